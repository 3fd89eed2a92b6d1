// Host-buffer sessions (astraea_step_host, csrc/api.cu) on a model of the CUDA runtime: a stream is a queue whose entries run in
// any order that streams and events allow (drawn from a seed) and not before somebody waits for them, device memory is host memory, and the
// kernels are stand-ins on whole numbers.  An output that was overtaken by a copy, a copy that a failed step leaves behind, or a copy
// that has to wait for the host shows here; no GPU is needed.
//
//   session_host steps B H d N_sel n_always shared seeds    dense, sparse, dense, sparse; shared: x_cur and out are one buffer
//   session_host fail  B H d N_sel n_always k_keep first    every call of a step fails once: the first step, or (0) the third
//   session_host modes B H d N_sel n_always                 steps with unknown modes
//
// Exit code 0, or 1 with the reason on standard output.  `steps` prints of the first dense step: copies in, copies back, copies
// in behind the first copy back, then the CTAs (256 query rows of a head) of every attention launch.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <memory>
#include <random>
#include <vector>

#define __device__
#define __forceinline__ inline
#define __global__
struct uint4 { uint32_t x, y, z, w; };
static float __uint_as_float(uint32_t) { return 0; }
struct dim3 { unsigned x = 1, y = 1, z = 1; };
enum cudaError_t { cudaSuccess = 0, cudaErrorUnknown = 999 };
enum cudaMemcpyKind { cudaMemcpyHostToDevice, cudaMemcpyDeviceToHost, cudaMemcpyDeviceToDevice };
enum { cudaStreamNonBlocking = 1, cudaEventDisableTiming = 2, cudaMemoryTypeHost = 1, cudaDevAttrMultiProcessorCount = 16, cudaEnableDefault = 0,
       cudaStreamCaptureModeThreadLocal = 1, cudaLaunchAttributeProgrammaticStreamSerialization = 6 };
enum cudaDriverEntryPointQueryResult { cudaDriverEntryPointSuccess, cudaDriverEntryPointSymbolNotFound };
struct cudaPointerAttributes { int type; void *devicePointer; };
struct cudaLaunchAttribute { int id; struct { int programmaticStreamSerializationAllowed; } val; };

namespace model {
struct Entry { std::function<bool()> ready; std::function<void()> run; };
struct Stream { std::deque<Entry> queue; };
struct Event { std::shared_ptr<bool> done = std::make_shared<bool>(true); };
std::vector<Stream *> streams;
std::mt19937 rng;
int calls = 0, fail_at = -1, copies_in = 0, copies_back = 0, copies_late = 0;
std::vector<int> attn_ctas;

void die(const char *why) { puts(why); exit(1); }
bool fails() { return calls++ == fail_at; }
void put(Stream *s, std::function<void()> run, std::function<bool()> ready = [] { return true; }) { s->queue.push_back({ready, run}); }
void wait_for(Stream *s) {
    while (!s->queue.empty()) {
        std::vector<Stream *> can;
        for (Stream *t : streams) if (!t->queue.empty() && t->queue.front().ready()) can.push_back(t);
        if (can.empty()) die("no stream can go on");
        Stream *t = can[rng() % can.size()];
        Entry e = t->queue.front();
        t->queue.pop_front();
        e.run();
    }
}
}  // namespace model
typedef model::Stream *cudaStream_t;
typedef model::Event *cudaEvent_t;
typedef void *cudaGraph_t, *cudaGraphExec_t;
struct cudaLaunchConfig_t { dim3 gridDim, blockDim; size_t dynamicSmemBytes; cudaStream_t stream; cudaLaunchAttribute *attrs; int numAttrs; };
template <class... A> cudaError_t cudaLaunchKernelEx(A...) { return cudaErrorUnknown; }

#define CALL() do { if (model::fails()) return cudaErrorUnknown; } while (0)
static const char *cudaGetErrorString(cudaError_t) { return "failed by the test"; }
static cudaError_t cudaGetLastError() { return cudaSuccess; }
static cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
static cudaError_t cudaDeviceGetAttribute(int *v, int, int) { *v = 148; return cudaSuccess; }
static cudaError_t cudaGetDriverEntryPoint(const char *, void **, int, cudaDriverEntryPointQueryResult *) { return cudaErrorUnknown; }
template <class T> cudaError_t cudaMalloc(T **p, size_t n) { *p = static_cast<T *>(malloc(n)); memset((void *)*p, 0xa5, n); return cudaSuccess; }
static cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
static cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = new model::Stream; model::streams.push_back(*s); return cudaSuccess; }
static cudaError_t cudaStreamDestroy(cudaStream_t s) {
    model::streams.erase(std::find(model::streams.begin(), model::streams.end(), s));
    delete s;
    return cudaSuccess;
}
static cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = new model::Event; return cudaSuccess; }
static cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; return cudaSuccess; }
static cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    CALL();
    auto done = std::make_shared<bool>(false);
    e->done = done;
    model::put(s, [done] { *done = true; });
    return cudaSuccess;
}
static cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    CALL();
    auto done = e->done;
    model::put(s, [] {}, [done] { return *done; });
    return cudaSuccess;
}
static cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (s) model::wait_for(s);
    CALL();
    return cudaSuccess;
}
static void count(cudaMemcpyKind kind) {
    model::copies_in += kind == cudaMemcpyHostToDevice;
    model::copies_back += kind == cudaMemcpyDeviceToHost;
    model::copies_late += kind == cudaMemcpyHostToDevice && model::copies_back > 0;
}
static cudaError_t cudaMemcpy2DAsync(void *dst, size_t dp, const void *src, size_t sp, size_t width, size_t rows, cudaMemcpyKind kind, cudaStream_t s) {
    CALL();
    count(kind);
    model::put(s, [=] { for (size_t r = 0; r < rows; ++r) memcpy((char *)dst + r * dp, (const char *)src + r * sp, width); });
    return cudaSuccess;
}
static cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t s) {
    CALL();
    count(kind);
    model::put(s, [=] { memcpy(dst, src, n); });
    return cudaSuccess;
}
static cudaError_t cudaMemsetAsync(void *dst, int v, size_t n, cudaStream_t s) { CALL(); model::put(s, [=] { memset(dst, v, n); }); return cudaSuccess; }
static cudaError_t cudaMemset(void *dst, int v, size_t n) { memset(dst, v, n); return cudaSuccess; }
static cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind) { memcpy(dst, src, n); return cudaSuccess; }
static cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) { a->type = cudaMemoryTypeHost; a->devicePointer = (void *)p; return cudaSuccess; }
static cudaError_t cudaStreamBeginCapture(cudaStream_t, int) { return cudaErrorUnknown; }
static cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorUnknown; }
static cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, int) { return cudaErrorUnknown; }
static cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorUnknown; }
static cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
static cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

#include "api.cu"

// ------------------------------------------------------------------ stand-ins for the kernels
namespace astraea {
#define LAUNCH() do { if (model::fails()) return ASTRAEA_ERR_CUDA; } while (0)
int32_t launch_score(const void *, const void *, const float *, const int32_t *, float *, int, int, int, int, int, float, float, int, int, cudaStream_t s, float *) {
    LAUNCH();
    model::put(s, [] {});
    return ASTRAEA_OK;
}
// the first k tokens and the always-kept ones
int32_t launch_select(const float *, int B, int N_sel, int k, int n_always, int32_t *sel, int32_t *, int32_t *n_skip, void *, cudaStream_t s) {
    LAUNCH();
    model::put(s, [=] {
        for (int b = 0; b < B; ++b) {
            for (int i = 0; i < k; ++i) sel[b * (k + n_always) + i] = i;
            for (int i = 0; i < n_always; ++i) sel[b * (k + n_always) + k + i] = N_sel + i;
            for (int i = 0; i < N_sel; ++i) n_skip[b * N_sel + i] = i < k ? 0 : n_skip[b * N_sel + i] + 1;
        }
    });
    return ASTRAEA_OK;
}
int32_t launch_scatter(void *cache, const void *rows, const int32_t *idx, int B, int N, int M, int elems, uint32_t, int *, cudaStream_t s, int pitch) {
    LAUNCH();
    const size_t p = pitch ? pitch : elems;
    model::put(s, [=] {
        for (int b = 0; b < B; ++b)
            for (int m = 0; m < M; ++m) {
                const size_t at = ((size_t)b * N + idx[b * M + m]) * p * 2;
                memcpy((char *)cache + at, (const char *)rows + at, (size_t)elems * 2);
            }
    });
    return ASTRAEA_OK;
}
// every output depends on its query and on all keys and values of its head
static uint16_t fold(const uint16_t *k, const uint16_t *v, int N, int d, int64_t sn) {
    uint16_t f = 0;
    for (int n = 0; n < N; ++n)
        for (int c = 0; c < d; ++c) f = (uint16_t)(f * 3 + k[n * sn + c] * 5 + v[n * sn + c]);
    return f;
}
int32_t launch_sparse_attn(const AttnArgs &a, cudaStream_t s) {
    LAUNCH();
    const int heads = a.head_count > 0 ? a.head_count : a.H;
    model::attn_ctas.push_back(a.B * heads * ((a.M + 255) / 256));
    model::put(s, [=] {
        const uint16_t *q = (const uint16_t *)a.q, *k = (const uint16_t *)a.k, *v = (const uint16_t *)a.v;
        for (int b = 0; b < a.B; ++b)
            for (int h = a.head_begin; h < a.head_begin + heads; ++h) {
                const uint16_t f = fold(k + b * a.k_sb + h * a.k_sh, v + b * a.v_sb + h * a.v_sh, a.N, a.d, a.k_sn);
                for (int m = 0; m < a.M; ++m) {
                    const int tok = a.q_idx ? a.q_idx[b * a.M + m] : m;
                    const uint16_t *row = q + b * a.q_sb + tok * a.q_sn + h * a.q_sh;
                    uint16_t *out = (uint16_t *)a.out + ((size_t)(b * a.N_tok + tok) * a.H + h) * a.d;
                    for (int c = 0; c < a.d; ++c) out[c] = (uint16_t)(row[c] * 7 + f);
                    a.lse_out[((size_t)b * a.H + h) * a.N_tok + tok] = out[0];
                }
            }
    });
    return ASTRAEA_OK;
}
size_t select_workspace_bytes(int, int) { return 256; }
size_t linear_workspace_bytes() { return 256; }
size_t attn_workspace_bytes(int, int, int, int, int) { return 256; }
size_t attn_kv_workspace_bytes(int, int, int, int) { return 256; }
void attn_plan(const AttnArgs &, int *, int *, int *) {}
int32_t launch_score_combine(const float *, const int32_t *, float *, int, int, int, int, int, float, float, cudaStream_t) { return ASTRAEA_ERR_CUDA; }
int32_t launch_gathered_linear(const void *, const int32_t *, int, const LinearLayer *, int, int, int, int, int, uint32_t, int *, cudaStream_t, const void *, const void *) { return ASTRAEA_ERR_CUDA; }
int32_t launch_layernorm_modulate(const void *, const int32_t *, int, const void *, const void *, void *, int, int, int, float, uint32_t, int *, cudaStream_t) { return ASTRAEA_ERR_CUDA; }
int32_t launch_wait_selftest(int *, uint64_t, int *, cudaStream_t) { return ASTRAEA_ERR_CUDA; }
int32_t launch_sparse_attn_kv(AttnArgs, const int32_t *, int, void *, cudaStream_t) { return ASTRAEA_ERR_CUDA; }
int32_t noalloc_scratch_address(void **) { return ASTRAEA_ERR_CUDA; }
}  // namespace astraea

// ------------------------------------------------------------------ the checks
struct Run {
    int B, H, d, N_sel, n_always, N, D;
    astraea_session *s = nullptr;
    std::vector<uint16_t> x, q, k, v, out, want, want_ref;
    std::vector<int> skip;
    std::mt19937 values{7};

    explicit Run(char **a) : B(atoi(a[0])), H(atoi(a[1])), d(atoi(a[2])), N_sel(atoi(a[3])), n_always(atoi(a[4])), N(N_sel + n_always), D(H * d) {
        if (astraea_session_create(&s, B, H, N, N_sel, d) != ASTRAEA_OK) model::die("no session");
        for (auto *t : {&x, &q, &k, &v, &out, &want, &want_ref}) t->resize((size_t)B * N * D);
        skip.assign((size_t)B * N_sel, 0);
    }
    ~Run() { astraea_session_destroy(s); }
    int32_t step(int k_keep, bool shared, int delta_mode = 0, int lse_mode = 0) {
        for (auto *t : {&x, &q, &k, &v}) for (auto &e : *t) e = (uint16_t)values();
        std::vector<uint16_t> x0 = x;
        for (int b = 0; b < B; ++b)
            for (int n = 0; n < N; ++n) {
                const bool sel = n < k_keep || n >= N_sel;
                if (n < N_sel) skip[b * N_sel + n] = sel ? 0 : skip[b * N_sel + n] + 1;
                if (sel) memcpy(&want_ref[((size_t)b * N + n) * D], &x0[((size_t)b * N + n) * D], (size_t)D * 2);
            }
        for (int b = 0; b < B; ++b)
            for (int h = 0; h < H; ++h) {
                const size_t base = (size_t)b * N * D + (size_t)h * d;
                const uint16_t f = astraea::fold(&k[base], &v[base], N, d, D);
                for (int n = 0; n < N; ++n)
                    if (n < k_keep || n >= N_sel)
                        for (int c = 0; c < d; ++c) want[base + (size_t)n * D + c] = (uint16_t)(q[base + (size_t)n * D + c] * 7 + f);
            }
        uint16_t *to = shared ? x.data() : out.data();
        const int32_t rc = astraea_step_host(s, x.data(), q.data(), k.data(), v.data(), to, k_keep, 1.f, 1.f, delta_mode, lse_mode);
        for (auto *t : model::streams) if (!t->queue.empty()) model::die("the call returned with work under way");
        if (shared) out = x;
        return rc;
    }
    void check() {
        if (out != want) model::die("outputs differ");
        if (memcmp(s->x_ref, want_ref.data(), want_ref.size() * 2)) model::die("reference inputs differ");
        if (memcmp(s->n_skip, skip.data(), skip.size() * 4)) model::die("skip counters differ");
    }
};

int main(int argc, char **argv)
{
    if (argc < 7) return 2;
    char **sizes = argv + 2;
    const int N_sel = atoi(sizes[3]);
    if (!strcmp(argv[1], "steps")) {
        for (int seed = 0; seed < atoi(argv[8]); ++seed) {
            Run run(sizes);
            model::rng.seed(seed);
            model::copies_in = model::copies_back = model::copies_late = 0;
            model::attn_ctas.clear();
            for (int i = 0; i < 4; ++i) {
                if (run.step(i % 2 ? N_sel / 3 : N_sel, atoi(argv[7]) != 0) != ASTRAEA_OK) model::die("a step failed");
                run.check();
                if (seed == 0 && i == 0) {
                    printf("%d %d %d", model::copies_in, model::copies_back, model::copies_late);
                    for (int c : model::attn_ctas) printf(" %d", c);
                    puts("");
                }
            }
        }
    } else if (!strcmp(argv[1], "fail")) {
        for (int at = 0;; ++at) {
            Run run(sizes);
            model::rng.seed(at);
            if (!atoi(argv[8])) { run.step(N_sel, false); run.step(N_sel / 2, false); }
            model::calls = 0;
            model::fail_at = at;
            const int32_t rc = run.step(atoi(argv[7]), false);
            model::fail_at = -1;
            if (at >= model::calls) { if (at < 10) model::die("hardly a call"); break; }       // a step without a failure
            if (rc != ASTRAEA_ERR_CUDA) model::die("a failed call was not reported");
        }
    } else {
        Run run(sizes);
        model::calls = 0;
        for (int i = 0; i < 2; ++i) {                                                            // the first step, and one behind it
            for (int delta : {-1, 3, 7}) if (run.step(N_sel, false, delta, 0) != ASTRAEA_ERR_UNSUPPORTED) model::die("an unknown delta_mode was taken");
            for (int lse : {-1, 2}) if (run.step(N_sel, false, 0, lse) != ASTRAEA_ERR_UNSUPPORTED) model::die("an unknown lse_mode was taken");
            if (i == 0 && model::calls != 0) model::die("something was sent for before the modes were looked at");
            if (run.step(N_sel, false) != ASTRAEA_OK) model::die("a step failed");
        }
    }
    return 0;
}
