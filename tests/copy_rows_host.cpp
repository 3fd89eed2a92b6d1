// The copying warp of the attention kernel, run on the host: 32 threads are its lanes, the primitives below a model of the
// device's (a load lands when its phase is waited for, the shared memory is an array, a warp-wide operation is a barrier that
// reports lanes that never come).
//
//   copy_rows_host rows tokens bytes blocks give_up
//
// give_up: number of the wait that runs out (-1: none).  It runs out while half of the lanes have passed it already.
// Exit code 0: every lane returned, no load was left in flight, and (no give-up) the rows were copied; 2: lanes parted.
#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

#define __device__
#define __forceinline__ inline
using std::max;
using std::min;
struct Dim { int x; };
static thread_local Dim threadIdx;
static Dim blockIdx, gridDim;

namespace model {
std::mutex mu;
std::condition_variable cv;
int here = 0, round_ = 0, waits[32], give_up = -1, next_vote = 0, vote = 0;
volatile int abort_flag = 0;
struct Load { uint32_t dst; const void *src; uint32_t bytes; };
std::map<uint32_t, std::vector<Load>> pending;          // by barrier
std::map<uint32_t, long long> expected;
std::vector<char> smem(1 << 16);

int meet(int bits) {                                     // all 32 lanes; returns the votes of this round
    std::unique_lock<std::mutex> lock(mu);
    const int mine = round_;
    next_vote |= bits;
    if (++here == 32) { vote = next_vote; next_vote = 0; here = 0; ++round_; cv.notify_all(); return vote; }
    cv.notify_all();
    if (!cv.wait_for(lock, std::chrono::seconds(5), [&] { return round_ != mine; })) { puts("lanes parted"); fflush(stdout); _Exit(2); }
    return vote;
}
void land(uint32_t bar) {                                // a phase is over when the bytes that it expects have been sent for
    std::unique_lock<std::mutex> lock(mu);
    auto &v = pending[bar];
    auto sent = [&] { long long n = 0; for (auto &l : v) n += l.bytes; return n; };
    if (!cv.wait_for(lock, std::chrono::seconds(5), [&] { return sent() == expected[bar]; })) { puts("bytes expected and loaded differ"); fflush(stdout); _Exit(3); }
    for (auto &l : v) memcpy(&smem[l.dst], l.src, l.bytes);
    v.clear();
    expected[bar] = 0;
}
}  // namespace model

static int __ldcg(const int *p) { return *p; }
static int __popc(unsigned v) { return __builtin_popcount(v); }
static unsigned __ballot_sync(unsigned, bool b) { return (unsigned)model::meet(b ? 1 << threadIdx.x : 0); }
static bool __any_sync(unsigned, bool b) { return model::meet(b ? 1 << threadIdx.x : 0) != 0; }
static void __syncwarp() { model::meet(0); }
static void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) { std::lock_guard<std::mutex> l(model::mu); model::expected[bar] = bytes; }
struct uint4 { uint32_t x, y, z, w; };
static void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    std::lock_guard<std::mutex> l(model::mu);
    if (dst % 16 || (uintptr_t)src % 16 || bytes % 16) { puts("misaligned copy"); fflush(stdout); _Exit(4); }
    model::pending[bar].push_back({dst, src, bytes});
    model::cv.notify_all();
}
static void bulk_store(void *dst, uint32_t src, uint32_t bytes) { std::lock_guard<std::mutex> l(model::mu); memcpy(dst, &model::smem[src], bytes); }
static void bulk_commit() {}
template <int N> static void bulk_wait_read() {}
template <int N> static void bulk_wait() {}
static void drain_bar(uint32_t bar, uint32_t) { model::land(bar); }
static void wait_bar(uint32_t bar, uint32_t, volatile int *abort_flag, int *) {
    const int lane = threadIdx.x, n = model::waits[lane]++;
    if (model::give_up < 0 || n < model::give_up) { model::land(bar); return; }
    if (*abort_flag || lane < 16) return;                // (the first half found the phase complete)
    std::unique_lock<std::mutex> lock(model::mu);        // the other half gives up once the first is on its way
    model::cv.wait_for(lock, std::chrono::seconds(1), [&] { return model::here >= 16 || model::abort_flag; });
    *abort_flag = 1;
}

#include "copy_rows.cuh"

struct Params {
    int copy_rows, M, N_tok;
    uint32_t copy_bytes;
    const int *q_idx;
    const uint4 *copy_src;
    uint4 *copy_dst;
    int *err_word;
};
struct Cfg { static constexpr int kCopyStages = STAGES, kCopyStageBytes = 4096; };

int main(int, char **argv) {
    const int rows = atoi(argv[1]), tokens = atoi(argv[2]), bytes = atoi(argv[3]), blocks = atoi(argv[4]);
    model::give_up = atoi(argv[5]);
    std::vector<int> idx(rows);
    for (int r = 0; r < rows; ++r) idx[r] = (int)((long long)r * tokens / rows);
    std::vector<uint4> src((size_t)tokens * bytes / 16), dst(src.size());
    for (size_t i = 0; i < src.size(); ++i) src[i] = {(uint32_t)i * 2654435761u, (uint32_t)i, 7u, 9u};
    Params p{rows, rows, tokens, (uint32_t)bytes, idx.data(), src.data(), dst.data(), nullptr};
    gridDim.x = blocks;
    for (blockIdx.x = 0; blockIdx.x < blocks; ++blockIdx.x) {
        model::abort_flag = 0;
        memset(model::waits, 0, sizeof(model::waits));
        std::vector<std::thread> lanes;
        for (int l = 0; l < 32; ++l) lanes.emplace_back([&, l] { threadIdx.x = l; copy_role<Cfg>(p, 0u, 1u << 20, &model::abort_flag); });
        for (auto &t : lanes) t.join();
        for (auto &v : model::pending) if (!v.second.empty()) { puts("a load is left in flight"); return 1; }
    }
    if (model::give_up >= 0) return 0;
    std::vector<char> listed(tokens, 0);
    for (int t : idx) listed[t] = 1;
    const std::vector<uint4> zero(bytes / 16);
    for (int t = 0; t < tokens; ++t)
        if (memcmp(&dst[(size_t)t * bytes / 16], listed[t] ? &src[(size_t)t * bytes / 16] : zero.data(), bytes)) { printf("row %d is wrong\n", t); return 1; }
    return 0;
}
