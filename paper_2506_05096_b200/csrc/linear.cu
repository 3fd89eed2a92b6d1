// astraea_gathered_linear: y[b, i, :] = x[b, i, :] W^T + bias for the listed token rows i = idx[b, r];
// the other rows of y keep the cached result (Algorithm 1 lines 4-7 applied to a linear layer of the
// block: the query projection of the selected tokens, the output projection and the MLP on selected
// rows; with idx == NULL the key / value projections of all tokens).
//
// A dense contraction, so it runs on the tcgen05 tensor cores.  Persistent CTA pairs (clusters of two, one CTA per SM)
// walk over 256-row x bn-column output tiles (column tiles of one row tile are neighbours in the walk, so the
// gathered rows stay in L2 while W, which is small, lives there anyway).  Both SMs of a pair work on one
// tcgen05.mma.cta_group::2 of 256 x bn x 16: each CTA holds 128 rows of A, half of the W tile and its 128 rows of the
// accumulator, so a W tile is read from shared memory once per pair instead of once per 128 rows, and the accumulator takes
// only half of a CTA's TMEM: there are two of them, and the epilogue of a tile runs under the main loop of the next.
// Warp roles of each CTA:
//   warps 0-15  epilogue: four threads per output row (every fourth group of 32 columns); TMEM -> registers -> (+ bias, GELU, gate,
//               residual) -> bf16 -> the row of y that idx names (fused scatter);
//   warp 16     TMA producer: this CTA's half of a W tile per stage (rows past N_out read as zero) and, when the rows
//               of x are a contiguous matrix (no list, or compact rows), the CTA's 128 rows of x as well; the bytes of both
//               CTAs are counted on the even one's barrier;
//   warp 17     even CTA: tcgen05.mma issuer for the pair, four MMAs per stage; odd CTA (listed rows only): passes on to the
//               even one that the gathered rows of a stage have landed;
//   warps 18-19 (listed rows only) gather of the A operand: the listed rows of x, 64 columns (128 bytes) per
//               pipeline stage, by 16-byte cp.async into the 128-byte-swizzled layout the MMA reads (rows past the end
//               and entries out of range are zero-filled); the copies arrive on the stage's barrier by themselves, so a
//               thread never waits for its own copies, only for a free stage.  (TMA gather4, one per lane and stage, was
//               measured at 331 us where this takes 119, 9001 x 3072 x 3072.)
// Layers of the same rows (the key and value projections; with SelectQ&K the query projection, too) share one launch: their column
// tiles follow one another, so that one partial round of tiles is paid instead of two or three, the rows of x are read once for all, and
// a launch is saved (7 us of set-up, first loads and last epilogue).  Keys and values of 4276 x 1536, four blocks (102 tiles on 74 pairs,
// eight times): 1070 -> 1047 us; of 32768 x 1152, the Open-Sora block: 1863 -> 1840; of 17776 x 3072, the CogVideoX block: 4469 -> 4434.
// Every mbarrier wait is bounded; on a timeout the CTA raises the error word, its remaining waits return at once, it sends
// for no further copy, the other CTA of the pair runs into its own limit, and both run out; they leave together, when the copies
// and MMAs that were under way have ended.
#include "common.cuh"
#include "linear_tiles.cuh"
#include "sm100_ptx.cuh"
#include "bounded_wait.cuh"

namespace astraea {
namespace {

using namespace ptx;

constexpr int kRowsCta = kBM / 2, kBK = 64;
constexpr int kAccSets = 2;                              // accumulators in TMEM: the epilogue runs under the next main loop
// Epilogue warps: four cover the CTA's 128 rows (one TMEM lane quarter each); kEpiSplit such groups share the columns.
// Four groups: a tile of a short contraction (K = 1152: 18 stages) is over in 5 us, and two groups take 6 us for its
// bias, GELU (erf), gate, residual and stores.
constexpr int kEpiSplit = 4;
constexpr int kEpiWarps = 4 * kEpiSplit, kGatherWarps = 2;
constexpr int kTmaWarp = kEpiWarps, kMmaWarp = kTmaWarp + 1, kFirstGatherWarp = kMmaWarp + 1;
constexpr int kEpiStageBytes = 32 * 64;                  // per epilogue warp: 32 rows x 32 bf16 columns on their way to / from global memory

constexpr int kStages = 6;
constexpr int kABytes = kRowsCta * kBK * 2, kBBytes = kMaxBN / 2 * kBK * 2;
constexpr int kBarBytes = 256;
static_assert(8 * (3 * kStages + 2 * kAccSets + 1) <= kBarBytes, "barrier area too small");
constexpr int kSmemBytes = kStages * (kABytes + kBBytes) + kBarBytes + kEpiWarps * kEpiStageBytes + 1024;
static_assert(kSmemBytes + 1536 <= 227 * 1024, "shared memory of one CTA");
constexpr int kMaxMats = 3;
constexpr uint32_t kAccCols = kMaxBN, kTmemCols = kAccSets * kAccCols;

struct LinParams {
    const __nv_bfloat16 *x;
    const int32_t *idx;
    int M;                       // rows listed per batch element (N when idx == nullptr)
    // Up to kMaxMats layers of the same rows in one launch: the column tiles run over the matrices one after the other, each
    // padded to mat_cols columns, a multiple of half a tile, so that each CTA's half of a W tile comes from one matrix.
    int n_mats, mat_cols;
    const __nv_bfloat16 *bias[kMaxMats];
    __nv_bfloat16 *y[kMaxMats];
    int B, N, K, N_out;
    int bn;                      // columns of an output tile
    uint32_t compact;            // bit i: y[i] is [B, M, N_out]
    int compact_in;              // x is [B, M, K]
    int gelu;                    // y = GELU(x W^T + bias), exact (erf) form
    const __nv_bfloat16 *residual;   // added to the result after the gate; [B, N, N_out] rows at idx, or compact [B, M, N_out]
    int res_compact;
    const __nv_bfloat16 *gate;       // [B, N_out]: multiplies act(x W^T + bias) before the residual is added
    int *err_word;
};

__device__ __forceinline__ void cp_async_16(uint32_t dst, const void *src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
// arrive on the mbarrier once every cp.async this thread has issued so far has landed (the arrival is one of
// those the barrier was initialised to expect)
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// GELU(x) = x (1 + erf(x / sqrt 2)) / 2 of two elements, with erf to 1.5e-7 absolute (rational approximation 7.1.26 of Abramowitz
// and Stegun: erf(z) = 1 - (a1 t + ... + a5 t^5) e^{-z^2} for z >= 0, t = 1 / (1 + p z)): with w = 1/2 + copysign(1/2 - (a1 t +
// ... + a5 t^5) e^{-z^2} / 2, z) it is x w.  Issue slots bind it (the epilogue of a tile has four warps on each SM sub-partition,
// and a main loop of K = 1152 is over in 5 us), so all but the XU operations and the signs are packed pairs: 10 instructions per
// element instead of 17.  z is rounded before it is squared and the halves only scale by powers of two, so the result is that of the
// same formula element by element, bit for bit (with 1 / sqrt 2 folded into the constants 9001 x 3072 x 12288 takes 488 us instead
// of 491, but outputs of a block move by single bf16 roundings; with |z| masked out of a packed product 493).  13106 x 1152 x 4608 took
// 110.0 us with the erf element by element and the epilogue's loads behind its wait, 101.6 now; 1846 x 1536 x 6144 32.2 -> 30.7.
__device__ __forceinline__ f32x2 both(float v) { return pack2(v, v); }
__device__ __forceinline__ f32x2 gelu2(f32x2 x) {
    float x0, x1, d0, d1, a0, a1, t0, t1, e0, e1;
    unpack2(x, x0, x1);
    const f32x2 az = pack2(__fmul_rn(fabsf(x0), 0.70710678118654752f), __fmul_rn(fabsf(x1), 0.70710678118654752f));     // |z|
    unpack2(fma2(az, both(0.3275911f), both(1.0f)), d0, d1);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t0) : "f"(d0));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t1) : "f"(d1));
    unpack2(mul2(mul2(az, az), both(-1.4426950408889634f)), a0, a1);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(a0));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(a1));
    const f32x2 t = pack2(t0, t1);
    f32x2 pl = fma2(both(-0.5f * 1.061405429f), t, both(0.5f * 1.453152027f));           // minus half the polynomial
    pl = fma2(pl, t, both(-0.5f * 1.421413741f));
    pl = fma2(pl, t, both(0.5f * 0.284496736f));
    pl = fma2(pl, t, both(-0.5f * 0.254829592f));
    const f32x2 half_erf = fma2(mul2(pl, t), pack2(e0, e1), both(0.5f));                // of |z|
    return mul2(x, add2(both(0.5f), (half_erf & 0x7fffffff7fffffffull) | (x & 0x8000000080000000ull)));
}

// A product that is rounded before anything is added to it, as the gate is before the residual: the product of packed pairs and the sum
// after it come out as one FMA even with .rn on both (same bits as fma2), a product of single elements does not.
__device__ __forceinline__ f32x2 mul2_alone(f32x2 a, f32x2 b) {
    float a0, a1, b0, b1;
    unpack2(a, a0, a1); unpack2(b, b0, b1);
    return pack2(__fmul_rn(a0, b0), __fmul_rn(a1, b1));
}

__device__ __forceinline__ uint4 shfl_vec(const uint4 &v, int lane) {
    return make_uint4(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane), __shfl_sync(0xffffffffu, v.z, lane),
                      __shfl_sync(0xffffffffu, v.w, lane));
}

// 2-D tiled load global -> this CTA's shared memory, completion counted in bytes on an mbarrier of either CTA of the pair
// (address from map_to_rank)
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *m, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(m), "r"(bar), "r"(c0), "r"(c1) : "memory");
}

// The g-th listed row (all batch elements in one list): its row of a [B, N, *] tensor, or -1 past the end of the list and for an
// index outside [0, N) or one that does not exceed its predecessor (*bad); *batch: the batch element.
__device__ __forceinline__ long long target_row(const LinParams &p, long long g, long long total, int *batch, bool *bad) {
    *bad = false;
    if (g >= total) return -1;
    const int b = (int)((unsigned)g / (unsigned)p.M), r = (int)((unsigned)g - (unsigned)b * (unsigned)p.M);   // fewer than 2^31 rows fit the device
    const int tok = p.idx ? __ldcg(p.idx + g) : r;
    const int before = (p.idx && r > 0) ? __ldcg(p.idx + g - 1) : -1;
    // not strictly ascending: a row would be written twice
    if ((unsigned)tok >= (unsigned)p.N || (r > 0 && before >= tok)) { *bad = true; return -1; }
    *batch = b;
    return (long long)b * p.N + tok;
}

// the matrix that column c of the launch belongs to (the last one for what is left of a last tile)
template <bool MULTI> __device__ __forceinline__ int mat_of(const LinParams &p, int c) {
    return MULTI ? min(c / p.mat_cols, p.n_mats - 1) : 0;
}

struct WMaps { CUtensorMap m[kMaxMats]; };

// What the epilogue does besides the bias, fixed at compile time for the plain layers and the GELU (with the tests inside its unrolled
// loops 1846 listed x 1536 x 1536 took 12.4 us where it takes 11.4, 13106 listed x 1152 x 1152 31.7 where 30.9).
enum { kNothing = 0, kGelu = 1, kAnything = 2 };

// DENSE: the rows of x are one contiguous matrix; MULTI: more than one layer (the registers of the listed form do not hold the
// choice between one and several)
template <bool DENSE> constexpr int kThreads = (kEpiWarps + 2 + (DENSE ? 0 : kGatherWarps)) * 32;

template <bool DENSE, bool MULTI, int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads<DENSE>, 1)
gathered_linear_kernel(const __grid_constant__ WMaps tmap_w, const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ LinParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ int stop;                                           // the stages that were sent for before the CTA gave up
    __shared__ int row_list[2][kRowsCta];                          // listed rows only: the rows of x of a tile

    // (both CTAs of a pair run the same kernel with the same static shared memory, so every offset below is the same in both)
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sA = smem_base, sB = sA + kStages * kABytes, bars = sB + kStages * kBBytes;
    const uint32_t bar_full = bars, bar_empty = bars + 8 * kStages, bar_peer = bars + 16 * kStages,
                   bar_acc_full = bars + 24 * kStages, bar_acc_empty = bar_acc_full + 8 * kAccSets,
                   bar_end = bar_acc_empty + 8 * kAccSets;

    const int tid = threadIdx.x;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);        // warp-uniform
    const int lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const long long total_rows = (long long)p.B * p.M;
    const int tiles_m = (int)((total_rows + kBM - 1) / kBM), tiles_n = ((MULTI ? p.n_mats * p.mat_cols : p.N_out) + p.bn - 1) / p.bn;
    const int total_tiles = tiles_m * tiles_n, k_steps = p.K / kBK;

    if (tid == 0) {
        abort_flag = 0;
        stop = 0x7fffffff;
        mbar_init(bar_end, 1);
        for (int s = 0; s < kStages; ++s) {
            // every gather thread + in the even CTA its TMA producer, for the bytes of both (odd CTA, contiguous rows: not used)
            mbar_init(bar_full + 8 * s, (DENSE ? 0 : kGatherWarps * 32) + (DENSE || rank == 0 ? 1 : 0));
            mbar_init(bar_empty + 8 * s, 1);                    // the issuer's commit
            mbar_init(bar_peer + 8 * s, 1);                     // even CTA: the odd CTA's gathered rows of the stage have landed
        }
        for (int a = 0; a < kAccSets; ++a) { mbar_init(bar_acc_full + 8 * a, 1); mbar_init(bar_acc_empty + 8 * a, 2 * kEpiWarps); }
        fence_barrier_init();
    }
    if (warp == kTmaWarp && elect_one()) { for (int i = 0; i < (MULTI ? p.n_mats : 1); ++i) prefetch_tensormap(&tmap_w.m[i]); if (DENSE) prefetch_tensormap(&tmap_x); }
    if (warp == kMmaWarp) {
        tmem_alloc_pair(smem_u32(&tmem_slot), kTmemCols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                            // the barriers of both CTAs are set up
    tc_fence_after();
    grid_dependency_wait();
    const uint32_t tmem = tmem_slot;

    if (warp < kEpiWarps) {
        // ------------------------------------------------ epilogue
        // TMEM lanes (rows of the CTA) by warp % 4; columns c0 + 32 (kEpiSplit j) .. + 31 of the tile by warp / 4
        const int part = warp >> 2;
        const int row = (int)rank * kRowsCta + (warp & 3) * 32 + lane;
        const int c0 = part * 32;
        const uint32_t t_row = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        uint8_t *stage = smem_raw + (bars + kBarBytes - smem_u32(smem_raw)) + warp * kEpiStageBytes;
        int it = 0;
        for (int tile = pair; tile < total_tiles; tile += n_pairs, ++it) {
            const int tm = tile / tiles_n, tn = tile - tm * tiles_n;
            const int acc = it % kAccSets;
            int batch = 0;
            bool bad;
            long long full_row = target_row(p, (long long)tm * kBM + row, total_rows, &batch, &bad);
            if (bad && tn == 0 && part == 0) atomicExch(p.err_word, kErrBadIndex);
            // What the epilogue reads is fetched while the main loop runs: behind the wait, each of the two groups of columns would pay
            // a round trip to L2 for its bias, and another one for the residual (rows x K x N_out 1846 x 1536 x 1536, a launch in a
            // chain: 12.24 -> 11.32 us; 2 x 6553 of 32768 x 1152 x 1152 34.3 -> 32.5; of 3.1 us from the last MMA to the last store).
            // The vectors that all rows share go round by shuffles: lanes 0-7 hold 8 columns of the bias each (0-3 of the first
            // group, 4-7 of the second), lanes 8-15 of the gate.
            const int q = lane & 3;
            const unsigned in_list = __ballot_sync(0xffffffffu, full_row >= 0);
            const int batch0 = __shfl_sync(0xffffffffu, batch, in_list ? __ffs(in_list) - 1 : 0);
            const bool one_batch = __all_sync(0xffffffffu, full_row < 0 || batch == batch0);       // (a gate belongs to a batch element)
            uint4 vec = make_uint4(0, 0, 0, 0);
            {
                const int c = c0 + ((lane >> 2) & 1) * (32 * kEpiSplit), mat = mat_of<MULTI>(p, tn * p.bn + c);
                const int col = tn * p.bn + c - mat * p.mat_cols + q * 8;
                const __nv_bfloat16 *src = lane < 8 ? p.bias[mat] : EPI == kAnything && lane < 16 && p.gate ? p.gate + (long long)batch0 * p.N_out : nullptr;
                if (src && c < p.bn && col < p.N_out) vec = ld_cached(reinterpret_cast<const uint4 *>(src + col));
            }
            uint4 rr[4];                                            // rows (lane >> 2) + 8 j of the residual, 8 columns each
            auto fetch_residual = [&](int colq) {
                const long long res_row = (full_row >= 0 && p.res_compact) ? (long long)tm * kBM + row : full_row;
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const long long rrow = __shfl_sync(0xffffffffu, res_row, (lane >> 2) + 8 * jj);
                    rr[jj] = (rrow >= 0 && colq < p.N_out) ? __ldcg(reinterpret_cast<const uint4 *>(p.residual + rrow * p.N_out + colq))
                                                           : make_uint4(0, 0, 0, 0);
                }
            };
            if (EPI == kAnything && p.residual && c0 < p.bn) fetch_residual(tn * p.bn + c0 + q * 8);
            wait_bar(bar_acc_full + 8 * acc, (it / kAccSets) & 1, &abort_flag, p.err_word);
            if (tile + n_pairs >= total_tiles) grid_launch_dependents();       // the last epilogue of this CTA
            tc_fence_after();
            if (abort_flag) full_row = -1;
            auto release = [&] {                                   // this warp's part of the accumulator has been read
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_rank(bar_acc_empty + 8 * acc, 0));
            };
            if (c0 >= p.bn) release();                             // narrow tiles: nothing for this group
            // Global memory is touched in a transposed layout: a thread owns a row of the accumulator, so a warp that
            // stored its rows directly would touch 32 lines per instruction, 16 bytes in each (measured: ~9 us of a
            // 36 us tile, 16 us with a residual).  Instead lane l moves the 16-byte piece l & 3 of rows (l >> 2) + 8 j:
            // 64 contiguous bytes per row, 8 rows per instruction, through 2 KB of shared memory per warp (pieces
            // swizzled by the row so that both directions are free of bank conflicts).
#pragma unroll 1
            for (int c = c0; c < p.bn; c += 32 * kEpiSplit) {
                const int mat = mat_of<MULTI>(p, tn * p.bn + c), n0 = tn * p.bn + c - mat * p.mat_cols;     // 32 columns of one matrix from n0
                const bool bias = p.bias[mat] != nullptr;
                const int first = c == c0 ? 0 : 4;                  // the lanes that hold this group's vectors
                __nv_bfloat16 *y = p.y[mat];
                // the row of a compact tensor is the row of the list
                const long long out_row = (full_row >= 0 && (p.compact >> mat & 1u)) ? (long long)tm * kBM + row : full_row;
                const int colq = n0 + q * 8;                        // the 8 columns this lane moves
                if (EPI == kAnything && p.residual) {
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        const int r = (lane >> 2) + 8 * jj;
                        *reinterpret_cast<uint4 *>(stage + r * 64 + ((q ^ ((r >> 1) & 3)) << 4)) = rr[jj];
                    }
                    __syncwarp();
                    if (c + 32 * kEpiSplit < p.bn) fetch_residual(colq + 32 * kEpiSplit);
                }
                uint32_t o[32];
                tmem_ld32(t_row + acc * kAccCols + c, o);
                tc_wait_ld();
                if (c + 32 * kEpiSplit >= p.bn) release();
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int col = n0 + v * 8;
                    uint4 *mine = reinterpret_cast<uint4 *>(stage + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4));     // residual in, result out
                    f32x2 f[4], t[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) f[i] = pack2(__uint_as_float(o[v * 8 + 2 * i]), __uint_as_float(o[v * 8 + 2 * i + 1]));
                    if (bias) {
                        unpack8(shfl_vec(vec, first + v), t);
#pragma unroll
                        for (int i = 0; i < 4; ++i) f[i] = add2(f[i], t[i]);
                    }
                    if (EPI == kGelu || (EPI == kAnything && p.gelu)) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) f[i] = gelu2(f[i]);
                    }
                    if (EPI == kAnything && p.gate) {
                        uint4 g = shfl_vec(vec, 8 + first + v);
                        if (!one_batch && col < p.N_out) g = ld_cached(reinterpret_cast<const uint4 *>(p.gate + (long long)batch * p.N_out + col));
                        unpack8(g, t);
                    }
                    if (EPI == kAnything && p.residual) {
                        f32x2 r[4];
                        unpack8(*mine, r);
#pragma unroll
                        for (int i = 0; i < 4; ++i) f[i] = add2(p.gate ? mul2_alone(f[i], t[i]) : f[i], r[i]);
                    } else if (EPI == kAnything && p.gate) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) f[i] = mul2(f[i], t[i]);
                    }
                    uint32_t w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float lo, hi;
                        unpack2(f[i], lo, hi);
                        __nv_bfloat162 v2 = __floats2bfloat162_rn(lo, hi);
                        w[i] = *reinterpret_cast<uint32_t *>(&v2);
                    }
                    *mine = make_uint4(w[0], w[1], w[2], w[3]);
                }
                __syncwarp();
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int r = (lane >> 2) + 8 * jj;
                    const long long orow = __shfl_sync(0xffffffffu, out_row, r);
                    const uint4 t = *reinterpret_cast<const uint4 *>(stage + r * 64 + ((q ^ ((r >> 1) & 3)) << 4));
                    if (orow >= 0 && colq < p.N_out) *reinterpret_cast<uint4 *>(y + orow * p.N_out + colq) = t;
                }
                __syncwarp();
            }
        }
    } else if (warp == kTmaWarp) {
        // ------------------------------------------------ TMA producer of the W tiles (and of contiguous rows of x)
        // (the odd CTA's bytes may arrive before the even one has said how many a stage gets: its phase cannot end before that)
        const uint32_t full0 = map_to_rank(bar_full, 0);
        auto gave_up = [&] { return *static_cast<volatile int *>(&abort_flag) != 0; };
        auto going = [&](int g) -> bool {                          // once the CTA has given up, stage g and those after it are not sent for
            if (gave_up()) stop = min(stop, g);
            return stop > g;
        };
        int g = 0;
        for (int tile = pair; tile < total_tiles; tile += n_pairs) {
            const int tm = tile / tiles_n, tn = tile - tm * tiles_n;
            const int col = tn * p.bn + (int)rank * (p.bn / 2), mat = mat_of<MULTI>(p, col);           // this CTA's half of the W tile
            for (int ks = 0; ks < k_steps; ++ks, ++g) {
                const int st = g % kStages;
                wait_bar(bar_empty + 8 * st, ((g / kStages) & 1) ^ 1, &abort_flag, p.err_word);
                if (elect_one() && going(g)) {
                    if (rank == 0) mbar_arrive_expect_tx(bar_full + 8 * st, 2 * (p.bn * kBK + (DENSE ? kABytes : 0)));
                    tma_load_2d(sB + st * kBBytes, &tmap_w.m[mat], full0 + 8 * st, ks * kBK, col - mat * p.mat_cols);
                    if (DENSE) tma_load_2d(sA + st * kABytes, &tmap_x, full0 + 8 * st, ks * kBK, tm * kBM + (int)rank * kRowsCta);
                }
                __syncwarp();
            }
        }
        // Every copy issued above must have landed before either CTA's shared memory is released.  (The odd CTA may be stages
        // ahead of one that gave up; the wait for one stage more, which does not come, outlasts them.)
        if (gave_up()) { __syncwarp(); g = min(g, stop) + 1; }
        for (int gs = (g > kStages ? g - kStages : 0); rank == 0 && gs < g; ++gs)
            drain_bar(bar_full + 8 * (gs % kStages), (gs / kStages) & 1);
    } else if (warp == kMmaWarp && rank == 0) {
        // ------------------------------------------------ MMA issuer of the pair
        const uint32_t idesc = idesc_bf16(kBM, p.bn, false);
        int g = 0, it = 0;
        for (int tile = pair; tile < total_tiles; tile += n_pairs, ++it) {
            const int acc = it % kAccSets;
            wait_bar<true>(bar_acc_empty + 8 * acc, ((it / kAccSets) & 1) ^ 1, &abort_flag, p.err_word);
            for (int ks = 0; ks < k_steps; ++ks, ++g) {
                const int st = g % kStages;
                wait_bar(bar_full + 8 * st, (g / kStages) & 1, &abort_flag, p.err_word);
                if (!DENSE) wait_bar<true>(bar_peer + 8 * st, (g / kStages) & 1, &abort_flag, p.err_word);
                fence_acquire_smem();                     // what landed in the odd CTA is in order before the MMAs too
                if (!DENSE) fence_proxy_async_smem();     // gathered rows were written through the generic proxy
                tc_fence_after();
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kBK / 16; ++kk)
                        mma_ss_pair(tmem + acc * kAccCols, smem_desc(sA + st * kABytes + kk * 32, 16, 1024, kSwizzle128B),
                                    smem_desc(sB + st * kBBytes + kk * 32, 16, 1024, kSwizzle128B), idesc, (ks > 0 || kk > 0) ? 1u : 0u);
                    tc_commit_pair(bar_empty + 8 * st);
                    if (ks == k_steps - 1) tc_commit_pair(bar_acc_full + 8 * acc);
                }
                __syncwarp();
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------ odd CTA: the gathered rows of a stage have landed
        const uint32_t peer0 = map_to_rank(bar_peer, 0);
        int g = 0;
        for (int tile = pair; !DENSE && tile < total_tiles; tile += n_pairs)
            for (int ks = 0; ks < k_steps; ++ks, ++g) {
                const int st = g % kStages;
                wait_bar(bar_full + 8 * st, (g / kStages) & 1, &abort_flag, p.err_word);
                fence_proxy_async_smem();                 // gathered rows were written through the generic proxy
                fence_release_smem();
                if (elect_one()) mbar_arrive_cluster(peer0 + 8 * st);
                __syncwarp();
            }
    } else if constexpr (!DENSE) {
        // ------------------------------------------------ gather of the A rows (cp.async, 128-byte swizzle)
        constexpr int kGatherThreads = kGatherWarps * 32, kRowStep = kGatherThreads / 8, kRowsThread = kRowsCta / kRowStep;
        static_assert(kRowStep % 8 == 0, "a row step keeps the swizzle phase of the thread's rows");
        const int t = tid - kFirstGatherWarp * 32;
        const int chunk = t & 7, row0 = t >> 3;               // this thread: 16-byte chunk `chunk` of rows row0 + kRowStep i
        const uint32_t off = row0 * 128 + ((chunk ^ (row0 & 7)) << 4);
        // The list entries of the next tile are fetched while this one is streamed (fetched where they are needed, two
        // dependent loads for each of a thread's rows, they cost 4-11 us a tile), each by one thread, and go round
        // through shared memory.
        constexpr int kEnt = kRowsCta / kGatherThreads;
        int ent[kEnt];
        auto fetch = [&](int tile) {
#pragma unroll
            for (int i = 0; i < kEnt; ++i) {
                const long long r = (long long)(tile / tiles_n) * kBM + (int)rank * kRowsCta + t + i * kGatherThreads;
                ent[i] = (tile < total_tiles && r < total_rows) ? __ldcg(p.idx + r) : -1;
            }
        };
        fetch(pair);
        int g = 0, it = 0;                                    // running stage and tile counts
        for (int tile = pair; tile < total_tiles; tile += n_pairs, ++it) {
            const int tm = tile / tiles_n;
            int *list = row_list[it & 1];
#pragma unroll
            for (int i = 0; i < kEnt; ++i) {
                // rows of 128 bytes or more: their number is below 2^31
                const unsigned r = (unsigned)tm * kBM + rank * kRowsCta + t + i * kGatherThreads;
                list[t + i * kGatherThreads] = (unsigned)ent[i] < (unsigned)p.N ? (int)(r / (unsigned)p.M * (unsigned)p.N) + ent[i] : -1;
            }
            fetch(tile + n_pairs);
            asm volatile("bar.sync 1, %0;" ::"n"(kGatherThreads) : "memory");      // two lists: one barrier per tile is enough
            int src[kRowsThread];
#pragma unroll
            for (int i = 0; i < kRowsThread; ++i) src[i] = list[row0 + kRowStep * i];
            const __nv_bfloat16 *xc = p.x + chunk * 8;
            for (int ks = 0; ks < k_steps; ++ks, ++g, xc += kBK) {
                const int st = g % kStages;
                wait_bar(bar_empty + 8 * st, ((g / kStages) & 1) ^ 1, &abort_flag, p.err_word);
#pragma unroll
                for (int i = 0; i < kRowsThread; ++i)
                    cp_async_16(sA + st * kABytes + off + i * (kRowStep * 128), xc + (size_t)(unsigned)max(src[i], 0) * (unsigned)p.K, src[i] >= 0);
                cp_async_arrive(bar_full + 8 * st);           // asynchronous: the thread goes on to the next free stage
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }

    // neither CTA leaves (or gives up its TMEM) while the other may still arrive on its barriers or read its shared memory
    tc_fence_before();
    __syncthreads();
    if (abort_flag && rank == 0 && warp == kMmaWarp) {             // MMAs that are under way end before their memory is given up
        if (elect_one()) { tc_commit_pair(bar_end); drain_bar(bar_end, 0); }
        __syncwarp();
    }
    cluster_sync_all();
    if (warp == kMmaWarp) tmem_dealloc_pair(tmem, kTmemCols);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// a row-major bf16 matrix [rows, K] with 128-byte-swizzled boxes of 64 columns x box_rows
int32_t make_matrix_map(CUtensorMap *map, const void *base, long long rows, int K, int box_rows, const char *what)
{
    const EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(tensor_map_encoder());
    if (!enc) return fail(ASTRAEA_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ASTRAEA_ERR_INVALID_ARG, "astraea_gathered_linear: tensor map of %s rejected (CUresult %d)", what, (int)r);
    return ASTRAEA_OK;
}

template <bool DENSE, bool MULTI, int EPI>
int32_t launch_linear(const LinParams &p, const void *x, const LinearLayer *layers, int pairs, cudaStream_t stream)
{
    WMaps mw;
    CUtensorMap mx;
    int32_t rc = ASTRAEA_OK;
    for (int i = 0; i < p.n_mats && rc == ASTRAEA_OK; ++i) rc = make_matrix_map(&mw.m[i], layers[i].w, p.N_out, p.K, p.bn / 2, "W");
    if (rc != ASTRAEA_OK) return rc;
    for (int i = p.n_mats; i < kMaxMats; ++i) mw.m[i] = mw.m[0];
    mx = mw.m[0];
    if (DENSE) rc = make_matrix_map(&mx, x, (long long)p.B * p.M, p.K, kRowsCta, "x");
    if (rc != ASTRAEA_OK) return rc;
    static PerDeviceOnce attrs;                   // the attribute is per device
    if (attrs.run([] { return cudaFuncSetAttribute(gathered_linear_kernel<DENSE, MULTI, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes); }) != cudaSuccess)
        return check_launch("astraea_gathered_linear (shared memory attribute)");
    const long long tiles = (((long long)p.B * p.M + kBM - 1) / kBM) * column_tiles(p.N_out, p.n_mats, p.bn);
    const int grid = 2 * (int)(tiles < pairs ? tiles : pairs);
    launch_overlapped(gathered_linear_kernel<DENSE, MULTI, EPI>, grid, kThreads<DENSE>, kSmemBytes, stream, mw, mx, p);
    return check_launch("astraea_gathered_linear");
}

}  // namespace

size_t linear_workspace_bytes() { return 256; }

int32_t launch_gathered_linear(const void *x, const int32_t *idx, int M, const LinearLayer *layers, int n_layers,
                               int B, int N, int K, int N_out, uint32_t flags, int *err_word, cudaStream_t stream,
                               const void *residual, const void *gate)
{
    LinParams p = {};
    p.x = reinterpret_cast<const __nv_bfloat16 *>(x);
    p.idx = idx;
    p.M = idx ? M : N;
    p.B = B; p.N = N; p.K = K; p.N_out = N_out;
    p.compact_in = (flags & ASTRAEA_LINEAR_COMPACT_IN) ? 1 : 0;
    p.gelu = (flags & ASTRAEA_LINEAR_GELU) ? 1 : 0;
    p.residual = reinterpret_cast<const __nv_bfloat16 *>(residual);
    p.res_compact = (flags & ASTRAEA_LINEAR_COMPACT_RES) ? 1 : 0;
    p.gate = reinterpret_cast<const __nv_bfloat16 *>(gate);
    p.err_word = err_word;
    const int pairs = sm_count() / 2 > 0 ? sm_count() / 2 : 1;
    p.n_mats = n_layers;
    p.bn = choose_bn((long long)B * p.M, N_out, n_layers, pairs);
    p.mat_cols = mat_columns(N_out, n_layers, p.bn);
    for (int i = 0; i < n_layers; ++i) {
        p.bias[i] = reinterpret_cast<const __nv_bfloat16 *>(layers[i].bias);
        p.y[i] = reinterpret_cast<__nv_bfloat16 *>(layers[i].y);
        if (layers[i].compact_out) p.compact |= 1u << i;
    }
    const bool dense = !idx || p.compact_in;
#define LAUNCH(MULTI, EPI) (dense ? launch_linear<true, MULTI, EPI>(p, x, layers, pairs, stream) : launch_linear<false, MULTI, EPI>(p, x, layers, pairs, stream))
    if (n_layers > 1) return LAUNCH(true, kNothing);
    if (!p.gelu && !p.residual && !p.gate) return LAUNCH(false, kNothing);
    if (p.gelu && !p.residual && !p.gate) return LAUNCH(false, kGelu);
    return LAUNCH(false, kAnything);
#undef LAUNCH
}

}  // namespace astraea
