// astraea_layernorm_modulate: y[r, :] = LayerNorm(x[r, :]) * (1 + scale[b, :]) + shift[b, :] for the listed token rows
// (Section 3.2: the layers of a compute block other than self-attention act on every token by itself, so the
// element-wise step in front of them runs for the selected tokens only; in front of the key / value projections it
// runs for all tokens).
//
// HBM-bound: every row is read once and written once.  One warp owns one row and keeps it packed in registers (16-byte
// loads, all in flight at once), takes mean and variance from the registers in one pass over shifted data, then
// normalises, modulates and stores in a second pass over the registers.  fp32 arithmetic, one rounding to bf16 at the end.
// Next to the bytes the issue slots bind it: element by element it is ~105 instructions per 16-byte vector, so the
// arithmetic is on packed fp32 pairs, and the register array has five and six vectors too, the widths of 1152 and 1536
// channels (32768 x 1152 36.4 -> 29.1 us, 17776 x 3072 44.7 -> 40.6, 4276 x 1536 7.8 -> 5.5), and whether there are modulation
// vectors is fixed at compile time (modulated now 26.5, 38.6 = 5.7 TB/s, 4.7).
// Four warps a block rather than eight even out short launches and are worth 2-5 % of the long ones; two rows a warp,
// sharing the unpacked modulation vectors, gain nothing.
#include "common.cuh"

namespace astraea {
namespace {

constexpr int kWarpsPerBlock = 4;
constexpr int kBlocksPerSM = 16;
constexpr int kMaxVecPerLane = 16;     // rows of up to 32 * 16 * 8 = 4096 channels

// What the launch knows of the modulation vectors, fixed when the kernel is compiled: with the tests inside the loop over a row's
// registers a plain norm took 20.7 us where it takes 15.6 now (9001 x 3072), a modulated one 24.1 (20.7 now); 32768 x 1152 27.5 ->
// 22.7 and 29.5 -> 26.5, 1846 x 1536 4.5 -> 3.5 and 5.2 -> 3.5.
enum { kPlain = 0,      // there are none
       kBoth = 1,       // both are there, read from L1 for every row
       kHeld = 2,       // both are there, each warp keeps its lane's part of them in registers: fewer blocks of an SM
       kEither = 3 };   // one of them (or both, see kTestedRows10)
template <int VPL, int MOD> constexpr int kBlocks = MOD == kHeld ? (VPL <= 2 ? 8 : VPL <= 5 ? 5 : VPL <= 6 ? 4 : VPL <= 12 ? 3 : 2)
                                                                 : VPL <= 6 ? 8 : VPL <= 8 ? 6 : 4;

// Ten times the rows a warp (of the blocks that the held form has room for) up to which a form is taken.  Held vectors pay where a warp
// has one row or so: their loads run beside the row's, not behind its statistics.  us with the vectors read per row / held, at 1.0, 1.2
// and 1.4 rows a warp: 512 channels 3.4 / 3.3, from 1.05 on 3.4 / 4.1; 1024 4.6 / 3.1, 4.7 / 4.0, 4.8 / 4.7; 1152 4.9 / 3.5, 5.1 / 4.7,
// 5.2 / 5.4; 1536 3.7 / 3.3, 4.8 / 4.5, 4.8 / 5.1; 2048 5.3 / 3.3, 5.5 / 4.6, 5.6 / 5.5; 3072 6.3 / 5.4, at 1.05 6.6 / 7.4; 4096 6.9 / 4.4, at
// 1.1 7.4 / 7.1, at 1.2 7.7 / 7.8.  Long launches: 13106 x 1152 11.3 / 12.8, 9001 x 3072 20.7 / 20.8.
template <int VPL> constexpr long long kHeldRows10 = VPL <= 2 || VPL == 12 ? 10 : VPL == 16 ? 11 : VPL == 8 ? 14 : 12;
// With three to five vectors a lane the form that tests for the vectors as it goes is the fastest between the two: 4144 x 1024 4.2 us where
// kBoth takes 4.8, 4144 x 1152 4.8 and 5.2; from 1.8 rows a warp on it is the slowest (5328 x 1024 6.0 and 4.6).
template <int VPL> constexpr long long kTestedRows10 = VPL == 4 ? 16 : VPL == 5 ? 14 : 0;

// VPL: 16-byte vectors per lane (vec_per_row <= 32 * VPL)
template <int VPL, int MOD>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, kBlocks<VPL, MOD>)
layernorm_modulate_kernel(const uint4 *__restrict__ x, const int32_t *__restrict__ idx, int M, const uint4 *__restrict__ scale,
                          const uint4 *__restrict__ shift, uint4 *__restrict__ y, int B, int N, int vec_per_row, float eps,
                          int compact_in, int compact_out, int *__restrict__ err_word)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long total = (long long)B * M;
    const float inv_D = 1.0f / (float)(vec_per_row * 8);
    constexpr bool kHold = MOD == kHeld;
    uint4 sc_v[kHold ? VPL : 1], sh_v[kHold ? VPL : 1];
    int batch = -1;                                                                          // that they belong to
    for (long long t = (long long)blockIdx.x * kWarpsPerBlock + warp; t < total; t += (long long)gridDim.x * kWarpsPerBlock) {
        const int b = (int)(t / M), r = (int)(t - (long long)b * M);
        if (kHold && b != batch) {
            batch = b;
#pragma unroll
            for (int u = 0; u < (kHold ? VPL : 0); ++u) {
                const int c = lane + 32 * u;
                sc_v[u] = c < vec_per_row ? ld_cached(scale + (long long)b * vec_per_row + c) : make_uint4(0, 0, 0, 0);
                sh_v[u] = c < vec_per_row ? ld_cached(shift + (long long)b * vec_per_row + c) : make_uint4(0, 0, 0, 0);
            }
        }
        const int tok = idx ? __ldcg(idx + t) : r;
        const int before = (idx && r > 0) ? __ldcg(idx + t - 1) : -1;
        if ((unsigned)tok >= (unsigned)N || before >= tok) {                               // see astraea_scatter_reuse
            if (lane == 0 && err_word) atomicExch(err_word, kErrBadIndex);
            continue;
        }
        const uint4 *src = x + (compact_in ? t : (long long)b * N + tok) * vec_per_row;
        uint4 *dst = y + (compact_out ? t : (long long)b * N + tok) * vec_per_row;
        uint4 v[VPL];
#pragma unroll
        for (int u = 0; u < VPL; ++u) v[u] = (lane + 32 * u < vec_per_row) ? ld_stream(src + lane + 32 * u) : make_uint4(0, 0, 0, 0);
        // mean and variance in one pass over the packed registers, on data shifted by the row's first element: the
        // shift takes the cancellation out of E[(x - x0)^2] - (E[x - x0])^2 whenever the mean is large against the spread
        const float x0 = __shfl_sync(0xffffffffu, __uint_as_float(v[0].x << 16), 0);
        const f32x2 minus_x0 = pack2(-x0, -x0);
        f32x2 a1 = 0ull, a2 = 0ull;
#pragma unroll
        for (int u = 0; u < VPL; ++u) {
            if (lane + 32 * u < vec_per_row) {
                f32x2 f[4];
                unpack8(v[u], f);
#pragma unroll
                for (int i = 0; i < 4; ++i) { const f32x2 c = add2(f[i], minus_x0); a1 = add2(a1, c); a2 = fma2(c, c, a2); }
            }
        }
        float lo, hi;
        unpack2(a1, lo, hi);
        float s1 = lo + hi;
        unpack2(a2, lo, hi);
        float s2 = lo + hi;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { s1 += __shfl_xor_sync(0xffffffffu, s1, o); s2 += __shfl_xor_sync(0xffffffffu, s2, o); }
        const float ms = s1 * inv_D, mean = x0 + ms;
        const float sq = fmaxf(s2 - s1 * ms, 0.f);                 // sum of squares about the mean
        const float rs = rsqrtf(sq * inv_D + eps);
        const f32x2 minus_mean = pack2(-mean, -mean), rstd = pack2(rs, rs);
#pragma unroll
        for (int u = 0; u < VPL; ++u) {
            const int c = lane + 32 * u;
            if (c < vec_per_row) {
                f32x2 f[4], sc[4], sh[4];
                unpack8(v[u], f);
                const bool scaled = MOD != kPlain && (MOD != kEither || scale), shifted = MOD != kPlain && (MOD != kEither || shift);
                if (scaled) unpack8(kHold ? sc_v[kHold ? u : 0] : ld_cached(scale + (long long)b * vec_per_row + c), sc);
                if (shifted) unpack8(kHold ? sh_v[kHold ? u : 0] : ld_cached(shift + (long long)b * vec_per_row + c), sh);
                uint32_t w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    f[i] = mul2(add2(f[i], minus_mean), rstd);
                    if (scaled) f[i] = fma2(f[i], sc[i], f[i]);
                    if (shifted) f[i] = add2(f[i], sh[i]);
                    unpack2(f[i], lo, hi);
                    __nv_bfloat162 v2 = __floats2bfloat162_rn(lo, hi);
                    w[i] = *reinterpret_cast<uint32_t *>(&v2);
                }
                dst[c] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
}

template <int VPL, int MOD>
void launch_ln(cudaStream_t stream, const uint4 *x, const int32_t *idx, int M, const uint4 *scale, const uint4 *shift, uint4 *y, int B, int N,
               int vec_per_row, float eps, int ci, int co, int *err_word)
{
    const long long want = ((long long)B * M + kWarpsPerBlock - 1) / kWarpsPerBlock, cap = (long long)sm_count() * (MOD == kHeld ? kBlocks<VPL, MOD> : kBlocksPerSM);
    launch_overlapped(layernorm_modulate_kernel<VPL, MOD>, (int)(want < cap ? want : cap), kWarpsPerBlock * 32, 0, stream, x, idx, M, scale, shift, y, B, N,
                      vec_per_row, eps, ci, co, err_word);
}

}  // namespace

int32_t launch_layernorm_modulate(const void *x, const int32_t *idx, int M, const void *scale, const void *shift, void *y,
                                  int B, int N, int D, float eps, uint32_t flags, int *err_word, cudaStream_t stream)
{
    const int rows = idx ? M : N;
    const long long total = (long long)B * rows;
    if (total == 0) return ASTRAEA_OK;
    const int vec_per_row = D >> 3;
    if (vec_per_row > 32 * kMaxVecPerLane)
        return fail(ASTRAEA_ERR_UNSUPPORTED, "astraea_layernorm_modulate: D=%d above %d", D, 32 * kMaxVecPerLane * 8);
    const uint4 *xs = reinterpret_cast<const uint4 *>(x), *sc = reinterpret_cast<const uint4 *>(scale), *sh = reinterpret_cast<const uint4 *>(shift);
    uint4 *ys = reinterpret_cast<uint4 *>(y);
    const int ci = (flags & ASTRAEA_LN_COMPACT_IN) ? 1 : 0, co = (flags & ASTRAEA_LN_COMPACT_OUT) ? 1 : 0;
    const int vpl = (vec_per_row + 31) / 32;
#define kHeldWarps(V) (sm_count() * kBlocks<V, kHeld> * kWarpsPerBlock)
#define LN1(V, MOD) launch_ln<V, MOD>(stream, xs, idx, rows, sc, sh, ys, B, N, vec_per_row, eps, ci, co, err_word)
#define LN(V) do { if (!sc && !sh) LN1(V, kPlain); else if (!sc || !sh) LN1(V, kEither); \
    else if (10 * total <= kHeldRows10<V> * kHeldWarps(V)) LN1(V, kHeld); \
    else if (10 * total <= kTestedRows10<V> * kHeldWarps(V)) LN1(V, kEither); else LN1(V, kBoth); } while (0)
    if (vpl <= 2) LN(2);
    else if (vpl <= 4) LN(4);
    else if (vpl <= 5) LN(5);
    else if (vpl <= 6) LN(6);
    else if (vpl <= 8) LN(8);
    else if (vpl <= 12) LN(12);
    else LN(16);
#undef LN
#undef LN1
#undef kHeldWarps
    return check_launch("astraea_layernorm_modulate");
}

}  // namespace astraea
