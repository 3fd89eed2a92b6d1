// The copying warp of the attention kernel.  (A file of its own, without includes: the primitives that it uses come from the
// kernel that includes it, or from a model of a warp on the host.)
#pragma once

// This CTA's even share of the listed rows goes from copy_src to copy_dst by bulk copies, through kCopyStages stages: the
// load of a batch is sent kCopyStages - 1 batches before its store.  A batch is as many rows as fit a stage, a lane each, or a
// piece of one row.  The standalone scatter is one more launch and a pass at memory speed in which the tensor cores idle;
// here the bytes move under the key loop (a batch takes ~1.5 us, a CTA has 5-30 of them in 30-900 us).
// When the CTA gives up, all lanes leave together, and not before the loads that have been sent have landed.
template <class C, class Params>
__device__ __forceinline__ void copy_role(const Params &p, uint32_t s_copy, uint32_t bar, volatile int *abort_flag)
{
    constexpr int kS = C::kCopyStages;
    const int lane = threadIdx.x & 31;
    const int r0 = (int)((long long)p.copy_rows * blockIdx.x / gridDim.x), r1 = (int)((long long)p.copy_rows * (blockIdx.x + 1) / gridDim.x);
    const int parts = (int)((p.copy_bytes + C::kCopyStageBytes - 1) / C::kCopyStageBytes);       // pieces of a row
    const int rows = parts > 1 ? 1 : min(32, (int)(C::kCopyStageBytes / p.copy_bytes));            // rows of a batch
    const int batches = parts > 1 ? (r1 - r0) * parts : (r1 - r0 + rows - 1) / rows;
    // 16-byte units ahead of this lane's piece of batch i in both tensors; -1: none, or a bad entry (reported by the softmax warps)
    auto piece = [&](int i) -> int {
        const int r = parts > 1 ? r0 + i / parts : r0 + i * rows + lane;
        if (i >= batches || lane >= rows || r >= r1) return -1;
        const int b = r / p.M, m = r - b * p.M;
        const int tok = __ldcg(p.q_idx + r), before = m > 0 ? __ldcg(p.q_idx + r - 1) : -1;
        if ((unsigned)tok >= (unsigned)p.N_tok || before >= tok) return -1;
        return (b * p.N_tok + tok) * (int)(p.copy_bytes >> 4) + (parts > 1 ? (i % parts) * (C::kCopyStageBytes / 16) : 0);
    };
    auto bytes = [&](int i) -> uint32_t {
        return parts > 1 ? min((uint32_t)C::kCopyStageBytes, p.copy_bytes - (uint32_t)(i % parts) * C::kCopyStageBytes) : p.copy_bytes;
    };
    const uint32_t slot = lane * (rows > 1 ? p.copy_bytes : 0u);
    int off[kS], next = piece(0);                 // off[u]: batch i - u
#pragma unroll
    for (int u = 0; u < kS; ++u) off[u] = -1;
    int gave_up = 0;                              // the round in which the CTA gave up
    for (int i = 0; i < batches + kS - 1; ++i) {
#pragma unroll
        for (int u = kS - 1; u > 0; --u) off[u] = off[u - 1];
        off[0] = next;
        next = piece(i + 1);
        const int j = i - (kS - 1);
        if (j >= 0) {
            wait_bar(bar + 8 * (j % kS), (j / kS) & 1, abort_flag, p.err_word);
            if (__any_sync(0xffffffffu, *abort_flag != 0)) {
                gave_up = i;
                break;
            }
            if (off[kS - 1] >= 0) bulk_store(p.copy_dst + off[kS - 1], s_copy + (j % kS) * C::kCopyStageBytes + slot, bytes(j));
        }
        bulk_commit();
        if (i < batches) {
            bulk_wait_read<1>();                        // the stage's last batch (stored one round ago) has left it
            const uint32_t n = __popc(__ballot_sync(0xffffffffu, off[0] >= 0));
            if (lane == 0) mbar_arrive_expect_tx(bar + 8 * (i % kS), n * bytes(i));
            __syncwarp();
            if (off[0] >= 0) bulk_load(s_copy + (i % kS) * C::kCopyStageBytes + slot, p.copy_src + off[0], bytes(i), bar + 8 * (i % kS));
        }
    }
    bulk_wait<0>();
    // (inside the loop this cost the whole kernel 0.7 %)
    for (int l = max(0, gave_up - (kS - 1)); l < min(gave_up, batches); ++l) drain_bar(bar + 8 * (l % kS), (l / kS) & 1);
}
