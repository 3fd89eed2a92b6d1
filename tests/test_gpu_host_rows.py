"""Host-buffer sessions: steps that compute every token move whole rows, in chunks of rows, or head groups."""
import pytest
import torch

from paper_2506_05096_b200 import binding as A

pytestmark = pytest.mark.gpu


# two chunks of a batch element with a ragged last one; one chunk, of few tokens and of more; four and three batch elements that go
# together; all of them; eight chunks, the last one of two tokens
@pytest.mark.parametrize("B,H,d,N_v,N_t", [(2, 6, 64, 4070, 30), (1, 2, 64, 300, 7), (1, 3, 128, 3074, 0), (7, 8, 64, 600, 0), (5, 2, 64, 300, 2),
                                           (1, 27, 128, 1790, 4),
                                           # by head groups: too many batch elements, a group a head and two heads in some (head_dim 64: the
                                           # bits of the others depend on the CTA shape, which a launch of fewer heads may change); N on both
                                           # sides of the line at 20000
                                           (13, 2, 64, 300, 3), (13, 14, 64, 200, 5), (1, 1, 64, 20090, 10), (1, 1, 64, 19980, 10)])
def test_dense_steps_equal_the_device_path(B, H, d, N_v, N_t):
    """A dense first step, a sparse one, a dense one again and a sparse one behind it, against the single calls on device buffers (all
    keys in every CTA, as in a session): bit-identical outputs, so the LSE cache, the counters and the reference inputs that the
    dense steps leave behind are right, too."""
    N, D = N_v + N_t, H * d
    g = torch.Generator("cuda").manual_seed(3)
    sess = A.Session(B, H, N, N_v, d)
    x_ref = None
    lse, n_skip = torch.zeros(B, H, N, device="cuda"), torch.zeros(B, N_v, dtype=torch.int32, device="cuda")
    out, score = torch.zeros(B, N, H, d, dtype=torch.bfloat16, device="cuda"), torch.empty(B, N_v, device="cuda")
    host_out = torch.empty(B, N, D, dtype=torch.bfloat16).pin_memory()
    s = A.bhnd_strides(N, H, d)
    for step, k in enumerate((N_v, N_v // 3, N_v, N_v // 2)):
        M = k + N_t
        x, q, kk, v = (torch.randn(B, N, D, dtype=torch.bfloat16, device="cuda", generator=g) for _ in range(4))
        host = [t.cpu() for t in (x, q, kk, v)]
        sess.step_host(*(host if step == 2 else (t.pin_memory() for t in host)), host_out, k)       # the second dense step from pageable memory
        if x_ref is None:
            x_ref = x.clone()
        sel = torch.empty(B, M, dtype=torch.int32, device="cuda")
        A.astraea_score(x, x_ref, lse, n_skip, score, B, N, N_v, D, H)
        A.astraea_select(score, B, N_v, k, N_t, sel, None, n_skip, A.new_workspace(A.OP_SELECT, B, 0, N_v, k, 0))
        ws = A.new_workspace(A.OP_SPARSE_ATTN, B, H, N, M, d)
        A.astraea_sparse_attn(q, kk, v, s, s, s, sel, M, out, lse, B, H, N, d, flags=A.ATTN_WHOLE_KEYS, workspace=ws)
        A.astraea_scatter_reuse(x_ref, x, sel, B, N, M, D, A.SCATTER_SRC_FULL, workspace=ws)
        A.astraea_poll_error(ws)
        assert torch.equal(host_out.view(torch.int16), out.view(B, N, D).cpu().view(torch.int16)), step
    sess.close()
