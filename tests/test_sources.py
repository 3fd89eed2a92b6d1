"""Rules of the CUDA sources that no run can show reliably: checked by reading them."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_05096_b200", "csrc")


def _code(name):
    """A source file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_no_load_takes_the_read_only_path():
    """Kernels start while the kernel before them still runs and wait inside: nothing they read is read-only for their whole
    life, so no load may go through the read-only path (a line of it may sit in L1 from before)."""
    names = [os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu*"))]
    assert len(names) >= 9
    for name in names:
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc|\bldg\b", _code(name)), name


def test_handshakes_between_ctas_have_cluster_scope():
    """An arrival on another CTA's barrier and the wait for it name the cluster as their scope (the default is the CTA, which
    promises the other one nothing), and where bytes in shared memory are passed on, a release and an acquire go with them."""
    ptx, lin = _code("sm100_ptx.cuh"), _code("linear.cu")
    for arrive in re.findall(r"mbarrier\.arrive\S*shared::cluster\S*", ptx):
        assert ".cluster.shared::cluster" in arrive, arrive
    remote = set(re.findall(r"map_to_rank\((bar_\w+)", lin)) - {"bar_full"}          # bar_full: bytes that TMA counts
    assert remote == {"bar_peer", "bar_acc_empty"}
    for bar in remote:
        waits = re.findall(r"wait_bar(<true>)?\(%s\b" % bar, lin)
        assert waits and all(waits), bar
    assert re.search(r"fence_release_smem\(\);\s*if \(elect_one\(\)\) mbar_arrive_cluster\(peer0", lin)
    assert re.search(r"wait_bar<true>\(bar_peer[^;]*;\s*fence_acquire_smem\(\);", lin)


def test_a_cta_that_gave_up_takes_no_further_unit():
    """Persistent attention CTAs: between the two CTA-wide barriers of a change of unit, the abort flag is looked at by every
    thread before any mbarrier is set up afresh."""
    attn = _code("attn.cu")
    body = attn[attn.index("auto next_unit"):attn.index("return true;")]
    flag, inval = body.index("(&abort_flag)) return false;"), body.index("mbar_inval")
    assert body.index("bar.sync 0") < flag < inval < body.rindex("bar.sync 0")


def _bodies(code, head):
    """The text of every block that starts with `head` (up to the brace that closes it)."""
    out, at = [], code.find(head)
    while at >= 0:
        depth, i = 0, code.index("{", at + len(head) - 1)
        start = i
        while True:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            if depth == 0:
                break
            i += 1
        out.append(code[start:i + 1])
        at = code.find(head, i)
    return out


def test_an_attention_cta_that_gave_up_sends_for_nothing_and_leaves_with_nothing_under_way():
    """Copies after the first tiles are sent for only while the CTA goes on; those that were sent are waited for without a look
    at the abort flag; the MMAs under way are committed and waited for before tensor memory is freed."""
    attn, wait = _code("attn.cu"), _code("bounded_wait.cuh")
    assert "abort" not in wait[wait.index("void drain_bar"):]
    for kv in "kv":
        (load,) = _bodies(attn, "auto load_%s = [&](int g, int j) {" % kv)
        assert load.index("wait_bar") < load.index("elect_one() && going(%s_stop, g)" % kv) < load.index("tma_load_4d")
        assert re.search(r"%s_loads = min\(%s_loads, %s_stop\)" % (kv, kv, kv), attn)
        assert "drain_bar(bar.%sf" % kv in attn
    end = attn[attn.rindex("if (abort_flag) {"):]
    assert end.index("tc_commit(bar_end") < end.index("drain_bar(bar_end") < end.index("__syncthreads()") < end.index("tmem_dealloc")


def test_a_gemm_pair_that_gave_up_sends_for_nothing_and_leaves_with_nothing_under_way():
    lin = _code("linear.cu")
    producer = lin[lin.index("const uint32_t full0"):lin.index("warp == kMmaWarp && rank == 0")]
    assert producer.index("wait_bar(bar_empty") < producer.index("elect_one() && going(g)") < producer.index("tma_load_2d")
    assert producer.index("min(g, stop)") < producer.index("drain_bar(bar_full") and "wait_bar(bar_full" not in producer
    end = lin[lin.rindex("if (abort_flag && rank == 0"):]
    assert end.index("tc_commit_pair(bar_end)") < end.index("drain_bar(bar_end") < end.index("cluster_sync_all()") < end.index("tmem_dealloc_pair")
