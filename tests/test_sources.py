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
