"""Rules that the CUDA sources have to keep and that no output shows."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32882_b200", "csrc")


def _code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_no_kernel_reads_as_constant_what_the_kernel_before_it_may_still_write():
    """Kernels are placed while the one ahead of them runs and wait in grid_enter: loads on the read-only path (__ldg, ld.global.nc, and what
    the compiler makes of `const __restrict__`) need not stay behind that wait.  (The self-tests are launched without overlap.)"""
    files = [f for f in glob.glob(os.path.join(CSRC, "*.cu*")) if not f.endswith("selftest.cu")]
    assert len(files) > 15
    for path in files:
        code = _code(path)
        assert "__ldg" not in code and "ld.global.nc" not in code, path
        assert not re.search(r"const\s+[\w:]+\s*\*\s*__restrict__", code), path


def test_every_kernel_is_launched_to_overlap_and_waits_for_the_one_before_it():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        if path.endswith("selftest.cu"):
            continue
        code = _code(path)
        assert "<<<" not in code, path
        kernels = re.findall(r"__global__[^;{]*?\b(\w+_kernel)\s*\([^{;]*\)\s*\{(.*?)\n\}", code, re.S)
        for name, body in kernels:
            assert "grid_enter" in body, (path, name)


def test_tensor_memory_is_touched_behind_a_fence_after_every_wait():
    """A tcgen05 operation (load, store, product) behind a wait for tcgen05 work of other threads needs tcgen05.fence::after_thread_sync between the
    two: without it the operation may run ahead of what was waited for.  In the order of the source, from each wait to the next operation; waits on
    vectors in shared memory (`stat_full`) and barriers of a group of threads (VSA2_GROUP_SYNC) stand behind a fence of their own."""
    token = re.compile(r"(?P<wait>\bVSA2_WAIT\w*\s*\(\s*(?!&misc->stat_full)|\bmbar_wait\w*\s*\()|(?P<fence>\btc_fence_after\s*\()"
                       r"|(?P<op>\btc::(?:tmem_ld_?\d\w*|tmem_st_\d\w*|mma_ts|mma_ss\w*)\s*\(|\bmma_pair\w*)")
    operations = 0
    for path in glob.glob(os.path.join(CSRC, "fine_*.cu")) + [os.path.join(CSRC, "router_tc.cu")]:
        pending = None
        for number, line in enumerate(_code_lines(path), 1):
            for m in token.finditer(line):
                if m.group("wait"):
                    pending = number
                elif m.group("fence"):
                    pending = None
                else:
                    assert pending is None, (path, f"line {number} follows the wait in line {pending} without a fence")
                    operations += 1
    assert operations > 50


def test_forward_kernels_keep_what_their_warps_share_of_an_item_by_its_parity():
    """Epilogue and softmax warps of the forward kernels are up to one item apart, so nothing that belongs to an item may lie in a single place."""
    for name in ("fine_fwd_rows_tc.cu", "fine_fwd_rows2_tc.cu"):
        code = "".join(_code_lines(os.path.join(CSRC, name)))
        uses = re.findall(r"misc->(m_ref|red|oc|tok|gate|list_head|rescued|tab_full|tab_free|m_full|sums_full)\b(\[\w+\])?", code)
        assert {u[0] for u in uses} >= {"m_ref", "red", "tok", "rescued"}
        assert all(index in ("[tb]", "[0]", "[1]", "[s]") for _, index in uses), (name, [u for u in uses if u[1] not in ("[tb]", "[0]", "[1]", "[s]")])


def test_waits_are_limited_by_a_timer_that_all_sms_share():
    """%clock counts on one SM; a thread that was preempted may go on on another one, whose count can be behind, and its wait would seem to have run out."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"%clock|\bclock(64)?\s*\(", _code(path)), path


def test_the_self_test_runs_out_every_wait_that_the_kernels_use():
    with open(os.path.join(CSRC, "tc05.cuh")) as f:
        waits = re.findall(r"bool (mbar_wait\w*)\(", f.read())
    code = _code(os.path.join(CSRC, "selftest.cu"))
    assert sorted(waits) == ["mbar_wait", "mbar_wait_parked"]
    for name in waits:
        assert re.search(rf"\b{name}\(&never, 0, &abort_flag, limit_ns\)", code), name


def _code_lines(path):
    with open(path) as f:
        return [re.sub(r"//.*", "", line) for line in f]
