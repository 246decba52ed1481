"""The order in which the two CTAs of a pair set up and release tensor memory.

An allocation for a pair of CTAs blocks without a limit, so a step of one CTA that is
not ordered against the other's can leave a kernel waiting for good.  The functions
that order them stand in one place; these tests read the sources.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_09165_gb300", "csrc")
RAW = ("tmem_alloc_pair(", "tmem_relinquish_pair(", "tmem_dealloc_pair(")


def _code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _sources():
    return {os.path.basename(p): _code(p) for ext in ("*.cu", "*.cuh", "*.h")
            for p in sorted(glob.glob(os.path.join(CSRC, ext)))}


def _body(code, name):
    start = code.index("{", code.index(" " + name + "("))
    depth = 0
    for i in range(start, len(code)):
        depth += {"{": 1, "}": -1}.get(code[i], 0)
        if depth == 0:
            return code[start:i]
    raise AssertionError(name)


def _order(body, *steps):
    at = 0
    for s in steps:
        assert s in body[at:], (s, "not found in its place")
        at = body.index(s, at) + len(s)
    return body[at:]


def test_both_ctas_run_before_the_allocation_and_have_it_before_the_permit_goes():
    body = _body(_sources()["ptx.cuh"], "tmem_pair_setup")
    _order(body, "barrier.cluster.wait", "tmem_alloc_pair(", "cluster_sync_all()", "tmem_relinquish_pair(")
    assert "barrier.cluster.arrive" in _body(_sources()["ptx.cuh"], "tmem_pair_enter")


def test_no_cta_leaves_while_the_other_releases():
    body = _body(_sources()["ptx.cuh"], "tmem_pair_teardown")
    rest = _order(body, "cluster_sync_all()", "tmem_dealloc_pair(", "cluster_sync_all()")
    assert "tmem_" not in rest


def test_kernels_on_pairs_use_nothing_else():
    kernels = 0
    for name, code in _sources().items():
        if name == "ptx.cuh":
            continue
        for raw in RAW:
            assert raw not in code, (name, raw)
        if "mma_commit_pair(" in code:
            kernels += 1
            for step in ("enter", "setup", "teardown"):
                assert code.count("tmem_pair_%s(" % step) == 1, name
            # the producer waits for the ring's last commits between the tiles and the release
            tail = _order(code, "tmem_pair_enter(", "tmem_pair_setup(", "tma_load_2d_pair(")
            m = re.search(r"for \(int q = 0; ok && q < kStages\w*; \+\+q\) \{\s*"
                          r"ok = wait_bounded\(empty_bar\(s\), ph \^ 1u, abort_flag\);", tail)
            assert m and m.start() < tail.index("tmem_pair_teardown("), name
    assert kernels == 3


def test_served_steps_run_on_single_sms():
    # beside the server's other streams no pair's allocation is made at all
    code = _sources()["server.cu"]
    for launch in ("launch_symgemm_pair(", "launch_symgemm_x3(", "launch_symgemm_f32("):
        assert launch not in code
    assert "launch_symgemm(" in code
