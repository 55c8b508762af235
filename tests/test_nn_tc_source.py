"""The tensor-core kernels' bounded waits, by their source: an instruction of a whole
warp (.sync.aligned: tensor-memory loads and allocations) may only follow a wait that
its lanes leave together, since each lane's time limit runs out by itself. (What
happens otherwise is not for a GPU to show.)"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _source():
    with open(os.path.join(ROOT, "paper_2401_17183_gb300", "csrc", "vlb_nn_tc.cuh")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(src, name):
    i = src.index("{", src.index(name + "("))
    depth = 0
    for k in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return src[i:k + 1]
    raise AssertionError(name)


def test_warp_roles_wait_as_warps():
    body = _body(_source(), " k_dgrad_mma")
    assert "mbar_wait_warp(" in body and not re.search(r"\bmbar_wait\(", body)
    assert "__all_sync" in _body(_source(), " mbar_wait_warp")


def test_aligned_instructions_follow_a_warp_sync():
    src = _source()
    for name in (" tmem_ld16", " tmem_ld24"):
        body = _body(src, name)
        assert 0 <= body.find("__syncwarp()") < body.index("tcgen05.ld.sync.aligned"), name
    for m in re.finditer(r'asm volatile\("tcgen05\.alloc', src):
        assert src[:m.start()].rstrip().endswith("__syncwarp();")
