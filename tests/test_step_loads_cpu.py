"""Consecutive steps overlap: a step's blocks start while the step before still
writes the state.  Its loads of the state have to be ordinary ones, because
non-coherent loads (__ldg, const __restrict__) are for data that nothing
writes during the kernel's lifetime.  Stands in for a test on a GPU, where a
stale value would be a matter of timing."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_13072_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_overlapped_steps_load_the_state_coherently():
    step = _code("fvlb_fused.cuh")
    assert "griddepcontrol.wait" in _code("fvlb_kernels.cuh") and "pdl_wait()" in step
    assert not re.findall(r"__ldg|\bld\.global\.nc|Store<S>::ld\(", step)
    bufs = re.search(r"struct Bufs \{(.*?)\};", _code("fvlb_lattice.cuh"), re.S).group(1)
    for name in ("f_in", "h_in"):
        decl = re.search(r"[^;]*\b%s;" % name, bufs).group(0)
        assert "__restrict__" not in decl, decl
