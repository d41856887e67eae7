"""Rules that the compiler does not enforce, checked on the kernels' source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_09608_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_only_constants_take_the_read_only_path():
    """Kernels start while the one before them still runs (programmatic dependent launch), so what an earlier kernel of the
    stream may write (inputs, positions, metadata) is loaded by svlm_ptx::ld_in and ld_l2, which stay behind the wait and are
    coherent.  The read-only path (__ldg, const __restrict__) is for the rotation table and the projections' weights."""
    constants = {"tab", "p", "wp"}      # p, wp: rows of W (svlm_gemv.cu)
    for name in sorted(os.listdir(CSRC)):
        src = _source(name)
        if "pdl_wait" not in src and name != "svlm_rope.cuh":
            continue
        used = set(re.findall(r"__ld(?:g|cg|ca|cs)\(\s*&?\s*(\w+)", src))
        assert used <= constants, (name, used - constants)
        restricted = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", src))
        assert restricted <= {"tab", "W"}, (name, restricted)
