"""Loads of the device code, read from its source.

Kernels launched by launch_following are placed while the kernel before them
still writes the arrays that they read, so none of their loads may be a
read-only (non-coherent) one: CUDA allows those only for data that nothing
writes as long as the kernel runs.  __ldg and ld.global.nc ask for one, and
a const __restrict__ pointer lets the compiler choose one."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2009_02044_gb300", "csrc")


def _code(path):
    text = re.sub(r"/\*.*?\*/", " ", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", " ", text)


def test_no_read_only_loads_in_kernels_placed_early():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
    assert any("griddepcontrol.wait" in _code(f) for f in files)
    bad = [(os.path.basename(f), w) for f in files
           for w in re.findall(r"__ldg\b|ld\.global\.nc|__restrict__|__ldca\b", _code(f))]
    # the loads of k_step_pair, which is placed once the step before it is over
    bad = [b for b in bad if b[0] != "step_pair.cuh"]
    assert not bad, bad
    pair = [m for f in files for m in re.findall(r"launch_following\([^;]*;|k_step_pair<NC><<<", _code(f))
            if "k_step_pair<" in m]
    assert pair == ["k_step_pair<NC><<<"], pair
