"""Orders between threads, launches and memory units that PTX asks for and that
no run can be trusted to show missing, read from the kernel sources.  Nothing
here needs a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_12115_gb300", "csrc")


def code(name):
    """A source without its comments."""
    with open(os.path.join(CSRC, name)) as fh:
        text = fh.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_dependent_launches_read_coherently():
    """A kernel launched as a programmatic dependent runs beside the launch
    before it, so no parameter of it may promise that memory does not change
    (const __restrict__), and nothing may take the read-only path (__ldg)."""
    sources = [f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))]
    dependent = [f for f in sources if "ProgrammaticStreamSerialization" in code(f)]
    assert sorted(dependent) == ["jac_adjoint.cu", "jfft.cu"]
    for f in dependent:
        text = code(f)
        assert "__restrict__" not in text and "__ldg" not in text and "ld.global.nc" not in text, f
        # and every kernel waits for the launches before it
        kernels = re.findall(r"__global__.*?\n}", text, flags=re.S)
        assert kernels and all("wait_prior_grids()" in k for k in kernels), f
