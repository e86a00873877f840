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


AFTER, BEFORE = "tmem_after_sync();", "tmem_before_sync();"


def test_tensor_memory_is_fenced_on_both_sides():
    """Every hand-over of tensor memory through a barrier is fenced by the
    warp that used it last and by the one that uses it next: sweep 1's stores
    to sweep 2's loads, sweep 2's loads to the stores that reuse a slot, and
    both to the deallocation."""
    text = code("jac_sweep2.cu")
    assert 'void tmem_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;"' in text
    assert 'void tmem_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;"' in text
    kernel = text[text.index("k_sweep2("):]
    sweep1 = kernel[kernel.index("const bool got_q"):]
    sweep2 = sweep1[sweep1.index("float *p_out;"):]
    sweep1 = sweep1[:sweep1.index("float *p_out;")]
    # sweep 1: the slot was read by sweep 2 before q_empty completed
    assert AFTER in sweep1[:sweep1.index("tmem_st16(")]
    assert BEFORE in sweep1[sweep1.index("tmem_wait_st()"):sweep1.index("mbar_arrive(&q_full")]
    # sweep 2
    assert AFTER in sweep2[:sweep2.index("tmem_ld16(")]
    assert BEFORE in sweep2[sweep2.rindex("tmem_wait_ld()"):sweep2.index("mbar_arrive(&q_empty")]
    # the deallocation, behind the CTA's last barrier
    end = sweep2[sweep2.index("__syncthreads();"):]
    assert AFTER in end[:end.index("tmem_dealloc(")]


def test_resident_halo_loads_follow_the_flag():
    """One lane of a communication warp acquires the neighbour's flag; the
    shuffle that tells the others does not order memory, so a warp barrier
    stands between it and their loads."""
    text = code("jac_resident.cu")
    wait = text[text.index("ld_acquire_gpu(nb_flag)"):]
    wait = wait[wait.index("__shfl_sync("):]
    assert "__syncwarp();" in wait[:wait.index("__ldcg(")]
