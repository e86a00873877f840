"""The failure path of the bounded device waits, made to run out on purpose
without faulting or hanging anything.

jac_inject_stall gives the next sweep call's launches a grid-barrier target
that no CTA ever reaches, and a wait limit of a few milliseconds.  The waits
for it -- of the streaming kernel's and the two-sweep kernel's producers, of
the resident kernel's communication warps -- then give up, every CTA drains its
own copies and exits, and the launch ends with the workspace error word set:
the residual written is NaN, jac_sync and jac_residual report JAC_ETIMEOUT
and clear the word, and the same context then sweeps normally again (the
result checked against the oracle).  This is the library's counterpart of
the offload search's measurement time limit (Section 5.1.2)."""
import numpy as np
import pytest

import jacobi_inputs as ji
from _util import TOL, oracle_ref, rel_g, rel_p

pytestmark = pytest.mark.gpu
WAIT_NS = 2_000_000          # 2 ms: far above any legitimate wait on these grids


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_12115_gb300 import _build
    _build.build()
    import paper_2002_12115_gb300 as p
    return p


@pytest.mark.parametrize("prec,dims,owned", [("f32", (70, 21, 19), False), ("bf16", (131, 9, 12), True),
                                             ("f64", (37, 33, 29), False)])
def test_stalled_barrier_times_out_and_context_recovers(pkg, prec, dims, owned):
    I, J, K = dims
    n = 4
    f = ji.himeno_fields(I, J, K, seed=300 + I)
    with pkg.Jacobi(I, J, K, prec, owned=owned) as jac:
        jac.upload(f)
        jac.inject_stall(WAIT_NS)
        jac.sweep(n)
        p_out = np.zeros((K, J, I))
        res = np.zeros(1)
        jac.download_async(p_out, res)
        with pytest.raises(pkg.JacError) as err:
            jac.sync()
        assert err.value.status == 5                      # JAC_ETIMEOUT
        assert np.isnan(res[0])                           # the launch wrote NaN, not stale partials
        jac.sync()                                        # the error word was cleared

        # the residual route reports it too
        jac.upload(f)
        jac.inject_stall(WAIT_NS)
        jac.sweep(n)
        with pytest.raises(pkg.JacError) as err:
            jac.residual()
        assert err.value.status == 5

        # and the context sweeps normally afterwards
        jac.upload(f)
        jac.sweep(n)
        g = jac.residual()
        p = jac.download()
    op, og = oracle_ref(f, n, prec)
    assert rel_p(p, op) <= TOL[prec] and rel_g(g, og) <= TOL[prec], (rel_p(p, op), rel_g(g, og))


def test_single_sweep_launch_has_no_barrier_to_stall(pkg):
    """One sweep per launch never waits on the grid barrier: the injection
    is consumed and the result is normal."""
    I, J, K = 40, 17, 11
    f = ji.himeno_fields(I, J, K, seed=333)
    with pkg.Jacobi(I, J, K, "f32") as jac:
        jac.upload(f)
        jac.inject_stall(WAIT_NS)
        jac.sweep(1)
        g = jac.residual()
        p = jac.download()
    op, og = oracle_ref(f, 1, "f32")
    assert rel_p(p, op) <= TOL["f32"] and rel_g(g, og) <= TOL["f32"]


def stall_and_recover(pkg, prec, dims, n, plan=None):
    """One stalled call (JAC_ETIMEOUT, a NaN residual, a partly swept state),
    then normal ones on the same context: bitwise the state of a context that
    was never stalled.  Returns the fields, the stalled call's state and the other
    state buffer after it."""
    I, J, K = dims
    f = ji.himeno_fields(I, J, K, seed=400 + I)
    with pkg.Jacobi(I, J, K, prec) as jac:
        if plan is not None:
            jac.set_plan(*plan)
        jac.upload(f)
        jac.inject_stall(WAIT_NS)
        jac.sweep(n)
        stalled, res = np.zeros((K, J, I)), np.zeros(1)
        jac.download_async(stalled, res)
        with pytest.raises(pkg.JacError) as err:
            jac.sync()
        assert err.value.status == 5 and np.isnan(res[0])
        raw = jac.storage[1 - n % 2].cpu().numpy().view(np.float64 if prec == "f64" else np.float32)
        other = raw.reshape(K, J, pkg.pitch(I))[:, :, :I].astype(np.float64)
        got = []
        for m in (n, n + 1):                              # the header is left as the next launch needs it
            jac.upload(f)
            jac.sweep(m)
            got.append((jac.download(), jac.residual()))
    with pkg.Jacobi(I, J, K, prec) as jac:
        if plan is not None:
            jac.set_plan(*plan)
        for m, (p, g) in zip((n, n + 1), got):
            jac.upload(f)
            jac.sweep(m)
            assert np.array_equal(jac.download(), p) and jac.residual() == g
    return f, stalled, other


@pytest.mark.parametrize("prec,dims", [("f32", (70, 21, 19)), ("bf16", (131, 9, 12)), ("f64", (37, 33, 29))])
def test_streaming_waits_run_out(pkg, prec, dims):
    """The streaming kernel's wait between sweeps: the first sweep is stored
    whole and no CTA starts the second."""
    n, plan = 4, (0, 0, 0, 1)
    assert pkg.sweep_route(*dims, prec, n, fuse=1)["single_sweeps"] == n
    f, stalled, other = stall_and_recover(pkg, prec, dims, n, plan)
    with pkg.Jacobi(*dims, prec) as jac:
        jac.upload(f)
        assert np.array_equal(stalled, jac.download())
        jac.sweep(1)
        assert np.array_equal(other, jac.download())


@pytest.mark.parametrize("prec,dims", [("f32", (77, 53, 101)), ("bf16", (61, 40, 50)), ("f64", (33, 33, 65))])
def test_resident_waits_run_out(pkg, prec, dims):
    """The resident kernel's waits: no box sees the barrier, so none gets past
    its first exchange.  Of its first sweep a box has stored the rows next to
    other boxes by then and no inner row (the streaming kernel stores all)."""
    n = 5                                                 # state n is in the buffer of state 1
    assert pkg.sweep_route(*dims, prec, n)["resident_sweeps"] == n
    f, stalled, _ = stall_and_recover(pkg, prec, dims, n)
    with pkg.Jacobi(*dims, prec) as jac:
        jac.upload(f)
        p0 = jac.download()
        jac.sweep(1)
        p1 = jac.download()
    inside = (slice(1, -1),) * 3
    swept, kept = np.all(stalled == p1, axis=2)[inside[:2]], np.all(stalled == p0, axis=2)[inside[:2]]
    assert np.all(swept | kept) and swept.any() and kept.any()


@pytest.mark.parametrize("dims,n,plan", [((129, 33, 20), 4, (0, 0, 0, 2)), ((130, 17, 23), 8, (0, 0, 0, 2)),
                                         ((129, 129, 140), 4, None)])
def test_pass_barrier_runs_out(pkg, dims, n, plan):
    """The two-sweep kernel's wait between passes: the first pass is stored --
    state 2, where single sweeps would have stored state 1 -- and no CTA starts
    the second.  Sweeps after the passes would run on that state, with a NaN
    residual."""
    assert pkg.sweep_route(*dims, "f32", n, fuse=plan[3] if plan else 0)["passes"] == n // 2
    f, stalled, other = stall_and_recover(pkg, "f32", dims, n, plan)
    with pkg.Jacobi(*dims, "f32") as jac:
        jac.set_plan(0, 0, 0, 1)
        jac.upload(f)
        assert np.array_equal(stalled, jac.download())
        jac.sweep(2)
        assert np.array_equal(other, jac.download())
