"""Resident sweeps (the library's own plan on grids that fit in shared memory)
against the streaming kernel (any explicit plan entry selects it).  Each
point-update is the same arithmetic, so the state must be bitwise the same.
The FP32 residual squares are summed in FP32 in groups of at most four points,
which the two kernels group differently: each square and each of three sums
rounds by 2^-24, so a residual of positive terms differs by at most 8 x 2^-24.
FP64 partial sums are over at most 1e6 positive terms with compensation beyond
a thread: 1e-12.  Shapes: one point, one box, boxes of one row, rows of more
and fewer points than a turn of the compute warps, the largest boxes that fit
and the first grids past them."""
import numpy as np
import pytest

import jacobi_inputs as ji
from _util import TOL, gpu_run, oracle_ref, rel_g, rel_p

pytestmark = pytest.mark.gpu

STREAM = (0, 0, 0, 1)
BAR = {"f64": 1e-12, "f32": 8 * 2.0 ** -24, "bf16": 8 * 2.0 ** -24}
SHAPES = [(3, 3, 3), (3, 17, 9), (5, 6, 7), (17, 17, 17), (33, 33, 65), (77, 53, 101), (700, 5, 6), (49, 49, 97),
          (65, 65, 129), (3, 90, 80), (130, 12, 40), (600, 3, 70)]
# they do not fit, or their boxes' halos take longer than streaming
STREAMING = {("f64", (77, 53, 101)), ("f64", (65, 65, 129)), ("f64", (700, 5, 6)), ("f32", (700, 5, 6))}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_12115_gb300 import _build
    _build.build()
    import oracle
    oracle.build()


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("dims", SHAPES)
def test_equals_streaming(dims, prec):
    I, J, K = dims
    f = ji.himeno_fields(I, J, K, seed=900 + I + J + K)
    from paper_2002_12115_gb300 import sweep_route
    for n in (3, 8, 9):
        if n > 3:                # three sweeps may not be worth the copy of the coefficients
            assert sweep_route(I, J, K, prec, n)["resident_sweeps"] == (0 if (prec, dims) in STREAMING else n)
        assert sweep_route(I, J, K, prec, n, fuse=1)["single_sweeps"] == n
        p1, g1 = gpu_run(f, n, prec, STREAM)
        p2, g2 = gpu_run(f, n, prec)
        assert np.array_equal(p1, p2), float(np.abs(p1 - p2).max())
        assert abs(g2 - g1) <= BAR[prec] * abs(g1), (g1, g2)


def test_many_sweeps_against_oracle_and_repeatable():
    """300 sweeps in calls of several lengths (both buffer parities), twice."""
    I, J, K = 61, 40, 50
    f = ji.himeno_fields(I, J, K, seed=31)
    from paper_2002_12115_gb300 import Jacobi
    got = []
    for _ in range(2):
        with Jacobi(I, J, K, "f32") as jac:
            jac.upload(f)
            for n in (4, 3, 1, 92, 200):
                jac.sweep(n)
            got.append((jac.download(), jac.residual()))
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
    wp, wg = oracle_ref(f, 300, "f32")
    assert rel_p(got[0][0], wp) <= TOL["f32"] and rel_g(got[0][1], wg) <= TOL["f32"]


def test_workspace_of_the_streaming_kernel_still_serves():
    """A workspace with room for the partials only takes the streaming kernel."""
    import torch

    import paper_2002_12115_gb300 as pkg
    I, J, K, n = 33, 20, 25, 6
    f = ji.himeno_fields(I, J, K, seed=8)
    want, _ = gpu_run(f, n, "f32")
    with pkg.Jacobi(I, J, K, "f32") as jac:
        jac.upload(f)
        g = jac.grid()
        small = pkg.workspace_size(g, 8 * 2, 4, 64)               # an explicit plan: partials of its CTAs
        full = pkg.workspace_size(g)
        assert full >= small
        ws = torch.zeros(256 + 256 * 8, dtype=torch.uint8, device="cuda")
        res = torch.zeros(1, dtype=torch.float64, device="cuda")
        pkg.sweep_dev(g, n, res.data_ptr(), ws.data_ptr(), ws.numel(), jac.stream)
        pkg.workspace_check(ws.data_ptr(), jac.stream)
        out = torch.empty((K, J, I), dtype=torch.float64, device="cuda")
        pkg.unpack_dev(I, J, K, "f32", 0, g.p[n % 2], out.data_ptr(), jac.stream)
        assert np.array_equal(out.cpu().numpy(), want)
