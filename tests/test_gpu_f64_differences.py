"""FP64 sweeps form each b bracket from differences along j and i that
neighbouring points and planes share through the warp's shared memory.  Against
the oracle at the widths where the halo of a tile's difference row matters: one
tile narrower than, as wide as and just past the grid, several tiles, rows of 1,
2 and 4 segments per warp, items of one and of several planes, balanced ranges;
with cross coefficients of up to 0.3, so that a wrong difference shows.

A point-update is at most 30 roundings of terms that add up to at most 4 max|p|
(six axis coefficients of 1 and twelve cross terms of 0.3, times a3 = 1/6 and
omega = 0.8, plus p): 30 x 4 x 2^-53 < 1.4e-14 a sweep."""
import numpy as np
import pytest

import jacobi_inputs as ji
from _util import gpu_run, rel_p

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_12115_gb300 import _build
    _build.build()
    import oracle
    oracle.build()


@pytest.mark.parametrize("tile_i", [16, 32, 64])
@pytest.mark.parametrize("over", [-1, 0, 1, 2, 3])
def test_tile_edges_against_oracle(tile_i, over):
    import oracle
    for tiles, warps, kdepth in ((1, 8, 0), (2, 4, 1), (3, 8, 3), (2, 8, -1)):
        I, J, K, n = tiles * tile_i + over, 21, 12, 2
        f = {k: np.array(v) for k, v in ji.himeno_fields(I, J, K, seed=1000 + I).items()}
        r = np.random.default_rng(I)
        for k in ("b0", "b1", "b2"):
            f[k] = r.uniform(-0.3, 0.3, (K, J, I))
        f["p"] = r.uniform(-1.0, 1.0, (K, J, I))
        got, _ = gpu_run(f, n, "f64", (64 * warps // tile_i, kdepth, tile_i, 1))
        want = oracle.run(f, n)
        want = want[0] if isinstance(want, tuple) else want
        assert rel_p(got, want) <= n * 1.4e-14, (I, warps, kdepth, rel_p(got, want))
