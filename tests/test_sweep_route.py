"""Which kernels a call runs (jac_sweep_route, no GPU): the rule that the sweep
itself follows, on a GB300's 152 SMs and 128 MiB of L2."""
import random

import pytest

from paper_2002_12115_gb300 import JacError, sweep_route

SMS = 152


def route(I, J, K, prec, n, **plan):
    r = sweep_route(I, J, K, prec, n, sm_count=SMS, **plan)
    return r["launches"], r["resident_sweeps"], r["passes"], r["single_sweeps"]


@pytest.mark.parametrize("dims,prec,n,want", [
    ((33, 33, 65), "f64", 200, (1, 200, 0, 0)),          # fits in shared memory
    ((33, 33, 65), "f64", 2, (1, 0, 0, 2)),              # but not for two sweeps
    ((77, 53, 101), "f32", 20, (1, 20, 0, 0)),
    ((65, 65, 129), "bf16", 3, (1, 3, 0, 0)),
    ((65, 65, 129), "f64", 50, (1, 0, 0, 50)),
    ((129, 129, 257), "f32", 100, (1, 0, 50, 0)),        # full tiles: passes, also where the state stays in L2
    ((129, 129, 257), "f32", 7, (2, 0, 2, 3)),
    ((513, 513, 1025), "f32", 102, (2, 0, 50, 2)),
    ((161, 161, 161), "f32", 100, (1, 0, 0, 100)),       # two tiles 62% full
    ((513, 513, 1025), "bf16", 10, (1, 0, 0, 10)),
    ((513, 513, 1025), "f64", 10, (1, 0, 0, 10)),
    ((513, 513, 1025), "f32", 0, (0, 0, 0, 0)),
])
def test_routes_without_a_plan(dims, prec, n, want):
    assert route(*dims, prec, n) == want


@pytest.mark.parametrize("dims,prec", [
    ((402, 145, 5), "bf16"), ((449, 160, 3), "f32"), ((147, 114, 11), "f32"), ((404, 44, 23), "f32"),
    ((143, 158, 9), "f32"), ((321, 22, 34), "f32"), ((254, 37, 51), "bf16"), ((264, 122, 8), "f64"),
    ((120, 40, 30), "f64")])
def test_wide_flat_grids_stream(dims, prec):
    """Their coefficients fit in shared memory, but a resident sweep takes 1.05
    to 1.6 times a streaming one: boxes without inner rows, and much halo."""
    for n in (4, 20, 100):
        assert route(*dims, prec, n)[1] == 0


@pytest.mark.parametrize("dims,prec,n", [
    ((17, 17, 17), "f64", 5), ((33, 33, 65), "f64", 5), ((49, 49, 97), "f64", 5), ((77, 53, 101), "f32", 5),
    ((65, 65, 129), "f32", 5), ((65, 65, 129), "bf16", 5), ((61, 40, 50), "bf16", 5), ((218, 133, 4), "f32", 20),
    ((80, 104, 3), "f64", 5), ((70, 20, 4), "bf16", 5)])
def test_small_grids_run_resident(dims, prec, n):
    assert route(*dims, prec, n)[1] == n


def test_routes_of_explicit_plans():
    """Any non-zero entry leaves out the resident kernel; fuse 1 and 2 decide
    the passes, fuse 0 beside another entry the size of the state."""
    assert route(33, 33, 65, "f64", 200, kdepth=4) == (1, 0, 0, 200)
    assert route(77, 53, 101, "f32", 20, fuse=1) == (1, 0, 0, 20)
    assert route(77, 53, 101, "f32", 22, fuse=2) == (2, 0, 10, 2)
    assert route(129, 129, 257, "f32", 100, kdepth=16) == (1, 0, 0, 100)
    assert route(513, 513, 1025, "f32", 100, kdepth=16) == (1, 0, 50, 0)
    assert route(513, 513, 1025, "f32", 100, fuse=1) == (1, 0, 0, 100)


def test_every_sweep_is_counted_once():
    rng = random.Random(4)
    for _ in range(300):
        I, J, K = (rng.randint(3, 300) for _ in range(3))
        n = rng.randint(1, 60)
        launches, resident, passes, single = route(I, J, K, rng.choice(["f64", "f32", "bf16"]), n)
        assert resident + 2 * passes + single == n and passes % 2 == 0
        assert launches == (resident > 0) + (passes > 0) + (single > 0)


@pytest.mark.parametrize("dims,n", [((185, 104, 421), 20), ((201, 124, 326), 4), ((129, 129, 257), 5),
                                    ((161, 161, 161), 8)])
def test_bench_names_the_kernel_that_runs(dims, n):
    """The bench's roofline counts the bytes of the kernel the library takes,
    also where the padded rows decide whether the state stays in L2."""
    import torch

    import bench
    if torch.cuda.is_available():
        pytest.skip("the bench asks for the present device")
    w = dict(I=dims[0], J=dims[1], K=dims[2])
    _, _, passes, single = route(*dims, "f32", n)
    r = bench.sweep_roofline(w, "f32", n, 1.0)
    assert r["kernel"].startswith("k_sweep2 " if passes else "k_sweep")
    assert r.get("passes_per_launch", 0) == passes
    per_point = 56 * (passes + single)
    assert r["algorithmic_bytes_per_launch"] == per_point * bench.n_interior(w)


@pytest.mark.parametrize("dims,prec,kw", [((33, 33, 65), "f64", dict(kdepth=4)), ((77, 53, 101), "f32", dict(fuse=1)),
                                          ((65, 65, 129), "bf16", dict(tile_j=16, tile_i=128, kdepth=8)),
                                          ((129, 129, 257), "f32", dict(kdepth=64))])
def test_workspace_of_an_explicit_plan_is_that_plan_s(dims, prec, kw):
    """256 bytes and a double per CTA of the plan, rounded up to 256 bytes; the
    flags of the resident kernel and a pass's partials only where the library
    may choose them."""
    import paper_2002_12115_gb300 as pkg
    g = pkg.jac_grid()
    g.I, g.J, g.K, g.prec, g.omega = *dims, pkg.PRECS[prec], 0.8
    for b in range(2):
        g.p[b] = 0x1000 * (b + 1)
    for q in range(1, len(g.coef)):
        g.coef[q] = 0x10000 * q
    p = pkg.resolve_plan(*dims, prec, **kw)
    items = (((dims[0] - 2) // p["tile_i"] + 1) * -(-(dims[1] - 2) // p["tile_j"]) * -(-(dims[2] - 2) // p["kdepth"]))
    size, default = pkg.workspace_size(g, **kw), pkg.workspace_size(g)
    assert size == 256 + -(-8 * min(items, 148) // 256) * 256        # 148 or 152 SMs: the same
    assert default >= size


@pytest.mark.parametrize("kw", [dict(tile_j=5), dict(kdepth=-2), dict(fuse=3)])
def test_bad_plans_and_counts_are_rejected(kw):
    with pytest.raises(JacError, match="JAC_EINVAL"):
        sweep_route(129, 129, 257, "f32", 10, sm_count=SMS, **kw)
    with pytest.raises(JacError, match="JAC_EINVAL"):
        sweep_route(129, 129, 257, "f32", -1, sm_count=SMS)
    with pytest.raises(JacError, match="JAC_EINVAL"):
        sweep_route(2, 9, 9, "f32", 1, sm_count=SMS)
