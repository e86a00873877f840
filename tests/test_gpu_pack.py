"""The packing kernel: every array of a copy-in in its storage layout, from
FP64 and FP32 sources, against torch's round-to-nearest conversions.  Exact:
rounding is RNE (BF16 through FP32) and the padding columns are zero.  Row
lengths from one point to more than a block's 2048 elements."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3, 3), (8, 5, 4), (31, 4, 3), (33, 3, 7), (120, 4, 3), (127, 5, 4), (129, 3, 5), (257, 9, 3), (2100, 3, 3)]


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_12115_gb300 import _build
    _build.build()
    import paper_2002_12115_gb300 as p
    return p


def _storage(jac, q, prec, pitch):
    """Storage array q of a borrowed context (0, 1: the state buffers) as (K, J, pitch)."""
    import torch
    dt = {"f64": torch.float64, "f32": torch.float32,
          "bf16": torch.float32 if q in (0, 1, 12) else torch.bfloat16}[prec]
    return jac.storage[q].view(dt).view(jac.K, jac.J, pitch)


@pytest.mark.parametrize("source", ["f64", "f32"])
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_storage_is_the_rounded_input(pkg, shape, prec, source):
    import torch
    I, J, K = shape
    g = torch.Generator().manual_seed(I + 1000 * J)
    f = {n: torch.randn((K, J, I), generator=g, dtype=torch.float64) for n in pkg.FIELDS}
    # ties, carries into the exponent, FP32 subnormals, overflow, signed zeros, infinities
    special = [1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 1 + 2.0 ** -24 + 2.0 ** -52, 2 - 2.0 ** -25, -(2 - 2.0 ** -25),
               1e-42, -2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -25), 2.0 ** -150, -3e38, 2.0 ** 128 - 2.0 ** 103,
               2.0 ** 128 - 2.0 ** 102, -1e300, 1e-320, -0.0, 0.0, float("inf"), -float("inf")]
    for n in ("p", "a0", "c1", "wrk1"):
        f[n].view(-1)[:len(special)] = torch.tensor(special, dtype=torch.float64)
    f = {n: v.to(torch.float32) for n, v in f.items()} if source == "f32" else f
    with pkg.Jacobi(I, J, K, prec, async_upload=source == "f32") as jac:
        for s in jac.storage:
            s.fill_(0xff)
        if source == "f64":
            jac.upload_tensors({n: v.cuda() for n, v in f.items()})
        else:
            jac.upload_f32_async({n: v.numpy() for n, v in f.items()})
        jac.sync()
        P = pkg.pitch(I)
        for q in range(14):
            got = _storage(jac, q, prec, P).cpu()
            src = f[pkg.FIELDS[max(q - 1, 0)]]
            want = torch.zeros((K, J, P), dtype=got.dtype)
            want[..., :I] = src.to(torch.float32).to(got.dtype) if got.dtype == torch.bfloat16 else src.to(got.dtype)
            assert torch.equal(got, want), (q, prec, source)
        out = jac.download()
        assert np.array_equal(out, _storage(jac, 0, prec, P)[..., :I].cpu().double().numpy())
