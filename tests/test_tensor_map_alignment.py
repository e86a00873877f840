"""Tensor maps are encoded at addresses that are multiples of 64 (the driver's
precondition), wherever the caller keeps the bytes of a batch's descriptor
table.  Host-only: without a driver the encoder reports that it is missing."""
import ctypes

import pytest

JAC_EINVAL = 1


@pytest.mark.parametrize("offset", [0, 8, 16, 32, 48])
def test_batch_descriptors_may_lie_anywhere(offset):
    import paper_2002_12115_gb300 as pkg
    L = pkg.lib()
    desc_bytes = getattr(L, "_ZN3jac17sweep2_desc_bytesEv")
    desc_bytes.restype = ctypes.c_size_t
    batch_desc = getattr(L, "_ZN3jac17sweep2_batch_descEPvPK8jac_gridiPi")
    batch_desc.restype = ctypes.c_int
    batch_desc.argtypes = [ctypes.c_void_p, ctypes.POINTER(pkg.jac_grid), ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    n = desc_bytes()
    assert n % 64 == 0                       # the records of a device table stay aligned
    raw = ctypes.create_string_buffer(n + 128)
    base = (ctypes.addressof(raw) + 63) // 64 * 64
    g = pkg.jac_grid()
    g.I, g.J, g.K, g.prec, g.omega = 129, 40, 20, 1, 0.8
    g.p[0], g.p[1] = 0x10000, 0x20000        # never dereferenced
    for q in range(1, len(g.coef)):
        g.coef[q] = 0x30000 + 0x10000 * q
    items = ctypes.c_int()
    st = batch_desc(base + offset, ctypes.byref(g), 8, ctypes.byref(items))
    assert st != JAC_EINVAL, L.jac_last_error(None)
    if st == 0:                              # one tile along i, five along j, three k-blocks
        assert items.value == 15


def test_misaligned_map_is_refused():
    import paper_2002_12115_gb300 as pkg
    L = pkg.lib()
    enc = getattr(L, "_ZN3jac14encode_box_mapEP14CUtensorMap_stPKvmiiiiii")
    enc.restype = ctypes.c_int
    enc.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t] + [ctypes.c_int] * 6
    raw = ctypes.create_string_buffer(256)
    at = (ctypes.addressof(raw) + 63) // 64 * 64 + 16
    assert enc(at, 0x10000, 4, 136, 136, 20, 20, 128, 8) == JAC_EINVAL
    assert b"64" in L.jac_last_error(None)
