"""Coarse vectors in device memory need no more than the 8 bytes of a double: every call of the C ABI that takes them
gives the same bits for arrays at odd multiples of 8 bytes as for arrays of 16-byte alignment (inputs, outputs and both)."""

import pytest
import torch

from paper_1610_02370_gb300 import synth

pytestmark = pytest.mark.gpu

DIMS, NV = (8, 8, 8, 16), 21


@pytest.fixture(scope="module")
def lib():
    from paper_1610_02370_gb300 import build
    build.build()
    from paper_1610_02370_gb300 import ddtm
    return ddtm


def place(x, odd):
    """x (complex128) as doubles on the device, at an odd multiple of 8 bytes if odd."""
    buf = torch.zeros(2 * x.numel() + 2, dtype=torch.float64, device="cuda")
    d = buf[1:-1] if odd else buf[:-2]
    d.copy_(torch.view_as_real(x).flatten())
    assert d.data_ptr() % 16 == (8 if odd else 0)
    return d


@pytest.mark.parametrize("coarse_prec,levels,nrhs", [(1, 2, 3), (2, 2, 3), (2, 2, 40), (1, 3, 5)])
def test_coarse_vectors_at_odd_doubles(lib, coarse_prec, levels, nrhs):
    import ctypes
    c, dev = lib._lib, lib.LOC_DEVICE
    dims = (16, 16, 16, 16) if levels == 3 else DIMS
    lat = (dims[0], dims[3], dims[2], dims[1])
    U = synth.gauge_field(dims, 0.2, seed=81, device="cuda")
    ctx = lib.ddtm_create(dims, (4, 4, 4, 4), 0)
    try:
        lib.ddtm_load_gauge(ctx, U, 0.134, 1.5755)
        p = lib.ddtm_get_params(ctx)
        p.n_levels, p.nv[0], p.nv[1], p.coarse_prec, p.coarse_tol = levels, NV, 8, coarse_prec, 1e-2
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_set_test_vectors(ctx, 0, synth.gaussian_vectors((NV,) + lat + (4, 3), seed=82, device="cuda"), NV)
        cl = tuple(n // 4 for n in lat)
        if levels == 3:
            lib.ddtm_set_test_vectors(ctx, 1, synth.gaussian_vectors((8,) + cl + (2 * NV,), seed=85, device="cuda"), 8)
        x = synth.gaussian_vectors((nrhs,) + cl + (2 * NV,), seed=83, device="cuda")
        f = synth.gaussian_spinor(dims, seed=84, nrhs=nrhs, device="cuda")
        it = ctypes.c_int(0)
        calls = {"apply_Dc": (x, x, lambda o, i: c.ddtm_apply_Dc(ctx, 1, o, i, nrhs, 0.02, dev)),
                 "restrict": (x, f, lambda o, i: c.ddtm_restrict(ctx, 0, o, i, nrhs, dev)),
                 "prolong": (f, x, lambda o, i: c.ddtm_prolong(ctx, 0, o, i, nrhs, dev))}
        if levels == 2:
            calls["solve"] = (x, x, lambda o, i: c.ddtm_coarse_solve_batch(ctx, o, i, nrhs, 0.02, dev, ctypes.byref(it)))
        else:
            calls["sap"] = (x, x, lambda o, i: c.ddtm_sap_coarse(ctx, 1, o, i, nrhs, 0.02, 2, 3, dev))
        for name, (out, inp, call) in calls.items():
            want = None
            for odd_in, odd_out in ((0, 0), (1, 0), (0, 1), (1, 1)):
                # the fine side (restrict in, prolong out) is read and written in 16-byte pieces and stays aligned
                if (inp is f and odd_in) or (out is f and odd_out):
                    continue
                i, o = place(inp, odd_in), place(torch.zeros_like(out), odd_out)
                assert call(o.data_ptr(), i.data_ptr()) == lib.OK, (name, lib.ddtm_last_error(ctx))
                torch.cuda.synchronize()
                want = o.clone() if want is None else want
                assert float(want.abs().max()) > 0 and torch.equal(o, want), (name, odd_in, odd_out)
    finally:
        lib.ddtm_destroy(ctx)
