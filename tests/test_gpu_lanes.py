"""The kernels for 4^4 blocks that hold one or two right-hand sides per thread
(csrc/stencil_lanes.cuh): the smoother and D(mu) against the CPU oracle at the edges of
their range -- one, two and an odd number of right-hand sides, antiperiodic time, unequal
lattice sides, no MR step and several -- and with the FP16 operator copies that FP16 fields fall
back to when the FP32 copies do not fit.  Tolerances as in the other parity tests: 2e-6
for FP32 (sums of a few dozen products, a handful of dependent steps), 2e-3 with FP16 storage.
"""

import numpy as np
import pytest
import torch

from oracle import sap as osap
from oracle.operators import FineOperator
from paper_1610_02370_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {1: 2e-6, 2: 2e-3}
DIMS, BLOCK, KAPPA, CSW, MU = (16, 8, 8, 24), (4, 4, 4, 4), 0.13, 1.2, 0.03


@pytest.fixture(scope="module")
def lib():
    from paper_1610_02370_gb300 import build
    build.build()
    from paper_1610_02370_gb300 import ddtm
    return ddtm


@pytest.fixture(scope="module")
def fields():
    U = synth.gauge_field(DIMS, 0.3, seed=21)
    b = synth.gaussian_spinor(DIMS, seed=22, nrhs=3)
    return U, b, FineOperator(U.numpy(), KAPPA, CSW, 1)


def relerr(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))


def smooth(ddtm, ctx, b, prec, ncycles, nmr):
    n = b.shape[0]
    fb, fx = ddtm.ddtm_field_create(ctx, prec, n), ddtm.ddtm_field_create(ctx, prec, n)
    try:
        ddtm.ddtm_field_import(ctx, fb, b)
        ddtm.ddtm_sap_field(ctx, fx, fb, MU, ncycles, nmr)
        x = torch.zeros_like(b)
        ddtm.ddtm_field_export(ctx, fx, x)
        torch.cuda.synchronize()
        return x.cpu().numpy()
    finally:
        ddtm.ddtm_field_destroy(fb)
        ddtm.ddtm_field_destroy(fx)


@pytest.mark.parametrize("nmr", [0, 1, 5])
@pytest.mark.parametrize("nrhs", [1, 2, 3])
def test_sap_edges(lib, fields, nrhs, nmr):
    U, b, op = fields
    ctx = lib.ddtm_create(DIMS, BLOCK, 1)
    try:
        lib.ddtm_load_gauge(ctx, U.cuda(), KAPPA, CSW)
        ref = osap.sap(op, b[nrhs - 1].numpy(), MU, BLOCK, 2, nmr, eo=True)
        for prec in (1, 2):
            x = smooth(lib, ctx, b[:nrhs].cuda(), prec, 2, nmr)
            assert relerr(x[nrhs - 1], ref) < TOL[prec], (prec, relerr(x[nrhs - 1], ref))
    finally:
        lib.ddtm_destroy(ctx)


@pytest.mark.parametrize("nrhs", [1, 3])
def test_sap_f16_operator_when_memory_is_short(lib, fields, nrhs):
    """Under a memory cap that leaves no room for FP32 operator copies, FP16 fields are smoothed with
    FP16 copies; the cap costs accuracy of the storage, not the call."""
    U, b, op = fields
    ctx = lib.ddtm_create(DIMS, BLOCK, 1)
    try:
        lib.ddtm_load_gauge(ctx, U.cuda(), KAPPA, CSW)
        V = int(np.prod(DIMS))
        # FP16 links, clover and even-site inverses (432 B per site), the fields and the canonical staging
        lib.ddtm_set_memory_limit(lib.ddtm_memory_in_use() + V * (432 + 2 * nrhs * 52) + (1 << 16))
        x = smooth(lib, ctx, b[:nrhs].cuda(), 2, 2, 3)
        ref = osap.sap(op, b[nrhs - 1].numpy(), MU, BLOCK, 2, 3, eo=True)
        assert relerr(x[nrhs - 1], ref) < TOL[2]
    finally:
        lib.ddtm_set_memory_limit(0)
        lib.ddtm_destroy(ctx)


@pytest.mark.parametrize("nrhs", [1, 2, 3])
def test_dirac_edges(lib, fields, nrhs):
    U, b, op = fields
    ctx = lib.ddtm_create(DIMS, BLOCK, 1)
    try:
        lib.ddtm_load_gauge(ctx, U.cuda(), KAPPA, CSW)
        ref = op.apply(b[nrhs - 1].numpy(), MU)
        for prec in (1, 2):
            fx, fy = lib.ddtm_field_create(ctx, prec, nrhs), lib.ddtm_field_create(ctx, prec, nrhs)
            x = b[:nrhs].cuda()
            lib.ddtm_field_import(ctx, fx, x)
            lib.ddtm_apply_D_field(ctx, fy, fx, MU)
            y = torch.zeros_like(x)
            lib.ddtm_field_export(ctx, fy, y)
            torch.cuda.synchronize()
            lib.ddtm_field_destroy(fx)
            lib.ddtm_field_destroy(fy)
            assert relerr(y[nrhs - 1].cpu().numpy(), ref) < TOL[prec]
    finally:
        lib.ddtm_destroy(ctx)
