"""Aggregation and the FP16-storage Galerkin product at the edges of their launch shapes, against the CPU oracle: 17 or
fewer vectors (all in shared memory), 24, 28 and 32 (some in registers; chunks of 32, 16 and 8 sites in the Galerkin
kernel), an odd number, and blocks of 16 and 64 sites, antiperiodic in t.  Tolerances as in the other parity tests: P
2e-6 (FP32 storage), D_c applications 2e-3 (FP16 operands)."""

import numpy as np
import pytest
import torch

from oracle import aggregation, coarse as ocoarse
from oracle.operators import FineOperator
from paper_1610_02370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1610_02370_gb300 import build
    build.build()
    from paper_1610_02370_gb300 import ddtm
    return ddtm


def relerr(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))


@pytest.mark.parametrize("dims,block,nv", [((8, 8, 8, 8), (4, 4, 4, 4), 9), ((8, 8, 8, 8), (4, 4, 4, 4), 24),
                                           ((8, 8, 8, 8), (4, 4, 4, 4), 28), ((8, 8, 8, 8), (4, 4, 4, 4), 32),
                                           ((8, 4, 4, 8), (2, 2, 2, 2), 5), ((8, 8, 8, 4), (4, 2, 4, 2), 21)])
def test_aggregation_and_galerkin(lib, dims, block, nv):
    U = synth.gauge_field(dims, 0.3, seed=41)
    op = FineOperator(U.numpy(), 0.13, 1.2, 1)
    v = synth.gaussian_vectors((nv,) + op.lat + (4, 3), seed=42)
    ctx = lib.ddtm_create(dims, block, 1)
    try:
        lib.ddtm_load_gauge(ctx, U.cuda(), 0.13, 1.2)
        p = lib.ddtm_get_params(ctx)
        p.nv[0], p.coarse_prec = nv, lib.PREC_F16
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_set_test_vectors(ctx, 0, v.cuda(), nv)
        W = aggregation.build_P(op, v.numpy(), block)
        got = torch.zeros((2, nv) + op.lat + (4, 3), dtype=torch.complex128, device="cuda")
        lib.ddtm_get_prolongator(ctx, 0, got)
        assert relerr(got.cpu().numpy(), W) < 2e-6
        cop = ocoarse.build_coarse_operator(op, W, block)
        x = synth.gaussian_vectors((2,) + cop.lat + (2 * nv,), seed=43)
        y = torch.zeros_like(x).cuda()
        lib.ddtm_apply_Dc(ctx, 1, y, x.cuda(), 2, 0.02)
        for r in range(2):
            assert relerr(y[r].cpu().numpy(), cop.apply(x[r].numpy(), 0.02)) < 2e-3
    finally:
        lib.ddtm_destroy(ctx)


@pytest.mark.parametrize("nv,nrhs", [(24, 1), (21, 5), (9, 40)])
def test_coarse_apply_in_place_and_host(lib, nv, nrhs):
    """D_c x from device arrays (straight between canonical vectors and operand images), in place and from host arrays
    (through the interleaved batch) is the same, bit for bit."""
    dims = (8, 8, 8, 16)
    U = synth.gauge_field(dims, 0.3, seed=44).cuda()
    ctx = lib.ddtm_create(dims, (4, 4, 4, 4), 0)
    try:
        lib.ddtm_load_gauge(ctx, U, 0.13, 1.2)
        p = lib.ddtm_get_params(ctx)
        p.nv[0], p.coarse_prec = nv, lib.PREC_F16
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_set_test_vectors(ctx, 0, synth.gaussian_vectors((nv, 8, 16, 8, 8, 4, 3), seed=45).cuda(), nv)
        x = synth.gaussian_vectors((nrhs, 2, 4, 2, 2, 2 * nv), seed=46)
        y = torch.zeros_like(x).cuda()
        lib.ddtm_apply_Dc(ctx, 1, y, x.cuda(), nrhs, 0.03)
        z = x.cuda()
        lib.ddtm_apply_Dc(ctx, 1, z, z, nrhs, 0.03)
        h = torch.zeros_like(x)
        lib.ddtm_apply_Dc(ctx, 1, h, x, nrhs, 0.03)
        assert torch.equal(y, z) and torch.equal(y.cpu(), h)
    finally:
        lib.ddtm_destroy(ctx)
