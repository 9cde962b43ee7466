"""Solves whose FP16 transfers run on the matrix instructions, at the edges of their tiles: fewer than 16 vectors,
an odd number, more than 32 (with the FP32 coarse operator, which allows them), one right-hand side and more than two
column tiles.  The transfers only precondition, so the check is the solution (FP64 residual 1e-10) in about as many outer
iterations as with FP32 transfers (a preconditioner with a wrong entry does not converge at that rate)."""

import pytest
import torch

from paper_1610_02370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1610_02370_gb300 import build
    build.build()
    from paper_1610_02370_gb300 import ddtm
    return ddtm


@pytest.mark.parametrize("nv,nrhs,coarse_prec", [(12, 1, 2), (21, 17, 2), (40, 3, 1)])
def test_solve_with_f16_transfers(lib, nv, nrhs, coarse_prec):
    dims, mu = (16, 8, 8, 8), 0.01
    U = synth.gauge_field(dims, 0.2, seed=51).cuda()
    b = synth.gaussian_spinor(dims, seed=52, nrhs=nrhs).cuda()
    iters = {}
    for smoother in (lib.PREC_F32, lib.PREC_F16):
        ctx = lib.ddtm_create(dims, (4, 4, 4, 4), 1)
        try:
            lib.ddtm_load_gauge(ctx, U, 0.134, 1.5755)
            p = lib.ddtm_get_params(ctx)
            p.nv[0], p.n_setup, p.post_smooth, p.coarse_prec, p.smoother_prec = nv, 3, 2, coarse_prec, smoother
            lib.ddtm_set_params(ctx, p)
            lib.ddtm_setup(ctx, mu, 7)
            x = torch.zeros_like(b)
            info, code = lib.ddtm_solve(ctx, x, b, nrhs, mu)
            assert code == lib.OK and info.max_relres <= 1e-10
            iters[smoother] = info.iters
        finally:
            lib.ddtm_destroy(ctx)
    print("outer iterations FP32 / FP16 smoother:", iters)
    assert iters[lib.PREC_F16] <= iters[lib.PREC_F32] + 3
