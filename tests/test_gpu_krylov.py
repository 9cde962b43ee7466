"""The coarsest even-odd GMRES on image-ordered vectors (csrc/krylov_tc.cu) at the edges of its launch shapes:
one right-hand side (padding columns, one CTA), a padded odd batch, dofs that do not fill a k group of 16, more
basis vectors than one shared-memory chunk, a restart, and more tiles than warps.  Every solution has to satisfy
D_c x = b to the requested tolerance, measured with ddtm_apply_Dc of the same operator.

Bound: the reduced system is solved to tol, its right-hand side is at most about twice b (||D_oe D_ee^-1|| is of
order one), and the FP16 operands of the products (unit roundoff 5e-4, a few dozen blocks) add up to 3e-3, the
margin of the coarse-solve parity test: 2 tol + 3e-3.
"""

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


# lattice, test vectors, right-hand sides, restart, tolerance
CASES = [
    ((16, 8, 8, 8), 24, 1, 100, 1e-1),
    ((16, 8, 8, 8), 21, 3, 100, 1e-2),
    ((16, 8, 8, 8), 21, 12, 25, 1e-2),
    ((16, 8, 8, 16), 24, 40, 100, 2e-3),
    ((32, 16, 16, 32), 24, 96, 100, 1e-1),
]


@pytest.mark.parametrize("dims,nv,nrhs,restart,tol", CASES)
def test_coarse_solve_shapes(lib, dims, nv, nrhs, restart, tol):
    mu = 0.004
    U = synth.gauge_field(dims, 0.2, seed=31, device="cuda")
    ctx = lib.ddtm_create(dims, (4, 4, 4, 4), 0)
    try:
        lib.ddtm_load_gauge(ctx, U, 0.134, 1.5755)
        p = lib.ddtm_get_params(ctx)
        p.nv[0], p.n_setup, p.post_smooth, p.coarse_prec = nv, 2, 2, lib.PREC_F16
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_setup(ctx, mu, 5)
        p.coarse_restart, p.coarse_max_restarts, p.coarse_tol = restart, 30, tol
        lib.ddtm_set_params(ctx, p)
        cl = (dims[0] // 4, dims[3] // 4, dims[2] // 4, dims[1] // 4)
        b = synth.gaussian_vectors((nrhs,) + cl + (2 * nv,), seed=32, device="cuda")
        x, y = torch.zeros_like(b), torch.zeros_like(b)
        iters, code = lib.ddtm_coarse_solve_batch(ctx, x, b, nrhs, 5.2 * mu)
        assert code == lib.OK and iters > 0
        lib.ddtm_apply_Dc(ctx, 1, y, x, nrhs, 5.2 * mu)
        res = torch.linalg.vector_norm((b - y).flatten(1), dim=1) / torch.linalg.vector_norm(b.flatten(1), dim=1)
        print(dims, nv, nrhs, "iterations", iters, "worst residual", float(res.max()))
        assert float(res.max()) < 2 * tol + 3e-3
        again = torch.zeros_like(b)
        assert lib.ddtm_coarse_solve_batch(ctx, again, b, nrhs, 5.2 * mu)[0] == iters
        assert torch.equal(x, again)  # fixed grids and summation orders
    finally:
        lib.ddtm_destroy(ctx)
