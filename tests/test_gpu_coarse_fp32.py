"""The FP32 coarse stencil and its even-odd steps at the edges of their launch shapes, against the CPU oracle: one column,
two, chunks of four that are full or not (odd and even numbers of right-hand sides), one and two units per hop, from 2 to
128 dofs; and the outer Gram-Schmidt over more than 32 basis vectors.  Tolerances as in the other parity tests: D_c
applications 1e-5, well-conditioned coarse solves to 1e-5 within 1e-4."""

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


@pytest.mark.parametrize("dims,block,nv,nrhs", [((8, 8, 8, 8), (4, 4, 4, 4), 1, 1), ((8, 8, 8, 8), (4, 4, 4, 4), 5, 2),
                                                ((8, 8, 8, 8), (4, 4, 4, 4), 24, 3), ((8, 8, 8, 8), (4, 4, 4, 4), 29, 6),
                                                ((8, 8, 8, 8), (4, 4, 4, 4), 57, 12), ((8, 8, 8, 8), (4, 4, 4, 4), 64, 9),
                                                ((8, 8, 8, 12), (2, 2, 2, 2), 5, 7)])
def test_apply_and_eo_solve(lib, dims, block, nv, nrhs):
    U = synth.gauge_field(dims, 0.3, seed=51)
    op = FineOperator(U.numpy(), 0.13, 1.2)
    v = synth.gaussian_vectors((nv,) + op.lat + (4, 3), seed=52)
    ctx = lib.ddtm_create(dims, block, 0)
    try:
        lib.ddtm_load_gauge(ctx, U.cuda(), 0.13, 1.2)
        p = lib.ddtm_get_params(ctx)
        p.nv[0], p.coarse_prec, p.coarse_tol = nv, lib.PREC_F32, 1e-5
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_set_test_vectors(ctx, 0, v.cuda(), nv)
        cop = ocoarse.build_coarse_operator(op, aggregation.build_P(op, v.numpy(), block), block)
        x = synth.gaussian_vectors((nrhs,) + cop.lat + (2 * nv,), seed=53)
        y = torch.zeros_like(x).cuda()
        lib.ddtm_apply_Dc(ctx, 1, y, x.cuda(), nrhs, 0.02)
        for r in range(nrhs):
            assert relerr(y[r].cpu().numpy(), cop.apply(x[r].numpy(), 0.02)) < 1e-5
        if nv > 42:  # the inverses of larger self blocks exceed the shared memory
            return
        s = torch.zeros_like(x).cuda()
        iters, code = lib.ddtm_coarse_solve_batch(ctx, s, x.cuda(), nrhs, 0.5)
        assert code == lib.OK and iters > 0
        for r in range(nrhs):
            assert relerr(cop.apply(s[r].cpu().numpy(), 0.5), x[r].numpy()) < 1e-4
    finally:
        lib.ddtm_destroy(ctx)


@pytest.mark.parametrize("dims,block", [((16, 8, 8, 8), (4, 4, 4, 4)), ((12, 4, 4, 4), (2, 2, 2, 2))])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_outer_gram_schmidt_long_cycles(lib, dims, block, nrhs):
    """A poor preconditioner (one test vector) makes outer cycles of far more than 32 basis vectors: the FP32 cycle stays
    orthogonal, so that it takes no more iterations to 1e-6 than the FP64 cycle (but for two, for its rounding)."""
    U = synth.gauge_field(dims, 0.2, seed=61, device="cuda")
    iters = {}
    for prec in (lib.PREC_F32, lib.PREC_F64):
        ctx = lib.ddtm_create(dims, block, 0)
        try:
            lib.ddtm_load_gauge(ctx, U, 0.134, 1.5755)
            p = lib.ddtm_get_params(ctx)
            p.nv[0], p.n_setup, p.post_smooth, p.nmr = 1, 1, 1, 1
            p.coarse_prec, p.smoother_prec = lib.PREC_F32, prec
            p.outer_restart, p.outer_tol, p.restart_tol = 100, 1e-6, 1e-6
            lib.ddtm_set_params(ctx, p)
            lib.ddtm_setup(ctx, 0.003, 5)
            b = synth.gaussian_spinor(dims, seed=62, nrhs=nrhs, device="cuda")
            x, y = torch.zeros_like(b), torch.zeros_like(b)
            info, code = lib.ddtm_solve(ctx, x, b, nrhs, 0.003)
            assert code == lib.OK
            lib.ddtm_apply_D(ctx, y, x, nrhs, 0.003, lib.PREC_F64)
            res = torch.linalg.vector_norm((b - y).reshape(nrhs, -1), dim=1) / torch.linalg.vector_norm(b.reshape(nrhs, -1), dim=1)
            assert float(res.max()) <= 1.001e-6
            assert abs(float(res.max()) - info.max_relres) < 1e-9
            iters[prec] = info.iters
        finally:
            lib.ddtm_destroy(ctx)
    assert iters[lib.PREC_F64] > 32 and iters[lib.PREC_F32] <= iters[lib.PREC_F64] + 2
