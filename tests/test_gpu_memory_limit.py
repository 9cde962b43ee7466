"""Under a memory limit the library keeps to the variants that need least: what the limit leaves room for is counted here from
the sizes of the arrays that a call cannot do without."""

import numpy as np
import pytest
import torch

from paper_1610_02370_gb300 import synth

pytestmark = pytest.mark.gpu

DIMS = (16, 16, 8, 8)
V = int(np.prod(DIMS))
SLACK = 1 << 16


@pytest.fixture(scope="module")
def lib():
    from paper_1610_02370_gb300 import build
    build.build()
    from paper_1610_02370_gb300 import ddtm
    return ddtm


@pytest.fixture()
def ctx(lib):
    h = lib.ddtm_create(DIMS, (4, 4, 4, 4), 0)
    try:
        lib.ddtm_load_gauge(h, synth.gauge_field(DIMS, 0.2, seed=101, device="cuda"), 0.134, 1.5755)
        yield h
    finally:
        lib.ddtm_set_memory_limit(0)
        lib.ddtm_destroy(h)


def limit(lib, nbytes):
    lib.ddtm_set_memory_limit(lib.ddtm_memory_in_use() + nbytes + SLACK)


def test_f16_smoothing_leaves_room_for_later_fields(lib, ctx):
    """FP16 links, clover and even-site inverses (432 B per site), two FP16 fields, and after the smoothing four FP64 ones
    (768 B per site): the FP32 copies (864) would fit when the smoother runs, and then the fields would not."""
    limit(lib, V * (432 + 2 * 52 + 4 * 192))
    b = synth.gaussian_spinor(DIMS, seed=102, nrhs=1, device="cuda")
    fb, fx = lib.ddtm_field_create(ctx, lib.PREC_F16, 1), lib.ddtm_field_create(ctx, lib.PREC_F16, 1)
    lib.ddtm_field_import(ctx, fb, b)
    lib.ddtm_sap_field(ctx, fx, fb, 0.003, 2, 3)
    later = [lib.ddtm_field_create(ctx, lib.PREC_F64, 1) for _ in range(4)]
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    lib.ddtm_field_export(ctx, fx, x)
    lib.ddtm_set_memory_limit(0)
    lib.ddtm_apply_D(ctx, y, x, 1, 0.003, lib.PREC_F64)
    assert float((b - y).norm() / b.norm()) < 0.7  # it did smooth
    for f in [fb, fx] + later:
        lib.ddtm_field_destroy(f)


def test_setup_and_solve_fit_in_what_they_need(lib):
    """The peak of a setup and a solve with FP16 smoothing, first without a limit, then in a new context under a limit of the
    same hierarchy and workspace with FP16 operator copies (144 B per site of inverses instead of 288)."""
    def run(ctx):
        p = lib.ddtm_get_params(ctx)
        p.nv[0], p.n_setup, p.post_smooth, p.coarse_prec = 20, 3, 2, lib.PREC_F16
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_setup(ctx, 0.003, 3)
        b = synth.gaussian_spinor(DIMS, seed=103, nrhs=2, device="cuda")
        x = torch.zeros_like(b)
        info, code = lib.ddtm_solve(ctx, x, b, 2, 0.003)
        assert code == lib.OK and info.max_relres <= 1e-10
        return x

    U = synth.gauge_field(DIMS, 0.2, seed=101, device="cuda")
    used = []
    for capped in (False, True):
        ctx = lib.ddtm_create(DIMS, (4, 4, 4, 4), 0)
        try:
            before = lib.ddtm_memory_in_use()
            if capped:
                limit(lib, used[0] - V * 144)
            lib.ddtm_load_gauge(ctx, U, 0.134, 1.5755)
            run(ctx)
            used.append(lib.ddtm_memory_in_use() - before)
        finally:
            lib.ddtm_set_memory_limit(0)
            lib.ddtm_destroy(ctx)
    assert used[1] <= used[0] - V * 144 + SLACK


@pytest.mark.parametrize("loc", ["cuda", "cpu"])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_canonical_calls_of_many_vectors(lib, ctx, prec, loc):
    """Operator copies, two fields of one right-hand side, and host arrays staged one vector each way: that is enough for
    twelve right-hand sides, and the same bits as without a limit."""
    one = {0: 192, 1: 96, 2: 52}[prec]
    b = synth.gaussian_spinor(DIMS, seed=104, nrhs=12, device=loc)
    want = []
    for limited in (False, True):
        for f in (lambda y: lib.ddtm_apply_D(ctx, y, b, 12, 0.003, prec),
                  lambda y: lib.ddtm_sap(ctx, y, b, 12, 0.003, 2, 3, prec)):
            y = torch.zeros_like(b)
            if limited:  # the operator copies are there from the calls before
                limit(lib, V * (2 * one + (2 * 192 if loc == "cpu" else 0)))
            f(y)
            torch.cuda.synchronize()
            lib.ddtm_set_memory_limit(0)
            want.append(y)
        lib.ddtm_release_workspace(ctx)
    assert torch.equal(want[0], want[2]) and torch.equal(want[1], want[3])


def hierarchy(lib, ctx, nv):
    p = lib.ddtm_get_params(ctx)
    p.nv[0], p.coarse_prec, p.coarse_tol = nv, lib.PREC_F16, 1e-2
    lib.ddtm_set_params(ctx, p)
    lat = (DIMS[0], DIMS[3], DIMS[2], DIMS[1])
    lib.ddtm_set_test_vectors(ctx, 0, synth.gaussian_vectors((nv,) + lat + (4, 3), seed=105, device="cuda"), nv)
    return p, synth.gaussian_vectors((1,) + tuple(n // 4 for n in lat) + (2 * nv,), seed=106, device="cuda")


def test_coarse_calls_of_one_vector(lib, ctx):
    """The FP16 operand image (8 columns of 48 padded dofs), two interleaved batches of one column, and for the solve the
    basis of one column: image order pads the vectors to four columns."""
    nv = 20
    n, Nc, m = 2 * nv, V // 256, 100
    p, b = hierarchy(lib, ctx, nv)
    want, x = torch.zeros_like(b), torch.zeros_like(b)
    lib.ddtm_apply_Dc(ctx, 1, want, b, 1, 0.02)
    p.coarse_restart = 1
    lib.ddtm_set_params(ctx, p)
    lib.ddtm_coarse_solve(ctx, x, b, 0.02)  # the inverses of the even sites belong to the operator
    p.coarse_restart = m
    lib.ddtm_set_params(ctx, p)
    lib.ddtm_release_workspace(ctx)

    image = Nc * 8 * 48 * 2
    limit(lib, image + 2 * Nc * n * 8)
    y = torch.zeros_like(b)
    lib.ddtm_apply_Dc(ctx, 1, y, b, 1, 0.02)
    assert torch.equal(y, want)
    lib.ddtm_set_memory_limit(0)
    lib.ddtm_release_workspace(ctx)

    # basis in FP16, eleven batches on half of the sites or their equivalent, both images, Krylov scalars
    limit(lib, (m + 1) * Nc // 2 * n * 4 + 11 * Nc // 2 * n * 8 + image + (m + 1) * (m + 8) * 16 + (1 << 20))
    iters, code = lib.ddtm_coarse_solve(ctx, x, b, 0.02)
    assert code == lib.OK and iters > 0
    lib.ddtm_set_memory_limit(0)
    lib.ddtm_apply_Dc(ctx, 1, y, x, 1, 0.02)
    assert float((b - y).norm() / b.norm()) < 2e-2 + 3e-3


def test_spare_buffers_make_room(lib, ctx):
    """What a coarse solve keeps only for speed is given back when another call needs the memory, and taken again later."""
    p, b = hierarchy(lib, ctx, 24)
    x, x2 = torch.zeros_like(b), torch.zeros_like(b)
    iters, code = lib.ddtm_coarse_solve(ctx, x, b, 0.02)
    assert code == lib.OK
    basis = 101 * (V // 512) * 8 * 48 * 2
    nrhs = basis // (V * 192) + 1  # the fields take more than the free room, and less than that and the basis
    limit(lib, nrhs * V * 192 - basis // 2)
    f = lib.ddtm_field_create(ctx, lib.PREC_F64, nrhs)
    lib.ddtm_field_destroy(f)
    lib.ddtm_set_memory_limit(0)
    assert lib.ddtm_coarse_solve(ctx, x2, b, 0.02) == (iters, code)
    assert torch.equal(x, x2)
