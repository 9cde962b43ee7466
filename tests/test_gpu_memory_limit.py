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
