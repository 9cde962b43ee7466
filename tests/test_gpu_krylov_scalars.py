"""Scalars of the coarsest even-odd GMRES on image-ordered vectors: the reciprocal square root of the norms, right-hand sides of
very different size (and zero) in one batch, and a coefficient block that no CTA can stage."""

import ctypes
import os
import subprocess

import pytest
import torch

from paper_1610_02370_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    from paper_1610_02370_gb300 import build
    so_path = build.build()
    from paper_1610_02370_gb300 import ddtm
    so = str(tmp_path_factory.mktemp("ik") / "internal_kernels.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "internal_kernels.cu")
    subprocess.check_call([build._nvcc(), "-shared", src, "-o", so] + build.ARCH + build.FLAGS +
                          ["-I", build.CSRC, so_path, "-Xlinker", "-rpath=" + os.path.dirname(so_path)])
    return ddtm, ctypes.CDLL(so)


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def test_inv_sqrt(libs):
    """Against 1 / sqrt(x) in FP64, on both sides of the switches at 1e-30 and 1e30 and out to subnormal numbers and the
    largest.  The last Newton step leaves the rounding of x y (1/2 unit of 2^-53 after halving) and its own (1 unit), the
    reference two more: 4 units of 2^-53."""
    _, ik = libs
    gen = torch.Generator().manual_seed(3)
    x = torch.cat([10.0 ** (600 * torch.rand(20000, generator=gen, dtype=torch.float64) - 300),
                   10.0 ** (62 * torch.rand(20000, generator=gen, dtype=torch.float64) - 31),
                   torch.tensor([1e-30, 1e30, 5e-324, 2.2e-308, 1.7e308, 1.0, 4.0, 1.0 - 2.0 ** -53], dtype=torch.float64)])
    for s in (1e-30, 1e30, 2.0 ** -100, 2.0 ** 100):
        x = torch.cat([x, torch.nextafter(torch.tensor([s, s], dtype=torch.float64), torch.tensor([0.0, 1e300], dtype=torch.float64))])
    x = x.cuda()
    y = torch.zeros_like(x)
    assert ik.ik_inv_sqrt(ptr(x), ptr(y), x.numel()) == 0
    assert float((y * torch.sqrt(x) - 1).abs().max()) <= 4 * 2.0 ** -53


def test_right_hand_sides_of_any_size(libs):
    """Columns scaled by powers of two from 2^-50 to 2^40 and a zero column: every column has the bits of the unscaled one
    (no rounding depends on the scale: norms are squares of FP32 numbers within their range) and the zero one gives zero."""
    lib, _ = libs
    dims, nv, mu = (8, 8, 8, 16), 24, 0.02
    scales = [1.0, 2.0 ** -50, 2.0 ** 40, 0.0, 2.0 ** -20, 2.0 ** 13, 1.0, 0.0]
    ctx = lib.ddtm_create(dims, (4, 4, 4, 4), 0)
    try:
        lib.ddtm_load_gauge(ctx, synth.gauge_field(dims, 0.2, seed=111).cuda(), 0.134, 1.5755)
        p = lib.ddtm_get_params(ctx)
        p.nv[0], p.coarse_prec, p.coarse_tol = nv, lib.PREC_F16, 1e-2
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_set_test_vectors(ctx, 0, synth.gaussian_vectors((nv, 8, 16, 8, 8, 4, 3), seed=112).cuda(), nv)
        b1 = synth.gaussian_vectors((2, 4, 2, 2, 2 * nv), seed=113).cuda()
        b = torch.stack([s * b1 for s in scales])
        x = torch.zeros_like(b)
        iters, code = lib.ddtm_coarse_solve_batch(ctx, x, b, len(scales), mu)
        assert code == lib.OK and iters > 0
        for s, xs in zip(scales, x):
            assert torch.equal(xs, s * x[0]), s
        y = torch.zeros_like(b1)
        lib.ddtm_apply_Dc(ctx, 1, y, x[0].contiguous(), 1, mu)
        assert float((b1 - y).norm() / b1.norm()) < 2e-2 + 3e-3
        zero = torch.zeros_like(b)
        assert lib.ddtm_coarse_solve_batch(ctx, x, zero, len(scales), mu) == (0, lib.OK)
        assert torch.equal(x, zero)
    finally:
        lib.ddtm_destroy(ctx)


def test_coefficient_block_too_large(libs):
    """250 basis vectors of 256 right-hand sides: refused like every coefficient block that exceeds the shared memory, and the
    next call is not affected.  A block that fits: FP32 sums of 100 products, 100 u of the absolute ones."""
    lib, ik = libs
    n, R, nsites = 8, 256, 1
    entries = nsites * R * 2 * 16
    V = torch.zeros(250, entries, dtype=torch.float16, device="cuda")
    x = torch.zeros(entries, device="cuda")
    y = torch.zeros(250, R, 2, dtype=torch.float64, device="cuda")
    assert ik.ik_img_combine(ptr(x), ptr(V), 250, ptr(y), n, R, nsites) == lib.ERR_ARG
    V.copy_(torch.randn(V.shape, generator=torch.Generator().manual_seed(5)))
    y.copy_(torch.randn(y.shape, generator=torch.Generator().manual_seed(6), dtype=torch.float64))
    x0 = torch.randn(entries, generator=torch.Generator().manual_seed(7)).cuda()
    x.copy_(x0)
    assert ik.ik_img_combine(ptr(x), ptr(V), 50, ptr(y), n, R, nsites) == 0
    # 8 dofs padded to 16: [group of 4 columns][k group][column][8 real, 8 imaginary parts]
    def split(t):
        t = t.double().view(t.shape[:-1] + (R // 4, 2, 4, 2, 8))
        return torch.complex(t[..., 0, :], t[..., 1, :])
    c = torch.view_as_complex(y[:50].float().double()).view(50, R // 4, 1, 4, 1)
    ref = split(x0) + (c * split(V[:50])).sum(0)
    size = split(x0).abs() + (c.abs() * split(V[:50]).abs()).sum(0)
    assert float(((split(x) - ref).abs() / (100 * 2.0 ** -24 * size)).max()) <= 1.0
