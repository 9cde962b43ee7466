"""Restriction and prolongation of FP16 fields with the FP16 copy of P (the transfers of an FP16 smoother, which the C ABI
reaches only inside solves) against 64-bit sums of the same operands, entry by entry.

u = 2^-24.  An entry of the restriction sums 6 Vb complex products, 12 Vb / 32 real ones per lane in a chain, then five
levels of a warp sum: n = 12 Vb / 32 + 5 roundings and one of the scaled field entry.  Worst case per entry: (n + 1) u times
the sum of the absolute products.  In the norm the roundings are independent, each at most u of a partial sum:
sqrt(n) u (sums that are cut off instead of rounded add up to n u / 2 and more).  An entry of the prolongation
sums 2 nv real products (n = 2 nv + 1, + 2 with add) and is stored in FP16 relative to the site's largest component:
half a unit of 11 bits of the entry, or half of the smallest subnormal, 2^-25, of the scale."""

import ctypes
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def ik(tmp_path_factory):
    from paper_1610_02370_gb300 import build
    lib = build.build()
    so = str(tmp_path_factory.mktemp("ik") / "internal_kernels.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "internal_kernels.cu")
    subprocess.check_call([build._nvcc(), "-shared", src, "-o", so] + build.ARCH + build.FLAGS +
                          ["-I", build.CSRC, lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)])
    return ctypes.CDLL(so)


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def draw(gen, *shape):
    return torch.randn(*shape, 2, generator=gen, dtype=torch.float64, device="cuda")


def cplx(x):
    return torch.view_as_complex(x.double().contiguous())


def operands(Vb, Nb, nv, R, seed):
    """P with columns of norm about one, and FP16 fields with scales over four orders of magnitude."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    P = (draw(gen, Nb, 2, nv, 6, Vb) / (12 * Vb) ** 0.5).half().contiguous()
    psi = draw(gen, R, Nb, 12, Vb) * 10.0 ** (4 * torch.rand(R, Nb, 1, Vb, 1, generator=gen, dtype=torch.float64, device="cuda") - 2)
    scale = psi.abs().amax(dim=(2, 4)).float().contiguous()
    h = (psi / scale.double()[:, :, None, :, None]).half().contiguous()
    return gen, P, h, scale


SHAPES = [(256, 32, 1, 1), (256, 32, 12, 3), (256, 32, 21, 8), (256, 32, 24, 9), (256, 32, 32, 17), (256, 32, 40, 1),
          (16, 64, 21, 3), (16, 64, 32, 9), (64, 32, 12, 1), (64, 32, 24, 17)]


@pytest.mark.parametrize("Vb,Nb,nv,R", SHAPES)
def test_restrict(ik, Vb, Nb, nv, R):
    _, P, h, scale = operands(Vb, Nb, nv, R, 91)
    Rs = (R + 3) // 4 * 4

    def restrict(h, scale, R, Rs):
        c = torch.full((Nb, 2 * nv, Rs, 2), 7.0, device="cuda")
        assert ik.ik_restrict(Vb, Nb, ptr(c), ptr(h), ptr(scale), ptr(P), nv, R, Rs) == 0
        assert bool((c[:, :, R:] == 7.0).all())  # columns beyond R are left alone
        return c[:, :, :R]

    c = restrict(h, scale, R, Rs)
    p, psi = cplx(P), (cplx(h) * scale.double()[:, :, None, :]).view(R, Nb, 2, 6, Vb)
    ref = torch.einsum("bsicx,rbscx->bsir", p.conj(), psi).reshape(Nb, 2 * nv, R)
    err = (cplx(c) - ref).abs()
    size = torch.einsum("bsicx,rbscx->bsir", p.abs(), psi.abs()).reshape(Nb, 2 * nv, R)
    n = 12 * Vb // 32 + 5
    # |p| |psi| bounds both |re re| + |im im| and |re im| + |im re|; sqrt 2 for the two parts of the error
    assert float((err / ((n + 1) * U32 * 2 ** 0.5 * size)).max()) <= 1.0
    rel = float(err.norm() / ref.norm())
    print(Vb, nv, R, "restrict", rel)
    assert rel <= U32 * n ** 0.5
    for r in range(0, R, 4):  # a right-hand side of a batch has the bits it has alone
        assert torch.equal(restrict(h[r:r + 1].contiguous(), scale[r:r + 1].contiguous(), 1, 1)[:, :, 0], c[:, :, r])


@pytest.mark.parametrize("add", [0, 1])
@pytest.mark.parametrize("Vb,Nb,nv,R", SHAPES)
def test_prolong(ik, Vb, Nb, nv, R, add):
    gen, P, h, scale = operands(Vb, Nb, nv, R, 92)
    Rs = (R + 3) // 4 * 4
    e = draw(gen, Nb, 2 * nv, Rs).float().contiguous()

    def prolong(h, scale, e, R, Rs):
        x, xn = h.clone(), scale.clone()
        assert ik.ik_prolong(Vb, Nb, ptr(x), ptr(xn), ptr(e), ptr(P), nv, R, Rs, add) == 0
        return x, xn

    x, xn = prolong(h, scale, e, R, Rs)
    p, ce = cplx(P), cplx(e)[:, :, :R].reshape(Nb, 2, nv, R)
    old = cplx(h) * scale.double()[:, :, None, :]
    ref = torch.einsum("bsicx,bsir->rbscx", p, ce).reshape(R, Nb, 12, Vb) + (old if add else 0)
    size = torch.einsum("bsicx,bsir->rbscx", p.abs(), ce.abs()).reshape(R, Nb, 12, Vb) + (old.abs() if add else 0)
    got = cplx(x) * xn.double()[:, :, None, :]
    sums = (2 * nv + 3 + 2) * U32 * size  # + 2: the scale and its reciprocal
    top = torch.view_as_real(ref).abs().amax(dim=(2, 4))
    sum_top = sums.amax(dim=2)
    assert float(((xn - top).abs() / sum_top).max()) <= 1.0
    err = torch.view_as_real(got - ref).abs()
    bound = (2.0 ** -11 * torch.view_as_real(ref).abs() * (1 + 2.0 ** -10) + 2.0 ** -25 * top[:, :, None, :, None] +
             sums[..., None] * (1 + 2.0 ** -10))
    assert float((err / bound).max()) <= 1.0
    for r in range(0, R, 4):
        x1, n1 = prolong(h[r:r + 1].contiguous(), scale[r:r + 1].contiguous(), e[:, :, r:r + 1].contiguous(), 1, 1)
        assert torch.equal(x1[0], x[r]) and torch.equal(n1[0], xn[r])
