"""The FP32 blocks of D_c that the Galerkin product of FP16 coarse storage leaves (before they become FP16 operand images),
against 64-bit arithmetic on the same operands: columns of P in FP32, its rows rounded to FP16 where an aggregate's rows fit
in shared memory (4^4 aggregates: up to 30 vectors) and in FP32 beyond.

Bound: u = 2^-24.  A column's stencil is FP32 (at most 8 hops of 3 complex products and the site term: about 50 roundings,
sqrt(50) u in the norm, averaged over the 6 Vb entries that an element sums), and a sum of 6 Vb complex products rounded
to nearest in FP32, by lanes and a tree, carries sqrt(12 Vb / 32 + 5) u, as in test_gpu_transfer_exact.py.  Sums that are
cut off instead of rounded miss this by a factor of ten to forty."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from oracle import blocks
from oracle.operators import FineOperator
from paper_1610_02370_gb300 import synth

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


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


def galerkin64(op, left, W, block):
    """Blocks (9,) + coarse lattice + (n, n) of left^+ D_W W."""
    nv = W.shape[1]
    cl = blocks.coarse_lat(op.lat, block)
    out = np.zeros((9,) + cl + (2 * nv, 2 * nv), complex)
    masks = [blocks.crossing_mask(op.lat, block, d, sg).reshape(op.lat + (1, 1)) for d in range(4) for sg in (1, -1)]
    for s in range(2):
        for j in range(nv):
            phi = W[s, j]
            hops = [op.hop_dir(phi, d, sg) for d in range(4) for sg in (1, -1)]
            parts = [op.site(phi, 0.0) + sum(h * ~m for h, m in zip(hops, masks))] + [h * m for h, m in zip(hops, masks)]
            for k, part in enumerate(parts):
                rows = blocks.block_sum_keep(np.conj(left) * part, op.lat, block, 2)
                out[k][..., :, s * nv + j] = np.moveaxis(rows.reshape((2 * nv,) + cl), 0, -1)
    return out


# one and two tiles of 16 x 8 per warp, chunks of 32, 16 and 8 sites, small and odd blocks, odd numbers of vectors
@pytest.mark.parametrize("dims,block,nv,rows16", [((8, 8, 8, 8), (4, 4, 4, 4), 1, True), ((8, 8, 8, 8), (4, 4, 4, 4), 9, True),
                                                  ((8, 8, 8, 8), (4, 4, 4, 4), 24, True), ((8, 8, 8, 8), (4, 4, 4, 4), 30, True),
                                                  ((8, 8, 8, 8), (4, 4, 4, 4), 31, False), ((8, 8, 8, 8), (4, 4, 4, 4), 32, False),
                                                  ((8, 4, 4, 8), (2, 2, 2, 2), 5, True), ((8, 4, 4, 8), (2, 2, 2, 2), 32, True),
                                                  ((8, 8, 8, 4), (4, 2, 4, 2), 21, True)])
def test_galerkin_blocks(libs, dims, block, nv, rows16):
    lib, ik = libs
    U = synth.gauge_field(dims, 0.2, seed=95)
    op = FineOperator(U.numpy(), 0.134, 1.5755, 0)
    ctx = lib.ddtm_create(dims, block, 0)
    try:
        lib.ddtm_load_gauge(ctx, U.cuda(), 0.134, 1.5755)
        p = lib.ddtm_get_params(ctx)
        p.nv[0], p.coarse_prec = nv, lib.PREC_F16
        lib.ddtm_set_params(ctx, p)
        lib.ddtm_set_test_vectors(ctx, 0, synth.gaussian_vectors((nv,) + op.lat + (4, 3), seed=96).cuda(), nv)
        W = torch.zeros((2, nv) + op.lat + (4, 3), dtype=torch.complex128, device="cuda")
        lib.ddtm_get_prolongator(ctx, 0, W)
        left = torch.view_as_complex(torch.view_as_real(W).float().half().double()) if rows16 else W
        left = left.cpu().numpy()
        cl = blocks.coarse_lat(op.lat, block)
        Nc, n = int(np.prod(cl)), 2 * nv
        got = torch.zeros(Nc, 9, n, n, 2, device="cuda")  # [site][part][column][row]
        assert ik.ik_coarse_blocks(ctx, ctypes.c_void_p(got.data_ptr())) == 0
        got = torch.view_as_complex(got.double()).cpu().numpy().transpose(1, 0, 3, 2)
    finally:
        lib.ddtm_destroy(ctx)
    ref = galerkin64(op, left, W.cpu().numpy(), block).reshape(9, Nc, n, n)
    bound = U32 * ((12 * int(np.prod(block)) / 32 + 5) ** 0.5 + 50 ** 0.5)
    rel = [float(np.linalg.norm(g - r) / np.linalg.norm(r)) for g, r in zip(got, ref)]
    print(dims, block, nv, "relative errors of the self and hop blocks", rel, "bound", bound)
    assert max(rel) <= bound
