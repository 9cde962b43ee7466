// Coarse operator D_c(mu) = P^dagger D P + i mu Gamma5_c (Sec. 2.3): Galerkin
// build, stencil, even-odd reduction pieces, and the self-block inverses of
// the even-odd coarsest solve (Sec. 2.5).
//
// Storage: Dc[((x*9 + d)*n + col)*n + row], complex FP32, n = 2 nv,
// d = 0 self (without the twist), d = 1 + k for hop k = 2 mu + (0 fwd, 1 bwd):
// the block coupling site x to its neighbour in direction +mu (k even) or
// -mu (k odd).  Column-major blocks make the per-row threads of the stencil
// read consecutive addresses.  The twist i mu_c Gamma5_c (Gamma5_c = +1 on
// dofs < nv, -1 above) is added on the fly, so one build serves +mu, -mu and
// the shifted coarsest twist delta*mu.  With FP16 coarse storage the stencil
// of the coarsest solve runs on tensor cores from FP16 images of these blocks
// (coarse_tc.cu); the FP32 blocks stay for the rest.
#include "common.cuh"
#include "ddtm_internal.h"
#include "timer.h"
#include "coarse.h"
#include "launch_shape.h"

namespace ddtm {

template <typename DS> __device__ __forceinline__ cplx<float> ldD(const DS* p);
template <> __device__ __forceinline__ cplx<float> ldD<float2>(const float2* p) { return ld(p); }
template <typename DS> __device__ __forceinline__ void stD(DS* p, cplx<float> v);
template <> __device__ __forceinline__ void stD<float2>(float2* p, cplx<float> v) { st(p, v); }

__device__ __forceinline__ size_t pix(int blk, int s, int i, int comp, int loc, int nv, int Vb) {
  return (((size_t)(blk * 2 + s) * nv + i) * 6 + comp) * Vb + loc;
}

// ---- Galerkin build ----------------------------------------------------------------
// One CTA per aggregate A, thread = site.  For every column (s', j) of P:
//   y0(x)  = S phi(x) + hops of phi that stay inside A          (self part)
//   yk(x)  = hop k of phi read in the neighbour aggregate, for x on face k
// with phi = column (s', j) of every aggregate; then
//   Dc[A][0][col][row]   = sum_{x in A} <P_row(x), y0(x)>
//   Dc[A][1+k][col][row] = sum_{x on face k} <P_row(x), yk(x)>
// Face k of a block = sites whose hop k leaves the block; faces are stored
// compactly (face_list / face_idx tables, offsets face_off).
struct FaceTables {
  const int* idx;   // [8][Vb]: slot of site in face k or -1
  const int* list;  // [face_off[8]]: site of each slot
  int off[9];
};

template <typename DS>
__global__ void k_galerkin(DS* __restrict__ Dc, const float2* __restrict__ P, Links<PREC_F32> U, Clover<PREC_F32> C,
                           Geo g, FaceTables f, int nv) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Vb = g.Vb;
  cplx<float>* y0 = reinterpret_cast<cplx<float>*>(smem_raw);  // [12][Vb]
  cplx<float>* yf = y0 + 12 * Vb;                                // [12][face slots]
  const int nf = f.off[8];
  const int A = blockIdx.x;
  const int n = 2 * nv;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int col = 0; col < n; col++) {
    const int sp = col / nv, j = col - sp * nv;
    for (int loc = threadIdx.x; loc < Vb; loc += blockDim.x) {
      cplx<float> phi[12], acc[12], out[12];
#pragma unroll
      for (int c = 0; c < 12; c++) { phi[c] = cplx<float>(0, 0); acc[c] = cplx<float>(0, 0); }
      for (int comp = 0; comp < 6; comp++) phi[6 * sp + comp] = ld(P + pix(A, sp, j, comp, loc, nv, Vb));
      C.apply(A, loc, phi, out);
      for (int k = 0; k < 8; k++) {
        const int mu = k >> 1;
        const bool fwd = (k & 1) == 0;
        Nbr nb = neighbour(g, A, loc, k);
        cplx<float> p[12], h[6], wv[6], u[9];
#pragma unroll
        for (int c = 0; c < 12; c++) p[c] = cplx<float>(0, 0);
        for (int comp = 0; comp < 6; comp++) p[6 * sp + comp] = ld(P + pix(nb.blk, sp, j, comp, nb.loc, nv, Vb));
        project<float>(mu, fwd, p, h);
        if (fwd) { U.load(A, loc, mu, u); mul_U<float>(u, h, wv); }
        else { U.load(nb.blk, nb.loc, mu, u); mul_Udag<float>(u, h, wv); }
        if (nb.flip)
          for (int q = 0; q < 6; q++) wv[q] = -wv[q];
        if (!nb.cross) {
          reconstruct<float>(mu, fwd, wv, acc);
        } else {
          cplx<float> part[12];
#pragma unroll
          for (int c = 0; c < 12; c++) part[c] = cplx<float>(0, 0);
          reconstruct<float>(mu, fwd, wv, part);
          int slot = f.off[k] + f.idx[k * Vb + loc];
#pragma unroll
          for (int c = 0; c < 12; c++) yf[c * nf + slot] = -0.5f * part[c];
        }
      }
#pragma unroll
      for (int c = 0; c < 12; c++) y0[c * Vb + loc] = out[c] + (-0.5f) * acc[c];
    }
    __syncthreads();
    // projections: a warp takes GR rows of one block d (independent loads of
    // GR rows of P per step), the lanes stride over the sites
    const int GR = 4, ngr = (n + GR - 1) / GR;
    for (int o = w; o < 9 * ngr; o += nw) {
      const int d = o / ngr, r0 = (o - d * ngr) * GR;
      cplx<float> acc[GR];
      int sr[GR], ir[GR];
#pragma unroll
      for (int r = 0; r < GR; r++) {
        acc[r] = cplx<float>(0, 0);
        const int row = r0 + r < n ? r0 + r : n - 1;
        sr[r] = row / nv;
        ir[r] = row - sr[r] * nv;
      }
      if (d == 0) {
        for (int comp = 0; comp < 6; comp++)
#pragma unroll 4
          for (int loc = lane; loc < Vb; loc += 32)
#pragma unroll
            for (int r = 0; r < GR; r++)
              cmac_conj(acc[r], ld(P + pix(A, sr[r], ir[r], comp, loc, nv, Vb)), y0[(6 * sr[r] + comp) * Vb + loc]);
      } else {
        const int k = d - 1;
        for (int comp = 0; comp < 6; comp++)
#pragma unroll 2
          for (int q = f.off[k] + lane; q < f.off[k + 1]; q += 32) {
            const int fl = f.list[q];
#pragma unroll
            for (int r = 0; r < GR; r++)
              cmac_conj(acc[r], ld(P + pix(A, sr[r], ir[r], comp, fl, nv, Vb)), yf[(6 * sr[r] + comp) * nf + q]);
          }
      }
#pragma unroll
      for (int r = 0; r < GR; r++) {
        acc[r].re = warp_sum(acc[r].re);
        acc[r].im = warp_sum(acc[r].im);
        if (lane == 0 && r0 + r < n) stD(Dc + (((size_t)A * 9 + d) * n + col) * n + r0 + r, acc[r]);
      }
    }
    __syncthreads();
  }
}

// ---- Galerkin build with matrix instructions -----------------------------------------
// The same products, for FP16 coarse storage: one CTA per (aggregate A, row chirality s) keeps the nv rows of P on A
// as FP16 in shared memory and forms, for each part d (self, then the faces) and X sites at a time, the
// chirality-s components y of all n columns in FP32; their projections are a dense contraction
//   D[i][j] = sum over (component, site) conj(P_i) y_j
// done by mma.sync m16n8k8 in TF32: P's FP16 entries are exact in TF32, y goes in as hi + lo (22 bits), and the sums keep
// what the unit cuts off (mma_sum): 2.5e-8 against 64-bit sums of the same operands (8^4, 24 vectors), sums by FP32 lanes
// and warps 4.7e-8, one chain of accumulators 2.3e-5.  (The operands sit in registers and shared memory
// where the FP32 stencil leaves them; the contraction is 43 GFLOP at 16^3 x 32, a small part of the time, so the
// tensor-memory path would not pay for staging operand images.)  16^3 x 32, n = 48: 3.17 ms (2.75 without the cut parts),
// with FP32 projections out of shared memory 6.95 ms (17 loads per 32 multiply-adds and a warp reduction per entry); what
// is left is the latency of the P and link loads at 12 warps per SM.  Columns are spread over the threads X sites x
// (GM_THREADS / X) column groups, GM_CPT columns per thread sharing each link.
static const int GM_THREADS = 384, GM_CPT = 4;

__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// (s, e) += A (hi + lo), the sum in s and what its rounding left out in e.  The unit cuts a sum off towards zero, which in
// one chain of the 768 products of an entry adds up to 2e-5; forming the product once more on top of (old sum - new
// sum) gives back what was cut.
__device__ __forceinline__ void mma_sum(float (&s)[4], float (&e)[4], const uint32_t (&a)[4], uint32_t hi0, uint32_t hi1,
                                        uint32_t lo0, uint32_t lo1) {
  float t[4];
#pragma unroll
  for (int k = 0; k < 4; k++) t[k] = s[k];
  mma_tf32(t, a, hi0, hi1);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    e[k] = __fadd_rn(__fsub_rn(s[k], t[k]), e[k]);
    s[k] = t[k];
  }
  mma_tf32(e, a, hi0, hi1);
  mma_tf32(e, a, lo0, lo1);
}

// acc[cc] += chirality-s part of the hop (MU, FWD) of GM_CPT columns col0 + cc cstep read at (blk, loc) of P
// (columns beyond n repeat the last one; they are not stored)
template <int MU, bool FWD>
__device__ __forceinline__ void galerkin_hop(cplx<float> (&acc)[GM_CPT][6], const float2* __restrict__ P, const Links<PREC_F32>& U,
                                             float sign, int s, int A, int own, int blk, int loc, int nv, int Vb, int n,
                                             int col0, int cstep) {
  cplx<float> u[9];
  if (FWD) U.load(A, own, MU, u);
  else U.load(blk, loc, MU, u);
#pragma unroll
  for (int cc = 0; cc < GM_CPT; cc++) {
    const int col = col0 + cc * cstep < n ? col0 + cc * cstep : n - 1;
    const int sp = col >= nv ? 1 : 0, j = col - sp * nv;
    cplx<float> v[6], h[6], w[6];
    const float2* src = P + pix(blk, sp, j, 0, loc, nv, Vb);
#pragma unroll
    for (int c = 0; c < 6; c++) v[c] = ld(src + (size_t)c * Vb);
    // upper half of the projection: sp = 0 the column itself, sp = 1 -G l (forward), +G l (backward)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      cplx<float> g0, g1;
      apply_G<float>(MU, v[c], v[3 + c], g0, g1);
      h[c] = sp ? (FWD ? -g0 : g0) : v[c];
      h[3 + c] = sp ? (FWD ? -g1 : g1) : v[3 + c];
    }
    if (FWD) mul_U<float>(u, h, w);
    else mul_Udag<float>(u, h, w);
    // s = 0: w; s = 1: mu = 0 forward -w, backward w; mu = k forward G w, backward -G w
    const float q = s ? (((MU == 0) == FWD) ? -sign : sign) : sign;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      cplx<float> g0, g1;
      apply_G<float>(MU, w[c], w[3 + c], g0, g1);
      const cplx<float> o0 = s ? g0 : w[c], o1 = s ? g1 : w[3 + c];
      acc[cc][c].re = fmaf(q, o0.re, acc[cc][c].re);
      acc[cc][c].im = fmaf(q, o0.im, acc[cc][c].im);
      acc[cc][3 + c].re = fmaf(q, o1.re, acc[cc][3 + c].re);
      acc[cc][3 + c].im = fmaf(q, o1.im, acc[cc][3 + c].im);
    }
  }
}

// acc[cc] += site term (chirality s, packed at cp) of the columns of that chirality
__device__ __forceinline__ void galerkin_site(cplx<float> (&acc)[GM_CPT][6], const float2* __restrict__ P,
                                              const float2* __restrict__ cp, int s, int A, int loc, int nv, int Vb, int n,
                                              int col0, int cstep) {
  cplx<float> t[18];
#pragma unroll
  for (int q = 0; q < 18; q++) t[q] = ld(cp + (size_t)q * Vb);
#pragma unroll
  for (int cc = 0; cc < GM_CPT; cc++) {
    const int col = col0 + cc * cstep;
    if (col < n && (col >= nv) == (s == 1)) {
      cplx<float> v[6];
#pragma unroll
      for (int c = 0; c < 6; c++) v[c] = ld(P + pix(A, s, col - s * nv, c, loc, nv, Vb));
#pragma unroll
      for (int q = 0; q < 3; q++) {
        acc[cc][2 * q] = acc[cc][2 * q] + t[q].re * v[2 * q];
        acc[cc][2 * q + 1] = acc[cc][2 * q + 1] + t[q].im * v[2 * q + 1];
      }
#pragma unroll
      for (int i = 0; i < 5; i++)
#pragma unroll
        for (int j = 1; j < 6; j++)
          if (j > i) {
            const int slot = 3 + i * 5 - i * (i - 1) / 2 + (j - i - 1);
            cmac(acc[cc][i], t[slot], v[j]);
            cmac_conj(acc[cc][j], t[slot], v[i]);
          }
    }
  }
}

// one 16 x 8 tile of the projections of a chunk of X sites; real and imaginary sums and what they leave out
struct GmAcc {
  float r[4], i[4], re[4], ie[4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 4; k++) r[k] = i[k] = re[k] = ie[k] = 0.f;
  }
  __device__ __forceinline__ float2 get(int k) const { return make_float2(__fadd_rn(r[k], re[k]), __fadd_rn(i[k], ie[k])); }
};
template <int X>
__device__ __forceinline__ void galerkin_tile(GmAcc& acc, const __half2* __restrict__ Ps, const float2* __restrict__ Bs,
                                              const int* sites, int tile, int ntile, int nv, int rs, int Vb, int lane) {
  constexpr int BS = 6 * X + 4;
  const int n = 2 * nv, mt = tile / ntile, nt = tile - mt * ntile, t = lane & 3, gr = lane >> 2;
  const int i0 = mt * 16 + gr < nv ? mt * 16 + gr : nv - 1, i1 = mt * 16 + gr + 8 < nv ? mt * 16 + gr + 8 : nv - 1;
  const int col = nt * 8 + gr < n ? nt * 8 + gr : n - 1;  // rows and columns beyond the edge are not stored
  const __half2 *pa = Ps + (size_t)i0 * rs, *pb = Ps + (size_t)i1 * rs;
  const float2* pc = Bs + (size_t)col * BS;
#pragma unroll 1
  for (int c = 0; c < 6; c++)
#pragma unroll
    for (int x0 = 0; x0 < X; x0 += 4) {
      const int st = c * Vb + sites[x0 + t];
      const float2 a = __half22float2(pa[st]), b = __half22float2(pb[st]), y = pc[c * X + x0 + t];
      const uint32_t ar = __float_as_uint(a.x), ai = __float_as_uint(a.y), br = __float_as_uint(b.x), bi = __float_as_uint(b.y);
      const uint32_t re[4] = {ar, br, ai, bi}, im[4] = {__float_as_uint(-a.y), __float_as_uint(-b.y), ar, br};
      const uint32_t hr = to_tf32(y.x), hi = to_tf32(y.y);
      const uint32_t lr = to_tf32(y.x - __uint_as_float(hr)), li = to_tf32(y.y - __uint_as_float(hi));
      mma_sum(acc.r, acc.re, re, hr, hi, lr, li);
      mma_sum(acc.i, acc.ie, im, hr, hi, lr, li);
    }
}

template <int X>
__global__ void __launch_bounds__(GM_THREADS, 1) k_galerkin_mma(float2* __restrict__ Dc, const float2* __restrict__ P,
                                                                Links<PREC_F32> U, Clover<PREC_F32> C, Geo g, FaceTables f,
                                                                int nv, int rs) {
  constexpr int BS = 6 * X + 4;    // entries per column of y
  constexpr int CG = GM_THREADS / X;  // column groups
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int sites[X];
  const int Vb = g.Vb, A = blockIdx.x >> 1, s = blockIdx.x & 1, n = 2 * nv;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __half2* Ps = reinterpret_cast<__half2*>(smem_raw);                       // [nv][rs], entry comp * Vb + site
  float2* Bs = reinterpret_cast<float2*>(smem_raw + (size_t)nv * rs * 4);   // [n][BS], entry comp * X + x
  for (int e = threadIdx.x; e < nv * 6 * Vb; e += GM_THREADS) {
    const int i = e / (6 * Vb), q = e - i * 6 * Vb;
    Ps[(size_t)i * rs + q] = __float22half2_rn(__ldg(P + pix(A, s, i, 0, 0, nv, Vb) + q));
  }
  const int x = threadIdx.x % X, cg = threadIdx.x / X;
  const int ntile = (n + 7) / 8, tiles = (nv + 15) / 16 * ntile;  // 16 x 8 tiles, at most two per warp
  for (int d = 0; d < 9; d++) {
    const int nsite = d ? f.off[d] - f.off[d - 1] : Vb;
    GmAcc acc0, acc1;
    acc0.clear();
    acc1.clear();
    for (int c0 = 0; c0 < nsite; c0 += X) {
      // ---- y of X sites, all columns
      const bool in = c0 + x < nsite;
      const int loc = !in ? 0 : d ? f.list[f.off[d - 1] + c0 + x] : c0 + x;
      __syncthreads();  // the previous chunk's reads of Bs and sites (and at first the rows) are done
      if (threadIdx.x < X) sites[x] = loc;
      for (int col0 = cg; col0 < n; col0 += GM_CPT * CG) {
        cplx<float> acc[GM_CPT][6];
#pragma unroll
        for (int cc = 0; cc < GM_CPT; cc++)
#pragma unroll
          for (int c = 0; c < 6; c++) acc[cc][c] = cplx<float>(0.f, 0.f);
        if (in) {
#pragma unroll 1
          for (int k = d ? d - 1 : 0; k < (d ? d : 8); k++) {
            const Nbr nb = neighbour(g, A, loc, k);
            if (nb.cross != (d > 0)) continue;
            const float sg = nb.flip ? 0.5f : -0.5f;
#define GM_HOP(K)                                                                                                      \
  case K: galerkin_hop<(K) / 2, ((K) & 1) == 0>(acc, P, U, sg, s, A, loc, nb.blk, nb.loc, nv, Vb, n, col0, CG); break;
            switch (k) {
              GM_HOP(0) GM_HOP(1) GM_HOP(2) GM_HOP(3) GM_HOP(4) GM_HOP(5) GM_HOP(6)
              default: galerkin_hop<3, false>(acc, P, U, sg, s, A, loc, nb.blk, nb.loc, nv, Vb, n, col0, CG);
            }
#undef GM_HOP
          }
          if (d == 0) galerkin_site(acc, P, C.d + ((size_t)A * 36 + 18 * s) * Vb + loc, s, A, loc, nv, Vb, n, col0, CG);
        }
#pragma unroll
        for (int cc = 0; cc < GM_CPT; cc++) {
          const int col = col0 + cc * CG;
          if (col < n)
#pragma unroll
            for (int c = 0; c < 6; c++) Bs[(size_t)col * BS + c * X + x] = make_float2(acc[cc][c].re, acc[cc][c].im);
        }
      }
      __syncthreads();
      // ---- projections: 4 sites of one component per instruction
      if (warp < tiles) galerkin_tile<X>(acc0, Ps, Bs, sites, warp, ntile, nv, rs, Vb, lane);
      if (warp + GM_THREADS / 32 < tiles)
        galerkin_tile<X>(acc1, Ps, Bs, sites, warp + GM_THREADS / 32, ntile, nv, rs, Vb, lane);
    }
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const int tile = warp + q * (GM_THREADS / 32), mt = tile / ntile, nt = tile - mt * ntile;
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int row = mt * 16 + (lane >> 2) + (k >> 1) * 8, col = nt * 8 + 2 * (lane & 3) + (k & 1);
        if (tile < tiles && row < nv && col < n)
          Dc[(((size_t)A * 9 + d) * n + col) * n + s * nv + row] = q ? acc1.get(k) : acc0.get(k);
      }
    }
  }
}

// words per row of P in shared memory: rows 4 banks apart
static int galerkin_mma_rs(const FineGeom& g) { return (6 * g.Vb + 31) / 32 * 32 + 4; }
static size_t galerkin_mma_smem(const FineGeom& g, int nv, int X) {
  return (size_t)nv * galerkin_mma_rs(g) * 4 + (size_t)2 * nv * (6 * X + 4) * sizeof(float2);
}
template <int X>
static bool try_galerkin_mma(const FineGeom& g, float2* Dc, const float2* P, Links<PREC_F32> U, Clover<PREC_F32> C, Geo q,
                             FaceTables f, int nv, cudaStream_t st) {
  const size_t smem = galerkin_mma_smem(g, nv, X);
  if (smem > 226 * 1024 || (nv + 15) / 16 * ((2 * nv + 7) / 8) > 2 * (GM_THREADS / 32)) return false;
  set_dynamic_smem((const void*)k_galerkin_mma<X>, smem);
  k_galerkin_mma<X><<<g.Nb * 2, GM_THREADS, smem, st>>>(Dc, P, U, C, q, f, nv, galerkin_mma_rs(g));
  return true;
}

void launch_galerkin(const FineGeom& g, const FaceDev& faces, int dprec, void* Dc, const float2* P, const void* links32,
                     const void* clover32, int nv, bool rows_fp16, cudaStream_t st) {
  ScopedTimer timer_("galerkin", st);
  Geo q{g.Vb, g.Nb, g.loc_nbr.as<uint32_t>(), g.blk_nbr.as<int>()};
  FaceTables f;
  f.idx = faces.idx.as<int>();
  f.list = faces.list.as<int>();
  for (int k = 0; k < 9; k++) f.off[k] = faces.off[k];
  size_t smem = (size_t)12 * (g.Vb + faces.off[8]) * sizeof(cplx<float>);
  int threads = g.Vb >= 256 ? 256 : ((g.Vb + 31) / 32) * 32;
  Links<PREC_F32> U{(const float2*)links32, g.Vb};
  Clover<PREC_F32> C{(const float2*)clover32, g.Vb};
  if (dprec != PREC_F32) throw Error(DDTM_ERR_ARG, "internal: Galerkin output is FP32");
  // FP16 rows of P where FP16 coarse storage is asked for and they take no more than 220 KB beside one column and its face
  // hops in FP32 (4^4 aggregates: up to 30 vectors).  Beyond that the rows stay FP32 (k_galerkin), although the
  // matrix instructions would hold two vectors more: FP16 rows cost D_c 2e-4.  Widest chunk of sites that fits.
  const size_t rows = (size_t)nv * 6 * g.Vb * sizeof(__half2) + (size_t)6 * (g.Vb + faces.off[8]) * sizeof(cplx<float>);
  const bool mma = rows_fp16 && rows <= 220 * 1024 &&
                   (try_galerkin_mma<32>(g, (float2*)Dc, P, U, C, q, f, nv, st) ||
                    try_galerkin_mma<16>(g, (float2*)Dc, P, U, C, q, f, nv, st) ||
                    try_galerkin_mma<8>(g, (float2*)Dc, P, U, C, q, f, nv, st));
  if (!mma) {
    set_dynamic_smem((const void*)k_galerkin<float2>, smem);
    k_galerkin<float2><<<g.Nb, threads, smem, st>>>((float2*)Dc, P, U, C, q, f, nv);
  }
  CKL("galerkin");
}

void build_faces(const FineGeom& g, FaceDev& faces) {
  std::vector<int> idx(8 * g.Vb, -1), list;
  for (int k = 0; k < 8; k++) {
    faces.off[k] = (int)list.size();
    for (int loc = 0; loc < g.Vb; loc++)
      if ((g.h_loc_nbr[k * g.Vb + loc] >> 16) & 1) {
        idx[k * g.Vb + loc] = (int)list.size() - faces.off[k];
        list.push_back(loc);
      }
  }
  faces.off[8] = (int)list.size();
  faces.idx.ensure(idx.size() * 4);
  faces.list.ensure(list.size() * 4 + 4);
  CK(cudaMemcpy(faces.idx.p, idx.data(), idx.size() * 4, cudaMemcpyHostToDevice));
  CK(cudaMemcpy(faces.list.p, list.data(), list.size() * 4, cudaMemcpyHostToDevice));
}

// ---- coarse stencil ---------------------------------------------------------------
// Coarse vectors of a batch of R right-hand sides are stored interleaved,
// v[(idx * n + k) * R + r], so the R values of one dof are contiguous.  A
// thread owns one row r of one site and RC consecutive right-hand sides
// (register blocking: each matrix entry read from HBM is used RC times by the
// thread and R / RC times by the site's threads); threads of a site are
// ordered row fastest, so a warp reads consecutive entries of a column-major
// block.  Output slot idx has lattice site osite[idx] (idx itself when
// osite == nullptr); the self term reads x_self[idx], hop d reads
// x_hop[tab[(d-1) * nout + idx]] (tab: full neighbour table for full-lattice
// vectors, or the parity-compact table into the other parity's vector).
//   mode & 1: self block + twist i mu_c Gamma5_c;  mode & 2: the 8 hops
//   y[idx] = sy * y[idx] + sres * result   (sy = 0 overwrites y)
template <int RC>
__device__ __forceinline__ void load_rc(const cplx<float>* p, cplx<float> v[RC]) {
  if (RC == 4) {
    const float4* q = reinterpret_cast<const float4*>(p);
    float4 a = q[0], b = q[1];
    v[0] = cplx<float>(a.x, a.y); v[1] = cplx<float>(a.z, a.w);
    v[2] = cplx<float>(b.x, b.y); v[3] = cplx<float>(b.z, b.w);
  } else if (RC == 2) {
    float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = cplx<float>(a.x, a.y); v[1] = cplx<float>(a.z, a.w);
  } else {
#pragma unroll
    for (int c = 0; c < RC; c++) v[c] = p[c];
  }
}

// Two consecutive rows (r, r+1) of column k of a column-major block: one
// 16-byte load.
template <typename DS> __device__ __forceinline__ void ld_rows2(const DS* p, cplx<float>& a0, cplx<float>& a1);
template <> __device__ __forceinline__ void ld_rows2<float2>(const float2* p, cplx<float>& a0, cplx<float>& a1) {
  float4 v = __ldg(reinterpret_cast<const float4*>(p));
  a0 = cplx<float>(v.x, v.y);
  a1 = cplx<float>(v.z, v.w);
}

// acc{0,1}[c] += A[r0 + {0,1}][k] v[k][c] for a column-major n x n block whose
// row r0 is at A; the column loop is unrolled so that many independent
// matrix loads are in flight per thread.
template <typename DS, int RC>
__device__ __forceinline__ void block_mv2(const DS* A, const cplx<float>* v, int n, int R, cplx<float> acc0[RC],
                                          cplx<float> acc1[RC]) {
#pragma unroll 8
  for (int k = 0; k < n; k++) {
    cplx<float> a0, a1;
    ld_rows2<DS>(A + (size_t)k * n, a0, a1);
    cplx<float> x[RC];
    load_rc<RC>(v + (size_t)k * R, x);
#pragma unroll
    for (int c = 0; c < RC; c++) {
      cmac(acc0[c], a0, x[c]);
      cmac(acc1[c], a1, x[c]);
    }
  }
}

// One hop of the stencil, y[site] = A_d(site) x[site + d].  Threads of a site: n/2 row pairs x G chunk slots, row pair
// fastest (a warp reads consecutive 16-byte pieces of a column); a thread takes the chunks ch = g, g + G, ... of RC
// right-hand sides (launch_shape.h); SPB sites per CTA.
template <int RC>
__global__ void __launch_bounds__(256) k_coarse_hop(cplx<float>* __restrict__ y, const cplx<float>* __restrict__ x,
                                                     const float2* __restrict__ Dc, const int* __restrict__ nbr, int nout, int n,
                                                     int R, int G, int d) {
  const int np = n / 2, nch = R / RC, per = np * G, spb = blockDim.x / per;
  const int t = threadIdx.x, rp = t % np, g = (t / np) % G, q = t / per;
  const int site = blockIdx.x * spb + q;
  if (q >= spb || site >= nout) return;
  const int r0 = 2 * rp, src = __ldg(nbr + (size_t)(d - 1) * nout + site);
  for (int ch = g; ch < nch; ch += G) {
    const int c0 = ch * RC;
    cplx<float> acc0[RC], acc1[RC];
#pragma unroll
    for (int c = 0; c < RC; c++) acc0[c] = acc1[c] = cplx<float>(0, 0);
    block_mv2<float2, RC>(Dc + ((size_t)site * 9 + d) * n * n + r0, x + (size_t)src * n * R + c0, n, R, acc0, acc1);
    cplx<float>* yo = y + ((size_t)site * n + r0) * R + c0;
#pragma unroll
    for (int c = 0; c < RC; c++) {
      yo[c] = acc0[c];
      yo[R + c] = acc1[c];
    }
  }
}

// The stencil with a CTA per site and chunk of RC right-hand sides: n/2 row pairs x S shares of the products.  Unit
// u = d H + h is part h of H (columns h n / H ...) of hop d (d = 0: the self block); share s takes units s, s + S, ...,
// and every unit's result goes to shared memory, where the units are summed in order: the result depends neither on S
// nor on the batch.  With an inverse (even sites, Dinv != null) the sum hs = sr rhs + sres (hops) is multiplied by it,
// the columns shared out in the same way.  The last chunk may have fewer columns than RC.
// One thread per row pair for all of the hops, as for single hops (k_coarse_hop), is a chain of 9 n loads of 16 bytes and leaves most SMs
// without work on coarse lattices of a few hundred sites.  Full stencil in FP32, before ->
// after, 48 dofs: 32 sites, 1 column 65 -> 10 us, 12 columns 70 -> 14; 512 sites 76 -> 24, 113 to 165 -> 86; 2592 sites
// 194 -> 129, 352 -> 350.  Bound by the matrices (430 MB at 2592 sites) with one column and by shared loads of the
// vectors' columns with many.
// COLS: 0 all RC columns are there, 1 nc <= RC of them (any R), 2 the same with an even R
template <int RC, int COLS>
__device__ __forceinline__ void load_cols(const cplx<float>* p, int nc, cplx<float> v[RC]) {
  if (COLS == 0) {
    load_rc<RC>(p, v);
  } else if (COLS == 1) {
#pragma unroll
    for (int c = 0; c < RC; c++) v[c] = c < nc ? p[c] : cplx<float>(0, 0);
  } else {
#pragma unroll
    for (int c = 0; c + 1 < RC; c += 2) {
      const float4 a = c < nc ? *reinterpret_cast<const float4*>(p + c) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[c] = cplx<float>(a.x, a.y);
      v[c + 1] = cplx<float>(a.z, a.w);
    }
  }
}
// part[row][c] = sum_k A[row][k] x[k][c] of the rows r0, r0 + 1 (x rows R apart) for kn columns
template <int RC, int COLS>
__device__ __forceinline__ void split_unit(cplx<float>* part, const float2* A, const cplx<float>* x, int n, int kn, int R, int nc) {
  cplx<float> acc0[RC], acc1[RC];
#pragma unroll
  for (int c = 0; c < RC; c++) acc0[c] = acc1[c] = cplx<float>(0, 0);
#pragma unroll 8
  for (int k = 0; k < kn; k++) {
    cplx<float> a0, a1, v[RC];
    ld_rows2<float2>(A + (size_t)k * n, a0, a1);
    load_cols<RC, COLS>(x + (size_t)k * R, nc, v);
#pragma unroll
    for (int c = 0; c < RC; c++) {
      cmac(acc0[c], a0, v[c]);
      cmac(acc1[c], a1, v[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < RC; c++) {
    part[c] = acc0[c];
    part[RC + c] = acc1[c];
  }
}
__device__ __forceinline__ cplx<float> split_sum(const cplx<float>* part, int units, int nrc, int k) {
  cplx<float> v = part[k];
  for (int u = 1; u < units; u++) v = v + part[(size_t)u * nrc + k];
  return v;
}
static const int SPLIT_KU = 8;  // shares of the inverse's columns
template <int RC, int COLS>
__global__ void __launch_bounds__(1024)
    k_coarse_split(cplx<float>* __restrict__ y, const cplx<float>* __restrict__ x_self, const cplx<float>* __restrict__ x_hop,
                   const float2* __restrict__ Dc, const int* __restrict__ tab, const int* __restrict__ osite, int nout, int n,
                   int nv, int R, int S, int H, float mu_c, int mode, float sres, float sy, const float2* __restrict__ Dinv,
                   const cplx<float>* __restrict__ rhs, float sr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int np = n / 2, nch = (R + RC - 1) / RC, nrc = n * RC;
  const int idx = blockIdx.x / nch, c0 = (blockIdx.x - idx * nch) * RC, nc = R - c0 < RC ? R - c0 : RC;
  const int t = threadIdx.x, rp = t % np, s = t / np, r0 = 2 * rp;
  const int site = osite ? osite[idx] : idx;
  const int d0 = mode & 1 ? 0 : 1, d1 = mode & 2 ? 9 : 1;  // hops d0 ... d1 - 1
  const int units = (d1 - d0) * H, kh = (n + H - 1) / H;
  cplx<float>* part = reinterpret_cast<cplx<float>*>(smem_raw);  // [9 H][n][RC]
  cplx<float>* hs = part + (size_t)9 * H * nrc;                  // [n][RC], with an inverse
  for (int u = s; u < units; u += S) {
    const int d = d0 + u / H, k0 = (u % H) * kh, kn = n - k0 < kh ? n - k0 : kh;
    const cplx<float>* x = d ? x_hop + (size_t)__ldg(tab + (size_t)(d - 1) * nout + idx) * n * R : x_self + (size_t)idx * n * R;
    split_unit<RC, COLS>(part + (size_t)u * nrc + (size_t)r0 * RC, Dc + (((size_t)site * 9 + d) * n + k0) * n + r0,
                        x + (size_t)k0 * R + c0, n, kn, R, nc);
  }
  __syncthreads();
  for (int k = t; k < nrc; k += blockDim.x) {
    const int row = k / RC, c = k - row * RC;
    const size_t o = ((size_t)idx * n + row) * R + c0 + c;
    cplx<float> v = units > 0 ? split_sum(part, units, nrc, k) : cplx<float>(0, 0);
    if (Dinv) {
      v = sres * v;
      if (rhs && c < nc) v = v + sr * rhs[o];
      hs[k] = v;
    } else if (c < nc) {
      if (mode & 1) v = v + (row < nv ? mu_c : -mu_c) * times_i(x_self[o]);
      v = sres * v;
      y[o] = sy == 0.f ? v : sy * y[o] + v;
    }
  }
  if (!Dinv) return;
  __syncthreads();
  const int ku = (n + SPLIT_KU - 1) / SPLIT_KU;
  for (int u = s; u < SPLIT_KU; u += S) {
    const int k0 = u * ku < n ? u * ku : n, kn = n - k0 < ku ? n - k0 : ku;
    split_unit<RC, 0>(part + (size_t)u * nrc + (size_t)r0 * RC, Dinv + ((size_t)idx * n + k0) * n + r0,
                                hs + (size_t)k0 * RC, n, kn, RC, RC);
  }
  __syncthreads();
  for (int k = t; k < nrc; k += blockDim.x) {
    const int row = k / RC, c = k - row * RC;
    if (c < nc) y[((size_t)idx * n + row) * R + c0 + c] = split_sum(part, SPLIT_KU, nrc, k);
  }
}

// gather (dir = 0: compact[i] = full[list[i]]) or scatter (dir = 1), n*R
// contiguous complex numbers per site
__global__ void k_parity_copy(cplx<float>* __restrict__ compact, cplx<float>* __restrict__ full, const int* __restrict__ list,
                              int cnt, int nr, int dir) {
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)cnt * nr) return;
  int i = (int)(t / nr), r = (int)(t - (size_t)i * nr);
  size_t f = (size_t)list[i] * nr + r;
  if (dir == 0) compact[t] = full[f];
  else full[f] = compact[t];
}

// Canonical FP64 coarse vectors c[r][nc] <-> columns r0 ... r0 + nr - 1 of the interleaved FP32 batch v[nc][R] (dir 0: c ->
// v, dir 1: v -> c): tiles of IL_T entries x IL_R columns turned through shared memory, so that both sides are contiguous.
static const int IL_T = 64, IL_R = 32;
template <bool A16>
__global__ void __launch_bounds__(256) k_coarse_interleave(float2* __restrict__ v, double* __restrict__ c, size_t nc, int r0,
                                                           int nr, int R, int dir) {
  __shared__ float2 t[IL_T * (IL_R + 1)];
  const size_t e0 = (size_t)blockIdx.x * IL_T;
  const int q0 = blockIdx.y * IL_R, nq = nr - q0 < IL_R ? nr - q0 : IL_R;
  const int ne = nc - e0 < (size_t)IL_T ? (int)(nc - e0) : IL_T;
  c += 2 * ((size_t)q0 * nc + e0);
  v += e0 * R + r0 + q0;
  if (dir == 0) {
    for (int k = threadIdx.x; k < IL_T * nq; k += blockDim.x) {
      const int q = k / IL_T, e = k - q * IL_T;
      if (e < ne) {
        const double2 a = ld_canon<A16>(c, (size_t)q * nc + e);
        t[e * (IL_R + 1) + q] = make_float2((float)a.x, (float)a.y);
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < ne * nq; k += blockDim.x) {
      const int e = k / nq, q = k - e * nq;
      v[(size_t)e * R + q] = t[e * (IL_R + 1) + q];
    }
  } else {
    for (int k = threadIdx.x; k < ne * nq; k += blockDim.x) {
      const int e = k / nq, q = k - e * nq;
      t[e * (IL_R + 1) + q] = v[(size_t)e * R + q];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < IL_T * nq; k += blockDim.x) {
      const int q = k / IL_T, e = k - q * IL_T;
      if (e < ne) {
        const float2 z = t[e * (IL_R + 1) + q];
        st_canon<A16>(c, (size_t)q * nc + e, (double)z.x, (double)z.y);
      }
    }
  }
}

// Inverse of (self block + i mu_c Gamma5_c) per even site by Gauss-Jordan
// elimination with partial pivoting in CT (FP64, or FP32 where the inverses
// only feed FP16 operator images); one CTA per site, thread = row.
template <typename DS, typename CT>
__global__ void k_self_inverse(float2* __restrict__ Dinv, const DS* __restrict__ Dc, const int* __restrict__ even, int n,
                               int nv, double mu_c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<CT>* M = reinterpret_cast<cplx<CT>*>(smem_raw);  // [n][2n] row-major augmented
  __shared__ int piv;
  const int e = blockIdx.x, site = even[e];
  const int r = threadIdx.x;
  const int w2 = 2 * n;
  if (r < n) {
    for (int c = 0; c < n; c++) {
      cplx<float> a = ldD<DS>(Dc + ((size_t)site * 9 * n + c) * n + r);  // d = 0, column c, row r
      M[r * w2 + c] = cplx<CT>((CT)a.re, (CT)a.im);
      M[r * w2 + n + c] = cplx<CT>(r == c ? CT(1) : CT(0), CT(0));
    }
    M[r * w2 + r].im += (CT)(r < nv ? mu_c : -mu_c);
  }
  __syncthreads();
  for (int c = 0; c < n; c++) {
    if (r == 0) {
      int p = c;
      CT best = norm2(M[c * w2 + c]);
      for (int k = c + 1; k < n; k++)
        if (norm2(M[k * w2 + c]) > best) { best = norm2(M[k * w2 + c]); p = k; }
      piv = p;
    }
    __syncthreads();
    const int p = piv;
    if (p != c && r < w2) {  // swap rows c and p, column r (and r + n) per thread
      for (int cc = r; cc < w2; cc += blockDim.x) {
        cplx<CT> tmp = M[c * w2 + cc];
        M[c * w2 + cc] = M[p * w2 + cc];
        M[p * w2 + cc] = tmp;
      }
    }
    __syncthreads();
    cplx<CT> d = M[c * w2 + c];
    CT dn = norm2(d);
    cplx<CT> inv(d.re / dn, -d.im / dn);
    __syncthreads();
    for (int cc = r; cc < w2; cc += blockDim.x) M[c * w2 + cc] = M[c * w2 + cc] * inv;
    __syncthreads();
    if (r < n && r != c) {
      cplx<CT> fct = M[r * w2 + c];
      for (int cc = 0; cc < w2; cc++) M[r * w2 + cc] = M[r * w2 + cc] - fct * M[c * w2 + cc];
    }
    __syncthreads();
  }
  if (r < n)
    for (int c = 0; c < n; c++) {
      cplx<CT> v = M[r * w2 + n + c];
      Dinv[((size_t)e * n + c) * n + r] = make_float2((float)v.re, (float)v.im);  // column-major
    }
}

template <int RC, int COLS>
static void coarse_split_t(const CoarseLevel& c, cplx<float>* y, const cplx<float>* xs, const cplx<float>* xh, const int* tab,
                           const int* osite, int nout, int R, int S, int H, size_t smem, double mu_c, int mode, float sres,
                           float sy, const float2* Dinv, const cplx<float>* rhs, float sr, cudaStream_t st) {
  set_dynamic_smem((const void*)k_coarse_split<RC, COLS>, 200 * 1024);
  k_coarse_split<RC, COLS><<<(unsigned)(nout * ((R + RC - 1) / RC)), c.n / 2 * S, smem, st>>>(
      y, xs, xh, c.Dc.as<float2>(), tab, osite, nout, c.n, c.nv, R, S, H, (float)mu_c, mode, sres, sy, Dinv, rhs, sr);
  CKL("coarse_split");
}
// Units of a hop: two on lattices of up to two sites per SM, where the chain of a unit's loads is what counts, and one
// beyond (2592 sites of 48 dofs, 12 columns: 350 us with one, 388 with two).  Four columns per CTA, fewer where R is 1 or
// 2 (with 12 columns a matrix entry is loaded once for 12 right-hand sides, but the registers leave too few warps: 421).
static void coarse_split(const CoarseLevel& c, cplx<float>* y, const cplx<float>* xs, const cplx<float>* xh, const int* tab,
                         const int* osite, int nout, int R, double mu_c, int mode, float sres, float sy, const float2* Dinv,
                         const cplx<float>* rhs, float sr, cudaStream_t st) {
  if (nout == 0) return;
  const int np = c.n / 2, H = 18 * np <= 1024 && nout <= 304 ? 2 : 1, S = std::max(1, std::min(9 * H, 1024 / np));
  const int rc = R < 3 ? R : 4;
  auto go = R == 1       ? coarse_split_t<1, 0>
            : R == 2     ? coarse_split_t<2, 0>
            : R % 4 == 0 ? coarse_split_t<4, 0>
            : R % 2 == 0 ? coarse_split_t<4, 2>
                         : coarse_split_t<4, 1>;
  const size_t smem = (size_t)(9 * H + 1) * c.n * rc * sizeof(cplx<float>);  // n <= 128: at most 74 KB
  go(c, y, xs, xh, tab, osite, nout, R, S, H, smem, mu_c, mode, sres, sy, Dinv, rhs, sr, st);
}

void launch_coarse_apply_hop(const CoarseLevel& c, cplx<float>* y, const cplx<float>* x, int R, int hop, cudaStream_t st) {
  ScopedTimer timer_("coarse_apply", st, R);
  const CoarseShape sh = coarse_shape(c.n, R);
  const unsigned grid = (unsigned)((c.Nc + sh.spb - 1) / sh.spb);
  auto kernel = sh.rc == 4 ? k_coarse_hop<4> : sh.rc == 2 ? k_coarse_hop<2> : k_coarse_hop<1>;
  kernel<<<grid, sh.threads, 0, st>>>(y, x, c.Dc.as<float2>(), c.nbr.as<int>(), c.Nc, c.n, R, sh.groups, hop + 1);
  CKL("coarse_hop");
}

void launch_coarse_apply_full(const CoarseLevel& c, cplx<float>* y, const cplx<float>* x, int R, double mu_c, int mode,
                              float sres, float sy, cudaStream_t st) {
  ScopedTimer timer_("coarse_apply", st, R);
  coarse_split(c, y, x, x, c.nbr.as<int>(), nullptr, c.Nc, R, mu_c, mode, sres, sy, nullptr, nullptr, 0.f, st);
}

void launch_coarse_apply_odd(const CoarseLevel& c, cplx<float>* y_o, const cplx<float>* x_o, const cplx<float>* x_e, int R,
                             double mu_c, int mode, float sres, float sy, cudaStream_t st) {
  ScopedTimer timer_("coarse_apply_odd_f32", st, R);
  coarse_split(c, y_o, x_o, x_e, c.nbr_oe.as<int>(), c.odd.as<int>(), (int)c.h_odd.size(), R, mu_c, mode, sres, sy, nullptr,
               nullptr, 0.f, st);
}

void launch_coarse_even(const CoarseLevel& c, cplx<float>* t, const cplx<float>* rhs, const cplx<float>* v, int R, float sr,
                        float sh, cudaStream_t st) {
  ScopedTimer timer_("coarse_even_f32", st, R);
  // Batches beyond this size are refused, as ever: they never fitted the shared-memory stage of the callers' even-site
  // kernel.  (k_coarse_split itself stages four columns at a time and would take them.)
  if ((size_t)coarse_shape(c.n, R).spb * c.n * R * sizeof(cplx<float>) > 200 * 1024)
    throw Error(DDTM_ERR_ARG, "coarse_even: " + std::to_string(R) + " right-hand sides of " + std::to_string(c.n) +
                                  " dofs exceed the shared-memory stage");
  coarse_split(c, t, nullptr, v, c.nbr_eo.as<int>(), c.even.as<int>(), (int)c.h_even.size(), R, 0.f, v ? 2 : 0, sh, 0.f,
               c.Dinv.as<float2>(), rhs, sr, st);
}

void launch_parity_copy(const CoarseLevel& c, int parity, cplx<float>* compact, cplx<float>* full, int R, int dir,
                        cudaStream_t st) {
  ScopedTimer timer_("parity_copy", st);
  int cnt = parity == 0 ? (int)c.h_even.size() : (int)c.h_odd.size();
  const int* list = parity == 0 ? c.even.as<int>() : c.odd.as<int>();
  size_t tot = (size_t)cnt * c.n * R;
  k_parity_copy<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(compact, full, list, cnt, c.n * R, dir);
  CKL("parity_copy");
}

void launch_coarse_interleave(const CoarseLevel& c, cplx<float>* v, double* canon, int r, int R, int dir,
                              cudaStream_t st, int nr) {
  ScopedTimer timer_("coarse_interleave", st, nr);
  const size_t nc = (size_t)c.Nc * c.n;
  for (int q = 0; q < nr; q += 65535 * IL_R) {  // grid.y
    const int n = nr - q < 65535 * IL_R ? nr - q : 65535 * IL_R;
    auto kernel = canon_a16(canon) ? k_coarse_interleave<true> : k_coarse_interleave<false>;
    kernel<<<dim3((unsigned)((nc + IL_T - 1) / IL_T), (n + IL_R - 1) / IL_R), 256, 0, st>>>(
        reinterpret_cast<float2*>(v), canon + 2 * (size_t)q * nc, nc, r + q, n, R, dir);
    CKL("coarse_interleave");
  }
}

void launch_self_inverse(CoarseLevel& c, double mu_c, cudaStream_t st) {
  ScopedTimer timer_("self_inverse", st);
  int ne = (int)c.h_even.size();
  c.Dinv.ensure((size_t)ne * c.n * c.n * sizeof(float2));
  size_t smem = (size_t)c.n * 2 * c.n * sizeof(cplx<double>);
  int threads = ((c.n + 31) / 32) * 32;
  if (c.prec == PREC_F16) {
    // the inverses feed FP16 operator images: Gauss-Jordan in FP32 (FP64 is slow on this GPU)
    const size_t smem32 = (size_t)c.n * 2 * c.n * sizeof(cplx<float>);
    set_dynamic_smem((const void*)k_self_inverse<float2, float>, smem32);
    k_self_inverse<float2, float><<<ne, threads, smem32, st>>>(c.Dinv.as<float2>(), c.Dc.as<float2>(), c.even.as<int>(),
                                                               c.n, c.nv, mu_c);
  } else {
    set_dynamic_smem((const void*)k_self_inverse<float2, double>, smem);
    k_self_inverse<float2, double><<<ne, threads, smem, st>>>(c.Dinv.as<float2>(), c.Dc.as<float2>(), c.even.as<int>(),
                                                                c.n, c.nv, mu_c);
  }
  CKL("self_inverse");
  if (c.prec == PREC_F16) build_inverse_images(c, st);
  c.inv_mu = mu_c;
  c.inv_valid = true;
}

}  // namespace ddtm
