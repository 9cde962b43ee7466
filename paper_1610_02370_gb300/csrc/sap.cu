// Red-black multiplicative SAP smoother (Sec. 2.4) with even-odd reduced
// block solves by minimal residual (Sec. 2.4, 2.5).
//
// One launch is one half-sweep over the blocks of one colour; one CTA owns one
// block and RG right-hand sides of it (one group of threads per right-hand
// side, synchronised by its own named barrier), so the groups read the same
// links, clover entries and inverses at about the same time and all but the
// first are served by L1.  Blocks of one colour never touch, so CTAs are
// independent: each reads x on its own block and on the neighbouring blocks of
// the other colour and writes x only on its own block.  Per block B:
//   r     = b - D(mu) x                 on B (full stencil, neighbours in HBM)
//   rhat  = r_o - A_oe A_ee^-1 r_e      (A = D_BB + i mu Gamma5, hops leaving B dropped)
//   e_o   = nmr MR steps on A_hat e_o = rhat from 0,
//           A_hat = A_oo - A_oe A_ee^-1 A_eo,  alpha = <p, rho> / <p, p>
//   e_e   = A_ee^-1 (r_e - A_eo e_o)
//   x_B  += e
// A_ee^-1 is the precomputed inverse of the site term + i mu gamma5 on even
// sites.  Vectors of the block solve live in shared memory as [12][Vh]; inner
// products are reduced per CTA in a fixed order (deterministic).
#include "common.cuh"
#include "ddtm_internal.h"
#include "timer.h"
#include "stencil.cuh"
#include "stencil_lanes.cuh"

namespace ddtm {

template <typename R>
struct SapArgs {
  const int* blocks;       // blocks of this colour
  int nrhs;                // right-hand sides of the batch
  const int* zero_blocks;  // first sweep from x = 0: blocks of the other colour to clear
  int zero_x;              // x is implicitly zero on entry
  int nmr;
  R mu;
  size_t fstride;          // store2 elements between right-hand sides (12 V)
  long V;                  // sites (stride of the FP16 scales between right-hand sides)
};

// shared memory of one right-hand-side group: four block vectors of 12 x Vh
// complex and the reduction slots, rounded to 16 bytes
template <typename R>
__host__ __device__ constexpr size_t sap_group_smem(int Vh) {
  return (4 * 12 * (size_t)Vh * 2 * sizeof(R) + 3 * 32 * sizeof(R) + 15) / 16 * 16;
}

// barrier of one right-hand-side group (gt threads, a multiple of 32): named
// barrier 1 + grp, or the whole CTA when it holds one group
template <int RG>
__device__ __forceinline__ void group_sync(int grp, int gt) {
  if (RG == 1) {
    __syncthreads();
    return;
  }
  switch (grp) {  // literal barrier ids, so the kernel reserves RG + 1 barriers, not all 16
    case 0: asm volatile("bar.sync 1, %0;" ::"r"(gt) : "memory"); break;
    case 1: asm volatile("bar.sync 2, %0;" ::"r"(gt) : "memory"); break;
    case 2: asm volatile("bar.sync 3, %0;" ::"r"(gt) : "memory"); break;
    default: asm volatile("bar.sync 4, %0;" ::"r"(gt) : "memory"); break;
  }
}

// sum over the thread group (gt threads from thread grp * gt) of three reals;
// every thread of the group receives the totals
template <int RG, typename R>
__device__ __forceinline__ void group_sum3(R& a, R& b, R& c, R* red, int grp, int gt) {
  a = warp_sum(a);
  b = warp_sum(b);
  c = warp_sum(c);
  const int w = (threadIdx.x - grp * gt) >> 5, nw = gt >> 5;
  group_sync<RG>(grp, gt);
  if ((threadIdx.x & 31) == 0) {
    red[3 * w] = a;
    red[3 * w + 1] = b;
    red[3 * w + 2] = c;
  }
  group_sync<RG>(grp, gt);
  a = b = c = 0;
  for (int i = 0; i < nw; i++) {
    a += red[3 * i];
    b += red[3 * i + 1];
    c += red[3 * i + 2];
  }
}

template <int P, int RG>
__global__ void __launch_bounds__(128 * RG, P == PREC_F64 ? 2 : 4 / RG)
    k_sap_half(Spinor<P> x, Spinor<P> b, Links<P> U, Clover<P> C, SiteInv<P> Ainv, Geo g,
               SapArgs<typename Prec<P>::real> a) {
  typedef typename Prec<P>::real R;
  typedef cplx<R> Z;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Vh = g.Vb / 2;
  const int gt = blockDim.x / RG, grp = threadIdx.x / gt;  // group size and this thread's group
  // grid: x = group of RG right-hand sides, y = block of this colour
  const int rhs = blockIdx.x * RG + grp;
  if (rhs >= a.nrhs) return;  // a ragged last group: its barrier has no other members
  Z* rho = reinterpret_cast<Z*>(smem_raw + (size_t)grp * sap_group_smem<R>(Vh));  // odd sites: residual of the reduced system
  Z* te = rho + 12 * Vh;                    // even sites: intermediate
  Z* re = te + 12 * Vh;                     // even sites: block residual r_e
  Z* eo = re + 12 * Vh;                     // odd sites: correction e_o
  R* red = reinterpret_cast<R*>(eo + 12 * Vh);

  x.d += (size_t)rhs * a.fstride;
  b.d += (size_t)rhs * a.fstride;
  if (x.nrm) x.nrm += (size_t)rhs * a.V;
  if (b.nrm) b.nrm += (size_t)rhs * a.V;
  const int blk = a.blocks[blockIdx.y];
  const int i = threadIdx.x - grp * gt;
  const bool act = i < Vh;
  const int le = i, lo = Vh + i;  // this thread's even and odd site

  if (a.zero_x && act) {  // clear one block of the other colour (x = 0 start)
    Z zero[12];
#pragma unroll
    for (int c = 0; c < 12; c++) zero[c] = Z(0, 0);
    int zb = a.zero_blocks[blockIdx.y];
    x.store(zb, le, zero);
    x.store(zb, lo, zero);
  }

  // 1. block residual r = b - D x on both parities
  if (act) {
    Z bb[12], dx[12];
    b.load(blk, le, bb);
    if (!a.zero_x) {
      dslash_site<P, 1>(x, U, C, g, a.mu, blk, le, dx);
#pragma unroll
      for (int c = 0; c < 12; c++) bb[c] = bb[c] - dx[c];
    }
#pragma unroll
    for (int c = 0; c < 12; c++) re[c * Vh + i] = bb[c];
    Z t[12];
    Ainv.apply(blk, le, bb, t);
#pragma unroll
    for (int c = 0; c < 12; c++) te[c * Vh + i] = t[c];
    b.load(blk, lo, bb);
    if (!a.zero_x) {
      dslash_site<P, 1>(x, U, C, g, a.mu, blk, lo, dx);
#pragma unroll
      for (int c = 0; c < 12; c++) bb[c] = bb[c] - dx[c];
    }
#pragma unroll
    for (int c = 0; c < 12; c++) {
      rho[c * Vh + i] = bb[c];
      eo[c * Vh + i] = Z(0, 0);
    }
  }
  group_sync<RG>(grp, gt);
  // 2. rhat = r_o - H_oe A_ee^-1 r_e
  if (act) {
    Z h[12];
    hop_block<P, R>(te, Vh, U, g, blk, lo, h);
#pragma unroll
    for (int c = 0; c < 12; c++) rho[c * Vh + i] = rho[c * Vh + i] - h[c];
  }
  group_sync<RG>(grp, gt);
  // 3. MR on the reduced block system
  for (int k = 0; k < a.nmr; k++) {
    if (act) {  // te = A_ee^-1 H_eo rho
      Z h[12], t[12];
      hop_block<P, R>(rho, Vh, U, g, blk, le, h);
      Ainv.apply(blk, le, h, t);
#pragma unroll
      for (int c = 0; c < 12; c++) te[c * Vh + i] = t[c];
    }
    group_sync<RG>(grp, gt);
    Z p[12];
    R pr_re = 0, pr_im = 0, pp = 0;
    if (act) {  // p = A_oo rho - H_oe te
      Z r[12], h[12];
#pragma unroll
      for (int c = 0; c < 12; c++) r[c] = rho[c * Vh + i];
      C.apply(blk, lo, r, p);
#pragma unroll
      for (int c = 0; c < 12; c++) {
        R m = c < 6 ? a.mu : -a.mu;
        p[c] = p[c] + m * times_i(r[c]);
      }
      hop_block<P, R>(te, Vh, U, g, blk, lo, h);
#pragma unroll
      for (int c = 0; c < 12; c++) {
        p[c] = p[c] - h[c];
        pr_re += p[c].re * r[c].re + p[c].im * r[c].im;  // <p, rho> = sum conj(p) rho
        pr_im += p[c].re * r[c].im - p[c].im * r[c].re;
        pp += norm2(p[c]);
      }
    }
    group_sum3<RG, R>(pr_re, pr_im, pp, red, grp, gt);
    Z alpha = pp > 0 ? Z(pr_re / pp, pr_im / pp) : Z(0, 0);
    if (act) {
#pragma unroll
      for (int c = 0; c < 12; c++) {
        Z r = rho[c * Vh + i];
        eo[c * Vh + i] = eo[c * Vh + i] + alpha * r;
        rho[c * Vh + i] = r - alpha * p[c];
      }
    }
    group_sync<RG>(grp, gt);
  }
  // 4. e_e = A_ee^-1 (r_e - H_eo e_o); 5. x_B += e
  if (act) {
    Z h[12], t[12], xv[12];
    hop_block<P, R>(eo, Vh, U, g, blk, le, h);
#pragma unroll
    for (int c = 0; c < 12; c++) h[c] = re[c * Vh + i] - h[c];
    Ainv.apply(blk, le, h, t);
    if (a.zero_x) {
      x.store(blk, le, t);
#pragma unroll
      for (int c = 0; c < 12; c++) xv[c] = eo[c * Vh + i];
      x.store(blk, lo, xv);
    } else {
      x.loadw(blk, le, xv);
#pragma unroll
      for (int c = 0; c < 12; c++) xv[c] = xv[c] + t[c];
      x.store(blk, le, xv);
      x.loadw(blk, lo, xv);
#pragma unroll
      for (int c = 0; c < 12; c++) xv[c] = xv[c] + eo[c * Vh + i];
      x.store(blk, lo, xv);
    }
  }
}

// ---- 4^4 blocks, FP32 arithmetic ---------------------------------------------------
// The same half-sweep, one CTA per block and right-hand side (V = float, k_sap_half_b4_one) or pair of
// right-hand sides (V = float2, k_sap_half_b4).  The correction of the even sites is accumulated as
//   e_e = A_ee^-1 r_e - sum_k alpha_k A_ee^-1 A_eo rho_k,
// whose terms the MR steps form anyway, so the closing hop and inverse of step 4 above are not needed.
// Shared memory: bufE, bufO (the vectors the hops read) and accE, accO, 12 x 128 complex each.
// Both kernels form every sum in the same order (forward hops, backward hops, their sum; inner products per
// chirality and warp, then over the eight of them), so a right-hand side gets the same bits from either.
//
// What bounds them (24^3 x 48, 12 right-hand sides, FP16 fields, one cycle of 3 MR steps: 2.77 ms, before
// 5.85 ms with k_sap_half; one right-hand side 0.34 ms, before 0.63 ms): the shared-memory data path (about
// 0.8 ms per half-sweep of spinor and operator reads) and, with 8 warps per SM for the pair, the latency of the
// operator reads from L2.  Packing two right-hand sides cut the instructions from 2.17 G to 0.71 G per half-sweep.
// Measured and not taken for the pair: accE and accO in local memory for more warps per SM (3.07 ms with 2 CTAs, 3.01
// with 3, 3.66 with 4 per SM), two pairs per CTA (2.96 ms: their phases coincide), two threads per site as below
// (2.97 ms: 128 registers spill), the faces of the residual staged in shared memory first (2.68 ms, no gain).
template <typename V>
__host__ __device__ constexpr size_t sap_b4_smem() {
  return 4 * 12 * B4_VH * sizeof(cv<V>) + 2 * 8 * 3 * sizeof(V);
}

// partial sums of <p, rho> = sum conj(p) rho (s0 + i s1) and <p, p> (s2) over one chirality
template <typename V>
__device__ __forceinline__ void sap_dots(const cv<V> p[6], const cv<V> r[6], V& s0, V& s1, V& s2) {
  s0 = s1 = s2 = vset<V>(0.f);
#pragma unroll
  for (int c = 0; c < 6; c++) {
    s0 = vfma(p[c].re, r[c].re, vfma(p[c].im, r[c].im, s0));
    s1 = vsub(vfma(p[c].re, r[c].im, s1), vmul(p[c].im, r[c].re));
    s2 = vfma(p[c].re, p[c].re, vfma(p[c].im, p[c].im, s2));
  }
#pragma unroll
  for (int l = 0; l < vlanes<V>(); l++) {
    const float t0 = warp_sum(vlane(s0, l)), t1 = warp_sum(vlane(s1, l)), t2 = warp_sum(vlane(s2, l));
    vput(s0, l, t0);
    vput(s1, l, t1);
    vput(s2, l, t2);
  }
}
// alpha = <p, rho> / <p, p> from the eight partial sums
template <typename V> __device__ __forceinline__ void sap_alpha(const V* rd, V& are, V& aim) {
  V s0 = vset<V>(0.f), s1 = s0, s2 = s0;
#pragma unroll
  for (int w = 0; w < 8; w++) {
    s0 = vadd(s0, rd[3 * w]);
    s1 = vadd(s1, rd[3 * w + 1]);
    s2 = vadd(s2, rd[3 * w + 2]);
  }
#pragma unroll
  for (int l = 0; l < vlanes<V>(); l++) {
    const float pp = vlane(s2, l);
    vput(are, l, pp > 0.f ? vlane(s0, l) / pp : 0.f);
    vput(aim, l, pp > 0.f ? vlane(s1, l) / pp : 0.f);
  }
}
// e_o += alpha rho, e_e -= alpha A_ee^-1 A_eo rho, rho -= alpha p for one chirality at slots o, o + 128, ...
template <typename V>
__device__ __forceinline__ void sap_update(cv<V>* accO, cv<V>* accE, cv<V>* bufO, const cv<V>* bufE, int o, V are, V aim,
                                           const cv<V> r[6], const cv<V> p[6]) {
  const V nre = vsub(vset<V>(0.f), are), nim = vsub(vset<V>(0.f), aim);
#pragma unroll
  for (int c = 0; c < 6; c++, o += B4_VH) {
    cv<V> e = accO[o], t = bufE[o], f = accE[o], q = r[c];
    e.re = vfma(are, q.re, vfma(nim, q.im, e.re));
    e.im = vfma(are, q.im, vfma(aim, q.re, e.im));
    f.re = vfma(nre, t.re, vfma(aim, t.im, f.re));
    f.im = vfma(nre, t.im, vfma(nim, t.re, f.im));
    q.re = vfma(nre, p[c].re, vfma(aim, p[c].im, q.re));
    q.im = vfma(nre, p[c].im, vfma(nim, p[c].re, q.im));
    accO[o] = e;
    accE[o] = f;
    bufO[o] = q;
  }
}
// r = b - D x at site i of parity par, from the staged x (own, oth: its two parities) into out
template <int P, int PO, typename V, typename SO>
__device__ __forceinline__ void sap_residual(cv<V>* out, const cv<V>* own, const cv<V>* oth, const LaneField<P, V>& x,
                                             const LaneField<P, V>& b, const SO* __restrict__ U, const SO* __restrict__ C,
                                             const Geo& g, float mu, int blk, int i, int par) {
  cv<V> acc[12], v[12], s[12];
  v_hops_full<P, PO>(oth, x, U, g, blk, i, par, acc);
#pragma unroll
  for (int c = 0; c < 12; c++) v[c] = own[c * B4_VH + i];
  v_clover<PO, B4_VB>(C + (size_t)blk * 36 * B4_VB + par * B4_VH + i, v, s);
  v_twist(mu, v, s);
  b.load(blk, par * B4_VH + i, v);
#pragma unroll
  for (int c = 0; c < 12; c++) {
    cv<V> o;
    o.re = vsub(vfma(vset<V>(0.5f), acc[c].re, v[c].re), s[c].re);
    o.im = vsub(vfma(vset<V>(0.5f), acc[c].im, v[c].im), s[c].im);
    out[c * B4_VH + i] = o;
  }
}
// x = e (zero_x) or x + e at site i of parity par
template <int P, typename V>
__device__ __forceinline__ void sap_store(const LaneField<P, V>& x, const cv<V>* e, int blk, int i, int par, int zero_x, int r0,
                                          int nrhs) {
  cv<V> v[12];
  if (zero_x) {
#pragma unroll
    for (int c = 0; c < 12; c++) v[c] = e[c * B4_VH + i];
  } else {
    x.load(blk, par * B4_VH + i, v);
#pragma unroll
    for (int c = 0; c < 12; c++) {
      const cv<V> q = e[c * B4_VH + i];
      v[c].re = vadd(v[c].re, q.re);
      v[c].im = vadd(v[c].im, q.im);
    }
  }
  x.store(blk, par * B4_VH + i, v, r0, nrhs);
}

// Two right-hand sides: one thread per pair of sites (even i, odd i).
template <int P, int PO, typename V>
__global__ void __launch_bounds__(128, 2)
    k_sap_half_b4(Spinor<P> xf, Spinor<P> bf, const typename Prec<PO>::store2* __restrict__ U,
                  const typename Prec<PO>::store2* __restrict__ C, const typename Prec<PO>::store2* __restrict__ Ainv,
                  Geo g, SapArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cv<V>* bufE = reinterpret_cast<cv<V>*>(smem_raw);
  cv<V>* bufO = bufE + 12 * B4_VH;
  cv<V>* accE = bufO + 12 * B4_VH;
  cv<V>* accO = accE + 12 * B4_VH;
  V* red = reinterpret_cast<V*>(accO + 12 * B4_VH);  // [2][2 chiralities][4 warps][3]
  const int i = threadIdx.x, r0 = blockIdx.x * vlanes<V>();
  const int blk = a.blocks[blockIdx.y];
  const LaneField<P, V> x(xf, r0, a.nrhs, a.fstride, a.V), b(bf, r0, a.nrhs, a.fstride, a.V);
  const typename Prec<PO>::store2* ub = U + (size_t)blk * 36 * B4_VB;
  const typename Prec<PO>::store2* cb = C + (size_t)blk * 36 * B4_VB + B4_VH + i;
  const typename Prec<PO>::store2* ib = Ainv + (size_t)blk * 72 * B4_VH + i;

  // block residual on both parities, into accE and accO
  if (a.zero_x) {
    const int zb = a.zero_blocks[blockIdx.y];  // one block of the other colour is cleared per CTA
    cv<V> v[12];
#pragma unroll
    for (int c = 0; c < 12; c++) v[c].re = v[c].im = vset<V>(0.f);
    x.store(zb, i, v, r0, a.nrhs);
    x.store(zb, B4_VH + i, v, r0, a.nrhs);
    b.load(blk, i, v);
#pragma unroll
    for (int c = 0; c < 12; c++) accE[c * B4_VH + i] = v[c];
    b.load(blk, B4_VH + i, v);
#pragma unroll
    for (int c = 0; c < 12; c++) accO[c * B4_VH + i] = v[c];
  } else {
    {
      cv<V> v[12];
      x.load(blk, i, v);
#pragma unroll
      for (int c = 0; c < 12; c++) bufE[c * B4_VH + i] = v[c];
      x.load(blk, B4_VH + i, v);
#pragma unroll
      for (int c = 0; c < 12; c++) bufO[c * B4_VH + i] = v[c];
    }
    __syncthreads();
#pragma unroll 1
    for (int par = 0; par < 2; par++)
      sap_residual<P, PO>(par ? accO : accE, par ? bufO : bufE, par ? bufE : bufO, x, b, U, C, g, a.mu, blk, i, par);
    __syncthreads();  // the reads of bufE and bufO are done
  }
  // step 0: bufE = A_ee^-1 r_e, rho = bufO = r_o - A_oe bufE; steps 1 ... nmr: minimal residual
#pragma unroll 1
  for (int k = 0; k <= a.nmr; k++) {
    {
      cv<V> h[12], t[12];
      if (k == 0) {
#pragma unroll
        for (int c = 0; c < 12; c++) h[c] = accE[c * B4_VH + i];
      } else {
        cv<V> q[12];
        v_hops_inside<PO, true>(bufO, ub, i, 0, h);
        v_hops_inside<PO, false>(bufO, ub, i, 0, q);
#pragma unroll
        for (int c = 0; c < 12; c++) {
          h[c].re = vmul(vset<V>(-0.5f), vadd(h[c].re, q[c].re));
          h[c].im = vmul(vset<V>(-0.5f), vadd(h[c].im, q[c].im));
        }
      }
      v_site_inv_half<PO, B4_VH>(ib, h, t);
      v_site_inv_half<PO, B4_VH>(ib + 36 * B4_VH, h + 6, t + 6);
#pragma unroll
      for (int c = 0; c < 12; c++) {
        bufE[c * B4_VH + i] = t[c];
        if (k == 0) accE[c * B4_VH + i] = t[c];
      }
    }
    __syncthreads();
    cv<V> h[12];
    {
      cv<V> q[12];
      v_hops_inside<PO, true>(bufE, ub, i, 1, h);
      v_hops_inside<PO, false>(bufE, ub, i, 1, q);
#pragma unroll
      for (int c = 0; c < 12; c++) {
        h[c].re = vadd(h[c].re, q[c].re);
        h[c].im = vadd(h[c].im, q[c].im);
      }
    }
    if (k == 0) {
#pragma unroll
      for (int c = 0; c < 12; c++) {
        cv<V> r = accO[c * B4_VH + i];
        r.re = vfma(vset<V>(0.5f), h[c].re, r.re);
        r.im = vfma(vset<V>(0.5f), h[c].im, r.im);
        bufO[c * B4_VH + i] = r;
        r.re = r.im = vset<V>(0.f);
        accO[c * B4_VH + i] = r;
      }
      __syncthreads();
      continue;
    }
    cv<V> r[12], p[12];
#pragma unroll
    for (int c = 0; c < 12; c++) r[c] = bufO[c * B4_VH + i];
    v_clover<PO, B4_VB>(cb, r, p);
#pragma unroll
    for (int c = 0; c < 12; c++) {
      const float mu = c < 6 ? a.mu : -a.mu;
      p[c].re = vfma(vset<V>(-mu), r[c].im, vfma(vset<V>(0.5f), h[c].re, p[c].re));
      p[c].im = vfma(vset<V>(mu), r[c].re, vfma(vset<V>(0.5f), h[c].im, p[c].im));
    }
    V* rd = red + (k & 1) * 24;
#pragma unroll
    for (int q = 0; q < 2; q++) {
      V s0, s1, s2;
      sap_dots(p + 6 * q, r + 6 * q, s0, s1, s2);
      if ((i & 31) == 0) {
        const int w = 4 * q + (i >> 5);
        rd[3 * w] = s0;
        rd[3 * w + 1] = s1;
        rd[3 * w + 2] = s2;
      }
    }
    __syncthreads();
    V are, aim;
    sap_alpha(rd, are, aim);
    sap_update(accO, accE, bufO, bufE, i, are, aim, r, p);
    sap_update(accO, accE, bufO, bufE, 6 * B4_VH + i, are, aim, r + 6, p + 6);
    __syncthreads();
  }
#pragma unroll 1
  for (int par = 0; par < 2; par++) sap_store(x, par ? accO : accE, blk, i, par, a.zero_x, r0, a.nrhs);
}

// One right-hand side, where latency counts: 256 threads.  The residual takes one thread per site; in the
// block solve two threads share a site, the first (half 0) sums the forward hops, the second the backward
// hops, they exchange the chirality the other one owns, and each goes on with its own chirality
// (inverse, clover, minimal-residual update).
template <int P, int PO, typename V>
__global__ void __launch_bounds__(256, 2)
    k_sap_half_b4_one(Spinor<P> xf, Spinor<P> bf, const typename Prec<PO>::store2* __restrict__ U,
                      const typename Prec<PO>::store2* __restrict__ C, const typename Prec<PO>::store2* __restrict__ Ainv,
                      Geo g, SapArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cv<V>* bufE = reinterpret_cast<cv<V>*>(smem_raw);
  cv<V>* bufO = bufE + 12 * B4_VH;
  cv<V>* accE = bufO + 12 * B4_VH;
  cv<V>* accO = accE + 12 * B4_VH;
  V* red = reinterpret_cast<V*>(accO + 12 * B4_VH);  // [2][8 warps][3]
  const int hf = threadIdx.x >> 7, i = threadIdx.x & 127, r0 = blockIdx.x * vlanes<V>();
  const int blk = a.blocks[blockIdx.y];
  const typename Prec<PO>::store2* ub = U + (size_t)blk * 36 * B4_VB;

  const LaneField<P, V> x(xf, r0, a.nrhs, a.fstride, a.V);
  // block residual, thread = site (half = parity), into accE and accO
  {
    const LaneField<P, V> b(bf, r0, a.nrhs, a.fstride, a.V);
    cv<V>* out = hf ? accO : accE;
    cv<V> v[12];
    if (a.zero_x) {
#pragma unroll
      for (int c = 0; c < 12; c++) v[c].re = v[c].im = vset<V>(0.f);
      x.store(a.zero_blocks[blockIdx.y], threadIdx.x, v, r0, a.nrhs);  // clear one block of the other colour
      b.load(blk, threadIdx.x, v);
#pragma unroll
      for (int c = 0; c < 12; c++) out[c * B4_VH + i] = v[c];
    } else {
      cv<V>* own = hf ? bufO : bufE;
      x.load(blk, threadIdx.x, v);
#pragma unroll
      for (int c = 0; c < 12; c++) own[c * B4_VH + i] = v[c];
      __syncthreads();
      sap_residual<P, PO>(out, own, hf ? bufE : bufO, x, b, U, C, g, a.mu, blk, i, hf);
    }
    __syncthreads();
  }
  const int o0 = 6 * hf * B4_VH + i, x0 = 6 * (hf ^ 1) * B4_VH + i;  // own chirality, the other one
  const typename Prec<PO>::store2* cb = C + ((size_t)blk * 36 + 18 * hf) * B4_VB + B4_VH + i;
  const typename Prec<PO>::store2* ib = Ainv + ((size_t)blk * 72 + 36 * hf) * B4_VH + i;
  const float mu = hf ? -a.mu : a.mu;
  // phases 0, 1: bufE = A_ee^-1 r_e, rho = bufO = r_o - A_oe bufE; phases 2 k, 2 k + 1: MR step k
#pragma unroll 1
  for (int ph = 0; ph < 2 * a.nmr + 2; ph++) {
    const int par = ph & 1;
    cv<V>* dst = par ? bufO : bufE;
    cv<V> r[6], h[6];
    if (ph == 0) {
#pragma unroll
      for (int c = 0; c < 6; c++) h[c] = accE[o0 + c * B4_VH];
    } else {
      cv<V> acc[12];
      if (par)
#pragma unroll
        for (int c = 0; c < 6; c++) r[c] = (ph == 1 ? accO : bufO)[o0 + c * B4_VH];
      // partial sums of the other chirality go to its owner: in an odd phase through the slots of bufO whose
      // entries are now in r, in an even phase through slots of bufE, whose entries are no longer needed
      cv<V>* put = dst + (par ? o0 : x0);
      const cv<V>* get = dst + (par ? x0 : o0);
      if (hf == 0) {
        v_hops_inside<PO, true>(par ? bufE : bufO, ub, i, par, acc);
#pragma unroll
        for (int c = 0; c < 6; c++) put[c * B4_VH] = acc[6 + c];
#pragma unroll
        for (int c = 0; c < 6; c++) h[c] = acc[c];
      } else {
        v_hops_inside<PO, false>(par ? bufE : bufO, ub, i, par, acc);
#pragma unroll
        for (int c = 0; c < 6; c++) put[c * B4_VH] = acc[c];
#pragma unroll
        for (int c = 0; c < 6; c++) h[c] = acc[6 + c];
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 6; c++) {
        const cv<V> q = get[c * B4_VH];
        h[c].re = vadd(h[c].re, q.re);
        h[c].im = vadd(h[c].im, q.im);
      }
    }
    if (par == 0) {  // bufE = A_ee^-1 h, h = r_e or H_eo rho
      cv<V> t[6];
      if (ph)
#pragma unroll
        for (int c = 0; c < 6; c++) {
          h[c].re = vmul(vset<V>(-0.5f), h[c].re);
          h[c].im = vmul(vset<V>(-0.5f), h[c].im);
        }
      v_site_inv_half<PO, B4_VH>(ib, h, t);
#pragma unroll
      for (int c = 0; c < 6; c++) {
        bufE[o0 + c * B4_VH] = t[c];
        if (ph == 0) accE[o0 + c * B4_VH] = t[c];
      }
      __syncthreads();
      continue;
    }
    if (ph == 1) {
      __syncthreads();  // the exchanged sums are read
#pragma unroll
      for (int c = 0; c < 6; c++) {
        r[c].re = vfma(vset<V>(0.5f), h[c].re, r[c].re);
        r[c].im = vfma(vset<V>(0.5f), h[c].im, r[c].im);
        bufO[o0 + c * B4_VH] = r[c];
        r[c].re = r[c].im = vset<V>(0.f);
        accO[o0 + c * B4_VH] = r[c];
      }
      __syncthreads();
      continue;
    }
    cv<V> p[6];
    v_clover_half<PO, B4_VB>(cb, r, p);
#pragma unroll
    for (int c = 0; c < 6; c++) {
      p[c].re = vfma(vset<V>(-mu), r[c].im, vfma(vset<V>(0.5f), h[c].re, p[c].re));
      p[c].im = vfma(vset<V>(mu), r[c].re, vfma(vset<V>(0.5f), h[c].im, p[c].im));
    }
    V s0, s1, s2;
    sap_dots(p, r, s0, s1, s2);
    V* rd = red + (ph & 2) * 12;  // alternates from step to step
    if ((i & 31) == 0) {
      const int w = threadIdx.x >> 5;
      rd[3 * w] = s0;
      rd[3 * w + 1] = s1;
      rd[3 * w + 2] = s2;
    }
    __syncthreads();
    V are, aim;
    sap_alpha(rd, are, aim);
    sap_update(accO, accE, bufO, bufE, o0, are, aim, r, p);
    __syncthreads();
  }
  sap_store(x, hf ? accO : accE, blk, i, hf, a.zero_x, r0, a.nrhs);
}

template <int P, int PO>
static void launch_sap_b4(const FineGeom& g, void* x, float* xn, const void* b, const float* bn, const void* links,
                          const void* clover, const void* sinv, const int* blocks, const int* zero_blocks, int nblocks,
                          int zero_x, int nmr, double mu, int nrhs, cudaStream_t s) {
  typedef typename Prec<P>::store2 S;
  typedef typename Prec<PO>::store2 SO;
  Geo q{g.Vb, g.Nb, g.loc_nbr.as<uint32_t>(), g.blk_nbr.as<int>()};
  const bool two = nrhs > 1;
  const void* kern = two ? (const void*)k_sap_half_b4<P, PO, float2> : (const void*)k_sap_half_b4_one<P, PO, float>;
  const size_t smem = two ? sap_b4_smem<float2>() : sap_b4_smem<float>();
  set_dynamic_smem(kern, smem);
  const Spinor<P> X{(S*)x, xn, g.Vb}, B{(S*)b, (float*)bn, g.Vb};
  for (int b0 = 0; b0 < nblocks; b0 += 65535) {  // grid.y, as below
    const int nb = nblocks - b0 < 65535 ? nblocks - b0 : 65535;
    SapArgs<float> a{blocks + b0, nrhs, zero_blocks + b0, zero_x, nmr, (float)mu, (size_t)g.V * 12, g.V};
    if (two)
      k_sap_half_b4<P, PO, float2><<<dim3((nrhs + 1) / 2, nb), 128, smem, s>>>(X, B, (const SO*)links, (const SO*)clover,
                                                                             (const SO*)sinv, q, a);
    else
      k_sap_half_b4_one<P, PO, float><<<dim3(1, nb), 256, smem, s>>>(X, B, (const SO*)links, (const SO*)clover,
                                                                    (const SO*)sinv, q, a);
    CKL("sap_half");
  }
}

bool sap_b4_blocks(const FineGeom& g) { return g.b[0] == 4 && g.b[1] == 4 && g.b[2] == 4 && g.b[3] == 4; }

size_t sap_smem_bytes(int Vb, int prec) {
  return prec == PREC_F64 ? sap_group_smem<double>(Vb / 2) : sap_group_smem<float>(Vb / 2);
}

int sap_threads(int Vb) {
  int Vh = Vb / 2;
  return ((Vh + 31) / 32) * 32;
}

template <int P, int RG>
static void launch_sap_rg(const FineGeom& g, void* x, float* xn, const void* b, const float* bn, const void* links,
                          const void* clover, const void* sinv, const int* blocks, const int* zero_blocks, int nblocks,
                          int zero_x, int nmr, double mu, int nrhs, cudaStream_t s) {
  typedef typename Prec<P>::store2 S;
  typedef typename Prec<P>::real R;
  Geo q{g.Vb, g.Nb, g.loc_nbr.as<uint32_t>(), g.blk_nbr.as<int>()};
  const size_t smem = (size_t)RG * sap_group_smem<R>(g.Vb / 2);
  set_dynamic_smem((const void*)k_sap_half<P, RG>, smem);
  // grid.y is at most 65535: on large lattices (e.g. 128 x 64^3 with 4^4 blocks, 65536 blocks per
  // colour) the blocks of the colour go in several launches, which is exact since they are independent
  for (int b0 = 0; b0 < nblocks; b0 += 65535) {
    const int nb = nblocks - b0 < 65535 ? nblocks - b0 : 65535;
    SapArgs<R> a{blocks + b0, nrhs, zero_blocks + b0, zero_x, nmr, (R)mu, (size_t)g.V * 12, g.V};
    dim3 grid((nrhs + RG - 1) / RG, nb);
    k_sap_half<P, RG><<<grid, RG * sap_threads(g.Vb), smem, s>>>(
        Spinor<P>{(S*)x, xn, g.Vb}, Spinor<P>{(S*)b, (float*)bn, g.Vb}, Links<P>{(const S*)links, g.Vb},
        Clover<P>{(const S*)clover, g.Vb}, SiteInv<P>{(const S*)sinv, g.Vb / 2}, q, a);
    CKL("sap_half");
  }
}

// Right-hand sides per CTA: up to DDTM_SAP_RG where the batch and the shared memory allow it, fewer
// otherwise; FP64 keeps one.  For blocks other than 4^4; measured on 4^4 blocks before these had kernels of
// their own: two per CTA (99 KB of FP32 block vectors, 2 CTAs per SM) was fastest at 32^3 x 64 with 12 and 24
// right-hand sides: 34.7 / 68.9 ms per two cycles, against 36.7 / 74.2 ms with one and 37.3 / 73.8 ms with
// four (whose 198 KB of shared memory leave little L1 for the shared operator data).
#ifndef DDTM_SAP_RG
#define DDTM_SAP_RG 2
#endif
static int sap_rhs_groups(const FineGeom& g, int prec, int nrhs) {
  if (prec == PREC_F64 || nrhs <= 1) return 1;
  const size_t grp = sap_group_smem<float>(g.Vb / 2);
  const int gt = sap_threads(g.Vb);
  if (DDTM_SAP_RG >= 4 && nrhs >= 3 && 4 * grp <= 200 * 1024 && 4 * gt <= 1024) return 4;
  if (DDTM_SAP_RG >= 2 && 2 * grp <= 200 * 1024 && 2 * gt <= 1024) return 2;
  return 1;
}

template <int P>
static void launch_sap_half_t(const FineGeom& g, int po, void* x, float* xn, const void* b, const float* bn, const void* links,
                              const void* clover, const void* sinv, const int* blocks, const int* zero_blocks,
                              int nblocks, int zero_x, int nmr, double mu, int nrhs, cudaStream_t s) {
  const int rg = sap_rhs_groups(g, P, nrhs);
  if constexpr (P != PREC_F64) {
    if (sap_b4_blocks(g)) {
      if (po == PREC_F32)
        launch_sap_b4<P, PREC_F32>(g, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
      else
        launch_sap_b4<P, P>(g, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
      return;
    }
    if (rg == 4) {
      launch_sap_rg<P, 4>(g, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
      return;
    }
    if (rg == 2) {
      launch_sap_rg<P, 2>(g, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
      return;
    }
  }
  launch_sap_rg<P, 1>(g, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
}

void launch_sap_half(const FineGeom& g, int prec, int po, void* x, float* xn, const void* b, const float* bn, const void* links,
                     const void* clover, const void* sinv, const int* blocks, const int* zero_blocks, int nblocks,
                     int zero_x, int nmr, double mu, int nrhs, cudaStream_t s) {
  ScopedTimer timer_(prec == PREC_F64 ? "sap_half_f64" : prec == PREC_F32 ? "sap_half_f32" : "sap_half_f16", s, nrhs);
  if (prec == PREC_F64)
    launch_sap_half_t<PREC_F64>(g, po, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
  else if (prec == PREC_F32)
    launch_sap_half_t<PREC_F32>(g, po, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
  else
    launch_sap_half_t<PREC_F16>(g, po, x, xn, b, bn, links, clover, sinv, blocks, zero_blocks, nblocks, zero_x, nmr, mu, nrhs, s);
}

}  // namespace ddtm
