// The Wilson hop, the site term and the even-site inverse for one or two
// right-hand sides per thread, on 4^4 lattice blocks (Sec. 2.1, 2.4).
//
// V = float holds one right-hand side, V = float2 two of them in the halves of
// packed f32x2 instructions: the two share every link, clover and inverse entry,
// so the loads, the conversions from FP16 storage and the address arithmetic are
// paid once for both and one issue slot carries two multiply-adds.  Every operation is an explicitly
// rounded add, sub or fma, so a right-hand side gets the same bits in either
// form and whatever its partner holds.
//
// Inside a 4^4 block the neighbour index is arithmetic: site i of a parity has
// lexicographic index 2 i + b with b = lx & 1 fixed by the parity, so a hop in
// y, z, t moves i by 2, 8, 32, a hop in x by 0 or 1, and the 32 lanes of a warp
// share one t (hops in t leave the block for whole warps).
#pragma once

#include "common.cuh"

namespace ddtm {

// ---- one or two FP32 lanes -----------------------------------------------------
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);  // a - b, rounded once
}
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
template <typename V> __device__ __forceinline__ V vset(float a);
template <> __device__ __forceinline__ float vset<float>(float a) { return a; }
template <> __device__ __forceinline__ float2 vset<float2>(float a) { return make_float2(a, a); }
template <typename V> __host__ __device__ constexpr int vlanes() { return (int)(sizeof(V) / sizeof(float)); }
__device__ __forceinline__ float vlane(float a, int) { return a; }
__device__ __forceinline__ float vlane(float2 a, int l) { return l ? a.y : a.x; }
__device__ __forceinline__ void vput(float& a, int, float v) { a = v; }
__device__ __forceinline__ void vput(float2& a, int l, float v) { if (l) a.y = v; else a.x = v; }
template <bool MINUS, typename V> __device__ __forceinline__ V vpm(V a, V b) { return MINUS ? vsub(a, b) : vadd(a, b); }

// one complex number per lane; 8 or 16 bytes, one shared-memory access
template <typename V> struct __align__(2 * sizeof(V)) cv { V re, im; };

// ---- FP32 or FP16 operator entries as loaded, converted where they are used -------
template <int P> struct Raw;
template <> struct Raw<PREC_F32> {
  float2 v;
  __device__ __forceinline__ void load(const float2* p) { v = __ldg(p); }
  __device__ __forceinline__ void zero() { v = make_float2(0.f, 0.f); }
  __device__ __forceinline__ float2 get() const { return v; }
};
template <> struct Raw<PREC_F16> {
  __half2 v;
  __device__ __forceinline__ void load(const __half2* p) { v = __ldg(p); }
  __device__ __forceinline__ void zero() { v = __half2half2(__ushort_as_half(0)); }
  __device__ __forceinline__ float2 get() const { return __half22float2(v); }
};

// ---- geometry of a 4^4 block -----------------------------------------------------
static const int B4_VB = 256, B4_VH = 128;
struct B4Nbr {
  int i;        // index of the neighbour within the other parity
  bool inside;  // the hop stays in the block (else i is the wrapped site of the neighbour block)
};
// neighbour of site i of parity par in direction mu
template <int MU, bool FWD> __device__ __forceinline__ B4Nbr b4_nbr(int i, int par) {
  B4Nbr n;
  if (MU == 1) {  // x: lx = 2 (i & 1) + b, b = parity of the site minus that of ly + lz + lt
    const int b = (par ^ (i >> 1) ^ (i >> 3) ^ (i >> 5)) & 1;
    if (FWD) {
      n.inside = !(b & i & 1);
      n.i = b ? (n.inside ? i + 1 : i - 1) : i;
    } else {
      n.inside = (b | (i & 1)) != 0;
      n.i = b ? i : (n.inside ? i - 1 : i + 1);
    }
  } else {
    const int sh = MU == 2 ? 1 : MU == 3 ? 3 : 5, step = 1 << sh, l = (i >> sh) & 3;
    n.inside = FWD ? l != 3 : l != 0;
    n.i = FWD ? (n.inside ? i + step : i - 3 * step) : (n.inside ? i - step : i + 3 * step);
  }
  return n;
}

// ---- spin algebra (gamma basis of common.cuh) ------------------------------------
// h = upper half of (1 -+ gamma_mu) p
template <int MU, bool FWD, typename V> __device__ __forceinline__ void v_project(const cv<V> p[12], cv<V> h[6]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const cv<V>&u0 = p[c], &u1 = p[3 + c], &l0 = p[6 + c], &l1 = p[9 + c];
    cv<V>&h0 = h[c], &h1 = h[3 + c];
    if (MU == 0) {  // G = 1
      h0.re = vpm<FWD>(u0.re, l0.re); h0.im = vpm<FWD>(u0.im, l0.im);
      h1.re = vpm<FWD>(u1.re, l1.re); h1.im = vpm<FWD>(u1.im, l1.im);
    } else if (MU == 1) {  // (i l1, i l0)
      h0.re = vpm<!FWD>(u0.re, l1.im); h0.im = vpm<FWD>(u0.im, l1.re);
      h1.re = vpm<!FWD>(u1.re, l0.im); h1.im = vpm<FWD>(u1.im, l0.re);
    } else if (MU == 2) {  // (l1, -l0)
      h0.re = vpm<FWD>(u0.re, l1.re); h0.im = vpm<FWD>(u0.im, l1.im);
      h1.re = vpm<!FWD>(u1.re, l0.re); h1.im = vpm<!FWD>(u1.im, l0.im);
    } else {  // (i l0, -i l1)
      h0.re = vpm<!FWD>(u0.re, l0.im); h0.im = vpm<FWD>(u0.im, l0.re);
      h1.re = vpm<FWD>(u1.re, l1.im); h1.im = vpm<!FWD>(u1.im, l1.re);
    }
  }
}
// acc += (w, lower(w)), w = U h (FWD) or U^+ h, colour by colour of w
template <int MU, bool FWD, int P, typename V>
__device__ __forceinline__ void v_link_hop(const Raw<P> u[9], const cv<V> h[6], cv<V> acc[12]) {
#pragma unroll
  for (int a = 0; a < 3; a++) {
    cv<V> w0, w1;  // the two spins of colour a
    V m0, m1;      // the part that is subtracted: ui h.im from the real part (FWD), ui h.re from the imaginary part
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const float2 f = u[FWD ? a * 3 + b : b * 3 + a].get();
      const V ur = vset<V>(f.x), ui = vset<V>(f.y);
      const cv<V>&x0 = h[b], &x1 = h[3 + b];
      w0.re = b ? vfma(ur, x0.re, w0.re) : vmul(ur, x0.re);
      w0.im = b ? vfma(ur, x0.im, w0.im) : vmul(ur, x0.im);
      w1.re = b ? vfma(ur, x1.re, w1.re) : vmul(ur, x1.re);
      w1.im = b ? vfma(ur, x1.im, w1.im) : vmul(ur, x1.im);
      if (FWD) {
        w0.im = vfma(ui, x0.re, w0.im);
        w1.im = vfma(ui, x1.re, w1.im);
        m0 = b ? vfma(ui, x0.im, m0) : vmul(ui, x0.im);
        m1 = b ? vfma(ui, x1.im, m1) : vmul(ui, x1.im);
      } else {
        w0.re = vfma(ui, x0.im, w0.re);
        w1.re = vfma(ui, x1.im, w1.re);
        m0 = b ? vfma(ui, x0.re, m0) : vmul(ui, x0.re);
        m1 = b ? vfma(ui, x1.re, m1) : vmul(ui, x1.re);
      }
    }
    if (FWD) {
      w0.re = vsub(w0.re, m0);
      w1.re = vsub(w1.re, m1);
    } else {
      w0.im = vsub(w0.im, m0);
      w1.im = vsub(w1.im, m1);
    }
    cv<V>&l0 = acc[6 + a], &l1 = acc[9 + a];
    acc[a].re = vadd(acc[a].re, w0.re); acc[a].im = vadd(acc[a].im, w0.im);
    acc[3 + a].re = vadd(acc[3 + a].re, w1.re); acc[3 + a].im = vadd(acc[3 + a].im, w1.im);
    if (MU == 0) {  // fwd -w, bwd +w
      l0.re = vpm<FWD>(l0.re, w0.re); l0.im = vpm<FWD>(l0.im, w0.im);
      l1.re = vpm<FWD>(l1.re, w1.re); l1.im = vpm<FWD>(l1.im, w1.im);
    } else if (MU == 1) {  // fwd +(i w1, i w0)
      l0.re = vpm<FWD>(l0.re, w1.im); l0.im = vpm<!FWD>(l0.im, w1.re);
      l1.re = vpm<FWD>(l1.re, w0.im); l1.im = vpm<!FWD>(l1.im, w0.re);
    } else if (MU == 2) {  // fwd +(w1, -w0)
      l0.re = vpm<!FWD>(l0.re, w1.re); l0.im = vpm<!FWD>(l0.im, w1.im);
      l1.re = vpm<FWD>(l1.re, w0.re); l1.im = vpm<FWD>(l1.im, w0.im);
    } else {  // fwd +(i w0, -i w1)
      l0.re = vpm<FWD>(l0.re, w0.im); l0.im = vpm<!FWD>(l0.im, w0.re);
      l1.re = vpm<!FWD>(l1.re, w1.im); l1.im = vpm<FWD>(l1.im, w1.re);
    }
  }
}

// y = S_h x for one packed Hermitian 6x6 block at p (component stride VB)
template <int P, int VB, typename V, typename S>
__device__ __forceinline__ void v_clover_half(const S* __restrict__ p, const cv<V> x[6], cv<V> y[6]) {
#pragma unroll
  for (int k = 0; k < 3; k++) {
    Raw<P> d;
    d.load(p + k * VB);
    const float2 f = d.get();
    const V a = vset<V>(f.x), b = vset<V>(f.y);
    y[2 * k].re = vmul(a, x[2 * k].re); y[2 * k].im = vmul(a, x[2 * k].im);
    y[2 * k + 1].re = vmul(b, x[2 * k + 1].re); y[2 * k + 1].im = vmul(b, x[2 * k + 1].im);
  }
  int slot = 3;
#pragma unroll
  for (int i = 0; i < 6; i++)
#pragma unroll
    for (int j = i + 1; j < 6; j++, slot++) {
      Raw<P> d;
      d.load(p + slot * VB);
      const float2 f = d.get();
      const V ur = vset<V>(f.x), ui = vset<V>(f.y), un = vset<V>(-f.y);
      y[i].re = vfma(ur, x[j].re, vfma(un, x[j].im, y[i].re));
      y[i].im = vfma(ur, x[j].im, vfma(ui, x[j].re, y[i].im));
      y[j].re = vfma(ur, x[i].re, vfma(ui, x[i].im, y[j].re));
      y[j].im = vfma(ur, x[i].im, vfma(un, x[i].re, y[j].im));
    }
}
template <int P, int VB, typename V, typename S>
__device__ __forceinline__ void v_clover(const S* __restrict__ p, const cv<V> x[12], cv<V> y[12]) {
  v_clover_half<P, VB>(p, x, y);
  v_clover_half<P, VB>(p + 18 * VB, x + 6, y + 6);
}
// y = (A_ee^-1)_h x, full 6x6 of one chirality at p (component stride VH)
template <int P, int VH, typename V, typename S>
__device__ __forceinline__ void v_site_inv_half(const S* __restrict__ p, const cv<V> x[6], cv<V> y[6]) {
  V n[6];
#pragma unroll
  for (int j = 0; j < 6; j++) n[j] = vsub(vset<V>(0.f), x[j].im);
#pragma unroll
  for (int i = 0; i < 6; i++)
#pragma unroll
    for (int j = 0; j < 6; j++) {
      Raw<P> d;
      d.load(p + (i * 6 + j) * VH);
      const float2 f = d.get();
      const V ur = vset<V>(f.x), ui = vset<V>(f.y);
      y[i].re = j ? vfma(ur, x[j].re, y[i].re) : vmul(ur, x[j].re);
      y[i].im = j ? vfma(ur, x[j].im, y[i].im) : vmul(ur, x[j].im);
      y[i].re = vfma(ui, n[j], y[i].re);
      y[i].im = vfma(ui, x[j].re, y[i].im);
    }
}
// y += i mu Gamma5 x
template <typename V> __device__ __forceinline__ void v_twist(float mu, const cv<V> x[12], cv<V> y[12]) {
#pragma unroll
  for (int c = 0; c < 12; c++) {
    const V m = vset<V>(c < 6 ? mu : -mu), q = vset<V>(c < 6 ? -mu : mu);
    y[c].re = vfma(q, x[c].im, y[c].re);
    y[c].im = vfma(m, x[c].re, y[c].im);
  }
}

// ---- fields: component c of site loc of block blk, V's lanes from consecutive rhs ------
// Lane l reads right-hand side r0 + l (the last one again where the batch ends).
template <int P, typename V> struct LaneField {
  typedef typename Prec<P>::store2 S;
  S* d[vlanes<V>()];
  float* nrm[vlanes<V>()];
  __device__ __forceinline__ LaneField(const Spinor<P>& f, int r0, int nrhs, size_t fstride, long Vs) {
#pragma unroll
    for (int l = 0; l < vlanes<V>(); l++) {
      const int r = r0 + l < nrhs ? r0 + l : nrhs - 1;
      d[l] = f.d + (size_t)r * fstride;
      nrm[l] = Prec<P>::scaled ? f.nrm + (size_t)r * Vs : nullptr;
    }
  }
  // plain loads: SAP writes some of these fields in the same launch
  __device__ __forceinline__ void load(int blk, int loc, cv<V> v[12]) const {
#pragma unroll
    for (int l = 0; l < vlanes<V>(); l++) {
      const S* p = d[l] + (size_t)blk * 12 * B4_VB + loc;
      const float s = Prec<P>::scaled ? nrm[l][(size_t)blk * B4_VB + loc] : 1.f;
#pragma unroll
      for (int c = 0; c < 12; c++) {
        const cplx<float> a = ldw(p + c * B4_VB);
        vput(v[c].re, l, Prec<P>::scaled ? __fmul_rn(s, a.re) : a.re);
        vput(v[c].im, l, Prec<P>::scaled ? __fmul_rn(s, a.im) : a.im);
      }
    }
  }
  __device__ __forceinline__ void store(int blk, int loc, const cv<V> v[12], int r0, int nrhs) const {
#pragma unroll
    for (int l = 0; l < vlanes<V>(); l++) {
      if (r0 + l >= nrhs) break;
      Spinor<P> f{d[l], nrm[l], B4_VB};
      cplx<float> a[12];
#pragma unroll
      for (int c = 0; c < 12; c++) a[c] = cplx<float>(vlane(v[c].re, l), vlane(v[c].im, l));
      f.store(blk, loc, a);
    }
  }
};

// acc += the hop of direction (MU, FWD) inside the block (0 where it leaves it): v = the
// other parity's block vector, v[c * B4_VH + i]; ub = the block's links
template <int P, int MU, bool FWD, typename V, typename S>
__device__ __forceinline__ void v_hop_inside(const cv<V>* v, const S* __restrict__ ub, int i, int par, cv<V> acc[12]) {
  const B4Nbr n = b4_nbr<MU, FWD>(i, par);
  if (MU == 0 && !n.inside) return;  // whole warps
  const S* ul = ub + MU * 9 * B4_VB + (FWD ? par * B4_VH + i : (par ^ 1) * B4_VH + n.i);
  Raw<P> u[9];
#pragma unroll
  for (int q = 0; q < 9; q++) {
    u[q].zero();
    if (n.inside) u[q].load(ul + q * B4_VB);
  }
  cv<V> h[6];
  {
    cv<V> p[12];
#pragma unroll
    for (int c = 0; c < 12; c++) p[c] = v[c * B4_VH + n.i];
    v_project<MU, FWD>(p, h);
  }
  v_link_hop<MU, FWD, P>(u, h, acc);
}
// acc = sum of the 4 forward or the 4 backward hops inside the block (without the factor -1/2)
template <int P, bool FWD, typename V, typename S>
__device__ __forceinline__ void v_hops_inside(const cv<V>* v, const S* __restrict__ ub, int i, int par, cv<V> acc[12]) {
#pragma unroll
  for (int c = 0; c < 12; c++) acc[c].re = acc[c].im = vset<V>(0.f);
  v_hop_inside<P, 0, FWD>(v, ub, i, par, acc);
  v_hop_inside<P, 1, FWD>(v, ub, i, par, acc);
  v_hop_inside<P, 2, FWD>(v, ub, i, par, acc);
  v_hop_inside<P, 3, FWD>(v, ub, i, par, acc);
}

// acc += the hop of the full stencil: neighbours in the block from shared memory (v, the other
// parity), neighbours outside from the field in memory
template <int P, int PO, int MU, bool FWD, typename V, typename S>
__device__ __forceinline__ void v_hop_full(const cv<V>* v, const LaneField<P, V>& x, const S* __restrict__ U,
                                           const Geo& g, int blk, int i, int par, cv<V> acc[12]) {
  const B4Nbr n = b4_nbr<MU, FWD>(i, par);
  const int b = __ldg(g.blk_nbr + (2 * MU + (FWD ? 0 : 1)) * g.Nb + blk);
  const int nblk = n.inside ? blk : b & 0x3fffffff, nloc = (par ^ 1) * B4_VH + n.i;
  const S* ul = FWD ? U + ((size_t)blk * 4 + MU) * 9 * B4_VB + par * B4_VH + i
                    : U + ((size_t)nblk * 4 + MU) * 9 * B4_VB + nloc;
  Raw<PO> u[9];
#pragma unroll
  for (int q = 0; q < 9; q++) u[q].load(ul + q * B4_VB);
  cv<V> h[6];
  {
    cv<V> p[12];
    if (n.inside) {
#pragma unroll
      for (int c = 0; c < 12; c++) p[c] = v[c * B4_VH + n.i];
    } else {
      x.load(nblk, nloc, p);
    }
    v_project<MU, FWD>(p, h);
  }
  if (MU == 0) {  // antiperiodic t: the sign of the hops that wrap
    const V s = vset<V>(!n.inside && ((b >> 30) & 1) ? -1.f : 1.f);
#pragma unroll
    for (int k = 0; k < 6; k++) {
      h[k].re = vmul(s, h[k].re);
      h[k].im = vmul(s, h[k].im);
    }
  }
  v_link_hop<MU, FWD, PO>(u, h, acc);
}
template <int P, int PO, typename V, typename S>
__device__ __forceinline__ void v_hops_full(const cv<V>* v, const LaneField<P, V>& x, const S* __restrict__ U,
                                            const Geo& g, int blk, int i, int par, cv<V> acc[12]) {
#pragma unroll
  for (int c = 0; c < 12; c++) acc[c].re = acc[c].im = vset<V>(0.f);
  v_hop_full<P, PO, 0, true>(v, x, U, g, blk, i, par, acc);
  v_hop_full<P, PO, 0, false>(v, x, U, g, blk, i, par, acc);
  v_hop_full<P, PO, 1, true>(v, x, U, g, blk, i, par, acc);
  v_hop_full<P, PO, 1, false>(v, x, U, g, blk, i, par, acc);
  v_hop_full<P, PO, 2, true>(v, x, U, g, blk, i, par, acc);
  v_hop_full<P, PO, 2, false>(v, x, U, g, blk, i, par, acc);
  v_hop_full<P, PO, 3, true>(v, x, U, g, blk, i, par, acc);
  v_hop_full<P, PO, 3, false>(v, x, U, g, blk, i, par, acc);
}

}  // namespace ddtm
