// Arnoldi step of the coarsest even-odd GMRES (Sec. 2.5) on image-ordered vectors: the Krylov basis is kept
// as the FP16 operand images the tensor-core stencil reads, so the operator takes a basis vector as it is,
// and one cooperative kernel does everything between two operator applications.
//
// k_gs_step: every warp owns tiles of 32 items; an item is 8 dofs of one right-hand side (32 bytes of a basis
// vector, 64 of w), so a lane always works for one right-hand side (lane % 4 within the warp's group of four)
// and sums over a tile take three shuffles.
//   A  partial <V_i, w> per CTA                     -> grid barrier -> summed over CTAs in FP64 -> barrier
//   B  w -= sum_i h_i V_i (w in registers), norms   -> barrier
//   C  V_next = w / ||w|| in FP16; one warp per right-hand side does the Givens update
// The grid is one wave, one CTA per SM at most (cooperative launch); barrier waits are bounded and a timeout sets
// *err like the tensor-core passes.  Every barrier has a counter of its own, clear when its first CTA arrives: a step
// clears the counters that its later barriers make free, and the launch of a cycle's first step (no basis vectors) clears all.
// Bound by reading the basis twice (HBM, or L2 where it fits) and, where it is small, by the latency of three
// barriers and of the FP64 tail (hence inv_sqrt and the warps that share a tile).  Measured per step over a solve with
// restarts of 100, between events: 24^3 x 48, 12 right-hand sides, 43 vectors on average: 68 us; before (multi-dot,
// multi-axpy, two reductions, Givens, scaling and image kernels, vectors interleaved by right-hand side) 126 us;
// 16^3 x 32, 21 vectors: 30 us, before 66; 16 x 8^3, one right-hand side, 12 vectors: 18 us, before 90.
// Shapes tried at 24^3 x 48: 4 CTAs of 256 threads per SM 107 us, one of 1024 with 4 vectors in flight 97 us
// (tiles bunched on some SMs, FP64 sums in the tail); now the fewest warps that cover the tiles, with the registers
// spent on vectors in flight.
#include <cuda_fp16.h>

#include "common.cuh"
#include "ddtm_internal.h"
#include "krylov_tc.h"
#include "solver.h"
#include "tc_ptx.cuh"
#include "timer.h"

namespace ddtm {

static const int GS_CHUNK = 64;  // basis vectors per pass through shared memory
static const uint64_t GS_WAIT_NS = 2000000000ull;

struct GsArgs {
  const char* V;
  size_t ldv;
  int nvec;
  float* w;
  char* vout;
  int per_g;      // items of one group of four right-hand sides: nsites * kg4
  int kg4;        // items of one site and group: 4 kpad / 8
  int ngj, R, gmod;    // groups, right-hand sides, CTAs mod groups
  int split;           // warps per tile
  int xb_off, turn_off;  // bytes before the shares of w and the Givens columns in shared memory
  int b_half, g_half;  // entries per site, per group of a site
  ArnoldiDev a;
  int first;
  double* est_host;
  float2* part;
  double2* h;
  double* npart;
  unsigned* bar;
  int* err;
};

// entry offset of item q of group g
__device__ __forceinline__ size_t item_off(const GsArgs& a, int g, int q) {
  const int s = q / a.kg4;
  return (size_t)s * a.b_half + (size_t)g * a.g_half + (q - s * a.kg4) * 16;
}
struct Item {
  float re[8], im[8];
};
__device__ __forceinline__ Item ld_item(const float* p) {
  const float4* q = reinterpret_cast<const float4*>(p);
  const float4 a = q[0], b = q[1], c = q[2], d = q[3];
  return Item{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}, {c.x, c.y, c.z, c.w, d.x, d.y, d.z, d.w}};
}
__device__ __forceinline__ void st_item(float* p, const Item& t) {
  float4* q = reinterpret_cast<float4*>(p);
  q[0] = make_float4(t.re[0], t.re[1], t.re[2], t.re[3]);
  q[1] = make_float4(t.re[4], t.re[5], t.re[6], t.re[7]);
  q[2] = make_float4(t.im[0], t.im[1], t.im[2], t.im[3]);
  q[3] = make_float4(t.im[4], t.im[5], t.im[6], t.im[7]);
}
struct HItem {
  uint4 re, im;
};
__device__ __forceinline__ HItem ld_hitem(const char* p) {
  const uint4* q = reinterpret_cast<const uint4*>(p);
  return HItem{__ldg(q), __ldg(q + 1)};
}
__device__ __forceinline__ void unpack8(const uint4& u, float v[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
    v[2 * k] = f.x;
    v[2 * k + 1] = f.y;
  }
}
__device__ __forceinline__ uint4 pack8(const float v[8], float s) {
  uint32_t w[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const __half2 h = __floats2half2_rn(s * v[2 * k], s * v[2 * k + 1]);
    w[k] = *reinterpret_cast<const uint32_t*>(&h);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
// sum over the eight lanes that work for the same right-hand side
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  v += __shfl_xor_sync(0xffffffffu, v, 16);
  return v;
}

// All CTAs of the grid arrive; false after a timeout (every CTA then returns).
__device__ __forceinline__ bool grid_barrier(unsigned* counter, int* err, int* ok_sh) {
  __syncthreads();
  if (gridDim.x == 1) return true;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(counter, 1u);
    const uint64_t t0 = ptx::globaltimer();
    int ok = 1;
    while (true) {
      unsigned v;
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
      if (v >= gridDim.x) break;
      if (ptx::globaltimer() - t0 > GS_WAIT_NS) {
        atomicExch(err, 1);
        ok = 0;
        break;
      }
    }
    __threadfence();
    *ok_sh = ok;
  }
  __syncthreads();
  return *ok_sh != 0;
}

// Column j = nvec - 1 of right-hand side r, by one warp: the new column turned by the previous rotations.
// s: shared scratch of 3 (j + 2) entries, the column first.
__device__ void givens_turn(const GsArgs& a, int r, cplx<float>* s, int lane) {
  const int j = a.nvec - 1, m = a.a.m, R = a.R;
  cplx<float>*col = s, *cs = s + j + 2, *sn = cs + j + 1;
  for (int i = lane; i <= j; i += 32) {
    const double2 v = __ldcg(a.h + (size_t)i * R + r);
    col[i] = cplx<float>((float)v.x, (float)v.y);
  }
  for (int i = lane; i < j; i += 32) {
    const double2 c = a.a.cs[(size_t)r * m + i], q = a.a.sn[(size_t)r * m + i];
    cs[i] = cplx<float>((float)c.x, (float)c.y);
    sn[i] = cplx<float>((float)q.x, (float)q.y);
  }
  __syncwarp();
  if (lane == 0) {
    cplx<float> x = col[0];
    for (int i = 0; i < j; i++) {
      const cplx<float> c = cs[i], q = sn[i], y = col[i + 1];
      col[i] = conj(c) * x + conj(q) * y;
      x = c * y - q * x;
    }
    col[j] = x;
  }
  __syncwarp();
  double2* H = a.a.H + (size_t)r * (m + 1) * m;
  for (int i = lane; i < j; i += 32) H[(size_t)i * m + j] = make_double2((double)col[i].re, (double)col[i].im);
}
// The new rotation, once the norm is known: one thread.  inv_n: 1 / norm (0 if it vanished)
__device__ void givens_close(const GsArgs& a, int r, double nr2, double inv_n, const cplx<float>* col) {
  const int j = a.nvec - 1, m = a.a.m;
  const double hn = nr2 * inv_n;
  const cplx<double> d((double)col[j].re, (double)col[j].im);
  const double rho2 = norm2(d) + nr2, inv = rho2 > 0 ? inv_sqrt(rho2) : rho2;
  const cplx<double> c = rho2 > 0 ? cplx<double>(d.re * inv, d.im * inv) : cplx<double>(1, 0);
  const double q = hn * inv;
  a.a.cs[(size_t)r * m + j] = make_double2(c.re, c.im);
  a.a.sn[(size_t)r * m + j] = make_double2(q, 0);
  double2* H = a.a.H + (size_t)r * (m + 1) * m;
  H[(size_t)j * m + j] = make_double2((double)(float)(rho2 * inv), 0);
  H[(size_t)(j + 1) * m + j] = make_double2(0, 0);
  double2* g = a.a.g + (size_t)r * (m + 1);
  const cplx<double> gj(g[j].x, g[j].y), gd = conj(c) * gj;
  g[j + 1] = make_double2(-q * gj.re, -q * gj.im);
  g[j] = make_double2(gd.re, gd.im);
  const double est = q * a.a.est[r];  // |g_{j+1}| = q |g_j|
  a.a.est[r] = est;
  a.est_host[r] = est;
}

__device__ __forceinline__ Item zero_item() {
  Item w;
#pragma unroll
  for (int k = 0; k < 8; k++) w.re[k] = w.im[k] = 0.f;
  return w;
}

// NT threads, U basis vectors in flight per lane.  S = a.split warps share a tile where there are few of them: each
// takes a share of the basis vectors.
template <int NT, int U>
__global__ void __launch_bounds__(NT, 1) k_gs_step(const GsArgs a) {
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int ok_sh;
  __shared__ double nsum[NW][4];
  __shared__ float scale_sh[kMaxBatch];
  __shared__ double nr_sh[kMaxBatch], inv_sh[kMaxBatch];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rr = lane & 3;
  const int G = gridDim.x, S = a.split, SL = NW / S, slot = warp / S, s_id = warp - slot * S;
  const int nvec = a.nvec, R = a.R, W = G * SL;
  // tile slots are numbered across the CTAs first, so that the tiles spread evenly over the SMs; slot wg works for
  // group g of four right-hand sides and takes every tstep-th tile of it
  const int wg = slot * G + blockIdx.x, g = wg % a.ngj, t0 = wg / a.ngj, tstep = (W - 1 - g) / a.ngj + 1;
  const int ntiles = (a.per_g + 31) / 32;
  const bool single = ntiles <= W / a.ngj;  // at most one tile per slot: w stays in registers
  // right-hand side whose Givens update this warp does (-1: none): warps from the last one down
  const int my_r = blockIdx.x + G * (NW - 1 - warp) < R ? (int)blockIdx.x + G * (NW - 1 - warp) : -1;
  const bool idle = t0 >= ntiles;  // no tile: the Givens column can be turned while the other warps update theirs
  float2* hs = reinterpret_cast<float2*>(smem_raw);  // [slot][GS_CHUNK][4], later [GS_CHUNK][4 ngj]
  float* xb = reinterpret_cast<float*>(smem_raw + a.xb_off) + (size_t)warp * 512 + lane;  // [warp][16][32]
  cplx<float>* turn = reinterpret_cast<cplx<float>*>(smem_raw + a.turn_off) + (size_t)(NW - 1 - warp) * 3 * (nvec + 1);
  Item w = zero_item();
  if (single && t0 < ntiles && 32 * t0 + lane < a.per_g) w = ld_item(a.w + item_off(a, g, 32 * t0 + lane));

  if (nvec > 0) {
    // ---- A: partial inner products
    for (int c0 = 0; c0 < nvec; c0 += GS_CHUNK) {
      const int cn = nvec - c0 < GS_CHUNK ? nvec - c0 : GS_CHUNK;
      const int sub = (cn + S - 1) / S, ib = s_id * sub, ie = ib + sub < cn ? ib + sub : cn;
      float2* hw = hs + (size_t)slot * GS_CHUNK * 4;
      for (int i = 4 * ib + lane; i < 4 * ie; i += 32) hw[i] = make_float2(0.f, 0.f);
      __syncwarp();
      for (int t = t0; t < ntiles; t += tstep) {
        const int q = 32 * t + lane;
        const bool in = q < a.per_g;
        const size_t off = item_off(a, g, in ? q : 0);
        if (!single) w = in ? ld_item(a.w + off) : zero_item();
        const char* v0 = a.V + 2 * off + (size_t)c0 * a.ldv;
        for (int i0 = ib; i0 < ie; i0 += U) {
          HItem hv[U];
#pragma unroll
          for (int u = 0; u < U; u++) hv[u] = ld_hitem(v0 + (size_t)(i0 + u < ie ? i0 + u : ie - 1) * a.ldv);
#pragma unroll
          for (int u = 0; u < U; u++) {
            float vr[8], vi[8], sr = 0.f, si = 0.f;
            unpack8(hv[u].re, vr);
            unpack8(hv[u].im, vi);
#pragma unroll
            for (int k = 0; k < 8; k++) {
              sr += vr[k] * w.re[k] + vi[k] * w.im[k];
              si += vr[k] * w.im[k] - vi[k] * w.re[k];
            }
            sr = quad_sum(sr);
            si = quad_sum(si);
            if (lane < 4 && i0 + u < ie) {
              float2* p = hw + (i0 + u) * 4 + lane;
              p->x += sr;
              p->y += si;
            }
          }
        }
      }
      __syncthreads();
      for (int v = threadIdx.x; v < cn * R; v += NT) {
        const int i = v / R, r = v - i * R, gr = r >> 2;
        float sr = 0.f, si = 0.f;
        // the slots of group gr: (k G + CTA) % ngj == gr
        for (int k = 0, m = blockIdx.x % a.ngj; k < SL; k++) {
          if (m == gr) {
            const float2 p = hs[((size_t)k * GS_CHUNK + i) * 4 + (r & 3)];
            sr += p.x;
            si += p.y;
          }
          m += a.gmod;
          if (m >= a.ngj) m -= a.ngj;
        }
        __stcg(a.part + (size_t)(c0 * R + v) * G + blockIdx.x, make_float2(sr, si));
      }
      __syncthreads();
    }
    if (!grid_barrier(a.bar, a.err, &ok_sh)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.bar[2] = 0;  // of the previous step, which has ended
    for (int v = warp * G + blockIdx.x; v < nvec * R; v += G * NW) {
      double sr = 0, si = 0;
      for (int c = lane; c < G; c += 32) {
        const float2 p = __ldcg(a.part + (size_t)v * G + c);
        sr += p.x;
        si += p.y;
      }
      if (G > 1) {
        sr = warp_sum(sr);
        si = warp_sum(si);
      }
      if (lane == 0) __stcg(a.h + v, make_double2(sr, si));
    }
    if (!grid_barrier(a.bar + 1, a.err, &ok_sh)) return;
  }
  // ---- B: w -= sum_i h_i V_i, last vectors first (they are the likeliest to be in L2 still)
  if (s_id) w = zero_item();
  for (int c0 = (nvec - 1) / GS_CHUNK * GS_CHUNK; nvec > 0 && c0 >= 0; c0 -= GS_CHUNK) {
    const int cn = nvec - c0 < GS_CHUNK ? nvec - c0 : GS_CHUNK;
    const int sub = (cn + S - 1) / S, ib = s_id * sub, ie = ib + sub < cn ? ib + sub : cn;
    for (int v = threadIdx.x; v < cn * 4 * a.ngj; v += NT) {
      const int i = v / (4 * a.ngj), r = v - i * 4 * a.ngj;  // columns beyond R are padding
      const double2 p = r < R ? __ldcg(a.h + (size_t)(c0 + i) * R + r) : make_double2(0, 0);
      hs[v] = make_float2((float)p.x, (float)p.y);
    }
    __syncthreads();
    if (idle && my_r >= 0 && c0 + GS_CHUNK >= nvec) givens_turn(a, my_r, turn, lane);
    for (int t = t0; t < ntiles; t += tstep) {
      const int q = 32 * t + lane;
      if (q >= a.per_g) continue;
      const size_t off = item_off(a, g, q);
      if (!single) w = ld_item(a.w + off);
      const char* v0 = a.V + 2 * off + (size_t)c0 * a.ldv;
      const float2* hc = hs + 4 * g + rr;
      for (int i0 = ie - 1; i0 >= ib; i0 -= U) {
        HItem hv[U];
#pragma unroll
        for (int u = 0; u < U; u++) hv[u] = ld_hitem(v0 + (size_t)(i0 - u >= ib ? i0 - u : ib) * a.ldv);
#pragma unroll
        for (int u = 0; u < U; u++) {
          if (i0 - u < ib) break;
          const float2 h = hc[(size_t)(i0 - u) * 4 * a.ngj];
          float vr[8], vi[8];
          unpack8(hv[u].re, vr);
          unpack8(hv[u].im, vi);
#pragma unroll
          for (int k = 0; k < 8; k++) {
            w.re[k] -= h.x * vr[k] - h.y * vi[k];
            w.im[k] -= h.x * vi[k] + h.y * vr[k];
          }
        }
      }
      if (!single) st_item(a.w + off, w);
    }
    if (c0 || S > 1) __syncthreads();
  }
  if (S > 1) {  // the shares of a tile; from here on its first warp goes on alone
    if (s_id)
#pragma unroll
      for (int k = 0; k < 8; k++) {
        xb[64 * k] = w.re[k];
        xb[64 * k + 32] = w.im[k];
      }
    __syncthreads();
    if (s_id == 0)
      for (int s2 = 1; s2 < S; s2++)
#pragma unroll
        for (int k = 0; k < 8; k++) {
          w.re[k] += xb[512 * s2 + 64 * k];
          w.im[k] += xb[512 * s2 + 64 * k + 32];
        }
  }
  double nn = 0;
  if (s_id == 0)
    for (int t = t0; t < ntiles; t += tstep) {
      const int q = 32 * t + lane;
      if (!single) w = q < a.per_g ? ld_item(a.w + item_off(a, g, q)) : zero_item();
      float s = 0.f;
#pragma unroll
      for (int k = 0; k < 8; k++) s += w.re[k] * w.re[k] + w.im[k] * w.im[k];
      nn += (double)quad_sum(s);  // w is zero beyond the last item
    }
  if (lane < 4 && s_id == 0) nsum[slot][lane] = nn;
  __syncthreads();
  for (int r = warp; r < R; r += NW) {
    double s = lane < SL && (lane * G + (int)blockIdx.x) % a.ngj == (r >> 2) ? nsum[lane][r & 3] : 0.0;
    s = warp_sum(s);
    if (lane == 0) __stcg(a.npart + (size_t)r * G + blockIdx.x, s);
  }
  if (nvec > 0 && my_r >= 0 && !idle) givens_turn(a, my_r, turn, lane);  // while the other CTAs arrive
  if (!grid_barrier(a.bar + 2, a.err, &ok_sh)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) a.bar[0] = a.bar[1] = 0;  // every CTA has passed them
  // ---- C: norms, the next basis vector, the Givens update
  for (int r = warp; r < R; r += NW) {
    double s = 0;
    for (int c = lane; c < G; c += 32) s += __ldcg(a.npart + (size_t)r * G + c);
    if (G > 1) s = warp_sum(s);
    if (lane == 0) {
      const double inv = s > 0 ? inv_sqrt(s) : s;
      nr_sh[r] = s;
      inv_sh[r] = inv;
      scale_sh[r] = (float)inv;
    }
  }
  __syncthreads();
  if (a.vout && s_id == 0) {
    const float sc = 4 * g + rr < R ? scale_sh[4 * g + rr] : 0.f;
    for (int t = t0; t < ntiles; t += tstep) {
      const int q = 32 * t + lane;
      if (q >= a.per_g) continue;
      const size_t off = item_off(a, g, q);
      if (!single) w = ld_item(a.w + off);
      uint4* o = reinterpret_cast<uint4*>(a.vout + 2 * off);
      o[0] = pack8(w.re, sc);
      o[1] = pack8(w.im, sc);
    }
  }
  if (my_r >= 0) {
    if (nvec == 0) {  // start of a cycle
      const double beta = nr_sh[my_r] * inv_sh[my_r];
      for (int i = lane; i <= a.a.m; i += 32) a.a.g[(size_t)my_r * (a.a.m + 1) + i] = make_double2(i == 0 ? beta : 0.0, 0);
      if (lane == 0) {
        if (a.first) a.a.bn[my_r] = beta;
        const double bn = a.first ? beta : a.a.bn[my_r], est = bn > 0 ? beta / bn : (bn == 0 ? 0.0 : bn);
        a.a.est[my_r] = est;
        a.est_host[my_r] = est;
      }
    } else if (lane == 0) {
      givens_close(a, my_r, nr_sh[my_r], inv_sh[my_r], turn);
    }
  }
}

// Launch shape: CTAs (one per SM at most), threads, warps per tile.
struct GsShape {
  int ctas, nt, split;
};
static GsShape gs_shape(const ImgVec& v, int sms) {
  const long tiles = (long)v.t.ngj * (((long)v.nsites * 4 * (v.t.kpad / 8) + 31) / 32);
  GsShape p;
  // few tiles: one CTA without grid barriers; else every SM, with as many warps as tiles call for (more registers
  // per thread hold more loads in flight), and idle warps sharing tiles
  const long least = (v.t.R > v.t.ngj ? v.t.R : v.t.ngj);  // a warp per Givens update, a slot per group
  long n = tiles <= 16 ? 1 : (tiles + 1) / 2;
  if (n * 16 < least) n = (least + 15) / 16;
  p.ctas = (int)(n < sms ? n : sms);
  const long per = (tiles + p.ctas - 1) / p.ctas;
  p.nt = per <= 16 ? 512 : per <= 24 ? 768 : 1024;
  p.split = 1;
  while (p.split < 8 && per * p.split * 2 <= p.nt / 32 && (long)p.ctas * (p.nt / 32) / (p.split * 2) >= v.t.ngj) p.split *= 2;
  return p;
}
static size_t gs_xb_off(const ImgVec& v, int nvec, const GsShape& p) {
  const size_t n = nvec < GS_CHUNK ? nvec : GS_CHUNK;
  const size_t s = nvec > 0 ? (size_t)(p.nt / 32 / p.split) * GS_CHUNK * 4 * sizeof(float2) : 0, c = n * 4 * v.t.ngj * sizeof(float2);
  return ((c > s ? c : s) + 15) / 16 * 16;
}
static size_t gs_turn_off(const ImgVec& v, int nvec, const GsShape& p) {
  return gs_xb_off(v, nvec, p) + (p.split > 1 ? (size_t)(p.nt / 32) * 512 * sizeof(float) : 0);
}
static size_t gs_smem(const ImgVec& v, int nvec, const GsShape& p) {
  return gs_turn_off(v, nvec, p) + (size_t)((v.t.R + p.ctas - 1) / p.ctas) * 3 * (nvec + 1) * sizeof(cplx<float>) + 16;
}
static const void* gs_kernel(int nt) {
  return nt == 512 ? (const void*)k_gs_step<512, 8> : nt == 768 ? (const void*)k_gs_step<768, 5> : (const void*)k_gs_step<1024, 4>;
}

int gs_ctas(const ImgVec& v, int m) {
  int dev = 0, sms = 0, smem_blk = 0, coop = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  CK(cudaDeviceGetAttribute(&smem_blk, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  const GsShape p = gs_shape(v, sms);
  const void* k = gs_kernel(p.nt);
  cudaFuncAttributes fa;
  CK(cudaFuncGetAttributes(&fa, k));
  const size_t smem = gs_smem(v, m, p);
  if (!coop || (long)p.ctas * (p.nt / 32) < v.t.R || smem + fa.sharedSizeBytes > (size_t)smem_blk) return 0;
  set_dynamic_smem(k, smem);
  int per = 0;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, p.nt, smem));
  return per < 1 ? 0 : p.ctas;
}

void launch_gs_step(const ImgVec& v, const void* V, size_t ldv, int nvec, float* w, void* vout, const ArnoldiDev& a,
                    int first, double* est_host, const GsBuffers& b, cudaStream_t st) {
  ScopedTimer timer_("gs_step", st, nvec, (double)v.entries() * (2.0 * 2 * nvec + 2 * 4 + (vout ? 2 : 0)));
  int dev = 0, sms = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const GsShape p = gs_shape(v, sms);
  GsArgs g;
  g.V = (const char*)V;
  g.ldv = ldv;
  g.nvec = nvec;
  g.w = w;
  g.vout = (char*)vout;
  g.kg4 = 4 * (v.t.kpad / 8);
  g.per_g = v.nsites * g.kg4;
  g.ngj = v.t.ngj;
  g.gmod = p.ctas % v.t.ngj;
  g.R = v.t.R;
  g.b_half = v.t.b_bytes / 2;
  g.g_half = v.t.sbo / 2;
  g.split = p.split;
  g.a = a;
  g.first = first;
  g.est_host = est_host;
  g.part = b.part;
  g.h = b.h;
  g.npart = b.npart;
  g.bar = b.bar;
  g.err = b.err;
  g.xb_off = (int)gs_xb_off(v, nvec, p);
  g.turn_off = (int)gs_turn_off(v, nvec, p);
  // The last step of a cycle leaves the counter of its norm barrier at the number of CTAs; steps with basis vectors clear it
  // themselves behind their first barrier, a step without any has no barrier before that one.  (Also after a timeout.)
  if (nvec == 0) CK(cudaMemsetAsync(b.bar, 0, 3 * sizeof(unsigned), st));
  void* args[] = {(void*)&g};
  CK(cudaLaunchCooperativeKernel(gs_kernel(p.nt), dim3(p.ctas), dim3(p.nt), args, gs_smem(v, nvec, p), st));
  CKL("gs_step");
}

// ---- the rest, elementwise ------------------------------------------------------------
__global__ void __launch_bounds__(256) k_img_combine(float* __restrict__ x, const char* __restrict__ V, size_t ldv, int nvec,
                                                     const double2* __restrict__ y, int R, int ngj, int kg4, int b_half,
                                                     int g_half, size_t items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* yc = reinterpret_cast<float2*>(smem_raw);  // [nvec][R]
  for (int k = threadIdx.x; k < nvec * R; k += blockDim.x) yc[k] = make_float2((float)y[k].x, (float)y[k].y);
  __syncthreads();
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < items; k += (size_t)gridDim.x * blockDim.x) {
    const int per = ngj * kg4, rem = (int)(k % per), g = rem / kg4, q = rem - g * kg4, r = 4 * g + (q & 3);
    if (r >= R) continue;
    const size_t off = (k / per) * b_half + (size_t)g * g_half + q * 16;
    Item w = ld_item(x + off);
#pragma unroll 2
    for (int i = 0; i < nvec; i++) {
      const HItem h = ld_hitem(V + (size_t)i * ldv + 2 * off);
      const float2 c = yc[i * R + r];
      float vr[8], vi[8];
      unpack8(h.re, vr);
      unpack8(h.im, vi);
#pragma unroll
      for (int e = 0; e < 8; e++) {
        w.re[e] += c.x * vr[e] - c.y * vi[e];
        w.im[e] += c.x * vi[e] + c.y * vr[e];
      }
    }
    st_item(x + off, w);
  }
}

__global__ void k_img_order(float* __restrict__ img, float2* __restrict__ v, int R, int n, int ngj, int kg4, int b_half,
                            int g_half, size_t items, int dir) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= items) return;
  const int per = ngj * kg4, rem = (int)(k % per), g = rem / kg4, q = rem - g * kg4, r = 4 * g + (q & 3), k0 = 8 * (q >> 2);
  const size_t s = k / per, off = s * b_half + (size_t)g * g_half + q * 16;
  if (dir == 0) {
    Item t;
#pragma unroll
    for (int e = 0; e < 8; e++) {
      const float2 z = r < R && k0 + e < n ? v[(s * n + k0 + e) * R + r] : make_float2(0.f, 0.f);
      t.re[e] = z.x;
      t.im[e] = z.y;
    }
    st_item(img + off, t);
  } else if (r < R) {
    const Item t = ld_item(img + off);
#pragma unroll
    for (int e = 0; e < 8; e++)
      if (k0 + e < n) v[(s * n + k0 + e) * R + r] = make_float2(t.re[e], t.im[e]);
  }
}

// canonical FP64 vectors <-> image order: one thread per complex entry of a site's vector, blockIdx.y takes every
// gridDim.y-th right-hand side; canonical memory in order, runs of 8 entries in image order
__device__ __forceinline__ size_t img_entry(int r, int q, int n, int b_half, int g_half) {
  const int s = q / n, k = q - s * n;
  return (size_t)s * b_half + (size_t)(r >> 2) * g_half + (k >> 3) * 64 + (r & 3) * 16 + (k & 7);
}
template <bool A16>
__global__ void k_img_from_canon(__half* __restrict__ image, float* __restrict__ img, const double* __restrict__ x, int nc, int n,
                                 int b_half, int g_half, int R) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nc) return;
  for (int r = blockIdx.y; r < R; r += gridDim.y) {
    const double2 z = ld_canon<A16>(x, (size_t)r * nc + q);
    const float re = (float)z.x, im = (float)z.y;
    const size_t o = img_entry(r, q, n, b_half, g_half);
    img[o] = re;
    img[o + 8] = im;
    image[o] = __float2half_rn(re);
    image[o + 8] = __float2half_rn(im);
  }
}
template <bool A16>
__global__ void k_img_to_canon(double* __restrict__ y, const float* __restrict__ img, int nc, int n, int b_half, int g_half, int R) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nc) return;
  for (int r = blockIdx.y; r < R; r += gridDim.y) {
    const size_t o = img_entry(r, q, n, b_half, g_half);
    st_canon<A16>(y, (size_t)r * nc + q, (double)img[o], (double)img[o + 8]);
  }
}

__global__ void k_img_half(uint4* __restrict__ out, const float4* __restrict__ in, size_t n8) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n8) return;
  const float4 a = in[2 * k], b = in[2 * k + 1];
  const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  out[k] = pack8(v, 1.f);
}

__global__ void k_img_residual(float4* __restrict__ w, const float4* __restrict__ b, size_t n4) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n4) return;
  const float4 x = b[k], y = w[k];
  w[k] = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
}

void launch_img_combine(const ImgVec& v, float* x, const void* V, size_t ldv, int nvec, const double2* y, cudaStream_t st) {
  ScopedTimer timer_("img_combine", st, nvec, (double)v.entries() * (2.0 * nvec + 8));
  if (nvec <= 0) return;
  const int kg4 = 4 * (v.t.kpad / 8);
  const size_t items = (size_t)v.nsites * v.t.ngj * kg4, smem = (size_t)nvec * v.t.R * sizeof(float2);
  if (smem > 200 * 1024) throw Error(DDTM_ERR_ARG, "internal: coefficient block too large");
  set_dynamic_smem((const void*)k_img_combine, smem);
  size_t grid = (items + 255) / 256;
  if (grid > 4096) grid = 4096;
  k_img_combine<<<(unsigned)grid, 256, smem, st>>>(x, (const char*)V, ldv, nvec, y, v.t.R, v.t.ngj, kg4, v.t.b_bytes / 2,
                                                   v.t.sbo / 2, items);
  CKL("img_combine");
}
void launch_img_order(const ImgVec& v, float* img, cplx<float>* inter, int dir, cudaStream_t st) {
  ScopedTimer timer_("img_order", st, v.t.R);
  const int kg4 = 4 * (v.t.kpad / 8);
  const size_t items = (size_t)v.nsites * v.t.ngj * kg4;
  k_img_order<<<(unsigned)((items + 127) / 128), 128, 0, st>>>(img, reinterpret_cast<float2*>(inter), v.t.R, v.t.n, v.t.ngj,
                                                               kg4, v.t.b_bytes / 2, v.t.sbo / 2, items, dir);
  CKL("img_order");
}
void launch_img_from_canon(const ImgVec& v, void* image, float* img, const double* x, cudaStream_t st) {
  ScopedTimer timer_("img_order", st, v.t.R);
  const int nc = v.nsites * v.t.n;
  if (v.t.n != v.t.kpad || v.t.R % 4) {  // padding entries
    CK(cudaMemsetAsync(image, 0, v.entries() * sizeof(__half), st));
    CK(cudaMemsetAsync(img, 0, v.entries() * sizeof(float), st));
  }
  auto kernel = canon_a16(x) ? k_img_from_canon<true> : k_img_from_canon<false>;
  kernel<<<dim3((nc + 255) / 256, v.t.R < 65535 ? v.t.R : 65535), 256, 0, st>>>((__half*)image, img, x, nc, v.t.n,
                                                                              v.t.b_bytes / 2, v.t.sbo / 2, v.t.R);
  CKL("img_from_canon");
}
void launch_img_to_canon(const ImgVec& v, double* y, const float* img, cudaStream_t st) {
  ScopedTimer timer_("img_order", st, v.t.R);
  const int nc = v.nsites * v.t.n;
  auto kernel = canon_a16(y) ? k_img_to_canon<true> : k_img_to_canon<false>;
  kernel<<<dim3((nc + 255) / 256, v.t.R < 65535 ? v.t.R : 65535), 256, 0, st>>>(y, img, nc, v.t.n, v.t.b_bytes / 2,
                                                                              v.t.sbo / 2, v.t.R);
  CKL("img_to_canon");
}
void launch_img_half(const ImgVec& v, void* out, const float* in, cudaStream_t st) {
  const size_t n8 = v.entries() / 8;
  k_img_half<<<(unsigned)((n8 + 255) / 256), 256, 0, st>>>((uint4*)out, (const float4*)in, n8);
  CKL("img_half");
}
void launch_img_residual(const ImgVec& v, float* w, const float* b, cudaStream_t st) {
  const size_t n4 = v.entries() / 4;
  k_img_residual<<<(unsigned)((n4 + 255) / 256), 256, 0, st>>>((float4*)w, (const float4*)b, n4);
  CKL("img_residual");
}

}  // namespace ddtm
