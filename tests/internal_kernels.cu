// Entry points for tests of launchers that the C ABI reaches only inside a solve; compiled by the test against csrc/ and
// linked with libddtm.so.  Pointers are device memory, work goes to the default stream; the return value is 0 or a
// DDTM_ERR_* code.
#include "coarse.h"
#include "common.cuh"
#include "ddtm_internal.h"
#include "krylov_tc.h"

using namespace ddtm;

template <typename F>
static int run(F f) {
  try {
    f();
    CK(cudaDeviceSynchronize());
  } catch (const Error& e) {
    return e.code;
  }
  return 0;
}
static void set_geom(FineGeom& g, int Vb, int Nb) {
  g.Vb = Vb;
  g.Nb = Nb;
  g.V = (long)Vb * Nb;
}

__global__ void k_inv_sqrt(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = inv_sqrt(x[i]);
}

extern "C" {
int ik_inv_sqrt(const double* x, double* y, int n) {
  return run([&] {
    k_inv_sqrt<<<(n + 127) / 128, 128>>>(x, y, n);
    CKL("inv_sqrt");
  });
}
// x += sum_i y[i R + r] V_i on image-ordered vectors of R right-hand sides, n dofs and nsites sites
int ik_img_combine(float* x, const void* V, int nvec, const double* y, int n, int R, int nsites) {
  return run([&] {
    const ImgVec v{tc_geom(n, R), nsites};
    launch_img_combine(v, x, V, v.entries() * sizeof(__half), nvec, (const double2*)y, 0);
  });
}
// FP16 fields (complex half [r][block][12][Vb], one scale per site) and FP16 P ([block][2][nv][6][Vb]); the coarse side is
// complex FP32, column r of Rs
int ik_restrict(int Vb, int Nb, void* c, const void* psi, const float* pn, const void* P, int nv, int R, int Rs) {
  return run([&] {
    FineGeom g;
    set_geom(g, Vb, Nb);
    launch_restrict(g, PREC_F16, (cplx<float>*)c, psi, pn, P, PREC_F16, nv, R, Rs, 0);
  });
}
int ik_prolong(int Vb, int Nb, void* x, float* xn, const void* e, const void* P, int nv, int R, int Rs, int add) {
  return run([&] {
    FineGeom g;
    set_geom(g, Vb, Nb);
    launch_prolong(g, PREC_F16, x, xn, (const cplx<float>*)e, P, PREC_F16, nv, R, Rs, add, 0);
  });
}
// the FP32 blocks of D_c: [site][9][column][row]
int ik_coarse_blocks(ddtm_ctx* c, void* out) {
  return run([&] {
    CK(cudaMemcpy(out, c->c1.Dc.p, (size_t)c->c1.Nc * 9 * c->c1.n * c->c1.n * sizeof(float2), cudaMemcpyDeviceToDevice));
  });
}
}
