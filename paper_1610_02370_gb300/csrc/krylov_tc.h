// Host interface of the coarsest-level Arnoldi kernels on image-ordered vectors (krylov_tc.cu).
#pragma once

#include "blas.h"
#include "coarse.h"

namespace ddtm {

// Image order: the order of the FP16 vector images of the tensor-core stencil (coarse_tc.cu).  A vector
// batch of R right-hand sides (R = 1 or a multiple of 4) on nsites sites takes b_bytes per site in FP16 and twice
// that in FP32; 16 consecutive entries hold the real and then the imaginary parts of 8 dofs of one right-hand
// side.  Padding entries are zero.
struct ImgVec {
  TcGeom t;
  int nsites;
  size_t entries() const { return (size_t)nsites * (t.b_bytes / 2); }
};

// Work buffers of the Arnoldi step: partial sums over the launch's CTAs, the coefficients h[i * R + r], grid
// barrier counters (cleared by the launch of a step without basis vectors) and the timeout flag.
struct GsBuffers {
  float2* part;
  double2* h;
  double* npart;
  unsigned* bar;
  int* err;
};
// CTAs of every step of a solve with up to m basis vectors (all resident at once); 0 where the step does not
// apply (its shared memory would not fit)
int gs_ctas(const ImgVec& v, int m);

// One Arnoldi step: w orthogonalised against the nvec basis vectors V (FP16 images, ldv bytes apart; classical
// Gram-Schmidt), its norm, the Givens update of column nvec - 1, the residual estimates (also to est_host,
// pinned) and, if vout, the normalised vector as the next image.  nvec = 0 starts a cycle: g_0 = ||w||,
// and with first also bn = ||w||.
void launch_gs_step(const ImgVec& v, const void* V, size_t ldv, int nvec, float* w, void* vout, const ArnoldiDev& a,
                    int first, double* est_host, const GsBuffers& b, cudaStream_t st);
// x += sum_i y[i * R + r] V_i
void launch_img_combine(const ImgVec& v, float* x, const void* V, size_t ldv, int nvec, const double2* y, cudaStream_t st);
// interleaved FP32 batch (element (e, r) at e R + r) <-> image-ordered FP32 (dir 0: in, 1: out)
void launch_img_order(const ImgVec& v, float* img, cplx<float>* inter, int dir, cudaStream_t st);
// R canonical FP64 vectors (x[r][site n + k]) -> FP16 image and image-ordered FP32 batch
void launch_img_from_canon(const ImgVec& v, void* image, float* img, const double* x, cudaStream_t st);
// image-ordered FP32 batch -> canonical FP64 vectors
void launch_img_to_canon(const ImgVec& v, double* y, const float* img, cudaStream_t st);
// FP16 image of an image-ordered FP32 batch
void launch_img_half(const ImgVec& v, void* out, const float* in, cudaStream_t st);
// w = b - w
void launch_img_residual(const ImgVec& v, float* w, const float* b, cudaStream_t st);

}  // namespace ddtm
