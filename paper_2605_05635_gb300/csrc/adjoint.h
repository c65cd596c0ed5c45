// adjoint.h -- data shared by the adjoint kernels (adjoint.cu) and the host
// orchestration of bh_trace_backward (api.cu).
#pragma once
#include <cuda_runtime.h>

#include "internal.h"

namespace bhrt {

constexpr int kCkptEvery = 64;
constexpr int kMaxCrossAdj = 32;
// device status of a ray that ran out of checkpoints or chunks (no bh_status)
constexpr int kAdjNoRoom = -1;

// Derivatives of per-image constants with respect to (chi, theta_o, halo1,
// halo2), computed on the host.
struct AdjImg {
  double d_sqgrr[4], d_sqgth[4], d_sqgph[4], d_N[4], d_w[4], d_Rin[4];
};

struct Ckpt {
  double y[6], f[6];
  double h, lam, lam_last;
  int32_t nacc, nrej, steps, ncross;
  int32_t rejected, have_trusted, pad0, pad1;
};

struct AdjArgs {
  const WsHeader* hdr;
  const ImgParams* ip;   // [1]
  AdjImg aj;
  int levels;
  int64_t npix;
  const double* Gpix;    // [npix] dL/dI per pixel
  const int32_t* base_child;
  LevelRecs lv[kMaxLevels + 1];
  Ckpt* ckpt;            // [threads][max_ckpt]
  int max_ckpt;
  double* grad;          // [10]
  unsigned long long* head;
  int* status;
};

// A crossing of a replayed ray: its accepted step, abscissa and the weight
// dL/dI dI/dR_em.
struct XRec {
  int32_t step;
  double sig;
  double Rbar;
};

// adjoint_warp.cu: a replayed ray (its trajectory's newest chunk, last accepted
// step and crossings, the direct adjoint of the crossing terms), the counters
// of one forward / reverse pair of launches, and its arguments.
constexpr int kAdjChunk = 64;  // steps per trajectory chunk
struct AdjRay {
  int32_t nx, chunk, last, pad;
  double X, Y, E, ell;
  double pdir[13];
  XRec x[kMaxCrossAdj];
};
struct AdjCtl {
  unsigned long long reserved, used;  // chunks
  unsigned long long claimed, rays, swept;
  int32_t done, pad;                  // every cell has been claimed
};
struct AdjWarpArgs {
  const WsHeader* hdr;
  const ImgParams* ip;   // [1]
  AdjImg aj;
  int levels;
  int64_t npix;
  const double* Gpix;    // [npix] dL/dI per pixel
  const int32_t* base_child;
  LevelRecs lv[kMaxLevels + 1];
  double* pool;          // [chunks][5][kAdjChunk]: R, theta, p_R, p_theta, h per step
  int32_t* prev;         // [chunks] the ray's chunk before
  int64_t chunks;
  int per_ray;           // chunks the longest ray may take
  AdjRay* ray;           // [max_rays]
  int64_t max_rays;
  AdjCtl* ctl;
  double* grad;          // [10]
  unsigned long long* head;
  int* status;
};

struct ImgAdj {
  int nx, ny;
  double x_min, y_min, dx, dy;
  const float* dLdI;    // optional
  double S, Xc, Yc, C;  // pixel sum of I, centroid
  double FRs, FLs;      // right / left pixel sums
  double cC, cA;        // dL/dC, dL/dA_LR
  int bstar, nbins;     // radial profile argmax and bins
  double drho[3];       // d rho_peak / d(mean of bins bstar-1, bstar, bstar+1)
  int cnt[3];
  double cR;            // dL/d rho_peak
  double uv[16];        // 8 baselines
  double Vre[8], Vim[8], Vabs[8], V0, cV[8];
  double* G;            // [npix] out
};


cudaError_t launch_adjoint(const AdjArgs& a, int blocks, int threads, cudaStream_t s);
cudaError_t launch_adj_forward(const AdjWarpArgs& a, int blocks, int threads, cudaStream_t s);
cudaError_t launch_adj_reverse(const AdjWarpArgs& a, cudaStream_t s);
cudaError_t launch_pixel_adjoint(const ImgAdj& a, cudaStream_t s);
cudaError_t launch_image_moments(const float* I, const ImgAdj& a, double* out3, cudaStream_t s);
cudaError_t launch_image_profile(const float* I, const ImgAdj& a, double* lr, double* hs,
                                 unsigned long long* hc, cudaStream_t s);

}  // namespace bhrt
