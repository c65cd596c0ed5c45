// adjoint_warp.cu -- the ray adjoint of Kerr and Einasto images with the reverse
// sweep spread over a warp (the method of adjoint.cu: the derivative of the
// forward rays as executed, adaptive decisions frozen).
//
// adjoint.cu gives a ray to a thread: a small image keeps a few warps busy for
// as long as its longest ray, every reverse sweep replays its steps first, and
// its stage Jacobians are dual numbers through the right-hand side, about four
// times the FP64 operations of the closed form used here.  Cored-NFW images
// stay there: that kernel replays them with step sizes that differ in the last
// bits from its forward pass (the compiler fuses the lapse's products
// differently in its two copies of the step), which shows as 1e-8 relative in
// their gradients; a consistent replay would change results.
//
// Measured (GB300, chi = 0.7, 50 deg, one refinement level, image and diagnostics
// loss; adjoint.cu before): Kerr 12^2 361 -> 32 ms, 48^2 506 -> 52 ms, 128^2 694
// -> 165 ms, 256^2 1,241 -> 295 ms; Einasto 428 -> 37, 518 -> 60, 777 -> 233,
// 1,432 -> 353 ms.  What is left is the
// forward replay, one FP64 instruction in 64 cycles per warp at these sizes (33
// ms of a 48^2 gradient; the reverse sweep takes 4 to 16 ms).
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "adjoint.h"
#include "adjoint_event.cuh"
#include "integrator.cuh"

namespace bhrt {

// One attempted FP64 step of the forward replay: ray_step64 with the crossing's
// abscissa reported instead of its intensity.  Returns 0 (continue) or status +
// 1.
__device__ __forceinline__ int adj_step_rolled(const ImgParams& ip, const MetricConsts<double>& m,
                                               Ray64& r, bool& crossed, double& sig_out,
                                               double& Rc_out, bool& reflected) {
  crossed = false;
  reflected = false;
  const double h = r.h;
  double k[6], q[6][4], s5[6], se[6], sd[3];  // sd: R, theta, p_theta
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    k[i] = r.f[i];
    s5[i] = se[i] = 0.0;
  }
  sd[0] = sd[1] = sd[2] = 0.0;
#pragma unroll
  for (int u = 0; u < 6; ++u)
#pragma unroll
    for (int x = 0; x < 4; ++x) q[u][x] = 0.0;
  bool bad = false;
  double W, P2;
  const RayC<double> kc = ray_consts(m, r.E, r.ell);
#pragma unroll 1
  for (int j = 0; j < 7; ++j) {
    if ((kDPr.bmask >> j) & 1) {
      const double bj = kDPr.b[j];
#pragma unroll
      for (int i = 0; i < 6; ++i) s5[i] = fma(bj, k[i], s5[i]);
    }
    if ((kDPr.emask >> j) & 1) {
      const double ej = kDPr.e[j];
#pragma unroll
      for (int i = 0; i < 6; ++i) se[i] = fma(ej, k[i], se[i]);
    }
    if ((kDPr.dmask >> j) & 1) {
      const double dj = kDPr.d[j];
      sd[0] = fma(dj, k[1], sd[0]);
      sd[1] = fma(dj, k[2], sd[1]);
      sd[2] = fma(dj, k[5], sd[2]);
    }
    if (j == 6) break;
    const int qm = kDPr.qmask[j];
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      if ((qm >> u) & 1) {
        const double c = kDPr.q[j][u];
#pragma unroll
        for (int x = 0; x < 4; ++x) q[u][x] = fma(c, k[kQC(x)], q[u][x]);
      }
    }
    double ys[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) ys[x] = r.y[kQC(x)] + h * q[0][x];
    double sth, cth;
    d_sincos(ys[1], &sth, &cth);
    bad |= !geo_rhs_sc(m, kc, ys[0], sth, cth, ys[2], ys[3], k, W, P2);
#pragma unroll
    for (int u = 0; u < 5; ++u) {
#pragma unroll
      for (int x = 0; x < 4; ++x) q[u][x] = q[u + 1][x];
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) q[5][x] = 0.0;
  }
  double y1[6];
  float err2 = 0.f;
  const float fatol = f32_trunc(ip.atol), frtol = f32_trunc(ip.rtol);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    y1[i] = r.y[i] + h * s5[i];
    err2 += err_term(r.y[i], y1[i], h * se[i], fatol, frtol);
  }
  const float err = sqrtf(err2 / 6.f);
  r.steps++;
  if (bad || !(err <= 1.f)) {
    r.h = bad ? 0.5 * h : h * f64_of_f32(step_factor(err, true));
    r.rejected = true;
    r.nrej++;
    return r.steps >= ip.max_steps ? 3 : 0;
  }
  r.nacc++;
  const double s0 = r.y[2] - kHalfPi, s1 = y1[2] - kHalfPi;
  if ((s0 > 0.0 && s1 <= 0.0) || (s0 < 0.0 && s1 >= 0.0)) {
    const double hd1 = h * sd[0], hd2 = h * sd[1], hd5 = h * sd[2];
    double sig = 1.0;
    if (s1 != 0.0) {
      double x0 = 0.0, f0 = s0, x1 = 1.0, f1 = s1;
      for (int it = 0; it < 80; ++it) {
        double x2 = x1 - f1 * (x1 - x0) / (f1 - f0);
        if (!(x2 > fmin(x0, x1) && x2 < fmax(x0, x1))) x2 = 0.5 * (x0 + x1);
        double f2 = dense1(r.y[2], y1[2], h * r.f[2], h * k[2], hd2, x2) - kHalfPi;
        if (f2 == 0.0) {
          x1 = x2;
          break;
        }
        if ((f2 > 0.0) != (f1 > 0.0)) {
          x0 = x1;
          f0 = f1;
        } else {
          f0 *= 0.5;
        }
        x1 = x2;
        f1 = f2;
        if (fabs(x1 - x0) <= 1e-15 || fabs(f2) <= 1e-15) break;
      }
      sig = x1;
    }
    const double Rc = dense1(r.y[1], y1[1], h * r.f[1], h * k[1], hd1, sig);
    const double thc = dense1(r.y[2], y1[2], h * r.f[2], h * k[2], hd2, sig);
    const double pthc = dense1(r.y[5], y1[5], h * r.f[5], h * k[5], hd5, sig);
    const double cth = cos(thc);
    const double thdot = pthc / (Rc * Rc + m.chi2 * cth * cth);
    const double lamc = r.lam + sig * h;
    if (Rc >= ip.R_cap && Rc <= ip.R_esc && fabs(thdot) >= ip.thdot_min &&
        (!r.cs.have_trusted || lamc - r.cs.lam_last >= ip.dlam_min)) {
      crossed = true;
      sig_out = sig;
      Rc_out = Rc;
      r.cs.ncross++;
      r.cs.lam_last = lamc;
      r.cs.have_trusted = true;
    }
  }
  r.lam += h;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    r.y[i] = y1[i];
    r.f[i] = k[i];
  }
  if (reflect_axis(r.y[2], r.y[5], r.y[3])) {
    reflected = true;
    rhs_f64_into(m, r.E, r.ell, r.y[1], r.y[2], r.y[4], r.y[5], r.f);
  }
  if (r.y[1] < ip.R_cap) return 2;
  if (r.y[1] > ip.R_esc) return 1;
  r.h = h * f64_of_f32(step_factor(err, r.rejected));
  r.rejected = false;
  return r.steps >= ip.max_steps ? 3 : 0;
}

// The flattened list of the image's traced cells (base pixels, then each
// level): screen position and weight dL/dI of cell idx; false past the end.
__device__ __forceinline__ bool adj_cell(const AdjWarpArgs& a, int64_t idx, double& X, double& Y,
                                         double& gI) {
  int level = 0;
  int64_t nc = a.npix;
  while (idx >= nc) {
    idx -= nc;
    if (++level > a.levels) return false;
    const unsigned long long c = a.hdr->count[level];
    nc = (int64_t)(c < (unsigned long long)a.lv[level].cap ? c : (unsigned long long)a.lv[level].cap);
  }
  uint64_t key;
  double w;
  if (level == 0) {
    key = (uint64_t)idx << 16;
    w = (a.levels > 0 && a.base_child[idx] >= 0) ? 0.0 : 1.0;
  } else {
    key = a.lv[level].key[idx];
    const bool leaf = level == a.levels || a.lv[level].child[idx] < 0;
    w = leaf ? 1.0 / (double)(1 << (4 * level)) : 0.0;
  }
  gI = w * a.Gpix[(int64_t)(key >> 16)];
  cell_centre(*a.ip, key, X, Y);
  return true;
}

// 1. Forward replay, one ray per thread: the accepted steps' start states and
// sizes go to chunks of the trajectory pool (kAdjChunk steps each, newest
// first in a list), the crossings to the ray's record.  A thread reserves the
// longest ray's chunks before it starts a ray and gives back what the ray did
// not use, so a ray never runs out of room; when the pool or the records are
// full the kernel ends and the next launch goes on after the reverse sweep.
__global__ void __launch_bounds__(128) adj_forward_kernel(AdjWarpArgs a) {
  const ImgParams& ip = *a.ip;
  const MetricConsts<double> m = metric_consts<double>(ip);
  const unsigned long long per = (unsigned long long)a.per_ray;
  while (true) {
    if (atomicAdd(&a.ctl->reserved, per) + per > (unsigned long long)a.chunks) {
      atomicAdd(&a.ctl->reserved, 0ull - per);
      break;
    }
    double X = 0.0, Y = 0.0, gI = 0.0;
    // a record first: the cell claimed below then has one
    bool more = atomicAdd(&a.ctl->claimed, 1ull) < (unsigned long long)a.max_rays;
    while (more) {
      const int64_t idx = (int64_t)atomicAdd(a.head, 1ull);
      more = adj_cell(a, idx, X, Y, gI);
      if (!more) a.ctl->done = 1;
      if (!more || gI != 0.0) break;
    }
    if (!more) {
      atomicAdd(&a.ctl->reserved, 0ull - per);
      break;
    }
    Ray64 r;
    ray_init64(ip, m, X, Y, r);
    double pdir[13];  // direct adjoint of the crossing terms (tangents of D13)
    for (int t = 0; t < 13; ++t) pdir[t] = 0.0;
    AdjRay& rec = a.ray[atomicAdd(&a.ctl->rays, 1ull)];
    int nx = 0, used = 0;
    int32_t chunk = -1;
    int overflow = 0;
    while (true) {
      const int n = r.nacc;
      const double y0 = r.y[1], y1 = r.y[2], y2 = r.y[4], y3 = r.y[5], h0 = r.h;
      bool crossed, refl;
      double sig, Rc;
      const int term = adj_step_rolled(ip, m, r, crossed, sig, Rc, refl);
      if (r.nacc > n) {
        const int i = n % kAdjChunk;
        if (i == 0) {
          if (used >= a.per_ray) {
            overflow = kAdjNoRoom;
            break;
          }
          const int32_t c = (int32_t)atomicAdd(&a.ctl->used, 1ull);  // reserved: there is one
          a.prev[c] = chunk;
          chunk = c;
          ++used;
        }
        double* d = a.pool + (int64_t)chunk * (5 * kAdjChunk) + i;
        d[0] = y0;
        d[kAdjChunk] = y1;
        d[2 * kAdjChunk] = y2;
        d[3 * kAdjChunk] = y3;
        d[4 * kAdjChunk] = refl ? -h0 : h0;  // the sign marks a reflection after the step
      }
      if (crossed) {
        D13 Ic;
        double Rb = 0.0;
        if (crossing_intensity_dual(ip, Rc, r.E, r.ell, Ic)) {
          Rb = gI * Ic.d[0];
          for (int t = 1; t < 13; ++t) pdir[t] += gI * Ic.d[t];
        }
        if (nx < kMaxCrossAdj) rec.x[nx++] = XRec{r.nacc - 1, sig, Rb};
        else overflow = (int)BH_ERR_WORKSPACE;
      }
      if (term) break;
    }
    if (overflow) {
      atomicCAS(a.status, 0, overflow);
      nx = 0;
    }
    rec.nx = nx;
    rec.chunk = chunk;
    rec.last = r.nacc - 1;
    rec.X = X;
    rec.Y = Y;
    rec.E = r.E;
    rec.ell = r.ell;
    for (int t = 0; t < 13; ++t) rec.pdir[t] = pdir[t];
    atomicAdd(&a.ctl->reserved, 0ull - (per - (unsigned long long)used));
  }
}

// Delta(R) with its derivatives: D, D_R, D_RR, and the derivatives of D and D_R
// with respect to lambda_E.  Einasto: D = R^2 - 2 R M(x) + chi^2, x = R /
// lambda_E, M = 1 - (1 + x + x^2/2) e^-x, M' = x^2 e^-x / 2.
struct DeltaJet {
  double D, D1, D2, Dh, D1h;  // the halo parameter: Einasto's lambda_E
};
__device__ __forceinline__ DeltaJet delta_jet(const ImgParams& ip, double R) {
  DeltaJet o;
  const MetricConsts<double>& m = ip.md;
  o.Dh = o.D1h = 0.0;
  if (m.metric == 1) {
    const double x = R * m.il, e = d_exp(-x), x2 = x * x;
    const double M = 1.0 - (1.0 + x + 0.5 * x2) * e, g = 0.5 * x2 * e;  // g = dM/dx
    const double gx = x * e - g;                                      // d(g)/dx
    o.D = R * R - 2.0 * R * M + m.chi2;
    o.D1 = 2.0 * R - 2.0 * M - 2.0 * x * g;                            // R dM/dR = x g
    o.D2 = 2.0 - 2.0 * m.il * (2.0 * g + x * gx);
    // dx/dlambda = -x / lambda
    const double xl = -x * m.il;
    o.Dh = -2.0 * R * g * xl;
    o.D1h = -2.0 * xl * (2.0 * g + x * gx);
  } else {
    o.D = R * R - 2.0 * R + m.chi2;
    o.D1 = 2.0 * R - 2.0;
    o.D2 = 2.0;
  }
  return o;
}

// Derivatives of the right-hand side's active components f = (dR, dtheta,
// dp_R, dp_theta)/dlambda (geo_rhs_sc) with respect to (R, theta, p_R,
// p_theta, E, ell, chi, lambda_E), by differentiating the closed form: with
// U = Delta' (p_R^2 + PD^2) - 4 E R PD, PD = P / Delta,
//   f_R = Delta p_R / Sigma,  f_th = p_th / Sigma,
//   f_pR = -U / (2 Sigma) + W R / Sigma^2,
//   f_pth = -Q Q_th / Sigma - W chi^2 s c / Sigma^2.
// About 300 FP64 operations; dual numbers through the same right-hand side
// took about four times that.
__device__ __forceinline__ void rhs_jacobian(const ImgParams& ip, double E, double ell,
                                             const double* Y, double J[4][8]) {
  const MetricConsts<double>& m = ip.md;
  const double R = Y[0], pR = Y[2], pth = Y[3], chi = m.chi, chi2 = m.chi2;
  double s, c;
  d_sincos(Y[1], &s, &c);
  const DeltaJet d = delta_jet(ip, R);
  const double iS = d_rcp(R * R + chi2 * c * c), iS2 = iS * iS;
  const double iD = d_rcp(d.D), is = d_rcp(s), is2 = is * is;
  const double ra = R * R + chi2, P = ra * E - chi * ell, PD = P * iD;
  const double Q = ell * is - chi * E * s, Qt = -c * (ell * is2 + chi * E);  // dQ/dtheta
  const double a2 = pR * pR + PD * PD;
  const double W = d.D * pR * pR - P * PD + pth * pth + Q * Q;
  const double U = d.D1 * a2 - 4.0 * E * R * PD;
  const double x = chi2 * s * c;                       // -dSigma/dtheta / 2
  const double WR = W * R, Wx = W * x, QQ = Q * Qt;
  // f_pR and f_pth for a change of (U, W, Sigma), the rest of their changes
  // added by the caller: -dU iS/2 + dW R iS^2 + (U/2 iS^2 - 2 W R iS^3) dSigma
  const double gU = -0.5 * iS, gW = R * iS2, gS = iS2 * (0.5 * U - 2.0 * WR * iS);
  const double hW = -x * iS2, hS = iS2 * (QQ + 2.0 * Wx * iS);
  const double U_PD = 2.0 * d.D1 * PD - 4.0 * E * R;   // dU/dPD
  const double W_D = pR * pR + PD * PD;                // dW/dDelta at fixed P
  const double W_P = -2.0 * PD;
  const double DpS = d.D * pR * iS2, pthS = pth * iS2;
  // a change of P: PD changes by dP / Delta
  const double U_P = U_PD * iD;
  // a change of Delta: PD changes by -PD dDelta / Delta
  const double U_D = -U_PD * PD * iD;
  {  // R
    const double dS = 2.0 * R, dP = 2.0 * R * E, dD = d.D1;
    const double dW = W_D * dD + W_P * dP;
    const double dU = d.D2 * a2 + U_D * dD + U_P * dP - 4.0 * E * PD;
    J[0][0] = d.D1 * pR * iS - DpS * dS;
    J[1][0] = -pthS * dS;
    J[2][0] = gU * dU + gW * dW + W * iS2 + gS * dS;
    J[3][0] = hW * dW + hS * dS;
  }
  {  // theta
    const double dS = -2.0 * x, dW = 2.0 * QQ;
    const double Qtt = s * (ell * is2 + chi * E) + 2.0 * ell * c * c * is2 * is;  // d2Q/dtheta2
    J[0][1] = -DpS * dS;
    J[1][1] = -pthS * dS;
    J[2][1] = gW * dW + gS * dS;
    J[3][1] = -(Qt * Qt + Q * Qtt) * iS + hW * dW + hS * dS - W * chi2 * (c * c - s * s) * iS2;
  }
  {  // p_R
    const double dW = 2.0 * d.D * pR, dU = 2.0 * d.D1 * pR;
    J[0][2] = d.D * iS;
    J[1][2] = 0.0;
    J[2][2] = gU * dU + gW * dW;
    J[3][2] = hW * dW;
  }
  {  // p_theta
    const double dW = 2.0 * pth;
    J[0][3] = 0.0;
    J[1][3] = iS;
    J[2][3] = gW * dW;
    J[3][3] = hW * dW;
  }
  {  // E: dP = ra, dQ = -chi s, dQ_th = -chi c
    const double dQ = -chi * s, dW = W_P * ra + 2.0 * Q * dQ;
    const double dU = U_P * ra - 4.0 * R * PD;
    J[0][4] = J[1][4] = 0.0;
    J[2][4] = gU * dU + gW * dW;
    J[3][4] = -(dQ * Qt - Q * chi * c) * iS + hW * dW;
  }
  {  // ell: dP = -chi, dQ = 1/s, dQ_th = -c/s^2
    const double dW = -W_P * chi + 2.0 * Q * is;
    J[0][5] = J[1][5] = 0.0;
    J[2][5] = -gU * U_P * chi + gW * dW;
    J[3][5] = -(is * Qt - Q * c * is2) * iS + hW * dW;
  }
  {  // chi: dSigma = 2 chi c^2, dP = 2 chi E - ell, dDelta = 2 chi
    const double dS = 2.0 * chi * c * c, dP = 2.0 * chi * E - ell, dD = 2.0 * chi;
    const double dQ = -E * s, dW = W_D * dD + W_P * dP + 2.0 * Q * dQ;
    const double dU = U_D * dD + U_P * dP;
    J[0][6] = dD * pR * iS - DpS * dS;
    J[1][6] = -pthS * dS;
    J[2][6] = gU * dU + gW * dW + gS * dS;
    J[3][6] = -(dQ * Qt - Q * E * c) * iS + hW * dW + hS * dS - W * 2.0 * chi * s * c * iS2;
  }
  {  // lambda_E: Delta and Delta' only
    const double dW = W_D * d.Dh, dU = d.D1h * a2 + U_D * d.Dh;
    J[0][7] = d.Dh * pR * iS;
    J[1][7] = 0.0;
    J[2][7] = gU * dU + gW * dW;
    J[3][7] = hW * dW;
  }
}

static __constant__ DPTab kDPc = kDP;

// The stage states Y_s and derivatives k_s (active components) of a step.
__device__ __forceinline__ void adj_stages(const ImgParams& ip, double E, double ell,
                                           const double* yn, double h, double Y[7][4],
                                           double kv[7][4]) {
  const RayC<double> kc = ray_consts(ip.md, E, ell);
#pragma unroll 1
  for (int s = 0; s < 7; ++s) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int j = 0; j < s; ++j) {
      const double aj = kDPc.a[s][j];
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[x] = fma(aj, kv[j][x], acc[x]);
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) Y[s][x] = yn[x] + h * acc[x];
    double d[6], W, P2, sth, cth;
    d_sincos(Y[s][1], &sth, &cth);
    geo_rhs_sc(ip.md, kc, Y[s][0], sth, cth, Y[s][2], Y[s][3], d, W, P2);
#pragma unroll
    for (int x = 0; x < 4; ++x) kv[s][x] = d[kQC(x)];
  }
}

// Reverse recursion of one step for NU adjoint vectors at once: kb[s][u] the
// adjoints of k_s on entry (without the update's h b_s ybar), yb[u] that of
// y_{n+1}; out[u] receives the adjoints of y_n (4, added to what yn_bar holds)
// and of (E, ell, chi, lambda_E).
template <int NU>
__device__ __forceinline__ void adj_reverse(const ImgParams& ip, double E, double ell, double h,
                                            const double Y[7][4], int s_top, double kb[7][NU][4],
                                            double out[NU][8]) {
#pragma unroll 1
  for (int s = s_top; s >= 0; --s) {
    double J[4][8];
    rhs_jacobian(ip, E, ell, Y[s], J);
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const double k0 = kb[s][u][0], k1 = kb[s][u][1], k2 = kb[s][u][2], k3 = kb[s][u][3];
      double Yb[4];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        // f_R does not depend on p_theta, E, ell; f_theta only on R, theta,
        // p_theta and chi
        double acc = fma(J[3][t], k3, J[2][t] * k2);
        if (t != 3 && t != 4 && t != 5) acc = fma(J[0][t], k0, acc);
        if (t == 0 || t == 1 || t == 3 || t == 6) acc = fma(J[1][t], k1, acc);
        if (t < 4) Yb[t] = acc;
        out[u][t] += acc;
      }
#pragma unroll 1
      for (int j = 0; j < s; ++j) {
        const double aj = h * kDPc.a[s][j];
#pragma unroll
        for (int x = 0; x < 4; ++x) kb[j][u][x] = fma(aj, Yb[x], kb[j][u][x]);
      }
    }
  }
}

// 2. Reverse sweep, one warp per ray: each lane forms the adjoint map of one of
// 32 consecutive steps, ybar_{n+1} -> (ybar_n, adjoints of E, ell, chi,
// lambda_E), as a 4 x 8 matrix (four unit vectors through the step's reverse
// recursion) with the crossing's own contribution; then the warp applies the
// 32 maps in order, eight lanes a matrix-vector product.  A thread per ray did
// the steps one after the other: a small image kept a few warps busy for as
// long as its longest ray, and each reverse sweep replayed its steps first.
constexpr int kAdjWarps = 4;
struct AdjMaps {
  double T[4][8][32];
  double c[8][32];
};
__global__ void __launch_bounds__(32 * kAdjWarps) adj_reverse_kernel(AdjWarpArgs a) {
  extern __shared__ unsigned char adj_smem[];
  const int lane = threadIdx.x & 31;
  AdjMaps& M = reinterpret_cast<AdjMaps*>(adj_smem)[threadIdx.x >> 5];
  const ImgParams& ip = *a.ip;
  double gacc = 0.0;  // lane t: gradient component t
  const unsigned long long n_rays = a.ctl->rays;
  while (true) {
    unsigned long long idx = 0;
    if (lane == 0) idx = atomicAdd(&a.ctl->swept, 1ull);
    idx = __shfl_sync(kFull, idx, 0);
    if (idx >= n_rays) break;
    const AdjRay& rec = a.ray[idx];
    const int nx = rec.nx;
    if (nx == 0) continue;
    const double E = rec.E, ell = rec.ell;
    const int last = rec.x[nx - 1].step;  // the sweep starts at the last crossing step
    int32_t chunk = rec.chunk;
    for (int k = rec.last / kAdjChunk; k > last / kAdjChunk; --k) chunk = a.prev[chunk];
    int at = last / kAdjChunk;            // chunk's place in the ray
    // lanes 0-3: adjoint of (R, theta, p_R, p_theta); lanes 4-7: of (E, ell,
    // chi, lambda_E), which the crossings' direct terms start
    double v = lane >= 4 && lane < 8 ? rec.pdir[lane - 3] : 0.0;
    for (int seg = last / 32; seg >= 0; --seg) {
      const int n = 32 * seg + lane;
      if (32 * seg / kAdjChunk != at) {
        chunk = a.prev[chunk];
        --at;
      }
      double h = 0.0;
      if (n <= last) {
        const double* d = a.pool + (int64_t)chunk * (5 * kAdjChunk) + n % kAdjChunk;
        double yn[4] = {d[0], d[kAdjChunk], d[2 * kAdjChunk], d[3 * kAdjChunk]};
        h = d[4 * kAdjChunk];
        const double ha = fabs(h);
        double Y[7][4], kv[7][4];
        adj_stages(ip, E, ell, yn, ha, Y, kv);
        {
          double kb[7][4][4], out[4][8];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int t = 0; t < 8; ++t) out[u][t] = t == u ? 1.0 : 0.0;
          }
#pragma unroll 1
          for (int s = 0; s < 7; ++s) {
            const double b = ha * kDPc.b[s];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int x = 0; x < 4; ++x) kb[s][u][x] = x == u ? b : 0.0;
          }
          adj_reverse<4>(ip, E, ell, ha, Y, 5, kb, out);  // b_6 = 0
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int t = 0; t < 8; ++t) M.T[u][t][lane] = out[u][t];
        }
        int x = -1;
        for (int i = 0; i < nx; ++i)
          if (rec.x[i].step == n) x = i;
        double cc[1][8];
#pragma unroll
        for (int t = 0; t < 8; ++t) cc[0][t] = 0.0;
        if (x >= 0) {
          // dense output y(sig) = c0 y_n + c1 y_{n+1} + c2 h k1 + c3 h k7 + c4 h
          // sum d_j k_j; the abscissa moves with theta (implicit derivative)
          const double sg = rec.x[x].sig, Rb = rec.x[x].Rbar, u = 1.0 - sg;
          const double c1 = sg * sg * (3.0 - 2.0 * sg), c0 = 1.0 - c1, c2 = sg * u * u,
                       c3 = -sg * sg * u, c4 = sg * sg * u * u;
          const double e1 = 6.0 * sg * u, e0 = -e1, e2 = u * (1.0 - 3.0 * sg),
                       e3 = sg * (3.0 * sg - 2.0), e4 = 2.0 * sg * u * (1.0 - 2.0 * sg);
          double w[2];
          {
            double dq[2];
            for (int q = 0; q < 2; ++q) {
              double acc = 0.0, dd = 0.0;
              for (int j = 0; j < 7; ++j) {
                acc += kDPc.b[j] * kv[j][q];
                dd += kDPc.d[j] * kv[j][q];
              }
              dq[q] = e0 * yn[q] + e1 * (yn[q] + ha * acc) + e2 * ha * kv[0][q] +
                      e3 * ha * kv[6][q] + e4 * ha * dd;
            }
            w[0] = Rb;
            w[1] = -Rb * dq[0] / dq[1];
          }
          double kb[7][1][4];
          for (int s = 0; s < 7; ++s) {
            const double b = ha * (kDPc.b[s] * c1 + kDPc.d[s] * c4) +
                             (s == 0 ? ha * c2 : 0.0) + (s == 6 ? ha * c3 : 0.0);
            kb[s][0][0] = b * w[0];
            kb[s][0][1] = b * w[1];
            kb[s][0][2] = kb[s][0][3] = 0.0;
          }
          cc[0][0] = w[0] * (c0 + c1);
          cc[0][1] = w[1] * (c0 + c1);
          adj_reverse<1>(ip, E, ell, ha, Y, 6, kb, cc);
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) M.c[t][lane] = cc[0][t];
      }
      const unsigned refl = __ballot_sync(kFull, h < 0.0);
      __syncwarp();
      for (int i = min(31, last - 32 * seg); i >= 0; --i) {
        double y0 = __shfl_sync(kFull, v, 0), y1 = __shfl_sync(kFull, v, 1),
               y2 = __shfl_sync(kFull, v, 2), y3 = __shfl_sync(kFull, v, 3);
        if ((refl >> i) & 1u) {  // reflection after the step: theta -> -theta, p_th -> -p_th
          y1 = -y1;
          y3 = -y3;
        }
        if (lane < 8) {
          const double o = fma(M.T[3][lane][i], y3,
                               fma(M.T[2][lane][i], y2,
                                   fma(M.T[1][lane][i], y1, fma(M.T[0][lane][i], y0, M.c[lane][i]))));
          v = lane < 4 ? o : v + o;
        }
      }
      __syncwarp();
    }
    // 3. launch: theta_0 = theta_o, p_R = sqrt(g_RR) n^R, p_th = sqrt(g_thth) n^th,
    //    ell = sqrt(g_phph) n^phi, E = N + omega ell (Eqs. 63-74)
    double w[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) w[t] = __shfl_sync(kFull, v, t);
    const double X = rec.X, Y = rec.Y;
    const double dd = sqrt(ip.r_obs * ip.r_obs + X * X + Y * Y);
    const double nR = -ip.r_obs / dd, nth = -Y / dd, nph = -X / dd;
    if (lane < 4) {
      const double dell = a.aj.d_sqgph[lane] * nph;
      const double dE = a.aj.d_N[lane] + a.aj.d_w[lane] * (ip.sq_gph * nph) + ip.zamo_w * dell;
      double g = w[2] * a.aj.d_sqgrr[lane] * nR + w[3] * a.aj.d_sqgth[lane] * nth + w[5] * dell +
                 w[4] * dE + rec.pdir[6] * a.aj.d_Rin[lane];
      if (lane == 1) g += w[1];
      if (lane == 0) g += w[6];
      if (lane == 2) g += w[7];
      gacc += g;
    } else if (lane < 10) {
      gacc += rec.pdir[3 + lane];
    }
  }
  if (lane < 10 && gacc != 0.0) atomicAdd(&a.grad[lane], gacc);
}

cudaError_t launch_adj_forward(const AdjWarpArgs& a, int blocks, int threads, cudaStream_t s) {
  adj_forward_kernel<<<blocks, threads, 0, s>>>(a);
  return cudaGetLastError();
}
cudaError_t launch_adj_reverse(const AdjWarpArgs& a, cudaStream_t s) {
  const int smem = (int)sizeof(AdjMaps) * kAdjWarps;
  cudaError_t e = cudaFuncSetAttribute(adj_reverse_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int nb = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, adj_reverse_kernel, 32 * kAdjWarps, smem);
  if (e != cudaSuccess) return e;
  adj_reverse_kernel<<<num_sms() * (nb > 0 ? nb : 1), 32 * kAdjWarps, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace bhrt
