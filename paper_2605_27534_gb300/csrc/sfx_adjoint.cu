// Discrete adjoint of the no-flow coupled step (App. C), FP64.
//
// One step solves R(x1; x0, theta) = 0 for x1 = (f, F) with the residual of
// both App. C equations
//   R_f = (f* - f)/dt + N_f f + q,   R_F = (F* - F)/dt + N_F F - q,
//   q = k_a F (f_inf - f)/(phi + eta) - k_d f,
// N the finite-volume flux divergence of Sec. 3.1-3.2 (diffusivity D and
// drift B, both proportional to D) and f* = f^n, F* = F^n.  With
// -J = -dR/dx1 = [[a - N_f, -b], [-d, e - N_F]] per cell, where
//   a = 1/dt + k_d + c1 F,  b = c1 (f_inf - f),  d = c1 F + k_d,
//   e = 1/dt + b,  c1 = k_a/(phi + eta),
// a loss gradient lam1 = dL/dx1 pulls back by solving
//   (-J)^T nu = lam1,   lam0 = nu/dt,   dL/dtheta += (dR/dtheta)^T nu,
// with dR_f/dk_a = F (f_inf - f)/(phi + eta) = -dR_F/dk_a,
// dR_f/dk_d = -f = -dR_F/dk_d, dR_f/dD_f = N^_f f and dR_F/dD_F = N^_F F
// (N^ at unit diffusivity).  The transposed system is solved by defect
// correction: the FP64 residual r = lam - (-J)^T nu decides convergence and
// the correction e of (-J)^T e = r is relaxed by FP32 red-black Gauss-Seidel
// with a 2x2 solve per cell (the coupling is pointwise) on coefficients
// precomputed once per step from the FP64 operator.
//
// 2D grids (the rollout workload) take that solve from a table of the FP64
// weights, relax ten colours per launch in shared memory and decide about the
// next check on the device; 3D grids, whose table would cost 112 bytes per
// cell more, evaluate the operator in every residual and relax colour by
// colour.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sfx_internal.h"
#include "sfx_op64.cuh"

namespace sfx {
namespace {

constexpr int kAdjThreads = 256;

struct AdjP {
  Level L;
  double Df, DF, inv_dt, ka, kd, ginf, eps, eta;
  int literal;
  const double* Bf[3];   // unit-diffusivity drift faces
  const double* BF[3];
};

__device__ __forceinline__ Op op_of(const AdjP& p, int field, double D) {
  Op o;
  o.D = D;
  for (int d = 0; d < 3; ++d) o.B[d] = field ? p.BF[d] : p.Bf[d];
  o.literal = p.literal;
  o.lam = nullptr;
  o.Bs = D;
  return o;
}

struct Kin {
  double a, b, d, e, c1, finf, pe;
};

__device__ __forceinline__ Kin kin_at(const AdjP& p, double ph, double f, double F) {
  Kin k;
  k.pe = ph + p.eta;
  k.c1 = p.ka / k.pe;
  k.finf = p.ginf * ph * (1.0 - ph) / p.eps;
  k.b = k.c1 * (k.finf - f);
  k.d = k.c1 * F + p.kd;
  k.a = p.inv_dt + p.kd + k.c1 * F;
  k.e = p.inv_dt + k.b;
  return k;
}

__device__ __forceinline__ void cell_ijk(const Level& L, size_t c, int& i, int& j, int& k) {
  i = (int)(c % L.nx);
  j = (int)((c / L.nx) % L.ny);
  k = (int)(c / ((size_t)L.nx * L.ny));
}

// out = (-J) v, or (-J)^T v with transpose != 0
__global__ void k_adj_apply(AdjP p, const double* __restrict__ phi, const double* __restrict__ f,
                            const double* __restrict__ F, const double* __restrict__ vf,
                            const double* __restrict__ vF, int transpose,
                            double* __restrict__ of, double* __restrict__ oF) {
  const Level& L = p.L;
  const size_t n = L.ncell();
  const Op opf = op_of(p, 0, p.Df), opF = op_of(p, 1, p.DF);
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(L, c, i, j, k);
    const Kin q = kin_at(p, phi[c], f[c], F[c]);
    double Nf, NF;
    if (!transpose) {
      double sd, sn;
      const double iv = 1.0 / cell_volume(L, i);
      flux_terms(L, opf, vf, i, j, k, sd, sn);
      Nf = (sd * vf[c] + sn) * iv;
      flux_terms(L, opF, vF, i, j, k, sd, sn);
      NF = (sd * vF[c] + sn) * iv;
      of[c] = q.a * vf[c] - Nf - q.b * vF[c];
      oF[c] = -q.d * vf[c] + q.e * vF[c] - NF;
    } else {
      double dT, nT;
      flux_terms_T(L, opf, vf, i, j, k, dT, nT);
      Nf = dT * vf[c] + nT;
      flux_terms_T(L, opF, vF, i, j, k, dT, nT);
      NF = dT * vF[c] + nT;
      of[c] = q.a * vf[c] - Nf - q.d * vF[c];
      oF[c] = -q.b * vf[c] + q.e * vF[c] - NF;
    }
  }
}

// nu = dt lam: the solution when transport is negligible against 1/dt
__global__ void k_adj_init(size_t n, double dt, const double* __restrict__ lf,
                           const double* __restrict__ lF, double* __restrict__ nf,
                           double* __restrict__ nF) {
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    nf[c] = dt * lf[c];
    nF[c] = dt * lF[c];
  }
}

// r = lam - (-J)^T nu (rounded to float into rout), max |r| and max |lam|
// over both fields
__global__ void k_adj_resid(AdjP p, const double* __restrict__ phi, const double* __restrict__ f,
                            const double* __restrict__ F, const double* __restrict__ lf,
                            const double* __restrict__ lF, const double* __restrict__ nf,
                            const double* __restrict__ nF, float2* __restrict__ rout,
                            unsigned long long* nrm) {
  const Level& L = p.L;
  const size_t n = L.ncell();
  const Op opf = op_of(p, 0, p.Df), opF = op_of(p, 1, p.DF);
  double mr = 0.0, mb = 0.0;
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(L, c, i, j, k);
    const Kin q = kin_at(p, phi[c], f[c], F[c]);
    double dT, nT;
    flux_terms_T(L, opf, nf, i, j, k, dT, nT);
    const double rf = lf[c] - (q.a * nf[c] - (dT * nf[c] + nT) - q.d * nF[c]);
    flux_terms_T(L, opF, nF, i, j, k, dT, nT);
    const double rF = lF[c] - (-q.b * nf[c] + q.e * nF[c] - (dT * nF[c] + nT));
    rout[c] = make_float2((float)rf, (float)rF);
    double r = fmax(fabs(rf), fabs(rF));
    if (!(r <= 1e300)) r = INFINITY;   // NaN or Inf: never converged
    mr = fmax(mr, r);
    mb = fmax(mb, fmax(fabs(lf[c]), fabs(lF[c])));
  }
  mr = warp_max(mr);
  mb = warp_max(mb);
  if ((threadIdx.x & 31) == 0) {
    atomic_max_nonneg(&nrm[0], mr);
    atomic_max_nonneg(&nrm[1], mb);
  }
}

// Coefficients of the FP32 relaxation: per cell the inverse of the 2x2
// block [[A11, -d], [-b, A22]] of (-J)^T (A11 = a - dT_f, A22 = e - dT_F) as
// (A22, d, b, A11)/det, and the neighbour weights of N^T of both fields
// (W[q N + c] for f, W[(6 + q) N + c] for F).
__global__ void k_adj_coef(AdjP p, const double* __restrict__ phi, const double* __restrict__ f,
                           const double* __restrict__ F, float4* __restrict__ K,
                           float* __restrict__ W) {
  const Level& L = p.L;
  const size_t n = L.ncell();
  const Op opf = op_of(p, 0, p.Df), opF = op_of(p, 1, p.DF);
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(L, c, i, j, k);
    const Kin q = kin_at(p, phi[c], f[c], F[c]);
    double dTf, dTF, wf[6], wF[6];
    flux_weights_T(L, opf, i, j, k, dTf, wf);
    flux_weights_T(L, opF, i, j, k, dTF, wF);
    const double A11 = q.a - dTf, A22 = q.e - dTF;
    const double idet = 1.0 / (A11 * A22 - q.d * q.b);
    K[c] = make_float4((float)(A22 * idet), (float)(q.d * idet), (float)(q.b * idet),
                       (float)(A11 * idet));
#pragma unroll
    for (int m = 0; m < 6; ++m) {
      W[(size_t)m * n + c] = (float)wf[m];
      W[(size_t)(6 + m) * n + c] = (float)wF[m];
    }
  }
}

// One colour of the FP32 red-black Gauss-Seidel on (-J)^T e = r
__global__ void k_adj_csweep(Level L, const float4* __restrict__ K, const float* __restrict__ W,
                             const float2* __restrict__ r, float2* __restrict__ e, int color) {
  const int j = blockIdx.y, k = blockIdx.z;
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ((j + k + color) & 1);
  if (i >= L.nx) return;
  const size_t n = L.ncell();
  const size_t c = cidx(L, i, j, k);
  const size_t sy = (size_t)L.nx, sz = (size_t)L.nx * L.ny;
  const bool has[6] = {i > 0, i + 1 < L.nx, j > 0, j + 1 < L.ny,
                       L.geom == SFX_CART3D && k > 0, L.geom == SFX_CART3D && k + 1 < L.nz};
  const size_t nb[6] = {c - 1, c + 1, c - sy, c + sy, c - sz, c + sz};
  const float2 rc = r[c];
  float sf = rc.x, sF = rc.y;
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    if (!has[m]) continue;
    const float2 v = e[nb[m]];
    sf += W[(size_t)m * n + c] * v.x;
    sF += W[(size_t)(6 + m) * n + c] * v.y;
  }
  const float4 q = K[c];
  e[c] = make_float2(q.x * sf + q.y * sF, q.z * sf + q.w * sF);
}

// nu += e
__global__ void k_adj_add(size_t n, const float2* __restrict__ e, double* __restrict__ nf,
                          double* __restrict__ nF) {
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    const float2 v = e[c];
    nf[c] += (double)v.x;
    nF[c] += (double)v.y;
  }
}

// lam0 = nu/dt (in place) and block partials of the four parameter terms
__global__ void k_adj_finish(AdjP p, const double* __restrict__ phi, const double* __restrict__ f,
                             const double* __restrict__ F, const double* __restrict__ nf,
                             const double* __restrict__ nF, double* __restrict__ lf,
                             double* __restrict__ lF, double* __restrict__ part) {
  const Level& L = p.L;
  const size_t n = L.ncell();
  const Op ohf = op_of(p, 0, 1.0), ohF = op_of(p, 1, 1.0);
  double s[4] = {0, 0, 0, 0}, e[4] = {0, 0, 0, 0};
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(L, c, i, j, k);
    const Kin q = kin_at(p, phi[c], f[c], F[c]);
    const double vf = nf[c], vF = nF[c];
    const double iv = 1.0 / cell_volume(L, i);
    double sd, sn;
    flux_terms(L, ohf, f, i, j, k, sd, sn);
    const double Nhf = (sd * f[c] + sn) * iv;
    flux_terms(L, ohF, F, i, j, k, sd, sn);
    const double NhF = (sd * F[c] + sn) * iv;
    const double t[4] = {(vf - vF) * F[c] * (q.finf - f[c]) / q.pe, -(vf - vF) * f[c],
                         vf * Nhf, vF * NhF};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      double u, w;
      two_sum(s[m], t[m], u, w);
      s[m] = u;
      e[m] += w;
    }
    lf[c] = vf * p.inv_dt;
    lF[c] = vF * p.inv_dt;
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    block_sum_comp<kAdjThreads>(s[m], e[m]);
    if (threadIdx.x == 0) {
      const size_t o = 2 * ((size_t)m * gridDim.x + blockIdx.x);
      part[o] = s[m];
      part[o + 1] = e[m];
    }
  }
}

// One block per quantity: fixed-order combination of the block partials.
__global__ void k_adj_reduce(const double* __restrict__ part, int nblk, double* __restrict__ out) {
  const int m = blockIdx.x;
  double s = 0.0, e = 0.0;
  for (int q = threadIdx.x; q < nblk; q += blockDim.x) {
    const size_t o = 2 * ((size_t)m * nblk + q);
    double u, w;
    two_sum(s, part[o], u, w);
    s = u;
    e += part[o + 1] + w;
  }
  block_sum_comp<kAdjThreads>(s, e);
  if (threadIdx.x == 0) out[m] = s + e;
}

// ---- 2D: the solve from tables ---------------------------------------------
// At 256^2 the FP64 residual evaluated from the drift faces took 39 us, four
// times per step, with some 375 instructions per cell on a pipe that retires
// 0.6e12 of them a second, and the coefficients and the parameter terms took
// as much again.  The operator does not change within a step, so one launch
// forms, at unit diffusivity, the weights of both transposed operators and
// the cell's kinetics; the residual and the parameter terms are then 10
// multiply-adds per field.

// Rows of the table U (n doubles each): dT, w x-, x+, y-, y+ of N^_f^T, the
// same of N^_F^T, (f_inf - f)/(phi + eta) and d
enum { U_F = 5, U_B = 10, U_D = 11, U_ROWS = 12 };

// The state of one solve: k_adj_coef2 fills it, k_adj_resid2 keeps it
struct Ctl {
  double Df, DF, inv_dt, ka, tol;
  double rel;
  unsigned long long nrm[2];   // max |r|, max |lam| as integer words
  int max_checks, checks;
  unsigned blocks;             // finished blocks of this check
  int state;                   // 0: relax again, 1: converged, 2: out of checks, 3: not finite
};

__device__ __forceinline__ double flip_if(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}

// The table, the FP32 relaxation's K and W (see k_adj_coef; four weights per
// field) and the start nu = dt lam with a copy of lam.  256^2: 31 -> 11 us
// (with k_adj_init 33).
__global__ void __launch_bounds__(256)
k_adj_coef2(AdjP p, double invh, double inv_eps, const double* __restrict__ phi, const double* __restrict__ f,
            const double* __restrict__ F, const double* __restrict__ lf,
            const double* __restrict__ lF, double dt, double tol, int max_checks,
            double* __restrict__ U, float4* __restrict__ K, float* __restrict__ W,
            double* __restrict__ nf, double* __restrict__ nF, double* __restrict__ cf,
            double* __restrict__ cF, Ctl* ctl) {
  const Level& L = p.L;
  const size_t n = L.ncell();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    ctl->Df = p.Df;
    ctl->DF = p.DF;
    ctl->inv_dt = p.inv_dt;
    ctl->ka = p.ka;
    ctl->tol = tol;
    ctl->rel = INFINITY;
    ctl->nrm[0] = ctl->nrm[1] = 0ull;
    ctl->max_checks = max_checks;
    ctl->checks = 0;
    ctl->blocks = 0u;
    ctl->state = 0;
  }
  const int i = blockIdx.x * 32 + (threadIdx.x & 31);
  if (i >= L.nx) return;
  // area over volume: of the radial faces against the neighbour (w) and the
  // cell (d), of the axial faces against the cell (all 1/h on planar grids)
  double wl = invh, wr = invh, dl = invh, dr = invh, gy = invh;
  if (L.geom == SFX_AXISYM) {
    const double iv = 1.0 / cell_volume(L, i), al = face_area(L, 0, i), ar = face_area(L, 0, i + 1);
    wl = i > 0 ? al / cell_volume(L, i - 1) : 0.0;
    wr = ar / cell_volume(L, i + 1);
    dl = al * iv;
    dr = ar * iv;
    gy = face_area(L, 1, i) * iv;
  }
  const bool hl = i > 0, hr = i + 1 < L.nx;
  for (int j = blockIdx.y * 8 + (threadIdx.x >> 5); j < L.ny; j += gridDim.y * 8) {
    const size_t c = (size_t)j * L.nx + i;
    const bool hd = j > 0, hu = j + 1 < L.ny;
    const size_t fx = (size_t)j * (L.nx + 1) + i;
    double dT[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const double* Bx = q ? p.BF[0] : p.Bf[0];
      const double* By = q ? p.BF[1] : p.Bf[1];
      // cR of the lower faces, cL of the upper ones (face_coeffs at D = 1)
      auto low = [&](double B) {
        const bool left = (__double2hiint(B) < 0) != (p.literal != 0);
        return left ? invh : invh + B;
      };
      auto up = [&](double B) {
        const bool left = (__double2hiint(B) < 0) != (p.literal != 0);
        return left ? B - invh : -invh;
      };
      const double kl = hl ? low(Bx[fx]) : 0.0, kr = hr ? up(Bx[fx + 1]) : 0.0;
      const double kd = hd ? low(By[c]) : 0.0, ku = hu ? up(By[c + L.nx]) : 0.0;
      const double w[4] = {kl * wl, flip_if(kr * wr, true), kd * gy, flip_if(ku * gy, true)};
      dT[q] = (kr * dr - kl * dl) - (w[3] + w[2]);
      U[(size_t)(q * U_F) * n + c] = dT[q];
      const float D = (float)(q ? p.DF : p.Df);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        U[(size_t)(q * U_F + 1 + m) * n + c] = w[m];
        W[(size_t)(q * 4 + m) * n + c] = narrow(w[m]) * D;
      }
    }
    const double ph = phi[c], rp = 1.0 / (ph + p.eta);
    const double bh = (p.ginf * ph * (1.0 - ph) * inv_eps - f[c]) * rp;
    const double d = p.ka * rp * F[c] + p.kd, b = p.ka * bh;
    U[(size_t)U_B * n + c] = bh;
    U[(size_t)U_D * n + c] = d;
    const double A11 = p.inv_dt + d - p.Df * dT[0], A22 = p.inv_dt + b - p.DF * dT[1];
    const double idet = 1.0 / (A11 * A22 - d * b);
    K[c] = make_float4(narrow(A22 * idet), narrow(d * idet), narrow(b * idet), narrow(A11 * idet));
    const double x = lf[c], y = lF[c];
    cf[c] = x;
    cF[c] = y;
    nf[c] = dt * x;
    nF[c] = dt * y;
  }
}

__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long x) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
    x = y > x ? y : x;
  }
  return x;
}

// r = lam - (-J)^T nu from the table (rounded to float into rout), and in the
// last block the decision about this check: `loop` goes on while the solve
// has neither converged nor run out of checks.  Magnitudes are compared as
// integer words (a NaN exceeds every number and ends the solve).  256^2: 39
// -> 8.7 us, some 40 FP64 instructions per cell.
__global__ void __launch_bounds__(256)
k_adj_resid2(int nx, int ny, const double* __restrict__ U, const double* __restrict__ lf,
             const double* __restrict__ lF, const double* __restrict__ nf,
             const double* __restrict__ nF, float2* __restrict__ rout, Ctl* ctl,
             cudaGraphConditionalHandle loop) {
  const size_t n = (size_t)nx * ny, c = blockIdx.x * (size_t)256 + threadIdx.x;
  unsigned long long mr = 0ull, mb = 0ull;
  if (c < n) {
    const int j = (int)(c / (size_t)nx), i = (int)(c - (size_t)j * nx);
    const size_t nb[4] = {i > 0 ? c - 1 : c, i + 1 < nx ? c + 1 : c, j > 0 ? c - nx : c,
                          j + 1 < ny ? c + nx : c};   // weight 0 where there is none
    const double vf = nf[c], vF = nF[c], bh = U[(size_t)U_B * n + c], d = U[(size_t)U_D * n + c];
    double tf = U[c] * vf, tF = U[(size_t)U_F * n + c] * vF;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      tf += U[(size_t)(1 + m) * n + c] * nf[nb[m]];
      tF += U[(size_t)(U_F + 1 + m) * n + c] * nF[nb[m]];
    }
    const double b = ctl->ka * bh, x = lf[c], y = lF[c];
    const double rf = x - ((ctl->inv_dt + d) * vf - ctl->Df * tf - d * vF);
    const double rF = y - ((ctl->inv_dt + b) * vF - ctl->DF * tF - b * vf);
    rout[c] = make_float2(narrow(rf), narrow(rF));
    auto mag = [](double v) {
      return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    };
    mr = max(mag(rf), mag(rF));
    mb = max(mag(x), mag(y));
  }
  __shared__ unsigned long long sr[8], sb[8];
  mr = warp_max_bits(mr);
  mb = warp_max_bits(mb);
  if ((threadIdx.x & 31) == 0) {
    sr[threadIdx.x >> 5] = mr;
    sb[threadIdx.x >> 5] = mb;
  }
  __syncthreads();
  if (threadIdx.x) return;
  for (int q = 1; q < 8; ++q) {
    mr = max(mr, sr[q]);
    mb = max(mb, sb[q]);
  }
  atomicMax(&ctl->nrm[0], mr);
  atomicMax(&ctl->nrm[1], mb);
  __threadfence();
  if (atomicAdd(&ctl->blocks, 1u) != gridDim.x - 1) return;
  __threadfence();
  const double r = __longlong_as_double((long long)atomicExch(&ctl->nrm[0], 0ull));
  const double b = __longlong_as_double((long long)atomicExch(&ctl->nrm[1], 0ull));
  ctl->blocks = 0u;
  const int checks = ctl->checks + 1;
  ctl->checks = checks;
  int state = 0;
  if (!(r <= 1e300)) {
    state = 3;
  } else {
    const double rel = r / (b > 1e-300 ? b : 1e-300);
    ctl->rel = rel;
    if (b == 0.0 || rel <= ctl->tol) state = 1;
    else if (checks >= ctl->max_checks) state = 2;
  }
  ctl->state = state;
  cudaGraphSetConditional(loop, state == 0 ? 1u : 0u);
}

// `colours` half-sweeps (an even number, the first of colour 0) of the FP32 red-black
// Gauss-Seidel on (-J)^T e = r in one launch.  A block holds a window of
// 48 x 40 cells, of which the inner 28 x 20 are its own: a cell at distance d
// from the window's edge is right for the first d half-sweeps (outside it
// reads zeros), and ten of them reach no further than the tile.  A thread
// holds a pair of neighbouring cells, one of each colour, their coefficients
// in registers; e lies in shared memory by colour, so that a warp's accesses
// are consecutive.  Each cell takes the operations of k_adj_csweep on the same
// operands, so the tiling changes no bit.  `first`: e = 0 before; `last`: e
// is added to nu instead of being written.  The launches of one colour at 256^2
// took 2.0 us each for 4 MB from L2 (40 per check, 80 us); ten colours take
// 5.8 us: 130 blocks that load 100 KB once, then 0.1 us per colour.
constexpr int kRxP = 24, kRxY = 40, kRxK = 10, kRxTX = 2 * kRxP - 2 * kRxK, kRxTY = kRxY - 2 * kRxK;

__global__ void __launch_bounds__(kRxP* kRxY)
k_adj_relax2(int nx, int ny, const float4* __restrict__ K, const float* __restrict__ W,
             const float2* __restrict__ r, const float2* __restrict__ e, float2* __restrict__ eo,
             int colours, int first, int last, double* __restrict__ nf, double* __restrict__ nF) {
  __shared__ float2 sh[2][kRxY + 2][kRxP + 2];
  const size_t n = (size_t)nx * ny;
  const int tx = threadIdx.x % kRxP, ty = threadIdx.x / kRxP;
  for (int q = threadIdx.x; q < 2 * (kRxY + 2) * (kRxP + 2); q += kRxP * kRxY)
    (&sh[0][0][0])[q] = make_float2(0.f, 0.f);
  __syncthreads();
  const int j = (int)blockIdx.y * kRxTY - kRxK + ty, i0 = (int)blockIdx.x * kRxTX - kRxK + 2 * tx;
  const int a = j & 1;                       // colour 0 is the cell i0 + a
  float4 k[2];
  float wf[2][4], wF[2][4];
  float2 rr[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = i0 + (a ^ q);
    const bool in = i >= 0 && i < nx && j >= 0 && j < ny;
    const size_t c = in ? (size_t)j * nx + i : 0;
    const float2 z = make_float2(0.f, 0.f);
    k[q] = in ? K[c] : make_float4(0.f, 0.f, 0.f, 0.f);
    rr[q] = in ? r[c] : z;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      wf[q][m] = in ? W[(size_t)m * n + c] : 0.f;
      wF[q][m] = in ? W[(size_t)(4 + m) * n + c] : 0.f;
    }
    if (!first && in) sh[q][ty + 1][tx + 1] = e[c];
  }
  __syncthreads();
  auto update = [&](int q, int xl) {         // xl: pair of the left neighbour
    const float2 v[4] = {sh[q ^ 1][ty + 1][xl + 1], sh[q ^ 1][ty + 1][xl + 2],
                         sh[q ^ 1][ty][tx + 1], sh[q ^ 1][ty + 2][tx + 1]};
    float sf = rr[q].x, sF = rr[q].y;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      sf += wf[q][m] * v[m].x;
      sF += wF[q][m] * v[m].y;
    }
    sh[q][ty + 1][tx + 1] = make_float2(k[q].x * sf + k[q].y * sF, k[q].z * sf + k[q].w * sF);
  };
  for (int q = 0; q < colours; q += 2) {
    update(0, tx + a - 1);
    __syncthreads();
    update(1, tx - a);
    __syncthreads();
  }
  if (ty < kRxK || ty >= kRxK + kRxTY || j >= ny) return;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = i0 + (a ^ q), x = 2 * tx + (a ^ q);
    if (x < kRxK || x >= kRxK + kRxTX || i >= nx) continue;
    const size_t c = (size_t)j * nx + i;
    const float2 v = sh[q][ty + 1][tx + 1];
    if (last) {
      nf[c] += widen(v.x);
      nF[c] += widen(v.y);
    } else {
      eo[c] = v;
    }
  }
}

// lam0 = nu/dt and the four parameter terms, whose operators N^ are the
// table's weights read from the neighbours; nothing is written where the
// solve met a value that is not finite.  256^2: 35 -> 21 us, most of
// it the chains of the compensated sums.
__global__ void __launch_bounds__(kAdjThreads)
k_adj_finish2(int nx, int ny, const double* __restrict__ U, const double* __restrict__ f,
              const double* __restrict__ F, const double* __restrict__ nf,
              const double* __restrict__ nF, Ctl* ctl, double* __restrict__ lf,
              double* __restrict__ lF, double* part, double* out) {
  if (ctl->state == 3) return;
  const size_t n = (size_t)nx * ny;
  const double inv_dt = ctl->inv_dt;
  double s[4] = {0, 0, 0, 0}, e[4] = {0, 0, 0, 0};
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(c / (size_t)nx), i = (int)(c - (size_t)j * nx);
    const bool has[4] = {i > 0, i + 1 < nx, j > 0, j + 1 < ny};
    const size_t nb[4] = {c - 1, c + 1, c - nx, c + nx};
    const double xf = f[c], xF = F[c], vf = nf[c], vF = nF[c];
    double tf = U[c] * xf, tF = U[(size_t)U_F * n + c] * xF;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (!has[m]) continue;                 // the neighbour's weight towards c
      tf += U[(size_t)(1 + (m ^ 1)) * n + nb[m]] * f[nb[m]];
      tF += U[(size_t)(U_F + 1 + (m ^ 1)) * n + nb[m]] * F[nb[m]];
    }
    const double dv = vf - vF;
    const double t[4] = {dv * xF * U[(size_t)U_B * n + c], flip_if(dv * xf, true), vf * tf, vF * tF};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      double u, w;
      two_sum(s[m], t[m], u, w);
      s[m] = u;
      e[m] += w;
    }
    lf[c] = vf * inv_dt;
    lF[c] = vF * inv_dt;
  }
  // one warp per quantity, across the block and, in the last block, across
  // the blocks (in a fixed order; the four chains of FP64 additions one after
  // another took a third of the kernel)
  __shared__ double ss[4][kAdjThreads], se[4][kAdjThreads];
  __shared__ bool last;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    ss[m][threadIdx.x] = s[m];
    se[m][threadIdx.x] = e[m];
  }
  __syncthreads();
  double x = 0.0, y = 0.0;
  if (w < 4) {
    for (int q = lane; q < kAdjThreads; q += 32) {
      double u, v;
      two_sum(x, ss[w][q], u, v);
      x = u;
      y += se[w][q] + v;
    }
    warp_sum_comp(x, y);
    if (lane == 0) {
      const size_t o = 2 * ((size_t)w * gridDim.x + blockIdx.x);
      part[o] = x;
      part[o + 1] = y;
      __threadfence();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&ctl->blocks, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last || w >= 4) return;
  __threadfence();
  x = y = 0.0;
  for (int q = lane; q < (int)gridDim.x; q += 32) {
    const size_t o = 2 * ((size_t)w * gridDim.x + q);
    double u, v;
    two_sum(x, part[o], u, v);
    x = u;
    y += part[o + 1] + v;
  }
  warp_sum_comp(x, y);
  if (lane == 0) out[w] = x + y;
}

__global__ void k_f_from_gamma(size_t n, double inv_eps, const double* __restrict__ gamma,
                               const double* __restrict__ phi, double* __restrict__ f) {
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    const double p = phi[c];
    f[c] = gamma[c] * (p * (1.0 - p) * inv_eps);
  }
}

AdjP make_params(sfx_ctx* c, const sfx_params* pr, double dt) {
  AdjP p;
  p.L = c->lev[0].lv;
  p.Df = pr->Df;
  p.DF = pr->DF;
  p.inv_dt = 1.0 / dt;
  p.ka = pr->ka;
  p.kd = pr->kd;
  p.ginf = pr->gamma_inf;
  p.eps = pr->eps;
  p.eta = pr->eta;
  p.literal = pr->literal_upwind;
  const int nd = p.L.ndim();
  for (int d = 0; d < 3; ++d) {
    p.Bf[d] = d < nd ? c->adj.Bf[d] : nullptr;
    p.BF[d] = d < nd ? c->adj.BF[d] : nullptr;
  }
  return p;
}

sfx_status unit_drifts(sfx_ctx* c, const sfx_params* pr, const double* phi, cudaStream_t s) {
  return drift_faces64(c, phi, 1.0, 1.0, pr->eps, c->adj.Bf, c->adj.BF, s);
}

// The relaxation of one check as a graph, captured once per context and
// sweep count: every argument is context scratch, so it never goes stale.
// A colour sweep takes a few microseconds, and issuing the 2 S + 2 launches one
// by one left the step bound by the host.
sfx_status relax_graph(sfx_ctx* c, const Level& L, int sweeps) {
  if (c->adj.relax && c->adj.relax_sweeps == sweeps) return SFX_OK;
  if (c->adj.relax) {
    cudaGraphExecDestroy(c->adj.relax);
    c->adj.relax = nullptr;
  }
  if (!c->adj.cap) SFX_CUDA(cudaStreamCreateWithFlags(&c->adj.cap, cudaStreamNonBlocking));
  cudaStream_t cs = c->adj.cap;
  const size_t n = L.ncell();
  dim3 blk(128), grd((unsigned)(((L.nx + 1) / 2 + 127) / 128), (unsigned)L.ny, (unsigned)L.nz);
  SFX_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
  cudaMemsetAsync(c->adj.e, 0, n * sizeof(float2), cs);
  for (int q = 0; q < sweeps; ++q)
    for (int color = 0; color < 2; ++color)
      k_adj_csweep<<<grd, blk, 0, cs>>>(L, c->adj.K, c->adj.W, c->adj.r, c->adj.e, color);
  k_adj_add<<<blocks_for(n, kAdjThreads), kAdjThreads, 0, cs>>>(n, c->adj.e, c->adj.nf,
                                                                c->adj.nF);
  const cudaError_t le = cudaGetLastError();
  cudaGraph_t g = nullptr;
  const cudaError_t ce = cudaStreamEndCapture(cs, &g);
  cudaError_t ie = cudaSuccess;
  cudaGraphExec_t ex = nullptr;
  if (le == cudaSuccess && ce == cudaSuccess) ie = cudaGraphInstantiate(&ex, g, 0);
  if (g) cudaGraphDestroy(g);
  SFX_CUDA(le);
  SFX_CUDA(ce);
  SFX_CUDA(ie);
  c->adj.relax = ex;
  c->adj.relax_sweeps = sweeps;
  return SFX_OK;
}

// The 2D solve as a graph, captured once per context and sweep count (every
// argument is context scratch): a residual, then relaxation and residual
// again while the residual's last block asks for it.  One launch and one host
// wait per step; the checks one by one cost a host wait of some 12 us each.
sfx_status solve_graph2(sfx_ctx* c, const Level& L, int sweeps) {
  AdjScratch& A = c->adj;
  if (A.relax && A.relax_sweeps == sweeps) return SFX_OK;
  if (A.relax) {
    cudaGraphExecDestroy(A.relax);
    A.relax = nullptr;
  }
  for (cudaStream_t* q : {&A.cap, &A.cap_body})
    if (!*q) SFX_CUDA(cudaStreamCreateWithFlags(q, cudaStreamNonBlocking));
  const size_t n = L.ncell();
  const unsigned nb = (unsigned)((n + 255) / 256);
  const dim3 tiles((unsigned)((L.nx + kRxTX - 1) / kRxTX), (unsigned)((L.ny + kRxTY - 1) / kRxTY));
  Ctl* ctl = (Ctl*)A.ctl;
  cudaGraph_t g = nullptr;
  cudaGraphExec_t ex = nullptr;
  SFX_CUDA(cudaGraphCreate(&g, 0));
  auto capture = [&]() -> sfx_status {
    cudaGraphConditionalHandle loop;
    SFX_CUDA(cudaGraphConditionalHandleCreate(&loop, g, 0u, cudaGraphCondAssignDefault));
    auto resid = [&](cudaStream_t s) {
      k_adj_resid2<<<nb, 256, 0, s>>>(L.nx, L.ny, A.U, A.sig, A.dm, A.nf, A.nF, A.r, ctl, loop);
    };
    cudaGraph_t out = nullptr;
    SFX_CUDA(cudaStreamBeginCaptureToGraph(A.cap, g, nullptr, nullptr, 0,
                                           cudaStreamCaptureModeThreadLocal));
    resid(A.cap);
    cudaError_t le = cudaGetLastError();
    cudaStreamCaptureStatus cs;
    const cudaGraphNode_t* deps = nullptr;
    size_t ndeps = 0;
    cudaGraphNode_t after = nullptr;
    cudaError_t ce = cudaStreamGetCaptureInfo(A.cap, &cs, nullptr, nullptr, &deps, nullptr, &ndeps);
    if (ce == cudaSuccess && ndeps == 1) after = deps[0];
    const cudaError_t ee = cudaStreamEndCapture(A.cap, &out);
    SFX_CUDA(le);
    SFX_CUDA(ce);
    SFX_CUDA(ee);
    if (!after) return SFX_ERR_CUDA;
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = loop;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    SFX_CUDA(cudaGraphAddNode(&node, g, &after, nullptr, 1, &cp));
    SFX_CUDA(cudaStreamBeginCaptureToGraph(A.cap_body, cp.conditional.phGraph_out[0], nullptr,
                                           nullptr, 0, cudaStreamCaptureModeThreadLocal));
    float2 *e = A.e, *eo = A.e + n;
    for (int q = 0; q < 2 * sweeps; q += kRxK) {
      const int colours = std::min(kRxK, 2 * sweeps - q);
      k_adj_relax2<<<tiles, kRxP * kRxY, 0, A.cap_body>>>(L.nx, L.ny, A.K, A.W, A.r, e, eo, colours,
                                                          q == 0, q + colours == 2 * sweeps, A.nf,
                                                          A.nF);
      std::swap(e, eo);
    }
    resid(A.cap_body);
    le = cudaGetLastError();
    ce = cudaStreamEndCapture(A.cap_body, &out);
    SFX_CUDA(le);
    SFX_CUDA(ce);
    SFX_CUDA(cudaGraphInstantiate(&ex, g, 0));
    return SFX_OK;
  };
  const sfx_status st = capture();
  cudaGraphDestroy(g);
  if (st != SFX_OK) return st;
  A.relax = ex;
  A.relax_sweeps = sweeps;
  return SFX_OK;
}

// The step of a 2D grid (scratch and drift faces are in place).
sfx_status adjoint_step2(sfx_ctx* c, const AdjP& p, const double* phi, const double* f,
                         const double* F, double dt, double* lf, double* lF, double* dparams,
                         const sfx_solve_opts* o, sfx_step_stats* stats, cudaStream_t s) {
  AdjScratch& A = c->adj;
  const Level& L = p.L;
  const int sweeps = std::max(1, o->nu1 + o->nu2);
  Ctl* ctl = (Ctl*)A.ctl;
  sfx_status st = solve_graph2(c, L, sweeps);
  if (st != SFX_OK) return st;
  const dim3 cg((unsigned)((L.nx + 31) / 32), (unsigned)std::min((L.ny + 7) / 8, 65535));
  SFX_KERNEL(c, K_SETUP, k_adj_coef2, cg, 256, s, p, 1.0 / L.h, 1.0 / p.eps, phi, f, F, lf, lF,
             dt, o->tol, o->max_cycles, A.U, A.K, A.W, A.nf, A.nF, A.sig, A.dm, ctl);
  if (o->max_cycles > 0) {   // the profile times the solve as a whole
    prof_before(c, K_SMOOTH_FINE, s);
    SFX_CUDA(cudaGraphLaunch(A.relax, s));
    prof_after(c, K_SMOOTH_FINE, s);
  }
  SFX_KERNEL(c, K_OTHER, k_adj_finish2, std::min(A.nblk, 2 * c->sm_count), kAdjThreads, s, L.nx, L.ny,
             A.U, f, F, A.nf, A.nF, ctl, lf, lF, A.part, A.d_out);
  SFX_LAUNCH_CHECK();
  SFX_CUDA(cudaMemcpyAsync(A.h_out, A.d_out, 4 * sizeof(double), cudaMemcpyDeviceToHost, s));
  SFX_CUDA(cudaMemcpyAsync(A.h_ctl, ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
  SFX_CUDA(cudaStreamSynchronize(s));
  const Ctl& h = *(const Ctl*)A.h_ctl;
  const int launches = (2 * sweeps + kRxK - 1) / kRxK, relaxed = std::max(h.checks - 1, 0);
  c->prof.launches[K_RESIDUAL] += h.checks;
  c->prof.launches[K_SMOOTH_FINE] += launches * relaxed - (o->max_cycles > 0 ? 1 : 0);
  if (h.state == 3) return SFX_ERR_NONFINITE;
  const bool conv = h.state == 1;
  if (dparams)
    for (int m = 0; m < 4; ++m) dparams[m] += A.h_out[m];
  if (stats) {
    stats->picard = h.checks;
    stats->vcycles = relaxed * sweeps;
    stats->res_f = h.rel;
    stats->res_F = h.rel;
    stats->mass_f = 0.0;
    stats->mass_F = 0.0;
    stats->converged = conv ? 1 : 0;
  }
  return conv ? SFX_OK : SFX_ERR_NOT_CONVERGED;
}

}  // namespace

sfx_status adj_ensure_scratch(sfx_ctx* c) {
  if (c->adj.ready) return SFX_OK;
  const Level& L = c->lev[0].lv;
  const size_t n = L.ncell();
  auto get = [&](size_t bytes, void** p) -> sfx_status {
    SFX_CUDA(cudaMalloc(p, bytes ? bytes : 8));
    c->allocations.push_back(*p);
    return SFX_OK;
  };
  sfx_status st;
  for (int d = 0; d < L.ndim(); ++d) {
    if ((st = get(L.nface(d) * sizeof(double), (void**)&c->adj.Bf[d])) != SFX_OK) return st;
    if ((st = get(L.nface(d) * sizeof(double), (void**)&c->adj.BF[d])) != SFX_OK) return st;
  }
  double** cells[4] = {&c->adj.nf, &c->adj.nF, &c->adj.sig, &c->adj.dm};
  for (double** q : cells)
    if ((st = get(n * sizeof(double), (void**)q)) != SFX_OK) return st;
  const bool flat = L.ndim() == 2;
  // force and G of the loss; a 2D solve keeps its table there
  if ((st = get((flat ? U_ROWS : 6) * n * sizeof(double), (void**)&c->adj.force)) != SFX_OK)
    return st;
  c->adj.G = c->adj.force + L.ndim() * n;
  c->adj.U = flat ? c->adj.force : nullptr;
  c->adj.nblk = std::min(blocks_for(n, kAdjThreads), 1024);
  if ((st = get((size_t)c->adj.nblk * 2 * 5 * sizeof(double), (void**)&c->adj.part)) != SFX_OK)
    return st;
  if ((st = get(8 * sizeof(double), (void**)&c->adj.d_out)) != SFX_OK) return st;
  if ((st = get(2 * sizeof(unsigned long long), (void**)&c->adj.d_nrm)) != SFX_OK) return st;
  if ((st = get(n * sizeof(float4), (void**)&c->adj.K)) != SFX_OK) return st;
  if ((st = get((flat ? 8 : 12) * n * sizeof(float), (void**)&c->adj.W)) != SFX_OK) return st;
  if ((st = get(n * sizeof(float2), (void**)&c->adj.r)) != SFX_OK) return st;
  if ((st = get((flat ? 2 : 1) * n * sizeof(float2), (void**)&c->adj.e)) != SFX_OK) return st;
  if ((st = get(sizeof(Ctl), &c->adj.ctl)) != SFX_OK) return st;
  SFX_CUDA(cudaMallocHost((void**)&c->adj.h_out, 8 * sizeof(double)));
  SFX_CUDA(cudaMallocHost((void**)&c->adj.h_nrm, 2 * sizeof(unsigned long long)));
  SFX_CUDA(cudaMallocHost(&c->adj.h_ctl, sizeof(Ctl)));
  c->adj.ready = true;
  return SFX_OK;
}

sfx_status f_from_gamma(sfx_ctx* c, const double* gamma, const double* phi, double eps,
                        double* f, cudaStream_t s) {
  const size_t n = c->lev[0].lv.ncell();
  SFX_KERNEL(c, K_OTHER, k_f_from_gamma, blocks_for(n, 256), 256, s, n, 1.0 / eps, gamma, phi, f);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

sfx_status adjoint_apply(sfx_ctx* c, const sfx_params* pr, const double* phi, const double* f,
                         const double* F, double dt, int transpose, const double* vf,
                         const double* vF, double* of, double* oF, cudaStream_t s) {
  sfx_status st = adj_ensure_scratch(c);
  if (st != SFX_OK) return st;
  if ((st = unit_drifts(c, pr, phi, s)) != SFX_OK) return st;
  const AdjP p = make_params(c, pr, dt);
  const size_t n = p.L.ncell();
  SFX_KERNEL(c, K_OTHER, k_adj_apply, blocks_for(n, 256), 256, s, p, phi, f, F, vf, vF,
             transpose, of, oF);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

sfx_status adjoint_step(sfx_ctx* c, const sfx_params* pr, const double* phi, const double* f,
                        const double* F, double dt, double* lf, double* lF, double* dparams,
                        const sfx_solve_opts* o, sfx_step_stats* stats, cudaStream_t s) {
  sfx_status st = adj_ensure_scratch(c);
  if (st != SFX_OK) return st;
  if ((st = unit_drifts(c, pr, phi, s)) != SFX_OK) return st;
  const AdjP p = make_params(c, pr, dt);
  const Level& L = p.L;
  if (L.ndim() == 2) return adjoint_step2(c, p, phi, f, F, dt, lf, lF, dparams, o, stats, s);
  const size_t n = L.ncell();
  const int nb = blocks_for(n, kAdjThreads);
  double* nf = c->adj.nf;
  double* nF = c->adj.nF;
  SFX_KERNEL(c, K_SETUP, k_adj_init, nb, kAdjThreads, s, n, dt, lf, lF, nf, nF);
  SFX_KERNEL(c, K_SETUP, k_adj_coef, nb, kAdjThreads, s, p, phi, f, F, c->adj.K, c->adj.W);
  const int sweeps = std::max(1, o->nu1 + o->nu2);
  if ((st = relax_graph(c, L, sweeps)) != SFX_OK) return st;
  bool conv = false;
  double rel = INFINITY;
  int checks = 0, total_sweeps = 0;
  for (checks = 1; checks <= o->max_cycles; ++checks) {
    // FP64 residual of the current nu: the convergence test and the defect
    SFX_CUDA(cudaMemsetAsync(c->adj.d_nrm, 0, 2 * sizeof(unsigned long long), s));
    SFX_KERNEL(c, K_RESIDUAL, k_adj_resid, nb, kAdjThreads, s, p, phi, f, F, lf, lF, nf, nF,
               c->adj.r, c->adj.d_nrm);
    SFX_LAUNCH_CHECK();
    SFX_CUDA(cudaMemcpyAsync(c->adj.h_nrm, c->adj.d_nrm, 2 * sizeof(unsigned long long),
                             cudaMemcpyDeviceToHost, s));
    SFX_CUDA(cudaStreamSynchronize(s));
    double r, b;
    memcpy(&r, &c->adj.h_nrm[0], sizeof(double));
    memcpy(&b, &c->adj.h_nrm[1], sizeof(double));
    if (!std::isfinite(r)) return SFX_ERR_NONFINITE;
    rel = r / (b > 1e-300 ? b : 1e-300);
    if (b == 0.0 || rel <= o->tol) {
      conv = true;
      break;
    }
    if (checks == o->max_cycles) break;
    // FP32 relaxation of the defect equation from e = 0, then nu += e (one
    // graph launch; the profile counts its kernels and times it as a whole)
    prof_before(c, K_SMOOTH_FINE, s);
    SFX_CUDA(cudaGraphLaunch(c->adj.relax, s));
    prof_after(c, K_SMOOTH_FINE, s);
    c->prof.launches[K_SMOOTH_FINE] += 2 * sweeps - 1;
    c->prof.launches[K_OTHER] += 1;
    total_sweeps += sweeps;
  }
  const int nbf = c->adj.nblk;
  SFX_KERNEL(c, K_OTHER, k_adj_finish, nbf, kAdjThreads, s, p, phi, f, F, nf, nF, lf, lF,
             c->adj.part);
  SFX_KERNEL(c, K_OTHER, k_adj_reduce, 4, kAdjThreads, s, c->adj.part, nbf, c->adj.d_out);
  SFX_LAUNCH_CHECK();
  SFX_CUDA(cudaMemcpyAsync(c->adj.h_out, c->adj.d_out, 4 * sizeof(double),
                           cudaMemcpyDeviceToHost, s));
  SFX_CUDA(cudaStreamSynchronize(s));
  if (dparams)
    for (int m = 0; m < 4; ++m) dparams[m] += c->adj.h_out[m];
  if (stats) {
    stats->picard = std::min(checks, o->max_cycles);
    stats->vcycles = total_sweeps;
    stats->res_f = rel;
    stats->res_F = rel;
    stats->mass_f = 0.0;
    stats->mass_F = 0.0;
    stats->converged = conv ? 1 : 0;
  }
  return conv ? SFX_OK : SFX_ERR_NOT_CONVERGED;
}

}  // namespace sfx
