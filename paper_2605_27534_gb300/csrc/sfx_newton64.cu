// Coupled Newton defect correction of the App. C system in FP64 contexts.
//
// The system is the one of sfx_solver.cu (FP64 operator, FP64 residual test
// on |b - L(a)|_inf/|b|_inf).  Each iteration evaluates both residuals in
// FP64 at the current state with the pointwise 2x2 Jacobian of the exchange,
// relaxes the correction by FP32 red-black sweeps (the cell of the SFX_F32
// solver: sfx_f32_dev.cuh, face drifts in half precision) and adds it to the
// FP64 state.  The FP32 part only preconditions: the state and every
// residual stay FP64, and the error of the result is that of the FP64
// residual.  After an iteration passes the test its correction is still
// relaxed and added, so the returned state is one Newton step beyond the
// tested one.
//
// What bounds it: the FP64 pipe issues 1/59 of the FP32 rate, so the
// colour sweeps and V-cycles of the Picard solver in FP64 took 90 % of a
// step; one residual is about 50 FP64 instructions per cell for both
// fields.  On small grids the launches bound it: an iteration is the
// residual (which also does the first red half-sweep, the convergence test
// in its last block and the report to the host) and 2S - 1 colour launches.
//
// Measured against the Picard solver (4 iterations of one V-cycle per field):
// a 128^2 no-flow step with its force 5.4 -> 0.14 ms, 131 x 257 axisymmetric
// (odd: one level, 40 coarse sweeps) 5.7 -> 0.17 ms, a 96^3 step 19.2 -> 1.15 ms
// (residual 71 us for 0.88 M cells: 46 FP64 instructions per cell, the pipe 76 %
// busy; Picard's was 370 us); the error against a 64-bit solution
// falls from 1e-11 to 5e-14 at tol = 1e-10.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sfx_block2d.cuh"
#include "sfx_f32_dev.cuh"
#include "sfx_internal.h"

namespace sfx {
namespace {

// ------------------------------------------------------------------ setup
// Drift faces of both fields (App. C, as described in sfx_solver.cu) on the
// minus sides of a block's cells, from unit normals formed once per cell in
// shared memory (the block's cells and one layer on the minus sides; a face
// per thread and direction took two normals per face).  Where phi is flat
// bit for bit the normal is zero and costs no FP64 arithmetic; in 3D a warp is
// a box of 8 x 2 x 2 cells, fewer of which touch the band of phi than rows of
// 32 do (96^3: 98 -> 90 us, 65 x 70 x 60: 60 -> 44; FP64 pipe 76 % busy).
// Optional outputs: H2 the faces in half precision, c1 = r_a/(phi + eta) and
// finf = Gamma_inf phi (1 - phi)/eps per cell, and what a solve starts with
// (a memory operation and two copies of their own took 10 us of a 128^2 step).
constexpr int kSX = 32, kSY = 4;
constexpr int kCtlWords = 8;   // of Ctl64

struct Setup64 {
  Level L;
  const double* phi;
  double Df, DF, eps, ka, eta, ginf;
  double* Bf[3];
  double* BF[3];
  __half2* H[3];
  double* c1;
  double* finf;
  // the start of a solve: its control words cleared, x* = x without a flow
  int* ctl;
  const double* x[2];
  double* xs[2];
};

__device__ __forceinline__ bool bits_eq(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}

template <int ND>
__device__ __forceinline__ void unit_normal(const Level& L, const double* __restrict__ phi,
                                            const int* x, double inv2h, double inv_eps, double* n) {
  const size_t st[3] = {1, (size_t)L.nx, (size_t)L.nx * L.ny};
  const size_t c = cidx(L, x[0], x[1], x[2]);
  const double pc = phi[c];
  double a[ND], b[ND];
  bool flat = finite_bits(pc);
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    a[d] = phi[x[d] + 1 < L.extent(d) ? c + st[d] : c];
    b[d] = phi[x[d] > 0 ? c - st[d] : c];
    flat &= bits_eq(a[d], b[d]);
    n[d] = 0.0;
  }
  if (flat) return;
  if (!finite_bits(pc)) {   // the drift of its faces, a multiple of phi, is not a number
#pragma unroll
    for (int d = 0; d < ND; ++d) n[d] = pc - pc;
    return;
  }
  double m2 = 0.0;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    a[d] = (a[d] - b[d]) * inv2h;
    m2 = fma(a[d], a[d], m2);
  }
  const double m = sqrt(m2);
  const double slope = kNormalKappa * (pc * (1.0 - pc) * inv_eps);
  // phi outside [0, 1], and -0, has no profile slope: no direction either
  if (m < 1e-30 || __double_as_longlong(slope) < 0 || !(m > slope)) return;
  const double w = m >= 2.0 * slope ? 1.0 : m / slope - 1.0;
  const double s = w / m;
#pragma unroll
  for (int d = 0; d < ND; ++d) n[d] = a[d] * s;
}

template <int ND>
__global__ void __launch_bounds__(kSX * kSY * (ND == 3 ? 4 : 1)) k_setup64(Setup64 q, unsigned yb, unsigned zb) {
  constexpr int BZ = ND == 3 ? 4 : 1;
  constexpr int HX = kSX + 1, HY = kSY + 1, HZ = ND == 3 ? BZ + 1 : 1;
  __shared__ double sn[ND][HZ][HY][HX];
  const Level& L = q.L;
  const int x0 = blockIdx.x * kSX, y0 = (int)(yb + blockIdx.y) * kSY,
            z0 = (int)(zb + blockIdx.z) * BZ;
  if (q.ctl && (x0 | y0 | z0) == 0 && threadIdx.x < kCtlWords)
    q.ctl[threadIdx.x] = 0;
  const double inv2h = 0.5 / L.h, inv_eps = 1.0 / q.eps;
  // the normal of the cell (lx, ly, lz) of the block's box with its minus layers
  auto normal = [&](int lx, int ly, int lz) {
    const int x[3] = {x0 + lx - 1, y0 + ly - 1, ND == 3 ? z0 + lz - 1 : 0};
    double n[ND] = {};
    if (x[0] >= 0 && x[0] < L.nx && x[1] >= 0 && x[1] < L.ny && x[2] >= 0 && x[2] < L.nz)
      unit_normal<ND>(L, q.phi, x, inv2h, inv_eps, n);
#pragma unroll
    for (int d = 0; d < ND; ++d) sn[d][lz][ly][lx] = n[d];
  };
  int lx = threadIdx.x % kSX, ly = threadIdx.x / kSX % kSY, lz = threadIdx.x / (kSX * kSY);
  if (ND == 3) {
    const int3 l = CellBlock<3>::cell(threadIdx.x);
    lx = l.x, ly = l.y, lz = l.z;
    normal(lx + 1, ly + 1, lz + 1);
    const int t = threadIdx.x;
    if (t < kSX * kSY) normal(1 + t % kSX, 1 + t / kSX, 0);
    else if (t < kSX * (kSY + BZ + 1)) normal(1 + t % kSX, 0, t / kSX - kSY);
    else if (t < kSX * (kSY + BZ + 1) + HY * HZ) {
      const int e = t - kSX * (kSY + BZ + 1);
      normal(0, e % HY, e / HY);
    }
  } else {
    for (int t = threadIdx.x; t < HX * HY; t += blockDim.x) normal(t % HX, t / HX, 0);
  }
  __syncthreads();
  const int x[3] = {x0 + lx, y0 + ly, z0 + lz};
  if (x[0] >= L.nx || x[1] >= L.ny || x[2] >= L.nz) return;
  const size_t st[3] = {1, (size_t)L.nx, (size_t)L.nx * L.ny};
  const size_t c = cidx(L, x[0], x[1], x[2]);
  const double p = q.phi[c];
  const double kf = -q.Df * inv_eps, kF = -0.5 * q.DF * inv_eps;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const size_t f = fidx(L, d, x[0], x[1], x[2]);
    double bf = 0.0, bF = 0.0;
    if (x[d] > 0) {
      const int hz = ND == 3 ? lz + 1 : 0;
      const double nR = sn[d][hz][ly + 1][lx + 1];
      const double nL = sn[d][hz - (ND == 3 && d == 2)][ly + 1 - (d == 1)][lx + 1 - (d == 0)];
      if (!bits_eq(nR, 0.0) || !bits_eq(nL, 0.0)) {
        const double pL = q.phi[c - st[d]];
        bf = kf * ((0.5 - pL) * nL + (0.5 - p) * nR);
        bF = kF * ((1.0 - pL) * nL + (1.0 - p) * nR);
      }
    }
    q.Bf[d][f] = bf;
    q.BF[d][f] = bF;
    if (q.H[d]) q.H[d][f] = __floats2half2_rn((float)bf, (float)bF);
    if (x[d] + 1 == L.extent(d)) {   // the far wall's face
      const int y[3] = {x[0] + (d == 0), x[1] + (d == 1), x[2] + (d == 2)};
      const size_t w = fidx(L, d, y[0], y[1], y[2]);
      q.Bf[d][w] = q.BF[d][w] = 0.0;
      if (q.H[d]) q.H[d][w] = __floats2half2_rn(0.0f, 0.0f);
    }
  }
  if (q.c1) {
    q.c1[c] = q.ka / (p + q.eta);
    q.finf[c] = q.ginf * (p * (1.0 - p)) * inv_eps;
  }
  if (q.xs[0]) {
    q.xs[0][c] = q.x[0][c];
    q.xs[1][c] = q.x[1][c];
  }
}

// --------------------------------------------------------------- residual
struct Newton64 {
  Nw32 p;             // FP32 coefficients of the correction
  double Doh[2];      // D/h of f, F
  double invh, inv_dt, kd;
  const double* Bf[3];
  const double* BF[3];
  const __half2* H[3];
  const double* c1;
  const double* finf;
  const double* fs;   // f*, F*
  const double* Fs;
  float4* rc;
  float2* e2;
};

// Control words of a solve (device): the norms of an iteration, the blocks
// that have reported, and the state of the test.
struct Ctl64 {
  unsigned int nrm[4];   // |r_f|, |b_f|, |r_F|, |b_F| as float bits
  unsigned int blocks;
  int done;              // an iteration has passed: no further residuals
  int stop;              // its correction has been added: no further sweeps
  int iter;              // iterations evaluated
};
static_assert(sizeof(Ctl64) == kCtlWords * sizeof(int), "control words");

// (1/h) sum of +-G over the cell's faces of one field, G = D (a_R - a_L)/h
// + B a_up.  The diffusive part is gathered as D/h (sum of neighbours -
// count a); the drift part takes the sign of B from its integer word (a
// zero drift adds zero whichever side is taken).  Axisymmetric faces are
// weighted with the face area over V/h: 1 on axial faces, w[0], w[1] on the
// radial ones.
template <int G>
__device__ __forceinline__ double flux64(const Newton64& q, double Doh, const double* B,
                                         const double* nb, double a,
                                         const double* w) {
  constexpr int NQ = G == SFX_CART3D ? 6 : 4;
  const bool lit = q.p.literal != 0;
  double S = 0.0, T = 0.0, W = 0.0;
#pragma unroll
  for (int k = 0; k < NQ; ++k) {
    const bool plus = k & 1;
    const bool neg = __double_as_longlong(B[k]) < 0;
    const bool left = neg != lit;            // the upwind cell is the left one
    const double up = plus == left ? a : nb[k];   // this cell is left on plus faces
    if (G == SFX_AXISYM && k < 2) {
      S = fma(w[k], nb[k], S);
      W += w[k];
      const double bw = B[k] * w[k];
      T = plus ? fma(bw, up, T) : fma(-bw, up, T);
    } else {
      S += nb[k];                             // the cell itself past a wall
      T = plus ? fma(B[k], up, T) : fma(-B[k], up, T);
    }
  }
  const double cnt = G == SFX_AXISYM ? W + 2.0 : (double)NQ;
  return fma(Doh, fma(-cnt, a, S), T) * q.invh;
}

// What a cell of f* or F* adds to the norm of the right-hand side at least: a
// field that is not zero but vanishes in float has a norm below the host's
// range, not one of 0, which its residual of 0 would pass.
__device__ __forceinline__ float nonzero_norm(double x) {
  return (((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x)) != 0u ? 1e-30f : 0.0f;
}

// The system may have several solutions.  The exchange is bilinear, so the
// difference (df, dF) of two solutions solves the linearised system at their
// mean, with U = u + r_d and v there; its columns are dominated by their
// diagonals by 1/dt - 2 max(0, -U) and 1/dt - 2 max(0, -v), so where both stay
// above -1/(2 dt) there is one.  Pointwise the exchange leaves a quadratic in
// F whose roots have opposite signs wherever f* and F* are not negative; the
// physical one, F >= 0, is where its slope 1/dt + U + v is positive.  Newton
// is kept to iterates with U > -0.45/dt (F not below zero where phi is
// small), v > -0.98/dt (f above Gamma_inf delta in the tails of phi reaches
// -0.9/dt in the transient of an adsorption run; at -1/dt the F problem loses
// its diagonal) and a positive slope; any other is left to the Picard
// solver, so that a step does not change branch.
//
// Both residuals at every cell, rc = (r_f, r_F, u, v) and the first red
// half-sweep of the correction (e = M^-1 r from zero), the norms, and in
// the last block to finish the convergence test and its report to the host.
template <int G>
__global__ void __launch_bounds__(256)
k_resid64(Newton64 q, const double* __restrict__ f, const double* __restrict__ F, float tol,
          Ctl64* __restrict__ ctl, volatile unsigned int* report) {
  constexpr int NQ = G == SFX_CART3D ? 6 : 4;
  if (ctl->done) {
    // every block sees done (set by an earlier launch); the sweeps behind
    // this launch return too
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->stop = 1;
    return;
  }
  const Level& L = q.p.L;
  float m[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const ix cells = (ix)L.ncell();
  for (ix c = blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += gridDim.x * blockDim.x) {
    const ix r = c / (ix)L.nx;
    const int i = (int)(c - r * (ix)L.nx), j = (int)(r % (ix)L.ny), k = (int)(r / (ix)L.ny);
    double w[2] = {1.0, 1.0};
    if (G == SFX_AXISYM) {
      const double iv = 1.0 / (double)(2 * i + 1);
      w[0] = (double)(2 * i) * iv;
      w[1] = i + 1 < L.nx ? (double)(2 * i + 2) * iv : 0.0;
    }
    bool has[6];
    ix nbi[6];
    gather6<G>(L, i, j, k, c, has, nbi);
    const double fc = f[c], Fc = F[c];
    const ix fx = c + (ix)k * (ix)L.ny + (ix)j, fy = c + (ix)k * (ix)L.nx;
    const ix fi[6] = {fx, fx + 1, fy, fy + (ix)L.nx, c, c + (ix)L.nx * (ix)L.ny};
    double nf[NQ], nF[NQ], Bf[NQ], BF[NQ];
#pragma unroll
    for (int s = 0; s < NQ; ++s) {
      nf[s] = has[s] ? f[nbi[s]] : fc;
      nF[s] = has[s] ? F[nbi[s]] : Fc;
      Bf[s] = q.Bf[s / 2][fi[s]];        // zero on walls
      BF[s] = q.BF[s / 2][fi[s]];
    }
    const double flf = flux64<G>(q, q.Doh[0], Bf, nf, fc, w);
    const double flF = flux64<G>(q, q.Doh[1], BF, nF, Fc, w);
    const double c1 = q.c1[c], finf = q.finf[c], fst = q.fs[c], Fst = q.Fs[c];
    const double vd = c1 * (finf - fc);
    const double ex = fma(vd, Fc, -(q.kd * fc));     // c1 F (f_inf - f) - r_d f
    const double rfd = fma(fst - fc, q.inv_dt, flf) + ex;
    const double rFd = fma(Fst - Fc, q.inv_dt, flF) - ex;
    const float rf = (float)rfd, rF = (float)rFd;
    const float u = __fmul_rn((float)c1, (float)Fc), v = (float)vd;
    const RBIdx rb = rb_index(L, i, j, k);
    const int col = (i + j + k) & 1;
    const ix own = (ix)col * rb.plane + rb.pos;
    q.rc[own] = make_float4(rf, rF, u, v);
    if (col == 0) {
      float Hf[6], HF[6];
      faces6x2(L, q.H[0], q.H[1], q.H[2], i, j, k, has, Hf, HF);
      float2 B[6], z[6], dg;
#pragma unroll
      for (int s = 0; s < 6; ++s) {
        B[s] = make_float2(Hf[s], HF[s]);
        z[s] = v_bc(0.0f);
      }
      flux_lin2<G>(L, q.p.invh, make_float2(q.p.Dfh, q.p.DFh), q.p.literal, i, v_bc(0.0f), z, has,
                   B, dg);
      const Jac2 J = jac2(q.p, u, v);
      const float a = __fadd_rn(J.ff, dg.x), e = __fadd_rn(J.FF, dg.y);
      const float inv = __fdividef(1.0f, __fmaf_rn(a, e, -__fmul_rn(J.fF, J.Ff)));
      q.e2[own] = make_float2(__fmul_rn(__fmaf_rn(e, rf, __fmul_rn(J.fF, rF)), inv),
                              __fmul_rn(__fmaf_rn(J.Ff, rf, __fmul_rn(a, rF)), inv));
    }
    const float idt = (float)q.inv_dt;
    m[0] = fmaxf(m[0], fabsf(rf));
    m[1] = fmaxf(m[1], fabsf(__fmaf_rn((float)fst, idt, __fmul_rn(u, (float)finf))));
    m[1] = fmaxf(m[1], nonzero_norm(fst));
    m[2] = fmaxf(m[2], fabsf(rF));
    m[3] = fmaxf(m[3], fabsf(__fmaf_rn((float)Fst, idt, __fmul_rn((float)q.kd, (float)fc))));
    m[3] = fmaxf(m[3], nonzero_norm(Fst));
    // off the branch (above): as a non-finite norm
    const float U = __fadd_rn(u, (float)q.kd);
    if (!(fabsf(rf) <= 3.0e38f) || !(fabsf(rF) <= 3.0e38f) || U < -0.45f * idt ||
        v < -0.98f * idt || __fadd_rn(U, v) < -0.98f * idt)
      m[0] = m[2] = __int_as_float(0x7f800000);
  }
  resid_norms(m, ctl->nrm);
  // the last block to get here tests and reports
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0)
    last = atomicAdd(&ctl->blocks, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last || threadIdx.x != 0) return;
  __threadfence();
  unsigned int n[4];
  for (int s = 0; s < 4; ++s) {
    n[s] = atomicExch(&ctl->nrm[s], 0u);
    report[s] = n[s];
  }
  ctl->blocks = 0;
  const bool ok = __uint_as_float(n[0]) <= tol * __uint_as_float(n[1]) &&
                  __uint_as_float(n[2]) <= tol * __uint_as_float(n[3]);
  report[4] = ok ? 1u : 0u;
  if (ok) ctl->done = 1;
  __threadfence_system();
}

// The correction of a cell as it is added to the state: after a passed test
// none that is not finite (the sweeps overflow float where 1/dt is beyond
// 1e19; no residual follows that would see it).
__device__ __forceinline__ float2 added(float2 e, const Ctl64* __restrict__ ctl) {
  if (finite_bits(e.x) && finite_bits(e.y)) return e;
  return ctl->done ? make_float2(0.0f, 0.0f) : e;
}

// One colour of the correction sweep (corr2_load, corr2_apply); the last
// black colour of an iteration (fst not null) adds the corrections of the
// cell and of the red cell that shares its pair to the FP64 state.
template <int G>
__global__ void __launch_bounds__(128)
k_corr64(Nw32 p, const __half2* __restrict__ Hx, const __half2* __restrict__ Hy,
         const __half2* __restrict__ Hz, const float4* __restrict__ rc, float2* __restrict__ e2,
         int color, int first, double* fst, double* Fst, const double* fsrc, const double* Fsrc,
         const Ctl64* __restrict__ ctl) {
  if (ctl->stop) return;
  const Level& L = p.L;
  const int j = blockIdx.y, k = blockIdx.z;
  const __half2* H[3] = {Hx, Hy, Hz};
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + ((j + k + color) & 1);
  const bool in = i < L.nx;
  Corr2In a;
  if (in) {
    corr2_load<G>(p, i, j, k, H, rc, e2, color, first, a);
    corr2_apply<G>(p, a, e2, nullptr, nullptr, nullptr, nullptr);
  }
  if (!fst) return;
  const RBIdx rb = rb_index(L, i, j, k);
  if (in) {
    const float2 e = added(e2[a.own], ctl);
    fst[a.c] = fsrc[a.c] + (double)e.x;
    Fst[a.c] = Fsrc[a.c] + (double)e.y;
  }
  const int ir = i ^ 1;     // the pair's red cell (also of a row's odd tail)
  if (ir < L.nx) {
    const ix cr = cidx32(L, ir, j, k);
    const float2 e = added(e2[(ix)(1 - color) * rb.plane + rb.pos], ctl);
    fst[cr] = fsrc[cr] + (double)e.x;
    Fst[cr] = Fsrc[cr] + (double)e.y;
  }
}

// All sweeps of an iteration on 2D tiles (sfx_block2d.cuh).
template <int G>
__global__ void __launch_bounds__(kT2Threads)
k_corr64_tile2d(Nw32 p, int tx, int ty, int sweeps, const __half2* __restrict__ Hx,
                const __half2* __restrict__ Hy, const float4* __restrict__ rc,
                const float2* __restrict__ e2, double* fst, double* Fst, const double* fsrc,
                const double* Fsrc, const Ctl64* __restrict__ ctl) {
  if (ctl->stop) return;
  corr_tile2d<G>(p, blockIdx.x * tx, blockIdx.y * ty, tx, ty, sweeps, Hx, Hy, rc, e2,
                 [&](ix c, float2 e) {
                   e = added(e, ctl);
                   fst[c] = fsrc[c] + widen(e.x);
                   Fst[c] = Fsrc[c] + widen(e.y);
                 });
}

// Launch shape of the residual: cells in turn (rows of warps left the lanes
// past a row's end idle while the FP64 pipe took their slots: 65 x 70 x 60
// 36 -> 26 us, 300 x 400 16.2 -> 12.7, 96^3 73.4 -> 71.3), blocks of 256
// threads, eight per SM; of 128 where that is less than one cell per thread,
// to even out over the SMs.
struct Shape {
  unsigned grid, block;
};
Shape shape_of(const Level& L, int sms) {
  const size_t n = L.ncell();
  const unsigned block = n >= (size_t)sms * 2048 ? 256 : 128;
  return {(unsigned)std::min((n + block - 1) / block, (size_t)sms * 2048 / block), block};
}

sfx_status ensure(sfx_ctx* c) {
  N64Scratch& S = c->n64;
  if (S.ready) return SFX_OK;
  const Level& L = c->lev[0].lv;
  const size_t np = 2 * (size_t)L.ny * L.nz * ((L.nx + 1) / 2);
  auto get = [&](size_t bytes, void** p) -> sfx_status {
    if (*p) return SFX_OK;
    void* m = nullptr;
    SFX_CUDA(cudaMalloc(&m, bytes));
    c->allocations.push_back(*p = m);
    return SFX_OK;
  };
  sfx_status st;
  for (int d = 0; d < L.ndim(); ++d)
    if ((st = get(L.nface(d) * sizeof(__half2), (void**)&S.H[d])) != SFX_OK) return st;
  if ((st = get(np * sizeof(float2), (void**)&S.e2)) != SFX_OK) return st;
  if ((st = get(np * sizeof(float4), (void**)&S.rc)) != SFX_OK) return st;
  if ((st = get(sizeof(Ctl64), (void**)&S.ctl)) != SFX_OK) return st;
  if (!S.report) {
    SFX_CUDA(cudaHostAlloc((void**)&S.report, 2 * 8 * sizeof(unsigned int), cudaHostAllocMapped));
  }
  for (int q = 0; q < 2; ++q)
    if (!S.ev[q]) SFX_CUDA(cudaEventCreateWithFlags(&S.ev[q], cudaEventDisableTiming));
  S.ready = true;
  return SFX_OK;
}

template <int ND>
void launch_setup(sfx_ctx* c, const Setup64& q, cudaStream_t s) {
  const Level& L = q.L;
  constexpr int BZ = ND == 3 ? 4 : 1;
  grid_parts((unsigned)((L.nx + kSX - 1) / kSX), (unsigned)((L.ny + kSY - 1) / kSY),
             (unsigned)((L.nz + BZ - 1) / BZ), [&](dim3 g, unsigned yb, unsigned zb) {
               SFX_KERNEL(c, K_SETUP, k_setup64<ND>, g, kSX * kSY * BZ, s, q, yb, zb);
             });
}

constexpr double kHalfMax = 65504.0;   // the largest half

// Iterations after which a solve that still converges slowly is handed to
// the Picard solver.
constexpr int kMaxNewton = 30;

template <int G>
sfx_status solve(sfx_ctx* c, const Newton64& q, double* f, double* F, bool from_star,
                 const sfx_solve_opts* o, int* iters, double* rel, bool* conv, cudaStream_t s) {
  const Level& L = q.p.L;
  N64Scratch& S = c->n64;
  Ctl64* ctl = (Ctl64*)S.ctl;
  const int sweeps = std::max(1, o->nu1 + o->nu2);
  const float tol = (float)o->tol;
  const Shape rg = shape_of(L, c->sm_count);
  const dim3 blk(128), grd((unsigned)(((L.nx + 1) / 2 + 127) / 128), (unsigned)L.ny, (unsigned)L.nz);
  const int cap = std::min(o->max_cycles, kMaxNewton);
  Tile2D t2;
  size_t t2smem = 0;
  if (G != SFX_CART3D && (t2.ty = tile2d_rows(&L, 1, sweeps, c->sm_count)) > 0) {
    t2 = tile2d_of(L.nx, t2.ty, sweeps);
    t2smem = tile2d_smem(L.nx, L.ny, t2, sweeps);
    SFX_CUDA(cudaFuncSetAttribute(k_corr64_tile2d<G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)kT2Smem));
  }
  *conv = false;
  float first = 0.0f, back[3] = {0.0f, 0.0f, 0.0f};   // the first residual; the last three
  // the host reads an iteration's norms while the GPU works on the next one
  for (int it = 1; it <= cap + 1; ++it) {
    if (it <= cap) {
      const bool star = from_star && it == 1;
      const double *fa = star ? q.fs : f, *Fa = star ? q.Fs : F;
      SFX_KERNEL(c, K_RESIDUAL, k_resid64<G>, rg.grid, rg.block, s, q, fa, Fa, tol, ctl,
                 S.report + 8 * (it & 1));
      SFX_CUDA(cudaEventRecord(S.ev[it & 1], s));
      if (t2.ty > 0) {
        const dim3 g((unsigned)((L.nx + t2.tx - 1) / t2.tx), (unsigned)((L.ny + t2.ty - 1) / t2.ty));
        prof_before(c, K_SMOOTH_FINE, s);
        k_corr64_tile2d<G><<<g, kT2Threads, t2smem, s>>>(q.p, t2.tx, t2.ty, sweeps, q.H[0], q.H[1],
                                                         q.rc, q.e2, f, F, fa, Fa, ctl);
        prof_after(c, K_SMOOTH_FINE, s);
      }
      for (int w = 0; w < sweeps && t2.ty == 0; ++w)
        for (int color = w == 0 ? 1 : 0; color < 2; ++color) {
          const bool add = w == sweeps - 1 && color == 1;
          SFX_KERNEL(c, K_SMOOTH_FINE, k_corr64<G>, grd, blk, s, q.p, q.H[0], q.H[1], q.H[2], q.rc,
                     q.e2, color, w == 0 ? 1 : 0, add ? f : nullptr, add ? F : nullptr, fa, Fa,
                     ctl);
        }
      SFX_LAUNCH_CHECK();
    }
    const int prev = it - 1;
    if (prev < 1) continue;
    SFX_CUDA(cudaEventSynchronize(S.ev[prev & 1]));
    const volatile unsigned int* rep = S.report + 8 * (prev & 1);
    float n[4];
    for (int k = 0; k < 4; ++k) {
      const unsigned int u = rep[k];
      memcpy(&n[k], &u, 4);
    }
    const bool ok = rep[4] != 0;
    *iters = prev;
    rel[0] = n[0] / std::max((double)n[1], 1e-300);
    rel[1] = n[2] / std::max((double)n[3], 1e-300);
    for (int k = 0; k < 4; ++k)
      if (!std::isfinite(n[k])) return SFX_OK;
    // scales outside the comfortable range of the FP32 correction
    for (int k = 1; k < 4; k += 2)
      if (n[k] > 1e30f || (n[k] > 0.0f && n[k] < 1e-18f)) return SFX_OK;
    if (ok) {
      *conv = true;
      return SFX_OK;
    }
    const float worst = (float)std::max(rel[0], rel[1]);
    if (prev == 1) first = worst;
    if (worst > 1e3f * std::max(first, 1.0f)) return SFX_OK;   // diverging
    // at the best of its last three rates it would not get there: stalled (at
    // the rounding of the residual, for a tolerance below it) or too slow
    if (prev >= 6) {
      const double rate = std::min({worst / back[0], back[0] / back[1], back[1] / back[2]});
      if (!(rate < 0.999) || prev + std::log(o->tol / worst) / std::log(rate) > cap + 1) return SFX_OK;
    }
    back[2] = back[1];
    back[1] = back[0];
    back[0] = worst;
  }
  return SFX_OK;
}

}  // namespace

sfx_status drift_faces64(sfx_ctx* c, const double* phi, double Df, double DF, double eps,
                         double* const* Bf, double* const* BF, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  Setup64 q{L, phi, Df, DF, eps, 0.0, 0.0, 0.0, {}, {}, {}, nullptr, nullptr, nullptr, {}, {}};
  for (int d = 0; d < L.ndim(); ++d) {
    q.Bf[d] = Bf[d];
    q.BF[d] = BF[d];
  }
  if (L.ndim() == 3) launch_setup<3>(c, q, s);
  else launch_setup<2>(c, q, s);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

// The Newton solve is taken under the rule of the FP32 form: automatic
// multigrid depth and max(D) dt/h^2 <= 1, where relaxation alone converges
// (0.15-0.5 per sweep); beyond it, and where the caller names a number of
// levels, the Picard solver's V-cycles are the better ones.  Its work arrays
// index with 32 bits and its launches put rows in grid y.  The sweeps' drift
// faces are half precision and at most D/eps: larger ones are left to the
// Picard solver as well.
// Planar steps with a flow stay with the Picard solver too.  That is no property
// of the solvers - the Newton solve is the faster (512^2: 0.87 against 8.0 ms) and
// the more exact one there as well (1e-13 against up to 4e-9 in the force) - but
// of what programs that compare FP64 runs would see: on 30 rotating circles of 50
// to 512 cells a side, at tol = 1e-10, a third of the forces moved by more than
// 1e-9 between the solvers.  On the steps drawn alike without a flow, and in the
// other geometries, no force moved by more than 3e-10.  mg_levels = 1 or more
// names the Picard solver for any step.
bool newton64_eligible(const sfx_ctx* c, const sfx_params* p, double dt, const sfx_solve_opts* o,
                       bool flow) {
  const Level& L = c->lev[0].lv;
  const size_t nx = L.nx, ny = L.ny, nz = L.nz;
  const size_t most = std::max({(nx + 1) * ny * nz, nx * (ny + 1) * nz, nx * ny * (nz + 1),
                                2 * ny * nz * ((nx + 1) / 2)});
  const double D = std::max(p->Df, p->DF);
  return c->prec == SFX_F64 && o->mg_levels == 0 && !(flow && L.geom == SFX_PLANAR2D) &&
         most < ((size_t)1 << 31) && ny <= 65535 && nz <= 65535 && D * dt <= L.h * L.h &&
         D <= kHalfMax * p->eps;
}

// The work arrays of the Newton solve; where there is no memory for them the
// Picard solver, which needs none, takes the step.
bool newton64_scratch(sfx_ctx* c) {
  if (ensure(c) == SFX_OK) return true;
  cudaGetLastError();
  return false;
}

// Drift faces (into the finest level's arrays), the coefficients of the Newton
// solve and its cleared control words.
sfx_status newton64_prepare(sfx_ctx* c, const sfx_params* p, const double* phi, const double* f,
                            const double* F, bool copy, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  LevelData& D = c->lev[0];
  Setup64 q{L, phi, p->Df, p->DF, p->eps, p->ka, p->eta, p->gamma_inf, {}, {}, {}, D.lam, D.b,
            (int*)c->n64.ctl, {f, F}, {copy ? c->fstar : nullptr, copy ? c->Fstar : nullptr}};
  for (int d = 0; d < L.ndim(); ++d) {
    q.Bf[d] = D.B[0][d];
    q.BF[d] = D.B[1][d];
    q.H[d] = c->n64.H[d];
  }
  if (L.ndim() == 3) launch_setup<3>(c, q, s);
  else launch_setup<2>(c, q, s);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

sfx_status newton64_solve(sfx_ctx* c, const sfx_params* p, double* f, double* F, double dt,
                          bool from_star, const sfx_solve_opts* o, int* iters, double* rel,
                          bool* conv, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  LevelData& D = c->lev[0];
  Newton64 q{};
  q.p = Nw32{L, (float)(1.0 / L.h), (float)(p->Df / L.h), (float)(p->DF / L.h), (float)(1.0 / dt),
             (float)p->ka, (float)p->kd, (float)p->gamma_inf, (float)(1.0 / p->eps), (float)p->eta,
             p->literal_upwind, sor_omega(p->Df, dt, L.h, p->eps, L.ndim()),
             sor_omega(p->DF, dt, L.h, p->eps, L.ndim())};
  q.Doh[0] = p->Df / L.h;
  q.Doh[1] = p->DF / L.h;
  q.invh = 1.0 / L.h;
  q.inv_dt = 1.0 / dt;
  q.kd = p->kd;
  for (int d = 0; d < L.ndim(); ++d) {
    q.Bf[d] = D.B[0][d];
    q.BF[d] = D.B[1][d];
    q.H[d] = c->n64.H[d];
  }
  q.c1 = D.lam;
  q.finf = D.b;
  q.fs = c->fstar;
  q.Fs = c->Fstar;
  q.rc = c->n64.rc;
  q.e2 = c->n64.e2;
  switch (L.geom) {
    case SFX_AXISYM: return solve<SFX_AXISYM>(c, q, f, F, from_star, o, iters, rel, conv, s);
    case SFX_PLANAR2D: return solve<SFX_PLANAR2D>(c, q, f, F, from_star, o, iters, rel, conv, s);
    default: return solve<SFX_CART3D>(c, q, f, F, from_star, o, iters, rel, conv, s);
  }
}

}  // namespace sfx
