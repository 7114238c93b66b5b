// ACDI transport of the phase field (Sec. 2.5):
//   d phi/dt + div(u phi) = div(zeta {eps grad phi
//                              - 1/4 (1 - tanh^2(psi/(2 eps))) grad psi/|grad psi|}),
//   psi = eps ln r,  r = (phi + veps)/(1 - phi + veps),  veps = 1e-6,
// FP64 in both context precisions (phi is double everywhere).  The
// advective part is the BCG step of the transported fields (inflow faces
// carry phi = 1); the regularisation is explicit, in flux form, with the
// central face fluxes
//   a_f = zeta [eps (phi*_R - phi*_L)/h - 1/4 w_f nbar_f],
// nbar_f the mean of the two cells' unit normals of psi along the face and
// w_f = 1 - tanh^2((psi_L + psi_R)/(4 eps)).  With s = sqrt(r_L r_R),
// tanh((psi_L + psi_R)/(4 eps)) = (s - 1)/(s + 1), so w_f = 4 s/(1 + s)^2:
// the face needs no transcendental beyond the square root.
//
// What bounds it is the FP64 pipe (1/59 of the FP32 rate): psi takes a
// logarithm and a quotient, the normal a root and a quotient, a face of the
// regularisation a quotient.  All of that matters only where psi has a
// direction, a band of a few cells around the interface, so the passes are
//   psi32: psi in float per cell, good to 1e-6 of |grad psi|;
//   mark: cells where the float |grad psi| comes near kAcdiKappa;
//   cell: r^(1/2) and psi in FP64 for marked cells and their neighbours;
//   normal: FP64 normals of marked cells, with the FP64 test;
//   update: diffusion everywhere, the sharpening flux on the faces of marked
//     cells, clipped to [0, 1] on request (the scheme overshoots by O(veps)
//     where phi saturates, and the surfactant step divides by phi + eta).
// A cell that is not marked has |grad psi| < kAcdiKappa, so its normal is 0
// whatever its last bits.  160^3 sphere: psi, normal and update 1.91 ms with
// every cell in FP64 and six faces of a root and a quotient each; now, with the
// marks, 0.28 ms with a band of nine cells marked, 0.74 ms once the profile has
// spread (after 40 steps: cells 0.29, normals 0.11, update 0.30 ms).
//
// SFX_F64 contexts (BITS) keep every rounding of the definition: on a plateau
// of phi its last bits set how far the normal of the forces is faded in, and
// the curvature, double there, moved by up to 4e-8 of its scale with the
// shorter forms.
#include <algorithm>

#include "sfx_internal.h"

namespace sfx {
namespace {

constexpr double kAcdiVeps = 1e-6;
// n is undefined where psi is flat: where phi saturates, the direction of
// grad psi is set by the last bits of phi while 1 - tanh^2 stays ~4 veps.
// n = 0 where |grad psi| is below kAcdiKappa times its equilibrium value 1
// (psi is a signed distance at equilibrium) or below 1e-30; |grad psi|
// falls below 0.1 only where veps dominates psi (phi or 1 - phi below
// ~0.1 veps).
constexpr double kAcdiKappa = 0.1;
// Grids of fewer cells do without marks: two launches less, and in cell blocks a
// launch of few blocks lasts as long as the fullest of them.  A step of a circle
// or sphere at rest without and with marks, in FP64 and FP32 contexts: 128^2 29,
// 51 and 23, 37 us, 32^3 33, 62 and 28, 40, 48^3 72, 80 and 45, 56, 64^3 147, 96
// and 81, 62.
constexpr size_t kAcdiMarkCells = (size_t)1 << 17;

// psi/(2h) in float from phi* in [0, 1]: phi* may overshoot by O(veps) where
// it saturates, and past 1 + veps psi would have no value.  1 - phi is taken
// in FP64 (near 1 it would lose every digit in float).
__global__ void k_acdi_psi32(size_t n, const double* __restrict__ ps, float scale,
                             float* __restrict__ psi) {
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    const double p = ps[c];
    const float a = fminf(fmaxf((float)p, 0.0f), 1.0f);
    const float b = fminf(fmaxf((float)(1.0 - p), 0.0f), 1.0f);
    psi[c] = scale * logf(__fdividef(a + (float)kAcdiVeps, b + (float)kAcdiVeps));
  }
}

// fmin(fmax(v, 0), 1), NaN included, without the FP64 pipe
__device__ __forceinline__ double clip01(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if (b > 0x7ff0000000000000ULL) return 0.0;   // below 0 or NaN
  return b < 0x3ff0000000000000ULL ? v : 1.0;
}

// The cell of this thread: with marks (MARK), in cell blocks, of which a block
// takes a quarter in FP64 contexts (BITS), whose passes are the FP64 pipe's
// throughout, to even out over the SMs; without, cells in turn.
template <int ND, bool BITS, bool MARK>
__device__ __forceinline__ bool acdi_at(const Level& L, int* x) {
  if (MARK && !BITS) return CellBlock<ND>::at(L, blockIdx.x, x);
  if (MARK) return CellBlock<ND>::at(L, blockIdx.x / 4, x, (int)(blockIdx.x % 4 * 128 + threadIdx.x));
  const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;   // (small grids)
  const unsigned r = c / (unsigned)L.nx;
  x[0] = (int)(c - r * (unsigned)L.nx);
  x[1] = (int)(r % (unsigned)L.ny);
  x[2] = (int)(r / (unsigned)L.ny);
  return x[2] < L.nz;
}

template <int ND>
__device__ __forceinline__ void neighbours(const Level& L, const int* x, size_t c, size_t* o,
                                           bool* has) {
  const size_t st[3] = {1, (size_t)L.nx, (size_t)L.nx * L.ny};
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    has[2 * d] = x[d] > 0;
    has[2 * d + 1] = x[d] + 1 < L.extent(d);
    o[2 * d] = has[2 * d] ? c - st[d] : c;
    o[2 * d + 1] = has[2 * d + 1] ? c + st[d] : c;
  }
}

// mark[c] = 1 where |grad psi| in float is not safely below kAcdiKappa (or
// not a number: the FP64 passes decide)
template <int ND, bool BITS>
__global__ void k_acdi_mark(Level L, const float* __restrict__ psi, float thr2,
                            unsigned char* __restrict__ mark) {
  int x[3];
  if (!acdi_at<ND, BITS, true>(L, x)) return;
  const size_t c = cidx(L, x[0], x[1], x[2]);
  size_t o[2 * ND];
  bool has[2 * ND];
  neighbours<ND>(L, x, c, o, has);
  float m2 = 0.0f;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const float g = psi[o[2 * d + 1]] - psi[o[2 * d]];
    m2 = fmaf(g, g, m2);
  }
  mark[c] = m2 < thr2 ? 0 : 1;
}

// The mark of cell c; without marks every cell counts as marked.
template <bool MARK>
__device__ __forceinline__ int marked(const unsigned char* __restrict__ mark, size_t c) {
  return MARK ? mark[c] : 1;
}

// r^(1/2) (BITS: r) and psi of the cells that a marked cell's normal or faces
// read
template <int ND, bool BITS, bool MARK>
__global__ void k_acdi_cell(Level L, const unsigned char* __restrict__ mark,
                            const double* __restrict__ ps, double eps, double* __restrict__ g,
                            double* __restrict__ psi) {
  int x[3];
  if (!acdi_at<ND, BITS, MARK>(L, x)) return;
  const size_t c = cidx(L, x[0], x[1], x[2]);
  size_t o[2 * ND];
  bool has[2 * ND];
  neighbours<ND>(L, x, c, o, has);
  int any = marked<MARK>(mark, c);
#pragma unroll
  for (int q = 0; q < 2 * ND; ++q) any |= marked<MARK>(mark, o[q]);
  if (!any) return;
  const double p = clip01(ps[c]);
  const double rc = (p + kAcdiVeps) / (1.0 - p + kAcdiVeps);
  g[c] = BITS ? rc : sqrt(rc);
  psi[c] = eps * log(rc);
}

// n = grad psi/|grad psi| of the marked cells (centred differences,
// zero-gradient ghosts), 0 where psi is flat (above)
template <int ND, bool BITS, bool MARK>
__global__ void k_acdi_normal(Level L, const unsigned char* __restrict__ mark,
                              const double* __restrict__ psi, double* __restrict__ nv) {
  int x[3];
  if (!acdi_at<ND, BITS, MARK>(L, x)) return;
  const size_t c = cidx(L, x[0], x[1], x[2]), n = L.ncell();
  if (!marked<MARK>(mark, c)) return;
  // the 1/(2h) of the differences cancels in n; the threshold takes it
  // (kAcdiKappa is far above the guard 1e-30)
  const double thr = kAcdiKappa * (2.0 * L.h);
  size_t o[2 * ND];
  bool has[2 * ND];
  neighbours<ND>(L, x, c, o, has);
  double v[ND], m2 = 0.0;
  if (BITS) {
    const double inv2h = 0.5 / L.h;
    for (int d = 0; d < ND; ++d) {
      v[d] = (psi[o[2 * d + 1]] - psi[o[2 * d]]) * inv2h;
      m2 += v[d] * v[d];
    }
    const double m = sqrt(m2);
    for (int d = 0; d < ND; ++d) nv[(size_t)d * n + c] = m < kAcdiKappa ? 0.0 : v[d] / m;
    return;
  }
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    v[d] = psi[o[2 * d + 1]] - psi[o[2 * d]];
    m2 = fma(v[d], v[d], m2);
  }
  const double s = m2 < thr * thr ? 0.0 : rsqrt(m2);
#pragma unroll
  for (int d = 0; d < ND; ++d) nv[(size_t)d * n + c] = v[d] * s;
}

// The BITS form of the update below: per face the flux
// zeta [eps (phi*_R - phi*_L)/h - 1/4 w_f nbar_f], w_f = 4 s/(1 + s)^2.
template <int ND, bool AXI, bool MARK>
__global__ void k_acdi_update_bits(Level L, const unsigned char* __restrict__ mark,
                                   const double* __restrict__ ps, const double* __restrict__ r,
                                   const double* __restrict__ nv, double zeta, double eps,
                                   double dt, int clip, double* __restrict__ phi) {
  int x[3];
  if (!acdi_at<ND, true, MARK>(L, x)) return;
  const size_t c = cidx(L, x[0], x[1], x[2]), n = L.ncell();
  size_t o[2 * ND];
  bool has[2 * ND];
  neighbours<ND>(L, x, c, o, has);
  const double invh = 1.0 / L.h, pc = ps[c];
  const int mc = marked<MARK>(mark, c);
  double div = 0.0;
  for (int q = 0; q < 2 * ND; ++q) {
    if (!has[q]) continue;
    const double s = q & 1 ? 1.0 : -1.0;
    double w = 1.0;
    if (AXI && q < 2) w = 2.0 * (double)(x[0] + q) / (double)(2 * x[0] + 1);
    const int mo = marked<MARK>(mark, o[q]);
    double af;
    if (mc | mo) {
      const double* nd = nv + (size_t)(q / 2) * n;
      const double sq = sqrt(r[c] * r[o[q]]);
      const double wt = 4.0 * sq / ((1.0 + sq) * (1.0 + sq));
      const double nbar = 0.5 * ((mc ? nd[c] : 0.0) + (mo ? nd[o[q]] : 0.0));
      af = zeta * (eps * s * (ps[o[q]] - pc) * invh - 0.25 * wt * nbar);
    } else {
      af = zeta * (eps * s * (ps[o[q]] - pc) * invh);
    }
    div += s * w * af;
  }
  const double v = pc + dt * div * invh;
  phi[c] = clip ? clip01(v) : v;
}

// phi = phi* + dt/V sum_f (+-) A_f a_f; wall faces carry nothing and the
// axis face has zero area.  k1 = dt zeta eps/h^2, k2 = dt zeta/(2h): with s =
// r_L^(1/2) r_R^(1/2) and nbar = (n_L + n_R)/2 a face's sharpening flux
// zeta/4 w_f nbar_f is zeta s/(1 + s)^2 (n_L + n_R)/2.
//
// A face's s/(1 + s)^2 costs a quotient, and six faces per cell took 84 of
// the pass's FP64 instructions, so a block evaluates each face once: a thread
// the minus sides of its cell, 272 threads (48 in 2D) the block's far sides,
// both factors of the product handed over through shared memory (a cell still
// fuses it into its own sum, so the bits are those of six faces per cell).
// Rows of 40 doubles keep the two rows of a half warp in different banks.
// 160^3 after 40 steps: 425 -> 304 us; after one 180 -> 145 us (with two instead
// of three blocks per SM 335 and 165; clipping on the FP64 pipe 319 and 160).
template <int ND, bool AXI, bool MARK>
__global__ void __launch_bounds__(512, 3)
k_acdi_update(Level L, const unsigned char* __restrict__ mark, const double* __restrict__ ps,
              const double* __restrict__ g, const double* __restrict__ nv, double k1, double k2,
              int clip, double* __restrict__ phi) {
  using B = CellBlock<ND>;
  constexpr int kRow = 40, kRows = ND == 3 ? B::by * (B::bz + 1) : B::by + 1;
  __shared__ double sa[ND][kRows * kRow], sn[ND][kRows * kRow];
  const size_t n = L.ncell();
  const size_t st[3] = {1, (size_t)L.nx, (size_t)L.nx * L.ny};
  const int3 l = B::cell(threadIdx.x);
  int x[3];
  const bool in = B::at(L, blockIdx.x, x);
  const size_t c = in ? cidx(L, x[0], x[1], x[2]) : 0;
  // face area over V/h of the radial faces
  double wr[2] = {1.0, 1.0};
  if (AXI) {
    wr[0] = (double)(2 * x[0]) / (double)(2 * x[0] + 1);
    wr[1] = (double)(2 * x[0] + 2) / (double)(2 * x[0] + 1);
  }
  int any = 0;
  double pc = 0.0, lap = 0.0, div = 0.0;
  if (in) {
    size_t o[2 * ND];
    bool has[2 * ND];
    neighbours<ND>(L, x, c, o, has);
    any = marked<MARK>(mark, c);
    pc = ps[c];
#pragma unroll
    for (int q = 0; q < 2 * ND; ++q) {
      any |= marked<MARK>(mark, o[q]);
      const double dp = ps[o[q]] - pc;      // 0 at a wall
      lap = AXI && q < 2 ? fma(wr[q], dp, lap) : lap + dp;
    }
  }
  const auto slot = [](int d, int lx, int ly, int lz) {
    return (lz * (B::by + (d == 1)) + ly) * kRow + lx;
  };
  // s/(1 + s)^2 and n_L + n_R of the minus side of cell y in direction d
  const auto face = [&](int d, int yx, int yy, int yz, int at) {
    double a = 0.0, nn = 0.0;
    const int yd = d == 0 ? yx : (d == 1 ? yy : yz);
    if (yd > 0 && yx < L.nx && yy < L.ny && yz < L.nz) {
      const size_t r = cidx(L, yx, yy, yz), m = r - st[d];
      const int mr = marked<MARK>(mark, r), mm = marked<MARK>(mark, m);
      if (mr | mm) {
        const double* nd = nv + (size_t)d * n;
        nn = (mr ? nd[r] : 0.0) + (mm ? nd[m] : 0.0);
        const double u = 1.0 / fma(g[r], g[m], 1.0);   // 1/(1 + s); s/(1 + s)^2 = u - u^2
        a = fma(-u, u, u);
      }
    }
    sa[d][at] = a;
    sn[d][at] = nn;
  };
  const bool sharp = __syncthreads_or(any);
  if (sharp) {
#pragma unroll
    for (int d = 0; d < ND; ++d) face(d, x[0], x[1], x[2], slot(d, l.x, l.y, l.z));
    const int x0 = x[0] - l.x, y0 = x[1] - l.y, z0 = x[2] - l.z, t = threadIdx.x;
    constexpr int fy = B::bx * B::bz, fz = ND == 3 ? B::bx * B::by : 0;
    if (t < fy) {
      const int a = t % B::bx, e = t / B::bx;
      face(1, x0 + a, y0 + B::by, z0 + e, slot(1, a, B::by, e));
    } else if (t < fy + fz) {
      const int a = (t - fy) % B::bx, e = (t - fy) / B::bx;
      face(ND - 1, x0 + a, y0 + e, z0 + B::bz, slot(ND - 1, a, e, B::bz));
    } else if (t < fy + fz + B::by * B::bz) {
      const int a = (t - fy - fz) % B::by, e = (t - fy - fz) / B::by;
      face(0, x0 + B::bx, y0 + a, z0 + e, slot(0, B::bx, a, e));
    }
    __syncthreads();
  }
  if (!in) return;
  if (any) {
#pragma unroll
    for (int q = 0; q < 2 * ND; ++q) {
      const int d = q / 2, p = q & 1;
      const int at = slot(d, l.x + (p && d == 0), l.y + (p && d == 1), l.z + (p && d == 2));
      double a = sa[d][at];
      if (AXI && q < 2) a *= wr[q];
      div = fma(p ? -a : a, sn[d][at], div);
    }
  }
  double v = fma(k1, lap, pc);
  if (any) v = fma(k2, div, v);
  phi[c] = clip ? clip01(v) : v;
}

template <int ND, bool AXI, bool MARK>
void acdi_passes(sfx_ctx* c, const double* ps, double* g, double* psi, double* nv,
                 const float* psi32, unsigned char* mark, float thr2, double zeta, double eps,
                 double dt, int clip, double* phi, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  constexpr int threads = CellBlock<ND>::threads;
  const int blocks = (int)CellBlock<ND>::count(L), turns = (int)((L.ncell() + 255) / 256);
  if (c->prec == SFX_F64) {
    const int nt = MARK ? threads / 4 : 256, nb = MARK ? 4 * blocks : turns;
    if (MARK) SFX_KERNEL(c, K_PHASE, (k_acdi_mark<ND, true>), nb, nt, s, L, psi32, thr2, mark);
    SFX_KERNEL(c, K_PHASE, (k_acdi_cell<ND, true, MARK>), nb, nt, s, L, mark, ps, eps, g, psi);
    SFX_KERNEL(c, K_PHASE, (k_acdi_normal<ND, true, MARK>), nb, nt, s, L, mark, psi, nv);
    SFX_KERNEL(c, K_PHASE, (k_acdi_update_bits<ND, AXI, MARK>), nb, nt, s, L, mark, ps, g, nv, zeta,
               eps, dt, clip, phi);
  } else {
    const double k1 = dt * zeta * eps / (L.h * L.h), k2 = 0.5 * dt * zeta / L.h;
    const int nt = MARK ? threads : 256, nb = MARK ? blocks : turns;
    if (MARK) SFX_KERNEL(c, K_PHASE, (k_acdi_mark<ND, false>), nb, nt, s, L, psi32, thr2, mark);
    SFX_KERNEL(c, K_PHASE, (k_acdi_cell<ND, false, MARK>), nb, nt, s, L, mark, ps, eps, g, psi);
    SFX_KERNEL(c, K_PHASE, (k_acdi_normal<ND, false, MARK>), nb, nt, s, L, mark, psi, nv);
    SFX_KERNEL(c, K_PHASE, (k_acdi_update<ND, AXI, MARK>), blocks, threads, s, L, mark, ps, g, nv, k1,
               k2, clip, phi);
  }
}

}  // namespace

sfx_status acdi_step(sfx_ctx* c, const void* ux, const void* uy, const void* uz, double dt,
                     double zeta, double eps, int clip, double* phi, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  const size_t n = L.ncell();
  if (!c->acdi) {
    SFX_CUDA(cudaMalloc((void**)&c->acdi, (size_t)(3 + L.ndim()) * n * sizeof(double) + n));
    c->allocations.push_back(c->acdi);
  }
  double* ps = c->acdi;
  double* g = ps + n;
  double* psi = g + n;
  double* nv = psi + n;
  float* psi32 = (float*)nv;              // read before the normals are written
  unsigned char* mark = n >= kAcdiMarkCells ? (unsigned char*)(nv + (size_t)L.ndim() * n) : nullptr;
  if (ux) {
    sfx_status st = advect_phi(c, ux, uy, uz, dt, phi, 1.0, ps, s);
    if (st != SFX_OK) return st;
  } else {
    SFX_CUDA(cudaMemcpyAsync(ps, phi, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
  }
  if (mark)
    SFX_KERNEL(c, K_PHASE, k_acdi_psi32, blocks_for(n, 256), 256, s, n, ps, (float)(0.5 * eps / L.h),
               psi32);
  // the float psi/(2h) is good to a few 1e-7 of its largest value 7 eps/h
  const double thr = std::max(0.0, 0.9 * kAcdiKappa - 1e-4 * eps / L.h);
  const float thr2 = (float)(thr * thr);
  const auto passes = [&](auto marked, auto every) {
    (mark ? marked : every)(c, ps, g, psi, nv, psi32, mark, thr2, zeta, eps, dt, clip, phi, s);
  };
  switch (L.geom) {
    case SFX_CART3D: passes(&acdi_passes<3, false, true>, &acdi_passes<3, false, false>); break;
    case SFX_AXISYM: passes(&acdi_passes<2, true, true>, &acdi_passes<2, true, false>); break;
    default: passes(&acdi_passes<2, false, true>, &acdi_passes<2, false, false>);
  }
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

}  // namespace sfx
