// Conserved totals (compensated, deterministic), the surface-tension EOS of
// Sec. 2.3 and the Marangoni force of Sec. 2.4.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sfx_internal.h"
#include "sfx_op64.cuh"
#include "sfx_plic.cuh"

namespace sfx {
namespace {

constexpr int kTotThreads = kTotalsThreads;

// The totals sum V x of the fields in grid.y, both stages in one launch.
struct TotalFields {
  const double* x[8];
};
__global__ void __launch_bounds__(kTotThreads)
k_totals(Level L, TotalFields f, double* __restrict__ partials, unsigned* __restrict__ tickets,
         double* __restrict__ out) {
  const int fi = blockIdx.y;
  double s, cc;
  totals_thread(L, f.x[fi], s, cc);
  if (last_block_total<kTotThreads>(partials + 2 * (size_t)fi * gridDim.x, blockIdx.x, gridDim.x,
                                    tickets + fi, s, cc))
    out[fi] = s + cc;
}

// One block: fixed-order combination of block partials.
__global__ void k_total_final(const double* __restrict__ partials, int nblk,
                              double* __restrict__ out) {
  double s, cc;
  warp_combine(partials, nblk, s, cc);
  if (threadIdx.x == 0) out[0] = s + cc;
}

struct EosArgs {
  double ginf, eps, sigma0, E;
  int eos;
};

// Gamma = f/delta_phi where delta_phi >= 1e-3/eps, else 0; sigma in double.
__global__ void k_eos(size_t n, EosArgs q, const double* __restrict__ f,
                      const double* __restrict__ phi, double* __restrict__ sigma) {
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    double p = phi[c];
    // phi within 5e-4 of 0 or 1 (or outside): delta_phi is half of 1e-3/eps,
    // Gamma = 0 and every EOS gives sigma0, told from the integer words
    // without the quotients and the logarithm (FP64 pipe)
    const long long b = __double_as_longlong(p);
    if (b < 0x3f40624dd2f1a9fcLL || b > 0x3feffbe76c8b4396LL) {
      sigma[c] = q.sigma0;
      continue;
    }
    const double pq = p * (1.0 - p);
    double del = pq / q.eps;
    double G = del >= 1e-3 / q.eps ? f[c] / del : 0.0;
    double x = G / q.ginf;
    double s;
    if (q.eos == SFX_EOS_LANGMUIR) {
      x = fmin(x, 1.0 - 1e-12);          // stay below saturation
      s = q.sigma0 * (1.0 + q.E * log1p(-x));
    } else if (q.eos == SFX_EOS_LINEAR) {
      s = q.sigma0 * (1.0 - q.E * x);
    } else {
      s = q.sigma0 * (1.0 - tanh(q.E * x));
    }
    sigma[c] = s;
  }
}

// d sigma/d Gamma of the EOS above (0 where the Langmuir sigma is clamped)
__device__ __forceinline__ double eos_slope(const EosArgs& q, double G) {
  const double x = G / q.ginf;
  if (q.eos == SFX_EOS_LANGMUIR)
    return x < 1.0 - 1e-12 ? -q.sigma0 * q.E / (q.ginf * (1.0 - x)) : 0.0;
  if (q.eos == SFX_EOS_LINEAR) return -q.sigma0 * q.E / q.ginf;
  const double t = tanh(q.E * x);
  return -q.sigma0 * q.E / q.ginf * (1.0 - t * t);
}

// Interface cells of the PLIC area: nearer fractions are the round-off of empty
// or full cells.
__device__ __forceinline__ bool plic_cell(double C) { return C > 1e-6 && C < 1.0 - 1e-6; }

// One cell of the Marangoni force with its delta_m.
__device__ __forceinline__ void force64_cell(const Level& L, const double* __restrict__ phi,
                                             const double* __restrict__ C,
                                             const double* __restrict__ sigma, int dm_mode,
                                             double eps, size_t c, double* __restrict__ force,
                                             double* __restrict__ dm_out) {
  const size_t n = L.ncell();
  const int nd = L.ndim();
  const double inv2h = 0.5 / L.h;
  int idx[3];
  idx[0] = (int)(c % L.nx);
  row_jk(c / L.nx, L.ny, idx[1], idx[2]);
  double gs[3] = {0, 0, 0}, nn[3], ndg = 0.0, q = 0.0;
  unit_normal64(L, phi, idx, eps, nn);
  for (int d = 0; d < nd; ++d) {
    int pp[3] = {idx[0], idx[1], idx[2]}, pm[3] = {idx[0], idx[1], idx[2]};
    pp[d] = min(pp[d] + 1, L.extent(d) - 1);
    pm[d] = max(pm[d] - 1, 0);
    const size_t cp = cidx(L, pp[0], pp[1], pp[2]), cm = cidx(L, pm[0], pm[1], pm[2]);
    gs[d] = (sigma[cp] - sigma[cm]) * inv2h;
    ndg += nn[d] * gs[d];
    if (dm_mode == 0) {
      const double g = (C[cp] - C[cm]) * inv2h;
      q += g * g;
    }
  }
  double dm;
  if (dm_mode == 0) {
    dm = sqrt(q);
  } else {
    double m[3];
    youngs_normal(L, C, idx[0], idx[1], idx[2], m);
    dm = plic_cell(C[c]) ? plic_unit_area(nd, m, C[c]) / L.h : 0.0;
  }
  for (int d = 0; d < nd; ++d) force[(size_t)d * n + c] = dm * (gs[d] - nn[d] * ndg);
  if (dm_out) dm_out[c] = dm;
}

// |grad C| instead of the PLIC area (dm_mode 0): every cell carries a force.
__global__ void __launch_bounds__(256)
k_force(Level L, const double* __restrict__ phi, const double* __restrict__ C,
        const double* __restrict__ sigma, double eps, double* __restrict__ force,
        double* __restrict__ dm_out) {
  const size_t n = L.ncell();
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x)
    force64_cell(L, phi, C, sigma, 0, eps, c, force, dm_out);
}

// With the PLIC area only interface cells carry a force.  A block gathers those
// of its 512 cells and takes them by full warps: a cell is a chain of about 600 FP64 instructions, an instruction occupies the SM's FP64 pipe for a
// whole warp however few lanes it serves, and in rows of 32 cells a warp held
// one or two interface cells.  The gathered cells stay in shared memory: the
// call has no scratch, so that calls on different streams may overlap.  With
// the EOS: 96^3 533 -> 133 us, 160^3 1874 -> 252, 128^2 109 -> 46 (a list of the
// context's cells: 119, 221, 50; boxes of 1024 and 2048 cells 140-167 at 96^3,
// of 256 cells 128-146: what is left is the chains of the fullest SMs).
template <int ND>
__global__ void __launch_bounds__(128)
k_force_cut(Level L, const double* __restrict__ phi, const double* __restrict__ C,
            const double* __restrict__ sigma, double eps, double* __restrict__ force,
            double* __restrict__ dm_out) {
  using B = CellBlock<ND>;
  __shared__ unsigned short list[B::threads];
  __shared__ unsigned count;
  const size_t n = L.ncell();
  const unsigned nbx = (L.nx + B::bx - 1) / B::bx, nby = (L.ny + B::by - 1) / B::by;
  const int x0 = (int)(blockIdx.x % nbx) * B::bx, y0 = (int)(blockIdx.x / nbx % nby) * B::by,
            z0 = (int)(blockIdx.x / nbx / nby) * B::bz;
  const auto cell = [&](int t) {
    return cidx(L, x0 + t % B::bx, y0 + t / B::bx % B::by, z0 + t / (B::bx * B::by));
  };
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int t = threadIdx.x; t < B::threads; t += 128) {   // rows of cells
    bool cut = false;
    if (x0 + t % B::bx < L.nx && y0 + t / B::bx % B::by < L.ny &&
        z0 + t / (B::bx * B::by) < L.nz) {
      const size_t c = cell(t);
      cut = plic_cell(C[c]);
      if (!cut) {
        // delta_m = 0 times a gradient or a normal that is not finite is NaN:
        // those cells are evaluated as well
        const int x[3] = {x0 + t % B::bx, y0 + t / B::bx % B::by, z0 + t / (B::bx * B::by)};
        const size_t st[3] = {1, (size_t)L.nx, (size_t)L.nx * L.ny};
        bool finite = true;
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          const size_t cp = x[d] + 1 < L.extent(d) ? c + st[d] : c, cm = x[d] > 0 ? c - st[d] : c;
          finite &= finite_bits(sigma[cp]);
          finite &= finite_bits(sigma[cm]);
          finite &= finite_bits(phi[cp]);
          finite &= finite_bits(phi[cm]);
        }
        cut = !finite;
      }
      if (!cut) {
#pragma unroll
        for (int d = 0; d < ND; ++d) force[(size_t)d * n + c] = 0.0;
        if (dm_out) dm_out[c] = 0.0;
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, cut);
    if (!m) continue;
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&count, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (cut) list[base + __popc(m & ((1u << lane) - 1))] = (unsigned short)t;
  }
  __syncthreads();
  for (unsigned q = threadIdx.x; q < count; q += 128)
    force64_cell(L, phi, C, sigma, 1, eps, cell(list[q]), force, dm_out);
}

// Loss L = sum_c V_c |F_Ma,c|^2: block partials of the sum and, when G is
// given, G_c = dL/d(grad sigma)_c = 2 V_c delta_m,c F_Ma,c (F_Ma is already
// tangential, so the projector (I - n n) maps it to itself).
__global__ void k_loss_partials(Level L, const double* __restrict__ force,
                                const double* __restrict__ dm, double* __restrict__ G,
                                double* __restrict__ part) {
  const size_t n = L.ncell();
  const int nd = L.ndim();
  double s = 0.0, e = 0.0;
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    const double V = cell_volume(L, (int)(c % L.nx));
    double q = 0.0;
    for (int d = 0; d < nd; ++d) {
      const double Fd = force[(size_t)d * n + c];
      q += Fd * Fd;
      if (G) G[(size_t)d * n + c] = 2.0 * V * dm[c] * Fd;
    }
    double u, w;
    two_sum(s, V * q, u, w);
    s = u;
    e += w;
  }
  block_sum_comp<kTotThreads>(s, e);
  if (threadIdx.x == 0) {
    part[2 * (size_t)blockIdx.x] = s;
    part[2 * (size_t)blockIdx.x + 1] = e;
  }
}

// dL/df: the transpose of the centred gradient with its one-sided copies at
// walls (grad sigma_c = (sigma_{c+} - sigma_{c-})/2h, c+ = c at the upper
// wall, c- = c at the lower one) gives dL/dsigma; then through the EOS and
// Gamma = f/delta_phi.
__global__ void k_loss_grad(Level L, EosArgs q, const double* __restrict__ f,
                            const double* __restrict__ phi, const double* __restrict__ G,
                            double* __restrict__ out) {
  const size_t n = L.ncell();
  const int nd = L.ndim();
  const double inv2h = 0.5 / L.h;
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    const int idx[3] = {(int)(c % L.nx), (int)((c / L.nx) % L.ny),
                        (int)(c / ((size_t)L.nx * L.ny))};
    double g = 0.0;
    for (int d = 0; d < nd; ++d) {
      const double* Gd = G + (size_t)d * n;
      const size_t st = d == 0 ? 1 : (d == 1 ? (size_t)L.nx : (size_t)L.nx * L.ny);
      const int p = idx[d], m = L.extent(d);
      if (p >= 1) g += Gd[c - st];
      if (p == m - 1) g += Gd[c];
      if (p <= m - 2) g -= Gd[c + st];
      if (p == 0) g -= Gd[c];
    }
    g *= inv2h;
    const double ph = phi[c];
    const double del = ph * (1.0 - ph) / q.eps;
    out[c] = del >= 1e-3 / q.eps ? g * eos_slope(q, f[c] / del) / del : 0.0;
  }
}

}  // namespace

unsigned* cell_list(sfx_ctx* c, unsigned** slot, int lists, cudaStream_t s) {
  const size_t n = c->lev[0].lv.ncell();
  cudaStreamCaptureStatus cap;
  if (*slot || n >= ((size_t)1 << 32)) return *slot;
  void* p = nullptr;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone ||
      cudaMalloc(&p, lists * (n + 1) * sizeof(unsigned)) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  c->allocations.push_back(p);
  return *slot = (unsigned*)p;
}

// sigma, the force and (dm not null) delta_m of an FP64 state
static sfx_status eos_force(sfx_ctx* c, const EosArgs& q, const double* f, const double* phi,
                            const double* C, int dm_mode, double* sigma, double* force, double* dm,
                            cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  const size_t n = L.ncell();
  const int nb = blocks_for(n, 256);
  SFX_KERNEL(c, K_FORCES, k_eos, nb, 256, s, n, q, f, phi, sigma);
  if (dm_mode == 0)
    SFX_KERNEL(c, K_FORCES, k_force, nb, 256, s, L, phi, C, sigma, q.eps, force, dm);
  else if (L.ndim() == 3)
    SFX_KERNEL(c, K_FORCES, k_force_cut<3>, (unsigned)CellBlock<3>::count(L), 128, s, L, phi, C,
               sigma, q.eps, force, dm);
  else
    SFX_KERNEL(c, K_FORCES, k_force_cut<2>, (unsigned)CellBlock<2>::count(L), 128, s, L, phi, C,
               sigma, q.eps, force, dm);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

sfx_status marangoni_loss(sfx_ctx* c, const sfx_params* p, const double* f, const double* phi,
                          const double* C, int dm_mode, double* loss, double* grad,
                          cudaStream_t s) {
  sfx_status st = adj_ensure_scratch(c);
  if (st != SFX_OK) return st;
  const Level& L = c->lev[0].lv;
  const size_t n = L.ncell();
  const int nb = blocks_for(n, 256);
  EosArgs q{p->gamma_inf, p->eps, p->sigma0, p->E, p->eos};
  st = eos_force(c, q, f, phi, C, dm_mode, c->adj.sig, c->adj.force, c->adj.dm, s);
  if (st != SFX_OK) return st;
  const int nbp = c->adj.nblk;
  SFX_KERNEL(c, K_FORCES, k_loss_partials, nbp, kTotThreads, s, L, c->adj.force, c->adj.dm,
             grad ? c->adj.G : nullptr, c->adj.part);
  SFX_KERNEL(c, K_FORCES, k_total_final, 1, 32, s, c->adj.part, nbp, c->adj.d_out);
  if (grad)
    SFX_KERNEL(c, K_FORCES, k_loss_grad, nb, 256, s, L, q, f, phi, c->adj.G, grad);
  SFX_LAUNCH_CHECK();
  SFX_CUDA(cudaMemcpyAsync(c->adj.h_out, c->adj.d_out, sizeof(double), cudaMemcpyDeviceToHost, s));
  SFX_CUDA(cudaStreamSynchronize(s));
  *loss = c->adj.h_out[0];
  return SFX_OK;
}

sfx_status totals(sfx_ctx* c, const double* const* fields, int nf, double* out, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  TotalFields f{};
  for (int i = 0; i < nf; ++i) f.x[i] = fields[i];
  SFX_KERNEL(c, K_TOTALS, k_totals, dim3(totals_blocks(L.ncell()), nf), kTotThreads, s, L, f,
             c->partials, c->tickets, c->h_sums);
  SFX_LAUNCH_CHECK();
  SFX_CUDA(cudaStreamSynchronize(s));
  memcpy(out, c->h_sums, nf * sizeof(double));
  return SFX_OK;
}

sfx_status marangoni(sfx_ctx* c, const sfx_params* p, const double* f, const void* phi,
                     const double* C, int dm_mode, double* sigma, double* force,
                     cudaStream_t s) {
  EosArgs q{p->gamma_inf, p->eps, p->sigma0, p->E, p->eos};
  return eos_force(c, q, f, (const double*)phi, C, dm_mode, sigma, force, nullptr, s);
}

}  // namespace sfx
