// Geometric VoF advection of the volume fraction C (the paper's interface
// tracking, Sec. 2): directionally split conservative PLIC advection.  For each direction d in turn, with face Courant numbers
// c_f = u_f dt/h,
//   C <- C - (Q_+ - Q_-) + H (c_+ - c_-),
// Q_f the volume fraction crossing face f (the fluid of the upwind cell's
// PLIC reconstruction within |c_f| h of the face, signed with u_f) and
// H = [C > 1/2] at the start of the step; the direction order alternates
// from step to step.  Walls carry no flux.  Planar 2D and 3D.  C is double
// in both precisions; SFX_F32 contexts evaluate the PLIC geometry of the
// fluxes in FP32.
#include <algorithm>

#include "sfx_internal.h"
#include "sfx_plic.cuh"

namespace sfx {
namespace {

// Only cells near fluid 1 change.  Where C is zero bit for bit every flux out
// of a cell is zero, so a block of cells (32 x 4 x 4; 32 x 16 in 2D) without
// fluid 1 in itself or an adjacent block stays as it is through the step (a
// pass moves fluid by one cell along its direction).  On large grids the
// blocks are classified once per step and the passes run over a list of the
// active ones; small grids, where a launch costs more than the sweep, take
// every block.  What bounds a pass on active blocks is the FP64 pipe
// (velocity times dt/h, the update), so signs and the tests for empty and
// full cells read the integer words and floats are widened without the
// conversion instruction.  256^3 sphere of radius 64 in float: 2.45 ms per step
// with every face and cell, 0.90 ms fresh and 1.35 ms once 500 steps have torn
// off wisps (flux 236, update 26 us per direction, classification 94 us).
constexpr size_t kVofListCells = (size_t)1 << 20;

__device__ __forceinline__ long long vbits(double v) { return __double_as_longlong(v); }

// flag[b] = 1 where block b holds fluid 1; eight cells of loads in flight
template <int ND>
__global__ void __launch_bounds__(512) k_vof_flags(Level L, const double* __restrict__ C,
                                                   unsigned char* __restrict__ flag) {
  int x[3];
  const bool in = CellBlock<ND>::at(L, blockIdx.x, x);
  const bool wet = in && vbits(C[cidx(L, x[0], x[1], x[2])]) != 0;
  const int any = __syncthreads_or(wet);
  if (threadIdx.x == 0) flag[blockIdx.x] = any ? 1 : 0;
}

// The blocks with a flagged block among themselves and their neighbours
// (diagonals included), each with a bit per direction whose plus-side
// neighbour block is active too; list[0] counts them.
template <int ND>
__global__ void k_vof_list(Level L, const unsigned char* __restrict__ flag, int2* __restrict__ list) {
  using B = CellBlock<ND>;
  const int nx = (L.nx + B::bx - 1) / B::bx, ny = (L.ny + B::by - 1) / B::by,
            nz = (L.nz + B::bz - 1) / B::bz;
  const int nb = nx * ny * nz;
  auto active = [&](int X, int Y, int Z) {
    if (X >= nx || Y >= ny || Z >= nz) return false;
    for (int c = max(Z - 1, 0); c <= min(Z + 1, nz - 1); ++c)
      for (int b = max(Y - 1, 0); b <= min(Y + 1, ny - 1); ++b)
        for (int a = max(X - 1, 0); a <= min(X + 1, nx - 1); ++a)
          if (flag[(c * ny + b) * nx + a]) return true;
    return false;
  };
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
    const int X = b % nx, Y = b / nx % ny, Z = b / nx / ny;
    if (!active(X, Y, Z)) continue;
    int m = 0;
    if (active(X + 1, Y, Z)) m |= 1;
    if (active(X, Y + 1, Z)) m |= 2;
    if (ND == 3 && active(X, Y, Z + 1)) m |= 4;
    list[1 + atomicAdd(&list[0].x, 1)] = make_int2(b, m);
  }
}

// Volume fraction crossing the minus-side face of every cell in direction d
// (0 on walls), stored by cell, and in the first pass of a step (H not
// null) the indicator H = [C > 1/2].  G is the arithmetic of the PLIC
// geometry (double in SFX_F64 contexts, float in SFX_F32 contexts: the
// fluxes then carry float rounding, while C and its update stay double and
// the update stays exactly conservative).
template <typename U, typename G, int ND>
__global__ void __launch_bounds__(512)
k_vof_flux(Level L, int d, const int2* __restrict__ list, const double* __restrict__ C,
           const U* __restrict__ u, double dt_h, double* __restrict__ Q,
           unsigned char* __restrict__ H) {
  const size_t st = d == 0 ? 1 : (d == 1 ? (size_t)L.nx : (size_t)L.nx * L.ny);
  const unsigned nb = list ? (unsigned)list[0].x : gridDim.x;
  for (unsigned q = blockIdx.x; q < nb; q += gridDim.x) {
    int x[3];
    if (!CellBlock<ND>::at(L, list ? (unsigned)list[1 + q].x : q, x)) continue;
    const size_t c = cidx(L, x[0], x[1], x[2]);
    const double cq = C[c];
    if (H) H[c] = cq > 0.5 ? 1 : 0;
    double flux = 0.0;
    if (x[d] > 0) {
      // both candidates for the upwind cell are loaded with u
      const double cm = C[c - st];
      const U uf = u[fidx(L, d, x[0], x[1], x[2])];
      if (vbits(cm) != 0 || vbits(cq) != 0) {
        const double cf = widen(uf) * dt_h;
        const bool pos = vbits(cf) > 0;
        const double cu = pos ? cm : cq;
        if (vbits(cf) << 1 != 0 && vbits(cu) > 0) {     // a flow out of a cell with fluid
          const int ui = pos && d == 0 ? x[0] - 1 : x[0];
          const int uj = pos && d == 1 ? x[1] - 1 : x[1];
          const int uk = pos && d == 2 ? x[2] - 1 : x[2];
          G m[3] = {G(0), G(0), G(0)};
          if (vbits(cu) < 0x3ff0000000000000LL) youngs_normal(L, C, ui, uj, uk, m);  // full: no plane
          const G cg = (G)cu;
          flux = pos ? widen(plic_slab<G>(ND, m, cg, d, G(1) - (G)cf, G(1)))
                     : -widen(plic_slab<G>(ND, m, cg, d, G(0), (G)(-cf)));
        }
      }
    }
    Q[c] = flux;
  }
}

template <typename U, int ND>
__global__ void __launch_bounds__(512)
k_vof_update(Level L, int d, const int2* __restrict__ list, const U* __restrict__ u, double dt_h,
             const double* __restrict__ Q, const unsigned char* __restrict__ H,
             double* __restrict__ C) {
  using B = CellBlock<ND>;
  const size_t st = d == 0 ? 1 : (d == 1 ? (size_t)L.nx : (size_t)L.nx * L.ny);
  const unsigned nb = list ? (unsigned)list[0].x : gridDim.x;
  const int ext = d == 0 ? B::bx : (d == 1 ? B::by : B::bz);
  for (unsigned q = blockIdx.x; q < nb; q += gridDim.x) {
    const int2 e = list ? list[1 + q] : make_int2((int)q, 7);
    int x[3];
    if (!B::at(L, (unsigned)e.x, x)) continue;
    const size_t c = cidx(L, x[0], x[1], x[2]);
    // no flux through the far wall and into an inactive block
    const bool plus = x[d] + 1 < L.extent(d) && (x[d] % ext + 1 < ext || (e.y >> d & 1));
    const double Qm = Q[c], Qp = plus ? Q[c + st] : 0.0;
    const bool h = H[c] != 0;
    if (!h && ((vbits(Qm) | vbits(Qp)) << 1) == 0) continue;
    double v = C[c] - (Qp - Qm);
    if (h) {
      const size_t fm = fidx(L, d, x[0], x[1], x[2]);
      const size_t fp = fidx(L, d, x[0] + (d == 0), x[1] + (d == 1), x[2] + (d == 2));
      v += widen(u[fp]) * dt_h - widen(u[fm]) * dt_h;
    }
    C[c] = v;
  }
}

template <typename U, typename G, int ND>
sfx_status vof_impl(sfx_ctx* c, const U* const* u, double dt, int order, double* C,
                    cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  const double dt_h = dt / L.h;
  const size_t nb = CellBlock<ND>::count(L);
  int2* list = nullptr;
  unsigned grid = (unsigned)nb;
  if (L.ncell() >= kVofListCells) {
    const sfx_status st = block_list(c, nb);
    if (st != SFX_OK) return st;
    list = (int2*)c->block_list;
    unsigned char* flag = (unsigned char*)(list + nb + 1);
    SFX_CUDA(cudaMemsetAsync(list, 0, sizeof(int2), s));
    SFX_KERNEL(c, K_OTHER, k_vof_flags<ND>, (unsigned)nb, 512, s, L, C, flag);
    SFX_KERNEL(c, K_OTHER, k_vof_list<ND>, blocks_for(nb, 128), 128, s, L, flag, list);
    grid = (unsigned)std::min(nb, (size_t)c->sm_count * 4);
  }
  for (int q = 0; q < ND; ++q) {
    const int d = order ? ND - 1 - q : q;
    SFX_KERNEL(c, K_OTHER, (k_vof_flux<U, G, ND>), grid, 512, s, L, d, list, C, u[d], dt_h, c->vofQ,
               q == 0 ? c->vofH : nullptr);
    SFX_KERNEL(c, K_OTHER, (k_vof_update<U, ND>), grid, 512, s, L, d, list, u[d], dt_h, c->vofQ,
               c->vofH, C);
  }
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

}  // namespace

sfx_status vof_advect(sfx_ctx* c, const void* ux, const void* uy, const void* uz, double dt,
                      int order, double* C, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  if (!c->vofH) {
    SFX_CUDA(cudaMalloc((void**)&c->vofH, L.ncell()));
    c->allocations.push_back(c->vofH);
    SFX_CUDA(cudaMalloc((void**)&c->vofQ, L.ncell() * sizeof(double)));
    c->allocations.push_back(c->vofQ);
  }
  const bool three = L.ndim() == 3;
  if (c->prec == SFX_F32) {
    const float* u[3] = {(const float*)ux, (const float*)uy, (const float*)uz};
    return three ? vof_impl<float, float, 3>(c, u, dt, order, C, s)
                 : vof_impl<float, float, 2>(c, u, dt, order, C, s);
  }
  const double* u[3] = {(const double*)ux, (const double*)uy, (const double*)uz};
  return three ? vof_impl<double, double, 3>(c, u, dt, order, C, s)
               : vof_impl<double, double, 2>(c, u, dt, order, C, s);
}

}  // namespace sfx
