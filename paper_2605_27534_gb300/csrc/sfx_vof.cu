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

// Only cells near fluid 1 change.  Every flux out of a cell with C <= 0 is
// zero, so a block of cells (32 x 4 x 4; 32 x 16 in 2D) without fluid 1 in
// itself or an adjacent block stays as it is through the step (a pass moves
// fluid by one cell along its direction).  On large grids the blocks are
// classified once per step and the passes run over a list of the active
// ones; small grids, where a launch costs more than the sweep, take every
// block.  What bounds a flux pass is the PLIC geometry (about 2000
// instructions in a chain for a plane offset where C is within float rounding
// of 0 or 1, as in a third of a drop's interior), so on large grids the faces
// that need it are listed first and then taken by full warps (gathered per
// block instead, the other warps of a block waited for the chains); signs and
// the tests for empty and full cells read the integer words and floats are
// widened without the conversion instruction, which issues at the FP64 rate.
// 256^3 sphere of radius 64 in float: 2.45 ms per step with every face and
// cell, 0.46 ms now (planes 69, other faces 39, update 24 us per direction,
// classification 30 us), 0.72 ms after 500 steps of wisps.  The geometry is
// inlined once per kernel, for the flow in either direction: twice, its code
// did not fit the instruction cache (planes 102 us; small grids, where a pass
// lasts one chain, 28 us instead of 24).
constexpr size_t kVofListCells = (size_t)1 << 20;

__device__ __forceinline__ long long vbits(double v) { return __double_as_longlong(v); }

// a cell that may give fluid: C > 0, or NaN of either sign
__device__ __forceinline__ bool wet(double C) {
  const long long b = vbits(C);
  return b > 0 || (unsigned long long)b > 0xfff0000000000000ULL;
}

__device__ __forceinline__ bool positive(double x) {   // false for NaN
  return (unsigned long long)vbits(x) - 1ULL < 0x7ff0000000000000ULL;
}

template <typename U>
struct VofVel {
  const U* u[3];
};

// list[0].y = 1 where a velocity is not finite: H (c_+ - c_-) of its cells is
// NaN then, with H = 0 too, and the passes behind it visit every block.  Block
// b of nb.
template <typename U, int ND>
__device__ __forceinline__ void vof_finite(const Level& L, const VofVel<U>& v, unsigned b,
                                           unsigned nb, int2* __restrict__ list) {
  constexpr int per = 16 / sizeof(U);
  struct alignas(16) Pack {
    U x[per];
  };
  bool ok = true;
  const size_t t0 = (size_t)b * blockDim.x + threadIdx.x, step = (size_t)nb * blockDim.x;
  for (int d = 0; d < ND; ++d) {
    const U* u = v.u[d];
    const size_t n = L.nface(d), m = ((size_t)u & 15) == 0 ? n / per : 0;
    size_t t = t0;
    for (; t + 7 * step < m; t += 8 * step) {
      Pack q[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) q[k] = reinterpret_cast<const Pack*>(u)[t + k * step];
#pragma unroll
      for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int e = 0; e < per; ++e) ok &= finite_bits(q[k].x[e]);
    }
    for (; t < m; t += step) {
      const Pack q = reinterpret_cast<const Pack*>(u)[t];
#pragma unroll
      for (int e = 0; e < per; ++e) ok &= finite_bits(q.x[e]);
    }
    for (t = m * per + t0; t < n; t += step) ok &= finite_bits(u[t]);
  }
  if (!ok) list[0].y = 1;
}
template <typename U, int ND>
__global__ void __launch_bounds__(128) k_vof_finite(Level L, VofVel<U> v, int2* list) {
  vof_finite<U, ND>(L, v, blockIdx.x, gridDim.x, list);
}

// flag[b] = 1 where block b holds fluid 1: a warp per block, its 16 rows of
// 32 cells in flight together
template <int ND>
__global__ void __launch_bounds__(256) k_vof_flags(Level L, unsigned nb, const double* __restrict__ C,
                                                   unsigned char* __restrict__ flag) {
  using B = CellBlock<ND>;
  const unsigned b = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (b >= nb) return;
  const unsigned nbx = (L.nx + B::bx - 1) / B::bx, nby = (L.ny + B::by - 1) / B::by;
  const int i = (int)(b % nbx) * B::bx + (threadIdx.x & 31);
  const int j0 = (int)(b / nbx % nby) * B::by, k0 = (int)(b / nbx / nby) * B::bz;
  bool any = false;
  if (i < L.nx) {
#pragma unroll
    for (int r = 0; r < B::by * B::bz; ++r) {
      const int j = j0 + r % B::by, k = k0 + r / B::by;
      if (j < L.ny && k < L.nz) any |= wet(C[cidx(L, i, j, k)]);
    }
  }
  any = __any_sync(0xffffffffu, any);
  if ((threadIdx.x & 31) == 0) flag[b] = any ? 1 : 0;
}

// act[b] = 1 where block b or a neighbour (diagonals included) is flagged
template <int ND>
__global__ void k_vof_active(Level L, const unsigned char* __restrict__ flag,
                             unsigned char* __restrict__ act) {
  using B = CellBlock<ND>;
  const int nx = (L.nx + B::bx - 1) / B::bx, ny = (L.ny + B::by - 1) / B::by,
            nz = (L.nz + B::bz - 1) / B::bz;
  const int nb = nx * ny * nz;
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
    const int X = b % nx, Y = b / nx % ny, Z = b / nx / ny;
    unsigned v = 0;
#pragma unroll
    for (int q = 0; q < (ND == 3 ? 27 : 9); ++q) {
      const int a = min(max(X + q % 3 - 1, 0), nx - 1), e = min(max(Y + q / 3 % 3 - 1, 0), ny - 1),
                f = min(max(Z + q / 9 - (ND == 3), 0), nz - 1);
      v |= flag[(f * ny + e) * nx + a];
    }
    act[b] = (unsigned char)v;
  }
}

// A bit per direction whose plus-side neighbour of block b is active too.
template <int ND>
__device__ __forceinline__ int vof_plus(const Level& L, const unsigned char* __restrict__ act,
                                        int b) {
  using B = CellBlock<ND>;
  const int nx = (L.nx + B::bx - 1) / B::bx, ny = (L.ny + B::by - 1) / B::by,
            nz = (L.nz + B::bz - 1) / B::bz;
  const int X = b % nx, Y = b / nx % ny, Z = b / nx / ny;
  int m = 0;
  if (X + 1 < nx && act[b + 1]) m |= 1;
  if (Y + 1 < ny && act[b + nx]) m |= 2;
  if (ND == 3 && Z + 1 < nz && act[b + nx * ny]) m |= 4;
  return m;
}

// The active blocks with those bits; list[0].x counts them.
template <int ND>
__global__ void k_vof_list(Level L, const unsigned char* __restrict__ act, int2* __restrict__ list) {
  const int nb = (int)CellBlock<ND>::count(L);
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x)
    if (act[b]) list[1 + atomicAdd(&list[0].x, 1)] = make_int2(b, vof_plus<ND>(L, act, b));
}

// Flux through the minus-side face of cell x in direction d (not a wall)
// from its upwind cell's plane.
template <typename U, typename G, int ND>
__device__ __forceinline__ double plic_flux(const Level& L, int d, const int* x, size_t st,
                                            const double* __restrict__ C,
                                            const U* __restrict__ u, double dt_h) {
  const size_t c = cidx(L, x[0], x[1], x[2]);
  const double cf = widen(u[fidx(L, d, x[0], x[1], x[2])]) * dt_h;
  const bool pos = positive(cf);
  int y[3] = {x[0], x[1], x[2]};
  if (pos) y[d] -= 1;
  G m[3];
  youngs_normal(L, C, y[0], y[1], y[2], m);
  const G g = (G)cf;
  const double v = widen(plic_slab<G>(ND, m, (G)C[pos ? c - st : c], d, pos ? G(1) - g : G(0),
                                      pos ? G(1) : -g));
  return pos ? v : -v;
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
           unsigned char* __restrict__ H, unsigned* __restrict__ cut) {
  const size_t st = d == 0 ? 1 : (d == 1 ? (size_t)L.nx : (size_t)L.nx * L.ny);
  // blocks of fewer threads take a share of a cell block each
  const unsigned sub = (unsigned)CellBlock<ND>::threads / blockDim.x, step = gridDim.x / sub;
  const int t = (int)(blockIdx.x % sub * blockDim.x + threadIdx.x);
  const bool every = list && list[0].y;   // NaN may come from any block (vof_finite)
  const unsigned nb = !list ? step : every ? (unsigned)CellBlock<ND>::count(L) : (unsigned)list[0].x;
  for (unsigned q = blockIdx.x / sub; q < nb; q += step) {
    const unsigned blk = list && !every ? (unsigned)list[1 + q].x : q;
    int x[3];
    bool plane = false;
    size_t c = 0;
    if (CellBlock<ND>::at(L, blk, x, t)) {
      c = cidx(L, x[0], x[1], x[2]);
      const double cq = C[c];
      if (H) H[c] = cq > 0.5 ? 1 : 0;
      double flux = 0.0;
      if (x[d] > 0) {
        // both candidates for the upwind cell are loaded with u
        const double cm = C[c - st];
        const U uf = u[fidx(L, d, x[0], x[1], x[2])];
        const double cu = uf > U(0) ? cm : cq;
        if (uf != U(0) && wet(cu)) {           // a flow out of a cell with fluid
          const double cf = widen(uf) * dt_h;
          // no plane in a cell that is full, in float also within rounding
          if (!((G)cu < G(1))) {
            // (plic_slab of a cell with C >= 1; a NaN is no fraction: C (b - a))
            const G g = (G)cf, w = positive(cf) ? G(1) - (G(1) - g) : -g;
            flux = widen((G)cu >= G(1) ? w : (G)cu * w);
            if (!positive(cf)) flux = -flux;
          } else {
            plane = true;
          }
        }
      }
      if (!plane) Q[c] = flux;
      else if (!cut) Q[c] = plic_flux<U, G, ND>(L, d, x, st, C, u, dt_h);
    }
    if (cut) warp_append(cut, plane, (unsigned)c);
  }
}

// The listed faces (cells whose minus-side face in direction d needs a
// plane): cut[0] of them.  In the first direction the first `look` blocks read
// the velocities instead (vof_finite): the chains of the planes leave HBM idle.
template <typename U, typename G, int ND>
__global__ void __launch_bounds__(128)
k_vof_planes(Level L, int d, const double* __restrict__ C, const U* __restrict__ u, double dt_h,
             const unsigned* __restrict__ cut, double* __restrict__ Q, unsigned look, VofVel<U> v,
             int2* __restrict__ list) {
  if (blockIdx.x < look) {
    vof_finite<U, ND>(L, v, blockIdx.x, look, list);
    return;
  }
  const unsigned n = cut[0], blocks = gridDim.x - look;
  const size_t st = d == 0 ? 1 : (d == 1 ? (size_t)L.nx : (size_t)L.nx * L.ny);
  for (unsigned q = (blockIdx.x - look) * blockDim.x + threadIdx.x; q < n; q += blocks * blockDim.x) {
    const unsigned c = cut[1 + q];
    const int x[3] = {(int)(c % (unsigned)L.nx), (int)(c / (unsigned)L.nx % (unsigned)L.ny),
                      (int)(c / (unsigned)L.nx / (unsigned)L.ny)};
    Q[c] = plic_flux<U, G, ND>(L, d, x, st, C, u, dt_h);
  }
}

template <typename U, int ND>
__global__ void __launch_bounds__(512)
k_vof_update(Level L, int d, bool first, const int2* __restrict__ list,
             const unsigned char* __restrict__ act, const U* __restrict__ u, double dt_h,
             const double* __restrict__ Q, const unsigned char* __restrict__ H,
             double* __restrict__ C) {
  using B = CellBlock<ND>;
  const size_t st = d == 0 ? 1 : (d == 1 ? (size_t)L.nx : (size_t)L.nx * L.ny);
  const int ext = d == 0 ? B::bx : (d == 1 ? B::by : B::bz);
  const bool every = list && list[0].y, all = !list || every;   // velocities may not be finite
  const unsigned nb = !list ? gridDim.x : every ? (unsigned)B::count(L) : (unsigned)list[0].x;
  for (unsigned q = blockIdx.x; q < nb; q += gridDim.x) {
    // (the fluxes of the first direction took the active blocks only)
    const int2 e = !list || (every && !first) ? make_int2((int)q, 7)
                   : every ? make_int2((int)q, vof_plus<ND>(L, act, (int)q)) : list[1 + q];
    const bool active = !every || act[q], fluxes = active || !first;
    int x[3];
    if (!B::at(L, (unsigned)e.x, x)) continue;
    const size_t c = cidx(L, x[0], x[1], x[2]);
    // no flux through the far wall and into an inactive block
    const bool plus = x[d] + 1 < L.extent(d) && (x[d] % ext + 1 < ext || (e.y >> d & 1));
    const double Qm = fluxes ? Q[c] : 0.0, Qp = fluxes && plus ? Q[c + st] : 0.0;
    const bool h = active && H[c] != 0;
    const bool flux = ((vbits(Qm) | vbits(Qp)) << 1) != 0;
    if (!h && !all && !flux) continue;
    double v = C[c] - (Qp - Qm);
    if (h || all) {
      const size_t fm = fidx(L, d, x[0], x[1], x[2]);
      const size_t fp = fidx(L, d, x[0] + (d == 0), x[1] + (d == 1), x[2] + (d == 2));
      const U um = u[fm], up = u[fp];
      if (h) v += widen(up) * dt_h - widen(um) * dt_h;
      else if (!finite_bits(up) || !finite_bits(um)) v = __longlong_as_double(0x7ff8000000000000LL);
      else if (!flux) continue;
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
  unsigned* cut = nullptr;
  const unsigned char* act = nullptr;
  const VofVel<U> v{{u[0], u[1], u[2]}};
  if (c->vof_blocks) {
    cut = cell_list(c, &c->vof_cut, 1, s);
    list = (int2*)c->vof_blocks;
    unsigned char* flag = (unsigned char*)(list + nb + 1);
    act = flag + nb;
    SFX_CUDA(cudaMemsetAsync(list, 0, sizeof(int2), s));
    SFX_KERNEL(c, K_OTHER, k_vof_flags<ND>, (unsigned)((nb + 7) / 8), 256, s, L, (unsigned)nb, C, flag);
    SFX_KERNEL(c, K_OTHER, k_vof_active<ND>, blocks_for(nb, 128), 128, s, L, flag, flag + nb);
    SFX_KERNEL(c, K_OTHER, k_vof_list<ND>, blocks_for(nb, 128), 128, s, L, flag + nb, list);
    grid = (unsigned)std::min(nb, (size_t)c->sm_count * 4);
  }
  for (int q = 0; q < ND; ++q) {
    const int d = order ? ND - 1 - q : q;
    if (cut) SFX_CUDA(cudaMemsetAsync(cut, 0, sizeof(unsigned), s));
    // without a list a block lasts as long as its longest chain: small ones
    SFX_KERNEL(c, K_OTHER, (k_vof_flux<U, G, ND>), list ? grid : 4 * grid, list ? 512 : 128, s, L, d,
               list, C, u[d], dt_h, c->vofQ, q == 0 ? c->vofH : nullptr, cut);
    const unsigned look = list && q == 0 ? (unsigned)c->sm_count * 2 : 0;
    if (cut)
      SFX_KERNEL(c, K_OTHER, (k_vof_planes<U, G, ND>), c->sm_count * 16 + look, 128, s, L, d, C, u[d],
                 dt_h, cut, c->vofQ, look, v, list);
    else if (look)
      SFX_KERNEL(c, K_OTHER, (k_vof_finite<U, ND>), look, 128, s, L, v, list);
    SFX_KERNEL(c, K_OTHER, (k_vof_update<U, ND>), grid, 512, s, L, d, q == 0, list, act, u[d],
               dt_h, c->vofQ, c->vofH, C);
  }
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

}  // namespace

sfx_status vof_advect(sfx_ctx* c, const void* ux, const void* uy, const void* uz, double dt,
                      int order, double* C, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  const bool three = L.ndim() == 3;
  if (!c->vofH) {
    SFX_CUDA(cudaMalloc((void**)&c->vofH, L.ncell()));
    c->allocations.push_back(c->vofH);
  }
  if (!c->vofQ) {
    SFX_CUDA(cudaMalloc((void**)&c->vofQ, L.ncell() * sizeof(double)));
    c->allocations.push_back(c->vofQ);
    // (without memory for the list every block is taken)
    const size_t nb = three ? CellBlock<3>::count(L) : CellBlock<2>::count(L);
    if (L.ncell() >= kVofListCells) {
      if (cudaMalloc(&c->vof_blocks, (nb + 1) * sizeof(int2) + 2 * nb) == cudaSuccess) {
        c->allocations.push_back(c->vof_blocks);
      } else {
        c->vof_blocks = nullptr;
        cudaGetLastError();
      }
    }
  }
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
