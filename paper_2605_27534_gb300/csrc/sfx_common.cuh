// Shared device helpers of libsfx: grid levels, metric (cell volumes and
// face areas of Sec. 3.2, App. A and App. B), indexing and reductions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sfx.h"

namespace sfx {

constexpr double kPi = 3.14159265358979323846;

// One uniform grid level, passed to kernels by value.
struct Level {
  int geom;
  int nx, ny, nz;
  double h;
  __host__ __device__ int ndim() const { return geom == SFX_CART3D ? 3 : 2; }
  __host__ __device__ size_t ncell() const { return (size_t)nx * ny * nz; }
  __host__ __device__ int extent(int d) const { return d == 0 ? nx : (d == 1 ? ny : nz); }
  __host__ __device__ size_t nface(int d) const {
    return (size_t)(nx + (d == 0)) * (ny + (d == 1)) * (nz + (d == 2));
  }
};

__host__ __device__ inline size_t cidx(const Level& L, int i, int j, int k) {
  return ((size_t)k * L.ny + j) * L.nx + i;
}
// face (i,j,k) in direction d: the face on the minus side of cell (i,j,k)
__host__ __device__ inline size_t fidx(const Level& L, int d, int i, int j, int k) {
  int fx = L.nx + (d == 0), fy = L.ny + (d == 1);
  return ((size_t)k * fy + j) * fx + i;
}

// Cell volume: h^2 (planar, unit depth), h^3 (3D), pi (2i+1) h^3 (ring).
__host__ __device__ inline double cell_volume(const Level& L, int i) {
  double h = L.h;
  if (L.geom == SFX_PLANAR2D) return h * h;
  if (L.geom == SFX_CART3D) return h * h * h;
  return kPi * (double)(2 * i + 1) * h * h * h;
}
// Area of the minus-side face of cell column i in direction d: planar h,
// 3D h^2, axisymmetric radial 2 pi (i h) h, axial pi (2i+1) h^2.
__host__ __device__ inline double face_area(const Level& L, int d, int i) {
  double h = L.h;
  if (L.geom == SFX_PLANAR2D) return h;
  if (L.geom == SFX_CART3D) return h * h;
  if (d == 0) return 2.0 * kPi * (double)i * h * h;
  return kPi * (double)(2 * i + 1) * h * h;
}

// float to double without the conversion instruction, which issues at the
// rate of the FP64 pipe (1/59 of the integer words'): sign, exponent + 896,
// mantissa << 29.  Zeros, denormals, infinities and NaN take the instruction.
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), e = b & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) return (b << 1) == 0u ? __hiloint2double((int)b, 0) : (double)x;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)),
                          (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }
// double to float, rounded to nearest even as the conversion instruction
// does, from the integer words (the same reason); values outside the normal
// floats take the instruction.
__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e - 897u < 253u) {
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29), r = lo & 0x1fffffffu;
    unsigned v = ((e - 896u) << 23) | m;
    if (r > 0x10000000u || (r == 0x10000000u && (m & 1u))) ++v;   // may carry into the exponent
    return __uint_as_float((hi & 0x80000000u) | v);
  }
  return ((hi << 1) | lo) == 0u ? __uint_as_float(hi) : (float)x;
}

// neither NaN nor infinite, from the integer words
__device__ __forceinline__ bool finite_bits(float x) {
  return (__float_as_uint(x) & 0x7f800000u) != 0x7f800000u;
}
__device__ __forceinline__ bool finite_bits(double x) {
  return ((unsigned)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u;
}

// Row r = k ny + j (64-bit division only past 2^32).
__device__ __forceinline__ void row_jk(size_t r, int ny, int& j, int& k) {
  if (r >> 32) {
    k = (int)(r / (size_t)ny);
    j = (int)(r - (size_t)k * ny);
  } else {
    k = (int)((unsigned)r / (unsigned)ny);
    j = (int)((unsigned)r - (unsigned)k * (unsigned)ny);
  }
}

// Blocks of 32 x 4 x 4 cells (32 x 16 in 2D) with 512 threads for kernels
// whose work sits in a band around the interface: a warp holds 8 x 2 x 2
// cells (8 x 4), so that few warps straddle the band's edge.
template <int ND>
struct CellBlock {
  static constexpr int bx = 32, by = ND == 3 ? 4 : 16, bz = ND == 3 ? 4 : 1, threads = 512;
  static __device__ __forceinline__ int3 cell(int t) {
    const int l = t & 31, w = t >> 5;
    return ND == 3 ? make_int3((w & 3) * 8 + (l & 7), (w >> 2 & 1) * 2 + (l >> 3 & 1),
                               (w >> 3) * 2 + (l >> 4))
                   : make_int3((w & 3) * 8 + (l & 7), (w >> 2) * 4 + (l >> 3), 0);
  }
  static __host__ __device__ __forceinline__ size_t count(const Level& L) {
    return (((size_t)L.nx + bx - 1) / bx) * (((size_t)L.ny + by - 1) / by) *
           (((size_t)L.nz + bz - 1) / bz);
  }
  // the cell of this thread (or of thread t) in block b; false past the grid
  static __device__ __forceinline__ bool at(const Level& L, unsigned b, int* x) {
    return at(L, b, x, threadIdx.x);
  }
  static __device__ __forceinline__ bool at(const Level& L, unsigned b, int* x, int t) {
    const unsigned nbx = (L.nx + bx - 1) / bx, nby = (L.ny + by - 1) / by;
    const int3 l = cell(t);
    x[0] = (int)(b % nbx) * bx + l.x;
    x[1] = (int)(b / nbx % nby) * by + l.y;
    x[2] = (int)(b / nbx / nby) * bz + l.z;
    return x[0] < L.nx && x[1] < L.ny && x[2] < L.nz;
  }
};

// ---------------------------------------------------------------- reductions
// Max of non-negative doubles via their bit patterns (order-independent,
// hence deterministic).  NaN sets the flag instead.
__device__ inline void atomic_max_nonneg(unsigned long long* slot, double v) {
  atomicMax(slot, (unsigned long long)__double_as_longlong(v));
}

template <typename T>
__device__ inline T warp_max(T v) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Error-free sum (Knuth two-sum).
__device__ inline void two_sum(double a, double b, double& s, double& e) {
  s = a + b;
  double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// Compensated pair reduction across a warp: (s, c) with value s + c.
__device__ inline void warp_sum_comp(double& s, double& c) {
  for (int o = 16; o > 0; o >>= 1) {
    double so = __shfl_down_sync(0xffffffffu, s, o);
    double co = __shfl_down_sync(0xffffffffu, c, o);
    double t, e;
    two_sum(s, so, t, e);
    s = t;
    c = c + co + e;
  }
}

// Compensated block reduction of (s, c) pairs in a fixed order; thread 0
// receives the block's pair in (s, c).  NT threads per block, a multiple of
// 32.  The first warp adds the others' pairs lane by lane and then across its
// lanes: an FP64 instruction occupies the SM's pipe for 16 cycles however
// few lanes it serves, and a shuffle tree in every warp cost four times as
// many (the totals of a 128^2 grid 17 us, nearly all of it this).
template <int NT>
__device__ __forceinline__ void block_sum_comp(double& s, double& c) {
  __shared__ double ss[NT], sc[NT];
  ss[threadIdx.x] = s;
  sc[threadIdx.x] = c;
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int q = 1; q < NT / 32; ++q) {
      double t, e;
      two_sum(s, ss[threadIdx.x + 32 * q], t, e);
      s = t;
      c += sc[threadIdx.x + 32 * q] + e;
    }
    warp_sum_comp(s, c);
  }
  __syncthreads();
}

// The pairs of `n` blocks (part[2 q], part[2 q + 1]) combined in a fixed
// order by the first warp of a block; lane 0 receives (s, c).
__device__ __forceinline__ void warp_combine(const double* part, int n, double& s, double& c) {
  s = 0.0;
  c = 0.0;
  for (int q = threadIdx.x; q < n; q += 32) {
    double t, e;
    two_sum(s, part[2 * q], t, e);
    s = t;
    c += part[2 * q + 1] + e;
  }
  warp_sum_comp(s, c);
}

// A block's pair stored as block `blk` of `n` for one total; the last block
// to do so combines them and gets true in thread 0, with the pair.  The
// ticket returns to zero for the next launch.
template <int NT>
__device__ __forceinline__ bool last_block_total(double* part, int blk, int n, unsigned* ticket,
                                                 double& s, double& c) {
  block_sum_comp<NT>(s, c);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    part[2 * blk] = s;
    part[2 * blk + 1] = c;
    __threadfence();
    last = atomicAdd(ticket, 1u) == (unsigned)n - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return false;
  __threadfence();
  warp_combine(part, n, s, c);
  if (threadIdx.x == 0) *ticket = 0u;
  return threadIdx.x == 0;
}

// A thread's compensated part of sum V x (blocks in x over the cells).
__device__ __forceinline__ void totals_thread(const Level& L, const double* __restrict__ x,
                                              double& s, double& c) {
  const size_t n = L.ncell();
  s = 0.0;
  c = 0.0;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
       q += (size_t)gridDim.x * blockDim.x) {
    const int i = L.geom == SFX_AXISYM ? (int)(q % (size_t)L.nx) : 0;
    double t, e;
    two_sum(s, cell_volume(L, i) * x[q], t, e);
    s = t;
    c += e;
  }
}

// n is undefined where phi is flat: beyond the redistancing band phi is
// flat up to variations far below its own profile slope phi (1 - phi)/eps,
// whose direction is set by the last bits of phi.  With q = |grad phi| /
// (phi (1 - phi)/eps), n fades out continuously: it is scaled by
// w = clamp(q/kNormalKappa - 1, 0, 1) (0 at or below kNormalKappa, the
// unit vector at or above twice it), and n = 0 where |grad phi| < 1e-30.
// A hard cut-off would make the step jump when a round-off change of phi
// moves q of a band-edge cell across it.
constexpr double kNormalKappa = 1e-3;

__device__ __forceinline__ double normal_fade(double m, double slope) {
  return m < 1e-30 ? 0.0 : fmin(fmax(m / (kNormalKappa * slope) - 1.0, 0.0), 1.0);
}

// Appends the indices of the lanes with `take` to list (list[0] counts), one
// atomic per warp; every lane of the warp calls it.
__device__ __forceinline__ void warp_append(unsigned* list, bool take, unsigned v) {
  const unsigned m = __ballot_sync(0xffffffffu, take);
  if (!m) return;
  const int lane = threadIdx.x & 31, lead = __ffs(m) - 1;
  unsigned base = 0;
  if (lane == lead) base = atomicAdd(list, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, lead);
  if (take) list[1 + base + __popc(m & ((1u << lane) - 1))] = v;
}

// Unit normal grad phi / |grad phi| at cell x: centred differences,
// zero-gradient walls, faded out where phi is flat (above).
__device__ __forceinline__ void unit_normal64(const Level& L, const double* __restrict__ phi,
                                              const int* x, double eps, double* n) {
  double g[3] = {0.0, 0.0, 0.0};
  const double inv2h = 0.5 / L.h;
  const int i = x[0], j = x[1], k = x[2];
  int ip = min(i + 1, L.nx - 1), im = max(i - 1, 0);
  int jp = min(j + 1, L.ny - 1), jm = max(j - 1, 0);
  g[0] = (phi[cidx(L, ip, j, k)] - phi[cidx(L, im, j, k)]) * inv2h;
  g[1] = (phi[cidx(L, i, jp, k)] - phi[cidx(L, i, jm, k)]) * inv2h;
  if (L.geom == SFX_CART3D) {
    int kp = min(k + 1, L.nz - 1), km = max(k - 1, 0);
    g[2] = (phi[cidx(L, i, j, kp)] - phi[cidx(L, i, j, km)]) * inv2h;
  }
  const double m = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
  const double pc = phi[cidx(L, i, j, k)];
  const double slope = pc * (1.0 - pc) / eps;
  const double w = normal_fade(m, slope);
  for (int d = 0; d < 3; ++d) n[d] = w > 0.0 ? w * (g[d] / m) : 0.0;
}

}  // namespace sfx
