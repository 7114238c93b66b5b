// Phase-field carrier from the VoF fraction (Sec. 2.5): signed distance by
// Hamilton-Jacobi redistancing, then the tanh profile and its regularised
// delta (Sec. 2.6).
//
// chi0 = 2h(C - 1/2) (positive inside fluid 1).  Each Jacobi step:
//   away from the interface  chi <- chi - dtau s (|grad chi|_G - 1)
//     with s = sign(chi0) and |grad chi|_G the first-order Godunov upwind
//     gradient;
//   in cells whose chi0 changes sign against a face neighbour (the
//   Russo-Smereka sub-cell fix)  chi <- chi - (dtau/h)(s |chi| - d)
//     with d = h chi0 / |Delta chi0| the distance estimated from chi0 alone.
#include <algorithm>
#include <cmath>

#include "sfx_internal.h"

namespace sfx {
namespace {

// phi = (1 - tanh(chi/(2 eps)))/2.  The logistic form 1/(1 + exp(chi/eps))
// takes half the FP64 instructions (512^2 cells: 14.9 against 19.3 us) but
// other last bits, and where phi is within 1e-15 of 1 they set the direction
// of grad phi and with it the drift of f: an expanding sphere's far field
// moved by 1.4e-12 over its run.  The profile keeps its form.
__device__ __forceinline__ double phi_of(double chi, double eps) {
  return 0.5 * (1.0 - tanh(chi / (2.0 * eps)));
}

__device__ __forceinline__ bool same_bits(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}
__device__ __forceinline__ bool same_bits(float a, float b) {
  return __float_as_int(a) == __float_as_int(b);
}

template <typename T> __device__ __forceinline__ T tiny_pos();
template <> __device__ __forceinline__ double tiny_pos<double>() { return 1e-300; }
template <> __device__ __forceinline__ float tiny_pos<float>() { return 1e-30f; }
template <typename T> __device__ __forceinline__ T least_pos();
template <> __device__ __forceinline__ double least_pos<double>() { return __longlong_as_double(1); }
template <> __device__ __forceinline__ float least_pos<float>() { return __int_as_float(1); }

// Whether chi0 (s0 here, zm and zp its neighbours', the cell's own past a wall)
// changes sign against a face neighbour, and then the sub-cell distance
// h chi0/|Delta chi0|.
template <typename T>
__device__ __forceinline__ bool redist_cut(int nd, T s0, const T* zm, const T* zp, const bool* hasm,
                                           const bool* hasp, T h, T& dist) {
  bool cut = false;
  T dsum = 0;
  for (int d = 0; d < nd; ++d) {
    if ((hasm[d] && s0 * zm[d] < (T)0) || (hasp[d] && s0 * zp[d] < (T)0)) cut = true;
    T q = fabs(zp[d] - zm[d]) * (T)0.5;
    q = fmax(q, fabs(zp[d] - s0));
    q = fmax(q, fabs(s0 - zm[d]));
    dsum += q * q;
  }
  if (cut) dist = h * s0 / fmax(sqrt(dsum), (T)tiny_pos<T>());
  return cut;
}

// ------------------------------------------------- redistancing by blocks
// The update reads face neighbours only, so after `iters` steps a cell
// depends on the cells within `iters` of it (in the 1-norm).  Where all of
// those hold one value of C every step just adds dtau to the distance, the
// same for every cell: far from the interface there is nothing to iterate.
// The grid is cut into blocks (32 x 4 x 4 cells, 32 x 16 in 2D); a block is
// rough if one of its cells differs from a face neighbour, and active if a
// rough block lies within ceil(iters / extent) blocks of it.  Only active
// blocks iterate; the others get the value of a uniform field.  A
// neighbour cell in an inactive block still has the value of the cell
// itself whenever it is read (else its block would be active), so it is
// taken as the cell.  The results are those of stepping every cell.
//
// What bounds a step is the FP64 pipe (1/59 of the FP32 rate), so a cell
// costs one FP64 minimum, subtraction, maximum, product and sum per
// direction and a root; the sub-cell distance is formed once (aux), and
// a warp whose cells all equal their neighbours (compared as bits) only
// adds dtau.  Blocks differ in cost (those in the band against flat ones) and
// the FP64 pipe idles in a last wave: a step takes resident blocks of 128
// threads, a quarter of a cell block each, 66 us at 192^3 (four blocks of 512
// threads per SM, of which three fit: 78 us, the SMs active 71 % of it; minima
// of the differences in the integer words instead of the FP64 pipe: 86 us).
// 192^3 sphere of radius 48, 24 steps: 31.5 ms stepping every cell from its
// definition, 1.59 ms with active blocks (the whole phase field 1.93 ms).
constexpr int kBx = 32;
template <int ND>
using RdBlk = CellBlock<ND>;   // (rows of 32 cells per warp stepped 1.6 times as many warps)

struct RdGrid {
  int nbx, nby, nbz;   // blocks per direction
};

// aux of a cell: the sub-cell distance h chi0/|Delta chi0| where chi0
// changes sign against a face neighbour, else an infinity of chi0's sign
// (0 where chi0 is 0).
template <typename T>
__device__ __forceinline__ T rd_inf();
template <> __device__ __forceinline__ double rd_inf<double>() { return __longlong_as_double(0x7ff0000000000000LL); }
template <> __device__ __forceinline__ float rd_inf<float>() { return __int_as_float(0x7f800000); }
// an infinity of x's sign, 0 where x is 0 or NaN (doubles by their integer
// words)
__device__ __forceinline__ double signed_inf(double x) {
  const long long b = __double_as_longlong(x), m = b & 0x7fffffffffffffffLL;
  if (m == 0 || m > 0x7ff0000000000000LL) return 0.0;
  return __longlong_as_double(0x7ff0000000000000LL | (b ^ m));
}
__device__ __forceinline__ float signed_inf(float x) {
  return x > 0.0f ? rd_inf<float>() : (x < 0.0f ? -rd_inf<float>() : 0.0f);
}

// What a uniform field of C = 0 and of C = 1 gives after all steps.
struct RdUniform {
  double chi[2], phi[2], delta[2];
};

template <typename T>
__device__ __forceinline__ T rd_uniform(double h, double C, T dtau, int iters) {
  T x = (T)(2.0 * h * (C - 0.5));
  const T sg = x > (T)0 ? (T)1 : (x < (T)0 ? (T)-1 : (T)0);
  for (int q = 0; q < iters; ++q) x = x + dtau * sg;
  return x;
}

// chi0 (the first iterate) and aux of every cell; rough[b] = 1 where a cell
// of block b differs from a face neighbour in C.  The last block also fills
// uni for the last pass.  (LIST false: chi0 and aux alone, in blocks of 128
// threads that take a quarter of a cell block each.)
template <typename T, int ND, bool LIST>
__global__ void __launch_bounds__(512) k_rd_init(Level L, RdGrid R, const double* __restrict__ C,
                                                 T* __restrict__ aux, T* __restrict__ chi,
                                                 unsigned char* __restrict__ rough, T dtau,
                                                 int iters, double eps, RdUniform* uni) {
  using B = RdBlk<ND>;
  const int nb = R.nbx * R.nby * R.nbz;
  constexpr int sub = LIST ? 1 : 4;
  const int3 lc = B::cell((int)(blockIdx.x % sub * (B::threads / sub) + threadIdx.x));
  const int lx = lc.x, ly = lc.y, lz = lc.z;
  const size_t st[3] = {1, (size_t)L.nx, (size_t)L.nx * L.ny};
  for (int b = (int)blockIdx.x / sub; b < nb; b += (int)gridDim.x / sub) {
    const int i = (b % R.nbx) * kBx + lx, j = (b / R.nbx % R.nby) * B::by + ly,
              k = b / R.nbx / R.nby * B::bz + lz;
    bool diff = false;
    if (i < L.nx && j < L.ny && k < L.nz) {
      const int idx[3] = {i, j, k};
      const size_t c = cidx(L, i, j, k);
      const double c0 = C[c];
      const T s0 = (T)(2.0 * L.h * (c0 - 0.5));
      bool cut = false;
      T q[ND];
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        const bool hm = idx[d] > 0, hp = idx[d] + 1 < L.extent(d);
        const double cm = hm ? C[c - st[d]] : c0, cp = hp ? C[c + st[d]] : c0;
        const bool eq = __double_as_longlong(cm) == __double_as_longlong(c0) &&
                        __double_as_longlong(cp) == __double_as_longlong(c0);
        q[d] = (T)0;
        if (!eq) {
          diff = true;
          const T zm = (T)(2.0 * L.h * (cm - 0.5)), zp = (T)(2.0 * L.h * (cp - 0.5));
          cut = cut || (hm && s0 * zm < (T)0) || (hp && s0 * zp < (T)0);
          // sub-cell estimate of |grad chi0| h along d
          q[d] = fmax(fmax(fabs(zp - zm) * (T)0.5, fabs(zp - s0)), fabs(s0 - zm));
        }
      }
      T a = signed_inf(s0);
      if (cut) {
        T dsum = 0;
#pragma unroll
        for (int d = 0; d < ND; ++d) dsum += q[d] * q[d];
        a = (T)L.h * s0 / fmax(sqrt(dsum), (T)tiny_pos<T>());
        // 0 (next to an infinite C) stands for chi0 = 0: the smallest distance
        if (a == (T)0) a = s0 > (T)0 ? least_pos<T>() : -least_pos<T>();
      }
      aux[c] = a;
      chi[c] = s0;
    }
    if (!LIST) continue;
    diff = __syncthreads_or(diff);
    if (threadIdx.x == 0) rough[b] = diff ? 1 : 0;
  }
  if (LIST && blockIdx.x == gridDim.x - 1 && threadIdx.x < 2) {
    const double x = (double)rd_uniform<T>(L.h, (double)threadIdx.x, dtau, iters), p = phi_of(x, eps);
    uni->chi[threadIdx.x] = x;
    uni->phi[threadIdx.x] = p;
    uni->delta[threadIdx.x] = p * (1.0 - p) / eps;
  }
}

// out[b] = 1 where in[] is set within r blocks of b along direction d
__global__ void k_rd_dilate(RdGrid R, int d, int r, const unsigned char* __restrict__ in,
                            unsigned char* __restrict__ out) {
  const int nb = R.nbx * R.nby * R.nbz;
  const int ext = d == 0 ? R.nbx : (d == 1 ? R.nby : R.nbz);
  const int st = d == 0 ? 1 : (d == 1 ? R.nbx : R.nbx * R.nby);
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
    const int p = b / st % ext;
    unsigned char v = 0;
    for (int q = max(p - r, 0); q <= min(p + r, ext - 1) && !v; ++q) v = in[b + (q - p) * st];
    out[b] = v;
  }
}

// The active blocks, each with a bit per direction whose neighbour block is
// active as well (x-, x+, y-, y+, z-, z+); list[0] counts them (order as it
// falls: the steps do not depend on it).
__global__ void k_rd_list(RdGrid R, const unsigned char* __restrict__ act, int2* __restrict__ list) {
  const int nb = R.nbx * R.nby * R.nbz;
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
    if (!act[b]) continue;
    const int x = b % R.nbx, y = b / R.nbx % R.nby, z = b / R.nbx / R.nby;
    const int sy = R.nbx, sz = R.nbx * R.nby;
    int m = 0;
    if (x > 0 && act[b - 1]) m |= 1;
    if (x + 1 < R.nbx && act[b + 1]) m |= 2;
    if (y > 0 && act[b - sy]) m |= 4;
    if (y + 1 < R.nby && act[b + sy]) m |= 8;
    if (z > 0 && act[b - sz]) m |= 16;
    if (z + 1 < R.nbz && act[b + sz]) m |= 32;
    list[1 + atomicAdd(&list[0].x, 1)] = make_int2(b, m);
  }
}

// A step away from the interface: x0 - dtau s (|grad chi| - 1) with the
// Godunov gradient.  With y = s x the upwind difference along a direction is
// max(0, y0 - min(y-, y+)) (the larger of the two one-sided squares), so a
// direction costs a minimum, a subtraction and one fused multiply-add; signs
// are tested and flipped in the integer words.  A neighbour that is NaN adds
// no slope, as in the definition's maxima with 0.
template <int ND>
__device__ __forceinline__ double rd_step(double a, double x0, const double* xm, const double* xp,
                                          double invh, double dtau) {
  const long long sb = __double_as_longlong(a) & (1LL << 63);
  const double y0 = __longlong_as_double(__double_as_longlong(x0) ^ sb);
  double g = 0.0;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const double ym = __longlong_as_double(__double_as_longlong(xm[d]) ^ sb);
    const double yp = __longlong_as_double(__double_as_longlong(xp[d]) ^ sb);
    double m = y0 - fmin(ym, yp);
    if ((unsigned)__double2hiint(m) > 0x7ff00000u) m = 0.0;   // negative or NaN
    g = fma(m, m, g);
  }
  const double y = fma(-dtau, fma(sqrt(g), invh, -1.0), y0);
  return __longlong_as_double(__double_as_longlong(y) ^ sb);
}
// the float iterate keeps every rounding of the step as defined
template <int ND>
__device__ __forceinline__ float rd_step(float a, float x0, const float* xm, const float* xp,
                                         float invh, float dtau) {
  const float sg = a > 0.0f ? 1.0f : -1.0f;
  float g = 0.0f;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const float m = sg > 0.0f ? x0 - fminf(xm[d], xp[d]) : fmaxf(xm[d], xp[d]) - x0;
    const float t = __fmul_rn(fmaxf(m, 0.0f), invh);
    g = __fadd_rn(g, __fmul_rn(t, t));
  }
  return x0 - dtau * sg * (sqrtf(g) - 1.0f);
}

__device__ __forceinline__ bool is_inf_bits(double a) {
  return (__double_as_longlong(a) & 0x7fffffffffffffffLL) == 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool is_inf_bits(float a) {
  return (__float_as_int(a) & 0x7fffffff) == 0x7f800000;
}
__device__ __forceinline__ bool is_neg_bits(double a) { return __double_as_longlong(a) < 0; }
__device__ __forceinline__ bool is_neg_bits(float a) { return __float_as_int(a) < 0; }

// One Jacobi step of every active block, or (LIST false) of every block.
template <typename T, int ND, bool LIST>
__global__ void __launch_bounds__(512) k_rd_step(Level L, RdGrid R, T dtau,
                                                 const int2* __restrict__ list,
                                                 const T* __restrict__ aux,
                                                 const T* __restrict__ cin, T* __restrict__ cout) {
  using B = RdBlk<ND>;
  const T h = (T)L.h, invh = (T)(1.0 / L.h), dtau_h = dtau / h;
  // blocks of fewer threads take a share of a cell block each
  const int sub = B::threads / (int)blockDim.x, step = (int)gridDim.x / sub;
  const int3 lc = B::cell((int)(blockIdx.x % sub * blockDim.x + threadIdx.x));
  const int lx = lc.x, ly = lc.y, lz = lc.z;
  const int lo[3] = {lx, ly, lz}, last[3] = {kBx - 1, B::by - 1, B::bz - 1};
  const size_t st[3] = {1, (size_t)L.nx, (size_t)L.nx * L.ny};
  const int count = LIST ? list[0].x : R.nbx * R.nby * R.nbz;
  for (int q = (int)blockIdx.x / sub; q < count; q += step) {
    const int2 e = LIST ? list[1 + q] : make_int2(q, 63);
    const int b = e.x;
    const int i = (b % R.nbx) * kBx + lx, j = (b / R.nbx % R.nby) * B::by + ly,
              k = b / R.nbx / R.nby * B::bz + lz;
    if (i >= L.nx || j >= L.ny || k >= L.nz) continue;
    const int idx[3] = {i, j, k};
    const size_t c = cidx(L, i, j, k);
    const T x0 = cin[c], a = aux[c];
    T xm[ND], xp[ND];
    bool flat = true;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      // the cell itself past a wall and for a cell of an inactive block
      const bool hm = idx[d] > 0 && (lo[d] > 0 || (e.y >> (2 * d) & 1));
      const bool hp = idx[d] + 1 < L.extent(d) && (lo[d] < last[d] || (e.y >> (2 * d + 1) & 1));
      xm[d] = hm ? cin[c - st[d]] : x0;
      xp[d] = hp ? cin[c + st[d]] : x0;
      flat = flat && same_bits(xm[d], x0) && same_bits(xp[d], x0);
    }
    T v;
    if (!is_inf_bits(a)) {
      // the sub-cell fix, or chi0 = 0 (the cell stays)
      v = same_bits(a, (T)0) ? x0 : x0 - dtau_h * ((is_neg_bits(a) ? -fabs(x0) : fabs(x0)) - a);
    } else if (flat) {
      v = x0 + (is_neg_bits(a) ? -dtau : dtau);
    } else {
      v = rd_step<ND>(a, x0, xm, xp, invh, dtau);
    }
    cout[c] = v;
  }
}

// chi, phi and delta (may be null) of every cell: active blocks from the
// iterate, the others from `iters` steps of a uniform field, taken once per
// block.  A tanh and two quotients are some sixty FP64 instructions, and
// half of the cells of active blocks are out of the interface's reach (the
// blocks are long in x, the reach is a distance in the 1-norm): those hold
// one of the two values of uni, and warps of them evaluate nothing.  192^3:
// 350 -> 181 us.
template <typename T, int ND>
__global__ void __launch_bounds__(512) k_rd_finish(Level L, RdGrid R, T dtau, int iters, double eps,
                                                   const unsigned char* __restrict__ act,
                                                   const RdUniform* __restrict__ uni,
                                                   const double* C, const T* it, double* chi,
                                                   double* phi, double* delta) {
  using B = RdBlk<ND>;
  __shared__ double u[3];
  const int nb = R.nbx * R.nby * R.nbz;
  const int3 lc = B::cell(threadIdx.x);
  const int lx = lc.x, ly = lc.y, lz = lc.z;
  const RdUniform U = *uni;
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const int i0 = (b % R.nbx) * kBx, j0 = (b / R.nbx % R.nby) * B::by, k0 = b / R.nbx / R.nby * B::bz;
    const bool active = act[b];
    if (!active && threadIdx.x == 0) {
      const double c0 = C[cidx(L, i0, j0, k0)];
      const int one = same_bits(c0, 1.0);
      if (one || same_bits(c0, 0.0)) {
        u[0] = U.chi[one];
        u[1] = U.phi[one];
        u[2] = U.delta[one];
      } else {
        u[0] = (double)rd_uniform<T>(L.h, c0, dtau, iters);
        u[1] = phi_of(u[0], eps);
        u[2] = u[1] * (1.0 - u[1]) / eps;
      }
    }
    __syncthreads();
    const int i = i0 + lx, j = j0 + ly, k = k0 + lz;
    if (i < L.nx && j < L.ny && k < L.nz) {
      const size_t c = cidx(L, i, j, k);
      double x, p, dl;
      if (active) {
        x = (double)it[c];
        const int one = same_bits(x, U.chi[1]);
        if (one || same_bits(x, U.chi[0])) {
          p = one ? U.phi[1] : U.phi[0];
          dl = one ? U.delta[1] : U.delta[0];
        } else {
          p = phi_of(x, eps);
          dl = delta ? p * (1.0 - p) / eps : 0.0;
        }
      } else {
        x = u[0];
        p = u[1];
        dl = u[2];
      }
      chi[c] = x;
      phi[c] = p;
      if (delta) delta[c] = dl;
    }
    __syncthreads();
  }
}

// Up to kRdK Jacobi steps of a 2D grid in one launch: a block loads a
// (kRdX + 2 kRdK) x (kRdY + 2 kRdK) window of chi0 and the iterate into
// shared memory and updates a window that shrinks by one cell per step, so
// that after `steps` steps its kRdX x kRdY core holds exactly the values of
// `steps` single-step launches (the same update of the same operands).  A
// thread keeps its column of the window (80 columns of 12 rows in turn) and
// what does not change with the steps: the sign of chi0, or where chi0
// changes sign the sub-cell distance.  One block per SM at 512^2, so the
// steps are bound by the latency of few warps: 960 threads instead of 256,
// 38 -> 16 us per launch at 512^2 (three launches).  `first`: chi0 and the iterate are formed from
// C here.
constexpr int kRdX = 64, kRdY = 32, kRdK = 8;
constexpr int kRdWX = kRdX + 2 * kRdK, kRdWY = kRdY + 2 * kRdK;
constexpr int kRdRows = 12, kRdPer = kRdWY / kRdRows;
static_assert(kRdWY % kRdRows == 0, "rows per thread");

__global__ void __launch_bounds__(kRdWX* kRdRows)
    k_redistance_fused2d(Level L, float dtau, const double* __restrict__ C, bool first,
                         float* __restrict__ chi0, const float* __restrict__ cin,
                         float* __restrict__ cout, double* __restrict__ chi, int steps) {
  __shared__ float sz[kRdWY][kRdWX];
  __shared__ float sx[2][kRdWY][kRdWX];
  const float h = (float)L.h, invh = (float)(1.0 / L.h), dtau_h = dtau / h;
  const int lx = threadIdx.x % kRdWX, ty = threadIdx.x / kRdWX;
  const int gx = blockIdx.x * kRdX - kRdK + lx, gy0 = blockIdx.y * kRdY - kRdK;
  const bool inx = gx >= 0 && gx < L.nx;
#pragma unroll
  for (int q = 0; q < kRdPer; ++q) {
    const int ly = ty + q * kRdRows, gy = gy0 + ly;
    float z = 0.0f, x = 0.0f;
    if (inx && gy >= 0 && gy < L.ny) {
      const size_t c = (size_t)gy * L.nx + gx;
      if (first) {
        z = x = (float)(2.0 * L.h * (C[c] - 0.5));
        // the core's values of chi0, for the launches after this one
        if (lx >= kRdK && lx < kRdK + kRdX && ly >= kRdK && ly < kRdK + kRdY) chi0[c] = z;
      } else {
        z = chi0[c];
        x = cin[c];
      }
    }
    sz[ly][lx] = z;
    sx[0][ly][lx] = x;
  }
  __syncthreads();
  const bool hm = gx > 0, hp = gx + 1 < L.nx;
  float s[kRdPer], dist[kRdPer];     // sign of chi0; the sub-cell distance where it is cut
  unsigned cut = 0;
#pragma unroll
  for (int q = 0; q < kRdPer; ++q) {
    const int ly = ty + q * kRdRows, gy = gy0 + ly;
    s[q] = dist[q] = 0.0f;
    if (!inx || gy < 0 || gy >= L.ny || lx < 1 || lx >= kRdWX - 1 || ly < 1 || ly >= kRdWY - 1) continue;
    const float s0 = sz[ly][lx];
    const bool hasm[2] = {hm, gy > 0}, hasp[2] = {hp, gy + 1 < L.ny};
    const float zm[2] = {hm ? sz[ly][lx - 1] : s0, gy > 0 ? sz[ly - 1][lx] : s0};
    const float zp[2] = {hp ? sz[ly][lx + 1] : s0, gy + 1 < L.ny ? sz[ly + 1][lx] : s0};
    s[q] = s0 > 0.0f ? 1.0f : (s0 < 0.0f ? -1.0f : 0.0f);
    if (redist_cut<float>(2, s0, zm, zp, hasm, hasp, h, dist[q])) cut |= 1u << q;
  }
  int cur = 0;
  for (int st = 0; st < steps; ++st) {
    // cells at least st + 1 away from the window edge can be updated
    const int lo = st + 1;
    if (inx && lx >= lo && lx < kRdWX - lo) {
#pragma unroll
      for (int q = 0; q < kRdPer; ++q) {
        const int ly = ty + q * kRdRows, gy = gy0 + ly;
        if (ly < lo || ly >= kRdWY - lo || gy < 0 || gy >= L.ny) continue;
        const float x0 = sx[cur][ly][lx];
        float v;
        if (cut >> q & 1) {
          v = x0 - dtau_h * (s[q] * fabsf(x0) - dist[q]);
        } else {
          const float xm[2] = {hm ? sx[cur][ly][lx - 1] : x0, gy > 0 ? sx[cur][ly - 1][lx] : x0};
          const float xp[2] = {hp ? sx[cur][ly][lx + 1] : x0,
                               gy + 1 < L.ny ? sx[cur][ly + 1][lx] : x0};
          v = s[q] == 0.0f ? x0 : rd_step<2>(s[q], x0, xm, xp, invh, dtau);
        }
        sx[cur ^ 1][ly][lx] = v;
      }
    }
    __syncthreads();
    cur ^= 1;
  }
  if (lx < kRdK || lx >= kRdK + kRdX || !inx) return;
#pragma unroll
  for (int q = 0; q < kRdPer; ++q) {
    const int ly = ty + q * kRdRows, gy = gy0 + ly;
    if (ly < kRdK || ly >= kRdK + kRdY || gy < 0 || gy >= L.ny) continue;
    const size_t c = (size_t)gy * L.nx + gx;
    if (chi) chi[c] = (double)sx[cur][ly][lx];      // the last launch
    else cout[c] = sx[cur][ly][lx];
  }
}

// phi and delta from chi, and (chi_out not null) chi from an iterate.  Far from
// the interface chi holds one value over whole blocks, so a block's first cell
// is evaluated once and its value shared: only the band pays an FP64 tanh per
// cell.
template <typename T>
__global__ void __launch_bounds__(256)
k_phi_delta64(size_t n, double eps, const T* chi, double* chi_out, double* phi, double* delta) {
  __shared__ double sx, sp;
  for (size_t b = blockIdx.x * (size_t)blockDim.x; b < n; b += (size_t)gridDim.x * blockDim.x) {
    const size_t c = b + threadIdx.x;
    const double x = c < n ? (double)chi[c] : 0.0;
    if (threadIdx.x == 0) {
      sx = x;
      sp = phi_of(x, eps);
    }
    __syncthreads();
    if (c < n) {
      const double p = same_bits(x, sx) ? sp : phi_of(x, eps);
      if (chi_out) chi_out[c] = x;
      phi[c] = p;
      if (delta) delta[c] = p * (1.0 - p) / eps;
    }
    __syncthreads();
  }
}

}  // namespace

// The redistancing of T iterates by active blocks (see above): a and b are
// iterate buffers, aux the sub-cell distances.  Unless `chi` is one of the
// iterate buffers they are scratch.
template <typename T, int ND>
static sfx_status redistance_blocks(sfx_ctx* c, const double* C, T* aux, T* a, T* b, double* chi,
                                    double* phi, double* delta, int iters, double dtau, double eps,
                                    cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  using B = RdBlk<ND>;
  const RdGrid R{(L.nx + kBx - 1) / kBx, (L.ny + B::by - 1) / B::by, (L.nz + B::bz - 1) / B::bz};
  const size_t nb = (size_t)R.nbx * R.nby * R.nbz;
  int2* list = (int2*)c->block_list;
  RdUniform* uni = (RdUniform*)(list + nb + 1);
  unsigned char* f0 = (unsigned char*)(uni + 1);
  unsigned char* f1 = f0 + nb;
  const int full = (int)std::min(nb, (size_t)c->sm_count * 64);
  // a step: resident blocks of 128 threads, each with a quarter of a cell
  // block in turn (12 to an SM fit by registers)
  constexpr int kStepThreads = 128;
  const size_t sub = B::threads / kStepThreads;
  const int grid = (int)std::min(nb * sub, (size_t)c->sm_count * 12 / sub * sub);
  const int sg = (int)std::min((nb + 255) / 256, (size_t)c->sm_count * 8);
  // where all blocks are resident at once inactive ones cost a step nothing, and
  // finding the active ones four to five launches: every block iterates (7 steps
  // of 35 x 86: 75 -> 58 us, 24 of 15 x 31 x 30 186 -> 163, of 48^3 325 -> 298)
  if (nb * sub <= (size_t)grid) {
    SFX_KERNEL(c, K_PHASE, (k_rd_init<T, ND, false>), grid, kStepThreads, s, L, R, C, aux, a,
               nullptr, (T)dtau, iters, eps, nullptr);
    for (int it = 0; it < iters; ++it) {
      SFX_KERNEL(c, K_PHASE, (k_rd_step<T, ND, false>), grid, kStepThreads, s, L, R, (T)dtau, nullptr,
                 aux, a, b);
      std::swap(a, b);
    }
    SFX_KERNEL(c, K_PHASE, k_phi_delta64<T>, blocks_for(L.ncell(), 256), 256, s, L.ncell(), eps, a, chi,
               phi, delta);
    SFX_LAUNCH_CHECK();
    return SFX_OK;
  }
  SFX_CUDA(cudaMemsetAsync(list, 0, sizeof(int2), s));
  SFX_KERNEL(c, K_PHASE, (k_rd_init<T, ND, true>), full, 512, s, L, R, C, aux, a, f0, (T)dtau,
             iters, eps, uni);
  const int ext[3] = {kBx, B::by, B::bz};
  unsigned char *fi = f0, *fo = f1;
  for (int d = 0; d < ND; ++d) {
    SFX_KERNEL(c, K_PHASE, k_rd_dilate, sg, 256, s, R, d, (iters + ext[d] - 1) / ext[d], fi, fo);
    std::swap(fi, fo);
  }
  SFX_KERNEL(c, K_PHASE, k_rd_list, sg, 256, s, R, fi, list);
  for (int it = 0; it < iters; ++it) {
    SFX_KERNEL(c, K_PHASE, (k_rd_step<T, ND, true>), grid, kStepThreads, s, L, R, (T)dtau, list, aux, a,
               b);
    std::swap(a, b);
  }
  SFX_KERNEL(c, K_PHASE, (k_rd_finish<T, ND>), full, 512, s, L, R, (T)dtau, iters, eps, fi, uni,
             C, a, chi, phi, delta);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

sfx_status block_list(sfx_ctx* c) {
  const Level& L = c->lev[0].lv;
  const size_t nb = L.ndim() == 3 ? CellBlock<3>::count(L) : CellBlock<2>::count(L);
  SFX_CUDA(cudaMalloc(&c->block_list, (nb + 1) * sizeof(int2) + sizeof(RdUniform) + 2 * nb));
  c->allocations.push_back(c->block_list);
  return SFX_OK;
}

sfx_status phase_field_build(sfx_ctx* c, const double* C, double* chi, void* phi, void* delta,
                             int iters, double dtau, double eps, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  const size_t n = L.ncell();
  const int nb = blocks_for(n, 256);
  double *ph = (double*)phi, *de = (double*)delta;
  if (c->prec == SFX_F32 && c->f32.redist32) {
    if (!c->chi32) {
      SFX_CUDA(cudaMalloc((void**)&c->chi32, 3 * n * sizeof(float)));
      c->allocations.push_back(c->chi32);
    }
    float* z0 = c->chi32;
    float* a = c->chi32 + n;
    float* b = c->chi32 + 2 * n;
    if (L.ndim() == 3)
      return redistance_blocks<float, 3>(c, C, z0, a, b, chi, ph, de, iters, dtau, eps, s);
    // kRdK steps per launch; the first forms chi0, the last writes chi (with
    // no step at all, chi0 itself; in place of C only after every block has
    // read it)
    const dim3 fg((unsigned)((L.nx + kRdX - 1) / kRdX), (unsigned)((L.ny + kRdY - 1) / kRdY));
    int it = 0;
    bool first = true, last_in_scratch = false;
    do {
      const int steps = first && chi == C ? 0 : std::min(kRdK, iters - it);
      it += steps;
      SFX_KERNEL(c, K_PHASE, k_redistance_fused2d, fg, kRdWX * kRdRows, s, L, (float)dtau, C, first,
                 z0, a, b, it == iters && !(first && chi == C) ? chi : nullptr, steps);
      last_in_scratch = it == iters && first && chi == C;
      first = false;
      std::swap(a, b);
    } while (it < iters || last_in_scratch);
    SFX_KERNEL(c, K_PHASE, k_phi_delta64<double>, nb, 256, s, n, eps, chi, nullptr, ph, de);
    SFX_LAUNCH_CHECK();
    return SFX_OK;
  }
  // chi may alias C, which the last pass still reads: iterate in scratch
  return L.ndim() == 3
             ? redistance_blocks<double, 3>(c, C, c->chi0, c->chi_tmp, chi, chi, ph, de, iters, dtau, eps, s)
             : redistance_blocks<double, 2>(c, C, c->chi0, c->chi_tmp, chi, chi, ph, de, iters, dtau, eps, s);
}

sfx_status phase_field_from_chi(sfx_ctx* c, const double* chi, double* phi, double* delta,
                                double eps, cudaStream_t s) {
  const size_t n = c->lev[0].lv.ncell();
  SFX_KERNEL(c, K_PHASE, k_phi_delta64<double>, blocks_for(n, 256), 256, s, n, eps, chi, nullptr, phi,
             delta);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

}  // namespace sfx
