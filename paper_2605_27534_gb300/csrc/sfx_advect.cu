// Explicit advection step of Sec. 3.1: xi* = xi - dt div(u xi) with the
// unsplit Bell-Colella-Glaz predictor for the face values.
//
// Face value at a face with normal velocity u and Courant number c = u dt/h:
// take the upwind cell U, extrapolate along the normal over half a step,
//   xi_U + (sign(u) - c)/2 * slope_U       (monotonised-central slope),
// and subtract half a step of transverse advection
//   - dt/2 * vbar_U * (upwinded transverse difference)/h
// with vbar_U the cell-centred transverse velocity.  Inflow walls carry
// bc_in; walls reuse the wall cell (zero gradient) for slopes.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sfx_internal.h"

namespace sfx {
namespace {

template <typename U>
struct Vel {
  const U* u[3];
};

// The step cell by cell, six face values each.  SFX_F64 contexts take phi of
// an ACDI step through it: where phi is a plateau its last bits set how far
// the normal is faded in, and with 1e3 of amplification the curvature (double
// there) moves by 2e-9 when the fluxes are rounded in another order.
// Everywhere else the tiles below give the same step several times faster.
__device__ __forceinline__ double mc_limited(double xm, double x0, double xp) {
  double dl = x0 - xm, dr = xp - x0;
  if (dl * dr <= 0.0) return 0.0;
  double dc = 0.5 * (xp - xm);
  double m = fmin(fabs(dc), 2.0 * fmin(fabs(dl), fabs(dr)));
  return dc > 0.0 ? m : -m;
}

// value of xi at cell idx shifted by s along d (the cell itself outside)
__device__ __forceinline__ double nb(const Level& L, const double* __restrict__ xi,
                                     const int* idx, size_t c, int d, int s) {
  int p = idx[d] + s;
  if (p < 0 || p >= L.extent(d)) return xi[c];
  size_t stride = d == 0 ? 1 : (d == 1 ? (size_t)L.nx : (size_t)L.nx * L.ny);
  return s > 0 ? xi[c + stride] : xi[c - stride];
}

// BCG face value on the face of direction d whose plus-side cell is f
// (f[d] in 0..extent; f[d] = 0 or extent is a wall).
template <typename U>
__device__ double face_value(const Level& L, const Vel<U>& v, double dt,
                             const double* __restrict__ xi, double bc_in, int d, const int* f,
                             double u) {
  int n = L.extent(d);
  int uc[3] = {f[0], f[1], f[2]};
  if (u > 0.0) {
    if (f[d] == 0) return bc_in;
    uc[d] -= 1;
  } else if (f[d] == n) {
    return bc_in;
  }
  size_t U_ = cidx(L, uc[0], uc[1], uc[2]);
  double x0 = xi[U_];
  double sgn = u > 0.0 ? 1.0 : -1.0;
  double slope = mc_limited(nb(L, xi, uc, U_, d, -1), x0, nb(L, xi, uc, U_, d, +1));
  double val = x0 + 0.5 * (sgn - u * dt / L.h) * slope;
  for (int t = 0; t < L.ndim(); ++t) {
    if (t == d) continue;
    int ap[3] = {uc[0], uc[1], uc[2]};
    ap[t] += 1;
    double vbar = 0.5 * ((double)v.u[t][fidx(L, t, uc[0], uc[1], uc[2])] +
                         (double)v.u[t][fidx(L, t, ap[0], ap[1], ap[2])]);
    double dif = vbar > 0.0 ? x0 - nb(L, xi, uc, U_, t, -1) : nb(L, xi, uc, U_, t, +1) - x0;
    val -= 0.5 * dt * vbar * dif / L.h;
  }
  return val;
}

template <typename U>
__global__ void k_advect(Level L, Vel<U> v, double dt, const double* __restrict__ xi,
                         double bc_in, double* __restrict__ out) {
  const size_t n = L.ncell();
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n;
       c += (size_t)gridDim.x * blockDim.x) {
    int idx[3] = {(int)(c % L.nx), (int)((c / L.nx) % L.ny), (int)(c / ((size_t)L.nx * L.ny))};
    double div = 0.0;
    for (int d = 0; d < L.ndim(); ++d) {
      const U* ud = v.u[d];
      double um = (double)ud[fidx(L, d, idx[0], idx[1], idx[2])];
      if (um != 0.0)
        div -= face_area(L, d, idx[0]) * um * face_value(L, v, dt, xi, bc_in, d, idx, um);
      int p[3] = {idx[0], idx[1], idx[2]};
      p[d] += 1;
      double up = (double)ud[fidx(L, d, p[0], p[1], p[2])];
      if (up != 0.0)
        div += face_area(L, d, p[0]) * up * face_value(L, v, dt, xi, bc_in, d, p, up);
    }
    out[c] = xi[c] - dt * div / cell_volume(L, idx[0]);
  }
}

// One step of NF fields (double) that share the velocities.
//
// Per cell and direction a face value needs only the cell value less the
// transverse terms, A_d = x - sum_{t != d} p_t with p_t = dt/(2h) vbar_t
// (upwinded difference along t), and the limited slope s_d; so a thread
// forms both once per cell, each face is evaluated once, by its plus-side
// cell, and the flux is handed to the minus-side cell: along x by warp
// shuffles (a warp is a row of 32 cells), along y through shared memory,
// along z by marching through planes.  A block covers 30 x (TY - 2) cells
// and one ring around them.  What bounds it is the FP64 pipe: 42 FP64
// instructions per cell and field in 3D instead of the 230 of six face
// values per cell, signs and minima taken in the integer words; a cell
// whose neighbours all hold its value bit for bit has no slopes and no
// transverse terms.  160^3 phi with float velocities 3.03 -> 0.635 ms, both fields of a
// 96^3 step 1.27 -> 0.29 ms (six face values per cell before); FP64 pipe 80 % of
// active cycles, 68 instructions per cell with the tiles' rings.
constexpr int kAX = 32;

__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }

// twice the monotonised-central slope: min(|dc|, 4 |dl|, 4 |dr|) with the
// sign of dc = xp - xm = dl + dr, 0 unless dl and dr have one sign.  The
// magnitudes compare as integers; 4 |d| adds 2 to the exponent.
__device__ __forceinline__ double slope2(double dl, double dr, double dc) {
  const long long bl = dbits(dl), br = dbits(dr), mask = 0x7fffffffffffffffLL;
  const long long al = bl & mask, ar = br & mask;
  if ((bl ^ br) < 0 || al == 0 || ar == 0) return 0.0;
  const long long four = 2LL << 52;
  const long long m = min(dbits(dc) & mask, min(al, ar) + four);
  return __longlong_as_double(m | (bl & ~mask));
}

template <int NF>
struct AdvFields {
  const double* x[NF];
  double* out[NF];
  double bc[NF];
};

template <typename U, int G, int NF, int TY>
__global__ void __launch_bounds__(kAX * TY, (NF == 1 ? 2 : 1) * (G == SFX_CART3D ? 16 / TY : 1))
k_bcg64(Level L, Vel<U> v, double dt, AdvFields<NF> P, int zc, unsigned yb, unsigned zb) {
  constexpr int ND = G == SFX_CART3D ? 3 : 2;
  __shared__ double sA[NF][TY][kAX], sS[NF][TY][kAX], sF[NF][TY][kAX];
  const unsigned full = 0xffffffffu;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i = blockIdx.x * (kAX - 2) + tx - 1, j = (int)(yb + blockIdx.y) * (TY - 2) + ty - 1;
  const bool cell = i >= 0 && i < L.nx && j >= 0 && j < L.ny;
  // minus-side faces of the cell, and the far walls' (of cells nx and ny)
  const bool fx = i >= 0 && i <= L.nx && j >= 0 && j < L.ny && tx > 0;
  const bool fy = j >= 0 && j <= L.ny && i >= 0 && i < L.nx && ty > 0;
  const bool inner = cell && tx > 0 && tx < kAX - 1 && ty > 0 && ty < TY - 1;
  const int k0 = ND == 3 ? (int)(zb + blockIdx.z) * zc : 0, k1 = ND == 3 ? min(k0 + zc, L.nz) : 1;
  const double dth = dt / L.h, kk = 0.25 * dth;
  // a radial face's area over V/h
  double wm = 1.0, wp = 1.0;
  if (G == SFX_AXISYM && inner) {
    wm = (double)(2 * i) / (double)(2 * i + 1);
    wp = (double)(2 * i + 2) / (double)(2 * i + 1);
  }
  const size_t sy = L.nx, sz = (size_t)L.nx * L.ny;
  double xb[NF], xc[NF], Az[NF], Sz[NF], acc[NF], xo[NF];   // plane below, this plane; plane k - 1
#pragma unroll
  for (int q = 0; q < NF; ++q) xb[q] = xc[q] = Az[q] = Sz[q] = acc[q] = xo[q] = 0.0;
  const int kb = ND == 3 ? k0 - 1 : 0, ke = ND == 3 ? k1 : 0;   // planes kb .. ke
  if (cell) {
    const size_t c = cidx(L, i, j, max(kb, 0));
#pragma unroll
    for (int q = 0; q < NF; ++q) {
      xc[q] = P.x[q][c];
      xb[q] = ND == 3 && kb > 0 ? P.x[q][c - sz] : xc[q];
    }
  }
  for (int k = kb; k <= ke; ++k) {
    const bool plane = ND == 2 || (k >= 0 && k < L.nz);   // the plane's cells exist
    const bool own = k >= k0 && k < k1;                   // and belong to the block
    const size_t c = cidx(L, i, j, k);
    double um[3] = {0.0, 0.0, 0.0}, kv[3] = {0.0, 0.0, 0.0};
    if (own) {
      if (fx) um[0] = widen(v.u[0][c + (size_t)k * L.ny + j]);
      if (fy) um[1] = widen(v.u[1][c + (size_t)k * L.nx]);
    }
    if (ND == 3 && k >= k0 && inner) um[2] = widen(v.u[2][c]);
    double A[NF][3], S[NF][3], xn[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q) {
      xn[q] = xc[q];
#pragma unroll
      for (int d = 0; d < 3; ++d) A[q][d] = S[q][d] = 0.0;
    }
    if (plane && cell) {
      double m[NF][3], p[NF][3];
      bool flat = true;
#pragma unroll
      for (int q = 0; q < NF; ++q) {
        const double x0 = xc[q];
        m[q][0] = i > 0 ? P.x[q][c - 1] : x0;
        p[q][0] = i + 1 < L.nx ? P.x[q][c + 1] : x0;
        m[q][1] = j > 0 ? P.x[q][c - sy] : x0;
        p[q][1] = j + 1 < L.ny ? P.x[q][c + sy] : x0;
        if (ND == 3) {
          if (k + 1 < L.nz) xn[q] = P.x[q][c + sz];
          m[q][2] = xb[q];
          p[q][2] = xn[q];
        }
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          flat = flat && dbits(m[q][d]) == dbits(x0) && dbits(p[q][d]) == dbits(x0);
          A[q][d] = x0;
        }
      }
      // no slopes, but a velocity that is not finite times 0 is a transverse term
      if (flat) {
        bool ok = finite_bits(v.u[0][c + (size_t)k * L.ny + j]);
        ok &= finite_bits(v.u[0][c + (size_t)k * L.ny + j + 1]);
        ok &= finite_bits(v.u[1][c + (size_t)k * L.nx]);
        ok &= finite_bits(v.u[1][c + (size_t)k * L.nx + L.nx]);
        if (ND == 3) {
          ok &= finite_bits(v.u[2][c]);
          ok &= finite_bits(v.u[2][c + sz]);
        }
        flat = ok;
      }
      if (!flat) {
        // mean velocities of the cell: dt/(2h) vbar
        kv[0] = (widen(v.u[0][c + (size_t)k * L.ny + j]) + widen(v.u[0][c + (size_t)k * L.ny + j + 1])) * kk;
        kv[1] = (widen(v.u[1][c + (size_t)k * L.nx]) + widen(v.u[1][c + (size_t)k * L.nx + L.nx])) * kk;
        if (ND == 3) kv[2] = (widen(v.u[2][c]) + widen(v.u[2][c + sz])) * kk;
#pragma unroll
        for (int q = 0; q < NF; ++q) {
          const double x0 = xc[q];
          double t[3] = {0.0, 0.0, 0.0};
#pragma unroll
          for (int d = 0; d < ND; ++d) {
            const double dl = x0 - m[q][d], dr = p[q][d] - x0;
            S[q][d] = slope2(dl, dr, p[q][d] - m[q][d]);
            t[d] = kv[d] * (dbits(kv[d]) > 0 ? dl : dr);
          }
          A[q][0] = x0 - (ND == 3 ? t[1] + t[2] : t[1]);
          A[q][1] = x0 - (ND == 3 ? t[0] + t[2] : t[0]);
          if (ND == 3) A[q][2] = x0 - (t[0] + t[1]);
        }
      }
    }
    // the face value: bc beyond an inflow wall, else the upwind cell's
    auto face = [&](double u, double AL, double SL, double AR, double SR, bool lo, bool hi,
                    double bc) {
      const bool pos = dbits(u) > 0;
      const double fac = fma(-u, kk, pos ? 0.25 : -0.25);
      double val = fma(fac, pos ? SL : SR, pos ? AL : AR);
      if ((pos && lo) || (!pos && hi)) val = bc;
      return (dbits(u) << 1) == 0 ? 0.0 : u * val;
    };
    double F0[NF];
    if (own) {
#pragma unroll
      for (int q = 0; q < NF; ++q) {
        const double AL = __shfl_up_sync(full, A[q][0], 1), SL = __shfl_up_sync(full, S[q][0], 1);
        F0[q] = fx ? face(um[0], AL, SL, A[q][0], S[q][0], i == 0, i == L.nx, P.bc[q]) : 0.0;
        sA[q][ty][tx] = A[q][1];
        sS[q][ty][tx] = S[q][1];
      }
    }
    __syncthreads();
    double F1[NF];
    if (own) {
#pragma unroll
      for (int q = 0; q < NF; ++q) {
        F1[q] = fy ? face(um[1], sA[q][ty - 1][tx], sS[q][ty - 1][tx], A[q][1], S[q][1], j == 0,
                          j == L.ny, P.bc[q]) : 0.0;
        sF[q][ty][tx] = F1[q];
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NF; ++q) {
      double F2 = 0.0;
      if (ND == 3 && k >= k0 && inner) {
        F2 = face(um[2], Az[q], Sz[q], A[q][2], S[q][2], k == 0, k == L.nz, P.bc[q]);
        if (k > k0) P.out[q][c - sz] = fma(-dth, acc[q] + F2, xo[q]);   // plane k - 1 is complete
      }
      const double Fp = __shfl_down_sync(full, own ? F0[q] : 0.0, 1);
      if (own && inner) {
        const double gx = G == SFX_AXISYM ? wp * Fp - wm * F0[q] : Fp - F0[q];
        acc[q] = gx + (sF[q][ty + 1][tx] - F1[q]);
        xo[q] = xc[q];
        if (ND == 3) acc[q] -= F2;
        else P.out[q][c] = fma(-dth, acc[q], xo[q]);
      }
      Az[q] = A[q][2];
      Sz[q] = S[q][2];
      if (plane) {
        xb[q] = xc[q];
        xc[q] = xn[q];
      }
    }
  }
}

// The 3D tiling: rows per block (16 or 8) and planes per chunk.  A block's
// rows times planes (a chunk steps about 1.5 planes more than it owns) are the
// FP64 work of its SM, so what decides is the most of it that an SM gets,
// over how well its resident warps keep the pipe busy (measured: 80 % with 32
// warp-fields, so w/(w + 8)).  40 x 33 x 50, both fields: six tiles of 16
// rows in chunks of 8 planes 142 us, as chosen here 51; 50 x 64 x 40, one field
// with float velocities: 79 and 39; 160^3 and 96^3 keep 16 rows, 40 and 20 planes.
struct Tiling {
  int ty, zc;
};
inline Tiling bcg64_tiling(const Level& L, int nf, int sms) {
  Tiling best{16, L.nz};
  double cost = 0.0;
  for (int ty = 16; ty >= 8; ty -= 8) {
    const long long tiles = (long long)((L.nx + kAX - 3) / (kAX - 2)) * ((L.ny + ty - 3) / (ty - 2));
    const int fit = (nf == 1 ? 2 : 1) * (16 / ty);      // blocks resident on an SM
    for (int n = 1; n <= std::min(L.nz, 64); ++n) {
      const int z = (L.nz + n - 1) / n;
      const long long per = (tiles * ((L.nz + z - 1) / z) + sms - 1) / sms;
      const double w = (double)(std::min<long long>(per, fit) * ty * nf);
      const double t = (double)(per * ty) * (z + 1.5) * (w + 8.0) / w;
      if (cost == 0.0 || t < cost) cost = t, best = {ty, z};
    }
  }
  return best;
}

template <typename U, int G, int NF, int TY>
void launch_bcg64(sfx_ctx* c, const Vel<U>& v, double dt, const AdvFields<NF>& P, int zc,
                  cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  grid_parts((unsigned)((L.nx + kAX - 3) / (kAX - 2)), (unsigned)((L.ny + TY - 3) / (TY - 2)),
             (unsigned)((L.nz + zc - 1) / zc), [&](dim3 g, unsigned yb, unsigned zb) {
               SFX_KERNEL(c, K_ADVECT, (k_bcg64<U, G, NF, TY>), g, dim3(kAX, TY), s, L, v, dt, P, zc,
                          yb, zb);
             });
}

template <typename U, int NF>
sfx_status bcg64(sfx_ctx* c, const Vel<U>& v, double dt, const AdvFields<NF>& P, cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  if (L.geom == SFX_CART3D) {
    const Tiling t = bcg64_tiling(L, NF, c->sm_count);
    if (t.ty == 16) launch_bcg64<U, SFX_CART3D, NF, 16>(c, v, dt, P, t.zc, s);
    else launch_bcg64<U, SFX_CART3D, NF, 8>(c, v, dt, P, t.zc, s);
  } else if (L.geom == SFX_AXISYM) {
    // shallower tiles: 2D grids are small and want more blocks
    launch_bcg64<U, SFX_AXISYM, NF, 8>(c, v, dt, P, 1, s);
  } else {
    launch_bcg64<U, SFX_PLANAR2D, NF, 8>(c, v, dt, P, 1, s);
  }
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

template <typename U>
__global__ void k_umax(size_t n, const U* __restrict__ u, unsigned long long* slot) {
  double m = 0.0;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n;
       q += (size_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs((double)u[q]));
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) atomic_max_nonneg(slot, m);
}

}  // namespace

sfx_status advect(sfx_ctx* c, const void* ux, const void* uy, const void* uz, double dt,
                  const double* xi, double bc_in, double* out, cudaStream_t s) {
  const AdvFields<1> P{{xi}, {out}, {bc_in}};
  if (c->prec == SFX_F64)
    return bcg64(c, Vel<double>{{(const double*)ux, (const double*)uy, (const double*)uz}}, dt, P, s);
  return bcg64(c, Vel<float>{{(const float*)ux, (const float*)uy, (const float*)uz}}, dt, P, s);
}

sfx_status advect_phi(sfx_ctx* c, const void* ux, const void* uy, const void* uz, double dt,
                      const double* xi, double bc_in, double* out, cudaStream_t s) {
  if (c->prec != SFX_F64) return advect(c, ux, uy, uz, dt, xi, bc_in, out, s);
  const Level& L = c->lev[0].lv;
  const Vel<double> v{{(const double*)ux, (const double*)uy, (const double*)uz}};
  SFX_KERNEL(c, K_ADVECT, k_advect<double>, blocks_for(L.ncell(), 256), 256, s, L, v, dt, xi, bc_in,
             out);
  SFX_LAUNCH_CHECK();
  return SFX_OK;
}

sfx_status advect2(sfx_ctx* c, const double* ux, const double* uy, const double* uz, double dt,
                   const double* f, const double* F, double bc_f, double bc_F, double* fout,
                   double* Fout, cudaStream_t s) {
  return bcg64(c, Vel<double>{{ux, uy, uz}}, dt, AdvFields<2>{{f, F}, {fout, Fout}, {bc_f, bc_F}}, s);
}

sfx_status cfl_umax(sfx_ctx* c, const void* ux, const void* uy, const void* uz, double* umax,
                    cudaStream_t s) {
  const Level& L = c->lev[0].lv;
  SFX_CUDA(cudaMemsetAsync(c->d_norms, 0, 8 * sizeof(unsigned long long), s));
  const void* u[3] = {ux, uy, uz};
  for (int d = 0; d < L.ndim(); ++d) {
    size_t n = L.nface(d);
    if (c->prec == SFX_F64)
      SFX_KERNEL(c, K_OTHER, k_umax<double>, blocks_for(n, 256), 256, s, n, (const double*)u[d], c->d_norms);
    else
      SFX_KERNEL(c, K_OTHER, k_umax<float>, blocks_for(n, 256), 256, s, n, (const float*)u[d], c->d_norms);
  }
  SFX_LAUNCH_CHECK();
  SFX_CUDA(cudaMemcpyAsync(c->h_norms, c->d_norms, sizeof(unsigned long long),
                           cudaMemcpyDeviceToHost, s));
  SFX_CUDA(cudaStreamSynchronize(s));
  unsigned long long b = c->h_norms[0];
  memcpy(umax, &b, sizeof(double));
  return SFX_OK;
}

}  // namespace sfx
