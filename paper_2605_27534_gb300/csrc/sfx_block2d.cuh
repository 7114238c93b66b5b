// All sweeps of a Newton correction on a 2D tile in one launch.
//
// The colour launches of an iteration (black, then red and black in turn, S
// sweeps, 2S - 1 launches) are each a few microseconds of latency on a 2D
// grid, and on large batches re-read the same residuals and faces from L2.
// A block here loads a tile and a halo of 2S - 1 cells into shared memory
// (the residuals with the exchange Jacobian, the half faces and the red
// half-sweep of the residual pass), runs every colour on a region that
// shrinks by one cell per colour, and adds the corrections of its tile to the
// state.  A cell's update is the one of the colour launches on the same
// operands, so the result is theirs bit for bit; neighbouring tiles compute
// their common halo cells alike.  The extra cells (a factor of 1.6 at four
// sweeps, none across an extent that fits the tile) cost FP32 arithmetic,
// which was idle.  Before and after, per Newton iteration: 128^2 (FP64 context)
// 7 launches of 2.0 us -> 6.3 us, 512 columns of 5 launches 58 -> 31 us, 512^2
// 18 -> 11 us, a batch of 64 cylindrical grids 120 -> 102 us.
#pragma once

#include "sfx_f32_dev.cuh"

namespace sfx {

// Tile of a grid: tx x ty cells (tx even or the whole extent).
struct Tile2D {
  int tx = 0, ty = 0;
};
constexpr int kT2Threads = 512;
constexpr int kT2Width = 64;            // cells of a row with its halo
constexpr size_t kT2Smem = 100 * 1024;  // two blocks per SM

inline size_t tile2d_smem(int nx, int ny, const Tile2D& t, int sweeps) {
  const int P = 2 * sweeps - 1, Pe = P + 1;
  const size_t wp = (size_t)(std::min(nx, t.tx + 2 * Pe) + 1) / 2, h = (size_t)std::min(ny, t.ty + 2 * P);
  return h * wp * 2 * (16 + 8) + h * (2 * wp + 1) * 4 + (h + 1) * 2 * wp * 4 + 16;
}

// Rows per tile for a set of grids (nx, ny): the fewest waves of two blocks
// per SM times the rows a block steps (its own, half its halo and about eight
// rows' worth of loads and barriers), within kT2Smem.  ty = 0 where no tile
// fits (many sweeps on a wide grid): the colour launches stay.
template <class Grid>
inline int tile2d_rows(const Grid* g, int n, int sweeps, int sms) {
  const int P = 2 * sweeps - 1;
  int best = 0;
  double cost = 0.0;
  for (int ty = 4; ty <= 512; ty += 4) {
    long long tiles = 0;
    bool fits = true;
    for (int q = 0; q < n && fits; ++q) {
      const int tx = g[q].nx <= kT2Width ? g[q].nx : kT2Width - 2 * (P + 1);
      fits = tx >= 32 || g[q].nx <= kT2Width;
      if (!fits) break;
      fits = tile2d_smem(g[q].nx, g[q].ny, Tile2D{tx, ty}, sweeps) <= kT2Smem;
      tiles += (long long)((g[q].nx + tx - 1) / tx) * ((g[q].ny + ty - 1) / ty);
    }
    if (!fits) break;
    const double c = (double)((tiles + 2 * sms - 1) / (2 * sms)) * (ty + P + 8);
    if (!best || c < cost) {
      best = ty;
      cost = c;
    }
  }
  return best;
}
inline Tile2D tile2d_of(int nx, int ty, int sweeps) {
  return Tile2D{nx <= kT2Width ? nx + (nx & 1) : kT2Width - 4 * sweeps, ty};
}

namespace {

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

// put(c, e): adds the correction e = (e_f, e_F) of cell c to the state.
template <int G, class Put>
__device__ __forceinline__ void corr_tile2d(const Nw32& p, int x0, int y0, int tx, int ty,
                                            int sweeps, const __half2* __restrict__ Hx,
                                            const __half2* __restrict__ Hy,
                                            const float4* __restrict__ rc,
                                            const float2* __restrict__ e2, Put put) {
  extern __shared__ __align__(16) unsigned char t2smem[];
  const Level& L = p.L;
  const int P = 2 * sweeps - 1, Pe = P + 1;
  const int xs = max(0, x0 - Pe), xe = min(L.nx, x0 + tx + Pe);
  const int ys = max(0, y0 - P), ye = min(L.ny, y0 + ty + P);
  const int Wp = (xe - xs + 1) / 2, H = ye - ys, n = H * Wp;
  float4* R = reinterpret_cast<float4*>(t2smem);           // [colour][row][pair]
  float2* E = reinterpret_cast<float2*>(R + 2 * n);        // the same
  __half2* X = reinterpret_cast<__half2*>(E + 2 * n);      // minus-x faces [row][2 Wp + 1]
  __half2* Y = X + H * (2 * Wp + 1);                       // minus-y faces [row][2 Wp]
  const int rps = blockDim.x / Wp;                         // rows the block takes at once
  const int px = threadIdx.x % Wp, pr = threadIdx.x / Wp;
  const bool act = pr < rps;
  const int half = (L.nx + 1) >> 1;
  const size_t plane = (size_t)L.ny * half;
  const int i0 = xs + 2 * px;
  if (act) {
    for (int r = pr; r <= H; r += rps) {
      const int j = ys + r;
      const __half2* gy = Hy + (size_t)j * L.nx + i0;
      cp_async4(&Y[r * 2 * Wp + 2 * px], gy);
      if (i0 + 1 < L.nx) cp_async4(&Y[r * 2 * Wp + 2 * px + 1], gy + 1);
      if (r == H) break;
      const size_t g = (size_t)j * half + (i0 >> 1);
      const int o = r * Wp + px;
      cp_async16(&R[o], rc + g);
      cp_async16(&R[n + o], rc + plane + g);
      cp_async8(&E[o], e2 + g);
      E[n + o] = make_float2(0.0f, 0.0f);
      const __half2* gx = Hx + (size_t)j * (L.nx + 1) + i0;
      __half2* X0 = &X[r * (2 * Wp + 1) + 2 * px];
      cp_async4(X0, gx);
      cp_async4(X0 + 1, gx + 1);
      if (px == Wp - 1 && i0 + 2 <= L.nx) cp_async4(X0 + 2, gx + 2);
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  for (int k = 0; k < P; ++k) {
    const int color = k & 1 ? 0 : 1, m = P - 1 - k;
    const int xa = x0 - m, xb = min(L.nx, x0 + tx + m);
    const int ra = max(0, y0 - m) - ys, rb = min(L.ny, y0 + ty + m) - ys;
    float2* own = E + color * n;
    const float2* oth = E + (1 - color) * n;
    if (act) {
      for (int r = pr; r < rb; r += rps) {
        const int j = ys + r, i = i0 + ((j + color) & 1);
        if (r < ra || i < xa || i >= xb) continue;
        const int o = r * Wp + px, a = i & 1, li = i - xs;
        const bool has[6] = {i > 0, i + 1 < L.nx, j > 0, j + 1 < L.ny, false, false};
        const float2 z = make_float2(0.0f, 0.0f);
        const float2 en[6] = {has[0] ? oth[o - 1 + a] : z, has[1] ? oth[o + a] : z,
                              has[2] ? oth[o - Wp] : z, has[3] ? oth[o + Wp] : z, z, z};
        const __half2* fx = X + r * (2 * Wp + 1) + li;
        const __half2* fy = Y + r * 2 * Wp + li;
        const float2 B[6] = {has[0] ? __half22float2(fx[0]) : z, has[1] ? __half22float2(fx[1]) : z,
                             has[2] ? __half22float2(fy[0]) : z,
                             has[3] ? __half22float2(fy[2 * Wp]) : z, z, z};
        const float2 ec = own[o];
        float2 dg;
        const float2 fl = flux_lin2<G>(L, p.invh, make_float2(p.Dfh, p.DFh), p.literal, i, ec, en,
                                       has, B, dg);
        float2 ne = corr2_block(p, R[color * n + o], ec, fl, dg);
        if (color == 0) ne = relax_red(p, ne, ec);
        own[o] = ne;
      }
    }
    __syncthreads();
  }
  if (!act) return;
  for (int r = y0 - ys + pr; r < min(L.ny, y0 + ty) - ys; r += rps) {
    const int j = ys + r;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = i0 + q;
      if (i < x0 || i >= min(L.nx, x0 + tx)) continue;
      put((ix)j * (ix)L.nx + (ix)i, E[((i + j) & 1) * n + r * Wp + px]);
    }
  }
}

}  // namespace
}  // namespace sfx
