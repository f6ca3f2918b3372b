// Tiled V-cycle passes of the 2D levels, shared by the single-design V-cycle
// (FP32 and FP64) and the batched one.  Each pass of Table 1 used to be a
// kernel of its own that gathered every operand of a node from global memory
// with bounds and Dirichlet tests per neighbour; the finest level's passes ran
// at 4-6 times their bytes' time and the coarse ones at the latency of a
// launch.  A block here stages a tile with its rim in shared memory (off-grid
// and fixed neighbours as zeros, so the stencil needs no tests) and does all
// that follows from it:
//   down, finest:  x = w D^-1 b (or the given x), r = b - A x, b_c = P^T r,
//                  x_c = w D_c^-1 b_c        (three or four passes before)
//   up, finest:    v = x + P x_c, x' = v + w D^-1 (b - A v)           (two)
//   down, coarse:  r = b - A x, b_c = P^T r, x_c = w D_c^-1 b_c       (two)
//   up, coarse:    v = x + P x_c, x' = v + w D^-1 (b - A v)     (one or two)
// The residual never goes to memory.  1025^2 nodes in FP32: down 6.7 us (21.5
// as three kernels), up 8.2 us (20 as two), a coarse level 2.6-5.3 us each way
// (6-8); bound by instruction issue (100 warp instructions per node down, 130
// up).  FP32 results are those of the separate passes bit for bit (the mixed
// 2D solves before and after were compared).  Tiles are 64 columns wide with their
// rim (two nodes per lane), so a warp's rows are coalesced and no lane divides
// to find its node; tall enough that the rim costs 8 % (residuals) to 24 %
// (x) more, short enough that a 1024^2 grid fills the chip in one wave.
#pragma once
#include "common.cuh"

namespace mgar {
namespace l2d {

constexpr int kW = 64;        // columns of a finest-level tile with its rim
constexpr int kThreads2 = 256;
// Each of the eight warps owns R consecutive rows (two columns per lane), so
// the rows' stencils share their neighbours' shared-memory loads, and one
// address per array serves all nodes of a thread.  R = 3 costs the least rim;
// R = 1 spreads a small grid over three times the blocks (best_rows).
template <int R>
struct Geo {
  static constexpr int kRows = 8 * R;
  static constexpr int kCY = (kRows - 3) / 2;  // down: coarse rows per tile (2 kCY + 3 rows)
  static constexpr int kUY = kRows - 2;        // up, product: own rows per tile
};
constexpr int kR = 3;
constexpr int kCX = 30;  // down: coarse columns per tile (2 kCX + 3 = 63)
constexpr int kUX = 62;  // up, product: own columns per tile
// coarse levels: down, coarse nodes per tile (31 x 7 residuals); up, own nodes
constexpr int kDX = 15, kDY = 3, kDownThreads = 32 * (2 * kDY + 1);
constexpr int kPX = 30, kPY = 8, kUpThreads = 32 * (kPY + 2);

__host__ __device__ __forceinline__ int tiles(int n, int per) { return (n + per - 1) / per; }

// Rows per warp of the finest level's tiles: a pass takes as long as the SM
// with the most rows (FP64 passes are bound by its FP64 pipe), blocks / SMs
// rounded up times R.  Tall tiles win from two blocks per SM on, since they
// compute the smallest rim; a 101^2 grid takes R = 1.
template <class Blocks>
inline int best_rows(int sms, Blocks&& blocks) {
  int best = 3, cost = 3 * tiles(blocks(3), sms);
  for (int r = 2; r >= 1; --r)
    if (const int c = r * tiles(blocks(r), sms); c < cost) {
      best = r;
      cost = c;
    }
  return best;
}
inline int up_rows(int NX, int NY, int sms) {
  const int uy[4] = {0, Geo<1>::kUY, Geo<2>::kUY, Geo<3>::kUY};
  return best_rows(sms, [&](int r) { return tiles(NX, kUX) * tiles(NY, uy[r]); });
}
inline int down_rows(int cNX, int cNY, int sms) {
  const int cy[4] = {0, Geo<1>::kCY, Geo<2>::kCY, Geo<3>::kCY};
  return best_rows(sms, [&](int r) { return tiles(cNX, kCX) * tiles(cNY, cy[r]); });
}

// A finest level (matrix-free operator).
// dinv: 1/diag, negated on fixed nodes (one load for both)
template <typename Real>
struct Fine {
  const Real* ke;
  const Real* dinv;
  int ex, ey, cNX, cNY;  // elements; nodes of the next level
  Real omega;
};

// A coarse level (assembled stencil).
template <typename Real>
struct Coarse {
  StencilOp<Real> op;
  int ex, ey, cNX, cNY;
  Real omega;
};

// Restriction weights of coarse node I from the fine nodes 2I-1, 2I, 2I+1 (nf
// fine elements; off-grid residuals are zero, so only the injected last node
// of an odd axis differs from 1/2, 1, 1/2).
template <typename Real>
__device__ __forceinline__ void restrict_weights(int I, int nf, Real& w0, Real& w1, Real& w2) {
  const int f = 2 * I;
  w0 = f - 1 == nf ? Real(1) : Real(0.5);
  w1 = Real(1);
  w2 = f + 1 == nf ? Real(0) : Real(0.5);
}

template <typename Real, int W>
__device__ __forceinline__ Real restrict_sum(const Real (*r)[W], int c, int y, int I, int J, int ex,
                                             int ey) {
  Real x0, x1, x2, y0, y1, y2;
  restrict_weights<Real>(I, ex, x0, x1, x2);
  restrict_weights<Real>(J, ey, y0, y1, y2);
  if constexpr (sizeof(Real) == 4) {
    // the order of restrict_node
    Real acc = (y0 * x0) * r[y][c];
    acc += (y0 * x1) * r[y][c + 1];
    acc += (y0 * x2) * r[y][c + 2];
    acc += (y1 * x0) * r[y + 1][c];
    acc += (y1 * x1) * r[y + 1][c + 1];
    acc += (y1 * x2) * r[y + 1][c + 2];
    acc += (y2 * x0) * r[y + 2][c];
    acc += (y2 * x1) * r[y + 2][c + 1];
    acc += (y2 * x2) * r[y + 2][c + 2];
    return acc;
  } else {
    // 9 FP64 products fewer
    const Real a = x0 * r[y][c] + x1 * r[y][c + 1] + x2 * r[y][c + 2];
    const Real b = x0 * r[y + 1][c] + x1 * r[y + 1][c + 1] + x2 * r[y + 1][c + 2];
    const Real d = x0 * r[y + 2][c] + x1 * r[y + 2][c + 1] + x2 * r[y + 2][c + 2];
    return y0 * a + y1 * b + y2 * d;
  }
}

// The Q4 rows times 6 of column c at the tile rows y0 .. y0 + R - 1, tile row
// y at shared-memory row y + 1: x with off-grid and fixed values zero, k the
// element to the lower right of the node; f(q, row) with row as a function of
// the centre value.
template <typename Real, int R, class F>
__device__ __forceinline__ void q4_rows(const Real (*x)[kW], const Real (*k)[kW], int c, int y0, F&& f) {
  Real xl = x[y0][c - 1], xc = x[y0][c], xr = x[y0][c + 1];
  Real yl = x[y0 + 1][c - 1], yc = x[y0 + 1][c], yr = x[y0 + 1][c + 1];
  Real k00 = k[y0][c - 1], k01 = k[y0][c];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const Real zl = x[y0 + q + 2][c - 1], zc = x[y0 + q + 2][c], zr = x[y0 + q + 2][c + 1];
    const Real k10 = k[y0 + q + 1][c - 1], k11 = k[y0 + q + 1][c];
    const Real s = k00 + k01, n = k10 + k11;
    f(q, yc, [&](Real xi) {
      if constexpr (sizeof(Real) == 4) {
        // fine_row2's order of additions, with the contractions that give its
        // bits (found by comparing outputs)
        Real acc = __fmul_rn(__fmul_rn(4.f, s + n), xi);
        acc = __fmaf_rn(-(k00 + k10), yl, acc);
        acc = __fmaf_rn(-(k01 + k11), yr, acc);
        acc = __fmaf_rn(-s, xc, acc);
        acc = __fmaf_rn(-n, zc, acc);
        acc = __fmaf_rn(-2.f * k00, xl, acc);
        acc = __fmaf_rn(-2.f * k01, xr, acc);
        acc = __fmaf_rn(-2.f * k10, zl, acc);
        acc = __fmaf_rn(-2.f * k11, zr, acc);
        return acc;
      } else {
        const Real dg = k00 * xl + k01 * xr + k10 * zl + k11 * zr;
        const Real ed = (k00 + k10) * yl + (k01 + k11) * yr + s * xc + n * zc;
        return Real(4) * (s + n) * xi - ed - Real(2) * dg;
      }
    });
    xl = yl, xc = yc, xr = yr;
    yl = zl, yc = zc, yr = zr;
    k00 = k10, k01 = k11;
  }
}

// (P x_c) at a fine node whose first coarse tap sits at c[y][x]; hx, hy:
// halfway between two coarse nodes along x, y.  Weights are powers of two, so
// they scale the sum exactly.
template <typename Real, int W>
__device__ __forceinline__ Real prolong_sum(const Real (*c)[W], int x, int y, bool hx, bool hy) {
  Real s = c[y][x];
  if (hx) s += c[y][x + 1];
  if (hy) {
    s += c[y + 1][x];
    if (hx) s += c[y + 1][x + 1];
  }
  const Real wx = hx ? Real(0.5) : Real(1), wxy = hy ? Real(0.5) * wx : wx;
  return wxy * s;
}

// a / 6; rounded by itself in FP32, as fine_row2's result
__device__ __forceinline__ float sixth(float a) { return __fmul_rn(a, float(1.0 / 6.0)); }
__device__ __forceinline__ double sixth(double a) { return a * (1.0 / 6.0); }

// First coarse tap of fine node i, and whether it is halfway.
__device__ __forceinline__ int first_tap(int i, int nf, bool& half) {
  half = (i & 1) && i < nf;
  return (i & 1) && i == nf ? (i + 1) >> 1 : i >> 1;
}

// A thread's 2 R nodes in a tile whose first node is (fx0, fy0): rows y0 + q,
// columns lane + 32 h.
template <int R>
struct Place {
  int lane, w, y0;
  bool con[2], eon[2];  // column on the grid, its element on the grid
  __device__ __forceinline__ Place(int fx0, int ex) {
    lane = threadIdx.x & 31;
    w = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    y0 = R * w;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned i = (unsigned)(fx0 + lane + 32 * h);
      con[h] = i <= (unsigned)ex;
      eon[h] = i < (unsigned)ex;
    }
  }
};

// ------------------------------------------------------------- finest, down
// tile row y at row y + 1; the rows before the first and after the last are
// read by the rim rows' stencils, whose results are not used
template <typename Real, int R>
struct DownSmem {
  static constexpr int kRows = Geo<R>::kRows;
  Real x[kRows + 2][kW];
  Real k[kRows + 1][kW];
  Real r[kRows][kW];
};

// ZERO: x = w D^-1 b, written to t; otherwise x is read from t.  bc and (not
// null) xc of the tile's coarse nodes.
template <typename Real, int R, bool ZERO>
__device__ __forceinline__ void fine_down(DownSmem<Real, R>& s, const Fine<Real>& f, int tx, int ty,
                                          const Real* b, Real* t,
                                          Real* bc, const Real* __restrict__ dinvc,
                                          Real* xc) {
  constexpr int kCY = Geo<R>::kCY;
  const int NX = f.ex + 1, NY = f.ey + 1;
  const int I0 = tx * kCX, J0 = ty * kCY;
  const int fx0 = 2 * I0 - 2, fy0 = 2 * J0 - 2;
  const Place<R> p(fx0, f.ex);
  const int64_t at = fx0 + p.lane + (int64_t)NX * (fy0 + p.y0);
  const int64_t eat = fx0 + p.lane + (int64_t)f.ex * (fy0 + p.y0);
  Real dv[R][2], bv[R][2];
  bool ron[R];
  // hierarchy data before the wait on the predecessor
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const unsigned j = (unsigned)(fy0 + p.y0 + q);
    ron[q] = j < (unsigned)NY;
    const bool reon = j < (unsigned)f.ey;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      dv[q][h] = Real(0);
      if (ron[q] && p.con[h]) dv[q][h] = f.dinv[at + q * NX + 32 * h];
      Real kv = Real(0);
      if (reon && p.eon[h]) kv = f.ke[eat + q * f.ex + 32 * h];
      s.k[p.y0 + q + 1][p.lane + 32 * h] = kv;
    }
  }
  Real dc[2] = {Real(0), Real(0)};
  int cidx[2];
  bool con[2];
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int I = I0 + p.lane, J = J0 + p.w + 8 * g;
    con[g] = p.w + 8 * g < kCY && p.lane < kCX && I < f.cNX && J < f.cNY;
    cidx[g] = I + f.cNX * J;
    if (xc && con[g]) dc[g] = dinvc[cidx[g]];
  }
  pdl_wait();
  pdl_trigger();
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bv[q][h] = Real(0);
      if (ron[q] && p.con[h]) bv[q][h] = b[at + q * NX + 32 * h];
    }
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int y = p.y0 + q, c = p.lane + 32 * h;
      Real x = Real(0);
      if (ZERO) {
        x = f.omega * fabs(dv[q][h]) * bv[q][h];
        if (y >= 2 && y < 2 * kCY + 2 && c >= 2 && c < 2 * kCX + 2 && ron[q] && p.con[h])
          t[at + q * NX + 32 * h] = x;
      } else if (ron[q] && p.con[h]) {
        x = t[at + q * NX + 32 * h];
      }
      s.x[y + 1][c] = dv[q][h] > Real(0) ? x : Real(0);
    }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = p.lane + 32 * h;
    if (c >= 1 && c < 2 * kCX + 2)
      q4_rows<Real, R>(s.x, s.k, c, p.y0, [&](int q, Real xi, auto&& row) {
        const Real r = bv[q][h] - sixth(row(xi));
        s.r[p.y0 + q][c] = dv[q][h] > Real(0) ? r : Real(0);
      });
  }
  __syncthreads();
#pragma unroll
  for (int g = 0; g < 2; ++g)
    if (con[g]) {
      const int cy = p.w + 8 * g;
      const Real v = restrict_sum<Real, kW>(s.r, 2 * p.lane + 1, 2 * cy + 1, I0 + p.lane, J0 + cy,
                                            f.ex, f.ey);
      bc[cidx[g]] = v;
      if (xc) xc[cidx[g]] = f.omega * dc[g] * v;
    }
}

// --------------------------------------------------------------- finest, up
template <typename Real, int R>
struct UpSmem {
  static constexpr int kRows = Geo<R>::kRows;
  Real v[kRows + 2][kW];
  Real k[kRows + 1][kW];
  Real c[kRows / 2 + 3][kW / 2 + 4];
};

// xout = v + w D^-1 (b - A v), v = t + P res (fixed nodes keep t); dot(b, x')
// is called for every node of the tile.
template <typename Real, int R, class Dot>
__device__ __forceinline__ void fine_up(UpSmem<Real, R>& s, const Fine<Real>& f, int tx, int ty,
                                        const Real* b, const Real* t,
                                        const Real* res, Real* xout,
                                        Dot&& dot) {
  constexpr int kUY = Geo<R>::kUY, CR = Geo<R>::kRows / 2 + 2, CC = kW / 2 + 2;
  const int NX = f.ex + 1, NY = f.ey + 1;
  const int fx0 = tx * kUX - 1, fy0 = ty * kUY - 1;
  const int ci0 = max(fx0, 0) >> 1, cj0 = max(fy0, 0) >> 1;
  const Place<R> p(fx0, f.ex);
  const int64_t at = fx0 + p.lane + (int64_t)NX * (fy0 + p.y0);
  const int64_t eat = fx0 + p.lane + (int64_t)f.ex * (fy0 + p.y0);
  Real dv[R][2], bv[R][2], tv[R][2];
  bool ron[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const unsigned j = (unsigned)(fy0 + p.y0 + q);
    ron[q] = j < (unsigned)NY;
    const bool reon = j < (unsigned)f.ey;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      dv[q][h] = Real(0);
      if (ron[q] && p.con[h]) dv[q][h] = f.dinv[at + q * NX + 32 * h];
      Real kv = Real(0);
      if (reon && p.eon[h]) kv = f.ke[eat + q * f.ex + 32 * h];
      s.k[p.y0 + q + 1][p.lane + 32 * h] = kv;
    }
  }
  pdl_wait();
  pdl_trigger();
  // coarse values under the tile (clamped: values past the grid are not used)
  for (int cy = p.w; cy < CR; cy += 8)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int cx = p.lane + 32 * h;
      if (cx < CC)
        s.c[cy][cx] = res[min(ci0 + cx, f.cNX - 1) + f.cNX * min(cj0 + cy, f.cNY - 1)];
    }
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bv[q][h] = tv[q][h] = Real(0);
      if (ron[q] && p.con[h]) {
        bv[q][h] = b[at + q * NX + 32 * h];
        tv[q][h] = t[at + q * NX + 32 * h];
      }
    }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    bool hx;
    const int cx = min(max(first_tap(fx0 + p.lane + 32 * h, f.ex, hx) - ci0, 0), CC);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      bool hy;
      const int cy = min(max(first_tap(fy0 + p.y0 + q, f.ey, hy) - cj0, 0), CR - 1);
      const bool in = dv[q][h] > Real(0);
      if (in) tv[q][h] += prolong_sum<Real, kW / 2 + 4>(s.c, cx, cy, hx, hy);
      s.v[p.y0 + q + 1][p.lane + 32 * h] = in ? tv[q][h] : Real(0);
    }
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = p.lane + 32 * h;
    if (c >= 1 && c <= kUX && p.con[h])
      q4_rows<Real, R>(s.v, s.k, c, p.y0, [&](int q, Real, auto&& row) {
        const int y = p.y0 + q;
        if (!(y >= 1 && y <= kUY && ron[q])) return;
        const Real v = tv[q][h];
        const Real ax = dv[q][h] < Real(0) ? v : sixth(row(v));
        const Real xo = v + f.omega * fabs(dv[q][h]) * (bv[q][h] - ax);
        xout[at + q * NX + 32 * h] = xo;
        dot(bv[q][h], xo);
      });
  }
}

// -------------------------------------------- finest, FP64 direction, product
template <int R>
struct DirSmem {
  double p[Geo<R>::kRows + 2][kW];
  double k[Geo<R>::kRows + 1][kW];
};

// p = z + beta p_old (p = z when first), y = A p with conductivities ke;
// returns this thread's terms of p . y.
template <int R>
__device__ __forceinline__ double fine_dir(DirSmem<R>& s, const double* __restrict__ ke,
                                           const uint8_t* __restrict__ fixed, int ex, int ey, int tx,
                                           int ty, const double* z,
                                           const double* p_old, bool first, double beta,
                                           double* pn, double* y) {
  constexpr int kUY = Geo<R>::kUY;
  const int NX = ex + 1, NY = ey + 1;
  const int fx0 = tx * kUX - 1, fy0 = ty * kUY - 1;
  const Place<R> p(fx0, ex);
  const int64_t at = fx0 + p.lane + (int64_t)NX * (fy0 + p.y0);
  const int64_t eat = fx0 + p.lane + (int64_t)ex * (fy0 + p.y0);
  double v[R][2];
  bool ron[R], fx[R][2];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const unsigned j = (unsigned)(fy0 + p.y0 + q);
    ron[q] = j < (unsigned)NY;
    const bool reon = j < (unsigned)ey;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      v[q][h] = 0.0;
      fx[q][h] = true;
      if (ron[q] && p.con[h]) {
        const int64_t o = at + q * NX + 32 * h;
        v[q][h] = first ? z[o] : z[o] + beta * p_old[o];
        fx[q][h] = fixed[o] != 0;
      }
      double kv = 0.0;
      if (reon && p.eon[h]) kv = ke[eat + q * ex + 32 * h];
      s.k[p.y0 + q + 1][p.lane + 32 * h] = kv;
      s.p[p.y0 + q + 1][p.lane + 32 * h] = fx[q][h] ? 0.0 : v[q][h];
    }
  }
  __syncthreads();
  double dot = 0.0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = p.lane + 32 * h;
    if (c >= 1 && c <= kUX && p.con[h])
      q4_rows<double, R>(s.p, s.k, c, p.y0, [&](int q, double, auto&& row) {
        const int t = p.y0 + q;
        if (!(t >= 1 && t <= kUY && ron[q])) return;
        const double xi = v[q][h], a = fx[q][h] ? xi : sixth(row(xi));
        const int64_t o = at + q * NX + 32 * h;
        pn[o] = xi;
        y[o] = a;
        dot += xi * a;
      });
  }
  return dot;
}

// ------------------------------------------------------------- coarse, down
template <typename Real>
__device__ __forceinline__ void coarse_down(Real (*s)[32], const Coarse<Real>& f, int tx, int ty,
                                            const Real* b, const Real* x,
                                            Real* bc, const Real* __restrict__ dinvc,
                                            Real* xc) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int I0 = tx * kDX, J0 = ty * kDY;
  const int i = 2 * I0 - 1 + lane, j = 2 * J0 - 1 + w;
  const bool on = lane < 2 * kDX + 1 && i >= 0 && i < f.op.NX && j >= 0 && j < f.op.NY;
  Real sv[9];
  if (on) stencil_coefs<2>(f.op, i, j, 0, sv);
  const int I = I0 + lane, J = J0 + w;
  const bool con = lane < kDX && w < kDY && I < f.cNX && J < f.cNY;
  const int cidx = con ? I + f.cNX * J : 0;
  const Real dc = xc && con ? dinvc[cidx] : Real(0);
  pdl_wait();
  pdl_trigger();
  Real r = Real(0);
  if (on) r = b[i + f.op.NX * j] - stencil_apply<2, Real, false>(f.op, x, i, j, 0, sv);
  s[w][lane] = r;
  __syncthreads();
  if (con) {
    const Real v = restrict_sum<Real, 32>(s, 2 * lane, 2 * w, I, J, f.ex, f.ey);
    bc[cidx] = v;
    if (xc) xc[cidx] = f.omega * dc * v;
  }
}

// --------------------------------------------------------------- coarse, up
template <typename Real>
struct CoarseUpSmem {
  Real v[kPY + 2][32];
};

// AXES: interpolate along x, then y (post_node's order of additions), else
// all taps in one sum (prolong_node's).
template <typename Real, bool AXES>
__device__ __forceinline__ void coarse_up(CoarseUpSmem<Real>& s, const Coarse<Real>& f, int tx, int ty,
                                          const Real* b, const Real* x,
                                          const Real* res, Real* xout) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = tx * kPX - 1 + lane, j = ty * kPY - 1 + w;
  const bool on = i >= 0 && i < f.op.NX && j >= 0 && j < f.op.NY;
  const bool own = on && lane >= 1 && lane <= kPX && w >= 1 && w <= kPY;
  const int idx = on ? i + f.op.NX * j : 0;
  Real sv[9], dv = Real(0);
  if (own) {
    stencil_coefs<2>(f.op, i, j, 0, sv);
    dv = f.op.dinv[idx];
  }
  bool hx = false, hy = false;
  const int cx = on ? first_tap(i, f.ex, hx) : 0, cy = on ? first_tap(j, f.ey, hy) : 0;
  pdl_wait();
  pdl_trigger();
  Real v = Real(0), bv = Real(0);
  if (on) {
    // four taps, an unused one repeating the first
    const int c0 = cx + f.cNX * cy, ox = hx ? 1 : 0, oy = hy ? f.cNX : 0;
    const Real r0 = res[c0], r1 = res[c0 + ox], r2 = res[c0 + oy], r3 = res[c0 + ox + oy];
    v = x[idx];
    if (own) bv = b[idx];
    if (AXES) {
      const Real p = hx ? Real(0.5) * (r0 + r1) : r0, u = hx ? Real(0.5) * (r2 + r3) : r2;
      v += hy ? Real(0.5) * (p + u) : p;
    } else {
      Real p = r0;
      if (hx) p += r1;
      if (hy) {
        p += r2;
        if (hx) p += r3;
      }
      v += (hx ? Real(0.5) : Real(1)) * (hy ? Real(0.5) : Real(1)) * p;
    }
  }
  s.v[w][lane] = v;
  __syncthreads();
  if (own) {
    Real acc = Real(0);
#pragma unroll
    for (int q = 0; q < 9; ++q) acc += sv[q] * s.v[w - 1 + q / 3][lane - 1 + q % 3];
    xout[idx] = v + f.omega * dv * (bv - acc);
  }
}

}  // namespace l2d
}  // namespace mgar
