// Tiled FP64 kernels of the finest 3D (H8) level: the FP64 path's V-cycle
// passes, products and CG direction update.
//
// GB300 runs FP64 at 1/58 of the FP32 rate (about 20 clocks per warp
// instruction and SM), so these kernels are bound by their count of FP64
// operations: a row gathered from its 8 conductivities and 20 neighbours took
// 45 of them (203-249 us a pass on 129^3 nodes).  Here the rows are split by
// element layer as in fine3d.cu,
//   row = up(layer k) + down(layer k-1),
//   up   = 4 S x_lo - C - E(hi),  down = 4 S x_hi - C - E(lo),
// and everything two threads need is formed once and passed through shared
// memory: the column sums x_lo + x_hi (C = sum of e_q times those at the
// in-plane diagonal neighbours) and the element pair sums along x and y (the
// weights of E, and S).  A node costs 22 operations:
//   2 pair sums, 1 column sum, 2 for 4 S, 4 for C, 6 for the row (dk - C -
//   E(hi) + 4 S x), 5 for the next row's down part, and the pass's own 2-4.
// A tile's rim adds one operation for about 150 threads per step.  Tiles and
// z runs are those of fine3d.cu (the fewest idle lanes: an idle lane's slot in
// the FP64 pipe is lost).
#include "common.cuh"
#include "tile3d.cuh"

namespace mgar {
namespace f64 {
using namespace tile;

enum Mode { PRE_SMOOTH = 0, RESIDUAL = 1, SWEEP = 2, DIRECTION = 3, APPLY = 4 };

struct Args {
  int ex, ey, ez, NX, NY, NZ, gz;
  const uint8_t* fixed;
  const double* ke;
  const double* ksub;  // APPLY: k_e - ksub_e, fixed rows zero (null: k_e, fixed rows identity)
  const double* b;     // PRE, RESID, SWEEP: right-hand side; DIR: z
  const double* dinv;  // PRE, SWEEP
  int full;            // RESID: r on fixed rows too (else 0), r . r into dout
  const double* x;     // RESID, SWEEP, APPLY: operand; DIR: p_old
  double* out0;        // PRE: x; RESID: r; SWEEP: x'; DIR: p; APPLY: y
  double* out1;        // PRE: r; DIR: A p
  double omega, scale;
  // DIR: *beta; p = z when first; odd *parity (may be null): p_old is x_alt
  // and p goes to out_alt (the two buffers swap each iteration)
  const double* beta;
  const double* parity;
  const double* x_alt;
  double* out_alt;
  int first;
  double* partials;
  unsigned int* counter;
  SumOut dout;         // SWEEP: b . x'; DIR: p . A p; APPLY: x . y
};

template <int MODE, class T>
__global__ void __launch_bounds__(T::NTB, T::NT <= 256 ? 3 : 2) k_fine64(Args a) {
  constexpr int TX = T::TX, TY = T::TY, NT = T::NT, XRING = T::XRING, KRING = T::KRING,
                KRING0 = T::KRING0;
  __shared__ double X[2][TY + 2][TX + 2];
  __shared__ double K[2][TY + 1][TX + 1];
  __shared__ double XS[TY + 2][TX + 2];  // x_lo + x_hi
  __shared__ double H[TY + 1][TX];       // K[r][c] + K[r][c + 1]
  __shared__ double V[TY][TX + 1];       // K[r][c] + K[r + 1][c]
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const bool real = tid < NT;
  // (a plane's tiles numbered along x alone: their rows may pass the second
  // dimension's 65535)
  const int ntx = (a.NX + TX - 1) / TX, by = blockIdx.x / ntx;
  const int i0 = (blockIdx.x - by * ntx) * TX, j0 = by * TY;
  const int kb = (int)(((int64_t)blockIdx.z * a.NZ) / a.gz);
  const int kend = (int)(((int64_t)(blockIdx.z + 1) * a.NZ) / a.gz);
  const int i = i0 + tx, j = j0 + ty, NXY = a.NX * a.NY;
  const bool mine = real && i < a.NX && j < a.NY;
  const bool xr = tid < XRING, kr = tid >= KRING0 && tid < KRING0 + KRING;
  int rxh = 0, ryh = 0, kxh = 0, kyh = 0;
  if (xr) T::xring(tid, rxh, ryh);
  if (kr) T::kring(tid - KRING0, kxh, kyh);
  const int ri = i0 - 1 + rxh, rj = j0 - 1 + ryh, ki = i0 - 1 + kxh, kj = j0 - 1 + kyh;
  const bool ron = xr && ri >= 0 && ri < a.NX && rj >= 0 && rj < a.NY;
  const bool eon = real && i < a.ex && j < a.ey;
  const bool kron = kr && ki >= 0 && ki < a.ex && kj >= 0 && kj < a.ey;
  const int ocol = i + a.NX * j, rcol = ri + a.NX * rj;
  const int ecol = i + a.ex * j, kcol = ki + a.ex * kj;
  const double om = MODE != DIRECTION ? a.omega : a.first ? 0.0 : *a.beta;
  if (MODE == DIRECTION && a.parity && is_set(a.parity)) {
    a.x = a.x_alt;
    a.out0 = a.out_alt;
  }

  // a node's operand: the value the stencil's centre takes, and (masked) what
  // its neighbours see of it
  struct Node {
    double v, b, d;
    bool on, fx;
  };
  auto fetch = [&](int col, bool in, int k, bool own) {
    Node n{0.0, 0.0, 0.0, in && k >= 0 && k < a.NZ, true};
    if (n.on) {
      const int64_t idx = col + (int64_t)NXY * k;
      n.fx = a.fixed[idx] != 0;
      if (MODE == PRE_SMOOTH) {
        n.b = a.b[idx];
        n.d = a.dinv[idx];
      } else if (MODE == DIRECTION) {
        n.b = a.b[idx];
        n.d = a.first ? 0.0 : a.x[idx];
      } else {
        n.v = a.x[idx];
        if (own && MODE != APPLY) {
          n.b = a.b[idx];
          if (MODE == SWEEP) n.d = a.dinv[idx];
        }
      }
    }
    return n;
  };
  auto value = [&](Node& n) {
    if (MODE == PRE_SMOOTH) n.v = om * n.d * n.b;
    if (MODE == DIRECTION) n.v = a.first ? n.b : n.b + om * n.d;
  };
  auto elem = [&](int col, bool in, int l) {
    double v = 0.0;
    if (in && l >= 0 && l < a.ez) {
      const int64_t e = col + (int64_t)a.ex * a.ey * l;
      v = a.ke[e];
      if (MODE == APPLY && a.ksub) v -= a.ksub[e];
    }
    return v;
  };
  auto put_plane = [&](int s, Node& own, Node& ring) {
    value(own);
    if (real) X[s][ty + 1][tx + 1] = own.on && !own.fx ? own.v : 0.0;
    if (xr) {
      value(ring);
      X[s][ryh][rxh] = ring.on && !ring.fx ? ring.v : 0.0;
    }
  };
  auto put_layer = [&](int s, double own, double ring) {
    if (real) K[s][ty + 1][tx + 1] = own;
    if (kr) K[s][kyh][kxh] = ring;
  };

  // the rim's sums, one per thread: column sums of the plane's ring, then the
  // first row of H and the first column of V
  constexpr int EXTRA = XRING + TX + TY;
  static_assert(EXTRA <= T::NTB, "one rim sum per thread");

  const bool sum = a.dout.out != nullptr;
  const double rscale = a.scale * (1.0 / 12.0);
  double acc[1] = {0.0};
  double dk = 0.0;              // down part of the current row
  double e_lo[4] = {0, 0, 0, 0};  // plane lo's in-plane edge neighbours
  Node lo = fetch(ocol, mine, kb - 1, true), lor = fetch(rcol, ron, kb - 1, false);
  Node hi = fetch(ocol, mine, kb, true), hir = fetch(rcol, ron, kb, false);
  double kown = elem(ecol, eon, kb - 1), kring = elem(kcol, kron, kb - 1);
  put_plane(0, lo, lor);
  // step s handles the layer between planes k - 1 + s (lo) and k + s (hi):
  // planes alternate slots
  int s = 0;
  for (int k = kb - 1; k < kend; ++k, s ^= 1) {
    // plane k in slot s (and lo), plane k + 1 in hi, layer k in kown
    put_plane(s ^ 1, hi, hir);
    put_layer(s, kown, kring);
    Node nxt{}, nxtr{};
    double kn = 0.0, krn = 0.0;
    if (k + 1 < kend) {
      nxt = fetch(ocol, mine, k + 2, true);
      nxtr = fetch(rcol, ron, k + 2, false);
      kn = elem(ecol, eon, k + 1);
      krn = elem(kcol, kron, k + 1);
    }
    __syncthreads();
    const double xlo = real ? X[s][ty + 1][tx + 1] : 0.0, xhi = real ? X[s ^ 1][ty + 1][tx + 1] : 0.0;
    double en = 0.0, ee = 0.0, e11 = 0.0, e01 = 0.0, e10 = 0.0;
    if (real) {
      e11 = K[s][ty + 1][tx + 1];
      e01 = K[s][ty][tx + 1];
      e10 = K[s][ty + 1][tx];
      en = e10 + e11;
      ee = e01 + e11;
      XS[ty + 1][tx + 1] = xlo + xhi;
      H[ty + 1][tx] = en;
      V[ty][tx + 1] = ee;
    }
    if (tid < EXTRA) {
      const double *p, *q;
      double* o;
      if (tid < XRING) {
        p = &X[0][ryh][rxh];
        q = &X[1][ryh][rxh];
        o = &XS[ryh][rxh];
      } else if (tid < XRING + TX) {
        const int c = tid - XRING;
        p = &K[s][0][c];
        q = &K[s][0][c + 1];
        o = &H[0][c];
      } else {
        const int r = tid - XRING - TX;
        p = &K[s][r][0];
        q = &K[s][r + 1][0];
        o = &V[r][0];
      }
      *o = *p + *q;
    }
    __syncthreads();
    if (mine) {
      const double e00 = K[s][ty][tx];
      const double es = H[ty][tx], ew = V[ty][tx];
      const double s4 = 4.0 * (es + en);
      const double* xs0 = XS[ty] + tx;  // row above-left
      const double* xs2 = XS[ty + 2] + tx;
      double cc = e00 * xs0[0];
      cc = fma(e01, xs0[2], cc);
      cc = fma(e10, xs2[0], cc);
      cc = fma(e11, xs2[2], cc);
      const double (*Xh)[TX + 2] = X[s ^ 1];
      const double h0 = Xh[ty + 1][tx], h1 = Xh[ty + 1][tx + 2], h2 = Xh[ty][tx + 1],
                   h3 = Xh[ty + 2][tx + 1];
      if (k >= kb) {
        double row = dk - cc;
        row = fma(-ew, h0, row);
        row = fma(-ee, h1, row);
        row = fma(-es, h2, row);
        row = fma(-en, h3, row);
        row = fma(s4, xlo, row);
        const int64_t idx = ocol + (int64_t)NXY * k;
        const double xi = lo.v;  // a fixed row is the identity
        if (MODE == PRE_SMOOTH) {
          a.out0[idx] = xi;
          a.out1[idx] = lo.fx ? 0.0 : fma(row, -1.0 / 12.0, lo.b);
        } else if (MODE == RESIDUAL) {
          const double r = lo.fx ? (a.full ? lo.b - xi : 0.0) : fma(row, -1.0 / 12.0, lo.b);
          a.out0[idx] = r;
          if (sum) acc[0] = fma(r, r, acc[0]);
        } else if (MODE == SWEEP) {
          const double r = lo.fx ? lo.b - xi : fma(row, -1.0 / 12.0, lo.b);
          const double xo = fma(om * lo.d, r, xi);
          a.out0[idx] = xo;
          if (sum) acc[0] = fma(lo.b, xo, acc[0]);
        } else if (MODE == DIRECTION) {
          const double y = lo.fx ? xi : row * (1.0 / 12.0);
          a.out0[idx] = xi;
          a.out1[idx] = y;
          acc[0] = fma(xi, y, acc[0]);
        } else {
          const double y = lo.fx ? (a.ksub ? 0.0 : a.scale * xi) : row * rscale;
          a.out0[idx] = y;
          if (sum) acc[0] = fma(xi, y, acc[0]);
        }
      }
      double dn = cc;
      dn = fma(ew, k < kb ? X[s][ty + 1][tx] : e_lo[0], dn);
      dn = fma(ee, k < kb ? X[s][ty + 1][tx + 2] : e_lo[1], dn);
      dn = fma(es, k < kb ? X[s][ty][tx + 1] : e_lo[2], dn);
      dn = fma(en, k < kb ? X[s][ty + 2][tx + 1] : e_lo[3], dn);
      dk = fma(s4, xhi, -dn);
      e_lo[0] = h0;
      e_lo[1] = h1;
      e_lo[2] = h2;
      e_lo[3] = h3;
    }
    lo = hi;
    hi = nxt;
    hir = nxtr;
    kown = kn;
    kring = krn;
    // the next step writes plane k + 2 into slot s, which only the first step
    // reads past its sums, layer k + 1 into the other K slot, and its sums after
    // its own barrier
    if (k < kb) __syncthreads();
  }
  if (sum) {
    const double other = sum_other(a.dout, tid == 0);
    double t[1];
    const int bid = blockIdx.x + gridDim.x * blockIdx.z;
    const int nb = gridDim.x * gridDim.z;
    if (block_sum_last_ids<1>(acc, a.partials, a.counter, t, tid, T::NTB, bid, nb) && tid == 0)
      sum_out(a.dout, t[0], other);
  }
}

bool wide_tile(const Dims& d) {
  return tile_use(d.NX, d.NY, T43x5::TX, T43x5::TY) > tile_use(d.NX, d.NY, T32x8::TX, T32x8::TY);
}

// z runs so that the grid fills the GPU once
template <int MODE, class T>
int runs_for(const Ctx& c) {
  const Dims& d = c.L[0];
  int per_sm = 0;
  MGAR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fine64<MODE, T>, T::NTB, 0));
  const int64_t cols = (int64_t)((d.NX + T::TX - 1) / T::TX) * ((d.NY + T::TY - 1) / T::TY);
  const int64_t gz = std::max<int64_t>(1, (int64_t)std::max(per_sm, 1) * c.sms / cols);
  return (int)std::min<int64_t>(gz, d.NZ);
}
template <class T>
void prepare(Ctx& c) {
  c.f64_gz[APPLY] = runs_for<APPLY, T>(c);
  if (c.p.precision != MGAR_FP64) return;  // a mixed handle takes no other FP64 pass
  c.f64_gz[PRE_SMOOTH] = runs_for<PRE_SMOOTH, T>(c);
  c.f64_gz[RESIDUAL] = runs_for<RESIDUAL, T>(c);
  c.f64_gz[SWEEP] = runs_for<SWEEP, T>(c);
  c.f64_gz[DIRECTION] = runs_for<DIRECTION, T>(c);
}

template <int MODE, class T>
void launch_t(Ctx& c, Args& a) {
  const Dims& d = c.L[0];
  a.gz = std::max(1, c.f64_gz[MODE]);
  const dim3 grid(((d.NX + T::TX - 1) / T::TX) * ((d.NY + T::TY - 1) / T::TY), 1, a.gz);
  launch_pdl(c.stream, c.use_pdl, k_fine64<MODE, T>, grid, dim3(T::NTB), a);
}
template <int MODE>
void launch(Ctx& c, Args& a) {
  if (wide_tile(c.L[0])) launch_t<MODE, T43x5>(c, a);
  else launch_t<MODE, T32x8>(c, a);
}

Args base(Ctx& c) {
  const Dims& d = c.L[0];
  Args a{};
  a.ex = d.ex;
  a.ey = d.ey;
  a.ez = d.ez;
  a.NX = d.NX;
  a.NY = d.NY;
  a.NZ = d.NZ;
  a.fixed = c.fixed;
  a.omega = c.p.omega;
  a.partials = c.partials;
  a.counter = c.counter;
  return a;
}

}  // namespace f64

// launch shapes (occupancy queries; call outside stream capture)
void fine3d64_prepare(Ctx& c) {
  if (f64::wide_tile(c.L[0])) f64::prepare<tile::T43x5>(c);
  else f64::prepare<tile::T32x8>(c);
}

void fine3d(Ctx& c, int mode, const double* ke, const double* b, const double* dinv, const double* x,
            const double*, double* out0, double* out1, const float2*, SumOut dout) {
  using namespace f64;
  Args a = base(c);
  a.ke = ke;
  a.b = b;
  a.dinv = dinv;
  a.x = x;
  a.out0 = out0;
  a.out1 = out1;
  a.dout = dout;
  if (mode == 0) launch<PRE_SMOOTH>(c, a);
  else if (mode == 2) launch<RESIDUAL>(c, a);
  else launch<SWEEP>(c, a);
  MGAR_LAUNCH_CHECK_AT(level_site(mode == 0 ? 6 : mode == 2 ? 9 : 8, 0));
}

void fine3d_residual64(Ctx& c, const double* q, const double* x, double* r, SumOut rr) {
  using namespace f64;
  Args a = base(c);
  a.ke = c.ke;
  a.b = q;
  a.x = x;
  a.out0 = r;
  a.full = 1;
  a.dout = rr;
  launch<RESIDUAL>(c, a);
  MGAR_LAUNCH_CHECK();
}

void fine3d_dir64(Ctx& c, const double* z, const double* p_old, double* p, const double* beta,
                  bool first, const double* parity, double* y, SumOut dot) {
  using namespace f64;
  Args a = base(c);
  a.ke = c.ke;
  a.b = z;
  a.x = p_old;
  a.beta = beta;
  a.first = first ? 1 : 0;
  a.parity = parity;
  a.x_alt = p;
  a.out_alt = const_cast<double*>(p_old);
  a.out0 = p;
  a.out1 = y;
  a.dout = dot;
  launch<DIRECTION>(c, a);
  MGAR_LAUNCH_CHECK();
}

void fine3d_apply64(Ctx& c, const double* ke, const double* ksub, const double* x, double* y,
                    double scale, SumOut dot) {
  using namespace f64;
  Args a = base(c);
  a.ke = ke;
  a.ksub = ksub;
  a.x = x;
  a.out0 = y;
  a.scale = scale;
  a.dout = dot;
  launch<APPLY>(c, a);
  MGAR_LAUNCH_CHECK();
}

}  // namespace mgar
