// V-cycle x <- MG(A, b, x, P) of Table 1 on the reference hierarchy, plus the
// fine-level operator applications used by the solvers.
//
// Per level (Table 1): pre-smooth with damped Jacobi
// x <- x + omega D^-1 (b - A x), residual restricted by P^T, coarse
// correction (recursively one V-cycle with zero initial guess, the coarsest
// level by its explicit inverse), interpolation x <- x + P x^c, post-smooth.
// The finest operator is matrix-free from the element conductivities; the
// coarse ones are assembled 3^d-point stencils.  Every kernel is templated on
// the working precision (FP64, or FP32 for the mixed preconditioner).
#include "common.cuh"
#include "level2d.cuh"
#include "levelops.cuh"

#include <type_traits>

namespace mgar {

const char* level_site(int kind, int level) {
  static const char* names[10] = {"jacobi0", "sweep", "residual", "restrict", "prolong",
                                  "coarse", "pre3d", "post3d", "sweep3d", "resid3d"};
  static char table[10][kMaxLevels][24];
  static bool init = false;
  if (!init) {
    for (int k = 0; k < 10; ++k)
      for (int l = 0; l < kMaxLevels; ++l) snprintf(table[k][l], 24, "vc %s L%d", names[k], l);
    init = true;
  }
  return table[kind % 10][level % kMaxLevels];
}

// ------------------------------------------------------------ row functors
template <typename Real, int DIM>
struct FineRow {
  FineOp<Real> op;
  __device__ __forceinline__ Real operator()(const Real* __restrict__ x, int idx) const {
    int i, j, k;
    coords(idx, op.fNX, op.fNXY, i, j, k);
    Real d;
    if (DIM == 2) return fine_row2(op, x, i, j, d);
    return fine_row3(op, x, i, j, k, d);
  }
  __device__ __forceinline__ int size() const { return op.n; }
};

template <typename Real, int DIM>
struct StencilRow {
  StencilOp<Real> op;
  __device__ __forceinline__ Real operator()(const Real* __restrict__ x, int idx) const {
    int i, j, k;
    coords(idx, op.fNX, op.fNXY, i, j, k);
    if (DIM == 2) return stencil_row2(op, x, i, j);
    return stencil_row3(op, x, i, j, k);
  }
  __device__ __forceinline__ int size() const { return op.n; }
};

// ----------------------------------------------------------------- kernels
template <class Row, typename Real>
__global__ void k_jacobi(Row row, const Real* __restrict__ b, const Real* __restrict__ xin,
                         Real* __restrict__ xout, const Real* __restrict__ dinv, Real omega) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= row.size()) return;
  const Real ax = row(xin, idx);
  xout[idx] = xin[idx] + omega * dinv[idx] * (b[idx] - ax);
}

template <typename Real>
__global__ void k_jacobi_zero(const Real* __restrict__ b, Real* __restrict__ x,
                              const Real* __restrict__ dinv, Real omega, int n) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < n) x[idx] = omega * dinv[idx] * b[idx];
}

template <class Row, typename Real>
__global__ void k_residual(Row row, const Real* __restrict__ b, const Real* __restrict__ x,
                           Real* __restrict__ r) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= row.size()) return;
  r[idx] = b[idx] - row(x, idx);
}

// y = A x, optionally with the deterministic sum of x.y into out.
template <class Row, typename Real, bool DOT>
__global__ void k_apply(Row row, const Real* __restrict__ x, Real* __restrict__ y, Real scale,
                        double* partials, unsigned int* counter, SumOut out) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (idx < row.size()) {
    const Real ax = scale * row(x, idx);
    y[idx] = ax;
    if (DOT) v = (double)x[idx] * (double)ax;
  }
  if (DOT) block_sum_finish(v, partials, counter, out);
}

// The 2D levels' tiled passes (level2d.cuh).
template <typename Real, int R, bool ZERO>
__global__ void __launch_bounds__(l2d::kThreads2) k_down2d(l2d::Fine<Real> f, const Real* b,
                                                           Real* t, Real* bc,
                                                           const Real* __restrict__ dinvc,
                                                           Real* xc) {
  __shared__ l2d::DownSmem<Real, R> s;
  l2d::fine_down<Real, R, ZERO>(s, f, blockIdx.x, blockIdx.y, b, t, bc, dinvc, xc);
}

// DOT (FP64): also b . xout into dout.
template <typename Real, int R, bool DOT>
__global__ void __launch_bounds__(l2d::kThreads2) k_up2d(l2d::Fine<Real> f, const Real* b,
                                                         const Real* t,
                                                         const Real* res,
                                                         Real* xout, double* partials,
                                                         unsigned int* counter, SumOut dout) {
  __shared__ l2d::UpSmem<Real, R> s;
  double acc[1] = {0.0};
  l2d::fine_up<Real, R>(s, f, blockIdx.x, blockIdx.y, b, t, res, xout,
                        [&](Real bv, Real xo) { if (DOT) acc[0] += bv * xo; });
  if (DOT) {
    const double other = sum_other(dout, threadIdx.x == 0);
    double v[1];
    if (block_sum_last_ids<1>(acc, partials, counter, v, threadIdx.x, l2d::kThreads2,
                              blockIdx.x + gridDim.x * blockIdx.y, gridDim.x * gridDim.y) &&
        threadIdx.x == 0)
      sum_out(dout, v[0], other);
  }
}

// r . x (r in df64 pairs, or r = b without them) over the nodes in memory
// order.  The mixed 2D CG is sensitive to its last bits: another order of this
// sum changes which FP32 roundings the V-cycle meets, and with them the
// iteration count of one design in sixty.  So the sum keeps the order of the
// nodes and does not follow the tiles, where it cost 6 us on 1025^2 nodes at
// the end of the pass.
__global__ void __launch_bounds__(kThreads) k_dot_rz(const float2* r, const float* b,
                                                     const float* x, int n,
                                                     double* partials, unsigned int* counter,
                                                     SumOut out) {
  pdl_wait();
  pdl_trigger();
  const double other = sum_other(out, threadIdx.x == 0);
  float2 rv[4 * kSumVB];
  float xv[4 * kSumVB];
  double t;
  if (ordered_sum<4>(
          n, blockIdx.x, partials, counter, t,
          [&](int q, int idx) {
            rv[q] = r ? r[idx] : make_float2(b[idx], 0.f);
            xv[q] = x[idx];
          },
          [&](int q) { return df_mulf(df{rv[q].x, rv[q].y}, xv[q]); }) &&
      threadIdx.x == 0)
    sum_out(out, t, other);
}

// FP64: p = z + beta p_old (p = z when first), y = A p, p . y into out; odd
// *parity (may be null) swaps p_old and p.
template <int R>
__global__ void __launch_bounds__(l2d::kThreads2) k_dir2d(const double* __restrict__ ke,
                                                          const uint8_t* __restrict__ fixed, int ex,
                                                          int ey, const double* z,
                                                          const double* p_old, double* p,
                                                          const double* beta, int first,
                                                          const double* parity,
                                                          double* y, double* partials,
                                                          unsigned int* counter, SumOut out) {
  __shared__ l2d::DirSmem<R> s;
  pdl_wait();
  pdl_trigger();
  if (parity && is_set(parity)) {
    double* t = const_cast<double*>(p_old);
    p_old = p;
    p = t;
  }
  const double other = sum_other(out, threadIdx.x == 0);
  double v[1], t[1];
  v[0] = l2d::fine_dir<R>(s, ke, fixed, ex, ey, blockIdx.x, blockIdx.y, z, p_old, first != 0,
                          first ? 0.0 : *beta, p, y);
  if (block_sum_last_ids<1>(v, partials, counter, t, threadIdx.x, l2d::kThreads2,
                            blockIdx.x + gridDim.x * blockIdx.y, gridDim.x * gridDim.y) &&
      threadIdx.x == 0)
    sum_out(out, t[0], other);
}

template <typename Real>
__global__ void __launch_bounds__(l2d::kDownThreads) k_coarse_down2d(l2d::Coarse<Real> f,
                                                                     const Real* b,
                                                                     const Real* x,
                                                                     Real* bc,
                                                                     const Real* __restrict__ dinvc,
                                                                     Real* xc) {
  __shared__ Real s[2 * l2d::kDY + 1][32];
  l2d::coarse_down<Real>(s, f, blockIdx.x, blockIdx.y, b, x, bc, dinvc, xc);
}

template <typename Real, bool AXES>
__global__ void __launch_bounds__(l2d::kUpThreads) k_coarse_up2d(l2d::Coarse<Real> f,
                                                                 const Real* b,
                                                                 const Real* x,
                                                                 const Real* res,
                                                                 Real* xout) {
  __shared__ l2d::CoarseUpSmem<Real> s;
  l2d::coarse_up<Real, AXES>(s, f, blockIdx.x, blockIdx.y, b, x, res, xout);
}

template <typename Real, int DIM>
__global__ void k_restrict(const Real* r, Real* bc, Dims f, Dims cd,
                           const uint8_t* __restrict__ fixed, const Real* __restrict__ dinvc = nullptr,
                           Real omega = Real(0), Real* xc = nullptr) {
  pdl_wait();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < cd.n) restrict_node<Real, DIM, false>(r, bc, f, cd, fixed, idx, dinvc, omega, xc);
  pdl_trigger();
}

// dst = cur + P xc (fixed fine nodes keep cur); dst may equal cur.
template <typename Real, int DIM>
__global__ void k_prolong(const Real* xc, const Real* cur, Real* dst, Dims f, Dims cd,
                          const uint8_t* __restrict__ fixed) {
  pdl_wait();
  pdl_trigger();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < f.n) prolong_node<Real, DIM>(xc, cur, dst, f, cd, fixed, idx);
}

// 3D interpolation by z-columns: a thread owns the fine nodes (i, j, k0 ..
// k0 + kProlongChunk - 1), k0 even, and interpolates each of the coarse
// planes k0/2 .. k0/2 + kProlongChunk/2 in x and y once (4 loads), so a
// fine node costs one or two plane values instead of 8 coarse loads.  Every
// load of the chunk is issued before the first use (compile-time slots), so
// the column costs one memory round trip.
constexpr int kProlongChunk = 8;

template <typename Real>
__global__ void k_prolong3(const Real* xc, const Real* cur, Real* dst, Dims f, Dims cd,
                           const uint8_t* __restrict__ fixed) {
  constexpr int KC = kProlongChunk, NP = KC / 2 + 1;
  pdl_wait();
  pdl_trigger();
  const int NXY = f.NX * f.NY;
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= NXY) return;
  const int i = col % f.NX, j = col / f.NX;
  int ix[2], iy[2];
  float wx[2], wy[2];
  prolong_taps(i, f.ex, ix, wx);
  prolong_taps(j, f.ey, iy, wy);
  Real wxy[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) wxy[q] = (Real)(wx[q & 1] * wy[q >> 1]);
  const int cNXY = cd.NX * cd.NY;
  const int k0 = blockIdx.y * KC, Kb = k0 >> 1;
  // coarse planes Kb .. Kb + NP - 1, interpolated in x and y
  Real P[NP];
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    P[t] = Real(0);
    const int K = Kb + t;
    if (K < cd.NZ) {
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const int o = ix[a] + cd.NX * iy[b] + cNXY * K;
          if (CK(o, cd.n)) P[t] += wxy[a + 2 * b] * xc[o];
        }
    }
  }
  Real cv[KC];
  uint8_t fx[KC];
#pragma unroll
  for (int u = 0; u < KC; ++u) {
    const int k = k0 + u;
    cv[u] = Real(0);
    fx[u] = 0;
    if (k < f.NZ) {
      const int idx = col + NXY * k;
      cv[u] = cur[idx];
      if (fixed) fx[u] = fixed[idx];
    }
  }
#pragma unroll
  for (int u = 0; u < KC; ++u) {
    const int k = k0 + u;
    if (k >= f.NZ) break;
    // taps along z: even k -> plane k/2; odd k -> halfway, or the top node
    // of an odd element count -> plane (k+1)/2
    Real pz;
    if ((u & 1) == 0) pz = P[u >> 1];
    else if (k < f.ez) pz = Real(0.5) * (P[u >> 1] + P[(u >> 1) + 1]);
    else pz = P[(u >> 1) + 1];
    dst[col + NXY * k] = fx[u] ? cv[u] : cv[u] + pz;
  }
}

// The coarse-level kernels gather what the hierarchy build wrote (stencil
// coefficients, D^-1, the coarsest inverse) before they wait on their
// predecessor: a kernel may start while its predecessor runs, and every
// kernel here waits before it lets its own successor start, so everything
// older than the predecessor is complete and visible by then.  The latency
// of those loads overlaps the predecessor's tail; the arithmetic and its
// order are unchanged.
template <typename Real, int DIM>
__global__ void k_resid_coarse(StencilOp<Real> op, const Real* b, const Real* x, Real* r) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const bool on = idx < op.n;
  int i = 0, j = 0, k = 0;
  Real sv[stencil_size<DIM>()];
  if constexpr (DIM == 3) {
    const int i0 = blockIdx.x * blockDim.x;
    if (stencil_flat(op, i0, i0 + (int)blockDim.x)) {
      stencil_coefs_flat(op, idx, sv);
      pdl_wait();
      r[idx] = b[idx] - stencil_apply_flat(op, x, idx, sv);
      pdl_trigger();
      return;
    }
  }
  if (on) {
    coords(idx, op.fNX, op.fNXY, i, j, k);
    stencil_coefs<DIM>(op, i, j, k, sv);
  }
  pdl_wait();
  if (on) r[idx] = b[idx] - stencil_apply<DIM, Real, false>(op, x, i, j, k, sv);
  pdl_trigger();
}

// Small FP32 levels, 3D: the residual and its restriction in one launch.  A
// level of at most split_coarse_nodes nodes takes 3 to 4 us in either kernel,
// launch and round trips; here a block forms the residuals that its 4^3 coarse
// nodes read (9^3, one per thread, a share of 0.42 of them also formed by a
// neighbour) in shared memory.  33^3 -> 17^3 nodes: 4.0 + 3.6 -> 6.0 us, 17^3
// -> 9^3: 3.7 + 3.3 -> 4.6 us.
constexpr int kRR = 4, kRRF = 2 * kRR + 1, kRRThreads = 736;  // 23 warps >= 9^3
__global__ void __launch_bounds__(kRRThreads) k_resid_restrict3(
    StencilOp<float> op, const float* b, const float* x, Dims f, Dims cd,
    const float* __restrict__ dinvc, float omega, float* bc, float* xc) {
  __shared__ float rs[kRRF][kRRF][kRRF];
  const int t = threadIdx.x;
  const int tx = t % kRRF, ty = (t / kRRF) % kRRF, tz = t / (kRRF * kRRF);
  const int i = 2 * kRR * blockIdx.x - 1 + tx, j = 2 * kRR * blockIdx.y - 1 + ty,
            k = 2 * kRR * blockIdx.z - 1 + tz;
  const bool tile = tz < kRRF;
  const bool on = tile && i >= 0 && i < f.NX && j >= 0 && j < f.NY && k >= 0 && k < f.NZ;
  const int idx = i + f.NX * (j + f.NY * k);
  float sv[27];
  if (on) stencil_coefs<3>(op, i, j, k, sv);
  // the coarse node of this thread
  const int I = kRR * blockIdx.x + t % kRR, J = kRR * blockIdx.y + (t / kRR) % kRR,
            K = kRR * blockIdx.z + t / (kRR * kRR);
  const bool coarse = t < kRR * kRR * kRR && I < cd.NX && J < cd.NY && K < cd.NZ;
  const int ci = I + cd.NX * (J + cd.NY * K);
  const float dc = coarse && xc ? dinvc[ci] : 0.f;
  pdl_wait();
  float rv = 0.f;
  if (on) rv = b[idx] - stencil_apply<3, float, false>(op, x, i, j, k, sv);
  if (tile) rs[tz][ty][tx] = rv;
  pdl_trigger();
  __syncthreads();
  if (!coarse) return;
  int ix[3], iy[3], iz[3];
  float wx[3], wy[3], wz[3];
  restrict_taps(I, f.ex, ix, wx);
  restrict_taps(J, f.ey, iy, wy);
  restrict_taps(K, f.ez, iz, wz);
  const int lx = 2 * (t % kRR), ly = 2 * ((t / kRR) % kRR), lz = 2 * (t / (kRR * kRR));
  float acc = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float wyz = wy[q] * wz[c];
#pragma unroll
      for (int a = 0; a < 3; ++a) acc += (wyz * wx[a]) * rs[lz + c][ly + q][lx + a];
    }
  bc[ci] = acc;
  if (xc) xc[ci] = omega * dc * acc;
}

// FP32 restriction of the finest level's residual, 3D: a thread owns a column
// of coarse nodes and kRestrictChunk coarse planes; each fine plane's 3 x 3
// weighted sum serves the one or two coarse planes that read it, so a coarse
// node costs 22 loads without clamps instead of 27 with a weight and an index
// formed for each (390 instructions).  65^3 coarse nodes: 7.6 -> 6.3 us,
// 129^3: 41 -> 27 us; on few nodes the chain of planes costs more (38 x 27 x 21
// coarse nodes: 3.1 -> 4.8 us), so it is taken above split_coarse_nodes.
constexpr int kRestrictChunk = 2;
__global__ void k_restrict3(const float* r, float* bc, Dims f, Dims cd,
                            const float* __restrict__ dinvc, float omega, float* xc) {
  constexpr int KC = kRestrictChunk, NP = 2 * KC + 1;
  // (blocks numbered along x alone: planes may pass the second dimension's 65535)
  const int cNXY = cd.NX * cd.NY, blocks = (cNXY + (int)blockDim.x - 1) / (int)blockDim.x;
  const int chunk = blockIdx.x / blocks, col = (blockIdx.x - chunk * blocks) * blockDim.x + threadIdx.x;
  const bool on = col < cNXY;
  const int J = on ? col / cd.NX : 0, I = on ? col - J * cd.NX : 0, K0 = chunk * KC;
  int ix[3], iy[3];
  float wx[3], wy[3];
  restrict_taps(I, f.ex, ix, wx);
  restrict_taps(J, f.ey, iy, wy);
  float dc[KC];
#pragma unroll
  for (int u = 0; u < KC; ++u) dc[u] = on && xc && K0 + u < cd.NZ ? dinvc[col + cNXY * (K0 + u)] : 0.f;
  pdl_wait();
  if (on) {
    float s[NP];  // fine planes 2 K0 - 1 .. 2 K0 + 2 KC - 1
#pragma unroll
    for (int t = 0; t < NP; ++t) {
      const int k = 2 * K0 - 1 + t;
      s[t] = 0.f;
      if (k < 0 || k >= f.NZ) continue;
      const float* plane = r + (int64_t)f.NX * f.NY * k;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float* row = plane + f.NX * iy[q];
        s[t] += wy[q] * (wx[0] * row[ix[0]] + wx[1] * row[ix[1]] + wx[2] * row[ix[2]]);
      }
    }
#pragma unroll
    for (int u = 0; u < KC; ++u) {
      const int K = K0 + u;
      if (K >= cd.NZ) break;
      int iz[3];
      float wz[3];
      restrict_taps(K, f.ez, iz, wz);
      const float acc = wz[0] * s[2 * u] + wz[1] * s[2 * u + 1] + wz[2] * s[2 * u + 2];
      bc[col + cNXY * K] = acc;
      if (xc) xc[col + cNXY * K] = omega * dc[u] * acc;
    }
  }
  pdl_trigger();
}

template <typename Real, int DIM>
__global__ void k_post_coarse(StencilOp<Real> op, const Real* xc,
                              const Real* cur, const Real* b,
                              const Real* __restrict__ dinv, Real omega, Real* dst,
                              Dims f, Dims cd) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const bool on = idx < op.n;
  Real sv[stencil_size<DIM>()];
  if (on) {
    int i, j, k;
    coords(idx, op.fNX, op.fNXY, i, j, k);
    stencil_coefs<DIM>(op, i, j, k, sv);
  }
  pdl_wait();
  if (on) post_node<Real, DIM, false, true>(op, xc, cur, b, dinv, omega, dst, f, cd, idx, sv);
  pdl_trigger();
}

// One damped-Jacobi sweep on an assembled level, x' = x + w D^-1 (b - A x).
template <typename Real, int DIM>
__global__ void k_jacobi_st(StencilOp<Real> op, const Real* b, const Real* xin, Real* xout,
                            const Real* __restrict__ dinv, Real omega) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const bool on = idx < op.n;
  int i = 0, j = 0, k = 0;
  Real sv[stencil_size<DIM>()];
  Real dv = Real(0);
  if constexpr (DIM == 3) {
    const int i0 = blockIdx.x * blockDim.x;
    if (stencil_flat(op, i0, i0 + (int)blockDim.x)) {
      stencil_coefs_flat(op, idx, sv);
      dv = dinv[idx];
      pdl_wait();
      const Real ax = stencil_apply_flat(op, xin, idx, sv);
      xout[idx] = xin[idx] + omega * dv * (b[idx] - ax);
      pdl_trigger();
      return;
    }
  }
  if (on) {
    coords(idx, op.fNX, op.fNXY, i, j, k);
    stencil_coefs<DIM>(op, i, j, k, sv);
    dv = dinv[idx];
  }
  pdl_wait();
  if (on) {
    const Real ax = stencil_apply<DIM, Real, false>(op, xin, i, j, k, sv);
    xout[idx] = xin[idx] + omega * dv * (b[idx] - ax);
  }
  pdl_trigger();
}

// x = C b with the explicit inverse of the coarsest operator: a warp per
// row, the row's entries loaded before the wait when it has at most 128
// (four per lane), summed in the same order as coarse_row.
template <typename Real, typename M>
__global__ void k_coarse_solve(const M* __restrict__ cinv, const Real* b,
                               Real* x, int n) {
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool pre = n <= 128;
  M cv[4] = {M(0), M(0), M(0), M(0)};
  if (pre && row < n) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int jj = lane + 32 * q;
      const int jc = min(jj, n - 1);  // a valid address even where the entry is unused
      if (jj < n && CK((int64_t)row * n + jc, (int64_t)n * n)) cv[q] = cinv[(int64_t)row * n + jc];
    }
  }
  pdl_wait();
  pdl_trigger();
  if (row >= n) return;
  if (!pre) {
    coarse_row<Real, false, M>(cinv, b, x, n, row, lane);
    return;
  }
  M s = M(0);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int jj = lane + 32 * q;
    if (jj < n) s += cv[q] * (M)b[jj];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) x[row] = (Real)s;
}

// ------------------------------------------- bottom of the V-cycle, one cluster
// Levels lb .. nl-1 (each at most kBottomNodes nodes) of the zero-guess
// V-cycle in one launch of a thread-block cluster: the CTAs of the cluster
// stride over each level's nodes, and the hardware cluster barrier (release
// on arrive, acquire on wait) separates the phases, so the small levels cost
// no kernel launches and no waits of this code's own.
constexpr int kBottomThreads = 512;
constexpr int kBottomClusterMax = 16;  // non-portable cluster size, used when it fits

template <typename Real>
struct BottomArgs {
  StencilOp<Real> op[kMaxLevels];
  Dims L[kMaxLevels];
  Real* b[kMaxLevels];
  Real* x[kMaxLevels];
  Real* t[kMaxLevels];
  Real* r[kMaxLevels];
  const typename CoarseT<Real>::T* cinv;
  int nc, lb, nl;
  Real omega;
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n"
      "barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

template <typename Real, int DIM>
__global__ void __launch_bounds__(kBottomThreads) k_bottom(BottomArgs<Real> a) {
  pdl_wait();
  pdl_trigger();
  const int nthr = gridDim.x * blockDim.x;
  const int vt = blockIdx.x * blockDim.x + threadIdx.x;
  // x_l = w D^-1 b_l is already in place (left by the restriction)
  for (int l = a.lb; l + 1 < a.nl; ++l) {
    for (int idx = vt; idx < a.L[l].n; idx += nthr)
      resid_node<Real, DIM, true>(a.op[l], a.b[l], a.x[l], a.r[l], idx);
    cluster_barrier();
    Real* xn = l + 2 < a.nl ? a.x[l + 1] : nullptr;  // the coarsest level is solved
    for (int idx = vt; idx < a.L[l + 1].n; idx += nthr)
      restrict_node<Real, DIM, true>(a.r[l], a.b[l + 1], a.L[l], a.L[l + 1], nullptr, idx,
                                     a.op[l + 1].dinv, a.omega, xn);
    cluster_barrier();
  }
  {
    const int l = a.nl - 1;
    const int warp = vt >> 5, nwarps = nthr >> 5, lane = threadIdx.x & 31;
    for (int row = warp; row < a.nc; row += nwarps)
      coarse_row<Real, true, typename CoarseT<Real>::T>(a.cinv, a.b[l], a.x[l], a.nc, row, lane);
  }
  const Real* res = a.x[a.nl - 1];
  for (int l = a.nl - 2; l >= a.lb; --l) {
    cluster_barrier();
    for (int idx = vt; idx < a.L[l].n; idx += nthr)
      post_node<Real, DIM, true>(a.op[l], res, a.x[l], a.b[l], a.op[l].dinv, a.omega, a.t[l], a.L[l],
                                 a.L[l + 1], idx);
    res = a.t[l];
  }
}

__global__ void k_convert_d2f(const double* __restrict__ a, float* __restrict__ b, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (float)a[i];
}
__global__ void k_convert_f2d(const float* __restrict__ a, double* __restrict__ b, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (double)a[i];
}

// -------------------------------------------------------------------- host
template <typename Real>
static LevelBuf<Real>* levels(Ctx& c);
template <>
LevelBuf<double>* levels<double>(Ctx& c) { return c.h64; }
template <>
LevelBuf<float>* levels<float>(Ctx& c) { return c.h32; }

template <typename Real>
static const Real* ref_ke(Ctx& c);
template <>
const double* ref_ke<double>(Ctx& c) { return c.ke0; }
template <>
const float* ref_ke<float>(Ctx& c) { return c.ke0_f; }

template <typename Real, int DIM>
static FineRow<Real, DIM> fine_row(Ctx& c, const Real* ke, const Real* ksub) {
  FineRow<Real, DIM> r;
  const Dims& d = c.L[0];
  r.op = FineOp<Real>{ke, ksub, c.fixed, d.ex, d.ey, d.ez, d.NX, d.NY, d.NZ, (int)d.n, d.fNX, d.fNXY};
  return r;
}

template <typename Real, int DIM>
static StencilRow<Real, DIM> stencil_row(Ctx& c, int l) {
  StencilRow<Real, DIM> r;
  const Dims& d = c.L[l];
  r.op = StencilOp<Real>{levels<Real>(c)[l].st, levels<Real>(c)[l].dinv, d.NX, d.NY, d.NZ, (int)d.n,
                         d.fNX, d.fNXY};
  return r;
}

// One damped-Jacobi sweep xout = xin + omega D^-1 (b - A xin) on level l.
template <typename Real, int DIM>
static void sweep(Ctx& c, int l, const Real* b, const Real* xin, Real* xout) {
  const Dims& d = c.L[l];
  LevelBuf<Real>* h = levels<Real>(c);
  const Real om = (Real)c.p.omega;
  ProfScope ps(c, l == 0 ? MGAR_KC_SMOOTH0 : -1);
  if (l == 0)
    k_jacobi<<<blocks_for(d.n), kThreads, 0, c.stream>>>(fine_row<Real, DIM>(c, ref_ke<Real>(c), nullptr),
                                                         b, xin, xout, h[0].dinv, om);
  else
    launch_pdl(c.stream, c.use_pdl, k_jacobi_st<Real, DIM>, dim3(blocks_for(d.n)), dim3(kThreads),
               stencil_row<Real, DIM>(c, l).op, b, xin, xout, (const Real*)h[l].dinv, om);
  MGAR_LAUNCH_CHECK_AT(level_site(1, l));
}

template <typename Real, int DIM>
static void residual(Ctx& c, int l, const Real* b, const Real* x, Real* r) {
  const Dims& d = c.L[l];
  ProfScope ps(c, l == 0 ? MGAR_KC_RESID0 : -1);
  if (l == 0)
    k_residual<<<blocks_for(d.n), kThreads, 0, c.stream>>>(fine_row<Real, DIM>(c, ref_ke<Real>(c), nullptr),
                                                           b, x, r);
  else
    k_residual<<<blocks_for(d.n), kThreads, 0, c.stream>>>(stencil_row<Real, DIM>(c, l), b, x, r);
  MGAR_LAUNCH_CHECK_AT(level_site(2, l));
}

// First level handled by the cluster kernel (nl if none).
static int bottom_level(const Ctx& c) {
  if (!c.bottom_ok) return c.nl;
  int lb = c.nl - 1;
  while (lb - 1 >= 1 && c.L[lb - 1].n <= c.bottom_nodes) --lb;
  return lb;
}

template <typename Real, int DIM>
static void launch_bottom(Ctx& c, int lb) {
  LevelBuf<Real>* h = levels<Real>(c);
  BottomArgs<Real> a{};
  for (int l = lb; l < c.nl; ++l) {
    a.op[l] = stencil_row<Real, DIM>(c, l).op;
    a.L[l] = c.L[l];
    a.b[l] = h[l].b;
    a.x[l] = h[l].x;
    a.t[l] = h[l].t;
    a.r[l] = h[l].r;
  }
  a.cinv = CoarseT<Real>::inv(c);
  a.nc = c.nc;
  a.lb = lb;
  a.nl = c.nl;
  a.omega = (Real)c.p.omega;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.bottom_cluster);
  cfg.blockDim = dim3(kBottomThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = c.stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c.bottom_cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = c.use_pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  MGAR_CUDA(cudaLaunchKernelEx(&cfg, k_bottom<Real, DIM>, a));
  MGAR_LAUNCH_CHECK_AT("vc bottom");
}

template <typename Real, int DIM>
static bool bottom_fits(int csize) {
  if (csize > 8 &&
      cudaFuncSetAttribute(k_bottom<Real, DIM>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize);
  cfg.blockDim = dim3(kBottomThreads);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k_bottom<Real, DIM>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  return clusters >= 1;
}

// Whether the cluster kernel can run here (FP32 V-cycle), and with how many
// CTAs (16 if the device allows the non-portable size, else 8); call outside
// stream capture.
void bottom_prepare(Ctx& c) {
  c.bottom_ok = false;
  for (int csize = kBottomClusterMax; csize >= 8 && !c.bottom_ok; csize /= 2) {
    c.bottom_ok = c.dim == 3 && bottom_fits<float, 3>(csize);
    if (c.bottom_ok) c.bottom_cluster = csize;
  }
}

// dst = cur + P xc on level f (P from level cd; fixed nodes of f keep cur).
template <typename Real, int DIM>
static void launch_prolong(Ctx& c, bool pdl, const Real* xc, const Real* cur, Real* dst,
                           const Dims& f, const Dims& cd, const uint8_t* fixed) {
  if (DIM == 3 && c.prolong_col) {
    const int64_t cols = (int64_t)f.NX * f.NY;
    const int gz = (f.NZ + kProlongChunk - 1) / kProlongChunk;
    launch_pdl(c.stream, pdl && c.use_pdl, k_prolong3<Real>, dim3(blocks_for(cols), gz),
               dim3(kThreads), xc, cur, dst, f, cd, fixed);
  } else {
    launch_pdl(c.stream, pdl && c.use_pdl, k_prolong<Real, DIM>, dim3(blocks_for(f.n)),
               dim3(kThreads), xc, cur, dst, f, cd, fixed);
  }
}

// The coarsest level by its explicit inverse.
template <typename Real>
static void coarse_solve(Ctx& c) {
  LevelBuf<Real>* h = levels<Real>(c);
  const int l = c.nl - 1, rows_per_block = kThreads / 32;
  launch_pdl(c.stream, c.use_pdl, k_coarse_solve<Real, typename CoarseT<Real>::T>,
             dim3((c.nc + rows_per_block - 1) / rows_per_block), dim3(kThreads),
             (const typename CoarseT<Real>::T*)CoarseT<Real>::inv(c), (const Real*)h[l].b, h[l].x, c.nc);
  MGAR_LAUNCH_CHECK_AT(level_site(5, l));
}

// f with the rows per warp (1, 2 or 3) as a constant
template <class F>
static void with_rows(int rows, F&& f) {
  if (rows == 3) f(std::integral_constant<int, 3>{});
  else if (rows == 2) f(std::integral_constant<int, 2>{});
  else f(std::integral_constant<int, 1>{});
}

// Whether the tiled 2D passes can be launched: their rows of tiles are a launch's
// second dimension, which ends at 65535 (a domain of some 390,000 rows; longer
// ones take the general kernels).
bool tiles2d_ok(const Ctx& c) {
  using namespace l2d;
  constexpr int kMax = 65535;
  const int cy[4] = {0, Geo<1>::kCY, Geo<2>::kCY, Geo<3>::kCY}, uy[4] = {0, Geo<1>::kUY, Geo<2>::kUY, Geo<3>::kUY};
  const Dims &d0 = c.L[0], &d1 = c.L[1];
  if (tiles(d1.NY, cy[down_rows(d1.NX, d1.NY, c.sms)]) > kMax) return false;
  if (tiles(d0.NY, uy[up_rows(d0.NX, d0.NY, c.sms)]) > kMax) return false;
  for (int l = 1; l + 1 < c.nl; ++l)
    if (tiles(c.L[l + 1].NY, kDY) > kMax || tiles(c.L[l].NY, kPY) > kMax) return false;
  return true;
}

// The 2D V-cycle with one pre- and one post-sweep in the tiled passes: one
// launch per level and direction and the coarsest solve, in either precision
// (FP64 gains from the passes saved and, on small grids, from 2 instead of 5
// launches per level; its rims cost 8 % more FP64 operations).  dout: r . x
// (r = b, or rdot's pairs when given).
template <typename Real>
static void vcycle_fused2(Ctx& c, const Real* b0, Real* x0, bool zero_guess,
                          const float2* rdot = nullptr, SumOut dout = {}) {
  LevelBuf<Real>* h = levels<Real>(c);
  const int nl = c.nl;
  const Real om = (Real)c.p.omega;
  const Dims& d0 = c.L[0];
  auto next_x = [&](int l) { return l + 2 < nl ? h[l + 1].x : (Real*)nullptr; };
  auto coarse = [&](int l) {
    return l2d::Coarse<Real>{stencil_row<Real, 2>(c, l).op, c.L[l].ex, c.L[l].ey, c.L[l + 1].NX,
                             c.L[l + 1].NY, om};
  };
  const l2d::Fine<Real> f{ref_ke<Real>(c), h[0].dinv_s, d0.ex, d0.ey, c.L[1].NX, c.L[1].NY, om};
  {
    ProfScope ps(c, MGAR_KC_SMOOTH0);
    if (!zero_guess) sweep<Real, 2>(c, 0, b0, x0, h[0].t);
    ProfScope pr(c, MGAR_KC_RESID0);
    auto down = [&](auto rows) {
      constexpr int R = decltype(rows)::value;
      const dim3 grid(l2d::tiles(c.L[1].NX, l2d::kCX), l2d::tiles(c.L[1].NY, l2d::Geo<R>::kCY));
      launch_pdl(c.stream, c.use_pdl, zero_guess ? k_down2d<Real, R, true> : k_down2d<Real, R, false>,
                 grid, dim3(l2d::kThreads2), f, b0, h[0].t, h[1].b, (const Real*)h[1].dinv, next_x(0));
    };
    with_rows(l2d::down_rows(c.L[1].NX, c.L[1].NY, c.sms), down);
    MGAR_LAUNCH_CHECK_AT(level_site(0, 0));
  }
  for (int l = 1; l + 1 < nl; ++l) {
    const dim3 grid(l2d::tiles(c.L[l + 1].NX, l2d::kDX), l2d::tiles(c.L[l + 1].NY, l2d::kDY));
    launch_pdl(c.stream, c.use_pdl, k_coarse_down2d<Real>, grid, dim3(l2d::kDownThreads), coarse(l),
               (const Real*)h[l].b, (const Real*)h[l].x, h[l + 1].b, (const Real*)h[l + 1].dinv,
               next_x(l));
    MGAR_LAUNCH_CHECK_AT(level_site(3, l));
  }
  coarse_solve<Real>(c);
  const Real* res = h[nl - 1].x;
  for (int l = nl - 2; l >= 1; --l) {
    const dim3 grid(l2d::tiles(c.L[l].NX, l2d::kPX), l2d::tiles(c.L[l].NY, l2d::kPY));
    // (large levels: the additions' order of the interpolation as a pass of its own)
    launch_pdl(c.stream, c.use_pdl,
               c.L[l].n > c.split_coarse_nodes ? k_coarse_up2d<Real, false> : k_coarse_up2d<Real, true>,
               grid, dim3(l2d::kUpThreads), coarse(l), (const Real*)h[l].b, (const Real*)h[l].x, res,
               h[l].t);
    MGAR_LAUNCH_CHECK_AT(level_site(4, l));
    res = h[l].t;
  }
  ProfScope ps(c, MGAR_KC_SMOOTH0);
  const bool fused = sizeof(Real) == 8 && dout.out;
  auto up = [&](auto rows) {
    constexpr int R = decltype(rows)::value;
    const dim3 grid(l2d::tiles(d0.NX, l2d::kUX), l2d::tiles(d0.NY, l2d::Geo<R>::kUY));
    launch_pdl(c.stream, c.use_pdl, fused ? k_up2d<Real, R, true> : k_up2d<Real, R, false>, grid,
               dim3(l2d::kThreads2), f, b0, (const Real*)h[0].t, res, x0, c.partials, c.counter, dout);
  };
  with_rows(l2d::up_rows(d0.NX, d0.NY, c.sms), up);
  MGAR_LAUNCH_CHECK_AT(level_site(1, 0));
  if constexpr (sizeof(Real) == 4) {
    if (dout.out) {
      launch_pdl(c.stream, c.use_pdl, k_dot_rz, dim3(sum_phys(d0.n, 4)), dim3(kThreads), rdot, b0, (const float*)x0, (int)d0.n, c.partials, c.counter, dout);
      MGAR_LAUNCH_CHECK();
    }
  }
}

// Table 1 with one pre- and one post-sweep and a zero guess below the finest
// level, 3D: the tiled passes on the finest level, per coarse level the
// residual, the restriction (which leaves the next level's zero-guess sweep)
// and one fused post kernel (interpolation + smooth) or two on large levels; on
// request the small levels at the bottom run in one cluster launch (FP32).
template <typename Real>
static void vcycle_fused3(Ctx& c, const Real* b0, Real* x0, bool zero_guess,
                          const float2* rdot = nullptr, SumOut dout = {}) {
  constexpr int DIM = 3;
  LevelBuf<Real>* h = levels<Real>(c);
  const int nl = c.nl;
  const Real om = (Real)c.p.omega;
  const Real* res[kMaxLevels] = {};  // each coarse level's correction
  const Dims& d0 = c.L[0];
  // finest level, pre
  Real* cur0;
  {
    ProfScope ps(c, MGAR_KC_SMOOTH0);
    if (zero_guess) {
      fine3d(c, 0, ref_ke<Real>(c), b0, h[0].dinv, (const Real*)nullptr, (const Real*)nullptr, h[0].t,
             h[0].r);
    } else {
      fine3d(c, 3, ref_ke<Real>(c), b0, h[0].dinv, (const Real*)x0, (const Real*)nullptr, h[0].t,
             (Real*)nullptr);
      fine3d(c, 2, ref_ke<Real>(c), b0, h[0].dinv, (const Real*)h[0].t, (const Real*)nullptr, h[0].r,
             (Real*)nullptr);
    }
    cur0 = h[0].t;
  }
  // the tiled 3D kernels leave r = 0 on fixed nodes, which P^T = (Z P)^T ignores
  // each restriction into a level above the coarsest also leaves that
  // level's zero-guess sweep x = w D^-1 b
  Real* const x1 = nl > 2 ? h[1].x : nullptr;
  const Dims& d1 = c.L[1];
  bool columns = false;
  if constexpr (std::is_same<Real, float>::value) {
    columns = d1.n > c.split_coarse_nodes;
    if (columns)
      launch_pdl(c.stream, c.use_pdl, k_restrict3,
                 dim3(blocks_for((int64_t)d1.NX * d1.NY) * ((d1.NZ + kRestrictChunk - 1) / kRestrictChunk)),
                 dim3(kThreads), (const float*)h[0].r, h[1].b, d0, d1, (const float*)h[1].dinv, om, x1);
  }
  if (!columns) {
    launch_pdl(c.stream, c.use_pdl, k_restrict<Real, DIM>, dim3(blocks_for(c.L[1].n)), dim3(kThreads),
               (const Real*)h[0].r, h[1].b, d0, c.L[1], (const uint8_t*)nullptr,
               (const Real*)h[1].dinv, om, x1);
  }
  MGAR_LAUNCH_CHECK_AT(level_site(3, 0));
  const int lb = sizeof(Real) == 4 ? bottom_level(c) : nl;
  // coarse levels, down
  for (int l = 1; l + 1 < nl && l < lb; ++l) {
    const Dims& d = c.L[l];
    if constexpr (std::is_same<Real, float>::value) {
      if (d.n <= c.split_coarse_nodes) {
        const Dims& e = c.L[l + 1];
        const auto tiles = [](int n) { return (unsigned)((n + kRR - 1) / kRR); };
        launch_pdl(c.stream, c.use_pdl, k_resid_restrict3, dim3(tiles(e.NX), tiles(e.NY), tiles(e.NZ)),
                   dim3(kRRThreads), stencil_row<Real, DIM>(c, l).op, (const float*)h[l].b,
                   (const float*)h[l].x, d, e, (const float*)h[l + 1].dinv, om, h[l + 1].b,
                   l + 2 < nl ? h[l + 1].x : (float*)nullptr);
        MGAR_LAUNCH_CHECK_AT(level_site(0, l));
        continue;
      }
    }
    launch_pdl(c.stream, c.use_pdl, k_resid_coarse<Real, DIM>, dim3(blocks_for(d.n)), dim3(kThreads),
               stencil_row<Real, DIM>(c, l).op, (const Real*)h[l].b, (const Real*)h[l].x, h[l].r);
    MGAR_LAUNCH_CHECK_AT(level_site(0, l));
    launch_pdl(c.stream, c.use_pdl, k_restrict<Real, DIM>, dim3(blocks_for(c.L[l + 1].n)),
               dim3(kThreads), (const Real*)h[l].r, h[l + 1].b, d, c.L[l + 1],
               (const uint8_t*)nullptr, (const Real*)h[l + 1].dinv, om,
               l + 2 < nl ? h[l + 1].x : (Real*)nullptr);
    MGAR_LAUNCH_CHECK_AT(level_site(3, l));
  }
  if (lb < nl) {
    // levels lb .. nl-1 in one cluster launch
    if constexpr (sizeof(Real) == 4) launch_bottom<Real, DIM>(c, lb);
    res[nl - 1] = h[nl - 1].x;
    for (int l = lb; l + 1 < nl; ++l) res[l] = h[l].t;
  } else {
    coarse_solve<Real>(c);
    const int l = nl - 1;
    res[l] = h[l].x;
  }
  // coarse levels, up
  for (int l = std::min(nl - 2, lb - 1); l >= 1; --l) {
    const Dims& d = c.L[l];
    // FP64: interpolating at each of 27 neighbours takes longer than a launch
    // on every level (24 us on 9^3 and on 17^3 nodes, against 11 for the two)
    if (sizeof(Real) == 8 || d.n > c.split_coarse_nodes) {
      // large level: thin interpolation in place on x_l, then the sweep into t_l
      launch_prolong<Real, DIM>(c, true, res[l + 1], (const Real*)h[l].x, h[l].x, d, c.L[l + 1],
                                (const uint8_t*)nullptr);
      MGAR_LAUNCH_CHECK_AT(level_site(4, l));
      sweep<Real, DIM>(c, l, h[l].b, h[l].x, h[l].t);
    } else {
      launch_pdl(c.stream, c.use_pdl, k_post_coarse<Real, DIM>, dim3(blocks_for(d.n)),
                 dim3(kThreads), stencil_row<Real, DIM>(c, l).op, res[l + 1], (const Real*)h[l].x,
                 (const Real*)h[l].b, (const Real*)h[l].dinv, om, h[l].t, d, c.L[l + 1]);
      MGAR_LAUNCH_CHECK_AT(level_site(4, l));
    }
    res[l] = h[l].t;
  }
  // finest level, post (the timed class is the tiled pass alone)
  if (sizeof(Real) == 4 && !c.split_post) {
    ProfScope ps(c, MGAR_KC_SMOOTH0);
    fine3d(c, 1, ref_ke<Real>(c), b0, h[0].dinv, (const Real*)cur0, res[1], x0, (Real*)nullptr, rdot,
           dout);
  } else {
    // interpolation in place on the pre-smoothed iterate, then the tiled sweep
    launch_prolong<Real, DIM>(c, true, (const Real*)res[1], (const Real*)cur0, cur0, d0, c.L[1],
                              (const uint8_t*)c.fixed);
    MGAR_LAUNCH_CHECK_AT(level_site(4, 0));
    ProfScope ps(c, MGAR_KC_SMOOTH0);
    fine3d(c, 3, ref_ke<Real>(c), b0, h[0].dinv, (const Real*)cur0, (const Real*)nullptr, x0,
           (Real*)nullptr, rdot, dout);
  }
}

// General Table 1 V-cycle (any numbers of pre- and post-sweeps).
template <typename Real, int DIM>
static void vcycle_dim(Ctx& c, const Real* b0, Real* x0, bool zero_guess) {
  if (c.p.nu_pre == 1 && c.p.nu_post == 1 && c.nl >= 2 && !c.untiled) {
    if constexpr (DIM == 2) vcycle_fused2<Real>(c, b0, x0, zero_guess);
    else vcycle_fused3<Real>(c, b0, x0, zero_guess);
    return;
  }
  LevelBuf<Real>* h = levels<Real>(c);
  const int nl = c.nl;
  const Real om = (Real)c.p.omega;
  Real* cur[kMaxLevels];
  // downward leg
  for (int l = 0; l + 1 < nl; ++l) {
    const Dims& d = c.L[l];
    const Real* b = l == 0 ? b0 : h[l].b;
    Real* x = l == 0 ? x0 : h[l].x;
    Real* other = h[l].t;
    Real* cu = x;
    int sweeps = c.p.nu_pre;
    if (l > 0 || zero_guess) {
      if (sweeps > 0) {
        ProfScope ps(c, l == 0 ? MGAR_KC_SMOOTH0 : -1);
        k_jacobi_zero<<<blocks_for(d.n), kThreads, 0, c.stream>>>(b, x, h[l].dinv, om, (int)d.n);
        MGAR_LAUNCH_CHECK_AT(level_site(0, l));
        --sweeps;
      } else {
        MGAR_CUDA(cudaMemsetAsync(x, 0, d.n * sizeof(Real), c.stream));
      }
    }
    for (; sweeps > 0; --sweeps) {
      Real* dst = (cu == x) ? other : x;
      sweep<Real, DIM>(c, l, b, cu, dst);
      cu = dst;
    }
    cur[l] = cu;
    residual<Real, DIM>(c, l, b, cu, h[l].r);
    k_restrict<Real, DIM><<<blocks_for(c.L[l + 1].n), kThreads, 0, c.stream>>>(
        h[l].r, h[l + 1].b, d, c.L[l + 1], l == 0 ? c.fixed : nullptr);
    MGAR_LAUNCH_CHECK_AT(level_site(3, l));
  }
  coarse_solve<Real>(c);
  // upward leg
  for (int l = nl - 2; l >= 0; --l) {
    const Dims& d = c.L[l];
    const Real* b = l == 0 ? b0 : h[l].b;
    Real* x = l == 0 ? x0 : h[l].x;
    Real* other = h[l].t;
    const int post = c.p.nu_post;
    Real* dst = (post % 2 == 0) ? x : other;
    launch_prolong<Real, DIM>(c, false, (const Real*)h[l + 1].x, (const Real*)cur[l], dst, d,
                              c.L[l + 1], l == 0 ? (const uint8_t*)c.fixed : nullptr);
    MGAR_LAUNCH_CHECK_AT(level_site(4, l));
    Real* cu = dst;
    for (int s = 0; s < post; ++s) {
      Real* nxt = (cu == x) ? other : x;
      sweep<Real, DIM>(c, l, b, cu, nxt);
      cu = nxt;
    }
  }
}

template <typename Real>
void vcycle(Ctx& c, const Real* b, Real* x, bool zero_guess) {
  if (c.dim == 2) vcycle_dim<Real, 2>(c, b, x, zero_guess);
  else vcycle_dim<Real, 3>(c, b, x, zero_guess);
}
template void vcycle<double>(Ctx&, const double*, double*, bool);
template void vcycle<float>(Ctx&, const float*, float*, bool);

void vcycle_dot(Ctx& c, const float* b, float* x, const float2* r, SumOut dout) {
  require(vcycle_dot_ok(c), MGAR_ERR_ARG,
          "fused r.z V-cycle needs one pre- and one post-sweep, two levels and the tiled 3D kernels");
  if (c.dim == 2) vcycle_fused2<float>(c, b, x, true, r, dout);
  else vcycle_fused3<float>(c, b, x, true, r, dout);
}

void vcycle_dot64(Ctx& c, const double* b, double* x, SumOut dout) {
  if (c.dim == 2) vcycle_fused2<double>(c, b, x, true, nullptr, dout);
  else vcycle_fused3<double>(c, b, x, true, nullptr, dout);
}

void cg_dir64(Ctx& c, const double* z, const double* p_old, double* p, const double* beta, bool first,
              const double* parity, double* y, SumOut dot) {
  ProfScope ps(c, MGAR_KC_APPLY64);
  if (c.dim == 3) {
    fine3d_dir64(c, z, p_old, p, beta, first, parity, y, dot);
    return;
  }
  const Dims& d = c.L[0];
  with_rows(l2d::up_rows(d.NX, d.NY, c.sms), [&](auto rows) {
    constexpr int R = decltype(rows)::value;
    const dim3 grid(l2d::tiles(d.NX, l2d::kUX), l2d::tiles(d.NY, l2d::Geo<R>::kUY));
    launch_pdl(c.stream, c.use_pdl, k_dir2d<R>, grid, dim3(l2d::kThreads2), (const double*)c.ke,
               (const uint8_t*)c.fixed, d.ex, d.ey, z, p_old, p, beta, first ? 1 : 0, parity, y,
               c.partials, c.counter, dot);
  });
  MGAR_LAUNCH_CHECK();
}

template <typename Real, int DIM>
static void apply_dim(Ctx& c, const Real* ke, const Real* ksub, const Real* x, Real* y, Real scale,
                      SumOut dot_out) {
  const Dims& d = c.L[0];
  auto row = fine_row<Real, DIM>(c, ke, ksub);
  if (dot_out.out)
    k_apply<FineRow<Real, DIM>, Real, true><<<blocks_for(d.n), kThreads, 0, c.stream>>>(
        row, x, y, scale, c.partials, c.counter, dot_out);
  else
    k_apply<FineRow<Real, DIM>, Real, false><<<blocks_for(d.n), kThreads, 0, c.stream>>>(
        row, x, y, scale, nullptr, nullptr, SumOut{});
  MGAR_LAUNCH_CHECK();
}

void apply_fine64(Ctx& c, const double* ke, const double* x, double* y, SumOut dot_out) {
  ProfScope ps(c, MGAR_KC_APPLY64);
  if (c.dim == 2) apply_dim<double, 2>(c, ke, nullptr, x, y, 1.0, dot_out);
  else if (!c.untiled) fine3d_apply64(c, ke, nullptr, x, y, 1.0, dot_out);
  else apply_dim<double, 3>(c, ke, nullptr, x, y, 1.0, dot_out);
}
// y = -(A - A0) x
void apply_dK64(Ctx& c, const double* x, double* y) {
  if (c.dim == 2) apply_dim<double, 2>(c, c.ke, c.ke0, x, y, -1.0, {});
  else if (!c.untiled) fine3d_apply64(c, c.ke, c.ke0, x, y, -1.0, {});
  else apply_dim<double, 3>(c, c.ke, c.ke0, x, y, -1.0, {});
}
void apply_dK32(Ctx& c, const float* x, float* y) {
  if (c.dim == 2) apply_dim<float, 2>(c, c.ke_f, c.ke0_f, x, y, -1.f, {});
  else apply_dim<float, 3>(c, c.ke_f, c.ke0_f, x, y, -1.f, {});
}

void convert_d2f(Ctx& c, const double* a, float* b, int64_t n) {
  k_convert_d2f<<<blocks_for(n), kThreads, 0, c.stream>>>(a, b, n);
  MGAR_LAUNCH_CHECK();
}
void convert_f2d(Ctx& c, const float* a, double* b, int64_t n) {
  k_convert_f2d<<<blocks_for(n), kThreads, 0, c.stream>>>(a, b, n);
  MGAR_LAUNCH_CHECK();
}

}  // namespace mgar
