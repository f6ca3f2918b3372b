// FP32 passes of the finest 3D (H8) level on linear segments of the node
// planes: the V-cycle's pre-smoothing, residual and sweep, and the CG's
// direction update and product.
//
// Conductivities stand at the pitch of the nodes, zero where a node has no
// element at its upper corner (kn: element (i, j, k) at node (i, j, k)), so the
// elements around node m of a layer are kn[m - NX - 1], kn[m - NX], kn[m - 1],
// kn[m], off-grid ones are zero by themselves, and whatever value stands at an
// off-grid neighbour's place (the end of the row before, a plane's last row) is
// multiplied by zero.  So a block takes a run of consecutive nodes of the
// plane, whatever its rows, and walks along z; it stages the run and NX + 1
// nodes on either side, and no thread looks at coordinates, rims or bounds
// other than the array's.  Fixed nodes are the negative entries of the signed
// inverse diagonal; neighbours see them as zero.
//
// These passes are bound by instruction issue: a tiled form with rim loads and
// bounds tests executes 226 warp instructions per 32 nodes.  On 257^3 nodes,
// tiled -> segments: pre 193 -> 90, sweep 208 -> 105, direction and product
// 195 -> 122 us (bytes alone: 53); on 129^3, whose runs of eight planes pay two
// of prologue each, 20.1 -> 16.0, 25.5 -> 21.5 and 24.6 -> 24.8 us.
//
// The row is split by element layer as in fine3d.cu: the layer between planes k
// and k+1 gives row k's "up" part and row k+1's "down" part, a step reads one
// plane and one layer (12 shared-memory loads per node), and the down part and
// plane k's eight in-plane neighbours are carried in registers.  Two slots of
// each and one barrier per plane.
#include "common.cuh"

namespace mgar {
namespace f3l {

enum Mode { PRE = 0, RESID = 1, SWEEP = 2, DIR = 3 };
constexpr int NT = 512, NPT = 2;  // threads, nodes per thread
constexpr int kMaxSL = 5;  // staged cells per thread: 40 KB of slots at 5

struct Args {
  int NX, NXY, NZ, n;
  int L, gz;            // nodes per segment, z runs
  const float* kn;      // conductivities at node pitch
  const float* dinv;    // 1/diag, negated on fixed nodes
  const float* b;       // DIR: z
  const float* x;       // RESID, SWEEP: iterate; DIR: p_old
  float* out0;          // PRE: x; RESID: r; SWEEP: x'; DIR: p
  float* out1;          // PRE: r; DIR: A p
  float omega;
  const float2* rdot;   // SWEEP: r of r . x' in df64 pairs (null: b)
  double* partials;
  unsigned int* counter;
  SumOut dout;          // SWEEP: r . x'; DIR: p . A p
  // DIR: beta (a df64 pair), or 0 while *first is nonzero; with *parity odd,
  // p_old is x_alt and p goes to out_alt; rz_set receives *rz_new
  const double* beta;
  const double* rz_new;
  const double* first;
  const double* parity;
  const float* x_alt;
  float* out_alt;
  double* rz_set;
};

// The up and down parts (times 12) of a node column's rows for one layer: e_q
// its four elements, nb plane lo's in-plane neighbours (four diagonal, then -x,
// +x, -y, +y) on entry and plane hi's on return.
__device__ __forceinline__ void layer_rows(const float* __restrict__ K, const float* __restrict__ X,
                                           int m, int NX, float (&nb)[8], float x_lo, float x_hi,
                                           float& up, float& down) {
  const float e00 = K[m - NX - 1], e01 = K[m - NX], e10 = K[m - 1], e11 = K[m];
  float h[8];
  h[0] = X[m - NX - 1];
  h[1] = X[m - NX + 1];
  h[2] = X[m + NX - 1];
  h[3] = X[m + NX + 1];
  h[4] = X[m - 1];
  h[5] = X[m + 1];
  h[6] = X[m - NX];
  h[7] = X[m + NX];
  const float ew = e00 + e10, ee = e01 + e11, es = e00 + e01, en = e10 + e11;
  const float s4 = 4.f * (es + en);
  const float cc = e00 * (nb[0] + h[0]) + e01 * (nb[1] + h[1]) + e10 * (nb[2] + h[2]) +
                   e11 * (nb[3] + h[3]);
  const float elo = ew * nb[4] + ee * nb[5] + es * nb[6] + en * nb[7];
  const float ehi = ew * h[4] + ee * h[5] + es * h[6] + en * h[7];
  up = s4 * x_lo - cc - ehi;
  down = s4 * x_hi - cc - elo;
#pragma unroll
  for (int q = 0; q < 8; ++q) nb[q] = h[q];
}

template <int MODE, int SL>
__global__ void __launch_bounds__(NT, 2) k_fine3l(Args a) {
  constexpr int S = NT * SL;
  extern __shared__ float sm[];  // X slots 0, 1, then K slots 0, 1, S cells each
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, NX = a.NX, NXY = a.NXY;
  const int seg = blockIdx.x * a.L;
  const int kb = (int)(((int64_t)blockIdx.y * a.NZ) / a.gz);
  const int kend = (int)(((int64_t)(blockIdx.y + 1) * a.NZ) / a.gz);
  float om = a.omega;
  const float* xsrc = a.x;
  float* pdst = a.out0;
  // DIR: p_old counts as zero, whatever it holds, for the first direction: a
  // mask and not a condition on the loads (129 -> 122 us on 257^3 nodes).
  unsigned keep = ~0u;
  auto kept = [&](float v) { return __uint_as_float(__float_as_uint(v) & keep); };
  if (MODE == DIR) {
    const bool first = is_set(a.first);
    keep = first ? 0u : ~0u;
    om = first ? 0.f : load_pair(a.beta).hi;
    if (a.parity && is_set(a.parity)) {
      xsrc = a.x_alt;
      pdst = a.out_alt;
    }
  }
  // staged cell q of this thread: plane-linear node lin0 + NT q
  const int lin0 = seg - NX - 1 + tid;
  float v0[SL], v1[SL], vk[SL];
  // loads of plane k (operands v0, v1) and of layer l (vk)
  auto load_plane = [&](int k) {
    const bool in = k >= 0 && k < a.NZ;
    const int at = k * NXY + lin0;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const int idx = at + NT * q;
      const bool ok = in && (unsigned)idx < (unsigned)a.n;
      v0[q] = 0.f;
      v1[q] = -1.f;
      if (ok) {
        v1[q] = a.dinv[idx];
        if (MODE == PRE) v0[q] = a.b[idx];
        else if (MODE == DIR) v0[q] = fmaf(om, kept(xsrc[idx]), a.b[idx]);
        else v0[q] = xsrc[idx];
      }
    }
  };
  auto load_layer = [&](int l) {
    const bool in = l >= 0;
    const int at = l * NXY + lin0;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const int idx = at + NT * q;
      vk[q] = in && (unsigned)idx < (unsigned)a.n ? a.kn[idx] : 0.f;
    }
  };
  auto put_plane = [&](int s) {
    float* X = sm + s * S;
#pragma unroll
    for (int q = 0; q < SL; ++q) {
      const float x = MODE == PRE ? om * v1[q] * v0[q] : v0[q];
      X[tid + NT * q] = v1[q] > 0.f ? x : 0.f;
    }
  };
  auto put_layer = [&](int s) {
    float* K = sm + (2 + s) * S;
#pragma unroll
    for (int q = 0; q < SL; ++q) K[tid + NT * q] = vk[q];
  };
  // own nodes: run cell m[u] (staged at m + NX + 1)
  bool mine[NPT];
  int m[NPT];
#pragma unroll
  for (int u = 0; u < NPT; ++u) {
    const int c = tid + NT * u;
    mine[u] = c < a.L && seg + c < NXY;
    m[u] = min(c, S - 2 * (NX + 1) - 1) + NX + 1;  // a valid cell either way
  }
  // own operands of plane k: b and the signed 1/diag
  float ob[NPT], od[NPT];
  auto load_own = [&](int k) {
#pragma unroll
    for (int u = 0; u < NPT; ++u) {
      ob[u] = 0.f;
      od[u] = -1.f;
      if (mine[u] && k < a.NZ) {
        const int idx = k * NXY + seg + tid + NT * u;
        od[u] = a.dinv[idx];
        if (MODE != DIR) ob[u] = a.b[idx];
      }
    }
  };
  const bool rdot = (MODE == SWEEP || MODE == DIR) && a.dout.out != nullptr;
  df dacc{0.f, 0.f};
  float facc = 0.f;

  // planes kb - 1 and kb, layer kb - 1; then plane kb + 1 and layer kb in flight
  load_plane(kb - 1);
  put_plane((kb + 1) & 1);
  load_plane(kb);
  load_layer(kb - 1);
  put_plane(kb & 1);
  put_layer((kb + 1) & 1);
  load_plane(kb + 1);
  load_layer(kb);
  load_own(kb);
  __syncthreads();
  float nb[NPT][8], dk[NPT], xl[NPT];
#pragma unroll
  for (int u = 0; u < NPT; ++u) {
    const float* X = sm + ((kb + 1) & 1) * S;
    const float* Xh = sm + (kb & 1) * S;
    nb[u][0] = X[m[u] - NX - 1];
    nb[u][1] = X[m[u] - NX + 1];
    nb[u][2] = X[m[u] + NX - 1];
    nb[u][3] = X[m[u] + NX + 1];
    nb[u][4] = X[m[u] - 1];
    nb[u][5] = X[m[u] + 1];
    nb[u][6] = X[m[u] - NX];
    nb[u][7] = X[m[u] + NX];
    float up;
    xl[u] = Xh[m[u]];
    layer_rows(sm + (2 + ((kb + 1) & 1)) * S, Xh, m[u], NX, nb[u], X[m[u]], xl[u], up, dk[u]);
  }
  __syncthreads();  // plane kb - 1's slot is written next
  for (int k = kb; k < kend; ++k) {
    put_plane((k + 1) & 1);
    put_layer(k & 1);
    float cb[NPT], cd[NPT];
#pragma unroll
    for (int u = 0; u < NPT; ++u) {
      cb[u] = ob[u];
      cd[u] = od[u];
    }
    if (k + 1 < kend) {
      load_plane(k + 2);
      load_layer(k + 1);
      load_own(k + 1);
    }
    __syncthreads();
    const float* X = sm + ((k + 1) & 1) * S;
    const float* K = sm + (2 + (k & 1)) * S;
#pragma unroll
    for (int u = 0; u < NPT; ++u) {
      float up, down;
      const float xh = X[m[u]];
      layer_rows(K, X, m[u], NX, nb[u], xl[u], xh, up, down);
      const float acc = up + dk[u];
      dk[u] = down;
      float xi = xl[u];
      xl[u] = xh;
      if (!mine[u]) continue;
      const int idx = k * NXY + seg + tid + NT * u;
      const bool fx = cd[u] < 0.f;
      if (fx) {  // a fixed row is the identity, its value not in the tile
        if (MODE == PRE) xi = om * cb[u];
        else if (MODE == DIR) xi = fmaf(om, kept(xsrc[idx]), a.b[idx]);
        else xi = xsrc[idx];
      }
      const float ax = fx ? xi : acc * float(1.0 / 12.0);
      // r = 0 on fixed nodes: the restriction P^T = (Z P)^T does not read them
      if (MODE == PRE) {
        a.out0[idx] = xi;
        a.out1[idx] = fx ? 0.f : cb[u] - ax;
      } else if (MODE == RESID) {
        a.out0[idx] = fx ? 0.f : cb[u] - ax;
      } else if (MODE == DIR) {
        pdst[idx] = xi;
        a.out1[idx] = ax;
        facc = fmaf(xi, ax, facc);
      } else {
        const float xo = xi + om * fabsf(cd[u]) * (cb[u] - ax);
        a.out0[idx] = xo;
        if (rdot) {
          if (a.rdot) {
            const float2 rv = a.rdot[idx];
            dacc = df_add(dacc, df_mulf(df{rv.x, rv.y}, xo));
          } else {
            facc = fmaf(cb[u], xo, facc);
          }
        }
      }
    }
  }
  if (rdot) {
    const double other = sum_other(a.dout, tid == 0);
    double t;
    const int bid = blockIdx.x + gridDim.x * blockIdx.y, nblk = gridDim.x * gridDim.y;
    if (block_sum_last_df(df_add(dacc, df{facc, 0.f}), a.partials, a.counter, t, tid, NT, bid, nblk) &&
        tid == 0) {
      sum_out(a.dout, t, other);
      if (MODE == DIR) *a.rz_set = *a.rz_new;
    }
  }
}

// Segment length and cells per thread: a segment of L nodes stages L + 2 NX + 2
// cells, NT at a time, and its cost is about 12 instructions per staged cell
// and 45 per node.
bool shape(const Dims& d, int& L, int& SL) {
  double best = 0.0;
  SL = 0;
  for (int s = 2; s <= kMaxSL; ++s) {
    const int l = std::min(NT * NPT, NT * s - 2 * (d.NX + 1));
    if (l < NT / 2) continue;
    const int64_t segs = ((int64_t)d.NX * d.NY + l - 1) / l;
    const double cost = (double)segs * (12.0 * s + 45.0 * NPT);
    if (SL == 0 || cost < best) {
      best = cost;
      SL = s;
      L = l;
    }
  }
  return SL != 0;
}

template <int MODE, int SL>
void launch_sl(Ctx& c, Args& a) {
  const Dims& d = c.L[0];
  const int segs = (int)(((int64_t)d.NX * d.NY + a.L - 1) / a.L);
  launch_pdl_smem(c.stream, c.use_pdl, k_fine3l<MODE, SL>, dim3(segs, a.gz), dim3(NT),
                  (size_t)4 * NT * SL * sizeof(float), a);
}
template <int MODE>
void launch(Ctx& c, Args& a) {
  a.L = c.f3l_L;
  a.gz = c.f3l_gz;
  switch (c.f3l_SL) {
    case 2: launch_sl<MODE, 2>(c, a); break;
    case 3: launch_sl<MODE, 3>(c, a); break;
    case 4: launch_sl<MODE, 4>(c, a); break;
    default: launch_sl<MODE, 5>(c, a); break;
  }
}

Args base(Ctx& c) {
  const Dims& d = c.L[0];
  Args a{};
  a.NX = d.NX;
  a.NXY = d.NX * d.NY;
  a.NZ = d.NZ;
  a.n = (int)d.n;
  a.kn = c.kn0;
  a.dinv = c.h32[0].dinv_s;
  a.omega = (float)c.p.omega;
  a.partials = c.partials;
  a.counter = c.counter;
  return a;
}

}  // namespace f3l

// Buffers and launch shape at creation (3D mixed handles); rows too long for
// the staging (NX above 1151) keep the tiled passes.
void fine3l_prepare(Ctx& c) {
  using namespace f3l;
  const Dims& d = c.L[0];
  int L = 0, SL = 0;
  if (!shape(d, L, SL)) return;
  MGAR_CUDA(cudaMalloc(&c.kn0, d.n * sizeof(float)));
  MGAR_CUDA(cudaMalloc(&c.h32[0].dinv_s, d.n * sizeof(float)));
  c.f3l_L = L;
  c.f3l_SL = SL;
  // z runs: rounds of two blocks per SM times planes per run and its two
  // planes of prologue
  const int64_t segs = ((int64_t)d.NX * d.NY + L - 1) / L;
  double best = 0.0;
  for (int g = 1; g <= d.NZ; ++g) {
    const double rounds = std::ceil((double)(segs * g) / (2.0 * c.sms));
    const double cost = rounds * (std::ceil((double)d.NZ / g) + 2.0);
    if (g == 1 || cost < best) {
      best = cost;
      c.f3l_gz = g;
    }
  }
}

void fine3l(Ctx& c, int mode, const float* b, const float* x, float* out0, float* out1,
            const float2* rdot, SumOut dout) {
  using namespace f3l;
  Args a = base(c);
  a.b = b;
  a.x = x;
  a.out0 = out0;
  a.out1 = out1;
  a.rdot = rdot;
  a.dout = dout;
  if (mode == 0) launch<PRE>(c, a);
  else if (mode == 2) launch<RESID>(c, a);
  else launch<SWEEP>(c, a);
  MGAR_LAUNCH_CHECK_AT(level_site(mode == 0 ? 6 : mode == 2 ? 9 : 8, 0));
}

void fine3l_dir(Ctx& c, const float* z, const float* p_old, float* p, const double* beta,
                const double* first, const double* parity, float* y, SumOut dot,
                const double* rz_new, double* rz_set) {
  using namespace f3l;
  Args a = base(c);
  a.b = z;
  a.x = p_old;
  a.out0 = p;
  a.x_alt = p;
  a.out_alt = const_cast<float*>(p_old);
  a.out1 = y;
  a.beta = beta;
  a.rz_new = rz_new;
  a.first = first;
  a.parity = parity;
  a.rz_set = rz_set;
  a.dout = dot;
  launch<DIR>(c, a);
  MGAR_LAUNCH_CHECK();
}

}  // namespace mgar
