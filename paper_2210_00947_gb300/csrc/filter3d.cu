// The 3D density filter and its transpose (Eq. 6-8) of the mixed path for radii
// above 2, in double-float arithmetic.
//
// The weight of an offset depends on its length alone, so of the (2R+1)^3
// offsets of a filter of reach R only those with 0 <= b <= a in the plane and
// 0 <= d across it differ.  A block owns a column of 32 x 8 elements and walks
// along z; per plane of the input a thread
//   sums the in-plane neighbours of each class (a, b) once (up to eight),
//   forms the plane's contribution at distance d, Q_d = sum_ab w(a,b,d) S_ab,
//   and adds Q_d to the outputs d planes below and above it, which it carries
//   in registers.
// With 1033 offsets (radius 6.27) that is 123 additions and 134 products per
// element instead of 1033 products, and 123 shared-memory loads instead of 1033
// loads through L1.  The kernels are bound by the FP32 pipe: 224 x 112 x 112
// elements, 2.90 ms per filter offset by offset.
//
// Radii up to 2 (reach 1: at most 27 offsets) stay with the offset-by-offset
// kernels, which are bound by memory there.
#include "common.cuh"
#include "filter3d.cuh"

namespace mgar {
namespace f3f {

constexpr int TX = 32, TY = 8, NT = TX * TY;
constexpr int kMaxR = 8;  // the tables hold 3072 offsets: radius below 9.1
constexpr int kMaxCls = (kMaxR + 1) * (kMaxR + 2) / 2;

struct Classes {
  int n8, n;           // classes of eight neighbours, then of four, then the centre
  int4 off[kMaxCls][2];  // tile offsets of the neighbours
  int dmax[kMaxCls];
  float2 w[kMaxCls][kMaxR + 1];
};

// Offsets and weights of radius r.
__global__ void k_filter_classes(Classes* c, double r, int R) {
  if (threadIdx.x == 0) {
    const int W = TX + 2 * R;
    int cnt8 = 0, cnt4 = 0;
    for (int pass = 0; pass < 3; ++pass)
      for (int a = 0; a <= R; ++a)
        for (int b = 0; b <= a; ++b) {
          const int n = a == 0 ? 1 : (b == 0 || a == b) ? 4 : 8;
          if (n != (pass == 0 ? 8 : pass == 1 ? 4 : 1)) continue;
          if (!(r - sqrt((double)(a * a + b * b)) > 0.0)) continue;
          const int q = cnt8 + cnt4;
          if (n == 8) ++cnt8;
          else ++cnt4;
          int4 o0, o1 = make_int4(0, 0, 0, 0);
          if (n == 8) {
            o0 = make_int4(a + W * b, -a + W * b, a - W * b, -a - W * b);
            o1 = make_int4(b + W * a, -b + W * a, b - W * a, -b - W * a);
          } else if (b == 0) {
            o0 = make_int4(a, -a, W * a, -W * a);
          } else {
            o0 = make_int4(a + W * a, -a + W * a, a - W * a, -a - W * a);
          }
          if (n == 1) o0 = make_int4(0, 0, 0, 0);
          c->off[q][0] = o0;
          c->off[q][1] = o1;
          int dm = 0;
          for (int d = 0; d <= R; ++d) {
            const double w = r - sqrt((double)(a * a + b * b + d * d));
            df v{0.f, 0.f};
            if (w > 0.0) {
              v = df_from_double(w);
              dm = d;
            }
            c->w[q][d] = make_float2(v.hi, v.lo);
          }
          c->dmax[q] = dm;
        }
    c->n8 = cnt8;
    c->n = cnt8 + cnt4;
  }
}

// (ah, al) += x, the rounding errors gathered in al
__device__ __forceinline__ void add_to(float& ah, float& al, float xh, float xl) {
  float t, e;
  two_sum(ah, xh, t, e);
  ah = t;
  al = __fadd_rn(al, __fadd_rn(e, xl));
}
// (ah, al) += w * (xh, xl)
__device__ __forceinline__ void add_prod(float& ah, float& al, float2 w, float xh, float xl) {
  float p, e;
  two_prod(w.x, xh, p, e);
  e = __fmaf_rn(w.x, xl, e);
  e = __fmaf_rn(w.y, xh, e);
  add_to(ah, al, p, e);
}

template <int R, class Out>
__global__ void __launch_bounds__(NT, R <= 4 ? 3 : 2)
    k_filter3(const float2* __restrict__ in, const Classes* __restrict__ cls, int ex, int ey, int ez,
              int runs, Out out) {
  constexpr int W = TX + 2 * R, H = TY + 2 * R, CELLS = W * H, LPT = (CELLS + NT - 1) / NT;
  __shared__ float2 P[2][CELLS];
  __shared__ int4 off[kMaxCls][2];
  __shared__ float2 wt[kMaxCls][R + 1];
  __shared__ int dmx[kMaxCls];
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const int n8 = cls->n8, n = cls->n;
  for (int q = tid; q < n; q += NT) {
    off[q][0] = cls->off[q][0];
    off[q][1] = cls->off[q][1];
    dmx[q] = cls->dmax[q];
    for (int d = 0; d <= R; ++d) wt[q][d] = cls->w[q][d];
  }
  // (a plane's tiles numbered along x alone: their rows may pass the second
  // dimension's 65535)
  const int ntx = (ex + TX - 1) / TX, by = blockIdx.x / ntx;
  const int i0 = (blockIdx.x - by * ntx) * TX, j0 = by * TY;
  const int z0 = (int)((int64_t)blockIdx.z * ez / runs), z1 = (int)((int64_t)(blockIdx.z + 1) * ez / runs);
  const int i = i0 + tx, j = j0 + ty;
  const bool mine = i < ex && j < ey;
  // this thread's cells of a plane tile
  int cell_at[LPT];
#pragma unroll
  for (int q = 0; q < LPT; ++q) {
    const int c = tid + q * NT, cy = c / W, cx = c - cy * W;
    const int ii = i0 - R + cx, jj = j0 - R + cy;
    cell_at[q] = c < CELLS && ii >= 0 && ii < ex && jj >= 0 && jj < ey ? ii + ex * jj : -1;
  }
  const int plane = ex * ey;
  float2 nxt[LPT];
  auto fetch = [&](int z) {
#pragma unroll
    for (int q = 0; q < LPT; ++q) {
      nxt[q] = make_float2(0.f, 0.f);
      if (cell_at[q] >= 0 && z >= 0 && z < ez) nxt[q] = in[cell_at[q] + (int64_t)plane * z];
    }
  };
  // outputs p - R .. p + R of the current plane p
  float ah[2 * R + 1], al[2 * R + 1];
#pragma unroll
  for (int q = 0; q <= 2 * R; ++q) ah[q] = al[q] = 0.f;
  const int centre = (tx + R) + W * (ty + R);
  // planes past the grid add nothing and only finish outputs
  fetch(z0 - R);
  int buf = 0;
  for (int p = z0 - R; p < z1 + R; ++p, buf ^= 1) {
#pragma unroll
    for (int q = 0; q < LPT; ++q)
      if (tid + q * NT < CELLS) P[buf][tid + q * NT] = nxt[q];
    fetch(p + 1);
    __syncthreads();
    if (p >= 0 && p < ez) {
      const float2* S = &P[buf][centre];
      float qh[R + 1], ql[R + 1];
#pragma unroll
      for (int d = 0; d <= R; ++d) qh[d] = ql[d] = 0.f;
      auto spread = [&](int c, float sh, float sl) {
        const int dm = dmx[c];
#pragma unroll
        for (int d = 0; d <= R; ++d)
          if (d <= dm) add_prod(qh[d], ql[d], wt[c][d], sh, sl);
      };
      for (int c = 0; c < n8; ++c) {
        const int4 o = off[c][0], u = off[c][1];
        const float2 v0 = S[o.x], v1 = S[o.y], v2 = S[o.z], v3 = S[o.w];
        const float2 v4 = S[u.x], v5 = S[u.y], v6 = S[u.z], v7 = S[u.w];
        // two chains of four
        float sh = v0.x, sl = v0.y, th = v4.x, tl = v4.y;
        add_to(sh, sl, v1.x, v1.y);
        add_to(th, tl, v5.x, v5.y);
        add_to(sh, sl, v2.x, v2.y);
        add_to(th, tl, v6.x, v6.y);
        add_to(sh, sl, v3.x, v3.y);
        add_to(th, tl, v7.x, v7.y);
        add_to(sh, sl, th, tl);
        spread(c, sh, sl);
      }
      for (int c = n8; c < n - 1; ++c) {
        const int4 o = off[c][0];
        const float2 v0 = S[o.x], v1 = S[o.y], v2 = S[o.z], v3 = S[o.w];
        float sh = v0.x, sl = v0.y, th = v2.x, tl = v2.y;
        add_to(sh, sl, v1.x, v1.y);
        add_to(th, tl, v3.x, v3.y);
        add_to(sh, sl, th, tl);
        spread(c, sh, sl);
      }
      {
        const float2 v = S[0];
        spread(n - 1, v.x, v.y);
      }
      add_to(ah[R], al[R], qh[0], ql[0]);
#pragma unroll
      for (int d = 1; d <= R; ++d) {
        add_to(ah[R + d], al[R + d], qh[d], ql[d]);
        add_to(ah[R - d], al[R - d], qh[d], ql[d]);
      }
    }
    if (mine && p - R >= z0) out(i + ex * j + plane * (p - R), df_make(ah[0], al[0]));
#pragma unroll
    for (int q = 0; q < 2 * R; ++q) {
      ah[q] = ah[q + 1];
      al[q] = al[q + 1];
    }
    ah[2 * R] = al[2 * R] = 0.f;
  }
}

int reach(double r) { return (int)std::ceil(r) - 1; }

template <int R, class Out>
void launch_r(Ctx& c, const float2* in, const Out& out) {
  const Dims& d = c.L[0];
  const int gx = (d.ex + TX - 1) / TX, gy = (d.ey + TY - 1) / TY;
  // one wave of resident blocks, but runs of no fewer than 2 R planes (each
  // run reads 2 R planes more than it owns)
  int per_sm = 1;
  MGAR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter3<R, Out>, NT, 0));
  const int want = std::max(1, std::max(per_sm, 1) * c.sms / (gx * gy));
  const int runs = std::max(1, std::min(want, d.ez / (2 * R)));
  k_filter3<R, Out><<<dim3(gx * gy, 1, runs), NT, 0, c.stream>>>(
      in, reinterpret_cast<const Classes*>(c.f_cls), d.ex, d.ey, d.ez, runs, out);
  MGAR_LAUNCH_CHECK();
}

template <class Out>
void launch(Ctx& c, const float2* in, const Out& out) {
  switch (reach(c.filter_r)) {
    case 2: launch_r<2>(c, in, out); break;
    case 3: launch_r<3>(c, in, out); break;
    case 4: launch_r<4>(c, in, out); break;
    case 5: launch_r<5>(c, in, out); break;
    case 6: launch_r<6>(c, in, out); break;
    case 7: launch_r<7>(c, in, out); break;
    default: launch_r<8>(c, in, out); break;
  }
}

struct SimpOut {
  SimpArgs a;
  __device__ __forceinline__ void operator()(int e, df s) const { simp_store(a, e, s); }
};

struct TransposeOut {
  double* out;
  float2* out_df;
  __device__ __forceinline__ void operator()(int e, df v) const {
    if (out_df) {
      // renormalised by TwoSum: the pair an FP64 round trip of hi + lo gives
      float sh, se;
      two_sum(v.hi, v.lo, sh, se);
      out_df[e] = make_float2(sh, se);
    } else {
      out[e] = df_to_double(v);
    }
  }
};

}  // namespace f3f

bool filter3d_ok(const Ctx& c) {
  const int R = f3f::reach(c.filter_r);
  return c.dim == 3 && c.f_cls && R >= 2 && R <= f3f::kMaxR;
}

void filter3d_classes(Ctx& c) {
  if (c.dim != 3 || c.p.precision != MGAR_MIXED) return;
  if (!c.f_cls) MGAR_CUDA(cudaMalloc(&c.f_cls, sizeof(f3f::Classes)));
  if (!filter3d_ok(c)) return;
  f3f::k_filter_classes<<<1, 32, 0, c.stream>>>(reinterpret_cast<f3f::Classes*>(c.f_cls), c.filter_r,
                                                f3f::reach(c.filter_r));
  MGAR_LAUNCH_CHECK();
}

void filter3d_simp(Ctx& c, const float2* rho, const SimpArgs& a) {
  f3f::launch(c, rho, f3f::SimpOut{a});
}

void filter3d_t(Ctx& c, const float2* in, double* out, float2* out_df) {
  f3f::launch(c, in, f3f::TransposeOut{out, out_df});
}

}  // namespace mgar
