// The mixed path's SIMP epilogue of a filtered density (Eq. 4), and the 3D
// filter of larger radii (filter3d.cu).
#pragma once
#include "common.cuh"

namespace mgar {

// k_e = kmin + (k0 - kmin) rho~^p.  The constants come as double-float pairs
// (kmin_df, dk_df = k0 - kmin) and 1/Hs as pairs, so no thread converts them
// from FP64 (1/58 of the FP32 rate).
struct SimpArgs {
  const float2* inv_hs;
  double k0, kmin, penal;
  int cubic;  // penal == 3, compared once on the host
  float2 kmin_df, dk_df;
  double* rho_phys;
  float2* rho_df;
  double* ke;
  float* kf;
  float2* kdf;
};

// rho~_e = s / Hs and k_e: FP64 values, pairs, and k_e in FP32.
__device__ __forceinline__ void simp_store(const SimpArgs& a, int e, df s) {
  const float2 h = a.inv_hs[e];
  const df r = df_mul(s, df{h.x, h.y});
  a.rho_phys[e] = df_to_double(r);
  a.rho_df[e] = make_float2(r.hi, r.lo);  // the pair k_e comes from (rho_phys: its FP64 rounding)
  df kv;
  if (a.cubic) {
    kv = df_add(df{a.kmin_df.x, a.kmin_df.y},
                df_mul(df{a.dk_df.x, a.dk_df.y}, df_mul(df_mul(r, r), r)));
  } else {
    kv = df_from_double(a.kmin + (a.k0 - a.kmin) * pow(df_to_double(r), a.penal));
  }
  a.ke[e] = df_to_double(kv);
  a.kf[e] = __fadd_rn(kv.hi, kv.lo);
  a.kdf[e] = make_float2(kv.hi, kv.lo);
}

// Whether the current radius has the class form (3D mixed handles, radius
// above 2), its tables for a new radius, the filter with the SIMP
// conductivities, and the transpose (of an input already scaled by 1/Hs; FP64
// out, or pairs when out_df is given).
bool filter3d_ok(const Ctx& c);
void filter3d_classes(Ctx& c);
void filter3d_simp(Ctx& c, const float2* rho, const SimpArgs& a);
void filter3d_t(Ctx& c, const float2* in, double* out, float2* out_df);

}  // namespace mgar
