// The level search's counters and the places in its list of lattice points
// (design.cu).  Grids of up
// to 2^26 nodes have up to 125 points per element, more than 2^32 in all, and a
// field of coinciding values offers every one of them to the list: the count
// is 64 bits wide, and a place is compared with the list's capacity as it is,
// never narrowed.  No CUDA header, so that a host program can check the rule.
#pragma once

#ifdef __CUDACC__
#define MGAR_PP_HD __host__ __device__ __forceinline__
#else
#define MGAR_PP_HD inline
#endif

namespace mgar {

using PpCount = unsigned long long;
constexpr int kPpBins = 4096;

struct PpCtrl {
  PpCount hist[2][kPpBins];
  PpCount above[3];       // points past the bracket of each histogram pass and of the listing
  unsigned lo[3], hi[3];  // bracket (bit patterns, inclusive) of each pass
  PpCount nlist;          // points met by the listing
  int bad;                // a nodal value is not in [0, 1e37]
};

// Whether the point that was given place `slot` (from 0) is in the list.
MGAR_PP_HD bool pp_listed(PpCount slot, int cap) { return slot < static_cast<PpCount>(cap); }

// Whether every point met so far is in the list.
MGAR_PP_HD bool pp_complete(PpCount count, int cap) { return count <= static_cast<PpCount>(cap); }

}  // namespace mgar
