// Worklist of the tensor-core attention launch: which (head, band) units the allocation executes and how many items
// (pairs of 128-row query tiles) each of them has.
#pragma once
#include "ff_internal.h"

constexpr int FF_TILE = 128;             // query rows per stream = key rows per tile
constexpr int FF_MAX_UNITS = 1024;       // units a worklist holds
constexpr size_t FF_WORK_INTS = 2 + 3 * FF_MAX_UNITS + 1;   // units, items, offsets[MAX + 1], desc[MAX], tiles[MAX]

// The residue classes of the mid band come in two sizes: the first `rem` = nb mod s classes hold
// one block more than the others.  Items of a (head, mid band) unit are numbered class by class.
struct MidShape {
  int rem;              // classes with the larger block count
  int nclass;           // residue classes that exist: min(nb, s)
  int nt_big, nt_small; // query (= key) tiles of a class of either size
  int pairs_big, pairs_small;
  int items;            // items of one head's mid band
};

__host__ __device__ __forceinline__ MidShape mid_shape(const FFDims& dm) {
  MidShape m;
  const long long q = dm.s > 0 ? dm.nb / dm.s : 0;
  m.rem = dm.s > 0 ? (int)(dm.nb % dm.s) : 0;
  m.nclass = (int)(dm.nb < dm.s ? dm.nb : dm.s);
  m.nt_big = (int)(((q + 1) * dm.b + FF_TILE - 1) / FF_TILE);
  m.nt_small = (int)((q * dm.b + FF_TILE - 1) / FF_TILE);
  m.pairs_big = (m.nt_big + 1) / 2;
  m.pairs_small = (m.nt_small + 1) / 2;
  m.items = m.rem * m.pairs_big + (m.nclass - m.rem) * m.pairs_small;
  return m;
}

#if defined(__CUDACC__)
// One unit per (head, band) that the allocation executes, called by a whole warp: the low band's units first (when
// `low_on`), then the mid band's (their items are the long ones), then the high band's.  The units of a band have
// equally many items (`mid_items` of the mid band), so a unit's number and first item follow from a ballot.
__device__ __forceinline__ void build_worklist(const FFDims& dm, const uint8_t* alloc, int low_on, int mid_items, int* work) {
  const int lane = threadIdx.x & 31;
  int* offsets = work + 2;
  int* desc = offsets + FF_MAX_UNITS + 1;
  int* tiles = desc + FF_MAX_UNITS;
  int nu = 0, total = 0;
  for (int band = low_on ? 0 : 1; band < 3; ++band) {
    // (the anchor pattern of the mid band is not a union of dense classes: those heads run on the generic kernel)
    if (band == 1 && dm.pattern != FF_MID_STRIDED) continue;
    const int nt = band == 1 ? 0 : (int)(((band == 0 ? dm.Nbar : dm.Nhigh) + FF_TILE - 1) / FF_TILE);
    const int items = band == 1 ? mid_items : (nt + 1) / 2;
    for (int base = 0; base < dm.BH; base += 32) {
      const int bh = base + lane;
      const bool has = bh < dm.BH && (alloc[bh] & (1 << band));
      const unsigned mask = __ballot_sync(0xffffffffu, has);
      const int before = __popc(mask & ((1u << lane) - 1u));
      if (has && nu + before < FF_MAX_UNITS) {
        offsets[nu + before] = total + before * items;
        desc[nu + before] = (bh << 12) | (band << 10);
        tiles[nu + before] = nt;
      }
      const int n = __popc(mask) < FF_MAX_UNITS - nu ? __popc(mask) : FF_MAX_UNITS - nu;
      nu += n; total += n * items;
    }
  }
  if (lane == 0) { offsets[nu] = total; work[0] = nu; work[1] = total; }
}
#endif
