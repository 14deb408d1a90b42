// Band attention on the 5th-generation tensor cores ("Hierarchical frequency-domain attention":
// strided block-sparse attention on the mid band, sliding-window attention on the high band, and
// dense attention on the pooled low band when that is at least a tile long), bf16 operands, fp32
// accumulation, head_dim 128 or 64 (template parameter HD).
//
// One persistent launch runs both branches from a worklist of (head, band, pair of query tiles)
// items that is rebuilt whenever the head-to-band allocation is (ff_worklist.cuh).  A CTA owns every
// gridDim-th item.  An item is two neighbouring 128-row query tiles ("streams" A and B) that walk
// one sequence of 128-key tiles together: both streams of a mid-band item see every key tile of
// their residue class; in the high band the union of the two windows is 2 + 2R/128 key tiles of
// which each stream takes part in 1 + 2R/128.  K and V tiles are therefore fetched once for two
// query tiles, and while the softmax warps of one stream work the tensor core runs the other's MMAs.
//   warp 0       TMA producer: the two Q tiles, K and V tiles (two stages each)
//   warp 1       tcgen05.mma issuer: S_x = Q_x K^T (operands from shared memory), O_x += P_x V
//                (A = P from tensor memory, B = V as an MN-major operand), issue order
//                PV_A[j], QK_A[j+1], PV_B[j], QK_B[j+1]; owns the tensor-memory allocation
//   warps 4..11  softmax: per stream one thread per query row (row = TMEM lane); the row's 128 scores are read into
//                registers once, key masks are generated from the row's band rank, P is written back to tensor memory
//                as bf16 over the scores; O accumulates in tensor memory and is rescaled only when a row maximum grows
//                by > 2^8.  The registers of the first warpgroup (104 are left of 168 a thread) go to these two
//                (200): 128 x 104 + 256 x 200 = 384 x 168.  With two threads a row, a shared-memory hand-shake for the
//                maximum and a second read of the scores the launch took 1.37 instead of 1.17 ms (64K tokens, 24 heads,
//                all bands)
// Tensor memory (512 columns): S/P of stream A, S/P of stream B, O of stream A, O of stream B.
// Every wait is bounded; when one runs out the CTA raises FF_ERR_TIMEOUT in the plan's status
// word, stops taking work, lets its copies drain, frees its tensor memory and returns.
#include <cuda.h>

#include "ff_clocks.cuh"
#include "ff_internal.h"
#include "ff_sm100.cuh"
#include "ff_worklist.cuh"

using namespace sm100;

namespace {

constexpr int TILE = FF_TILE;        // query rows per stream = key rows per tile
constexpr int HD_MAX = 128;          // largest head_dim; the shared-memory slots are sized for it
constexpr int TILE_BYTES = TILE * HD_MAX * 2;
constexpr int HALF_BYTES = TILE_BYTES / 2;
constexpr int MAX_UNITS = FF_MAX_UNITS;
constexpr int TC_THREADS = 128 + 2 * 128;            // warpgroups: TMA and MMA warp (and two idle ones), softmax of streams A and B
constexpr float LAZY_LOG2 = 8.0f;    // rescale O only when the running max grows by more than this (log2 units)

struct TcParams {
  FFDims dm;
  const uint8_t* alloc;
  int* work;          // the worklist (ff_worklist.cuh)
  __nv_bfloat16* y_mid;
  __nv_bfloat16* y_high;
  float* y_low;       // [BH][Nbar][d] fp32, written when low_on
  int low_on;         // heads whose mask has the low band run it here (band code 0: dense over Nbar pooled tokens)
  int* status;
  int rb_mid;         // rows per TMA box of the mid map = min(b, 128)
};

// (ff_high_attention_noalloc only; the plan's worklist is built where its allocation is decided)
__global__ void build_worklist_kernel(TcParams P) { build_worklist(P.dm, P.alloc, 0, 0, P.work); }

struct Item {
  int band, bh, c;
  int tile_a;         // query tile of stream A; stream B takes tile_a + 1
  int has_b;          // stream B exists
  int nk;             // key tiles of the item
  long long n;        // band length
  long long ks;       // high: first key rank of key tile 0
  int lo[2], hi[2];   // key tiles lo .. hi that streams A and B take part in
};

struct Shared {
  uint64_t q_full, q_empty, k_full[2], k_empty[2], v_full[2], v_empty[2];
  uint64_t s_full[2], p_half[2], p_full[2], o_full[2], o_empty[2];      // per stream
  uint32_t tmem_base;
  int abort_flag;
  int n_units, total;
  MidShape ms;        // kept here rather than in every thread's registers
  int offsets[MAX_UNITS + 1];
  int desc[MAX_UNITS];
  int ntile[MAX_UNITS];
};

template <bool HAS_LOW>
__device__ __forceinline__ Item decode_item(const Shared& sh, const FFDims& dm, int it) {
  const MidShape& ms = sh.ms;
  int lo = 0, hi = sh.n_units - 1;
  while (lo < hi) {                       // last unit whose offset <= it
    const int mid = (lo + hi + 1) >> 1;
    if (sh.offsets[mid] <= it) lo = mid; else hi = mid - 1;
  }
  Item x;
  const int dsc = sh.desc[lo];
  x.bh = dsc >> 12; x.band = (dsc >> 10) & 3; x.c = 0;
  const int local = it - sh.offsets[lo];
  if (x.band == 1) {
    int pr, nt;
    if (local < ms.rem * ms.pairs_big) { x.c = local / ms.pairs_big; pr = local % ms.pairs_big; nt = ms.nt_big; }
    else {
      const int l2 = local - ms.rem * ms.pairs_big;
      x.c = ms.rem + l2 / ms.pairs_small; pr = l2 % ms.pairs_small; nt = ms.nt_small;
    }
    x.tile_a = 2 * pr;
    x.has_b = x.tile_a + 1 < nt;
    x.n = dm.Nmid;
    x.nk = nt;                            // every query tile of a class sees all its key tiles
    x.ks = 0;
  } else if (HAS_LOW && x.band == 0) {
    x.tile_a = 2 * local;
    x.has_b = x.tile_a + 1 < sh.ntile[lo];
    x.n = dm.Nbar;
    x.nk = sh.ntile[lo];                  // dense: every query tile sees every key tile
    x.ks = 0;
  } else {
    x.tile_a = 2 * local;
    x.has_b = x.tile_a + 1 < sh.ntile[lo];
    x.n = dm.Nhigh;
    const long long q0 = (long long)x.tile_a * TILE;
    x.ks = q0 - dm.R > 0 ? q0 - dm.R : 0;
    long long ke = q0 + (x.has_b ? 2 : 1) * TILE + dm.R;
    if (ke > x.n) ke = x.n;
    x.nk = (int)((ke - x.ks + TILE - 1) / TILE);
  }
  // Mid and low band: every tile.  High band: the tiles that meet the window of the stream's 128 query rows.
#pragma unroll
  for (int sx = 0; sx < 2; ++sx) {
    x.lo[sx] = 0; x.hi[sx] = x.nk - 1;
    if (x.band == 2) {
      const long long q0 = (long long)(x.tile_a + sx) * TILE, q1 = q0 + TILE - 1 + dm.R < x.n - 1 ? q0 + TILE - 1 + dm.R : x.n - 1;
      const long long first = q0 - dm.R - x.ks;             // (tile 0 holds it or what is left of it)
      x.lo[sx] = first > 0 ? (int)(first / TILE) : 0;
      x.hi[sx] = (int)((q1 - x.ks) / TILE);
    }
    if (sx == 1 && !x.has_b) { x.lo[1] = 1; x.hi[1] = 0; }
  }
  return x;
}

__device__ __forceinline__ bool stream_active(const Item& x, int sx, int j) { return j >= x.lo[sx] && j <= x.hi[sx]; }

// Band rank of class-local position u of residue class c (mid band).
// (32-bit arithmetic: positions and ranks stay below 2^32 for every supported size.)
__device__ __forceinline__ long long mid_rank(const FFDims& dm, int c, long long u) {
  const unsigned uu = (unsigned)u, b = (unsigned)dm.b;
  const unsigned blk = uu / b;
  return (long long)(((unsigned)c + blk * (unsigned)dm.s) * b + (uu - blk * b));
}

// Issues the TMA loads of one 128-row tile (two 64-column halves) into `dst`; the caller has
// already announced the bytes on `bar`.  `first` = class-local position (mid) or band rank (high).
// `halves` = head_dim / 64.
__device__ __forceinline__ void load_tile(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, const FFDims& dm,
                                          const Item& x, int slice, long long first, int rb, int halves, int* status) {
  // (debug build) a tile starts inside its band (rows past the end are zero-filled by the copy); the bytes were
  // announced on `bar` already, so a refused copy ends in the bounded wait of its consumer, not in a fault
  if (!FF_DBG_OK(first >= 0 && first < x.n + TILE && slice >= 0, status, 1)) return;
  if (x.band != 1) {
    tma_load_3d(dst, map, bar, 0, (int)first, slice);
    if (halves > 1) tma_load_3d(dst + HALF_BYTES, map, bar, 64, (int)first, slice);
  } else {
    for (int i = 0; i < TILE / rb; ++i) {
      const long long row = mid_rank(dm, x.c, first + (long long)i * rb);
      // a block past the end of the band starts beyond the tensor: the copy fills zeros
      const int y = row < dm.Nmid ? (int)row : (int)dm.Nmid;
      tma_load_3d(dst + i * rb * 128, map, bar, 0, y, slice);
      if (halves > 1) tma_load_3d(dst + HALF_BYTES + i * rb * 128, map, bar, 64, y, slice);
    }
  }
}

// The kernel body.  QKV_MAPS = false: map_a / map_b cover the plan's mid / high coefficient buffers,
// which hold Q~, K~ and V~ of head bh in slices bh, BH + bh and 2 BH + bh.  QKV_MAPS = true (the entry
// point that allocates nothing): map_a, map_b, map_c are the caller's separate Q, K, V tensors of one
// band, head bh in slice bh.
// HAS_LOW: the worklist may hold low-band items (band code 0).
template <int HD, bool QKV_MAPS, bool HAS_LOW>
__device__ __forceinline__ void attention_tc_body(const CUtensorMap& map_a, const CUtensorMap& map_b,
                                                  const CUtensorMap& map_c, const TcParams& P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;                       // stream A, stream B: 2 x 32 KB
  uint8_t* sK = smem + 2 * TILE_BYTES;      // 2 stages x 32 KB
  uint8_t* sV = smem + 4 * TILE_BYTES;      // 2 stages x 32 KB
  Shared& sh = *(Shared*)(smem + 6 * TILE_BYTES);
  const FFDims& dm = P.dm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int HALVES = HD / 64;                  // 64-channel halves of a row
  constexpr int TB = TILE * HD * 2;                // bytes of one tile

  if (threadIdx.x == 0) {
    mbar_init(&sh.q_full, 1); mbar_init(&sh.q_empty, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.k_full[i], 1); mbar_init(&sh.k_empty[i], 1);
      mbar_init(&sh.v_full[i], 1); mbar_init(&sh.v_empty[i], 1);
      mbar_init(&sh.s_full[i], 1); mbar_init(&sh.p_half[i], 128); mbar_init(&sh.p_full[i], 128);
      mbar_init(&sh.o_full[i], 1); mbar_init(&sh.o_empty[i], 128);
    }
    sh.abort_flag = 0;
    sh.ms = mid_shape(dm);
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
  ff_pdl_join();
  if (threadIdx.x == 0) { sh.n_units = P.work[0]; sh.total = P.work[1]; }
  __syncthreads();
  for (int i = threadIdx.x; i <= sh.n_units; i += TC_THREADS) {
    sh.offsets[i] = P.work[2 + i];
    if (i < sh.n_units) {
      sh.desc[i] = P.work[2 + MAX_UNITS + 1 + i];
      sh.ntile[i] = P.work[2 + MAX_UNITS + 1 + MAX_UNITS + i];
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sh.tmem_base;
  const int total = sh.total;
  volatile int* abort_flag = &sh.abort_flag;

  if (warp < 4) {
  reg_dec<104>();
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&map_a); tma_prefetch_desc(&map_b); tma_prefetch_desc(&map_c);
      int iter = 0; unsigned g = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < total && ok; it += gridDim.x, ++iter) {
        const Item x = decode_item<HAS_LOW>(sh, dm, it);
        const CUtensorMap* map = x.band == 1 ? &map_a : (!HAS_LOW || x.band == 2 || QKV_MAPS ? &map_b : &map_c);
        const CUtensorMap* mapq = QKV_MAPS ? &map_a : map;
        const CUtensorMap* mapk = QKV_MAPS ? &map_b : map;
        const CUtensorMap* mapv = QKV_MAPS ? &map_c : map;
        const int slice_k = QKV_MAPS ? x.bh : dm.BH + x.bh, slice_v = QKV_MAPS ? x.bh : 2 * dm.BH + x.bh;
        const int rb = x.band == 1 ? P.rb_mid : TILE;
        if (iter >= 1) ok = mbar_wait(&sh.q_empty, (iter - 1) & 1, abort_flag);
        if (!ok) break;
        mbar_arrive_expect_tx(&sh.q_full, x.has_b ? 2 * TB : TB);
        load_tile(sQ, mapq, &sh.q_full, dm, x, x.bh, (long long)x.tile_a * TILE, rb, HALVES, P.status);
        if (x.has_b) load_tile(sQ + TILE_BYTES, mapq, &sh.q_full, dm, x, x.bh, (long long)(x.tile_a + 1) * TILE, rb, HALVES, P.status);
        for (int j = 0; j < x.nk && ok; ++j, ++g) {
          const int st = g & 1;
          const long long first = x.band == 2 ? x.ks + (long long)j * TILE : (long long)j * TILE;
          if (g >= 2) ok = mbar_wait(&sh.k_empty[st], ((g >> 1) - 1) & 1, abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(&sh.k_full[st], TB);
          load_tile(sK + st * TILE_BYTES, mapk, &sh.k_full[st], dm, x, slice_k, first, rb, HALVES, P.status);
          if (g >= 2) ok = mbar_wait(&sh.v_empty[st], ((g >> 1) - 1) & 1, abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(&sh.v_full[st], TB);
          load_tile(sV + st * TILE_BYTES, mapv, &sh.v_full[st], dm, x, slice_v, first, rb, HALVES, P.status);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    {
      const uint32_t idesc_qk = idesc_bf16_f32(TILE, TILE, false, false);
      const uint32_t idesc_pv = idesc_bf16_f32(TILE, HD, false, true);
      int iter = 0; unsigned g = 0;
      unsigned cp[2] = {0, 0};          // P phases consumed per stream
      unsigned ce[2] = {0, 0};          // items seen per stream (for the O buffer hand-back)
      bool ok = true;
      // Operand descriptors of the first slots, once: an instruction then takes an add each (a step inside a slot or a
      // slot is a constant in the address field).  Assembled anew for every instruction they made the issuing
      // thread the limit, 135 cycles an instruction where the tensor core takes 64.
      const uint64_t q_desc = smem_desc_sw128(smem_u32(sQ), 16, 1024), k_desc = smem_desc_sw128(smem_u32(sK), 16, 1024);
      const uint64_t v_desc = smem_desc_sw128(smem_u32(sV), HALF_BYTES, 1024);
      // S_x = Q_x K[tile]^T; `last` = no further QK uses this K stage
      auto issue_qk = [&](int sx, unsigned gt, bool last, bool release_q) {
        const int st = gt & 1;
        const uint64_t qd = q_desc + (uint64_t)(sx * (TILE_BYTES >> 4)), kd = k_desc + (uint64_t)(st * (TILE_BYTES >> 4));
        const uint32_t d_tm = tm + sx * 128;
        FF_CLOCK(c_qk);
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint64_t off = (uint64_t)(((k >> 2) * HALF_BYTES + (k & 3) * 32) >> 4);
          umma_ss(d_tm, qd + off, kd + off, idesc_qk, k > 0 ? 1u : 0u);
        }
        umma_commit(&sh.s_full[sx]);
        FF_CLOCK_ADD(lane == 0, 0, c_qk);
        if (last) umma_commit(&sh.k_empty[st]);
        if (release_q) umma_commit(&sh.q_empty);
      };
      // O_x (+)= P_x V[tile]: the first 64 keys while the softmax works on the others
      auto issue_pv = [&](int sx, unsigned gt, bool first_of_item, bool last, bool last_of_item) -> bool {
        const int st = gt & 1;
        FF_CLOCK(c_half);
        if (!mbar_wait_warp(&sh.p_half[sx], cp[sx] & 1, abort_flag)) return false;
        FF_CLOCK_ADD(lane == 0, 2, c_half);
        if (first_of_item && ce[sx] >= 1 && !mbar_wait_warp(&sh.o_empty[sx], (ce[sx] - 1) & 1, abort_flag)) return false;
        tc_fence_after();
        const uint64_t vd = v_desc + (uint64_t)(st * (TILE_BYTES >> 4));
        const uint32_t p_tm = tm + sx * 128, d_tm = p_tm + 256, first = first_of_item ? 0u : 1u;
        FF_CLOCK(c_pv);                                    // (with the wait for the second half)
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (k == 4) {
            FF_CLOCK(c_full);
            if (!mbar_wait_warp(&sh.p_full[sx], cp[sx] & 1, abort_flag)) return false;
            FF_CLOCK_ADD(lane == 0, 3, c_full);
            ++cp[sx];
            tc_fence_after();
          }
          umma_ts(d_tm, p_tm + k * 8,                      // (P of keys 16 k .. 16 k + 15: eight columns)
                  vd + (uint64_t)(k * (2048 >> 4)), idesc_pv, k == 0 ? first : 1u);
        }
        if (last_of_item) umma_commit(&sh.o_full[sx]);
        if (last) umma_commit(&sh.v_empty[st]);
        FF_CLOCK_ADD(lane == 0, 1, c_pv);
        return true;
      };
      for (int it = blockIdx.x; it < total && ok; it += gridDim.x, ++iter) {
        const Item x = decode_item<HAS_LOW>(sh, dm, it);
        ok = mbar_wait_warp(&sh.q_full, iter & 1, abort_flag);
        if (!ok) break;
        const unsigned g0 = g;
        bool started[2] = {false, false};
        // key tile 0: QK of both streams
        ok = mbar_wait_warp(&sh.k_full[g0 & 1], (g0 >> 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        {
          const bool a0 = stream_active(x, 0, 0), b0 = stream_active(x, 1, 0);
          if (a0) issue_qk(0, g0, !b0, x.nk == 1 && !b0);
          if (b0) issue_qk(1, g0, true, x.nk == 1);
        }
        for (int j = 0; j < x.nk && ok; ++j) {
          FF_CLOCK(c_tile);
          const unsigned gt = g0 + j;
          const bool aj = stream_active(x, 0, j), bj = stream_active(x, 1, j);
          const bool more = j + 1 < x.nk;
          const bool an = more && stream_active(x, 0, j + 1), bn = more && stream_active(x, 1, j + 1);
          bool v_ready = false, k_ready = false;
#pragma unroll
          for (int sx = 0; sx < 2; ++sx) {
            if (!ok) break;
            const bool act = sx ? bj : aj, nxt = sx ? bn : an;
            if (act) {
              if (!v_ready) { ok = mbar_wait_warp(&sh.v_full[gt & 1], (gt >> 1) & 1, abort_flag); v_ready = true; if (!ok) break; }
              const bool last_pv = sx == 1 || !bj;
              ok = issue_pv(sx, gt, !started[sx], last_pv, !nxt);
              started[sx] = true;
              if (!ok) break;
            }
            if (nxt) {
              if (!k_ready) { ok = mbar_wait_warp(&sh.k_full[(gt + 1) & 1], ((gt + 1) >> 1) & 1, abort_flag); k_ready = true; if (!ok) break; tc_fence_after(); }
              const bool last_qk = sx == 1 || !bn;
              issue_qk(sx, gt + 1, last_qk, last_qk && j + 2 == x.nk);
            }
          }
          FF_CLOCK_ADD(lane == 0, 4, c_tile);
        }
        g = g0 + x.nk;
        ce[0] += 1;
        if (x.has_b) ce[1] += 1;
      }
    }
  }
  } else {
    reg_inc<200>();
    // ------------------------------------------------------------------ softmax
    // Warps 4..7 serve stream A, 8..11 stream B (a warp reaches the TMEM lanes 32*(warp%4)..+31).
    const int quarter = warp & 3;
    const int sx = (warp - 4) >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const uint32_t s_addr = tm + lane_addr + sx * 128;
    const uint32_t o_addr = tm + lane_addr + 256 + sx * 128;
    const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;
    unsigned cs = 0;                  // key tiles this stream has processed (phases of s_full / p_full)
    unsigned co = 0;                  // phases of o_full consumed: one per item
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      const Item x = decode_item<HAS_LOW>(sh, dm, it);
      if (sx == 1 && !x.has_b) continue;
      const int tile = x.tile_a + sx;
      // band rank of this thread's query row
      const long long u_q = (long long)tile * TILE + row;
      const long long p = x.band == 1 ? mid_rank(dm, x.c, u_q) : u_q;
      float m_ref = -1e30f, l = 0.f;
      bool first = true;
      const int j_lo = sx ? x.lo[1] : x.lo[0], j_hi = sx ? x.hi[1] : x.hi[0];
      for (int j = j_lo; j <= j_hi && ok; ++j) {
        // valid key columns [clo, chi] of this row in this tile
        int clo = 0, chi = TILE - 1;
        bool full;
        if (x.band == 1) {
          const long long u0 = (long long)j * TILE;
          // ranks grow with the class-local position, so the valid keys are a prefix; a class is a whole number
          // of blocks and blocks tile the 128 rows, so only its last tile can hold keys past the band end
          full = j + 1 < x.nk || mid_rank(dm, x.c, u0 + TILE - 1) < dm.Nmid;
          if (!full) {
            chi = -1;
            for (int cc = TILE - 1; cc >= 0; --cc)
              if (mid_rank(dm, x.c, u0 + cc) < dm.Nmid) { chi = cc; break; }
          }
        } else if (HAS_LOW && x.band == 0) {
          const long long left = x.n - (long long)j * TILE;     // pooled tokens from this tile on
          full = left >= TILE;
          if (!full) chi = (int)left - 1;
        } else {
          const long long t0 = x.ks + (long long)j * TILE;
          const long long q0 = (long long)tile * TILE;
          full = (t0 >= q0 + TILE - 1 - dm.R) && (t0 + TILE - 1 <= q0 + dm.R) && (t0 + TILE <= x.n);
          if (!full) {
            const long long lo = p - dm.R - t0, hi = (p + dm.R < x.n - 1 ? p + dm.R : x.n - 1) - t0;
            clo = lo > 0 ? (int)(lo < TILE ? lo : TILE) : 0;
            chi = hi < TILE - 1 ? (int)(hi < -1 ? -1 : hi) : TILE - 1;
          }
        }
        FF_CLOCK(c_wait);
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.s_full[sx], cs & 1, abort_flag));
        if (!ok) break;
        FF_CLOCK_ADD((threadIdx.x & 127) == 0, 8, c_wait);
        FF_CLOCK(c_max);
        tc_fence_after();
        // the row's scores, and their maximum in four chains
        uint32_t r[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + c * 32, r[c]);
        tmem_wait_ld();
        if (!full) {
          // (edge tiles) columns outside [clo, chi] count as -inf
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int a = clo - c * 32, b = chi - c * 32;                        // valid bits [a, b] of the chunk
            const uint32_t lo_m = a <= 0 ? 0xffffffffu : (a >= 32 ? 0u : 0xffffffffu << a);
            const uint32_t hi_m = b >= 31 ? 0xffffffffu : (b < 0 ? 0u : 0xffffffffu >> (31 - b));
            const uint32_t valid = lo_m & hi_m;
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (!(valid & (1u << i))) r[c][i] = 0xff800000u;
          }
        }
        float t4[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) t4[c] = fmaxf(__uint_as_float(r[c][0]), __uint_as_float(r[c][1]));
#pragma unroll
        for (int i = 2; i < 32; i += 2)
#pragma unroll
          for (int c = 0; c < 4; ++c) t4[c] = max3f(t4[c], __uint_as_float(r[c][i]), __uint_as_float(r[c][i + 1]));
        const float tmax = fmaxf(max3f(t4[0], t4[1], t4[2]), t4[3]);
        const float m_new = fmaxf(m_ref, tmax);
        const bool need = (m_new - m_ref) * sl2 > LAZY_LOG2;
        const float alpha = need ? ex2((m_ref - m_new) * sl2) : 1.f;
        FF_CLOCK_ADD((threadIdx.x & 127) == 0, 9, c_max);
        FF_CLOCK(c_scale);
        // The previous PV of this stream has completed: the scores of this tile, which s_full announces, were issued
        // behind it by the same thread.  So O may be rescaled in place.
        if (!first && __any_sync(0xffffffffu, need)) {
#pragma unroll
          for (int c = 0; c < HD / 16; ++c) {               // (16 columns at a time: the scores stay in registers)
            uint32_t v[16];
            tmem_ld16(o_addr + c * 16, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
            tmem_st16(o_addr + c * 16, v);
          }
          tmem_wait_st();
        }
        if (need) { l *= alpha; m_ref = m_new; }
        FF_CLOCK_ADD((threadIdx.x & 127) == 0, 10, c_scale);
        FF_CLOCK(c_exp);
        // P = 2^(s*scale*log2e - m) as bf16 over the scores, partial row sum
        const float mb = m_ref * sl2;
        float2 sum2 = make_float2(0.f, 0.f);              // (two scores per FMA / add: packed fp32 instructions)
        const float2 sl22 = make_float2(sl2, sl2), nmb2 = make_float2(-mb, -mb);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t pk[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float2 arg = __ffma2_rn(make_float2(__uint_as_float(r[c][2 * i]), __uint_as_float(r[c][2 * i + 1])), sl22, nmb2);
            const float2 pp = make_float2(ex2(arg.x), ex2(arg.y));
            sum2 = __fadd2_rn(sum2, pp);
            const __nv_bfloat162 v = __floats2bfloat162_rn(pp.x, pp.y);
            pk[i] = *(const uint32_t*)&v;
          }
          tmem_st16(s_addr + c * 16, pk);
          if (c & 1) {                                    // 64 keys are there
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(c == 1 ? &sh.p_half[sx] : &sh.p_full[sx]);
          }
        }
        FF_CLOCK_ADD((threadIdx.x & 127) == 0, 11, c_exp);
        l += sum2.x + sum2.y;
        first = false;
        ++cs;
      }
      if (!ok) break;
      // epilogue: O / l -> Y, once the item's last PV has landed
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.o_full[sx], co & 1, abort_flag));
      ++co;
      if (!ok) break;
      tc_fence_after();
      const float inv = 1.f / l;
      const bool store = p < x.n && FF_DBG_OK(p >= 0 && x.bh >= 0 && x.bh < dm.BH, P.status, 1);
      __nv_bfloat16* y = (x.band == 1 ? P.y_mid : P.y_high) + ((size_t)x.bh * x.n + (store ? p : 0)) * HD;
      float* yl = HAS_LOW && x.band == 0 ? P.y_low + ((size_t)x.bh * x.n + (store ? p : 0)) * HD : nullptr;   // low band: fp32
#pragma unroll
      for (int c = 0; c < HD / 32; ++c) {
        uint32_t r[32];
        tmem_ld32(o_addr + c * 32, r);
        tmem_wait_ld();
        if (store && yl) {
#pragma unroll
          for (int v4 = 0; v4 < 8; ++v4)
            *(float4*)(yl + c * 32 + v4 * 4) = make_float4(__uint_as_float(r[v4 * 4]) * inv, __uint_as_float(r[v4 * 4 + 1]) * inv,
                                                           __uint_as_float(r[v4 * 4 + 2]) * inv, __uint_as_float(r[v4 * 4 + 3]) * inv);
        } else if (store) {
#pragma unroll
          for (int v4 = 0; v4 < 4; ++v4) {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(r[v4 * 8 + 2 * i]) * inv,
                                                             __uint_as_float(r[v4 * 8 + 2 * i + 1]) * inv);
              w[i] = *(const uint32_t*)&v;
            }
            *(uint4*)(y + c * 32 + v4 * 8) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      }
      tc_fence_before();
      mbar_arrive(&sh.o_empty[sx]);
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (sh.abort_flag) {
    if (threadIdx.x == 0) atomicExch(P.status, FF_ERR_TIMEOUT | 0x100);   // low byte: status, next byte: which kernel
    // let copies that were already issued land before the shared memory is released
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

template <int HD, bool HAS_LOW>
__global__ void __launch_bounds__(TC_THREADS, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap map_mid, const __grid_constant__ CUtensorMap map_high,
                    const __grid_constant__ CUtensorMap map_low,
                    const TcParams P) {
  attention_tc_body<HD, false, HAS_LOW>(map_mid, map_high, map_low, P);
}

// Same kernel on the caller's separate Q, K, V tensors of one band (see ff_high_attention_noalloc).
__global__ void __launch_bounds__(TC_THREADS, 1)
attention_tc_qkv_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                        const __grid_constant__ CUtensorMap map_v, const TcParams P) {
  attention_tc_body<HD_MAX, true, false>(map_q, map_k, map_v, P);
}

// Scratch of ff_high_attention_noalloc: the worklist, one band mask per head and a status word.
// 13,824 bytes in every GPU context that loads this library, held until the process exits.
constexpr int NOALLOC_MAX_HEADS = MAX_UNITS;
constexpr size_t NOALLOC_WORK_BYTES = (FF_WORK_INTS * sizeof(int) + 255) / 256 * 256;
constexpr size_t NOALLOC_BYTES = NOALLOC_WORK_BYTES + NOALLOC_MAX_HEADS + 256;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

bool encode_band_map(CUtensorMap* map, void* base, long long rows, int slices, int box_rows, int hd = HD_MAX) {
  cuuint64_t dims[3] = {(cuuint64_t)hd, (cuuint64_t)rows, (cuuint64_t)slices};
  cuuint64_t strides[2] = {(cuuint64_t)hd * 2, (cuuint64_t)rows * hd * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

}  // namespace

// The tensor-core kernel covers bf16, head_dim 128 or 64 and block sizes that tile 128 rows evenly.
bool ffk_tc_supported(const FFDims& dm) {
  if (dm.fp32 || (dm.d != 128 && dm.d != 64)) return false;
  const bool b_ok = (dm.b <= TILE) ? (dm.b >= 8 && TILE % dm.b == 0) : (dm.b % TILE == 0);
  if (!b_ok) return false;
  if ((long long)dm.BH * 2 > MAX_UNITS || dm.BH >= (1 << 19)) return false;
  if ((long long)dm.BH * (mid_shape(dm).items + (dm.Nhigh + 2 * TILE - 1) / (2 * TILE)) >= (1LL << 31)) return false;
  if (dm.Nmid >= (1LL << 31) - 256 || dm.Nhigh >= (1LL << 31) - 256) return false;
  return true;
}

cudaError_t ffk_attention_tc_init() {
  cudaError_t e = cudaSuccess;
#define FF_ATT(D, LOW) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(attention_tc_kernel<D, LOW>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                                 (int)(6 * TILE_BYTES + sizeof(Shared) + 1024))
  FF_ATT(128, true); FF_ATT(128, false); FF_ATT(64, true); FF_ATT(64, false);
#undef FF_ATT
  return e;
}

bool ffk_tc_prepare(ff_plan* p) {
  static_assert(sizeof(CUtensorMap) <= sizeof(p->tmap_mid), "tensor map storage too small");
  const FFDims& dm = p->dm;
  const int rb = dm.b < TILE ? dm.b : TILE;
  // (an empty mid band has no items; its map is encoded over one row of the high band's buffer and never used)
  if (!encode_band_map((CUtensorMap*)p->tmap_mid, dm.Nmid > 0 ? p->buf.spec_mid : p->buf.spec_high, dm.Nmid > 0 ? dm.Nmid : 1,
                       3 * dm.BH, dm.Nmid > 0 ? rb : 1, dm.d) ||
      !encode_band_map((CUtensorMap*)p->tmap_high, p->buf.spec_high, dm.Nhigh, 3 * dm.BH, TILE, dm.d))
    return false;
  // The low branch joins this launch when the pooled band is at least one tile long (shorter ones are attended in fp32 by
  // the summary launch, or by the generic kernel where there are no summaries).
  p->low_tc_ok = p->buf.pooled_bf && dm.Nbar >= TILE && dm.Nbar < (1LL << 31) - 256 && (long long)dm.BH * 3 <= MAX_UNITS &&
                 encode_band_map((CUtensorMap*)p->tmap_low, p->buf.pooled_bf, dm.Nbar, 3 * dm.BH, TILE, dm.d);
  return true;
}

cudaError_t ffk_attention_tc(ff_plan* p, cudaStream_t st) {
  const FFDims& dm = p->dm;
  TcParams P;
  P.dm = dm; P.alloc = p->buf.alloc; P.work = p->buf.work;
  P.y_mid = (__nv_bfloat16*)p->buf.y_mid; P.y_high = (__nv_bfloat16*)p->buf.y_high;
  P.y_low = p->buf.y_low; P.low_on = p->low_tc_ok ? 1 : 0;
  P.status = p->buf.status; P.rb_mid = dm.b < TILE ? dm.b : TILE;
  const size_t smem = 6 * TILE_BYTES + sizeof(Shared) + 1024;
  const CUtensorMap& mm = *(const CUtensorMap*)p->tmap_mid;
  const CUtensorMap& mh = *(const CUtensorMap*)p->tmap_high;
  const CUtensorMap& ml = p->low_tc_ok ? *(const CUtensorMap*)p->tmap_low : mh;
  p->launches += 1;
#define FF_ATT(D, LOW) return ff_launch(attention_tc_kernel<D, LOW>, dim3(p->sm_count), dim3(TC_THREADS), smem, st, mm, mh, ml, P)
  if (dm.d == 128) { if (p->low_tc_ok) FF_ATT(128, true); FF_ATT(128, false); }
  if (p->low_tc_ok) FF_ATT(64, true);
  FF_ATT(64, false);
#undef FF_ATT
}

// ------------------------------------------------------------------------------------------------
// ff_high_attention_noalloc: the high-band operator for callers that cannot allocate.
// ------------------------------------------------------------------------------------------------
#include <mutex>

extern "C" ff_status_t ff_high_attention_noalloc(const void* q, const void* k, const void* v, void* y, int32_t heads,
                                                 int64_t n, int32_t radius, int32_t sync, void* cuda_stream) {
  if (!q || !k || !v || !y) { ff_set_thread_error("ff_high_attention_noalloc: a tensor pointer is NULL"); return FF_ERR_INVALID_ARG; }
  if ((((uintptr_t)q) | ((uintptr_t)k) | ((uintptr_t)v) | ((uintptr_t)y)) & 15) {
    ff_set_thread_error("ff_high_attention_noalloc: tensors must be 16-byte aligned");
    return FF_ERR_INVALID_ARG;
  }
  if (heads < 1 || n < 1 || radius < 0) {
    ff_set_thread_error("ff_high_attention_noalloc: need heads >= 1, n >= 1, radius >= 0");
    return FF_ERR_INVALID_ARG;
  }
  if (heads > NOALLOC_MAX_HEADS || n >= (1LL << 31) - 256) {
    ff_set_thread_error("ff_high_attention_noalloc: the built-in scratch covers at most 1024 heads and 2^31-257 tokens per head");
    return FF_ERR_UNSUPPORTED;
  }
  // the worklist counts items (pairs of 128-row query tiles) of all heads in 32 bits
  if ((long long)heads * ((n + 2 * TILE - 1) / (2 * TILE)) >= (1LL << 31)) {
    ff_set_thread_error("ff_high_attention_noalloc: heads x ceil(n / 256) must stay below 2^31");
    return FF_ERR_UNSUPPORTED;
  }
  // Device address of the scratch array, looked up once per device with that device current: in host
  // code the array's name is only a handle, not an address a kernel could use.
  static std::mutex mu;
  static unsigned char* dev_scratch[64] = {};
  static int sm_counts[64] = {};
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) { ff_set_thread_error("ff_high_attention_noalloc: no usable current device"); return FF_ERR_CUDA; }
  unsigned char* scratch = nullptr;
  int sms = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!dev_scratch[dev]) {
      void* ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_counts[dev], cudaDevAttrMultiProcessorCount, dev);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(attention_tc_qkv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(6 * TILE_BYTES + sizeof(Shared) + 1024));
      if (e != cudaSuccess || !ptr) { ff_set_thread_error(cudaGetErrorString(e)); return FF_ERR_CUDA; }
      dev_scratch[dev] = (unsigned char*)ptr;
    }
    scratch = dev_scratch[dev];
    sms = sm_counts[dev];
  }
  CUtensorMap mq, mk, mv;
  if (!encode_band_map(&mq, const_cast<void*>(q), n, heads, TILE) || !encode_band_map(&mk, const_cast<void*>(k), n, heads, TILE) ||
      !encode_band_map(&mv, const_cast<void*>(v), n, heads, TILE)) {
    ff_set_thread_error("ff_high_attention_noalloc: could not encode the tensor maps");
    return FF_ERR_CUDA;
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  TcParams P{};
  P.dm.B = 1; P.dm.heads = heads; P.dm.BH = heads; P.dm.d = HD_MAX; P.dm.R = radius;
  P.dm.Nhigh = n; P.dm.Nmid = 0; P.dm.nb = 0; P.dm.s = 1; P.dm.b = TILE; P.dm.r = 1;
  P.work = (int*)scratch;
  uint8_t* masks = scratch + NOALLOC_WORK_BYTES;
  P.alloc = masks;
  P.status = (int*)(scratch + NOALLOC_WORK_BYTES + NOALLOC_MAX_HEADS);
  P.y_mid = nullptr; P.y_high = (__nv_bfloat16*)y; P.rb_mid = TILE;
  // The array keeps the previous call's contents: rewrite the masks and clear the status word; the
  // worklist is rebuilt by its kernel.
  e = cudaMemsetAsync(masks, FF_BAND_HIGH, (size_t)heads, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(P.status, 0, sizeof(int), st);
  if (e == cudaSuccess) { build_worklist_kernel<<<1, 32, 0, st>>>(P); e = cudaGetLastError(); }
  if (e == cudaSuccess) {
    attention_tc_qkv_kernel<<<sms, TC_THREADS, 6 * TILE_BYTES + sizeof(Shared) + 1024, st>>>(mq, mk, mv, P);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) { ff_set_thread_error(cudaGetErrorString(e)); return FF_ERR_CUDA; }
  if (sync) {
    int word = 0;
    e = cudaMemcpyAsync(&word, P.status, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { ff_set_thread_error(cudaGetErrorString(e)); return FF_ERR_CUDA; }
    if (word != 0) { ff_set_thread_error("ff_high_attention_noalloc: a bounded device-side wait expired"); return FF_ERR_TIMEOUT; }
  }
  return FF_OK;
}

FF_CLOCKS_READ(attention)
