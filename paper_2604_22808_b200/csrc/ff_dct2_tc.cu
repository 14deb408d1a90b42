// Two axis passes of the separable transform in one launch ("Separable spectral decomposition",
// "Reconstruction"): the w axis and a second axis (h or t, whichever is shorter), with the
// intermediate between them kept in shared memory.  bf16 storage, 32 or 16 channels per work item.
//
// A work item is one plane of the grid (all positions of the two axes at one coordinate of the third
// axis) of one tensor-head, for one chunk of C channels (template parameter).  A CTA owns the item: the plane's
// intermediate (hi/lo bf16, 4 bytes per value) takes 128 KB or less of its shared memory, so planes of up to 1024
// positions go in chunks of 32 channels and planes of up to 2048 in chunks of 16 (32-byte rows).  Two tiles of 16 channels
// are handled like one of 32 (a group): the launch issues as many copies, instructions and stores per byte.
//   phase 1  transforms the plane's w lines (tiles of 128 positions = 128/W lines, fetched by TMA) and
//            scatters each result row, as a hi/lo bf16 pair, into the plane buffer; the rows land in
//            the operand layout of phase 2
//   phase 2  transforms the second axis (tiles of 128/n2 neighbouring w coefficients x all n2
//            positions), straight from the buffer, and stores the result with tensor stores (hi/lo
//            grids, or the caller's tensor)
// Both contractions are D[j][c] = sum_r A[j][r] X[r][c] over tiles of 128 positions x C channels
// with the matrix A = I kron Mat (w lines follow one another) or Mat kron I (lines of the second
// axis interleave) held in TENSOR MEMORY as the A operand (hi and lo bf16 parts, 64 columns each),
// so that a tile costs no shared-memory traffic for the matrix; the data tile is the MN-major B
// operand in place (64- or 32-byte rows, swizzled); up to four groups share one instruction (N = 128: an
// instruction takes the same time for any N up to 128).
//
//   warp 0        TMA producer (ring of 8 groups, or 4 hi/lo pairs)
//   warp 1        tcgen05.mma issuer of phase 1; owns the tensor-memory allocation
//   warp 2        idle
//   warp 3        tcgen05.mma issuer of phase 2
//   warps 4..11   phase-1 epilogue (a thread owns one position of a tile; the first four warps take
//                 the first group of a pair, the next four the second)
//   warps 12..19  phase-2 epilogue
// so that phase 1 of the next item runs while phase 2 of the current one drains.
// Every wait is bounded.
#include <cuda.h>

#include <vector>

#include "ff_clocks.cuh"
#include "ff_internal.h"
#include "ff_sm100.cuh"

using namespace sm100;

namespace {

constexpr int ROWS = 128;                     // positions per tile
// A group is what a ring slot, a TMA box and a step of an epilogue warp take: one tile of 32 channels or two of 16.
constexpr int GCOLS = 32;                     // accumulator columns of a group
constexpr int GROUP_B = ROWS * GCOLS * 2;     // 8 KB as bf16
constexpr int NSTG = 8;                       // input ring: at most 8 groups (64 KB: 8 bf16 groups or 4 hi/lo pairs)
constexpr int RING_B = NSTG * GROUP_B;
constexpr int MAX_GPI = 8;                    // groups of an item (128 KB of hi/lo buffer)
constexpr int D2_THREADS = 640;                 // TMA, MMA 1, idle, MMA 2, 8 phase-1 and 8 phase-2 epilogue warps
constexpr int ACC_GROUPS = 4;                 // groups that fit a phase's 128 accumulator columns: one batch of 4, or 2 of 2
constexpr int IMG_CELLS = 64;                 // 32-bit tensor-memory cells per matrix row: two bf16 K elements each
constexpr int STG_B = 32 * GCOLS * 2;         // bytes an epilogue warp stages at a time (its 32 rows of a group), hi or lo

struct Dct2Params {
  FFDims dm;
  const uint32_t* img1;    // w-axis matrix: hi [128][64] cells, then lo
  const uint32_t* img2;    // second-axis matrix: hi, then lo
  int axis2;               // 1 = h, 0 = t
  int n1, n2, n3;          // W, length of the second axis, length of the remaining axis
  int in_split;            // input is a hi/lo pair of grids (map0 = hi, map1 = lo); otherwise Q, K, V
  int last;                // output is the caller's tensor (bf16, no lo part)
  int group, group_start;
  int nchunk;              // channel chunks: head_dim / 32 or / 16
  int gpi;                 // groups of an item
  int bt1, bt2;            // groups per instruction batch of the two phases: 2 or 4
  double* clear;           // band energies to clear for the sums that follow (first launch of a routed forward), or NULL
  int* status;
};

struct D2Shared {
  uint64_t in_full[NSTG], in_empty[NSTG], acc1_full[2], acc1_empty[2], acc2_full[2], acc2_empty[2];
  // The plane buffer has one slot of 8 groups or two of 4 (items alternate): phase 1 of the next item fills one
  // slot while phase 2 of the current item reads the other.
  uint64_t buf_full[2];    // all rows of the item have landed in the slot
  uint64_t buf_half[2];    // the rows of the first half of the second axis have landed
  uint64_t half_free[2];   // phase 2 has finished reading those rows (its k-steps 0..3 of every batch)
  uint64_t buf_free[2];    // phase 2 of the item has finished reading the slot
  uint32_t tmem_base;
  int abort_flag;
};

// Shared-memory descriptor of an MN-major operand stored as rows of C bf16 (64 or 32 bytes) with the swizzle of that width:
// 8-row groups 8 rows apart (SBO); `lbo` = distance between the chunks of C elements along N.
template <int C>
__device__ __forceinline__ uint64_t smem_desc_rows(uint32_t smem_addr, uint32_t lbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)(8 * C * 2 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)(C == 32 ? 4 : 6) << 61;   // SWIZZLE_64B, SWIZZLE_32B
  return d;
}
// Position of 16-byte piece `i` of row `row` under that swizzle.
template <int C> __device__ __forceinline__ int swizzled(int i, int row) { return C == 32 ? i ^ ((row >> 1) & 3) : i ^ ((row >> 2) & 1); }

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// Item `it` of the launch: chunk fastest (CTAs that run side by side read neighbouring pieces of the same
// rows), then the coordinate of the remaining axis, then the tensor-head.
__device__ __forceinline__ void decode_item(const Dct2Params& P, int it, int& gi, int& a3, int& chunk) {
  chunk = it % P.nchunk;
  const int rest = it / P.nchunk;
  a3 = rest % P.n3;
  gi = rest / P.n3;
}

// fp32 accumulators of a thread's 32 columns -> bf16 hi and lo words (two channels per word)
__device__ __forceinline__ void split_hi_lo(const uint32_t (&r)[32], uint32_t (&hi)[16], uint32_t (&lo)[16], bool want_lo) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const __nv_bfloat162 hp = __floats2bfloat162_rn(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
    hi[i] = *(const uint32_t*)&hp;
  }
  if (want_lo) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const __nv_bfloat162 lp = __floats2bfloat162_rn(__uint_as_float(r[2 * i]) - __uint_as_float(hi[i] << 16),
                                                     __uint_as_float(r[2 * i + 1]) - __uint_as_float(hi[i] & 0xffff0000u));
      lo[i] = *(const uint32_t*)&lp;
    }
  }
}

// map0..map2: sources (Q, K, V; or hi, lo, -).  map_oh / map_ol: destinations (hi / lo grids, or the
// caller's tensor in map_oh), box = what an epilogue warp holds of a group.
template <int C>
__global__ void __launch_bounds__(D2_THREADS, 1)
dct2_tc_kernel(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap map1,
               const __grid_constant__ CUtensorMap map2, const __grid_constant__ CUtensorMap map_oh,
               const __grid_constant__ CUtensorMap map_ol, const Dct2Params P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const FFDims& dm = P.dm;
  constexpr int RT = GCOLS / C;                                    // tiles of a group
  constexpr int TILE_B = ROWS * C * 2;
  constexpr uint32_t KSTEP = 16 * C * 2 >> 4;                      // a descriptor's way to the next 16 rows of K
  const int gpi = P.gpi;
  uint8_t* sBuf = smem;                                            // tiles of the plane, hi and lo of each in turn: its intermediate
  uint8_t* sStage = smem + MAX_GPI * 2 * GROUP_B;                  // 8 phase-2 warps x (hi 2 KB, lo 2 KB), 1024-byte aligned
  uint8_t* sIn = sStage + 8 * 2 * STG_B;                           // ring: 8 groups, or 4 and behind them their lo parts
  D2Shared& sh = *(D2Shared*)(sIn + RING_B);
  const int lslot = P.in_split ? 2 : 3, nslot = 1 << lslot;
  static_assert(NSTG == 8, "ring slots");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n1 = P.n1, n2 = P.n2;
  const int ln1 = 31 - __clz(n1);
  const int kf1 = ROWS / n1, kf2 = ROWS / n2;
  const int lkf2 = 31 - __clz(kf2);
  const int total = P.group * P.n3 * P.nchunk;
  const int nsl = gpi <= MAX_GPI / 2 ? 2 : 1;                      // slots of the plane buffer
  // groups per instruction batch (N = 32 groups columns), batches of an item, and the accumulator buffers: one, or two with
  // batches of two (as logarithms: divisions by launch parameters would stand in front of every wait)
  const int bt1 = P.bt1, nb1 = gpi / bt1, la1 = bt1 <= ACC_GROUPS / 2, m1 = (1 << la1) - 1;
  const int bt2 = P.bt2, nb2 = gpi / bt2, la2 = bt2 <= ACC_GROUPS / 2, m2 = (1 << la2) - 1;
  // With an even number of batches, the first half of the phase-1 batches holds the first half
  // of the second axis, i.e. rows 0..63 of every phase-2 tile = its k-steps 0..3.  Phase 2 of the item's first
  // batch starts on those while phase 1 still works on the second half.
  const bool half_start = nb1 >= 2 && (nb1 & 1) == 0;
  // ... and phase 1 of the next item may overwrite those rows as soon as phase 2 has read them (forward launch:
  // measured slower for the inverse, whose phase 1 issues half as many instructions again)
  const bool half_release = half_start && !P.in_split;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSTG; ++i) { mbar_init(&sh.in_full[i], 1); mbar_init(&sh.in_empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&sh.acc1_full[i], 1); mbar_init(&sh.acc1_empty[i], 256); }
    for (int i = 0; i < 2; ++i) { mbar_init(&sh.acc2_full[i], 1); mbar_init(&sh.acc2_empty[i], 256); }
    for (int i = 0; i < 2; ++i) { mbar_init(&sh.buf_full[i], 8); mbar_init(&sh.buf_free[i], 1); mbar_init(&sh.buf_half[i], 8); }
    mbar_init(&sh.half_free[0], 1); mbar_init(&sh.half_free[1], 1);
    sh.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sh.tmem_base;
  volatile int* abort_flag = &sh.abort_flag;
  // tensor-memory columns: matrix images [0,256): w hi, w lo, second axis hi, lo; phase-1 accumulators
  // (128 columns: one or two batches) from 256; phase-2 accumulators behind them
  constexpr uint32_t COL_A1H = 0, COL_A1L = 64, COL_A2H = 128, COL_A2L = 192, COL_ACC1 = 256, COL_ACC2 = COL_ACC1 + ACC_GROUPS * GCOLS;
  static_assert(COL_ACC2 + ACC_GROUPS * GCOLS <= 512, "tensor memory has 512 columns");

  if (warp >= 4 && warp < 8) {
    // the four matrix images into tensor memory: a thread loads the row of its lane
    const int quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
#pragma unroll 1
    for (int im = 0; im < 4; ++im) {
      const uint32_t* src = (im < 2 ? P.img1 : P.img2) + (size_t)(im & 1) * FF_IMAGE_PART + (size_t)row * IMG_CELLS;
#pragma unroll
      for (int c0 = 0; c0 < IMG_CELLS; c0 += 32) {
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 v = *(const uint4*)(src + c0 + 4 * i);
          r[4 * i] = v.x; r[4 * i + 1] = v.y; r[4 * i + 2] = v.z; r[4 * i + 3] = v.w;
        }
        tmem_st32(tm + lane_addr + im * 64 + c0, r);
      }
    }
    tmem_wait_st();
  }
  ff_pdl_wait();
  if (P.clear && blockIdx.x == 0) for (int i = threadIdx.x; i < dm.B * 3 * dm.d; i += D2_THREADS) P.clear[i] = 0.0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  const int cid = (int)blockIdx.x, ncta = (int)gridDim.x;
  FF_CLOCK(t_all);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&map0);
      unsigned n = 0;
      bool ok = true;
      for (int it = cid; it < total && ok; it += ncta) {
        int gi, a3, chunk; decode_item(P, it, gi, a3, chunk);
        const CUtensorMap* map = &map0;
        int slice = gi;
        if (!P.in_split) {
          const int th = P.group_start + gi;
          const int tensor = th / dm.BH;
          map = tensor == 0 ? &map0 : (tensor == 1 ? &map1 : &map2);
          slice = th % dm.BH;
        }
        for (int k = 0; k < gpi && ok; ++k, ++n) {
          const int slot = n & (nslot - 1);
          FF_CLOCK(tp0);
          if (n >= (unsigned)nslot) ok = mbar_wait(&sh.in_empty[slot], ((n >> lslot) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 12, tp0);
          if (!ok) break;
          uint8_t* dst = sIn + slot * GROUP_B;
          const int b0 = k * RT * kf1;                             // first line of the group
          const int ch = P.axis2 == 1 ? b0 : a3, ct = P.axis2 == 1 ? a3 : b0;
          mbar_arrive_expect_tx(&sh.in_full[slot], P.in_split ? 2 * GROUP_B : GROUP_B);
          tma_load_5d(dst, map, &sh.in_full[slot], chunk * C, 0, ch, ct, slice);
          if (P.in_split) tma_load_5d(dst + RING_B / 2, &map1, &sh.in_full[slot], chunk * C, 0, ch, ct, slice);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer, phase 1
    // batches of bt1 groups (neighbouring slots of the ring), N = 32 bt1
    {
      const uint32_t idesc = idesc_bf16_f32(ROWS, bt1 * GCOLS, /*a_mn_major=*/false, /*b_mn_major=*/true);
      const uint32_t in_base = smem_u32(sIn);
      unsigned n1b = 0;
      bool ok = true;
      for (int it = cid; it < total && ok; it += ncta) {
        for (int kb = 0; kb < nb1 && ok; ++kb, ++n1b) {
          const int ab = n1b & m1;
          const unsigned nt = bt1 * n1b;                            // index of the batch's first group in the ring sequence
          FF_CLOCK(tm0);
          for (int i = 0; i < bt1 && ok; ++i) ok = mbar_wait_warp(&sh.in_full[(nt + i) & (nslot - 1)], ((nt + i) >> lslot) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 7, tm0);
          FF_CLOCK(tm1);
          if (ok && n1b > (unsigned)m1) ok = mbar_wait_warp(&sh.acc1_empty[ab], ((n1b >> la1) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 8, tm1);
          if (!ok) break;
          tc_fence_after();
          const uint32_t x0 = in_base + (uint32_t)(nt & (nslot - 1)) * GROUP_B;
          const uint64_t xh = smem_desc_rows<C>(x0, TILE_B), xl = smem_desc_rows<C>(x0 + RING_B / 2, TILE_B);
          const uint32_t d_tm = tm + COL_ACC1 + ab * bt1 * GCOLS;
          if (P.in_split) {
#pragma unroll
            for (int ks = 0; ks < ROWS / 16; ++ks) {
              umma_ts(d_tm, tm + COL_A1H + ks * 8, xh + (uint64_t)(ks * KSTEP), idesc, ks > 0 ? 1u : 0u);
              umma_ts(d_tm, tm + COL_A1L + ks * 8, xh + (uint64_t)(ks * KSTEP), idesc, 1u);
              umma_ts(d_tm, tm + COL_A1H + ks * 8, xl + (uint64_t)(ks * KSTEP), idesc, 1u);
            }
          } else {
#pragma unroll
            for (int ks = 0; ks < ROWS / 16; ++ks) {
              umma_ts(d_tm, tm + COL_A1H + ks * 8, xh + (uint64_t)(ks * KSTEP), idesc, ks > 0 ? 1u : 0u);
              umma_ts(d_tm, tm + COL_A1L + ks * 8, xh + (uint64_t)(ks * KSTEP), idesc, 1u);
            }
          }
          for (int i = 0; i < bt1; ++i) umma_commit(&sh.in_empty[(nt + i) & (nslot - 1)]);
          umma_commit(&sh.acc1_full[ab]);
        }
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ MMA issuer, phase 2
    // (a warp of its own: phase 2 of an item waits for all of its phase 1, phase 1 of the next item does not)
    {
      const uint32_t idesc = idesc_bf16_f32(ROWS, bt2 * GCOLS, /*a_mn_major=*/false, /*b_mn_major=*/true);
      const uint32_t buf_base = smem_u32(sBuf);
      unsigned n2b = 0, ni = 0;
      bool ok = true;
      for (int it = cid; it < total && ok; it += ncta, ++ni) {
        // the plane's rows have landed in this CTA's buffer
        FF_CLOCK(tm2);
        const int sl = (int)(ni & (nsl - 1));                             // the item's slot of the plane buffer
        ok = mbar_wait_warp(half_start ? &sh.buf_half[sl] : &sh.buf_full[sl], (ni >> (nsl - 1)) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 9, tm2);
        if (!ok) break;
        fence_proxy_async();
        for (int kb = 0; kb < nb2 && ok; ++kb, ++n2b) {
          const int ab = n2b & m2;
          FF_CLOCK(tm3);
          if (n2b > (unsigned)m2) ok = mbar_wait_warp(&sh.acc2_empty[ab], ((n2b >> la2) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 10, tm3);
          if (!ok) break;
          tc_fence_after();
          const uint32_t x0 = buf_base + (uint32_t)(sl * gpi + bt2 * kb) * 2 * GROUP_B;   // hi, lo of each tile in turn
          const uint64_t xh = smem_desc_rows<C>(x0, 2 * TILE_B), xl = smem_desc_rows<C>(x0 + TILE_B, 2 * TILE_B);
          const uint32_t d_tm = tm + COL_ACC2 + ab * bt2 * GCOLS;
#pragma unroll
          for (int ks = 0; ks < ROWS / 16; ++ks) {
            if (ks == ROWS / 32 && kb == 0 && half_start) {          // the second half of the rows
              FF_CLOCK(tm4);
              ok = mbar_wait_warp(&sh.buf_full[sl], (ni >> (nsl - 1)) & 1, abort_flag);
              FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 11, tm4);
              if (!ok) break;
              fence_proxy_async();
              tc_fence_after();
            }
            umma_ts(d_tm, tm + COL_A2H + ks * 8, xh + (uint64_t)(ks * KSTEP), idesc, ks > 0 ? 1u : 0u);
            umma_ts(d_tm, tm + COL_A2L + ks * 8, xh + (uint64_t)(ks * KSTEP), idesc, 1u);
            umma_ts(d_tm, tm + COL_A2H + ks * 8, xl + (uint64_t)(ks * KSTEP), idesc, 1u);
            // rows 0..63 of every tile have been read once the last batch's k-step 3 is done: phase 1 of the next
            // item may overwrite them
            if (ks == ROWS / 32 - 1 && kb == nb2 - 1 && half_release) umma_commit(&sh.half_free[sl]);
          }
          if (!ok) break;
          umma_commit(&sh.acc2_full[ab]);
        }
        umma_commit(&sh.buf_free[sl]);
      }
    }
  } else if (warp >= 4 && warp < 12) {
    // ------------------------------------------------------------------ phase-1 epilogue
    // accumulators -> hi/lo rows in the plane buffer.  A thread owns row (line l1, w coefficient a1)
    // of every tile of its group and sends it as 16-byte pieces of hi and of lo, straight from registers.
    const int ew = warp - 4;                               // 0..7
    const int half = ew >> 2;                              // which group of a pair
    const int quarter = warp & 3;
    const int j = quarter * 32 + lane;                     // position of this thread inside a tile
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const uint32_t buf_base = smem_u32(sBuf);
    const int l1 = j >> ln1, a1 = j & (n1 - 1);
    const int u2 = a1 >> lkf2;                             // phase-2 tile of the plane that takes coefficient a1
    // Eight neighbouring lanes store at once; their rows are kf2 per tile, and rows of different tiles
    // with the same swizzle would meet in the same banks: the lanes of tile t of the eight start
    // their pieces at piece `rot` instead of 0, which spreads them over the banks.
    constexpr int PIECES = C / 8;                          // 16-byte pieces of a row
    const int rot = (kf2 >= 8 ? 0 : ((lane & 7) >> lkf2) * (C == 32 && kf2 == 4 ? 2 : 1)) & (PIECES - 1);
    unsigned n1b = 0, ni = 0;
    bool ok = true;
    for (int it = cid; it < total && ok; it += ncta, ++ni) {
      FF_CLOCK(te0);
      const int sl = (int)(ni & (nsl - 1));                         // the item's slot: free once phase 2 of item ni - nsl is done
      if (ni >= (unsigned)nsl) {
        // (half_release: the first half of the batches writes rows phase 2 releases earlier; the rest waits below)
        ok = mbar_wait_warp(half_release ? &sh.half_free[sl] : &sh.buf_free[sl], ((ni >> (nsl - 1)) - 1) & 1, abort_flag);
        if (!ok) break;
      }
      FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 1, te0);
      for (int kb = 0; kb < nb1 && ok; ++kb, ++n1b) {
        if (half_release && kb == nb1 / 2 && ni >= (unsigned)nsl) {
          ok = mbar_wait_warp(&sh.buf_free[sl], ((ni >> (nsl - 1)) - 1) & 1, abort_flag);
          if (!ok) break;
        }
        const int ab = n1b & m1;
        FF_CLOCK(te1);
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc1_full[ab], (n1b >> la1) & 1, abort_flag));
        if (!ok) break;
        FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 0, te1);
        FF_CLOCK(te2);
        tc_fence_after();
        for (int tb = half; tb < bt1; tb += 2) {            // this warp's groups of the batch
        uint32_t r[32];
        tmem_ld32(tm + lane_addr + COL_ACC1 + ab * bt1 * GCOLS + tb * 32, r);
        tmem_wait_ld();
        if (tb + 2 >= bt1) {                                // the accumulators are free once the warp's last group is read
          tc_fence_before();
          mbar_arrive(&sh.acc1_empty[ab]);
        }
        uint32_t hi[16], lo[16];
        split_hi_lo(r, hi, lo, true);
        // rotate the pieces by `rot` (conditional swaps), then piece i of the registers is piece (i + rot) % PIECES of the row
        if (C == 16 && rot) {
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (!(q & 4)) {
              const uint32_t h0 = hi[q], l0 = lo[q];
              hi[q] = hi[q + 4]; hi[q + 4] = h0;
              lo[q] = lo[q + 4]; lo[q + 4] = l0;
            }
        }
        if (C == 32 && (rot & 1)) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t h0 = hi[q], l0 = lo[q];
            hi[q] = hi[4 + q]; hi[4 + q] = hi[8 + q]; hi[8 + q] = hi[12 + q]; hi[12 + q] = h0;
            lo[q] = lo[4 + q]; lo[4 + q] = lo[8 + q]; lo[8 + q] = lo[12 + q]; lo[12 + q] = l0;
          }
        }
        if (C == 32 && (rot & 2)) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const uint32_t h0 = hi[q], l0 = lo[q];
            hi[q] = hi[8 + q]; hi[8 + q] = h0;
            lo[q] = lo[8 + q]; lo[8 + q] = l0;
          }
        }
#pragma unroll
        for (int t = 0; t < RT; ++t) {
          // where the row goes: position b of the second axis, row b kf2 + (a1 mod kf2) of tile u2
          const int b = ((bt1 * kb + tb) * RT + t) * kf1 + l1;
          const int drow = (b << lkf2) | (a1 & (kf2 - 1));
          const uint32_t daddr = buf_base + (uint32_t)(sl * gpi * RT + u2) * 2 * TILE_B + (uint32_t)drow * (C * 2);
          // (debug build) the row lies inside a tile of the buffer
          if (!FF_DBG_OK(drow >= 0 && drow < ROWS && u2 >= 0 && u2 < gpi * RT && b < n2, P.status, 4)) continue;
#pragma unroll
          for (int i = 0; i < PIECES; ++i) {
            const uint32_t dst = daddr + (uint32_t)(swizzled<C>((i + rot) & (PIECES - 1), drow) << 4);
            const int w = (t * PIECES + i) * 4;
            st_shared_v4(dst, make_uint4(hi[w], hi[w + 1], hi[w + 2], hi[w + 3]));
            st_shared_v4(dst + TILE_B, make_uint4(lo[w], lo[w + 1], lo[w + 2], lo[w + 3]));
          }
        }
        }
        FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 2, te2);
        if (half_start && kb == nb1 / 2 - 1) {               // this warp's rows of the first half are written
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.buf_half[sl]);
        }
      }
      if (!ok) break;
      // this warp's rows of the item are written
      FF_CLOCK(te4);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.buf_full[sl]);
      FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 6, te4);
    }
  } else if (warp >= 12) {
    // ------------------------------------------------------------------ phase-2 epilogue
    // accumulators -> destination grids.  Rows 32 quarter .. + 31 of the tiles of a group are the box [a2 = a0 .., w ..]
    // of the store map; the warp stages them (w fastest) and one lane issues the tensor stores.
    const int ew = warp - 12;                              // 0..7
    const int half = ew >> 2;
    const int quarter = warp & 3;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    uint8_t* st_hi = sStage + ew * 2 * STG_B;
    uint8_t* st_lo = st_hi + STG_B;
    const int a0 = (quarter * 32) >> lkf2;
    constexpr int PIECES = C / 8;
    const int row0 = (lane >> lkf2) * RT * kf2 + (lane & (kf2 - 1));      // row of the box; kf2 more for the group's second tile
    const bool flip = C == 16 && kf2 == 4 && (lane & 4);   // (rows 8 apart meet in the same banks: these lanes start at piece 1)
    unsigned n2b = 0;
    bool ok = true;
    for (int it = cid; it < total && ok; it += ncta) {
      int gi, a3, chunk; decode_item(P, it, gi, a3, chunk);
      const int out_slice = P.last ? P.group_start + gi : gi;
      for (int kb = 0; kb < nb2 && ok; ++kb, ++n2b) {
        const int ab = n2b & m2;
        FF_CLOCK(te5);
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc2_full[ab], (n2b >> la2) & 1, abort_flag));
        if (!ok) break;
        FF_CLOCK_ADD(threadIdx.x == 384, P.in_split * 16 + 3, te5);
        FF_CLOCK(te6);
        tc_fence_after();
        for (int tb = half; tb < bt2; tb += 2) {            // this warp's groups of the batch
        uint32_t r[32];
        tmem_ld32(tm + lane_addr + COL_ACC2 + ab * bt2 * GCOLS + tb * 32, r);
        tmem_wait_ld();
        if (tb + 2 >= bt2) {
          tc_fence_before();
          mbar_arrive(&sh.acc2_empty[ab]);
        }
        uint32_t hi[16], lo[16];
        split_hi_lo(r, hi, lo, !P.last);
        // the previous tensor store of this warp must have read the staging area
        FF_CLOCK(te7);
        if (lane == 0) bulk_wait_read0();
        __syncwarp();
        FF_CLOCK_ADD(threadIdx.x == 384, P.in_split * 16 + 4, te7);
        if (flip) {
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (!(q & 4)) {
              const uint32_t h0 = hi[q], l1 = lo[q];
              hi[q] = hi[q + 4]; hi[q + 4] = h0;
              lo[q] = lo[q + 4]; lo[q + 4] = l1;
            }
        }
#pragma unroll
        for (int t = 0; t < RT; ++t)
#pragma unroll
          for (int i = 0; i < PIECES; ++i) {
            const int row = row0 + t * kf2, w = (t * PIECES + i) * 4;
            const int so = row * (C * 2) + (swizzled<C>(i ^ (flip ? 1 : 0), row) << 4);
            *(uint4*)(st_hi + so) = make_uint4(hi[w], hi[w + 1], hi[w + 2], hi[w + 3]);
            if (!P.last) *(uint4*)(st_lo + so) = make_uint4(lo[w], lo[w + 1], lo[w + 2], lo[w + 3]);
          }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          const int cw = (bt2 * kb + tb) * RT * kf2;         // first w coefficient of the group
          const int ch = P.axis2 == 1 ? a0 : a3, ct = P.axis2 == 1 ? a3 : a0;
          tma_store_5d(st_hi, &map_oh, chunk * C, cw, ch, ct, out_slice);
          if (!P.last) tma_store_5d(st_lo, &map_ol, chunk * C, cw, ch, ct, out_slice);
          bulk_commit();
        }
        }
        FF_CLOCK_ADD(threadIdx.x == 384, P.in_split * 16 + 5, te6);
      }
    }
    if (lane == 0) bulk_wait0();
  }

  // ------------------------------------------------------------------ teardown
  FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 15, t_all);
  tc_fence_before();
  __syncthreads();
  if (sh.abort_flag) {
    if (threadIdx.x == 0) atomicExch(P.status, FF_ERR_TIMEOUT | 0x400);   // low byte: status, next byte: which kernel
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

// 5-D map over a [slices][T][H][W][d] bf16 grid.  Load box: one group of phase 1, C channels of 32/C tiles of 128/W
// whole w lines that are neighbours along the second axis.
bool encode_in_map(CUtensorMap* map, const void* base, const FFDims& dm, int slices, int axis2, int C) {
  const cuuint64_t CH = (cuuint64_t)dm.d;
  cuuint64_t dims[5] = {CH, (cuuint64_t)dm.W, (cuuint64_t)dm.H, (cuuint64_t)dm.T, (cuuint64_t)slices};
  cuuint64_t strides[4] = {CH * 2, (cuuint64_t)dm.W * CH * 2, (cuuint64_t)dm.H * dm.W * CH * 2, (cuuint64_t)dm.N * CH * 2};
  cuuint32_t box[5] = {(cuuint32_t)C, (cuuint32_t)dm.W, 1, 1, 1};
  box[axis2 == 1 ? 2 : 3] = (cuuint32_t)(ROWS / dm.W * (GCOLS / C));
  return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box,
                       C == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

// Store box: what one epilogue warp holds of a group after phase 2, C channels of tile rows 32 q .. 32 q + 31 of its
// tiles, row of a tile = (position along the second axis) * kf2 + (w coefficient inside the tile).
bool encode_out_map(CUtensorMap* map, const void* base, const FFDims& dm, int slices, int axis2, int C) {
  const cuuint64_t CH = (cuuint64_t)dm.d;
  cuuint64_t dims[5] = {CH, (cuuint64_t)dm.W, (cuuint64_t)dm.H, (cuuint64_t)dm.T, (cuuint64_t)slices};
  cuuint64_t strides[4] = {CH * 2, (cuuint64_t)dm.W * CH * 2, (cuuint64_t)dm.H * dm.W * CH * 2, (cuuint64_t)dm.N * CH * 2};
  const int n2 = axis2 == 1 ? dm.H : dm.T;
  const int kf2 = ROWS / n2;                       // at most 8
  cuuint32_t box[5] = {(cuuint32_t)C, (cuuint32_t)(kf2 * (GCOLS / C)), 1, 1, 1};
  box[axis2 == 1 ? 2 : 3] = (cuuint32_t)(32 / kf2);
  return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box,
                       C == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_NONE);
}

// (the staging areas of the tensor stores sit 1024-byte aligned: their swizzle is a function of the address)
constexpr size_t D2_SMEM = 1024 + (size_t)MAX_GPI * 2 * GROUP_B + (size_t)8 * 2 * STG_B + (size_t)RING_B + sizeof(D2Shared) + 64;

cudaError_t launch(ff_plan* p, const CUtensorMap& m0, const CUtensorMap& m1, const CUtensorMap& m2, const CUtensorMap& moh,
                   const CUtensorMap& mol, Dct2Params& P, cudaStream_t st) {
  P.nchunk = P.dm.d / p->dct2_chunk;
  P.gpi = P.dm.W * P.n2 / ROWS * p->dct2_chunk / GCOLS;
  // Groups per instruction batch.  Four make N = 128, which costs the tensor core the least, and one accumulator buffer; two
  // make N = 64 and two buffers.  The inverse's ring holds four groups as hi/lo pairs: a batch of four waits for the whole
  // ring and empties it, and the latency of the loads stands between two batches, so its phase 1 takes two (stage at
  // 1.6 GHz, 24 heads of 64K tokens 932 -> 868 us, 48 of 128K 3825 -> 3507).  The forward's ring holds two batches of four
  // (two at a time: 1483 -> 1532 us of the 64K transform stage).  Phase 2 with 16 channels is bound by its epilogue's twice as
  // many short rows, which two buffers keep busy (forward, 128K tokens 6763 -> 6415 us; with 32 channels 1477 and 1479).
  const int most = P.gpi < ACC_GROUPS ? P.gpi : ACC_GROUPS;
  P.bt1 = P.in_split ? 2 : most;
  P.bt2 = p->dct2_chunk == 16 ? 2 : most;
  const int items = P.group * P.n3 * P.nchunk;
  const dim3 grid((unsigned)(items < p->sm_count ? items : p->sm_count));
  const cudaError_t e = ff_launch(p->dct2_chunk == 32 ? dct2_tc_kernel<32> : dct2_tc_kernel<16>, grid, dim3(D2_THREADS), D2_SMEM, st,
                                  m0, m1, m2, moh, mol, P);
  if (e != cudaSuccess) return e;
  p->launches += 1;
  return cudaSuccess;
}

// (through the plan's cache)
bool in_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, int axis2) {
  return p->maps.get(map, base, 32 | axis2, slices, [&] { return encode_in_map(map, base, p->dm, slices, axis2, p->dct2_chunk); });
}
bool out_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, int axis2) {
  return p->maps.get(map, base, 40 | axis2, slices, [&] { return encode_out_map(map, base, p->dm, slices, axis2, p->dct2_chunk); });
}

}  // namespace

cudaError_t ffk_dct2_init() {
  const cudaError_t e = cudaFuncSetAttribute(dct2_tc_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D2_SMEM);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(dct2_tc_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D2_SMEM);
}

// Which second axis the fused launch takes, and the channels of a work item: the shorter of h and t (smaller planes),
// an even number of groups, up to 2048 positions (W x n2).  Up to 1024 of them, 32 channels: 23% faster than the separate
// passes (T = 16, W = 64).  Up to 2048, 16 channels: two samples of 32 x 64 x 64 tokens, 24 heads, 10.8 ms at 1.6 GHz; the
// plane of 32 channels divided between two CTAs, whose rows cross the cluster, took 12.9, the separate passes 13.9 with
// intermediates of the same precision.
bool ffk_dct2_supported(const FFDims& dm, int* axis2, int* chunk) {
  if (dm.fp32 || (dm.d != 128 && dm.d != 64) || ff_fp32_grid(dm)) return false;
  const int a2 = dm.T < dm.H ? 0 : 1;
  const int n2 = a2 == 1 ? dm.H : dm.T;
  const int tiles = dm.W * n2 / ROWS, c = tiles > MAX_GPI ? 16 : 32, groups = tiles * c / GCOLS;
  if (groups > MAX_GPI || groups % 2 != 0) return false;
  *axis2 = a2;
  *chunk = c;
  return true;
}

// Matrix image of one axis and direction as the tensor-memory A operand: row j = output position
// of a tile, cell c = the bf16 pair (A[j][2c], A[j][2c+1]); three parts [128][64], each the bf16 next to what the parts
// before it leave.
// w axis: lines follow one another, A = I kron Mat (index = line*n + a); h, t: A = Mat kron I
// (index = a*kf + line); rows and columns past the tile's kf*n positions are zero.  `mat` is the host matrix
// [n][n], out[a] = sum_b mat[a][b] in[b].
bool ffk_dct2_build_image(ff_plan* p, int axis, int inverse, const float* mat, int n) {
  const size_t per = FF_IMAGE_CELLS;
  const int parts = ff_fp32_grid(p->dm) ? 3 : 2;        // (the third is read on those grids only)
  if (!p->dct2_images && cudaMalloc((void**)&p->dct2_images, FF_IMAGES * per * sizeof(uint32_t)) != cudaSuccess) return false;
  const FFPassShape g = ff_pass_shape(p->dm, axis);
  const int kf = g.kf;
  const bool seq = axis == 2;
  std::vector<uint32_t> img(parts * FF_IMAGE_PART);
  for (int j = 0; j < g.rows; ++j)
    for (int r = 0; r < g.rows; ++r) {
      float v;
      if (seq) v = (j / n == r / n) ? mat[(j % n) * n + (r % n)] : 0.f;
      else v = (j % kf == r % kf) ? mat[(j / kf) * n + (r / kf)] : 0.f;
      size_t cell = (size_t)j * IMG_CELLS + (r >> 1);
      for (int part = 0; part < parts; ++part, cell += FF_IMAGE_PART) {
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        const uint32_t hb = *(const uint16_t*)&h;
        img[cell] |= (r & 1) ? hb << 16 : hb;
        v -= __bfloat162float(h);
      }
    }
  const int slot = (inverse ? 3 : 0) + axis;
  return cudaMemcpy(p->dct2_images + slot * per, img.data(), img.size() * sizeof(uint32_t), cudaMemcpyHostToDevice) == cudaSuccess;
}

// Forward: Q, K, V of tensor-heads [g0, g0 + g) -> w and second-axis transform -> hi/lo grids.
cudaError_t ffk_dct2_forward(ff_plan* p, const void* Q, const void* K, const void* V, int g0, int g, void* out_hi, void* out_lo,
                             bool clear_energy, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int G = p->dct_group;
  const int axis2 = p->dct2_axis2;
  CUtensorMap mq, mk, mv, oh, ol;
  if (!in_map(p, &mq, Q, dm.BH, axis2) || !in_map(p, &mk, K, dm.BH, axis2) ||
      !in_map(p, &mv, V, dm.BH, axis2) || !out_map(p, &oh, out_hi, G, axis2) ||
      !out_map(p, &ol, out_lo, G, axis2))
    return cudaErrorInvalidValue;
  const size_t per = FF_IMAGE_CELLS;
  Dct2Params P{};
  P.dm = dm; P.status = p->buf.status;
  P.img1 = p->dct2_images + (size_t)(0 + 2) * per; P.img2 = p->dct2_images + (size_t)(0 + axis2) * per;
  P.axis2 = axis2; P.n1 = dm.W; P.n2 = axis2 == 1 ? dm.H : dm.T; P.n3 = axis2 == 1 ? dm.T : dm.H;
  P.clear = clear_energy ? p->buf.energy : nullptr;
  P.in_split = 0; P.last = 0; P.group = g; P.group_start = g0;
  return launch(p, mq, mk, mv, oh, ol, P, st);
}

// Inverse: hi/lo grids of heads [h0, h0 + g) -> w and second-axis inverse transform -> out.
cudaError_t ffk_dct2_inverse(ff_plan* p, const void* in_hi, const void* in_lo, int h0, int g, void* out, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int G = p->dct_group;
  const int axis2 = p->dct2_axis2;
  CUtensorMap mh, ml, mo;
  if (!in_map(p, &mh, in_hi, G, axis2) || !in_map(p, &ml, in_lo, G, axis2) ||
      !out_map(p, &mo, out, dm.BH, axis2))
    return cudaErrorInvalidValue;
  const size_t per = FF_IMAGE_CELLS;
  Dct2Params P{};
  P.dm = dm; P.status = p->buf.status;
  P.img1 = p->dct2_images + (size_t)(3 + 2) * per; P.img2 = p->dct2_images + (size_t)(3 + axis2) * per;
  P.axis2 = axis2; P.n1 = dm.W; P.n2 = axis2 == 1 ? dm.H : dm.T; P.n3 = axis2 == 1 ? dm.T : dm.H;
  P.in_split = 1; P.last = 1; P.group = g; P.group_start = h0;
  return launch(p, mh, ml, ml, mo, mo, P, st);
}

FF_CLOCKS_READ(transform_plane)
