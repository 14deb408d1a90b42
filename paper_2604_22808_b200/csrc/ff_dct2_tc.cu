// Two axis passes of the separable transform in one launch ("Separable spectral decomposition",
// "Reconstruction"): the w axis and a second axis (h or t, whichever is shorter), with the
// intermediate between them kept in shared memory.  bf16 storage, 32 channels per work item.
//
// A work item is one plane of the grid (all positions of the two axes at one coordinate of the third
// axis) of one tensor-head, for one chunk of 32 channels.  A CTA owns the item: the plane's
// intermediate (hi/lo bf16, 4 bytes per value) takes 128 KB or less of its shared memory.  A plane of twice that
// belongs to a cluster of two CTAs (template parameter PAIR): each transforms half of its lines in phase 1, sends a
// result row to the CTA that owns the row's w coefficient (st.shared::cluster), and takes half of the w coefficients in
// phase 2; the buffer is handed over with barriers that the other CTA arrives at.
//   phase 1  transforms the plane's w lines (tiles of 128 positions = 128/W lines, fetched by TMA) and
//            scatters each result row, as a hi/lo bf16 pair, into the plane buffer; the rows land in
//            the operand layout of phase 2
//   phase 2  transforms the second axis (tiles of 128/n2 neighbouring w coefficients x all n2
//            positions), straight from the buffer, and stores the result with tensor stores (hi/lo
//            grids, or the caller's tensor)
// Both contractions are D[j][c] = sum_r A[j][r] X[r][c] over tiles of 128 positions x 32 channels
// with the matrix A = I kron Mat (w lines follow one another) or Mat kron I (lines of the second
// axis interleave) held in TENSOR MEMORY as the A operand (hi and lo bf16 parts, 64 columns each),
// so that a tile costs no shared-memory traffic for the matrix; the data tile is the MN-major B
// operand in place (64-byte rows, 64-byte swizzle); four tiles share one instruction (N = 128: an
// instruction takes the same time for any N up to 128).
//
//   warp 0        TMA producer (ring of 8 tiles, or 4 hi/lo pairs)
//   warp 1        tcgen05.mma issuer of phase 1; owns the tensor-memory allocation
//   warp 2        idle (PAIR: tells both CTAs when this one has finished reading its part of the buffer)
//   warp 3        tcgen05.mma issuer of phase 2
//   warps 4..11   phase-1 epilogue (a thread owns one position of a tile; the first four warps take
//                 the first tile of a pair, the next four the second)
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

constexpr int CHK = 32;                       // channels per work item
constexpr int ROWS = 128;                     // positions per tile
constexpr int TILE_B = ROWS * CHK * 2;        // 8 KB: one bf16 tile
constexpr int NSTG = 8;                       // input ring: at most 8 tiles (64 KB: 8 bf16 tiles or 4 hi/lo pairs)
constexpr int RING_B = NSTG * TILE_B;
constexpr int MAX_TPC = 8;                    // tiles per CTA and item (128 KB of hi/lo buffer)
constexpr int D2_THREADS = 640;                 // TMA, MMA 1, release, MMA 2, 8 phase-1 and 8 phase-2 epilogue warps
constexpr int NA1 = 1, NA2 = 1;               // accumulator buffers (batches of 128 columns) of the two phases
constexpr int IMG_CELLS = 64;                 // 32-bit tensor-memory cells per matrix row: two bf16 K elements each
constexpr int STG_ROW = 64;                   // bytes per staged row (32 channels)

struct Dct2Params {
  FFDims dm;
  const uint32_t* img1;    // w-axis matrix: hi [128][64] cells, then lo
  const uint32_t* img2;    // second-axis matrix: hi, then lo
  int axis2;               // 1 = h, 0 = t
  int n1, n2, n3;          // W, length of the second axis, length of the remaining axis
  int in_split;            // input is a hi/lo pair of grids (map0 = hi, map1 = lo); otherwise Q, K, V
  int last;                // output is the caller's tensor (bf16, no lo part)
  int group, group_start;
  int nchunk;              // head_dim / 32
  int tpc;                 // tiles per CTA and item
  double* clear;           // band energies to clear for the sums that follow (first launch of a routed forward), or NULL
  int* status;
};

struct D2Shared {
  uint64_t in_full[NSTG], in_empty[NSTG], acc1_full[NA1], acc1_empty[NA1], acc2_full[NA2], acc2_empty[NA2];
  // The plane buffer has one slot of 8 tiles or two of 4 (items alternate): phase 1 of the next item fills one
  // slot while phase 2 of the current item reads the other.
  uint64_t buf_full[2];    // all rows of the item have landed in the slot
  uint64_t buf_half[2];    // the rows of the first half of the second axis have landed
  uint64_t half_free[2];   // phase 2 has finished reading those rows (its k-steps 0..3 of every batch)
  uint64_t buf_free[2];    // phase 2 of the item has finished reading the slot (PAIR: in both CTAs)
  uint64_t mma2_done[2];   // (PAIR) this CTA's phase-2 instructions of the item (by slot) have completed
  uint32_t tmem_base;
  int abort_flag;
};

// Shared-memory descriptor of an MN-major operand stored as 64-byte rows (32 bf16) with the 64-byte
// swizzle: 8-row groups 512 bytes apart (SBO); `lbo` = distance between 32-element chunks along N.
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;   // SWIZZLE_64B
  return d;
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar_addr) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait of a whole warp on a barrier of the plane buffer; with PAIR its arrivals come from both CTAs.
template <bool PAIR>
__device__ __forceinline__ bool wait_buffer(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (!PAIR) return mbar_wait_warp(bar, parity, abort_flag);
  bool ok = mbar_try_wait_cluster(bar, parity);
  const long long t0 = clock64();
  while (!ok && !*abort_flag) {
    ok = mbar_try_wait_cluster(bar, parity);
    if (!ok && clock64() - t0 > kWaitLimitCycles) *abort_flag = 1;
  }
  return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// (rows that the other CTA wrote, or that go there)
template <bool PAIR> __device__ __forceinline__ void fence_buffer() {
  if (PAIR) asm volatile("fence.proxy.async;" ::: "memory");
  else fence_proxy_async();
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// Item `it` of the launch: chunk fastest (CTAs that run side by side read neighbouring 64-byte
// pieces of the same rows), then the coordinate of the remaining axis, then the tensor-head.
__device__ __forceinline__ void decode_item(const Dct2Params& P, int it, int& gi, int& a3, int& chunk) {
  chunk = it % P.nchunk;
  const int rest = it / P.nchunk;
  a3 = rest % P.n3;
  gi = rest / P.n3;
}

// fp32 accumulators of one row (32 channels) -> bf16 hi and lo words (two channels per word)
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
// caller's tensor in map_oh), box = the 32 positions x 32 channels an epilogue warp holds.
template <bool PAIR>
__global__ void __launch_bounds__(D2_THREADS, 1)
dct2_tc_kernel(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap map1,
               const __grid_constant__ CUtensorMap map2, const __grid_constant__ CUtensorMap map_oh,
               const __grid_constant__ CUtensorMap map_ol, const Dct2Params P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const FFDims& dm = P.dm;
  const int tpc = P.tpc;
  const int STAGE_B = P.in_split ? 2 * TILE_B : TILE_B;            // hi tile, then lo tile
  uint8_t* sBuf = smem;                                            // tpc x (hi 8 KB, lo 8 KB): the plane's intermediate
  uint8_t* sStage = smem + MAX_TPC * 2 * TILE_B;                   // 8 phase-2 warps x (hi 2 KB, lo 2 KB), 1024-byte aligned
  uint8_t* sIn = sStage + 8 * 2 * 32 * STG_ROW;                    // NSTG x STAGE_B
  D2Shared& sh = *(D2Shared*)(sIn + RING_B);
  const int nslot = RING_B / STAGE_B;                              // ring slots: 8 tiles, or 4 hi/lo pairs
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int cs = PAIR ? 2 : 1;                                 // CTAs of a plane
  const int rank = PAIR ? (int)cluster_ctarank() : 0;
  const int n1 = P.n1, n2 = P.n2;
  const int ln1 = 31 - __clz(n1);
  const int kf1 = ROWS / n1, kf2 = ROWS / n2;
  const int lkf2 = 31 - __clz(kf2);
  const int total = P.group * P.n3 * P.nchunk;
  const int nsl = !PAIR && tpc <= MAX_TPC / 2 ? 2 : 1;             // slots of the plane buffer
  const int bt = tpc < 4 ? tpc : 4;                                // tiles per instruction batch (N = 32 bt columns): an
  const int nb = tpc / bt;                                         // instruction costs the same for any N up to 128
  // One CTA per plane and an even number of batches: the first half of the phase-1 batches holds the first half
  // of the second axis, i.e. rows 0..63 of every phase-2 tile = its k-steps 0..3.  Phase 2 of the item's first
  // batch starts on those while phase 1 still works on the second half.
  const bool half_start = !PAIR && nb >= 2 && (nb & 1) == 0;
  // ... and phase 1 of the next item may overwrite those rows as soon as phase 2 has read them (forward launch:
  // measured slower for the inverse, whose phase 1 issues half as many instructions again)
  const bool half_release = half_start && !P.in_split;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSTG; ++i) { mbar_init(&sh.in_full[i], 1); mbar_init(&sh.in_empty[i], 1); }
    for (int i = 0; i < NA1; ++i) { mbar_init(&sh.acc1_full[i], 1); mbar_init(&sh.acc1_empty[i], 256); }
    for (int i = 0; i < NA2; ++i) { mbar_init(&sh.acc2_full[i], 1); mbar_init(&sh.acc2_empty[i], 256); }
    for (int i = 0; i < 2; ++i) { mbar_init(&sh.buf_full[i], 8 * cs); mbar_init(&sh.buf_free[i], cs); mbar_init(&sh.buf_half[i], 8); }
    if (PAIR) { mbar_init(&sh.mma2_done[0], 1); mbar_init(&sh.mma2_done[1], 1); }
    mbar_init(&sh.half_free[0], 1); mbar_init(&sh.half_free[1], 1);
    sh.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_barrier();                                     // the other CTA's barriers exist before anyone arrives there
  tc_fence_after();
  const uint32_t tm = sh.tmem_base;
  volatile int* abort_flag = &sh.abort_flag;
  // tensor-memory columns: matrix images [0,256): w hi, w lo, second axis hi, lo; phase-1 accumulators
  // (NA1 batches of 128 columns) from 256; phase-2 accumulators (NA2 batches) behind them
  constexpr uint32_t COL_A1H = 0, COL_A1L = 64, COL_A2H = 128, COL_A2L = 192, COL_ACC1 = 256, COL_ACC2 = 256 + NA1 * 128;
  static_assert(COL_ACC2 + NA2 * 128 <= 512, "tensor memory has 512 columns");

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

  const int cid = (int)blockIdx.x / cs, ncl = (int)gridDim.x / cs;
  FF_CLOCK(t_all);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&map0);
      unsigned n = 0;
      bool ok = true;
      for (int it = cid; it < total && ok; it += ncl) {
        int gi, a3, chunk; decode_item(P, it, gi, a3, chunk);
        const CUtensorMap* map = &map0;
        int slice = gi;
        if (!P.in_split) {
          const int th = P.group_start + gi;
          const int tensor = th / dm.BH;
          map = tensor == 0 ? &map0 : (tensor == 1 ? &map1 : &map2);
          slice = th % dm.BH;
        }
        for (int k = 0; k < tpc && ok; ++k, ++n) {
          const int slot = n % nslot;
          FF_CLOCK(tp0);
          if (n >= (unsigned)nslot) ok = mbar_wait(&sh.in_empty[slot], ((n / nslot) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 12, tp0);
          if (!ok) break;
          uint8_t* dst = sIn + slot * STAGE_B;
          const int u1 = rank * tpc + k;                           // tile of the plane: lines u1 kf1 .. + kf1
          const int b0 = u1 * kf1;
          const int ch = P.axis2 == 1 ? b0 : a3, ct = P.axis2 == 1 ? a3 : b0;
          mbar_arrive_expect_tx(&sh.in_full[slot], STAGE_B);
          tma_load_5d(dst, map, &sh.in_full[slot], chunk * CHK, 0, ch, ct, slice);
          if (P.in_split) tma_load_5d(dst + TILE_B, &map1, &sh.in_full[slot], chunk * CHK, 0, ch, ct, slice);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer, phase 1
    // batches of bt input tiles (neighbouring slots of the ring), N = 32 bt.  A descriptor advances by
    // 1024 bytes (64 in its address field) per 16 rows of K.
    {
      const uint32_t idesc = idesc_bf16_f32(ROWS, bt * CHK, /*a_mn_major=*/false, /*b_mn_major=*/true);
      const uint32_t in_base = smem_u32(sIn);
      unsigned n1b = 0;
      bool ok = true;
      for (int it = cid; it < total && ok; it += ncl) {
        for (int kb = 0; kb < nb && ok; ++kb, ++n1b) {
          const int ab = n1b % NA1;
          const unsigned nt = bt * n1b;                            // index of the batch's first tile in the ring sequence
          FF_CLOCK(tm0);
          for (int i = 0; i < bt && ok; ++i) ok = mbar_wait_warp(&sh.in_full[(nt + i) % nslot], ((nt + i) / nslot) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 7, tm0);
          FF_CLOCK(tm1);
          if (ok && n1b >= (unsigned)NA1) ok = mbar_wait_warp(&sh.acc1_empty[ab], ((n1b / NA1) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 8, tm1);
          if (!ok) break;
          tc_fence_after();
          const uint32_t x0 = in_base + (uint32_t)(nt % nslot) * STAGE_B;
          const uint64_t xh = smem_desc_sw64(x0, STAGE_B, 512), xl = smem_desc_sw64(x0 + TILE_B, STAGE_B, 512);
          const uint32_t d_tm = tm + COL_ACC1 + ab * 128;
          if (P.in_split) {
#pragma unroll
            for (int ks = 0; ks < ROWS / 16; ++ks) {
              umma_ts(d_tm, tm + COL_A1H + ks * 8, xh + (uint64_t)(ks * 64), idesc, ks > 0 ? 1u : 0u);
              umma_ts(d_tm, tm + COL_A1L + ks * 8, xh + (uint64_t)(ks * 64), idesc, 1u);
              umma_ts(d_tm, tm + COL_A1H + ks * 8, xl + (uint64_t)(ks * 64), idesc, 1u);
            }
          } else {
#pragma unroll
            for (int ks = 0; ks < ROWS / 16; ++ks) {
              umma_ts(d_tm, tm + COL_A1H + ks * 8, xh + (uint64_t)(ks * 64), idesc, ks > 0 ? 1u : 0u);
              umma_ts(d_tm, tm + COL_A1L + ks * 8, xh + (uint64_t)(ks * 64), idesc, 1u);
            }
          }
          for (int i = 0; i < bt; ++i) umma_commit(&sh.in_empty[(nt + i) % nslot]);
          umma_commit(&sh.acc1_full[ab]);
        }
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ MMA issuer, phase 2
    // (a warp of its own: phase 2 of an item waits for all of its phase 1, phase 1 of the next item does not)
    {
      const uint32_t idesc = idesc_bf16_f32(ROWS, bt * CHK, /*a_mn_major=*/false, /*b_mn_major=*/true);
      const uint32_t buf_base = smem_u32(sBuf);
      unsigned n2b = 0, ni = 0;
      bool ok = true;
      for (int it = cid; it < total && ok; it += ncl, ++ni) {
        // the plane's rows have landed in this CTA's buffer
        FF_CLOCK(tm2);
        const int sl = (int)(ni % nsl);                             // the item's slot of the plane buffer
        ok = half_start ? mbar_wait_warp(&sh.buf_half[sl], (ni / nsl) & 1, abort_flag)
                        : wait_buffer<PAIR>(&sh.buf_full[sl], (ni / nsl) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 9, tm2);
        if (!ok) break;
        fence_buffer<PAIR>();
        for (int kb = 0; kb < nb && ok; ++kb, ++n2b) {
          const int ab = n2b % NA2;
          FF_CLOCK(tm3);
          if (n2b >= (unsigned)NA2) ok = mbar_wait_warp(&sh.acc2_empty[ab], ((n2b / NA2) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 10, tm3);
          if (!ok) break;
          tc_fence_after();
          const uint32_t x0 = buf_base + (uint32_t)(sl * tpc + bt * kb) * 2 * TILE_B;   // tiles bt kb ..: hi, lo of each in turn
          const uint64_t xh = smem_desc_sw64(x0, 2 * TILE_B, 512), xl = smem_desc_sw64(x0 + TILE_B, 2 * TILE_B, 512);
          const uint32_t d_tm = tm + COL_ACC2 + ab * 128;
#pragma unroll
          for (int ks = 0; ks < ROWS / 16; ++ks) {
            if (ks == ROWS / 32 && kb == 0 && half_start) {          // the second half of the rows
              FF_CLOCK(tm4);
              ok = mbar_wait_warp(&sh.buf_full[sl], (ni / nsl) & 1, abort_flag);
              FF_CLOCK_ADD(lane == 0, P.in_split * 16 + 11, tm4);
              if (!ok) break;
              fence_proxy_async();
              tc_fence_after();
            }
            umma_ts(d_tm, tm + COL_A2H + ks * 8, xh + (uint64_t)(ks * 64), idesc, ks > 0 ? 1u : 0u);
            umma_ts(d_tm, tm + COL_A2L + ks * 8, xh + (uint64_t)(ks * 64), idesc, 1u);
            umma_ts(d_tm, tm + COL_A2H + ks * 8, xl + (uint64_t)(ks * 64), idesc, 1u);
            // rows 0..63 of every tile have been read once the last batch's k-step 3 is done: phase 1 of the next
            // item may overwrite them
            if (ks == ROWS / 32 - 1 && kb == nb - 1 && half_release) umma_commit(&sh.half_free[sl]);
          }
          if (!ok) break;
          umma_commit(&sh.acc2_full[ab]);
        }
        umma_commit(PAIR ? &sh.mma2_done[sl] : &sh.buf_free[sl]);
      }
    }
  } else if (PAIR && warp == 2) {
    // ------------------------------------------------------------------ buffer release, to both CTAs
    if (lane == 0) {
      unsigned ni = 0;
      bool ok = true;
      for (int it = cid; it < total && ok; it += ncl, ++ni) {
        ok = mbar_wait(&sh.mma2_done[ni % nsl], (ni / nsl) & 1, abort_flag);
        if (!ok) break;
        for (int rk = 0; rk < cs; ++rk) mbar_arrive_cluster(mapa(smem_u32(&sh.buf_free[ni % nsl]), (uint32_t)rk));
      }
    }
  } else if (warp >= 4 && warp < 12) {
    // ------------------------------------------------------------------ phase-1 epilogue
    // accumulators -> hi/lo rows in the plane buffer.  A thread owns row (line l1, w coefficient a1)
    // of its tile and sends it as four 16-byte pieces of hi and four of lo, straight from registers.
    const int ew = warp - 4;                               // 0..7
    const int half = ew >> 2;                              // which tile of a pair
    const int quarter = warp & 3;
    const int j = quarter * 32 + lane;                     // position of this thread inside a tile
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const uint32_t buf_base = smem_u32(sBuf);
    const int l1 = j >> ln1, a1 = j & (n1 - 1);
    const int u2g = a1 >> lkf2;                            // phase-2 tile of the plane that takes coefficient a1
    const int owner = PAIR ? u2g / tpc : 0, u2 = u2g - owner * tpc;      // its CTA, its tile there
    // Eight neighbouring lanes store at once; their rows are kf2 per tile, and rows of different tiles
    // that share (row / 2) % 4 would meet in the same banks: the lanes of tile t of the eight start
    // their four pieces at piece `rot` instead of 0, which spreads them over the banks.
    const int rot = (kf2 >= 8 ? 0 : ((lane & 7) >> lkf2) * (kf2 == 4 ? 2 : 1)) & 3;
    unsigned n1b = 0, ni = 0;
    bool ok = true;
    for (int it = cid; it < total && ok; it += ncl, ++ni) {
      FF_CLOCK(te0);
      const int sl = (int)(ni % nsl);                         // the item's slot: free once phase 2 of item ni - nsl is done
      if (ni >= (unsigned)nsl) {
        // (half_release: the first half of the batches writes rows phase 2 releases earlier; the rest waits below)
        ok = half_release ? __all_sync(0xffffffffu, mbar_wait(&sh.half_free[sl], ((ni / nsl) - 1) & 1, abort_flag))
                        : wait_buffer<PAIR>(&sh.buf_free[sl], ((ni / nsl) - 1) & 1, abort_flag);
        if (!ok) break;
      }
      FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 1, te0);
      for (int kb = 0; kb < nb && ok; ++kb, ++n1b) {
        if (half_release && kb == nb / 2 && ni >= (unsigned)nsl) {
          ok = mbar_wait_warp(&sh.buf_free[sl], ((ni / nsl) - 1) & 1, abort_flag);
          if (!ok) break;
        }
        const int ab = n1b % NA1;
        FF_CLOCK(te1);
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc1_full[ab], (n1b / NA1) & 1, abort_flag));
        if (!ok) break;
        FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 0, te1);
        FF_CLOCK(te2);
        tc_fence_after();
        for (int tb = half; tb < bt; tb += 2) {            // this warp's tiles of the batch
        uint32_t r[32];
        tmem_ld32(tm + lane_addr + COL_ACC1 + ab * 128 + tb * 32, r);
        tmem_wait_ld();
        if (tb + 2 >= bt) {                                // the accumulators are free once the warp's last tile is read
          tc_fence_before();
          mbar_arrive(&sh.acc1_empty[ab]);
        }
        uint32_t hi[16], lo[16];
        split_hi_lo(r, hi, lo, true);
        // where the row goes: position b of the second axis, row b kf2 + (a1 mod kf2) of tile u2
        const int u1 = rank * tpc + bt * kb + tb;
        const int b = u1 * kf1 + l1;
        const int drow = (b << lkf2) | (a1 & (kf2 - 1));
        uint32_t daddr = buf_base + (uint32_t)(sl * tpc + u2) * 2 * TILE_B + (uint32_t)drow * STG_ROW;
        if (PAIR) daddr = mapa(daddr, (uint32_t)owner);
        const int swz = (drow >> 1) & 3;
        // (debug build) the row lies inside a tile of the buffer
        if (!FF_DBG_OK(drow >= 0 && drow < ROWS && u2 >= 0 && u2 < tpc && owner < cs && b < n2, P.status, 4)) continue;
        // rotate the pieces by `rot` (two conditional swaps), then piece i of the registers is piece (i + rot) % 4 of the row
        if (rot & 1) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t h0 = hi[q], l0 = lo[q];
            hi[q] = hi[4 + q]; hi[4 + q] = hi[8 + q]; hi[8 + q] = hi[12 + q]; hi[12 + q] = h0;
            lo[q] = lo[4 + q]; lo[4 + q] = lo[8 + q]; lo[8 + q] = lo[12 + q]; lo[12 + q] = l0;
          }
        }
        if (rot & 2) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const uint32_t h0 = hi[q], l0 = lo[q];
            hi[q] = hi[8 + q]; hi[8 + q] = h0;
            lo[q] = lo[8 + q]; lo[8 + q] = l0;
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t dst = daddr + (uint32_t)((((i + rot) & 3) ^ swz) << 4);
          const uint4 vh = make_uint4(hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
          const uint4 vl = make_uint4(lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
          if (PAIR) { st_cluster_v4(dst, vh); st_cluster_v4(dst + TILE_B, vl); }
          else { st_shared_v4(dst, vh); st_shared_v4(dst + TILE_B, vl); }
        }
        }
        FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 2, te2);
        if (half_start && kb == nb / 2 - 1) {               // this warp's rows of the first half are written
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.buf_half[sl]);
        }
      }
      if (!ok) break;
      // this warp's rows of the item are written
      FF_CLOCK(te4);
      fence_buffer<PAIR>();
      __syncwarp();
      if (PAIR) { if (lane < cs) mbar_arrive_cluster(mapa(smem_u32(&sh.buf_full[sl]), (uint32_t)lane)); }
      else if (lane == 0) mbar_arrive(&sh.buf_full[sl]);
      FF_CLOCK_ADD(threadIdx.x == 128, P.in_split * 16 + 6, te4);
    }
  } else if (warp >= 12) {
    // ------------------------------------------------------------------ phase-2 epilogue
    // accumulators -> destination grids.  Rows 32 quarter .. + 31 of a tile are the box [a2 = a0 .., w = l0 ..]
    // of the store map; the warp stages them (64-byte swizzle) and one lane issues the tensor stores.
    const int ew = warp - 12;                              // 0..7
    const int half = ew >> 2;
    const int quarter = warp & 3;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    uint8_t* st_hi = sStage + ew * 2 * 32 * STG_ROW;
    uint8_t* st_lo = st_hi + 32 * STG_ROW;
    const int j0 = quarter * 32;
    const int a0 = j0 >> lkf2, l0 = j0 & (kf2 - 1);
    unsigned n2b = 0;
    bool ok = true;
    for (int it = cid; it < total && ok; it += ncl) {
      int gi, a3, chunk; decode_item(P, it, gi, a3, chunk);
      const int out_slice = P.last ? P.group_start + gi : gi;
      for (int kb = 0; kb < nb && ok; ++kb, ++n2b) {
        const int ab = n2b % NA2;
        FF_CLOCK(te5);
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc2_full[ab], (n2b / NA2) & 1, abort_flag));
        if (!ok) break;
        FF_CLOCK_ADD(threadIdx.x == 384, P.in_split * 16 + 3, te5);
        FF_CLOCK(te6);
        tc_fence_after();
        for (int tb = half; tb < bt; tb += 2) {            // this warp's tiles of the batch
        uint32_t r[32];
        tmem_ld32(tm + lane_addr + COL_ACC2 + ab * 128 + tb * 32, r);
        tmem_wait_ld();
        if (tb + 2 >= bt) {
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
        // 16-byte chunk i of row `lane` at chunk position i ^ (lane / 2 % 4): the 64-byte swizzle
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int so = lane * STG_ROW + ((i ^ ((lane >> 1) & 3)) << 4);
          *(uint4*)(st_hi + so) = make_uint4(hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
          if (!P.last) *(uint4*)(st_lo + so) = make_uint4(lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          const int u2g = rank * tpc + bt * kb + tb;        // tile of the plane: w coefficients u2g kf2 .. + kf2
          const int cw = u2g * kf2 + l0;
          const int ch = P.axis2 == 1 ? a0 : a3, ct = P.axis2 == 1 ? a3 : a0;
          tma_store_5d(st_hi, &map_oh, chunk * CHK, cw, ch, ct, out_slice);
          if (!P.last) tma_store_5d(st_lo, &map_ol, chunk * CHK, cw, ch, ct, out_slice);
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
  if (PAIR) cluster_barrier();      // no CTA leaves while the other may still write into its shared memory or arrive at its barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

// 5-D map over a [slices][T][H][W][d] bf16 grid.  Load box: one phase-1 tile, 32 channels of 128/W
// whole w lines that are neighbours along the second axis.
bool encode_in_map(CUtensorMap* map, const void* base, const FFDims& dm, int slices, int axis2) {
  const cuuint64_t CH = (cuuint64_t)dm.d;
  cuuint64_t dims[5] = {CH, (cuuint64_t)dm.W, (cuuint64_t)dm.H, (cuuint64_t)dm.T, (cuuint64_t)slices};
  cuuint64_t strides[4] = {CH * 2, (cuuint64_t)dm.W * CH * 2, (cuuint64_t)dm.H * dm.W * CH * 2, (cuuint64_t)dm.N * CH * 2};
  cuuint32_t box[5] = {CHK, (cuuint32_t)dm.W, 1, 1, 1};
  box[axis2 == 1 ? 2 : 3] = (cuuint32_t)(ROWS / dm.W);
  return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

// Store box: what one epilogue warp holds after phase 2, 32 channels of tile rows 32 q .. 32 q + 31,
// row = (position along the second axis) * kf2 + (w coefficient inside the tile).
bool encode_out_map(CUtensorMap* map, const void* base, const FFDims& dm, int slices, int axis2) {
  const cuuint64_t CH = (cuuint64_t)dm.d;
  cuuint64_t dims[5] = {CH, (cuuint64_t)dm.W, (cuuint64_t)dm.H, (cuuint64_t)dm.T, (cuuint64_t)slices};
  cuuint64_t strides[4] = {CH * 2, (cuuint64_t)dm.W * CH * 2, (cuuint64_t)dm.H * dm.W * CH * 2, (cuuint64_t)dm.N * CH * 2};
  const int n2 = axis2 == 1 ? dm.H : dm.T;
  const int kf2 = ROWS / n2;                       // at most 8
  cuuint32_t box[5] = {CHK, (cuuint32_t)kf2, 1, 1, 1};
  box[axis2 == 1 ? 2 : 3] = (cuuint32_t)(32 / kf2);
  return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B,
                       CU_TENSOR_MAP_L2_PROMOTION_NONE);
}

// (the staging areas of the tensor stores sit 1024-byte aligned: their 64-byte swizzle is a function of the address)
constexpr size_t D2_SMEM = 1024 + (size_t)MAX_TPC * 2 * TILE_B + (size_t)8 * 2 * 32 * STG_ROW + (size_t)RING_B + sizeof(D2Shared) + 64;

cudaError_t launch(ff_plan* p, const CUtensorMap& m0, const CUtensorMap& m1, const CUtensorMap& m2, const CUtensorMap& moh,
                   const CUtensorMap& mol, Dct2Params& P, cudaStream_t st) {
  const int items = P.group * P.n3 * P.nchunk, cs = p->dct2_pair ? 2 : 1;
  const int most = p->sm_count / cs, ncl = items < most ? items : most;
  const dim3 grid((unsigned)(ncl * cs));
  const cudaError_t e = p->dct2_pair
      ? ff_launch_cluster(dct2_tc_kernel<true>, cs, grid, dim3(D2_THREADS), D2_SMEM, st, m0, m1, m2, moh, mol, P)
      : ff_launch(dct2_tc_kernel<false>, grid, dim3(D2_THREADS), D2_SMEM, st, m0, m1, m2, moh, mol, P);
  if (e != cudaSuccess) return e;
  p->launches += 1;
  return cudaSuccess;
}

// (through the plan's cache)
bool in_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, int axis2) {
  return p->maps.get(map, base, 32 | axis2, slices, [&] { return encode_in_map(map, base, p->dm, slices, axis2); });
}
bool out_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, int axis2) {
  return p->maps.get(map, base, 40 | axis2, slices, [&] { return encode_out_map(map, base, p->dm, slices, axis2); });
}

}  // namespace

cudaError_t ffk_dct2_init() {
  const cudaError_t e = cudaFuncSetAttribute(dct2_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D2_SMEM);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(dct2_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D2_SMEM);
}

// Which second axis the fused launch takes, and whether two CTAs share a plane: the shorter of h and t (smaller planes),
// an even number of tiles a CTA, up to 2048 positions (W x n2).  One CTA a plane (up to 1024): 23% faster than the separate
// passes (T = 16, W = 64).  Two CTAs: two samples of 32 x 64 x 64 tokens, 24 heads, 12.91 ms against 13.88 with passes that
// hand on bf16 pairs.  (With byte-form intermediates those take 12.52 ms, but lose a bit: low coefficients 9.6e-6 instead
// of 6.3e-6 from fp64.)  From four CTAs on the launch loses to the passes with bytes, which the
// larger planes take (64 x 64 x 64: 10.9 against 8.7 ms for the transform): the remote stores of phase 1 and their
// cluster-scope release cost more than the saved round trip.
bool ffk_dct2_supported(const FFDims& dm, int* axis2, bool* pair) {
  if (dm.fp32 || dm.d % CHK != 0 || (dm.d != 128 && dm.d != 64) || ff_fp32_grid(dm)) return false;
  const int a2 = dm.T < dm.H ? 0 : 1;
  const int n2 = a2 == 1 ? dm.H : dm.T;
  const int tiles = dm.W * n2 / ROWS, cs = tiles > MAX_TPC ? 2 : 1;
  if (tiles / cs > MAX_TPC || tiles / cs % 2 != 0) return false;
  *axis2 = a2;
  *pair = cs == 2;
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
  if (!p->dct2_images && cudaMalloc((void**)&p->dct2_images, 6 * per * sizeof(uint32_t)) != cudaSuccess) return false;
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
  P.in_split = 0; P.last = 0; P.group = g; P.group_start = g0; P.nchunk = dm.d / CHK;
  P.tpc = dm.W * P.n2 / ROWS / (p->dct2_pair ? 2 : 1);
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
  P.in_split = 1; P.last = 1; P.group = g; P.group_start = h0; P.nchunk = dm.d / CHK;
  P.tpc = dm.W * P.n2 / ROWS / (p->dct2_pair ? 2 : 1);
  return launch(p, mh, ml, ml, mo, mo, P, st);
}

FF_CLOCKS_READ(transform_plane)
