// Separable transform on the tensor cores ("Separable spectral decomposition", "Reconstruction"),
// bf16 storage, head_dim 128 or 64 (template parameter CH).  Every axis pass is a batched contraction over "lines" of n grid
// positions along the axis (all other coordinates fixed): out[a][c] = sum_b Mat[a][b] in[b][c].
// A CTA works on tiles of 128 grid positions = 128/n adjacent lines, fetched by one TMA box per
// 64-channel half (a contiguous run of memory for the w axis; 128/n neighbouring w positions per
// axis position for the h and t axes, so that the strided axes also read contiguous pieces).
// One tile is one 128 x 128 x 128 contraction
//     D[j][c] = sum_r A[j][r] * X[r][c],   A = Mat kron I (or I kron Mat) over the lines of the tile
// with A held in tensor memory for the whole launch (loaded once per CTA), X the TMA tile used in place as
// the MN-major B operand, and D in tensor memory with one output position per lane, so that an
// epilogue thread owns a whole 256-byte output row and stores it with 16-byte accesses.
//
// Precision: the transform matrix is split into bf16 hi + lo parts, and so is every intermediate
// between two axis passes (two bf16 grids, hi = bf16(v), lo = bf16(v - hi)); a pass then issues
// C_hi*X_hi + C_lo*X_hi + C_hi*X_lo per k-step.  Intermediates can be far larger than the final
// values (low-frequency content, the constant offset the exchange adds to a whole band), so a
// single bf16 rounding between passes would not meet the output tolerance.
//
// Three-byte intermediates.  Where the three axes run as separate passes (planes above 2048 positions, or asked for), the
// pair written by the first forward pass and the pairs between the inverse passes are stored as the fp32 value
// rounded to 24 bits: the upper 16 bits (a bf16 by truncation) in the hi grid and the next 8 bits in a byte grid.  hi
// and (value - hi) are both exact bf16 operands, together they carry 16 significant bits, one less than a bf16 hi/lo
// pair, and a pass moves 3 instead of 4 bytes per value.  A launch whose input has the byte form (FORM_BYTES) runs four more
// warps that expand the bytes of every arriving tile to the bf16 lo operand in shared memory before the MMAs
// read it (128 channels: in place, the bytes of a row arrive inside the row's own bf16 space).  The expansion
// competes with the epilogue for issue slots; measured per launch at 1M tokens (3 tensor-heads): a middle pass
// 0.55 -> 0.48 ms with byte-form input and output, the band-split pass 0.43 -> 0.67 ms and the last inverse
// pass 0.38 -> 0.42 ms with byte-form input.  So the band-split pass always reads a bf16 pair (the second
// forward pass writes one), and the fused two-axis launches keep bf16 pairs on both sides.
//
// Any grid.  A line of any length up to 128 fits a tile, so the passes run on every grid: floor(128 / n) lines
// per tile, the left-over rows zero in the matrix and in shared memory, partial last tiles filled with zeros and
// clipped by the copies.  Grids with an axis other than 16, 32, 64 or 128 ran on fp32 kernels, and the precision stays
// that of fp32 numbers: the passes hand on fp32 grids (FORM_EXACT1 and FORM_EXACT), matrix and data are three bf16 parts
// each, which hold all 24 bits, and six of their nine products are summed, the small ones first (the others are below
// 2^-24).  The parts of the data are made by warps of their own: truncations, so that they
// add up to the value.  A pass moves 4 bytes per value like a bf16 pair, and 48 instructions a tile keep the tensor core
// below the copies' time.  21 x 45 x 80 tokens, 16 heads: forward transform 1.94 ms and inverse with the exchange 0.94
// (fp32 kernels: 4.46 and 2.83; 16-bit intermediates: 1.54 and 0.67).
// What bounds the passes that read fp32 is the way of a tile through its stage: copy, parts, instructions, 10 300 cycles
// with 128 channels.  A stage there holds only the rows in use and no third part, which lives from its making to the
// instructions and has two slots: three stages of 96 rows or less fit where two of 96 KB did, two of 128 rows still.  And eight
// warps make the parts instead of four (not beside the band split, whose epilogue needs the registers).  The first pass waited for
// its one staging area: it has two, and a stage less.  Six heads of that grid, the passes alone, us: w 176 -> 172 (6.1 TB/s),
// h 296 -> 245 (5.7), t with the band split 271 -> 264 (4.0), inverse t 96 -> 94, h 107 -> 89, w 107 -> 96; layers (16 heads 3640 ->
// 3474, eight of 7 x 90 x 127 tokens 1970 -> 1873).  With 64 channels the smaller stages lost (20 x 30 x 52 tokens, eight heads, 481 ->
// 501, 16 x 45 x 80, four, 487 -> 502; and two staging areas, 504 and 508): they keep four stages of whole tiles.  With few tiles a launch whose code no SM has run yet costs more than eight warps gain: the
// middle pass and the band split then share theirs, four warps in both (rule: FEW_TILES).
//
// Order of the tiles.  A pass that reads what the previous launch wrote walks its tiles from the last to the
// first (P.reverse), the next one forward again: the end of the previous launch's output is still in L2.
//
//   warp 0      TMA producer (ring of 2-8 stages)
//   warp 1      tcgen05.mma issuer (A from tensor memory), 3 accumulator buffers of 128 TMEM columns (2 beside three
//               matrix parts)
//   warps 2..9  epilogue: tcgen05.ld, convert to the output's form, store; a thread owns one output position
//   warps 10..13  (FORM_BYTES, FORM_EXACT) operands of an arriving tile; FORM_EXACT with 128 channels: 10..17
// Output path (FIRST, MIDDLE, LAST): an epilogue warp's 32 rows are 32 grid positions that form a
// box of the grid, so the warp writes 32 channels of them (64 bytes per row, 64-byte swizzle, no
// bank conflicts) into its own staging area and one lane sends them out with a tensor store; the
// area is reused when that store has read it.  SPLIT scatters rows to band positions: staged the
// same way, then stored by all lanes with four lanes per 64-byte row piece.
// Modes: FIRST  caller's Q/K/V -> intermediate
//        MIDDLE intermediate -> intermediate
//        SPLIT  intermediate -> band-major coefficient buffers (rank evaluated in registers): mid and
//               high band in bf16, low band in fp32 straight from the accumulators (hi/lo
//               intermediates carry 16 or 17 bits); the router's mid and high band energies are
//               accumulated here from the stored bf16 coefficients (the low band's, few values per
//               channel, by the band-statistics kernel from the fp32 coefficients)
//        LAST   intermediate -> the caller's out tensor
#include <cuda.h>

#include <vector>

#include "ff_clocks.cuh"
#include "ff_internal.h"
#include "ff_sm100.cuh"
#include "ff_three_byte.cuh"
#include "ff_two_buffers.h"

using namespace sm100;

namespace {

constexpr int CH_MAX = 128;                          // largest head_dim; shared-memory tiles are sized for it
constexpr int TILE_ROWS = 128;
constexpr int TILE_BYTES = TILE_ROWS * CH_MAX * 2; // 32 KB: 128 rows of bf16
constexpr int HALF_BYTES = TILE_BYTES / 2;
constexpr int MAX_STAGE = 8;

constexpr int NACC_MAX = 3;
constexpr int IMG_CELLS = 64;               // 32-bit tensor-memory cells per matrix row: two bf16 K elements each

// What a pass reads and, with it, the parts of its operands.
enum {
  FORM_PAIR,      // bf16: the caller's tensor, or a hi/lo pair of grids
  FORM_BYTES,     // a pair in the three-byte form
  FORM_EXACT1,    // any grid: the caller's bf16 tensor, handed on as fp32
  FORM_EXACT,     // any grid: an fp32 grid
  FORM_EXACT_SPLIT,  // ... and the band split follows (128 channels; with 64 it is a mode of FORM_EXACT)
  FORM_EXACT_FEW     // ... either of them (128 channels, few tiles)
};
template <int CH, int FORM> struct Shape {
  static constexpr bool any_grid = FORM >= FORM_EXACT1;
  static constexpr bool convert = FORM == FORM_BYTES || FORM >= FORM_EXACT;
  // TMA warp, MMA warp, 8 epilogue warps; then those that make operands of the data: 128 threads, with FORM_EXACT as many for
  // every 64 channels
  static constexpr int makers = !convert ? 0 : (FORM == FORM_EXACT ? 2 * CH : 128);
  static constexpr int threads = 320 + makers;
  static constexpr int parts = any_grid ? 3 : 2;           // of the matrix, 64 tensor-memory columns each
  static constexpr uint32_t col_acc = parts * 64;          // accumulator buffers of 128 columns behind them
  static constexpr int nacc = any_grid ? 2 : NACC_MAX;
  static_assert(col_acc + nacc * 128 <= 512, "tensor memory has 512 columns");
};

enum { MODE_FIRST = 0, MODE_MIDDLE = 1, MODE_SPLIT = 2, MODE_LAST = 3 };

struct DctTcParams {
  FFDims dm;
  const uint32_t* image;   // matrix image as the tensor-memory A operand: parts of [128][64] cells
  FFPassShape g;           // lines and tiles of the pass
  FFFastDiv by_tiles, by_inner;   // tiles of a tensor-head; tiles along the inner extent
  FFFastDiv by_line;       // (SPLIT) unravels a line index: by W for the t axis, by H for the w axis
  int axis;                // 0 = t, 1 = h, 2 = w
  int mode;
  int group;               // tensor-heads in this launch
  int group_start;         // index of the first one (tensor * BH + bh for the forward, bh for the inverse)
  int in_split;            // input is a hi/lo pair of grids (map0 = hi, map1 = lo)
  int out_lo8;             // the lo part of the output pair is one byte per value (see "Three-byte intermediates")
  int nstage;              // ring depth
  int early;               // the next launch comes in behind this one's wait, not when its blocks end
  int reverse;             // walk the tiles from the last to the first (what the previous launch wrote last is still in L2)
  __nv_bfloat16* spec_mid; __nv_bfloat16* spec_high;
  float* spec_low;         // MODE_SPLIT: [3 BH][N_low][d] fp32
  double* energy;          // (SPLIT) [B][3][CH], or NULL
  double* clear;           // (FIRST) band energies to clear for the sums that follow, or NULL
  int* status;
};

constexpr int STG_PITCH = 64;                       // bytes per staged row piece; the 16-byte chunks are rotated by row/2 against bank conflicts

struct DctShared {
  uint64_t full[MAX_STAGE], empty[MAX_STAGE], acc_full[NACC_MAX], acc_empty[NACC_MAX], conv[MAX_STAGE];
  uint64_t third_empty[2];                 // (F32) a slot of the third part has been read
  uint64_t stg_full[2][FFTwoBuffers::FULL], stg_free[2];       // (any grid) staging areas of four epilogue warps: written / read by the store
  uint32_t tmem_base;
  int abort_flag;
  int e_sample;            // (SPLIT) sample of the CTA's last tile
  // per epilogue warp: 32 rows x 64 bytes of hi and of lo, to turn one-row-per-thread registers
  // into stores where four lanes cover a row's 64 contiguous bytes
  alignas(1024) uint8_t stage[8][2][32 * STG_PITCH];
};

// (F32) rows of a tile in shared memory: whole k-steps.
__host__ __device__ constexpr int exact_rows(int rows) { return (rows + 15) / 16 * 16; }

// First line of tile `u` of a tensor-head: index along the inner extent and along the outer one.
__device__ __forceinline__ void tile_origin(const DctTcParams& P, unsigned u, int& i0, int& o0) {
  if (P.g.seq) { i0 = 0; o0 = (int)u * P.g.kf; }
  else { const unsigned o = ff_div(u, P.by_inner); o0 = (int)o; i0 = (int)(u - o * (unsigned)P.g.tiles_inner) * P.g.kf; }
}

// Three source maps (Q, K, V) in MODE_FIRST; otherwise map0 (= hi) and, for split input, map1 (= lo).
// map_oh / map_ol: destination hi / lo grids with the box of one epilogue warp (32 positions x 32
// channels), all modes but SPLIT; MODE_LAST and the EXACT forms have no lo grid.
// RAG (any grid): tiles of kf * n < 128 rows, or a last tile that is not full.  The rows past kf * n are zero in shared
// memory (cleared once, no copy writes them) and zero in the matrix; lines past the end of the grid arrive as zeros and
// are clipped by the stores.  32 rows are then no box of the grid, so the four warps of a channel half stage a
// whole tile (32 channels) and one thread stores it.
template <int CH, int FORM>
__global__ void __launch_bounds__(Shape<CH, FORM>::threads, 1)
dct_tc_kernel(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap map1,
              const __grid_constant__ CUtensorMap map2, const __grid_constant__ CUtensorMap map_oh,
              const __grid_constant__ CUtensorMap map_ol, const DctTcParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr bool LO8 = FORM == FORM_BYTES, F32 = FORM >= FORM_EXACT, RAG = Shape<CH, FORM>::any_grid, CONVERT = Shape<CH, FORM>::convert;
  constexpr int NACC = Shape<CH, FORM>::nacc, THREADS = Shape<CH, FORM>::threads;
  constexpr uint32_t COL_ACC = Shape<CH, FORM>::col_acc;
  const FFDims& dm = P.dm;
  const int n = P.g.n, kf = P.g.kf;                       // axis length, lines per tile
  const bool seq = P.g.seq;                               // lines follow one another (w axis) or interleave
  const int rows = RAG ? P.g.rows : TILE_ROWS;
  const int NSTAGE = P.nstage;
  const bool split = FORM == FORM_EXACT_SPLIT || ((FORM == FORM_PAIR || FORM == FORM_EXACT_FEW || (FORM == FORM_EXACT && CH == 64)) && P.mode == MODE_SPLIT);     // (the band-split pass never reads the byte form)
  const bool tma_out = !split;
  constexpr int TB = TILE_ROWS * CH * 2;                  // bytes of one data tile (16 KB for 64 channels)
  constexpr int LO8_OFF = CH == 128 ? TB : 2 * TB;         // where a stage takes the lo bytes
  // (F32) blocks of 128-byte rows, as many as the instructions read; the third part of the data has two slots of its own, or
  // lies behind the other two (64 channels: stages of whole tiles are small enough)
  constexpr bool SLOTS = F32 && CH == 128;
  const int RB = SLOTS ? exact_rows(rows) * 128 : HALF_BYTES, THIRD_BYTES = SLOTS ? RB * (CH / 64) : 0;
  const int STAGE_BYTES = LO8 ? LO8_OFF + TB / 2 + (CH == 128 ? TB / 2 : 0) : (SLOTS ? RB * (CH / 32) : F32 ? 3 * TB : (P.in_split ? 2 * TB : TB));   // hi tile, lo tile
  uint8_t* sData = smem;                                  // NSTAGE x STAGE_BYTES
  uint8_t* sThird = smem + NSTAGE * STAGE_BYTES;
  DctShared& sh = *(DctShared*)(sThird + 2 * THIRD_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned tiles_per_th = (unsigned)P.g.tiles;
  const int total_tiles = P.group * P.g.tiles;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSTAGE; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 1); mbar_init(&sh.conv[i], CONVERT ? Shape<CH, FORM>::makers : 1); }
    for (int i = 0; i < NACC; ++i) { mbar_init(&sh.acc_full[i], 1); mbar_init(&sh.acc_empty[i], 256); }
    if (RAG)
      for (int i = 0; i < 2; ++i) {
        for (int b = 0; b < FFTwoBuffers::FULL; ++b) mbar_init(&sh.stg_full[i][b], 128);
        mbar_init(&sh.stg_free[i], 1); mbar_init(&sh.third_empty[i], 1);
      }
    sh.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
  if (RAG) {                                              // rows that no copy writes must not hold NaN patterns
    for (int i = threadIdx.x * 16; i < NSTAGE * STAGE_BYTES + 2 * THIRD_BYTES; i += blockDim.x * 16) *(uint4*)(sData + i) = make_uint4(0, 0, 0, 0);
    fence_proxy_async();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sh.tmem_base;
  volatile int* abort_flag = &sh.abort_flag;

  if (warp >= 2 && warp < 6) {
    // The matrix (its bf16 parts) into tensor memory, where it is the A operand of every tile: a thread
    // loads the row of its lane (prepared at plan creation as pairs of bf16 K elements per 32-bit cell).
    const int quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
#pragma unroll 1
    for (int im = 0; im < Shape<CH, FORM>::parts; ++im) {
      const uint32_t* src = P.image + (size_t)im * FF_IMAGE_PART + (size_t)row * IMG_CELLS;
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
  if (P.early) ff_pdl_wait(); else ff_pdl_join();
  if (!CONVERT && P.clear && blockIdx.x == 0) for (int i = threadIdx.x; i < dm.B * 3 * CH; i += THREADS) P.clear[i] = 0.0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&map0);
      unsigned it = 0;
      bool ok = true;
      for (int sl = blockIdx.x; sl < total_tiles && ok; sl += gridDim.x, ++it) {
        const int s = P.reverse ? total_tiles - 1 - sl : sl;
        const int slot = it % NSTAGE;
        FF_CLOCK(pt);
        if (it >= (unsigned)NSTAGE) ok = mbar_wait(&sh.empty[slot], ((it / NSTAGE) - 1) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, P.mode * 16 + 6, pt);
        if (!ok) break;
        uint8_t* dst = sData + slot * STAGE_BYTES;
        const int gi = (int)ff_div((unsigned)s, P.by_tiles);
        int i0, o0; tile_origin(P, (unsigned)s - (unsigned)gi * tiles_per_th, i0, o0);
        const CUtensorMap* map = &map0;
        int slice = gi;
        if (P.mode == MODE_FIRST) {
          const int th = P.group_start + gi;
          const int tensor = (th >= dm.BH) + (th >= 2 * dm.BH);
          map = tensor == 0 ? &map0 : (tensor == 1 ? &map1 : &map2);
          slice = th - tensor * dm.BH;
        }
        mbar_arrive_expect_tx(&sh.full[slot], (uint32_t)(rows * CH) * (LO8 ? 3u : (F32 || P.in_split ? 4u : 2u)));
        if (F32) {                                         // blocks of 32 channels: rows of 128 bytes
#pragma unroll
          for (int b = 0; b < CH / 32; ++b) tma_load_5d(dst + b * RB, map, &sh.full[slot], 32 * b, i0, 0, o0, slice);
          continue;
        }
        tma_load_5d(dst, map, &sh.full[slot], 0, i0, 0, o0, slice);
        if (CH == 128) tma_load_5d(dst + HALF_BYTES, map, &sh.full[slot], 64, i0, 0, o0, slice);
        if (LO8) {
          tma_load_5d(dst + LO8_OFF, &map1, &sh.full[slot], 0, i0, 0, o0, slice);     // the lo bytes: rows of CH bytes
        } else if (P.in_split) {
          tma_load_5d(dst + TB, &map1, &sh.full[slot], 0, i0, 0, o0, slice);
          if (CH == 128) tma_load_5d(dst + TB + HALF_BYTES, &map1, &sh.full[slot], 64, i0, 0, o0, slice);
        }
      }
    }
  } else if (warp == 1) {
    {
      const uint32_t idesc = idesc_bf16_f32(TILE_ROWS, CH, /*a_mn_major=*/false, /*b_mn_major=*/true);
      unsigned it = 0;
      bool ok = true;
      for (int sl = blockIdx.x; sl < total_tiles && ok; sl += gridDim.x, ++it) {
        const int slot = it % NSTAGE, ab = it % NACC;
        FF_CLOCK(pm);
        ok = mbar_wait_warp(CONVERT ? &sh.conv[slot] : &sh.full[slot], (it / NSTAGE) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, P.mode * 16 + 2, pm);
        FF_CLOCK(pm2);
        if (ok && it >= NACC) ok = mbar_wait_warp(&sh.acc_empty[ab], ((it / NACC) - 1) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, P.mode * 16 + 3, pm2);
        if (!ok) break;
        tc_fence_after();
        const uint32_t dbase = smem_u32(sData + slot * STAGE_BYTES);
        const uint32_t d_tm = tm + COL_ACC + ab * 128;
        const int ksteps = (rows + 15) >> 4;               // (the rows behind them are zero)
        // k-steps of matrix part `part` times the operand at `x` (a descriptor advances by 2048 bytes = 128 in its address
        // field per 16 rows of K)
        auto product = [&](int part, uint64_t x, bool first) {
#pragma unroll
          for (int ks = 0; ks < TILE_ROWS / 16; ++ks)
            if (ks < ksteps) umma_ts(d_tm, tm + part * 64 + ks * 8, x + (uint64_t)(ks * 128), idesc, first && ks == 0 ? 0u : 1u);
        };
        if (F32) {
          // (the halves of 64 channels of the first two parts alternate, those of the third follow one another)
          const uint64_t x0 = smem_desc_sw128(dbase, 2 * RB, 1024), x1 = smem_desc_sw128(dbase + RB, 2 * RB, 1024);
          const uint64_t x2 = smem_desc_sw128(SLOTS ? smem_u32(sThird + (it & 1) * THIRD_BYTES) : dbase + 2 * TB, RB, 1024);
          product(2, x0, true);
          product(1, x1, false);
          product(0, x2, false);
          product(1, x0, false);
          product(0, x1, false);
          product(0, x0, false);
        } else if (RAG) {
          const uint64_t x = smem_desc_sw128(dbase, HALF_BYTES, 1024);
          product(2, x, true);
          product(1, x, false);
          product(0, x, false);
        } else {
          const uint64_t xh0 = smem_desc_sw128(dbase, HALF_BYTES, 1024), xl0 = smem_desc_sw128(dbase + TB, HALF_BYTES, 1024);
#pragma unroll
          for (int ks = 0; ks < TILE_ROWS / 16; ++ks) {
            umma_ts(d_tm, tm + ks * 8, xh0 + (uint64_t)(ks * 128), idesc, ks > 0 ? 1u : 0u);
            umma_ts(d_tm, tm + 64 + ks * 8, xh0 + (uint64_t)(ks * 128), idesc, 1u);
            if (P.in_split) umma_ts(d_tm, tm + ks * 8, xl0 + (uint64_t)(ks * 128), idesc, 1u);
          }
        }
        umma_commit(&sh.empty[slot]);
        if (SLOTS) umma_commit(&sh.third_empty[it & 1]);
        umma_commit(&sh.acc_full[ab]);
      }
    }
  } else if (F32 && warp >= 10) {
    // ------------------------------------------------------------------ fp32 -> three bf16 parts, in place
    // A thread owns 64 channels of a row of the tile: they arrive in two blocks of 32 channels, the first and the
    // second part go where they were (64 channels a block), the third part into its slot; all with the 128-byte swizzle.
    const int r0 = (threadIdx.x - 320) & 127, h0 = (threadIdx.x - 320) >> 7;
    unsigned it = 0;
    bool ok = true;
    for (int sl = blockIdx.x; sl < total_tiles && ok; sl += gridDim.x, ++it) {
      const int slot = it % NSTAGE;
      FF_CLOCK(pc0);
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[slot], (it / NSTAGE) & 1, abort_flag));
      if (SLOTS && ok && it >= 2) ok = mbar_wait_warp(&sh.third_empty[it & 1], ((it >> 1) - 1) & 1, abort_flag);
      FF_CLOCK_ADD(threadIdx.x == 320, P.mode * 16 + 0, pc0);
      if (!ok) break;
      FF_CLOCK(pc1);
      if (r0 < rows) {
#pragma unroll 1
        for (int h = h0; h < CH / 64; h += Shape<CH, FORM>::makers / 128) {
          uint8_t* b0 = sData + slot * STAGE_BYTES + h * 2 * RB + r0 * 128;
          uint8_t* b2 = (SLOTS ? sThird + (it & 1) * THIRD_BYTES : sData + slot * STAGE_BYTES + 2 * TB) + h * RB + r0 * 128;
          // The first 32 channels go to registers.  Then eight channels at a time, those of the second block from its end, so
          // that no chunk is written before it has been read.
          uint4 x[8];                                      // four channels each
#pragma unroll
          for (int c = 0; c < 8; ++c) x[c] = *(const uint4*)(b0 + ((c ^ (r0 & 7)) << 4));
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int c = k < 4 ? 7 - k : k - 4;           // 16-byte chunk of each part
            uint4 xa, xb;
            if (c >= 4) {
              xa = *(const uint4*)(b0 + RB + (((2 * c - 8) ^ (r0 & 7)) << 4));
              xb = *(const uint4*)(b0 + RB + (((2 * c - 7) ^ (r0 & 7)) << 4));
            } else {
              xa = x[2 * (c & 3)]; xb = x[2 * (c & 3) + 1];
            }
            const uint32_t v[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
            uint32_t p0[4], p1[4], p2[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint32_t va = v[2 * i], vb = v[2 * i + 1];
              const uint32_t ra = __float_as_uint(__uint_as_float(va) - __uint_as_float(va & 0xffff0000u));
              const uint32_t rb = __float_as_uint(__uint_as_float(vb) - __uint_as_float(vb & 0xffff0000u));
              const float ta = __uint_as_float(ra) - __uint_as_float(ra & 0xffff0000u), tb = __uint_as_float(rb) - __uint_as_float(rb & 0xffff0000u);
              p0[i] = __byte_perm(va, vb, 0x7632);
              p1[i] = __byte_perm(ra, rb, 0x7632);
              p2[i] = __byte_perm(__float_as_uint(ta), __float_as_uint(tb), 0x7632);
            }
            const uint32_t off = (uint32_t)((c ^ (r0 & 7)) << 4);
            *(uint4*)(b0 + off) = make_uint4(p0[0], p0[1], p0[2], p0[3]);
            *(uint4*)(b0 + RB + off) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
            *(uint4*)(b2 + off) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
          }
        }
      }
      fence_proxy_async();
      mbar_arrive(&sh.conv[slot]);
      FF_CLOCK_ADD(threadIdx.x == 320, P.mode * 16 + 1, pc1);
    }
  } else if (LO8 && warp >= 10) {
    // ------------------------------------------------------------------ lo bytes -> bf16 lo operand
    // A thread owns a row of the tile.  For every value v24 = (hi << 16) | (byte << 8) as fp32: lo = v24 - hi =
    // +-byte 2^(E-15) with hi's sign and exponent E, exact in bf16.  A byte in the low half of a bf16 is byte 2^-133
    // (below 128 as a subnormal number), so two packed multiplications give two values: by 2^118, and by hi without
    // its mantissa (+-2^E).  Four instructions a pair; as two fp32 differences and a conversion it took eight.  The bytes arrive as rows of CH bytes (128-byte swizzle for 128 channels, 64-byte for 64),
    // the bf16 tiles as 64-channel halves of 128-byte rows (128-byte swizzle).
    const int r0 = threadIdx.x - 320;
    const __nv_bfloat162 up = __float2bfloat162_rn(0x1p118f);
    unsigned it = 0;
    bool ok = true;
    for (int sl = blockIdx.x; sl < total_tiles && ok; sl += gridDim.x, ++it) {
      const int slot = it % NSTAGE;
      FF_CLOCK(pc0);
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.full[slot], (it / NSTAGE) & 1, abort_flag));
      FF_CLOCK_ADD(threadIdx.x == 320, P.mode * 16 + 0, pc0);
      if (!ok) break;
      FF_CLOCK(pc1);
      uint8_t* base = sData + slot * STAGE_BYTES;
#pragma unroll 1
      for (int r = r0; r < TILE_ROWS; r += 128) {
      // 128 channels: the bytes arrive where the bf16 lo tile goes, row r's 128 bytes inside the first half of its
      // own bf16 row, so a thread takes them into registers before it writes the row (no other thread touches
      // it).  64 channels: the bytes have their own 8 KB behind the two tiles.
      const uint8_t* lob = base + LO8_OFF + r * CH;
      uint32_t lw[CH / 4];
#pragma unroll
      for (int cc = 0; cc < CH / 16; ++cc) {                 // 16-byte chunk cc of the row (16 channels)
        const int pc = CH == 128 ? (cc ^ (r & 7)) : (cc ^ ((r >> 1) & 3));
        const uint4 lb = *(const uint4*)(lob + (pc << 4));
        lw[4 * cc] = lb.x; lw[4 * cc + 1] = lb.y; lw[4 * cc + 2] = lb.z; lw[4 * cc + 3] = lb.w;
      }
#pragma unroll
      for (int c8 = 0; c8 < CH / 8; ++c8) {                  // 8-channel chunk of the row: one 16-byte chunk of bf16
        const uint32_t off = (uint32_t)(c8 >> 3) * HALF_BYTES + (uint32_t)r * 128 + (uint32_t)(((c8 & 7) ^ (r & 7)) << 4);
        const uint4 hv = *(const uint4*)(base + off);
        const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
        uint32_t ow[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t b2 = __byte_perm(lw[2 * c8 + (i >> 1)], 0u, (i & 1) ? 0x4342 : 0x4140);     // 0x00b1'00b0
          const uint32_t e2 = hw[i] & 0xff80ff80u;
          const __nv_bfloat162 lp = __hmul2(__hmul2(*(const __nv_bfloat162*)&b2, up), *(const __nv_bfloat162*)&e2);
          ow[i] = *(const uint32_t*)&lp;
        }
        *(uint4*)(base + TB + off) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
      }
      }
      fence_proxy_async();
      mbar_arrive(&sh.conv[slot]);
      FF_CLOCK_ADD(threadIdx.x == 320, P.mode * 16 + 1, pc1);
    }
  } else {
    const int quarter = warp & 3;
    const int j = quarter * 32 + lane;                    // output position of this thread inside a tile
    const int a = seq ? j % n : j / kf;                   // output index along the axis
    const int l = seq ? j / n : j % kf;                   // line of the tile
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int ew = warp - 2;                              // epilogue warp 0..7: warps 0-3 take channels 0..63, 4-7 channels 64..127
    constexpr int NQ = CH / 64;                           // 32-channel chunks per thread
    const int q_lo = (ew >> 2) * NQ;
    // Position along the axis and line of the warp's first row (tile row 32 quarter): the warp's 32
    // rows are the box [32 channels] x [from there .. + the extents the store map was built with]
    const int j0 = quarter * 32;
    const int a0 = seq ? j0 % n : j0 / kf, l0 = seq ? j0 / n : j0 % kf;
    unsigned nchunk = 0;                                  // (any grid) chunks this channel half has staged
    const int Lhw = dm.L[1] * dm.L[2], Mhw = dm.M[1] * dm.M[2];
    // (SPLIT) lane k of a warp accumulates the energies of channels 32 q + 2 (k % 16) + {0, 1} over the
    // warp's rows of parity k / 16: ea = mid + high rows, em = mid rows
    float ea[NQ][2] = {}, em[NQ][2] = {};                 // [chunk of the thread][channel of the pair]
    int e_sample = -1, sample_th = -1, sample_of_th = 0;
    unsigned it = 0;
    bool ok = true;
    auto flush_energy = [&]() {
      if (!LO8 && e_sample >= 0 && P.energy) {
#pragma unroll
        for (int qi = 0; qi < NQ; ++qi)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int c = (q_lo + qi) * 32 + 2 * (lane & 15) + e;
            atomicAdd(P.energy + ((size_t)e_sample * 3 + 1) * CH + c, (double)em[qi][e]);
            atomicAdd(P.energy + ((size_t)e_sample * 3 + 2) * CH + c, (double)(ea[qi][e] - em[qi][e]));
            ea[qi][e] = em[qi][e] = 0.f;
          }
      }
    };
    for (int sl = blockIdx.x; sl < total_tiles && ok; sl += gridDim.x, ++it) {
      const int s = P.reverse ? total_tiles - 1 - sl : sl;
      const int ab = it % NACC;
      FF_CLOCK(pe0);
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.acc_full[ab], (it / NACC) & 1, abort_flag));
      FF_CLOCK_ADD(threadIdx.x == 64, P.mode * 16 + 4, pe0);
      if (!ok) break;
      tc_fence_after();
      FF_CLOCK(pe1);
      const int gi = (int)ff_div((unsigned)s, P.by_tiles);
      int i0, o0; tile_origin(P, (unsigned)s - (unsigned)gi * tiles_per_th, i0, o0);
      const int th = P.group_start + gi;
      const int tensor = (th >= dm.BH) + (th >= 2 * dm.BH), bh = th - tensor * dm.BH;
      // where this thread's row goes
      __nv_bfloat16* row_hi = nullptr; float* row_f32 = nullptr;
      int band = -1;
      if (split) {
        if (th != sample_th) { sample_th = th; sample_of_th = bh / dm.heads; }
        const int sample = sample_of_th;
        if (sample != e_sample) { flush_energy(); e_sample = sample; }
        // Band and rank of this row's coefficient: the pass axis supplies index a, the line the other two.
        // The counts of box members below a coefficient are piecewise linear in the coordinates.
        int kt = a, h_ = a, ww = a;
        bool inside = true;
        if (P.axis == 0) {
          const unsigned line = (unsigned)(i0 + l);
          h_ = (int)ff_div(line, P.by_line); ww = (int)(line - (unsigned)h_ * P.by_line.d);
          if (RAG) inside = j < rows && (int)line < P.g.inner;
        } else if (P.axis == 1) {
          kt = o0; ww = i0 + l;
          if (RAG) inside = j < rows && ww < dm.W;
        } else {
          const unsigned line = (unsigned)(o0 + l);
          kt = (int)ff_div(line, P.by_line); h_ = (int)(line - (unsigned)kt * P.by_line.d);
          if (RAG) inside = j < rows && (int)line < P.g.outer;
        }
        const bool hw_low = h_ < dm.L[1] && ww < dm.L[2], hw_mid = h_ < dm.M[1] && ww < dm.M[2];
        const int offM = (h_ < dm.M[1] ? h_ : dm.M[1]) * dm.M[2] + (h_ < dm.M[1] ? (ww < dm.M[2] ? ww : dm.M[2]) : 0);
        // (axis lengths are at most 128, so every count fits 32 bits)
        const int cm = kt < dm.M[0] ? kt * Mhw + offM : dm.M[0] * Mhw;
        const size_t th_slice = (size_t)tensor * dm.BH + bh;
        long long rk = 0, nband = 1;                                                 // band-local rank, band length
        if (RAG && !inside) {
          kt = h_ = ww = 0;                                                          // no position of the grid: not stored
        } else if (kt < dm.L[0] && hw_low) {
          band = 0;                                                                  // low band: fp32
          rk = (kt * dm.L[1] + h_) * dm.L[2] + ww; nband = dm.Nlow;
          row_f32 = P.spec_low + (th_slice * dm.Nlow + (unsigned)rk) * CH;
        } else if (kt < dm.M[0] && hw_mid) {
          const int offL = (h_ < dm.L[1] ? h_ : dm.L[1]) * dm.L[2] + (h_ < dm.L[1] ? (ww < dm.L[2] ? ww : dm.L[2]) : 0);
          const int cl = kt < dm.L[0] ? kt * Lhw + offL : (int)dm.Nlow;
          band = 1;
          rk = cm - cl; nband = dm.Nmid;
          row_hi = P.spec_mid + (th_slice * dm.Nmid + (unsigned)rk) * CH;
        } else {
          band = 2;
          rk = ((kt * dm.H + h_) * dm.W + ww) - cm; nband = dm.Nhigh;
          row_hi = P.spec_high + (th_slice * dm.Nhigh + (unsigned)rk) * CH;
        }
        // (debug build) the rank must lie inside its band and the coordinates inside the grid
        if (!FF_DBG_OK(kt >= 0 && kt < dm.T && h_ >= 0 && h_ < dm.H && ww >= 0 && ww < dm.W && rk >= 0 && rk < nband &&
                       th_slice < (size_t)3 * dm.BH, P.status, 2)) {
          row_hi = nullptr; row_f32 = nullptr; band = -1;
        }
      }
      // (SPLIT) lane L stores for rows 8 i + L/4 of its warp: fetch those rows' destinations
      __nv_bfloat16* dst_hi[4];
      if (split)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int src = 8 * i + (lane >> 2);
        dst_hi[i] = (__nv_bfloat16*)__shfl_sync(0xffffffffu, (unsigned long long)row_hi, src);
      }
      const int out_slice = P.mode == MODE_LAST ? th : gi;
      const unsigned nonlow_rows = __ballot_sync(0xffffffffu, band > 0), mid_rows = __ballot_sync(0xffffffffu, band == 1);
      // both 32-channel chunks of the row at once; the accumulator buffer is free as soon as they are read
      constexpr bool EACH = FORM >= FORM_EXACT_SPLIT;      // (for want of registers one after the other)
      uint32_t rr2[EACH ? 1 : NQ][32];
      if (!EACH) {
        FF_CLOCK(pl);
#pragma unroll
        for (int qi = 0; qi < NQ; ++qi) tmem_ld32(tm + lane_addr + COL_ACC + ab * 128 + (q_lo + qi) * 32, rr2[EACH ? 0 : qi]);
        tmem_wait_ld();
        FF_CLOCK_ADD(threadIdx.x == 64, P.mode * 16 + 8, pl);
        tc_fence_before();
        mbar_arrive(&sh.acc_empty[ab]);
      }
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi) {
        const int q = q_lo + qi;
        uint32_t (&r)[32] = rr2[EACH ? 0 : qi];
        if (EACH) {
          tmem_ld32(tm + lane_addr + COL_ACC + ab * 128 + q * 32, r);
          tmem_wait_ld();
          if (qi == NQ - 1) { tc_fence_before(); mbar_arrive(&sh.acc_empty[ab]); }
        }
        if (!LO8 && row_f32) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *(uint4*)(row_f32 + q * 32 + i * 4) = make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
        }
        if (RAG && tma_out) {
          // four warps stage one tile, 32 channels of 128 rows: fp32 in rows of 128 bytes (128-byte swizzle), or the caller's
          // bf16 in rows of 64 (64-byte swizzle).  (Two areas of half the size in turn: 3470 against 3300 us for the
          // 76K-token layer; two whole ones for the bf16 rows: 96 -> 103 us.)
          const int grp = ew >> 2;
          // The first pass has two areas in turn (the second pair behind the barriers) and five instead of six stages.
          constexpr bool TWO = FORM == FORM_EXACT1 && CH == 128;
          uint8_t* area = TWO && FFTwoBuffers::buffer(nchunk) ? (uint8_t*)(&sh + 1) + grp * HALF_BYTES : sh.stage[grp * 4][0];
          uint64_t* filled = &sh.stg_full[grp][TWO ? FFTwoBuffers::full(nchunk) : 0];
          if (TWO ? FFTwoBuffers::waits_free(nchunk) : nchunk > 0) {
            if (quarter == 0 && lane == 0) {
              if (TWO) bulk_wait_read1(); else bulk_wait_read0();
              mbar_arrive(&sh.stg_free[grp]);
            }
            ok = __all_sync(0xffffffffu, mbar_wait(&sh.stg_free[grp], TWO ? FFTwoBuffers::free_parity(nchunk) : (nchunk - 1) & 1, abort_flag));
            if (!ok) break;
          }
          if (FORM == FORM_EXACT1 || P.mode == MODE_MIDDLE) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              *(uint4*)(area + j * 128 + ((i ^ (j & 7)) << 4)) = make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              uint32_t w[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) w[k] = bf16_pair(r[8 * i + 2 * k], r[8 * i + 2 * k + 1]);
              *(uint4*)(area + j * STG_PITCH + ((i ^ ((j >> 1) & 3)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
          fence_proxy_async();
          mbar_arrive(filled);
          if (quarter == 0) {
            ok = __all_sync(0xffffffffu, mbar_wait(filled, TWO ? FFTwoBuffers::full_parity(nchunk) : nchunk & 1, abort_flag));
            if (!ok) break;
            if (lane == 0) {
              tma_store_5d(area, &map_oh, q * 32, i0, 0, o0, out_slice);
              bulk_commit();
            }
            __syncwarp();
          }
          ++nchunk;
        } else {
          const bool want_lo = !RAG && (P.mode == MODE_FIRST || P.mode == MODE_MIDDLE);
          const bool lo8 = want_lo && P.out_lo8;
          uint32_t hi[16], lo[16];
          if (lo8) {
#pragma unroll
            for (int i = 0; i < 32; ++i) r[i] = ff_round24(r[i]);
#pragma unroll
            for (int i = 0; i < 16; ++i) hi[i] = ff_hi2(r[2 * i], r[2 * i + 1]);
#pragma unroll
            for (int i = 0; i < 8; ++i) lo[i] = ff_lo4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) hi[i] = bf16_pair(r[2 * i], r[2 * i + 1]);
          }
          if (want_lo && !lo8) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const __nv_bfloat162 lp = __floats2bfloat162_rn(__uint_as_float(r[2 * i]) - __uint_as_float(hi[i] << 16),
                                                             __uint_as_float(r[2 * i + 1]) - __uint_as_float(hi[i] & 0xffff0000u));
              lo[i] = *(const uint32_t*)&lp;
            }
          }
          uint8_t* st_hi = sh.stage[ew][0];
          uint8_t* st_lo = sh.stage[ew][1];
          if (tma_out) {
            // the previous store of this warp must have read the staging area
            FF_CLOCK(pw);
            if (lane == 0) bulk_wait_read0();
            __syncwarp();
            FF_CLOCK_ADD(threadIdx.x == 64, P.mode * 16 + 7, pw);
          }
          // 16-byte chunk i of row `lane` at chunk position i ^ (lane / 2 % 4): the 64-byte swizzle
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            *(uint4*)(st_hi + lane * STG_PITCH + ((i ^ ((lane >> 1) & 3)) << 4)) = make_uint4(hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
            if (want_lo && !lo8)
              *(uint4*)(st_lo + lane * STG_PITCH + ((i ^ ((lane >> 1) & 3)) << 4)) = make_uint4(lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
          }
          if (lo8) {                                        // 32 bytes per row, rows 32 bytes apart (no swizzle)
            *(uint4*)(st_lo + lane * 32) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            *(uint4*)(st_lo + lane * 32 + 16) = make_uint4(lo[4], lo[5], lo[6], lo[7]);
          }
          if (tma_out) {
            FF_CLOCK(pf);
            fence_proxy_async();
            __syncwarp();
            FF_CLOCK_ADD(threadIdx.x == 64, P.mode * 16 + 10, pf);
            if (lane == 0) {
              tma_store_5d(st_hi, &map_oh, q * 32, i0 + (seq ? 0 : l0), a0, o0 + (seq ? l0 : 0), out_slice);
              if (want_lo) tma_store_5d(st_lo, &map_ol, q * 32, i0 + (seq ? 0 : l0), a0, o0 + (seq ? l0 : 0), out_slice);
              bulk_commit();
            }
          } else if (!LO8) {
            __syncwarp();
            if (P.energy) {
              // Router statistics: channel energies of the staged (bf16) coefficients, summed down the
              // columns of the warp's 32 x 32 block; a lane reads one channel pair of every other row.
              const int par = lane >> 4, cp = lane & 15;
              float a0 = 0.f, a1 = 0.f, m0 = 0.f, m1 = 0.f;
              if (nonlow_rows == 0xffffffffu && (mid_rows == 0u || mid_rows == 0xffffffffu)) {
                // (almost every block: its 32 rows lie in one band, mid or high)
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  const uint32_t wd = *(const uint32_t*)(st_hi + (2 * i + par) * STG_PITCH + (((cp >> 2) ^ (i & 3)) << 4) + (cp & 3) * 4);
                  const float v0 = __uint_as_float(wd << 16), v1 = __uint_as_float(wd & 0xffff0000u);
                  a0 = fmaf(v0, v0, a0); a1 = fmaf(v1, v1, a1);
                }
                if (mid_rows) { m0 = a0; m1 = a1; }
              } else {
                const unsigned nl = nonlow_rows >> par, md = mid_rows >> par;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  const uint32_t wd = *(const uint32_t*)(st_hi + (2 * i + par) * STG_PITCH + (((cp >> 2) ^ (i & 3)) << 4) + (cp & 3) * 4);
                  const float v0 = __uint_as_float(wd << 16), v1 = __uint_as_float(wd & 0xffff0000u);
                  const float s0 = v0 * v0, s1 = v1 * v1;
                  if ((nl >> (2 * i)) & 1) { a0 += s0; a1 += s1; }
                  if ((md >> (2 * i)) & 1) { m0 += s0; m1 += s1; }
                }
              }
              ea[qi][0] += a0; ea[qi][1] += a1; em[qi][0] += m0; em[qi][1] += m1;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int rr = 8 * i + (lane >> 2), piece = lane & 3;      // row of the warp, 16-byte piece of its 64 bytes
              if (dst_hi[i]) *(uint4*)(dst_hi[i] + q * 32 + piece * 8) = *(const uint4*)(st_hi + rr * STG_PITCH + ((piece ^ ((rr >> 1) & 3)) << 4));
            }
            __syncwarp();
          }
        }
      }
      FF_CLOCK_ADD(threadIdx.x == 64, P.mode * 16 + 5, pe1);
    }
    if (split && P.energy) {
      // the CTA's last sample: the warp's sums into its staging area ([row parity][band][channel of the half]),
      // added up below with one atomic per channel and CTA (1184 atomics per address took 40 us at the kernel's end)
      if (lane == 0 && ew == 0) sh.e_sample = e_sample;
      float* part = (float*)sh.stage[ew] + (lane >> 4) * CH;
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int c = qi * 32 + 2 * (lane & 15) + e;
          part[c] = em[qi][e];
          part[CH / 2 + c] = ea[qi][e] - em[qi][e];
        }
    }
    if (tma_out && lane == 0) bulk_wait0();
  }

  tc_fence_before();
  __syncthreads();
  if (split && P.energy && threadIdx.x < 2 * CH && sh.e_sample >= 0) {
    const int band = threadIdx.x / CH, half = threadIdx.x % CH / (CH / 2), c = threadIdx.x % (CH / 2);
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += (double)((const float*)sh.stage[half * 4 + (i >> 1)])[(i & 1) * CH + band * (CH / 2) + c];
    atomicAdd(P.energy + ((size_t)sh.e_sample * 3 + 1) * CH + threadIdx.x, s);     // mid band, then high band
  }
  if (sh.abort_flag) {
    if (threadIdx.x == 0) atomicExch(P.status, FF_ERR_TIMEOUT | 0x200);   // low byte: status, next byte: which kernel
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

enum { T_BF16, T_BYTE, T_F32 };
// 5-D map over a grid [slices][outer][n][inner][d] seen along `axis`.  Load map: the box is one tile, kf whole lines of
// 64 (bf16), 32 (fp32) or all channels (bytes: the lo part of the three-byte form), 128-byte rows but for the 64 bytes of
// head_dim 64.  Store map: 32 channels of what one epilogue warp holds (tile rows 32 q .. 32 q + 31), or of a whole tile
// where 32 rows are not a box of the grid.
bool encode_map(CUtensorMap* map, const void* base, const FFDims& dm, int slices, int axis, int type, bool store) {
  const FFPassShape g = ff_pass_shape(dm, axis);
  const cuuint64_t CH = (cuuint64_t)dm.d, eb = type == T_BYTE ? 1 : (type == T_BF16 ? 2 : 4);
  const cuuint64_t line = (cuuint64_t)g.inner * CH * eb;
  cuuint64_t dims[5] = {CH, (cuuint64_t)g.inner, (cuuint64_t)g.n, (cuuint64_t)g.outer, (cuuint64_t)slices};
  cuuint64_t strides[4] = {CH * eb, line, line * g.n, (cuuint64_t)dm.N * CH * eb};
  cuuint32_t box[5] = {store || type == T_F32 ? 32u : (type == T_BYTE ? (cuuint32_t)dm.d : 64u), (cuuint32_t)(g.seq ? 1 : g.kf), (cuuint32_t)g.n,
                       (cuuint32_t)(g.seq ? g.kf : 1), 1};
  if (store && !ff_fp32_grid(dm)) {        // 32 consecutive tile rows
    if (g.seq) { box[2] = (cuuint32_t)(g.n < 32 ? g.n : 32); box[3] = (cuuint32_t)(g.n < 32 ? 32 / g.n : 1); }
    else { box[1] = (cuuint32_t)(g.kf < 32 ? g.kf : 32); box[2] = (cuuint32_t)(g.kf < 32 ? 32 / g.kf : 1); }
  }
  const cuuint32_t row = box[0] * (cuuint32_t)eb;      // bytes of a row in shared memory
  const CUtensorMapSwizzle swz = row == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (row == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE);
  const CUtensorMapDataType element = type == T_BYTE ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                      : type == T_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  return ff_encode_map(map, element, 5, base, dims, strides, box, swz,
                       store ? CU_TENSOR_MAP_L2_PROMOTION_NONE : CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}
// (through the plan's cache)
bool map_for(ff_plan* p, CUtensorMap* map, const void* base, int slices, int axis, int type, bool store) {
  return p->maps.get(map, base, axis | (type << 2) | (store ? 16 : 0), slices,
                     [&] { return encode_map(map, base, p->dm, slices, axis, type, store); });
}
bool grid_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, int axis, int type = T_BF16) {
  return map_for(p, map, base, slices, axis, type, false);
}
bool store_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, int axis, int type = T_BF16) {
  return map_for(p, map, base, slices, axis, type, true);
}

// `form`: what the pass reads.
cudaError_t launch_pass(ff_plan* p, const CUtensorMap& m0, const CUtensorMap& m1, const CUtensorMap& m2,
                        const CUtensorMap& moh, const CUtensorMap& mol, DctTcParams& P, int form, cudaStream_t st) {
  P.g = ff_pass_shape(P.dm, P.axis);
  const size_t tile = (size_t)TILE_ROWS * P.dm.d * 2, third = form >= FORM_EXACT && P.dm.d == 128 ? (size_t)exact_rows(P.g.rows) * P.dm.d * 2 : 0;
  const size_t stage = third ? 2 * third : form >= FORM_EXACT ? 3 * tile : (form == FORM_BYTES ? (P.dm.d == 128 ? 2 * tile : 2 * tile + tile / 2) : (size_t)(P.in_split ? 2 : 1) * tile);
  const size_t second = form == FORM_EXACT1 && P.dm.d == 128 ? 2 * HALF_BYTES : 0;      // the second pair of staging areas
  const size_t fixed = sizeof(DctShared) + 1024 + 2 * third + second;
  int nstage = (int)((232448 - 256 - fixed) / stage);   // 227 KB of shared memory per CTA
  if (nstage > MAX_STAGE) nstage = MAX_STAGE;
  P.nstage = nstage;
  // (see ff_internal.h; any other grid: level)
  P.early = ff_fp32_grid(P.dm) || p->masks_given;
  const size_t smem = nstage * stage + fixed;
  P.by_tiles = ff_fast_div((unsigned)P.g.tiles); P.by_inner = ff_fast_div((unsigned)P.g.tiles_inner);
  P.by_line = ff_fast_div((unsigned)(P.axis == 2 ? P.dm.H : P.dm.W));
  const int tiles = P.group * P.g.tiles;
  const int grid = tiles < p->sm_count ? tiles : p->sm_count;
  cudaError_t e;
#define FF_DCT(D, F) e = ff_launch(dct_tc_kernel<D, F>, dim3(grid), dim3(Shape<D, F>::threads), smem, st, m0, m1, m2, moh, mol, P)
#define FF_DCT_D(F) do { if (P.dm.d == 128) FF_DCT(128, F); else FF_DCT(64, F); } while (0)
  switch (form) {
    case FORM_PAIR: FF_DCT_D(FORM_PAIR); break;
    case FORM_BYTES: FF_DCT_D(FORM_BYTES); break;
    case FORM_EXACT1: FF_DCT_D(FORM_EXACT1); break;
    case FORM_EXACT: FF_DCT_D(FORM_EXACT); break;
    case FORM_EXACT_SPLIT: FF_DCT(128, FORM_EXACT_SPLIT); break;
    default: FF_DCT(128, FORM_EXACT_FEW);
  }
#undef FF_DCT_D
#undef FF_DCT
  if (e != cudaSuccess) return e;
  p->launches += 1;
  return cudaSuccess;
}

}  // namespace

// Any grid, 128 channels: tiles an SM of the middle pass, all tensor-heads together, up to which it and the band split run the
// same code.  Layers, us, each its own / the same (tiles): 5 x 33 x 20 tokens, eight heads, all bands 159.5 / 154.0 (6); 12 x 40 x 100,
// one 231.7 / 222.9 (8), two 354.4 / 350.1 (16); 21 x 45 x 80, one 297.2 / 285.9 (17).  10 x 50 x 110, two 403.6 / 399.2 (22),
// 48 x 24 x 60, two 490.1 / 494.0 (23), 21 x 45 x 80, two, routed 471.2 / 476.7 (34), four 994.5 / 1004.7 (68).
constexpr int FEW_TILES = 20;
static bool few_tiles(const FFDims& dm, int sm_count) {
  return dm.d == 128 && 3LL * dm.BH * ff_pass_shape(dm, 1).tiles <= (long long)FEW_TILES * sm_count;
}

cudaError_t ffk_dct_tc_init(const FFDims& dm, int sm_count) {
  cudaError_t e = cudaSuccess;
#define FF_DCT(D, F) \
  if (e == cudaSuccess && dm.d == D) e = cudaFuncSetAttribute(dct_tc_kernel<D, F>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448 - 256)
  if (!ffk_dct_tc_supported(dm)) return e;
  if (ff_fp32_grid(dm)) {
    FF_DCT(128, FORM_EXACT1); FF_DCT(128, FORM_EXACT); FF_DCT(64, FORM_EXACT1); FF_DCT(64, FORM_EXACT);
    if (few_tiles(dm, sm_count)) { FF_DCT(128, FORM_EXACT_FEW); } else { FF_DCT(128, FORM_EXACT_SPLIT); }
  } else { FF_DCT(128, FORM_PAIR); FF_DCT(128, FORM_BYTES); FF_DCT(64, FORM_PAIR); FF_DCT(64, FORM_BYTES); }
#undef FF_DCT
  return e;
}

// bf16, head_dim 128 or 64; any axis lengths (at most 128: a line fits a tile).
bool ffk_dct_tc_supported(const FFDims& dm) {
  if (dm.fp32 || (dm.d != 128 && dm.d != 64)) return false;
  long long tiles = 0;
  for (int a = 0; a < 3; ++a) { const FFPassShape g = ff_pass_shape(dm, a); if (g.tiles > tiles) tiles = g.tiles; }
  return 3LL * dm.BH * tiles < (1LL << 31);              // tile numbers of a launch are 31-bit
}

// The matrix of axis `axis` (0 = t, 1 = h, 2 = w), forward or inverse, as the tensor-memory operand image the
// plan holds (built at plan creation by ffk_dct2_build_image: w lines follow one another, A = I kron Mat;
// h and t lines interleave, A = Mat kron I).
static const uint32_t* matrix_image(const ff_plan* p, int axis, int inverse) {
  return p->dct2_images + (size_t)((inverse ? 3 : 0) + axis) * FF_IMAGE_CELLS;
}

// Scratch: two hi/lo pairs of bf16 grids for `group` tensor-heads, or two fp32 grids.
size_t ffk_dct_tc_scratch_bytes(const FFDims& dm, int group) {
  const size_t grid = (size_t)group * dm.N * dm.d * 2;
  return 4 * ((grid + 255) / 256 * 256);
}

namespace {
struct Scratch { __nv_bfloat16 *a_hi, *a_lo, *b_hi, *b_lo; };
Scratch carve(ff_plan* p) {
  const size_t grid_bytes = ((size_t)p->dct_group * p->dm.N * p->dm.d * 2 + 255) / 256 * 256;
  char* base = (char*)p->buf.scratchA;
  Scratch s;
  s.a_hi = (__nv_bfloat16*)base; s.a_lo = (__nv_bfloat16*)(base + grid_bytes);
  s.b_hi = (__nv_bfloat16*)(base + 2 * grid_bytes); s.b_lo = (__nv_bfloat16*)(base + 3 * grid_bytes);
  return s;
}
}  // namespace

cudaError_t ffk_forward_transform_tc(ff_plan* p, const void* Q, const void* K, const void* V, bool want_energy,
                                     cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int G = p->dct_group;
  const Scratch sc = carve(p);
  // Default: w and the shorter of h, t in one launch (intermediate on chip), then the band-split pass
  // along the remaining axis.  Kernel-select bit 4: the three axes as separate passes w, h, t.
  const bool fused = p->dct2_ok && !(p->attn_impl & 4);
  const int last_axis = fused ? (p->dct2_axis2 == 1 ? 0 : 1) : 0;
  // mXh/mXl: load maps of a pass's input pair; oXh/oXl: store maps of a pass's output pair (the box
  // follows the axis of the pass that uses the map)
  const bool exact = ff_fp32_grid(dm);        // fp32 grids between the passes (in the place of a pair)
  CUtensorMap mq, mk, mv, m1h, m1l, m2h, m2l, o0h, o0l, o1h, o1l, m3h, m3l;
  // (otherwise the first pass writes the byte form; the second one a pair, measured: the band-split pass is slower with a
  // byte-form input)
  if (!fused && !(grid_map(p, &mq, Q, dm.BH, 2) && grid_map(p, &mk, K, dm.BH, 2) && grid_map(p, &mv, V, dm.BH, 2))) return cudaErrorInvalidValue;
  if (fused   ? !(grid_map(p, &m3h, sc.a_hi, G, last_axis) && grid_map(p, &m3l, sc.a_lo, G, last_axis))
      : exact ? !(store_map(p, &o0h, sc.a_hi, G, 2, T_F32) && grid_map(p, &m1h, sc.a_hi, G, 1, T_F32) &&
                  store_map(p, &o1h, sc.b_hi, G, 1, T_F32) && grid_map(p, &m2h, sc.b_hi, G, 0, T_F32))
              : !(store_map(p, &o0h, sc.a_hi, G, 2) && store_map(p, &o0l, sc.a_lo, G, 2, T_BYTE) &&
                  grid_map(p, &m1h, sc.a_hi, G, 1) && grid_map(p, &m1l, sc.a_lo, G, 1, T_BYTE) &&
                  store_map(p, &o1h, sc.b_hi, G, 1) && store_map(p, &o1l, sc.b_lo, G, 1) &&
                  grid_map(p, &m2h, sc.b_hi, G, 0) && grid_map(p, &m2l, sc.b_lo, G, 0)))
    return cudaErrorInvalidValue;
  if (exact) { o0l = o0h; m1l = m1h; o1l = o1h; m2l = m2h; }     // (not used)
  const int total = 3 * dm.BH;
  const bool few = few_tiles(dm, p->sm_count);
  DctTcParams P{};
  P.dm = dm; P.status = p->buf.status;
  P.spec_mid = (__nv_bfloat16*)p->buf.spec_mid; P.spec_high = (__nv_bfloat16*)p->buf.spec_high;
  P.energy = want_energy ? p->buf.energy : nullptr;
  P.spec_low = p->buf.spec_low;
  for (int g0 = 0; g0 < total; g0 += G) {
    const int g = total - g0 < G ? total - g0 : G;
    P.group = g; P.group_start = g0;
    cudaError_t e;
    if (p->pipe_in) {                              // host-buffer entry point: this group's copy must have landed
      e = cudaStreamWaitEvent(st, p->ev_copy[g0 / G], 0);
      if (e != cudaSuccess) return e;
    }
    if (fused) {
      e = (p->fold ? ffk_dct_fold_forward : ffk_dct2_forward)(p, Q, K, V, g0, g, sc.a_hi, sc.a_lo, want_energy && g0 == 0, st);
      if (e != cudaSuccess) return e;
      P.in_split = 1; P.out_lo8 = 0; P.reverse = 1;
      P.mode = MODE_SPLIT; P.axis = last_axis; P.image = matrix_image(p, last_axis, 0);
      e = launch_pass(p, m3h, m3l, m3l, m3h, m3l, P, FORM_PAIR, st);    // (no tensor stores in this mode)
      if (e != cudaSuccess) return e;
      continue;
    }
    P.clear = want_energy && g0 == 0 ? p->buf.energy : nullptr;
    P.mode = MODE_FIRST; P.in_split = 0; P.out_lo8 = 1; P.reverse = 0; P.axis = 2; P.image = matrix_image(p, 2, 0);
    e = launch_pass(p, mq, mk, mv, o0h, o0l, P, exact ? FORM_EXACT1 : FORM_PAIR, st);
    if (e != cudaSuccess) return e;
    P.clear = nullptr;
    P.mode = MODE_MIDDLE; P.in_split = 1; P.out_lo8 = 0; P.reverse = 1; P.axis = 1; P.image = matrix_image(p, 1, 0);
    e = launch_pass(p, m1h, m1l, m1l, o1h, o1l, P, exact ? (few ? FORM_EXACT_FEW : FORM_EXACT) : FORM_BYTES, st);
    if (e != cudaSuccess) return e;
    P.in_split = 1; P.out_lo8 = 0; P.reverse = 0;
    P.mode = MODE_SPLIT; P.axis = 0; P.image = matrix_image(p, 0, 0);
    e = launch_pass(p, m2h, m2l, m2l, m2h, m2l, P, exact ? (few ? FORM_EXACT_FEW : dm.d == 128 ? FORM_EXACT_SPLIT : FORM_EXACT) : FORM_PAIR, st);    // (no tensor stores in this mode)
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Inverse transform of `g` recombined grids (in the first scratch pair, written by the exchange: three-byte form or
// fp32) into out[h0 .. h0+g).
cudaError_t ffk_inverse_transform_tc(ff_plan* p, int h0, int g, void* out, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int G = p->dct_group;
  const Scratch sc = carve(p);
  const bool fused = p->dct2_ok && !(p->attn_impl & 4), exact = ff_fp32_grid(dm);
  // Order of the axes: the one that the fused launch leaves out, and it; or three passes.  Those go w, h, t on the grids with
  // the byte form: the pass along t reads and writes rows that lie H W positions apart, which costs it most where it
  // also moves the bytes of both sides (64 x 128 x 128, 16 heads, whole inverse stage: t, h, w 10.48 ms; h, w, t 9.93;
  // w, h, t 9.75.  64 x 64 x 64: 3.33, 3.27, 3.27).  With fp32 grids every order takes the same time (1085 to 1090 us).
  const bool w_first = !fused && !exact;
  const int first_axis = fused ? (p->dct2_axis2 == 1 ? 0 : 1) : (w_first ? 2 : 0), last_axis = w_first ? 0 : 2;
  // (the exchange writes the three-byte form; three passes hand it on, the fused launch takes a bf16 pair)
  const int hi = exact ? T_F32 : T_BF16, lo = fused ? T_BF16 : T_BYTE;
  const int form = exact ? FORM_EXACT : FORM_BYTES;
  CUtensorMap m_in, m_inl, mbh, mbl, mah, mal, obh, obl, oah, oal, mout;
  if (!grid_map(p, &m_in, sc.a_hi, G, first_axis, hi) || !store_map(p, &obh, sc.b_hi, G, first_axis, hi) ||
      (!fused && (!grid_map(p, &mbh, sc.b_hi, G, 1, hi) || !store_map(p, &oah, sc.a_hi, G, 1, hi) ||
                  !grid_map(p, &mah, sc.a_hi, G, last_axis, hi) || !store_map(p, &mout, out, dm.BH, last_axis))))
    return cudaErrorInvalidValue;
  if (exact) { m_inl = m_in; obl = obh; mbl = mbh; oal = oah; mal = mah; }     // (not used)
  else if (!grid_map(p, &m_inl, sc.a_lo, G, first_axis, T_BYTE) || !store_map(p, &obl, sc.b_lo, G, first_axis, lo) ||
           (!fused && (!grid_map(p, &mbl, sc.b_lo, G, 1, lo) || !store_map(p, &oal, sc.a_lo, G, 1, lo) ||
                       !grid_map(p, &mal, sc.a_lo, G, last_axis, lo))))
    return cudaErrorInvalidValue;
  DctTcParams P{};
  P.dm = dm; P.status = p->buf.status; P.group = g; P.group_start = h0;
  P.mode = MODE_MIDDLE; P.in_split = 1; P.out_lo8 = fused ? 0 : 1; P.reverse = 1; P.axis = first_axis;
  P.image = matrix_image(p, first_axis, 1);
  cudaError_t e = launch_pass(p, m_in, m_inl, m_inl, obh, obl, P, form, st);
  if (e != cudaSuccess) return e;
  if (fused) return (p->t16 ? ffk_dct_t16_inverse : ffk_dct2_inverse)(p, sc.b_hi, sc.b_lo, h0, g, out, st);
  P.reverse = 0; P.axis = 1; P.image = matrix_image(p, 1, 1);
  e = launch_pass(p, mbh, mbl, mbl, oah, oal, P, form, st);
  if (e != cudaSuccess) return e;
  P.mode = MODE_LAST; P.out_lo8 = 0; P.reverse = 1; P.axis = last_axis; P.image = matrix_image(p, last_axis, 1);
  return launch_pass(p, mah, mal, mal, mout, mout, P, form, st);
}

FF_CLOCKS_READ(transform_pass)
