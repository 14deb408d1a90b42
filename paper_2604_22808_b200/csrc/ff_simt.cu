// Generic FP32-arithmetic kernels of the FreqFormer forward.  They cover every configuration the
// ABI accepts (any storage type, head_dim, block/stride/radius) and are the path of the fp32
// workloads; the bf16 workloads replace them with the tensor-core kernels where those apply.
#include "ff_bands.cuh"
#include "ff_internal.h"
#include "ff_three_byte.cuh"
#include "ff_worklist.cuh"

namespace {

__device__ __forceinline__ void fma4(float4& acc, float m, const float4& x) {
  acc.x = fmaf(m, x.x, acc.x); acc.y = fmaf(m, x.y, acc.y); acc.z = fmaf(m, x.z, acc.z); acc.w = fmaf(m, x.w, acc.w);
}

// ff_band_rank_of in 32 bits (axis lengths are at most 128).
__device__ __forceinline__ int band_rank(const FFDims& dm, int kt, int kh, int kw, int& rank) {
  auto below = [&](const int (&A)[3]) {
    if (kt >= A[0]) return A[0] * A[1] * A[2];
    return kt * A[1] * A[2] + min(kh, A[1]) * A[2] + (kh < A[1] ? min(kw, A[2]) : 0);
  };
  const int cl = below(dm.L), cm = below(dm.M);
  if (kt < dm.L[0] && kh < dm.L[1] && kw < dm.L[2]) { rank = cl; return 0; }
  if (kt < dm.M[0] && kh < dm.M[1] && kw < dm.M[2]) { rank = cm - cl; return 1; }
  rank = (kt * dm.H + kh) * dm.W + kw - cm;
  return 2;
}

// Where coefficient (kt, kh, kw) of tensor-head th goes: four channels from `ch` on.
template <typename ST>
__device__ __forceinline__ void store_coefficient(const FFDims& dm, float* spec_low, void* spec_mid, void* spec_high, int th, int kt,
                                                  int kh, int kw, int ch, const float4& v) {
  int rank;
  const int band = band_rank(dm, kt, kh, kw, rank);
  if (band == 0) st4(spec_low + ((size_t)th * dm.Nlow + rank) * dm.d + ch, v);
  else if (band == 1) st4((ST*)spec_mid + ((size_t)th * dm.Nmid + rank) * dm.d + ch, v);
  else st4((ST*)spec_high + ((size_t)th * dm.Nhigh + rank) * dm.d + ch, v);
}

// ------------------------------------------------------------------------------------------------
// One axis of the separable transform ("Separable spectral decomposition"):
//   out[o][a][c] = sum_b Mat[a][b] * in[o][b][c],   a, b in [0,n), c in [0,inner), o in [0,outer)
// with the tensor-head as the slowest index.  Mat is C (forward) or C^T (inverse).
// MODE 0: `in` is the caller's Q/K/V (storage type), `out` an fp32 scratch grid.
// MODE 1: fp32 scratch -> fp32 scratch.
// MODE 2: fp32 scratch -> band-major coefficient buffers (forward, last axis = t).
// MODE 3: fp32 scratch -> the caller's `out` tensor (storage type).
//
// A block stages tiles of n positions x V groups of four neighbouring columns (o, c) with asynchronous copies, the next
// tile while it works on this one; a thread computes eight outputs of one group, V = 256 / (output groups), so any n
// keeps the lanes busy.  Bound by the FMA pipe next to the shared-memory reads (one of the tile, two broadcasts of the
// matrix per 32 FMA); straight from global memory, as before, it waited for loads two thirds of the time (w pass of
// 12 x 9 x 30 x 40 x 64 floats 44 us).
// ------------------------------------------------------------------------------------------------
constexpr int DCT_THREADS = 256;

struct DctPassParams {
  const void* src[3];   // MODE 0: Q, K, V; otherwise src[0] = scratch
  void* dst;            // MODE 0/1: scratch; MODE 3: out tensor
  const float* mat_t;   // [b][a] = Mat[a][b]
  int n, inner, outer;
  int group_start;      // first tensor-head index of this launch
  int BH;
  int V, tiles;         // column groups per tile; tiles of a tensor-head
  int nbuf;             // tile buffers: 2, or 1 where two would leave an SM with a single block
  int group;            // tensor-heads of the launch
  long long N_d;        // elements per tensor-head
  FFDims dm;
  // MODE 2
  float* spec_low; void* spec_mid; void* spec_high;
  double* clear;        // MODE 0, first launch of a routed call: the band energies, cleared for the sums that follow
};

// The matrix, rows padded to a multiple of eight outputs.
__device__ __forceinline__ void stage_matrix(float* mt, const float* mat_t, int n, int npad) {
  for (int idx = threadIdx.x; idx < n * npad; idx += blockDim.x) {
    const int b = idx / npad, a = idx - b * npad;
    mt[idx] = a < n ? mat_t[b * n + a] : 0.f;
  }
}

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename ST, int MODE>
__global__ void __launch_bounds__(DCT_THREADS, 3) dct_pass_kernel(const __grid_constant__ DctPassParams P) {
  extern __shared__ float mt[];
  const int n = P.n, npad = (n + 7) & ~7, groups = npad / 8, V = P.V;
  float* buf = mt + n * npad;               // nbuf x [n][4 V]
  stage_matrix(mt, P.mat_t, n, npad);
  ff_pdl_wait();
  if (MODE == 0 && P.clear && blockIdx.x == 0)
    for (int i = threadIdx.x; i < P.dm.B * 3 * P.dm.d; i += DCT_THREADS) P.clear[i] = 0.0;
  const unsigned inner = (unsigned)P.inner, cols = inner * (unsigned)P.outer;
  const int total = P.tiles * P.group;
  const int g = (int)threadIdx.x / V, v = (int)threadIdx.x - g * V, rstep = DCT_THREADS / V;
  auto load = [&](int t, float* dst) {
    if (t < total && g < rstep) {
      const int gi = t / P.tiles, th = P.group_start + gi;     // tensor-head inside the group; tensor * BH + bh
      const unsigned col = (unsigned)((t - gi * P.tiles) * V + v) * 4;
      const bool on = col < cols;
      const unsigned o = on ? col / inner : 0, c = on ? col - o * inner : 0;
      const size_t line = (size_t)o * n * inner + c;
      if (MODE == 0 && sizeof(ST) == 2) {
        const ST* src = (const ST*)P.src[th / P.BH] + (size_t)(th % P.BH) * P.N_d + line;
#pragma unroll 4
        for (int b = g; b < n; b += rstep) *(float4*)(dst + (b * V + v) * 4) = ld4(src + (size_t)b * inner);
      } else {
        const float* src = (MODE == 0 ? (const float*)P.src[th / P.BH] + (size_t)(th % P.BH) * P.N_d : (const float*)P.src[0] + (size_t)gi * P.N_d) + line;
#pragma unroll 4
        for (int b = g; b < n; b += rstep) cp_async16(dst + (b * V + v) * 4, src + (size_t)b * inner, on);
      }
    }
    cp_async_commit();
  };
  int cur = 0;
  load(blockIdx.x, buf);
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    const float* tile = buf + (size_t)cur * n * V * 4;
    if (P.nbuf == 2) {
      load(t + gridDim.x, buf + (size_t)(cur ^ 1) * n * V * 4);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int gi = t / P.tiles, th = P.group_start + gi;
    const unsigned col = (unsigned)((t - gi * P.tiles) * V + v) * 4;
    if (g < groups && col < cols) {
      const unsigned o = col / inner, c = col - o * inner;
      const size_t line = (size_t)o * n * inner + c;
      float4 acc[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      const float* m = mt + g * 8;
      const float* xs = tile + v * 4;
#pragma unroll 4
      for (int b = 0; b < n; ++b) {
        const float4 x = *(const float4*)(xs + b * V * 4);
        const float4 m0 = *(const float4*)(m + b * npad), m1 = *(const float4*)(m + b * npad + 4);
        fma4(acc[0], m0.x, x); fma4(acc[1], m0.y, x); fma4(acc[2], m0.z, x); fma4(acc[3], m0.w, x);
        fma4(acc[4], m1.x, x); fma4(acc[5], m1.y, x); fma4(acc[6], m1.z, x); fma4(acc[7], m1.w, x);
      }
      int ch = 0, kw = 0, kh = 0;
      if (MODE == 2) {                      // a = k_t, column = (k_h, k_w, channel)
        const unsigned p = c / (unsigned)P.dm.d;
        ch = (int)(c - p * (unsigned)P.dm.d);
        kh = (int)(p / (unsigned)P.dm.W); kw = (int)(p - (unsigned)kh * (unsigned)P.dm.W);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int a = g * 8 + i;
        if (a >= n) break;
        if (MODE <= 1) st4((float*)P.dst + (size_t)gi * P.N_d + line + (size_t)a * inner, acc[i]);
        else if (MODE == 3) st4((ST*)P.dst + (size_t)th * P.N_d + line + (size_t)a * inner, acc[i]);
        else store_coefficient<ST>(P.dm, P.spec_low, P.spec_mid, P.spec_high, th, a, kh, kw, ch, acc[i]);
      }
    }
    __syncthreads();
    if (P.nbuf == 2) cur ^= 1; else load(t + gridDim.x, buf);
  }
  cp_async_wait<0>();
}

template <typename ST, int MODE>
cudaError_t launch_dct_pass(ff_plan* p, DctPassParams& P, int group, cudaStream_t st) {
  const int npad = (P.n + 7) & ~7;
  P.V = DCT_THREADS / (npad / 8);
  P.tiles = (int)(((long long)P.inner * P.outer / 4 + P.V - 1) / P.V);
  P.group = group;
  const size_t mat = (size_t)P.n * npad * sizeof(float), tile = (size_t)P.n * P.V * 4 * sizeof(float);
  P.nbuf = mat + 2 * tile <= 112 * 1024 ? 2 : 1;
  const size_t smem = mat + P.nbuf * tile;
  const int per_sm = smem <= 75 * 1024 ? 3 : 2;
  const long long total = (long long)P.tiles * group, most = (long long)per_sm * p->sm_count;
  p->launches += 1;
  return ff_launch(dct_pass_kernel<ST, MODE>, dim3((unsigned)(total < most ? total : most)), dim3(DCT_THREADS), smem, st, P);
}

// ------------------------------------------------------------------------------------------------
// All three axes of a small grid in one launch: a block holds eight channels of a tensor-head's whole grid in shared
// memory and transforms it in place, axis by axis (lines are handled in rounds: everything a round reads is in
// registers before any of it is overwritten).  Small grids are bound by launches and latency: 4 x 8 x 8 tokens take
// one launch of 6 us instead of three of 5.  On the smallest grids a thread computes two outputs instead of eight, which keep a
// quarter of the threads or fewer busy (rule: vol_fine).
// ------------------------------------------------------------------------------------------------
constexpr int VOL_CH = 8, VOL_THREADS = 256;
constexpr int VOL_MAX = 2304;            // positions: 72 KB, so that three blocks share an SM

struct VolParams {
  const void* src[3];      // forward: Q, K, V; inverse: src[0] = fp32 grids [g][N][d]
  void* out;               // inverse: the caller's tensor
  const float* mat_t[3];   // per axis (t, h, w): [b][a]
  int group_start;
  FFDims dm;
  float* spec_low; void* spec_mid; void* spec_high;
  double* clear;
};

// OUT: outputs (of four channels each) that a thread computes of a line.
template <typename ST, bool INVERSE, int OUT>
__global__ void __launch_bounds__(VOL_THREADS) dct_volume_kernel(const __grid_constant__ VolParams P) {
  extern __shared__ float4 vol[];                      // [N][2]
  const FFDims& dm = P.dm;
  const int N = (int)dm.N, tid = threadIdx.x;
  float* mats = (float*)(vol + 2 * N);                 // the matrices of the three axes, before anything is waited for
  for (int axis = 0, at = 0; axis < 3; ++axis) {
    const int n = axis == 2 ? dm.W : (axis == 1 ? dm.H : dm.T), npad = (n + 7) & ~7;
    stage_matrix(mats + at, P.mat_t[axis], n, npad);
    at += n * npad;
  }
  ff_pdl_wait();
  if (!INVERSE && P.clear && blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = tid; i < dm.B * 3 * dm.d; i += VOL_THREADS) P.clear[i] = 0.0;
  const int th = P.group_start + blockIdx.y, c0 = blockIdx.x * VOL_CH;
  const size_t per = (size_t)N * dm.d;
  for (int i = tid; i < 2 * N; i += VOL_THREADS) {
    const size_t o = (size_t)(i >> 1) * dm.d + c0 + (i & 1) * 4;
    vol[i] = INVERSE ? ld4((const float*)P.src[0] + (size_t)blockIdx.y * per + o)
                     : ld4((const ST*)P.src[th / dm.BH] + (size_t)(th % dm.BH) * per + o);
  }
  __syncthreads();
  for (int step = 0; step < 3; ++step) {
    const int axis = INVERSE ? step : 2 - step;
    const int n = axis == 2 ? dm.W : (axis == 1 ? dm.H : dm.T), stride = axis == 2 ? 1 : (axis == 1 ? dm.W : dm.H * dm.W);
    const int npad = (n + 7) & ~7, groups = OUT == 8 ? npad / 8 : (n + OUT - 1) / OUT;
    const int at = axis == 0 ? 0 : dm.T * ((dm.T + 7) & ~7) + (axis == 1 ? 0 : dm.H * ((dm.H + 7) & ~7));
    const float* mt = mats + at;
    const int upl = 2 * groups, lines = N / n;           // units (OUT outputs x 4 channels) of a line
    const int lpr = VOL_THREADS / upl;                   // lines per round
    const int l = tid / upl, u = tid - l * upl, cg = u & 1, g = u >> 1;
    for (int l0 = 0; l0 < lines; l0 += lpr) {
      const int line = l0 + l;
      const bool on = l < lpr && line < lines;
      const int base = axis == 0 ? line : (line / stride) * stride * n + line % stride;
      float4* x = vol + 2 * base + cg;
      float4 acc[OUT];
#pragma unroll
      for (int i = 0; i < OUT; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (on)
#pragma unroll 4
        for (int b = 0; b < n; ++b) {
          const float4 v = x[2 * b * stride];
          if (OUT == 2) {
            const float2 m = *(const float2*)(mt + b * npad + g * 2);
            fma4(acc[0], m.x, v); fma4(acc[1], m.y, v);
          } else {
            const float4 m0 = *(const float4*)(mt + b * npad + g * 8), m1 = *(const float4*)(mt + b * npad + g * 8 + 4);
            fma4(acc[0], m0.x, v); fma4(acc[1], m0.y, v); fma4(acc[2 % OUT], m0.z, v); fma4(acc[3 % OUT], m0.w, v);
            fma4(acc[4 % OUT], m1.x, v); fma4(acc[5 % OUT], m1.y, v); fma4(acc[6 % OUT], m1.z, v); fma4(acc[7 % OUT], m1.w, v);
          }
        }
      __syncthreads();
      if (on)
#pragma unroll
        for (int i = 0; i < OUT; ++i)
          if (g * OUT + i < n) x[2 * (g * OUT + i) * stride] = acc[i];
    }
    __syncthreads();
  }
  for (int i = tid; i < 2 * N; i += VOL_THREADS) {
    const int f = i >> 1, ch = c0 + (i & 1) * 4;
    if (INVERSE) st4((ST*)P.out + (size_t)th * per + (size_t)f * dm.d + ch, vol[i]);
    else store_coefficient<ST>(dm, P.spec_low, P.spec_mid, P.spec_high, th, f / (dm.H * dm.W), f / dm.W % dm.H, f % dm.W, ch, vol[i]);
  }
}

size_t vol_smem(const FFDims& dm) {
  size_t m = 0;
  const int n[3] = {dm.T, dm.H, dm.W};
  for (int a = 0; a < 3; ++a) m += (size_t)n[a] * ((n[a] + 7) & ~7);
  return (size_t)dm.N * VOL_CH * sizeof(float) + m * sizeof(float);
}
bool vol_fits(const FFDims& dm) { return dm.N <= VOL_MAX; }

// Two outputs a thread, both ways (a layer of this size is bound by fetching code, too), where they cover the axes in one round, up
// to an eighth of the steps.  Layers, fp32, all bands, us, eight / two: 4 x 8 x 8 tokens, two heads of 32 channels 27.3 / 26.2, 24 of
// 64 59.4 / 58.2, 96 of 64 125.3 / 112.2; 3 x 5 x 7, twelve of 64 29.3 / 27.2; 2 x 3 x 40 (two rounds of h), 24 of 64 65.5 / 62.2.  In more
// rounds they gain once there are blocks enough to fill the SMs: 3 x 9 x 9, four heads of 64, routed 32.6 / 33.8, 24 of 128 (2.6 blocks
// an SM, inverse) 74.7 / 76.8, 48 of 128 122.5 / 113.9; 5 x 9 x 10, 450 positions, 40.7 / 41.2.  And not where every SM has one block or
// two of the inverse launch, of more than half of 256 positions: 4 x 8 x 8, nine heads of 128 (0.97 an SM) 36.6 / 38.5, 36 of 32
// 48.3 / 52.4, 24 of 96 (1.95) 59.8 / 62.5, 30 of 64 (1.6) 61.5 / 63.4; 42 of 64 (2.3) 71.9 / 69.2.
bool vol_fine(const FFDims& dm, int sm_count) {
  if (dm.N > VOL_THREADS) return false;
  const double blocks = (double)dm.BH * (dm.d / VOL_CH) / sm_count;
  int steps = 0, more = 0;
  for (const int n : {dm.T, dm.H, dm.W}) {
    const int per_round = VOL_THREADS / ((n + 1) / 2 * 2), rounds = ((int)(dm.N / n) + per_round - 1) / per_round;
    steps += n; more += (rounds - 1) * n;
  }
  if (8 * more > steps) return blocks > 4;
  return dm.N <= VOL_THREADS / 2 || !((blocks > 0.875 && blocks < 1.2) || (blocks > 1.5 && blocks < 2.2));
}

// ------------------------------------------------------------------------------------------------
// Band operators ("Hierarchical frequency-domain attention") in fp32: a block takes 64 query rows of one (head, band)
// and walks key tiles with an online softmax.  The key set of a row is generated from its rank: all pooled tokens
// (low), the blocks at block distance 0 mod s (mid; query tiles then run along a residue class, so its keys are one
// dense range of class positions), own and anchor blocks (mid, anchor pattern), the window |p - p'| <= R (high).
//
// Bound by the FMA pipe (5.3 GFLOP of tiles at 9 x 30 x 40 tokens, 4 heads of 64 channels, all bands: 78 us at full
// rate).  A thread holds 8 rows x KT / 16 keys of scores, so that a step of four channels is 12 16-byte shared reads for
// 128 FMA (4 x 4 scores per thread were bound by those reads: 233 us), then 8 rows x d / 16 output channels.  Rows lie
// as they are in memory, padded by 16 bytes against bank conflicts, so copies are asynchronous: the next keys arrive
// during the softmax and P V, the values during Q K.  P is only read by the half warp that wrote it.  64 keys a tile up
// to head_dim 64, 32 above (three blocks, two blocks per SM).  Measured there: 196 us, 70% of the issue slots; packed
// pairs of FMA gained nothing (204 us).
// ------------------------------------------------------------------------------------------------
constexpr int AT = 64, AT_THREADS = 128, AT_PITCH = AT + 4;

template <int DPL> struct AtShape {
  static constexpr int d = DPL * 32, KT = DPL <= 2 ? 64 : 32, KJ = KT / 16, PITCH = d + 4;
  static constexpr size_t smem = (size_t)(AT * PITCH + 2 * KT * PITCH + KT * AT_PITCH) * sizeof(float);
};

template <typename KT_, int DPL>
__device__ __forceinline__ void attend_tile(const KT_* Qp, const KT_* Kp, const KT_* Vp, KT_* Yp, const FFDims& dm, int band, int n, int tile,
                                            float* sm) {
  using S = AtShape<DPL>;
  constexpr int d = S::d, KT = S::KT, KJ = S::KJ, PITCH = S::PITCH, VEC = d / 4;
  float* Qs = sm;                                        // [AT][PITCH]
  float* Ks = Qs + AT * PITCH;                           // [KT][PITCH]
  float* Vs = Ks + KT * PITCH;                           // [KT][PITCH]
  float* Ps = Vs + KT * PITCH;                           // [KT][AT_PITCH]: P transposed
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const float scale = rsqrtf((float)d);
  const int blk_rows = min(dm.b, n), R = min(dm.R, n);   // (so that sums of positions stay in 32 bits)
  const bool strided = band == 1 && dm.pattern == FF_MID_STRIDED;
  const bool anchor = band == 1 && !strided;
  // class-local (strided mid band) or band positions of the tile, and the range of key positions
  int cls = 0, q0 = tile * AT, len = n, ks = 0, ke = n;
  if (strided) {
    const int per = (int)(dm.nb / dm.s), rem = (int)(dm.nb % dm.s);                   // blocks of a class: per or per + 1
    const int t_big = ((per + 1) * blk_rows + AT - 1) / AT, t_small = (per * blk_rows + AT - 1) / AT;
    int t;
    if (tile < rem * t_big) { cls = tile / t_big; t = tile % t_big; len = (per + 1) * blk_rows; }
    else {
      const int rest = tile - rem * t_big;
      if (t_small == 0 || rest >= (dm.s - rem) * t_small) return;
      cls = rem + rest / t_small; t = rest % t_small; len = per * blk_rows;
    }
    q0 = t * AT; ke = len;
  } else {
    if (q0 >= n) return;
    if (band == 2) {
      ks = q0 > R ? q0 - R : 0;
      ke = n - q0 - AT < R ? n : q0 + AT + R;
    }
  }
  auto rank_of = [&](int u) -> int {                     // band rank of a position
    if (!strided) return u;
    const unsigned blk = (unsigned)u / (unsigned)blk_rows;
    return (int)(((unsigned)cls + blk * (unsigned)dm.s) * (unsigned)blk_rows + ((unsigned)u - blk * (unsigned)blk_rows));
  };
  // rows u0 .. u0 + ROWS of the positions below `end`, zeros past them
  auto load = [&](float* dst, const KT_* src, int rows, int u0, int end) {
#pragma unroll 4
    for (int i = tid; i < rows * VEC; i += AT_THREADS) {
      const int r = i / VEC, v = i - r * VEC, rk = u0 + r < end ? rank_of(u0 + r) : n;
      const bool on = rk < n;
      const KT_* from = src + (size_t)(on ? rk : 0) * d + v * 4;
      float* to = dst + r * PITCH + v * 4;
      if (sizeof(KT_) == 4) cp_async16(to, (const float*)from, on);
      else *(float4*)to = on ? ld4(from) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    cp_async_commit();
  };
  // (anchor) anchor blocks are s blocks apart: skip key tiles without one and without any of the rows' own blocks
  auto next_tile = [&](int k0) {
    for (; anchor && k0 < ke; k0 += KT) {
      const int b0 = k0 / blk_rows, b1 = (min(k0 + KT, n) - 1) / blk_rows;
      const bool any = (b1 + 1) / dm.s > b0 / dm.s;      // some block J in [b0, b1] has J = s - 1 mod s
      if (any || !(b1 < q0 / blk_rows || b0 > (min(q0 + AT, n) - 1) / blk_rows)) break;
    }
    return k0;
  };
  int k0 = next_tile(ks);
  load(Qs, Qp, AT, q0, len);
  load(Ks, Kp, KT, k0, ke);
  int pq[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) pq[i] = q0 + ty * 8 + i < len ? rank_of(q0 + ty * 8 + i) : n;
  float mx[8], den[8], o[8][DPL][2];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    mx[i] = -INFINITY; den[i] = 0.f;
#pragma unroll
    for (int j = 0; j < DPL; ++j) o[i][j][0] = o[i][j][1] = 0.f;
  }
  while (k0 < ke) {
    load(Vs, Vp, KT, k0, ke);                            // (P V of the previous tile has been read: barrier below)
    cp_async_wait<1>();
    __syncthreads();
    float s[8][KJ];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < KJ; ++j) s[i][j] = 0.f;
#pragma unroll 2
    for (int c = 0; c < d; c += 4) {
      float4 k[KJ];
#pragma unroll
      for (int j = 0; j < KJ; ++j) k[j] = *(const float4*)(Ks + (tx + 16 * j) * PITCH + c);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 q = *(const float4*)(Qs + (ty * 8 + i) * PITCH + c);
#pragma unroll
        for (int j = 0; j < KJ; ++j)
          s[i][j] = fmaf(q.x, k[j].x, fmaf(q.y, k[j].y, fmaf(q.z, k[j].z, fmaf(q.w, k[j].w, s[i][j]))));
      }
    }
    __syncthreads();                                     // K has been read
    const int k1 = next_tile(k0 + KT);
    if (k1 < ke) load(Ks, Kp, KT, k1, ke);
    // which pairs exist: all of them, except in edge tiles
    bool full = k0 + KT <= ke && !anchor;
    if (band == 2) full = full && k0 >= q0 + AT - 1 - R && k0 + KT - 1 <= q0 + R;
    else if (strided) full = full && rank_of(k0 + KT - 1) < n;
    if (full) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < KJ; ++j) s[i][j] *= scale;
    } else {
#pragma unroll
      for (int j = 0; j < KJ; ++j) {
        const int u = k0 + tx + 16 * j, rk = u < ke ? rank_of(u) : n;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          bool ok = rk < n;
          if (band == 2) ok = ok && rk - pq[i] <= R && pq[i] - rk <= R;
          else if (anchor) { const int J = rk / blk_rows; ok = ok && (J == pq[i] / blk_rows || J % dm.s == dm.s - 1); }
          s[i][j] = ok ? s[i][j] * scale : -INFINITY;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float nm = s[i][0];
#pragma unroll
      for (int j = 1; j < KJ; ++j) nm = fmaxf(nm, s[i][j]);
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) nm = fmaxf(nm, __shfl_xor_sync(0xffffffffu, nm, w));
      nm = fmaxf(nm, mx[i]);
      const float ref = nm == -INFINITY ? 0.f : nm;      // (no key of the row so far)
      const float corr = expf(mx[i] - ref);
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < KJ; ++j) { s[i][j] = expf(s[i][j] - ref); sum += s[i][j]; }
      den[i] = den[i] * corr + sum;                      // (this thread's share of the row sum)
      mx[i] = nm;
#pragma unroll
      for (int j = 0; j < DPL; ++j) { o[i][j][0] *= corr; o[i][j][1] *= corr; }
    }
#pragma unroll
    for (int j = 0; j < KJ; ++j) {
      float* p = Ps + (tx + 16 * j) * AT_PITCH + ty * 8;
      *(float4*)p = make_float4(s[0][j], s[1][j], s[2][j], s[3][j]);
      *(float4*)(p + 4) = make_float4(s[4][j], s[5][j], s[6][j], s[7][j]);
    }
    if (k1 < ke) cp_async_wait<1>(); else cp_async_wait<0>();      // V has arrived (the next K may still be on its way)
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < KT; ++k) {
      const float4 p0 = *(const float4*)(Ps + k * AT_PITCH + ty * 8), p1 = *(const float4*)(Ps + k * AT_PITCH + ty * 8 + 4);
      const float pp[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
      for (int j = 0; j < DPL; ++j) {
        const float2 v = *(const float2*)(Vs + k * PITCH + 32 * j + 2 * tx);
#pragma unroll
        for (int i = 0; i < 8; ++i) { o[i][j][0] = fmaf(pp[i], v.x, o[i][j][0]); o[i][j][1] = fmaf(pp[i], v.y, o[i][j][1]); }
      }
    }
    __syncthreads();                                     // V has been read
    k0 = k1;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int w = 8; w > 0; w >>= 1) den[i] += __shfl_xor_sync(0xffffffffu, den[i], w);
    if (pq[i] >= n) continue;
    KT_* y = Yp + (size_t)pq[i] * d + 2 * tx;
#pragma unroll
    for (int j = 0; j < DPL; ++j) { stf<KT_>(y + 32 * j, o[i][j][0] / den[i]); stf<KT_>(y + 32 * j + 1, o[i][j][1] / den[i]); }
  }
}

template <typename ST, int DPL>
__global__ void __launch_bounds__(AT_THREADS, DPL <= 2 ? 3 : 2) attention_simt_kernel(FFBuffers buf, FFDims dm, int band_bits) {
  extern __shared__ float sm[];
  ff_pdl_wait();
  const int band = blockIdx.z == 0 ? 1 : (blockIdx.z == 1 ? 2 : 0);      // the mid band's items are the long ones
  const int bh = blockIdx.y;
  if (!(buf.alloc[bh] & band_bits & (1 << band))) return;
  const int n = (int)(band == 0 ? dm.Nbar : (band == 1 ? dm.Nmid : dm.Nhigh));
  if (n == 0) return;
  const size_t one = (size_t)n * DPL * 32, tensor = (size_t)dm.BH * one;  // a head's, a tensor's extent in the band's buffer
  if (sizeof(ST) == 4) {                          // (one copy of the code: small launches are bound by fetching it)
    const float* Q = (band == 0 ? buf.pooled : (const float*)(band == 1 ? buf.spec_mid : buf.spec_high)) + bh * one;
    float* Y = (band == 0 ? buf.y_low : (float*)(band == 1 ? buf.y_mid : buf.y_high)) + bh * one;
    attend_tile<float, DPL>(Q, Q + tensor, Q + 2 * tensor, Y, dm, band, n, blockIdx.x, sm);
  } else if (band == 0) {
    const float* Q = buf.pooled + bh * one;
    attend_tile<float, DPL>(Q, Q + tensor, Q + 2 * tensor, buf.y_low + bh * one, dm, band, n, blockIdx.x, sm);
  } else {
    const ST* Q = (const ST*)(band == 1 ? buf.spec_mid : buf.spec_high) + bh * one;
    attend_tile<ST, DPL>(Q, Q + tensor, Q + 2 * tensor, (ST*)(band == 1 ? buf.y_mid : buf.y_high) + bh * one, dm, band, n, blockIdx.x, sm);
  }
}

// Small launches (up to ROW_PAIRS scored pairs, if every head ran every band): one warp per query row, eight keys side by
// side, merged into the running softmax as a group.  Little code and as many warps as rows; the tiled kernel above spends
// most of its 17 us there on fetching its instructions (256 tokens, 2 heads of 32 channels).  Whole layer with the tiled
// kernel / with this one, us, all bands: 23K pairs 42.2 / 32.3 (head_dim 64) and 48.5 / 31.1 (128), 73K 44.0 / 45.8 and
// 51.0 / 43.8, 90K 46.4 / 50.3 and 58.4 / 50.5, 103K 42.5 / 47.4 (32), 227K 52.7 / 77.3 and 66.7 / 82.8, 492K 58.5 / 99.9
// and 79.6 / 101.3.  (head_dim 96: 206K 74.8 / 58.4, 492K 83.6 / 89.7.)
constexpr int ROW_WARPS = 4;
constexpr long long ROW_PAIRS = 3 << 15;

template <typename KT_, int DPL>
__device__ __forceinline__ void attend_row(const KT_* Qp, const KT_* Kp, const KT_* Vp, KT_* Yp, const FFDims& dm, int band, int n, int p) {
  const int lane = threadIdx.x & 31, d = DPL * 32;
  const int b = min(dm.b, n), R = min(dm.R, n);
  const bool strided = band == 1;
  // keys: positions of the row's residue class, or a range of ranks
  int cls = 0, k_lo = 0, k_hi = n;
  if (strided) { cls = (int)((p / b) % dm.s); k_hi = (int)((dm.nb - cls + dm.s - 1) / dm.s) * b; }
  else if (band == 2) { k_lo = max(p - R, 0); k_hi = min(p + R + 1, n); }
  const float scale = rsqrtf((float)d);
  float q[DPL], o[DPL], mx = -INFINITY, den = 0.f;
#pragma unroll
  for (int j = 0; j < DPL; ++j) { q[j] = ldf<KT_>(Qp + (size_t)p * d + lane + 32 * j); o[j] = 0.f; }
#pragma unroll 1
  for (int k0 = k_lo; k0 < k_hi; k0 += 8) {
    float sc[8], v[8][DPL];
    bool on[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int u = k0 + k;
      int rk = u;
      if (strided) { const unsigned blk = (unsigned)u / (unsigned)b; rk = (int)(((unsigned)cls + blk * (unsigned)dm.s) * (unsigned)b + ((unsigned)u - blk * (unsigned)b)); }
      on[k] = u < k_hi && rk < n;
      const size_t at = (size_t)(on[k] ? rk : p) * d + lane;
      float part = 0.f;
#pragma unroll
      for (int j = 0; j < DPL; ++j) { part = fmaf(q[j], ldf<KT_>(Kp + at + 32 * j), part); v[k][j] = ldf<KT_>(Vp + at + 32 * j); }
      sc[k] = part;
    }
#pragma unroll
    for (int w = 16; w > 0; w >>= 1)
#pragma unroll
      for (int k = 0; k < 8; ++k) sc[k] += __shfl_xor_sync(0xffffffffu, sc[k], w);
    float nm = mx;
#pragma unroll
    for (int k = 0; k < 8; ++k) { sc[k] = on[k] ? sc[k] * scale : -INFINITY; nm = fmaxf(nm, sc[k]); }
    const float ref = nm == -INFINITY ? 0.f : nm;        // (no key of the row so far)
    const float corr = expf(mx - ref);
    // (every lane has all eight scores: lane k takes the exponential of key k)
    float mine = sc[0];
#pragma unroll
    for (int k = 1; k < 8; ++k) mine = (lane & 7) == k ? sc[k] : mine;
    mine = expf(mine - ref);
    den *= corr;
#pragma unroll
    for (int j = 0; j < DPL; ++j) o[j] *= corr;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float pr = __shfl_sync(0xffffffffu, mine, k);
      den += pr;
#pragma unroll
      for (int j = 0; j < DPL; ++j) o[j] = fmaf(pr, v[k][j], o[j]);
    }
    mx = nm;
  }
#pragma unroll
  for (int j = 0; j < DPL; ++j) stf<KT_>(Yp + (size_t)p * d + lane + 32 * j, o[j] / den);
}

template <typename ST, int DPL>
__global__ void __launch_bounds__(ROW_WARPS * 32) attention_row_kernel(FFBuffers buf, FFDims dm, int band_bits) {
  ff_pdl_wait();
  const int band = blockIdx.z == 0 ? 1 : (blockIdx.z == 1 ? 2 : 0), bh = blockIdx.y;
  if (!(buf.alloc[bh] & band_bits & (1 << band))) return;
  const int n = (int)(band == 0 ? dm.Nbar : (band == 1 ? dm.Nmid : dm.Nhigh)), p = blockIdx.x * ROW_WARPS + (threadIdx.x >> 5);
  if (p >= n) return;
  const size_t one = (size_t)n * DPL * 32, tensor = (size_t)dm.BH * one;
  if (sizeof(ST) == 4 || band == 0) {
    const float* Q = (band == 0 ? buf.pooled : (const float*)(band == 1 ? buf.spec_mid : buf.spec_high)) + bh * one;
    float* Y = (band == 0 ? buf.y_low : (float*)(band == 1 ? buf.y_mid : buf.y_high)) + bh * one;
    attend_row<float, DPL>(Q, Q + tensor, Q + 2 * tensor, Y, dm, band, n, p);
  } else {
    const ST* Q = (const ST*)(band == 1 ? buf.spec_mid : buf.spec_high) + bh * one;
    attend_row<ST, DPL>(Q, Q + tensor, Q + 2 * tensor, (ST*)(band == 1 ? buf.y_mid : buf.y_high) + bh * one, dm, band, n, p);
  }
}

// Exchange + recombination ("Cross-band residual exchange", "Reconstruction"): for every
// coefficient of the grid, fetch its band token, add softmax(y Z^T / sqrt(d)) Z over the 2m summary
// tokens of the other two bands, and write the row at its coefficient position.
// Eight lanes share a token (lane s holds channels 4 s + 32 i .. + 3): a score takes three shuffles for four tokens.
// The four tokens of a warp may lie in different bands, so all 3m summaries are scored and a token's own band masked.
constexpr int EXC_WARPS = 8;
constexpr int EXC_TOKENS = EXC_WARPS * 4;      // per block and round

template <typename ST, int DPL, typename OT>
__global__ void __launch_bounds__(EXC_WARPS * 32, 2) exchange_recombine_kernel(FFBuffers buf, FFDims dm, int bh0, OT* grid_out,
                                                                               void* grid_lo, int rounds) {
  extern __shared__ float4 Z[];                // [3 m][d]
  constexpr int d = DPL * 32, KB = DPL >= 3 ? 4 : 8;       // keys scored side by side (registers)
  ff_pdl_wait();
  const int gi = blockIdx.y, bh = bh0 + gi, m = dm.m;
  const float4* zsrc = (const float4*)(buf.summary + (size_t)bh * 3 * m * d);
#pragma unroll 4
  for (int i = threadIdx.x; i < 3 * m * (d / 4); i += EXC_WARPS * 32) Z[i] = zsrc[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, s = lane & 7;
  const float scale = rsqrtf((float)d);
  const int N = (int)dm.N;
  for (int round = 0; round < rounds; ++round) {
    const int f0 = ((int)blockIdx.x * rounds + round) * EXC_TOKENS + warp * 4;
    if (f0 >= N) return;
    const int f = f0 + (lane >> 3) < N ? f0 + (lane >> 3) : N - 1;
    const int row_w = f / dm.W, kw = f - row_w * dm.W, kt = row_w / dm.H, kh = row_w - kt * dm.H;
    int rank;
    const int band = band_rank(dm, kt, kh, kw, rank);
    const BandView<ST> v = band_view<ST>(buf, dm, bh, band);
    float4 y[DPL], acc[DPL];
    const size_t at = (size_t)(v.compressed ? rank / dm.r : rank) * d + 4 * s;
#pragma unroll
    for (int i = 0; i < DPL; ++i) {
      y[i] = v.f32 ? ld4(v.f32 + at + 32 * i) : ld4(v.st + at + 32 * i);
      acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (m > 0) {
      // keys of the token: not its own band's, and none of an empty mid band
      const int skip0 = band * m, skip1 = dm.Nmid == 0 ? m : skip0;
      float mx = -INFINITY, den = 0.f;
      for (int k0 = 0; k0 < 3 * m; k0 += KB) {
        float sc[KB];
#pragma unroll
        for (int k = 0; k < KB; ++k) {
          const float4* z = Z + (k0 + k < 3 * m ? k0 + k : 0) * (d / 4) + s;
          float part = 0.f;
#pragma unroll
          for (int i = 0; i < DPL; ++i) {
            const float4 zz = z[8 * i];
            part = fmaf(y[i].x, zz.x, part); part = fmaf(y[i].y, zz.y, part);
            part = fmaf(y[i].z, zz.z, part); part = fmaf(y[i].w, zz.w, part);
          }
          sc[k] = part;
        }
#pragma unroll
        for (int w = 4; w > 0; w >>= 1)
#pragma unroll
          for (int k = 0; k < KB; ++k) sc[k] += __shfl_xor_sync(0xffffffffu, sc[k], w);
        float nm = mx;
#pragma unroll
        for (int k = 0; k < KB; ++k) {
          const int key = k0 + k;
          const bool on = key < 3 * m && !(key >= skip0 && key < skip0 + m) && !(key >= skip1 && key < skip1 + m);
          sc[k] = on ? sc[k] * scale : -INFINITY;
          nm = fmaxf(nm, sc[k]);
        }
        const float ref = nm == -INFINITY ? 0.f : nm;           // (no key so far)
        const float corr = expf(mx - ref);
        den *= corr;
#pragma unroll
        for (int i = 0; i < DPL; ++i) { acc[i].x *= corr; acc[i].y *= corr; acc[i].z *= corr; acc[i].w *= corr; }
#pragma unroll
        for (int k = 0; k < KB; ++k) {
          const float pr = expf(sc[k] - ref);
          const float4* z = Z + (k0 + k < 3 * m ? k0 + k : 0) * (d / 4) + s;
          den += pr;
#pragma unroll
          for (int i = 0; i < DPL; ++i) fma4(acc[i], pr, z[8 * i]);
        }
        mx = nm;
      }
      if (den > 0.f)
#pragma unroll
        for (int i = 0; i < DPL; ++i) { acc[i].x /= den; acc[i].y /= den; acc[i].z /= den; acc[i].w /= den; }
    }
    if (f0 + (lane >> 3) >= N) continue;
    // With a second grid (bf16 output) the value is stored in three bytes.  A band's tokens share almost the same
    // exchange offset, so a single bf16 rounding would bias whole bands coherently and the inverse transform would
    // focus that bias on a few tokens.
    const size_t o = ((size_t)gi * N + f) * d + 4 * s;
#pragma unroll
    for (int i = 0; i < DPL; ++i) {
      const float4 w = make_float4(y[i].x + acc[i].x, y[i].y + acc[i].y, y[i].z + acc[i].z, y[i].w + acc[i].w);
      if (grid_lo) {
        const uint32_t u0 = ff_round24(w.x), u1 = ff_round24(w.y), u2 = ff_round24(w.z), u3 = ff_round24(w.w);
        *(uint2*)((uint16_t*)grid_out + o + 32 * i) = make_uint2(ff_hi2(u0, u1), ff_hi2(u2, u3));
        *(uint32_t*)((uint8_t*)grid_lo + o + 32 * i) = ff_lo4(u0, u1, u2, u3);
      } else {
        st4(grid_out + o + 32 * i, w);
      }
    }
  }
}

// Rounds per block: up to 8, fewer when the launch would otherwise have too few blocks.
int exc_rounds(long long tokens, int g, int sm_count) {
  const long long r = tokens * g / ((long long)EXC_TOKENS * 8 * sm_count);
  return r < 1 ? 1 : (r > 8 ? 8 : (int)r);
}

template <typename ST, int DPL, typename OT>
cudaError_t launch_exchange(ff_plan* p, int g, int h0, OT* grid_hi, void* grid_lo, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int rounds = exc_rounds(dm.N, g, p->sm_count);
  const long long per_block = (long long)EXC_TOKENS * rounds;
  p->launches += 1;
  return ff_launch(exchange_recombine_kernel<ST, DPL, OT>, dim3((unsigned)((dm.N + per_block - 1) / per_block), (unsigned)g),
                   dim3(EXC_WARPS * 32), (size_t)3 * dm.m * dm.d * sizeof(float), st, p->buf, dm, h0, grid_hi, grid_lo, rounds);
}

}  // namespace

// ================================================================================================
// Launchers
// ================================================================================================
template <typename ST>
static cudaError_t forward_transform_t(ff_plan* p, const void* Q, const void* K, const void* V, bool want_energy, cudaStream_t st) {
  const FFDims& dm = p->dm;
  if (vol_fits(dm)) {
    VolParams P{};
    P.src[0] = Q; P.src[1] = K; P.src[2] = V; P.dm = dm;
    for (int a = 0; a < 3; ++a) P.mat_t[a] = p->basis_t[a];
    P.spec_low = p->buf.spec_low; P.spec_mid = p->buf.spec_mid; P.spec_high = p->buf.spec_high;
    P.clear = want_energy ? p->buf.energy : nullptr;
    p->launches += 1;
    return ff_launch(vol_fine(dm, p->sm_count) ? dct_volume_kernel<ST, false, 2> : dct_volume_kernel<ST, false, 8>, dim3((unsigned)(dm.d / VOL_CH), (unsigned)(3 * dm.BH)), dim3(VOL_THREADS),
                     vol_smem(dm), st, P);
  }
  const int total = 3 * dm.BH, G = p->lay.group;
  DctPassParams P{};
  P.BH = dm.BH; P.N_d = dm.N * dm.d; P.dm = dm;
  P.spec_low = p->buf.spec_low; P.spec_mid = p->buf.spec_mid; P.spec_high = p->buf.spec_high;
  for (int g0 = 0; g0 < total; g0 += G) {
    const int g = (total - g0 < G) ? total - g0 : G;
    P.group_start = g0;
    // w axis: lines of W elements with stride d
    P.src[0] = Q; P.src[1] = K; P.src[2] = V; P.dst = p->buf.scratchA; P.mat_t = p->basis_t[2];
    P.n = dm.W; P.inner = dm.d; P.outer = dm.T * dm.H;
    P.clear = want_energy && g0 == 0 ? p->buf.energy : nullptr;
    cudaError_t e = launch_dct_pass<ST, 0>(p, P, g, st);
    if (e != cudaSuccess) return e;
    // h axis
    P.src[0] = p->buf.scratchA; P.dst = p->buf.scratchB; P.mat_t = p->basis_t[1];
    P.n = dm.H; P.inner = dm.W * dm.d; P.outer = dm.T;
    e = launch_dct_pass<ST, 1>(p, P, g, st);
    if (e != cudaSuccess) return e;
    // t axis + band split
    P.src[0] = p->buf.scratchB; P.dst = nullptr; P.mat_t = p->basis_t[0];
    P.n = dm.T; P.inner = dm.H * dm.W * dm.d; P.outer = 1;
    e = launch_dct_pass<ST, 2>(p, P, g, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t ffk_forward_transform(ff_plan* p, const void* Q, const void* K, const void* V, bool want_energy, cudaStream_t st) {
  return p->dm.fp32 ? forward_transform_t<float>(p, Q, K, V, want_energy, st)
                    : forward_transform_t<__nv_bfloat16>(p, Q, K, V, want_energy, st);
}

template <typename ST>
static cudaError_t attention_simt_t(ff_plan* p, int band_bits, cudaStream_t st) {
  const FFDims& dm = p->dm;
  // the longest of the bands asked for, in tiles of 64 query rows (strided mid band: per residue class)
  auto tiles = [](long long n) { return (n + AT - 1) / AT; };
  long long most = 0;
  if ((band_bits & FF_BAND_LOW) && tiles(dm.Nbar) > most) most = tiles(dm.Nbar);
  if (band_bits & FF_BAND_MID) {
    const long long per = dm.nb / dm.s, rem = dm.nb % dm.s;
    const long long b = dm.b < dm.Nmid ? dm.b : dm.Nmid;
    const long long t = dm.pattern == FF_MID_STRIDED ? rem * tiles((per + 1) * b) + (dm.s - rem) * tiles(per * b) : tiles(dm.Nmid);
    if (dm.Nmid > 0 && t > most) most = t;
  }
  if ((band_bits & FF_BAND_HIGH) && tiles(dm.Nhigh) > most) most = tiles(dm.Nhigh);
  if (most == 0) return cudaSuccess;                 // (only an empty band was asked for)
  const unsigned bands = (band_bits & FF_BAND_LOW) ? 3 : ((band_bits & FF_BAND_HIGH) ? 2 : 1);
  p->launches += 1;
  // scored pairs, if every head ran every band asked for
  long long rows = 0, pairs = 0;
  auto add = [&](long long n, long long keys) { rows = n > rows ? n : rows; pairs += dm.BH * n * (keys < n ? keys : n); };
  if (band_bits & FF_BAND_LOW) add(dm.Nbar, dm.Nbar);
  if (band_bits & FF_BAND_MID) add(dm.Nmid, (dm.nb + dm.s - 1) / dm.s * dm.b);
  if (band_bits & FF_BAND_HIGH) add(dm.Nhigh, 2LL * dm.R + 1);
  if (pairs <= ROW_PAIRS && !((band_bits & FF_BAND_MID) && dm.pattern == FF_MID_ANCHOR)) {
    const dim3 grid((unsigned)((rows + ROW_WARPS - 1) / ROW_WARPS), (unsigned)dm.BH, bands);
    switch (dm.d / 32) {
      case 1: return ff_launch(attention_row_kernel<ST, 1>, grid, dim3(ROW_WARPS * 32), 0, st, p->buf, dm, band_bits);
      case 2: return ff_launch(attention_row_kernel<ST, 2>, grid, dim3(ROW_WARPS * 32), 0, st, p->buf, dm, band_bits);
      case 3: return ff_launch(attention_row_kernel<ST, 3>, grid, dim3(ROW_WARPS * 32), 0, st, p->buf, dm, band_bits);
      default: return ff_launch(attention_row_kernel<ST, 4>, grid, dim3(ROW_WARPS * 32), 0, st, p->buf, dm, band_bits);
    }
  }
  const dim3 grid((unsigned)most, (unsigned)dm.BH, bands);
  switch (dm.d / 32) {
    case 1: return ff_launch(attention_simt_kernel<ST, 1>, grid, dim3(AT_THREADS), AtShape<1>::smem, st, p->buf, dm, band_bits);
    case 2: return ff_launch(attention_simt_kernel<ST, 2>, grid, dim3(AT_THREADS), AtShape<2>::smem, st, p->buf, dm, band_bits);
    case 3: return ff_launch(attention_simt_kernel<ST, 3>, grid, dim3(AT_THREADS), AtShape<3>::smem, st, p->buf, dm, band_bits);
    default: return ff_launch(attention_simt_kernel<ST, 4>, grid, dim3(AT_THREADS), AtShape<4>::smem, st, p->buf, dm, band_bits);
  }
}

cudaError_t ffk_attention_simt(ff_plan* p, int band_bits, cudaStream_t st) {
  return p->dm.fp32 ? attention_simt_t<float>(p, band_bits, st) : attention_simt_t<__nv_bfloat16>(p, band_bits, st);
}

// Tensor-core inverse: exchange + recombination into the three-byte grids (or one of fp32, ff_fp32_grid), then the axis passes.
static cudaError_t exchange_inverse_tc(ff_plan* p, void* out, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int G = p->dct_group;
  cudaError_t e = cudaSuccess;
  for (int h0 = 0; h0 < dm.BH; h0 += G) {
    const int g = (dm.BH - h0 < G) ? dm.BH - h0 : G;
    const size_t grid_bytes = ((size_t)G * dm.N * dm.d * 2 + 255) / 256 * 256;
    __nv_bfloat16* ghi = (__nv_bfloat16*)p->buf.scratchA;
    uint8_t* glo = ff_fp32_grid(dm) ? nullptr : (uint8_t*)p->buf.scratchA + grid_bytes;
    if (p->xtc_ok) {
      // mid and high bands on the tensor cores, the fp32 low band with its own kernel
      e = ffk_exchange_low(p, h0, g, ghi, glo, st);
      if (e == cudaSuccess) e = ffk_exchange_tc(p, h0, g, ghi, glo, st);
    } else if (glo) {
      e = dm.d == 128 ? launch_exchange<__nv_bfloat16, 4>(p, g, h0, ghi, glo, st) : launch_exchange<__nv_bfloat16, 2>(p, g, h0, ghi, glo, st);
    } else {
      e = dm.d == 128 ? launch_exchange<__nv_bfloat16, 4>(p, g, h0, p->buf.scratchA, nullptr, st)
                      : launch_exchange<__nv_bfloat16, 2>(p, g, h0, p->buf.scratchA, nullptr, st);
    }
    if (e != cudaSuccess) return e;
    e = ffk_inverse_transform_tc(p, h0, g, out, st);
    if (e != cudaSuccess) return e;
    if (p->pipe_out) {                             // host-buffer entry point: hand this group of heads to the copy stream
      cudaEvent_t ev = p->ev_copy[FF_COPY_EVENTS + h0 / G];
      e = cudaEventRecord(ev, st);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(p->copy_stream, ev, 0);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync((char*)p->pipe_out_host + (size_t)h0 * p->pipe_head_bytes, (const char*)out + (size_t)h0 * p->pipe_head_bytes,
                            (size_t)g * p->pipe_head_bytes, cudaMemcpyDeviceToHost, p->copy_stream);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

template <typename ST>
static cudaError_t exchange_inverse_t(ff_plan* p, void* out, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int G = p->lay.group;
  DctPassParams P{};
  P.BH = dm.BH; P.N_d = dm.N * dm.d; P.dm = dm;
  for (int h0 = 0; h0 < dm.BH; h0 += G) {
    const int g = (dm.BH - h0 < G) ? dm.BH - h0 : G;
    cudaError_t e;
    switch (dm.d / 32) {
      case 1: e = launch_exchange<ST, 1>(p, g, h0, p->buf.scratchA, nullptr, st); break;
      case 2: e = launch_exchange<ST, 2>(p, g, h0, p->buf.scratchA, nullptr, st); break;
      case 3: e = launch_exchange<ST, 3>(p, g, h0, p->buf.scratchA, nullptr, st); break;
      default: e = launch_exchange<ST, 4>(p, g, h0, p->buf.scratchA, nullptr, st); break;
    }
    if (e != cudaSuccess) return e;
    // inverse along t, h, w with the transposed matrices
    if (vol_fits(dm)) {
      VolParams P{};
      P.src[0] = p->buf.scratchA; P.out = out; P.dm = dm; P.group_start = h0;
      for (int a = 0; a < 3; ++a) P.mat_t[a] = p->basis[a];
      p->launches += 1;
      e = ff_launch(vol_fine(dm, p->sm_count) ? dct_volume_kernel<ST, true, 2> : dct_volume_kernel<ST, true, 8>, dim3((unsigned)(dm.d / VOL_CH), (unsigned)g), dim3(VOL_THREADS), vol_smem(dm), st, P);
      if (e != cudaSuccess) return e;
      continue;
    }
    P.group_start = h0;
    P.src[0] = p->buf.scratchA; P.dst = p->buf.scratchB; P.mat_t = p->basis[0];
    P.n = dm.T; P.inner = dm.H * dm.W * dm.d; P.outer = 1;
    e = launch_dct_pass<ST, 1>(p, P, g, st);
    if (e != cudaSuccess) return e;
    P.src[0] = p->buf.scratchB; P.dst = p->buf.scratchA; P.mat_t = p->basis[1];
    P.n = dm.H; P.inner = dm.W * dm.d; P.outer = dm.T;
    e = launch_dct_pass<ST, 1>(p, P, g, st);
    if (e != cudaSuccess) return e;
    P.src[0] = p->buf.scratchA; P.dst = out; P.mat_t = p->basis[2];
    P.n = dm.W; P.inner = dm.d; P.outer = dm.T * dm.H;
    e = launch_dct_pass<ST, 3>(p, P, g, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t ffk_exchange_inverse(ff_plan* p, void* out, cudaStream_t st) {
  if (p->dct_tc_ok && !(p->attn_impl & 2)) return exchange_inverse_tc(p, out, st);
  return p->dm.fp32 ? exchange_inverse_t<float>(p, out, st) : exchange_inverse_t<__nv_bfloat16>(p, out, st);
}

cudaError_t ffk_simt_init() {
  cudaError_t e = cudaSuccess;
  const int most = 144 * 1024;       // the largest: a 72 KB volume and a 128 x 128 matrix
#define FF_SET(...) if (e == cudaSuccess) e = cudaFuncSetAttribute(__VA_ARGS__, cudaFuncAttributeMaxDynamicSharedMemorySize, most)
#define FF_SET_D(T, D)                                                                         \
  FF_SET(attention_simt_kernel<T, D>); FF_SET(exchange_recombine_kernel<T, D, float>)
#define FF_SET_T(T)                                                                            \
  FF_SET(dct_pass_kernel<T, 0>); FF_SET(dct_pass_kernel<T, 1>); FF_SET(dct_pass_kernel<T, 2>); FF_SET(dct_pass_kernel<T, 3>); \
  FF_SET(dct_volume_kernel<T, false, 2>); FF_SET(dct_volume_kernel<T, true, 2>);               \
  FF_SET(dct_volume_kernel<T, false, 8>); FF_SET(dct_volume_kernel<T, true, 8>);               \
  FF_SET_D(T, 1); FF_SET_D(T, 2); FF_SET_D(T, 3); FF_SET_D(T, 4)
  FF_SET_T(float); FF_SET_T(__nv_bfloat16);
  FF_SET(exchange_recombine_kernel<__nv_bfloat16, 2, __nv_bfloat16>); FF_SET(exchange_recombine_kernel<__nv_bfloat16, 4, __nv_bfloat16>);
#undef FF_SET_T
#undef FF_SET_D
#undef FF_SET
  return e;
}
