// Summary tokens ("Cross-band residual exchange"), the attention of a short pooled low band, and the low band's part of
// the exchange.
//
// Summaries: S = U_l Pool(Y^(l)), segment j of a band's n working tokens = [floor(j n / m), max(a + 1, floor((j + 1) n / m))).
// A block sums one piece of a segment (16-byte loads, eight rows in flight per thread); the piece that finishes last
// adds the pieces up, projects the mean and writes the token twice: fp32 for the low band's exchange and bf16 hi + lo in
// the operand layout of the tensor-core exchange.  One launch without cleared buffers or atomics on data, bound by
// reading Y (N d bytes 2 per head).
//
// Short pooled low bands (below a 128-row tile) take their attention along: a segment holds a few pooled tokens, so the
// block that needs them computes their rows, dense softmax over all pooled tokens, one warp per row.  As a launch of
// its own in front of the tensor-core kernel it cost 6 - 27 us of the step for microseconds of work.
#include "ff_bands.cuh"
#include "ff_internal.h"
#include "ff_sm100.cuh"
#include "ff_three_byte.cuh"

namespace {

constexpr int SUM_THREADS = 256;
constexpr int SUM_WARPS = SUM_THREADS / 32;
constexpr int LOW_MAX = 128;             // pooled low bands below this are attended here

struct SumParams {
  FFBuffers buf;
  FFDims dm;
  const float* U;
  int identity_u;
  unsigned* tickets;      // [BH][3][m], zero between launches
  int pieces;             // most pieces per segment (grid.x = m * pieces)
  int piece_rows;         // rows a piece should have
  int low_attention;
  int nkeys;              // rows of an operand image (0: no image wanted)
};

// Row `row` of the pooled low band's dense attention by a whole warp, lane + 32 j = channel: scores of eight keys at a
// time reduced side by side, merged into the running softmax as a group.
template <int DPL>
__device__ __forceinline__ void low_row(const FFBuffers& buf, const FFDims& dm, int bh, long long row, int lane, float (&o)[DPL]) {
  const int d = DPL * 32;
  const int n = (int)dm.Nbar;
  const float* Q = buf.pooled + ((size_t)bh * n + row) * d + lane;
  const float* K = buf.pooled + ((size_t)dm.BH + bh) * n * d + lane;
  const float* V = buf.pooled + ((size_t)2 * dm.BH + bh) * n * d + lane;
  const float scale = rsqrtf((float)d);
  float q[DPL], mx = -INFINITY, den = 0.f;
#pragma unroll
  for (int j = 0; j < DPL; ++j) { q[j] = Q[32 * j]; o[j] = 0.f; }
  for (int k0 = 0; k0 < n; k0 += 8) {
    float sc[8], v[8][DPL];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const size_t at = (size_t)(k0 + k < n ? k0 + k : k0) * d;
      float part = 0.f;
#pragma unroll
      for (int j = 0; j < DPL; ++j) { part = fmaf(q[j], K[at + 32 * j], part); v[k][j] = V[at + 32 * j]; }
      sc[k] = part;
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
#pragma unroll
      for (int k = 0; k < 8; ++k) sc[k] += __shfl_xor_sync(0xffffffffu, sc[k], s);
    float nm = mx;
#pragma unroll
    for (int k = 0; k < 8; ++k) { sc[k] = k0 + k < n ? sc[k] * scale : -INFINITY; nm = fmaxf(nm, sc[k]); }
    const float corr = expf(mx - nm);
    den *= corr;
#pragma unroll
    for (int j = 0; j < DPL; ++j) o[j] *= corr;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float p = expf(sc[k] - nm);                       // (0 for the keys past the end)
      den += p;
#pragma unroll
      for (int j = 0; j < DPL; ++j) o[j] = fmaf(p, v[k][j], o[j]);
    }
    mx = nm;
  }
#pragma unroll
  for (int j = 0; j < DPL; ++j) o[j] /= den;
}

// Row `key` of the head's operand images: 64 channels per 128-byte row, 16-byte chunks XOR-swizzled with the row.
__device__ __forceinline__ void store_image(const SumParams& P, int bh, int key, int c, float v) {
  const __nv_bfloat16 hi = __float2bfloat16_rn(v);
  const __nv_bfloat16 lo = __float2bfloat16_rn(v - __bfloat162float(hi));
  const int half = c >> 6, ck = c & 63;
  uint8_t* img = P.buf.zimg + (size_t)bh * 4 * P.nkeys * 128;
  const uint32_t off = half * (P.nkeys * 128) + key * 128 + ((((ck >> 3) ^ (key & 7)) << 4) | ((ck & 7) << 1));
  *(__nv_bfloat16*)(img + off) = hi;
  *(__nv_bfloat16*)(img + 2 * P.nkeys * 128 + off) = lo;
}

template <typename ST, int DPL>
__global__ void __launch_bounds__(SUM_THREADS) summary_kernel(const __grid_constant__ SumParams P) {
  constexpr int d = DPL * 32, vecs = d / 8;          // 8-channel vectors per row
  constexpr int nrs = SUM_THREADS / vecs;            // rows in flight
  __shared__ float red[nrs * d];
  __shared__ float mean[d];
  __shared__ bool last;
  ff_pdl_wait();
  const FFDims& dm = P.dm;
  const int m = dm.m;
  const int j = blockIdx.x / P.pieces, piece = blockIdx.x % P.pieces, band = blockIdx.y, bh = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const BandView<ST> v = band_view<ST>(P.buf, dm, bh, band);
  const bool attend = band == 0 && P.low_attention && v.compressed;
  const long long a = ((long long)j * v.n) / m;
  long long e = ((long long)(j + 1) * v.n) / m;
  if (e < a + 1) e = a + 1;
  int pieces = attend || v.n == 0 ? 1 : (int)((e - a + P.piece_rows - 1) / P.piece_rows);
  if (pieces > P.pieces) pieces = P.pieces;
  if (piece >= pieces) return;
  const size_t seg = ((size_t)bh * 3 + band) * m + j;
  int nred = nrs;                                    // rows of `red` in use
  if (v.n == 0) {
    // empty band (two-band layer): its tokens are zero and never attended
    for (int i = tid; i < d; i += SUM_THREADS) red[i] = 0.f;
    nred = 1;
  } else if (attend) {
    float acc[DPL];
#pragma unroll
    for (int i = 0; i < DPL; ++i) acc[i] = 0.f;
    for (long long row = a + warp; row < e; row += SUM_WARPS) {
      float o[DPL];
      low_row<DPL>(P.buf, dm, bh, row, lane, o);
      float* y = P.buf.y_low + ((size_t)bh * dm.Nbar + row) * d + lane;
#pragma unroll
      for (int i = 0; i < DPL; ++i) { y[32 * i] = o[i]; acc[i] += o[i]; }
    }
#pragma unroll
    for (int i = 0; i < DPL; ++i) red[warp * d + lane + 32 * i] = acc[i];
    nred = SUM_WARPS;
  } else {
    const long long chunk = (e - a + pieces - 1) / pieces;
    const long long r0 = a + piece * chunk, r1 = r0 + chunk < e ? r0 + chunk : e;
    const int vec = tid % vecs, sub = tid / vecs;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (sub < nrs) {
      long long p = r0 + sub;
      if (v.f32 || sizeof(ST) == 4) {
        const float* base = (v.f32 ? v.f32 : (const float*)v.st) + vec * 8;
        auto add = [&](const float4& x0, const float4& x1) {
          acc[0] += x0.x; acc[1] += x0.y; acc[2] += x0.z; acc[3] += x0.w;
          acc[4] += x1.x; acc[5] += x1.y; acc[6] += x1.z; acc[7] += x1.w;
        };
        for (; p + 3 * nrs < r1; p += 4 * nrs) {
          float4 x[8];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            x[2 * u] = __ldcs((const float4*)(base + (size_t)(p + u * nrs) * d));
            x[2 * u + 1] = __ldcs((const float4*)(base + (size_t)(p + u * nrs) * d + 4));
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) add(x[2 * u], x[2 * u + 1]);
        }
        for (; p < r1; p += nrs) add(*(const float4*)(base + (size_t)p * d), *(const float4*)(base + (size_t)p * d + 4));
      } else {
        const __nv_bfloat16* base = (const __nv_bfloat16*)v.st + vec * 8;
        auto add = [&](const uint4& x) {
          const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            acc[2 * i] += __uint_as_float(w[i] << 16);
            acc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
          }
        };
        for (; p + 7 * nrs < r1; p += 8 * nrs) {
          uint4 x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = __ldcs((const uint4*)(base + (size_t)(p + u * nrs) * d));
#pragma unroll
          for (int u = 0; u < 8; ++u) add(x[u]);
        }
        for (; p < r1; p += nrs) add(*(const uint4*)(base + (size_t)p * d));
      }
      *(float4*)(red + sub * d + vec * 8) = make_float4(acc[0], acc[1], acc[2], acc[3]);
      *(float4*)(red + sub * d + vec * 8 + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
  }
  __syncthreads();
  float sum = 0.f;
  if (tid < d) for (int i = 0; i < nred; ++i) sum += red[i * d + tid];
  if (pieces > 1) {
    float* part = P.buf.sum_part + seg * P.pieces * d;
    if (tid < d) part[(size_t)piece * d + tid] = sum;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(P.tickets + seg, 1u) == (unsigned)pieces - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (tid == 0) P.tickets[seg] = 0;
    if (tid < d) {
      sum = 0.f;
      for (int i = 0; i < pieces; ++i) sum += __ldcg(part + (size_t)i * d + tid);
    }
  }
  if (tid < d) mean[tid] = sum / (float)(e - a);
  __syncthreads();
  float* S = P.buf.summary + seg * d;
  if (P.identity_u) {
    if (tid < d) {
      S[tid] = mean[tid];
      if (P.nkeys) store_image(P, bh, band * m + j, tid, mean[tid]);
    }
  } else {
    // one output channel per warp at a time: coalesced rows of U
    for (int c = warp; c < d; c += SUM_WARPS) {
      const float* u = P.U + ((size_t)band * d + c) * d + lane;
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < DPL; ++i) s = fmaf(u[32 * i], mean[lane + 32 * i], s);
      s = warp_sum(s);
      if (lane == 0) {
        S[c] = s;
        if (P.nkeys) store_image(P, bh, band * m + j, c, s);
      }
    }
  }
  if (P.nkeys && band == 2 && j == m - 1)                    // the rows that round the images up to a k-step
    for (int i = tid; i < (P.nkeys - 3 * m) * d; i += SUM_THREADS) store_image(P, bh, 3 * m + i / d, i % d, 0.f);
}

// Low band of the tensor-core inverse ("Cross-band residual exchange", "Reconstruction"): exchange + recombination of the
// low band's coefficients into the three-byte grids (F32: into one of fp32).  A head that executes the low band has one pooled output row for
// every r consecutive coefficient ranks, so its update is computed once and written r times; other heads carry V~ low,
// one row per rank.  Eight lanes share a row (lane s holds channels 4 s + 32 i .. + 3), so that a score takes three
// shuffles for four rows at once: with a whole warp per row the kernel was bound by its five shuffles per score and row
// (131 072 rows of 64 channels, 16 keys: 106 us).  Scores of four or eight keys are reduced side by side and merged into the
// running softmax as a group, exponentials by ex2.approx on scores in log2 units, like the tensor-core kernel's.
constexpr int XL_WARPS = 8;
template <int DPL, bool F32>
__global__ void __launch_bounds__(XL_WARPS * 32, 2) exchange_low_kernel(FFBuffers buf, FFDims dm, int bh0, __nv_bfloat16* grid_hi,
                                                                      uint8_t* grid_lo, float* grid_f32, int rounds) {
  extern __shared__ float4 Z[];                 // the summaries of the other bands, [keys][d]
  constexpr int d = DPL * 32, V = DPL;          // float4 per lane and row
  constexpr int KB = DPL >= 4 ? 4 : 8;          // keys scored side by side (registers)
  ff_pdl_wait();
  const int gi = blockIdx.y, bh = bh0 + gi, m = dm.m;
  // the summaries of the other bands: the mid band's (none if it is empty), then the high band's
  const int k_first = dm.Nmid == 0 ? 2 * m : m, nkeys = 3 * m - k_first;
  const float4* src_z = (const float4*)(buf.summary + ((size_t)bh * 3 * m + k_first) * d);
#pragma unroll 4
  for (int i = threadIdx.x; i < nkeys * (d / 4); i += XL_WARPS * 32) Z[i] = src_z[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, s = lane & 7;
  const bool exec = buf.alloc[bh] & FF_BAND_LOW;
  const float* src = exec ? buf.y_low + (size_t)bh * dm.Nbar * d : buf.spec_low + ((size_t)2 * dm.BH + bh) * dm.Nlow * d;
  const int rows = (int)(exec ? dm.Nbar : dm.Nlow);
  const int rep = exec ? dm.r : 1;
  const float scale = rsqrtf((float)d) * 1.4426950408889634f;
  for (int round = 0; round < rounds; ++round) {
    const int row0 = ((int)blockIdx.x * rounds + round) * XL_WARPS * 4 + warp * 4;
    if (row0 >= rows) return;
    const int row = row0 + (lane >> 3);
    const bool live = row < rows;
    const float4* yr = (const float4*)(src + (size_t)(live ? row : row0) * d) + s;
    float4 y[V], acc[V];
#pragma unroll
    for (int i = 0; i < V; ++i) { y[i] = yr[8 * i]; acc[i] = make_float4(0.f, 0.f, 0.f, 0.f); }
    float mx = -INFINITY, den = 0.f;
    for (int k0 = 0; k0 < nkeys; k0 += KB) {
      float sc[KB];
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        const float4* z = Z + (size_t)(k0 + k < nkeys ? k0 + k : 0) * (d / 4) + s;
        float part = 0.f;
#pragma unroll
        for (int i = 0; i < V; ++i) {
          const float4 zz = z[8 * i];
          part = fmaf(y[i].x, zz.x, part); part = fmaf(y[i].y, zz.y, part);
          part = fmaf(y[i].z, zz.z, part); part = fmaf(y[i].w, zz.w, part);
        }
        sc[k] = part;
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < KB; ++k) sc[k] += __shfl_xor_sync(0xffffffffu, sc[k], o);
      float nm = mx;
#pragma unroll
      for (int k = 0; k < KB; ++k) { sc[k] = k0 + k < nkeys ? sc[k] * scale : -INFINITY; nm = fmaxf(nm, sc[k]); }
      const float corr = sm100::ex2(mx - nm);
      den *= corr;
#pragma unroll
      for (int i = 0; i < V; ++i) { acc[i].x *= corr; acc[i].y *= corr; acc[i].z *= corr; acc[i].w *= corr; }
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        const float p = sm100::ex2(sc[k] - nm);               // (0 for the keys past the end)
        const float4* z = Z + (size_t)(k0 + k < nkeys ? k0 + k : 0) * (d / 4) + s;
        den += p;
#pragma unroll
        for (int i = 0; i < V; ++i) {
          const float4 zz = z[8 * i];
          acc[i].x = fmaf(p, zz.x, acc[i].x); acc[i].y = fmaf(p, zz.y, acc[i].y);
          acc[i].z = fmaf(p, zz.z, acc[i].z); acc[i].w = fmaf(p, zz.w, acc[i].w);
        }
      }
      mx = nm;
    }
    const float inv = nkeys > 0 ? 1.f / den : 0.f;
    // the value, in three bytes or as it is, at every rank the row stands for
    uint2 hi[V]; uint32_t lo[V];
#pragma unroll
    for (int i = 0; i < V; ++i) {
      if (F32) {
        y[i] = make_float4(fmaf(acc[i].x, inv, y[i].x), fmaf(acc[i].y, inv, y[i].y), fmaf(acc[i].z, inv, y[i].z), fmaf(acc[i].w, inv, y[i].w));
        continue;
      }
      const uint32_t u0 = ff_round24(fmaf(acc[i].x, inv, y[i].x)), u1 = ff_round24(fmaf(acc[i].y, inv, y[i].y));
      const uint32_t u2 = ff_round24(fmaf(acc[i].z, inv, y[i].z)), u3 = ff_round24(fmaf(acc[i].w, inv, y[i].w));
      hi[i] = make_uint2(ff_hi2(u0, u1), ff_hi2(u2, u3));
      lo[i] = ff_lo4(u0, u1, u2, u3);
    }
    if (!live) continue;
    unsigned p = (unsigned)row * (unsigned)rep;
    const unsigned Lw = (unsigned)dm.L[2], Lh = (unsigned)dm.L[1];
    unsigned kw = p % Lw, kh = p / Lw % Lh, kt = p / (Lw * Lh);
    for (int i = 0; i < rep && p < (unsigned)dm.Nlow; ++i, ++p) {
      const size_t o = ((size_t)gi * dm.N + ((size_t)kt * dm.H + kh) * dm.W + kw) * d + 4 * s;
#pragma unroll
      for (int q = 0; q < V; ++q) {
        if (F32) { *(float4*)(grid_f32 + o + 32 * q) = y[q]; continue; }
        *(uint2*)(grid_hi + o + 32 * q) = hi[q];
        *(uint32_t*)(grid_lo + o + 32 * q) = lo[q];
      }
      if (++kw == Lw) { kw = 0; if (++kh == Lh) { kh = 0; ++kt; } }
    }
  }
}

// Rows a piece of a segment should have: about the three blocks an SM holds over all bands while that leaves 128 rows or
// more (a block's own latency is three to four microseconds), at most 1024 (256 KB of bf16 at head_dim 128).
int piece_rows(const FFDims& dm) {
  const long long rows = (long long)dm.BH * dm.N / (FF_B200_SMS * 3);
  return (int)(rows < 128 ? 128 : (rows > 1024 ? 1024 : rows));
}

}  // namespace

int ffk_summary_pieces(const FFDims& dm) {
  if (dm.m < 1) return 1;
  long long longest = dm.Nhigh > dm.Nmid ? dm.Nhigh : dm.Nmid;
  if (dm.Nlow > longest) longest = dm.Nlow;
  const long long n = (longest / dm.m + piece_rows(dm)) / piece_rows(dm);
  return (int)(n < 1 ? 1 : (n > 64 ? 64 : n));
}

bool ffk_low_in_summary(const ff_plan* p) {
  const bool tc = p->tc_ok && !(p->attn_impl & 1);
  return p->dm.m > 0 && p->dm.Nbar < LOW_MAX && !(tc && p->low_tc_ok);
}

cudaError_t ffk_summaries(ff_plan* p, cudaStream_t st) {
  const FFDims& dm = p->dm;
  SumParams P{};
  P.buf = p->buf; P.dm = dm; P.U = p->U; P.identity_u = p->identity_u;
  P.tickets = p->tickets + 64;
  P.pieces = ffk_summary_pieces(dm); P.piece_rows = piece_rows(dm);
  P.low_attention = ffk_low_in_summary(p) ? 1 : 0;
  P.nkeys = p->xtc_ok ? ff_exchange_keys(dm.m) : 0;
  const dim3 grid((unsigned)(dm.m * P.pieces), 3, (unsigned)dm.BH), block(SUM_THREADS);
  p->launches += 1;
#define FF_SUM(T)                                                              \
  switch (dm.d / 32) {                                                         \
    case 1: return ff_launch(summary_kernel<T, 1>, grid, block, 0, st, P);     \
    case 2: return ff_launch(summary_kernel<T, 2>, grid, block, 0, st, P);     \
    case 3: return ff_launch(summary_kernel<T, 3>, grid, block, 0, st, P);     \
    default: return ff_launch(summary_kernel<T, 4>, grid, block, 0, st, P);    \
  }
  if (dm.fp32) FF_SUM(float)
  FF_SUM(__nv_bfloat16)
#undef FF_SUM
}

cudaError_t ffk_exchange_low(ff_plan* p, int h0, int g, void* grid_hi, void* grid_lo, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const size_t smem = (size_t)2 * dm.m * dm.d * sizeof(float);           // at most 32 KB (m <= 32)
  const long long per_round = XL_WARPS * 4;
  long long rounds = dm.Nlow * g / (per_round * 8 * p->sm_count);        // up to eight, fewer while the launch is small
  rounds = rounds < 1 ? 1 : (rounds > 8 ? 8 : rounds);
  const dim3 grid((unsigned)((dm.Nlow + per_round * rounds - 1) / (per_round * rounds)), (unsigned)g);
  p->launches += 1;
  auto* kernel = grid_lo ? (dm.d == 128 ? exchange_low_kernel<4, false> : exchange_low_kernel<2, false>)
                         : (dm.d == 128 ? exchange_low_kernel<4, true> : exchange_low_kernel<2, true>);
  return ff_launch(kernel, grid, dim3(XL_WARPS * 32), smem, st, p->buf, dm, h0, (__nv_bfloat16*)grid_hi, (uint8_t*)grid_lo, (float*)grid_hi,
                   (int)rounds);
}
