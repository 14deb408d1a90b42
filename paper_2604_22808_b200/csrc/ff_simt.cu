// Generic FP32-arithmetic kernels of the FreqFormer forward.  They cover every configuration the
// ABI accepts (any storage type, head_dim, block/stride/radius) and are the path of the fp32
// workload; the bf16 workloads replace the attention step with the tensor-core kernel.
#include "ff_bands.cuh"
#include "ff_internal.h"

namespace {

// ------------------------------------------------------------------------------------------------
// One axis of the separable transform ("Separable spectral decomposition"):
//   out[o][a][c] = sum_b Mat[a][b] * in[o][b][c],   a, b in [0,n), c in [0,inner), o in [0,outer)
// with the tensor-head as the slowest index.  Mat is C (forward) or C^T (inverse).
// MODE 0: `in` is the caller's Q/K/V (storage type), `out` an fp32 scratch grid.
// MODE 1: fp32 scratch -> fp32 scratch.
// MODE 2: fp32 scratch -> band-major coefficient buffers (forward, last axis = t): the rank of
//         every coefficient is evaluated in registers from the nested-box closed form.
// MODE 3: fp32 scratch -> the caller's `out` tensor (storage type).
// ------------------------------------------------------------------------------------------------
constexpr int DCT_IC = 64;       // columns per CTA tile
constexpr int DCT_THREADS = 256;

struct DctPassParams {
  const void* src[3];   // MODE 0: Q, K, V; otherwise src[0] = scratch
  void* dst;            // MODE 0/1: scratch; MODE 3: out tensor
  const float* mat;     // [n][n]
  int n, inner, outer;
  int group_start;      // first tensor-head index of this launch
  int BH;
  long long N_d;        // elements per tensor-head
  // MODE 2
  FFDims dm;
  float* spec_low; void* spec_mid; void* spec_high;
  double* clear;        // MODE 0, first launch of a routed call: the band energies, cleared for the sums that follow
};

template <typename ST, int MODE>
__global__ void __launch_bounds__(DCT_THREADS) dct_pass_kernel(const DctPassParams P) {
  ff_pdl_wait();
  extern __shared__ float smem[];
  if (MODE == 0 && P.clear && blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = threadIdx.x; i < P.dm.B * 3 * P.dm.d; i += DCT_THREADS) P.clear[i] = 0.0;
  const int n = P.n;
  const int npad = (n + 7) & ~7;
  float* matT = smem;                       // [b][npad]: matT[b][a] = Mat[a][b]
  float* tile = smem + (size_t)n * npad;    // [b][DCT_IC]
  const int chunks = (P.inner + DCT_IC - 1) / DCT_IC;
  const int o = blockIdx.x / chunks;
  const int c0 = (blockIdx.x % chunks) * DCT_IC;
  const int gi = blockIdx.y;                // tensor-head inside the group
  const int th = P.group_start + gi;        // global tensor-head index: tensor * BH + bh
  const int tid = threadIdx.x;

  for (int idx = tid; idx < n * npad; idx += DCT_THREADS) {
    const int b = idx / npad, a = idx % npad;
    matT[idx] = (a < n) ? P.mat[(size_t)a * n + b] : 0.f;
  }
  const size_t line0 = ((size_t)o * n) * P.inner + c0;
  if (MODE == 0) {
    const ST* src = (const ST*)P.src[th / P.BH] + (size_t)(th % P.BH) * P.N_d + line0;
    for (int idx = tid; idx < n * DCT_IC; idx += DCT_THREADS) {
      const int b = idx / DCT_IC, c = idx % DCT_IC;
      tile[idx] = (c0 + c < P.inner) ? ldf<ST>(src + (size_t)b * P.inner + c) : 0.f;
    }
  } else {
    const float* src = (const float*)P.src[0] + (size_t)gi * P.N_d + line0;
    for (int idx = tid; idx < n * DCT_IC; idx += DCT_THREADS) {
      const int b = idx / DCT_IC, c = idx % DCT_IC;
      tile[idx] = (c0 + c < P.inner) ? src[(size_t)b * P.inner + c] : 0.f;
    }
  }
  __syncthreads();

  const int agroups = npad / 8;
  for (int w = tid; w < agroups * (DCT_IC / 4); w += DCT_THREADS) {
    const int ag = w / (DCT_IC / 4), cg = w % (DCT_IC / 4);
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int b = 0; b < n; ++b) {
      const float4 x = *(const float4*)(tile + b * DCT_IC + cg * 4);
      const float4 m0 = *(const float4*)(matT + b * npad + ag * 8);
      const float4 m1 = *(const float4*)(matT + b * npad + ag * 8 + 4);
      const float mm[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
      const float xx[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(mm[i], xx[j], acc[i][j]);
    }
    const int c = c0 + cg * 4;
    if (c >= P.inner) continue;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int a = ag * 8 + i;
      if (a >= n) break;
      if (MODE == 0 || MODE == 1) {
        float* dst = (float*)P.dst + (size_t)gi * P.N_d + ((size_t)o * n + a) * P.inner + c;
        *(float4*)dst = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      } else if (MODE == 3) {
        ST* dst = (ST*)P.dst + (size_t)th * P.N_d + ((size_t)o * n + a) * P.inner + c;
#pragma unroll
        for (int j = 0; j < 4; ++j) stf<ST>(dst + j, acc[i][j]);
      } else {  // MODE 2: a = k_t, column = (k_h, k_w, channel)
        const int d = P.dm.d;
        const int ch = c % d;
        const int kw = (c / d) % P.dm.W;
        const int kh = c / (d * P.dm.W);
        long long rank;
        const int band = ff_band_rank_of(P.dm, a, kh, kw, &rank);
        const int tensor = th / P.BH, bh = th % P.BH;
        if (band == 0) {
          float* dst = P.spec_low + (((size_t)tensor * P.BH + bh) * P.dm.Nlow + rank) * d + ch;
          *(float4*)dst = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        } else {
          const long long nl = (band == 1) ? P.dm.Nmid : P.dm.Nhigh;
          ST* dst = (ST*)(band == 1 ? P.spec_mid : P.spec_high) + (((size_t)tensor * P.BH + bh) * nl + rank) * d + ch;
#pragma unroll
          for (int j = 0; j < 4; ++j) stf<ST>(dst + j, acc[i][j]);
        }
      }
    }
  }
}

template <typename ST, int MODE>
cudaError_t launch_dct_pass(const DctPassParams& P, int group, cudaStream_t st) {
  const int npad = (P.n + 7) & ~7;
  const size_t smem = ((size_t)P.n * npad + (size_t)P.n * DCT_IC) * sizeof(float);
  const int chunks = (P.inner + DCT_IC - 1) / DCT_IC;
  dim3 grid((unsigned)((size_t)P.outer * chunks), (unsigned)group);
  return ff_launch(dct_pass_kernel<ST, MODE>, grid, dim3(DCT_THREADS), smem, st, P);
}

// ------------------------------------------------------------------------------------------------
// Band operators ("Hierarchical frequency-domain attention"), one warp per query row, online
// softmax with the score reduced by warp shuffles.  The key set of a row is generated from its
// rank: all pooled tokens (low), the blocks at block distance 0 mod s (mid), the window
// |p - p'| <= R (high).
// ------------------------------------------------------------------------------------------------
constexpr int ATT_WARPS = 8;

template <typename KT, int DPL>   // DPL = d / 32 channels per lane
__device__ __forceinline__ void attend_range(const KT* __restrict__ Kp, const KT* __restrict__ Vp, long long k0,
                                             long long k1, int d, const float (&q)[DPL], float scale, float& mx,
                                             float& den, float (&o)[DPL], int lane) {
  for (long long k = k0; k < k1; ++k) {
    const KT* kr = Kp + (size_t)k * d;
    float part = 0.f;
#pragma unroll
    for (int j = 0; j < DPL; ++j) part = fmaf(q[j], ldf<KT>(kr + lane + 32 * j), part);
    const float sc = warp_sum(part) * scale;
    const float nm = fmaxf(mx, sc);
    const float corr = expf(mx - nm);
    const float pr = expf(sc - nm);
    den = den * corr + pr;
    const KT* vr = Vp + (size_t)k * d;
#pragma unroll
    for (int j = 0; j < DPL; ++j) o[j] = fmaf(pr, ldf<KT>(vr + lane + 32 * j), o[j] * corr);
    mx = nm;
  }
}

template <typename ST, int DPL>
__global__ void __launch_bounds__(ATT_WARPS * 32) attention_simt_kernel(FFBuffers buf, FFDims dm, int band_bits) {
  ff_pdl_wait();
  const int band = blockIdx.z, bh = blockIdx.y;
  if (!(buf.alloc[bh] & band_bits & (1 << band))) return;
  const long long n = band == 0 ? dm.Nbar : (band == 1 ? dm.Nmid : dm.Nhigh);
  const long long p = (long long)blockIdx.x * ATT_WARPS + (threadIdx.x >> 5);
  if (p >= n) return;
  const int lane = threadIdx.x & 31;
  const int d = dm.d;
  const float scale = rsqrtf((float)d);
  float q[DPL], o[DPL];
  float mx = -INFINITY, den = 0.f;
#pragma unroll
  for (int j = 0; j < DPL; ++j) o[j] = 0.f;
  const size_t BHn = (size_t)dm.BH * n * d;   // one tensor's extent in this band's buffer
  if (band == 0) {
    const float* Qp = buf.pooled + (size_t)bh * n * d;
    const float* Kp = Qp + BHn;
    const float* Vp = Kp + BHn;
#pragma unroll
    for (int j = 0; j < DPL; ++j) q[j] = Qp[(size_t)p * d + lane + 32 * j];
    attend_range<float, DPL>(Kp, Vp, 0, n, d, q, scale, mx, den, o, lane);
    float* y = buf.y_low + ((size_t)bh * n + p) * d;
#pragma unroll
    for (int j = 0; j < DPL; ++j) y[lane + 32 * j] = o[j] / den;
  } else {
    const ST* Qp = (const ST*)(band == 1 ? buf.spec_mid : buf.spec_high) + (size_t)bh * n * d;
    const ST* Kp = Qp + BHn;
    const ST* Vp = Kp + BHn;
#pragma unroll
    for (int j = 0; j < DPL; ++j) q[j] = ldf<ST>(Qp + (size_t)p * d + lane + 32 * j);
    if (band == 1 && dm.pattern == FF_MID_ANCHOR) {
      // own block and every anchor block (block index = s-1 mod s)
      const long long J = p / dm.b;
      for (long long Jk = 0; Jk < dm.nb; ++Jk) {
        if (Jk != J && Jk % dm.s != dm.s - 1) continue;
        const long long k0 = Jk * dm.b;
        const long long k1 = (k0 + dm.b < n) ? k0 + dm.b : n;
        attend_range<ST, DPL>(Kp, Vp, k0, k1, d, q, scale, mx, den, o, lane);
      }
    } else if (band == 1) {
      const long long J = p / dm.b;
      for (long long Jk = J % dm.s; Jk < dm.nb; Jk += dm.s) {
        const long long k0 = Jk * dm.b;
        const long long k1 = (k0 + dm.b < n) ? k0 + dm.b : n;
        attend_range<ST, DPL>(Kp, Vp, k0, k1, d, q, scale, mx, den, o, lane);
      }
    } else {
      const long long k0 = (p - dm.R > 0) ? p - dm.R : 0;
      const long long k1 = (p + dm.R + 1 < n) ? p + dm.R + 1 : n;
      attend_range<ST, DPL>(Kp, Vp, k0, k1, d, q, scale, mx, den, o, lane);
    }
    ST* y = (ST*)(band == 1 ? buf.y_mid : buf.y_high) + ((size_t)bh * n + p) * d;
#pragma unroll
    for (int j = 0; j < DPL; ++j) stf<ST>(y + lane + 32 * j, o[j] / den);
  }
}

// Exchange + recombination ("Cross-band residual exchange", "Reconstruction"): for every
// coefficient of the grid, fetch its band token, add softmax(y Z^T / sqrt(d)) Z over the 2m summary
// tokens of the other two bands, and write the row at its coefficient position (fp32 grid).
constexpr int EXC_WARPS = 8;

// Coefficients per warp: up to 8, fewer when the launch would otherwise have too few blocks.
static int exc_rounds(long long tokens, int g, int sm_count) {
  long long r = tokens * g / ((long long)EXC_WARPS * 8 * sm_count);
  return r < 1 ? 1 : (r > 8 ? 8 : (int)r);
}

template <typename ST, int DPL, typename OT>
__global__ void __launch_bounds__(EXC_WARPS * 32) exchange_recombine_kernel(FFBuffers buf, FFDims dm, int bh0,
                                                                             OT* grid_out, void* grid_lo, int low_only, int rounds) {
  ff_pdl_wait();
  extern __shared__ float S[];   // [3][m][d]
  const int gi = blockIdx.y, bh = bh0 + gi;
  const int d = dm.d, m = dm.m;
  for (int i = threadIdx.x; i < 3 * m * d; i += blockDim.x) S[i] = buf.summary[(size_t)bh * 3 * m * d + i];
  __syncthreads();
  // low_only: the launch covers the low band's coefficients only (the other bands are exchanged
  // by the tensor-core kernel); the index is then a low rank, unravelled inside the low box.
  const int lane = threadIdx.x & 31;
  // a block stages the summaries once and then works through rounds x EXC_WARPS coefficients
  for (int round = 0; round < rounds; ++round) {
  long long f = ((long long)blockIdx.x * rounds + round) * EXC_WARPS + (threadIdx.x >> 5);
  if (f >= (low_only ? dm.Nlow : dm.N)) return;
  int kw, kh, kt;
  if (low_only) {
    kw = (int)(f % dm.L[2]); kh = (int)((f / dm.L[2]) % dm.L[1]); kt = (int)(f / ((long long)dm.L[2] * dm.L[1]));
    f = ((long long)kt * dm.H + kh) * dm.W + kw;
  } else {
    kw = (int)(f % dm.W); kh = (int)((f / dm.W) % dm.H); kt = (int)(f / ((long long)dm.W * dm.H));
  }
  long long rank;
  const int band = ff_band_rank_of(dm, kt, kh, kw, &rank);
  const BandView<ST> v = band_view<ST>(buf, dm, bh, band);
  const long long row = v.compressed ? rank / dm.r : rank;
  float y[DPL], acc[DPL];
#pragma unroll
  for (int j = 0; j < DPL; ++j) {
    y[j] = v.f32 ? v.f32[(size_t)row * d + lane + 32 * j] : ldf<ST>(v.st + (size_t)row * d + lane + 32 * j);
    acc[j] = 0.f;
  }
  if (m > 0) {
    const float scale = rsqrtf((float)d);
    float mx = -INFINITY, den = 0.f;
    for (int ob = 0; ob < 3; ++ob) {
      if (ob == band || (ob == 1 && dm.Nmid == 0)) continue;     // own band; an empty mid band has no summaries
      for (int j2 = 0; j2 < m; ++j2) {
        const float* z = S + ((size_t)ob * m + j2) * d;
        float part = 0.f;
#pragma unroll
        for (int j = 0; j < DPL; ++j) part = fmaf(y[j], z[lane + 32 * j], part);
        const float sc = warp_sum(part) * scale;
        const float nm = fmaxf(mx, sc);
        const float corr = expf(mx - nm), pr = expf(sc - nm);
        den = den * corr + pr;
#pragma unroll
        for (int j = 0; j < DPL; ++j) acc[j] = fmaf(pr, z[lane + 32 * j], acc[j] * corr);
        mx = nm;
      }
    }
#pragma unroll
    for (int j = 0; j < DPL; ++j) acc[j] /= den;
  }
  // With a second grid (bf16 output) the value is stored in three bytes, rounded to 24 bits: its upper 16 bits
  // in grid_out, the next 8 bits in the byte grid.  A band's tokens share almost the same exchange offset, so a
  // single bf16 rounding would bias whole bands coherently and the inverse transform would focus that bias on a
  // few tokens.
  OT* dst = grid_out + ((size_t)gi * dm.N + f) * d;
#pragma unroll
  for (int j = 0; j < DPL; ++j) {
    const float v = y[j] + acc[j];
    if (grid_lo) {
      const uint32_t u = __float_as_uint(v) + 0x80u;
      ((uint16_t*)dst)[lane + 32 * j] = (uint16_t)(u >> 16);
      ((uint8_t*)grid_lo)[((size_t)gi * dm.N + f) * d + lane + 32 * j] = (uint8_t)(u >> 8);
    } else {
      stf<OT>(dst + lane + 32 * j, v);
    }
  }
  }
}

}  // namespace

// ================================================================================================
// Launchers
// ================================================================================================
template <typename ST>
static cudaError_t forward_transform_t(ff_plan* p, const void* Q, const void* K, const void* V, bool want_energy, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int total = 3 * dm.BH, G = p->lay.group;
  DctPassParams P{};
  P.BH = dm.BH; P.N_d = dm.N * dm.d; P.dm = dm;
  P.spec_low = p->buf.spec_low; P.spec_mid = p->buf.spec_mid; P.spec_high = p->buf.spec_high;
  for (int g0 = 0; g0 < total; g0 += G) {
    const int g = (total - g0 < G) ? total - g0 : G;
    P.group_start = g0;
    // w axis: lines of W elements with stride d
    P.src[0] = Q; P.src[1] = K; P.src[2] = V; P.dst = p->buf.scratchA; P.mat = p->basis[2];
    P.n = dm.W; P.inner = dm.d; P.outer = dm.T * dm.H;
    P.clear = want_energy && g0 == 0 ? p->buf.energy : nullptr;
    cudaError_t e = launch_dct_pass<ST, 0>(P, g, st);
    if (e != cudaSuccess) return e;
    // h axis
    P.src[0] = p->buf.scratchA; P.dst = p->buf.scratchB; P.mat = p->basis[1];
    P.n = dm.H; P.inner = dm.W * dm.d; P.outer = dm.T;
    e = launch_dct_pass<ST, 1>(P, g, st);
    if (e != cudaSuccess) return e;
    // t axis + band split
    P.src[0] = p->buf.scratchB; P.dst = nullptr; P.mat = p->basis[0];
    P.n = dm.T; P.inner = dm.H * dm.W * dm.d; P.outer = 1;
    e = launch_dct_pass<ST, 2>(P, g, st);
    if (e != cudaSuccess) return e;
    p->launches += 3;
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
  long long nmax = 0;
  if ((band_bits & FF_BAND_LOW) && dm.Nbar > nmax) nmax = dm.Nbar;
  if ((band_bits & FF_BAND_MID) && dm.Nmid > nmax) nmax = dm.Nmid;
  if ((band_bits & FF_BAND_HIGH) && dm.Nhigh > nmax) nmax = dm.Nhigh;
  if (nmax == 0) return cudaSuccess;                 // (only an empty band was asked for)
  const int zdim = (band_bits & FF_BAND_HIGH) ? 3 : ((band_bits & FF_BAND_MID) ? 2 : 1);
  dim3 grid((unsigned)((nmax + ATT_WARPS - 1) / ATT_WARPS), (unsigned)dm.BH, zdim);
  p->launches += 1;
  switch (dm.d / 32) {
    case 1: return ff_launch(attention_simt_kernel<ST, 1>, grid, dim3(ATT_WARPS * 32), 0, st, p->buf, dm, band_bits);
    case 2: return ff_launch(attention_simt_kernel<ST, 2>, grid, dim3(ATT_WARPS * 32), 0, st, p->buf, dm, band_bits);
    case 3: return ff_launch(attention_simt_kernel<ST, 3>, grid, dim3(ATT_WARPS * 32), 0, st, p->buf, dm, band_bits);
    default: return ff_launch(attention_simt_kernel<ST, 4>, grid, dim3(ATT_WARPS * 32), 0, st, p->buf, dm, band_bits);
  }
}

cudaError_t ffk_attention_simt(ff_plan* p, int band_bits, cudaStream_t st) {
  return p->dm.fp32 ? attention_simt_t<float>(p, band_bits, st) : attention_simt_t<__nv_bfloat16>(p, band_bits, st);
}

// Generic exchange + recombination into the hi/lo bf16 grids of the tensor-core inverse; DPL = d / 32.
template <int DPL>
static cudaError_t exchange_to_grids(ff_plan* p, long long tokens, int g, size_t smem, int h0, __nv_bfloat16* ghi,
                                     __nv_bfloat16* glo, int low_only, cudaStream_t st) {
  const int rounds = exc_rounds(tokens, g, p->sm_count);
  const long long per_block = (long long)EXC_WARPS * rounds;
  dim3 grid((unsigned)((tokens + per_block - 1) / per_block), (unsigned)g);
  p->launches += 1;
  return ff_launch(exchange_recombine_kernel<__nv_bfloat16, DPL, __nv_bfloat16>, grid, dim3(EXC_WARPS * 32), smem, st, p->buf, p->dm,
                   h0, ghi, (void*)glo, low_only, rounds);
}

// Tensor-core inverse: exchange + recombination into a bf16 grid, then the three axis passes.
static cudaError_t exchange_inverse_tc(ff_plan* p, void* out, cudaStream_t st) {
  const FFDims& dm = p->dm;
  const int G = p->dct_group;
  const size_t smem = (size_t)3 * dm.m * dm.d * sizeof(float);
  cudaError_t e = cudaSuccess;
  for (int h0 = 0; h0 < dm.BH; h0 += G) {
    const int g = (dm.BH - h0 < G) ? dm.BH - h0 : G;
    const size_t grid_bytes = ((size_t)G * dm.N * dm.d * 2 + 255) / 256 * 256;
    __nv_bfloat16* ghi = (__nv_bfloat16*)p->buf.scratchA;
    __nv_bfloat16* glo = (__nv_bfloat16*)((char*)p->buf.scratchA + grid_bytes);
    if (p->xtc_ok) {
      // mid and high bands on the tensor cores, the fp32 low band with its own kernel (one warp per source row)
      e = ffk_exchange_low(p, h0, g, ghi, glo, st);
      if (e == cudaSuccess) e = ffk_exchange_tc(p, h0, g, ghi, glo, st);
    } else {
      e = dm.d == 128 ? exchange_to_grids<4>(p, dm.N, g, smem, h0, ghi, glo, 0, st) : exchange_to_grids<2>(p, dm.N, g, smem, h0, ghi, glo, 0, st);
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
  const size_t smem = (size_t)3 * dm.m * dm.d * sizeof(float);
  for (int h0 = 0; h0 < dm.BH; h0 += G) {
    const int g = (dm.BH - h0 < G) ? dm.BH - h0 : G;
    const int rounds = exc_rounds(dm.N, g, p->sm_count);
    dim3 grid((unsigned)((dm.N + (long long)EXC_WARPS * rounds - 1) / ((long long)EXC_WARPS * rounds)), (unsigned)g);
    cudaError_t e = cudaSuccess;
#define FF_EXC(DPL)                                                                                                     \
  ff_launch(exchange_recombine_kernel<ST, DPL, float>, grid, dim3(EXC_WARPS * 32), smem, st, p->buf, dm, h0, p->buf.scratchA, \
            (void*)nullptr, 0, rounds)
    switch (dm.d / 32) {
      case 1: e = FF_EXC(1); break;
      case 2: e = FF_EXC(2); break;
      case 3: e = FF_EXC(3); break;
      default: e = FF_EXC(4); break;
    }
#undef FF_EXC
    if (e != cudaSuccess) return e;
    P.group_start = h0;
    // inverse along t, h, w with the transposed matrices
    P.src[0] = p->buf.scratchA; P.dst = p->buf.scratchB; P.mat = p->basis_t[0];
    P.n = dm.T; P.inner = dm.H * dm.W * dm.d; P.outer = 1;
    e = launch_dct_pass<ST, 1>(P, g, st);
    if (e != cudaSuccess) return e;
    P.src[0] = p->buf.scratchB; P.dst = p->buf.scratchA; P.mat = p->basis_t[1];
    P.n = dm.H; P.inner = dm.W * dm.d; P.outer = dm.T;
    e = launch_dct_pass<ST, 1>(P, g, st);
    if (e != cudaSuccess) return e;
    P.src[0] = p->buf.scratchA; P.dst = out; P.mat = p->basis_t[2];
    P.n = dm.W; P.inner = dm.d; P.outer = dm.T * dm.H;
    e = launch_dct_pass<ST, 3>(P, g, st);
    if (e != cudaSuccess) return e;
    p->launches += 4;
  }
  return cudaSuccess;
}

cudaError_t ffk_exchange_inverse(ff_plan* p, void* out, cudaStream_t st) {
  if (p->dct_tc_ok && !(p->attn_impl & 2)) return exchange_inverse_tc(p, out, st);
  return p->dm.fp32 ? exchange_inverse_t<float>(p, out, st) : exchange_inverse_t<__nv_bfloat16>(p, out, st);
}

cudaError_t ffk_simt_init() {
  cudaError_t e = cudaSuccess;
  const int most = 3 * 64 * 128 * (int)sizeof(float);       // summaries of a head; a transform tile and its matrix need no more
#define FF_SET(k) if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most)
#define FF_SET_T(T)                                                                                                    \
  FF_SET((dct_pass_kernel<T, 0>)); FF_SET((dct_pass_kernel<T, 1>)); FF_SET((dct_pass_kernel<T, 2>)); FF_SET((dct_pass_kernel<T, 3>)); \
  FF_SET((exchange_recombine_kernel<T, 1, float>)); FF_SET((exchange_recombine_kernel<T, 2, float>));                  \
  FF_SET((exchange_recombine_kernel<T, 3, float>)); FF_SET((exchange_recombine_kernel<T, 4, float>))
  FF_SET_T(float); FF_SET_T(__nv_bfloat16);
  FF_SET((exchange_recombine_kernel<__nv_bfloat16, 2, __nv_bfloat16>)); FF_SET((exchange_recombine_kernel<__nv_bfloat16, 4, __nv_bfloat16>));
#undef FF_SET_T
#undef FF_SET
  return e;
}
