// From the coefficients to the head-to-band allocation in one launch ("Low band: dense global attention on compressed
// tokens", "Spectral routing network"): r:1 pooling of the low band, the channel energies the transform's epilogue has
// not summed, the router MLP with its head quota, and the worklist of the attention launch.
//
// The router needs the energies of every block, so the block that finishes last (a ticket counter owned by the plan)
// runs it.  What these steps cost is latency, not work: as five launches (low-band energy, router, pooling, worklist
// and the fp32 path's energies) they took 53 us of a 16K-token layer, the router alone 29 us with its second layer
// read by three threads.  By clocks of the last block (six heads of 16K tokens, 27 000 cycles) the hidden layer took 9400, its
// weights read in rounds of eight inputs and then one by one, the second layer 2800, e(t) 2300 before the launch's wait, which
// nothing overlaps there: now the weights are asked for ahead, e(t) is made beside the energies.  The launch alone 14.6 -> 10.2 us,
// layers 188.5 -> 184.8 (four heads of 8K 118.5 -> 115.4, 256 fp32 tokens 29.6 -> 28.7).
#include "ff_bands.cuh"
#include "ff_internal.h"
#include "ff_worklist.cuh"

namespace {

constexpr int ST_THREADS = 512;
constexpr int ST_MASKS = 512;            // band masks kept in shared memory for the worklist
constexpr int ST_ROWS = 8;               // rows of a pooled token that a thread reads at a time
constexpr int ST_STEPS = 8;              // rows per thread of a mid / high block

struct StatsParams {
  FFDims dm;
  const float* spec_low; const void* spec_mid; const void* spec_high;
  float* pooled; __nv_bfloat16* pooled_bf;
  double* energy;                        // NULL: no statistics wanted (the caller gave the allocation)
  const float* W1; const float* b1; const float* W2; const float* b2;
  const float* timestep;                 // device, [B]; NULL: they are in ts
  float ts[FF_TS_INLINE];
  const uint8_t* alloc_in;               // the caller's masks, or NULL to route
  uint8_t* alloc; float* pi;
  int* work; int low_on;                 // attention worklist (NULL: the tensor-core kernel does not run)
  int mid_items;                         // items of one head's mid band in it
  unsigned* ticket;
  int n_low, n_mid;                      // blocks of the low and of the mid band (the rest: high band); 0: not covered
  int low_steps;                         // pooled tokens per thread of a low block
};

__device__ __forceinline__ void add_squares(float4& e, const float4& x) {
  e.x = fmaf(x.x, x.x, e.x); e.y = fmaf(x.y, x.y, e.y); e.z = fmaf(x.z, x.z, e.z); e.w = fmaf(x.w, x.w, e.w);
}

// Line `line` of 128 bytes of n floats into L2.
__device__ __forceinline__ void prefetch_line(const float* p, int line, int n) {
  if (line < (n + 31) / 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + line * 32));
}

// Sinusoidal embedding of the sample's timestep into et[dt], in double precision; by as many of the block's last warps as it takes.
__device__ void embed_timestep(const StatsParams& P, int sample, float* et) {
  const int half = P.dm.dt / 2, threads = half < ST_THREADS ? (half + 31) / 32 * 32 : ST_THREADS;
  for (int k = (int)threadIdx.x - (ST_THREADS - threads); k >= 0 && k < half; k += threads) {
    const double t = (double)(P.timestep ? P.timestep[sample] : P.ts[sample]);
    const double om = exp2(-(double)k / (double)half * 13.287712379549449);     // 10000^(-k/half); log2(10000)
    double sn, cs;
    sincos(t * om, &sn, &cs);
    et[k] = (float)sn;
    et[half + k] = (float)cs;
  }
}

// z = W2 relu(W1 [g; e(t)] + b1) + b2, pi = softmax(z), largest-remainder quota, one-hot masks; a whole block.  A chain of
// latencies: under way before the step that needs them are the weights of the first 224 inputs of the first 64 hidden units (all of
// them with head_dim 32 and an embedding of up to 128), those of the second layer's first 64, and e(t) on warps of its own.  The other
// weights are loaded eight inputs at a time, without a test where eight are left: in chunks of seven tested ones layers took, us,
// 256 fp32 tokens, 1024 hidden units 52.4 for 44.2, 512 with t_embed_dim 512 45.7 for 39.7, head_dim 128 with 256 38.8 for 38.4.
constexpr int ST_AHEAD = 7;              // inputs of a hidden unit that a lane holds weights of (28 registers of 64)
__device__ void route_sample(const StatsParams& P, int sample, bool embedded, float* sm, uint8_t* masks) {
  const FFDims& dm = P.dm;
  const int d = dm.d, nin = 3 * d + dm.dt, hid = dm.hid;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* x = sm;            // [nin]
  float* h = sm + nin;      // [hid]
  __shared__ float z[3];
  __shared__ int first[4];  // first head of each band
  // hidden layer: four units per warp at a time, lanes stride over the inputs (coalesced rows of W1)
  float w[4][ST_AHEAD];
#pragma unroll
  for (int t = 0; t < ST_AHEAD; ++t)
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k][t] = 32 * t + lane < nin && warp * 4 + k < hid ? P.W1[(size_t)(warp * 4 + k) * nin + 32 * t + lane] : 0.f;
  const float w2 = warp < 3 && lane < hid ? P.W2[warp * hid + lane] : 0.f, w2b = warp < 3 && lane + 32 < hid ? P.W2[warp * hid + lane + 32] : 0.f;
  const float bias2 = warp < 3 ? P.b2[warp] : 0.f;
  float bias1 = lane < 4 && warp * 4 + lane < hid ? P.b1[warp * 4 + lane] : 0.f;
  if (!embedded) embed_timestep(P, sample, x + 3 * d);
  for (int i = tid; i < 3 * d; i += ST_THREADS) {
    const int band = i / d;
    const long long cnt = band == 0 ? dm.Nlow : (band == 1 ? dm.Nmid : dm.Nhigh);
    const double terms = 3.0 * dm.heads * (double)(cnt > 0 ? cnt : 1);          // an empty band (two-band layer) has g = 0
    x[i] = (float)log1p(__ldcg(P.energy + (size_t)sample * 3 * d + i) / terms);
  }
  __syncthreads();
  // (the first units' inputs so far; from there on as many loads at a time as fit)
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int t = 0; t < ST_AHEAD; ++t) {
    const float v = 32 * t + lane < nin ? x[32 * t + lane] : 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = fmaf(w[k][t], v, acc[k]);
  }
  int i0 = 32 * ST_AHEAD;
  for (int j0 = warp * 4; j0 < hid; j0 += (ST_THREADS / 32) * 4) {
    const float* row = P.W1 + (size_t)j0 * nin + lane;
    const int o1 = j0 + 1 < hid ? nin : 0, o2 = j0 + 2 < hid ? 2 * nin : 0, o3 = j0 + 3 < hid ? 3 * nin : 0;
    auto add = [&](int i, bool on) {
      const float v = on ? x[i + lane] : 0.f;
      acc[0] = fmaf(on ? row[i] : 0.f, v, acc[0]); acc[1] = fmaf(on ? row[i + o1] : 0.f, v, acc[1]);
      acc[2] = fmaf(on ? row[i + o2] : 0.f, v, acc[2]); acc[3] = fmaf(on ? row[i + o3] : 0.f, v, acc[3]);
    };
    for (; i0 + 32 * 8 <= nin; i0 += 32 * 8)
#pragma unroll
      for (int t = 0; t < 8; ++t) add(i0 + 32 * t, true);
    if (i0 < nin)
#pragma unroll
      for (int t = 0; t < 8; ++t) add(i0 + 32 * t, i0 + 32 * t + lane < nin);
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = warp_sum(acc[k]);
    if (lane < 4 && j0 + lane < hid) {
      const float v = lane == 0 ? acc[0] : (lane == 1 ? acc[1] : (lane == 2 ? acc[2] : acc[3]));
      if (j0 != warp * 4) bias1 = P.b1[j0 + lane];
      h[j0 + lane] = fmaxf(v + bias1, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = 0.f;
    i0 = 0;
  }
  __syncthreads();
  if (warp < 3) {
    float acc = lane < hid ? w2 * h[lane] : 0.f;
    if (lane + 32 < hid) acc = fmaf(w2b, h[lane + 32], acc);
    for (int j = lane + 64; j < hid; j += 32) acc = fmaf(P.W2[warp * hid + j], h[j], acc);
    acc = warp_sum(acc);
    if (lane == 0) z[warp] = acc + bias2;
  }
  __syncthreads();
  if (tid == 0) {
    const float mx = fmaxf(z[0], fmaxf(z[1], z[2]));
    float e[3], frac[3], sum = 0.f;
    int base[3], total = 0;
    for (int l = 0; l < 3; ++l) { e[l] = expf(z[l] - mx); sum += e[l]; }
    for (int l = 0; l < 3; ++l) {
      const float p = e[l] / sum, q = p * (float)dm.heads;
      P.pi[sample * 3 + l] = p;
      base[l] = (int)floorf(q);
      frac[l] = q - floorf(q);
      total += base[l];
    }
    for (int left = dm.heads - total; left > 0; --left) {   // leftover heads: largest fraction, ties to the lower band
      int best = 0;
      for (int l = 1; l < 3; ++l) if (frac[l] > frac[best]) best = l;
      base[best] += 1;
      frac[best] = -1.f;
    }
    first[0] = 0; first[1] = base[0]; first[2] = base[0] + base[1]; first[3] = 0;
  }
  __syncthreads();
  for (int hix = tid; hix < dm.heads; hix += ST_THREADS) {
    const uint8_t mask = hix < first[1] ? FF_BAND_LOW : (hix < first[2] ? FF_BAND_MID : FF_BAND_HIGH);
    P.alloc[sample * dm.heads + hix] = mask;
    if (sample * dm.heads + hix < ST_MASKS) masks[sample * dm.heads + hix] = mask;
  }
  __syncthreads();                                          // (the next sample reuses the shared memory; the worklist reads the masks)
}

template <typename ST>
__global__ void __launch_bounds__(ST_THREADS, 2) band_stats_kernel(const __grid_constant__ StatsParams P) {
  extern __shared__ float sm[];
  __shared__ bool last;
  __shared__ uint8_t masks[ST_MASKS];
  const FFDims& dm = P.dm;
  // (any block may turn out to be the one that routes; the sums below use other shared memory)
  float* mlp = sm + (ST_THREADS / (dm.d / 4)) * dm.d;
  // (an embedding that takes more than half of the threads is not overlapped with the energies: 1024, 33.1 us a layer, here 32.3)
  const bool early = !P.timestep && dm.dt > ST_THREADS;
  if (!P.alloc_in) {
    // A transform that has gone through L2 leaves none of the router's weights there: the first blocks ask for them while
    // the sums are made.
    const int line = (int)(blockIdx.y * gridDim.x + blockIdx.x) * ST_THREADS + (int)threadIdx.x;
    prefetch_line(P.W1, line, dm.hid * (3 * dm.d + dm.dt));
    prefetch_line(P.W2, line, 3 * dm.hid);
    prefetch_line(P.b1, line, dm.hid);
    prefetch_line(P.b2, line, 3);
    if (early) embed_timestep(P, 0, mlp + 3 * dm.d);
  }
  // (a router keeps one block busy long after the others: let in early, the next launch's blocks settle unevenly meanwhile.
  // With masks given there is little to wait for: 4 x 19 x 16 fp32 tokens, six heads, all bands, 55.6 us, let in late 61.1)
  if (P.alloc_in) ff_pdl_wait(); else ff_pdl_join();
  const int d = dm.d, vecs = d / 4;                         // four channels per thread
  const int vec = threadIdx.x % vecs, sub = threadIdx.x / vecs, nsub = ST_THREADS / vecs;
  const int th = blockIdx.y;
  float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
  int band = 0;
  if ((int)blockIdx.x < P.n_low) {
    if (sub < nsub)
      for (int k = 0; k < P.low_steps; ++k) {
        const long long g = ((long long)blockIdx.x * P.low_steps + k) * nsub + sub;
        if (g >= dm.Nbar) break;
        const long long p0 = g * dm.r, p1 = p0 + dm.r < dm.Nlow ? p0 + dm.r : dm.Nlow;
        const float* src = P.spec_low + ((size_t)th * dm.Nlow + p0) * d + vec * 4;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        const int n = (int)(p1 - p0);
        for (int i0 = 0; i0 < n; i0 += ST_ROWS) {
          float4 x[ST_ROWS];
#pragma unroll
          for (int i = 0; i < ST_ROWS; ++i) x[i] = i0 + i < n ? ld4(src + (size_t)(i0 + i) * d) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int i = 0; i < ST_ROWS; ++i) {
            acc.x += x[i].x; acc.y += x[i].y; acc.z += x[i].z; acc.w += x[i].w;
            add_squares(e, x[i]);
          }
        }
        const float fn = (float)n;
        acc = make_float4(acc.x / fn, acc.y / fn, acc.z / fn, acc.w / fn);
        const size_t o = ((size_t)th * dm.Nbar + g) * d + vec * 4;
        *(float4*)(P.pooled + o) = acc;
        if (P.pooled_bf) {
          __nv_bfloat162 a = __floats2bfloat162_rn(acc.x, acc.y), b = __floats2bfloat162_rn(acc.z, acc.w);
          *(uint2*)(P.pooled_bf + o) = make_uint2(*(uint32_t*)&a, *(uint32_t*)&b);
        }
      }
  } else {
    const int bx = (int)blockIdx.x - P.n_low;
    band = bx < P.n_mid ? 1 : 2;
    const long long nl = band == 1 ? dm.Nmid : dm.Nhigh;
    const long long r0 = (long long)(band == 1 ? bx : bx - P.n_mid) * nsub * ST_STEPS + sub;
    const ST* src = (const ST*)(band == 1 ? P.spec_mid : P.spec_high) + (size_t)th * nl * d + vec * 4;
    if (sub < nsub)
#pragma unroll
      for (int k = 0; k < ST_STEPS; ++k)
        if (r0 + k * nsub < nl) add_squares(e, ld4(src + (size_t)(r0 + k * nsub) * d));
  }
  if (P.energy) {
    if (sub < nsub) *(float4*)(sm + sub * d + vec * 4) = e;
    __syncthreads();
    if ((int)threadIdx.x < d) {
      double s = 0.0;
      for (int i = 0; i < nsub; ++i) s += (double)sm[i * d + threadIdx.x];
      atomicAdd(P.energy + ((size_t)((th % dm.BH) / dm.heads) * 3 + band) * d + threadIdx.x, s);
    }
  }
  if (P.alloc_in) {                                          // nothing to wait for: one block copies the masks and lists the work
    if (blockIdx.x == 0 && blockIdx.y == 0) {
      for (int i = threadIdx.x; i < dm.BH; i += ST_THREADS) P.alloc[i] = P.alloc_in[i];
      __syncthreads();
      if (P.work && threadIdx.x < 32) build_worklist(dm, P.alloc, P.low_on, P.mid_items, P.work);
    }
    return;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(P.ticket, 1u) == gridDim.x * gridDim.y - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) *P.ticket = 0;
  for (int sample = 0; sample < dm.B; ++sample) {
    route_sample(P, sample, early && sample == 0, mlp, masks);
  }
  if (P.work && threadIdx.x < 32) build_worklist(dm, dm.BH <= ST_MASKS ? masks : P.alloc, P.low_on, P.mid_items, P.work);
}

// More timesteps than fit the statistics' arguments, in launches of their own: a copy from the caller's memory would be
// read again when a captured call is replayed.
struct TimestepChunk { float v[256]; };
__global__ void set_timesteps_kernel(const __grid_constant__ TimestepChunk c, float* dst, int n) {
  ff_pdl_wait();
  if ((int)threadIdx.x < n) dst[threadIdx.x] = c.v[threadIdx.x];
}

// Shared memory of a block: a row of channels per thread group for the sums, and the router's input and hidden layer.
size_t sums_bytes(const FFDims& dm) { return (size_t)(ST_THREADS / (dm.d / 4)) * dm.d * sizeof(float); }
size_t router_bytes(const FFDims& dm) { return (size_t)(3 * dm.d + dm.dt + dm.hid) * sizeof(float); }

}  // namespace

// (routers up to what a block can have; a wider one fails where it is used, with the launch's error.  The 48 KB of a launch that asked
// for nothing hold the kernel's static arrays, too: 544 bytes.  The most and not this plan's need: the attribute is the kernel's, and
// a plan made later must not take it back from an earlier, wider one.)
cudaError_t ffk_stats_init(const FFDims& dm) {
  constexpr size_t most = 226 * 1024, beside = 1024;       // (of 227 KB)
  if (sums_bytes(dm) + router_bytes(dm) + beside <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(dm.fp32 ? band_stats_kernel<float> : band_stats_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)most);
}

cudaError_t ffk_set_timesteps(ff_plan* p, const float* host, cudaStream_t st) {
  for (int b0 = 0; b0 < p->dm.B; b0 += 256) {
    TimestepChunk c;
    const int n = p->dm.B - b0 < 256 ? p->dm.B - b0 : 256;
    memcpy(c.v, host + b0, n * sizeof(float));
    p->launches += 1;
    const cudaError_t e = ff_launch(set_timesteps_kernel, dim3(1), dim3(256), 0, st, c, p->buf.timestep + b0, n);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Pooling, statistics, router or copy of the caller's masks, worklist.  `bands_summed`: the transform's epilogue has
// summed the energies of the mid and high bands already.
cudaError_t ffk_band_stats(ff_plan* p, const uint8_t* alloc_in, const float* timestep_host, bool bands_summed, cudaStream_t st) {
  const FFDims& dm = p->dm;
  StatsParams P{};
  P.dm = dm;
  P.spec_low = p->buf.spec_low; P.spec_mid = p->buf.spec_mid; P.spec_high = p->buf.spec_high;
  P.pooled = p->buf.pooled; P.pooled_bf = p->low_tc_ok ? p->buf.pooled_bf : nullptr;
  P.alloc_in = alloc_in; P.alloc = p->buf.alloc; P.pi = p->buf.pi;
  P.ticket = p->tickets;
  const bool tc = p->tc_ok && !(p->attn_impl & 1);
  P.work = tc ? p->buf.work : nullptr; P.low_on = p->low_tc_ok ? 1 : 0;
  P.mid_items = mid_shape(dm).items;
  if (!alloc_in) {
    P.energy = p->buf.energy;
    P.W1 = p->W1; P.b1 = p->b1; P.W2 = p->W2; P.b2 = p->b2;
    if (dm.B <= FF_TS_INLINE) for (int i = 0; i < dm.B; ++i) P.ts[i] = timestep_host[i];
    else P.timestep = p->buf.timestep;
  }
  const int nsub = ST_THREADS / (dm.d / 4);
  // a low block takes one round of pooled tokens while the launch stays below three blocks per SM, then up to 16 (a
  // block ends with one atomic per channel, all blocks on the same addresses: 64K tokens, head_dim 64, 98,304 pooled
  // tokens, 48 us at eight blocks per SM, 41 us at three)
  long long steps = dm.Nbar * 3 * dm.BH / ((long long)nsub * 3 * p->sm_count);
  P.low_steps = (int)(steps < 1 ? 1 : (steps > 16 ? 16 : steps));
  P.n_low = (int)((dm.Nbar + (long long)nsub * P.low_steps - 1) / ((long long)nsub * P.low_steps));
  long long blocks = P.n_low;
  if (!alloc_in && !bands_summed) {
    P.n_mid = (int)((dm.Nmid + nsub * ST_STEPS - 1) / (nsub * ST_STEPS));
    blocks += P.n_mid + (dm.Nhigh + nsub * ST_STEPS - 1) / (nsub * ST_STEPS);
  }
  p->launches += 1;
  return ff_launch(dm.fp32 ? band_stats_kernel<float> : band_stats_kernel<__nv_bfloat16>, dim3((unsigned)blocks, (unsigned)(3 * dm.BH)),
                   dim3(ST_THREADS), sums_bytes(dm) + (alloc_in ? 0 : router_bytes(dm)), st, P);
}
