// Internal declarations shared by the host API and the kernel translation units.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <utility>

#include "ff_tensor_map.h"
#include "freqformer.h"

#if defined(__CUDACC__)
#define FF_HD __host__ __device__ __forceinline__
#else
#define FF_HD inline
#endif

// Debug build (-DFF_DEBUG): every computed band rank, row offset and tile coordinate is range-checked on
// the device before it is used; a value out of range is not used for the access (the store or copy is
// skipped) and FF_ERR_INVALID_ARG together with the kernel's id is raised in the plan's status word, where
// ff_plan_device_status reports it.  The release build compiles the checks away.
#if defined(FF_DEBUG) && defined(__CUDACC__)
#define FF_DBG_OK(cond, status_ptr, kernel_id) \
  ((cond) ? true : (atomicExch((status_ptr), FF_ERR_INVALID_ARG | ((kernel_id) << 8)), false))
#else
#define FF_DBG_OK(cond, status_ptr, kernel_id) (true)
#endif

// Problem sizes derived from ff_config_t ("Frequency band partitioning": N_low + N_mid + N_high = N).
struct FFDims {
  int B, T, H, W, heads, d, BH;
  int L[3], M[3];
  int r, b, s, R, m, hid, dt;
  int fp32;              // storage type of Q,K,V,out and of the mid/high band buffers
  int pattern;           // mid-band sparse pattern: FF_MID_STRIDED or FF_MID_ANCHOR
  long long N, Nlow, Nbar, Nmid, Nhigh;
  long long nb;          // number of mid blocks
};

// Number of members of the box A = [0,A_t) x [0,A_h) x [0,A_w) whose flat index is below that of k.
FF_HD long long ff_box_count_below(int At, int Ah, int Aw, int kt, int kh, int kw) {
  long long c = (long long)(kt < At ? kt : At) * Ah * Aw;
  if (kt < At) {
    c += (long long)(kh < Ah ? kh : Ah) * Aw;
    if (kh < Ah) c += (kw < Aw ? kw : Aw);
  }
  return c;
}

// Band (0 low, 1 mid, 2 high) and band-local rank of coefficient (kt,kh,kw): nested boxes, band
// order = increasing flat index.
FF_HD int ff_band_rank_of(const FFDims& dm, int kt, int kh, int kw, long long* rank) {
  const long long cl = ff_box_count_below(dm.L[0], dm.L[1], dm.L[2], kt, kh, kw);
  const long long cm = ff_box_count_below(dm.M[0], dm.M[1], dm.M[2], kt, kh, kw);
  const bool in_low = kt < dm.L[0] && kh < dm.L[1] && kw < dm.L[2];
  const bool in_mid = kt < dm.M[0] && kh < dm.M[1] && kw < dm.M[2];
  if (in_low) { *rank = cl; return 0; }
  if (in_mid) { *rank = cm - cl; return 1; }
  *rank = ((long long)kt * dm.H + kh) * dm.W + kw - cm;
  return 2;
}

// Division of a 31-bit number by a number fixed on the host, as a multiply-high, an add and a shift (Granlund and
// Montgomery, "Division by Invariant Integers using Multiplication", 1994).
struct FFFastDiv { unsigned d, m, s; };
inline FFFastDiv ff_fast_div(unsigned d) {
  FFFastDiv f;
  f.d = d; f.s = 0;
  while ((1ull << f.s) < d) ++f.s;
  f.m = (unsigned)(((((1ull << f.s) - d) << 32) / d) + 1);
  return f;
}
#if defined(__CUDACC__)
// Programmatic dependent launch.  Every kernel of the path is launched with the attribute, does what does not
// depend on earlier kernels (barriers, tensor memory, matrices of the plan), then waits until the kernel
// before it in the stream has finished and its writes are visible.  It reads or writes nothing another kernel
// touches before the wait.  Here it then lets the next kernel start its own prologue.
__device__ __forceinline__ void ff_pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The two halves on their own.  The exchange of the mid and high bands starts with the trigger and ends with the join: it
// does not depend on the launch before it, the low band's exchange, but on the ones before that, and whoever waits for it
// has waited for both.  That holds only while the launch before it triggers behind its own wait, or not at all.
//
// A kernel with the join alone lets the next one in when its own blocks have ended.  The one-axis passes of the grids with
// 16, 32, 64 or 128 positions an axis and the statistics, both in a routed call, the inverse launch with t in registers and the
// attention do: what follows them has little to do ahead of its wait, and let in early it cost more than the start-up it hid (layers, us,
// with the trigger behind the wait / without: six heads of 16K tokens 214.2 / 203.1, 24 of 64K 2815 / 2770, 16 of 64K with
// head_dim 64 1010 / 990, fp32 7 x 16 x 12, six heads, 111 / 100).  The summaries keep it (16K tokens: 211, without 218), the
// two-axis launch too (203, 206).  With masks given there is no router to wait for, and the passes let the next launch in behind
// their wait (all bands, when their blocks end / behind the wait: six heads of 16 x 16 x 16 110.7 / 106.9, four of 16 x 16 x 32
// 130.1 / 127.2, of 16 x 32 x 32 with head_dim 64 135.1 / 131.6, six of 64 x 16 x 64 901 / 889, of 16 x 32 x 32 228.0 / 229.7,
// four of 64 x 64 x 64 3368 / 3358; routed calls lose by it: six of 16 x 32 x 32 217 / 224, of 64 x 16 x 64 681 / 695).
__device__ __forceinline__ void ff_pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void ff_pdl_join() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// (an event wait in the stream before the launch, the library's own or the caller's, holds the whole kernel back)
template <class... K, class... A>
inline cudaError_t ff_launch(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

__device__ __forceinline__ unsigned ff_div(unsigned n, const FFFastDiv& f) { return (__umulhi(f.m, n) + n) >> f.s; }
#endif

// One axis of a tensor-core transform pass as a grid [outer][n][inner] of positions.  A tile is kf whole lines:
// neighbours along `inner` (t and h axes: row = a * kf + line) or, where inner is 1 (w axis), along `outer`
// (row = line * n + a).
struct FFPassShape {
  int n, kf, rows;          // axis length, lines per tile, rows in use (kf * n <= 128)
  int inner, outer;
  int seq;                  // w axis
  int tiles_inner;          // tiles along `inner` (1 for the w axis)
  int tiles;                // tiles of one tensor-head
};
inline FFPassShape ff_pass_shape(const FFDims& dm, int axis) {
  FFPassShape g;
  g.n = axis == 2 ? dm.W : (axis == 1 ? dm.H : dm.T);
  g.inner = axis == 2 ? 1 : (axis == 1 ? dm.W : dm.H * dm.W);
  g.outer = axis == 2 ? dm.T * dm.H : (axis == 1 ? dm.T : 1);
  g.seq = axis == 2;
  const int lines = g.seq ? g.outer : g.inner;
  g.kf = 128 / g.n < lines ? 128 / g.n : lines;
  g.rows = g.kf * g.n;
  g.tiles_inner = g.seq ? 1 : (g.inner + g.kf - 1) / g.kf;
  g.tiles = g.seq ? (g.outer + g.kf - 1) / g.kf : g.outer * g.tiles_inner;
  return g;
}
// Axes that divide a tile of 128 rows into boxes of whole lines.  With any other axis the values between the passes of
// the tensor-core transform are fp32 numbers, and its operands three bf16 parts (ff_dct_tc.cu).
FF_HD bool ff_tile_axis(int n) { return n == 16 || n == 32 || n == 64 || n == 128; }
FF_HD bool ff_fp32_grid(const FFDims& dm) { return !(ff_tile_axis(dm.T) && ff_tile_axis(dm.H) && ff_tile_axis(dm.W)); }

// Transform matrix of an axis as tensor-memory operand images: [3 parts][128 rows][64 cells of two bf16]; the first two
// parts are the bf16 pair, all three the fp32 value.
constexpr size_t FF_IMAGE_PART = (size_t)128 * 64, FF_IMAGE_CELLS = 3 * FF_IMAGE_PART;
constexpr int FF_IMAGES = 6;

// SMs for the rules that shape the workspace: its size is a function of the configuration alone (it is asked for without
// a device).  Rules that shape only a launch take the device's count.
constexpr int FF_B200_SMS = 148;

// Device buffers inside the caller's workspace.
struct FFBuffers {
  float* spec_low;   // [3][BH][Nlow][d]
  void* spec_mid;    // st [3][BH][Nmid][d]
  void* spec_high;   // st [3][BH][Nhigh][d]
  float* pooled;     // [3][BH][Nbar][d]
  __nv_bfloat16* pooled_bf;  // the same values as bf16, operands of the tensor-core low branch (NULL if unused)
  float* y_low;      // [BH][Nbar][d]
  void* y_mid;       // st [BH][Nmid][d]
  void* y_high;      // st [BH][Nhigh][d]
  float* summary;    // [BH][3][m][d]
  uint8_t* zimg;     // [BH][hi, lo] summaries of a head as operand images of the tensor-core exchange
  float* sum_part;   // [BH][3][m][pieces][d] partial segment sums
  double* energy;    // [B][3][d]
  uint8_t* alloc;    // [BH]
  float* pi;         // [B][3]
  float* timestep;   // [B]
  int* status;       // device status word
  int* work;         // worklist of the tensor-core attention kernel
  float* scratchA;   // [G][N][d]
  float* scratchB;   // [G][N][d]
  void* stage_q;     // host-call staging (st [BH][N][d]) or NULL
  void* stage_k;
  void* stage_v;
  void* stage_out;
};

struct FFLayout {
  size_t off[24];
  size_t total;
  int group;         // G: tensor-heads processed per generic transform launch
  int tc_group;      // tensor-heads per tensor-core transform launch
  int tc_group_pipe; // ... when the launches are pipelined with host copies (host-buffer entry point)
};

constexpr int FF_COPY_EVENTS = 64;
constexpr int FF_TS_INLINE = 32;     // timesteps of up to this many samples travel as kernel arguments

struct ff_plan {
  ff_config_t cfg;
  FFDims dm;
  int device;
  // device tables owned by the plan
  float* basis[3];    // C_T, C_H, C_W  [n][n], C[k][i]
  float* basis_t[3];  // transposes
  float* W1; float* b1; float* W2; float* b2; float* U;
  bool has_router;
  int identity_u;     // no summary projections were given: U_l = I
  // workspace
  void* ws; size_t ws_bytes;
  FFBuffers buf;
  FFLayout lay;
  bool ws_has_staging;
  int attn_impl;
  int sm_count;
  bool tc_ok;                                  // tensor-core attention usable with this plan + workspace
  bool dct_tc_ok;                              // tensor-core transform usable
  int dct_group;                               // tensor-heads per tensor-core transform launch
  bool xtc_ok;                                 // tensor-core exchange usable
  unsigned* tickets;                           // "last block" counters, zero between launches (plan-owned)
  int* pos_table;                              // rank -> flat coefficient index of the mid, then the high band (plan-owned)
  alignas(64) unsigned char tmap_x[4][128];    // CUtensorMaps of the exchange kernel (Y / V~ of the mid and high bands)
  uint32_t* dct2_images;                       // transform matrices as tensor-memory operand images (plan-owned): three axes forward,
                                               // inverse; in unused parts the folded one of ff_dct_t16.cu
  FFMapCache maps;                             // tensor maps of the transform passes, by shape
  bool dct2_ok;                                // the fused two-axis launch covers this configuration
  int dct2_axis2;                              // its second axis (1 = h, 0 = t); the remaining axis gets a pass of its own
  bool t16, fold;                              // ... and the inverse, the forward one is ff_dct_t16.cu
  float t16_mat[16][8];                        // C_T[k][i], i < 8
  float fold_mat[32 * 16];                     // C[k][i] of the second axis, i < n2 / 2
  int dct2_chunk;                              // channels of its work items: 32, or 16 for the larger planes
  alignas(64) unsigned char tmap_mid[128];     // CUtensorMap over the mid-band / high-band coefficient buffers
  alignas(64) unsigned char tmap_high[128];
  alignas(64) unsigned char tmap_low[128];     // ... over the pooled low band (bf16 copy), when low_tc_ok
  bool low_tc_ok;                              // the low branch runs in the tensor-core attention launch
  long long launches;
  bool masks_given;                            // the call has the caller's masks (set by every call before its first launch)
  // ff_forward_host on the tensor-core path: copies run on a second stream, one event per launch
  // group of the forward transform (host -> device) and of the inverse transform (device -> host)
  cudaStream_t copy_stream;
  cudaEvent_t ev_copy[2 * FF_COPY_EVENTS + 1];   // [0,64) input groups, [64,128) output groups, [128] start
  bool pipe_in, pipe_out;                      // set for the duration of one ff_forward_host
  void* pipe_out_host;                         // host destination of `out`
  size_t pipe_head_bytes;                      // bytes of one (batch, head) slice of Q / K / V / out
  bool profiling;
  cudaEvent_t ev[FF_STAGE_COUNT + 1];
  long long stage_launches[FF_STAGE_COUNT];
  char err[512];
};

// Records `msg` as the calling thread's plan-less error (what ff_last_error(NULL) returns).
void ff_set_thread_error(const char* msg);

void ff_compute_layout(const FFDims& dm, bool with_staging, FFLayout* lay);

// ---- kernel launchers (ff_simt.cu).  Each returns the cudaError_t of its launches. --------------
// (..._init: kernel attributes on the current device, set at plan creation; of the forms the configuration uses where
// there are many: the first look at a kernel loads it)
cudaError_t ffk_simt_init();
cudaError_t ffk_attention_tc_init();
cudaError_t ffk_exchange_tc_init(const FFDims& dm);
cudaError_t ffk_dct_tc_init(const FFDims& dm, int sm_count);
cudaError_t ffk_dct2_init();
cudaError_t ffk_proj_init();
cudaError_t ffk_stats_init(const FFDims& dm);
cudaError_t ffk_forward_transform(ff_plan* p, const void* Q, const void* K, const void* V, bool want_energy, cudaStream_t st);
// ---- pooling, band statistics, router, worklist (ff_stats.cu) ---------------------------------------
cudaError_t ffk_set_timesteps(ff_plan* p, const float* host, cudaStream_t st);     // (more than FF_TS_INLINE samples)
cudaError_t ffk_band_stats(ff_plan* p, const uint8_t* alloc_in, const float* timestep_host, bool bands_summed, cudaStream_t st);
cudaError_t ffk_attention_simt(ff_plan* p, int band_bits, cudaStream_t st);   // band_bits: which bands to run
// ---- tensor-core attention (ff_attn_tc.cu) -------------------------------------------------------
bool ffk_tc_supported(const FFDims& dm);
bool ffk_tc_prepare(ff_plan* p);               // builds the tensor maps over the workspace
cudaError_t ffk_attention_tc(ff_plan* p, cudaStream_t st);
// ---- tensor-core exchange (ff_exchange_tc.cu) -----------------------------------------------------
bool ffk_exchange_tc_supported(const FFDims& dm);
bool ffk_exchange_tc_build_tables(ff_plan* p);
bool ffk_exchange_tc_prepare(ff_plan* p);
cudaError_t ffk_exchange_tc(ff_plan* p, int h0, int g, void* grid_hi, void* grid_lo, cudaStream_t st);
// ---- tensor-core transform (ff_dct_tc.cu) --------------------------------------------------------
bool ffk_dct_tc_supported(const FFDims& dm);
size_t ffk_dct_tc_scratch_bytes(const FFDims& dm, int group);
cudaError_t ffk_forward_transform_tc(ff_plan* p, const void* Q, const void* K, const void* V, bool want_energy,
                                     cudaStream_t st);
cudaError_t ffk_inverse_transform_tc(ff_plan* p, int h0, int g, void* out, cudaStream_t st);
// ---- two axis passes in one launch, intermediate in shared memory (ff_dct2_tc.cu) --------------------
bool ffk_dct2_supported(const FFDims& dm, int* axis2, int* chunk);
bool ffk_dct2_build_image(ff_plan* p, int axis, int inverse, const float* mat_host, int n);
cudaError_t ffk_dct2_forward(ff_plan* p, const void* Q, const void* K, const void* V, int g0, int g, void* out_hi, void* out_lo,
                             bool clear_energy, cudaStream_t st);
cudaError_t ffk_dct2_inverse(ff_plan* p, const void* in_hi, const void* in_lo, int h0, int g, void* out, cudaStream_t st);
// ---- the same with the second axis in registers (ff_dct_t16.cu): inverse with t = 16, forward with 16 or 32 positions --
cudaError_t ffk_dct_t16_init();
bool ffk_dct_t16_supported(const ff_plan* p);
bool ffk_dct_fold_supported(const ff_plan* p);
bool ffk_dct_fold_build_image(ff_plan* p, const float* mat_host);
cudaError_t ffk_dct_fold_forward(ff_plan* p, const void* Q, const void* K, const void* V, int g0, int g, void* out_hi, void* out_lo,
                                 bool clear_energy, cudaStream_t st);
cudaError_t ffk_dct_t16_inverse(ff_plan* p, const void* in_hi, const void* in_lo, int h0, int g, void* out, cudaStream_t st);
// ---- projections around the path (ff_proj_tc.cu) -------------------------------------------------------
bool ffk_proj_supported(const FFDims& dm);
cudaError_t ffk_project_qkv(ff_plan* p, const void* X, const void* Wqkv, void* Q, void* K, void* V, cudaStream_t st);
cudaError_t ffk_project_out(ff_plan* p, const void* O, const void* Wo, void* out, cudaStream_t st);
// ---- summary tokens and the low band's part of the exchange (ff_summary.cu) ----------------------------
int ffk_summary_pieces(const FFDims& dm);
bool ffk_low_in_summary(const ff_plan* p);     // the summary launch computes the (short) pooled low band's attention too
cudaError_t ffk_summaries(ff_plan* p, cudaStream_t st);
cudaError_t ffk_exchange_low(ff_plan* p, int h0, int g, void* grid_hi, void* grid_lo, cudaStream_t st);
// Keys of the tensor-core exchange: the 3m summaries of a head, rounded up to a k-step; bytes of one operand image
// pair (hi, lo; two 64-channel halves of 128-byte rows each).
FF_HD int ff_exchange_keys(int m) { return (3 * m + 15) / 16 * 16; }
FF_HD size_t ff_zimg_bytes(int m) { return (size_t)4 * ff_exchange_keys(m) * 128; }
cudaError_t ffk_exchange_inverse(ff_plan* p, void* out, cudaStream_t st);
