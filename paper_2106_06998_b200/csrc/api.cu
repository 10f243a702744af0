// libxconv C ABI: argument checks, workspace planning and kernel dispatch.
#include <cmath>
#include "../../include/xconv.h"

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>

#include "common.cuh"
#include "simt_kernels.cuh"
#include "conv_fma.h"
#include "conv_split.h"
#include "contract_split.h"
#include "gemm_split.h"
#include "small_f32.h"
#include "tc_api.h"
#include <type_traits>

namespace xconv {

thread_local int g_last_cuda_error = 0;
thread_local int g_launches = 0;

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
static inline long cdiv(long a, long b) { return (a + b - 1) / b; }
static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static xconv_status check_launch() {
  ++g_launches;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

// A fresh non-zero tag per API call (see the workspace header in common.cuh).
static std::atomic<unsigned int> g_call_tag{0x51u};
thread_local unsigned int g_tag = 1u;
static void new_call() {
  g_launches = 0;
  g_tag = g_call_tag.fetch_add(2u) | 1u;
}
unsigned int call_tag() { return g_tag; }

// Depth of the volume and of the kernel (0 and 1 both mean a planar layer).
static inline int depth(const xconv_desc* d) { return d->D > 1 ? d->D : 1; }
static inline int kdepth(const xconv_desc* d) { return d->KD > 1 ? d->KD : 1; }

static xconv_status validate(const xconv_desc* d) {
  if (!d) return XCONV_ERR_INVALID_ARG;
  if (d->B <= 0 || d->Cin <= 0 || d->Cout <= 0 || d->H <= 0 || d->W <= 0 || d->r <= 0 || d->KH <= 0 || d->KW <= 0)
    return XCONV_ERR_INVALID_ARG;
  if (d->dtype != XCONV_F32 && d->dtype != XCONV_BF16 && d->dtype != XCONV_F16) return XCONV_ERR_INVALID_ARG;
  if (d->pad_h < 0 || d->pad_w < 0 || d->D < 0 || d->KD < 0 || d->pad_d < 0) return XCONV_ERR_INVALID_ARG;
  if (d->circular != 0 && d->circular != 1) return XCONV_ERR_INVALID_ARG;
  if (d->KH != d->KW || (d->KH != 1 && d->KH != 3 && d->KH != 5)) return XCONV_ERR_UNSUPPORTED;
  if (2 * d->pad_h != d->KH - 1 || 2 * d->pad_w != d->KW - 1) return XCONV_ERR_UNSUPPORTED;
  // kernels over volumes: 3 x 3 x 3, or planar kernels (1 x K x K) applied to every plane
  if (kdepth(d) != 1 && !(kdepth(d) == 3 && d->KH == 3)) return XCONV_ERR_UNSUPPORTED;
  if (2 * d->pad_d != kdepth(d) - 1) return XCONV_ERR_UNSUPPORTED;
  // circular shifts (the operator T_k of the paper's Section 3) are served for planar layers only
  if (d->circular && (depth(d) > 1 || kdepth(d) > 1)) return XCONV_ERR_UNSUPPORTED;
  // 32-bit grid and index limits of the kernels.  r, B and the channel counts land on the y axis of a
  // grid (at most 65535 blocks of 16 or more) in the FP32-FMA kernels, and r and B trade places when
  // xconv_wgrad sums over the probes first.
  const long px = (long)depth(d) * d->H * d->W;
  const long Kdim = px * d->Cin, Q = px * d->Cout;
  if (Kdim > (1L << 40) || Q > (1L << 40) || (long)d->B * depth(d) * d->H * cdiv(d->W, 32) > 2000000000L ||
      (long)depth(d) * d->H > 2000000000L)
    return XCONV_ERR_UNSUPPORTED;
  const long axis_limit = 65535L * 16;
  if (d->r > axis_limit || d->B > axis_limit || d->Cin > axis_limit || d->Cout > axis_limit ||
      (long)d->r * d->B > (1L << 40) || (long)d->r * depth(d) > 2000000000L || (long)d->B * depth(d) > 2000000000L)
    return XCONV_ERR_UNSUPPORTED;
  return XCONV_OK;
}

// The sketch, the back-probe and the per-channel kernels see the pixels of a sample as one flat axis: for
// them a volume is an image with D*H rows.
static xconv_desc flat(const xconv_desc* d) {
  xconv_desc f = *d;
  f.H = d->H * depth(d);
  f.D = 1; f.KD = 1; f.pad_d = 0;
  f.zero_blocks = nullptr;
  return f;
}
// The tensor-core contraction works plane by plane, on D times the probes.  A planar kernel on a volume treats every plane as an image of its
// own (D = 1 from there on); a 3 x 3 x 3 kernel keeps D, so that the kernels know where a volume ends.
static xconv_desc planes_ct(const xconv_desc* d) {
  xconv_desc f = *d;
  f.r = d->r * depth(d);
  if (kdepth(d) == 1) {
    f.D = 1; f.KD = 1; f.pad_d = 0;
    if (depth(d) > 1) f.zero_blocks = nullptr;      // the mask is per probe, and r now counts planes
  }
  return f;
}
static inline bool volumetric(const xconv_desc* d) { return kdepth(d) == 3; }

// ----------------------------------------------------------------------------------- plans
// A plan fixes every launch shape and workspace offset from the descriptor alone, so that
// xconv_workspace_bytes and the entry points always agree.

static const size_t WS_HEADER = 256;   // word 0: status left by pipelined kernels

struct SketchPlan {
  bool tc;
  bool stream; StreamSketchPlan s;     // few samples or few probes (stream_tc.cu)
  bool split; GemmSplitPlan g;         // float rows on the tensor cores (gemm_split.cu)
  int splits; long k_per_split;        // simt
  TcSketchPlan t;                      // tcgen05
  size_t part_off, bytes;
};

// Float layers whose sketch and back-probe go to the tensor cores (gemm_split.cu): where their clocks, at the part of the rates they were
// measured at and with 5000 more for launches and first copies, are below those of the multiply-adds.  Those take 70 a clock
// and SM on tiles of 64 x 64 (sketch), and in the back-probe 310 clocks a term of a wave of blocks, or the bytes at 16 a clock and SM.
// On 160 layers this picks within 1.5 % (sketch) and 1 % (back-probe) of the faster kernel of each; us, multiply-adds -> this:
// sketch 128 x 64 rows, 65536 terms 39 -> 26, 512 x 4, 1.6 M terms 3500 -> 1300, but 86 x 128 rows, 4624 terms 10.4 -> 14.2; back-probe
// 16 rows, 512 terms 84 -> 17, 256 rows, 64 terms, 48672 positions 57 -> 41, but 16 rows, 4 terms, 3.3 M positions 66 -> 308.
static bool plan_sketch_f32(const xconv_desc* d, GemmSplitPlan* p) {
  const double macs = (double)align_up(d->r, 64) * align_up(d->B, 64) * depth(d) * d->H * d->W * d->Cin;
  return d->dtype == XCONV_F32 && plan_sketch_split(d, p) && 1.8 * p->clocks + 5000.0 < macs / (148.0 * 70.0);
}
static bool plan_backprobe_f32(const xconv_desc* d, GemmSplitPlan* p) {
  if (d->dtype != XCONV_F32 || !plan_backprobe_split(d, p)) return false;
  const double Q = (double)depth(d) * d->H * d->W * d->Cout;
  const double waves = (double)cdiv(cdiv((long)Q, 1024) * cdiv(d->r, 16), 296);
  return 1.5 * p->clocks + 5000.0 < std::max(waves * d->B * 310.0, ((double)d->B + d->r) * 4.0 * Q / (148.0 * 16.0));
}

// The back-probe of 16-bit layers that neither tc_plan_wgrad's nor the streaming one serves: where the clocks of gemm_split.cu, with 5000 more for
// the launch that splits S, are below those of the multiply-adds, 1270 a term of a wave of blocks or the stores of L at 7 bytes a clock and SM.  us,
// multiply-adds -> this: 118 rows, 5 terms, 3.5 M positions 675 -> 371, 512 rows, 11 terms, 3136 positions 10.4 -> 7.2, 128 rows, 187
// terms, 750000 positions 2325 -> 214, but 256 rows, 4 terms, 2400 positions 6.4 -> 7.5, 157 rows, 6 terms, 89856 positions 18.7 -> 19.7.
static bool plan_backprobe_whole(const xconv_desc* d, GemmSplitPlan* p) {
  if (d->dtype == XCONV_F32 || !plan_backprobe_split(d, p)) return false;
  const double Q = (double)depth(d) * d->H * d->W * d->Cout;
  const double waves = (double)cdiv(cdiv((long)Q, 1024) * cdiv(d->r, 16), 296);
  return p->clocks + 5000.0 < std::max(waves * d->B * 1270.0, d->r * 2.0 * Q / (148.0 * 7.0));
}

static SketchPlan plan_sketch(const xconv_desc* d_, bool seeded = false) {
  const xconv_desc fl = flat(d_);
  const xconv_desc* d = &fl;
  SketchPlan p{};
  const long K = (long)d->H * d->W * d->Cin;
  p.part_off = WS_HEADER;
  p.stream = tc_plan_sketch_stream(d, seeded, &p.s);
  if (p.stream) {
    p.bytes = p.part_off + align_up(p.s.part_bytes, 256);
    return p;
  }
  p.tc = tc_plan_sketch(d, &p.t, seeded && tc_sketch_can_redraw(d));
  if (p.tc) {
    p.bytes = p.part_off + align_up(p.t.part_bytes, 256);
    return p;
  }
  if (plan_sketch_f32(d, &p.g)) {
    p.split = true;
    p.bytes = p.part_off + align_up(p.g.bytes, 256);
    return p;
  }
  const long tiles = cdiv(d->r, 64) * cdiv(d->B, 64);
  // short chains: a block walks its k-range step by step with one step of loads in flight, so the time of a
  // sketch is (steps per block) x (load latency) unless the range is dealt to many blocks
  // one full wave of the grid: four blocks of the transposing kernel fit an SM, three of the cp.async kernel that
  // serves float rows on 16-byte boundaries (80 registers, 54 KB)
  const long per_sm = (d->dtype == XCONV_F32 && K % 4 == 0) ? 3 : 4;
  long splits = std::max(1L, std::min(cdiv(per_sm * 148, tiles), cdiv(K, 128)));
  splits = std::min(splits, 2048L);
  p.k_per_split = align_up((size_t)cdiv(K, splits), 32);
  p.splits = (int)cdiv(K, p.k_per_split);
  p.bytes = p.part_off + align_up((size_t)p.splits * d->r * d->B * sizeof(float), 256);
  return p;
}

// 16-bit tensors whose channel count is not a multiple of 8 have rows the copy engine cannot step through (16-byte rule).
// The tensor-core kernels then get a copy in the workspace with the channels padded by zeros to the next multiple of 8.
static inline int pad8(int c) { return (c + 7) / 8 * 8; }
static size_t padded_bytes(long rows, int c) { return c % 8 ? align_up((size_t)rows * pad8(c) * 2, 256) : 0; }

// One or two tensors of C channels; a thread writes one 16-byte piece.
struct PadJob { const unsigned short* in; unsigned short* out; long pieces; };
static __global__ void __launch_bounds__(256) pad_channels_kernel(const PadJob one, const PadJob two, int C, int per_row) {
  const long at = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool second = at >= one.pieces;
  const long i = second ? at - one.pieces : at;
  const unsigned short* in = second ? two.in : one.in;
  unsigned short* out = second ? two.out : one.out;
  const long row = i / per_row;
  const int c0 = (int)(i - row * per_row) * 8;
  pdl_wait();
  pdl_trigger();
  if (i >= (second ? two.pieces : one.pieces)) return;
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (c0 + k < C) w[k >> 1] |= (uint32_t)in[row * C + c0 + k] << (16 * (k & 1));
  *reinterpret_cast<uint4*>(out + i * 8) = make_uint4(w[0], w[1], w[2], w[3]);
}

// `t` (and `u`, where there is one) themselves, or their padded copies at *ws (which then moves on behind them).
static xconv_status pad_channels(const void*& t, long rows, int C, char*& ws, cudaStream_t st, const void** u = nullptr, long rows_u = 0) {
  if (C % 8 == 0) return XCONV_OK;
  const int per_row = pad8(C) / 8;
  PadJob one{static_cast<const unsigned short*>(t), reinterpret_cast<unsigned short*>(ws), rows * per_row}, two{nullptr, nullptr, 0};
  t = ws;
  ws += padded_bytes(rows, C);
  if (u) {
    two = PadJob{static_cast<const unsigned short*>(*u), reinterpret_cast<unsigned short*>(ws), rows_u * per_row};
    *u = ws;
    ws += padded_bytes(rows_u, C);
  }
  const cudaError_t e = launch_pdl(pad_channels_kernel, dim3((unsigned)cdiv(one.pieces + two.pieces, 256)), dim3(256), 0, st, one, two, C, per_row);
  ++g_launches;
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

struct WgradPlan {
  bool tc_bp, tc_ct;
  bool split_bp; GemmSplitPlan g;      // back-probe with S in parts (gemm_split.cu): float layers, 16-bit ones that the others do not serve
  bool stream_bp;                      // back-probe of few rows (stream_tc.cu)
  bool halo;                           // contraction of few channels (contract_tc.cu) instead of the one of tc_kernels.cu
  TcHaloPlan h;                        // ... on the layer with its channels padded to multiples of 8
  bool split; ContractSplitPlan c;     // contraction of float layers on the tensor cores (contract_split.cu)
  size_t ct_bytes;                     // scratch of the contraction: partial sums, padded copies
  int splits; long items_per_split;    // simt contraction
  TcWgradPlan t;                       // tcgen05: contraction fields (planned on the per-plane layer)
  TcWgradPlan tb;                      // tcgen05: back-probe fields (planned on the flattened layer)
  size_t l_off, sb_off, part_off, bytes;
};

// Float layers whose contraction goes to the tensor cores (contract_split.cu).  It was faster on every one of 160 layers (us: 84 -> 72 to
// 2680 -> 520, two thirds of them more than threefold).  The limit (multiply-adds at 70 a clock and SM on tiles of 64 x 32 channels and 32 pixels
// for 15000 clocks) is not where the two cross, which is below it: it leaves the layer 16 -> 16 channels, 32 x 32, 8 probes on the kernel that
// the parity tests name for it, and gives up a few microseconds on layers of that size.
static bool plan_contract_f32(const xconv_desc* d, ContractSplitPlan* p) {
  const double macs = (double)d->r * depth(d) * d->H * cdiv(d->W, 32) * 32 * kdepth(d) * d->KH * d->KW * align_up(d->Cin, 64) * align_up(d->Cout, 32);
  return d->dtype == XCONV_F32 && macs > 15000.0 * 148 * 70 && plan_contract_split(d, p);
}

static WgradPlan plan_wgrad_core(const xconv_desc* d) {
  WgradPlan p{};
  const long Q = (long)depth(d) * d->H * d->W * d->Cout;
  const int T = kdepth(d) * d->KH * d->KW;
  const size_t lsz = d->dtype == XCONV_F32 ? 4 : 2;
  p.l_off = WS_HEADER;
  p.sb_off = p.l_off + align_up((size_t)d->r * Q * lsz, 256);
  const xconv_desc f = flat(d);
  p.tc_bp = (tc_plan_wgrad(&f, &p.tb) & 1) != 0;
  p.stream_bp = tc_backprobe_streams(&f, p.tc_bp);
  p.split_bp = d->dtype == XCONV_F32 ? plan_backprobe_f32(&f, &p.g) : !p.tc_bp && !p.stream_bp && plan_backprobe_whole(&f, &p.g);
  p.part_off = p.sb_off + align_up(p.split_bp ? p.g.bytes : (size_t)d->r * d->B * 2, 256);
  const xconv_desc c = planes_ct(d);    // the tensor-core contraction works plane by plane
  p.tc_ct = (tc_plan_wgrad(&c, &p.t) & 2) != 0;
  // The contraction for few channels: where the other one does not go (drained; if its channel blocks are not mostly padding, see
  // halo_channels), and where that one leaves MMA rows empty or copies Z once per offset.  Measured, other -> this, us: 3 x 3, 32 -> 32 channels, 64 probes of 64 x 64: 27.6 -> 17.0, 128 -> 32
  // channels out 35 -> 22 (but 32 -> 256 31 -> 37, 128 -> 128 35 -> 41, 64 -> 64 20.8 -> 20.7); 5 x 5, 32 channels 58 -> 20,
  // 128: 36.4 -> 36.5; pointwise, 64 channels 12.6 -> 9.9, 128: 14.7 -> 19.4; 3 x 3 x 3, 32 -> 64 73 -> 30, 128 -> 128 38 -> 28,
  // 96 -> 96, a quarter of it padding, 43 -> 47.  (A list of zero blocks is only read by the other one.)
  xconv_desc e = *d;
  e.Cin = pad8(d->Cin); e.Cout = pad8(d->Cout);
  const int most = std::max(d->Cin, d->Cout);
  const bool whole = (d->Cin == 32 || d->Cin % 64 == 0) && (d->Cout == 32 || d->Cout % 64 == 0);
  const bool few = volumetric(d) ? most <= 128 && whole : d->KH == 3 ? d->Cout <= 32 : most <= 64;
  const bool other = p.tc_ct && (p.t.ct_masked || !few);
  if (!other && tc_plan_halo(&e, !p.tc_ct, &p.h)) {
    p.halo = true;
    const long px = (long)depth(d) * d->H * d->W * d->r;
    p.ct_bytes = align_up(p.h.part_bytes, 256) + padded_bytes(px, d->Cin) + padded_bytes(px, d->Cout);
    p.bytes = p.part_off + p.ct_bytes;
    return p;
  }
  if (p.tc_ct) {
    p.ct_bytes = align_up(p.t.part_bytes, 256);
    p.bytes = p.part_off + p.ct_bytes;
    return p;
  }
  if (plan_contract_f32(d, &p.c)) {
    p.split = true;
    p.ct_bytes = align_up(p.c.bytes, 256);
    p.bytes = p.part_off + p.ct_bytes;
    return p;
  }
  const long items = (long)d->r * depth(d) * d->H * cdiv(d->W, 32);
  // blocks per split: 5 x 5 kernels take one offset row per block, 3 x 3 x 3 kernels three
  const long tiles = cdiv(d->Cin, 64) * cdiv(d->Cout, 32) * (d->KH == 5 ? 5 : volumetric(d) ? 3 : 1);
  // one wave of the grid: two blocks of this kernel fit an SM (its 72 accumulators per thread)
  long splits = std::max(1L, std::min(std::max(1L, 2L * 148 / tiles), cdiv(items, 2)));
  splits = std::min(splits, 4096L);
  p.items_per_split = cdiv(items, splits);
  p.splits = (int)cdiv(items, p.items_per_split);
  p.ct_bytes = align_up((size_t)p.splits * d->Cout * T * d->Cin * sizeof(float), 256);
  p.bytes = p.part_off + p.ct_bytes;
  return p;
}

// Re-association for r > B.  The estimate is one bilinear form,
//   dW[m,n,k] = scale_n * sum_{j,b,q} S[j,b] dY[b,m,q] Z[j,n,q+k],
// and Algorithm 1 sums over b first (L = S dY^T, cost r*Cout*N*(B + 9*Cin)).  Summing over j first
// gives Xr[b,n,p] = sum_j S[j,b] Z[j,n,p] -- the activation rebuilt from its sketch -- followed by the
// same offset contraction over the batch, dW = scale * sum_{b,q} dY[b,m,q] Xr[b,n,q+k]
// (cost B*Cin*N*(r + 9*Cout)): cheaper exactly when r > B.  Both steps are the kernels of the other
// order with the roles of the tensors swapped, so xconv_wgrad picks the cheaper order; the explicit
// halves xconv_backprobe / xconv_contract always follow the paper's order.
struct SwappedWgrad {
  bool on;
  xconv_desc d1, d2;       // d1: "back-probe" producing Xr; d2: contraction over the batch
  WgradPlan p1, p2;
  size_t x_off, st_off, sb_off, part_off, bytes;
};

static SwappedWgrad plan_wgrad_swapped(const xconv_desc* d) {
  SwappedWgrad w{};
  w.on = d->r > d->B;
  if (!w.on) return w;
  w.d1 = *d; w.d1.B = d->r; w.d1.r = d->B; w.d1.Cout = d->Cin; w.d1.chan_scale = nullptr;
  w.d2 = *d; w.d2.r = d->B;
  w.d1.zero_blocks = w.d2.zero_blocks = nullptr;      // neither step sums over the probes block by block
  w.p1 = plan_wgrad_core(&w.d1);
  w.p2 = plan_wgrad_core(&w.d2);
  const size_t es = d->dtype == XCONV_F32 ? 4 : 2;
  w.x_off = WS_HEADER;
  w.st_off = w.x_off + align_up((size_t)d->B * depth(d) * d->H * d->W * d->Cin * es, 256);
  w.sb_off = w.st_off + align_up((size_t)d->r * d->B * 4, 256);
  w.part_off = w.sb_off + align_up(w.p1.split_bp ? w.p1.g.bytes : (size_t)d->r * d->B * 2, 256);
  w.bytes = w.part_off + w.p2.ct_bytes;
  return w;
}

static WgradPlan plan_wgrad(const xconv_desc* d, SwappedWgrad* swapped = nullptr) {
  WgradPlan p = plan_wgrad_core(d);
  const SwappedWgrad w = plan_wgrad_swapped(d);
  if (w.on) p.bytes = std::max(p.bytes, w.bytes);
  if (swapped) *swapped = w;
  return p;
}

// ----------------------------------------------------------------------------------- probes from a seed

// Z redrawn from a seed: entry e (in memory order) is +1 if bit (e mod 128) of Philox block (e div 128) is 0,
// -1 if it is 1; bit b is bit (b mod 32) of output word (b div 32).  One thread writes eight entries.
template <typename T>
__global__ void __launch_bounds__(256) probes_from_seed_kernel(T* __restrict__ Z, long total, uint32_t k0, uint32_t k1) {
  pdl_trigger();
  pdl_wait();
  const long e0 = ((long)blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (e0 >= total) return;
  const unsigned long long blk = (unsigned long long)e0 >> 7;
  const uint4 w = philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), k0, k1);
  const int word = (int)((e0 & 127) >> 5);
  const uint32_t wv = word == 0 ? w.x : word == 1 ? w.y : word == 2 ? w.z : w.w;
  const uint32_t bits = (wv >> (e0 & 31)) & 0xFFu;
  if (e0 + 8 <= total) {                     // Z is 16-byte aligned and e0 a multiple of 8: vector stores
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = ((bits >> i) & 1u) ? -1.0f : 1.0f;
    st4(Z + e0, make_float4(v[0], v[1], v[2], v[3]));
    st4(Z + e0 + 4, make_float4(v[4], v[5], v[6], v[7]));
    return;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (e0 + i < total) Z[e0 + i] = from_f<T>(((bits >> i) & 1u) ? -1.0f : 1.0f);
}

static xconv_status run_probes_from_seed(const xconv_desc* d, unsigned long long seed, void* Z, cudaStream_t st) {
  const long total = (long)d->r * depth(d) * d->H * d->W * d->Cin;
  const unsigned grid = (unsigned)cdiv(cdiv(total, 8), 256);
  const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
  cudaError_t e = d->dtype == XCONV_F32
      ? launch_pdl(probes_from_seed_kernel<float>, dim3(grid), dim3(256), 0, st, static_cast<float*>(Z), total, k0, k1)
      : d->dtype == XCONV_F16
      ? launch_pdl(probes_from_seed_kernel<f16>, dim3(grid), dim3(256), 0, st, static_cast<f16*>(Z), total, k0, k1)
      : launch_pdl(probes_from_seed_kernel<bf16>, dim3(grid), dim3(256), 0, st, static_cast<bf16*>(Z), total, k0, k1);
  ++g_launches;
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

// Z with standard normal entries from a seed: Philox block b (counter word 2 = 1, which keeps the stream apart from
// the Rademacher one) gives entries 4b .. 4b+3, two Box-Muller pairs.  One thread per block.
template <typename T>
__global__ void __launch_bounds__(256) gaussian_probes_kernel(T* __restrict__ Z, long total, uint32_t k0, uint32_t k1) {
  pdl_trigger();
  pdl_wait();
  const long b = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long e0 = b * 4;
  if (e0 >= total) return;
  const uint4 w = philox4x32_10((uint32_t)b, (uint32_t)((unsigned long long)b >> 32), k0, k1, 1u);
  const float2 p0 = box_muller_u24(w.x, w.y), p1 = box_muller_u24(w.z, w.w);
  if (e0 + 4 <= total) { st4(Z + e0, make_float4(p0.x, p0.y, p1.x, p1.y)); return; }
  const float v[4] = {p0.x, p0.y, p1.x, p1.y};
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (e0 + i < total) Z[e0 + i] = from_f<T>(v[i]);
}

static xconv_status run_gaussian_probes(const xconv_desc* d, unsigned long long seed, void* Z, cudaStream_t st) {
  const long total = (long)d->r * depth(d) * d->H * d->W * d->Cin;
  const unsigned grid = (unsigned)cdiv(cdiv(total, 4), 256);
  const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
  cudaError_t e = d->dtype == XCONV_F32
      ? launch_pdl(gaussian_probes_kernel<float>, dim3(grid), dim3(256), 0, st, static_cast<float*>(Z), total, k0, k1)
      : d->dtype == XCONV_F16
      ? launch_pdl(gaussian_probes_kernel<f16>, dim3(grid), dim3(256), 0, st, static_cast<f16*>(Z), total, k0, k1)
      : launch_pdl(gaussian_probes_kernel<bf16>, dim3(grid), dim3(256), 0, st, static_cast<bf16*>(Z), total, k0, k1);
  ++g_launches;
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

// Block-sparse probing vectors (Eq. 7) from a seed.  keep[g], g = j * Cin + n: block n of probing vector j is non-zero
// iff word (g mod 4) of Philox block (g div 4) -- counter word 2 = 2, apart from the two value streams -- is below the
// threshold floor(p * 2^32).
__global__ void __launch_bounds__(256) block_keep_kernel(unsigned char* __restrict__ keep, long total, uint32_t k0,
                                                         uint32_t k1, unsigned long long threshold) {
  const long b = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (b * 4 >= total) return;
  const uint4 w = philox4x32_10((uint32_t)b, (uint32_t)((unsigned long long)b >> 32), k0, k1, 2u);
  const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (b * 4 + i < total) keep[b * 4 + i] = (unsigned long long)v[i] < threshold ? 1 : 0;
}
// scale[n] = 1 / nnz(Z_n), the number of probing vectors whose block n is kept (Eq. 8); 0 for a channel no vector probes.
__global__ void __launch_bounds__(256) keep_scale_kernel(const unsigned char* __restrict__ keep, int r, int Cin,
                                                         float* __restrict__ scale) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= Cin) return;
  int nnz = 0;
  for (int j = 0; j < r; ++j) nnz += keep[(long)j * Cin + n];
  scale[n] = nnz > 0 ? __fdiv_rn(1.0f, (float)nnz) : 0.0f;
}
// The dropped blocks of a dense Z set to +0.  Entry e belongs to probe e / per_probe and channel e % Cin.
template <typename T>
__global__ void __launch_bounds__(256) drop_blocks_kernel(T* __restrict__ Z, const unsigned char* __restrict__ keep,
                                                          long total, long per_probe, int Cin) {
  const long e0 = ((long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long e = e0 + i;
    if (e < total && !keep[(e / per_probe) * Cin + e % Cin]) Z[e] = from_f<T>(0.0f);
  }
}

static size_t probes_bytes(const xconv_desc* d) {
  return align_up((size_t)d->r * depth(d) * d->H * d->W * d->Cin * (d->dtype == XCONV_F32 ? 4 : 2), 256);
}

// ----------------------------------------------------------------------------------- launchers

// Every block of a dependent launch pays for its go-ahead and its wait: 51200 blocks (5 x 5, 128 -> 512 channels) 34 us without,
// 54 with; 36000 blocks 26 and 38; 18000 14 and 20.  It saves 2 us of launch (1280 blocks 22.6 without, 20.3 with).
static const unsigned REDUCE_PDL_BLOCKS = 6000;
// Many splits of up to 16384 outputs are added in pairs, with eight loads of a thread in flight (few splits, or more outputs, lose with that many: us a launch,
// 65536 of 7 3.8 -> 5.1, of 200 18.6 -> 24.6).  32 threads share an output while their blocks are one wave, eight to an SM: 9472 outputs.  Steps of 32 layers
// with 440 to 16384 outputs of 64 to 296 splits take 0.996 of what they take with that line at 2304; behind a kernel that ends first, 8 threads -> 32, us: 64 outputs
// of 200 splits 6.3 -> 5.2, of 2048 21 -> 16.5, 8192 of 64 to 200 the same or 1.9 more, but 12960 of 140 8.2 -> 10.3, of 512 14.5 -> 18.6.
static bool paired_sums(long count, int splits) { return splits >= 64 && count <= 16384; }
static bool wide_sums(long count, int splits) { return paired_sums(count, splits) && count <= 148L * 8 * 8; }
static xconv_status run_reduce(const float* part, float* out, long count, int splits, float alpha, const float* chan_scale,
                               int period, cudaStream_t st) {
  const bool wide = wide_sums(count, splits);
  const dim3 grid((unsigned)cdiv(count, wide ? 8 : 32)), block(256);
  cudaError_t e;
  if (wide) {
    e = launch_pdl(reduce_partials<true, 32, true>, grid, block, 0, st, part, out, count, splits, alpha, chan_scale, period);
  } else if (paired_sums(count, splits)) {
    e = launch_pdl(reduce_partials<true, 8, true>, grid, block, 0, st, part, out, count, splits, alpha, chan_scale, period);
  } else if (grid.x <= REDUCE_PDL_BLOCKS) {
    e = launch_pdl(reduce_partials<true, 8, false>, grid, block, 0, st, part, out, count, splits, alpha, chan_scale, period);
  } else {
    reduce_partials<false, 8, false><<<grid, block, 0, st>>>(part, out, count, splits, alpha, chan_scale, period);
    e = cudaGetLastError();
  }
  ++g_launches;
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

template <typename T>
static xconv_status run_sketch_simt(const xconv_desc* d, const SketchPlan& p, const void* X, const void* Z,
                                    float* S, char* ws, cudaStream_t st, bool held) {
  const long K = (long)d->H * d->W * d->Cin;
  float* part = reinterpret_cast<float*>(ws + p.part_off);
  dim3 grid((unsigned)cdiv(d->B, 64), (unsigned)cdiv(d->r, 64), (unsigned)p.splits);
  // (Started under the kernel before only if it is over at once: grids of a whole wave are dealt unevenly to SMs that that one still uses, 512 x 32 rows, 1176
  // terms 10 -> 12.8 us, and the copies go through what L1 it leaves, 16 x 53 rows, 10816 terms in a training step 83 -> 86; 8 x 8 rows, 16384 terms 10.3 -> 8.0.
  // Behind a convolution that holds whole SMs that is next to nothing: the forward call of 16 -> 96 channels, 78 images of 4 x 34, r = 6, started under it 22.9 -> 28.5.)
  const bool small = !held && (long)grid.x * grid.y * grid.z <= 148 && (d->r + d->B) * K <= 1L << 19;
  if (std::is_same<T, float>::value && K % 4 == 0 && p.k_per_split % GT_KS == 0) {
    const size_t smem = (size_t)GT_STAGES * 128 * GT_LD * sizeof(float);
    cudaError_t ea = cudaFuncSetAttribute(gemm_tn_simt_async, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ea != cudaSuccess) { g_last_cuda_error = (int)ea; return XCONV_ERR_CUDA; }
    ea = launch_if_pdl(small, gemm_tn_simt_async, grid, dim3(256), smem, st, reinterpret_cast<const float*>(Z), reinterpret_cast<const float*>(X), part,
                    d->r, d->B, K, p.k_per_split);
    if (ea != cudaSuccess) { g_last_cuda_error = (int)ea; return XCONV_ERR_CUDA; }
  } else {
    // (an ordinary launch: it loads through L1, of which SMs split for the kernel before have little; 16 x 8 rows, 1440 terms behind a convolution 8 us, 17 started under it)
    gemm_tn_simt<T><<<grid, 256, 0, st>>>(static_cast<const T*>(Z), static_cast<const T*>(X), part, d->r, d->B, K,
                                          p.k_per_split, (K % 4 == 0) ? 1 : 0);
  }
  xconv_status s = check_launch();
  if (s != XCONV_OK) return s;
  return run_reduce(part, S, (long)d->r * d->B, p.splits, 1.0f, nullptr, 1, st);
}

// Whether the sketch kernel of this layer redraws Z itself; otherwise the seeded call first writes Z
// into the workspace (behind the regular scratch) and runs the regular kernels on it.
static bool sketch_redraws(const xconv_desc* d, const SketchPlan& p) {
  const xconv_desc fl = flat(d);
  return p.stream || (p.tc && tc_sketch_can_redraw(&fl));
}

// `held`: the kernel before is one of the call's own that holds the SMs it runs on.
static xconv_status run_sketch(const xconv_desc* d_, const void* X, const void* Z, float* S, void* ws,
                               size_t ws_bytes, cudaStream_t st, const unsigned long long* seed = nullptr, bool held = false) {
  const xconv_desc fl = flat(d_);
  const xconv_desc* d = &fl;
  const SketchPlan p = plan_sketch(d, seed != nullptr);
  const bool redraw = seed && sketch_redraws(d, p);
  const size_t need = p.bytes + (seed && !redraw ? probes_bytes(d) : 0);
  if (!ws || ws_bytes < need) return XCONV_ERR_WORKSPACE;
  if (!aligned16(ws)) return XCONV_ERR_ALIGNMENT;
  char* w = static_cast<char*>(ws);
  if (seed && !redraw) {
    xconv_status s = run_probes_from_seed(d, *seed, w + p.bytes, st);
    if (s != XCONV_OK) return s;
    Z = w + p.bytes;
  }
  if (p.stream) {
    float* part = reinterpret_cast<float*>(w + p.part_off);
    xconv_status s = tc_run_sketch_stream(d, p.s, X, Z, part, w, st, redraw ? seed : nullptr);
    return s == XCONV_OK ? run_reduce(part, S, (long)d->r * d->B, p.s.splits, 1.0f, nullptr, 1, st) : s;
  }
  if (p.tc) return tc_run_sketch(d, p.t, X, Z, S, w, w + p.part_off, st, redraw ? seed : nullptr);
  if (p.split) {
    float* part = reinterpret_cast<float*>(w + p.part_off);
    xconv_status s = run_sketch_split(d, p.g, static_cast<const float*>(X), static_cast<const float*>(Z), part, w, st);
    return s == XCONV_OK ? run_reduce(part, S, (long)d->r * d->B, (int)p.g.splits, 1.0f, nullptr, 1, st) : s;
  }
  return d->dtype == XCONV_F32 ? run_sketch_simt<float>(d, p, X, Z, S, w, st, held)
         : d->dtype == XCONV_F16 ? run_sketch_simt<f16>(d, p, X, Z, S, w, st, held)
                                 : run_sketch_simt<bf16>(d, p, X, Z, S, w, st, held);
}

template <typename T, typename TL>
static xconv_status run_backprobe_simt(const xconv_desc* d, const float* S, const void* dY, void* Lv,
                                       cudaStream_t st) {
  const long Q = (long)depth(d) * d->H * d->W * d->Cout;
  // Block size: the kernel holds about 126 registers per thread, so an SM runs floor(65536 / (126 t)) blocks of t
  // threads; the time goes with (waves of the grid) x (threads an SM runs at once).  256 threads leave the last
  // wave of a small layer part empty (256 blocks for 296 places on the 64-channel 32 x 32 layer; 224 threads fill it).
  int threads = 256;
  long best = -1;
  for (int t = 256; t >= 128; t -= 32) {
    const long per_sm = std::min<long>(65536 / (126L * t), 2048 / t);
    const long blocks = cdiv(cdiv(Q, 4), t) * cdiv(d->r, 16);
    const long cost = cdiv(blocks, 148 * per_sm) * per_sm * t;
    if (best < 0 || cost < best) { best = cost; threads = t; }
  }
  dim3 g1((unsigned)cdiv(cdiv(Q, 4), threads), (unsigned)cdiv(d->r, 16));
  // Small ones start under the kernel before.  Large ones would find their SMs split for that one, with little of the L1 that their loads are in flight
  // through (us with the contraction behind, ordinary -> dependent: 8 rows of 8 terms, 57600 positions 20.4 -> 19.2, but 16 rows of 22, 251008 positions 84 -> 105).
  const bool small = (long)g1.x * g1.y <= 296 && (d->r + d->B) * Q <= 1L << 20;
  const cudaError_t e = launch_if_pdl(small, backprobe_simt<T, TL>, g1, dim3(threads), 0, st, S, static_cast<const T*>(dY), static_cast<TL*>(Lv), d->r, d->B, Q,
                                      (Q % 4 == 0) ? 1 : 0);
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return check_launch();
}

template <typename T, typename TL>
static xconv_status run_contract_simt(const xconv_desc* d, const WgradPlan& p, const void* Lv, const void* Z,
                                      float* dW, float alpha, float* part, cudaStream_t st) {
  const int T9 = kdepth(d) * d->KH * d->KW;
  const TL* L = static_cast<const TL*>(Lv);
  const T* Zt = static_cast<const T*>(Z);
  const bool vec = d->Cin % 4 == 0 && d->Cout % 4 == 0;      // rows of L and Z then start on 4-element boundaries
  const unsigned gx = (unsigned)cdiv(d->Cin, 64), gy = (unsigned)cdiv(d->Cout, 32), gz = (unsigned)p.splits;
  if constexpr (std::is_same<T, float>::value)
    if (small_contract_serves(d)) {
      const xconv_status ss = run_small_contract(d, p.splits, p.items_per_split, L, Zt, part, st);
      return ss == XCONV_OK ? run_reduce(part, dW, (long)d->Cout * T9 * d->Cin, p.splits, alpha, d->chan_scale, d->Cin, st) : ss;
    }
#define XC_CONTRACT(KS, KD, DYS) do { \
    dim3 g2(gx * (KD * KS / DYS), gy, gz); \
    if (vec && std::is_same<TL, float>::value && std::is_same<T, float>::value) { \
      const size_t smem = 2 * contract_async_tile_floats<KS, DYS>() * sizeof(float); \
      auto kern = contract_simt_async<KS, KD, DYS>; \
      cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
      if (ea != cudaSuccess) { g_last_cuda_error = (int)ea; return XCONV_ERR_CUDA; } \
      kern<<<g2, 256, smem, st>>>(reinterpret_cast<const float*>(L), reinterpret_cast<const float*>(Zt), part, d->r, depth(d), d->H, d->W, d->Cin, d->Cout, p.items_per_split, d->circular); \
    } else if (vec) contract_simt<TL, T, KS, KD, DYS, true><<<g2, 256, 0, st>>>(L, Zt, part, d->r, depth(d), d->H, d->W, d->Cin, d->Cout, p.items_per_split, d->circular); \
    else contract_simt<TL, T, KS, KD, DYS, false><<<g2, 256, 0, st>>>(L, Zt, part, d->r, depth(d), d->H, d->W, d->Cin, d->Cout, p.items_per_split, d->circular); \
  } while (0)
  if (volumetric(d)) XC_CONTRACT(3, 3, 3);
  else if (d->KH == 3) XC_CONTRACT(3, 1, 3);
  else if (d->KH == 5) XC_CONTRACT(5, 1, 1);
  else XC_CONTRACT(1, 1, 1);
#undef XC_CONTRACT
  xconv_status s = check_launch();
  if (s != XCONV_OK) return s;
  return run_reduce(part, dW, (long)d->Cout * T9 * d->Cin, p.splits, alpha, d->chan_scale, d->Cin, st);
}

template <typename T>
static xconv_status run_conv_simt(const xconv_desc* d, bool dgrad, const void* in, const void* Wt, void* out,
                                  cudaStream_t st) {
  const int Ci = dgrad ? d->Cout : d->Cin, Co = dgrad ? d->Cin : d->Cout;
  const int D = depth(d), planes = d->B * D;
  ConvFma g;
  if constexpr (std::is_same<T, float>::value) {
    if (small_conv_serves(d))
      return run_small_conv(d, dgrad, static_cast<const float*>(in), static_cast<const float*>(Wt), static_cast<float*>(out), st);
    if (plan_conv_fma(d, dgrad, &g))
      return run_conv_fma(d, g, dgrad, static_cast<const float*>(in), static_cast<const float*>(Wt), static_cast<float*>(out), st);
  }
  dim3 grid((unsigned)((long)planes * d->H * cdiv(d->W, 32)), (unsigned)cdiv(Co, 64));
  const T* i_ = static_cast<const T*>(in);
  const T* w_ = static_cast<const T*>(Wt);
  T* o_ = static_cast<T*>(out);
#define XC_CONV(KS, KD) do { \
    if (dgrad) conv_simt<T, KS, KD, true><<<grid, 256, 0, st>>>(i_, w_, o_, planes, D, d->H, d->W, Ci, Co, d->Cin, d->circular); \
    else       conv_simt<T, KS, KD, false><<<grid, 256, 0, st>>>(i_, w_, o_, planes, D, d->H, d->W, Ci, Co, d->Cin, d->circular); \
  } while (0)
  if (volumetric(d)) XC_CONV(3, 3);
  else if (d->KH == 3) XC_CONV(3, 1);
  else if (d->KH == 5) XC_CONV(5, 1);
  else XC_CONV(1, 1);
#undef XC_CONV
  return check_launch();
}

// Float layers whose convolution goes to the tensor cores (conv_split.cu): all but the smallest.  The call alone is faster from a
// microsecond of multiply-adds on (us, multiply-adds -> this, 160 layers: 8 x 16 -> 16 channels of 32 x 32 12.5 -> 8.6, 4 x 192 -> 48, 37 x 37,
// 1 x 1 14.5 -> 8.9, larger ones 236 -> 57; but 9 x 1 -> 128 channels of 13 x 13, 1 x 1, with the copies before it 15.5 -> 18.6).  The line, 3000
// clocks of 75 multiply-adds a clock and SM, was drawn against those kernels (conv_simt, conv_fma); below it small_f32.cu is the faster one, the first
// of these in 4.8.  From there to twice the line multiply-adds in its tiles would still be faster, but with two to three times the error.
static bool plan_conv_f32(const xconv_desc* d, bool dgrad, ConvSplitPlan* p) {
  const double macs = (double)d->B * depth(d) * d->H * d->W * d->Cin * d->Cout * kdepth(d) * d->KH * d->KW;
  if (d->dtype != XCONV_F32 || macs <= 3000.0 * 148 * 75) return false;
  // Image channels: a block of 16 is nearly all padding.  3 x 3, 1 or 3 -> 64 to 256 channels 376 -> 257, 69 -> 48, 38 -> 31 us, but 3 -> 16
  // 142 -> 290, 1 -> 32 55 -> 72, 5 x 5 3 -> 32 388 -> 889, 3 x 3 x 3 3 -> 64 109 -> 145.
  if ((dgrad ? d->Cout : d->Cin) < 8 && ((dgrad ? d->Cin : d->Cout) < 64 || d->KH == 5 || kdepth(d) == 3)) return false;
  return plan_conv_split(d, dgrad, p);
}

// The convolution with its input channels padded (see pad8) and the scratch its copies take behind the header; the output
// channels have to be a multiple of 8 themselves.
static xconv_desc conv_padded(const xconv_desc* d) {
  xconv_desc e = *d;
  e.Cin = pad8(d->Cin);
  return e;
}
// Pointwise layers of few input channels with one block of conv_simt (32 pixels of a row x 64 channels) per SM at most are done
// there before conv_tc has its tensor maps and its tensor memory: 17 pixels, 8 -> 384 channels 5.7 against 7.2 us a call, 48
// pixels, 24 -> 384 5.8 against 8.2, 96 blocks, 8 -> 200 4.7 against 6.8; but 270 blocks, 24 -> 72 6.2 against 5.2.
static bool conv_tiny(const xconv_desc* d, bool dgrad) {
  const int Ci = dgrad ? d->Cout : d->Cin, Co = dgrad ? d->Cin : d->Cout;
  return d->KH == 1 && kdepth(d) == 1 && Ci <= 24 && (long)d->B * depth(d) * d->H * cdiv(d->W, 32) * cdiv(Co, 64) <= 148;
}
// The tensor-core convolution of this layer, if it goes there.
static bool plan_conv(const xconv_desc* d, bool dgrad, xconv_desc* e, TcConvPlan* t) {
  *e = conv_padded(d);
  return (!dgrad || d->Cin % 8 == 0) && !conv_tiny(d, dgrad) && tc_plan_conv(e, dgrad, t);
}
// (Scratch that a call cannot do without; a float layer with less than `conv_ws_wish` stays on multiply-adds.)
static size_t conv_ws_wish(const xconv_desc* d, bool dgrad) {
  ConvSplitPlan p;
  return plan_conv_f32(d, dgrad, &p) ? WS_HEADER + p.bytes : WS_HEADER;
}
static size_t conv_ws_bytes(const xconv_desc* d, bool dgrad) {
  xconv_desc e;
  TcConvPlan t;
  if (dgrad || d->Cin % 8 == 0 || !plan_conv(d, dgrad, &e, &t)) return WS_HEADER;
  return WS_HEADER + padded_bytes((long)d->B * depth(d) * d->H * d->W, d->Cin) +
         padded_bytes((long)d->Cout * kdepth(d) * d->KH * d->KW, d->Cin);
}

static xconv_status run_conv(const xconv_desc* d, bool dgrad, const void* in, const void* Wt, void* out,
                             char* ws, size_t ws_bytes, cudaStream_t st, bool* held = nullptr) {
  ConvSplitPlan f;
  const bool split = plan_conv_f32(d, dgrad, &f) && ws_bytes >= WS_HEADER + f.bytes;
  if (held) *held = split;
  if (split)
    return run_conv_split(d, f, dgrad, static_cast<const float*>(in), static_cast<const float*>(Wt), static_cast<float*>(out), ws,
                          ws + WS_HEADER, st);
  TcConvPlan t;
  xconv_desc e;
  if (plan_conv(d, dgrad, &e, &t)) {
    char* copies = ws + WS_HEADER;
    if (!dgrad) {
      const xconv_status s = pad_channels(in, (long)d->B * depth(d) * d->H * d->W, d->Cin, copies, st, &Wt, (long)d->Cout * kdepth(d) * d->KH * d->KW);
      if (s != XCONV_OK) return s;
    }
    return tc_run_conv(&e, t, dgrad, in, Wt, out, ws, st);
  }
  return d->dtype == XCONV_F32 ? run_conv_simt<float>(d, dgrad, in, Wt, out, st)
         : d->dtype == XCONV_F16 ? run_conv_simt<f16>(d, dgrad, in, Wt, out, st)
                                 : run_conv_simt<bf16>(d, dgrad, in, Wt, out, st);
}

// L = S dY^T into `L`; `Sb` receives the 16-bit copy or the parts of S that the tensor-core kernels read.
static xconv_status run_backprobe(const xconv_desc* d, const WgradPlan& p, const float* S, const void* dY,
                                  void* L, void* Sb_, char* w, cudaStream_t st, const unsigned long long* seed = nullptr) {
  if (p.split_bp) {
    const xconv_desc f = flat(d);
    return run_backprobe_split(&f, p.g, S, d->B, 1, dY, L, w, static_cast<char*>(Sb_), st);
  }
  if (p.stream_bp) {
    const xconv_desc f = flat(d);
    return tc_run_backprobe_stream(&f, S, d->B, 1, dY, L, !p.tc_bp, w, st, nullptr);
  }
  if (p.tc_bp) {
    const long n = (long)d->r * d->B;
    cudaError_t e = d->dtype == XCONV_F16
        ? launch_pdl(cast_f32_to_16<f16>, dim3((unsigned)cdiv(n, 256)), dim3(256), 0, st, S, static_cast<f16*>(Sb_), n)
        : launch_pdl(cast_f32_to_16<bf16>, dim3((unsigned)cdiv(n, 256)), dim3(256), 0, st, S, static_cast<bf16*>(Sb_), n);
    ++g_launches;
    if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
    const xconv_desc f = flat(d);
    return tc_run_backprobe(&f, p.tb, Sb_, dY, L, w, st, seed);
  }
  return d->dtype == XCONV_F32 ? run_backprobe_simt<float, float>(d, S, dY, L, st)
         : d->dtype == XCONV_F16 ? run_backprobe_simt<f16, f16>(d, S, dY, L, st)
                                 : run_backprobe_simt<bf16, bf16>(d, S, dY, L, st);
}

static xconv_status run_contract(const xconv_desc* d, const WgradPlan& p, const void* L, const void* Z,
                                 float* dW, float alpha, char* part, char* w, cudaStream_t st) {
  if (p.halo) {
    xconv_desc e = *d;
    e.Cin = pad8(d->Cin); e.Cout = pad8(d->Cout);
    const long px = (long)depth(d) * d->H * d->W * d->r;
    char* copies = part + align_up(p.h.part_bytes, 256);
    xconv_status s = pad_channels(Z, px, d->Cin, copies, st);
    if (s == XCONV_OK) s = pad_channels(L, px, d->Cout, copies, st);
    if (s != XCONV_OK) return s;
    return tc_run_halo(&e, p.h, L, Z, d->Cout, d->Cin, dW, alpha, w, part, st);
  }
  if (p.split)
    return run_contract_split(d, p.c, static_cast<const float*>(L), static_cast<const float*>(Z), dW, alpha, w, part, st);
  if (p.tc_ct) {
    const xconv_desc c = planes_ct(d);
    return tc_run_contract(&c, p.t, L, Z, dW, alpha, w, part, st);
  }
  return d->dtype == XCONV_F32
             ? run_contract_simt<float, float>(d, p, L, Z, dW, alpha, reinterpret_cast<float*>(part), st)
         : d->dtype == XCONV_F16
             ? run_contract_simt<f16, f16>(d, p, L, Z, dW, alpha, reinterpret_cast<float*>(part), st)
             : run_contract_simt<bf16, bf16>(d, p, L, Z, dW, alpha, reinterpret_cast<float*>(part), st);
}

static xconv_status check_ws(void* ws, size_t ws_bytes, size_t need) {
  if (!ws || ws_bytes < need) return XCONV_ERR_WORKSPACE;
  if (!aligned16(ws)) return XCONV_ERR_ALIGNMENT;
  return XCONV_OK;
}

// Whether xconv_wgrad_seeded redraws the probing vectors inside its first kernel (the estimator summed over the
// probes first, r > B, with that step on the tensor cores) instead of writing them to the workspace first.
static bool wgrad_redraws(const xconv_desc* d) {
  const SwappedWgrad sw = plan_wgrad_swapped(d);
  return sw.on && (sw.p1.stream_bp ? ((long)depth(d) * d->H * d->W * d->Cin) % 64 == 0 : sw.p1.tc_bp);
}

// `seed` != nullptr (only where wgrad_redraws holds): Z is not read.
static xconv_status run_wgrad(const xconv_desc* d, const float* S, const void* dY, const void* Z, float* dW,
                              void* ws, size_t ws_bytes, cudaStream_t st, const unsigned long long* seed = nullptr) {
  SwappedWgrad sw;
  const WgradPlan p = plan_wgrad(d, &sw);
  xconv_status s = check_ws(ws, ws_bytes, p.bytes);
  if (s != XCONV_OK) return s;
  char* w = static_cast<char*>(ws);
  const float alpha = 1.0f / (float)d->r;
  if (sw.on) {
    // Xr = S^T Z, then the offset contraction over the batch (see plan_wgrad_swapped)
    if ((s = validate(&sw.d1)) != XCONV_OK || (s = validate(&sw.d2)) != XCONV_OK) return s;
    if (sw.p1.stream_bp) {                 // reads S by its columns itself
      const xconv_desc f = flat(&sw.d1);
      s = tc_run_backprobe_stream(&f, S, 1, d->B, Z, w + sw.x_off, !sw.p1.tc_bp, w, st, seed);
    } else if (sw.p1.split_bp) {           // (so does this one)
      const xconv_desc f = flat(&sw.d1);
      s = run_backprobe_split(&f, sw.p1.g, S, 1, d->B, Z, w + sw.x_off, w, w + sw.sb_off, st);
    } else {
      // the transposed sketch, in the form that its reader takes
      const dim3 grid((unsigned)cdiv(d->B, 32), (unsigned)cdiv(d->r, 32)), block(32, 8);
      float* St = reinterpret_cast<float*>(w + sw.st_off);
      cudaError_t e;
      if (!sw.p1.tc_bp) e = launch_pdl(transpose_sketch<float>, grid, block, 0, st, S, St, (int)d->r, (int)d->B);
      else if (d->dtype == XCONV_F16) e = launch_pdl(transpose_sketch<f16>, grid, block, 0, st, S, reinterpret_cast<f16*>(w + sw.sb_off), (int)d->r, (int)d->B);
      else e = launch_pdl(transpose_sketch<bf16>, grid, block, 0, st, S, reinterpret_cast<bf16*>(w + sw.sb_off), (int)d->r, (int)d->B);
      ++g_launches;
      if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
      if (sw.p1.tc_bp) {
        const xconv_desc f = flat(&sw.d1);
        s = tc_run_backprobe(&f, sw.p1.tb, w + sw.sb_off, Z, w + sw.x_off, w, st, seed);
      } else {
        s = run_backprobe(&sw.d1, sw.p1, St, Z, w + sw.x_off, w + sw.sb_off, w, st, seed);
      }
    }
    if (s != XCONV_OK) return s;
    return run_contract(&sw.d2, sw.p2, dY, w + sw.x_off, dW, alpha, w + sw.part_off, w, st);
  }
  s = run_backprobe(d, p, S, dY, w + p.l_off, w + p.sb_off, w, st);
  if (s != XCONV_OK) return s;
  return run_contract(d, p, w + p.l_off, Z, dW, alpha, w + p.part_off, w, st);
}

// One block per (probe, 64-channel group): do the H*W (volumes: D*H*W) rows of 64 channels hold anything but +-0?
template <typename T>
__global__ void __launch_bounds__(256) zero_blocks_kernel(const T* __restrict__ Z, unsigned char* __restrict__ mask,
                                                           long pixels, int Cin) {
  constexpr int PER_ROW = 64 * (int)sizeof(T) / 16;          // 16-byte pieces of one row of the block
  constexpr uint32_t ABS = sizeof(T) == 4 ? 0x7FFFFFFFu : 0x7FFF7FFFu;      // a negative zero is a zero
  const int groups = Cin / 64;
  const long j = blockIdx.x / groups;
  const int g = (int)(blockIdx.x % groups);
  const T* base = Z + j * pixels * Cin + (long)g * 64;
  int any = 0;
  for (long i = threadIdx.x; i < pixels * PER_ROW; i += blockDim.x) {
    const uint4 v = *reinterpret_cast<const uint4*>(base + (i / PER_ROW) * Cin + (i % PER_ROW) * (16 / (int)sizeof(T)));
    any |= ((v.x | v.y | v.z | v.w) & ABS) != 0u;
  }
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) mask[blockIdx.x] = any ? 0 : 1;
}

// FP32 FMA throughput probe: every thread runs 16 independent chains of dependent FMAs on registers (no
// memory traffic), 4 blocks of 256 threads per SM's worth of grid; the result is stored so that the
// compiler keeps the arithmetic.
__global__ void __launch_bounds__(256) fma_rate_kernel(float* __restrict__ sink, int iters, float a, float b) {
  float v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = (float)(threadIdx.x + i);
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = fmaf(v[i], a, b);
  }
  float t = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) t += v[i];
  sink[(long)blockIdx.x * blockDim.x + threadIdx.x] = t;
}

// ----------------------------------------------------------------------------------- per-pair ("independent") probing

// Layout of the scratch of xconv_wgrad_independent: header | Xr (the activation rebuilt per channel) | partial sums
struct IndepPlan { xconv_desc d2; WgradPlan p2; size_t x_off, part_off, bytes; };

static IndepPlan plan_indep(const xconv_desc* d) {
  IndepPlan ip{};
  ip.d2 = *d; ip.d2.r = d->B; ip.d2.chan_scale = nullptr;     // the contraction runs over the batch
  ip.d2.zero_blocks = nullptr;
  ip.p2 = plan_wgrad_core(&ip.d2);
  const size_t es = d->dtype == XCONV_F32 ? 4 : 2;
  ip.x_off = WS_HEADER;
  ip.part_off = ip.x_off + align_up((size_t)d->B * depth(d) * d->H * d->W * d->Cin * es, 256);
  ip.bytes = ip.part_off + ip.p2.ct_bytes;
  return ip;
}

static xconv_status validate_indep(const xconv_desc* d) {
  xconv_status s = validate(d);
  if (s != XCONV_OK) return s;
  if (d->r > 65535L * IS_JT || d->B > 65535L * IR_BT) return XCONV_ERR_UNSUPPORTED;     // grid z axes
  return XCONV_OK;
}

template <typename T>
static xconv_status run_sketch_indep(const xconv_desc* d, const void* X, const void* Z, float* S, cudaStream_t st) {
  const long N = (long)depth(d) * d->H * d->W;
  dim3 grid((unsigned)cdiv(d->B, IS_BT), (unsigned)cdiv(d->Cin, 32), (unsigned)cdiv(d->r, IS_JT));
  sketch_indep_simt<T><<<grid, 256, 0, st>>>(static_cast<const T*>(X), static_cast<const T*>(Z), S, d->r, d->B, N, d->Cin);
  return check_launch();
}

template <typename T>
static xconv_status run_rebuild_indep(const xconv_desc* d, const float* S, const void* Z, void* Xr, cudaStream_t st) {
  const long N = (long)depth(d) * d->H * d->W;
  dim3 grid((unsigned)cdiv(N, 8), (unsigned)cdiv(d->Cin, 32), (unsigned)cdiv(d->B, IR_BT));
  rebuild_indep_simt<T><<<grid, 256, 0, st>>>(S, static_cast<const T*>(Z), static_cast<T*>(Xr), d->r, d->B, N, d->Cin);
  return check_launch();
}

// Forms of the kernels (see xconv_variants_for), step by step as the plans and the launchers above choose them.
static int sketch_variants(const xconv_desc* d, const SketchPlan& p) {
  if (p.tc) return p.t.row_boxes ? XCONV_VARIANT_ROW_BOXES : 0;
  const int splits = p.stream ? p.s.splits : p.split ? (int)p.g.splits : p.splits;
  return (p.stream ? XCONV_VARIANT_STREAM : 0) | (wide_sums((long)d->r * d->B, splits) ? XCONV_VARIANT_WIDE_SUMS : 0);
}
static int backprobe_variants(const xconv_desc* d, const WgradPlan& p, bool redrawn) {
  const xconv_desc f = flat(d);
  if (p.split_bp) return 0;
  if (p.stream_bp) return XCONV_VARIANT_STREAM | (redrawn && tc_stream_draws_pairs(&f) ? XCONV_VARIANT_SIGN_PAIRS : 0);
  return p.tc_bp && tc_backprobe_row_boxes(&f, redrawn) ? XCONV_VARIANT_ROW_BOXES : 0;
}
static int contract_variants(const xconv_desc* d, const WgradPlan& p) {
  if (p.halo || p.split || p.tc_ct) return 0;
  return (small_contract_serves(d) ? XCONV_VARIANT_SMALL_TILES : 0) |
         (wide_sums((long)d->Cout * d->Cin * kdepth(d) * d->KH * d->KW, p.splits) ? XCONV_VARIANT_WIDE_SUMS : 0);
}
static int wgrad_variants(const xconv_desc* d, bool seeded) {
  SwappedWgrad sw;
  const WgradPlan p = plan_wgrad(d, &sw);
  if (sw.on) return backprobe_variants(&sw.d1, sw.p1, seeded && wgrad_redraws(d)) | contract_variants(&sw.d2, sw.p2);
  return backprobe_variants(d, p, false) | contract_variants(d, p);
}
static int conv_variants(const xconv_desc* d, bool dgrad) {
  xconv_desc e;
  TcConvPlan t;
  ConvSplitPlan f;
  if (plan_conv_f32(d, dgrad, &f)) return 0;
  if (plan_conv(d, dgrad, &e, &t)) return t.slide ? XCONV_VARIANT_WALK : 0;
  return d->dtype == XCONV_F32 && small_conv_serves(d) ? XCONV_VARIANT_SMALL_TILES : 0;
}

int launches() { return g_launches; }
void count_launch() { ++g_launches; }
void set_cuda_error(int e) { g_last_cuda_error = e; }

}  // namespace xconv

using namespace xconv;

extern "C" {

size_t xconv_workspace_bytes(const xconv_desc* desc, int op) {
  if (validate(desc) != XCONV_OK) return 0;
  switch (op) {
    case XCONV_OP_FORWARD: return std::max({plan_sketch(desc).bytes, conv_ws_bytes(desc, false), conv_ws_wish(desc, false)});
    case XCONV_OP_SKETCH: return plan_sketch(desc).bytes;
    case XCONV_OP_WGRAD_SEEDED: return plan_wgrad(desc).bytes + (wgrad_redraws(desc) ? 0 : probes_bytes(desc));
    case XCONV_OP_SKETCH_SEEDED: {
      const SketchPlan p = plan_sketch(desc, true);
      return p.bytes + (sketch_redraws(desc, p) ? 0 : probes_bytes(desc));
    }
    case XCONV_OP_SKETCH_SEEDED_GAUSSIAN: return plan_sketch(desc).bytes + probes_bytes(desc);
    case XCONV_OP_WGRAD_SEEDED_GAUSSIAN: return plan_wgrad(desc).bytes + probes_bytes(desc);
    case XCONV_OP_WGRAD:
    case XCONV_OP_BACKPROBE:
    case XCONV_OP_CONTRACT: return plan_wgrad(desc).bytes;
    case XCONV_OP_DGRAD: return conv_ws_wish(desc, true);
    case XCONV_OP_WGRAD_INDEPENDENT: return validate_indep(desc) == XCONV_OK ? plan_indep(desc).bytes : 0;
    default: return 0;
  }
}

int xconv_engine_for(const xconv_desc* desc, int op) {
  if (validate(desc) != XCONV_OK) return XCONV_ENGINE_NONE;
  const int tc = desc->dtype == XCONV_F16 ? XCONV_ENGINE_TCGEN05_F16 : XCONV_ENGINE_TCGEN05_BF16;
  const int f32 = XCONV_ENGINE_TCGEN05_F32;
  switch (op) {
    case XCONV_OP_SKETCH: {
      const SketchPlan p = plan_sketch(desc);
      return p.split ? f32 : p.stream || p.tc ? tc : XCONV_ENGINE_SIMT_F32;
    }
    case XCONV_OP_WGRAD:
    case XCONV_OP_CONTRACT: {
      const WgradPlan p = plan_wgrad(desc);
      return p.split ? f32 : p.halo || p.tc_ct ? tc : XCONV_ENGINE_SIMT_F32;
    }
    case XCONV_OP_BACKPROBE: {
      const WgradPlan p = plan_wgrad(desc);
      return p.split_bp && desc->dtype == XCONV_F32 ? f32 : p.split_bp || p.stream_bp || p.tc_bp ? tc : XCONV_ENGINE_SIMT_F32;
    }
    case XCONV_OP_FORWARD:
    case XCONV_OP_DGRAD: {
      TcConvPlan t;
      xconv_desc e;
      ConvSplitPlan f;
      if (plan_conv_f32(desc, op == XCONV_OP_DGRAD, &f)) return f32;
      return plan_conv(desc, op == XCONV_OP_DGRAD, &e, &t) ? tc : XCONV_ENGINE_SIMT_F32;
    }
    default: return XCONV_ENGINE_NONE;
  }
}

int xconv_variants_for(const xconv_desc* desc, int op) {
  if (validate(desc) != XCONV_OK) return 0;
  switch (op) {
    case XCONV_OP_FORWARD: return conv_variants(desc, false);
    case XCONV_OP_DGRAD: return conv_variants(desc, true);
    case XCONV_OP_SKETCH: {
      const xconv_desc f = flat(desc);
      return sketch_variants(&f, plan_sketch(desc));
    }
    case XCONV_OP_SKETCH_SEEDED: {
      const xconv_desc f = flat(desc);
      return sketch_variants(&f, plan_sketch(desc, true));
    }
    case XCONV_OP_BACKPROBE: return backprobe_variants(desc, plan_wgrad(desc), false);
    case XCONV_OP_CONTRACT: return contract_variants(desc, plan_wgrad(desc));
    case XCONV_OP_WGRAD: return wgrad_variants(desc, false);
    case XCONV_OP_WGRAD_SEEDED: return wgrad_variants(desc, true);
    default: return 0;
  }
}

xconv_status xconv_sketch(const xconv_desc* desc, const void* X, const void* Z, float* sketch, void* ws,
                          size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!X || !Z || !sketch) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(Z) || !aligned16(sketch)) return XCONV_ERR_ALIGNMENT;
  new_call();
  return run_sketch(desc, X, Z, sketch, ws, ws_bytes, static_cast<cudaStream_t>(cuda_stream));
}

xconv_status xconv_probes_from_seed(const xconv_desc* desc, unsigned long long seed, void* Z, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!Z) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(Z)) return XCONV_ERR_ALIGNMENT;
  new_call();
  return run_probes_from_seed(desc, seed, Z, static_cast<cudaStream_t>(cuda_stream));
}

xconv_status xconv_sketch_seeded(const xconv_desc* desc, const void* X, unsigned long long seed, float* sketch,
                                 void* ws, size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!X || !sketch) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(sketch)) return XCONV_ERR_ALIGNMENT;
  new_call();
  return run_sketch(desc, X, nullptr, sketch, ws, ws_bytes, static_cast<cudaStream_t>(cuda_stream), &seed);
}

xconv_status xconv_wgrad_seeded(const xconv_desc* desc, const float* sketch, const void* dY, unsigned long long seed,
                                float* dW, void* ws, size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!sketch || !dY || !dW) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(sketch) || !aligned16(dY) || !aligned16(dW)) return XCONV_ERR_ALIGNMENT;
  const size_t base = plan_wgrad(desc).bytes;
  const bool redraw = wgrad_redraws(desc);
  s = check_ws(ws, ws_bytes, base + (redraw ? 0 : probes_bytes(desc)));
  if (s != XCONV_OK) return s;
  new_call();
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // r > B on the tensor cores: the first kernel of the estimator redraws its tiles of Z on chip
  if (redraw) return run_wgrad(desc, sketch, dY, nullptr, dW, ws, base, st, &seed);
  // Algorithm 1 backward step 2: redraw Z from the seed (behind the regular scratch), then steps 3-4
  char* Z = static_cast<char*>(ws) + base;
  s = run_probes_from_seed(desc, seed, Z, st);
  if (s != XCONV_OK) return s;
  return run_wgrad(desc, sketch, dY, Z, dW, ws, base, st);
}

xconv_status xconv_gaussian_probes_from_seed(const xconv_desc* desc, unsigned long long seed, void* Z,
                                             void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!Z) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(Z)) return XCONV_ERR_ALIGNMENT;
  new_call();
  return run_gaussian_probes(desc, seed, Z, static_cast<cudaStream_t>(cuda_stream));
}

xconv_status xconv_block_sparse_probes_from_seed(const xconv_desc* desc, unsigned long long seed, int gaussian, double p,
                                                 void* Z, unsigned char* keep, float* chan_scale, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!Z || !keep || !chan_scale || !(p >= 0.0 && p <= 1.0) || (gaussian != 0 && gaussian != 1)) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(Z)) return XCONV_ERR_ALIGNMENT;
  new_call();
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  s = gaussian ? run_gaussian_probes(desc, seed, Z, st) : run_probes_from_seed(desc, seed, Z, st);
  if (s != XCONV_OK) return s;
  const long blocks = (long)desc->r * desc->Cin;
  const unsigned long long threshold = (unsigned long long)std::floor(p * 4294967296.0);
  block_keep_kernel<<<(unsigned)cdiv(cdiv(blocks, 4), 256), 256, 0, st>>>(keep, blocks, (uint32_t)(seed & 0xFFFFFFFFull),
                                                                          (uint32_t)(seed >> 32), threshold);
  if ((s = check_launch()) != XCONV_OK) return s;
  keep_scale_kernel<<<(unsigned)cdiv(desc->Cin, 256), 256, 0, st>>>(keep, desc->r, desc->Cin, chan_scale);
  if ((s = check_launch()) != XCONV_OK) return s;
  const long per_probe = (long)depth(desc) * desc->H * desc->W * desc->Cin, total = per_probe * desc->r;
  const unsigned grid = (unsigned)cdiv(cdiv(total, 4), 256);
  if (desc->dtype == XCONV_F32) drop_blocks_kernel<float><<<grid, 256, 0, st>>>(static_cast<float*>(Z), keep, total, per_probe, desc->Cin);
  else if (desc->dtype == XCONV_F16) drop_blocks_kernel<f16><<<grid, 256, 0, st>>>(static_cast<f16*>(Z), keep, total, per_probe, desc->Cin);
  else drop_blocks_kernel<bf16><<<grid, 256, 0, st>>>(static_cast<bf16*>(Z), keep, total, per_probe, desc->Cin);
  return check_launch();
}

xconv_status xconv_sketch_seeded_gaussian(const xconv_desc* desc, const void* X, unsigned long long seed,
                                          float* sketch, void* ws, size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!X || !sketch) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(sketch)) return XCONV_ERR_ALIGNMENT;
  const size_t base = plan_sketch(desc).bytes;
  s = check_ws(ws, ws_bytes, base + probes_bytes(desc));
  if (s != XCONV_OK) return s;
  new_call();
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  char* Z = static_cast<char*>(ws) + base;             // Z[seed] behind the regular scratch, then the regular kernels
  s = run_gaussian_probes(desc, seed, Z, st);
  if (s != XCONV_OK) return s;
  return run_sketch(desc, X, Z, sketch, ws, base, st);
}

xconv_status xconv_wgrad_seeded_gaussian(const xconv_desc* desc, const float* sketch, const void* dY,
                                         unsigned long long seed, float* dW, void* ws, size_t ws_bytes,
                                         void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!sketch || !dY || !dW) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(sketch) || !aligned16(dY) || !aligned16(dW)) return XCONV_ERR_ALIGNMENT;
  const size_t base = plan_wgrad(desc).bytes;
  s = check_ws(ws, ws_bytes, base + probes_bytes(desc));
  if (s != XCONV_OK) return s;
  new_call();
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  char* Z = static_cast<char*>(ws) + base;             // Algorithm 1 backward step 2, then steps 3-4
  s = run_gaussian_probes(desc, seed, Z, st);
  if (s != XCONV_OK) return s;
  return run_wgrad(desc, sketch, dY, Z, dW, ws, base, st);
}

xconv_status xconv_sketch_independent(const xconv_desc* desc, const void* X, const void* Z, float* sketch,
                                      void* cuda_stream) {
  xconv_status s = validate_indep(desc);
  if (s != XCONV_OK) return s;
  if (!X || !Z || !sketch) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(Z) || !aligned16(sketch)) return XCONV_ERR_ALIGNMENT;
  new_call();
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  return desc->dtype == XCONV_F32 ? run_sketch_indep<float>(desc, X, Z, sketch, st)
         : desc->dtype == XCONV_F16 ? run_sketch_indep<f16>(desc, X, Z, sketch, st)
                                    : run_sketch_indep<bf16>(desc, X, Z, sketch, st);
}

xconv_status xconv_wgrad_independent(const xconv_desc* desc, const float* sketch, const void* dY, const void* Z,
                                     float* dW, void* ws, size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate_indep(desc);
  if (s != XCONV_OK) return s;
  if (!sketch || !dY || !Z || !dW) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(sketch) || !aligned16(dY) || !aligned16(Z) || !aligned16(dW)) return XCONV_ERR_ALIGNMENT;
  const IndepPlan ip = plan_indep(desc);
  if ((s = validate(&ip.d2)) != XCONV_OK) return s;
  s = check_ws(ws, ws_bytes, ip.bytes);
  if (s != XCONV_OK) return s;
  new_call();
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  char* w = static_cast<char*>(ws);
  s = desc->dtype == XCONV_F32 ? run_rebuild_indep<float>(desc, sketch, Z, w + ip.x_off, st)
      : desc->dtype == XCONV_F16 ? run_rebuild_indep<f16>(desc, sketch, Z, w + ip.x_off, st)
                                 : run_rebuild_indep<bf16>(desc, sketch, Z, w + ip.x_off, st);
  if (s != XCONV_OK) return s;
  return run_contract(&ip.d2, ip.p2, dY, w + ip.x_off, dW, 1.0f / (float)desc->r, w + ip.part_off, w, st);
}

xconv_status xconv_forward(const xconv_desc* desc, const void* X, const void* W, const void* Z, void* Y,
                           float* sketch, void* ws, size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!X || !W || !Z || !Y || !sketch) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(W) || !aligned16(Z) || !aligned16(Y) || !aligned16(sketch))
    return XCONV_ERR_ALIGNMENT;
  if (!ws || ws_bytes < std::max(plan_sketch(desc).bytes, conv_ws_bytes(desc, false))) return XCONV_ERR_WORKSPACE;
  if (!aligned16(ws)) return XCONV_ERR_ALIGNMENT;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  new_call();
  bool held;
  s = run_conv(desc, false, X, W, Y, static_cast<char*>(ws), ws_bytes, st, &held);
  if (s != XCONV_OK) return s;
  return run_sketch(desc, X, Z, sketch, ws, ws_bytes, st, nullptr, held);
}

xconv_status xconv_wgrad(const xconv_desc* desc, const float* sketch, const void* dY, const void* Z, float* dW,
                         void* ws, size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!sketch || !dY || !Z || !dW) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(sketch) || !aligned16(dY) || !aligned16(Z) || !aligned16(dW)) return XCONV_ERR_ALIGNMENT;
  if (desc->chan_scale && (reinterpret_cast<uintptr_t>(desc->chan_scale) & 3u)) return XCONV_ERR_ALIGNMENT;
  new_call();
  return run_wgrad(desc, sketch, dY, Z, dW, ws, ws_bytes, static_cast<cudaStream_t>(cuda_stream));
}

size_t xconv_backprobe_bytes(const xconv_desc* desc) {
  if (validate(desc) != XCONV_OK) return 0;
  return (size_t)desc->r * depth(desc) * desc->H * desc->W * desc->Cout * (desc->dtype == XCONV_F32 ? 4 : 2);
}

xconv_status xconv_backprobe(const xconv_desc* desc, const float* sketch, const void* dY, void* L, void* ws,
                             size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!sketch || !dY || !L) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(sketch) || !aligned16(dY) || !aligned16(L)) return XCONV_ERR_ALIGNMENT;
  const WgradPlan p = plan_wgrad(desc);
  s = check_ws(ws, ws_bytes, p.bytes);
  if (s != XCONV_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  new_call();
  return run_backprobe(desc, p, sketch, dY, L, static_cast<char*>(ws) + p.sb_off, static_cast<char*>(ws), st);
}

xconv_status xconv_contract(const xconv_desc* desc, const void* L, const void* Z, float* dW, void* ws,
                            size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!L || !Z || !dW) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(L) || !aligned16(Z) || !aligned16(dW)) return XCONV_ERR_ALIGNMENT;
  if (desc->chan_scale && (reinterpret_cast<uintptr_t>(desc->chan_scale) & 3u)) return XCONV_ERR_ALIGNMENT;
  const WgradPlan p = plan_wgrad(desc);
  s = check_ws(ws, ws_bytes, p.bytes);
  if (s != XCONV_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  new_call();
  return run_contract(desc, p, L, Z, dW, 1.0f / (float)desc->r, static_cast<char*>(ws) + p.part_off,
                      static_cast<char*>(ws), st);
}

xconv_status xconv_dgrad(const xconv_desc* desc, const void* dY, const void* W, void* dX, void* ws,
                         size_t ws_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!dY || !W || !dX) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(dY) || !aligned16(W) || !aligned16(dX)) return XCONV_ERR_ALIGNMENT;
  if (!ws || ws_bytes < WS_HEADER) return XCONV_ERR_WORKSPACE;
  if (!aligned16(ws)) return XCONV_ERR_ALIGNMENT;
  new_call();
  return run_conv(desc, true, dY, W, dX, static_cast<char*>(ws), ws_bytes, static_cast<cudaStream_t>(cuda_stream));
}

// Arena layout of the host-buffer entry point: X | dY | Z | S | dW | workspace, each 256-aligned.
struct HostArena { size_t x, dy, z, s, dw, ws, ws_bytes, total, xb, dyb, zb, sb, dwb; };
static HostArena host_arena(const xconv_desc* d) {
  HostArena a{};
  const size_t es = d->dtype == XCONV_F32 ? 4 : 2;
  const size_t px = (size_t)depth(d) * d->H * d->W;
  a.xb = (size_t)d->B * px * d->Cin * es;
  a.dyb = (size_t)d->B * px * d->Cout * es;
  a.zb = (size_t)d->r * px * d->Cin * es;
  a.sb = (size_t)d->r * d->B * 4;
  a.dwb = (size_t)d->Cout * kdepth(d) * d->KH * d->KW * d->Cin * 4;
  a.x = 0;
  a.dy = a.x + align_up(a.xb, 256);
  a.z = a.dy + align_up(a.dyb, 256);
  a.s = a.z + align_up(a.zb, 256);
  a.dw = a.s + align_up(a.sb, 256);
  a.ws = a.dw + align_up(a.dwb, 256);
  a.ws_bytes = std::max(plan_sketch(d).bytes, plan_wgrad(d).bytes);
  a.total = a.ws + a.ws_bytes;
  return a;
}

size_t xconv_host_arena_bytes(const xconv_desc* desc) {
  if (validate(desc) != XCONV_OK) return 0;
  return host_arena(desc).total;
}

xconv_status xconv_sketch_wgrad_host(const xconv_desc* desc, const void* hX, const void* hdY, const void* hZ,
                                     float* hS, float* hdW, void* arena, size_t arena_bytes, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!hX || !hdY || !hZ || !hS || !hdW || !arena) return XCONV_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(arena) & 255u) return XCONV_ERR_ALIGNMENT;
  const HostArena a = host_arena(desc);
  if (arena_bytes < a.total) return XCONV_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  char* base = static_cast<char*>(arena);
  cudaError_t e;
  if ((e = cudaMemcpyAsync(base + a.x, hX, a.xb, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(base + a.z, hZ, a.zb, cudaMemcpyHostToDevice, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(base + a.dy, hdY, a.dyb, cudaMemcpyHostToDevice, st)) != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return XCONV_ERR_CUDA;
  }
  new_call();
  float* S = reinterpret_cast<float*>(base + a.s);
  float* dW = reinterpret_cast<float*>(base + a.dw);
  s = run_sketch(desc, base + a.x, base + a.z, S, base + a.ws, a.ws_bytes, st);
  if (s != XCONV_OK) return s;
  s = run_wgrad(desc, S, base + a.dy, base + a.z, dW, base + a.ws, a.ws_bytes, st);
  if (s != XCONV_OK) return s;
  if ((e = cudaMemcpyAsync(hS, S, a.sb, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(hdW, dW, a.dwb, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(st)) != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return XCONV_ERR_CUDA;
  }
  return XCONV_OK;
}

xconv_status xconv_selftest_wait_limit(void* ws, size_t ws_bytes, unsigned int limit_ms, void* cuda_stream) {
  if (!ws || ws_bytes < WS_HEADER) return XCONV_ERR_WORKSPACE;
  if (!aligned16(ws)) return XCONV_ERR_ALIGNMENT;
  if (limit_ms == 0 || limit_ms > 2000) return XCONV_ERR_INVALID_ARG;
  new_call();
  return tc_run_wait_selftest(static_cast<char*>(ws), (unsigned long long)limit_ms * 1000000ull,
                              static_cast<cudaStream_t>(cuda_stream));
}

xconv_status xconv_workspace_status(const void* ws, void* cuda_stream) {
  if (!ws) return XCONV_ERR_INVALID_ARG;
  unsigned int word[2] = {0, 0};
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaMemcpyAsync(word, ws, sizeof(word), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return (word[0] != WS_OK && word[0] == word[1]) ? XCONV_ERR_TIMEOUT : XCONV_OK;
}

int xconv_zero_blocks_used(const xconv_desc* desc) {
  if (validate(desc) != XCONV_OK || desc->zero_blocks == nullptr) return 0;
  const WgradPlan p = plan_wgrad(desc);
  return (p.tc_ct && p.t.ct_masked) ? 1 : 0;
}

xconv_status xconv_zero_blocks(const xconv_desc* desc, const void* Z, unsigned char* mask, void* cuda_stream) {
  xconv_status s = validate(desc);
  if (s != XCONV_OK) return s;
  if (!Z || !mask) return XCONV_ERR_INVALID_ARG;
  if (!aligned16(Z)) return XCONV_ERR_ALIGNMENT;
  if (desc->Cin % 64 != 0 || (long)desc->r * (desc->Cin / 64) > 2000000000L) return XCONV_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const long pixels = (long)depth(desc) * desc->H * desc->W;
  const unsigned blocks = (unsigned)((long)desc->r * (desc->Cin / 64));
  new_call();
  if (desc->dtype == XCONV_F32) zero_blocks_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(Z), mask, pixels, desc->Cin);
  else zero_blocks_kernel<unsigned short><<<blocks, 256, 0, st>>>(static_cast<const unsigned short*>(Z), mask, pixels, desc->Cin);
  ++g_launches;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

xconv_status xconv_measure_fma_rate(void* scratch, size_t scratch_bytes, double* tflops, void* cuda_stream) {
  const int blocks = 148 * 16, threads = 256, iters = 4096;
  if (!scratch || !tflops) return XCONV_ERR_INVALID_ARG;
  if (scratch_bytes < (size_t)blocks * threads * sizeof(float)) return XCONV_ERR_WORKSPACE;
  if (!aligned16(scratch)) return XCONV_ERR_ALIGNMENT;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  float best_ms = 0.f;
  new_call();
  for (int rep = 0; rep < 6 && e == cudaSuccess; ++rep) {      // the first repetition warms up
    cudaEventRecord(e0, st);
    fma_rate_kernel<<<blocks, threads, 0, st>>>(static_cast<float*>(scratch), iters, 0.999f, 0.001f);
    ++g_launches;
    cudaEventRecord(e1, st);
    e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (rep > 0 && (best_ms == 0.f || ms < best_ms)) best_ms = ms;
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (e != cudaSuccess || best_ms <= 0.f) { g_last_cuda_error = (int)e; return XCONV_ERR_CUDA; }
  *tflops = 2.0 * 16.0 * iters * (double)blocks * threads / (best_ms * 1e-3) / 1e12;
  return XCONV_OK;
}

int xconv_last_launch_count(void) { return g_launches; }
int xconv_last_cuda_error(void) { return g_last_cuda_error; }

const char* xconv_status_string(xconv_status s) {
  switch (s) {
    case XCONV_OK: return "ok";
    case XCONV_ERR_INVALID_ARG: return "invalid argument";
    case XCONV_ERR_UNSUPPORTED: return "unsupported layer or option (no kernel; there is no fallback)";
    case XCONV_ERR_ALIGNMENT: return "pointer not 16-byte aligned";
    case XCONV_ERR_WORKSPACE: return "workspace missing or too small";
    case XCONV_ERR_CUDA: return "CUDA call failed";
    case XCONV_ERR_TIMEOUT: return "a bounded device-side wait ran out";
    default: return "unknown status";
  }
}

}  // extern "C"
