// The exact convolution Y = conv(X, w) and the exact input gradient dX of float layers on the tensor cores (sm_100a): every
// float as three bfloat16 parts, a product as six (split_f32.cuh).
//
// Patches, offsets and the walk are those of conv_tc.cu: an MMA row tile is a patch of pw x ph pixels, its input lies in shared
// memory once with its halo, and the A tile of an offset is the same memory read from dy * P + dx rows further on.  Here the
// copy engine brings the floats of the patch and twelve warps write their parts as three tiles (one block of 32 or 16 channels of one
// plane per stage; an offset in depth is a stage of its own), so the input crosses the memory system once, as floats.
// The weights are split once per call into tile images in the workspace -- [column tile][block][depth offset][offset], each
// the 3n rows (h of n channels out, m, l) as they lie in shared memory -- which plain bulk copies bring in.
//
// Three MMAs per k-step of 16 channels form the six products, in three groups of n accumulator columns:
//   h x [h | m | l] -> columns 0..3n,   m x [h | m] -> columns n..3n,   l x h -> columns 2n..3n.
// The A tile is then read three times instead of six (what bounds narrow MMAs), and the products hh have a column group of their
// own (which also decides results that are not finite: split_f32.cuh).  Two accumulator sets take rows of offsets in turn (1 x 1: four blocks
// of channels), an issuing warp each; eight epilogue warps add the three groups of a set to float registers.
//
// Error against 64 bits on 120 random layers, times that of the FP32 multiply-adds (conv_fma.cu): 0.35 in the median, nowhere more
// than 1; 1e-7 where those have 1e-6.  What bounds it: the MMAs, 204 clocks per k-step and 64 channels out (an MMA of N columns holds the
// tensor pipe N / 2 clocks, or shared memory 32 + N / 4).  The tensor pipe is active 0.54 of the time on 64 -> 64 channels, 128 images of 32 x 32 from a
// cold cache (0.64 of the warm call): the rest are the issuing warps' waits for weights (336 MB from L2 there) and for the conversion.
// us, multiply-adds -> this: 64 -> 64 channels, 128 images of 32 x 32 236 -> 57 (the MMAs alone 36); 96 -> 160, 39 x 39 286 -> 53; 5 x 5,
// 64 -> 128 617 -> 130; 1 x 1, 48 -> 128, 4 images of 168 x 190 138 -> 48.
#include "conv_split.h"

#include <algorithm>

#include "conv_walk.cuh"
#include "split_f32.cuh"

namespace xconv {

constexpr int CS_A_SLOTS = 4, CS_W_SLOTS = 5;      // (weights: of each issuer's ring)

struct ConvSplitParams {
  const float* wt;
  const uint8_t* wimg;
  int Co, Cw, dgrad;                               // channels out and in of the weights
  int KD, T, pad, pad_d;
  int P, pw, ph, patches_x, patches_y, depth;
  uint32_t patches, items;
  int npos, nb, cw, ks_full, ks_last, chain;       // positions of the box; channel blocks; k-steps of a block and of the last; rows of offsets per chain
  int n;                                           // channels out per column tile
  uint32_t a_plane, a_slot; int a_slots;
  uint32_t w_tile, w_slot; int w_slots;
  uint32_t f_off, f_slot, f_bytes; int f_slots;    // the floats
  uint32_t w_off, o_off, o_bytes;
  int ocw;
  uint32_t hi, lo0, idesc;
  int tmem_cols;
  unsigned int *status, tag;
};

__device__ __forceinline__ void cs_epi_sync() { asm volatile("barrier.cta.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ bool cs_epi_all(bool ok) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 1, 256, p;\n\t"
               "selp.b32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"(ok ? 1u : 0u) : "memory");
  return r != 0;
}
// The weight of the sum: Y reads w(co, ci, t), dX w(ci, co, T-1-t).
__device__ __forceinline__ float cs_weight(const ConvSplitParams& p, int co, int ci, int t) {
  return p.dgrad ? p.wt[((size_t)ci * p.T + (p.T - 1 - t)) * p.Co + co] : p.wt[((size_t)co * p.T + t) * p.Cw + ci];
}

// The weights' tile images, a thread per four channels in of one row.  T here counts the offsets of all depths.
__global__ void __launch_bounds__(256) conv_split_weights(const ConvSplitParams p, uint8_t* __restrict__ img, int tiles_n) {
  pdl_wait();
  pdl_trigger();
  const int quads = p.cw >> 2, T2 = p.T / p.KD;
  const uint32_t total = (uint32_t)(tiles_n * p.nb * p.T) * (uint32_t)(p.n * quads);
  for (uint32_t i = blockIdx.x * 256 + threadIdx.x; i < total; i += gridDim.x * 256) {
    const int q = (int)(i % (uint32_t)quads);
    uint32_t r = i / (uint32_t)quads;
    const int row = (int)(r % (uint32_t)p.n);
    const uint32_t tile = r / (uint32_t)p.n;
    r = tile;
    const int t2 = (int)(r % (uint32_t)T2); r /= (uint32_t)T2;
    const int dz = (int)(r % (uint32_t)p.KD); r /= (uint32_t)p.KD;
    const int blk = (int)(r % (uint32_t)p.nb), tn = (int)(r / (uint32_t)p.nb);
    const int co = tn * p.n + row, c = blk * p.cw + 4 * q, t = dz * T2 + t2;
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = co < p.Co && c + k < p.Cw ? cs_weight(p, co, c + k, t) : 0.f;
    const Split4 s = split4_apart<Bf16Parts>(make_float4(v[0], v[1], v[2], v[3]));
    uint8_t* base = img + (size_t)tile * p.w_tile;
    const auto at = [&](int plane) {
      const uint32_t rr = (uint32_t)(plane * p.n + row);
      return base + swizzled(p.cw == 32 ? 6 : 5, rr, 8 * q);
    };
    *reinterpret_cast<uint2*>(at(0)) = s.h;
    *reinterpret_cast<uint2*>(at(1)) = s.m;
    *reinterpret_cast<uint2*>(at(2)) = s.l;
  }
}

// The MMAs of one offset.
template <int KSTEPS>
__device__ __forceinline__ void cs_offset(const ConvSplitParams& p, uint32_t d, uint32_t a, uint32_t b, uint32_t acc) {
  const uint32_t plane16 = p.a_plane >> 4, n = (uint32_t)p.n, narrower = (n >> 3) << 17;
#pragma unroll
  for (int k = 0; k < KSTEPS; ++k) {
    umma_warp(d, a + 2 * k, p.hi, b + 2 * k, p.hi, p.idesc, acc);
    umma_warp(d + n, a + plane16 + 2 * k, p.hi, b + 2 * k, p.hi, p.idesc - narrower, 1u);
    umma_warp(d + 2 * n, a + 2 * plane16 + 2 * k, p.hi, b + 2 * k, p.hi, p.idesc - 2 * narrower, 1u);
    acc = 1u;
  }
}

template <int KS, int RB>
__global__ void __launch_bounds__(SP_THREADS, 1) conv_split_kernel(const __grid_constant__ CUtensorMap map_in, const __grid_constant__ CUtensorMap map_out,
                                                                 const __grid_constant__ ConvSplitParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t a_full[CS_A_SLOTS], a_empty[CS_A_SLOTS], w_full[2][CS_W_SLOTS], w_empty[2][CS_W_SLOTS], t_full[2], t_empty[2];
  __shared__ __align__(8) uint64_t f_full[SP_FLOATS], f_empty[SP_FLOATS];
  __shared__ uint32_t tmem_slot;
  __shared__ int go;
  constexpr int T2 = KS * KS;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  if (threadIdx.x == 0) {
    for (int s = 0; s < CS_A_SLOTS; ++s) { mbar_init(&a_full[s], SP_CONVERTERS / 32); mbar_init(&a_empty[s], 2); }
    for (int s = 0; s < 2 * CS_W_SLOTS; ++s) { mbar_init(&w_full[0][s], 1); mbar_init(&w_empty[0][s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&t_full[b], 1); mbar_init(&t_empty[b], 8); }
    for (int f = 0; f < SP_FLOATS; ++f) { mbar_init(&f_full[f], 1); mbar_init(&f_empty[f], SP_CONVERTERS / 32); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    prefetch_tmap(&map_in);
    prefetch_tmap(&map_out);
  }
  const uint32_t tmem_base = split_begin(warp, &tmem_slot, (uint32_t)p.tmem_cols, 0u, 0u, p.status, p.tag, &go);
  const uint32_t i0 = (uint32_t)((unsigned long long)p.items * blockIdx.x / gridDim.x);
  const uint32_t i1 = (uint32_t)((unsigned long long)p.items * (blockIdx.x + 1) / gridDim.x);
  const int stages = p.nb * p.KD;                   // of a unit: blocks of channels, one depth offset after the other

  if (!go) {
    // fall through to the teardown
  } else if (warp == 0) {
    // ------------------------------------------------------------------ weights
    if (lane == 0) {
      uint32_t s[2] = {0, 0}, par[2] = {1, 1}, cnt[2] = {0, 0}, ring = 0;      // (a wait for the phase before the first returns at once)
      bool ok = true;
      const uint32_t per_tn = (uint32_t)(stages * T2);
      for (uint32_t it = i0; it < i1 && ok; ++it) {
        const uint32_t tn = it / p.patches;
        int left = p.chain;
        for (int dz = 0; dz < p.KD && ok; ++dz)
          for (int blk = 0; blk < p.nb && ok; ++blk) {
            const uint8_t* src = p.wimg + (size_t)(tn * per_tn + (uint32_t)((blk * p.KD + dz) * T2)) * p.w_tile;
            for (int t = 0; t < T2; ++t) {
              const uint32_t at = ring ? s[1] : s[0];
              ok = mbar_wait(&w_empty[ring][at], ring ? par[1] : par[0], p.status, p.tag);
              if (!ok) break;
              mbar_arrive_expect_tx(&w_full[ring][at], p.w_tile);
              bulk_load(base + p.w_off + (ring * (uint32_t)p.w_slots + at) * p.w_slot, src + (size_t)t * p.w_tile, p.w_tile, &w_full[ring][at]);
              const bool wrap = at + 1 == (uint32_t)p.w_slots;
              if (ring) { ++cnt[1]; s[1] = wrap ? 0 : at + 1; par[1] ^= wrap ? 1u : 0u; }
              else { ++cnt[0]; s[0] = wrap ? 0 : at + 1; par[0] ^= wrap ? 1u : 0u; }
              if (t % KS == KS - 1 && --left == 0) { left = p.chain; ring ^= 1u; }
            }
          }
        if (left != p.chain) ring ^= 1u;             // (the unit's last chain)
      }
      // every copy issued must have landed before the CTA exits
      for (int r = 0; r < 2; ++r)
        for (uint32_t n = r ? cnt[1] : cnt[0], i = n > (uint32_t)p.w_slots ? n - p.w_slots : 0; i < n; ++i)
          if (!mbar_wait(&w_full[r][i % p.w_slots], (i / p.w_slots) & 1u, p.status, p.tag)) break;
    }
  } else if (warp <= 2) {
    // ------------------------------------------------------------------ MMA issuers (whole warps): every other chain each
    const uint32_t own = (uint32_t)warp - 1;
    const uint32_t a0 = p.lo0 | ((base & 0x3FFFFu) >> 4);
    const uint32_t w0 = p.lo0 | (((base + p.w_off + own * (uint32_t)p.w_slots * p.w_slot) & 0x3FFFFu) >> 4);
    const uint32_t a_slot16 = p.a_slot >> 4, w_slot16 = p.w_slot >> 4, row16 = (uint32_t)p.P * (RB >> 4);
    const uint32_t d = tmem_base + own * (uint32_t)(3 * p.n);
    uint64_t *full = w_full[own], *empty = w_empty[own];
    uint32_t s = 0, a_par = 0, a_at = a0, ws = 0, w_par = 0, w_at = w0, chain = 0, t_par = 1;
    bool ok = true;
    for (uint32_t it = i0; it < i1 && ok; ++it) {
      int rows = 0, blk = 0;                         // rows of offsets in the chain so far
      for (int st = 0; st < stages && ok; ++st) {
        ok = mbar_wait_warp(&a_full[s], a_par, p.status, p.tag);
        if (!ok) break;
        tc_fence_after();
        const int ks = blk == p.nb - 1 ? p.ks_last : p.ks_full;
        if (++blk == p.nb) blk = 0;
        uint32_t a = a_at;
#pragma unroll 1
        for (int dy = 0; dy < KS; ++dy, a += row16) {
          const bool last = rows + 1 == p.chain || (st == stages - 1 && dy == KS - 1);
          if (chain == own) {
            if (rows == 0) {
              ok = mbar_wait_warp(&t_empty[own], t_par, p.status, p.tag);
              if (!ok) break;
            }
            bool ready = mbar_wait_warp(&full[ws], w_par, p.status, p.tag);
#pragma unroll
            for (int dx = 0; dx < KS; ++dx) {
              if (dx > 0 && !ready) ready = mbar_wait_warp(&full[ws], w_par, p.status, p.tag);
              ok = ok && ready;
              tc_fence_after();
              const bool wrap = ws + 1 == (uint32_t)p.w_slots;
              const uint32_t here = ws, w_here = w_at;
              ws = wrap ? 0u : ws + 1;
              w_par ^= wrap ? 1u : 0u;
              w_at = wrap ? w0 : w_at + w_slot16;
              // the next weights are asked for before this offset's MMAs: the answer's way is behind them
              if (dx + 1 < KS) ready = mbar_try_wait(&full[ws], w_par);
              const uint32_t acc = rows > 0 || dx > 0 ? 1u : 0u;
              if (RB == 64 && ks == 2) cs_offset<2>(p, d, a + (uint32_t)dx * (RB >> 4), w_here, acc);
              else cs_offset<1>(p, d, a + (uint32_t)dx * (RB >> 4), w_here, acc);
              umma_commit_warp(&empty[here]);
              if (dx + 1 < KS) ready = __all_sync(0xffffffffu, ready);
            }
            if (!ok) break;
            if (last) { umma_commit_warp(&t_full[own]); t_par ^= 1u; }
          }
          rows = last ? 0 : rows + 1;
          chain ^= last ? 1u : 0u;
        }
        if (!ok) break;
        umma_commit_warp(&a_empty[s]);
        a_at += a_slot16;
        if (++s == (uint32_t)p.a_slots) { s = 0; a_par ^= 1u; a_at = a0; }
      }
    }
  } else if (warp == SP_LOAD) {
    // ------------------------------------------------------------------ copies of the floats
    if (lane == 0) {
      uint32_t f = 0, par = 1, cnt = 0;
      bool ok = true;
      for (CvWalk w(p, i0, i1); w.it < i1 && ok; w.step(p))
        for (int dz = 0; dz < p.KD && ok; ++dz)
          for (int blk = 0; blk < p.nb; ++blk) {
            ok = mbar_wait(&f_empty[f], par, p.status, p.tag);
            if (!ok) break;
            mbar_arrive_expect_tx(&f_full[f], p.f_bytes);
            tma_load_5d(base + p.f_off + f * p.f_slot, &map_in, blk * p.cw, w.x - p.pad, w.y - p.pad, w.z + dz - p.pad_d, w.b, &f_full[f]);
            ++cnt;
            if (++f == (uint32_t)p.f_slots) { f = 0; par ^= 1u; }
          }
      for (uint32_t i = cnt > (uint32_t)p.f_slots ? cnt - p.f_slots : 0; i < cnt; ++i)
        if (!mbar_wait(&f_full[i % p.f_slots], (i / p.f_slots) & 1u, p.status, p.tag)) break;
    }
  } else if (warp >= SP_EPILOGUE && warp < SP_CONVERT) {
    // ------------------------------------------------------------------ epilogue: chains to registers, registers to the result
    const int quad = warp & 3, half = (warp - SP_EPILOGUE) >> 2, groups = p.n >> 4;
    const int m = quad * 32 + lane, my = m / p.P, mx = m - my * p.P;      // this thread's position in the box
    const bool live = mx < p.pw && my < p.ph;
    const uint32_t v = (uint32_t)(my * p.pw + mx), orb = (uint32_t)p.ocw * 4;
    const uint32_t swz = p.ocw == 32 ? v & 7u : (v >> 1) & 3u;
    const uint32_t tmem_q = tmem_base + ((uint32_t)(quad * 32) << 16);
    const int chains = (stages * KS + p.chain - 1) / p.chain;
    const bool leader = warp == SP_EPILOGUE && lane == 0;
    uint32_t buf = 0, par = 0;
    bool ok = true;
    for (CvWalk w(p, i0, i1); w.it < i1; w.step(p)) {
      float2 sum[2][8];                              // channel groups half, half + 2 of 16
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int e = 0; e < 8; ++e) sum[k][e] = make_float2(0.f, 0.f);
      for (int c = 0; c < chains && ok; ++c) {
        ok = split_wait(&t_full[buf], par, p.status, p.tag);
        if (!ok) break;
        tc_fence_after();
        split_add_set<Bf16Parts>(tmem_q + buf * (uint32_t)(3 * p.n), (uint32_t)p.n, half, sum, &t_empty[buf]);
        par ^= buf;
        buf ^= 1u;
      }
      if (leader) bulk_wait_read<0>();               // the last stores have read the staging tile
      if (!cs_epi_all(ok)) break;                    // the warps leave together
      const int n0 = (int)w.tn * p.n;
      if (live) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int g = half + 2 * k;
          if (g >= groups) break;
          const uint32_t row = base + p.o_off + (uint32_t)(p.ocw == 32 ? g >> 1 : g) * p.o_bytes + v * orb;
          const uint32_t piece = p.ocw == 32 ? (uint32_t)(g & 1) * 4 : 0u;
#pragma unroll
          for (int e = 0; e < 16; e += 4)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row + (((piece + (e >> 2)) ^ swz) << 4)),
                         "f"(sum[k][e / 2].x), "f"(sum[k][e / 2].y), "f"(sum[k][e / 2 + 1].x), "f"(sum[k][e / 2 + 1].y) : "memory");
        }
      }
      fence_async_smem();
      cs_epi_sync();
      if (leader) {
        for (int c = 0; c < p.n && n0 + c < p.Co; c += p.ocw)
          tma_store_5d(&map_out, base + p.o_off + (uint32_t)(c / p.ocw) * p.o_bytes, n0 + c, w.x, w.y, w.z, w.b);
        bulk_commit();
      }
    }
    if (leader) bulk_wait_all();
  } else if (warp >= SP_CONVERT) {
    // ------------------------------------------------------------------ conversion
    const uint32_t total = (i1 - i0) * (uint32_t)stages;
    uint32_t s = 0, par = 1, f = 0, f_par = 0;
    for (uint32_t j = 0; j < total; ++j) {
      if (!split_wait(&a_empty[s], par, p.status, p.tag) || !split_wait(&f_full[f], f_par, p.status, p.tag)) break;
      const SplitBox box{base + p.f_off + f * p.f_slot, p.npos, base + s * p.a_slot, p.a_plane, 0u, 0u, 0u};
      float2 check = make_float2(0.f, 0.f);
      split_box<RB == 64 ? 6 : 5, RB == 64 ? 3 : 2, false>(box, check);
      split_stage_done(&a_full[s], &f_empty[f], check, [&] { split_box_again<RB == 64 ? 6 : 5, RB == 64 ? 3 : 2, false>(box); });
      if (++s == (uint32_t)p.a_slots) { s = 0; par ^= 1u; }
      if (++f == (uint32_t)p.f_slots) { f = 0; f_par ^= 1u; }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// [rows][C] floats to [rows][C4], C4 the next multiple of 4, with zeros: the copy engine steps through rows of 16 bytes.
__global__ void __launch_bounds__(256) pad_floats_kernel(const float* in, float4* __restrict__ out, long pieces, int C, int per_row) {
  pdl_trigger();
  pdl_wait();
  const long i = (long)blockIdx.x * 256 + threadIdx.x;
  if (i >= pieces) return;
  const long row = i / per_row;
  const int c = (int)(i - row * per_row) * 4;
  float v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = c + k < C ? in[row * C + c + k] : 0.f;
  out[i] = make_float4(v[0], v[1], v[2], v[3]);
}

// ------------------------------------------------------------------------------------ host side

size_t padded_float_bytes(long rows, int C) { return C % 4 ? ((size_t)rows * round_up(C, 4) * 4 + 255) / 256 * 256 : 0; }
xconv_status pad_floats(const float*& t, float* copy, long rows, int C, cudaStream_t st) {
  if (C % 4 == 0) return XCONV_OK;
  const long pieces = rows * (round_up(C, 4) / 4);
  const cudaError_t e = launch_pdl(pad_floats_kernel, dim3((unsigned)cdivl(pieces, 256)), dim3(256), 0, st, t, reinterpret_cast<float4*>(copy),
                                   pieces, C, round_up(C, 4) / 4);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  t = copy;
  return XCONV_OK;
}

bool plan_conv_split(const xconv_desc* d, bool dgrad, ConvSplitPlan* p) {
  if (d->dtype != XCONV_F32 || d->circular) return false;
  const int Ci = dgrad ? d->Cout : d->Cin, Co = dgrad ? d->Cin : d->Cout;
  if (Co % 4 != 0) return false;                     // rows of the result on 16-byte boundaries
  const ConvGeo g = conv_geo(d);
  if (g.W >= (1L << 30) || g.B >= (1L << 31) || g.W * g.H >= (1L << 31)) return false;
  const int K = d->KH, KD = d->KD > 1 ? d->KD : 1, T2 = K * K;
  p->cw = Ci > 16 ? 32 : 16;
  p->nb = (int)cdivl(Ci, p->cw);
  p->ks_last = (int)cdivl(Ci - (p->nb - 1) * p->cw, 16);
  p->tiles_n = (int)cdivl(Co, SP_MAX_N);
  p->n = round_up((int)cdivl(Co, p->tiles_n), 16);
  p->ocw = p->n % 32 == 0 ? 32 : 16;
  if ((long)p->tiles_n * p->nb * KD * T2 * p->n * (p->cw / 4) >= 1L << 31) return false;      // (conv_split_weights counts pieces in 32 bits)
  const uint32_t rb = 2 * (uint32_t)p->cw;
  p->w_tile = 3 * (uint32_t)p->n * rb;
  const uint32_t w_slot = up1k(p->w_tile), budget = SMEM_LIMIT - 4096;
  const long ksteps = (long)KD * T2 * ((p->nb - 1) * (p->cw / 16) + p->ks_last);
  long best = -1;
  for (long nx = cdivl(g.W, 128); nx <= std::max(cdivl(g.W, 128), std::min(32L, g.W)); ++nx) {
    const int pw = (int)cdivl(g.W, nx), P = pw + K - 1;
    const int ph_max = (int)std::min<long>(g.H, (128 - pw) / P + 1), ph = (int)cdivl(g.H, cdivl(g.H, ph_max));
    const int npos = P * (ph + K - 1);
    const uint32_t need = (uint32_t)std::max(npos, (K - 1) * P + (K - 1) + TILE_M);
    const uint32_t a_plane = up1k(need * rb), a_slot = 3 * a_plane;
    const uint32_t o_all = up1k((uint32_t)(pw * ph) * 4 * p->ocw) * (uint32_t)(p->n / p->ocw), f_slot = up1k((uint32_t)npos * 4 * p->cw);
    if (P > 256 || 2 * a_slot + 4 * w_slot + o_all + 2 * f_slot > budget) continue;
    const long patches = cdivl(g.W, pw) * cdivl(g.H, ph) * g.D * g.B, items = patches * p->tiles_n;
    if (items >= (1L << 32) - 1) continue;
    // conversion: some 45 instructions for four values, on four schedulers at two thirds of their rate
    const long convert = (long)npos * KD * p->nb * p->cw / 4 * 45 / 85;
    const long cost = cdivl(items, NUM_SMS) * std::max(ksteps * split_kstep_clocks(p->n), convert);
    if (best >= 0 && cost >= best) continue;
    best = cost;
    p->pw = pw; p->ph = ph; p->patches = patches;
    p->a_plane = a_plane;
    // two of everything, two more weight tiles, a third box of floats, weights up to a chain and a half, a third patch
    uint32_t room = budget - o_all - 2 * f_slot - 2 * a_slot;
    p->w_slots = room >= 6 * w_slot ? 3 : 2;
    room -= 2 * (uint32_t)p->w_slots * w_slot;
    p->f_slots = 2;
    while (p->f_slots < SP_FLOATS && room >= f_slot) { ++p->f_slots; room -= f_slot; }
    while (p->w_slots < CS_W_SLOTS && room >= 2 * w_slot) { ++p->w_slots; room -= 2 * w_slot; }
    p->a_slots = (int)std::min<uint32_t>(CS_A_SLOTS, 2 + room / a_slot);
    p->f_slot = f_slot;
  }
  if (best < 0) return false;
  p->img_bytes = ((size_t)p->tiles_n * p->nb * KD * T2 * p->w_tile + 255) / 256 * 256;
  p->bytes = p->img_bytes + padded_float_bytes(g.W * g.H * g.D * g.B, Ci);
  return true;
}

xconv_status run_conv_split(const xconv_desc* d, const ConvSplitPlan& pl, bool dgrad, const float* in, const float* Wt, float* out,
                            char* ws_head, char* scratch, cudaStream_t st) {
  const int K = d->KH, KD = d->KD > 1 ? d->KD : 1;
  const int Ci = dgrad ? d->Cout : d->Cin, Co = dgrad ? d->Cin : d->Cout;
  const ConvGeo g = conv_geo(d);
  if (xconv_status s = pad_floats(in, reinterpret_cast<float*>(scratch + pl.img_bytes), g.W * g.H * g.D * g.B, Ci, st)) return s;
  ConvSplitParams p{};
  p.wt = Wt;
  p.wimg = reinterpret_cast<const uint8_t*>(scratch);
  p.Cw = Ci; p.Co = Co; p.dgrad = dgrad ? 1 : 0;
  p.KD = KD; p.T = KD * K * K; p.pad = (K - 1) / 2; p.pad_d = (KD - 1) / 2;
  p.pw = pl.pw; p.ph = pl.ph; p.P = pl.pw + K - 1;
  p.patches_x = (int)cdivl(g.W, p.pw); p.patches_y = (int)cdivl(g.H, p.ph); p.depth = (int)g.D;
  p.patches = (uint32_t)pl.patches; p.items = (uint32_t)(pl.patches * pl.tiles_n);
  p.npos = p.P * (p.ph + K - 1);
  p.nb = pl.nb; p.cw = pl.cw; p.ks_full = pl.cw / 16; p.ks_last = pl.ks_last; p.chain = K > 1 ? 1 : 4;
  p.n = pl.n; p.ocw = pl.ocw;
  p.a_plane = pl.a_plane; p.a_slot = 3 * pl.a_plane; p.a_slots = pl.a_slots;
  p.w_tile = pl.w_tile; p.w_slot = up1k(pl.w_tile); p.w_slots = pl.w_slots;
  p.w_off = (uint32_t)p.a_slots * p.a_slot;
  p.o_off = p.w_off + 2 * (uint32_t)p.w_slots * p.w_slot;
  p.o_bytes = up1k((uint32_t)(p.pw * p.ph) * 4 * (uint32_t)p.ocw);
  p.f_off = p.o_off + p.o_bytes * (uint32_t)(p.n / p.ocw);
  p.f_slot = pl.f_slot; p.f_slots = pl.f_slots; p.f_bytes = (uint32_t)p.npos * 4 * (uint32_t)p.cw;
  const uint32_t rb = 2 * (uint32_t)p.cw;
  p.hi = ((8 * rb) >> 4) | (1u << 14) | ((p.cw == 32 ? 4u : 6u) << 29);
  p.lo0 = 1u << 16;
  p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(3 * p.n >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24);
  p.tmem_cols = pow2_cols(6 * p.n);
  p.status = reinterpret_cast<unsigned int*>(ws_head);
  p.tag = call_tag();

  const uint32_t pieces = (uint32_t)(pl.tiles_n * p.nb * p.T) * (uint32_t)(p.n * (p.cw / 4));
  const unsigned wblocks = (unsigned)std::min<long>(2 * NUM_SMS, cdivl(pieces, 256));
  CUtensorMap mi, mo;
  auto image_map = [&](CUtensorMap* m, const float* ptr, int C, int cb, int bw, int bh, CUtensorMapSwizzle swizzle) {
    const uint64_t row = (uint64_t)C * 4;
    const uint64_t dims[5] = {(uint64_t)C, (uint64_t)g.W, (uint64_t)g.H, (uint64_t)g.D, (uint64_t)g.B};
    const uint64_t str[4] = {row, row * g.W, row * g.W * g.H, row * g.W * g.H * g.D};
    const uint32_t box[5] = {(uint32_t)cb, (uint32_t)bw, (uint32_t)bh, 1, 1};
    return make_map_f32(m, ptr, 5, dims, str, box, swizzle);
  };
  if (!image_map(&mi, in, round_up(Ci, 4), p.cw, p.P, p.ph + K - 1, CU_TENSOR_MAP_SWIZZLE_NONE) ||
      !image_map(&mo, out, Co, p.ocw, p.pw, p.ph, p.ocw == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B))
    return XCONV_ERR_CUDA;
  const size_t smem = 1024 + (size_t)p.f_off + (size_t)p.f_slots * p.f_slot;
  if (smem > (size_t)(SMEM_LIMIT - 1024)) return XCONV_ERR_UNSUPPORTED;
  cudaError_t e = launch_pdl(conv_split_weights, dim3(wblocks), dim3(256), 0, st, p, reinterpret_cast<uint8_t*>(scratch), pl.tiles_n);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  void (*kernel)(CUtensorMap, CUtensorMap, ConvSplitParams) =
      p.cw == 32 ? (K == 3 ? conv_split_kernel<3, 64> : K == 5 ? conv_split_kernel<5, 64> : conv_split_kernel<1, 64>)
                 : (K == 3 ? conv_split_kernel<3, 32> : K == 5 ? conv_split_kernel<5, 32> : conv_split_kernel<1, 32>);
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT - 1024);
  const unsigned grid = std::min<uint32_t>(p.items, NUM_SMS);
  if (e == cudaSuccess) e = launch_pdl(kernel, dim3(grid), dim3(SP_THREADS), smem_of_grid(smem, grid), st, mi, mo, p);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

}  // namespace xconv
