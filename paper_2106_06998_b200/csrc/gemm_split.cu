// Sketch S = Z^T X and back-probe L = S dY^T with float operands on the tensor cores (sm_100a): every float as three bfloat16 parts, a
// product as six (split_f32.cuh).
//
// Both read one or two large float matrices once: the copy engine brings boxes of 32 terms of the reduction, twelve warps in three
// teams split them and write the parts as MMA tiles.  The columns' parts lie one under another, so that three MMAs per k-step of 16 form the six products
// in three groups of n accumulator columns, as in conv_split.cu; two accumulator sets take chains of four k-steps (two stages) in
// turn and eight epilogue warps add them in float registers.
// Error against 64 bits, times that of the FP32 multiply-adds: 0.47 in the median, nowhere more than 1.  us, multiply-adds -> this: sketch of
// 128 x 64 rows, 65536 terms 39 -> 20 (memory 8: the stages' chain of copy, split and MMA is some 2000 clocks, and a CTA has 14), back-probe
// of 64 rows, 128 terms, 65536 positions 37 -> 23 (memory 8).  Long sketches run at 3 to 4 TB/s: the conversion.
//   sketch      rows = the larger of probes and samples (tiles of 128), columns = the other (up to 64); both K-major; the k-blocks are dealt
//               to the splits in turn, so that the CTAs read neighbouring bytes of every row at a time
//   back-probe  rows = 128 positions of the flat (pixel, channel) axis, MN-major, columns = up to 64 rows of S, whose parts a small
//               kernel writes as tile images; a CTA walks its tiles, a warp stores 128 bytes of a row of L at a time
//   back-probe of 16-bit layers (those the kernels of tc_kernels.cu and stream_tc.cu do not serve; they were on multiply-adds, and S is
//               not to be rounded): Y's tiles are copied as they are, two boxes of 64 positions, S goes in three parts (float16: its rows
//               scaled first), one MMA a k-step.  us, multiply-adds -> this: 256 rows, 461 terms, 68208 positions 916 -> 91, 167 rows, 31 terms,
//               591872 positions 353 -> 101 (memory 36), 512 rows, 4 terms, 295840 positions 180 -> 126 (memory 47).  Bound by S's
//               images from L2 (20 KB a stage, 750 clocks) where the reduction is long, by the epilogue's chain of waits, loads and
//               conversions (1850 clocks a tile) where it is short.
#include "gemm_split.h"

#include <algorithm>

#include "split_f32.cuh"

namespace xconv {

constexpr int GS_STAGES = 8, GS_TERMS = 32, GS_TEAMS = 3;
constexpr uint32_t GS_OUT = 2048;                  // a staging tile of 16-bit results: 32 columns of 32 positions
enum : int { GS_SKETCH = 0, GS_BACK = 1, GS_BACK_BF16 = 2, GS_BACK_F16 = 3 };
template <int KIND> struct GsElement { using type = float; using parts = Bf16Parts; };
template <> struct GsElement<GS_BACK_BF16> { using type = bf16; using parts = Bf16Parts; };
template <> struct GsElement<GS_BACK_F16> { using type = f16; using parts = F16Parts; };

struct GemmSplitParams {
  const float* B; const void* Y;                   // back-probe: S, and Y [K][M]
  const uint8_t* img; const float* scale;
  void* out;
  long M, K, N;
  long s_row, s_k;                                 // back-probe: S(j, k) = B[j * s_row + k * s_k]
  long o_m, o_n;                                   // out[m * o_m + n * o_n]
  long kblocks, tiles_m, splits;
  int n, tiles_n, stages, ks_last;
  uint32_t a_plane, b_plane, a_bytes, b_bytes, stage_bytes;
  uint32_t f_off, f_slot, f_b, f_bytes; int f_slots;      // the floats of a stage: the rows' box, the columns' f_b bytes behind it
  int f_rows_a, f_rows_b;
  uint32_t a_hi, a_lo0, a_step, idesc;
  int tmem_cols;
  unsigned int *status, tag;
};

// The tile images of S for the back-probe: [column tile][k-block][3n rows of 32 terms], four terms at a time.
template <int KIND>
__device__ __forceinline__ void write_image(const GemmSplitParams& p, uint8_t* img, long j, long kb, int q, float scale) {
  const long tn = j / p.n, k = kb * GS_TERMS + 4 * q;
  const int row = (int)(j - tn * p.n);
  float v[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) v[e] = j < p.N && k + e < p.K ? p.B[j * p.s_row + (k + e) * p.s_k] * scale : 0.f;
  const Split4 s = split4_apart<typename GsElement<KIND>::parts>(make_float4(v[0], v[1], v[2], v[3]));
  uint8_t* base = img + (tn * p.kblocks + kb) * (long)p.b_bytes;
  *reinterpret_cast<uint2*>(base + swizzled(6, (uint32_t)row, 8 * q)) = s.h;
  *reinterpret_cast<uint2*>(base + swizzled(6, (uint32_t)(p.n + row), 8 * q)) = s.m;
  *reinterpret_cast<uint2*>(base + swizzled(6, (uint32_t)(2 * p.n + row), 8 * q)) = s.l;
}

__global__ void __launch_bounds__(256) split_sketch_images(const GemmSplitParams p, uint8_t* __restrict__ img) {
  pdl_wait();
  pdl_trigger();
  const long total = (long)p.tiles_n * p.n * p.kblocks * 8;
  for (long i = (long)blockIdx.x * 256 + threadIdx.x; i < total; i += (long)gridDim.x * 256) {
    const long j = i / (p.kblocks * 8), k = i - j * (p.kblocks * 8);
    write_image<GS_BACK>(p, img, j, k >> 3, (int)(k & 7), 1.0f);
  }
}

// float16 parts.  A row of S is scaled by the power of two that brings its largest finite value to 2^14 (infinities and NaN stay what they are).
// Its parts then hold it down to 2^-61 of that value, all 24 bits of entries above 2^-36 of it.  A row with smaller entries than that (they
// count where the large ones meet zeros of Y) is marked by the sign of its scale: its sums are taken by multiply-adds.  A warp per row.
__global__ void __launch_bounds__(256) split_sketch_images_f16(const GemmSplitParams p, uint8_t* __restrict__ img, float* __restrict__ scale) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  for (long j = (long)blockIdx.x * 8 + (threadIdx.x >> 5); j < (long)p.tiles_n * p.n; j += (long)gridDim.x * 8) {
    float top = 0.f, low = INFINITY;
    if (j < p.N)
      for (long k = lane; k < p.K; k += 32) {
        const float v = fabsf(p.B[j * p.s_row + k * p.s_k]);
        if (v - v == 0.f) top = fmaxf(top, v);
        if (v > 0.f) low = fminf(low, v);
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
      low = fminf(low, __shfl_xor_sync(0xffffffffu, low, o));
    }
    const int e = top > 0.f ? max(-100, (int)(__float_as_uint(top) >> 23) - 127 - 14) : 0;
    if (lane == 0) scale[j] = copysignf(__uint_as_float((uint32_t)(127 + e) << 23), low - top * 1.4551915228366852e-11f);      // 2^-36
    const float down = __uint_as_float((uint32_t)(127 - e) << 23);
    for (long i = lane; i < p.kblocks * 8; i += 32) write_image<GS_BACK_F16>(p, img, j, i >> 3, (int)(i & 7), down);
  }
}

// The results of marked columns (a bit per column of an epilogue warp's staging tile) at 32 positions, by multiply-adds: Q columns, U terms under
// way at a time.  us, 256 rows, 461 terms, 68208 positions: no row marked 97, one 440, all 8000.  (No more registers than the kernel has: with
// 150 a thread the next one no longer fits beside it, 12.6 -> 14.4 us for 70 rows, 131 terms.)
template <int Q, int U>
__device__ __noinline__ unsigned gs_wide_columns(const GemmSplitParams& p, uint32_t stage, unsigned wide, long n0, long m, int lane) {
  const f16* Y = static_cast<const f16*>(p.Y) + min(m, p.M - 1);
  int c[Q];
  const float* S[Q];
  float acc[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    c[q] = __ffs(wide) - 1;
    wide &= wide - 1;
    S[q] = p.B + (n0 + c[q] + (c[q] & 16)) * p.s_row;
    acc[q] = 0.f;
  }
#pragma unroll 1
  for (long k = 0; k < p.K; k += U) {
    f16 y[U];
    float s[U][Q];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const long at = min(k + i, p.K - 1);
      y[i] = Y[at * p.M];
#pragma unroll
      for (int q = 0; q < Q; ++q) s[i][q] = S[q][at * p.s_k];
    }
#pragma unroll
    for (int i = 0; i < U; ++i)
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (k + i < p.K) acc[q] = fmaf(s[i][q], to_f(y[i]), acc[q]);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) st_shared_16(stage + (uint32_t)(c[q] * 64 + lane * 2), from_f<f16>(acc[q]));
  return wide;
}

template <int KIND>
__global__ void __launch_bounds__(KIND >= GS_BACK_BF16 ? SP_CONVERT * 32 : SP_THREADS, 1)
gemm_split_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ GemmSplitParams p) {
  using T = typename GsElement<KIND>::type;
  constexpr int TEAMS = GS_TEAMS;
  constexpr bool BACK = KIND != GS_SKETCH, WHOLE = KIND >= GS_BACK_BF16;      // WHOLE: Y's tiles are copied as they are
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[GS_STAGES], empty[GS_STAGES], acc_full[2], acc_empty[2];
  __shared__ __align__(8) uint64_t f_full[SP_FLOATS], f_empty[SP_FLOATS];
  __shared__ uint32_t tmem_slot;
  __shared__ int go;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  if (threadIdx.x == 0) {
    for (int s = 0; s < GS_STAGES; ++s) { mbar_init(&full[s], WHOLE ? 2 : SP_CONVERTERS / 32 / TEAMS + (BACK ? 1 : 0)); mbar_init(&empty[s], 2); }
    for (int f = 0; f < SP_FLOATS; ++f) { mbar_init(&f_full[f], 1); mbar_init(&f_empty[f], SP_CONVERTERS / 32 / TEAMS); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    prefetch_tmap(&map_a);
    if (!BACK) prefetch_tmap(&map_b);
  }
  // (the sketch: rows that no conversion writes are multiplied all the same)
  const uint32_t tmem_base = split_begin(warp, &tmem_slot, (uint32_t)p.tmem_cols, base, BACK ? 0u : (uint32_t)p.stages * p.stage_bytes, p.status, p.tag, &go);
  // this CTA's units -- back-probe: a run of tiles; sketch: one -- and the k-blocks of a unit
  const long tiles = p.tiles_m * p.tiles_n;
  const long t0 = BACK ? tiles * blockIdx.x / gridDim.x : (long)blockIdx.x / p.splits;
  const long t1 = BACK ? tiles * (blockIdx.x + 1) / gridDim.x : t0 + 1;
  const long kb0 = BACK ? 0 : blockIdx.x - t0 * p.splits, kstep = BACK ? 1 : p.splits;
  const uint32_t per_unit = (uint32_t)((p.kblocks - kb0 + kstep - 1) / kstep), total = (uint32_t)(t1 - t0) * per_unit;

  if (!go) {
    // fall through to the teardown
  } else if (warp == 0) {
    // ------------------------------------------------------------------ S's tile images (back-probe)
    if (BACK && lane == 0) {
      uint32_t s = 0, par = 1, i = 0, kb = 0;        // (a wait for the phase before the first returns at once)
      long tn = t0 / p.tiles_m, m = t0 - tn * p.tiles_m;      // (counted along: a division of longs for every stage held the copies up)
      const uint8_t* tile = p.img + tn * p.kblocks * (long)p.b_bytes;
      const uint8_t* src = tile;
      for (; i < total; ++i) {
        if (!mbar_wait(&empty[s], par, p.status, p.tag)) break;
        mbar_arrive_expect_tx(&full[s], p.b_bytes);
        bulk_load(base + s * p.stage_bytes + p.a_bytes, src, p.b_bytes, &full[s]);
        src += p.b_bytes;
        if (++kb == per_unit) {
          kb = 0;
          if (++m == p.tiles_m) { m = 0; tile = src; }
          src = tile;
        }
        if (++s == (uint32_t)p.stages) { s = 0; par ^= 1u; }
      }
      // every copy issued must have landed before the CTA exits
      for (uint32_t k = i > (uint32_t)p.stages ? i - p.stages : 0; k < i; ++k)
        if (!mbar_wait(&full[k % p.stages], (k / p.stages) & 1u, p.status, p.tag)) break;
    }
  } else if (warp <= 2) {
    // ------------------------------------------------------------------ MMA issuers (whole warps): every other chain each
    const uint32_t own = (uint32_t)warp - 1;
    const uint32_t s0 = (base & 0x3FFFFu) >> 4, stage16 = p.stage_bytes >> 4, ap = p.a_plane >> 4, n = (uint32_t)p.n;
    const uint32_t narrower = (n >> 3) << 17, b_add = (1u << 16) + (p.a_bytes >> 4);
    const uint32_t a_hi = p.a_hi, b_hi = (512u >> 4) | (1u << 14) | (4u << 29), d = tmem_base + own * 3 * n;
    uint32_t s = 0, par = 0, t_par = 1, chain = 0, kb = 0, acc = 0, left = 0;
    for (uint32_t i = 0; i < total; ++i) {
      if (left == 0) {                               // a chain: two stages, or the unit's last one
        left = min(2u, per_unit - kb);
        acc = 0;
        if (chain == own && !mbar_wait_warp(&acc_empty[own], t_par, p.status, p.tag)) break;
      }
      if (!mbar_wait_warp(&full[s], par, p.status, p.tag)) break;
      if (chain == own) {
        tc_fence_after();
        const bool two = kb0 + (long)kb * kstep != p.kblocks - 1 || p.ks_last == 2;
        const uint32_t a = s0 + s * stage16 + p.a_lo0, b = s0 + s * stage16 + b_add;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (k == 1 && !two) break;
          const uint32_t ak = a + (k ? p.a_step : 0u);
          umma_warp(d, ak, a_hi, b + 2 * k, b_hi, p.idesc, acc);
          if (!WHOLE) umma_warp(d + n, ak + ap, a_hi, b + 2 * k, b_hi, p.idesc - narrower, 1u);
          if (!WHOLE) umma_warp(d + 2 * n, ak + 2 * ap, a_hi, b + 2 * k, b_hi, p.idesc - 2 * narrower, 1u);
          acc = 1u;
        }
        umma_commit_warp(&empty[s]);
      } else if (lane == 0) {
        mbar_arrive(&empty[s]);
      }
      if (--left == 0) {
        if (chain == own) { umma_commit_warp(&acc_full[own]); t_par ^= 1u; }
        chain ^= 1u;
      }
      if (++kb == per_unit) kb = 0;
      if (++s == (uint32_t)p.stages) { s = 0; par ^= 1u; }
    }
  } else if (WHOLE && warp == SP_LOAD) {
    // ------------------------------------------------------------------ copies of Y's tiles, as they are
    if (lane == 0) {
      long m = (t0 % p.tiles_m) * TILE_M;
      uint32_t s = 0, par = 1, kb = 0, i = 0;
      for (; i < total; ++i) {
        if (!mbar_wait(&empty[s], par, p.status, p.tag)) break;
        const uint32_t dst = base + s * p.stage_bytes;
        mbar_arrive_expect_tx(&full[s], p.a_bytes);
        tma_load_2d(dst, &map_a, (int)m, (int)(kb * GS_TERMS), &full[s]);
        tma_load_2d(dst + (p.a_bytes >> 1), &map_a, (int)m + 64, (int)(kb * GS_TERMS), &full[s]);
        if (++kb == per_unit) {
          kb = 0;
          if ((m += TILE_M) >= p.M) m = 0;
        }
        if (++s == (uint32_t)p.stages) { s = 0; par ^= 1u; }
      }
      // every copy issued must have landed before the CTA exits
      for (uint32_t k = i > (uint32_t)p.stages ? i - p.stages : 0; k < i; ++k)
        if (!mbar_wait(&full[k % p.stages], (k / p.stages) & 1u, p.status, p.tag)) break;
    }
  } else if (warp == SP_LOAD) {
    // ------------------------------------------------------------------ copies of the floats
    if (lane == 0) {
      const long tn0 = t0 / p.tiles_m;
      long m = (t0 - tn0 * p.tiles_m) * TILE_M;
      uint32_t f = 0, par = 1, kb = 0, i = 0;
      for (; i < total; ++i) {
        if (!mbar_wait(&f_empty[f], par, p.status, p.tag)) break;
        const uint32_t dst = base + p.f_off + f * p.f_slot;
        const int k = (int)((kb0 + (long)kb * kstep) * GS_TERMS);
        mbar_arrive_expect_tx(&f_full[f], p.f_bytes);
        if (BACK) {
          tma_load_2d(dst, &map_a, (int)m, k, &f_full[f]);
        } else {
          tma_load_2d(dst, &map_a, k, (int)m, &f_full[f]);
          tma_load_2d(dst + p.f_b, &map_b, k, (int)(tn0 * p.n), &f_full[f]);
        }
        if (++kb == per_unit) {
          kb = 0;
          if ((m += TILE_M) >= p.M) m = 0;
        }
        if (++f == (uint32_t)p.f_slots) { f = 0; par ^= 1u; }
      }
      // every copy issued must have landed before the CTA exits
      for (uint32_t k = i > (uint32_t)p.f_slots ? i - p.f_slots : 0; k < i; ++k)
        if (!mbar_wait(&f_full[k % p.f_slots], (k / p.f_slots) & 1u, p.status, p.tag)) break;
    }
  } else if (warp >= SP_EPILOGUE && warp < SP_CONVERT) {
    // ------------------------------------------------------------------ epilogue
    const int quad = warp & 3, half = (warp - SP_EPILOGUE) >> 2, groups = p.n >> 4;      // column groups half, half + 2 of 16
    const uint32_t tmem_q = tmem_base + ((uint32_t)(quad * 32) << 16);
    uint32_t buf = 0, par = 0;
    const uint32_t stage = base + p.f_off + (uint32_t)(warp - SP_EPILOGUE) * GS_OUT;      // (WHOLE)
    bool ok = true;
    long tn_at = t0 / p.tiles_m, m_at = (t0 - tn_at * p.tiles_m) * TILE_M;       // (WHOLE: counted along; the others have no registers for it)
    for (long t = t0; t < t1 && ok; ++t) {
      const long tn = WHOLE ? tn_at : t / p.tiles_m, m = (WHOLE ? m_at : (t - tn * p.tiles_m) * TILE_M) + quad * 32 + lane;
      if ((m_at += TILE_M) >= p.M) { m_at = 0; ++tn_at; }
      float scale = 0.f;                             // (float16) of column half * 16 + lane + (lane & 16), given to the others when it is needed
      // (an ordinary load: the kernel before this one, which this one may start beside, writes the scales)
      if (KIND == GS_BACK_F16 && half * 16 + lane + (lane & 16) < p.n)
        scale = *const_cast<const volatile float*>(p.scale + tn * p.n + half * 16 + lane + (lane & 16));
      float2 sum[2][8];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int e = 0; e < 8; ++e) sum[k][e] = make_float2(0.f, 0.f);
      for (uint32_t i = 0; i < per_unit; i += 2) {
        ok = split_wait(&acc_full[buf], par, p.status, p.tag);
        if (!ok) break;
        tc_fence_after();
        split_add_set<typename GsElement<KIND>::parts, WHOLE>(tmem_q + buf * (uint32_t)(3 * p.n), (uint32_t)p.n, half, sum, &acc_empty[buf]);
        par ^= buf;
        buf ^= 1u;
      }
      if (!ok) break;
      if (WHOLE) {
        // Results of 16 bits go through shared memory, so that a lane stores 16 bytes of a row (2 bytes a lane and store: 4900 clocks a tile;
        // boxes of 16 rows of 64 bytes by the copy engine: 2080).
        __syncwarp();                                // the last tile is read
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (half + 2 * k >= groups) break;
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            float v = split_sum(sum, k, e);
            if (KIND == GS_BACK_F16) v *= __shfl_sync(0xffffffffu, fabsf(scale), k * 16 + e);
            st_shared_16(stage + (uint32_t)((k * 16 + e) * 64 + lane * 2), from_f<T>(v));
          }
        }
        if (KIND == GS_BACK_F16) {
          unsigned wide = __ballot_sync(0xffffffffu, scale < 0.f);
          while (wide) wide = __popc(wide) >= 4 ? gs_wide_columns<4, 4>(p, stage, wide, tn * p.n + half * 16, m, lane)
                                                : gs_wide_columns<1, 8>(p, stage, wide, tn * p.n + half * 16, m, lane);
        }
        __syncwarp();
        const long at = m - lane + (lane & 3) * 8;   // (rows have a multiple of 8 positions)
        T* to = static_cast<T*>(p.out) + at;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = i * 8 + (lane >> 2), c = half * 16 + row + (row & 16);
          const long n = tn * p.n + c;
          if (c < p.n && n < p.N && at < p.M) *reinterpret_cast<uint4*>(to + n * p.M) = ld_shared_v4(stage + (uint32_t)(row * 64 + (lane & 3) * 16));
        }
        continue;
      }
      if (m >= p.M) continue;
      T* out = static_cast<T*>(p.out) + (BACK ? 0 : kb0 * p.M * p.N) + m * p.o_m;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (half + 2 * k >= groups) break;
        const long n0 = tn * p.n + (half + 2 * k) * 16;
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (n0 + e < p.N) out[(n0 + e) * p.o_n] = from_f<T>(split_sum(sum, k, e));
      }
    }
  } else if (!WHOLE && warp >= SP_CONVERT) {
    // ------------------------------------------------------------------ conversion
    // In three teams of four warps that take the stages in turn: with all twelve on each a stage took 1500 to 1800 clocks whatever its rows (two waits,
    // the way through shared memory, the proxy's fence, the arrivals), and nothing hid them.  us, one team -> two -> three:
    // sketch of 64 x 16 rows, 2^21 terms 355 -> 225 -> 226, 64 x 64, 131072 terms 36.1 -> 29.6 -> 27.8, 300 x 100, 51200 terms 76.5 -> 60.8 -> 58.3.
    // A ring has as many stages as there are teams, so that a stage's barriers see one team: the parity of a lap tells it from the lap before only.
    // (Float boxes, three or four, change teams: that the stage `f_slots` before is converted is known from `empty`, which says that the MMAs have
    // gone through all stages up to three before.)
    constexpr int THREADS = SP_CONVERTERS / TEAMS;
    const uint32_t team = (uint32_t)(warp - SP_CONVERT) / (THREADS / 32);
    SplitTurn turn(team, (uint32_t)p.stages), f_turn(team, (uint32_t)p.f_slots);
    for (uint32_t i = team; i < total; i += TEAMS) {
      const uint32_t s = turn.at, f = f_turn.at;
      if (!split_wait(&empty[s], turn.lap ^ 1u, p.status, p.tag) || !split_wait(&f_full[f], f_turn.lap, p.status, p.tag)) break;
      const uint32_t from = base + p.f_off + f * p.f_slot, to = base + s * p.stage_bytes;
      float2 check = make_float2(0.f, 0.f);
      if (BACK) {
        const SplitBox box{from, GS_TERMS, to, p.a_plane, p.a_plane >> 1, 0u, 0u};
        split_box<7, 5, false, THREADS>(box, check);
        split_stage_done(&full[s], &f_empty[f], check, [&] { split_box_again<7, 5, false, THREADS>(box); });
      } else {
        const SplitBox rows{from, p.f_rows_a, to, p.a_plane, 0u, 0u, 0u}, cols{from + p.f_b, p.f_rows_b, to + p.a_bytes, p.b_plane, 0u, 0u, 0u};
        split_box<6, 3, false, THREADS>(rows, check);
        split_box<6, 3, false, THREADS>(cols, check);
        split_stage_done(&full[s], &f_empty[f], check, [&] { split_box_again<6, 3, false, THREADS>(rows); split_box_again<6, 3, false, THREADS>(cols); });
      }
      turn.next(TEAMS); f_turn.next(TEAMS);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// ------------------------------------------------------------------------------------ host side

static void plan_columns(long M, long N, int kind, GemmSplitPlan* p) {
  const bool back = kind != GS_SKETCH, whole = kind >= GS_BACK_BF16;
  p->tiles_n = (int)cdivl(N, SP_MAX_N);
  p->n = round_up((int)cdivl(N, p->tiles_n), 16);
  p->f_rows_a = back ? GS_TERMS : (int)std::min<long>(TILE_M, (M + 7) / 8 * 8);
  p->f_rows_b = back ? 0 : (int)std::min<long>(p->n, (N + 7) / 8 * 8);
  const int f_slot = whole ? (int)GS_OUT * 4 : back ? GS_TERMS * 512 : (int)up1k((uint32_t)p->f_rows_a * 128) + (int)up1k((uint32_t)p->f_rows_b * 128);
  const int stage = (whole ? 1 : 3) * 8192 + (int)up1k(3u * 64 * (uint32_t)p->n), room = SMEM_LIMIT - 4096 - 2 * stage - 2 * f_slot;
  if (whole) {
    p->f_slots = 2;                                  // (the results' staging tiles)
    p->stages = 2 + std::min(GS_STAGES - 2, room / stage);
  } else {                                           // (every n has room for that: 3 x 36 KB and 3 x 24 KB)
    p->stages = GS_TEAMS;
    p->f_slots = 2 + std::min(SP_FLOATS - 2, (room - (GS_TEAMS - 2) * stage) / f_slot);
  }
}
static const double HBM_SM = 22.0;                  // bytes per clock and SM from memory

bool plan_sketch_split(const xconv_desc* d, GemmSplitPlan* p) {
  const long K = (long)(d->D > 1 ? d->D : 1) * d->H * d->W * d->Cin;
  if (d->dtype != XCONV_F32 || K % 4 != 0 || K >= (1L << 31) - 64) return false;      // (rows on 16-byte boundaries)
  p->swap = d->B > d->r ? 1 : 0;
  const long M = std::max(d->B, d->r), N = std::min(d->B, d->r);
  plan_columns(M, N, GS_SKETCH, p);
  p->tiles_m = cdivl(M, TILE_M);
  p->kblocks = cdivl(K, GS_TERMS);
  const long tiles = p->tiles_m * p->tiles_n;
  if (tiles > (1L << 20)) return false;
  p->splits = std::max(1L, std::min(p->kblocks, NUM_SMS / tiles));
  const long rows = p->f_rows_a + p->f_rows_b;
  const double clk = std::max({2.0 * split_kstep_clocks(p->n), rows * 8 * 45.0 / 85, rows * 128 / HBM_SM});
  p->clocks = (long)((double)cdivl(p->kblocks, p->splits) * clk * cdivl(tiles * p->splits, NUM_SMS));
  p->bytes = (size_t)p->splits * d->r * d->B * sizeof(float);
  return true;
}

static int back_kind(const xconv_desc* d) {
  return d->dtype == XCONV_F32 ? GS_BACK : d->dtype == XCONV_F16 ? GS_BACK_F16 : GS_BACK_BF16;
}

bool plan_backprobe_split(const xconv_desc* d, GemmSplitPlan* p) {
  const long Q = (long)(d->D > 1 ? d->D : 1) * d->H * d->W * d->Cout;
  const int kind = back_kind(d);
  p->swap = 0;
  plan_columns(0, d->r, kind, p);
  p->tiles_m = cdivl(Q, TILE_M);
  p->kblocks = cdivl(d->B, GS_TERMS);
  p->splits = 1;
  if (Q % (kind == GS_BACK ? 4 : 8) != 0 || Q >= (1L << 31) - 128) return false;      // (rows on 16-byte boundaries)
  // (float16: a tile whose rows of S are all marked takes its sums by multiply-adds in the epilogue, some 1500 clocks a term, and the other warps
  // wait for a second at most)
  if (kind == GS_BACK_F16 && d->B > 1 << 18) return false;
  const long tiles = p->tiles_m * p->tiles_n, ksteps = cdivl(d->B, 16);
  // (whole rows: measured, 1850 clocks a tile of one k-block, 3000 of three, 10800 of fifteen)
  const double clk = kind == GS_BACK ? std::max({(double)ksteps * split_kstep_clocks(p->n), ksteps * 16 * 32 * 45.0 / 85,
                                                 (d->B + std::min(d->r, p->n)) * 512 / HBM_SM}) + 200.0
                                     : std::max(p->kblocks * 750.0 + 500.0, 1900.0);
  p->clocks = (long)((double)cdivl(tiles, NUM_SMS) * clk);
  p->bytes = (size_t)p->tiles_n * p->kblocks * 3 * p->n * 64 + (kind == GS_BACK_F16 ? (size_t)p->tiles_n * p->n * sizeof(float) : 0);
  return true;
}

static void fill_common(const GemmSplitPlan& pl, int kind, char* ws_head, GemmSplitParams* p) {
  p->kblocks = pl.kblocks; p->tiles_m = pl.tiles_m; p->splits = pl.splits;
  p->n = pl.n; p->tiles_n = pl.tiles_n; p->stages = pl.stages;
  p->ks_last = (int)cdivl(p->K - (pl.kblocks - 1) * GS_TERMS, 16);
  p->a_plane = 8192; p->b_plane = 64 * (uint32_t)pl.n;
  p->a_bytes = (kind >= GS_BACK_BF16 ? 1 : 3) * p->a_plane; p->b_bytes = 3 * p->b_plane;
  p->stage_bytes = p->a_bytes + up1k(p->b_bytes);
  p->f_off = (uint32_t)pl.stages * p->stage_bytes;
  p->f_rows_a = pl.f_rows_a; p->f_rows_b = pl.f_rows_b; p->f_slots = pl.f_slots;
  p->a_hi = (512u >> 4) | (1u << 14) | (4u << 29);
  p->idesc = (1u << 4) | (kind == GS_BACK_F16 ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)(3 * pl.n >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24);
  p->tmem_cols = pow2_cols(6 * pl.n);
  p->status = reinterpret_cast<unsigned int*>(ws_head);
  p->tag = call_tag();
}

static bool matrix_map(CUtensorMap* m, const float* ptr, long cols, long rows, int box_cols, int box_rows) {
  const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows}, str[1] = {(uint64_t)cols * 4};
  const uint32_t box[2] = {(uint32_t)box_cols, (uint32_t)box_rows};
  return make_map_f32(m, ptr, 2, dims, str, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

template <int KIND>
static xconv_status launch_gemm_split(const CUtensorMap& ma, const CUtensorMap& mb, const GemmSplitParams& p, unsigned grid, cudaStream_t st) {
  const size_t smem = 1024 + (size_t)p.f_off + (size_t)p.f_slots * p.f_slot;
  const int threads = KIND >= GS_BACK_BF16 ? SP_CONVERT * 32 : SP_THREADS;
  if (smem > (size_t)(SMEM_LIMIT - 1024) || (KIND < GS_BACK_BF16 && (p.stages != GS_TEAMS || p.f_slots < GS_TEAMS))) return XCONV_ERR_UNSUPPORTED;
  cudaError_t e = cudaFuncSetAttribute(gemm_split_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT - 1024);
  if (e == cudaSuccess) e = launch_pdl(gemm_split_kernel<KIND>, dim3(grid), dim3(threads), smem_of_grid(smem, grid), st, ma, mb, p);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

xconv_status run_sketch_split(const xconv_desc* d, const GemmSplitPlan& pl, const float* X, const float* Z, float* part, char* ws_head,
                              cudaStream_t st) {
  GemmSplitParams p{};
  const float *rows = pl.swap ? X : Z, *cols = pl.swap ? Z : X;
  p.out = part;
  p.M = pl.swap ? d->B : d->r;
  p.N = pl.swap ? d->r : d->B;
  p.K = (long)(d->D > 1 ? d->D : 1) * d->H * d->W * d->Cin;
  p.o_m = pl.swap ? 1 : d->B;
  p.o_n = pl.swap ? d->B : 1;
  fill_common(pl, GS_SKETCH, ws_head, &p);
  p.a_lo0 = 1u << 16; p.a_step = 2;
  p.f_b = up1k((uint32_t)p.f_rows_a * 128);
  p.f_slot = p.f_b + up1k((uint32_t)p.f_rows_b * 128);
  p.f_bytes = (uint32_t)(p.f_rows_a + p.f_rows_b) * 128;
  CUtensorMap ma, mb;
  if (!matrix_map(&ma, rows, p.K, p.M, GS_TERMS, p.f_rows_a) || !matrix_map(&mb, cols, p.K, p.N, GS_TERMS, p.f_rows_b)) return XCONV_ERR_CUDA;
  return launch_gemm_split<GS_SKETCH>(ma, mb, p, (unsigned)(pl.tiles_m * pl.tiles_n * pl.splits), st);
}

xconv_status run_backprobe_split(const xconv_desc* d, const GemmSplitPlan& pl, const float* S, long s_row, long s_k, const void* Y, void* L,
                                 char* ws_head, char* scratch, cudaStream_t st) {
  const int kind = back_kind(d);
  GemmSplitParams p{};
  p.B = S; p.Y = Y; p.s_row = s_row; p.s_k = s_k;
  p.img = reinterpret_cast<const uint8_t*>(scratch);
  p.out = L;
  p.M = (long)(d->D > 1 ? d->D : 1) * d->H * d->W * d->Cout;
  p.N = d->r; p.K = d->B;
  p.o_m = 1; p.o_n = p.M;
  fill_common(pl, kind, ws_head, &p);
  p.a_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
  p.a_lo0 = (4096u >> 4) << 16; p.a_step = (16 * 128) >> 4; p.idesc |= 1u << 15;
  float* scale = reinterpret_cast<float*>(scratch + (size_t)pl.tiles_n * pl.kblocks * p.b_bytes);
  p.scale = scale;
  CUtensorMap ma;
  if (kind == GS_BACK) {
    p.f_slot = p.f_bytes = GS_TERMS * 512;
    if (!matrix_map(&ma, static_cast<const float*>(Y), p.M, p.K, TILE_M, GS_TERMS)) return XCONV_ERR_CUDA;
  } else {
    const uint64_t dims[2] = {(uint64_t)p.M, (uint64_t)p.K}, str[1] = {(uint64_t)p.M * 2};
    const uint32_t box[2] = {64, GS_TERMS};
    if (!make_map(&ma, Y, 2, dims, str, box, kind == GS_BACK_F16)) return XCONV_ERR_CUDA;
    p.f_slot = 4 * GS_OUT;
  }
  const long pieces = (long)p.tiles_n * p.kblocks * p.n * 8;
  const dim3 block(256);
  const cudaError_t e = kind == GS_BACK_F16
      ? launch_pdl(split_sketch_images_f16, dim3((unsigned)cdivl((long)p.tiles_n * p.n, 8)), block, 0, st, p, reinterpret_cast<uint8_t*>(scratch), scale)
      : launch_pdl(split_sketch_images, dim3((unsigned)std::min<long>(2 * NUM_SMS, cdivl(pieces, 256))), block, 0, st, p,
                   reinterpret_cast<uint8_t*>(scratch));
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  const unsigned grid = (unsigned)std::min<long>(pl.tiles_m * pl.tiles_n, NUM_SMS);
  return kind == GS_BACK ? launch_gemm_split<GS_BACK>(ma, ma, p, grid, st)
         : kind == GS_BACK_F16 ? launch_gemm_split<GS_BACK_F16>(ma, ma, p, grid, st) : launch_gemm_split<GS_BACK_BF16>(ma, ma, p, grid, st);
}

}  // namespace xconv
