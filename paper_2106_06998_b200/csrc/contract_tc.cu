// The offset contraction (Algorithm 1 backward step 4, Eq. 6) on the tensor cores for layers of few channels, 16-bit
// storage (sm_100a):
//
//   dW[m, n, (dz, dy, dx)] = scale * sum over positions q of L[q, m] * Z[q + (dz, dy, dx) - pad, n]
//
// (with dY and the rebuilt activation in the places of L and Z when the estimate sums over the probes first).  With a
// tile per kernel offset, 32 output channels fill a quarter of the 128 MMA rows and every offset copies Z again.  Here a
// patch of pw x ph positions of both tensors is copied once, with a halo, and the offsets are spread over BOTH sides of
// one MMA: rows (i, m) = L moved by i rows of the image, columns (j, n) = Z moved by j pixels,
//
//   D[(i, m), (j, n)] += sum over the 16 pixels of a k-step of L[q + (i - p) rows, m] * Z[q + (j - p) pixels, n]
//                        which is the offset dy = KS - 1 - i, dx = j.
//
// Both tiles are MN-major (rows = pixels, 2*cw bytes of channels each), and the shifted copies are the same shared memory
// again: the descriptor's stride between column blocks (its leading byte offset) is one image row of the patch on the L
// side and one pixel on the Z side.  Positions outside the image are zero-filled by the copy engine on at least one side of
// every product that must vanish.  A k-step lies inside one image row, so pw is a multiple of 16.
//
// Where the rows are full without it (more than 64 output channels) L is not moved and a work unit holds one dy; volumes
// put dz on the column side, in one unit while the accumulators fit tensor memory.  Channel blocks are 64 (or 32) wide, the
// last one padded with zeros by the copy engine.  The patches are dealt evenly to k-splits, whose partial sums (in the
// order they leave tensor memory) a second kernel adds in fixed order.
//
// The accumulators of the tensor cores are not rounded to nearest, and a chain of 2700 k-steps left 5e-5 of a sum (about 2e-8 a
// k-step) where FP32 multiply-adds leave 2e-6.  Layers whose contraction was on those before (channels off the multiples of
// 32) are therefore *drained*: two accumulator sets take CH_DRAIN k-steps in turn, and eight epilogue warps add each up in
// float registers, 128 of them a thread, which is why a unit then has at most 256 columns (more row tiles or pixel shifts become
// units of their own).  Against 64 bits, xconv_contract alone, 180 random layers, times the error of the FP32-FMA kernel: median 2.6
// and largest 24 undrained, 0.95 and 4.3 with 32 k-steps, 0.5 to 1 and 3.4 with 16 (all above 2.2 below 6e-7 in itself).  us,
// FP32-FMA kernel -> undrained -> drained: 3 -> 64 channels 112 x 112, 64 probes 2568 -> 72 -> 57; 16 -> 32, 5 x 5 86 -> 15 -> 14;
// 48 -> 48, 64 x 64 378 -> 26 -> 31; 24 -> 96 326 -> 19 -> 23; volumes 16 -> 16 6976 -> 224 -> 244.
//
// What bounds it: with 32 channels a side one MMA of 96 columns per 16 pixels serves nine offsets (the tile per offset took
// three times the tensor time and ten copied tiles where this takes two), and the copies from memory remain: 256 x 256 images,
// 16 samples, 134 MB: 87 -> 33 us (4.1 TB/s); 48^3 volumes, 27 offsets, 57 MB: 249 -> 55 us.  From 64 channels a side on the
// partial sums of the splits weigh as much as the mainloop.  It also serves the channel counts that only the FP32-FMA
// kernel took (16 -> 32 channels 5 x 5: 89 -> 12 us; 3 -> 64 channels of 112 x 112 images, 32 samples: 1295 -> 28 us).
#include "common.cuh"
#include "tc_api.h"
#include "tc_ptx.cuh"

namespace xconv {

constexpr int CH_STAGES = 6, CH_PIECES = 12;
constexpr int CH_DRAIN = 16;                      // k-steps a drained accumulator holds
constexpr int halo_threads(bool drain) { return drain ? 320 : 192; }

struct HaloParams {
  int KS, pad, pad_d;
  int pw, ph, patches_x, patches_y, depth;
  uint32_t items, splits;
  int rows_on_a;                                   // L moved by image rows on the MMA rows; else one dy per unit
  int dy_n, dz_n, dz_per, ng_n, ng_per, mg_n, mt;  // work units: dy, groups of dz, of channel blocks of Z, of MMA row tiles,
  int j_n, j_per;                                  // ... of pixel shifts
  int chunk_rows, chunk_patches;                   // drained: what an accumulator set holds (several patches, or some rows of one)
  int a_boxes, b_boxes;                            // channel blocks copied per stage
  int cwa, cwb;
  uint32_t a_blk, b_blk, a_bytes, stage_bytes, tx_bytes;
  int stages;
  uint32_t a_row16, b_row16;                       // image row of the patch in the two tiles (bytes >> 4)
  uint32_t a_step16, b_step16;                     // 16 pixels
  uint32_t a_mt16, a_lo0, b_lo0, a_hi, b_hi;
  int pieces, cols, tmem_cols;                     // MMAs per k-step and row tile; accumulator columns per row tile
  uint32_t piece_off[CH_PIECES], piece_col[CH_PIECES], piece_idesc[CH_PIECES];
  int Cout, Cin, T;
  float* part;
  unsigned int* status;
  unsigned int tag;
};

struct HaloUnit { int dy, dzg, ng, mg, jg; };
__host__ __device__ __forceinline__ HaloUnit halo_unit(const HaloParams& p, uint32_t ug) {
  HaloUnit u;
  u.ng = (int)(ug % (uint32_t)p.ng_n); ug /= (uint32_t)p.ng_n;
  u.jg = (int)(ug % (uint32_t)p.j_n); ug /= (uint32_t)p.j_n;
  u.dzg = (int)(ug % (uint32_t)p.dz_n); ug /= (uint32_t)p.dz_n;
  u.dy = (int)(ug % (uint32_t)p.dy_n); ug /= (uint32_t)p.dy_n;
  u.mg = (int)ug;
  return u;
}

// The MMAs of `rows` image rows of a patch.  FORM 1 and 2: as many row tiles and one piece; 12 and 13: one row tile, two or three
// pieces; 0: any number of both.  KX: k-steps of a row, 0 for any number.  The warp issues an instruction per some six clocks, so a loop that looks the
// pieces up took 135 clocks an MMA of 56 (volumes of 48^3, 32 channels 49 -> 34 us), and a loop over a row's k-steps 143 an MMA of 62 where there is one (images of 16 columns), 96
// for two, 69 for three.  us a call with its reduction, that loop -> rows unrolled: 64 -> 16 channels, 12 planes of 13 x 13, 290 probes 112 -> 73; 48 -> 64, 256 images of 86 x 86 36.6 -> 27.8;
// volumes of 48^3, 32 channels 44 -> 36; 32 -> 32, 64 probes of 256 x 256 106 -> 90.  (Asking for the next patch before this one's commit gains 1 % where the MMAs bound it
// and loses 5 % where the copies do.)
template <int FORM, int KX>
__device__ __forceinline__ void halo_mmas(const HaloParams& p, int rows, uint32_t tmem, uint32_t a0, uint32_t b0, uint32_t& acc,
                                          uint32_t id0) {
  const int kx = KX > 0 ? KX : p.pw >> 4;
  const uint32_t a_step = p.a_step16, b_step = p.b_step16;
  auto kstep = [&](uint32_t a, uint32_t b) {
    if (FORM > 10) {
#pragma unroll
      for (int i = 0; i < FORM - 10; ++i)
        umma_warp(tmem + p.piece_col[i], a, p.a_hi, b + p.piece_off[i], p.b_hi, p.piece_idesc[i], acc);
    } else if (FORM > 0) {
      umma_warp(tmem, a, p.a_hi, b, p.b_hi, id0, acc);
      if (FORM == 2) umma_warp(tmem + (uint32_t)p.cols, a + p.a_mt16, p.a_hi, b, p.b_hi, id0, acc);
    } else {
      for (int i = 0; i < p.pieces; ++i) {
        const uint32_t bb = b + p.piece_off[i], d = tmem + p.piece_col[i], id = p.piece_idesc[i];
        umma_warp(d, a, p.a_hi, bb, p.b_hi, id, acc);
        if (p.mt > 1) umma_warp(d + (uint32_t)p.cols, a + p.a_mt16, p.a_hi, bb, p.b_hi, id, acc);
        if (p.mt > 2) umma_warp(d + 2u * (uint32_t)p.cols, a + 2u * p.a_mt16, p.a_hi, bb, p.b_hi, id, acc);
      }
    }
    acc = 1u;
  };
  if (KX > 0) {
    constexpr int ROWS = KX == 1 ? 4 : KX == 2 ? 2 : 1;            // unrolled together
    int y = 0;
#pragma unroll 1
    for (; y + ROWS <= rows; y += ROWS) {
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
#pragma unroll
        for (int x = 0; x < KX; ++x) kstep(a0 + (uint32_t)x * a_step, b0 + (uint32_t)x * b_step);
        a0 += p.a_row16;
        b0 += p.b_row16;
      }
    }
    if (ROWS > 1)
#pragma unroll 1
      for (; y < rows; ++y) {
#pragma unroll
        for (int x = 0; x < KX; ++x) kstep(a0 + (uint32_t)x * a_step, b0 + (uint32_t)x * b_step);
        a0 += p.a_row16;
        b0 += p.b_row16;
      }
  } else {
    for (int y = 0; y < rows; ++y) {
      uint32_t a = a0, b = b0;
      for (int x = 0; x < kx; ++x) {
        kstep(a, b);
        a += a_step;
        b += b_step;
      }
      a0 += p.a_row16;
      b0 += p.b_row16;
    }
  }
}

struct HaloBars { uint64_t *full, *empty, *acc_full, *acc_empty; };

// The issuing warp of a drained contraction: two accumulator sets in turn, each for chunk_patches patches or for chunk_rows rows
// of one (a loop per chunk and nothing to decide per row: the warp issues an instruction per some six clocks).  `a_add`, `b_add`,
// `id0`: what the unit moves the two tiles by, and the instruction descriptor for its pixel shifts (FORM > 0).
template <int FORM, int KX>
__device__ __forceinline__ void halo_issue_drained(const HaloParams& p, const HaloBars& bar, uint32_t n, uint32_t tmem_base,
                                                   uint32_t s0, uint32_t a_add, uint32_t b_add, uint32_t id0) {
  const uint32_t stage16 = p.stage_bytes >> 4, set_cols = (uint32_t)(p.mt * p.cols);
  uint32_t s = 0, par = 0, acc = 0, st = s0, tmem = tmem_base, buf = 0, buf_par = 1;   // (a wait for the phase before the first returns at once)
  int left = 0;
  for (uint32_t i = 0; i < n; ++i) {
    if (!mbar_wait_warp(&bar.full[s], par, p.status, p.tag)) return;
    tc_fence_after();
    uint32_t a = (p.a_lo0 | st) + a_add, b = (p.b_lo0 | st) + b_add;
    for (int y = 0; y < p.ph; y += p.chunk_rows) {
      if (left == 0) {
        if (!mbar_wait_warp(&bar.acc_empty[buf], buf_par, p.status, p.tag)) return;
        tc_fence_after();
        acc = 0;
        left = p.chunk_patches;
      }
      halo_mmas<FORM, KX>(p, min(p.chunk_rows, p.ph - y), tmem, a, b, acc, id0);
      if (--left == 0 || (i + 1 == n && y + p.chunk_rows >= p.ph)) {
        umma_commit_warp(&bar.acc_full[buf]);
        left = 0;
        buf_par ^= buf;
        buf ^= 1u;
        tmem = tmem_base + buf * set_cols;
      }
      a += p.a_row16 * (uint32_t)p.chunk_rows;
      b += p.b_row16 * (uint32_t)p.chunk_rows;
    }
    umma_commit_warp(&bar.empty[s]);
    st += stage16;
    if (++s == (uint32_t)p.stages) { s = 0; par ^= 1u; st = s0; }
  }
}

// ... of an undrained one: a single chain.
template <int FORM, int KX>
__device__ __forceinline__ void halo_issue_chain(const HaloParams& p, const HaloBars& bar, uint32_t n, uint32_t tmem_base, uint32_t b0, uint32_t a_bytes16) {
  const uint32_t stage16 = p.stage_bytes >> 4;
  uint32_t s = 0, par = 0, acc = 0, st = b0;
  for (uint32_t i = 0; i < n; ++i) {
    if (!mbar_wait_warp(&bar.full[s], par, p.status, p.tag)) return;
    tc_fence_after();
    halo_mmas<FORM, KX>(p, p.ph, tmem_base, p.a_lo0 | st, p.b_lo0 | (st + a_bytes16), acc, p.piece_idesc[0]);
    umma_commit_warp(&bar.empty[s]);
    st += stage16;
    if (++s == (uint32_t)p.stages) { s = 0; par ^= 1u; st = b0; }
  }
  umma_commit_warp(&bar.acc_full[0]);
}

template <bool F16, bool DRAIN>
__global__ void __launch_bounds__(halo_threads(DRAIN), 1)
contract_halo_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const HaloParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[CH_STAGES], empty[CH_STAGES], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int go;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  if (threadIdx.x == 0) {
    for (int s = 0; s < CH_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    prefetch_tmap(&map_a);
    prefetch_tmap(&map_b);
  }
  if (warp == 1) tmem_alloc_then_trigger(&tmem_slot, (uint32_t)p.tmem_cols);
  pdl_wait();
  if (threadIdx.x == 0) {
    go = (*reinterpret_cast<volatile unsigned int*>(p.status) != p.tag) ? 1 : 0;
    if (blockIdx.x == 0) reinterpret_cast<volatile unsigned int*>(p.status)[1] = p.tag;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  const uint32_t ug = blockIdx.x / p.splits, split = blockIdx.x - ug * p.splits;
  const uint32_t i0 = (uint32_t)((unsigned long long)p.items * split / p.splits);
  const uint32_t n = (uint32_t)((unsigned long long)p.items * (split + 1) / p.splits) - i0;     // patches of this CTA (>= 1)

  if (!go) {
    // fall through to the teardown
  } else if (warp == 0) {
    // ------------------------------------------------------------------ copies
    if (lane == 0) {
      const HaloUnit u = halo_unit(p, ug);
      const uint32_t qa = i0 / (uint32_t)p.patches_x, qb = qa / (uint32_t)p.patches_y, qc = qb / (uint32_t)p.depth;
      int x = (int)(i0 - qa * p.patches_x) * p.pw, y = (int)(qa - qb * p.patches_y) * p.ph;
      int z = (int)(qb - qc * p.depth), b = (int)qc;
      const int a_c0 = p.rows_on_a ? 0 : u.mg * p.a_boxes * p.cwa, b_c0 = u.ng * p.ng_per * p.cwb;
      const int a_dy = p.rows_on_a ? -p.pad : 0, b_dy = p.rows_on_a ? 0 : u.dy - p.pad;
      const int b_dz = u.dzg * p.dz_per - p.pad_d;
      int s = 0;
      uint32_t par = 1;                            // (a wait for the phase before the first returns at once)
      uint32_t i = 0;
      for (; i < n; ++i) {
        if (!mbar_wait(&empty[s], par, p.status, p.tag)) break;
        const uint32_t dst = base + (uint32_t)s * p.stage_bytes;
        mbar_arrive_expect_tx(&full[s], p.tx_bytes);
        for (int g = 0; g < p.a_boxes; ++g)
          tma_load_5d(dst + (uint32_t)g * p.a_blk, &map_a, a_c0 + g * p.cwa, x, y + a_dy, z, b, &full[s]);
        for (int g = 0; g < p.b_boxes; ++g)
          tma_load_5d(dst + p.a_bytes + (uint32_t)g * p.b_blk, &map_b, b_c0 + g * p.cwb, x - p.pad, y + b_dy, z + b_dz, b, &full[s]);
        if ((x += p.pw) >= p.patches_x * p.pw) {
          x = 0;
          if ((y += p.ph) >= p.patches_y * p.ph) { y = 0; if (++z == p.depth) { z = 0; ++b; } }
        }
        if (++s == p.stages) { s = 0; par ^= 1u; }
      }
      // every copy issued must have landed before the CTA exits
      for (uint32_t k = i > (uint32_t)p.stages ? i - p.stages : 0; k < i; ++k)
        if (!mbar_wait(&full[k % p.stages], (k / p.stages) & 1u, p.status, p.tag)) break;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the whole warp)
    const uint32_t b0 = ((base & 0x3FFFFu) >> 4), a_bytes16 = p.a_bytes >> 4;
    const bool one = p.mt == 1 && p.pieces == 1;
    if (DRAIN) {
      const HaloUnit u = halo_unit(p, ug);
      const HaloBars bar{full, empty, acc_full, acc_empty};
      const uint32_t a_add = p.rows_on_a ? (uint32_t)(u.mg * p.mt) * p.a_mt16 : 0u;
      const uint32_t b_add = a_bytes16 + (uint32_t)(u.jg * p.j_per) * (p.b_step16 >> 4);
      const int fewer = max(0, (u.jg + 1) * p.j_per - p.KS) * p.cwb;           // columns of shifts behind the last one
      const uint32_t id0 = p.piece_idesc[0] - ((uint32_t)(fewer >> 3) << 17);
#define XC_ISSUE(FORM, KX) halo_issue_drained<FORM, KX>(p, bar, n, tmem_base, b0, a_add, b_add, id0)
#define XC_ROWS(FORM) switch (p.pw >> 4) { case 1: XC_ISSUE(FORM, 1); break; case 2: XC_ISSUE(FORM, 2); break; case 3: XC_ISSUE(FORM, 3); break; \
                                           case 4: XC_ISSUE(FORM, 4); break; default: XC_ISSUE(FORM, 0); }
      if (one) XC_ROWS(1)
      else if (p.mt == 2 && p.pieces == 1) XC_ROWS(2)
      else if (p.mt == 1 && p.pieces == 2) XC_ROWS(12)
      else if (p.mt == 1 && p.pieces == 3) XC_ROWS(13)
      else XC_ISSUE(0, 0);
#undef XC_ISSUE
    } else {
      const HaloBars bar{full, empty, acc_full, acc_empty};
#define XC_ISSUE(FORM, KX) halo_issue_chain<FORM, KX>(p, bar, n, tmem_base, b0, a_bytes16)
      if (one) XC_ROWS(1)
      else if (p.mt == 2 && p.pieces == 1) XC_ROWS(2)
      else if (p.mt == 1 && p.pieces == 2) XC_ROWS(12)
      else if (p.mt == 1 && p.pieces == 3) XC_ROWS(13)
      else XC_ISSUE(0, 0);
#undef XC_ROWS
#undef XC_ISSUE
    }
  } else {
    // ------------------------------------------------------------------ epilogue: partial sums in accumulator order
    const int quad = warp & 3;
    // rows behind the last shift or channel are not stored
    const int row_w = halo_unit(p, ug).mg * p.mt * TILE_M + quad * 32, row_end = p.rows_on_a ? p.KS * p.cwa : p.Cout;
    float* part = p.part + ((((size_t)ug * p.splits + split) * p.mt) * (p.cols >> 2) * TILE_M + quad * 32 + lane) * 4;
    bool ok = true;
    if (DRAIN) {
      // two warps per quadrant take the 32-column chunks of the row tiles in turn and add up each set in registers
      const int half = (warp - 2) >> 2, chunks = p.cols >> 5, all = p.mt * chunks;
      const uint32_t tmem_q = tmem_base + ((uint32_t)(quad * 32) << 16);
      const uint32_t per_patch = (uint32_t)((p.ph + p.chunk_rows - 1) / p.chunk_rows);
      const uint32_t sets = per_patch > 1 ? n * per_patch : (n + (uint32_t)p.chunk_patches - 1) / (uint32_t)p.chunk_patches;
      float sum[4][32];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int e = 0; e < 32; ++e) sum[k][e] = 0.f;
      for (uint32_t c = 0; c < sets; ++c) {
        const uint32_t buf = c & 1u;
        if (lane == 0) ok = mbar_wait(&acc_full[buf], (c >> 1) & 1u, p.status, p.tag);
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (half + 2 * k >= all) break;
          uint32_t v[32];
          tmem_ld32(tmem_q + buf * (uint32_t)(p.mt * p.cols) + (uint32_t)(half + 2 * k) * 32, v);
#pragma unroll
          for (int e = 0; e < 32; ++e) sum[k][e] += __uint_as_float(v[e]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[buf]);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int at = half + 2 * k, t = at / chunks;
        if (!ok || at >= all) break;
        if (row_w + t * TILE_M >= row_end) continue;
        float* dst = part + ((size_t)t * (p.cols >> 2) + (size_t)(at - t * chunks) * 8) * TILE_M * 4;
#pragma unroll
        for (int e = 0; e < 32; e += 4)
          *reinterpret_cast<float4*>(dst + (size_t)(e >> 2) * TILE_M * 4) = make_float4(sum[k][e], sum[k][e + 1], sum[k][e + 2], sum[k][e + 3]);
      }
    } else {
      if (lane == 0) ok = mbar_wait(&acc_full[0], 0, p.status, p.tag);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      tc_fence_after();
      if (ok)
        for (int t = 0; t < p.mt; ++t) {
          if (row_w + t * TILE_M >= row_end) continue;
          float* dst = part + (size_t)t * (p.cols >> 2) * TILE_M * 4;
          for (int c = 0; c < p.cols; c += 32) {
            uint32_t v[32];
            tmem_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(t * p.cols + c), v);
#pragma unroll
            for (int k = 0; k < 32; k += 4)
              *reinterpret_cast<float4*>(dst + (size_t)((c + k) >> 2) * TILE_M * 4) =
                  make_float4(__uint_as_float(v[k]), __uint_as_float(v[k + 1]), __uint_as_float(v[k + 2]), __uint_as_float(v[k + 3]));
          }
        }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// dW[m][offset][n] = scale(n) * sum over splits, four neighbouring columns of one accumulator row per group.  LANES
// threads share a group and take the splits in turn; their sums are added in lane order.  `cout_out`, `cin_out`: channels
// of dW (the padded channels behind them have no place in it).
template <int LANES>
__global__ void __launch_bounds__(256) reduce_halo_partials(const HaloParams p, float* out, uint32_t groups, int cout_out, int cin_out, float alpha,
                                                            const float* chan_scale) {
  constexpr int GROUPS = 256 / LANES;
  __shared__ float4 acc[LANES][GROUPS];
  const int o = threadIdx.x % GROUPS, g = threadIdx.x / GROUPS;
  const uint32_t idx = blockIdx.x * GROUPS + o;
  const uint32_t row = idx % TILE_M, q4 = (uint32_t)p.cols >> 2;
  uint32_t t = idx / TILE_M;
  const uint32_t q = t % q4; t /= q4;
  const uint32_t mt = t % (uint32_t)p.mt, ug = t / (uint32_t)p.mt;
  const HaloUnit u = halo_unit(p, ug);
  int m, dy;
  if (p.rows_on_a) {
    const int i = (int)((u.mg * p.mt + mt) * TILE_M + row) / p.cwa;
    m = (int)row % p.cwa;
    dy = p.KS - 1 - i;
  } else {
    m = (u.mg * p.mt + (int)mt) * TILE_M + (int)row;
    dy = u.dy;
  }
  const int c = (int)q * 4, per = p.j_per * p.cwb, grp = c / per, j = u.jg * p.j_per + (c - grp * per) / p.cwb;
  const int nb = u.ng * p.ng_per + grp % p.ng_per, dz = u.dzg * p.dz_per + grp / p.ng_per;
  const int n = nb * p.cwb + (c - grp * per) % p.cwb;
  const bool live = idx < groups && dy >= 0 && j < p.KS && m < cout_out && n < cin_out;
  const size_t tile = (size_t)p.mt * p.cols * TILE_M;
  const float* src = p.part + (size_t)ug * p.splits * tile + ((size_t)mt * q4 * TILE_M + (size_t)q * TILE_M + row) * 4;
  pdl_wait();                                        // (what is above runs under the kernel before)
  float4 s = live ? sum_splits4<LANES>(src, tile, g, (int)p.splits) : make_float4(0.f, 0.f, 0.f, 0.f);
  pdl_trigger();
  if (LANES > 1) {
    acc[g][o] = s;
    __syncthreads();
    if (g != 0) return;
#pragma unroll
    for (int l = 1; l < LANES; ++l) { s.x += acc[l][o].x; s.y += acc[l][o].y; s.z += acc[l][o].z; s.w += acc[l][o].w; }
  }
  if (!live) return;
  const float r[4] = {s.x, s.y, s.z, s.w};
  float* dst = out + ((size_t)m * p.T + (dz * p.KS + dy) * p.KS + j) * cin_out + n;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (n + k < cin_out) dst[k] = r[k] * (chan_scale ? chan_scale[n + k] : alpha);
}

// ------------------------------------------------------------------------------------ host side

static uint32_t up1k(uint32_t v) { return (v + 1023u) & ~1023u; }

// Channel counts whose blocks are at least three quarters full (one block of 32 always).  The line was drawn against the wide
// layers' contraction (96 -> 96 channels, 3 x 3 x 3, a quarter of it padding: 43 -> 47 us); 40, 72, 80, 88 and 136 channels, where
// that one does not go either, have not been measured here and stay on FP32 multiply-adds.
static bool halo_channels(int c) { return c % 8 == 0 && (c <= 32 || 4 * c >= 3 * round_up(c, 64)); }

// `d`: r planes groups (probes, or samples in the other order), D planes each.
// `drain`: the accumulators are emptied every CH_DRAIN k-steps; the two sets then share tensor memory, and the epilogue warps
// hold one in registers (256 columns).
bool tc_plan_halo(const xconv_desc* d, bool drain, TcHaloPlan* p) {
  if ((d->dtype != XCONV_BF16 && d->dtype != XCONV_F16) || d->circular) return false;
  if (!halo_channels(d->Cin) || !halo_channels(d->Cout)) return false;
  const int KS = d->KH, KD = d->KD > 1 ? d->KD : 1;
  const long depth = KD > 1 ? (d->D > 1 ? d->D : 1) : 1, outer = KD > 1 ? d->r : (long)d->r * (d->D > 1 ? d->D : 1);
  if ((long)d->H * d->W < 16 || outer * depth >= (1L << 31)) return false;
  p->cwa = d->Cout > 32 ? 64 : 32;
  p->cwb = d->Cin > 32 ? 64 : 32;
  const int ga = (int)cdivl(d->Cout, p->cwa), gb = (int)cdivl(d->Cin, p->cwb);
  const int limit = drain ? 256 : 512;
  p->drain = drain ? 1 : 0;
  p->j_per = KS * p->cwb <= limit ? KS : 3;                          // pixel shifts of a unit
  p->j_n = (int)cdivl(KS, p->j_per);
  const int per = p->j_per * p->cwb;                                 // columns of one (dz, channel block)
  p->rows_on_a = ga == 1 ? 1 : 0;
  int nblk = 0;                                                      // moved copies of L the MMA rows read
  for (;;) {
    const int tiles = p->rows_on_a ? (int)cdivl(KS * p->cwa, TILE_M) : (int)cdivl(d->Cout, TILE_M);
    p->mt = p->rows_on_a ? tiles : std::min(tiles, 2);
    p->dz_per = KD; p->ng_per = gb;
    auto fits = [&]() { return p->mt * p->dz_per * p->ng_per * per <= limit && p->dz_per * p->ng_per * (per > 256 ? 2 : 1) <= CH_PIECES; };
    if (!fits() && KD > 1) p->dz_per = 1;
    while (!fits() && p->ng_per > 1) --p->ng_per;
    if (!fits() && (!p->rows_on_a || drain)) p->mt = 1;
    p->mg_n = (int)cdivl(tiles, p->mt);
    nblk = tiles * (TILE_M / p->cwa);
    if (fits()) break;
    if (!p->rows_on_a) return false;
    p->rows_on_a = 0;
  }
  p->ng_n = (int)cdivl(gb, p->ng_per);
  p->dz_n = KD / p->dz_per;
  p->dy_n = p->rows_on_a ? 1 : KS;
  p->cols = p->dz_per * p->ng_per * per;
  const long units = (long)p->mg_n * p->dy_n * p->dz_n * p->ng_n * p->j_n;
  // Patch: clocks of its MMAs (half a clock per column, at least the 50 between two issues) or of its copies (45 bytes
  // per clock and SM from L2), by the number of patches.
  const int pieces = p->dz_per * p->ng_per * (per > 256 ? 2 : 1);
  const long kstep = (long)p->mt * std::max(50L * pieces, (long)p->cols / 2);
  const int a_blocks = p->rows_on_a ? 1 : (p->mg_n > 1 || p->mt > 1 || ga > 1 ? 2 * p->mt : 1);
  long best = -1;
  const long nx0 = cdivl(d->W, 128), nx1 = std::min(cdivl(d->W, 16), std::max(4 * nx0, 12L));
  for (long nx = nx0; nx <= nx1; ++nx) {
    const int pw = round_up((int)cdivl(d->W, nx), 16);
    for (int ph = std::min(d->H, 16); ph >= 1; ph = ph > 1 ? (ph + 1) / 2 : 0) {
      const int a_rows = p->rows_on_a ? pw * (ph + KS - 1) : pw * ph, a_need = p->rows_on_a ? pw * (ph + nblk - 1) : a_rows;
      const int b_rows = (pw + KS - 1) * ph * p->dz_per;
      const uint32_t a_blk = up1k((uint32_t)std::max(a_rows, a_need) * 2 * p->cwa), b_blk = up1k((uint32_t)b_rows * 2 * p->cwb);
      const uint32_t stage = a_blk * a_blocks + b_blk * p->ng_per;
      const int stages = (int)std::min<long>(CH_STAGES, (SMEM_LIMIT - 4096) / stage);
      if (stages < 2 || (pw + KS - 1) > 256) continue;
      const long patches = cdivl(d->W, pw) * cdivl(d->H, ph) * depth * outer;
      if (patches >= (1L << 31)) return false;
      const long bytes = (long)a_rows * 2 * p->cwa * std::min(ga, p->rows_on_a ? 1 : 2 * p->mt) + (long)b_rows * 2 * p->cwb * p->ng_per;
      const long clk = std::max(kstep * (pw / 16) * ph, bytes / 45) + 250 + (stages < 3 ? 300 : 0);
      const long splits = std::max(1L, std::min((long)NUM_SMS / units, patches));
      const long cost = cdivl(patches, splits) * clk;
      if (best >= 0 && cost >= best) continue;
      best = cost;
      p->pw = pw; p->ph = ph; p->stages = stages; p->a_blk = a_blk; p->b_blk = b_blk; p->a_blocks = a_blocks;
      p->patches = patches; p->splits = splits;
    }
  }
  if (best < 0) return false;
  // a split has to be long enough to be worth its partial tile
  p->splits = std::max(1L, std::min(p->splits, p->patches / 2));
  p->units = units;
  p->part_bytes = (size_t)units * p->splits * p->mt * p->cols * TILE_M * sizeof(float);
  return true;
}

xconv_status tc_run_halo(const xconv_desc* d, const TcHaloPlan& pl, const void* L, const void* Z, int cout_out, int cin_out, float* dW,
                         float alpha, char* ws_head, char* part, cudaStream_t st) {
  const int KS = d->KH, KD = d->KD > 1 ? d->KD : 1;
  const bool f16 = d->dtype == XCONV_F16;
  const long depth = KD > 1 ? (d->D > 1 ? d->D : 1) : 1, outer = KD > 1 ? d->r : (long)d->r * (d->D > 1 ? d->D : 1);
  HaloParams p{};
  p.KS = KS; p.pad = (KS - 1) / 2; p.pad_d = (KD - 1) / 2;
  p.pw = pl.pw; p.ph = pl.ph; p.patches_x = (int)cdivl(d->W, pl.pw); p.patches_y = (int)cdivl(d->H, pl.ph); p.depth = (int)depth;
  p.items = (uint32_t)pl.patches; p.splits = (uint32_t)pl.splits;
  p.rows_on_a = pl.rows_on_a;
  p.dy_n = pl.dy_n; p.dz_n = pl.dz_n; p.dz_per = pl.dz_per; p.ng_n = pl.ng_n; p.ng_per = pl.ng_per; p.mg_n = pl.mg_n; p.mt = pl.mt;
  p.j_n = pl.j_n; p.j_per = pl.j_per;
  p.chunk_rows = std::min(pl.ph, std::max(1, CH_DRAIN / (pl.pw / 16)));
  p.chunk_patches = p.chunk_rows == pl.ph ? std::max(1, CH_DRAIN / (pl.pw / 16 * pl.ph)) : 1;
  p.cwa = pl.cwa; p.cwb = pl.cwb;
  const uint32_t rba = 2 * (uint32_t)pl.cwa, rbb = 2 * (uint32_t)pl.cwb;
  p.a_boxes = pl.a_blocks; p.b_boxes = pl.ng_per;
  p.a_blk = pl.a_blk; p.b_blk = pl.b_blk;
  p.a_bytes = pl.a_blk * (uint32_t)pl.a_blocks;
  p.stage_bytes = p.a_bytes + pl.b_blk * (uint32_t)pl.ng_per;
  p.stages = pl.stages;
  const int a_rows = pl.ph + (pl.rows_on_a ? KS - 1 : 0), PB = pl.pw + KS - 1;
  // (a box that lies wholly beyond the last channel still arrives, as zeros)
  p.tx_bytes = (uint32_t)(a_rows * pl.pw) * rba * (uint32_t)p.a_boxes + (uint32_t)(pl.ph * PB * pl.dz_per) * rbb * (uint32_t)p.b_boxes;
  p.a_row16 = ((uint32_t)pl.pw * rba) >> 4; p.b_row16 = ((uint32_t)PB * rbb) >> 4;
  p.a_step16 = (16 * rba) >> 4; p.b_step16 = (16 * rbb) >> 4;
  // MMA rows: moved copies of the one block, an image row apart, or neighbouring channel blocks (a single one: read twice)
  const uint32_t a_lbo = pl.rows_on_a ? (uint32_t)pl.pw * rba : pl.a_blocks > 1 ? pl.a_blk : 0u;
  p.a_mt16 = (pl.rows_on_a ? (uint32_t)(TILE_M / pl.cwa) * pl.pw * rba : 2 * pl.a_blk) >> 4;
  p.a_lo0 = (a_lbo >> 4) << 16;
  p.b_lo0 = (rbb >> 4) << 16;                                        // columns: copies of a block, one pixel apart
  const uint32_t la = pl.cwa == 64 ? 2u : 4u, lb = pl.cwb == 64 ? 2u : 4u;
  p.a_hi = ((8 * rba) >> 4) | (1u << 14) | (la << 29);
  p.b_hi = ((8 * rbb) >> 4) | (1u << 14) | (lb << 29);
  const int per = pl.j_per * pl.cwb;
  p.cols = pl.cols;
  for (int dz = 0; dz < pl.dz_per; ++dz)
    for (int g = 0; g < pl.ng_per; ++g)
      for (int j = 0; j < pl.j_per;) {
        const int nj = std::min(pl.j_per - j, per > 256 ? 3 : pl.j_per), i = p.pieces++;
        p.piece_off[i] = ((uint32_t)g * pl.b_blk + (uint32_t)(dz * pl.ph * PB + j) * rbb) >> 4;
        p.piece_col[i] = (uint32_t)((dz * pl.ng_per + g) * per + j * pl.cwb);
        p.piece_idesc[i] = (1u << 4) | (f16 ? 0u : (1u << 7) | (1u << 10)) | (1u << 15) | (1u << 16) |
                           ((uint32_t)(nj * pl.cwb >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24);
        j += nj;
      }
  p.tmem_cols = pow2_cols((pl.drain ? 2 : 1) * pl.mt * pl.cols);
  p.Cout = d->Cout; p.Cin = d->Cin; p.T = KD * KS * KS;
  p.part = reinterpret_cast<float*>(part);
  p.status = reinterpret_cast<unsigned int*>(ws_head);
  p.tag = call_tag();

  CUtensorMap ma, mb;
  auto map = [&](CUtensorMap* m, const void* ptr, int C, int cw, int bw, int bh, int bd) {
    const uint64_t row = (uint64_t)C * 2;
    const uint64_t dims[5] = {(uint64_t)C, (uint64_t)d->W, (uint64_t)d->H, (uint64_t)depth, (uint64_t)outer};
    const uint64_t str[4] = {row, row * d->W, row * d->W * d->H, row * d->W * d->H * depth};
    const uint32_t box[5] = {(uint32_t)cw, (uint32_t)bw, (uint32_t)bh, (uint32_t)bd, 1};
    return make_map(m, ptr, 5, dims, str, box, f16, cw == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B);
  };
  if (!map(&ma, L, d->Cout, pl.cwa, pl.pw, a_rows, 1) || !map(&mb, Z, d->Cin, pl.cwb, PB, pl.ph, pl.dz_per)) return XCONV_ERR_CUDA;
  const size_t smem = 1024 + (size_t)p.stages * p.stage_bytes;
  if (smem > (size_t)(SMEM_LIMIT - 1024)) return XCONV_ERR_UNSUPPORTED;
  const unsigned grid = (unsigned)(pl.units * pl.splits);
  void (*kernel)(CUtensorMap, CUtensorMap, HaloParams) =
      pl.drain ? (f16 ? contract_halo_kernel<true, true> : contract_halo_kernel<false, true>)
               : (f16 ? contract_halo_kernel<true, false> : contract_halo_kernel<false, false>);
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT - 1024);
  if (e == cudaSuccess) e = launch_pdl(kernel, dim3(grid), dim3(halo_threads(pl.drain != 0)), smem_of_grid(smem, grid), st, ma, mb, p);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  const uint32_t groups = (uint32_t)(pl.units * pl.mt * (pl.cols / 4) * TILE_M);
#define XC_REDUCE(LANES) launch_pdl(reduce_halo_partials<LANES>, dim3((unsigned)cdivl(groups, 256 / LANES)), dim3(256), 0, st, p, dW, \
                                    groups, cout_out, cin_out, alpha, d->chan_scale)
  if (pl.splits >= 64) e = XC_REDUCE(16);
  else if (pl.splits >= 12) e = XC_REDUCE(4);
  else e = XC_REDUCE(1);
#undef XC_REDUCE
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

}  // namespace xconv
