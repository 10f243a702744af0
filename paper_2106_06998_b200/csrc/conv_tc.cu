// The exact convolution Y = conv(X, w) (Algorithm 1 forward step 1, Eq. 5) and the exact input gradient dX on the
// tensor cores, for 16-bit storage (sm_100a).
//
//   D[pixel, co] = sum over (offset, ci) of In[pixel + offset, ci] * w(co, ci, offset)
//
// An MMA row tile is one patch of pw x ph output pixels.  Its input is copied ONCE per block of cw channels, with its
// halo: a box of P = pw + K - 1 columns, ph + K - 1 rows (and KD planes), one tile row of 2*cw bytes per pixel.  The
// MMA rows are the positions m = y * P + x of that box, so the A tile of the offset (dz, dy, dx) is the same shared
// memory, read from dz * plane + dy * P + dx rows further on: K*K*KD offsets cost one copy instead of one each.  (Rows
// m with x >= pw are wasted, their sums are not stored; a tile start inside an 8-row swizzle group is fine because the
// swizzle is a function of the shared-memory address.)  The box is zero-filled outside the image and beyond the last
// channel, which is the zero padding of the convolution and makes any multiple of 8 channels a whole number of MMA steps.
//
// The weights of an offset are a [channels out x channels in] tile, K-major for Y (w as stored) and MN-major for dX (the
// same w, rows = the reduction index, offsets mirrored: no transposed copy is made).  Where all tiles fit beside two
// input boxes they stay in shared memory for the whole launch, otherwise they pass through a ring.
//
// A CTA walks a contiguous run of patches (one CTA per SM).  Warp 0 copies input boxes, warp 2 weights, warp 1 issues
// the MMAs and owns tensor memory, warps 4..7 write the results: tensor memory -> 16 bits -> swizzled staging tile of the
// patch's pixels -> one tensor store per block of channels, which clips at the image border.
// Every wait is bounded as in tc_kernels.cu.
//
// What bounds it: wide layers the tensor pipe under the power cap (256 channels, 28 x 28, batch 512: 437 -> 370 us,
// 1.28 PFLOP/s of the 1.38 that the library GEMM sustains); narrow layers the issuing warp (32 channels: about 50 clocks
// per MMA of 32 columns where its operands take 32; 256 x 256 images 148 -> 43 us, 48^3 volumes 293 -> 44 us).  Two things
// made the difference to copying a box per offset with the MMAs issued by one thread: the halo (a ninth of the copies,
// which the copy engine took some 150 clocks each for), and issuing from a converged warp (the same kernel issued under
// `if (lane == 0)` took 215 us and 380 us on those two layers).
#include "common.cuh"
#include "tc_api.h"
#include "tc_ptx.cuh"
#include "conv_walk.cuh"
#include "conv_slide.cuh"

namespace xconv {

constexpr int CV_THREADS = 384;            // launch bound; a launch has 128 + 128 * groups threads
constexpr int CV_A_SLOTS = 8, CV_W_SLOTS = 8, CV_RING = 32;

struct ConvParams {
  int KD, T, pad, pad_d, dgrad;
  int P, pw, ph, patches_x, patches_y, depth;     // patch geometry
  uint32_t patches, items;                        // patches of the layer; items = patches x column tiles
  uint32_t plane_rows;                            // tile rows of one plane of the box
  int m_sub, acc_bufs, groups, tile_n, tmem_cols; // groups: of epilogue warps
  int o_per;                                      // staging tiles per group of epilogue warps
  int nb, cw, ks_full, ks_last;                   // channel blocks; MMA k-steps of a block and of the last one
  uint32_t rb;                                    // bytes of an input tile row
  uint32_t a_sub_bytes, a_tx; int a_slots;        // one patch's box in shared memory; bytes copied for it
  int w_resident, w_slots, w_boxes, w_nbw;        // w_nbw: columns per MN-major block
  uint32_t w_tile_bytes, w_box_bytes;
  uint32_t w_off, o_off, o_bytes;                 // shared memory behind the input ring: weights, staging tiles
  uint32_t a_hi, b_hi, b_lo0, b_step, idesc;      // descriptor words
  int ocw, co;                                    // channels per staging tile, channels of the output
  // walking along an axis (conv_slide.cuh): its extent, padding and kernel offsets; rows of offsets in the plane; images per tile; accumulators
  int extent, pad_s, ks, ki, planar, img_step, ring;
  uint32_t w_blk_bytes;                           // weights of one of the ks offsets that an MMA takes together
  unsigned int* status;
  unsigned int tag;
};

// The MMAs of one channel block: every offset, KSTEPS k-steps for each of the unit's patches (TWO: two, which share the
// weight tile).  Run by the whole warp.  Returns false if a wait ran out.  The warp issues one instruction per some six
// clocks and a narrow MMA takes 32, so its loops are unrolled over a row of offsets and step by additions only.
struct CvIssue { uint32_t d, a, w, acc, ws, w_par; };
template <int KS, int KSTEPS, bool TWO, bool RES>
__device__ __forceinline__ bool cv_block(const ConvParams& p, CvIssue& q, uint32_t w0, uint64_t* w_full, uint64_t* w_empty) {
  const uint32_t rb16 = p.rb >> 4, a_sub16 = p.a_sub_bytes >> 4, w_tile16 = p.w_tile_bytes >> 4;
  const uint32_t row16 = (uint32_t)p.P * rb16, plane_back = p.plane_rows * rb16 - KS * row16;
  const uint32_t d = q.d, tile_n = (uint32_t)p.tile_n, a_hi = p.a_hi, b_hi = p.b_hi, b_step = p.b_step, idesc = p.idesc;
  uint32_t a_lo = (1u << 16) | q.a, b_lo = p.b_lo0 | q.w, acc = q.acc;
  for (int dz = 0; dz < p.KD; ++dz) {
#pragma unroll 1
    for (int dy = 0; dy < KS; ++dy) {
#pragma unroll
      for (int dx = 0; dx < KS; ++dx) {
        if (!RES) {
          if (!mbar_wait_warp(&w_full[q.ws], q.w_par, p.status, p.tag)) return false;
          tc_fence_after();
          b_lo = p.b_lo0 | (w0 + q.ws * w_tile16);
        }
#pragma unroll
        for (int k = 0; k < KSTEPS; ++k) {                        // 16 channels = 32 bytes of a tile row
          const uint32_t a = a_lo + (uint32_t)dx * rb16 + 2 * k, b = b_lo + k * b_step;
          umma_warp(d, a, a_hi, b, b_hi, idesc, acc);
          if (TWO) umma_warp(d + tile_n, a + a_sub16, a_hi, b, b_hi, idesc, acc);
          acc = 1u;
        }
        if (RES) {
          b_lo += w_tile16;
        } else {
          umma_commit_warp(&w_empty[q.ws]);
          if (++q.ws == (uint32_t)p.w_slots) { q.ws = 0; q.w_par ^= 1u; }
        }
      }
      a_lo += row16;
    }
    a_lo += plane_back;
  }
  q.acc = 1u;
  q.w = b_lo & 0xFFFFu;
  return true;
}

struct CvBars { uint64_t *a_full, *a_empty, *w_full, *w_empty, *t_full, *t_empty; };

// The issuing warp where one channel block holds all input channels and the weights stay: one patch per unit, two
// accumulator sets, nothing to decide per unit.
template <int KS, int KSTEPS>
__device__ __forceinline__ void cv_issue_one_block(const ConvParams& p, const CvBars& bar, uint32_t units, uint32_t tmem_base,
                                                   uint32_t a0, uint32_t w0, uint32_t a_slot16) {
  CvIssue q{};
  uint32_t s = 0, a_par = 0, buf = 0, t_par = 1;        // (a wait for the phase before the first returns at once)
  q.a = a0;
  q.d = tmem_base;
  for (uint32_t left = units; left > 0; --left) {
    if (!mbar_wait_warp(&bar.t_empty[buf], t_par, p.status, p.tag)) return;
    if (!mbar_wait_warp(&bar.a_full[s], a_par, p.status, p.tag)) return;
    tc_fence_after();
    q.acc = 0;
    q.w = w0;
    cv_block<KS, KSTEPS, false, true>(p, q, w0, nullptr, nullptr);
    umma_commit_warp(&bar.a_empty[s]);
    umma_commit_warp(&bar.t_full[buf]);
    q.a += a_slot16;
    if (++s == (uint32_t)p.a_slots) { s = 0; a_par ^= 1u; q.a = a0; }
    q.d = buf ? tmem_base : tmem_base + (uint32_t)p.tile_n;
    t_par ^= buf;
    buf ^= 1u;
  }
}

// SLIDE: the layer is walked along an axis (conv_slide.cuh).
template <bool F16, int KS, bool SLIDE>
__global__ void __launch_bounds__(CV_THREADS, 1)
conv_tc_kernel(const __grid_constant__ CUtensorMap map_in, const __grid_constant__ CUtensorMap map_w,
               const __grid_constant__ CUtensorMap map_out, const __grid_constant__ ConvParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t a_full[CV_A_SLOTS], a_empty[CV_A_SLOTS];
  __shared__ __align__(8) uint64_t w_full[CV_W_SLOTS], w_empty[CV_W_SLOTS];
  constexpr int SETS = SLIDE ? CV_RING : 2;          // accumulators that change hands
  __shared__ __align__(8) uint64_t t_full[SETS], t_empty[SETS];
  __shared__ uint32_t tmem_slot;
  __shared__ int go;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  if (threadIdx.x == 0) {
    for (int s = 0; s < CV_A_SLOTS; ++s) { mbar_init(&a_full[s], 1); mbar_init(&a_empty[s], 1); }
    for (int s = 0; s < CV_W_SLOTS; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); }
    for (int b = 0; b < SETS; ++b) { mbar_init(&t_full[b], 1); mbar_init(&t_empty[b], SLIDE || p.acc_bufs == 2 ? 4 : 4 * p.groups); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    prefetch_tmap(&map_in);
    prefetch_tmap(&map_w);
    prefetch_tmap(&map_out);
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
  // this CTA's run of items (the runs differ by one item at most)
  const uint32_t i0 = (uint32_t)((unsigned long long)p.items * blockIdx.x / gridDim.x);
  const uint32_t i1 = (uint32_t)((unsigned long long)p.items * (blockIdx.x + 1) / gridDim.x);
  const uint32_t a_slot_bytes = p.a_sub_bytes * (uint32_t)p.m_sub;

  if (!go) {
    // fall through to the teardown
  } else if (SLIDE) {
    if (warp == 0) {
      if (lane == 0) sl_copy(p, &map_in, base, i0, i1, a_full, a_empty);
    } else if (warp == 2) {
      if (lane == 0 && i0 < i1) {                // all weights once: per block of channels and offset in the plane the ks offsets, the last first
        mbar_arrive_expect_tx(&w_full[0], (uint32_t)(p.nb * p.ki * KS) * p.w_tile_bytes);
        uint32_t dst = base + p.w_off;
        for (int blk = 0; blk < p.nb; ++blk)
          for (int o = 0; o < p.ki * KS; ++o)
            for (int k = p.ks - 1; k >= 0; --k) {
              const int t = k * p.ki * KS + o;
              if (!p.dgrad) tma_load_3d(dst, &map_w, blk * p.cw, t, 0, &w_full[0]);
              else
                for (int j = 0; j < p.w_boxes; ++j) tma_load_3d(dst + (uint32_t)j * p.w_box_bytes, &map_w, j * p.w_nbw, p.T - 1 - t, blk * p.cw, &w_full[0]);
              dst += p.w_blk_bytes;
            }
        mbar_wait(&w_full[0], 0, p.status, p.tag);
      }
    } else if (warp == 1) {
      if (i0 < i1 && mbar_wait_warp(&w_full[0], 0, p.status, p.tag)) {
        tc_fence_after();
        sl_issue<KS>(p, tmem_base, (base & 0x3FFFFu) >> 4, ((base + p.w_off) & 0x3FFFFu) >> 4, i0, i1,
                     SlBars{a_full, a_empty, t_full, t_empty});
      }
    } else if (warp >= 4) {
      sl_epilogue<F16>(p, &map_out, base, tmem_base, i0, i1, t_full, t_empty);
    }
  } else if (warp == 0) {
    // ------------------------------------------------------------------ input boxes
    if (lane == 0) {
      int s = 0;
      uint32_t fill = 0, cnt = 0;
      bool ok = true;
      for (CvWalk w0(p, i0, i1); w0.it < i1 && ok;) {
        const int n = w0.unit(p);
        CvWalk w1 = w0;
        if (n > 1) w1.step(p);
        for (int blk = 0; blk < p.nb; ++blk) {
          if (fill > 0) {
            ok = mbar_wait(&a_empty[s], (fill - 1) & 1u, p.status, p.tag);
            if (!ok) break;
          }
          const uint32_t dst = base + (uint32_t)s * a_slot_bytes;
          mbar_arrive_expect_tx(&a_full[s], (uint32_t)n * p.a_tx);
          tma_load_5d(dst, &map_in, blk * p.cw, w0.x - p.pad, w0.y - p.pad, w0.z - p.pad_d, w0.b, &a_full[s]);
          if (n > 1)
            tma_load_5d(dst + p.a_sub_bytes, &map_in, blk * p.cw, w1.x - p.pad, w1.y - p.pad, w1.z - p.pad_d, w1.b, &a_full[s]);
          ++cnt;
          if (++s == p.a_slots) { s = 0; ++fill; }
        }
        w0 = w1;
        w0.step(p);
      }
      // every copy issued must have landed before the CTA exits
      for (uint32_t i = cnt > (uint32_t)p.a_slots ? cnt - p.a_slots : 0; i < cnt; ++i)
        if (!mbar_wait(&a_full[i % p.a_slots], (i / p.a_slots) & 1u, p.status, p.tag)) break;
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ weights
    if (lane == 0) {
      auto fetch = [&](uint32_t dst, int blk, int t, uint32_t tn, uint64_t* bar) {
        const int n0 = (int)tn * p.tile_n;
        if (p.dgrad)
          for (int j = 0; j < p.w_boxes; ++j)
            tma_load_3d(dst + (uint32_t)j * p.w_box_bytes, &map_w, n0 + j * p.w_nbw, p.T - 1 - t, blk * p.cw, bar);
        else
          tma_load_3d(dst, &map_w, blk * p.cw, t, n0, bar);
      };
      if (p.w_resident) {                        // one column tile: all weight tiles once
        if (i0 < i1) {
          mbar_arrive_expect_tx(&w_full[0], (uint32_t)(p.nb * p.T) * p.w_tile_bytes);
          for (int blk = 0; blk < p.nb; ++blk)
            for (int t = 0; t < p.T; ++t)
              fetch(base + p.w_off + (uint32_t)(blk * p.T + t) * p.w_tile_bytes, blk, t, 0, &w_full[0]);
          mbar_wait(&w_full[0], 0, p.status, p.tag);
        }
      } else {
        int s = 0;
        uint32_t fill = 0, cnt = 0;
        bool ok = true;
        for (CvWalk w(p, i0, i1); w.it < i1 && ok;) {
          const int n = w.unit(p);
          for (int blk = 0; blk < p.nb && ok; ++blk)
            for (int t = 0; t < p.T; ++t) {
              if (fill > 0) {
                ok = mbar_wait(&w_empty[s], (fill - 1) & 1u, p.status, p.tag);
                if (!ok) break;
              }
              mbar_arrive_expect_tx(&w_full[s], p.w_tile_bytes);
              fetch(base + p.w_off + (uint32_t)s * p.w_tile_bytes, blk, t, w.tn, &w_full[s]);
              ++cnt;
              if (++s == p.w_slots) { s = 0; ++fill; }
            }
          for (int i = 0; i < n; ++i) w.step(p);
        }
        for (uint32_t i = cnt > (uint32_t)p.w_slots ? cnt - p.w_slots : 0; i < cnt; ++i)
          if (!mbar_wait(&w_full[i % p.w_slots], (i / p.w_slots) & 1u, p.status, p.tag)) break;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the whole warp)
    const uint32_t a_slot16 = a_slot_bytes >> 4;
    const uint32_t a0 = (base & 0x3FFFFu) >> 4, w0 = ((base + p.w_off) & 0x3FFFFu) >> 4;
    const uint32_t set_cols = (uint32_t)(p.tile_n * p.m_sub);
    bool ok = true;
    if (p.w_resident && i0 < i1) { ok = mbar_wait_warp(&w_full[0], 0, p.status, p.tag); tc_fence_after(); }
    if (p.w_resident && p.nb == 1) {              // (one column tile, one patch per unit, two accumulator sets)
      const CvBars bar{a_full, a_empty, w_full, w_empty, t_full, t_empty};
      const uint32_t units = ok ? i1 - i0 : 0;
      switch (p.ks_last) {
        case 1: cv_issue_one_block<KS, 1>(p, bar, units, tmem_base, a0, w0, a_slot16); break;
        case 2: cv_issue_one_block<KS, 2>(p, bar, units, tmem_base, a0, w0, a_slot16); break;
        case 3: cv_issue_one_block<KS, 3>(p, bar, units, tmem_base, a0, w0, a_slot16); break;
        default: cv_issue_one_block<KS, 4>(p, bar, units, tmem_base, a0, w0, a_slot16);
      }
    } else {
      CvIssue q{};
      uint32_t s = 0, a_par = 0, lu = 0;
      uint32_t in_tile = i0 < i1 ? p.patches - i0 % p.patches : 0;      // items left in this column tile
      for (uint32_t left = i1 - i0; left > 0 && ok; ++lu) {
        const uint32_t n = min((uint32_t)p.m_sub, min(left, in_tile));
        const uint32_t buf = p.acc_bufs == 2 ? lu & 1u : 0u, use = p.acc_bufs == 2 ? lu >> 1 : lu;
        if (use > 0) {
          ok = mbar_wait_warp(&t_empty[buf], (use - 1) & 1u, p.status, p.tag);
          if (!ok) break;
          tc_fence_after();
        }
        q.d = tmem_base + buf * set_cols;
        q.acc = 0;
        q.w = w0;
        for (int blk = 0; blk < p.nb; ++blk) {
          ok = mbar_wait_warp(&a_full[s], a_par, p.status, p.tag);
          if (!ok) break;
          tc_fence_after();
          q.a = a0 + s * a_slot16;
          const int shape = (blk == p.nb - 1 ? p.ks_last : p.ks_full) * 4 + (n > 1 ? 2 : 0) + p.w_resident;
#define XC_BLOCK(KT, TWO, RES) case KT * 4 + TWO * 2 + RES: ok = cv_block<KS, KT, TWO != 0, RES != 0>(p, q, w0, w_full, w_empty); break;
#define XC_BLOCKS(KT) XC_BLOCK(KT, 0, 0) XC_BLOCK(KT, 0, 1) XC_BLOCK(KT, 1, 0)
          switch (shape) { XC_BLOCKS(1) XC_BLOCKS(2) XC_BLOCKS(3) XC_BLOCKS(4) }
#undef XC_BLOCKS
#undef XC_BLOCK
          if (!ok) break;
          umma_commit_warp(&a_empty[s]);
          if (++s == (uint32_t)p.a_slots) { s = 0; a_par ^= 1u; }
        }
        if (ok) umma_commit_warp(&t_full[buf]);
        left -= n;
        in_tile -= n;
        if (in_tile == 0) in_tile = p.patches;
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ epilogue
    const int quad = warp & 3, group = (warp - 4) >> 2;
    const uint32_t set_cols = (uint32_t)(p.tile_n * p.m_sub);
    const EpiPixel px(p, quad * 32 + lane);                               // this thread's pixel
    const bool leader = quad == 0 && lane == 0;
    uint32_t lu = 0, ob = 0;                                              // ob: which of the group's staging tiles
    for (CvWalk w(p, i0, i1); w.it < i1; ++lu) {
      const int n = w.unit(p);
      const uint32_t buf = p.acc_bufs == 2 ? lu & 1u : 0u, use = p.acc_bufs == 2 ? lu >> 1 : lu;
      if (p.acc_bufs == 2 && p.groups == 2 && buf != (uint32_t)group) {                    // the other group's unit
        for (int i = 0; i < n; ++i) w.step(p);
        continue;
      }
      bool ok = true;
      if (lane == 0) ok = mbar_wait(&t_full[buf], use & 1u, p.status, p.tag);
      if (!epi_all(group, ok)) break;                                     // the four warps leave together
      tc_fence_after();
      const int n0 = (int)w.tn * p.tile_n, cols = min(p.tile_n, p.co - n0);
      const bool share = p.acc_bufs == 1 && p.groups == 2;
      const int last = share ? group : n - 1;                             // this group's last patch of the unit
      for (int sub = 0; sub < n; ++sub, w.step(p)) {
        if (share && sub != group) continue;
        for (int c = 0; c < cols; c += p.ocw) {
          const uint32_t tile = base + p.o_off + ((uint32_t)(group * p.o_per) + ob) * p.o_bytes;
          if (leader) { if (p.o_per == 1) bulk_wait_read<0>(); else bulk_wait_read<1>(); }     // the tile's last store has read it
          epi_sync(group);
          epi_row<F16>(p, px, tile, tmem_base + ((uint32_t)(quad * 32) << 16) + buf * set_cols + (uint32_t)(sub * p.tile_n + c), p.tile_n - c);
          if (sub == last && c + p.ocw >= cols) {                         // this group has read what it reads of the set
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&t_empty[buf]);
          }
          fence_async_smem();
          epi_sync(group);
          if (leader) {
            tma_store_5d(&map_out, tile, n0 + c, w.x, w.y, w.z, w.b);
            bulk_commit();
          }
          if (p.o_per == 2) ob ^= 1u;
        }
      }
      if (last >= n) {                                                    // one accumulator set, a unit of one patch
        __syncwarp();
        if (lane == 0) mbar_arrive(&t_empty[buf]);
      }
    }
    if (leader) bulk_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// ------------------------------------------------------------------------------------ host side

static uint32_t align1k(uint32_t v) { return (v + 1023u) & ~1023u; }
static CUtensorMapSwizzle swizzle_of(int row_elems) {
  return row_elems == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : row_elems == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}
static uint32_t layout_of(int row_elems) { return row_elems == 64 ? 2u : row_elems == 32 ? 4u : 6u; }
static int block_width(int c) { return c > 32 ? 64 : c > 16 ? 32 : 16; }

// The plan of conv_slide.cuh and the clocks of its busiest CTA, as measured: the MMAs of a plane hold the pipe N/2 clocks each or as long as their operands take
// from shared memory, or the warp that issues them some 45 and 230 a plane; the planes at the ends of a CTA's segments and where the ring of accumulators
// ends take 750 and 105 an MMA; an epilogue warp waits some 250 clocks for its turn beside what its columns take, and there are two groups.
static long plan_slide(const xconv_desc* d, bool dgrad, TcConvPlan* p) {
  const int Ci = dgrad ? d->Cout : d->Cin, Co = dgrad ? d->Cin : d->Cout;
  const ConvGeo g = conv_geo(d);
  const int K = d->KH, ks = K, planar = d->KD > 1 ? 0 : 1, ki = planar ? 1 : K;
  if (K < 3) return -1;
  const long extent = planar ? g.H : g.D;
  const int nbw = dgrad ? (Co % 64 == 0 ? 64 : 32) : 16, tile_n = round_up(Co, nbw), ocw = block_width(Co);
  if (ks * tile_n > 256) return -1;
  const int ring = std::min(CV_RING, 512 / tile_n);
  const uint32_t budget = SMEM_LIMIT - 4096;
  long best = -1;
  for (int cw = block_width(Ci); cw >= 16 && best < 0; cw /= 2) {      // (narrower blocks only where no plan fits)
    const int nb = (int)cdivl(Ci, cw), ksteps = (nb - 1) * (cw / 16) + (int)cdivl(Ci - (nb - 1) * cw, 16);
    const uint32_t rb = 2 * (uint32_t)cw;
    const long w_bytes = (long)nb * ki * K * ks * tile_n * rb;
    for (long nx = cdivl(g.W, 128); nx <= std::max(cdivl(g.W, 128), std::min(32L, g.W)); ++nx) {
      const int pw = (int)cdivl(g.W, nx), P = pw + K - 1;
      if (P > 256) continue;
      const long across = planar ? g.B : g.H;                       // what a tile takes several rows of: images or rows
      const int ph_max = (int)std::min<long>(across, (128 - pw) / P + 1), ph = (int)cdivl(across, cdivl(across, ph_max));
      const int box_rows = P * (planar ? ph : ph + K - 1), need_rows = (ki - 1) * P + K - 1 + TILE_M;
      const uint32_t a_sub = align1k((uint32_t)std::max(box_rows, need_rows) * rb), o_bytes = align1k((uint32_t)(pw * ph) * 2 * ocw);
      const long room = (long)budget - w_bytes - 1024 - 2L * o_bytes;
      if (room < 2L * a_sub) continue;
      const int o_per = room >= 4L * a_sub + 2L * o_bytes ? 2 : 1;
      const int a_slots = (int)std::min<long>(CV_A_SLOTS, (room - (o_per - 1) * 2L * o_bytes) / a_sub);
      const long columns = cdivl(g.W, pw) * cdivl(across, ph) * (planar ? 1 : g.B), items = columns * extent;
      if (items >= (1L << 31)) continue;
      const long per_cta = cdivl(items, std::min<long>(items, NUM_SMS));
      const long segments = per_cta >= extent ? cdivl(per_cta, extent) : (extent % per_cta ? 2 : 1), planes = per_cta + (ks - 1) * std::min(2L, segments);
      const long products = (long)ki * K * ksteps + 1, pipe = std::max({62, ks * tile_n / 2, 40 + ks * tile_n / 4});
      const long bytes = (long)nb * box_rows * rb, copy = std::max(bytes / 45, bytes * 2200 / ((long)a_slots * a_sub));
      const long odd = std::min(planes, nb > 1 ? planes : 2 * (ks - 1) * segments + per_cta * (ks - 1) / ring);      // planes that are not like the one before
      const long inner = std::max({230 + 45 * products, products * pipe, copy, (250 + 7L * tile_n) / 2}), other = 750 + 500 * (nb - 1) + products * std::max(105L, pipe);
      const long cost = (planes - odd) * inner + odd * std::max(other, copy) + w_bytes / 45;
      if (best >= 0 && cost >= best) continue;
      best = cost;
      p->slide = 1; p->ring = ring;
      p->cw = cw; p->m_sub = 1; p->tile_n = tile_n; p->tiles_n = 1; p->acc_bufs = 2; p->patch_w = pw; p->patch_h = ph;
      p->resident = 1; p->w_slots = 0; p->groups = 2; p->nbw = nbw; p->ocw = ocw; p->patches = items; p->o_per = o_per; p->a_slots = a_slots; p->a_sub_bytes = a_sub;
    }
  }
  return best;
}

// Picks patch, column tile, patches per weight tile and the place of the weights by the time a CTA would take, in
// clocks: the MMAs (a k-step of N columns holds the pipe N/2 clocks, and at least the 34 it takes to read its A tile),
// or the copies where they take longer (an SM pulls about 45 bytes per clock from L2), times the items of the busiest CTA.
bool tc_plan_conv(const xconv_desc* d, bool dgrad, TcConvPlan* p) {
  if (d->dtype != XCONV_BF16 && d->dtype != XCONV_F16) return false;
  const int Ci = dgrad ? d->Cout : d->Cin, Co = dgrad ? d->Cin : d->Cout;
  if (Ci % 8 != 0 || Co % 8 != 0 || d->circular) return false;      // circular padding: FP32-FMA kernels
  const ConvGeo g = conv_geo(d);
  if (g.W >= (1L << 31) || g.B >= (1L << 31)) return false;
  const int K = d->KH, KD = d->KD > 1 ? d->KD : 1, T = KD * K * K;
  const uint32_t budget = SMEM_LIMIT - 4096;
  long best = -1, real = 0;
  for (int cw = block_width(Ci); cw >= 16 && best < 0; cw /= 2) {   // (narrower blocks only where no plan fits)
    const int nb = (int)cdivl(Ci, cw), ks_last = (int)cdivl(Ci - (nb - 1) * cw, 16), ksteps = (nb - 1) * (cw / 16) + ks_last;
    const uint32_t rb = 2 * (uint32_t)cw;
    const int nbw = dgrad ? (Co % 64 == 0 ? 64 : 32) : 16;          // dX: the weight tile comes in blocks of nbw columns
    const int n_full = std::min(256, round_up(Co, nbw)), ocw = block_width(std::min(Co, n_full));
    for (int variant = 0; variant < 4; ++variant) {
      const int m_sub = 1 + (variant & 1), tile_n = variant & 2 ? 128 : n_full;
      if ((variant & 2) && n_full <= 128) break;
      if (m_sub * tile_n > 512) continue;
      const int tiles_n = (int)cdivl(Co, tile_n), acc_bufs = 2 * m_sub * tile_n <= 512 ? 2 : 1;
      const uint32_t w_tile = (uint32_t)tile_n * rb;
      const uint32_t w_all = align1k((uint32_t)std::min(1L << 20, (long)nb * T * w_tile));
      for (long nx = cdivl(g.W, 128); nx <= std::max(cdivl(g.W, 128), std::min(32L, g.W)); ++nx) {
        const int pw = (int)cdivl(g.W, nx), P = pw + K - 1;
        if (P > 256) continue;
        const int ph_max = (int)std::min<long>(g.H, (128 - pw) / P + 1);
        const int ph = (int)cdivl(g.H, cdivl(g.H, ph_max));
        const uint32_t plane_rows = (uint32_t)(P * (ph + K - 1)), box_rows = plane_rows * KD;
        const uint32_t need_rows = (uint32_t)((KD - 1) * plane_rows + (K - 1) * P + (K - 1) + TILE_M);
        const uint32_t a_sub = align1k(std::max(box_rows, need_rows) * rb), a_slot = a_sub * m_sub;
        const uint32_t o_bytes = align1k((uint32_t)(pw * ph) * 2 * ocw);
        if (a_slot * 2 + o_bytes * 2 > budget) continue;
        const uint32_t room = budget - 2 * a_slot - 2 * o_bytes;
        const bool resident = tiles_n == 1 && w_all <= room;
        if (!resident && room < 3 * w_tile) continue;
        if (resident && m_sub == 2) continue;                       // nothing to share
        const long patches = cdivl(g.W, pw) * cdivl(g.H, ph) * g.D * g.B, items = patches * tiles_n;
        if (items >= (1L << 32) - 1) continue;
        const long per_cta = cdivl(items, std::min<long>(items, NUM_SMS));
        const long mma = (long)T * ksteps * std::max(34, tile_n / 2);
        const long copy = ((long)box_rows * rb * nb + (resident ? 0 : (long)nb * T * w_tile / m_sub)) / 45;
        const long epi = 200 + 6L * tile_n;                         // one patch through the epilogue
        const long cost = per_cta * (std::max(std::max(mma, copy), epi) + (acc_bufs == 1 ? epi : 0)) +
                          (resident ? (long)w_all / 45 : 0);
        if (best >= 0 && cost >= best) continue;
        best = cost;
        p->cw = cw; p->m_sub = m_sub; p->tile_n = tile_n; p->tiles_n = tiles_n; p->acc_bufs = acc_bufs;
        p->patch_w = pw; p->patch_h = ph; p->resident = resident ? 1 : 0; p->groups = resident || acc_bufs == 1 ? 2 : 1; p->nbw = nbw; p->ocw = ocw;
        p->patches = patches;
        p->o_per = p->groups == 1 ? 2 : 1;
        if (resident) {
          // Two more staging tiles where they fit beside four input boxes: with one, a group waits for its last store to have read it
          // before every tile (1 x 1, 64 -> 256 channels, 64 images of 56 x 56 28.5 -> 25.6 us, 24 -> 160, 3 x 3 122 -> 105 with the
          // sketch; in the place of boxes 256 -> 192 channels, 1 x 1 53.4 -> 55.9).
          p->w_slots = 0;
          if (room - w_all >= 2 * o_bytes + 2 * a_slot) p->o_per = 2;
          // Long runs of patches get as many boxes in flight as fit: four narrow ones leave the copies waiting for memory (1 x 1, 192 -> 24 channels,
          // 46 images of 129 x 129 75.9 -> 66.1 us, dX of 96 -> 16, 3 x 3, 16 of 188 x 256 46.9 -> 42.3; with runs of six 11.6 -> 12.0;
          // 1 x 1 with more channels out than in is bound by its stores: 128 -> 192, 102 of 59 x 59 40.2 -> 41.3; with as many, 18 convolutions of
          // 16 to 256, 1.006 of the time: dX of 96, 64 of 97 x 97 47.4 -> 42.2, but of 64, 300 of 90 x 90 101 -> 118).
          p->a_slots = (int)std::min<uint32_t>(per_cta >= 16 && (K > 1 || Ci > Co) ? CV_A_SLOTS : 4, 2 + (room - w_all - (p->o_per == 2 ? 2 * o_bytes : 0)) / a_slot);
        } else {
          p->a_slots = room >= a_slot + 4 * w_tile ? 3 : 2;
          p->w_slots = (int)std::min<uint32_t>(CV_W_SLOTS, (budget - (uint32_t)p->a_slots * a_slot - 2 * o_bytes) / w_tile);
        }
        p->a_sub_bytes = a_sub;
        p->slide = 0;
        // ... and what its patches take as measured: an MMA 56 clocks at least, 250 from one patch to the next, a ring of weight tiles hands on as many as
        // it holds in the time of one copy, and a box of one plane comes in at 5 clocks a pixel however narrow its rows are (16 -> 16 channels, 3 x 3, 25 images of
        // 154 x 154: walked 20.7 us where it was taken for slower than patches at 23.8, 64 of 95 x 157 36.8 -> 32.2)
        const long turns = std::max({(long)T * ksteps * m_sub * std::max(56, tile_n / 2) + 250, KD == 1 ? 5L * nb * m_sub * box_rows : 0, resident ? 0 : (long)nb * T * 2200 / p->w_slots, m_sub * copy, m_sub * epi});
        real = cdivl(per_cta, m_sub) * turns + (resident ? (long)w_all / 45 : 0);
      }
    }
  }
  // Both counts leave out the same 5 us of launch, first copies and last stores, and the walk's last planes complete several outputs at once: it is taken
  // for a tenth and 2000 clocks less, or where the weights would be streamed.  (Of 104 convolutions with at most 64 channels on one side 14 are walked,
  // 0.39 to 0.95 of the time; without the 2000 clocks also 5 x 5, 8 -> 16 channels of 4 images of 224 x 224, 20.2 -> 22.6 us.)
  TcConvPlan slide{};
  const long sliding = best >= 0 && real < 8000 ? -1 : plan_slide(d, dgrad, &slide);      // (a walk takes that much for its first and last planes)
  if (sliding >= 0 && (best < 0 || sliding + 2000 < (p->resident ? real - real / 10 : real))) { *p = slide; return true; }
  return best >= 0;
}

xconv_status tc_run_conv(const xconv_desc* d, const TcConvPlan& pl, bool dgrad, const void* in, const void* W,
                         void* out, char* ws_head, cudaStream_t st) {
  const int K = d->KH, KD = d->KD > 1 ? d->KD : 1, T = KD * K * K;
  const int Ci = dgrad ? d->Cout : d->Cin, Co = dgrad ? d->Cin : d->Cout;
  const bool f16 = d->dtype == XCONV_F16;
  const ConvGeo g = conv_geo(d);
  ConvParams p{};
  p.KD = KD; p.T = T; p.pad = (K - 1) / 2; p.pad_d = (KD - 1) / 2; p.dgrad = dgrad ? 1 : 0;
  p.pw = pl.patch_w; p.ph = pl.patch_h; p.P = pl.patch_w + K - 1;
  p.patches_x = (int)cdivl(g.W, p.pw); p.patches_y = (int)cdivl(g.H, p.ph); p.depth = (int)g.D;
  if (pl.slide) {
    p.planar = KD == 1 ? 1 : 0;
    p.ks = K; p.ki = p.planar ? 1 : K; p.pad_s = (K - 1) / 2; p.ring = pl.ring;
    p.extent = (int)(p.planar ? g.H : g.D); p.img_step = p.planar ? p.ph : 1;
    if (p.planar) p.patches_y = 1;
  }
  p.patches = (uint32_t)pl.patches; p.items = (uint32_t)(pl.patches * pl.tiles_n);
  p.plane_rows = (uint32_t)(p.P * (p.ph + K - 1));
  p.m_sub = pl.m_sub; p.acc_bufs = pl.acc_bufs; p.groups = pl.groups; p.tile_n = pl.tile_n;
  p.o_per = pl.o_per;
  p.tmem_cols = pow2_cols(pl.slide ? pl.ring * pl.tile_n : pl.acc_bufs * pl.m_sub * pl.tile_n);
  p.cw = pl.cw; p.nb = (int)cdivl(Ci, pl.cw); p.ks_full = pl.cw / 16; p.ks_last = (int)cdivl(Ci - (p.nb - 1) * pl.cw, 16);
  p.rb = 2 * (uint32_t)pl.cw;
  p.a_sub_bytes = pl.a_sub_bytes; p.a_tx = p.plane_rows * KD * p.rb; p.a_slots = pl.a_slots;
  p.w_resident = pl.resident; p.w_slots = pl.w_slots; p.w_nbw = pl.nbw;
  p.w_tile_bytes = (uint32_t)pl.tile_n * p.rb;
  p.w_boxes = dgrad ? pl.tile_n / pl.nbw : 1;
  p.w_box_bytes = p.w_tile_bytes / (uint32_t)p.w_boxes;
  p.w_blk_bytes = p.w_tile_bytes;
  if (pl.slide) {                                // a tile: the weights of the axis' ks offsets
    p.w_tile_bytes *= (uint32_t)p.ks;
    p.a_tx = (uint32_t)(p.P * (p.planar ? p.ph : p.ph + K - 1)) * p.rb;
  }
  p.w_off = (uint32_t)(pl.a_slots * pl.m_sub) * pl.a_sub_bytes;
  p.o_off = align1k(p.w_off + (uint32_t)(pl.resident ? p.nb * T : pl.w_slots) * p.w_blk_bytes);
  p.ocw = pl.ocw; p.co = Co;
  p.o_bytes = align1k((uint32_t)(p.pw * p.ph * 2 * pl.ocw));
  p.a_hi = ((8 * p.rb) >> 4) | (1u << 14) | (layout_of(pl.cw) << 29);
  if (dgrad) {                                   // MN-major weight tile: rows = the reduction index, blocks of nbw columns
    const uint32_t nrb = 2 * (uint32_t)pl.nbw;
    p.b_hi = ((8 * nrb) >> 4) | (1u << 14) | (layout_of(pl.nbw) << 29);
    p.b_lo0 = (p.w_box_bytes >> 4) << 16;
    p.b_step = (16 * nrb) >> 4;
  } else {
    p.b_hi = p.a_hi;
    p.b_lo0 = 1u << 16;
    p.b_step = 2;
  }
  p.idesc = (1u << 4) | (f16 ? 0u : (1u << 7) | (1u << 10)) | (dgrad ? 1u << 16 : 0u) | (pl.slide ? 0u : (uint32_t)(pl.tile_n >> 3) << 17) |
            ((uint32_t)(TILE_M >> 4) << 24);
  p.status = reinterpret_cast<unsigned int*>(ws_head);
  p.tag = call_tag();

  CUtensorMap mi, mw, mo;
  auto image_map = [&](CUtensorMap* m, const void* ptr, int C, int cb, int bw, int bh, int bd, int bb) {
    const uint64_t dims[5] = {(uint64_t)C, (uint64_t)g.W, (uint64_t)g.H, (uint64_t)g.D, (uint64_t)g.B};
    const uint64_t row = (uint64_t)C * 2;
    const uint64_t str[4] = {row, row * g.W, row * g.W * g.H, row * g.W * g.H * g.D};
    const uint32_t box[5] = {(uint32_t)cb, (uint32_t)bw, (uint32_t)bh, (uint32_t)bd, (uint32_t)bb};
    return make_map(m, ptr, 5, dims, str, box, f16, swizzle_of(cb));
  };
  const uint64_t dw[3] = {(uint64_t)d->Cin, (uint64_t)T, (uint64_t)d->Cout};
  const uint64_t sw[2] = {(uint64_t)d->Cin * 2, (uint64_t)T * d->Cin * 2};
  const uint32_t bw[3] = {(uint32_t)(dgrad ? pl.nbw : pl.cw), 1, (uint32_t)(dgrad ? pl.cw : pl.tile_n)};
  const bool rows = pl.slide && p.planar;        // a tile's rows are of several images
  if (!image_map(&mi, in, Ci, pl.cw, p.P, rows ? 1 : p.ph + K - 1, pl.slide ? 1 : KD, rows ? p.ph : 1) ||
      !image_map(&mo, out, Co, pl.ocw, p.pw, rows ? 1 : p.ph, 1, rows ? p.ph : 1) ||
      !make_map(&mw, W, 3, dw, sw, bw, f16, swizzle_of(dgrad ? pl.nbw : pl.cw)))
    return XCONV_ERR_CUDA;
  const size_t smem = 1024 + (size_t)p.o_off + (size_t)(p.groups * p.o_per) * p.o_bytes;
  if (smem > (size_t)(SMEM_LIMIT - 1024)) return XCONV_ERR_UNSUPPORTED;
  const unsigned grid = std::min<uint32_t>(p.items, NUM_SMS);
  void (*kernel)(CUtensorMap, CUtensorMap, CUtensorMap, ConvParams) =
      K == 1 ? (f16 ? conv_tc_kernel<true, 1, false> : conv_tc_kernel<false, 1, false>)
      : pl.slide ? (K == 3 ? (f16 ? conv_tc_kernel<true, 3, true> : conv_tc_kernel<false, 3, true>)
                           : (f16 ? conv_tc_kernel<true, 5, true> : conv_tc_kernel<false, 5, true>))
      : K == 3 ? (f16 ? conv_tc_kernel<true, 3, false> : conv_tc_kernel<false, 3, false>)
               : (f16 ? conv_tc_kernel<true, 5, false> : conv_tc_kernel<false, 5, false>);
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT - 1024);
  if (e == cudaSuccess)
    e = launch_pdl(kernel, dim3(grid), dim3(128 + 128 * p.groups), smem_of_grid(smem, grid), st, mi, mw, mo, p);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

}  // namespace xconv
