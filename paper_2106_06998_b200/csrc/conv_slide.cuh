// The exact convolutions of layers with few channels out (conv_tc.cu), along one axis of the image.
//
// An MMA needs shared memory for 32 clocks and a quarter of its columns to be handed 128 rows of the input (40 clocks for 32 columns, 56 for 96), and one follows
// another no sooner than some 56 to 62 clocks in the kernels measured here, whatever its width up to 96.  So one MMA here serves the KS kernel offsets along one axis, the image
// rows (planar layers) or the planes (3 x 3 x 3 kernels): the input plane s, moved by one of the other offsets, is multiplied with the weights of
// all KS offsets side by side, and the sums go to the KS outputs s - pad .. s + pad, whose accumulators lie side by side in tensor memory:
//
//   D[pixel, (s', co)] += sum over ci of In_s[pixel + (dy, dx), ci] * w(co, ci, (s - s' + pad, dy, dx)),   s' = s - pad .. s + pad
//
// A CTA walks along the axis; every input plane is copied once and used for all its offsets, an output is complete with the last plane that
// reaches it.  The accumulators are a ring of as many outputs as tensor memory holds, so the MMAs run ahead of the epilogue; where the ring's end
// lies between the outputs an MMA is done in two, and so is the first one of a plane, which starts the newest output's sum instead of adding
// to it.  A planar layer's tile has no halo along the axis and takes rows of several images where one is shorter than 128 pixels.
//
// What bounds it (tensor pipe active 0.25 on 256 x 256, 0.32 in volumes; memory at 0.4 and 0.1 of its rate): 3 x 3 kernels of 32 channels the issuing warp (some 230 clocks a plane beside 45 an MMA), volumes and wider layers the pipe (62 clocks an MMA
// of 96 columns, 96 one of 192).  us a launch, one MMA per offset -> this: 16 images of 256 x 256, 32 -> 32 channels 42.2 -> 33.4; 4 volumes of 48^3,
// 32 -> 32 46.2 -> 36.5; 208 images of 123 x 126, 16 -> 24 108 -> 82; 5 x 5, 375 of 97 x 97, 32 -> 16 328 -> 208; 5 volumes of 22 x 34 x 34, 96 -> 24 (weights kept
// here, streamed there) 153 -> 60.
#pragma once

#include "tc_api.h"
#include "tc_ptx.cuh"

namespace xconv {

// The 128 threads of one group of epilogue warps: true if `ok` holds in every one of them.
__device__ __forceinline__ bool epi_all(int group, bool ok) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, %2, 128, p;\n\t"
               "selp.b32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"(ok ? 1u : 0u), "r"(1 + group) : "memory");
  return r != 0;
}
__device__ __forceinline__ void epi_sync(int group) { asm volatile("barrier.cta.sync %0, 128;" ::"r"(1 + group) : "memory"); }

// The pixel of the patch that an epilogue thread writes: the accumulator's row m is position m of the box.
struct EpiPixel {
  bool live;
  uint32_t v, swz;                  // pixel of the patch; swizzle of its row in a staging tile
  template <class Params>
  __device__ __forceinline__ EpiPixel(const Params& p, int m) {
    const int my = m / p.P, mx = m - my * p.P;
    live = mx < p.pw && my < p.ph;
    v = (uint32_t)(my * p.pw + mx);
    swz = p.ocw == 64 ? v & 7u : p.ocw == 32 ? (v >> 1) & 3u : (v >> 2) & 1u;
  }
};
// Up to ocw columns of an accumulator (`left` of them there are) to the pixel's row of a staging tile, rounded to storage.
template <bool F16, class Params>
__device__ __forceinline__ void epi_row(const Params& p, const EpiPixel& px, uint32_t tile, uint32_t taddr, int left) {
  const uint32_t row = tile + px.v * (uint32_t)p.ocw * 2;
  for (int h = 0; h < p.ocw && h < left; h += 32) {
    uint32_t r[32];
    if (left - h >= 32) tmem_ld32(taddr + (uint32_t)h, r);
    else tmem_ld16(taddr + (uint32_t)h, r);
    const int n16 = min(32, min(p.ocw, left) - h) >> 3;   // 16-byte pieces
    if (px.live) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (i >= n16) break;
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row + ((((uint32_t)(h >> 3) + i) ^ px.swz) << 4)),
                     "r"(pack2(r[8 * i + 0], r[8 * i + 1], F16)), "r"(pack2(r[8 * i + 2], r[8 * i + 3], F16)),
                     "r"(pack2(r[8 * i + 4], r[8 * i + 5], F16)), "r"(pack2(r[8 * i + 6], r[8 * i + 7], F16)) : "memory");
      }
    }
  }
}

// A walk over a CTA's run of outputs: the column (a patch of pixels of one or several images) and the position along the axis.
struct SlWalk {
  uint32_t it;
  int s, x, y, b;
  template <class Params>
  __device__ __forceinline__ SlWalk(const Params& p, uint32_t i0) : it(i0) {
    const uint32_t col = i0 / (uint32_t)p.extent, row = col / (uint32_t)p.patches_x, grp = row / (uint32_t)p.patches_y;
    s = (int)(i0 - col * (uint32_t)p.extent);
    x = (int)(col - row * (uint32_t)p.patches_x) * p.pw;
    y = (int)(row - grp * (uint32_t)p.patches_y) * p.ph;
    b = (int)grp * p.img_step;
  }
  // the next column (the walk stands at its first position then)
  template <class Params>
  __device__ __forceinline__ void next_column(const Params& p) {
    s = 0;
    x += p.pw;
    if (x < p.patches_x * p.pw) return;
    x = 0; y += p.ph;
    if (y < p.patches_y * p.ph) return;
    y = 0; b += p.img_step;
  }
  template <class Params>
  __device__ __forceinline__ void step(const Params& p) {
    ++it;
    if (++s == p.extent) next_column(p);
  }
};

// The outputs of one column that a CTA computes, and the input planes they need.
struct SlSegment {
  int s0, s1, first, last;          // outputs s0 .. s1-1, planes first .. last
  template <class Params>
  __device__ __forceinline__ SlSegment(const Params& p, const SlWalk& w, uint32_t i1) {
    s0 = w.s;
    s1 = (int)min((uint32_t)p.extent, (uint32_t)w.s + (i1 - w.it));
    first = max(0, s0 - p.pad_s);
    last = min(p.extent - 1, s1 - 1 + p.pad_s);
  }
};

// Input planes, one box per block of channels.  One thread.
template <class Params>
__device__ __forceinline__ void sl_copy(const Params& p, const CUtensorMap* map_in, uint32_t base, uint32_t i0, uint32_t i1, uint64_t* a_full, uint64_t* a_empty) {
  int s = 0;
  uint32_t fill = 0, cnt = 0;
  bool ok = true;
  for (SlWalk w(p, i0); w.it < i1 && ok;) {
    const SlSegment g(p, w, i1);
    for (int si = g.first; si <= g.last && ok; ++si)
      for (int blk = 0; blk < p.nb; ++blk) {
        if (fill > 0) {
          ok = mbar_wait(&a_empty[s], (fill - 1) & 1u, p.status, p.tag);
          if (!ok) break;
        }
        mbar_arrive_expect_tx(&a_full[s], p.a_tx);
        tma_load_5d(base + (uint32_t)s * p.a_sub_bytes, map_in, blk * p.cw, w.x - p.pad, p.planar ? si : w.y - p.pad, p.planar ? 0 : si, w.b, &a_full[s]);
        ++cnt;
        if (++s == p.a_slots) { s = 0; ++fill; }
      }
    w.it += (uint32_t)(g.s1 - g.s0);
    w.s = g.s1;
    if (w.s == p.extent) w.next_column(p);
  }
  for (uint32_t i = cnt > (uint32_t)p.a_slots ? cnt - p.a_slots : 0; i < cnt; ++i)      // every copy issued must have landed before the CTA exits
    if (!mbar_wait(&a_full[i % p.a_slots], (i / p.a_slots) & 1u, p.status, p.tag)) break;
}

// The products of one plane and its only block of channels for K accumulators side by side, but for those of the first offset and k-step.
template <int K, int KSTEPS, class Params>
__device__ __forceinline__ void sl_products(const Params& p, uint32_t d, uint32_t idesc, uint32_t a_lo, uint32_t b_lo) {
  const uint32_t rb16 = p.rb >> 4, row16 = (uint32_t)p.P * rb16, a_hi = p.a_hi, b_hi = p.b_hi, b_step = p.b_step, tile16 = p.w_tile_bytes >> 4;
  bool first = true;
#pragma unroll 1
  for (int dy = 0; dy < p.ki; ++dy) {
#pragma unroll
    for (int dx = 0; dx < K; ++dx) {
#pragma unroll
      for (int k = 0; k < KSTEPS; ++k) {                        // 16 channels = 32 bytes of a tile row
        if (dx == 0 && k == 0 && first) { first = false; continue; }
        umma_warp(d, a_lo + (uint32_t)dx * rb16 + 2 * k, a_hi, b_lo + k * b_step, b_hi, idesc, 1u);
      }
      b_lo += tile16;
    }
    a_lo += row16;
  }
}

// What the issuing warp carries from plane to plane.
struct SlState {
  uint32_t s, a_par;                 // input box and its phase
  uint32_t slot, used;               // accumulator of the lowest output that the plane reaches; a bit per slot that flips with each output it takes
};
struct SlBars { uint64_t *a_full, *a_empty, *t_full, *t_empty; };

// One plane, whatever it reaches: n outputs from q.slot on, those from `fresh` on with their first product; the weights of the lowest one at block
// first_block of a tile (the largest offset first).  `done` of them get no more.  False if a wait ran out.
template <int K, class Params>
__device__ __forceinline__ bool sl_plane(const Params& p, SlState& q, uint32_t tmem_base, uint32_t a0, uint32_t w0, uint32_t n, uint32_t fresh, uint32_t first_block, uint32_t done,
                                         const SlBars& bar) {
  const uint32_t ring = (uint32_t)p.ring, tile_n = (uint32_t)p.tile_n, idesc_n = (tile_n >> 3) << 17, blk16 = p.w_blk_bytes >> 4, slot = q.slot;
  const uint32_t before = min(n, ring - slot), b0 = first_block * blk16;
#pragma unroll 1
  for (uint32_t i = fresh; i < n; ++i) {
    const uint32_t t = i < before ? slot + i : slot + i - ring;
    if (!mbar_wait_warp(&bar.t_empty[t], ((q.used >> t) & 1u) ^ 1u, p.status, p.tag)) return false;
    q.used ^= 1u << t;
  }
  // the accumulators up to the ring's end, and those from its start
  const uint32_t d_lower = tmem_base + slot * tile_n, idesc_lower = p.idesc + before * idesc_n, idesc_upper = p.idesc + (n - before) * idesc_n, b_upper = before * blk16;
#pragma unroll 1
  for (int blk = 0; blk < p.nb; ++blk) {
    if (!mbar_wait_warp(&bar.a_full[q.s], q.a_par, p.status, p.tag)) return false;
    tc_fence_after();
    const uint32_t a = a0 + q.s * (p.a_sub_bytes >> 4), wt = w0 + (uint32_t)(blk * p.ki * K) * (p.w_tile_bytes >> 4);
    if (blk == 0) {                                   // the first product, in parts that start sums and parts that add to them
      const uint32_t c1 = min(fresh, before), c2 = max(fresh, before);
      auto part = [&](uint32_t i, uint32_t e) {
        if (i < e)
          umma_warp(tmem_base + (i < before ? slot + i : slot + i - ring) * tile_n, (1u << 16) | a, p.a_hi, (p.b_lo0 | wt) + b0 + i * blk16, p.b_hi,
                    p.idesc + (e - i) * idesc_n, i < fresh ? 1u : 0u);
      };
      part(0, c1);
      part(c1, c2);
      part(c2, n);
    }
    // (rolled up: a CTA comes here a few times, and finds the instructions in memory)
    const int ksteps = blk == p.nb - 1 ? p.ks_last : p.ks_full;
    uint32_t a_row = (1u << 16) | a, b_lo = (p.b_lo0 | wt) + b0;
    bool first = blk == 0;
#pragma unroll 1
    for (int dy = 0; dy < p.ki; ++dy, a_row += (uint32_t)p.P * (p.rb >> 4)) {
      uint32_t a_lo = a_row;
#pragma unroll 1
      for (int dx = 0; dx < K; ++dx, a_lo += p.rb >> 4, b_lo += p.w_tile_bytes >> 4) {
#pragma unroll 1
        for (int k = first ? 1 : 0; k < ksteps; ++k) {
          umma_warp(d_lower, a_lo + 2 * (uint32_t)k, p.a_hi, b_lo + (uint32_t)k * p.b_step, p.b_hi, idesc_lower, 1u);
          if (before < n) umma_warp(tmem_base, a_lo + 2 * (uint32_t)k, p.a_hi, b_lo + b_upper + (uint32_t)k * p.b_step, p.b_hi, idesc_upper, 1u);
        }
        first = false;
      }
    }
    umma_commit_warp(&bar.a_empty[q.s]);
    if (++q.s == (uint32_t)p.a_slots) { q.s = 0; q.a_par ^= 1u; }
  }
#pragma unroll 1
  for (uint32_t i = 0; i < done; ++i) umma_commit_warp(&bar.t_full[i < before ? slot + i : slot + i - ring]);      // outputs that no later plane reaches
  return true;
}

// Planes away from the ends of a segment, one block of channels, accumulators that lie side by side: everything but the addresses is fixed, and the
// barriers of the next plane are asked while this one's products run.  `count` of them; q.slot is that of the first one's lowest output.
template <int K, int KSTEPS, class Params>
__device__ __forceinline__ bool sl_inner_planes(const Params& p, SlState& q, uint32_t tmem_base, uint32_t a0, uint32_t w0, uint32_t count, const SlBars& bar) {
  const uint32_t tile_n = (uint32_t)p.tile_n, idesc_n = (tile_n >> 3) << 17, a_slot16 = p.a_sub_bytes >> 4;
  const uint32_t idesc_all = p.idesc + K * idesc_n, idesc_old = p.idesc + (K - 1) * idesc_n, idesc_new = p.idesc + idesc_n;
  const uint32_t b_lo = p.b_lo0 | w0, b_new = b_lo + (K - 1) * (p.w_blk_bytes >> 4);
  uint32_t s = q.s, a_par = q.a_par, slot = q.slot, used = q.used, d = tmem_base + q.slot * tile_n, a = a0 + q.s * a_slot16;
  bool t_ready = mbar_try_wait(&bar.t_empty[slot + K - 1], ((used >> (slot + K - 1)) & 1u) ^ 1u), a_ready = mbar_try_wait(&bar.a_full[s], a_par);
#pragma unroll 1
  for (;;) {
    if (!__all_sync(0xffffffffu, t_ready & a_ready)) {
      if (!mbar_wait_warp(&bar.t_empty[slot + K - 1], ((used >> (slot + K - 1)) & 1u) ^ 1u, p.status, p.tag)) return false;
      if (!mbar_wait_warp(&bar.a_full[s], a_par, p.status, p.tag)) return false;
    }
    tc_fence_after();
    used ^= 1u << (slot + K - 1);
    umma_warp(d, (1u << 16) | a, p.a_hi, b_lo, p.b_hi, idesc_old, 1u);
    umma_warp(d + (K - 1) * tile_n, (1u << 16) | a, p.a_hi, b_new, p.b_hi, idesc_new, 0u);
    sl_products<K, KSTEPS>(p, d, idesc_all, (1u << 16) | a, b_lo);
    uint64_t *a_done = &bar.a_empty[s], *t_done = &bar.t_full[slot];
    ++slot;
    d += tile_n;
    a += a_slot16;
    if (++s == (uint32_t)p.a_slots) { s = 0; a_par ^= 1u; a = a0; }
    if (--count == 0) {
      umma_commit_warp(a_done);
      umma_commit_warp(t_done);
      break;
    }
    t_ready = mbar_try_wait(&bar.t_empty[slot + K - 1], ((used >> (slot + K - 1)) & 1u) ^ 1u);
    a_ready = mbar_try_wait(&bar.a_full[s], a_par);
    umma_commit_warp(a_done);
    umma_commit_warp(t_done);
  }
  q.s = s; q.a_par = a_par; q.slot = slot; q.used = used;
  return true;
}

// The issuing warp, converged.  (K offsets along the axis, too: p.ks == K.)
template <int K, class Params>
__device__ __forceinline__ void sl_issue(const Params& p, uint32_t tmem_base, uint32_t a0, uint32_t w0, uint32_t i0, uint32_t i1, const SlBars& bar) {
  const uint32_t ring = (uint32_t)p.ring;
  SlState q{};
  uint32_t slot0 = 0;                                    // of the segment's first output
  for (SlWalk w(p, i0); w.it < i1;) {
    const SlSegment g(p, w, i1);
    q.slot = slot0;
    int lo = g.s0;
    for (int si = g.first; si <= g.last;) {
      if (si - p.pad_s > lo) { ++lo; if (++q.slot == ring) q.slot = 0; }
      const int hi = min(g.s1 - 1, si + p.pad_s);
      bool ok;
      if (p.nb == 1 && si != g.first && hi - lo == K - 1 && q.slot + K <= ring) {
        // planes from here on that reach K outputs, one of them new, up to the ring's end
        const int inner = min(g.s1 - p.pad_s - si, (int)(ring - K - q.slot) + 1);
        switch (p.ks_last) {
#define XC_PLANES(KT) ok = sl_inner_planes<K, KT>(p, q, tmem_base, a0, w0, (uint32_t)inner, bar); break;
          case 1: XC_PLANES(1) case 2: XC_PLANES(2) case 3: XC_PLANES(3) default: XC_PLANES(4)
#undef XC_PLANES
        }
        si += inner;
        lo += inner;                                     // (and q.slot is that of this output)
        if (q.slot == ring) q.slot = 0;
      } else {
        const uint32_t n = (uint32_t)(hi - lo + 1), fresh = si == g.first ? 0u : hi == si + p.pad_s ? n - 1 : n;
        ok = sl_plane<K>(p, q, tmem_base, a0, w0, n, fresh, (uint32_t)(K - 1 - (si - lo + p.pad_s)), si == g.last ? n : si - p.pad_s == lo ? 1u : 0u, bar);
        ++si;
      }
      if (!ok) return;
    }
    const uint32_t outputs = (uint32_t)(g.s1 - g.s0);
    slot0 = (slot0 + outputs) % ring;
    w.it += outputs;
    w.s = g.s1;
    if (w.s == p.extent) w.next_column(p);
  }
}

// One group of four epilogue warps: every other output of the CTA.
template <bool F16, class Params>
__device__ __forceinline__ void sl_epilogue(const Params& p, const CUtensorMap* map_out, uint32_t base, uint32_t tmem_base, uint32_t i0, uint32_t i1,
                                            uint64_t* t_full, uint64_t* t_empty) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, quad = warp & 3, group = (warp - 4) >> 2;
  const EpiPixel px(p, quad * 32 + lane);
  const bool leader = quad == 0 && lane == 0;
  uint32_t slot = (uint32_t)group, par = 0, ob = 0;      // (the ring has at least four slots)
  SlWalk w(p, i0);
  if (group == 1) w.step(p);
  for (; w.it < i1; w.step(p), w.step(p)) {
    bool ok = true;
    if (lane == 0) ok = mbar_wait(&t_full[slot], par, p.status, p.tag);
    if (!epi_all(group, ok)) break;                      // the four warps leave together
    tc_fence_after();
    const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + slot * (uint32_t)p.tile_n;
    for (int c = 0; c < p.co; c += p.ocw) {
      const uint32_t tile = base + p.o_off + ((uint32_t)(group * p.o_per) + ob) * p.o_bytes;
      if (leader) { if (p.o_per == 1) bulk_wait_read<0>(); else bulk_wait_read<1>(); }     // the tile's last store has read it
      epi_sync(group);
      epi_row<F16>(p, px, tile, taddr + (uint32_t)c, p.tile_n - c);
      if (c + p.ocw >= p.co) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&t_empty[slot]);
      }
      fence_async_smem();
      epi_sync(group);
      if (leader) {
        tma_store_5d(map_out, tile, c, w.x, p.planar ? w.s : w.y, p.planar ? 0 : w.s, w.b);
        bulk_commit();
      }
      if (p.o_per == 2) ob ^= 1u;
    }
    slot += 2;
    if (slot >= (uint32_t)p.ring) { slot -= (uint32_t)p.ring; par ^= 1u; }
  }
  if (leader) bulk_wait_all();
}

}  // namespace xconv
