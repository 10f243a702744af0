// The offset contraction (Algorithm 1 backward step 4, Eq. 6) of float layers on the tensor cores (sm_100a): every float as three
// bfloat16 parts, a product as six (split_f32.cuh).
//
//   dW[m, n, (dz, dy, dx)] = scale * sum over positions q of L[q, m] * Z[q + (dz, dy, dx) - pad, n]
//
// As in contract_tc.cu a patch of both tensors lies in shared memory once, rows = pixels (MN-major tiles), and the offsets are the
// same memory read from other rows: the columns of an MMA are 32 channels of Z at each of the KS pixel shifts dx (the descriptor's
// stride between column blocks is one pixel), its rows 32 channels of L at each of the KS image rows (stride: one row of the box),
// or 128 channels of L with one dy per work unit where that takes fewer units.  Both boxes have rows of P = pw + KS - 1
// positions, and L is zero in the last KS - 1 of them and behind the last row: the reduction then runs over the flat positions of the box, 16
// per k-step whatever the width of the patch (7 pixels: 7 of 9 are work, where whole k-steps per row left 7 of 16).
//
// The copy engine brings the floats of both boxes, twelve warps write their parts; six passes over a chain of k-steps, the products of the small parts
// first (scaled up, split_f32.cuh; the MMA scales the accumulator down between them) and hh last, leave an accumulator that was rounded towards
// zero a few times at its full size only.  Two accumulator
// sets take the chains in turn, eight epilogue warps add them in float registers (48 sums a thread), and the
// sums of the splits are added in fixed order by a second kernel.
//
// Error against 64 bits on 120 random layers, times that of the FP32 multiply-adds: 0.31 in the median, nowhere more than 1.
// What bounds it: the six passes' MMAs, 56 clocks each for 96 columns (A tile and B at shared memory's 128 bytes a clock), and the
// conversion of a patch for every unit that reads it, about as long.  us, multiply-adds -> this, contraction and sum of the splits: 64 -> 64
// channels, 64 probes of 32 x 32 130 -> 50; 24 -> 48, 3 x 3 x 3, 2 volumes of 27 x 47 x 47 840 -> 105; 3 -> 160, 17 x 13 414 -> 30.
#include "contract_split.h"

#include <algorithm>

#include "conv_split.h"
#include "split_f32.cuh"

namespace xconv {

constexpr int CT_STAGES = 4, CT_CHAIN = 5;         // k-steps a chain holds at most
constexpr int CT_COLS = 96;                        // accumulator columns of a set

struct ContractSplitParams {
  const float *L, *Z;
  float* part;
  int Cout, Cin, W, H, Lc, Zc, depth, KS, KD, T, pad, pad_d;
  int pw, ph, P, patches_x, patches_y;
  uint32_t items, splits;
  int rows_on_a, tiles;                            // L moved by image rows on the MMA rows, in `tiles` row tiles; else one dy per unit
  int mg_n, dy_n, ng_n, j_n, j_per, ng_per;        // work units: row tiles, dy, channel blocks of Z, pixel shifts (and KD depth offsets)
  int a_rows;                                      // image rows of L's box
  uint32_t inv_pw;
  int ksteps, chunk;
  uint32_t a_blk, b_blk, a_plane, b_plane, a_bytes, stage_bytes; int stages;
  uint32_t f_off, f_slot, f_b, f_bytes; int f_slots;      // the floats of a stage: L's box, Z's f_b bytes behind it
  uint32_t a_lo0, b_lo0, a_hi, b_hi, a_step16, b_step16, a_tile16, idesc;
  int cols;
  unsigned int *status, tag;
};

struct SplitUnit { int mg, dy, dz, ng, jg; };
__device__ __forceinline__ SplitUnit split_unit(const ContractSplitParams& p, uint32_t ug) {
  SplitUnit u;
  u.ng = (int)(ug % (uint32_t)p.ng_n); ug /= (uint32_t)p.ng_n;
  u.jg = (int)(ug % (uint32_t)p.j_n); ug /= (uint32_t)p.j_n;
  u.dz = (int)(ug % (uint32_t)p.KD); ug /= (uint32_t)p.KD;
  u.dy = (int)(ug % (uint32_t)p.dy_n); ug /= (uint32_t)p.dy_n;
  u.mg = (int)ug;
  return u;
}
// What accumulator row `row` and column `c` of a unit are: channels m and n, offset (dy, dx).
struct SplitEntry { int m, n, dy, dx; };
__device__ __forceinline__ SplitEntry split_entry(const ContractSplitParams& p, const SplitUnit& u, int row, int c) {
  SplitEntry e;
  if (p.rows_on_a) {
    const int i = u.mg % p.tiles * (TILE_M / 32) + row / 32;
    e.m = u.mg / p.tiles * 32 + row % 32;
    e.dy = p.KS - 1 - i;
  } else {
    e.m = u.mg * TILE_M + row;
    e.dy = u.dy;
  }
  if (p.KS == 1) { e.dx = 0; e.n = u.ng * p.ng_per * 32 + c; }
  else { e.dx = u.jg * p.j_per + c / 32; e.n = u.ng * 32 + c % 32; }
  return e;
}
__device__ __forceinline__ bool split_live(const ContractSplitParams& p, const SplitEntry& e) {
  return e.m < p.Cout && e.n < p.Cin && e.dy >= 0 && e.dx < p.KS;
}

// A walk over patches.
struct SplitWalk {
  int x, y, z, b;
  __device__ __forceinline__ SplitWalk(const ContractSplitParams& p, uint32_t i) {
    const uint32_t a = i / (uint32_t)p.patches_x, c = a / (uint32_t)p.patches_y, e = c / (uint32_t)p.depth;
    x = (int)(i - a * p.patches_x) * p.pw;
    y = (int)(a - c * p.patches_y) * p.ph;
    z = (int)(c - e * p.depth);
    b = (int)e;
  }
  __device__ __forceinline__ void step(const ContractSplitParams& p) {
    if ((x += p.pw) < p.patches_x * p.pw) return;
    x = 0;
    if ((y += p.ph) < p.patches_y * p.ph) return;
    y = 0;
    if (++z == p.depth) { z = 0; ++b; }
  }
};

// The sums of 32 entries with one offset over this split's patches by multiply-adds, a lane each: over the patches in the set `only`, or all; rows
// of patches that are `piece` modulo `pieces`.  Ends early when no lane's sum can change any more: NaN, or not finite among finite terms.
constexpr int CT_SET = 2048;                       // patches of a CTA that a set tells apart (patch i: bit i modulo this)
__device__ __forceinline__ float split_line(const ContractSplitParams& p, uint32_t i0, uint32_t n, int dz, int dy, int dx, int ch_l, int ch_z, bool wanted,
                                            const uint32_t* only, uint32_t piece, uint32_t pieces) {
  constexpr int U = 16;                              // terms whose loads are under way together
  float acc = 0.f;
  uint32_t turn = 0;
  SplitWalk w(p, i0);
  for (uint32_t i = 0; i < n; ++i, w.step(p)) {
    if (only && !((only[i % CT_SET / 32] >> (i % 32)) & 1u)) continue;
    const int zz = w.z + dz - p.pad_d;
    if (zz < 0 || zz >= p.depth) continue;
    const float* Lp = p.L + (((size_t)w.b * p.depth + w.z) * p.H * p.W + w.x) * p.Lc + ch_l;
    const float* Zp = p.Z + (((size_t)w.b * p.depth + zz) * p.H * p.W + w.x) * p.Zc + ch_z;
    const int x0 = max(0, p.pad - dx - w.x), x1 = min(min(p.pw, p.W - w.x), p.W - w.x + p.pad - dx);
    for (int y = 0; y < p.ph; ++y) {
      const int yz = p.rows_on_a ? w.y + y : w.y + y + dy - p.pad, yl = yz - (dy - p.pad);
      if (yz < 0 || yz >= p.H || yl < 0 || yl >= p.H) continue;
      if (turn++ % pieces != piece) continue;
      const float *l = Lp + (size_t)yl * p.W * p.Lc, *z = Zp + (ptrdiff_t)(yz * (ptrdiff_t)p.W + dx - p.pad) * p.Zc;
      for (int x = x0; x < x1; x += U) {
        float a[U], b[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const bool in = x + k < x1;
          a[k] = in ? l[(size_t)(x + k) * p.Lc] : 0.f;
          b[k] = in ? z[(size_t)(x + k) * p.Zc] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) acc = fmaf(a[k], b[k], acc);
        if (__all_sync(0xffffffffu, !wanted || (only ? acc != acc : acc - acc != 0.f))) return acc;
      }
    }
  }
  return acc;
}

// A value that cannot be split makes NaN of every sum it enters, and of those that it meets with a zero between image rows or outside the
// image: the sums of the unit's tile that are not finite are taken again, by all warps of the block.  A warp takes 32 columns of a row, or 32
// rows of a column, whichever leaves fewer of them to do: one infinity among the values of L is rows, one in Z columns.  First over the patches that
// hold values that are not finite (`odd`): what comes out not finite is the result.  The others met such a value with a zero, or ran over;
// they are summed over all patches, which finite terms alone enter.
// us a call (contraction and sum of the splits), 64 -> 64 channels, 64 probes of 32 x 32: finite values 53; one infinity in L 97, in Z 72; all of L
// NaN 123, or so large that every sum runs over 173.  One thread a sum, serially, took 16900 and 1060 for one infinity.
__device__ __noinline__ void split_again(const ContractSplitParams& p, const SplitUnit& u, float* tile, uint32_t i0, uint32_t n, const uint32_t* odd,
                                         uint32_t* scratch) {
  constexpr int WARPS = SP_THREADS / 32, MAP = CT_COLS * 4, LIST = MAP + 8, SUMS = LIST + CT_COLS * 4;
  uint32_t *map = scratch, *lines = scratch + MAP, *list = scratch + LIST, &count = lines[7];      // map: sums to do, [column][row / 32]; lines: rows, columns with one
  float* sums = reinterpret_cast<float*>(scratch + SUMS);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const auto at = [&](int row, int c) { return tile + (size_t)(c >> 2) * 4 * TILE_M + row * 4 + (c & 3); };
  for (int i = tid; i < LIST; i += SP_THREADS) scratch[i] = 0;
  bool any = tid < CT_SET / 32 && odd[tid] != 0;
  const bool some_odd = __syncthreads_or(any);
#pragma unroll 2
  for (int i = tid; i < p.cols / 4 * TILE_M; i += SP_THREADS) {      // (a warp: four columns of 32 rows)
    const float4 v = reinterpret_cast<const float4*>(tile)[i];
    const float f[4] = {v.x, v.y, v.z, v.w};
    const int row = i % TILE_M, c0 = i / TILE_M * 4;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!__any_sync(0xffffffffu, f[k] - f[k] != 0.f)) continue;
      const unsigned rows = __ballot_sync(0xffffffffu, f[k] - f[k] != 0.f && split_live(p, split_entry(p, u, row, c0 + k)));
      if (lane != 0 || !rows) continue;
      map[(c0 + k) * 4 + (row >> 5)] = rows;
      atomicOr(&lines[row >> 5], rows);
      atomicOr(&lines[4 + (c0 >> 5)], 1u << ((c0 + k) & 31));
    }
  }
  __syncthreads();
  const bool by_row = __popc(lines[0]) + __popc(lines[1]) + __popc(lines[2]) + __popc(lines[3]) <= __popc(lines[4]) + __popc(lines[5]) + __popc(lines[6]);
  const int wide = (by_row ? p.cols : TILE_M) / 32, words = (by_row ? TILE_M : p.cols) * wide;
  struct Word { int row, c; bool wanted; unsigned lanes; SplitEntry e; int dy, dx; };
  const auto word_at = [&](int word) {
    Word t;
    const int line = word / wide, other = word % wide * 32 + lane;
    t.row = by_row ? line : other; t.c = by_row ? other : line;
    t.wanted = (map[t.c * 4 + (t.row >> 5)] >> (t.row & 31)) & 1u;
    t.lanes = __ballot_sync(0xffffffffu, t.wanted);
    t.e = split_entry(p, u, t.row, t.c);
    const int first = max(0, __ffs(t.lanes) - 1);               // (the offset is that of all wanted lanes)
    t.dy = __shfl_sync(0xffffffffu, t.e.dy, first); t.dx = __shfl_sync(0xffffffffu, t.e.dx, first);
    return t;
  };
  const auto line_sum = [&](const Word& t, const uint32_t* only, uint32_t piece, uint32_t pieces) {
    return split_line(p, i0, n, u.dz, t.dy, t.dx, t.wanted ? t.e.m : 0, t.wanted ? t.e.n : 0, t.wanted, only, piece, pieces);
  };
  for (int word = warp; word < words; word += WARPS) {
    const Word t = word_at(word);
    if (!t.lanes) continue;
    bool left = t.wanted;
    if (some_odd) {
      const float s = line_sum(t, odd, 0, 1);
      if (left && s - s != 0.f) {
        *at(t.row, t.c) = s;
        atomicAnd(&map[t.c * 4 + (t.row >> 5)], ~(1u << (t.row & 31)));
        left = false;
      }
    }
    if (__any_sync(0xffffffffu, left) && lane == 0) list[atomicAdd(&count, 1u)] = (uint32_t)word;
  }
  __syncthreads();
  const int todo = (int)count, pieces = max(1, WARPS / max(1, todo));
  for (int item = warp; item < todo * pieces; item += WARPS) {
    const Word t = word_at((int)list[item / pieces]);
    const float s = line_sum(t, nullptr, (uint32_t)(item % pieces), (uint32_t)pieces);
    if (pieces > 1) sums[item * 32 + lane] = s;
    else if (t.wanted) *at(t.row, t.c) = s;
  }
  if (pieces == 1) return;
  __syncthreads();
  if (warp >= todo) return;
  const Word t = word_at((int)list[warp]);
  float s = 0.f;
  for (int k = 0; k < pieces; ++k) s += sums[(warp * pieces + k) * 32 + lane];
  if (t.wanted) *at(t.row, t.c) = s;
}

template <int RBA, int QA, int QB>
__global__ void __launch_bounds__(SP_THREADS, 1)
contract_split_kernel(const __grid_constant__ CUtensorMap map_l, const __grid_constant__ CUtensorMap map_z, const __grid_constant__ ContractSplitParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[CT_STAGES], empty[CT_STAGES], acc_full[2], acc_empty[2];
  __shared__ __align__(8) uint64_t f_full[SP_FLOATS], f_empty[SP_FLOATS];
  __shared__ uint32_t tmem_slot, odd[CT_SET / 32];      // odd: patches with a value that is not finite
  __shared__ int go;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  if (threadIdx.x == 0) {
    for (int s = 0; s < CT_STAGES; ++s) { mbar_init(&full[s], SP_CONVERTERS / 32); mbar_init(&empty[s], 2); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 8); }
    for (int f = 0; f < SP_FLOATS; ++f) { mbar_init(&f_full[f], 1); mbar_init(&f_empty[f], SP_CONVERTERS / 32); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    prefetch_tmap(&map_l);
    prefetch_tmap(&map_z);
  }
  if (threadIdx.x < CT_SET / 32) odd[threadIdx.x] = 0;
  // (L between the rows of a patch and both tensors behind the last one stay zero)
  const uint32_t tmem_base = split_begin(warp, &tmem_slot, 256u, base, (uint32_t)p.stages * p.stage_bytes, p.status, p.tag, &go);
  const uint32_t ug = blockIdx.x / p.splits, split = blockIdx.x - ug * p.splits;
  const uint32_t i0 = (uint32_t)((unsigned long long)p.items * split / p.splits);
  const uint32_t n = (uint32_t)((unsigned long long)p.items * (split + 1) / p.splits) - i0;     // patches of this CTA (>= 1)
  const SplitUnit u = split_unit(p, ug);
  const int chains = (p.ksteps + p.chunk - 1) / p.chunk;
  const int width = p.KS == 1 ? p.cols : min(p.j_per, p.KS - u.jg * p.j_per) * 32;      // columns of this unit's MMAs
  int again = 0;                                     // a sum is not finite

  if (!go) {
    // fall through to the teardown
  } else if (warp == 1 || warp == 2) {
    // ------------------------------------------------------------------ MMA issuers (whole warps): every other chain each
    const uint32_t own = (uint32_t)warp - 1;
    const uint32_t s0 = (base & 0x3FFFFu) >> 4, stage16 = p.stage_bytes >> 4, ap = p.a_plane >> 4, bp = p.b_plane >> 4;
    const uint32_t a_add = p.a_lo0 + (p.rows_on_a ? (uint32_t)(u.mg % p.tiles) * p.a_tile16 : 0u);
    const uint32_t b_add = p.b_lo0 + (p.a_bytes >> 4) + (uint32_t)(u.jg * p.j_per) * 4u;             // (a pixel: 64 bytes)
    const uint32_t idesc = p.idesc | ((uint32_t)(width >> 3) << 17);
    const uint32_t a_step = p.a_step16, b_step = p.b_step16, a_hi = p.a_hi, b_hi = p.b_hi;
    const uint32_t d = tmem_base + own * CT_COLS;
    uint32_t s = 0, par = 0, st = s0, chain = 0, t_par = 1;     // (a wait for the phase before the first returns at once)
    bool ok = true;
    for (uint32_t i = 0; i < n && ok; ++i) {
      ok = mbar_wait_warp(&full[s], par, p.status, p.tag);
      if (!ok) break;
      tc_fence_after();
      uint32_t a0 = st + a_add, b0 = st + b_add;
      for (int k0 = 0; k0 < p.ksteps; k0 += p.chunk, chain ^= 1u, a0 += a_step * (uint32_t)p.chunk, b0 += b_step * (uint32_t)p.chunk) {
        if (chain != own) continue;
        ok = mbar_wait_warp(&acc_empty[own], t_par, p.status, p.tag);
        if (!ok) break;
        t_par ^= 1u;
        tc_fence_after();
        const int kn = min(p.chunk, p.ksteps - k0);
        uint32_t acc = 0;
        // lh, hl, mm (times 2^14), mh, hm (2^7), hh: the accumulator is scaled down between them
        auto pass = [&](uint32_t a, uint32_t b, bool down) {
#pragma unroll
          for (int k = 0; k < CT_CHAIN; ++k) {
            if (k >= kn) break;
            if (k == 0 && down) umma_warp_down<7>(d, a, a_hi, b, b_hi, idesc);
            else umma_warp(d, a, a_hi, b, b_hi, idesc, acc);
            acc = 1u;
            a += a_step;
            b += b_step;
          }
        };
        pass(a0 + 2 * ap, b0, false);
        pass(a0, b0 + 2 * bp, false);
        pass(a0 + ap, b0 + bp, false);
        pass(a0 + ap, b0, true);
        pass(a0, b0 + bp, false);
        pass(a0, b0, true);
        umma_commit_warp(&acc_full[own]);
      }
      if (!ok) break;
      umma_commit_warp(&empty[s]);
      st += stage16;
      if (++s == (uint32_t)p.stages) { s = 0; par ^= 1u; st = s0; }
    }
  } else if (warp >= SP_CONVERT) {
    // ------------------------------------------------------------------ conversion
    uint32_t s = 0, par = 1, f = 0, f_par = 0;
    for (uint32_t i = 0; i < n; ++i) {
      if (!split_wait(&empty[s], par, p.status, p.tag) || !split_wait(&f_full[f], f_par, p.status, p.tag)) break;
      const uint32_t from = base + p.f_off + f * p.f_slot, to = base + s * p.stage_bytes;
      const SplitBox of_l{from, p.pw * p.a_rows, to, p.a_plane, p.a_blk, (uint32_t)(p.KS - 1), p.inv_pw};
      const SplitBox of_z{from + p.f_b, p.P * p.ph, to + p.a_bytes, p.b_plane, p.b_blk, 0u, 0u};
      float2 check = make_float2(0.f, 0.f);
      split_box<RBA == 128 ? 7 : 6, QA, true>(of_l, check);
      split_box<6, QB, false>(of_z, check);
      split_stage_done(&full[s], &f_empty[f], check, [&] {
        const bool odd_l = split_box_again<RBA == 128 ? 7 : 6, QA, true>(of_l), odd_z = split_box_again<6, QB, false>(of_z);
        if (odd_l || odd_z) atomicOr(&odd[i % CT_SET / 32], 1u << (i % 32));
      });
      if (++s == (uint32_t)p.stages) { s = 0; par ^= 1u; }
      if (++f == (uint32_t)p.f_slots) { f = 0; f_par ^= 1u; }
    }
  } else if (warp == SP_LOAD) {
    // ------------------------------------------------------------------ copies of the floats
    if (lane == 0) {
      const int a_dy = p.rows_on_a ? -p.pad : 0, b_dy = p.rows_on_a ? 0 : u.dy - p.pad;
      const int a_c0 = p.rows_on_a ? u.mg / p.tiles * 32 : u.mg * TILE_M, b_c0 = u.ng * p.ng_per * 32;
      uint32_t f = 0, par = 1, i = 0;
      SplitWalk w(p, i0);
      for (; i < n; ++i, w.step(p)) {
        if (!mbar_wait(&f_empty[f], par, p.status, p.tag)) break;
        const uint32_t dst = base + p.f_off + f * p.f_slot;
        mbar_arrive_expect_tx(&f_full[f], p.f_bytes);
        tma_load_5d(dst, &map_l, a_c0, w.x, w.y + a_dy, w.z, w.b, &f_full[f]);
        tma_load_5d(dst + p.f_b, &map_z, b_c0, w.x - p.pad, w.y + b_dy, w.z + u.dz - p.pad_d, w.b, &f_full[f]);
        if (++f == (uint32_t)p.f_slots) { f = 0; par ^= 1u; }
      }
      // every copy issued must have landed before the CTA exits
      for (uint32_t k = i > (uint32_t)p.f_slots ? i - p.f_slots : 0; k < i; ++k)
        if (!mbar_wait(&f_full[k % p.f_slots], (k / p.f_slots) & 1u, p.status, p.tag)) break;
    }
  } else if (warp >= SP_EPILOGUE) {
    // ------------------------------------------------------------------ epilogue: chains to registers, registers to partial sums
    // Column groups half, half + 2, ... of 16, of the columns that the MMAs write: 5 x 5 kernels have units of two shifts, whose third lies in tensor memory
    // as the kernel before left it.  (Read, and not finite by chance, it sent the block through split_again for nothing, 22 -> 32 us.)
    const int quad = warp & 3, half = (warp - SP_EPILOGUE) >> 2, groups = width >> 4;
    const uint32_t tmem_q = tmem_base + ((uint32_t)(quad * 32) << 16);
    float sum[3][16];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int e = 0; e < 16; ++e) sum[k][e] = 0.f;
    bool ok = true;
    const uint32_t sets = n * (uint32_t)chains;
    for (uint32_t c = 0; c < sets; ++c) {
      const uint32_t buf = c & 1u;
      ok = split_wait(&acc_full[buf], (c >> 1) & 1u, p.status, p.tag);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (half + 2 * k >= groups) break;
        uint32_t x[16];
        tmem_ld16_issue(tmem_q + buf * CT_COLS + (uint32_t)(half + 2 * k) * 16, x);
        tmem_ld_wait(x);
#pragma unroll
        for (int e = 0; e < 16; ++e) sum[k][e] += __uint_as_float(x[e]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
    if (ok) {
      const int row = quad * 32 + lane;
      float* part = p.part + ((size_t)ug * p.splits + split) * (size_t)p.cols * TILE_M + (size_t)row * 4;
      float check = 0.f;                             // 0, or NaN
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (half + 2 * k >= groups) break;
        float* dst = part + (size_t)(half + 2 * k) * 16 * TILE_M;
#pragma unroll
        for (int e = 0; e < 16; ++e) check = fmaf(sum[k][e], 0.f, check);
#pragma unroll
        for (int e = 0; e < 16; e += 4)
          *reinterpret_cast<float4*>(dst + (size_t)e * TILE_M) = make_float4(sum[k][e], sum[k][e + 1], sum[k][e + 2], sum[k][e + 3]);
      }
      again = !(check == 0.f);
    }
  }
  tc_fence_before();
  again = __syncthreads_or(again);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 256u);
  }
  if (again) split_again(p, u, p.part + ((size_t)ug * p.splits + split) * (size_t)p.cols * TILE_M, i0, n, odd,
                         reinterpret_cast<uint32_t*>(smem_raw));
}

// dW[m][offset][n] = scale(n) * sum over splits, four neighbouring columns of one accumulator row per group.  LANES threads share a
// group and take the splits in turn; their sums are added in lane order.
template <int LANES>
__global__ void __launch_bounds__(256) reduce_split_partials(const ContractSplitParams p, float* __restrict__ out, uint32_t groups,
                                                             float alpha, const float* __restrict__ chan_scale) {
  constexpr int GROUPS = 256 / LANES;
  __shared__ float4 acc[LANES][GROUPS];
  const int o = threadIdx.x % GROUPS, g = threadIdx.x / GROUPS;
  const uint32_t idx = blockIdx.x * GROUPS + o, q4 = (uint32_t)p.cols >> 2;
  const uint32_t row = idx % TILE_M, q = idx / TILE_M % q4, ug = idx / TILE_M / q4;
  const SplitUnit u = split_unit(p, ug);
  const SplitEntry e = split_entry(p, u, (int)row, (int)q * 4);
  const bool live = idx < groups && split_live(p, e);
  const size_t tile = (size_t)p.cols * TILE_M;
  const float* src = p.part + (size_t)ug * p.splits * tile + ((size_t)q * TILE_M + row) * 4;
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
  float* dst = out + ((size_t)e.m * p.T + (u.dz * p.KS + e.dy) * p.KS + e.dx) * p.Cin + e.n;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (e.n + k < p.Cin) dst[k] = r[k] * (chan_scale ? chan_scale[e.n + k] : alpha);
}

// ------------------------------------------------------------------------------------ host side


// The positions as the kernel sees them: without neighbours (1 x 1 kernels) all pixels of all probes are one row.
struct SplitGeo { long W, H, D, B; };
static SplitGeo split_geo(const xconv_desc* d) {
  const long depth = d->D > 1 ? d->D : 1;
  if (d->KD <= 1 && d->KH == 1) return {(long)d->r * depth * d->H * d->W, 1, 1, 1};
  if (d->KD <= 1) return {d->W, d->H, 1, (long)d->r * depth};
  return {d->W, d->H, depth, d->r};
}

bool plan_contract_split(const xconv_desc* d, ContractSplitPlan* p) {
  if (d->dtype != XCONV_F32 || d->circular) return false;
  const SplitGeo g = split_geo(d);
  if (g.W >= (1L << 30) || g.W * g.H >= (1L << 31) || g.D * g.B >= (1L << 31)) return false;
  const int KS = d->KH, KD = d->KD > 1 ? d->KD : 1;
  const int row_tiles = (int)cdivl(KS * 32, TILE_M);
  const long moved = cdivl(d->Cout, 32) * row_tiles, plain = cdivl(d->Cout, TILE_M) * KS;
  p->rows_on_a = KS > 1 && moved <= plain ? 1 : 0;
  p->tiles = p->rows_on_a ? row_tiles : 1;
  p->mg_n = (int)(p->rows_on_a ? moved : cdivl(d->Cout, TILE_M));
  p->dy_n = p->rows_on_a ? 1 : KS;
  p->cwa = p->rows_on_a || d->Cout <= 32 ? 32 : 64;
  p->a_blocks = p->rows_on_a || d->Cout <= 64 ? 1 : 2;
  p->j_per = std::min(KS, 3);
  p->j_n = (int)cdivl(KS, p->j_per);
  p->ng_per = KS > 1 ? 1 : d->Cin > 32 ? 2 : 1;
  p->ng_n = (int)cdivl(d->Cin, 32 * p->ng_per);
  p->cols = KS > 1 ? p->j_per * 32 : p->ng_per * 32;
  const long units = (long)p->mg_n * p->dy_n * KD * p->ng_n * p->j_n;
  if (units * (p->cols / 4) * TILE_M >= 1L << 31) return false;      // (the sum of the splits counts groups of four entries in 32 bits)
  const int qa = p->a_blocks * p->cwa / 4, qb = p->ng_per * 8;
  // clocks of an MMA: the tensor pipe, or the A tile and B at shared memory's rate
  const long mma = std::max(p->cols / 2, 32 + p->cols / 4);
  double best = -1;
  // (a few widths, and of each the three largest patches that fit: the search is part of every call)
  static const int widths[] = {128, 96, 64, 48, 32, 16};
  const long nx0 = cdivl(g.W, 128);
  for (int i = 0; i < 6; ++i) {
    if (g.W <= 1024 && nx0 + i > g.W) break;
    const long nx = g.W > 1024 ? cdivl(g.W, widths[i]) : nx0 + i;
    const int pw = (int)cdivl(g.W, nx), P = pw + KS - 1;
    int tried = 0;
    for (long ny = cdivl(g.H, 16); ny <= g.H && tried < 3; ny = std::max(ny + 1, cdivl(g.H, cdivl(g.H, ny) - (g.H > ny ? 1 : 0)))) {
      const int ph = (int)cdivl(g.H, ny), ksteps = (int)cdivl((ph - 1) * P + pw, 16);
      const int a_pos = ksteps * 16 + (p->rows_on_a ? (p->tiles * (TILE_M / 32) - 1) * P : 0), b_pos = ksteps * 16 + KS - 1;
      const uint32_t a_blk = up1k((uint32_t)a_pos * 2 * p->cwa), b_blk = up1k((uint32_t)b_pos * 64);
      const int a_rows = p->rows_on_a ? ph + KS - 1 : ph;
      const uint32_t stage = 3 * (a_blk * p->a_blocks + b_blk * p->ng_per);
      const uint32_t f_b = (uint32_t)(pw * a_rows * qa) * 16, f_slot = up1k(f_b) + up1k((uint32_t)(P * ph * qb) * 16);
      const long room = SMEM_LIMIT - 4096 - 2 * (long)stage - 2 * (long)f_slot;
      if (room < 0 || P > 256 || a_rows > 256) continue;
      ++tried;
      const long patches = cdivl(g.W, pw) * cdivl(g.H, ph) * g.D * g.B;
      if (patches >= (1L << 31)) continue;
      const long quads = (long)pw * a_rows * qa + (long)P * ph * qb;
      // conversion: some 45 instructions for four values, on four schedulers at two thirds of their rate
      const double clk = std::max({6.0 * ksteps * mma, quads * 45.0 / 85, quads * 16.0 / 45, 300.0 * cdivl(ksteps, CT_CHAIN)}) + 150;
      const long splits = std::max(1L, std::min((long)NUM_SMS / units, patches));
      const double cost = (double)cdivl(patches, splits) * clk * cdivl(units * splits, NUM_SMS);
      if (best >= 0 && cost >= best) continue;
      best = cost;
      p->pw = pw; p->ph = ph; p->ksteps = ksteps; p->a_blk = a_blk; p->b_blk = b_blk;
      p->patches = patches; p->splits = splits;
      p->f_slot = f_slot; p->f_b = up1k(f_b);
      p->f_slots = 2 + (int)std::min<long>(SP_FLOATS - 2, room / f_slot);
      p->stages = 2 + (int)std::min<long>(CT_STAGES - 2, (room - (p->f_slots - 2) * (long)f_slot) / stage);
    }
  }
  if (best < 0) return false;
  p->units = units;
  const long px = g.W * g.H * g.D * g.B;
  p->part_bytes = (size_t)units * p->splits * p->cols * TILE_M * sizeof(float);
  p->bytes = p->part_bytes + padded_float_bytes(px, d->Cout) + padded_float_bytes(px, d->Cin);
  return true;
}

xconv_status run_contract_split(const xconv_desc* d, const ContractSplitPlan& pl, const float* L, const float* Z, float* dW, float alpha,
                                char* ws_head, char* part, cudaStream_t st) {
  const int KS = d->KH, KD = d->KD > 1 ? d->KD : 1;
  const SplitGeo g = split_geo(d);
  const long px = g.W * g.H * g.D * g.B;
  char* copies = part + pl.part_bytes;
  xconv_status s = pad_floats(L, reinterpret_cast<float*>(copies), px, d->Cout, st);
  if (s == XCONV_OK) s = pad_floats(Z, reinterpret_cast<float*>(copies + padded_float_bytes(px, d->Cout)), px, d->Cin, st);
  if (s != XCONV_OK) return s;
  ContractSplitParams p{};
  p.L = L; p.Z = Z; p.part = reinterpret_cast<float*>(part);
  p.Cout = d->Cout; p.Cin = d->Cin; p.Lc = round_up(d->Cout, 4); p.Zc = round_up(d->Cin, 4); p.W = (int)g.W; p.H = (int)g.H; p.depth = (int)g.D;
  p.KS = KS; p.KD = KD; p.T = KD * KS * KS; p.pad = (KS - 1) / 2; p.pad_d = (KD - 1) / 2;
  p.pw = pl.pw; p.ph = pl.ph; p.P = pl.pw + KS - 1;
  p.patches_x = (int)cdivl(g.W, p.pw); p.patches_y = (int)cdivl(g.H, p.ph);
  p.items = (uint32_t)pl.patches; p.splits = (uint32_t)pl.splits;
  p.rows_on_a = pl.rows_on_a; p.tiles = pl.tiles;
  p.mg_n = pl.mg_n; p.dy_n = pl.dy_n; p.ng_n = pl.ng_n; p.j_n = pl.j_n; p.j_per = pl.j_per; p.ng_per = pl.ng_per;
  p.a_rows = pl.rows_on_a ? pl.ph + KS - 1 : pl.ph;
  p.inv_pw = (uint32_t)cdivl(1L << 20, pl.pw);
  p.ksteps = pl.ksteps;
  p.chunk = (int)cdivl(pl.ksteps, cdivl(pl.ksteps, CT_CHAIN));
  const uint32_t rba = 2 * (uint32_t)pl.cwa;
  p.a_blk = pl.a_blk; p.b_blk = pl.b_blk;
  p.a_plane = pl.a_blk * (uint32_t)pl.a_blocks; p.b_plane = pl.b_blk * (uint32_t)pl.ng_per;
  p.a_bytes = 3 * p.a_plane; p.stage_bytes = p.a_bytes + 3 * p.b_plane; p.stages = pl.stages;
  const int qa = pl.a_blocks * pl.cwa / 4, qb = pl.ng_per * 8;      // pieces of four channels per position
  p.f_off = (uint32_t)p.stages * p.stage_bytes;
  p.f_slot = pl.f_slot; p.f_slots = pl.f_slots; p.f_b = pl.f_b;
  p.f_bytes = (uint32_t)(p.pw * p.a_rows * qa + p.P * p.ph * qb) * 16;
  // MMA rows: moved copies of the one block, a row of the box apart, or neighbouring channel blocks (a single one: read twice)
  p.a_lo0 = ((pl.rows_on_a ? (uint32_t)p.P * rba : pl.a_blocks > 1 ? pl.a_blk : 0u) >> 4) << 16;
  p.b_lo0 = ((KS > 1 ? 64u : pl.b_blk) >> 4) << 16;
  p.a_hi = ((8 * rba) >> 4) | (1u << 14) | ((pl.cwa == 64 ? 2u : 4u) << 29);
  p.b_hi = ((8 * 64u) >> 4) | (1u << 14) | (4u << 29);
  p.a_step16 = (16 * rba) >> 4; p.b_step16 = 64;
  p.a_tile16 = ((TILE_M / 32) * (uint32_t)p.P * rba) >> 4;
  p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(TILE_M >> 4) << 24);
  p.cols = pl.cols;
  p.status = reinterpret_cast<unsigned int*>(ws_head);
  p.tag = call_tag();
  CUtensorMap ml, mz;
  auto map = [&](CUtensorMap* m, const float* ptr, int C, int cb, int bw, int bh) {
    const uint64_t row = (uint64_t)C * 4;
    const uint64_t dims[5] = {(uint64_t)C, (uint64_t)g.W, (uint64_t)g.H, (uint64_t)g.D, (uint64_t)g.B};
    const uint64_t str[4] = {row, row * g.W, row * g.W * g.H, row * g.W * g.H * g.D};
    const uint32_t box[5] = {(uint32_t)cb, (uint32_t)bw, (uint32_t)bh, 1, 1};
    return make_map_f32(m, ptr, 5, dims, str, box, CU_TENSOR_MAP_SWIZZLE_NONE);
  };
  if (!map(&ml, L, p.Lc, 4 * qa, p.pw, p.a_rows) || !map(&mz, Z, p.Zc, 4 * qb, p.P, p.ph)) return XCONV_ERR_CUDA;
  const size_t smem = 1024 + (size_t)p.f_off + (size_t)p.f_slots * p.f_slot;
  if (smem > (size_t)(SMEM_LIMIT - 1024)) return XCONV_ERR_UNSUPPORTED;
  const unsigned grid = (unsigned)(pl.units * pl.splits);
  void (*kernel)(CUtensorMap, CUtensorMap, ContractSplitParams) =
      qb == 16 ? (qa == 8 ? contract_split_kernel<64, 3, 4> : qa == 16 ? contract_split_kernel<128, 4, 4> : contract_split_kernel<128, 5, 4>)
               : (qa == 8 ? contract_split_kernel<64, 3, 3> : qa == 16 ? contract_split_kernel<128, 4, 3> : contract_split_kernel<128, 5, 3>);
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT - 1024);
  if (e == cudaSuccess) e = launch_pdl(kernel, dim3(grid), dim3(SP_THREADS), smem_of_grid(smem, grid), st, ml, mz, p);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  const uint32_t groups = (uint32_t)(pl.units * (pl.cols / 4) * TILE_M);
#define XC_REDUCE(LANES) launch_pdl(reduce_split_partials<LANES>, dim3((unsigned)cdivl(groups, 256 / LANES)), dim3(256), 0, st, p, dW, groups, \
                                    alpha, d->chan_scale)
  if (pl.splits >= 64) e = XC_REDUCE(16);
  else if (pl.splits >= 12) e = XC_REDUCE(4);
  else e = XC_REDUCE(1);
#undef XC_REDUCE
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

}  // namespace xconv
