// Float operands for the tensor cores: every float as the sum of three bfloat16 values,
//
//   x = h + m + l,   h = rn(x), m = rn(x - h), l = rn(x - h - m)      (8 + 8 + 8 significand bits: exact)
//
// and a product of two floats as the six products hh, hm, mh, hl, mm, lh of their parts (each exact in a float; the three
// left out are below 2^-24 of the product together: |m| <= 2^-8 |x|, |l| <= 2^-17 |x|).  The second and third parts are kept times 2^7 and
// 2^14, so that they have the range of the first one: floats below 2^-110 would lose bits of their last part otherwise.  hm and mh then carry
// 2^7, hl, mm and lh 2^14, none larger than the product itself, and their sums are scaled back (exactly) where they are added.
//
// What keeps the sums as precise as FP32 multiply-adds is where they are taken: the accumulators of the tensor cores are not rounded to
// nearest and lose about 2e-8 of their value with every MMA, so the products hh are summed apart from the small ones, or behind them, in
// chains of a few MMAs, and the chains are added in float registers (see the kernels for the errors measured).
//
// Values that are not finite.  The first part of an infinity or NaN is the value itself, so the products hh are what the definition makes of
// it; the other parts are NaN then.  Where the products hh have a column group of their own, a chain whose group is not finite counts
// with that group alone (split_add_set): results that are not finite cost no more than others, and no other result changes.  The contraction, whose
// products share an accumulator, and whose zeros between image rows would meet them, takes sums that are not finite again.
// The first part of a finite value is finite (a value that would round up to an infinity is cut to the largest bfloat16 instead).
#pragma once

#include <type_traits>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace xconv {

// The parts of four neighbouring floats, packed in pairs.
struct Split4 { uint2 h, m, l; };
struct Bf16Parts {
  static constexpr float STEP = 128.f;               // between the scales of two parts
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  static __device__ __forceinline__ float2 floats(uint32_t v) { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u)); }
};
// Three float16 parts (11 + 11 + 11 bits, of values that the caller scales to below 2^15; the second part times 2^12, the third times 2^24, so
// that what is left of a value below 2^15 is below 2^-47 whatever its size).
struct F16Parts {
  static constexpr float STEP = 4096.f;
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  static __device__ __forceinline__ float2 floats(uint32_t v) { return __half22float2(*reinterpret_cast<const __half2*>(&v)); }
};
// (a, b) - (the two values of v), times the scale of the next part; two floats an instruction.
template <class Parts>
__device__ __forceinline__ void take_part(float& a, float& b, uint32_t v) {
  const float2 left = __fmul2_rn(__ffma2_rn(Parts::floats(v), make_float2(-1.f, -1.f), make_float2(a, b)), make_float2(Parts::STEP, Parts::STEP));
  a = left.x; b = left.y;
}
// The parts of v, the first one given; `v` is what is left of it behind the second one then.
template <class Parts>
__device__ __forceinline__ Split4 split_behind(float4& v, uint2 h) {
  Split4 s;
  s.h = h;
  take_part<Parts>(v.x, v.y, h.x); take_part<Parts>(v.z, v.w, h.y);
  s.m = make_uint2(Parts::pack(v.x, v.y), Parts::pack(v.z, v.w));
  take_part<Parts>(v.x, v.y, s.m.x); take_part<Parts>(v.z, v.w, s.m.y);
  s.l = make_uint2(Parts::pack(v.x, v.y), Parts::pack(v.z, v.w));
  return s;
}
constexpr float BF16_MAX = 3.3895313892515355e38f;
__device__ __forceinline__ float cut_to_bf16(float v) { return v - v == 0.f ? fminf(fmaxf(v, -BF16_MAX), BF16_MAX) : v; }
// 2^7 (c - the two values of v): the multiply-add takes the bfloat16 halves as they are (unpacking them cost four instructions of ten).
__device__ __forceinline__ float2 left_behind(float2 c, uint32_t v) {
  const float2 up = __fmul2_rn(c, make_float2(Bf16Parts::STEP, Bf16Parts::STEP));
  float2 d;
  asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tfma.rn.f32.bf16 %0, l, %5, %3;\n\tfma.rn.f32.bf16 %1, h, %5, %4;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "r"(v), "f"(up.x), "f"(up.y), "h"((uint16_t)0xC300));      // -128
  return d;
}
// The parts where the first part of every value is finite and 2^7 times the value is; `check` becomes NaN where not.
__device__ __forceinline__ Split4 split4(float4 v, float2& check) {
  Split4 s;
  s.h = make_uint2(Bf16Parts::pack(v.x, v.y), Bf16Parts::pack(v.z, v.w));
  float2 a = left_behind(make_float2(v.x, v.y), s.h.x), b = left_behind(make_float2(v.z, v.w), s.h.y);
  s.m = make_uint2(Bf16Parts::pack(a.x, a.y), Bf16Parts::pack(b.x, b.y));
  a = left_behind(a, s.m.x); b = left_behind(b, s.m.y);
  s.l = make_uint2(Bf16Parts::pack(a.x, a.y), Bf16Parts::pack(b.x, b.y));
  check = __ffma2_rn(a, b, check);
  return s;
}
// A first part that rounded to zero of values that are not zero becomes the type's smallest number, so that an infinity times it is
// one.  (For operands that a kernel of their own splits.  Where the boxes are split, an infinity times a float below 2^-134 is NaN.)
__device__ __forceinline__ uint32_t never_zero(uint32_t h, float a, float b) {
  if (a != 0.f && !(h & 0x7FFFu)) h |= 1u;
  if (b != 0.f && !(h & 0x7FFF0000u)) h |= 0x10000u;
  return h;
}
template <class Parts, bool NEVER_ZERO = true>
__device__ __forceinline__ Split4 split4_apart(float4 v) {
  const float4 c = std::is_same<Parts, Bf16Parts>::value ? make_float4(cut_to_bf16(v.x), cut_to_bf16(v.y), cut_to_bf16(v.z), cut_to_bf16(v.w)) : v;
  uint2 h = make_uint2(Parts::pack(c.x, c.y), Parts::pack(c.z, c.w));
  if (NEVER_ZERO) h = make_uint2(never_zero(h.x, v.x, v.y), never_zero(h.y, v.z, v.w));
  return split_behind<Parts>(v, h);
}
__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint2 v) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}
template <typename T>
__device__ __forceinline__ void st_shared_16(uint32_t addr, T v) {
  asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"(*reinterpret_cast<const uint16_t*>(&v)) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
// Byte offset of byte `b` of tile row `row` (2^rbs bytes a row, swizzled as the copy engine and the MMA descriptors have it).
__device__ __forceinline__ uint32_t swizzled(int rbs, uint32_t row, uint32_t b) {
  return (row << rbs) + (b ^ (((row >> (7 - rbs)) & ((1u << (rbs - 4)) - 1u)) << 4));
}

// Loads of 16 columns each, and the wait for them (the registers pass through it, so that nothing reads them before).
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
               "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                 "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]),
                 "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]) :: "memory");
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// The roles of a block's 24 warps (80 registers a thread): 0 copies operands that were split before, 1 and 2 issue MMAs -- the chains of
// accumulator set 0 and those of set 1, since one warp's instructions (some 40 clocks an MMA, and the waits between) do not keep the
// tensor pipe busy beside the other warps -- 3 copies the floats, 4..11 add chains up, two per quarter of the MMA rows, 12..23 convert.
constexpr int SP_THREADS = 768, SP_LOAD = 3, SP_EPILOGUE = 4, SP_CONVERT = 12, SP_CONVERTERS = 384;
constexpr int SP_MAX_N = 64;                         // columns of a group (two groups of 16 per epilogue warp)
constexpr int SP_FLOATS = 4;                         // float boxes under way at most

// A box of floats as the copy engine left it at `src` (2^QSHIFT pieces of four per position, one position behind the other), converted to
// three tiles of 2^RBS bytes a row in blocks `block` bytes apart, the parts `plane` bytes apart.  Position i goes to row i, or with PITCH to
// row i + (KS - 1) floor(i / width): `gap` = KS - 1, `inv` = ceil(2^20 / width).  By the twelve conversion warps; some 35 instructions for four
// values (with copies of single pieces by the threads, their addresses and bounds, it was 100, and the conversion bounded every kernel).
// `check` becomes NaN where this form cannot split a value: the box then goes through split_box_again.
struct SplitBox { uint32_t src; int positions; uint32_t dst, plane, block, gap, inv; };
template <int RBS, int QSHIFT, bool PITCH>
struct SplitPlaces {
  uint32_t to, byte, plane, gap, inv;
  __device__ __forceinline__ SplitPlaces(const SplitBox& b, int tid) : plane(b.plane), gap(b.gap), inv(b.inv) {
    const uint32_t q = (uint32_t)tid & ((1u << QSHIFT) - 1u);
    byte = (q & ((1u << (RBS - 3)) - 1u)) * 8;
    to = b.dst + (QSHIFT > RBS - 3 ? (q >> (RBS - 3)) * b.block : 0u);
  }
  __device__ __forceinline__ uint32_t of(int i) const {
    uint32_t row = (uint32_t)i >> QSHIFT;
    if (PITCH) row += ((row * inv) >> 20) * gap;
    return to + swizzled(RBS, row, byte);
  }
  __device__ __forceinline__ void store(uint32_t at, const Split4& s) const {
    st_shared_v2(at, s.h);
    st_shared_v2(at + plane, s.m);
    st_shared_v2(at + 2 * plane, s.l);
  }
};
// Where the converting warps take stages in turn, in teams: the slot of a ring that a team comes to next, and the parity of its lap.
struct SplitTurn {
  uint32_t at, lap, slots;
  __device__ __forceinline__ SplitTurn(uint32_t first, uint32_t n) : at(first), lap(0), slots(n) { next(0); }
  __device__ __forceinline__ void next(uint32_t teams) {
    at += teams;
    while (at >= slots) { at -= slots; lap ^= 1u; }
  }
};
template <int RBS, int QSHIFT, bool PITCH, int THREADS = SP_CONVERTERS>
__device__ __forceinline__ void split_box(const SplitBox& b, float2& check) {
  constexpr int U = 4;
  // Without PITCH the items of a thread lie ROWS rows apart, and the swizzle of every other one differs in one bit at most: the addresses are
  // constants apart, where working each out took five instructions of forty.
  constexpr uint32_t ROWS = THREADS >> QSHIFT, FLIP = ((ROWS >> (7 - RBS)) & ((1u << (RBS - 4)) - 1u)) << 4;
  static_assert(PITCH || ((FLIP == 0 || FLIP == 64) && (2 * ROWS >> (7 - RBS)) % (1u << (RBS - 4)) == 0), "two items ahead the swizzle is the same");
  const int tid = (threadIdx.x - SP_CONVERT * 32) % THREADS, items = b.positions << QSHIFT;
  const SplitPlaces<RBS, QSHIFT, PITCH> places(b, tid);
  uint32_t from = b.src + (uint32_t)tid * 16, at = PITCH ? 0u : places.of(tid);
  for (int i = tid; i < items; i += U * THREADS, from += U * THREADS * 16, at += U * ROWS << RBS) {
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u == 0 || i + u * THREADS < items) v[u] = ld_shared_f4(from + u * THREADS * 16);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (u > 0 && i + u * THREADS >= items) break;
      places.store(PITCH ? places.of(i + u * THREADS) : (u & 1 ? at ^ FLIP : at) + (u * ROWS << RBS), split4(v[u], check));
    }
  }
}
// The thread's part of a box again, any values; returns whether one is not finite.
template <int RBS, int QSHIFT, bool PITCH, int THREADS = SP_CONVERTERS>
__device__ __noinline__ bool split_box_again(const SplitBox b) {
  const int tid = (threadIdx.x - SP_CONVERT * 32) % THREADS, items = b.positions << QSHIFT;
  const SplitPlaces<RBS, QSHIFT, PITCH> places(b, tid);
  bool odd = false;
#pragma unroll 2
  for (int i = tid; i < items; i += THREADS) {
    const float4 v = ld_shared_f4(b.src + (uint32_t)i * 16);
    odd = odd || (v.x - v.x) + (v.y - v.y) + (v.z - v.z) + (v.w - v.w) != 0.f;
    places.store(places.of(i), split4_apart<Bf16Parts, false>(v));
  }
  return odd;
}
// What the converters do when a stage's tiles are written and its floats read: `again` converts them once more, where a value asks for that
// (behind the fence, whose time hides the check's).
template <class Again>
__device__ __forceinline__ void split_stage_done(uint64_t* full, uint64_t* floats_empty, float2 check, const Again& again) {
  fence_async_smem();
  const float c = check.x + check.y;
  if (c != c) {
    again();
    fence_async_smem();
  }
  __syncwarp();
  if ((threadIdx.x & 31) == 0) { mbar_arrive(full); mbar_arrive(floats_empty); }
}
// A wait by a whole warp, one lane at the barrier.  What the barrier guards is ordered before the other lanes' reads by the warp barrier (a
// shuffle orders no memory).
__device__ __forceinline__ bool split_wait(uint64_t* bar, uint32_t parity, unsigned int* status, unsigned int tag) {
  bool ok = true;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, status, tag);
  ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
  __syncwarp();
  return ok;
}
__device__ __forceinline__ void split_zero(uint32_t base, uint32_t bytes) {
  for (uint32_t i = threadIdx.x * 16; i < bytes; i += SP_THREADS * 16)
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(base + i), "r"(0) : "memory");
  fence_async_smem();
}
// What a block does between its barriers' set-up and its roles: the accumulators' columns of tensor memory (the go-ahead for the next kernel is
// given behind them), `bytes` of zeros at `at`, the wait for the kernel before, the tag of this call in the header.  Returns where the
// columns are; *go: no earlier kernel of the call ran into its time limit.
__device__ __forceinline__ uint32_t split_begin(int warp, uint32_t* slot, uint32_t columns, uint32_t at, uint32_t bytes, unsigned int* status, unsigned int tag, int* go) {
  if (warp == 1) tmem_alloc_then_trigger(slot, columns);
  if (bytes) split_zero(at, bytes);
  pdl_wait();
  if (threadIdx.x == 0) {
    *go = (*reinterpret_cast<volatile unsigned int*>(status) != tag) ? 1 : 0;
    if (blockIdx.x == 0) reinterpret_cast<volatile unsigned int*>(status)[1] = tag;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return *reinterpret_cast<volatile uint32_t*>(slot);
}
// An accumulator set's three groups of n columns added to the sums of an epilogue warp's column groups (`half`, `half` + 2 of 16).  A sum
// of products hh that is not finite counts alone.  AT_ONCE: all three groups are loaded together, where there are registers for it.  The set is
// given back to the MMAs (`empty`) as soon as it is read: they do not wait for the look at its sums.
template <class Parts, bool AT_ONCE = false>
__device__ __forceinline__ void split_add_set(uint32_t set, uint32_t n, int half, float2 (&sum)[2][8], uint64_t* empty) {
  const float2 down = make_float2(1.f / Parts::STEP, 1.f / Parts::STEP), zero = make_float2(0.f, 0.f);
  const auto pair = [](const uint32_t (&v)[16], int e) { return make_float2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])); };
  const auto give_back = [&] {
    tc_fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(empty);
  };
  if ((uint32_t)half * 16 >= n) {                    // (a warp without columns)
    give_back();
    return;
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const uint32_t c = (uint32_t)(half + 2 * k) * 16;
    if (c >= n) break;
    uint32_t x[16], y[16], z[16];
    tmem_ld16_issue(set + n + c, y);
    tmem_ld16_issue(set + 2 * n + c, z);
    if (AT_ONCE) tmem_ld16_issue(set + c, x);
    tmem_ld_wait(y); tmem_ld_wait(z);
    float2 t[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) t[e] = __ffma2_rn(pair(z, e), down, pair(y, e));
    if (!AT_ONCE) tmem_ld16_issue(set + c, x);
    tmem_ld_wait(x);
    if (k == 1 || c + 32 >= n) give_back();
    constexpr int CHECKS = AT_ONCE ? 4 : 2;          // (chains of multiply-adds: their latency counts)
    float2 check[CHECKS];                            // 0, or NaN
#pragma unroll
    for (int i = 0; i < CHECKS; ++i) check[i] = zero;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      t[e] = __ffma2_rn(t[e], down, pair(x, e));
      check[e & (CHECKS - 1)] = __ffma2_rn(t[e], zero, check[e & (CHECKS - 1)]);
    }
#pragma unroll
    for (int i = CHECKS / 2; i > 0; i >>= 1)
#pragma unroll
      for (int j = 0; j < i; ++j) check[j] = __fadd2_rn(check[j], check[j + i]);
    if (!(check[0].x + check[0].y == 0.f)) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float2 hh = pair(x, e);
        if (hh.x - hh.x != 0.f) t[e].x = hh.x;
        if (hh.y - hh.y != 0.f) t[e].y = hh.y;
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) sum[k][e] = __fadd2_rn(sum[k][e], t[e]);
  }
}
__device__ __forceinline__ float split_sum(const float2 (&sum)[2][8], int k, int e) { return e & 1 ? sum[k][e >> 1].y : sum[k][e >> 1].x; }

static inline uint32_t up1k(uint32_t v) { return (v + 1023u) & ~1023u; }
// Clocks of the three MMAs of a k-step with n columns per group: the tensor pipe's half clock per column, or shared memory's 128 bytes a clock.
static inline long split_kstep_clocks(int n) {
  long c = 0;
  for (int g = 1; g <= 3; ++g) c += std::max(g * n / 2, 32 + g * n / 4);
  return c;
}

// A tensor map over floats.
static inline bool make_map_f32(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides, const uint32_t* box,
                         CUtensorMapSwizzle swizzle) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint32_t estr[5] = {1, 1, 1, 1, 1}, bx[5];
  cuuint64_t d[5], st[4];
  for (int i = 0; i < rank; ++i) { d[i] = dims[i]; bx[i] = box[i]; }
  for (int i = 0; i + 1 < rank; ++i) st[i] = strides[i];
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, const_cast<void*>(base), d, st, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace xconv
