// Sketch and back-probe of layers with few samples or few probes, 16-bit storage: kernels that stream one large operand
// from memory through registers.
//
// A row of the small side (16 samples, say) leaves the tcgen05 kernels one narrow MMA per 128-byte row piece, and their
// time goes with the hand-shakes of a CTA's roles per tile, a multiple of the time the bytes take.  These kernels have no
// roles, no stages and no barriers: every warp loads its operands straight into the fragments of mma.sync (16 x 8 x 16, float
// accumulators), whose rate -- far below tcgen05's, far above what is needed at 16 multiply-adds per byte -- is not
// what bounds them.  Two facts make the fragments free:
//  - the order of the reduction index is ours, as long as both operands use the same: a thread's fragments of two k-steps
//    are then 16 consecutive bytes of a row (sketch);
//  - the order of the columns is ours too: a thread that holds 8 neighbouring columns of two rows pairs them into the B
//    fragments of 8 column tiles with one byte permutation each, and its accumulators are 16 neighbouring columns of the
//    result (back-probe).
// Probing vectors redrawn from a seed are drawn into the fragments: a fragment register is two sign bits of a Philox word
// moved to bits 15 and 31, a multiplication and a logic instruction.
#include "common.cuh"
#include "tc_api.h"

#include <algorithm>

namespace xconv {

// (FREE: the compiler may move it among other instructions; the loads of the kernels with stored operands run ahead in program order.)
template <bool F16, bool FREE = false>
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
#define XC_MMA(T) "mma.sync.aligned.m16n8k16.row.col.f32." T "." T ".f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};" \
                : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1)
  if (F16) {
    if (FREE) asm(XC_MMA("f16")); else asm volatile(XC_MMA("f16"));
  } else {
    if (FREE) asm(XC_MMA("bf16")); else asm volatile(XC_MMA("bf16"));
  }
#undef XC_MMA
}
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
template <bool F16>
__device__ __forceinline__ unsigned short to16(float v) {
  if (F16) { const __half h = __float2half_rn(v); return *reinterpret_cast<const unsigned short*>(&h); }
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  return *reinterpret_cast<const unsigned short*>(&h);
}
template <bool F16>
__device__ __forceinline__ float from16(unsigned short v) {
  if (F16) return __half2float(__ushort_as_half(v));
  return __uint_as_float((uint32_t)v << 16);
}
template <bool F16>
__device__ __forceinline__ uint32_t pack16(float a, float b) { return (uint32_t)to16<F16>(a) | ((uint32_t)to16<F16>(b) << 16); }

// Two signs at bits 15 and 31 of `bits`, as two values +-1: one instruction, with both constants in registers (as constants they are put
// into two instructions).
struct SignPair { uint32_t mask, ones; };
template <bool F16>
__device__ __forceinline__ SignPair sign_pair() {
  SignPair s;
  asm volatile("mov.b32 %0, %1;" : "=r"(s.mask) : "n"(0x80008000u));
  asm volatile("mov.b32 %0, %1;" : "=r"(s.ones) : "n"(F16 ? 0x3C003C00u : 0x3F803F80u));
  return s;
}
__device__ __forceinline__ uint32_t signed_ones(uint32_t bits, const SignPair& s) {
  uint32_t v;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(v) : "r"(bits), "r"(s.mask), "r"(s.ones));       // (bits & mask) | ones
  return v;
}

// Two packed values with infinities and NaN replaced by zeros.
template <bool F16>
__device__ __forceinline__ uint32_t finite16(uint32_t v) {
  if (F16) {
    const __half2 h = *reinterpret_cast<const __half2*>(&v);
    return v & __hlt2_mask(__habs2(h), __half2(__ushort_as_half(0x7C00), __ushort_as_half(0x7C00)));
  }
  const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&v);
  return v & __hlt2_mask(__habs2(h), __nv_bfloat162(__ushort_as_bfloat16(0x7F80), __ushort_as_bfloat16(0x7F80)));
}

// What the kernels that draw signs take from constant memory: the keys of the ten rounds (added up per block they are a fifth of Philox's
// instructions), and powers of two.  Signs are moved into place by multiplications with these: what bounds the drawing is the pipe of
// shifts and logic (60 % busy, two instructions a register), and a multiplication goes to another.  (A constant factor the compiler would
// make a shift again.)
struct SignKeys {
  uint32_t key[10][2], pow2[16];
  void set(unsigned long long seed) {
    uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
    for (auto& k : key) { k[0] = k0; k[1] = k1; k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    for (int i = 0; i < 16; ++i) pow2[i] = 1u << i;
  }
};
// Philox block b (philox4x32_10 in common.cuh).
__device__ __forceinline__ uint4 sign_block(unsigned long long b, const SignKeys& s) {
  uint32_t c0 = (uint32_t)b, c1 = (uint32_t)(b >> 32), c2 = 0u, c3 = 0u;
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const unsigned long long m0 = (unsigned long long)0xD2511F53u * c0, m1 = (unsigned long long)0xCD9E8D57u * c2;
    c0 = (uint32_t)(m1 >> 32) ^ c1 ^ s.key[i][0]; c1 = (uint32_t)m1;
    c2 = (uint32_t)(m0 >> 32) ^ c3 ^ s.key[i][1]; c3 = (uint32_t)m0;
  }
  return make_uint4(c0, c1, c2, c3);
}
// The 128 sign bits of entries e0 .. e0+127 of Z (e0 a multiple of 64, `whole`: of 128).
__device__ __forceinline__ uint4 sign_bits128(unsigned long long e0, bool whole, const SignKeys& s) {
  uint4 w = sign_block(e0 >> 7, s);
  if (!whole && (e0 & 64)) {                          // the second half of this block, the first of the next
    const uint4 v = sign_block((e0 >> 7) + 1, s);
    w = make_uint4(w.z, w.w, v.x, v.y);
  }
  return w;
}

// ------------------------------------------------------------------------------------ sketch

// part[split][m][n] (or [n][m] if `swap`) = sum over this block's k of A[m,k] Bm[n,k]: 16 MT rows of A per block, up to
// 8 NT rows of Bm.  The blocks take the pieces of the k axis in turn and the eight warps the k-steps of a piece, so that at
// any time the GPU reads neighbouring bytes of every row; the warps' tiles are added in warp order.
struct SketchStream {
  const uint16_t *A, *Bm;
  float* part;
  int M, N, swap;
  long K;
  SignKeys signs;
  unsigned int *status, tag;                          // workspace header: this call is the last to use it
};

template <bool F16, int MT, int NT, bool SEEDED>
__global__ void __launch_bounds__(256, 2) sketch_stream_kernel(const SketchStream p) {
  __shared__ float red[8][16 * 8 + 1];
  __shared__ uint4 bits[SEEDED ? 8 : 1][SEEDED ? 16 * MT : 1];
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) p.status[1] = p.tag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int m0 = blockIdx.y * 16 * MT;
  float acc[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);

  if (!SEEDED) {
    // k-step of 32: thread (g, t) holds k = 8t .. 8t+7 of its rows, the pairs in order
    constexpr int U = MT * 2 + NT <= 3 ? 4 : MT * 2 + NT <= 6 ? 2 : 1;       // k-steps whose loads are in flight together
    const uint16_t* arow = p.A + (long)(m0 + g) * p.K + 8 * t;
    const uint16_t* brow = p.Bm + (long)g * p.K + 8 * t;
    for (long k0 = (long)blockIdx.x * 256 * U + warp * 32; k0 < p.K; k0 += (long)gridDim.x * 256 * U) {
      uint4 a[U][MT][2], b[U][NT];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const long k = k0 + 256 * u;
        const bool in = k + 8 * t < p.K;                                    // (K is a multiple of 8)
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            a[u][i][h] = in && m0 + 16 * i + 8 * h + g < p.M ? ldg_stream(arow + (long)(16 * i + 8 * h) * p.K + k) : zero;
#pragma unroll
        for (int j = 0; j < NT; ++j) b[u][j] = in && 8 * j + g < p.N ? ldg_stream(brow + (long)(8 * j) * p.K + k) : zero;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          const uint4 lo = a[u][i][0], hi = a[u][i][1];
          const uint32_t f0[4] = {lo.x, hi.x, lo.y, hi.y}, f1[4] = {lo.z, hi.z, lo.w, hi.w};
#pragma unroll
          for (int j = 0; j < NT; ++j) {
            mma16816<F16>(acc[i][j], f0, b[u][j].x, b[u][j].y);
            mma16816<F16>(acc[i][j], f1, b[u][j].z, b[u][j].w);
          }
        }
    }
  } else {
    // A = the signs of the seed.  128 k at a time: each lane draws one row's 128 signs (MT / 2 of them), the rows' words go
    // through shared memory.  In a step of 32 k (one word) the pairs are (s, s + 16), s = 4t .. 4t+3.
    // What bounds it: a product holds a scheduler for some 8 clocks, and the instructions beside it, 8 a product, take theirs one after
    // the other (17 of 19 clocks a product; no pipe above 43 %).  256 probes x 16 samples, 2.1 M terms 91 -> 80 us against two logic
    // instructions and an addition of keys more.
    const SignPair pm = sign_pair<F16>();
    const uint32_t place = p.signs.pow2[12 - 4 * t];
    const bool whole = (p.K & 127) == 0;
    const uint16_t* brow = p.Bm + (long)g * p.K + 4 * t;
    constexpr int DR = (16 * MT + 31) / 32;            // rows a lane draws
    uint4 drawn[DR];
    auto draw = [&](long k) {
#pragma unroll
      for (int i = 0; i < DR; ++i)
        drawn[i] = sign_bits128((unsigned long long)(m0 + 32 * i + lane) * (unsigned long long)p.K + (unsigned long long)k, whole, p.signs);
    };
    long k0 = (long)blockIdx.x * 1024 + warp * 128;
    if (k0 < p.K) draw(k0);
    for (; k0 < p.K; k0 += (long)gridDim.x * 1024) {
      uint2 x[4][NT][2];
#pragma unroll
      for (int w = 0; w < 4; ++w)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            x[w][j][h] = k0 + 32 * w < p.K && 8 * j + g < p.N                // (K is a multiple of 64)
                             ? *reinterpret_cast<const uint2*>(brow + (long)(8 * j) * p.K + k0 + 32 * w + 16 * h) : make_uint2(0u, 0u);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < DR; ++i)
        if (32 * i + lane < 16 * MT) bits[warp][32 * i + lane] = drawn[i];
      __syncwarp();
      if (k0 + (long)gridDim.x * 1024 < p.K) draw(k0 + (long)gridDim.x * 1024);      // the next piece's signs, between this one's products
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        uint32_t b[NT][4], w0[MT], w1[MT];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          const uint2 lo = x[w][j][0], hi = x[w][j][1];
          b[j][0] = __byte_perm(lo.x, hi.x, 0x5410); b[j][1] = __byte_perm(lo.x, hi.x, 0x7632);
          b[j][2] = __byte_perm(lo.y, hi.y, 0x5410); b[j][3] = __byte_perm(lo.y, hi.y, 0x7632);
        }
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          w0[i] = reinterpret_cast<const uint32_t*>(&bits[warp][16 * i + g])[w] * place;
          w1[i] = reinterpret_cast<const uint32_t*>(&bits[warp][16 * i + 8 + g])[w] * place;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)                    // all row tiles of one half, so that no product waits for the one before it
#pragma unroll
          for (int i = 0; i < MT; ++i) {
            const uint32_t c0 = p.signs.pow2[3 - 2 * h], c1 = h ? 1u : p.signs.pow2[2];
            const uint32_t f[4] = {signed_ones(w0[i] * c0, pm), signed_ones(w1[i] * c0, pm), signed_ones(w0[i] * c1, pm),
                                   signed_ones(w1[i] * c1, pm)};
#pragma unroll
            for (int j = 0; j < NT; ++j) mma16816<F16, true>(acc[i][j], f, b[j][2 * h], b[j][2 * h + 1]);
          }
      }
    }
  }
  // the warps' tiles, 16 x 8 at a time
  float* out = p.part + (long)blockIdx.x * p.M * p.N;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      __syncthreads();
#pragma unroll
      for (int e = 0; e < 4; ++e) red[warp][(g + 8 * (e >> 1)) * 8 + 2 * t + (e & 1)] = acc[i][j][e];
      __syncthreads();
      if (threadIdx.x < 128) {
        float s = red[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < 8; ++w) s += red[w][threadIdx.x];
        const int m = m0 + 16 * i + (int)threadIdx.x / 8, n = 8 * j + (int)threadIdx.x % 8;
        if (m < p.M && n < p.N) out[p.swap ? (long)n * p.M + m : (long)m * p.N + n] = s;
      }
    }
}

// ------------------------------------------------------------------------------------ back-probe

// L[row][q] = sum over k of S(row, k) * Y[k][q], rounded to storage: up to 16 MT rows, a warp owns 64 columns.  S(row, k) =
// S[row * s_row + k * s_k] (float, rounded to storage in shared memory, so that neither a transposed nor a 16-bit copy of it
// is written).
struct BackprobeStream {
  const float* S;
  long s_row, s_k;
  const uint16_t* Y;
  uint16_t* L;
  int rows, K, K16, ld;                               // K16: K rounded up to 64; ld: row pitch of S in shared memory
  long Q, groups;                                     // groups of 64 columns
  unsigned int *status, tag;
};

// S in shared memory, rounded to storage (SPLIT: as two values, the second ones at s16lo, and what the sums of a row are multiplied by in `unscale`).
template <bool F16, int MT, bool SPLIT>
__device__ __forceinline__ void stage_sketch(const BackprobeStream& p, uint16_t* s16, uint16_t* s16lo, float* unscale) {
  if (SPLIT) {
    // a warp's rows side by side, so that their loads are in flight together (one row after the other, a wait for memory
    // each: 64 rows of 5 terms 11.8 us a launch in float16)
    constexpr int R = 2 * MT;
    const int row0 = threadIdx.x >> 5, lane0 = threadIdx.x & 31;
    float up[R];
#pragma unroll
    for (int i = 0; i < R; ++i) up[i] = 1.0f;
    if (F16) {
      float most[R];
#pragma unroll
      for (int i = 0; i < R; ++i) most[i] = 0.f;
      for (int k = lane0; k < p.K; k += 32) {
        float a[R];
#pragma unroll
        for (int i = 0; i < R; ++i) a[i] = row0 + 8 * i < p.rows ? fabsf(p.S[(row0 + 8 * i) * p.s_row + k * p.s_k]) : 0.f;
#pragma unroll
        for (int i = 0; i < R; ++i)
          if (a[i] < __int_as_float(0x7F800000)) most[i] = fmaxf(most[i], a[i]);
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) most[i] = fmaxf(most[i], __shfl_xor_sync(0xffffffffu, most[i], o));
        const int e = most[i] > 0.f ? min(126, max(-126, 14 - ilogbf(most[i]))) : 0;
        up[i] = __int_as_float((127 + e) << 23);
        if (lane0 == 0) unscale[row0 + 8 * i] = __int_as_float((127 - e) << 23);
      }
    }
    for (int k = lane0; k < p.K16; k += 32) {
      float v[R];
#pragma unroll
      for (int i = 0; i < R; ++i)
        v[i] = row0 + 8 * i < p.rows && k < p.K ? p.S[(row0 + 8 * i) * p.s_row + k * p.s_k] * up[i] : 0.f;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        uint16_t hi = to16<F16>(v[i]);
        if (v[i] != 0.f && (hi & 0x7FFFu) == 0) hi |= 1u;
        const float h = from16<F16>(hi);
        s16[(row0 + 8 * i) * p.ld + k] = hi;
        s16lo[(row0 + 8 * i) * p.ld + k] = fabsf(h) < __int_as_float(0x7F800000) ? to16<F16>(v[i] - h) : (uint16_t)0;
      }
    }
  } else {
    for (int i = threadIdx.x; i < 16 * MT * p.K16; i += 256) {
      const int row = p.s_k == 1 ? i / p.K16 : i % (16 * MT), k = p.s_k == 1 ? i % p.K16 : i / (16 * MT);
      s16[row * p.ld + k] = row < p.rows && k < p.K ? to16<F16>(p.S[row * p.s_row + k * p.s_k]) : (uint16_t)0;
    }
  }
  __syncthreads();
}

// SPLIT: S as the sum of two 16-bit values, multiplied one after the other: for the layers whose sums used the float S (24 bits)
// before.  The two keep 16 bits of it in bfloat16 and 22 in float16 (where every row is scaled by a power of two into the range
// first), far below the rounding of the result: relative error against 64 bits on 76 random layers 1.6e-3 to 1.7e-3 (bfloat16)
// and 2.1e-4 (float16), 1.00001 times that of the float S at most; 2.4e-3 with S rounded once.
// Y's infinities and NaN count once, with the first value: the second is zero or of either sign, and its product with an
// infinity would make a NaN of the sum.  So an entry of S that is not zero has a first value that is not zero either.
// KC: k-steps of 16 that are loaded together.  ALL: they are the whole reduction; a warp then takes 4 / KC groups of
// columns at a time, so that as many bytes are in flight as with a long reduction.  Otherwise the loads of the next
// KC k-steps (of the next group behind the last) are under way while these are multiplied.
template <bool F16, int MT, int KC, bool ALL, bool SPLIT>
__global__ void __launch_bounds__(256, MT >= 4 ? 1 : 2) backprobe_stream_kernel(const BackprobeStream p) {
  extern __shared__ __align__(16) uint16_t s16[];     // [16 MT][ld]
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x == 0) p.status[1] = p.tag;
  __shared__ float unscale[SPLIT ? 16 * MT : 1];      // SPLIT: what the row's sums are multiplied by
  uint16_t* s16lo = s16 + 16 * MT * p.ld;             // SPLIT: the second values
  stage_sketch<F16, MT, SPLIT>(p, s16, s16lo, unscale);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  constexpr int GB = ALL ? 4 / KC : 1, VB = ALL ? GB : 2;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  float acc[MT][8][4];
  uint4 v[VB][KC][4];
  auto fetch = [&](int gb, long grp, int k0) {        // rows 2t, 2t+1, 2t+8, 2t+9 of every k-step, 8 columns of each
    const long q = grp * 64 + 8 * g;
#pragma unroll
    for (int u = 0; u < KC; ++u)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int k = k0 + 16 * u + 2 * t + (r & 1) + 8 * (r >> 1);
        v[gb][u][r] = k < p.K && q < p.Q ? ldg_stream(p.Y + (long)k * p.Q + q) : zero;
      }
  };
  auto multiply = [&](int gb, int k0) {
#pragma unroll
    for (int u = 0; u < KC; ++u) {
      uint32_t a[SPLIT ? 2 * MT : MT][4];
#pragma unroll
      for (int i = 0; i < (SPLIT ? 2 * MT : MT); ++i) {
        const uint16_t* s = s16 + (16 * i + g) * p.ld + k0 + 16 * u + 2 * t;      // (the second values follow the first)
        a[i][0] = *reinterpret_cast<const uint32_t*>(s);
        a[i][1] = *reinterpret_cast<const uint32_t*>(s + 8 * p.ld);
        a[i][2] = *reinterpret_cast<const uint32_t*>(s + 8);
        a[i][3] = *reinterpret_cast<const uint32_t*>(s + 8 * p.ld + 8);
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) {                   // column 8 g + c is column g of tile c
        uint32_t b0 = __byte_perm(word(v[gb][u][0], c >> 1), word(v[gb][u][1], c >> 1), (c & 1) ? 0x7632 : 0x5410);
        uint32_t b1 = __byte_perm(word(v[gb][u][2], c >> 1), word(v[gb][u][3], c >> 1), (c & 1) ? 0x7632 : 0x5410);
#pragma unroll
        for (int i = 0; i < MT; ++i) mma16816<F16>(acc[i][c], a[i], b0, b1);
        if (SPLIT) {
          b0 = finite16<F16>(b0); b1 = finite16<F16>(b1);
#pragma unroll
          for (int i = 0; i < MT; ++i) mma16816<F16>(acc[i][c], a[MT + i], b0, b1);
        }
      }
    }
  };
  if (!ALL) fetch(0, (long)blockIdx.x * 8 + warp, 0);
  for (long grp0 = ((long)blockIdx.x * 8 + warp) * GB; grp0 < p.groups; grp0 += (long)gridDim.x * 8 * GB) {
    if (ALL)
#pragma unroll
      for (int gb = 0; gb < GB; ++gb) fetch(gb, grp0 + gb, 0);
#pragma unroll
    for (int gb = 0; gb < GB; ++gb) {
      const long grp = grp0 + gb;
      if (grp >= p.groups) break;
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[i][c][e] = 0.f;
      if (ALL) {
        multiply(gb, 0);
      } else {
        for (int k0 = 0; k0 < p.K16; k0 += 32 * KC) {       // (K16 is a multiple of 64)
          fetch(1, grp, k0 + 16 * KC);
          multiply(0, k0);
          const bool last = k0 + 32 * KC >= p.K16;
          fetch(0, last ? grp + (long)gridDim.x * 8 : grp, last ? 0 : k0 + 32 * KC);
          // (padding of the reduction: zeros; left out by halves, a test per k-step keeps the loads from running ahead)
          if (!SPLIT || k0 + 16 * KC < p.K) multiply(1, k0 + 16 * KC);
        }
      }
      // accumulator columns 2t and 2t+1 of tile c are the columns 16 t + c and 16 t + 8 + c
      const long qo = grp * 64 + 16 * t;
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row = 16 * i + 8 * h + g;
          if (row >= p.rows) continue;
          if (SPLIT && F16) {
            const float d = unscale[row];
#pragma unroll
            for (int c = 0; c < 8; ++c) { acc[i][c][2 * h] *= d; acc[i][c][2 * h + 1] *= d; }
          }
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            if (qo + 8 * s >= p.Q) continue;
            uint4 o;
            o.x = pack16<F16>(acc[i][0][2 * h + s], acc[i][1][2 * h + s]); o.y = pack16<F16>(acc[i][2][2 * h + s], acc[i][3][2 * h + s]);
            o.z = pack16<F16>(acc[i][4][2 * h + s], acc[i][5][2 * h + s]); o.w = pack16<F16>(acc[i][6][2 * h + s], acc[i][7][2 * h + s]);
            *reinterpret_cast<uint4*>(p.L + (long)row * p.Q + qo + 8 * s) = o;
          }
        }
    }
  }
}

// The same with Y = the signs of the seed.  Bounded as the sketch that draws them (above); 16 rows, 256 terms, 2.1 M columns 96 -> 76 us, 16 rows,
// 8 terms, 3.5 M columns 45 -> 24.
template <bool F16, int MT, int GP, bool SPLIT>
__global__ void __launch_bounds__(256, MT >= 4 ? 1 : 2) backprobe_seeded_kernel(const BackprobeStream p, const __grid_constant__ SignKeys signs) {
  extern __shared__ __align__(16) uint16_t s16[];     // [16 MT][ld], then 8 warps x 32 rows x 16 bytes of signs
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x == 0) p.status[1] = p.tag;
  __shared__ float unscale[SPLIT ? 16 * MT : 1];
  stage_sketch<F16, MT, SPLIT>(p, s16, s16 + 16 * MT * p.ld, unscale);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  // S of k-step k: the first values in a[0 .. MT-1], the second ones behind
  auto load_s = [&](uint32_t (&a)[SPLIT ? 2 * MT : MT][4], int k) {
#pragma unroll
    for (int i = 0; i < (SPLIT ? 2 * MT : MT); ++i) {
      const uint16_t* s = s16 + (16 * i + g) * p.ld + k + 2 * t;
      a[i][0] = *reinterpret_cast<const uint32_t*>(s);
      a[i][1] = *reinterpret_cast<const uint32_t*>(s + 8 * p.ld);
      a[i][2] = *reinterpret_cast<const uint32_t*>(s + 8);
      a[i][3] = *reinterpret_cast<const uint32_t*>(s + 8 * p.ld + 8);
    }
  };
  // accumulator columns 2t and 2t+1 of tile c are the columns 16 t + c and 16 t + 8 + c
  auto store = [&](float (&acc)[MT][8][4], long grp) {
    const long qo = grp * 64 + 16 * t;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = 16 * i + 8 * h + g;
        if (row >= p.rows) continue;
        if (SPLIT && F16) {
          const float d = unscale[row];
#pragma unroll
          for (int c = 0; c < 8; ++c) { acc[i][c][2 * h] *= d; acc[i][c][2 * h + 1] *= d; }
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          if (qo + 8 * s >= p.Q) continue;
          uint4 o;
          o.x = pack16<F16>(acc[i][0][2 * h + s], acc[i][1][2 * h + s]); o.y = pack16<F16>(acc[i][2][2 * h + s], acc[i][3][2 * h + s]);
          o.z = pack16<F16>(acc[i][4][2 * h + s], acc[i][5][2 * h + s]); o.w = pack16<F16>(acc[i][6][2 * h + s], acc[i][7][2 * h + s]);
          *reinterpret_cast<uint4*>(p.L + (long)row * p.Q + qo + 8 * s) = o;
        }
      }
  };
  // A warp takes GP groups side by side, a whole Philox block of every row where GP is 2.  The signs of 32 rows, a row per lane, go
  // through shared memory, and the next 32 are drawn between the products of these.
  const SignPair pm = sign_pair<F16>();
  uint4* bits = reinterpret_cast<uint4*>(s16 + (SPLIT ? 2 : 1) * 16 * MT * p.ld) + warp * 32;
  const bool whole = GP == 2 && (p.Q & 127) == 0;
  for (long grp0 = ((long)blockIdx.x * 8 + warp) * GP; grp0 < p.groups; grp0 += (long)gridDim.x * 8 * GP) {
    float acc[GP][MT][8][4];
#pragma unroll
    for (int gp = 0; gp < GP; ++gp)
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[gp][i][c][e] = 0.f;
    uint4 drawn;
    auto draw = [&](int k0) {
      const unsigned long long e0 = (unsigned long long)(k0 + lane) * (unsigned long long)p.Q + (unsigned long long)(grp0 * 64);
      if (GP == 2) {
        drawn = sign_bits128(e0, whole, signs);
      } else {
        const uint4 w = sign_block(e0 >> 7, signs);
        drawn = (e0 & 64) ? make_uint4(w.z, w.w, 0u, 0u) : make_uint4(w.x, w.y, 0u, 0u);
      }
    };
    draw(0);
    for (int k0 = 0; k0 < p.K; k0 += 32) {                // (S is padded with zeros to a multiple of 64 terms)
      __syncwarp();
      bits[lane] = drawn;
      __syncwarp();
      if (k0 + 32 < p.K) draw(k0 + 32);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        uint32_t a[SPLIT ? 2 * MT : MT][4];
        load_s(a, k0 + 16 * u);
#pragma unroll
        for (int gp = 0; gp < GP; ++gp) {
          // eight signs of the two rows of a pair, at bits 0 and 16
          const uint8_t* sb = reinterpret_cast<const uint8_t*>(bits) + (16 * u + 2 * t) * 16 + 8 * gp + g;
          const uint32_t x0 = (uint32_t)sb[0] | ((uint32_t)sb[16] << 16), x1 = (uint32_t)sb[128] | ((uint32_t)sb[144] << 16);
#pragma unroll
          for (int c = 0; c < 8; ++c) {                   // column 8 g + c is column g of tile c
            const uint32_t place = signs.pow2[15 - c], b0 = signed_ones(x0 * place, pm), b1 = signed_ones(x1 * place, pm);
#pragma unroll
            for (int i = 0; i < (SPLIT ? 2 * MT : MT); ++i) mma16816<F16, true>(acc[gp][i % MT][c], a[i], b0, b1);
          }
        }
      }
    }
#pragma unroll
    for (int gp = 0; gp < GP; ++gp)
      if (grp0 + gp < p.groups) store(acc[gp], grp0 + gp);
  }
}

// ------------------------------------------------------------------------------------ host side

static long cdiv_(long a, long b) { return (a + b - 1) / b; }

// These kernels want their SM's memory as L1, where their loads in flight live.  Without the wish they were placed on SMs still
// split for the kernel before them (nearly all shared memory, for a tensor-core kernel) and kept that split as long as its CTAs
// and theirs overlapped: sketch of 4 volumes of 48^3 behind the convolution 85 -> 65 us for both, back-probe of 16 samples x 64
// probes of 256 x 256 x 32 with the contraction 105 -> 96, of 16 probes x 256 samples 116 -> 91.  (An ordinary launch, behind the end of
// the kernel before, gives the same and costs 2 us.)  The rest is shared memory for two blocks.
static cudaError_t want_l1(const void* kernel, size_t smem) {
  const int share = (int)std::min<size_t>(100, std::max<size_t>(30, 2 * (smem + 2048) * 100 / (228 * 1024) + 1));
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, share);
}

// Measured against the tcgen05 sketch, other -> this, us: 8 x 4 (probes x samples), 3.5 M terms 178 -> 22; 512 x 8, 65536 terms
// 14.5 -> 10.0; 256 x 16, 25600 terms 10.0 -> 8.0; 164 x 16, 93312 terms 13.7 -> 10.8; but 64 x 16, 2.1 M terms 76 -> 113 (a load
// instruction touches eight rows, and many rows far apart cost it more than the bytes do): more than 32 rows only up to
// 131072 terms.  With a second column tile the rows' loads are fewer in flight: 380 x 13, 91200 terms 17.0 -> 18.8, 512 x 15,
// 92160 terms 20.1 -> 22.6, so there up to 32 M values only (512 x 8, 97344 terms 21.6 -> 19.2).  (Left out by the limit: 64 x
// 16, 200704 terms 13.3 -> 11.5; 128 x 16, 262144 terms 16.3 -> 15.8.)  Redrawn from the seed only the few samples are read: 64 x
// 16 64 -> 31, 256 x 16 190 -> 90.
bool tc_plan_sketch_stream(const xconv_desc* d, bool seeded, StreamSketchPlan* p) {
  if (d->dtype != XCONV_BF16 && d->dtype != XCONV_F16) return false;
  const long K = (long)d->H * d->W * d->Cin;
  if (K % 8 != 0 || K < 2048 || std::min(d->r, d->B) > 16) return false;
  if (seeded && (d->B > 16 || K % 64 != 0)) return false;            // the signs are drawn on the row side
  p->swap = d->B <= d->r || seeded ? 0 : 1;                          // 0: rows = probes
  if (!p->swap && d->B > 16) return false;
  const int M = p->swap ? d->B : d->r, N = p->swap ? d->r : d->B;
  if (!seeded && M > 32 && (K > 131072 || (N > 8 && (long)M * K > 32000000))) return false;
  p->mt = seeded || M > 32 ? 4 : M > 16 ? 2 : 1;
  p->nt = N > 8 ? 2 : 1;
  p->tiles_m = (int)cdiv_(M, 16 * p->mt);
  // two blocks per SM, and at least one k-step of 32 per warp and block
  const long splits = std::max(1L, std::min(cdiv_(2L * 148, p->tiles_m), cdiv_(K, seeded ? 1024 : 256)));
  p->splits = (int)splits;
  p->part_bytes = (size_t)p->splits * d->r * d->B * sizeof(float);
  return true;
}

template <bool F16>
static cudaError_t launch_sketch_stream(const StreamSketchPlan& pl, bool seeded, const SketchStream& q, cudaStream_t st) {
  const dim3 grid((unsigned)pl.splits, (unsigned)pl.tiles_m), block(256);
  void (*kernel)(SketchStream) =
      seeded ? (pl.nt == 2 ? sketch_stream_kernel<F16, 4, 2, true> : sketch_stream_kernel<F16, 4, 1, true>)
      : pl.mt == 4 ? (pl.nt == 2 ? sketch_stream_kernel<F16, 4, 2, false> : sketch_stream_kernel<F16, 4, 1, false>)
      : pl.mt == 2 ? (pl.nt == 2 ? sketch_stream_kernel<F16, 2, 2, false> : sketch_stream_kernel<F16, 2, 1, false>)
                   : (pl.nt == 2 ? sketch_stream_kernel<F16, 1, 2, false> : sketch_stream_kernel<F16, 1, 1, false>);
  const cudaError_t e = want_l1(reinterpret_cast<const void*>(kernel), 12 * 1024);      // (static shared memory)
  return e != cudaSuccess ? e : launch_pdl(kernel, grid, block, 0, st, q);
}

xconv_status tc_run_sketch_stream(const xconv_desc* d, const StreamSketchPlan& pl, const void* X, const void* Z, float* part,
                                  char* ws_head, cudaStream_t st, const unsigned long long* seed) {
  SketchStream q{};
  q.status = reinterpret_cast<unsigned int*>(ws_head);
  q.tag = call_tag();
  q.A = static_cast<const uint16_t*>(pl.swap ? X : Z);
  q.Bm = static_cast<const uint16_t*>(pl.swap ? Z : X);
  q.part = part;
  q.M = pl.swap ? d->B : d->r;
  q.N = pl.swap ? d->r : d->B;
  q.swap = pl.swap;
  q.K = (long)d->H * d->W * d->Cin;
  if (seed) q.signs.set(*seed);
  const cudaError_t e = d->dtype == XCONV_F16 ? launch_sketch_stream<true>(pl, seed != nullptr, q, st)
                                              : launch_sketch_stream<false>(pl, seed != nullptr, q, st);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

static int stream_k(int K) { return (int)(cdiv_(K, 64) * 64); }
static size_t stream_smem(int mt, int K, bool seeded, bool split) {
  return (size_t)(16 * mt) * (stream_k(K) + 8) * (split ? 4 : 2) + (seeded ? 8 * 32 * 16 : 0);
}

// `other`: the tcgen05 back-probe serves the layer.  Up to 16 rows this one is faster where every warp has two groups of columns
// or the reduction is short; measured, other -> this, us: 4 rows, 8 terms, 3.5 M columns 76 -> 21; 16 rows, 64 terms, 2.1 M
// columns 76 -> 62, 256 terms 269 -> 192; but 8 rows, 512 terms, 65536 columns 14.5 -> 24; 32 rows, 128 terms, 200704 columns
// 15 -> 20; 64 rows, 128 terms, 802816 columns 56 -> 88 (mma.sync holds its pipe for some 20 clocks or more, whatever feeds it).
// Where the choice is between this and the FP32-FMA kernel: 50 rows, 50 terms, 153760 columns 61 -> 16.
bool tc_backprobe_streams(const xconv_desc* d, bool other) {
  if (d->dtype != XCONV_BF16 && d->dtype != XCONV_F16) return false;
  const long Q = (long)d->H * d->W * d->Cout;
  if (Q % 8 != 0 || Q < 2048 || d->r > 64 || stream_smem(d->r > 32 ? 4 : d->r > 16 ? 2 : 1, d->B, true, !other) > 98 * 1024) return false;
  return !other || (d->r <= 16 && (d->B <= 64 || Q >= 2L * 64 * 16 * 148));
}

// Pairs of groups draw half the blocks, but only where every warp of the grid has a group of its own all the same (16 rows: 256 terms, 2.1 M
// columns 91 -> 77 us, 498 terms, 4608 columns 28 -> 34).  Above 16 rows their accumulators would not fit the registers.
bool tc_stream_draws_pairs(const xconv_desc* d) { return d->r <= 16 && cdiv_((long)d->H * d->W * d->Cout, 64) > 8L * 148 * 2; }

template <bool F16, int MT>
static cudaError_t launch_backprobe_seeded(const BackprobeStream& q, const SignKeys& signs, bool pairs, bool split, unsigned grid, size_t smem, cudaStream_t st) {
  constexpr int PAIR = MT == 1 ? 2 : 1;
  void (*kernel)(BackprobeStream, SignKeys);
  if (split) kernel = pairs ? backprobe_seeded_kernel<F16, MT, PAIR, true> : backprobe_seeded_kernel<F16, MT, 1, true>;
  else if (MT > 1) return cudaErrorInvalidValue;
  else kernel = pairs ? backprobe_seeded_kernel<F16, 1, 2, false> : backprobe_seeded_kernel<F16, 1, 1, false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
  if (e == cudaSuccess) e = want_l1(reinterpret_cast<const void*>(kernel), smem);
  return e != cudaSuccess ? e : launch_pdl(kernel, dim3(grid), dim3(256), smem, st, q, signs);
}

template <bool F16, int MT>
static cudaError_t launch_backprobe_stream(const BackprobeStream& q, const SignKeys* signs, bool pairs, bool split, unsigned grid, size_t smem, cudaStream_t st) {
  if (signs) return launch_backprobe_seeded<F16, MT>(q, *signs, pairs, split, grid, smem, st);
  constexpr int KC = MT == 1 ? 2 : 1;
  void (*kernel)(BackprobeStream);
  if (split) kernel = backprobe_stream_kernel<F16, MT, KC, false, true>;
  else if (MT > 1) return cudaErrorInvalidValue;      // (one value per entry of S: up to 16 rows only)
  else
    kernel = q.K <= 16 ? backprobe_stream_kernel<F16, 1, 1, true, false>
             : q.K <= 32 ? backprobe_stream_kernel<F16, 1, 2, true, false>
             : q.K <= 64 ? backprobe_stream_kernel<F16, 1, 4, true, false> : backprobe_stream_kernel<F16, 1, 2, false, false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
  if (e == cudaSuccess) e = want_l1(reinterpret_cast<const void*>(kernel), smem);
  return e != cudaSuccess ? e : launch_pdl(kernel, dim3(grid), dim3(256), smem, st, q);
}

xconv_status tc_run_backprobe_stream(const xconv_desc* d, const float* S, long s_row, long s_k, const void* dY, void* L,
                                     bool split, char* ws_head, cudaStream_t st, const unsigned long long* seed) {
  BackprobeStream q{};
  q.status = reinterpret_cast<unsigned int*>(ws_head);
  q.tag = call_tag();
  q.S = S; q.s_row = s_row; q.s_k = s_k;
  q.Y = static_cast<const uint16_t*>(dY);
  q.L = static_cast<uint16_t*>(L);
  q.rows = d->r; q.K = d->B; q.K16 = stream_k(d->B); q.ld = q.K16 + 8;
  q.Q = (long)d->H * d->W * d->Cout;
  q.groups = cdiv_(q.Q, 64);
  SignKeys keys;
  if (seed) keys.set(*seed);
  const SignKeys* signs = seed ? &keys : nullptr;
  const int mt = d->r > 32 ? 4 : d->r > 16 ? 2 : 1;
  const unsigned grid = (unsigned)std::min<long>(cdiv_(q.groups, 8), 148L * (mt == 4 ? 1 : 2));
  const size_t smem = stream_smem(mt, d->B, seed != nullptr, split);
  const bool pairs = tc_stream_draws_pairs(d);
  cudaError_t e;
  if (d->dtype == XCONV_F16)
    e = mt == 4 ? launch_backprobe_stream<true, 4>(q, signs, pairs, split, grid, smem, st)
        : mt == 2 ? launch_backprobe_stream<true, 2>(q, signs, pairs, split, grid, smem, st)
                  : launch_backprobe_stream<true, 1>(q, signs, pairs, split, grid, smem, st);
  else
    e = mt == 4 ? launch_backprobe_stream<false, 4>(q, signs, pairs, split, grid, smem, st)
        : mt == 2 ? launch_backprobe_stream<false, 2>(q, signs, pairs, split, grid, smem, st)
                  : launch_backprobe_stream<false, 1>(q, signs, pairs, split, grid, smem, st);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

}  // namespace xconv
