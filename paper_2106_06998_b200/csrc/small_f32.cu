// FP32 multiply-adds for float layers that are done in a few microseconds whatever the arithmetic takes: a few thousand pixels, a few channels.
// What bounds them is the chain of a block -- launch, one round of loads, the products, the stores -- and work done for padding, so the tiles are
// small, every load of a step is in flight at once (cp.async, 16 bytes, zeros outside the image), the next step's loads run under this step's products,
// and the kernels start under the kernel before them.  Operands are read by loads that see what that kernel wrote (no pointer is __restrict__).
#include "small_f32.h"

#include <algorithm>

#include "common.cuh"
#include "simt_kernels.cuh"
#include "tc_api.h"

namespace xconv {

static long cdiv_(long a, long b) { return (a + b - 1) / b; }

// ------------------------------------------------------------------------------------ convolution

// out[b,y,x,co] = sum over (offset, ci) of w(co, ci, offset) * in[b, y + dy - p, x + dx - p, ci]; weights as in conv_simt.  A block owns NS strips of
// four pixels of a row (of any rows: each strip has its window in shared memory) and CO channels; a thread four pixels, two channels and every KG-th four of the
// channels in, whose sums are added through shared memory: with KG = 4 a block takes a quarter of the strips, so that few pixels still make many blocks.
// Both operands are read four channels at a time, 6 + 6 128-bit loads for 96 multiply-adds (3 x 3).
// 8 images of 32 x 32, 16 -> 16 channels, conv_simt -> this: 11.4 -> 4.8 us, input gradient 10.5 -> 4.7; 128 -> 16 channels of 8 images of 9 x 9
// 46 -> 12.
template <int KS, int KD, bool DGRAD, int CO, int KG>
struct SmallConv {
  static constexpr int CP = CO / 2, NS = 128 / CP / KG, WIN = 4 + KS - 1, R = KD * KS, T = R * KS, CK = KG == 4 || T < 25 ? 16 : 8;
  static constexpr int X_FLOATS = NS * R * WIN * CK;
  static constexpr int W_PITCH = T * CK + 4;                    // (rows of eight lanes' channels then start in different banks)
  static constexpr int W_FLOATS = DGRAD ? CK * T * CO : CO * W_PITCH;
  static constexpr size_t SMEM = (size_t)2 * (X_FLOATS + W_FLOATS) * sizeof(float);
};

template <int KS, int KD, bool DGRAD, int CO, int KG>
__global__ void __launch_bounds__(128) small_conv_kernel(const float* in, const float* Wt, float* out, long strips, int D, int H, int W, int Ci, int Co) {
  using G = SmallConv<KS, KD, DGRAD, CO, KG>;
  constexpr int P = (KS - 1) / 2, PD = (KD - 1) / 2;
  extern __shared__ __align__(16) float small_smem[];           // [2][ X: strip, offset row, pixel, channel | W ]
  __shared__ int sx[G::NS], sy[G::NS], sz[G::NS];
  __shared__ long sb[G::NS];                                    // the strip's plane, or -1
  const int tid = threadIdx.x, per_row = (W + 3) / 4;
  if (tid < G::NS) {
    const long s = (long)blockIdx.x * G::NS + tid, row = s / per_row, plane = row / H;
    sx[tid] = (int)(s - row * per_row) * 4;
    sy[tid] = (int)(row - plane * H);
    sz[tid] = (int)(plane % D);
    sb[tid] = s < strips ? plane : -1;
  }
  __syncthreads();
  pdl_wait();
  const int co0 = blockIdx.y * CO, cp = tid % G::CP, strip = (tid / G::CP) % G::NS, kg = tid / (G::CP * G::NS);

  auto fetch = [&](int buf, int ci0) {
    float* X = small_smem + buf * (G::X_FLOATS + G::W_FLOATS);
    float* Wb = X + G::X_FLOATS;
    for (int i = tid; i < G::NS * G::R * G::WIN * (G::CK / 4); i += 128) {
      const int c = (i % (G::CK / 4)) * 4, px = (i / (G::CK / 4)) % G::WIN, rho = (i / (G::CK / 4 * G::WIN)) % G::R, s = i / (G::CK / 4 * G::WIN * G::R);
      const int dz = rho / KS - PD, y = sy[s] + rho % KS - P, x = sx[s] + px - P, z = sz[s] + dz;
      const bool ok = sb[s] >= 0 && z >= 0 && z < D && y >= 0 && y < H && x >= 0 && x < W && ci0 + c < Ci;
      cp_async16_f(X + i * 4, ok ? in + (((sb[s] + dz) * H + y) * W + x) * Ci + ci0 + c : in, ok);
    }
    if (DGRAD) {                                                // w(co, ci, t) = Wt[ci][T-1-t][co]
      for (int i = tid; i < G::CK * G::T * (CO / 4); i += 128) {
        const int co = (i % (CO / 4)) * 4, t = (i / (CO / 4)) % G::T, ci = i / (CO / 4 * G::T);
        const bool ok = ci0 + ci < Ci && co0 + co < Co;
        cp_async16_f(Wb + i * 4, ok ? Wt + ((long)(ci0 + ci) * G::T + (G::T - 1 - t)) * Co + co0 + co : Wt, ok);
      }
    } else {                                                    // w(co, ci, t) = Wt[co][t][ci]
      for (int i = tid; i < CO * G::T * (G::CK / 4); i += 128) {
        const int c = (i % (G::CK / 4)) * 4, t = (i / (G::CK / 4)) % G::T, co = i / (G::CK / 4 * G::T);
        const bool ok = ci0 + c < Ci && co0 + co < Co;
        cp_async16_f(Wb + co * G::W_PITCH + t * G::CK + c, ok ? Wt + ((long)(co0 + co) * G::T + t) * Ci + ci0 + c : Wt, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  float acc[4][2];
#pragma unroll
  for (int p = 0; p < 4; ++p) acc[p][0] = acc[p][1] = 0.f;
  fetch(0, 0);
  int buf = 0;
  for (int ci0 = 0; ci0 < Ci; ci0 += G::CK, buf ^= 1) {
    if (ci0 + G::CK < Ci) {
      fetch(buf ^ 1, ci0 + G::CK);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float* X = small_smem + buf * (G::X_FLOATS + G::W_FLOATS);
    const float* Wb = X + G::X_FLOATS;
    X += strip * G::R * G::WIN * G::CK;
#pragma unroll 1
    for (int c = 4 * kg; c < G::CK; c += 4 * KG) {
#pragma unroll(G::R > 3 ? 1 : G::R)
      for (int rho = 0; rho < G::R; ++rho) {
        float4 x[G::WIN];
#pragma unroll
        for (int i = 0; i < G::WIN; ++i) x[i] = ld4(X + (rho * G::WIN + i) * G::CK + c);
#pragma unroll
        for (int dx = 0; dx < KS; ++dx) {
          float w[4][2];                                        // [channel in][channel out]
          if (DGRAD) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float2 v = *reinterpret_cast<const float2*>(Wb + ((c + k) * G::T + rho * KS + dx) * CO + 2 * cp);
              w[k][0] = v.x; w[k][1] = v.y;
            }
          } else {
#pragma unroll
            for (int o = 0; o < 2; ++o) {
              const float4 v = ld4(Wb + (cp + o * G::CP) * G::W_PITCH + (rho * KS + dx) * G::CK + c);
              w[0][o] = v.x; w[1][o] = v.y; w[2][o] = v.z; w[3][o] = v.w;
            }
          }
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int o = 0; o < 2; ++o) {
              float a = acc[p][o];
              a = fmaf(x[p + dx].x, w[0][o], a); a = fmaf(x[p + dx].y, w[1][o], a);
              a = fmaf(x[p + dx].z, w[2][o], a); a = fmaf(x[p + dx].w, w[3][o], a);
              acc[p][o] = a;
            }
        }
      }
    }
    __syncthreads();             // all reads of this buffer are done before the copies of the step after next land in it
  }
  pdl_trigger();
  int p0 = 0, p1 = 4;                                           // the pixels that this thread writes
  if (KG == 4) {
    float* red = small_smem;                                    // [channels in][pixel, channel][thread]
    const int t = tid % (G::CP * G::NS);
#pragma unroll
    for (int p = 0; p < 4; ++p) { red[(kg * 8 + 2 * p) * 32 + t] = acc[p][0]; red[(kg * 8 + 2 * p + 1) * 32 + t] = acc[p][1]; }
    __syncthreads();
    float s0 = red[2 * kg * 32 + t], s1 = red[(2 * kg + 1) * 32 + t];
#pragma unroll
    for (int g = 1; g < 4; ++g) { s0 += red[(g * 8 + 2 * kg) * 32 + t]; s1 += red[(g * 8 + 2 * kg + 1) * 32 + t]; }
#pragma unroll
    for (int p = 0; p < 4; ++p) { acc[p][0] = s0; acc[p][1] = s1; }
    p0 = kg; p1 = kg + 1;
  }
  if (sb[strip] < 0) return;
  float* o = out + ((sb[strip] * H + sy[strip]) * W + sx[strip]) * Co + co0;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    if (p < p0 || p >= p1 || sx[strip] + p >= W) continue;
    if (DGRAD) {
      if (co0 + 2 * cp < Co) *reinterpret_cast<float2*>(o + (long)p * Co + 2 * cp) = make_float2(acc[p][0], acc[p][1]);
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (co0 + cp + i * G::CP < Co) o[(long)p * Co + cp + i * G::CP] = acc[p][i];
    }
  }
}

// Small: up to the 3000 clocks of 75 multiply-adds a clock and SM from which conv_split.cu serves.  (It would be faster up to twice that, 128 -> 128 channels,
// 8 images of 8 x 8 18 -> 15 us, but with the rounding of plain multiply-adds where that kernel has a third of it.)  Every layer below was faster here than on
// conv_fma and conv_simt: 1 x 1, 16 -> 16 channels of 128 images of 14 x 14 6.4 -> 3.3 us; 3 x 3, 96 -> 48 of 6 of 10 x 10 41 -> 11.
bool small_conv_serves(const xconv_desc* d) {
  const long planes = (long)d->B * (d->D > 1 ? d->D : 1), KD = d->KD > 1 ? d->KD : 1;
  const double macs = (double)planes * d->H * d->W * d->Cin * d->Cout * (KD * d->KH * d->KW);
  return d->dtype == XCONV_F32 && !d->circular && d->Cin % 4 == 0 && d->Cout % 4 == 0 && macs <= 3000.0 * 148 * 75;
}

template <int KS, int KD, bool DGRAD, int CO, int KG>
static cudaError_t launch_small_conv(const xconv_desc* d, const float* in, const float* Wt, float* out, cudaStream_t st) {
  using G = SmallConv<KS, KD, DGRAD, CO, KG>;
  const int Ci = DGRAD ? d->Cout : d->Cin, Co = DGRAD ? d->Cin : d->Cout, D = d->D > 1 ? d->D : 1;
  const long strips = (long)d->B * D * d->H * cdiv_(d->W, 4);
  auto kernel = small_conv_kernel<KS, KD, DGRAD, CO, KG>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3((unsigned)cdiv_(strips, G::NS), (unsigned)cdiv_(Co, CO)), dim3(128), G::SMEM, st, in, Wt, out, strips, D, d->H, d->W, Ci, Co);
}
template <int KS, int KD, bool DGRAD>
static cudaError_t launch_small_conv(const xconv_desc* d, const float* in, const float* Wt, float* out, cudaStream_t st) {
  const int Co = DGRAD ? d->Cin : d->Cout;
  const long strips = (long)d->B * (d->D > 1 ? d->D : 1) * d->H * cdiv_(d->W, 4), blocks = cdiv_(strips, Co <= 16 ? 16 : 8) * cdiv_(Co, Co <= 16 ? 16 : 32);
  const bool split = blocks <= 148;                             // (8 images of 32 x 32, 16 -> 16 channels, 128 blocks: 5.3 -> 4.8 us; 784 blocks 3.8 -> 5.5)
  if (Co <= 16) return split ? launch_small_conv<KS, KD, DGRAD, 16, 4>(d, in, Wt, out, st) : launch_small_conv<KS, KD, DGRAD, 16, 1>(d, in, Wt, out, st);
  return split ? launch_small_conv<KS, KD, DGRAD, 32, 4>(d, in, Wt, out, st) : launch_small_conv<KS, KD, DGRAD, 32, 1>(d, in, Wt, out, st);
}
template <int KS, int KD>
static cudaError_t launch_small_conv(const xconv_desc* d, bool dgrad, const float* in, const float* Wt, float* out, cudaStream_t st) {
  return dgrad ? launch_small_conv<KS, KD, true>(d, in, Wt, out, st) : launch_small_conv<KS, KD, false>(d, in, Wt, out, st);
}

static xconv_status launched(cudaError_t e) {
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

xconv_status run_small_conv(const xconv_desc* d, bool dgrad, const float* in, const float* Wt, float* out, cudaStream_t st) {
  return launched(d->KD > 1 ? launch_small_conv<3, 3>(d, dgrad, in, Wt, out, st)
                  : d->KH == 3 ? launch_small_conv<3, 1>(d, dgrad, in, Wt, out, st)
                  : d->KH == 5 ? launch_small_conv<5, 1>(d, dgrad, in, Wt, out, st) : launch_small_conv<1, 1>(d, dgrad, in, Wt, out, st));
}

// ------------------------------------------------------------------------------------ contraction

// part[split][m][offset][n] = sum over the split's (probe, row, 32 pixels) of L[j,y,x,m] * Z[j,y+dy-p,x+dx-p,n] (contract_simt's sums).  A block owns
// 16 x 16 channels and a row of planes of offsets (all of a planar kernel's), a thread one pair of channels and all offsets, whose window of Z slides along the
// row in registers: KS + 1 loads for KS * KS multiply-adds.  8 probes of 32 x 32, 16 -> 16 channels, contract_simt_async -> this: 11.6 -> 4.7 us.
constexpr int SC_X = 32;
template <int KS, int KD>
__global__ void __launch_bounds__(256) small_contract_kernel(const float* L, const float* Z, float* part, long items, long items_per_split, int D, int H, int W, int Cin, int Cout,
                                                             int circ) {
  constexpr int P = (KS - 1) / 2, PD = (KD - 1) / 2, ZW = SC_X + KS - 1, T = KS * KS, TALL = KD * T;
  __shared__ __align__(16) float Ls[2][SC_X][16], Zs[2][KS][ZW][16];
  const int tid = threadIdx.x, n = tid & 15, m = tid >> 4;
  const int nblocks = (Cin + 15) / 16, kz = blockIdx.x / nblocks, n0 = (int)(blockIdx.x % nblocks) * 16, m0 = blockIdx.y * 16;
  const int chunks = (W + SC_X - 1) / SC_X;
  const long ib = (long)blockIdx.z * items_per_split, ie = min(items, ib + items_per_split);
  // coordinates of the item whose tiles are fetched next
  int xc = (int)(ib % chunks), y = (int)((ib / chunks) % H);
  long jz = ib / ((long)chunks * H);                            // plane: probe * D + z
  int z = (int)(jz % D);
  pdl_wait();
  auto fetch = [&](int buf) {
    const int x0 = xc * SC_X;
    for (int i = tid; i < SC_X * 4; i += 256) {
      const int c = (i & 3) * 4, px = i >> 2;
      const bool ok = x0 + px < W && m0 + c < Cout;
      cp_async16_f(&Ls[buf][px][c], ok ? L + ((jz * H + y) * W + x0 + px) * Cout + m0 + c : L, ok);
    }
    const int zz = z + kz - PD;
    for (int i = tid; i < KS * ZW * 4; i += 256) {
      const int c = (i & 3) * 4, px = (i >> 2) % ZW, dy = (i >> 2) / ZW;
      int yy = y + dy - P, xx = x0 + px - P;
      if (circ) { yy = wrap_index(yy, H); xx = wrap_index(xx, W); }
      const bool ok = zz >= 0 && zz < D && yy >= 0 && yy < H && xx >= 0 && xx < W && n0 + c < Cin;
      cp_async16_f(&Zs[buf][dy][px][c], ok ? Z + (((jz + kz - PD) * H + yy) * W + xx) * Cin + n0 + c : Z, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (++xc == chunks) { xc = 0; if (++y == H) { y = 0; ++jz; if (++z == D) z = 0; } }
  };
  float acc[KS][KS];
#pragma unroll
  for (int i = 0; i < KS; ++i)
#pragma unroll
    for (int j = 0; j < KS; ++j) acc[i][j] = 0.f;
  int buf = 0;
  if (ib < ie) fetch(0);
  for (long it = ib; it < ie; ++it, buf ^= 1) {
    if (it + 1 < ie) {
      fetch(buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    float w[KS][KS];                                            // Z at offsets (dy, dx) of the pixel
#pragma unroll
    for (int dy = 0; dy < KS; ++dy)
#pragma unroll
      for (int dx = 1; dx < KS; ++dx) w[dy][dx] = Zs[buf][dy][dx - 1][n];
#pragma unroll 8
    for (int px = 0; px < SC_X; ++px) {
      const float l = Ls[buf][px][m];
#pragma unroll
      for (int dy = 0; dy < KS; ++dy) {
#pragma unroll
        for (int dx = 0; dx + 1 < KS; ++dx) w[dy][dx] = w[dy][dx + 1];
        w[dy][KS - 1] = Zs[buf][dy][px + KS - 1][n];
#pragma unroll
        for (int dx = 0; dx < KS; ++dx) acc[dy][dx] = fmaf(l, w[dy][dx], acc[dy][dx]);
      }
    }
    __syncthreads();             // all reads of this buffer are done before the copies of the item after next land in it
  }
  pdl_trigger();
  if (m0 + m >= Cout || n0 + n >= Cin) return;
  float* o = part + ((long)blockIdx.z * Cout * TALL + (long)(m0 + m) * TALL + kz * T) * Cin + n0 + n;
#pragma unroll
  for (int dy = 0; dy < KS; ++dy)
#pragma unroll
    for (int dx = 0; dx < KS; ++dx) o[(long)(dy * KS + dx) * Cin] = acc[dy][dx];
}

// (A 16 x 16 block takes a fifth of the instructions of a 32 x 64 one.)
bool small_contract_serves(const xconv_desc* d) {
  return d->dtype == XCONV_F32 && d->Cin % 4 == 0 && d->Cout % 4 == 0 && cdiv_(d->Cin, 16) * cdiv_(d->Cout, 16) <= 5 * cdiv_(d->Cin, 64) * cdiv_(d->Cout, 32);
}

template <int KS, int KD>
static cudaError_t launch_small_contract(const xconv_desc* d, int splits, long items_per_split, const float* L, const float* Z, float* part, cudaStream_t st) {
  const int D = d->D > 1 ? d->D : 1;
  const dim3 grid((unsigned)(cdiv_(d->Cin, 16) * KD), (unsigned)cdiv_(d->Cout, 16), (unsigned)splits);
  return launch_pdl(small_contract_kernel<KS, KD>, grid, dim3(256), 0, st, L, Z, part, (long)d->r * D * d->H * cdiv_(d->W, SC_X), items_per_split, D, d->H, d->W, d->Cin, d->Cout,
                    d->circular);
}

xconv_status run_small_contract(const xconv_desc* d, int splits, long items_per_split, const float* L, const float* Z, float* part, cudaStream_t st) {
  return launched(d->KD > 1 ? launch_small_contract<3, 3>(d, splits, items_per_split, L, Z, part, st)
                  : d->KH == 3 ? launch_small_contract<3, 1>(d, splits, items_per_split, L, Z, part, st)
                  : d->KH == 5 ? launch_small_contract<5, 1>(d, splits, items_per_split, L, Z, part, st) : launch_small_contract<1, 1>(d, splits, items_per_split, L, Z, part, st));
}

}  // namespace xconv
