// Direct convolution (and, with the weights read transposed and mirrored, the exact input gradient) on FP32 multiply-adds
// for float layers that neither conv_split.cu nor small_f32.cu takes (channels off the multiples of 4, circular shifts, and calls whose
// scratch is the header alone); conv_simt (simt_kernels.cuh) serves the layers too small for its tiles, and the 16-bit layers of odd
// channel counts or circular shifts.
//
//   out[b,y,x,co] = sum over (offset, ci) of w(co,ci,offset) * in[b,y+dy-p,x+dx-p,ci]
//
// A thread owns a strip of 8 pixels of one image row and 8 output channels.  Per input channel and offset row it loads the
// strip's window (8 + KS - 1 values, three 128-bit loads) once for all KS offsets, and per offset its 8 weights (two 128-bit
// loads): 64 KS multiply-adds for 3 + 2 KS loads, all of them broadcasts or conflict-free.  Of a block's THREADS threads TN
// stand side by side in the channels (8 TN channels), the THREADS / TN groups on strips of a patch of SW strips x RH rows x NI
// planes (NI > 1 for images smaller than a patch).  Input channels go by CK through shared memory, transposed so that the
// pixels of a row are consecutive; where the pixels of the patch lie in memory is worked out once (`tab`).  Two blocks of
// 256 threads per SM, so that one loads while the other multiplies, except where their shared memory allows only one (3 x 3 x 3
// layers with few channels out: up to 126 KB; the plan's cost does not know that).
// The sums are taken in the order of conv_simt (same bits).  64 -> 64 channels, 32 x 32 images, batch 128: 560 -> 236 us (41
// of the 68 TFLOP/s that register-only chains reach; three quarters of the rest is the last wave of blocks, then the
// loads); 3 -> 64 channels of 112 x 112 images 457 -> 102 us; 5 x 5, 32 channels 891 -> 155 us.
#include "conv_fma.h"

#include <algorithm>

#include "simt_kernels.cuh"

namespace xconv {


template <int KS, int KD>
__host__ __device__ constexpr int conv_fma_ck() { return KS * KS * KD >= 25 ? 4 : KS == 1 ? 16 : 8; }

template <int KS, int KD, bool DGRAD, int TN, int THREADS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) conv_fma(const float* __restrict__ in, const float* __restrict__ Wt, float* __restrict__ out,
                                                   int planes, int D, int H, int W, int Ci, int Co, int Cin_w, int circ,
                                                   const ConvFma g) {
  constexpr int P = (KS - 1) / 2, PD = (KD - 1) / 2, T = KD * KS * KS, CK = conv_fma_ck<KS, KD>(), CO = 8 * TN;
  constexpr int WIN = (8 + KS - 1 + 3) / 4 * 4;
  extern __shared__ __align__(16) float fma_smem[];
  float* Ws = fma_smem;                                // [T][CK][CO]
  float* Xs = Ws + T * CK * CO;                        // [CK][NI][KD][RH + KS - 1][pitch]
  int2* tab = reinterpret_cast<int2*>(Xs + CK * g.plane); // per position of the patch: pixel index of the input or -1, place in Xs
  const int tid = threadIdx.x;
  const int nx = (W + 8 * g.SW - 1) / (8 * g.SW), ny = (H + g.RH - 1) / g.RH;
  const int x0 = (int)(blockIdx.x % nx) * 8 * g.SW, y0 = (int)((blockIdx.x / nx) % ny) * g.RH, b0 = (int)(blockIdx.x / (nx * ny)) * g.NI;
  const int co0 = blockIdx.y * CO;
  const int width = 8 * g.SW + KS - 1, rows = g.RH + KS - 1, npos = g.NI * KD * rows * width;
  // (pixel indexes count from the block's first plane less PD, so that they fit 32 bits)
  for (int i = tid; i < npos; i += THREADS) {
    const int px = i % width, rr = (i / width) % rows, dz = (i / (width * rows)) % KD, im = i / (width * rows * KD);
    const int b = b0 + im, z = b % D + dz - PD;
    int yy = y0 + rr - P, xx = x0 + px - P;
    if (circ) { yy = wrap_index(yy, H); xx = wrap_index(xx, W); }
    const bool ok = b < planes && z >= 0 && z < D && yy >= 0 && yy < H && xx >= 0 && xx < W;
    tab[i] = make_int2(ok ? ((im + dz) * H + yy) * W + xx : -1, i / width * g.pitch + px);
  }
  const float* in0 = in + (long)(b0 - PD) * H * W * Ci;   // (only dereferenced where tab says so)
  const int tn = tid % TN, s = tid / TN, sx = s % g.SW, r = (s / g.SW) % g.RH, im = s / (g.SW * g.RH);
  float acc[8][8];
#pragma unroll
  for (int p = 0; p < 8; ++p)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[p][c] = 0.f;
  const bool vec_in = Ci % 4 == 0, vec_w = Cin_w % 4 == 0;
  __syncthreads();

  for (int ci0 = 0; ci0 < Ci; ci0 += CK) {
    // input: four channels of one pixel per step
    for (int i = tid; i < npos * (CK / 4); i += THREADS) {
      const int c4 = (i % (CK / 4)) * 4, c = ci0 + c4;
      const int2 at = tab[i / (CK / 4)];
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (at.x >= 0 && c < Ci) v = ld4_guard(in0 + (long)at.x * Ci, c, Ci, vec_in);
      float* dst = Xs + c4 * g.plane + at.y;
      dst[0] = v.x; dst[g.plane] = v.y; dst[2 * g.plane] = v.z; dst[3 * g.plane] = v.w;
    }
    if (DGRAD) {                                       // w(co, ci, t) = Wt[ci][T-1-t][co]: channels out are consecutive
      for (int i = tid; i < T * CK * (CO / 4); i += THREADS) {
        const int c4 = (i % (CO / 4)) * 4, ci = (i / (CO / 4)) % CK, t = i / (CO / 4 * CK);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ci0 + ci < Ci) v = ld4_guard(Wt + ((long)(ci0 + ci) * T + (T - 1 - t)) * Cin_w, co0 + c4, Co, vec_w);
        *reinterpret_cast<float4*>(Ws + (t * CK + ci) * CO + c4) = v;
      }
    } else {                                           // w(co, ci, t) = Wt[co][t][ci]: transposed on the way
      for (int i = tid; i < T * (CK / 4) * CO; i += THREADS) {
        const int co = i % CO, c4 = ((i / CO) % (CK / 4)) * 4, t = i / (CO * (CK / 4));
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (co0 + co < Co) v = ld4_guard(Wt + ((long)(co0 + co) * T + t) * Cin_w, ci0 + c4, Ci, vec_w);
        float* dst = Ws + (t * CK + c4) * CO + co;
        dst[0] = v.x; dst[CO] = v.y; dst[2 * CO] = v.z; dst[3 * CO] = v.w;
      }
    }
    __syncthreads();
    const float* xb = Xs + (im * KD * rows + r) * g.pitch + 8 * sx;
    const float* wb = Ws + 4 * tn;
#pragma unroll 1
    for (int ci = 0; ci < CK; ++ci, xb += g.plane, wb += CO) {
#pragma unroll
      for (int dz = 0; dz < KD; ++dz)
#pragma unroll
        for (int dy = 0; dy < KS; ++dy) {
          float xv[WIN];
#pragma unroll
          for (int i = 0; i < WIN; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(xb + (dz * rows + dy) * g.pitch + i);
            xv[i] = v.x; xv[i + 1] = v.y; xv[i + 2] = v.z; xv[i + 3] = v.w;
          }
#pragma unroll
          for (int dx = 0; dx < KS; ++dx) {
            const float* w = wb + ((dz * KS + dy) * KS + dx) * CK * CO;
            const float4 lo = *reinterpret_cast<const float4*>(w), hi = *reinterpret_cast<const float4*>(w + 4 * TN);
#pragma unroll
            for (int p = 0; p < 8; ++p) {
              const float x = xv[p + dx];
              acc[p][0] = fmaf(x, lo.x, acc[p][0]); acc[p][1] = fmaf(x, lo.y, acc[p][1]);
              acc[p][2] = fmaf(x, lo.z, acc[p][2]); acc[p][3] = fmaf(x, lo.w, acc[p][3]);
              acc[p][4] = fmaf(x, hi.x, acc[p][4]); acc[p][5] = fmaf(x, hi.y, acc[p][5]);
              acc[p][6] = fmaf(x, hi.z, acc[p][6]); acc[p][7] = fmaf(x, hi.w, acc[p][7]);
            }
          }
        }
    }
    __syncthreads();
  }
  const int b = b0 + im, y = y0 + r;
  if (b >= planes || y >= H) return;
  const bool vec_out = Co % 4 == 0;
  float* o = out + (((long)b * H + y) * W + x0 + 8 * sx) * Co;
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    if (x0 + 8 * sx + p >= W) continue;
    const int c = co0 + 4 * tn;
    if (c < Co) st4_guard(o + (long)p * Co, c, Co, vec_out, make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]));
    if (c + 4 * TN < Co) st4_guard(o + (long)p * Co, c + 4 * TN, Co, vec_out, make_float4(acc[p][4], acc[p][5], acc[p][6], acc[p][7]));
  }
}

static const int FMA_SMEM_MAX = 227 * 1024;           // (the largest plan takes 126 KB)

static long cd(long a, long b) { return (a + b - 1) / b; }

// Threads of a block, patch and channel tile by the time of the busiest SM: outputs computed there (padding counts), more per
// output where few warps share the SM, where a block or the channel tile is small (more loads per multiply-add: on the
// 64 -> 64 layer blocks of 256, 128 and 64 threads take 234, 240 and 275 us) and for the halo.
// False where conv_simt, which takes about 2.4 times as long per output (2.1 in pointwise layers: with 2.4 four layers of
// one wave and 160 to 200 channels took 20.6 -> 22.6, 26.7 -> 29.1 us) but has blocks of 2048, would be done sooner, or where
// the pixel indexes of a block would not fit 32 bits.  The least a plan below can cost is one block of 128 threads per SM, so
// small layers are told apart without the search (1 us of a 5 us call).
bool plan_conv_fma(const xconv_desc* d, bool dgrad, ConvFma* g) {
  const int K = d->KH, KD = d->KD > 1 ? d->KD : 1, Co = dgrad ? d->Cin : d->Cout;
  const long planes = (long)d->B * (d->D > 1 ? d->D : 1);
  if (d->dtype != XCONV_F32 || (long)d->H * d->W * 64 > 2000000000L) return false;
  double best = (K == 1 ? 2.1 : 2.4) * 2048.0 * (double)cd(planes * d->H * cd(d->W, 32) * cd(Co, 64), 148);
  if (best <= 64.0 * 128 * 2.0 * 1.08) return false;
  bool found = false;
  for (int threads = 256; threads >= 64; threads /= 2)
    for (int t = 8; t >= 2; t /= 2) {
      const long tiles = cd(Co, 8 * t);
      for (int sw = 1; sw <= 4; sw *= 2)
        for (int ni = 1; ni <= 8; ni *= 2) {
          const int rh = threads / t / sw / ni;
          if (rh < 1 || (ni > 1 && rh > 2 * d->H)) continue;
          const long blocks = cd(d->W, 8L * sw) * cd(d->H, rh) * cd(planes, ni) * tiles;
          if (blocks / tiles > 2000000000L) continue;
          const long per_sm = cd(blocks, 148);
          const long warps = std::min<long>(per_sm * threads, 512) / 32;
          const double halo = (double)(8 * sw + K - 1) * (rh + K - 1) / (8.0 * sw * rh);
          const double cost = 64.0 * threads * per_sm * (warps >= 16 ? 1.0 : warps >= 8 ? 1.25 : warps >= 4 ? 2.0 : 3.7) *
                              (threads == 256 ? 1.0 : threads == 128 ? 1.08 : 1.25) * (t == 8 ? 1.0 : t == 4 ? 1.06 : 1.2) * (1.0 + 0.04 * (halo - 1.0));
          if (cost >= best) continue;
          best = cost;
          found = true;
          g->threads = threads; g->tn = t;
          g->SW = sw; g->RH = rh; g->NI = ni;
          g->pitch = 8 * sw + (K > 1 ? 4 : 0);
          g->plane = ni * KD * (rh + K - 1) * g->pitch + 4;
        }
    }
  return found;
}

template <int KS, int KD, bool DGRAD, int TN, int THREADS>
static cudaError_t launch_one(const xconv_desc* d, const ConvFma& g, const float* in, const float* Wt, float* out, cudaStream_t st) {
  const int Ci = DGRAD ? d->Cout : d->Cin, Co = DGRAD ? d->Cin : d->Cout, D = d->D > 1 ? d->D : 1, planes = d->B * D;
  const size_t smem = ((size_t)KS * KS * KD * conv_fma_ck<KS, KD>() * 8 * TN + (size_t)conv_fma_ck<KS, KD>() * g.plane +
                       (size_t)2 * g.NI * KD * (g.RH + KS - 1) * (8 * g.SW + KS - 1)) * 4;
  auto kern = conv_fma<KS, KD, DGRAD, TN, THREADS>;
  // (the limit belongs to the kernel, not to this launch: the same for every patch, so that no other thread finds it lowered)
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FMA_SMEM_MAX);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)(cd(d->W, 8L * g.SW) * cd(d->H, g.RH) * cd(planes, g.NI)), (unsigned)cd(Co, 8 * TN));
  kern<<<grid, THREADS, smem, st>>>(in, Wt, out, planes, D, d->H, d->W, Ci, Co, d->Cin, d->circular, g);
  return cudaGetLastError();
}
template <int KS, int KD, bool DGRAD, int TN>
static cudaError_t launch_threads(const xconv_desc* d, const ConvFma& g, const float* in, const float* Wt, float* out, cudaStream_t st) {
  return g.threads == 256 ? launch_one<KS, KD, DGRAD, TN, 256>(d, g, in, Wt, out, st)
         : g.threads == 128 ? launch_one<KS, KD, DGRAD, TN, 128>(d, g, in, Wt, out, st)
                            : launch_one<KS, KD, DGRAD, TN, 64>(d, g, in, Wt, out, st);
}
template <int KS, int KD>
static cudaError_t launch_kernel(const xconv_desc* d, const ConvFma& g, bool dgrad, const float* in, const float* Wt, float* out,
                                 cudaStream_t st) {
  if (dgrad) return g.tn == 8 ? launch_threads<KS, KD, true, 8>(d, g, in, Wt, out, st)
                    : g.tn == 4 ? launch_threads<KS, KD, true, 4>(d, g, in, Wt, out, st) : launch_threads<KS, KD, true, 2>(d, g, in, Wt, out, st);
  return g.tn == 8 ? launch_threads<KS, KD, false, 8>(d, g, in, Wt, out, st)
         : g.tn == 4 ? launch_threads<KS, KD, false, 4>(d, g, in, Wt, out, st) : launch_threads<KS, KD, false, 2>(d, g, in, Wt, out, st);
}

xconv_status run_conv_fma(const xconv_desc* d, const ConvFma& g, bool dgrad, const float* in, const float* Wt, float* out,
                          cudaStream_t st) {
  const cudaError_t e = d->KD > 1 ? launch_kernel<3, 3>(d, g, dgrad, in, Wt, out, st)
                        : d->KH == 3 ? launch_kernel<3, 1>(d, g, dgrad, in, Wt, out, st)
                        : d->KH == 5 ? launch_kernel<5, 1>(d, g, dgrad, in, Wt, out, st) : launch_kernel<1, 1>(d, g, dgrad, in, Wt, out, st);
  count_launch();
  if (e != cudaSuccess) { set_cuda_error((int)e); return XCONV_ERR_CUDA; }
  return XCONV_OK;
}

}  // namespace xconv
