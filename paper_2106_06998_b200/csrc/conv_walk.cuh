// How the tensor-core convolutions (conv_tc.cu, conv_split.cu) see a layer and walk over it.
#pragma once

#include "tc_api.h"

namespace xconv {

// A walk over a CTA's run of items: the patch under way and its first pixel.  A step costs a few additions (the roles of
// a CTA walk on their critical paths; decoding every item by divisions took them some 300 clocks each).
template <class Params>
struct CvWalk {
  uint32_t it, end, patch, tn;
  int x, y, z, b;
  __device__ __forceinline__ CvWalk(const Params& p, uint32_t i0, uint32_t i1) : it(i0), end(i1) {
    tn = i0 / p.patches;
    patch = i0 - tn * p.patches;
    const uint32_t a = patch / (uint32_t)p.patches_x, c = a / (uint32_t)p.patches_y, e = c / (uint32_t)p.depth;
    x = (int)(patch - a * p.patches_x) * p.pw;
    y = (int)(a - c * p.patches_y) * p.ph;
    z = (int)(c - e * p.depth);
    b = (int)e;
  }
  __device__ __forceinline__ int unit(const Params& p) const {      // patches of the unit that starts here
    return (int)min(min((uint32_t)p.m_sub, end - it), p.patches - patch);
  }
  __device__ __forceinline__ void step(const Params& p) {
    ++it;
    if (++patch == p.patches) { patch = 0; ++tn; x = y = z = b = 0; return; }
    x += p.pw;
    if (x < p.patches_x * p.pw) return;
    x = 0; y += p.ph;
    if (y < p.patches_y * p.ph) return;
    y = 0;
    if (++z == p.depth) { z = 0; ++b; }
  }
};

// The image the kernel sees: a 1 x 1 kernel has no neighbours, so all pixels of the batch are one row of one image.
struct ConvGeo { long W, H, D, B; };
static ConvGeo conv_geo(const xconv_desc* d) {
  const long depth = d->D > 1 ? d->D : 1, kd = d->KD > 1 ? d->KD : 1;
  if (kd == 1 && d->KH == 1 && (long)d->B * depth * d->H * d->W < (1L << 31) - 256) return {(long)d->B * depth * d->H * d->W, 1, 1, 1};
  if (kd == 1) return {d->W, d->H, 1, (long)d->B * depth};        // a planar kernel takes every plane as an image
  return {d->W, d->H, depth, d->B};
}

}  // namespace xconv
