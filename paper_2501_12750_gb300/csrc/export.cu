// export.cu -- headless image export: the rendered colour and id planes packed
// into interleaved 8-bit RGBA with a background of chosen transparency (the
// alpha of pixels where no primitive was hit), ready to be written to an
// image file by the host.
#include "vtx_internal.h"

namespace vtx {

__device__ __forceinline__ uint32_t rgba_word(float r, float g, float b, uint32_t id, uint32_t bg_a) {
  const uint32_t x = __float2uint_rn(fminf(fmaxf(r, 0.0f), 1.0f) * 255.0f);
  const uint32_t y = __float2uint_rn(fminf(fmaxf(g, 0.0f), 1.0f) * 255.0f);
  const uint32_t z = __float2uint_rn(fminf(fmaxf(b, 0.0f), 1.0f) * 255.0f);
  return x | y << 8 | z << 16 | (id == kNoId ? bg_a : 255u) << 24;
}

// P pixels per thread and step, image blockIdx.y: three colour planes and the id plane read coalesced, one 32-bit
// RGBA word per pixel written.  HBM-bound (16 B read + 4 B written per pixel).  P = 4 (16-byte loads and stores)
// where the planes and the image allow it: 7680 x 4320 (664 MB) 102 us against 174 us at P = 1, whose four 4-byte
// loads a thread and 64-bit division by the image size a pixel keep too little in flight.
template <int P>
__global__ __launch_bounds__(256) void k_export_rgba8(const float *__restrict__ rgb, const uint32_t *__restrict__ id,
                                                      uint32_t ppi, int n_img, uint32_t bg_a,
                                                      uint32_t *__restrict__ out) {
  const uint32_t units = ppi / P, stride = gridDim.x * blockDim.x;
  for (long long img = blockIdx.y; img < n_img; img += gridDim.y) {
    const float *c = rgb + img * 3 * ppi;
    const uint32_t *d = id + img * ppi;
    uint32_t *o = out + img * ppi;
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < units; u += stride) {
      const size_t q = (size_t)u * P;
      if (P == 4) {
        const float4 r = __ldcs(reinterpret_cast<const float4 *>(c + q));
        const float4 g = __ldcs(reinterpret_cast<const float4 *>(c + ppi + q));
        const float4 b = __ldcs(reinterpret_cast<const float4 *>(c + 2 * (size_t)ppi + q));
        const uint4 i = __ldcs(reinterpret_cast<const uint4 *>(d + q));
        __stcs(reinterpret_cast<uint4 *>(o + q),
               make_uint4(rgba_word(r.x, g.x, b.x, i.x, bg_a), rgba_word(r.y, g.y, b.y, i.y, bg_a),
                          rgba_word(r.z, g.z, b.z, i.z, bg_a), rgba_word(r.w, g.w, b.w, i.w, bg_a)));
      } else {
        __stcs(o + q, rgba_word(__ldcs(c + q), __ldcs(c + ppi + q), __ldcs(c + 2 * (size_t)ppi + q), __ldcs(d + q), bg_a));
      }
    }
  }
}

cudaError_t run_export_rgba8(const float *rgb, const uint32_t *id, long long ppi, long long n_img, unsigned char bg_a,
                             uint8_t *rgba, cudaStream_t st) {
  if (ppi * n_img == 0) return cudaSuccess;
  // ppi <= 2^28.  Four pixels at a time: every image's planes then start on 16-byte boundaries
  const bool vec = ppi % 4 == 0 && (((uintptr_t)rgb | (uintptr_t)id | (uintptr_t)rgba) & 15u) == 0;
  const long long units = vec ? ppi / 4 : ppi;
  const long long cap = 8LL * sm_count();
  const long long rows = n_img < 65535 ? n_img : 65535;
  long long bx = (units + 255) / 256;
  const long long share = cap / rows > 0 ? cap / rows : 1;
  bx = bx < share ? bx : share;
  const dim3 grid((unsigned)bx, (unsigned)rows);
  if (vec)
    k_export_rgba8<4><<<grid, 256, 0, st>>>(rgb, id, (uint32_t)ppi, (int)n_img, bg_a, reinterpret_cast<uint32_t *>(rgba));
  else
    k_export_rgba8<1><<<grid, 256, 0, st>>>(rgb, id, (uint32_t)ppi, (int)n_img, bg_a, reinterpret_cast<uint32_t *>(rgba));
  return cudaGetLastError();
}

}  // namespace vtx
