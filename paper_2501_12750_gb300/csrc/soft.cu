// soft.cu -- soft-edge (differentiable) sphere renderer, forward and backward.
//
// Per pixel, the spheres whose signed pixel distance to their silhouette is
// at least -4 px are composited front to back in centre-depth order (ties:
// smaller id):
//   delta = (r - sqrt(rho^2 + 1e-12)) f / z_c        (rho: centre-to-ray distance)
//   alpha = min(0.99, sigmoid(delta / sigma))
//   g     = sqrt(max(r^2 - rho^2, 0) + eta^2) - eta,  eta = 0.05 r
//   t_i   = t_c - g / |u|         (smoothed entry depth; t_c = closest approach)
//   n_i   = (t_i u - C) / r
//   w_i = alpha_i T_i, T_{i+1} = T_i (1 - alpha_i), stop once T < 1e-4;
//   coverage = sum w_i, depth = sum w_i t_i, normal = sum w_i n_i.
// Binning (cull with 4 px dilation, precise setup, per-tile counting sort)
// is shared with the hard-edge path.  Then
//   k_soft_sort  one CTA per non-empty tile orders its list by (centre depth
//        key, id) in shared memory (bucket pass plus per-bucket insertion sort;
//        in global memory for lists longer than shared memory holds) and
//        writes it back; other CTAs fill the planes of the empty tiles;
//   k_soft_fwd   each warp takes (tile, 8x4 block) items from a queue, longest
//        lists first, and walks the sorted list on its own, staging 32 entries
//        at a time -- those that can reach its pixels, in pairs -- with their
//        per-sphere constants (f / z_c, 1 / r and a bound on rho^2 that rejects
//        most before any square root or division), and takes a pair per step
//        on the paired FP32 pipes.  It can leave per pixel its final
//        transmittance and last contributor (the state);
//   k_soft_bwd   likewise over the forward's sorted lists or rebuilt ones: it
//        takes the last contributor and final transmittance from the state, or
//        re-walks each pixel front to back for them, then walks back to front
//        with the carry R_i = alpha_{i+1} c_{i+1} + (1 - alpha_{i+1}) R_{i+1},
//        recovering T_i from T_{i+1} / (1 - alpha_i) (alpha <= 0.99 keeps this
//        safe), and accumulates d/d(x, y, z, r) per sphere as a warp sum (one
//        reduce-scatter of nine shuffles per pair) and one 16-byte FP32 atomic
//        per sphere and warp.
#include "vtx_internal.h"

namespace vtx {

cudaError_t run_binning(const Geometry &g, const Scene &sc, const Scratch &s, cudaStream_t st, StageEvents *evs,
                        bool soft);

constexpr int kSoftCap = 4096;
constexpr int kSoftNT = 256;
constexpr float kTStop = 1e-4f;
constexpr float kAMax = 0.99f;

// The entries of a warp's window as its pixel loop reads them: pairs of consecutive kept entries (a, b), every field
// of both side by side, so that a 16-byte read gives two fields of the pair ready for the paired FP32 pipes.  A field
// of entry e (0 or 1) of pair p is at float 2 (field) + e of pair p's seven 16-byte words.
enum SoftField {
  kFU0h, kFU0l,      // projected reference point x (pixels), double-float, negated
  kFV0h, kFV0l,      // and y
  kFK, kFDz,         // A per pixel at zr; zr - centre depth
  kFZr, kFRad,       // reference depth; radius
  kFFz, kFInvRad,    // f / centre depth; 1 / radius
  kFEta, kFRej2,     // 0.05 radius; bound on rho^2 of a used sphere
  kFRpx2, kFPos,     // rej2 / k^2 (px^2) when dz = 0, else +inf: the pixel-distance pre-test; list position (int bits)
  kSoftFields
};
static_assert(kSoftFields == 14, "seven 16-byte words");
constexpr int kPairWords = kSoftFields / 2;  // 112 bytes: pairs start 28 banks apart, so staging stores conflict 2-way
constexpr int kWindowBytes = 2048;           // per warp: 16 pairs and 32 atom ids
static_assert(16 * kPairWords * 16 + 32 * 4 <= kWindowBytes, "a window");

struct SoftWindow {
  float4 *pair;     // [16][kPairWords]
  uint32_t *id;     // [32] atom of each kept entry
  __device__ __forceinline__ explicit SoftWindow(unsigned char *warp_base)
      : pair(reinterpret_cast<float4 *>(warp_base)),
        id(reinterpret_cast<uint32_t *>(warp_base + 16 * kPairWords * 16)) {}
  __device__ __forceinline__ float *slot(int s) const {  // field f of kept entry s at slot(s)[2 f]
    return reinterpret_cast<float *>(pair + (s >> 1) * kPairWords) + (s & 1);
  }
};

// Per-pixel ray constants.
struct SoftPix {
  PixRay r;
  float inv_uu, inv_un;  // 1 / |u|^2, 1 / |u|
};

__device__ __forceinline__ SoftPix soft_pix(const ViewParams &v, int px, int py) {
  SoftPix x;
  x.r = pix_ray(v, px, py);
  x.inv_uu = 1.0f / x.r.uu;
  x.inv_un = 1.0f / sqrtf(x.r.uu);
  return x;
}

// The soft terms of a pair of spheres for one pixel (x: sphere a, y: sphere b); false where delta < -4 px.
struct SoftPair {
  bool ha, hb;
  int posa, posb;          // list positions
  float2 ovx, ovy, dz;     // ray origin minus centre (internal frame)
  float2 sst;              // ray parameter of the closest approach, relative to zr
  float2 rho2s, irho;      // rho^2 + 1e-12 and its inverse root
  float2 delta, sg, alpha, m, ism, t, nx, ny, nz;  // n: internal frame
  float2 fz, inv_rad, eta, rad;
};

__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// nl2s = -log2(e) / sigma, so that exp(-delta / sigma) = 2^(delta nl2s).  Every product-sum is one paired operation;
// lane for lane they are the operations of one sphere's term.
__device__ __forceinline__ void soft_pair(const float4 *w, const SoftPix &x, float nl2s, bool act, SoftPair &o) {
  const PixRay &r = x.r;
  const float4 u = w[0], v = w[1], rp = w[6];
  const float2 ox = __fadd2_rn(__fadd2_rn(bc2(r.pxc), make_float2(u.x, u.y)), make_float2(u.z, u.w));
  const float2 oyn = __fadd2_rn(__fadd2_rn(make_float2(v.x, v.y), bc2(-r.pyc)), make_float2(v.z, v.w));  // minus oy
  const float2 d2 = __ffma2_rn(ox, ox, __fmul2_rn(oyn, oyn));
  const float2 lim = __fmul2_rn(make_float2(rp.x, rp.y), bc2(r.uu));
  o.ha = act && !(d2.x > lim.x);  // pixel-distance pre-test
  o.hb = act && !(d2.y > lim.y);
  if (!(o.ha || o.hb)) return;
  o.posa = __float_as_int(rp.z);
  o.posb = __float_as_int(rp.w);
  const float4 kd = w[2], zr = w[3], fi = w[4], er = w[5];
  const float2 k = make_float2(kd.x, kd.y);
  o.dz = make_float2(kd.z, kd.w);
  o.rad = make_float2(zr.z, zr.w);
  o.fz = make_float2(fi.x, fi.y);
  o.inv_rad = make_float2(fi.z, fi.w);
  o.eta = make_float2(er.x, er.y);
  o.ovx = __fmul2_rn(k, ox);  // local_o
  o.ovy = __fmul2_rn(k, oyn);
  const float2 ou = __ffma2_rn(o.ovx, bc2(r.a), __ffma2_rn(o.ovy, bc2(r.b), o.dz));
  const float2 oo = __ffma2_rn(o.ovx, o.ovx, __ffma2_rn(o.ovy, o.ovy, __fmul2_rn(o.dz, o.dz)));
  o.sst = __fmul2_rn(ou, bc2(-x.inv_uu));
  float2 rho2 = __ffma2_rn(ou, o.sst, oo);  // |o|^2 - (o.u)^2 / |u|^2
  rho2 = make_float2(fmaxf(rho2.x, 0.0f), fmaxf(rho2.y, 0.0f));
  o.ha = o.ha && !(rho2.x > er.z);
  o.hb = o.hb && !(rho2.y > er.w);
  o.rho2s = __fadd2_rn(rho2, bc2(1e-12f));
  // hardware approximations (relative errors near 1e-7; the outputs' tolerance is 5e-5): sqrt as x rsqrt(x),
  // the sigmoid through ex2.approx and rcp.approx
  o.irho = make_float2(rsqrt_approx(o.rho2s.x), rsqrt_approx(o.rho2s.y));
  o.delta = __fmul2_rn(__ffma2_rn(neg2(o.rho2s), o.irho, o.rad), o.fz);
  o.ha = o.ha && o.delta.x >= -4.0f;
  o.hb = o.hb && o.delta.y >= -4.0f;
  const float2 ex = __fmul2_rn(o.delta, bc2(nl2s));
  const float2 den = __fadd2_rn(bc2(1.0f), make_float2(exp2_approx(ex.x), exp2_approx(ex.y)));
  o.sg = make_float2(rcp_approx(den.x), rcp_approx(den.y));
  o.alpha = make_float2(fminf(kAMax, o.sg.x), fminf(kAMax, o.sg.y));
  const float2 m = __ffma2_rn(o.rad, o.rad, neg2(rho2));
  o.m = make_float2(fmaxf(m.x, 0.0f), fmaxf(m.y, 0.0f));
  const float2 m2 = __ffma2_rn(o.eta, o.eta, o.m);
  o.ism = make_float2(rsqrt_approx(m2.x), rsqrt_approx(m2.y));
  const float2 g = __ffma2_rn(m2, o.ism, neg2(o.eta));
  const float2 si = __ffma2_rn(neg2(g), bc2(x.inv_un), o.sst);  // smoothed entry, relative to zr
  o.t = __fadd2_rn(make_float2(zr.x, zr.y), si);
  o.nx = __fmul2_rn(__ffma2_rn(si, bc2(r.a), o.ovx), o.inv_rad);
  o.ny = __fmul2_rn(__ffma2_rn(si, bc2(r.b), o.ovy), o.inv_rad);
  o.nz = __fmul2_rn(__fadd2_rn(o.dz, si), o.inv_rad);
}

// A warp's share of a tile: an 8x4 pixel block, lane l its pixel (l & 7, l >> 3), and the tile's list.
struct SoftTile {
  int img, px, py, m;
  float col0, row0;  // centre of the block's first pixel
  bool inside;
  const unsigned long long *list;  // the tile's entries in (centre-depth key, id) order
};

__device__ __forceinline__ uint32_t soft_count(const uint32_t *__restrict__ tile_count,
                                               const uint32_t *__restrict__ tile_start, long long gt,
                                               unsigned long long cap_entries, uint32_t &start) {
  uint32_t cnt = tile_count[gt];
  start = tile_start[gt];
  if ((unsigned long long)start >= cap_entries) cnt = 0;
  else if ((unsigned long long)start + cnt > cap_entries) cnt = (uint32_t)(cap_entries - start);
  return cnt;
}

__device__ __forceinline__ SoftTile soft_block(const Geometry &g, long long gt, int blk,
                                               const unsigned long long *__restrict__ entries,
                                               unsigned long long cap_entries, const uint32_t *__restrict__ tile_count,
                                               const uint32_t *__restrict__ tile_start) {
  SoftTile T;
  const int lane = threadIdx.x & 31;
  T.img = (int)(gt / g.tiles_per_img);
  const int t = (int)(gt % g.tiles_per_img);
  const int px0 = (t % g.tiles_x) * 16 + 8 * (blk & 1), py0 = (t / g.tiles_x) * 16 + 4 * (blk >> 1);
  T.px = px0 + (lane & 7);
  T.py = py0 + (lane >> 3);
  T.col0 = (float)px0 + 0.5f;
  T.row0 = (float)py0 + 0.5f;
  T.inside = T.px < g.W && T.py < g.H;
  uint32_t start;
  T.m = (int)soft_count(tile_count, tile_start, gt, cap_entries, start);
  T.list = entries + start;
  return T;
}

// Exact ascending order of a tile's m entries (centre-depth key << 32 | id)
// in s_e.  A one-pass counting sort first places the entries into 1024 buckets
// of the tile's key range by a monotone FP32 map (every key of a bucket is <=
// every key of a later bucket, and equal keys share a bucket); each thread
// then insertion-sorts its four buckets.  A tile whose fullest bucket holds more
// than 32 entries is finished by a bitonic sort instead.  src is the list in
// global memory (read three times, L1 hits after the first); s_off (2 bytes
// per entry) is scratch.  1024 buckets because the insertion sorts took 60 % of
// the cycles at 256 (lists of 540 entries on average: fullest bucket 11).
constexpr int kSoftBuckets = 1024;
__device__ __forceinline__ void soft_order(const unsigned long long *__restrict__ src, int m,
                                           unsigned long long *s_e, uint16_t *s_off) {
  constexpr int NB = kSoftBuckets, PER = NB / kSoftNT;
  __shared__ uint32_t s_cnt[NB], s_red[3], s_wt[kSoftNT / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (int i = threadIdx.x; i < m; i += kSoftNT) {
    const uint32_t k = (uint32_t)(src[i] >> 32);
    lo = min(lo, k);
    hi = max(hi, k);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
#pragma unroll
  for (int j = 0; j < PER; ++j) s_cnt[threadIdx.x * PER + j] = 0u;
  if (threadIdx.x == 0) {
    s_red[0] = 0xffffffffu;
    s_red[1] = 0u;
    s_red[2] = 0u;
  }
  __syncthreads();
  if (lane == 0) {
    atomicMin(s_red, lo);
    atomicMax(s_red + 1, hi);
  }
  __syncthreads();
  lo = s_red[0];
  hi = s_red[1];
  const float scale = (float)NB / ((float)(hi - lo) + 1.0f);
  for (int i = threadIdx.x; i < m; i += kSoftNT) {
    const uint32_t k = (uint32_t)(src[i] >> 32);
    s_off[i] = (uint16_t)atomicAdd(s_cnt + min(NB - 1, (int)((float)(k - lo) * scale)), 1u);
  }
  __syncthreads();
  uint32_t c[PER], sum = 0u, cm = 0u;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    c[j] = s_cnt[threadIdx.x * PER + j];
    sum += c[j];
    cm = max(cm, c[j]);
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  const uint32_t cmax = __reduce_max_sync(0xffffffffu, cm);
  if (lane == 31) s_wt[wid] = inc;
  if (lane == 0) atomicMax(s_red + 2, cmax);
  __syncthreads();
  uint32_t base = inc - sum;
  for (int w = 0; w < wid; ++w) base += s_wt[w];
  uint32_t at = base;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    s_cnt[threadIdx.x * PER + j] = at;
    at += c[j];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += kSoftNT) {
    const unsigned long long e = src[i];
    const uint32_t k = (uint32_t)(e >> 32);
    s_e[s_cnt[min(NB - 1, (int)((float)(k - lo) * scale))] + s_off[i]] = e;
  }
  const bool small = s_red[2] <= 32u;
  __syncthreads();
  if (small) {
    // the thread's buckets follow one another, so no entry moves past the start of its own bucket
    for (int i = (int)base + 1; i < (int)(base + sum); ++i) {
      const unsigned long long x = s_e[i];
      int j = i - 1;
      while (j >= (int)base && s_e[j] > x) {
        s_e[j + 1] = s_e[j];
        --j;
      }
      s_e[j + 1] = x;
    }
    __syncthreads();
    return;
  }
  int n2 = 1;
  while (n2 < m) n2 <<= 1;
  for (int i = m + threadIdx.x; i < n2; i += kSoftNT) s_e[i] = ~0ull;
  __syncthreads();
  for (int k = 2; k <= n2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < n2; i += kSoftNT) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = s_e[i], b2 = s_e[ixj];
          const bool up = (i & k) == 0;
          if ((a > b2) == up) {
            s_e[i] = b2;
            s_e[ixj] = a;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Ascending order of a list too long for shared memory, sorted in place in global memory by the whole CTA:
// a bitonic network written with ascending comparisons only (each stage first compares i with
// i ^ (k - 1), then i with i + j), so that padding the list to a power of two with virtual +inf entries
// never moves anything: no element is compared with a partner at or beyond m.
__device__ __noinline__ void soft_sort_global(unsigned long long *a, int m) {
  int n2 = 1;
  while (n2 < m) n2 <<= 1;
  const int half = n2 >> 1;
  for (int k = 2; k <= n2; k <<= 1) {
    const int hk = k >> 1;
    for (int t = threadIdx.x; t < half; t += blockDim.x) {
      const int i = (t / hk) * k + (t % hk);
      const int q = i ^ (k - 1);
      if (q < m) {
        const unsigned long long x = a[i], y = a[q];
        if (x > y) {
          a[i] = y;
          a[q] = x;
        }
      }
    }
    __syncthreads();
    for (int j = k >> 2; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < half; t += blockDim.x) {
        const int i = (t / j) * 2 * j + (t % j);
        const int q = i + j;
        if (q < m) {
          const unsigned long long x = a[i], y = a[q];
          if (x > y) {
            a[i] = y;
            a[q] = x;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Zeros (state: full transmittance, no contributor) into the planes of empty tile gt, by one warp: whole 64-byte rows of
// eight (state: 128-byte rows of four) tile rows per store.  vec: every row starts on a 16-byte boundary and holds a
// multiple of four pixels.
__device__ __forceinline__ void soft_fill_tile(const Geometry &g, long long gt, bool vec, float *cov, float *dep,
                                               float *nrm, uint2 *state) {
  const int lane = threadIdx.x & 31;
  const int img = (int)(gt / g.tiles_per_img), t = (int)(gt % g.tiles_per_img);
  const int px0 = (t % g.tiles_x) * 16, py0 = (t / g.tiles_x) * 16;
  const long long ppi = g.pix_per_img;
  float *plane[5] = {cov + img * ppi, dep + img * ppi, nrm + img * 3 * ppi, nrm + (img * 3 + 1) * ppi,
                     nrm + (img * 3 + 2) * ppi};
  uint2 *st = state ? state + img * ppi : nullptr;
  const uint32_t one = __float_as_uint(1.0f);
  if (vec) {
    const int px = px0 + 4 * (lane & 3), sx = px0 + 2 * (lane & 7);
    for (int y = lane >> 2; y < 16; y += 8)
      if (px < g.W && py0 + y < g.H)
#pragma unroll
        for (int q = 0; q < 5; ++q)
          *reinterpret_cast<float4 *>(plane[q] + (long long)(py0 + y) * g.W + px) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (st)
      for (int y = lane >> 3; y < 16; y += 4)
        if (sx < g.W && py0 + y < g.H)
          *reinterpret_cast<uint4 *>(st + (long long)(py0 + y) * g.W + sx) = make_uint4(one, 0u, one, 0u);
  } else {
    const int px = px0 + (lane & 15);
    for (int y = lane >> 4; y < 16; y += 2) {
      if (px >= g.W || py0 + y >= g.H) continue;
      const long long p = (long long)(py0 + y) * g.W + px;
      for (int q = 0; q < 5; ++q) plane[q][p] = 0.0f;
      if (st) st[p] = make_uint2(one, 0u);
    }
  }
}

// Orders the lists of the n_list non-empty tiles in place: n_sort CTAs take every n_sort-th of them, longest first.  With
// output planes (the forward), every warp of the CTAs behind them fills one tile's planes if it is empty.  n_sort is
// bounded (a CTA per tile of the image, most of which ended at once, made a backward that rebuilds the lists of four
// views at 4096x4096 take 898 us instead of 664, and the forward 1125 instead of 865).
__global__ __launch_bounds__(kSoftNT) void k_soft_sort(Geometry g, unsigned long long *entries,
                                                      unsigned long long cap_entries,
                                                      const uint32_t *__restrict__ tile_count,
                                                      const uint32_t *__restrict__ tile_start,
                                                      const uint32_t *__restrict__ tile_list, long long pitch,
                                                      Status *status, unsigned n_sort, float *cov, float *dep, float *nrm,
                                                      uint2 *state, int vec) {
  pdl_enter();
  __shared__ unsigned long long s_e[kSoftCap];
  __shared__ uint16_t s_off[kSoftCap];
  if (blockIdx.x >= n_sort) {
    const long long gt = (long long)(blockIdx.x - n_sort) * (kSoftNT / 32) + (threadIdx.x >> 5);
    if (gt < (long long)g.n_img * g.tiles_per_img && tile_count[gt] == 0u)
      soft_fill_tile(g, gt, vec != 0, cov, dep, nrm, state);
    return;
  }
  const uint32_t n_list = status->n_list;
  const TileOrder order(status, pitch);
  for (uint32_t li = blockIdx.x; li < n_list; li += n_sort) {
    const long long gt = order.tile(tile_list, pitch, li);
    uint32_t start;
    const int m = (int)soft_count(tile_count, tile_start, gt, cap_entries, start);
    if (threadIdx.x == 0) atomicMax(&status->max_list, (unsigned)m);
    if (m == 0) continue;
    if (m > kSoftCap) {
      soft_sort_global(entries + start, m);
      continue;
    }
    __syncthreads();  // the previous list has left shared memory
    soft_order(entries + start, m, s_e, s_off);
    for (int i = threadIdx.x; i < m; i += kSoftNT) entries[start + i] = s_e[i];
  }
}

// Each warp walks the sorted list on its own (no block barrier after the
// sort, so a warp of saturated pixels never waits for a warp of silhouette
// pixels): it stages 32 entries at a time, lane i converting entry c0 + i, in
// its private 32-slot window of shared memory.
//
// Staging also culls the window for the warp.  The warp covers an 8x4 pixel
// block (lane l at column l & 7, row l >> 3); `am` marks the lanes still
// compositing.  For a sphere whose reference
// point is its centre (dz = 0) the offset at the reference depth is
// o = k (du, -dv, 0) with (du, dv) the pixel offset from the projected centre,
// and rho^2 = |o|^2 - (o.u)^2 / |u|^2 >= |o|^2 / |u|^2 (Cauchy-Schwarz on the
// x, y part), so rho^2 > rej2 whenever k^2 d^2 > rej2 |u|^2_max.  Entries whose
// disc of that radius misses the bounding rectangle of the active lanes'
// pixel centres are dropped from the returned mask; the radius is widened
// (0.01 % plus 1e-3 px plus 2e-7 of the coordinates) to cover FP32 rounding.
// The record index of entry j of the tile's list (0 outside it); loaded two windows ahead of its use, and the record
// itself brought into L1 one window ahead.
__device__ __forceinline__ uint32_t soft_rec_index(const Geometry &g, const uint32_t *__restrict__ rec_of,
                                                   const SoftTile &T, int j) {
  return (j >= 0 && j < T.m) ? rec_of[(long long)T.img * g.n_atoms + (uint32_t)T.list[j]] : 0u;
}
__device__ __forceinline__ void soft_prefetch(const PrimRec *__restrict__ recs, uint32_t ridx) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(recs + ridx));
}

// Stages the window [c0, c0 + 32): the entries that lanes `am` can use (and lists before `end`), in order, as pairs;
// returns their number.  An odd last entry is paired with one that no pixel accepts.
__device__ __forceinline__ int soft_stage(const PrimRec *__restrict__ recs, uint32_t ridx, const SoftTile &T, int c0,
                                          int end, float f, const SoftWindow &W, unsigned am, float col0, float row0,
                                          float uu_max) {
  const int lane = threadIdx.x & 31;
  const int j = c0 + lane;
  bool keep = false;
  PrimRec p;
  float fz = 0.0f, rej2 = 0.0f;
  if (j < end) {
    p = recs[ridx];
    fz = f / (p.zr - p.dz);
    // delta >= -4 px needs sqrt(rho^2) <= rad + 4 / fz; the bound is widened by
    // 0.05 % so that rounding never drops a sphere the exact test keeps.
    const float reach = p.rad + 4.0f / fz;
    rej2 = reach * reach * 1.001f + 1e-6f;
    const unsigned cols = (am | (am >> 8) | (am >> 16) | (am >> 24)) & 0xffu;
    const unsigned rows = ((am & 0xffu) ? 1u : 0u) | ((am & 0xff00u) ? 2u : 0u) | ((am & 0xff0000u) ? 4u : 0u) |
                          ((am & 0xff000000u) ? 8u : 0u);
    const float rx0 = col0 + (float)(__ffs(cols) - 1), rx1 = col0 + (float)(31 - __clz(cols));
    const float ry0 = row0 + (float)(__ffs(rows) - 1), ry1 = row0 + (float)(31 - __clz(rows));
    const float cu = p.u0h + p.u0l, cv = p.v0h + p.v0l;
    const float dx = fmaxf(fmaxf(rx0 - cu, cu - rx1), 0.0f);
    const float dy = fmaxf(fmaxf(ry0 - cv, cv - ry1), 0.0f);
    const float r2 = rej2 * uu_max;  // approximate root and quotient: the 0.01 % widening covers their error
    const float rt = __fdividef(r2 * rsqrtf(r2), p.k) * 1.0001f + 1e-3f + 2e-7f * (fabsf(cu) + fabsf(cv));
    keep = p.dz != 0.0f || !(dx * dx + dy * dy > rt * rt);
  }
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  const int n = __popc(m);
  const int at = __popc(m & ((1u << lane) - 1u));
  if (keep) {
    float *s = W.slot(at);
    s[2 * kFU0h] = -p.u0h;
    s[2 * kFU0l] = -p.u0l;
    s[2 * kFV0h] = p.v0h;
    s[2 * kFV0l] = p.v0l;
    s[2 * kFK] = p.k;
    s[2 * kFDz] = p.dz;
    s[2 * kFZr] = p.zr;
    s[2 * kFRad] = p.rad;
    s[2 * kFFz] = fz;
    s[2 * kFInvRad] = 1.0f / p.rad;
    s[2 * kFEta] = 0.05f * p.rad;
    s[2 * kFRej2] = rej2;
    // with dz = 0 the offset is o = k (dx, -dy, 0) and rho^2 >= |o|^2 / |u|^2 (Cauchy-Schwarz on its x, y part),
    // so d^2 > rej2 |u|^2 / k^2 (d: pixel distance to the projected centre) rejects the sphere; the 0.1 % in
    // rej2 covers the FP32 rounding of this quotient
    s[2 * kFRpx2] = p.dz == 0.0f ? rej2 / (p.k * p.k) : __int_as_float(0x7f800000);
    s[2 * kFPos] = __int_as_float(j);
    W.id[at] = p.id;
  }
  if ((n & 1) && lane < kSoftFields) W.slot(n)[2 * lane] = lane == kFRpx2 ? -1.0f : 0.0f;
  __syncwarp();
  return n;
}

// state (optional, [n_img][H][W]): per pixel the final transmittance (float
// bits) and 1 + the sorted-list position of its last contributor (0: none),
// which lets the backward pass start its back-to-front walk directly.
// The forward of one warp's block.
__device__ __forceinline__ void soft_fwd_walk(const Geometry &g, const SoftTile &T, const PrimRec *__restrict__ recs,
                                              const uint32_t *__restrict__ rec_of, Status *status, float *cov,
                                              float *dep, float *nrm, uint2 *state, const SoftWindow &W) {
  const ViewParams &v = g.views[T.img % g.n_views];
  const SoftPix x = soft_pix(v, T.px, T.py);
  const float inv_sigma = 1.0f / g.sigma;
  const float nl2s = -1.4426950408889634f * inv_sigma;  // exp(-delta / sigma) = 2^(delta nl2s)
  const float uu_max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x.r.uu)));
  const int lane = threadIdx.x & 31;
  float A = 0.0f, D = 0.0f, N0 = 0.0f, N1 = 0.0f, N2 = 0.0f, Tr = 1.0f;
  int last = -1;
  unsigned used = 0u;
  bool done = !T.inside;
  {
    uint32_t ridx = soft_rec_index(g, rec_of, T, lane), next = soft_rec_index(g, rec_of, T, 32 + lane);
    for (int c0 = 0; c0 < T.m; c0 += 32) {
      const unsigned am = __ballot_sync(0xffffffffu, !done);
      if (am == 0u) break;
      const uint32_t next2 = soft_rec_index(g, rec_of, T, c0 + 64 + lane);  // in flight during this window
      soft_prefetch(recs, next);
      const int n = soft_stage(recs, ridx, T, c0, T.m, v.f, W, am, T.col0, T.row0, uu_max);
      ridx = next;
      next = next2;
      for (int q = 0; q < n; q += 2) {
        SoftPair o;
        soft_pair(W.pair + (q >> 1) * kPairWords, x, nl2s, !done, o);
        if (o.ha) {
          const float w = o.alpha.x * Tr;
          A += w;
          D = fmaf(w, o.t.x, D);
          N0 = fmaf(w, o.nx.x, N0);
          N1 = fmaf(w, o.ny.x, N1);
          N2 = fmaf(-w, o.nz.x, N2);
          Tr *= 1.0f - o.alpha.x;
          last = o.posa;
          ++used;
          if (Tr < kTStop) done = true;
        }
        if (o.hb && !done) {
          const float w = o.alpha.y * Tr;
          A += w;
          D = fmaf(w, o.t.y, D);
          N0 = fmaf(w, o.nx.y, N0);
          N1 = fmaf(w, o.ny.y, N1);
          N2 = fmaf(-w, o.nz.y, N2);
          Tr *= 1.0f - o.alpha.y;
          last = o.posb;
          ++used;
          if (Tr < kTStop) done = true;
        }
      }
      __syncwarp();
    }
  }
  // composited terms, one atomic per warp (the algorithmic work of the pass)
  const unsigned wused = __reduce_add_sync(0xffffffffu, used);
  if (lane == 0 && wused) atomicAdd(&status->n_terms, (unsigned long long)wused);
  if (T.inside) {
    if (state)
      state[(long long)T.img * g.pix_per_img + (long long)T.py * g.W + T.px] =
          make_uint2(__float_as_uint(Tr), (uint32_t)(last + 1));
    const long long ppi = g.pix_per_img;
    const long long p = (long long)T.py * g.W + T.px;
    cov[(long long)T.img * ppi + p] = A;
    dep[(long long)T.img * ppi + p] = D;
    float *nb = nrm + (long long)T.img * 3 * ppi + p;
    nb[0] = N0;
    nb[ppi] = N1;
    nb[2 * ppi] = N2;
  }
}

// Warps take (tile, 8x4 block) items from a queue: the non-empty tiles longest first, eight blocks each.  No step needs
// the whole tile, so a warp that finishes its block early takes the next item instead of waiting for the tile's
// slowest warp (a quarter of the time with a CTA per tile, of 20,000 atoms from 16 views), and the sort before it keeps
// neither its registers nor its shared memory.
// Forward CTAs per SM: 3 (80 registers).  Bound by issue and the pairs' dependent steps (65 % of the issue slots, 21 of 32
// lanes).
//
// 20,000 atoms from 16 views at 512x512: 143 us after 38 us of sorting and filling, forward call 229 us; 284 us with a
// CTA per tile that sorted, walked and (empty ones) filled; 309 us with one entry per step on the scalar pipes.
#ifndef VTX_SOFT_FWD_MINB
#define VTX_SOFT_FWD_MINB 3
#endif
__global__ __launch_bounds__(kSoftNT, VTX_SOFT_FWD_MINB) void k_soft_fwd(Geometry g, const PrimRec *__restrict__ recs,
                                                      const uint32_t *__restrict__ rec_of,
                                                      const unsigned long long *__restrict__ entries,
                                                      unsigned long long cap_entries,
                                                      const uint32_t *__restrict__ tile_count,
                                                      const uint32_t *__restrict__ tile_start,
                                                      const uint32_t *__restrict__ tile_list, long long pitch,
                                                      Status *status, float *cov, float *dep, float *nrm,
                                                      uint2 *state) {
  pdl_enter();
  __shared__ __align__(16) unsigned char s_win[(kSoftNT / 32) * kWindowBytes];  // a window per warp
  const SoftWindow W(s_win + (threadIdx.x >> 5) * kWindowBytes);
  const int lane = threadIdx.x & 31;
  const uint32_t n_items = status->n_list * 8u;
  const TileOrder order(status, pitch);
  for (;;) {
    uint32_t item = 0u;
    if (lane == 0) item = atomicAdd(&status->tile_next, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) break;
    const SoftTile T = soft_block(g, order.tile(tile_list, pitch, item >> 3), (int)(item & 7u), entries, cap_entries,
                                  tile_count, tile_start);
    soft_fwd_walk(g, T, recs, rec_of, status, cov, dep, nrm, state, W);
    __syncwarp();
  }
}

// Sums over the warp of four per-lane values of sphere a and four of sphere b, scattered: lanes 0, 4, 8, 12 receive
// a's sums in order and lanes 16, 20, 24, 28 b's (nine shuffles).
__device__ __forceinline__ float warp_sum8_scatter(const float2 (&v)[4], int lane) {
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0, h4 = (lane & 4) != 0;
  float k[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    k[c] = h16 ? v[c].y : v[c].x;
    k[c] += __shfl_xor_sync(0xffffffffu, h16 ? v[c].x : v[c].y, 16);
  }
  float p0 = h8 ? k[2] : k[0], p1 = h8 ? k[3] : k[1];
  p0 += __shfl_xor_sync(0xffffffffu, h8 ? k[0] : k[2], 8);
  p1 += __shfl_xor_sync(0xffffffffu, h8 ? k[1] : k[3], 8);
  float s = h4 ? p1 : p0;
  s += __shfl_xor_sync(0xffffffffu, h4 ? p0 : p1, 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// The backward of one warp's block; W is the warp's window.
__device__ __forceinline__ void soft_bwd_walk(const Geometry &g, const SoftTile &T,
                                              const PrimRec *__restrict__ recs, const uint32_t *__restrict__ rec_of,
                                              const float *gcov, const float *gdep, const float *gnrm,
                                              const uint2 *__restrict__ state, float *grad, const SoftWindow &W) {
  const ViewParams &v = g.views[T.img % g.n_views];
  const SoftPix x = soft_pix(v, T.px, T.py);
  const PixRay &r = x.r;
  const float inv_sigma = 1.0f / g.sigma;
  const float nl2s = -1.4426950408889634f * inv_sigma;
  const long long ppi = g.pix_per_img;
  const long long p = (long long)T.py * g.W + T.px;
  float gA = 0.0f, gD = 0.0f;
  float3 gN = make_float3(0.0f, 0.0f, 0.0f);
  if (T.inside) {
    const long long q = (long long)T.img * ppi + p;
    if (gcov) gA = gcov[q];
    if (gdep) gD = gdep[q];
    if (gnrm) {
      const float *b = gnrm + (long long)T.img * 3 * ppi + p;
      gN = make_float3(b[0], b[ppi], -b[2 * ppi]);  // to the internal frame
    }
  }
  const bool need = T.inside && (gA != 0.0f || gD != 0.0f || gN.x != 0.0f || gN.y != 0.0f || gN.z != 0.0f);
  // pass 1: front to back, last contributor and final transmittance (read from the forward call's state
  // when it left one)
  const float uu_max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(r.uu)));
  float Tr = 1.0f;
  int last = -1;
  bool done = !need;
  if (state) {
    if (need) {
      const uint2 sv = state[(long long)T.img * ppi + p];
      Tr = __uint_as_float(sv.x);
      last = min((int)sv.y - 1, T.m - 1);
    }
    done = true;
  }
  const int lane = threadIdx.x & 31;
  if (!__all_sync(0xffffffffu, done)) {
    uint32_t ridx = soft_rec_index(g, rec_of, T, lane), next = soft_rec_index(g, rec_of, T, 32 + lane);
    for (int c0 = 0; c0 < T.m; c0 += 32) {
      const unsigned am = __ballot_sync(0xffffffffu, !done);
      if (am == 0u) break;
      const uint32_t next2 = soft_rec_index(g, rec_of, T, c0 + 64 + lane);
      soft_prefetch(recs, next);
      const int n = soft_stage(recs, ridx, T, c0, T.m, v.f, W, am, T.col0, T.row0, uu_max);
      ridx = next;
      next = next2;
      for (int q = 0; q < n; q += 2) {
        SoftPair o;
        soft_pair(W.pair + (q >> 1) * kPairWords, x, nl2s, !done, o);
        if (o.ha) {
          Tr *= 1.0f - o.alpha.x;
          last = o.posa;
          if (Tr < kTStop) done = true;
        }
        if (o.hb && !done) {
          Tr *= 1.0f - o.alpha.y;
          last = o.posb;
          if (Tr < kTStop) done = true;
        }
      }
      __syncwarp();
    }
  }
  const int wlast = __reduce_max_sync(0xffffffffu, last);
  if (wlast < 0) return;
  // pass 2: back to front, a pair per step, its later sphere first; per-sphere sums leave the warp as one 16-byte
  // atomic
  const float ugn0 = fmaf(r.a, gN.x, fmaf(r.b, gN.y, gN.z));
  float R = 0.0f, Tc = Tr;
  const int w0 = (wlast / 32) * 32;
  uint32_t ridx = soft_rec_index(g, rec_of, T, w0 + lane), prev = soft_rec_index(g, rec_of, T, w0 - 32 + lane);
  for (int c0 = w0; c0 >= 0; c0 -= 32) {
    const unsigned am = __ballot_sync(0xffffffffu, last >= c0);
    const uint32_t prev2 = soft_rec_index(g, rec_of, T, c0 - 64 + lane);  // in flight during this window
    soft_prefetch(recs, prev);
    const uint32_t cur = ridx;
    ridx = prev;
    prev = prev2;
    if (am == 0u) continue;
    const int n = soft_stage(recs, cur, T, c0, wlast + 1, v.f, W, am, T.col0, T.row0, uu_max);
    for (int q = (n - 1) & ~1; q >= 0; q -= 2) {
      const float4 *pw = W.pair + (q >> 1) * kPairWords;
      float2 gr[4];  // d/d(x, y, z) in the internal frame and d/dr, of spheres a and b
      bool nz = false;
      SoftPair o;
      soft_pair(pw, x, nl2s, c0 <= last, o);
      o.ha = o.ha && o.posa <= last;
      o.hb = o.hb && o.posb <= last;
      if (o.ha || o.hb) {
        // c_i, then back to front through the pair: b, then a
        float2 ci = __ffma2_rn(bc2(gD), o.t, bc2(gA));
        const float2 gn = __ffma2_rn(bc2(gN.x), o.nx, __ffma2_rn(bc2(gN.y), o.ny, __fmul2_rn(bc2(gN.z), o.nz)));
        ci = __fadd2_rn(ci, gn);
        float2 w = make_float2(0.0f, 0.0f), dal = w;
        if (o.hb) {
          const float Ti = Tc / (1.0f - o.alpha.y);
          w.y = o.alpha.y * Ti;
          dal.y = Ti * (ci.y - R);
          R = o.alpha.y * ci.y + (1.0f - o.alpha.y) * R;
          Tc = Ti;
        }
        if (o.ha) {
          const float Ti = Tc / (1.0f - o.alpha.x);
          w.x = o.alpha.x * Ti;
          dal.x = Ti * (ci.x - R);
          R = o.alpha.x * ci.x + (1.0f - o.alpha.x) * R;
          Tc = Ti;
        }
        float2 dadd = __fmul2_rn(__fmul2_rn(o.sg, __fadd2_rn(bc2(1.0f), neg2(o.sg))), bc2(inv_sigma));
        dadd = make_float2(o.sg.x < kAMax ? dadd.x : 0.0f, o.sg.y < kAMax ? dadd.y : 0.0f);
        const float2 ddf = __fmul2_rn(__fmul2_rn(dal, dadd), o.fz);
        // closest-approach offset minus q = (o + s u) - C, |q|^2 = rho^2
        const float2 qx = __ffma2_rn(o.sst, bc2(r.a), o.ovx), qy = __ffma2_rn(o.sst, bc2(r.b), o.ovy);
        const float2 qz = __fadd2_rn(o.dz, o.sst);
        // delta(C, r): d delta / dC = minus q's offset over rho, d delta / d zc = -delta / zc = -delta fz / f
        const float2 dq = __fmul2_rn(ddf, o.irho);
        gr[0] = __fmul2_rn(dq, qx);
        gr[1] = __fmul2_rn(dq, qy);
        gr[2] = __ffma2_rn(dq, qz, __fmul2_rn(__fmul2_rn(neg2(ddf), o.delta), bc2(v.inv_f)));
        gr[3] = ddf;
        // t_i(C, r) and n_i = (t_i u - C) / r
        const float2 c2 = make_float2(o.m.x > 0.0f ? -o.ism.x * x.inv_un : 0.0f,
                                      o.m.y > 0.0f ? -o.ism.y * x.inv_un : 0.0f);  // 2 (dg / drho^2) / |u|
        float2 dg = __ffma2_rn(__ffma2_rn(bc2(0.05f), o.eta, o.rad), o.ism, bc2(-0.05f));
        dg = make_float2(o.m.x > 0.0f ? dg.x : 0.0f, o.m.y > 0.0f ? dg.y : 0.0f);
        const float2 dtx = __ffma2_rn(c2, qx, bc2(r.a * x.inv_uu)), dty = __ffma2_rn(c2, qy, bc2(r.b * x.inv_uu));
        const float2 dtz = __ffma2_rn(c2, qz, bc2(x.inv_uu)), dtr = __fmul2_rn(neg2(dg), bc2(x.inv_un));
        const float2 ut = __fmul2_rn(w, bc2(gD));
        // through the depth and the normal alike: (w gD + w (u.gN) / r) dt, and -w gN / r for the centre itself
        const float2 wr = __fmul2_rn(w, o.inv_rad), s = __ffma2_rn(wr, bc2(ugn0), ut), mwr = neg2(wr);
        gr[0] = __fadd2_rn(gr[0], __ffma2_rn(s, dtx, __fmul2_rn(mwr, bc2(gN.x))));
        gr[1] = __fadd2_rn(gr[1], __ffma2_rn(s, dty, __fmul2_rn(mwr, bc2(gN.y))));
        gr[2] = __fadd2_rn(gr[2], __ffma2_rn(s, dtz, __fmul2_rn(mwr, bc2(gN.z))));
        gr[3] = __fadd2_rn(gr[3], __ffma2_rn(s, dtr, __fmul2_rn(mwr, gn)));
#pragma unroll
        for (int c = 0; c < 4; ++c) gr[c] = make_float2(o.ha ? gr[c].x : 0.0f, o.hb ? gr[c].y : 0.0f);
        nz = gr[0].x != 0.0f || gr[1].x != 0.0f || gr[2].x != 0.0f || gr[3].x != 0.0f || gr[0].y != 0.0f ||
             gr[1].y != 0.0f || gr[2].y != 0.0f || gr[3].y != 0.0f;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) gr[c] = make_float2(0.0f, 0.0f);
      }
      if (__any_sync(0xffffffffu, nz)) {
        const float sum = warp_sum8_scatter(gr, lane);
        const float sy = __shfl_down_sync(0xffffffffu, sum, 4);
        const float sz = __shfl_down_sync(0xffffffffu, sum, 8);
        const float sr = __shfl_down_sync(0xffffffffu, sum, 12);
        const int e = q + (lane >> 4);
        if ((lane & 15) == 0 && e < n) {
          const float4 wv = make_float4(v.R[0] * sum + v.U[0] * sy + v.F[0] * sz,
                                        v.R[1] * sum + v.U[1] * sy + v.F[1] * sz,
                                        v.R[2] * sum + v.U[2] * sy + v.F[2] * sz, sr);
          if (wv.x != 0.0f || wv.y != 0.0f || wv.z != 0.0f || wv.w != 0.0f)
            atomicAdd(reinterpret_cast<float4 *>(grad) + W.id[e], wv);
        }
      }
    }
    __syncwarp();  // every lane is done with the window before it is refilled
  }
}

// Items and queue as the forward's.
// Bound by each warp's chain of pairs and by issue (59 % of the slots at 24 % of the warps, 19 of 32 lanes; on small
// problems 21 % of the slots, the chain alone).  CTAS per SM: two (120 registers, nothing spilled) up to 32,768 tiles,
// where the chain counts, three (80 registers) above, where items are short and many and their waits count.  At 2 / 3 /
// 4: 1,000 atoms from 16 views at 256x256 85 / 101 / 114 us, 20,000 from 16 views at 512x512 336 / 331 / 395, at 1024x1024
// 391 / 361 / 395, 20,000 from 4 views at 4096x4096 489 / 424 / 404, 2,000 from 8 at 2048x2048 156 / 143 / 139.  One
// entry per step, its atom id read from the list in global memory, took 362 us at 512x512 (348 at 4096x4096).
template <int CTAS>
__global__ __launch_bounds__(kSoftNT, CTAS) void k_soft_bwd(Geometry g, const PrimRec *__restrict__ recs,
                                                            const uint32_t *__restrict__ rec_of,
                                                            const unsigned long long *__restrict__ entries,
                                                            unsigned long long cap_entries,
                                                            const uint32_t *__restrict__ tile_count,
                                                            const uint32_t *__restrict__ tile_start,
                                                            const uint32_t *__restrict__ tile_list, long long pitch,
                                                            Status *status,
                                                            const float *gcov, const float *gdep, const float *gnrm,
                                                            const uint2 *__restrict__ state, float *grad) {
  pdl_enter();
  __shared__ __align__(16) unsigned char s_win[(kSoftNT / 32) * kWindowBytes];  // a window per warp
  const SoftWindow W(s_win + (threadIdx.x >> 5) * kWindowBytes);
  const int lane = threadIdx.x & 31;
  const uint32_t n_items = status->n_list * 8u;
  const TileOrder order(status, pitch);
  for (;;) {
    uint32_t item = 0u;
    if (lane == 0) item = atomicAdd(&status->soft_next, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) break;
    const SoftTile T = soft_block(g, order.tile(tile_list, pitch, item >> 3), (int)(item & 7u), entries, cap_entries,
                                  tile_count, tile_start);
    if (T.m > 0) soft_bwd_walk(g, T, recs, rec_of, gcov, gdep, gnrm, state, grad, W);
    __syncwarp();
  }
}

cudaError_t run_soft_pipeline(const Geometry &g, const Scene &sc, const Scratch &s, float *cov, float *depth,
                              float *normal, const float *g_cov, const float *g_depth, const float *g_normal,
                              float *grad, uint2 *state, bool reuse_lists, cudaStream_t st, StageEvents *evs) {
  const bool reuse = reuse_lists && grad != nullptr;
  if (reuse) {
    // the lists, records and tile order of the forward call are still in place; only the backward's tile
    // queue counter (which the forward leaves untouched) is reset
    cudaMemsetAsync(&s.status->soft_next, 0, sizeof(s.status->soft_next), st);
  } else {
    cudaError_t e = run_binning(g, sc, s, st, evs, true);
    if (e != cudaSuccess) return e;
  }
  const long long n_tiles = (long long)g.n_img * g.tiles_per_img, pitch = tile_pitch(n_tiles);
  const bool fwd = grad == nullptr;
  if (!reuse) {
    const bool vec = fwd && g.W % 4 == 0 &&
                     ((uintptr_t)cov | (uintptr_t)depth | (uintptr_t)normal | (uintptr_t)state) % 16 == 0;
    // sorting CTAs: about three times as many as are resident (44 KB of shared memory each); then, forward, a filling
    // warp per tile
    const long long most = 16LL * sm_count(), n_sort = n_tiles < most ? n_tiles : most;
    const long long fill = fwd ? (n_tiles + kSoftNT / 32 - 1) / (kSoftNT / 32) : 0;
    launch_pdl(k_soft_sort, (unsigned)(n_sort + fill), kSoftNT, 0, st, g, s.entries, s.cap_entries, s.tile_count,
               s.tile_start, s.tile_list, pitch, s.status, n_sort, cov, depth, normal, state, vec ? 1 : 0);
  }
  // persistent CTAs: as many as are resident at once, never more than eight items of a tile each
  const int ctas = fwd ? VTX_SOFT_FWD_MINB : (n_tiles > 32768 ? 3 : 2);
  const long long most = (long long)ctas * sm_count();
  const unsigned grid = (unsigned)(n_tiles < most ? n_tiles : most);
  if (fwd) {
    launch_pdl(k_soft_fwd, grid, kSoftNT, 0, st, g, s.recs, s.rec_of, s.entries, s.cap_entries, s.tile_count,
               s.tile_start, s.tile_list, pitch, s.status, cov, depth, normal, state);
  } else {
    cudaMemsetAsync(grad, 0, sizeof(float) * 4 * (size_t)g.n_atoms, st);
    launch_pdl(ctas == 3 ? k_soft_bwd<3> : k_soft_bwd<2>, grid, kSoftNT, 0, st, g, s.recs, s.rec_of, s.entries, s.cap_entries, s.tile_count,
               s.tile_start, s.tile_list, pitch, s.status, g_cov, g_depth, g_normal, state, grad);
  }
  if (evs && evs->ev && evs->n > 5) cudaEventRecord(evs->ev[5], st);
  if (evs && evs->ev && evs->n > 6) cudaEventRecord(evs->ev[6], st);
  if (evs && evs->ev && evs->n > 7) cudaEventRecord(evs->ev[7], st);
  return cudaGetLastError();
}

}  // namespace vtx
