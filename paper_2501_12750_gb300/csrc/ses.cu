// ses.cu -- solvent excluded surface (SES) on a grid, extracted by marching
// cubes (Methods, "Cartoon and SES representations": a discrete approach in
// the manner of Lindow et al., surface by Lorensen-Cline marching cubes).
//
//   1. SAS interior: a grid point X = o + h (i, j, k) is inside when some atom
//      has ((X-c)_x^2 + (X-c)_y^2) + (X-c)_z^2 < (r + p)^2, evaluated in FP64
//      with every operation explicitly rounded (no contraction), so the
//      decision is a pure function of the inputs.  One warp per atom, one
//      lane per grid row of the atom's box; the interior is one bit per point.
//   2. Squared distance (grid units) to the nearest point outside the SAS
//      interior, exact inside a (2K+1)^3 window (K = ceil(p/h) + 1) and
//      K^2 + 1 beyond, integers only.  Marching cubes only ever needs values
//      <= K^2.  Windows of K <= 6 (p/h <= 5): 32 points at a time, as bit
//      sets of the points within each possible distance; larger windows: three
//      separable min-plus passes (x, y, z).
//   3. SES interior: edt2 >= 1 and edt2 h^2 >= p^2 (FP64; an integer threshold
//      here, as the product is monotone in edt2).  Marching cubes in two passes:
//      each CTA classifies a run of cells (one case byte per cell) and counts
//      their triangles, one CTA scans the counts, then each CTA writes its
//      cells' triangles in cell order, so the output order is deterministic.  The per-case
//      loops come from a table built once on the host: faces with four
//      crossings cut their inside corners apart, segments are directed by the
//      face's outward normal so loops turn counter-clockwise about the
//      outward (inside to outside) normal, and loops longer than three edges
//      become a star of triangles around their mean vertex.
#include <cmath>
#include <mutex>
#include <utility>

#include "vtx_internal.h"

namespace vtx {

constexpr int kSesThreads = 256;
constexpr int kSesCellsPerThread = 4;
constexpr int kSesCellsPerBlock = kSesThreads * kSesCellsPerThread;
constexpr uint16_t kSesInf = 0xffffu;

// Per case: number of loops, their lengths, and their edges back to back.
struct SesCase {
  unsigned char n_loops;
  unsigned char n_tris;
  unsigned char len[4];
  unsigned char edge[12];
};
__constant__ SesCase c_ses_case[256];

// Corners (x, y, z offsets) and edges (corner pairs) of a cell.
__constant__ int c_corner[8][3] = {{0, 0, 0}, {1, 0, 0}, {1, 1, 0}, {0, 1, 0}, {0, 0, 1}, {1, 0, 1}, {1, 1, 1}, {0, 1, 1}};
__constant__ int c_edge[12][2] = {{0, 1}, {1, 2}, {2, 3}, {3, 0}, {4, 5}, {5, 6},
                                  {6, 7}, {7, 4}, {0, 4}, {1, 5}, {2, 6}, {3, 7}};

// ------------------------------------------------------------ case table --

namespace {

const int kCorner[8][3] = {{0, 0, 0}, {1, 0, 0}, {1, 1, 0}, {0, 1, 0}, {0, 0, 1}, {1, 0, 1}, {1, 1, 1}, {0, 1, 1}};
const int kEdge[12][2] = {{0, 1}, {1, 2}, {2, 3}, {3, 0}, {4, 5}, {5, 6}, {6, 7}, {7, 4}, {0, 4}, {1, 5}, {2, 6}, {3, 7}};
// Faces: corner cycle and outward normal.
const int kFace[6][4] = {{0, 3, 2, 1}, {4, 5, 6, 7}, {0, 1, 5, 4}, {2, 3, 7, 6}, {0, 4, 7, 3}, {1, 2, 6, 5}};
const int kFaceN[6][3] = {{0, 0, -1}, {0, 0, 1}, {0, -1, 0}, {0, 1, 0}, {-1, 0, 0}, {1, 0, 0}};

int edge_between(int a, int b) {
  for (int e = 0; e < 12; ++e)
    if ((kEdge[e][0] == a && kEdge[e][1] == b) || (kEdge[e][1] == a && kEdge[e][0] == b)) return e;
  return -1;
}

// Twice the midpoint of edge e (integral).
void mid2(int e, long m[3]) {
  for (int k = 0; k < 3; ++k) m[k] = kCorner[kEdge[e][0]][k] + kCorner[kEdge[e][1]][k];
}

// Link crossing edges ea and eb on face f, the segment cutting off the inside
// corners cut[0..nc): direction d = m x n, m from the cut corners' mean to
// the segment's midpoint (all scaled to integers).
void link(int f, int ea, int eb, const int *cut, int nc, int next[12]) {
  long pa[3], pb[3], m[3];
  mid2(ea, pa);
  mid2(eb, pb);
  for (int k = 0; k < 3; ++k) {
    long c = 0;
    for (int q = 0; q < nc; ++q) c += 2 * kCorner[cut[q]][k];
    m[k] = (pa[k] + pb[k]) * nc - 2 * c;
  }
  const int *n = kFaceN[f];
  const long d[3] = {m[1] * n[2] - m[2] * n[1], m[2] * n[0] - m[0] * n[2], m[0] * n[1] - m[1] * n[0]};
  const long along = (pb[0] - pa[0]) * d[0] + (pb[1] - pa[1]) * d[1] + (pb[2] - pa[2]) * d[2];
  if (along > 0)
    next[ea] = eb;
  else
    next[eb] = ea;
}

SesCase build_case(int cs) {
  SesCase out{};
  if (cs == 0 || cs == 255) return out;
  int next[12];
  for (int e = 0; e < 12; ++e) next[e] = -1;
  for (int f = 0; f < 6; ++f) {
    const int *q = kFace[f];
    int crossing[4], n_cross = 0, in_c[4], n_in = 0;
    for (int s = 0; s < 4; ++s) {
      const bool a_in = (cs >> q[s]) & 1, b_in = (cs >> q[(s + 1) % 4]) & 1;
      if (a_in != b_in) crossing[n_cross++] = edge_between(q[s], q[(s + 1) % 4]);
      if (a_in) in_c[n_in++] = q[s];
    }
    if (n_cross == 2) {
      link(f, crossing[0], crossing[1], in_c, n_in, next);
    } else if (n_cross == 4) {
      for (int s = 0; s < 4; ++s)
        if ((cs >> q[s]) & 1) {
          const int c = q[s];
          link(f, edge_between(q[(s + 3) % 4], c), edge_between(c, q[(s + 1) % 4]), &c, 1, next);
        }
    }
  }
  bool seen[12] = {};
  int at = 0;
  for (int s = 0; s < 12; ++s) {
    if (next[s] < 0 || seen[s]) continue;
    int L = 0;
    for (int e = s; !seen[e]; e = next[e]) {
      seen[e] = true;
      out.edge[at + L++] = (unsigned char)e;
    }
    out.len[out.n_loops++] = (unsigned char)L;
    out.n_tris += (unsigned char)(L == 3 ? 1 : L);
    at += L;
  }
  return out;
}

std::once_flag g_table_once[64];
bool g_table_ok[64];

}  // namespace

// Upload the case table to this device's constant memory (once per device).
static bool ses_table_ready(int device) {
  if (device < 0 || device >= 64) return false;
  std::call_once(g_table_once[device], [device] {
    SesCase t[256];
    for (int cs = 0; cs < 256; ++cs) t[cs] = build_case(cs);
    g_table_ok[device] = cudaMemcpyToSymbol(c_ses_case, t, sizeof(t)) == cudaSuccess;
  });
  return g_table_ok[device];
}

// --------------------------------------------------------------- kernels --

struct SesGrid {
  float ox, oy, oz, h, p;
  int nx, ny, nz;
  int wx;        // 32-bit words per row of the interior bits: ceil(nx / 32)
  int K;
  int t_in;      // smallest edt2 with edt2 * h^2 >= p^2 in FP64 (the SES test, monotone in edt2)
  float xmax;    // largest |coordinate| of any grid point (bounds the FP32 rounding of the SAS filter)
};

__device__ __forceinline__ double grid_coord(float o, float h, long long i) {
  return __dadd_rn((double)o, __dmul_rn((double)h, (double)i));
}

__device__ __forceinline__ bool sas_exact(const SesGrid &G, long long i, double dy2, double dz2, double cx, double R2) {
  const double dx = __dsub_rn(grid_coord(G.ox, G.h, i), cx);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), dy2), dz2) < R2;
}

// SAS interior, one bit per grid point (bit i & 31 of word i >> 5 of a row; wx words a row): one warp per atom
// (`parts` warps when there are few atoms), lanes over the (j, k) rows of its box.  A row meets the sphere in a
// chord: with t = R^2 - dy^2 - dz^2 in FP32 and M the bound on the FP32 error of d^2 (coordinates, differences
// and squares, all at most a few ulps of numbers <= xmax + R + 2h, and of R^2 itself), every point with
// |dx| <= sqrt(t - M) is inside and none with |dx| > sqrt(t + M) is; the index bounds of both are widened by the
// rounding of the index itself.  The points between the two (a few in a thousand rows have one) are decided by
// the exact FP64 test, so every decision equals the FP64 one.  The chord's bits are set with one atomic a word.
//
// Bound by the row loop's issue and its atomics, not by memory: the bits of 3.4e7 points are 4.6 MB and stay in
// L2.  1e5 atoms at 0.5 A (3.4e7 points): 179 us; 1302 us with a byte per point, each point classified on its own.
__global__ __launch_bounds__(256) void k_ses_sas(SesGrid G, const float4 *__restrict__ X, long long n, int parts,
                                                 uint32_t *__restrict__ bits) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long item = warp; item < n * parts; item += n_warps) {
    const float4 c = X[item / parts];
    // FP32 throughout except on the rare points the filter cannot decide (the
    // FP64 pipes are a small fraction of the FP32 ones on this part)
    const float Rf = c.w + G.p, R2f = Rf * Rf;
    const float span = G.xmax + Rf + 2.0f * G.h;
    const float delta = 4e-7f * span;                      // |FP32 difference - exact| per axis
    const float ext = fabsf(Rf) + 2.0f * G.h;
    const float M = 8.0f * ext * delta + 4.0f * delta * delta + 1e-6f * ext * ext + 1e-6f;
    // candidate index ranges, two points wider than the sphere's extent on each side
    const float inv_h = 1.0f / G.h;
    const float cf[3] = {c.x, c.y, c.z};
    const float of[3] = {G.ox, G.oy, G.oz};
    const int nn[3] = {G.nx, G.ny, G.nz};
    int lo[3], hi[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      // clamped as floats first, so that the conversions cannot overflow
      const float top = (float)nn[d];
      lo[d] = max((int)fminf(fmaxf(floorf((cf[d] - Rf - of[d]) * inv_h) - 2.0f, 0.0f), top), 0);
      hi[d] = min((int)fminf(fmaxf(ceilf((cf[d] + Rf - of[d]) * inv_h) + 2.0f, -1.0f), top), nn[d] - 1);
    }
    if (lo[0] > hi[0] || lo[1] > hi[1] || lo[2] > hi[2]) continue;
    // rounding of a chord end's grid index: FP32 sums and products of numbers <= |c| + |o| + R
    const float eps = 1e-5f + 2e-6f * (fabsf(c.x) + fabsf(G.ox) + fabsf(Rf)) * inv_h;
    // row r of the box is (lo[1] + r % ny_box, lo[2] + r / ny_box); this lane takes every (32 parts)-th
    const unsigned ny_box = (unsigned)(hi[1] - lo[1] + 1), step = 32u * (unsigned)parts;
    const unsigned r0 = 32u * (unsigned)(item % parts) + (unsigned)lane;
    const int step_j = (int)(step % ny_box), step_k = (int)(step / ny_box);
    int j = lo[1] + (int)(r0 % ny_box), k = lo[2] + (int)(r0 / ny_box);
    for (; k <= hi[2]; k += step_k) {
      const float dyf = __fsub_rn(__fmaf_rn(G.h, (float)j, G.oy), c.y);
      const float dzf = __fsub_rn(__fmaf_rn(G.h, (float)k, G.oz), c.z);
      const float yz = __fmaf_rn(dyf, dyf, __fmul_rn(dzf, dzf));
      const float t = R2f - yz;
      if (!(t < -M)) {  // else the whole row is outside
        const float w_out = sqrtf(fmaxf(t + M, 0.0f)) * 1.000001f + 2.0f * delta;
        const float w_in = t > M ? sqrt_approx(t - M) * 0.999999f - 2.0f * delta : -1.0f;
        const float top = (float)(hi[0] + 1);
        const int i0 = max((int)fminf(fmaxf(ceilf((c.x - w_out - G.ox) * inv_h - eps), 0.0f), top), lo[0]);
        const int i1 = min((int)fminf(fmaxf(floorf((c.x + w_out - G.ox) * inv_h + eps), -1.0f), top), hi[0]);
        int a = i1 + 1, b = i1;  // the certain points [a, b] (none yet)
        if (w_in >= 0.0f) {
          const int ca = (int)fminf(fmaxf(ceilf((c.x - w_in - G.ox) * inv_h + eps), 0.0f), top);
          const int cb = (int)fminf(fmaxf(floorf((c.x + w_in - G.ox) * inv_h - eps), -1.0f), top);
          if (max(ca, i0) <= min(cb, i1)) {
            a = max(ca, i0);
            b = min(cb, i1);
          }
        }
        uint32_t *row = bits + ((size_t)k * (size_t)G.ny + (size_t)j) * (size_t)G.wx;
        if (a <= b) {
          const int wa = a >> 5, wb = b >> 5;
          for (int w = wa; w <= wb; ++w) {
            uint32_t m = 0xffffffffu;
            if (w == wa) m <<= a & 31;
            if (w == wb) m &= 0xffffffffu >> (31 - (b & 31));
            atomicOr(row + w, m);
          }
        }
        if (a > i0 || b < i1) {
          const double dy = __dsub_rn(grid_coord(G.oy, G.h, j), (double)c.y);
          const double dz = __dsub_rn(grid_coord(G.oz, G.h, k), (double)c.z);
          const double dy2 = __dmul_rn(dy, dy), dz2 = __dmul_rn(dz, dz);
          const double R = __dadd_rn((double)c.w, (double)G.p);
          const double R2 = __dmul_rn(R, R);
          for (int i = i0; i <= i1; ++i) {
            if (i == a) {  // past the certain points
              i = b;
              continue;
            }
            if (sas_exact(G, i, dy2, dz2, (double)c.x, R2)) atomicOr(row + (i >> 5), 1u << (i & 31));
          }
        }
      }
      j += step_j;
      if (j > hi[1]) {
        j -= (int)ny_box;
        ++k;
      }
    }
  }
}

// The interior as one byte per point (only when the caller asks for the plane).
__global__ __launch_bounds__(256) void k_ses_sas_bytes(SesGrid G, const uint32_t *__restrict__ bits, long long n_pts,
                                                       uint8_t *__restrict__ sas) {
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n_pts;
       q += (long long)gridDim.x * blockDim.x) {
    const long long row = q / G.nx, i = q - row * G.nx;
    sas[q] = (uint8_t)((bits[row * G.wx + (i >> 5)] >> (i & 31)) & 1u);
  }
}

// ------------------------------------------------- distances as bit sets --

// Largest window of the bit-set distance pass.
constexpr int kSesBitK = 6;

// The lattice offsets (dx >= 0, dy, dz) of squared length <= K^2 in ascending order of length ("steps"), and the
// distinct squared lengths ("levels": sums of three squares).  Offsets are those of the pass's shared-memory tile.
template <int K>
struct SesSteps {
  static constexpr int TY = 32, TZ = 8;                           // rows of a tile
  static constexpr int PY = TY + 2 * K, PZ = TZ + 2 * K, PL = PY * PZ;  // with their halo; one plane per dx
  static constexpr int max_steps = (K + 1) * (2 * K + 1) * (2 * K + 1);
  int n = 0, n_levels = 0;
  int off[max_steps] = {};
  int level[max_steps + 1] = {};   // level of each step
  int value[K * K + 2] = {};       // squared length of each level, then the sentinel K^2 + 1
  constexpr SesSteps() {
    for (int m = 0; m <= K * K; ++m) {
      bool any = false;
      for (int dx = 0; dx <= K; ++dx)
        for (int dz = -K; dz <= K; ++dz)
          for (int dy = -K; dy <= K; ++dy)
            if (dx * dx + dy * dy + dz * dz == m) {
              off[n] = dx * PL + dz * PY + dy;
              level[n++] = n_levels;
              any = true;
            }
      if (any) value[n_levels++] = m;
    }
    level[n] = n_levels;
    value[n_levels] = K * K + 1;
  }
};
template <int K>
constexpr SesSteps<K> kSesSteps{};

template <int K>
struct SesLevelState {
  uint32_t acc = 0u, prev = 0u;  // points within the levels so far; within the levels before the current one
  uint32_t plane[6] = {};        // binary digits of each point's level
};

template <int K, int I>
__device__ __forceinline__ void ses_step(const uint32_t *e, SesLevelState<K> &s) {
  constexpr int off = kSesSteps<K>.off[I], lv = kSesSteps<K>.level[I];
  constexpr bool last = kSesSteps<K>.level[I + 1] != lv;
  s.acc |= e[off];
  if constexpr (last) {
    const uint32_t newly = s.acc & ~s.prev;
    if constexpr ((lv & 1) != 0) s.plane[0] |= newly;
    if constexpr ((lv & 2) != 0) s.plane[1] |= newly;
    if constexpr ((lv & 4) != 0) s.plane[2] |= newly;
    if constexpr ((lv & 8) != 0) s.plane[3] |= newly;
    if constexpr ((lv & 16) != 0) s.plane[4] |= newly;
    if constexpr ((lv & 32) != 0) s.plane[5] |= newly;
    s.prev = s.acc;
  }
}

template <int K, int... I>
__device__ __forceinline__ void ses_steps(const uint32_t *e, SesLevelState<K> &s, std::integer_sequence<int, I...>) {
  (ses_step<K, I>(e, s), ...);
}

// s_val[level] = its squared length (the last one: the sentinel).
template <int K, int I>
__device__ __forceinline__ void ses_value(uint16_t *s_val) {
  constexpr int v = kSesSteps<K>.value[I];
  if (threadIdx.x == I) s_val[I] = (uint16_t)v;
}
template <int K, int... I>
__device__ __forceinline__ void ses_values(uint16_t *s_val, std::integer_sequence<int, I...>) {
  (ses_value<K, I>(s_val), ...);
}

// Windowed squared distance for windows K <= 6, 32 points at a time.  A CTA takes one word of 32 x 8 rows (y, z).
// E_d, d = 0..K, is the set of points with a point outside the SAS interior exactly d along x; the points within
// squared distance m are the union of E_dx over the rows (dy, dz) with dx^2 + dy^2 + dz^2 <= m, so going through
// the lattice offsets by length, one shared-memory read and one OR give 32 points' worth of each.  A point's
// level (the ordinal of its distance) is kept as binary digit planes and spread to one 16-bit value per point at
// the end.  Points beyond the grid are not outside points.
//
// Bound by shared-memory reads and issue (K = 4: 153 reads a word).  3.4e7 points at K = 4: 60 us; the three
// separable passes over 16-bit planes (one point per thread) take 105 + 2 x 172 us.  K <= 6 because the offsets
// grow with K^3 (519 at K = 6) and every one is an unrolled instruction.
template <int K>
__global__ __launch_bounds__(256) void k_ses_levels(SesGrid G, const uint32_t *__restrict__ bits,
                                                    uint16_t *__restrict__ edt2) {
  using S = SesSteps<K>;
  constexpr int n_levels = kSesSteps<K>.n_levels;
  __shared__ uint32_t s_e[(K + 1) * S::PL];
  __shared__ uint16_t s_val[64];
  const int lane = threadIdx.x & 31, zw = threadIdx.x >> 5;
  const unsigned ty = (unsigned)(G.ny + S::TY - 1) / S::TY;
  const unsigned b = blockIdx.x;
  const int w = (int)(b % (unsigned)G.wx);
  const unsigned q = b / (unsigned)G.wx;
  const long long y0 = (long long)(q % ty) * S::TY, z0 = (long long)(q / ty) * S::TZ;
  const int tail = G.nx - 32 * (G.wx - 1);  // points of a row's last word
  const uint32_t last_mask = 0xffffffffu >> (32 - tail);
  ses_values<K>(s_val, std::make_integer_sequence<int, n_levels + 1>{});
  for (int r = threadIdx.x; r < S::PL; r += 256) {
    const int yy = r % S::PY, zz = r / S::PY;
    const long long y = y0 + yy - K, z = z0 + zz - K;
    uint32_t zp = 0u, zc = 0u, zn = 0u;  // points outside the interior: the words before, at and after w
    if (y >= 0 && y < G.ny && z >= 0 && z < G.nz) {
      const uint32_t *p = bits + (z * G.ny + y) * G.wx + w;
      zc = ~p[0] & (w == G.wx - 1 ? last_mask : 0xffffffffu);
      if (w > 0) zp = ~p[-1];
      if (w + 1 < G.wx) zn = ~p[1] & (w + 1 == G.wx - 1 ? last_mask : 0xffffffffu);
    }
    s_e[r] = zc;
#pragma unroll
    for (int d = 1; d <= K; ++d) s_e[d * S::PL + r] = __funnelshift_r(zc, zn, d) | __funnelshift_l(zp, zc, d);
  }
  __syncthreads();
  SesLevelState<K> st;
  ses_steps<K>(s_e + (zw + K) * S::PY + lane + K, st, std::make_integer_sequence<int, kSesSteps<K>.n>{});
  const uint32_t rest = ~st.acc;  // farther than K: the last level
#pragma unroll
  for (int p = 0; p < 6; ++p)
    if ((n_levels >> p) & 1) st.plane[p] |= rest;
  // spread: row r of the warp's 32 (y0 + r), one point per lane
  constexpr int planes = n_levels < 2 ? 1 : n_levels < 4 ? 2 : n_levels < 8 ? 3 : n_levels < 16 ? 4 : n_levels < 32 ? 5 : 6;
  const long long z = z0 + zw, x = 32LL * w + lane;
  if (z >= G.nz) return;  // uniform in the warp; no barrier follows
  const int rows = (int)min((long long)S::TY, G.ny - y0);
  uint16_t *dst = edt2 + (z * G.ny + y0) * G.nx + x;
  for (int r = 0; r < rows; ++r, dst += G.nx) {
    unsigned lv = 0u;
#pragma unroll
    for (int p = 0; p < planes; ++p) lv |= ((__shfl_sync(0xffffffffu, st.plane[p], r) >> lane) & 1u) << p;
    if (x < G.nx) *dst = s_val[lv];
  }
}

// --------------------------------------------- distances in three passes --

// Pass x: distance^2 along x to the nearest point outside the SAS interior, within K.
__global__ __launch_bounds__(256) void k_ses_edt_x(SesGrid G, const uint32_t *__restrict__ bits,
                                                   uint16_t *__restrict__ g1, long long n_pts) {
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n_pts;
       q += (long long)gridDim.x * blockDim.x) {
    const long long r = q / G.nx;
    const int i = (int)(q - r * G.nx);
    const uint32_t *row = bits + r * G.wx;
    auto out = [&](int at) { return ((row[at >> 5] >> (at & 31)) & 1u) == 0u; };
    uint16_t best = kSesInf;
    if (out(i)) {
      best = 0;
    } else {
      for (int d = 1; d <= G.K; ++d) {
        const bool l = i - d >= 0 && out(i - d), rt = i + d < G.nx && out(i + d);
        if (l || rt) {
          best = (uint16_t)(d * d);
          break;
        }
      }
    }
    g1[q] = best;
  }
}

// Passes y and z: min over |d| <= K of d^2 + src[q + d * stride] (kSesInf = none).
// The last pass maps values above K^2 to the sentinel K^2 + 1.
__global__ __launch_bounds__(256) void k_ses_edt_yz(SesGrid G, const uint16_t *__restrict__ src,
                                                    uint16_t *__restrict__ dst, long long n_pts, long long stride,
                                                    long long extent, int last) {
  const int K2 = G.K * G.K;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n_pts;
       q += (long long)gridDim.x * blockDim.x) {
    const long long c = (q / stride) % extent;
    int best = src[q] == kSesInf ? 0x7fffffff : (int)src[q];
    for (int d = 1; d <= G.K; ++d) {
      const int dd = d * d;
      if (dd >= best) break;
      if (c - d >= 0) {
        const uint16_t v = src[q - d * stride];
        if (v != kSesInf && dd + (int)v < best) best = dd + (int)v;
      }
      if (c + d < extent) {
        const uint16_t v = src[q + d * stride];
        if (v != kSesInf && dd + (int)v < best) best = dd + (int)v;
      }
    }
    if (last)
      dst[q] = (uint16_t)(best > K2 ? K2 + 1 : best);
    else
      dst[q] = (uint16_t)(best > 0xfffe ? kSesInf : best);
  }
}



__device__ __forceinline__ int cell_case(const SesGrid &G, const uint16_t *__restrict__ edt, long long i, long long j,
                                         long long k) {
  int cs = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const long long q = ((k + c_corner[c][2]) * G.ny + (j + c_corner[c][1])) * (long long)G.nx + (i + c_corner[c][0]);
    if ((int)edt[q] >= G.t_in) cs |= 1 << c;
  }
  return cs;
}

// Triangles of the cells [c0, c0 + kSesCellsPerThread) of a thread; their cases
// are stored (one byte per cell) for the emit pass.
__device__ __forceinline__ int thread_cells_count(const SesGrid &G, const uint16_t *__restrict__ edt, long long c0,
                                                  long long n_cells, uint8_t *__restrict__ cases) {
  int n = 0;
  const long long cx = G.nx - 1, cy = G.ny - 1;
  for (int u = 0; u < kSesCellsPerThread; ++u) {
    const long long c = c0 + u;
    if (c >= n_cells) break;
    const long long i = c % cx, j = (c / cx) % cy, k = c / (cx * cy);
    const int cs = cell_case(G, edt, i, j, k);
    cases[c] = (uint8_t)cs;
    n += c_ses_case[cs].n_tris;
  }
  return n;
}

__device__ __forceinline__ unsigned block_exclusive_sum(unsigned v, unsigned *total) {
  __shared__ unsigned s_warp[kSesThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[w] = x;
  __syncthreads();
  if (w == 0) {
    unsigned s = lane < kSesThreads / 32 ? s_warp[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < kSesThreads / 32) s_warp[lane] = s;
  }
  __syncthreads();
  const unsigned before = (w > 0 ? s_warp[w - 1] : 0u) + x - v;
  if (total) *total = s_warp[kSesThreads / 32 - 1];
  __syncthreads();
  return before;
}

__global__ __launch_bounds__(kSesThreads) void k_ses_count(SesGrid G, const uint16_t *__restrict__ edt,
                                                           long long n_cells, uint8_t *__restrict__ cases,
                                                           unsigned *__restrict__ block_tris) {
  const long long c0 = (long long)blockIdx.x * kSesCellsPerBlock + (long long)threadIdx.x * kSesCellsPerThread;
  unsigned total;
  block_exclusive_sum((unsigned)thread_cells_count(G, edt, c0, n_cells, cases), &total);
  if (threadIdx.x == 0) block_tris[blockIdx.x] = total;
}

// Exclusive scan of the per-block counts in one CTA (64-bit totals).
__global__ __launch_bounds__(kSesThreads) void k_ses_scan(const unsigned *__restrict__ block_tris, long long n_blocks,
                                                          unsigned long long *__restrict__ block_base,
                                                          unsigned long long *__restrict__ total) {
  __shared__ unsigned long long s_carry;
  if (threadIdx.x == 0) s_carry = 0ull;
  __syncthreads();
  for (long long b0 = 0; b0 < n_blocks; b0 += kSesThreads) {
    const long long b = b0 + threadIdx.x;
    const unsigned v = b < n_blocks ? block_tris[b] : 0u;
    unsigned tot;
    const unsigned ex = block_exclusive_sum(v, &tot);
    if (b < n_blocks) block_base[b] = s_carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) s_carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = s_carry;
}

__device__ __forceinline__ void store_tri(float *__restrict__ tris, long long *__restrict__ labels,
                                          unsigned long long t, unsigned long long max_tris, const float3 &a,
                                          const float3 &b, const float3 &c, long long la, long long lb, long long lc) {
  if (t >= max_tris) return;
  float *o = tris + t * 9;
  o[0] = a.x, o[1] = a.y, o[2] = a.z;
  o[3] = b.x, o[4] = b.y, o[5] = b.z;
  o[6] = c.x, o[7] = c.y, o[8] = c.z;
  if (labels) {
    labels[t * 3] = la;
    labels[t * 3 + 1] = lb;
    labels[t * 3 + 2] = lc;
  }
}

// Vertex on edge e of cell (i, j, k): X_a + t (X_b - X_a), t = f_a / (f_a - f_b) clamped.
__device__ __forceinline__ float3 edge_vertex(const SesGrid &G, const uint16_t *__restrict__ edt, long long i,
                                              long long j, long long k, int e) {
  const int a = c_edge[e][0], b = c_edge[e][1];
  const long long ai = i + c_corner[a][0], aj = j + c_corner[a][1], ak = k + c_corner[a][2];
  const long long bi = i + c_corner[b][0], bj = j + c_corner[b][1], bk = k + c_corner[b][2];
  const float fa = sqrtf((float)edt[(ak * G.ny + aj) * (long long)G.nx + ai]) * G.h - G.p;
  const float fb = sqrtf((float)edt[(bk * G.ny + bj) * (long long)G.nx + bi]) * G.h - G.p;
  float s = fa == fb ? 0.5f : fa / (fa - fb);
  s = fminf(fmaxf(s, 0.0f), 1.0f);
  const float3 A = make_float3(G.ox + G.h * (float)ai, G.oy + G.h * (float)aj, G.oz + G.h * (float)ak);
  const float3 B = make_float3(G.ox + G.h * (float)bi, G.oy + G.h * (float)bj, G.oz + G.h * (float)bk);
  return make_float3(A.x + s * (B.x - A.x), A.y + s * (B.y - A.y), A.z + s * (B.z - A.z));
}

// One thread per output triangle of the CTA's run of cells: the cells'
// triangle offsets are scanned into shared memory, each thread finds its cell
// by binary search, its loop and fan position from the case table, and writes
// its triangle next to its neighbours' (coalesced).
__global__ __launch_bounds__(kSesThreads) void k_ses_emit(SesGrid G, const uint16_t *__restrict__ edt,
                                                          const uint8_t *__restrict__ cases, long long n_cells,
                                                          const unsigned long long *__restrict__ block_base,
                                                          float *__restrict__ tris, long long *__restrict__ labels,
                                                          unsigned long long max_tris) {
  __shared__ unsigned s_off[kSesCellsPerBlock + 1];
  __shared__ unsigned char s_case[kSesCellsPerBlock];
  const long long cb = (long long)blockIdx.x * kSesCellsPerBlock;
  unsigned n4[kSesCellsPerThread];
  unsigned mine = 0;
  for (int u = 0; u < kSesCellsPerThread; ++u) {
    const int lc = threadIdx.x * kSesCellsPerThread + u;
    const unsigned char cs = cb + lc < n_cells ? cases[cb + lc] : 0;
    s_case[lc] = cs;
    n4[u] = c_ses_case[cs].n_tris;
    mine += n4[u];
  }
  unsigned total;
  unsigned run = block_exclusive_sum(mine, &total);
  for (int u = 0; u < kSesCellsPerThread; ++u) {
    s_off[threadIdx.x * kSesCellsPerThread + u] = run;
    run += n4[u];
  }
  if (threadIdx.x == 0) s_off[kSesCellsPerBlock] = total;
  __syncthreads();
  const unsigned long long base_t = block_base[blockIdx.x];
  const long long cx = G.nx - 1, cy = G.ny - 1;
  for (unsigned q = threadIdx.x; q < total; q += kSesThreads) {
    int lo = 0, hi = kSesCellsPerBlock - 1;  // last cell with s_off <= q
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_off[mid] <= q) lo = mid; else hi = mid - 1;
    }
    const long long c = cb + lo;
    const SesCase &tc = c_ses_case[s_case[lo]];
    unsigned r = q - s_off[lo];
    int at = 0, l = 0;
    while (l < tc.n_loops) {
      const unsigned nt = tc.len[l] == 3 ? 1u : tc.len[l];
      if (r < nt) break;
      r -= nt;
      at += tc.len[l];
      ++l;
    }
    const long long i = c % cx, j = (c / cx) % cy, k = c / (cx * cy);
    const long long base = c * 16;
    const int L = tc.len[l];
    if (L == 3) {
      const int e0 = tc.edge[at], e1 = tc.edge[at + 1], e2 = tc.edge[at + 2];
      store_tri(tris, labels, base_t + q, max_tris, edge_vertex(G, edt, i, j, k, e0), edge_vertex(G, edt, i, j, k, e1),
                edge_vertex(G, edt, i, j, k, e2), base + e0, base + e1, base + e2);
    } else {
      float3 M = make_float3(0.0f, 0.0f, 0.0f);
      for (int v = 0; v < L; ++v) {
        const float3 p = edge_vertex(G, edt, i, j, k, tc.edge[at + v]);
        M.x += p.x;
        M.y += p.y;
        M.z += p.z;
      }
      const float inv = 1.0f / (float)L;
      M = make_float3(M.x * inv, M.y * inv, M.z * inv);
      const int q0 = (int)r, q1 = q0 + 1 == L ? 0 : q0 + 1;
      const int ea = tc.edge[at + q0], eb = tc.edge[at + q1];
      store_tri(tris, labels, base_t + q, max_tris, M, edge_vertex(G, edt, i, j, k, ea),
                edge_vertex(G, edt, i, j, k, eb), base + 12 + l, base + ea, base + eb);
    }
  }
}

// Bounding box of the SAS spheres: min and max of c -/+ (r + p), as float bits of
// non-negative-shifted values would be awkward, so each CTA reduces and writes one
// partial; the host finishes the (small) reduction.
__global__ __launch_bounds__(256) void k_ses_bbox(const float4 *__restrict__ X, long long n, float p,
                                                  float *__restrict__ partial) {
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < n; a += (long long)gridDim.x * blockDim.x) {
    const float4 c = X[a];
    const float R = c.w + p;
    lo[0] = fminf(lo[0], c.x - R), hi[0] = fmaxf(hi[0], c.x + R);
    lo[1] = fminf(lo[1], c.y - R), hi[1] = fmaxf(hi[1], c.y + R);
    lo[2] = fminf(lo[2], c.z - R), hi[2] = fmaxf(hi[2], c.z + R);
  }
  __shared__ float s[6][8];
  for (int d = 0; d < 3; ++d) {
    for (int o = 16; o > 0; o >>= 1) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
    }
  }
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0)
    for (int d = 0; d < 3; ++d) {
      s[d][w] = lo[d];
      s[3 + d][w] = hi[d];
    }
  __syncthreads();
  if (threadIdx.x < 6) {
    float v = s[threadIdx.x][0];
    for (int q = 1; q < 8; ++q) v = threadIdx.x < 3 ? fminf(v, s[threadIdx.x][q]) : fmaxf(v, s[threadIdx.x][q]);
    partial[blockIdx.x * 6 + threadIdx.x] = v;
  }
}

// ------------------------------------------------------------- launchers --

int ses_window(float probe, float h) { return (int)std::ceil((double)probe / (double)h) + 1; }

bool ses_three_pass(float probe, float h) { return ses_window(probe, h) > kSesBitK; }

long long ses_words(const int32_t dims[3]) { return ((long long)dims[0] + 31) / 32 * dims[1] * dims[2]; }

template <int K>
static void launch_levels(const SesGrid &G, const SesLaunch &L, cudaStream_t st) {
  using S = SesSteps<K>;
  const long long tiles = (long long)G.wx * (((long long)G.ny + S::TY - 1) / S::TY) * (((long long)G.nz + S::TZ - 1) / S::TZ);
  k_ses_levels<K><<<(unsigned)tiles, 256, 0, st>>>(G, L.bits, L.edt2);
}

cudaError_t run_ses_bbox(const float4 *X, long long n, float probe, float *partial, int n_blocks, cudaStream_t st) {
  k_ses_bbox<<<n_blocks, 256, 0, st>>>(X, n, probe, partial);
  return cudaGetLastError();
}

cudaError_t run_ses_grid(const SesLaunch &L, cudaStream_t st) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (!ses_table_ready(dev)) return cudaErrorInvalidValue;
  SesGrid G{L.origin[0], L.origin[1], L.origin[2], L.h, L.probe, L.dims[0], L.dims[1], L.dims[2],
            (int)(((long long)L.dims[0] + 31) / 32), ses_window(L.probe, L.h), 1, 0.0f};
  {
    // SES interior <=> edt2 >= 1 (inside the SAS) and edt2 * h^2 >= p^2 in FP64: the product is monotone in
    // edt2, so the test is edt2 >= t_in for the smallest such integer
    const double hh = (double)L.h * (double)L.h, pp = (double)L.probe * (double)L.probe;
    long long t = (long long)std::floor(pp / hh);
    while (t > 0 && (double)(t - 1) * hh >= pp) --t;
    while ((double)t * hh < pp) ++t;
    G.t_in = (int)(t < 1 ? 1 : t);
    double xm = 0.0;
    for (int d = 0; d < 3; ++d) {
      const double a0 = std::fabs((double)L.origin[d]);
      const double a1 = std::fabs((double)L.origin[d] + (double)L.h * (double)(L.dims[d] - 1));
      xm = std::fmax(xm, std::fmax(a0, a1));
    }
    G.xmax = (float)(xm * 1.001 + 1.0);
  }
  const long long n_pts = (long long)G.nx * G.ny * G.nz;
  const int sms = sm_count();
  cudaError_t e = cudaMemsetAsync(L.bits, 0, 4 * (size_t)ses_words(L.dims), st);
  if (e != cudaSuccess) return e;
  if (L.n_atoms > 0) {
    // one warp per atom, or up to 8 when the atoms alone would not fill the GPU (8 CTAs of 8 warps per SM)
    const long long fill = 64LL * sms;
    const long long share = fill / L.n_atoms;
    const int parts = (int)(share < 1 ? 1 : (share > 8 ? 8 : share));
    const long long warps = L.n_atoms * parts < 8 * fill ? L.n_atoms * parts : 8 * fill;
    k_ses_sas<<<(int)((warps * 32 + 255) / 256), 256, 0, st>>>(G, L.X, L.n_atoms, parts, L.bits);
  }
  const long long pb = (n_pts + 255) / 256;
  const int grid = (int)(pb < 16LL * sms ? pb : 16LL * sms);
  if (L.sas) k_ses_sas_bytes<<<grid, 256, 0, st>>>(G, L.bits, n_pts, L.sas);
  if (G.K <= kSesBitK) {
    switch (G.K) {
      case 1: launch_levels<1>(G, L, st); break;
      case 2: launch_levels<2>(G, L, st); break;
      case 3: launch_levels<3>(G, L, st); break;
      case 4: launch_levels<4>(G, L, st); break;
      case 5: launch_levels<5>(G, L, st); break;
      default: launch_levels<6>(G, L, st); break;
    }
  } else {
    k_ses_edt_x<<<grid, 256, 0, st>>>(G, L.bits, L.g_a, n_pts);
    k_ses_edt_yz<<<grid, 256, 0, st>>>(G, L.g_a, L.g_b, n_pts, (long long)G.nx, (long long)G.ny, 0);
    k_ses_edt_yz<<<grid, 256, 0, st>>>(G, L.g_b, L.edt2, n_pts, (long long)G.nx * G.ny, (long long)G.nz, 1);
  }
  const long long n_cells = (long long)(G.nx - 1) * (G.ny - 1) * (G.nz - 1);
  const long long n_blocks = (n_cells + kSesCellsPerBlock - 1) / kSesCellsPerBlock;
  if (n_blocks > 0) {
    k_ses_count<<<(unsigned)n_blocks, kSesThreads, 0, st>>>(G, L.edt2, n_cells, L.cases, L.block_tris);
    k_ses_scan<<<1, kSesThreads, 0, st>>>(L.block_tris, n_blocks, L.block_base, L.total);
    k_ses_emit<<<(unsigned)n_blocks, kSesThreads, 0, st>>>(G, L.edt2, L.cases, n_cells, L.block_base, L.tris,
                                                           L.labels, (unsigned long long)L.max_tris);
  } else {
    cudaMemsetAsync(L.total, 0, sizeof(unsigned long long), st);
  }
  return cudaGetLastError();
}

long long ses_blocks(const int32_t dims[3]) {
  const long long n_cells = (long long)(dims[0] - 1) * (dims[1] - 1) * (dims[2] - 1);
  return (n_cells + kSesCellsPerBlock - 1) / kSesCellsPerBlock;
}

}  // namespace vtx
