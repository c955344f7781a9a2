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
//      here, as the product is monotone in edt2), again one bit per point.
//      Marching cubes in two passes over "groups" of 32 cells of a row: one
//      counts the triangles of every CTA's groups (the last CTA scans the
//      counts), the other writes them in cell order, so the output order is
//      deterministic.  The per-case loops come from a table built once on the
//      host: faces with four crossings cut their inside corners apart, segments
//      are directed by the face's outward normal so loops turn
//      counter-clockwise about the outward (inside to outside) normal, and
//      loops longer than three edges become a star of triangles around their
//      mean vertex.
#include <cmath>
#include <mutex>
#include <utility>

#include "vtx_internal.h"

namespace vtx {

constexpr int kSesThreads = 256;
constexpr uint16_t kSesInf = 0xffffu;

// Per case: number of loops, their lengths, their edges back to back, and the triangles as three 4-bit vertex
// codes each (0..11: the vertex on that edge; 12 + l: the mean of loop l).
struct __align__(16) SesCase {
  unsigned char n_loops;
  unsigned char n_tris;
  unsigned char len[4];
  unsigned char edge[12];
  unsigned short tri[12];
};
__device__ SesCase g_ses_case[256];

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
    const unsigned char *e = out.edge + at;
    if (L == 3) {
      out.tri[out.n_tris++] = (unsigned short)(e[0] | e[1] << 4 | e[2] << 8);
    } else {
      for (int v = 0; v < L; ++v)
        out.tri[out.n_tris++] = (unsigned short)((12 + out.n_loops) | e[v] << 4 | e[v + 1 == L ? 0 : v + 1] << 8);
    }
    out.len[out.n_loops++] = (unsigned char)L;
    at += L;
  }
  return out;
}

std::once_flag g_table_once[64];
bool g_table_ok[64];

}  // namespace

// Upload the case table to this device's memory (once per device).
static bool ses_table_ready(int device) {
  if (device < 0 || device >= 64) return false;
  std::call_once(g_table_once[device], [device] {
    SesCase t[256];
    for (int cs = 0; cs < 256; ++cs) t[cs] = build_case(cs);
    g_table_ok[device] = cudaMemcpyToSymbol(g_ses_case, t, sizeof(t)) == cudaSuccess;
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

__device__ __forceinline__ bool sas_exact(float ox, float h, long long i, double dy2, double dz2, double cx, double R2) {
  const double dx = __dsub_rn(grid_coord(ox, h, i), cx);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), dy2), dz2) < R2;
}

// The points of one row that FP32 cannot decide, [i0, i1] but for the certain ones [a, b], by the exact FP64 test.
static __device__ __noinline__ void sas_row_exact(float ox, float oy, float oz, float h, float p, float4 c, int j, int k,
                                                  int i0, int i1, int a, int b, uint32_t *row) {
  const double dy = __dsub_rn(grid_coord(oy, h, j), (double)c.y);
  const double dz = __dsub_rn(grid_coord(oz, h, k), (double)c.z);
  const double dy2 = __dmul_rn(dy, dy), dz2 = __dmul_rn(dz, dz);
  const double R = __dadd_rn((double)c.w, (double)p);
  const double R2 = __dmul_rn(R, R);
  for (int i = i0; i <= i1; ++i) {
    if (i >= a && i <= b) {
      i = b;
      continue;
    }
    if (sas_exact(ox, h, i, dy2, dz2, (double)c.x, R2)) atomicOr(row + (i >> 5), 1u << (i & 31));
  }
}

// SAS interior, one bit per grid point (bit i & 31 of word i >> 5 of a row; wx words a row): one warp per atom
// (`parts` warps when there are few atoms), lanes over the (j, k) rows of its box.  A row meets the sphere in a
// chord: with t = R^2 - dy^2 - dz^2 in FP32 and M the bound on the FP32 error of t (below), every point with
// dx^2 <= t - M is inside and none with dx^2 > t + M is.  For t > 4 M both ends lie within M / sqrt(t) of sqrt(t).
// The ends are compared as grid indices, xc -/+ w with xc = (c.x - o.x) / h and w = sqrt(t) / h, so y and z enter
// through M alone.  In units of 2^-24 = 6e-8 xc carries 3 |xc| (difference, 1 / h, product), w carries 7 w (rsqrt 2
// ulps, the two products, 1 / h) and the sums xc -/+ w -/+ u 2 (|xc| + w + u); the ends are therefore known to within
//   u = 1.001 M / (h sqrt(t)) + eps + 1e-6 w,  eps = 1e-6 + 4e-7 (|xc| + R / h).
// The points within u of an end (a few in a thousand rows have one), and every point of a row with t <= 4 M, are
// decided by the exact FP64 test, so every decision equals the FP64 one.  The bounds are kept near the roundings they
// stand for: an exact test costs its warp some 300 cycles of the FP64 pipe (four times wider bounds took 262 us
// instead of 102).  The chord's bits are set with one atomic a word.
//
// Bound by issue (83 % of the slots; FP64 pipe 42 %).  1e5 atoms at 0.5 A (3.4e7 points): 105 us; 179 us with both ends
// of both bounds computed per row over a box two points wider on each side; 1302 us with a byte per point, each point
// classified on its own.
__global__ __launch_bounds__(256, 6) void k_ses_sas(SesGrid G, const float4 *__restrict__ X, long long n, int parts,
                                                    uint32_t *__restrict__ bits) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
  const float inv_h = 1.0f / G.h;
  const long long plane = (long long)G.ny * G.wx;
  for (long long item = warp; item < n * parts; item += n_warps) {
    const float4 c = X[item / parts];
    // FP32 throughout except on the rare points the filter cannot decide (the
    // FP64 pipes are a small fraction of the FP32 ones on this part)
    const float Rf = c.w + G.p, R2f = Rf * Rf;
    // error of an FP32 difference X - c along y or z: the roundings of the grid index and coordinate and of the
    // difference, at most three times 2^-24 of the largest number; M: of dy^2 + dz^2 (2 |d| delta an axis, with
    // |dy| + |dz| <= sqrt(2) ext) and the relative roundings of the squares, of R, R^2 and of t
    const float ext = fabsf(Rf) + 2.0f * G.h;
    const float delta = 2e-7f * (G.xmax + ext);
    float M = 2.9f * ext * delta + 4.0f * delta * delta + 6e-7f * ext * ext;
    // candidate index ranges, two points wider than the sphere's extent on each side
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
      if (d > 0) {
        // rows farther than sqrt(R^2 + M) from the centre are outside as a whole: the box without them
        const float w = sqrtf(R2f + M) * 1.000001f + 2.0f * delta;
        const float e = 1e-5f + 2e-6f * (fabsf(cf[d]) + fabsf(of[d]) + w) * inv_h;
        lo[d] = max(lo[d], (int)fminf(fmaxf(ceilf((cf[d] - w - of[d]) * inv_h - e), 0.0f), top));
        hi[d] = min(hi[d], (int)fminf(fmaxf(floorf((cf[d] + w - of[d]) * inv_h + e), -1.0f), top));
      }
    }
    if (lo[0] > hi[0] || lo[1] > hi[1] || lo[2] > hi[2]) continue;
    // the centre's grid index, and the rounding of a chord end's index: of the difference, of 1 / h and the product,
    // and of the end's sum, each 2^-24 of numbers <= (|c - o| + R) / h
    const float xc = (c.x - G.ox) * inv_h;
    const float eps = 1e-6f + 4e-7f * (fabsf(xc) + fabsf(Rf) * inv_h);
    // no usable index (1 / h overflows) or chord (R^2 does): the exact test decides every point
    if (!(fabsf(xc) < 1e30f && R2f < 1e30f)) M = INFINITY;
    const float Mh = M * inv_h * 1.001f;
    // row r of the box is (lo[1] + r % ny_box, lo[2] + r / ny_box); this lane takes every (32 parts)-th
    const unsigned ny_box = (unsigned)(hi[1] - lo[1] + 1), step = 32u * (unsigned)parts;
    const unsigned r0 = 32u * (unsigned)(item % parts) + (unsigned)lane;
    const int step_j = (int)(step % ny_box), step_k = (int)(step / ny_box);
    int j = lo[1] + (int)(r0 % ny_box), k = lo[2] + (int)(r0 / ny_box);
    uint32_t *row = bits + (long long)k * plane + (long long)j * G.wx;
    const long long step_row = (long long)step_k * plane + (long long)step_j * G.wx;
    const long long wrap_row = plane - (long long)ny_box * G.wx;
    for (; k <= hi[2]; k += step_k) {
      const float dyf = __fsub_rn(__fmaf_rn(G.h, (float)j, G.oy), c.y);
      const float dzf = __fsub_rn(__fmaf_rn(G.h, (float)k, G.oz), c.z);
      const float yz = __fmaf_rn(dyf, dyf, __fmul_rn(dzf, dzf));
      const float t = R2f - yz;
      if (t > 4.0f * M) {
        const float rs = rsqrtf(t);
        const float w = t * rs * inv_h, u = fmaf(Mh, rs, eps + 1e-6f * w);
        const int i0 = max(__float2int_ru(xc - w - u), lo[0]), a = max(__float2int_ru(xc - w + u), lo[0]);
        const int i1 = min(__float2int_rd(xc + w + u), hi[0]), b = min(__float2int_rd(xc + w - u), hi[0]);
        if (a <= b) {
          const int wa = a >> 5, wb = b >> 5;
          const uint32_t ma = 0xffffffffu << (a & 31), mb = 0xffffffffu >> (31 - (b & 31));
          if (wa == wb) {
            atomicOr(row + wa, ma & mb);
          } else {
            atomicOr(row + wa, ma);
            for (int q = wa + 1; q < wb; ++q) atomicOr(row + q, 0xffffffffu);
            atomicOr(row + wb, mb);
          }
        }
        if (a != i0 || b != i1) sas_row_exact(G.ox, G.oy, G.oz, G.h, G.p, c, j, k, i0, i1, a, b, row);
      } else if (!(t < -M)) {  // else the whole row is outside
        const float w = sqrtf(fmaxf(t + M, 0.0f)) * 1.000001f * inv_h;
        const bool all = !(t + M < INFINITY);
        const int i0 = all ? lo[0] : max(__float2int_ru(xc - w - eps), lo[0]);
        const int i1 = all ? hi[0] : min(__float2int_rd(xc + w + eps), hi[0]);
        sas_row_exact(G.ox, G.oy, G.oz, G.h, G.p, c, j, k, i0, i1, 1, 0, row);
      }
      j += step_j;
      row += step_row;
      if (j > hi[1]) {
        j -= (int)ny_box;
        ++k;
        row += wrap_row;
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
  uint32_t outside = 0u;         // points whose distance is below the SES threshold
  uint32_t plane[6] = {};        // binary digits of each point's level
};

template <int K, int I>
__device__ __forceinline__ void ses_step(const uint32_t *e, int t_in, SesLevelState<K> &s) {
  constexpr int off = kSesSteps<K>.off[I], lv = kSesSteps<K>.level[I];
  constexpr bool last = kSesSteps<K>.level[I + 1] != lv;
  s.acc |= e[off];
  if constexpr (last) {
    constexpr int value = kSesSteps<K>.value[lv];
    if (value < t_in) s.outside = s.acc;
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
__device__ __forceinline__ void ses_steps(const uint32_t *e, int t_in, SesLevelState<K> &s,
                                          std::integer_sequence<int, I...>) {
  (ses_step<K, I>(e, t_in, s), ...);
}

// Transpose of a 32 x 32 bit matrix, row l in lane l: lane l receives bit l of every row (blocks of 16, 8, 4, 2, 1
// columns exchanged between lanes that far apart).
__device__ __forceinline__ uint32_t warp_transpose(uint32_t v, int lane) {
  uint32_t m = 0x0000ffffu;  // the columns whose index has bit s clear
#pragma unroll
  for (int s = 16; s > 0; s >>= 1, m ^= m << s) {
    const uint32_t o = __shfl_xor_sync(0xffffffffu, v, s);
    v = (lane & s) ? ((v & ~m) | ((o >> s) & m)) : ((v & m) | ((o << s) & ~m));
  }
  return v;
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
// Bound by issue (K = 4: 153 reads and ORs a word; 79 % of the issue slots, ALU 70 %, shared memory 58 %).  3.4e7 points at
// K = 4: 66 us; the three separable passes over 16-bit planes (one point per thread) take 105 + 2 x 172 us.  K <= 6
// because the offsets grow with K^3 (519 at K = 6) and every one is an unrolled instruction.
template <int K>
__global__ __launch_bounds__(256) void k_ses_levels(SesGrid G, const uint32_t *__restrict__ bits,
                                                    uint16_t *__restrict__ edt2, uint32_t *__restrict__ inside) {
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
  ses_steps<K>(s_e + (zw + K) * S::PY + lane + K, G.t_in, st, std::make_integer_sequence<int, kSesSteps<K>.n>{});
  const uint32_t rest = ~st.acc;  // farther than K: the last level
#pragma unroll
  for (int p = 0; p < 6; ++p)
    if ((n_levels >> p) & 1) st.plane[p] |= rest;
  // spread: one point per lane and row.  Each digit plane's 32 x 32 bits (row r in lane r) are transposed across
  // the warp, so that lane x holds point x of every row; a row's level is then a bit of each plane.
  constexpr int planes = n_levels < 2 ? 1 : n_levels < 4 ? 2 : n_levels < 8 ? 3 : n_levels < 16 ? 4 : n_levels < 32 ? 5 : 6;
  const long long z = z0 + zw, x = 32LL * w + lane;
  if (z >= G.nz) return;  // uniform in the warp; no barrier follows
  const int rows = (int)min((long long)S::TY, G.ny - y0);
  if (lane < rows) inside[(z * G.ny + y0 + lane) * G.wx + w] = ~st.outside;
#pragma unroll
  for (int p = 0; p < planes; ++p) st.plane[p] = warp_transpose(st.plane[p], lane);
  uint16_t *dst = edt2 + (z * G.ny + y0) * G.nx + x;
  const bool mine = x < G.nx;
#pragma unroll 8
  for (int r = 0; r < rows; ++r, dst += G.nx) {
    unsigned lv = 0u;
#pragma unroll
    for (int p = planes - 1; p >= 0; --p) lv = 2u * lv + ((st.plane[p] >> r) & 1u);
    if (mine) *dst = s_val[lv];
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

// SES interior bits from the distances (three-pass windows): one warp per word.
__global__ __launch_bounds__(256) void k_ses_inside(SesGrid G, const uint16_t *__restrict__ edt2, long long n_words,
                                                    uint32_t *__restrict__ inside) {
  const int lane = threadIdx.x & 31;
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long q = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < n_words; q += n_warps) {
    const long long row = q / G.wx;
    const int x = 32 * (int)(q - row * G.wx) + lane;
    const unsigned m = __ballot_sync(0xffffffffu, x < G.nx && (int)edt2[row * G.nx + x] >= G.t_in);
    if (lane == 0) inside[q] = m;
  }
}

// --------------------------------------------------------- marching cubes --

// The corner bits of a group's 32 cells (i0 .. i0 + 31 of row (j, k)) and which of the cells cross the surface.
struct SesGroup {
  int i0, j, k;
  uint32_t c[8];   // c[q] bit t: corner q of cell i0 + t is inside
  uint32_t active;
};

__device__ __forceinline__ SesGroup ses_group(const SesGrid &G, const uint32_t *__restrict__ inside, uint32_t g,
                                              uint32_t n_groups) {
  SesGroup s;
  const uint32_t wc = (uint32_t)(G.nx + 30) / 32u;  // groups per row of nx - 1 cells
  const uint32_t row = g / wc, w = g - row * wc;
  s.i0 = (int)(w * 32u);
  s.k = (int)(row / (uint32_t)(G.ny - 1));
  s.j = (int)(row - (uint32_t)s.k * (uint32_t)(G.ny - 1));
  s.active = 0u;
  if (g >= n_groups) return s;
  const uint32_t *p = inside + ((size_t)s.k * G.ny + s.j) * G.wx + w;
  const size_t up = (size_t)G.ny * G.wx;
  const bool next = (int)w + 1 < G.wx;
  const uint32_t r0 = p[0], r1 = p[G.wx], r2 = p[up], r3 = p[up + G.wx];
  const uint32_t n0 = next ? p[1] : 0u, n1 = next ? p[G.wx + 1] : 0u;
  const uint32_t n2 = next ? p[up + 1] : 0u, n3 = next ? p[up + G.wx + 1] : 0u;
  s.c[0] = r0;
  s.c[3] = r1;
  s.c[4] = r2;
  s.c[7] = r3;
  s.c[1] = __funnelshift_r(r0, n0, 1);
  s.c[2] = __funnelshift_r(r1, n1, 1);
  s.c[5] = __funnelshift_r(r2, n2, 1);
  s.c[6] = __funnelshift_r(r3, n3, 1);
  const uint32_t any = s.c[0] | s.c[1] | s.c[2] | s.c[3] | s.c[4] | s.c[5] | s.c[6] | s.c[7];
  const uint32_t all = s.c[0] & s.c[1] & s.c[2] & s.c[3] & s.c[4] & s.c[5] & s.c[6] & s.c[7];
  const int cells = G.nx - 1 - s.i0;  // > 0
  s.active = any & ~all & (cells >= 32 ? 0xffffffffu : (1u << cells) - 1u);
  return s;
}

__device__ __forceinline__ unsigned ses_case_of(const SesGroup &s, int t) {
  unsigned cs = 0u;
#pragma unroll
  for (int q = 0; q < 8; ++q) cs |= ((s.c[q] >> t) & 1u) << q;
  return cs;
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
  unsigned before = x - v, sum = 0u;
#pragma unroll
  for (int q = 0; q < kSesThreads / 32; ++q) {
    const unsigned t = s_warp[q];
    if (q < w) before += t;
    sum += t;
  }
  __syncthreads();
  *total = sum;
  return before;
}

// Triangles of every `per_cta` <= 256 groups (one group per thread, going through its crossing cells), and, in the last
// CTA to finish, their exclusive scan: block_base[b] is the first triangle of CTA b's groups.  *done counts finished
// CTAs (zero at launch); no CTA waits for another.  3.4e7 points: 27 us, ALU at 64 % with half of the lanes idle
// (groups differ in crossing cells); 307 us with one thread per four cells reading the distance plane, and 100 us
// for the scan of its eight times as many counts in a launch of its own.
__global__ __launch_bounds__(kSesThreads) void k_ses_count(SesGrid G, const uint32_t *__restrict__ inside,
                                                           uint32_t n_groups, unsigned per_cta,
                                                           unsigned *__restrict__ block_tris,
                                                           unsigned long long *__restrict__ block_base,
                                                           unsigned long long *__restrict__ total, unsigned *done) {
  __shared__ unsigned char s_tris[256];
  __shared__ bool s_last;
  s_tris[threadIdx.x] = g_ses_case[threadIdx.x].n_tris;
  __syncthreads();
  const SesGroup s = ses_group(G, inside, blockIdx.x * per_cta + threadIdx.x,
                               threadIdx.x < per_cta ? n_groups : 0u);
  unsigned n = 0u;
  for (uint32_t m = s.active; m != 0u; m &= m - 1u) n += s_tris[ses_case_of(s, __ffs(m) - 1)];
  unsigned sum;
  block_exclusive_sum(n, &sum);
  if (threadIdx.x == 0) {
    block_tris[blockIdx.x] = sum;
    __threadfence();
    s_last = atomicAdd(done, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!s_last) return;
  // consecutive counts per thread: their sum, a block scan of the sums (64 bits in two halves), then the bases
  __threadfence();
  const unsigned nb = gridDim.x, per = (nb + kSesThreads - 1) / kSesThreads;
  const unsigned b0 = min(threadIdx.x * per, nb), b1 = min(b0 + per, nb);
  unsigned long long mine = 0ull;
#pragma unroll 8
  for (unsigned b = b0; b < b1; ++b) mine += __ldcg(block_tris + b);
  __shared__ unsigned long long s_sum[kSesThreads];
  s_sum[threadIdx.x] = mine;
  __syncthreads();
  for (int o = 1; o < kSesThreads; o <<= 1) {
    const unsigned long long y = (int)threadIdx.x >= o ? s_sum[threadIdx.x - o] : 0ull;
    __syncthreads();
    s_sum[threadIdx.x] += y;
    __syncthreads();
  }
  unsigned long long run = s_sum[threadIdx.x] - mine;
#pragma unroll 8
  for (unsigned b = b0; b < b1; ++b) {
    block_base[b] = run;
    run += __ldcg(block_tris + b);
  }
  if (threadIdx.x == kSesThreads - 1) *total = s_sum[threadIdx.x];
}

// Shared memory of the emit pass, for 256 crossing cells at a time.
struct SesEmitShared {
  float at[12][kSesThreads];       // the vertex of every crossing edge of each cell: its coordinate along the edge
  float mean[12][kSesThreads];     // means of its loops: x, y, z of loop l at 3 l
  float grid[6][kSesThreads];      // its lower and upper grid coordinates: x, y, z at 2 axis + upper
  float stage[kSesThreads / 32][32 * 9];  // per warp: 32 triangles on their way out
  int ci[kSesThreads], cj[kSesThreads], ck[kSesThreads];
  unsigned off[kSesThreads];       // first triangle of each cell
  unsigned char cs[kSesThreads];   // case
  unsigned char cell_of[kSesThreads * 12];  // cell of each triangle
};
static_assert(sizeof(SesEmitShared) <= 48 * 1024, "static shared memory");

// Edges by direction (bit e): along x, y, z; and by the upper side of the cell that they lie on.  An edge runs from
// its first corner to its second: along x 0, 2, 4, 6 (2 and 6 downward), along y 1, 3, 5, 7 (3 and 7 downward).
constexpr unsigned kEdgeX = 0x055u, kEdgeY = 0x0aau, kEdgeZ = 0xf00u;
constexpr unsigned kEdgeUpX = 0x622u, kEdgeUpY = 0xc44u, kEdgeUpZ = 0x0f0u;

// The vertex on edge e of a cell.
__device__ __forceinline__ float3 edge_point(const SesEmitShared &sh, int cell, int e) {
  const float v = sh.at[e][cell];
  const float x = sh.grid[(kEdgeUpX >> e) & 1u][cell], y = sh.grid[2 + ((kEdgeUpY >> e) & 1u)][cell];
  const float z = sh.grid[4 + ((kEdgeUpZ >> e) & 1u)][cell];
  return make_float3((kEdgeX >> e) & 1u ? v : x, (kEdgeY >> e) & 1u ? v : y, (kEdgeZ >> e) & 1u ? v : z);
}

// Triangles of the groups of CTA blockIdx.x, in cell order.  The groups' crossing cells are taken 256 at a time,
// one per thread: the eight distances are read once and give the parameter of every crossing edge and the means
// of the longer loops; then one thread per triangle puts its three vertices together and the warp writes its 32
// triangles as one run of floats.
//
// Bound by shared memory, issue and the barriers between the steps: L1 63 %, 66 % of the issue slots, 22 of 32 lanes; DRAM
// 17 %.  5.9e6 triangles (212 MB): 123 us, with f read from a table of the window's distances and the vertices kept
// as one coordinate along their edge; 146 us with a root per corner and positions worked out per triangle; 789 us with
// one thread per triangle finding its cell by binary search over a case byte per cell, recomputing its loop's vertices
// from the distance plane and storing 36-byte strides.
__global__ __launch_bounds__(kSesThreads) void k_ses_emit(SesGrid G, const uint16_t *__restrict__ edt,
                                                          const uint32_t *__restrict__ inside, uint32_t n_groups,
                                                          unsigned per_cta,
                                                          const unsigned long long *__restrict__ block_base,
                                                          float *__restrict__ tris, long long *__restrict__ labels,
                                                          unsigned long long max_tris) {
  __shared__ SesEmitShared sh;
  __shared__ float s_f[kSesBitK * kSesBitK + 2];  // f of every distance that a bit-set window has
  const bool table = G.K <= kSesBitK;
  unsigned long long base = block_base[blockIdx.x];
  if (base >= max_tris) return;
  if (threadIdx.x <= kSesBitK * kSesBitK + 1) s_f[threadIdx.x] = fmaf(sqrtf((float)threadIdx.x), G.h, -G.p);
  const SesGroup s = ses_group(G, inside, blockIdx.x * per_cta + threadIdx.x,
                               threadIdx.x < per_cta ? n_groups : 0u);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  unsigned n_cells;
  unsigned rank = block_exclusive_sum((unsigned)__popc(s.active), &n_cells);
  uint32_t rem = s.active;
  const size_t ny = (size_t)G.ny, nx = (size_t)G.nx;
  for (unsigned c0 = 0; c0 < n_cells; c0 += kSesThreads) {
    for (; rem != 0u && rank < c0 + kSesThreads; rem &= rem - 1u, ++rank) {
      const int t = __ffs(rem) - 1;
      const unsigned at = rank - c0;
      sh.ci[at] = s.i0 + t;
      sh.cj[at] = s.j;
      sh.ck[at] = s.k;
      sh.cs[at] = (unsigned char)ses_case_of(s, t);
    }
    __syncthreads();
    unsigned n_tri = 0u;
    const bool have = c0 + tid < n_cells;
    if (have) {
      const int i = sh.ci[tid], j = sh.cj[tid], k = sh.ck[tid];
      const unsigned cs = sh.cs[tid];
      const SesCase &tc = g_ses_case[cs];
      n_tri = tc.n_tris;
      const uint16_t *q = edt + ((size_t)k * ny + (size_t)j) * nx + (size_t)i;
      const size_t up = ny * nx;
      const int d[8] = {q[0], q[1], q[nx + 1], q[nx], q[up], q[up + 1], q[up + nx + 1], q[up + nx]};
      float f[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) f[c] = table ? s_f[d[c]] : fmaf(sqrtf((float)d[c]), G.h, -G.p);
      float g[6];
      g[0] = fmaf(G.h, (float)i, G.ox);
      g[1] = fmaf(G.h, (float)(i + 1), G.ox);
      g[2] = fmaf(G.h, (float)j, G.oy);
      g[3] = fmaf(G.h, (float)(j + 1), G.oy);
      g[4] = fmaf(G.h, (float)k, G.oz);
      g[5] = fmaf(G.h, (float)(k + 1), G.oz);
#pragma unroll
      for (int c = 0; c < 6; ++c) sh.grid[c][tid] = g[c];
      constexpr int ea[12] = {0, 1, 2, 3, 4, 5, 6, 7, 0, 1, 2, 3};
      constexpr int eb[12] = {1, 2, 3, 0, 5, 6, 7, 4, 4, 5, 6, 7};
#pragma unroll
      for (int e = 0; e < 12; ++e) {
        if (((cs >> ea[e]) ^ (cs >> eb[e])) & 1u) {
          // X_a + t (X_b - X_a) along the edge's axis, t = f_a / (f_a - f_b)
          const float fa = f[ea[e]], fb = f[eb[e]];
          const float t = fminf(fmaxf(fa == fb ? 0.5f : fa / (fa - fb), 0.0f), 1.0f);
          const int axis = e >= 8 ? 4 : ((e & 1) ? 2 : 0);
          const bool down = e < 8 && (e & 2);
          const float xa = down ? g[axis + 1] : g[axis], xb = down ? g[axis] : g[axis + 1];
          sh.at[e][tid] = fmaf(t, xb - xa, xa);
        }
      }
      for (int l = 0, at = 0; l < tc.n_loops; at += tc.len[l], ++l) {
        const int len = tc.len[l];
        if (len == 3) continue;
        float3 M = make_float3(0.0f, 0.0f, 0.0f);
        for (int v = 0; v < len; ++v) {
          const int e = tc.edge[at + v];
          const float3 p = edge_point(sh, tid, e);
          M.x += p.x;
          M.y += p.y;
          M.z += p.z;
        }
        const float inv = 1.0f / (float)len;
        sh.mean[3 * l][tid] = M.x * inv;
        sh.mean[3 * l + 1][tid] = M.y * inv;
        sh.mean[3 * l + 2][tid] = M.z * inv;
      }
    }
    unsigned total;
    const unsigned off = block_exclusive_sum(n_tri, &total);
    sh.off[tid] = off;
    for (unsigned t = 0; t < n_tri; ++t) sh.cell_of[off + t] = (unsigned char)tid;
    __syncthreads();
    for (unsigned q0 = 32u * wid; q0 < total && base + q0 < max_tris; q0 += kSesThreads) {
      const unsigned q = q0 + lane;
      const unsigned live = min(min(32u, total - q0), (unsigned)min(max_tris - (base + q0), 32ull));
      if (lane < live) {
        const int cell = sh.cell_of[q];
        const unsigned code = g_ses_case[sh.cs[cell]].tri[q - sh.off[cell]];
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          const int e = (int)((code >> (4 * v)) & 15u);
          float3 p;
          if (e < 12)
            p = edge_point(sh, cell, e);
          else
            p = make_float3(sh.mean[3 * (e - 12)][cell], sh.mean[3 * (e - 12) + 1][cell], sh.mean[3 * (e - 12) + 2][cell]);
          sh.stage[wid][9 * lane + 3 * v] = p.x;
          sh.stage[wid][9 * lane + 3 * v + 1] = p.y;
          sh.stage[wid][9 * lane + 3 * v + 2] = p.z;
          if (labels) {
            const long long cell_id = ((long long)sh.ck[cell] * (G.ny - 1) + sh.cj[cell]) * (G.nx - 1) + sh.ci[cell];
            labels[(base + q) * 3 + v] = cell_id * 16 + e;
          }
        }
      }
      __syncwarp();
      float *out = tris + (base + q0) * 9;
#pragma unroll
      for (unsigned o = 0; o < 9; ++o)
        if (32u * o + lane < 9u * live) out[32u * o + lane] = sh.stage[wid][32u * o + lane];
      __syncwarp();
    }
    base += total;
    __syncthreads();  // the cells are read before the next ones replace them
  }
}

// Bounding box of the SAS spheres: min and max of c -/+ (r + p).  Each CTA leaves its bounds, and the last one to
// finish reduces them into box[0..5]: one launch and 24 bytes for the host.  *done counts finished CTAs (zero at
// launch).
constexpr int kSesBoxCtas = 512;

__device__ __forceinline__ void ses_box_reduce(float (&lo)[3], float (&hi)[3], float *out) {
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
    out[threadIdx.x] = v;
  }
  __syncthreads();
}

__global__ __launch_bounds__(256) void k_ses_bbox(const float4 *__restrict__ X, long long n, float p, float *box,
                                                  float *partial, unsigned *done) {
  __shared__ bool s_last;
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x; a < n; a += (long long)gridDim.x * blockDim.x) {
    const float4 c = X[a];
    const float R = c.w + p;
    lo[0] = fminf(lo[0], c.x - R), hi[0] = fmaxf(hi[0], c.x + R);
    lo[1] = fminf(lo[1], c.y - R), hi[1] = fmaxf(hi[1], c.y + R);
    lo[2] = fminf(lo[2], c.z - R), hi[2] = fmaxf(hi[2], c.z + R);
  }
  ses_box_reduce(lo, hi, partial + 6 * blockIdx.x);
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int d = 0; d < 3; ++d) {
    lo[d] = INFINITY;
    hi[d] = -INFINITY;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
      lo[d] = fminf(lo[d], __ldcg(partial + 6 * b + d));
      hi[d] = fmaxf(hi[d], __ldcg(partial + 6 * b + 3 + d));
    }
  }
  ses_box_reduce(lo, hi, box);
}

// ------------------------------------------------------------- launchers --

int ses_window(float probe, float h) { return (int)std::ceil((double)probe / (double)h) + 1; }

bool ses_three_pass(float probe, float h) { return ses_window(probe, h) > kSesBitK; }

// Groups of 32 cells (dims >= 2 and at most 2^32 points: at most 2^31 groups).
static long long ses_groups(const int32_t dims[3]) {
  return ((long long)dims[0] + 30) / 32 * (dims[1] - 1) * (dims[2] - 1);
}

// Groups per CTA of the count and emit passes: 256, or fewer (down to 32) while that leaves less than four CTAs per SM,
// so that a small grid's cells spread over the chip (1,200 atoms at 0.6 A, 16,000 groups: emit 25 us at 256, 10 at 32).
static unsigned ses_per_cta(const int32_t dims[3]) {
  unsigned per = kSesThreads;
  while (per > 32 && ses_groups(dims) / per < 4LL * sm_count()) per >>= 1;
  return per;
}

long long ses_words(const int32_t dims[3]) { return ((long long)dims[0] + 31) / 32 * dims[1] * dims[2]; }

template <int K>
static void launch_levels(const SesGrid &G, const SesLaunch &L, cudaStream_t st) {
  using S = SesSteps<K>;
  const long long tiles = (long long)G.wx * (((long long)G.ny + S::TY - 1) / S::TY) * (((long long)G.nz + S::TZ - 1) / S::TZ);
  k_ses_levels<K><<<(unsigned)tiles, 256, 0, st>>>(G, L.bits, L.edt2, L.inside);
}

size_t ses_bbox_bytes() { return sizeof(float) * (8 + 6 * (size_t)kSesBoxCtas); }

cudaError_t run_ses_bbox(const float4 *X, long long n, float probe, float *box, cudaStream_t st) {
  // box: six bounds, the counter, one unused word, then the CTAs' bounds
  unsigned *done = reinterpret_cast<unsigned *>(box + 6);
  cudaError_t e = cudaMemsetAsync(done, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  const long long want = (n + 255) / 256;
  k_ses_bbox<<<(int)(want < kSesBoxCtas ? want : kSesBoxCtas), 256, 0, st>>>(X, n, probe, box, box + 8, done);
  return cudaGetLastError();
}

static SesGrid make_grid(const SesLaunch &L) {
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
  return G;
}

cudaError_t run_ses_count(const SesLaunch &L, cudaStream_t st) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (!ses_table_ready(dev)) return cudaErrorInvalidValue;
  const SesGrid G = make_grid(L);
  const long long n_pts = (long long)G.nx * G.ny * G.nz;
  const int sms = sm_count();
  cudaError_t e = cudaMemsetAsync(L.bits, 0, 4 * (size_t)(ses_words(L.dims) + 1), st);  // and the counter after them
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
    const long long n_words = ses_words(L.dims);
    const long long wb = (n_words + 7) / 8;
    k_ses_inside<<<(int)(wb < 16LL * sms ? wb : 16LL * sms), 256, 0, st>>>(G, L.edt2, n_words, L.inside);
  }
  if (L.edt2_copy) {
    e = cudaMemcpyAsync(L.edt2_copy, L.edt2, 2 * (size_t)n_pts, cudaMemcpyDefault, st);
    if (e != cudaSuccess) return e;
  }
  const long long n_blocks = ses_blocks(L.dims);
  unsigned *done = reinterpret_cast<unsigned *>(L.bits + ses_words(L.dims));  // cleared with the bits
  k_ses_count<<<(unsigned)n_blocks, kSesThreads, 0, st>>>(G, L.inside, (uint32_t)ses_groups(L.dims),
                                                          ses_per_cta(L.dims), L.block_tris, L.block_base, L.total, done);
  return cudaGetLastError();
}

cudaError_t run_ses_emit(const SesLaunch &L, cudaStream_t st) {
  if (L.max_tris == 0) return cudaSuccess;
  k_ses_emit<<<(unsigned)ses_blocks(L.dims), kSesThreads, 0, st>>>(
      make_grid(L), L.edt2, L.inside, (uint32_t)ses_groups(L.dims), ses_per_cta(L.dims), L.block_base, L.tris, L.labels,
      (unsigned long long)L.max_tris);
  return cudaGetLastError();
}

long long ses_blocks(const int32_t dims[3]) {
  const long long per = ses_per_cta(dims);
  return (ses_groups(dims) + per - 1) / per;
}

}  // namespace vtx
