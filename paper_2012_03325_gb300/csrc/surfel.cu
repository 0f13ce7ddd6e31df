// The G-buffer pass of surfel rendering (Sec. 4.3): oriented elliptical disks splatted into the
// FP32 G-buffer, the surfels within a depth window of the nearest one blended.
//   k_surfel_count  one thread per surfel: view-space frame, the near rule, the pixel box of the
//                   projected ellipse (its image conic's extent, widened by 1/8 pixel), and the
//                   number of surfels per cell of a pyramid of grids, 8 x 4 pixels at level 0,
//                   doubled from level to level; a surfel is listed in the cells its box meets on
//                   the finest level where these are at most 24
//   k_surfel_alloc  every cell's range of the list (ranges in any order: a block sum and one
//                   atomicAdd per 256 cells), and the heavy tiles: those whose lists would keep one warp
//                   busy after the others are done
//   k_surfel_fill   the surfels' indices into their cells' ranges
//   k_surfel_tile   one warp per 8 x 4 pixels, a lane per pixel: the surfels listed in the tile's
//                   cells, 32 at a time, their frames computed by one lane each into shared memory,
//                   their box pixels tested a lane per (surfel, pixel); nearest depth, blended sums
//                   and count stay in the pixel's lane, the means are written as the FP32 G-buffer.
//                   A heavy tile is shared out, units of its list to many warps, which only find the
//                   nearest depths here
//   k_surfel_heavy  the heavy tiles' units again, with the depth windows known: the sums, and the means by
//                   the warp that finishes a tile's last unit
// The decisions evaluate the oracle's FP32 expressions with each product, sum, quotient and
// square root rounded in the same order, so which pixels a surfel covers, the nearest depth and
// the window reproduce bit for bit; only the order of the attribute sums varies (the lists' order).
#include <string.h>

#include <algorithm>
#include <cmath>

#include "epbr_internal.cuh"

namespace epbr {

// A surfel as the pixel test reads it.
struct SurfelFrame {
  float4 n;   // view-space unit normal, 1 / a^2
  float4 t;   // view-space unit tangent, 1 / b^2
  float4 b;   // bitangent n^ x t^, c . t^
  float cb, nc;  // c . b^, n^ . c (c the view-space centre)
};

struct SurfelCam {
  float axes[9];  // the view axes in world space, axis k at 3 k
  float eye[3];
  float kx, ky, hw, hh, near, f;  // f = 1 + depth tolerance, rounded to FP32
  int W, H;
};

__device__ __forceinline__ float dot_rn(float a0, float a1, float a2, float b0, float b1, float b2) {
  return __fadd_rn(__fadd_rn(__fmul_rn(a0, b0), __fmul_rn(a1, b1)), __fmul_rn(a2, b2));
}

// View-space frame of a surfel from the first three quarters of its record; false when it is
// dropped (degenerate, or nearer than the near rule allows).
__device__ __forceinline__ bool surfel_frame(const float4 r0, const float4 r1, const float4 r2, const SurfelCam& cam,
                                             SurfelFrame& s, float (&c)[3]) {
  const float inf = __int_as_float(0x7f800000);
  const float d0 = __fsub_rn(r0.x, cam.eye[0]), d1 = __fsub_rn(r0.y, cam.eye[1]), d2 = __fsub_rn(r0.z, cam.eye[2]);
  float nv[3], tv[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float* ax = cam.axes + 3 * k;
    c[k] = dot_rn(ax[0], ax[1], ax[2], d0, d1, d2);
    nv[k] = dot_rn(ax[0], ax[1], ax[2], r1.x, r1.y, r1.z);
    tv[k] = dot_rn(ax[0], ax[1], ax[2], r2.x, r2.y, r2.z);
  }
  const float a = r0.w, b = r1.w;
  bool ok = a > 0.0f && b > 0.0f && a < inf && b < inf;
  const float nn = dot_rn(nv[0], nv[1], nv[2], nv[0], nv[1], nv[2]);
  ok = ok && nn > 0.0f && nn < inf;
  const float inv = __fdiv_rn(1.0f, __fsqrt_rn(nn));
  const float n0 = __fmul_rn(nv[0], inv), n1 = __fmul_rn(nv[1], inv), n2 = __fmul_rn(nv[2], inv);
  const float dt = dot_rn(tv[0], tv[1], tv[2], n0, n1, n2);
  const float p0 = __fsub_rn(tv[0], __fmul_rn(n0, dt)), p1 = __fsub_rn(tv[1], __fmul_rn(n1, dt)),
              p2 = __fsub_rn(tv[2], __fmul_rn(n2, dt));
  const float tt = dot_rn(p0, p1, p2, p0, p1, p2);
  ok = ok && tt > 0.0f && tt < inf;
  const float invt = __fdiv_rn(1.0f, __fsqrt_rn(tt));
  const float t0 = __fmul_rn(p0, invt), t1 = __fmul_rn(p1, invt), t2 = __fmul_rn(p2, invt);
  const float b0 = __fsub_rn(__fmul_rn(n1, t2), __fmul_rn(n2, t1));
  const float b1 = __fsub_rn(__fmul_rn(n2, t0), __fmul_rn(n0, t2));
  const float b2 = __fsub_rn(__fmul_rn(n0, t1), __fmul_rn(n1, t0));
  s.n = make_float4(n0, n1, n2, __fdiv_rn(1.0f, __fmul_rn(a, a)));
  s.t = make_float4(t0, t1, t2, __fdiv_rn(1.0f, __fmul_rn(b, b)));
  s.b = make_float4(b0, b1, b2, dot_rn(c[0], c[1], c[2], t0, t1, t2));
  s.cb = dot_rn(c[0], c[1], c[2], b0, b1, b2);
  s.nc = dot_rn(n0, n1, n2, c[0], c[1], c[2]);
  return ok && __fsub_rn(-c[2], __fadd_rn(a, b)) >= cam.near;
}

// Pixel box of the projected ellipse (the whole disk lies at eye depth >= near), clipped to the
// image: (x0, y0, width, height), width 0 when it holds no pixel.  With
// G = [a t^, b b^, c] the disk's boundary is G (cos, sin, 1); M maps view space to
// homogeneous pixel coordinates taken relative to the projected centre (Xc, Yc), so
// H = M G maps the unit circle onto the image conic, whose tangent lines l satisfy
// l^T H D H^T l = 0 with D = diag(1, 1, -1).  The lines X' = x are l = (1, 0, -x): the
// silhouette's extent along x is the two roots of C00 - 2 x C02 + x^2 C22 = 0 (C = H D H^T),
// likewise along y.  The box holds every pixel whose centre lies within 1/8 pixel (plus 1e-4
// of the extent) of that range: FP32 errors of these bounds are below 1e-3 pixel, and pixels
// that the rounded ellipse test accepts lie within ~1e-6 of the ellipse's size of it.
__device__ __forceinline__ int4 surfel_box(const SurfelFrame& s, const float (&c)[3], float a, float b,
                                           const SurfelCam& cam) {
  const float ec = -c[2];
  const float Xc = cam.hw * (1.0f + cam.kx * c[0] / ec), Yc = cam.hh * (1.0f - cam.ky * c[1] / ec);
  const float g0[3] = {a * s.t.x, b * s.b.x, c[0]}, g1[3] = {a * s.t.y, b * s.b.y, c[1]},
              g2[3] = {a * s.t.z, b * s.b.z, c[2]};
  float h0[3], h1[3], h2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    h0[k] = cam.hw * cam.kx * g0[k] + (Xc - cam.hw) * g2[k];
    h1[k] = -cam.hh * cam.ky * g1[k] + (Yc - cam.hh) * g2[k];
    h2[k] = -g2[k];
  }
  auto dd = [](const float* u, const float* v) { return u[0] * v[0] + u[1] * v[1] - u[2] * v[2]; };
  const float C22 = dd(h2, h2);  // a^2 t_z^2 + b^2 b_z^2 - e_c^2 < 0 for a disk in front of the eye
  float lo[2], hi[2];
  const float* hr[2] = {h0, h1};
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float C00 = dd(hr[q], hr[q]), C02 = dd(hr[q], h2);
    const float sq = sqrtf(fmaxf(C02 * C02 - C00 * C22, 0.0f));
    const float r0 = (C02 + sq) / C22, r1 = (C02 - sq) / C22;
    const float m = 0.125f + 1e-4f * fabsf(r1 - r0);
    lo[q] = fminf(r0, r1) - m;
    hi[q] = fmaxf(r0, r1) + m;
  }
  float fx0 = fmaxf(ceilf(Xc + lo[0] - 0.5f), 0.0f), fy0 = fmaxf(ceilf(Yc + lo[1] - 0.5f), 0.0f);
  float fx1 = fminf(floorf(Xc + hi[0] - 0.5f), (float)(cam.W - 1));
  float fy1 = fminf(floorf(Yc + hi[1] - 0.5f), (float)(cam.H - 1));
  if (!(C22 < 0.0f)) {  // a disk grazing the eye plane (rounding only): the whole view
    fx0 = fy0 = 0.0f;
    fx1 = (float)(cam.W - 1);
    fy1 = (float)(cam.H - 1);
  }
  if (!(fx1 >= fx0 && fy1 >= fy0)) return make_int4(0, 0, 0, 0);  // or a NaN bound
  const int x0 = (int)fx0, y0 = (int)fy0;
  return make_int4(x0, y0, (int)fx1 - x0 + 1, (int)fy1 - y0 + 1);
}

// Eye depth at which the pixel ray d = (ux, uy, -1) meets the surfel inside its ellipse, else 0:
// with U = (n^.c)(d.t^) - (n^.d)(c.t^), V likewise with b^, covered when (n^.c)(n^.d) > 0 and
// U^2 / a^2 + V^2 / b^2 <= (n^.d)^2; the depth (n^.c) / (n^.d) is formed only then.
__device__ __forceinline__ float surfel_hit(const SurfelFrame& s, float ux, float uy) {
  const float nd = __fsub_rn(__fadd_rn(__fmul_rn(s.n.x, ux), __fmul_rn(s.n.y, uy)), s.n.z);
  const float dt = __fsub_rn(__fadd_rn(__fmul_rn(s.t.x, ux), __fmul_rn(s.t.y, uy)), s.t.z);
  const float db = __fsub_rn(__fadd_rn(__fmul_rn(s.b.x, ux), __fmul_rn(s.b.y, uy)), s.b.z);
  if (!(__fmul_rn(s.nc, nd) > 0.0f)) return 0.0f;
  const float U = __fsub_rn(__fmul_rn(s.nc, dt), __fmul_rn(nd, s.b.w));
  const float V = __fsub_rn(__fmul_rn(s.nc, db), __fmul_rn(nd, s.cb));
  const float e = __fadd_rn(__fmul_rn(__fmul_rn(U, U), s.n.w), __fmul_rn(__fmul_rn(V, V), s.t.w));
  if (!(e <= __fmul_rn(nd, nd))) return 0.0f;
  const float sd = __fdiv_rn(s.nc, nd);
  return (sd > 0.0f && sd < __int_as_float(0x7f800000)) ? sd : 0.0f;
}

// ---- the pyramid of cells --------------------------------------------------------------------
constexpr int kTileW = 8, kTileH = 4;     // pixels of a level-0 cell: one warp's tile
constexpr int kSurfelLevels = 14;         // enough for 32768 rows: the last level has one row of cells
constexpr int kSurfelCells = 24;          // list entries per surfel: 96 bytes of workspace
// Atomics on one counter, or on counters of one 128-byte line, follow each other at 0.7 and 0.2 ns: with many
// surfels for the cells the counts, not the tiles, bound the pass.  1.2 M surfels over a 64 x 64 view take
// 1828 us with dense counters and 687 us with a line for each.  Arrays of at most 2^16, 2^17, 2^18 or 2^19 words:
// 1.2 M surfels in the middle tenth of a 640 x 480 view 1012, 846, 805, 781 us; 70,000 over all of it 92, 82,
// 79, 85.
constexpr int kSurfelSpread = 131072;

struct SurfelGrid {
  int levels;
  int stride;                       // words from one cell's counter to the next
  int most;                         // cells a surfel is listed in at most
  int nx[kSurfelLevels];            // cells per row of a level
  int first[kSurfelLevels + 1];     // its first cell
  __device__ __forceinline__ int at(int k) const { return k * stride; }
};

// Packed box: x0 | y0 << 16, width | height << 16 (each at most 32768; width 0: not drawn).
__device__ __forceinline__ uint2 pack_box(int4 b) {
  return make_uint2((unsigned)b.x | ((unsigned)b.y << 16), (unsigned)b.z | ((unsigned)b.w << 16));
}

// Cells of 8 x 4 pixels: a box of the usual few pixels meets about two, and one warp owns a tile.
// The limit per surfel bounds the list by the workspace whatever the boxes are.
// The cells a box is listed in: the finest level on which it meets at most g.most of them.
struct SurfelCellRange {
  int i0, i1, j0, j1, base, nx, level;
  // the range as one number (at most 24 cells across; an extent of the last level's few cells)
  __device__ __forceinline__ unsigned long long key() const {
    return (unsigned long long)(unsigned)(base + j0 * nx + i0) << 10 | (unsigned)((i1 - i0) << 5 | (j1 - j0));
  }
};
__device__ __forceinline__ SurfelCellRange surfel_cells(const SurfelGrid& g, uint2 box) {
  const int x0 = box.x & 0xffff, y0 = box.x >> 16, x1 = x0 + (int)(box.y & 0xffff) - 1, y1 = y0 + (int)(box.y >> 16) - 1;
  SurfelCellRange r;
  int l = 0;
  for (;; ++l) {
    r.i0 = x0 >> (3 + l), r.i1 = x1 >> (3 + l), r.j0 = y0 >> (2 + l), r.j1 = y1 >> (2 + l);
    if (l == g.levels - 1 || (r.i1 - r.i0 + 1) * (r.j1 - r.j0 + 1) <= g.most) break;
  }
  r.base = g.first[l];
  r.nx = g.nx[l];
  r.level = l;
  return r;
}

// ---- heavy tiles -----------------------------------------------------------------------------
// A warp owns a tile and goes over its list alone, 0.05 (surfels of a pixel) to 0.4 us (of a whole tile) per
// entry, so a tile with a list far above the average holds up the pass: 1.2 M surfels of a pixel projected
// to one point of a 640 x 480 view took 64.7 ms that way, 0.20 ms with the list shared out (two passes of
// global atomics over the surfels' pixels, before the tiles: 0.49 ms).  A tile is heavy when its list has
// more than 1.5 times a warp's share of all tiles' entries (at most 2/3 of the warps can then own one),
// and kHeavyMin entries.  Its list is cut into units of a 16th of the share, kHeavyUnit at least, so there are
// at most about 16 units per warp.  Times (us) with the line at 1, 1.5, 2 and 3 shares: 1080p surfels of 1.2 M
// in two scenes 267, 256, 259, 282 and 252, 247, 252, 252; 300,000 surfels of 30 pixels in the middle tenth of
// 1080p 9540, 10100, 11200, 12700.  kHeavyMin 64, 96, 128: 70,000 surfels over 128 x 96 57, 58, 58; 160,000
// over 300 x 200 72, 65, 81.  The second pass costs about 13 us, so the heavy tiles are shared out only when
// the longest list has more than 3 shares and kHeavyTrigger entries: else each is left to its warp
// (1992 x 195, 25,000 surfels, longest list 150: 51 us instead of 68; 1080p, longest 2.2 shares: 236 instead
// of 247; but 1080p, longest 3.4 shares: 294 instead of 257, longest 1478 entries, 21 shares: 202 instead of
// 102).
constexpr unsigned kHeavyMin = 96, kHeavyUnit = 32, kHeavyTrigger = 288;
constexpr unsigned kHeavyFlag = 1u << 31;  // of a level-0 cell's count (at most 2^28): its tile is heavy

struct SurfelHeader {  // all zero before k_surfel_count
  unsigned long long heavy;  // their units << 32 | heavy tiles
  unsigned long long work;   // entries of all tiles' lists together
  unsigned listed;           // entries of the list
  unsigned used;             // of them, those given to cells
  unsigned longest;          // entries of the longest list of a heavy tile
  unsigned pad;
};

// A heavy tile, from the end of the workspace backwards, as far as the list leaves room (a tile without
// room is not heavy).  Its nearest depths (as bits) and sums are gathered in the G-buffer's own pixels.
struct SurfelHeavy {
  float w[32];            // per pixel: the number of blended surfels
  unsigned first, units;  // its first unit of all heavy tiles' (ascending), their number
  unsigned tile, entries;
  unsigned done, pad[3];  // units whose surfels are in the sums
};

struct HeavyRule {
  unsigned limit, unit;  // a tile with more than `limit` entries is heavy; entries per unit
  unsigned trigger;      // the heavy tiles are shared out when one has more entries than this
};
__device__ __forceinline__ HeavyRule heavy_rule(const SurfelHeader* h, unsigned warps) {
  const unsigned share = (unsigned)fminf(__fdividef((float)__ldcg(&h->work), (float)warps), 268435456.0f);
  return HeavyRule{max(kHeavyMin, share + share / 2), max(kHeavyUnit, (share / 16 + 31) & ~31u), max(kHeavyTrigger, 3 * share)};
}
__device__ __forceinline__ bool heavy_shared(const SurfelHeader* h, unsigned warps) {
  const unsigned longest = __ldcg(&h->longest);
  return longest > kHeavyTrigger && longest > heavy_rule(h, warps).trigger;
}
__device__ __forceinline__ SurfelHeavy* heavy_at(char* end, unsigned slot) { return (SurfelHeavy*)end - (slot + 1); }
__device__ __forceinline__ unsigned heavy_room(const SurfelHeader* h, const unsigned* list, const char* end) {
  return (unsigned)min((size_t)(end - (const char*)(list + __ldcg(&h->listed))) / sizeof(SurfelHeavy), (size_t)(1u << 30));
}

// HEAVY: whether a tile can be heavy, here and below: the host's rule is more than kHeavyCloud surfels (a
// tile of 100 surfels of 3 pixels takes 57 us alone, 68 shared out).
constexpr int kHeavyCloud = 256;
template <bool HEAVY>
__global__ void __launch_bounds__(256) k_surfel_count(const float4* __restrict__ rec, int N, const SurfelCam cam,
                                                      const __grid_constant__ SurfelGrid g, uint2* __restrict__ boxes,
                                                      unsigned* __restrict__ counts, SurfelHeader* __restrict__ head) {
  __shared__ unsigned s_tiles[8], s_cells[8];
  griddep_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  uint2 box = make_uint2(0, 0);
  if (i < N) {
    const float4 r0 = __ldg(rec + 4 * (size_t)i), r1 = __ldg(rec + 4 * (size_t)i + 1), r2 = __ldg(rec + 4 * (size_t)i + 2);
    SurfelFrame s;
    float c[3];
    if (surfel_frame(r0, r1, r2, cam, s, c)) {
      const int4 b = surfel_box(s, c, r0.w, r1.w, cam);
      if (b.z > 0) box = pack_box(b);
    }
    boxes[i] = box;
  }
  unsigned tiles = 0, cells = 0;
  const unsigned drawn = __ballot_sync(0xffffffffu, box.y != 0u);
  if (box.y != 0u) {
    const SurfelCellRange r = surfel_cells(g, box);
    // surfels of a warp that all meet the same cells are counted together
    int same;
    __match_all_sync(drawn, r.key(), &same);
    const unsigned by = same ? __popc(drawn) : 1u;
    if (!same || (threadIdx.x & 31) == __ffs(drawn) - 1)
      for (int y = r.j0; y <= r.j1; ++y)
        for (int x = r.i0; x <= r.i1; ++x) atomicAdd(counts + g.at(r.base + y * r.nx + x), by);
    cells = (r.i1 - r.i0 + 1) * (r.j1 - r.j0 + 1);
    tiles = (min((r.i1 + 1) << r.level, g.nx[0]) - (r.i0 << r.level)) *
            (min((r.j1 + 1) << r.level, (cam.H + kTileH - 1) / kTileH) - (r.j0 << r.level));
  }
  if (!HEAVY) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  tiles = __reduce_add_sync(0xffffffffu, tiles);  // at most 2^25 each
  cells = __reduce_add_sync(0xffffffffu, cells);
  if (lane == 0) s_tiles[warp] = tiles, s_cells[warp] = cells;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    unsigned k = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += s_tiles[w], k += s_cells[w];
    atomicAdd(&head->work, t);
    atomicAdd(&head->listed, k);
  }
}

__device__ __forceinline__ float4* surfel_a(const GbufDev& out, int x, int y) {
  return (float4*)(const_cast<char*>(out.rt[0]) + (size_t)y * out.pitch[0]) + x;
}
__device__ __forceinline__ float4* surfel_n(const GbufDev& out, int x, int y) {
  return (float4*)(const_cast<char*>(out.rt[1]) + (size_t)y * out.pitch[1]) + x;
}
__device__ __forceinline__ float* surfel_depth(const GbufDev& out, int x, int y) {
  return (float*)(const_cast<char*>(out.rt[3]) + (size_t)y * out.pitch[3]) + x;
}

// Whether tile k is heavy, and its entry if so.
__device__ __forceinline__ void surfel_weigh(int k, unsigned* __restrict__ counts, SurfelHeader* __restrict__ head,
                                             const SurfelGrid& g, const unsigned* list, char* end, unsigned warps,
                                             const GbufDev& out) {
  const int y = k / g.nx[0], x = k - y * g.nx[0];
  unsigned entries = __ldcg(counts + g.at(k));  // on all levels; only this thread sets the flag of this cell
  const unsigned own = entries;
#pragma unroll
  for (int l = 1; l < kSurfelLevels; ++l)
    if (l < g.levels) entries += __ldcg(counts + g.at(g.first[l] + (y >> l) * g.nx[l] + (x >> l)));
  const HeavyRule rule = heavy_rule(head, warps);
  if (entries <= rule.limit) return;
  const unsigned units = (entries + rule.unit - 1) / rule.unit;
  const unsigned long long old = atomicAdd(&head->heavy, ((unsigned long long)units << 32) | 1ull);
  const unsigned slot = (unsigned)old;
  if (slot >= heavy_room(head, list, end)) return;
  atomicMax(&head->longest, entries);
  SurfelHeavy* h = heavy_at(end, slot);
  for (int q = 0; q < 32; ++q) {
    const int px = x * kTileW + (q & 7), py = y * kTileH + (q >> 3);
    h->w[q] = 0.0f;
    if (px >= out.W || py >= out.H) continue;
    *surfel_a(out, px, py) = *surfel_n(out, px, py) = make_float4(0, 0, 0, 0);
    *(unsigned*)surfel_depth(out, px, py) = 0xffffffffu;
  }
  h->first = (unsigned)(old >> 32);
  h->units = units;
  h->tile = k;
  h->entries = entries;
  h->done = 0;
  counts[g.at(k)] = own | kHeavyFlag;
}

// cursor[k] = the first list entry of cell k.  The blocks after those of the cells weigh the tiles.
template <bool HEAVY>
__global__ void __launch_bounds__(256) k_surfel_alloc(unsigned* __restrict__ counts, int cells,
                                                      unsigned* __restrict__ cursor, SurfelHeader* __restrict__ head,
                                                      const __grid_constant__ SurfelGrid g, const unsigned* list, char* end,
                                                      unsigned warps, GbufDev out) {
  __shared__ unsigned s_warp[8];
  __shared__ unsigned s_base;
  griddep_wait();
  griddep_launch_dependents();
  int k = blockIdx.x * 256 + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (HEAVY) {
    const int blocks = (cells + 255) / 256;
    if (blockIdx.x >= blocks) {
      k -= blocks * 256;
      if (k < g.first[1]) surfel_weigh(k, counts, head, g, list, end, warps, out);
      return;
    }
  }
  const unsigned n = k < cells ? __ldcg(counts + g.at(k)) & ~kHeavyFlag : 0u;
  unsigned incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned sum = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const unsigned v = s_warp[w];
      s_warp[w] = sum;
      sum += v;
    }
    s_base = atomicAdd(&head->used, sum);
  }
  __syncthreads();
  if (k < cells) cursor[g.at(k)] = s_base + s_warp[warp] + incl - n;
}

// Afterwards cursor[k] is the end of cell k's range.
__global__ void __launch_bounds__(256) k_surfel_fill(const uint2* __restrict__ boxes, int N,
                                                     const __grid_constant__ SurfelGrid g, unsigned* __restrict__ cursor,
                                                     unsigned* __restrict__ list) {
  griddep_wait();
  griddep_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const uint2 box = i < N ? __ldcg(boxes + i) : make_uint2(0, 0);
  const unsigned drawn = __ballot_sync(0xffffffffu, box.y != 0u);
  if (box.y == 0u) return;
  const SurfelCellRange r = surfel_cells(g, box);
  const int nx = r.i1 - r.i0 + 1, n = nx * (r.j1 - r.j0 + 1);
  int cx = r.i0, cell = r.base + r.j0 * r.nx + r.i0;
  int same;
  __match_all_sync(drawn, r.key(), &same);
  if (same && __popc(drawn) > 1) {  // together, as they were counted
    const int lane = threadIdx.x & 31, leader = __ffs(drawn) - 1, rank = __popc(drawn & ((1u << lane) - 1u));
    for (int q = 0; q < n; ++q) {
      unsigned at = 0;
      if (lane == leader) at = atomicAdd(cursor + g.at(cell), (unsigned)__popc(drawn));
      list[__shfl_sync(drawn, at, leader) + rank] = (unsigned)i;
      ++cell;
      if (++cx > r.i1) cx = r.i0, cell += r.nx - nx;
    }
    return;
  }
  // four at a time, so that four atomics are under way before the first result is used
  for (int q = 0; q < n; q += 4) {
    unsigned at[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (q + u < n) at[u] = atomicAdd(cursor + g.at(cell), 1u);
      ++cell;
      if (++cx > r.i1) cx = r.i0, cell += r.nx - nx;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (q + u < n) list[at[u]] = (unsigned)i;
  }
}

constexpr int kSurfelTileWarps = 4;  // a block covers 4 x 1 tiles: 32 x 4 pixels

// A warp's shared memory: up to 32 surfels of its tile.  Row strides of 80 and 48 bytes keep the
// 16-byte reads of eight different rows free of bank conflicts, 33 words the per-pixel depths.
struct SurfelWarp {
  float frame[32][20];  // SurfelFrame: n, t, b, (cb, nc), then the packed items, a row per surfel with any
  float mat[32][12];    // world normal and metal, albedo and rough
  float depth[32][33];  // [pixel][surfel]: depth of the hits
  unsigned hits[32];    // per pixel: the surfels that cover it
  unsigned nearest[32];  // per pixel: bits of the smallest depth so far
  float2 ray[32];        // per pixel: (ux, uy)
};

// A pixel's nearest depth so far and the window's end below it, the farthest blended depth, the sums.
struct SurfelPixel {
  float dmin, lim, far, w;
  float a0, a1, a2, a3, n0, n1, n2, n3;
  bool redo;
  __device__ __forceinline__ void clear() { w = a0 = a1 = a2 = a3 = n0 = n1 = n2 = n3 = 0.0f; }
};

// kOnce blends as it goes: a surfel behind the window of the nearest so far stays out, since that window
// only moves nearer.  When a nearer surfel moves it past some, but not all, of the blended ones, the
// tile is gone over again with the window known (`redo`).  kNearest only finds the nearest depths (in
// st.nearest), kBlend only blends, in a window that is known.
enum SurfelPass { kOnce, kNearest, kBlend };

// A surfel at depth d, nearer than all before, moves the window (kOnce).
__device__ __forceinline__ void surfel_nearer(SurfelPixel& p, float d, float f) {
  const float end = __fmul_rn(d, f);
  if (p.far > end) {
    p.redo = p.redo || p.dmin <= end;  // some blended surfels stay in the window, some do not
    p.clear();
    p.far = 0.0f;
  }
  p.dmin = d;
  p.lim = end;
}

template <int PASS>
__device__ __forceinline__ void surfel_add(SurfelPixel& p, const float* mat, float d) {
  if (PASS == kOnce) p.far = fmaxf(p.far, d);
  const float4 nw = *(const float4*)mat, al = *(const float4*)(mat + 4);
  p.a0 += al.x, p.a1 += al.y, p.a2 += al.z, p.a3 += nw.w;
  p.n0 += nw.x, p.n1 += nw.y, p.n2 += nw.z, p.n3 += al.w;
  p.w += 1.0f;
}

// Up to 32 surfels (idx, where `valid`) against the tile whose first pixel is (tx, ty), a pixel per lane.
template <int PASS>
__device__ __forceinline__ void surfel_batch(SurfelWarp& st, const float4* __restrict__ rec, const uint2* __restrict__ boxes,
                                             const SurfelCam& cam, unsigned idx, bool valid, int tx, int ty, int lane,
                                             SurfelPixel& p) {
  // a lane per surfel: its box clipped to the tile, its frame
  int cx = 0, cy = 0, cw = 0, ch = 0;
  if (valid) {
    const uint2 box = __ldcg(boxes + idx);
    cx = max((int)(box.x & 0xffffu) - tx, 0), cy = max((int)(box.x >> 16) - ty, 0);
    cw = min((int)((box.x & 0xffffu) + (box.y & 0xffffu)) - tx, kTileW) - cx;
    ch = min((int)((box.x >> 16) + (box.y >> 16)) - ty, kTileH) - cy;
  }
  const int mine = cw > 0 && ch > 0 ? cw * ch : 0;
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const unsigned live = __ballot_sync(0xffffffffu, mine > 0);
  if (live == 0u) return;
  const int total = __shfl_sync(0xffffffffu, incl, 31), excl = incl - mine;
  if (mine > 0) {
    const float4 r0 = __ldg(rec + 4 * (size_t)idx), r1 = __ldg(rec + 4 * (size_t)idx + 1);
    const float4 r2 = __ldg(rec + 4 * (size_t)idx + 2);
    SurfelFrame s;
    float c[3];
    surfel_frame(r0, r1, r2, cam, s, c);
    // the surfels with items, in consecutive rows; packed: clipped origin, width, its reciprocal
    // (exact quotients of items below 32 by widths up to 8) and the first item (below 1024)
    const int row = __popc(live & ((1u << lane) - 1u));
    const unsigned items = (unsigned)cx | ((unsigned)cy << 3) | ((unsigned)cw << 5) |
                           (((255u + cw) / (unsigned)cw) << 9) | ((unsigned)excl << 18);
    float4* f = (float4*)st.frame[row];
    // and the box as a mask of the tile's pixels
    const unsigned mask = (((1u << cw) - 1u) << cx) * 0x01010101u & (0xffffffffu >> (32 - kTileW * ch)) << (kTileW * cy);
    f[0] = s.n, f[1] = s.t, f[2] = s.b;
    f[3] = make_float4(s.cb, s.nc, __uint_as_float(items), __uint_as_float(mask));
    if (PASS != kNearest) {
      const float4 r3 = __ldg(rec + 4 * (size_t)idx + 3);
      const float rw = rsqrtf(fmaf(r1.x, r1.x, fmaf(r1.y, r1.y, r1.z * r1.z)));
      float4* m = (float4*)st.mat[row];
      m[0] = make_float4(r1.x * rw, r1.y * rw, r1.z * rw, r2.w);
      m[1] = r3;
    }
  }
  if (2 * total > 32 * __popc(live)) {
    // boxes that cover most of the tile: every lane tests its own pixel, one surfel at a time
    __syncwarp();
    const float2 ray = st.ray[lane];
    for (int k = 0; k < __popc(live); ++k) {
      const float4* f = (const float4*)st.frame[k];
      const float4 q = f[3];
      SurfelFrame s;
      s.n = f[0], s.t = f[1], s.b = f[2];
      s.cb = q.x, s.nc = q.y;
      const float d = surfel_hit(s, ray.x, ray.y);
      if (d > 0.0f && (__float_as_uint(q.w) >> lane & 1u)) {
        if (PASS != kBlend && d < p.dmin) {
          if (PASS == kOnce) surfel_nearer(p, d, cam.f);
          p.dmin = d;
        }
        if (PASS != kNearest && d <= p.lim) surfel_add<PASS>(p, st.mat[k], d);
      }
    }
    if (PASS != kBlend) st.nearest[lane] = min(st.nearest[lane], __float_as_uint(p.dmin));
    __syncwarp();
    return;
  }
  if (PASS != kNearest) st.hits[lane] = 0u;
  __syncwarp();
  // a lane per (surfel, box pixel)
  int begun = -1;  // rows whose items begin before j0, less one
  for (int j0 = 0; j0 < total; j0 += 32) {
    const int j = j0 + lane;
    const unsigned at = (unsigned)(excl - j0);
    const unsigned begins = __reduce_or_sync(0xffffffffu, mine > 0 && at < 32u ? 1u << at : 0u);
    const int k = begun + __popc(begins & ((2u << lane) - 1u));  // the row whose items hold j
    begun += __popc(begins);
    if (j < total) {
      const float4* f = (const float4*)st.frame[k];
      const float4 q = f[3];
      const unsigned m = __float_as_uint(q.z);
      const int local = j - (int)(m >> 18);
      const int ly = (local * (int)((m >> 9) & 511u)) >> 8, lx = local - ly * (int)((m >> 5) & 15u);
      const int px = ((int)((m >> 3) & 3u) + ly) * kTileW + (int)(m & 7u) + lx;
      const float2 ray = st.ray[px];
      SurfelFrame s;
      s.n = f[0], s.t = f[1], s.b = f[2];
      s.cb = q.x, s.nc = q.y;
      const float sd = surfel_hit(s, ray.x, ray.y);
      if (sd > 0.0f) {
        if (PASS != kBlend) atomicMin(&st.nearest[px], __float_as_uint(sd));  // positive floats order as their bits
        if (PASS != kNearest) {
          atomicOr(&st.hits[px], 1u << k);
          st.depth[px][k] = sd;
        }
      }
    }
  }
  __syncwarp();
  if (PASS == kNearest) return;
  // a lane per pixel
  unsigned hits = st.hits[lane];
  if (hits) {
    if (PASS == kOnce) {
      const float sd = __uint_as_float(st.nearest[lane]);
      if (sd < p.dmin) surfel_nearer(p, sd, cam.f);
    }
    do {
      const int k = __ffs(hits) - 1;
      hits &= hits - 1;
      const float d = st.depth[lane][k];
      if (d <= p.lim) surfel_add<PASS>(p, st.mat[k], d);
    } while (hits);
  }
  __syncwarp();
}

// A tile and its list: lane l holds the length and the end of the list of the tile's cell on level l.
struct SurfelTile {
  int tx, ty;
  unsigned n, end;
};

__device__ __forceinline__ SurfelTile surfel_tile(const SurfelGrid& g, int tx, int ty, int lane,
                                                  const unsigned* __restrict__ counts,
                                                  const unsigned* __restrict__ cursor) {
  SurfelTile t = {tx, ty, 0, 0};
  if (lane < g.levels) {
    const int k = g.first[lane] + (ty >> (2 + lane)) * g.nx[lane] + (tx >> (3 + lane));
    t.n = __ldcg(counts + g.at(k));
    t.end = __ldcg(cursor + g.at(k));
  }
  return t;
}

__device__ __forceinline__ float2 surfel_ray(const SurfelCam& cam, int x, int y) {
  return make_float2(__fdiv_rn(__fsub_rn(__fdiv_rn(__fadd_rn((float)x, 0.5f), cam.hw), 1.0f), cam.kx),
                     __fdiv_rn(__fsub_rn(1.0f, __fdiv_rn(__fadd_rn((float)y, 0.5f), cam.hh)), cam.ky));
}

// Entries from .. to - 1 of the tile's lists, one level after the other.
template <int PASS>
__device__ __forceinline__ void surfel_walk(SurfelWarp& st, const float4* __restrict__ rec, const uint2* __restrict__ boxes,
                                            const SurfelCam& cam, const SurfelGrid& g, const SurfelTile& t,
                                            const unsigned* __restrict__ list, unsigned from, unsigned to, int lane,
                                            SurfelPixel& p) {
  unsigned base = 0;
  for (int l = 0; l < g.levels; ++l) {
    unsigned n = __shfl_sync(0xffffffffu, t.n, l), first = __shfl_sync(0xffffffffu, t.end, l) - n;
    if (PASS != kOnce) {  // the level's share of from .. to - 1
      const unsigned a = min(max(from, base) - base, n), b = min(max(to, base) - base, n);
      base += n;
      first += a;
      n = b - a;
    }
    unsigned next = 0;
    if (lane < n) next = __ldcg(list + first + lane);
    for (unsigned q0 = 0; q0 < n; q0 += 32) {
      const unsigned idx = next;
      if (q0 + 32 + lane < n) next = __ldcg(list + first + q0 + 32 + lane);
      surfel_batch<PASS>(st, rec, boxes, cam, idx, q0 + lane < n, t.tx, t.ty, lane, p);
    }
  }
}

// The means of a pixel (w surfels, the sums a and n) as the FP32 G-buffer.
__device__ __forceinline__ void surfel_store(const GbufDev& out, float* __restrict__ weight, long long weight_pitch, int x,
                                             int y, float w, float4 a, float4 n, float depth) {
  float4 *rt0 = surfel_a(out, x, y), *rt1 = surfel_n(out, x, y);
  float* dep = surfel_depth(out, x, y);
  if (weight) ((float*)((char*)weight + (size_t)y * weight_pitch))[x] = w;
  if (w == 0.0f) {
    *rt0 = make_float4(0, 0, 0, 0);
    *rt1 = make_float4(0, 0, 0, 0);
    *dep = __int_as_float(0x7f800000);
    return;
  }
  const float iw = 1.0f / w;
  const float nn = fmaf(n.x, n.x, fmaf(n.y, n.y, n.z * n.z));
  const float rn = nn > 0.0f ? rsqrtf(nn) : 0.0f;
  *rt0 = make_float4(a.x * iw, a.y * iw, a.z * iw, a.w * iw);
  *rt1 = make_float4(n.x * rn, n.y * rn, n.z * rn, n.w * iw);
  *dep = depth;
}

struct SurfelArgs {
  const float4* rec;
  const uint2* boxes;
  const unsigned *counts, *cursor, *list;
  const SurfelHeader* head;
  char* end;       // of the workspace
  unsigned warps;  // that share the work (heavy_rule)
};

// The heavy tiles' units in runs of equal length, two per warp (one unit at least): runs warp, warp + warps, ...
template <int PASS>
__device__ __forceinline__ void surfel_runs(SurfelWarp& st, const SurfelArgs& s, const SurfelCam& cam, const SurfelGrid& g,
                                            unsigned warp, unsigned warps, int lane, const GbufDev& out,
                                            float* __restrict__ weight, long long weight_pitch) {
  if (!heavy_shared(s.head, s.warps)) return;
  const unsigned long long heavy = __ldcg(&s.head->heavy);
  const unsigned total = (unsigned)(heavy >> 32), slots = min((unsigned)heavy, heavy_room(s.head, s.list, s.end));
  const unsigned unit = heavy_rule(s.head, s.warps).unit, run = (total + 2 * warps - 1) / (2 * warps);
  for (unsigned u0 = warp * run; u0 < total; u0 += warps * run) {
    const unsigned u1 = min(total, u0 + run);
    // the last tile whose first unit is not above u0 (they ascend), 32 candidates at a time
    unsigned slot = 0, hi = slots;
    while (hi - slot > 1) {
      const unsigned step = (hi - slot + 31) / 32, at = slot + lane * step;
      const unsigned below = __ballot_sync(0xffffffffu, at < hi && __ldcg(&heavy_at(s.end, at)->first) <= u0);
      slot += (31 - __clz(below)) * step;
      hi = min(hi, slot + step);
    }
    for (unsigned u = u0; u < u1 && slot < slots; ++slot) {
      SurfelHeavy* h = heavy_at(s.end, slot);
      const unsigned first = __ldcg(&h->first), units = __ldcg(&h->units), tile = __ldcg(&h->tile);
      const unsigned k0 = u - first, k1 = min(units, u1 - first);
      if (k0 >= units) break;  // units of tiles without room follow those of the others
      u = first + k1;
      const int tx = (int)(tile % g.nx[0]) * kTileW, ty = (int)(tile / g.nx[0]) * kTileH;
      const int x = tx + (lane & 7), y = ty + (lane >> 3);
      SurfelTile t = surfel_tile(g, tx, ty, lane, s.counts, s.cursor);
      t.n &= ~kHeavyFlag;
      st.nearest[lane] = 0xffffffffu;
      st.ray[lane] = surfel_ray(cam, x, y);
      SurfelPixel p;
      p.clear();
      p.dmin = __int_as_float(0x7f800000);
      const bool inside = x < cam.W && y < cam.H;
      if (PASS == kBlend) {
        const unsigned bits = inside ? __ldcg((const unsigned*)surfel_depth(out, x, y)) : 0xffffffffu;
        if (bits != 0xffffffffu) p.dmin = __uint_as_float(bits);
        p.lim = __fmul_rn(p.dmin, cam.f);
      }
      __syncwarp();
      surfel_walk<PASS>(st, s.rec, s.boxes, cam, g, t, s.list, k0 * unit, min(k1 * unit, __ldcg(&h->entries)), lane, p);
      __syncwarp();
      if (PASS == kNearest) {
        if (st.nearest[lane] != 0xffffffffu) atomicMin((unsigned*)surfel_depth(out, x, y), st.nearest[lane]);
      } else {
        if (p.w > 0.0f) {
          atomicAdd(surfel_a(out, x, y), make_float4(p.a0, p.a1, p.a2, p.a3));
          atomicAdd(surfel_n(out, x, y), make_float4(p.n0, p.n1, p.n2, p.n3));
          atomicAdd(h->w + lane, p.w);
        }
        __threadfence();
        __syncwarp();
        unsigned done = 0;
        if (lane == 0) done = atomicAdd(&h->done, k1 - k0);
        done = __shfl_sync(0xffffffffu, done, 0);
        if (done + (k1 - k0) == units) {  // the tile's last units
          __threadfence();
          if (inside)
            surfel_store(out, weight, weight_pitch, x, y, __ldcg(h->w + lane), __ldcg(surfel_a(out, x, y)),
                         __ldcg(surfel_n(out, x, y)), p.dmin);
        }
      }
      __syncwarp();
    }
  }
}

// Bound by issue and latency at 6 blocks per SM (35 KB of shared memory).  A surfel's hits are found a lane per
// (surfel, pixel) unless the batch's boxes cover half of the tile's pixels on average; then a lane per pixel
// (300,000 surfels of 30 pixels over 1080p 4080 -> 3060 us; with a line at a third of the pixels the 1.2 M
// surfels at 1080p take 271 us instead of 268).  A lane per pixel for every surfel took 563 us there, blocks
// of 1, 2, 4 and 5 warps 307, 294, 279 and 300 us, two passes of global atomics 627 us.
// The first `heavy_rows` rows of blocks take the heavy tiles' units.
template <bool HEAVY>
__global__ void __launch_bounds__(32 * kSurfelTileWarps)
    k_surfel_tile(const __grid_constant__ SurfelArgs s, const SurfelCam cam, const __grid_constant__ SurfelGrid g,
                  int heavy_rows, GbufDev out, float* __restrict__ weight, long long weight_pitch) {
  __shared__ __align__(16) SurfelWarp s_all[kSurfelTileWarps];
  // k_surfel_alloc, which writes the header, was complete before k_surfel_fill let this kernel begin
  if (HEAVY && blockIdx.y < heavy_rows && !heavy_shared(s.head, s.warps)) return;
  griddep_wait();
  if (HEAVY) griddep_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  SurfelWarp& st = s_all[warp];
  if (HEAVY && blockIdx.y < heavy_rows) {
    surfel_runs<kNearest>(st, s, cam, g, (blockIdx.y * gridDim.x + blockIdx.x) * kSurfelTileWarps + warp,
                           heavy_rows * gridDim.x * kSurfelTileWarps, lane, out, weight, weight_pitch);
    return;
  }
  const int tx = (blockIdx.x * kSurfelTileWarps + warp) * kTileW, ty = (blockIdx.y - heavy_rows) * kTileH;
  if (tx >= cam.W) return;  // warp-uniform, no block barrier below
  const int x = tx + (lane & 7), y = ty + (lane >> 3);
  SurfelTile t = surfel_tile(g, tx, ty, lane, s.counts, s.cursor);
  if (HEAVY && (__shfl_sync(0xffffffffu, t.n, 0) & kHeavyFlag)) {
    if (heavy_shared(s.head, s.warps)) return;
    t.n &= ~kHeavyFlag;
  }
  st.nearest[lane] = 0xffffffffu;
  st.ray[lane] = surfel_ray(cam, x, y);
  SurfelPixel p;
  p.clear();
  p.dmin = p.lim = __int_as_float(0x7f800000);
  p.far = 0.0f;
  p.redo = false;
  for (int pass = 0; pass < 2; ++pass) {
    surfel_walk<kOnce>(st, s.rec, s.boxes, cam, g, t, s.list, 0, 0, lane, p);
    if (!__any_sync(0xffffffffu, p.redo)) break;
    p.clear();
    p.redo = false;
  }
  if (x < cam.W && y < cam.H)
    surfel_store(out, weight, weight_pitch, x, y, p.w, make_float4(p.a0, p.a1, p.a2, p.a3),
                 make_float4(p.n0, p.n1, p.n2, p.n3), p.dmin);
}

__global__ void __launch_bounds__(32 * kSurfelTileWarps, 6)
    k_surfel_heavy(const __grid_constant__ SurfelArgs s, const SurfelCam cam, const __grid_constant__ SurfelGrid g,
                   GbufDev out, float* __restrict__ weight, long long weight_pitch) {
  __shared__ __align__(16) SurfelWarp s_all[kSurfelTileWarps];
  // the header, as in k_surfel_tile; one block waits, so that this kernel is not complete before the tiles
  if (!heavy_shared(s.head, s.warps) && blockIdx.x > 0) return;
  griddep_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  surfel_runs<kBlend>(s_all[warp], s, cam, g, blockIdx.x * kSurfelTileWarps + warp, gridDim.x * kSurfelTileWarps, lane, out,
                      weight, weight_pitch);
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct SurfelLayout {
  size_t head, counters, counts, cursor, boxes, list, bytes;
  SurfelGrid grid;
};

// The workspace: the header, cell counts and cursors, 8 bytes of box and kSurfelCells
// list entries per surfel; heavy tiles (160 bytes each) from its end down to the entries that are used.  `bytes` is the size callers have always been told, 40 B per pixel, 4 B
// per column and row, 104 B per surfel and 8 B per 1024 of them: the list takes 96 B per surfel, the
// cells less than 4 B per pixel plus 1 KB.
static SurfelLayout surfel_layout(long long N, int W, int H) {
  SurfelLayout l;
  const size_t px = (size_t)W * H;
  l.bytes = align256(4 * px) + align256(36 * px) + align256(4 * (size_t)W) + align256(4 * (size_t)H) +
            align256(96 * (size_t)N) + align256(8 * (size_t)(N + 1)) + align256(8 * (size_t)((N + 1023) / 1024 + 1));
  SurfelGrid& g = l.grid;
  // list positions fit 32 bits
  g.most = (int)std::min<long long>(kSurfelCells, N > 0 ? 0xffffffffLL / N : kSurfelCells);
  g.first[0] = 0;
  for (g.levels = 0; g.levels < kSurfelLevels;) {
    const int k = g.levels++;
    g.nx[k] = (W + (kTileW << k) - 1) / (kTileW << k);
    const int ny = (H + (kTileH << k) - 1) / (kTileH << k);
    g.first[k + 1] = g.first[k] + g.nx[k] * ny;
    if (g.nx[k] * ny <= 4) break;
  }
  const size_t cells = (size_t)g.first[g.levels];
  l.head = 0;
  l.counts = sizeof(SurfelHeader);  // reset together
  g.stride = 1;
  const size_t room = sizeof(SurfelHeavy) * (size_t)g.first[1] + 1024;
  // few cells: their counters apart, up to kSurfelSpread words, as far as the 40 B per pixel hold both arrays
  // and the heavy tiles
  while (g.stride < 32 && 2 * cells * g.stride <= kSurfelSpread && 2 * 8 * cells * g.stride + room <= 40 * px) g.stride *= 2;
  l.counters = cells * g.stride;
  l.cursor = align256(l.counts + 4 * l.counters);
  l.boxes = l.cursor + align256(4 * l.counters);
  l.list = l.boxes + align256(8 * (size_t)N);
  return l;
}

}  // namespace epbr

using namespace epbr;

extern "C" epbr_status epbr_surfel_workspace_size(int32_t num_surfels, int32_t width, int32_t height, size_t* bytes) {
  if (!bytes || num_surfels < 0 || num_surfels > (1 << 28) || width < 1 || height < 1 || width > (1 << 15) ||
      height > (1 << 15))
    return fail(EPBR_ERR_INVALID_ARG, "surfels: bytes NULL, num_surfels outside [0, 2^28] or size outside [1, 32768]");
  *bytes = surfel_layout(num_surfels, width, height).bytes;
  return ok();
}

extern "C" epbr_status epbr_surfel_gbuffer(const epbr_surfels* surfels, const epbr_camera* camera, float near_depth,
                                           float depth_tolerance, const epbr_gbuffer* out, float* weight,
                                           int64_t weight_pitch, void* workspace, size_t workspace_bytes,
                                           void* stream) {
  if (!surfels || !out) return fail(EPBR_ERR_INVALID_ARG, "surfels: surfels or gbuffer is NULL");
  epbr_status st = validate_camera(camera, out);
  if (st) return st;
  if (out->format != EPBR_GBUFFER_FP32) return fail(EPBR_ERR_INVALID_ARG, "surfels: the output G-buffer must be FP32");
  if ((st = validate_gbuffer(out, true))) return st;
  const int N = surfels->num_surfels;
  if (N < 0 || N > (1 << 28) || (N > 0 && !surfels->records) || (uintptr_t)surfels->records % 16)
    return fail(EPBR_ERR_INVALID_ARG, "surfels: records NULL, not 16-byte aligned or count outside [0, 2^28]");
  if (!(near_depth > 0.0f) || !std::isfinite(near_depth))
    return fail(EPBR_ERR_INVALID_ARG, "surfels: near must be > 0");
  if (!(depth_tolerance >= 0.0f) || !std::isfinite(depth_tolerance))
    return fail(EPBR_ERR_INVALID_ARG, "surfels: depth tolerance must be finite and >= 0");
  if (weight && (weight_pitch < 4LL * out->width || weight_pitch % 4 || (uintptr_t)weight % 4))
    return fail(EPBR_ERR_INVALID_ARG, "surfels: weight misaligned or pitch too small");
  const int W = out->width, H = out->height;
  const SurfelLayout l = surfel_layout(N, W, H);
  if (!workspace || (uintptr_t)workspace % 256 || workspace_bytes < l.bytes)
    return fail(EPBR_ERR_INVALID_ARG, "surfels: workspace NULL, not 256-byte aligned or below %zu bytes", l.bytes);
  char* ws = (char*)workspace;
  unsigned* counts = (unsigned*)(ws + l.counts);
  unsigned* cursor = (unsigned*)(ws + l.cursor);
  uint2* boxes = (uint2*)(ws + l.boxes);
  unsigned* list = (unsigned*)(ws + l.list);
  SurfelCam sc;
  const CamDev cd = make_cam(*camera);
  for (int k = 0; k < 3; ++k) {
    for (int i = 0; i < 3; ++i) sc.axes[3 * k + i] = cd.r[3 * i + k];  // column k of the rotation
    sc.eye[k] = cd.eye[k];
  }
  const double t = std::tan(0.5 * (double)camera->fov_y);
  sc.ky = (float)(1.0 / t);
  sc.kx = (float)((double)H / ((double)W * t));
  sc.hw = (float)(0.5 * W);
  sc.hh = (float)(0.5 * H);
  sc.near = near_depth;
  sc.f = 1.0f + depth_tolerance;
  sc.W = W;
  sc.H = H;
  cudaStream_t s = (cudaStream_t)stream;
  const SurfelGrid& g = l.grid;
  const int cells = g.first[g.levels];
  if (cudaMemsetAsync(ws + l.head, 0, l.counts + 4 * l.counters, s) != cudaSuccess)
    return fail(EPBR_ERR_CUDA, "surfels: memset failed");
  const GbufDev gd = make_gbuf(*out);
  const float4* rec = (const float4*)surfels->records;
  SurfelHeader* head = (SurfelHeader*)(ws + l.head);
  const bool heavy = N > kHeavyCloud;
  const int heavy_blocks = num_sms() * 6;  // as many as are resident
  const SurfelArgs a = {rec, boxes, counts, cursor, list, head, ws + l.bytes, (unsigned)(heavy_blocks * kSurfelTileWarps)};
  cudaError_t e = cudaSuccess;
  if (N > 0) {
    const dim3 per_surfel((N + 255) / 256), per_cell((cells + 255) / 256 + (heavy ? (g.first[1] + 255) / 256 : 0));
    if (heavy)
      k_surfel_count<true><<<per_surfel, 256, 0, s>>>(rec, N, sc, g, boxes, counts, head);
    else
      k_surfel_count<false><<<per_surfel, 256, 0, s>>>(rec, N, sc, g, boxes, counts, head);
    e = launch_kernel(heavy ? k_surfel_alloc<true> : k_surfel_alloc<false>, per_cell, dim3(256), 0, s, true, counts, cells,
                      cursor, head, g, (const unsigned*)list, a.end, a.warps, gd);
    if (e == cudaSuccess)
      e = launch_kernel(k_surfel_fill, per_surfel, dim3(256), 0, s, true, (const uint2*)boxes, N, g, cursor, list);
  }
  const dim3 blk(32 * kSurfelTileWarps);
  dim3 grd((W + kSurfelTileWarps * kTileW - 1) / (kSurfelTileWarps * kTileW), (H + kTileH - 1) / kTileH);
  const int heavy_rows = heavy ? (heavy_blocks + (int)grd.x - 1) / (int)grd.x : 0;
  grd.y += heavy_rows;
  if (e == cudaSuccess)
    e = launch_kernel(heavy ? k_surfel_tile<true> : k_surfel_tile<false>, grd, blk, 0, s, N > 0, a, sc, g, heavy_rows, gd,
                      weight, (long long)weight_pitch);
  if (e == cudaSuccess && heavy)
    e = launch_kernel(k_surfel_heavy, dim3(heavy_blocks), blk, 0, s, true, a, sc, g, gd, weight, (long long)weight_pitch);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(EPBR_ERR_CUDA, "surfels: %s", cudaGetErrorString(e));
  }
  if ((st = check_launch("surfels"))) return st;
  return ok();
}
