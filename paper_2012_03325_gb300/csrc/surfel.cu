// The G-buffer pass of surfel rendering (Sec. 4.3): oriented elliptical disks splatted into the
// FP32 G-buffer, the surfels within a depth window of the nearest one blended.
//   k_surfel_count  one thread per surfel: view-space frame, the near rule, the pixel box of the
//                   projected ellipse (its image conic's extent, widened by 1/8 pixel), and the
//                   number of surfels per cell of a pyramid of grids, 8 x 4 pixels at level 0,
//                   doubled from level to level; a surfel is listed in the cells its box meets on
//                   the finest level where these are at most 24
//   k_surfel_alloc  every cell's range of the list (ranges in any order: a block sum and one
//                   atomicAdd per 256 cells)
//   k_surfel_fill   the surfels' indices into their cells' ranges
//   k_surfel_tile   one warp per 8 x 4 pixels, a lane per pixel: the surfels listed in the tile's
//                   cells, 32 at a time, their frames computed by one lane each into shared memory,
//                   their box pixels tested a lane per (surfel, pixel); nearest depth, blended sums
//                   and count stay in the pixel's lane, the means are written as the FP32 G-buffer
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

struct SurfelGrid {
  int levels;
  int most;                         // cells a surfel is listed in at most
  int nx[kSurfelLevels];            // cells per row of a level
  int first[kSurfelLevels + 1];     // its first cell
};

// Packed box: x0 | y0 << 16, width | height << 16 (each at most 32768; width 0: not drawn).
__device__ __forceinline__ uint2 pack_box(int4 b) {
  return make_uint2((unsigned)b.x | ((unsigned)b.y << 16), (unsigned)b.z | ((unsigned)b.w << 16));
}

// Cells of 8 x 4 pixels: a box of the usual few pixels meets about two, and one warp owns a tile.
// The limit per surfel bounds the list by the workspace whatever the boxes are.
// The cells a box is listed in: the finest level on which it meets at most g.most of them.
struct SurfelCellRange {
  int i0, i1, j0, j1, base, nx;
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
  return r;
}

__global__ void __launch_bounds__(256) k_surfel_count(const float4* __restrict__ rec, int N, const SurfelCam cam,
                                                      const __grid_constant__ SurfelGrid g, uint2* __restrict__ boxes,
                                                      unsigned* __restrict__ counts) {
  griddep_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float4 r0 = __ldg(rec + 4 * (size_t)i), r1 = __ldg(rec + 4 * (size_t)i + 1), r2 = __ldg(rec + 4 * (size_t)i + 2);
  SurfelFrame s;
  float c[3];
  uint2 box = make_uint2(0, 0);
  if (surfel_frame(r0, r1, r2, cam, s, c)) {
    const int4 b = surfel_box(s, c, r0.w, r1.w, cam);
    if (b.z > 0) {
      box = pack_box(b);
      const SurfelCellRange r = surfel_cells(g, box);
      for (int y = r.j0; y <= r.j1; ++y)
        for (int x = r.i0; x <= r.i1; ++x) atomicAdd(counts + r.base + y * r.nx + x, 1u);
    }
  }
  boxes[i] = box;
}

// cursor[k] = the first list entry of cell k.
__global__ void __launch_bounds__(256) k_surfel_alloc(const unsigned* __restrict__ counts, int cells,
                                                      unsigned* __restrict__ cursor, unsigned* __restrict__ used) {
  __shared__ unsigned s_warp[8];
  __shared__ unsigned s_base;
  griddep_wait();
  griddep_launch_dependents();
  const int k = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned n = k < cells ? __ldcg(counts + k) : 0u;
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
    s_base = atomicAdd(used, sum);
  }
  __syncthreads();
  if (k < cells) cursor[k] = s_base + s_warp[warp] + incl - n;
}

// Afterwards cursor[k] is the end of cell k's range.
__global__ void __launch_bounds__(256) k_surfel_fill(const uint2* __restrict__ boxes, int N,
                                                     const __grid_constant__ SurfelGrid g, unsigned* __restrict__ cursor,
                                                     unsigned* __restrict__ list) {
  griddep_wait();
  griddep_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const uint2 box = __ldcg(boxes + i);
  if ((box.y & 0xffffu) == 0) return;
  const SurfelCellRange r = surfel_cells(g, box);
  // four at a time, so that four atomics are under way before the first result is used
  const int nx = r.i1 - r.i0 + 1, n = nx * (r.j1 - r.j0 + 1);
  int cx = r.i0, cell = r.base + r.j0 * r.nx + r.i0;
  for (int q = 0; q < n; q += 4) {
    unsigned at[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (q + u < n) at[u] = atomicAdd(cursor + cell, 1u);
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

// Replaces two coverage passes of global atomics (an atomicMin, then two float4 and one float atomic
// add per covered pixel, 13.5 M of them in the 1.2 M-surfel 1080p scene), their set-up store, resets
// and resolve: 627 -> 256 us for the whole pass.  Bound by issue and latency at 6 blocks per SM (35 KB of
// shared memory, 79 registers; ncu before the surfels with items took consecutive rows, an item's
// surfel and ray then coming from nine shuffles, 269 us: 124 M warp instructions, 0.54 per scheduler
// and cycle; long scoreboard 2.4, fixed latency 2.1, short scoreboard 1.9 per issue).  Blocks of 1, 2, 4, 5
// warps then
// measured 307, 294, 279, 300 us, and a lane per pixel testing every listed surfel 563 us (tiles with
// 2000 small surfels then take the launch's tail).
__global__ void __launch_bounds__(32 * kSurfelTileWarps)
    k_surfel_tile(const float4* __restrict__ rec, const uint2* __restrict__ boxes, const SurfelCam cam,
                  const __grid_constant__ SurfelGrid g, const unsigned* __restrict__ counts,
                  const unsigned* __restrict__ cursor, const unsigned* __restrict__ list, GbufDev out,
                  float* __restrict__ weight, long long weight_pitch) {
  __shared__ __align__(16) SurfelWarp s_all[kSurfelTileWarps];
  griddep_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tx = (blockIdx.x * kSurfelTileWarps + warp) * kTileW, ty = blockIdx.y * kTileH;
  if (tx >= cam.W) return;  // warp-uniform, no block barrier below
  SurfelWarp& st = s_all[warp];
  const int x = tx + (lane & 7), y = ty + (lane >> 3);
  const float ux = __fdiv_rn(__fsub_rn(__fdiv_rn(__fadd_rn((float)x, 0.5f), cam.hw), 1.0f), cam.kx);
  const float uy = __fdiv_rn(__fsub_rn(1.0f, __fdiv_rn(__fadd_rn((float)y, 0.5f), cam.hh)), cam.ky);
  unsigned my_n = 0, my_end = 0;  // lane l: the tile's cell of level l
  if (lane < g.levels) {
    const int k = g.first[lane] + (ty >> (2 + lane)) * g.nx[lane] + (tx >> (3 + lane));
    my_n = __ldcg(counts + k);
    my_end = __ldcg(cursor + k);
  }
  const float inf = __int_as_float(0x7f800000);
  st.nearest[lane] = 0xffffffffu;
  st.ray[lane] = make_float2(ux, uy);
  // nearest depth so far and the window's end below it, the farthest blended depth, the sums
  float dmin = inf, lim = inf, far = 0.0f, w = 0.0f;
  float a0 = 0, a1 = 0, a2 = 0, a3 = 0, n0 = 0, n1 = 0, n2 = 0, n3 = 0;
  bool redo = false;
  // One pass blends as it goes: a surfel behind the window of the nearest so far stays out, since
  // that window only moves nearer.  When a nearer surfel moves it past some, but not all, of the
  // blended ones, the tile is gone over again with the window known.
  for (int pass = 0; pass < 2; ++pass) {
    for (int l = 0; l < g.levels; ++l) {
      const unsigned n = __shfl_sync(0xffffffffu, my_n, l), first = __shfl_sync(0xffffffffu, my_end, l) - n;
      unsigned next = 0;
      if (lane < n) next = __ldcg(list + first + lane);
      for (unsigned q0 = 0; q0 < n; q0 += 32) {
        // a lane per surfel: its box clipped to the tile, its frame
        const unsigned idx = next;
        if (q0 + 32 + lane < n) next = __ldcg(list + first + q0 + 32 + lane);
        int cx = 0, cy = 0, cw = 0, ch = 0;
        if (q0 + lane < n) {
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
        if (live == 0u) continue;
        const int total = __shfl_sync(0xffffffffu, incl, 31), excl = incl - mine;
        if (mine > 0) {
          const float4 r0 = __ldg(rec + 4 * (size_t)idx), r1 = __ldg(rec + 4 * (size_t)idx + 1);
          const float4 r2 = __ldg(rec + 4 * (size_t)idx + 2), r3 = __ldg(rec + 4 * (size_t)idx + 3);
          SurfelFrame s;
          float c[3];
          surfel_frame(r0, r1, r2, cam, s, c);
          // the surfels with items, in consecutive rows; packed: clipped origin, width, its reciprocal
          // (exact quotients of items below 32 by widths up to 8) and the first item (below 1024)
          const int row = __popc(live & ((1u << lane) - 1u));
          const unsigned items = (unsigned)cx | ((unsigned)cy << 3) | ((unsigned)cw << 5) |
                                 (((255u + cw) / (unsigned)cw) << 9) | ((unsigned)excl << 18);
          float4* f = (float4*)st.frame[row];
          f[0] = s.n, f[1] = s.t, f[2] = s.b, f[3] = make_float4(s.cb, s.nc, __uint_as_float(items), 0.0f);
          const float rw = rsqrtf(fmaf(r1.x, r1.x, fmaf(r1.y, r1.y, r1.z * r1.z)));
          float4* m = (float4*)st.mat[row];
          m[0] = make_float4(r1.x * rw, r1.y * rw, r1.z * rw, r2.w);
          m[1] = r3;
        }
        st.hits[lane] = 0u;
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
              atomicMin(&st.nearest[px], __float_as_uint(sd));  // positive floats order as their bits
              atomicOr(&st.hits[px], 1u << k);
              st.depth[px][k] = sd;
            }
          }
        }
        __syncwarp();
        // a lane per pixel
        unsigned hits = st.hits[lane];
        if (hits) {
          const float sd = __uint_as_float(st.nearest[lane]);
          if (sd < dmin) {
            const float end = __fmul_rn(sd, cam.f);
            if (far > end) {
              redo = redo || dmin <= end;  // some blended surfels stay in the window, some do not
              w = far = a0 = a1 = a2 = a3 = n0 = n1 = n2 = n3 = 0.0f;
            }
            dmin = sd;
            lim = end;
          }
          do {
            const int k = __ffs(hits) - 1;
            hits &= hits - 1;
            const float d = st.depth[lane][k];
            if (d <= lim) {
              far = fmaxf(far, d);
              const float4 nw = *(const float4*)st.mat[k], al = *(const float4*)(st.mat[k] + 4);
              a0 += al.x, a1 += al.y, a2 += al.z, a3 += nw.w;
              n0 += nw.x, n1 += nw.y, n2 += nw.z, n3 += al.w;
              w += 1.0f;
            }
          } while (hits);
        }
        __syncwarp();
      }
    }
    if (!__any_sync(0xffffffffu, redo)) break;
    w = a0 = a1 = a2 = a3 = n0 = n1 = n2 = n3 = 0.0f;
    redo = false;
  }
  if (x >= cam.W || y >= cam.H) return;
  float4* rt0 = (float4*)(const_cast<char*>(out.rt[0]) + (size_t)y * out.pitch[0]) + x;
  float4* rt1 = (float4*)(const_cast<char*>(out.rt[1]) + (size_t)y * out.pitch[1]) + x;
  float* dep = (float*)(const_cast<char*>(out.rt[3]) + (size_t)y * out.pitch[3]) + x;
  if (weight) ((float*)((char*)weight + (size_t)y * weight_pitch))[x] = w;
  if (w == 0.0f) {
    *rt0 = make_float4(0, 0, 0, 0);
    *rt1 = make_float4(0, 0, 0, 0);
    *dep = inf;
    return;
  }
  const float iw = 1.0f / w;
  const float nn = fmaf(n0, n0, fmaf(n1, n1, n2 * n2));
  const float rn = nn > 0.0f ? rsqrtf(nn) : 0.0f;
  *rt0 = make_float4(a0 * iw, a1 * iw, a2 * iw, a3 * iw);
  *rt1 = make_float4(n0 * rn, n1 * rn, n2 * rn, n3 * iw);
  *dep = dmin;
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct SurfelLayout {
  size_t counts, cursor, boxes, list, bytes;
  SurfelGrid grid;
};

// The workspace: cell counts (then the list's length) and cursors, 8 bytes of box and kSurfelCells
// list entries per surfel.  `bytes` is the size callers have always been told, 40 B per pixel, 4 B
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
  l.counts = 0;
  l.cursor = align256(4 * (cells + 1));
  l.boxes = l.cursor + align256(4 * cells);
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
  if (cudaMemsetAsync(counts, 0, 4 * (size_t)(cells + 1), s) != cudaSuccess)
    return fail(EPBR_ERR_CUDA, "surfels: memset failed");
  const GbufDev gd = make_gbuf(*out);
  const float4* rec = (const float4*)surfels->records;
  cudaError_t e = cudaSuccess;
  if (N > 0) {
    const dim3 per_surfel((N + 255) / 256), per_cell((cells + 255) / 256);
    k_surfel_count<<<per_surfel, 256, 0, s>>>(rec, N, sc, g, boxes, counts);
    e = launch_kernel(k_surfel_alloc, per_cell, dim3(256), 0, s, true, (const unsigned*)counts, cells, cursor,
                      counts + cells);
    if (e == cudaSuccess)
      e = launch_kernel(k_surfel_fill, per_surfel, dim3(256), 0, s, true, (const uint2*)boxes, N, g, cursor, list);
  }
  if (e == cudaSuccess)
    e = launch_kernel(k_surfel_tile, dim3((W + kSurfelTileWarps * kTileW - 1) / (kSurfelTileWarps * kTileW), (H + kTileH - 1) / kTileH),
                      dim3(32 * kSurfelTileWarps), 0, s, N > 0, rec, (const uint2*)boxes, sc, g, (const unsigned*)counts,
                      (const unsigned*)cursor, (const unsigned*)list, gd, weight, (long long)weight_pitch);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(EPBR_ERR_CUDA, "surfels: %s", cudaGetErrorString(e));
  }
  if ((st = check_launch("surfels"))) return st;
  return ok();
}
