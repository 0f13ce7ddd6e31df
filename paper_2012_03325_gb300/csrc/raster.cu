// The G-buffer pass of mesh rendering (Sec. 4.1): triangles rasterised into the FP32 G-buffer.
//   k_raster_tri       one thread per triangle and view: view transform and projection in FP32 with
//                      every operation rounded, vertices snapped to 1/256 px, orientation, pixel
//                      box; a box of at most kSerialPx pixels is tested by the thread itself, a
//                      larger one is queued
//   k_raster_large     the queued triangles: one warp per box of at most kChunkPx pixels, one warp per
//                      kChunkPx pixels of the others (a binary search over their task offsets)
//   k_raster_resolve   one thread per pixel: the winning triangle's perspective-correct weights
//                      and interpolated attributes, written as the FP32 G-buffer
//   k_fill_inf         the shadow maps' initial value; the coverage then lowers the maps' depths in
//                      place (Sec. 5.1 renders the scene "as a depth map" from each point light as
//                      from a normal camera)
// A G-buffer view keeps the nearest (depth bits, index) per pixel with a 64-bit atomicMin, a shadow
// map its smallest depth with a 32-bit one.  The coverage and depth decisions evaluate exactly the
// expressions of the oracle (integer edge functions; FP32 products, sums and quotients each
// rounded), so the covering triangle of every pixel is reproducible bit for bit.
#include <string.h>

#include <algorithm>
#include <cmath>

#include "epbr_internal.cuh"

namespace epbr {

// 64 bytes, two 32-byte sectors for the coverage's read of a triangle
struct TriSetup {
  int4 qab;    // snapped screen positions of a and b (1/256 px)
  int4 qc_xy;  // c, then the box origin x0, y0
  float4 iz;   // 1/z of a, b, c, then the area as a float
  int4 meta;   // box width | height << 16 (each at most 32768), then the vertex indices of a, b, c
};

__device__ __forceinline__ int box_width(const TriSetup& s) { return s.meta.x & 0xffff; }
__device__ __forceinline__ int box_height(const TriSetup& s) { return (int)((unsigned)s.meta.x >> 16); }

// Boxes of at most kSerialPx pixels are tested by their triangle's thread; k_raster_large takes the
// others, in tasks of kChunkPx pixels (more where the task count must fit its bits).  Neighbouring
// triangles of a mesh have boxes of similar size, so the lanes' loops end together, and the queue
// balances the rest over the GPU.  Measured (1080p pass of a 200,192-triangle mesh / 64 maps of 512^2
// of the same mesh, us): 8, 16, 24, 32, 48, 64 pixels 82, 73, 69, 67, 68, 69 / 541, 488, 485, 487,
// 490, 499 (chunks of 512); chunks of 256, 512, 1024, 2048, 4096 at 32 pixels 74, 67, 63, 71, 86 /
// 557, 487, 472, 499, 612.
constexpr int kSerialPx = 32, kChunkPx = 1024;
// Extent (1/256 px, in x and in y) up to which 32 bits hold the edge functions at the pixels of a
// triangle's box: extent^2 < 2^31 (181 pixels).
constexpr unsigned kNarrowExtent = 46340;

struct RasterCam {
  float r[9];  // view_to_world rotation, row-major
  float eye[3];
  float kx, ky, hw, hh, near;
  int W, H;
};

// The cameras of a group of views rendered by one set of launches (the lights' shadow maps);
// a single view uses c[0].  The shadow maps' workspace is sized for kMaxViews views with their
// keys; a launch takes up to kMaxGroup (2.4 KB of kernel parameters).
constexpr int kMaxViews = 8, kMaxGroup = 32;
struct RasterCams {
  RasterCam c[kMaxGroup];
};

struct RVert {
  float iz;
  int qx, qy;
  bool ok;
};

__device__ __forceinline__ RVert raster_vertex(const float* __restrict__ v, const RasterCam& c) {
  float dx = __fsub_rn(v[0], c.eye[0]), dy = __fsub_rn(v[1], c.eye[1]), dz = __fsub_rn(v[2], c.eye[2]);
  // view axis k = column k of the view_to_world rotation: r[k], r[3 + k], r[6 + k]
  float ax = __fadd_rn(__fadd_rn(__fmul_rn(c.r[0], dx), __fmul_rn(c.r[3], dy)), __fmul_rn(c.r[6], dz));
  float ay = __fadd_rn(__fadd_rn(__fmul_rn(c.r[1], dx), __fmul_rn(c.r[4], dy)), __fmul_rn(c.r[7], dz));
  float az = __fadd_rn(__fadd_rn(__fmul_rn(c.r[2], dx), __fmul_rn(c.r[5], dy)), __fmul_rn(c.r[8], dz));
  RVert o = {0.0f, 0, 0, false};
  const float e = -az;
  if (!(e >= c.near)) return o;
  o.iz = __frcp_rn(e);  // 1 / e, correctly rounded
  float u = __fmul_rn(ax, o.iz), w = __fmul_rn(ay, o.iz);
  float X = __fmul_rn(c.hw, __fadd_rn(1.0f, __fmul_rn(u, c.kx)));
  float Y = __fmul_rn(c.hh, __fsub_rn(1.0f, __fmul_rn(w, c.ky)));
  o.ok = fabsf(X) < 4194304.0f && fabsf(Y) < 4194304.0f;
  o.qx = __float2int_rn(X * 256.0f);  // below 2^30 in magnitude when ok
  o.qy = __float2int_rn(Y * 256.0f);
  return o;
}

__device__ __forceinline__ long long edge_fn(long long ax, long long ay, long long bx, long long by, long long px,
                                             long long py) {
  return (bx - ax) * (py - ay) - (by - ay) * (px - ax);
}

// top-left rule: 0 for an edge whose zero-weight centres belong to the triangle, else 1.  A centre
// is covered by an edge when its (integer) edge function is >= this value.
__device__ __forceinline__ int edge_excl(int ax, int ay, int bx, int by) {
  int dx = bx - ax, dy = by - ay;
  return (dy < 0 || (dy == 0 && dx > 0)) ? 0 : 1;
}

// Where the coverage keeps the nearest surface of a view: DEPTH 0, (depth bits, triangle) keys; 1,
// the shadow maps themselves (positive floats order as their bits).
template <int DEPTH>
__device__ __forceinline__ void raster_put(void* img, size_t p, float z, int tri) {
  if (DEPTH)
    atomicMin((unsigned*)img + p, __float_as_uint(z));
  else
    atomicMin((unsigned long long*)img + p, ((unsigned long long)__float_as_uint(z) << 32) | (unsigned)tri);
}

// The edge functions of a triangle as values at a pixel and steps per pixel in x and y, each less
// the edge's top-left exclusion, so that a pixel is covered when none is negative.  Kept modulo 2^32
// (U = unsigned) or 2^64: the value at a pixel of the triangle's box is twice the area of a triangle
// inside that box, at most extent_x * extent_y in magnitude, so 32 bits hold it when that product is
// below 2^31, whatever a step outside the box wraps to.
template <typename U>
struct Edges {
  U c, a, b, cx, ax, bx, cy, ay, by;
  U xc, xa, xb;  // the exclusions
  __device__ __forceinline__ bool covers() const {
    return sizeof(U) == 4 ? (int)(c | a | b) >= 0 : (long long)(c | a | b) >= 0;
  }
};

template <typename U>
__device__ __forceinline__ Edges<U> raster_edges(const int4 qab, const int4 qc_xy, int x, int y) {
  Edges<U> e;
  // sign-extended to the width of U
  const U px = (U)(256 * x + 128), py = (U)(256 * y + 128);
  const U ax = (U)qab.x, ay = (U)qab.y, bx = (U)qab.z, by = (U)qab.w, cx = (U)qc_xy.x, cy = (U)qc_xy.y;
  e.xc = (U)edge_excl(qab.x, qab.y, qab.z, qab.w);
  e.xa = (U)edge_excl(qab.z, qab.w, qc_xy.x, qc_xy.y);
  e.xb = (U)edge_excl(qc_xy.x, qc_xy.y, qab.x, qab.y);
  e.c = (bx - ax) * (py - ay) - (by - ay) * (px - ax) - e.xc;
  e.a = (cx - bx) * (py - by) - (cy - by) * (px - bx) - e.xa;
  e.b = (ax - cx) * (py - cy) - (ay - cy) * (px - cx) - e.xb;
  e.cx = (ay - by) * 256u, e.ax = (by - cy) * 256u, e.bx = (cy - ay) * 256u;
  e.cy = (bx - ax) * 256u, e.ay = (cx - bx) * 256u, e.by = (ax - cx) * 256u;
  return e;
}

// Eye depth of a covered pixel from its edge functions (non-negative, their sum the area).  NARROW:
// the area, so each of them, is below 2^32 and converts to float from 32 bits (the same value).
template <bool NARROW, typename U>
__device__ __forceinline__ float raster_depth(const Edges<U>& e, float4 iz) {
  const U wa = e.a + e.xa, wb = e.b + e.xb, wc = e.c + e.xc;
  const float fa = NARROW ? (float)(unsigned)wa : (float)wa, fb = NARROW ? (float)(unsigned)wb : (float)wb;
  const float fc = NARROW ? (float)(unsigned)wc : (float)wc;
  const float s0 = __fmul_rn(fa, iz.x), s1 = __fmul_rn(fb, iz.y), s2 = __fmul_rn(fc, iz.z);
  return __fdiv_rn(iz.w, __fadd_rn(__fadd_rn(s0, s1), s2));
}

// Pixels first + lane, first + lane + 32, ... below last of a box (row order), for a whole warp.
template <int DEPTH, bool NARROW, typename U>
__device__ __forceinline__ void raster_box_warp(const int4 qab, const int4 qc_xy, float4 iz, int w, int first, int last,
                                                int lane, int tri, int W, void* img) {
  int j = first + lane;
  // quotients by the box width: below 2^15 the FP32 product is within 0.01 / w of (j + 1/2) / w,
  // whose distance to an integer is at least 1 / (2 w)
  const float rw = __frcp_rn((float)w);
  const int ly = j < (1 << 15) ? __float2int_rd(((float)j + 0.5f) * rw) : j / w;
  int lx = j - ly * w;
  const int dy = __float2int_rd(32.5f * rw), dx = 32 - dy * w;
  Edges<U> e = raster_edges<U>(qab, qc_xy, qc_xy.z + lx, qc_xy.w + ly);
  const U sc = (U)dx * e.cx + (U)dy * e.cy, sa = (U)dx * e.ax + (U)dy * e.ay, sb = (U)dx * e.bx + (U)dy * e.by;
  const U rc = e.cy - (U)w * e.cx, ra = e.ay - (U)w * e.ax, rb = e.by - (U)w * e.bx;  // on to the next row
  size_t p = (size_t)(qc_xy.w + ly) * W + (qc_xy.z + lx);
  const size_t sp = (size_t)dy * W + dx;
  for (; j < last; j += 32) {
    if (e.covers()) raster_put<DEPTH>(img, p, raster_depth<NARROW, U>(e, iz), tri);
    lx += dx;
    p += sp;
    e.c += sc, e.a += sa, e.b += sb;
    if (lx >= w) {
      lx -= w;
      p += W - w;
      e.c += rc, e.a += ra, e.b += rb;
    }
  }
}

// Queue of the triangles k_raster_tri leaves to k_raster_large, n entries for at most n set-ups: those of
// one task as set-up indices from the end (count[1] + 1 of them), those of several from the front:
// count[0] + 1 holds their number in its low `bits` bits and their tasks above (one atomicAdd
// takes an entry and its task range, so the task offsets ascend), entry k is (its first task <<
// bits) | set-up index.  The counters start at all ones, the value the keys' memset writes.
struct RasterQueue {
  unsigned long long* count;
  unsigned long long* entry;
  long long n;
  int bits, chunk;  // chunk: box pixels per task
};

// Bound by instruction issue: about 600 warp instructions per 32 triangles and view (three vertex
// transforms, the box, the serial pixels; ncu: 0.76 per scheduler and cycle), so the edge functions
// are 32-bit wherever they fit and a triangle that no pixel centre can hit stops at its box.  62 us for
// the 1080p pass, 460 us for the 64 maps; 122 and 1650 us with a set-up pass, scans over the item counts and a
// search per run of box pixels.
// blockIdx.y = the view: its set-ups follow the previous views' (set-up view * T + t), its image
// starts at view * view_px.  Set-ups are stored for the resolve (DEPTH 0) and for the queued ones.
template <int DEPTH>
__global__ void __launch_bounds__(256) k_raster_tri(const float* __restrict__ verts, int V, const int* __restrict__ tris,
                                                    int T, const __grid_constant__ RasterCams cams,
                                                    TriSetup* __restrict__ setup, RasterQueue queue, long long view_px,
                                                    void* __restrict__ img) {
  griddep_launch_dependents();
  const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const RasterCam& cam = cams.c[blockIdx.y];
  const int W = cam.W;
  img = DEPTH ? (void*)((unsigned*)img + blockIdx.y * view_px) : (void*)((unsigned long long*)img + blockIdx.y * view_px);
  int4 qab = make_int4(0, 0, 0, 0), qc_xy = qab;
  float4 iz = make_float4(0, 0, 0, 0);
  int w = 1, area_px = 0;  // box width and pixels
  bool queued = false;     // as a single task
  const unsigned idx = blockIdx.y * (unsigned)T + t;  // set-up index, below 2^31
  int i[3] = {-1, -1, -1};
  if (t < T)
#pragma unroll
    for (int k = 0; k < 3; ++k) i[k] = __ldg(tris + 3 * (size_t)t + k);
  if (i[0] >= 0 && i[1] >= 0 && i[2] >= 0 && i[0] < V && i[1] < V && i[2] < V) {
    RVert a = raster_vertex(verts + 12 * (size_t)i[0], cam), b = raster_vertex(verts + 12 * (size_t)i[1], cam),
          c = raster_vertex(verts + 12 * (size_t)i[2], cam);
    if (a.ok && b.ok && c.ok) {
      const int xmin = min(a.qx, min(b.qx, c.qx)), xmax = max(a.qx, max(b.qx, c.qx));
      const int ymin = min(a.qy, min(b.qy, c.qy)), ymax = max(a.qy, max(b.qy, c.qy));
      // pixels whose centre 256 x + 128 lies in [min, max], clipped to the image
      const int x0 = max((xmin + 127) >> 8, 0), x1 = min((xmax - 128) >> 8, W - 1);
      const int y0 = max((ymin + 127) >> 8, 0), y1 = min((ymax - 128) >> 8, cam.H - 1);
      if (x1 >= x0 && y1 >= y0) {
        const unsigned ex = (unsigned)xmax - (unsigned)xmin, ey = (unsigned)ymax - (unsigned)ymin;
        const bool narrow = ex <= kNarrowExtent && ey <= kNarrowExtent;
        long long area = narrow ? (long long)(int)((unsigned)(b.qx - a.qx) * (unsigned)(c.qy - a.qy) -
                                                     (unsigned)(b.qy - a.qy) * (unsigned)(c.qx - a.qx))
                                : edge_fn(a.qx, a.qy, b.qx, b.qy, c.qx, c.qy);
        if (area != 0) {
          int ib = i[1], ic = i[2];
          if (area < 0) {  // orient so that the area is positive
            RVert tmp = b;
            b = c;
            c = tmp;
            ib = i[2];
            ic = i[1];
            area = -area;
          }
          const int h = y1 - y0 + 1;
          w = x1 - x0 + 1;
          area_px = w * h;  // at most 2^30
          const bool here = narrow && area_px <= kSerialPx;
          qab = make_int4(a.qx, a.qy, b.qx, b.qy);
          qc_xy = make_int4(c.qx, c.qy, x0, y0);
          iz = make_float4(a.iz, b.iz, c.iz, __ll2float_rn(area));
          if (!DEPTH || !here) {
            TriSetup s;
            s.qab = qab, s.qc_xy = qc_xy, s.iz = iz;
            s.meta = make_int4((int)((unsigned)w | ((unsigned)h << 16)), i[0], ib, ic);
            setup[idx] = s;
          }
          if (!here) {
            queued = area_px <= queue.chunk;
            if (!queued) {
              const unsigned long long tasks = (unsigned)(area_px + queue.chunk - 1) / (unsigned)queue.chunk;
              const unsigned long long at = atomicAdd(queue.count, (tasks << queue.bits) + 1ull) + 1ull;
              const unsigned long long mask = (1ull << queue.bits) - 1ull;
              queue.entry[at & mask] = (at & ~mask) | idx;
            }
            area_px = 0;  // nothing left for this thread
          }
        } else {
          area_px = 0;
        }
      }
    }
  }
  const unsigned q = __ballot_sync(0xffffffffu, queued);
  if (q) {  // one atomic per warp
    unsigned long long base = 0;
    if (lane == __ffs(q) - 1) base = atomicAdd(queue.count + 1, (unsigned long long)__popc(q)) + 1ull;
    base = __shfl_sync(0xffffffffu, base, __ffs(q) - 1);
    if (queued) queue.entry[queue.n - 1 - (long long)base - __popc(q & ((1u << lane) - 1u))] = idx;
  }
  if (area_px > 0) {
    Edges<unsigned> e = raster_edges<unsigned>(qab, qc_xy, qc_xy.z, qc_xy.w);
    const unsigned rc = e.cy - w * e.cx, ra = e.ay - w * e.ax, rb = e.by - w * e.bx;
    size_t p = (size_t)qc_xy.w * W + qc_xy.z;
    int lx = 0;
    for (int k = 0; k < area_px; ++k) {
      if (e.covers()) raster_put<DEPTH>(img, p, raster_depth<true, unsigned>(e, iz), t);
      ++p, e.c += e.cx, e.a += e.ax, e.b += e.bx;
      if (++lx == w) lx = 0, p += W - w, e.c += rc, e.a += ra, e.b += rb;
    }
  }
}

// Box pixels first .. last - 1 of a queued triangle, by one warp.
template <int DEPTH>
__device__ __forceinline__ void raster_task(const TriSetup& s, unsigned idx, int first, int last, int lane, unsigned T,
                                            int W, long long view_px, void* img) {
  const unsigned v = idx / T;
  const int w = box_width(s), tri = (int)(idx - v * T);
  img = DEPTH ? (void*)((unsigned*)img + v * view_px) : (void*)((unsigned long long*)img + v * view_px);
  const unsigned ex = (unsigned)max(s.qab.x, max(s.qab.z, s.qc_xy.x)) - (unsigned)min(s.qab.x, min(s.qab.z, s.qc_xy.x));
  const unsigned ey = (unsigned)max(s.qab.y, max(s.qab.w, s.qc_xy.y)) - (unsigned)min(s.qab.y, min(s.qab.w, s.qc_xy.y));
  if (ex <= kNarrowExtent && ey <= kNarrowExtent)
    raster_box_warp<DEPTH, true, unsigned>(s.qab, s.qc_xy, s.iz, w, first, last, lane, tri, W, img);
  else if (s.iz.w < 4e9f)
    raster_box_warp<DEPTH, true, unsigned long long>(s.qab, s.qc_xy, s.iz, w, first, last, lane, tri, W, img);
  else
    raster_box_warp<DEPTH, false, unsigned long long>(s.qab, s.qc_xy, s.iz, w, first, last, lane, tri, W, img);
}

// Balances the queue over the grid.  Three blocks per SM (80 registers): four or five at 64 or 48
// registers measured 66 and 70 us for the 1080p pass against 62 (461 and 486 against 467 us for the
// maps).
template <int DEPTH>
__global__ void __launch_bounds__(256, 3) k_raster_large(const TriSetup* __restrict__ setup, RasterQueue queue, int T, int W,
                                                      long long view_px, void* __restrict__ img) {
  griddep_wait();  // launched early: the queue is complete when k_raster_tri has finished
  if (!DEPTH) griddep_launch_dependents();  // the resolve; the maps' last kernel lets nothing begin early
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long singles = (long long)(queue.count[1] + 1ull);
  // the tasks of the larger boxes first (they are the longer ones), then the boxes of one task,
  // whose next set-up is loaded while the current one is tested
  const unsigned long long n = queue.count[0] + 1ull;
  const long long total = (long long)(n >> queue.bits);
  const unsigned long long mask = (1ull << queue.bits) - 1ull;
  const int entries = (int)(n & mask);
  for (long long task = warp; task < total; task += warps) {
    int lo = 0, hi = entries - 1;  // the last entry whose first task is <= task (warp-uniform)
    while (lo < hi) {
      const int mid = lo + (hi - lo + 1) / 2;
      if ((long long)(__ldcg(queue.entry + mid) >> queue.bits) <= task) lo = mid;
      else hi = mid - 1;
    }
    const unsigned long long q = __ldcg(queue.entry + lo);
    const unsigned idx = (unsigned)(q & mask);
    const TriSetup s = setup[idx];
    const int first = (int)((task - (long long)(q >> queue.bits)) * queue.chunk);
    const int last = (int)min((long long)first + queue.chunk, (long long)box_width(s) * box_height(s));
    raster_task<DEPTH>(s, idx, first, last, lane, (unsigned)T, W, view_px, img);
  }
  const unsigned long long* one = queue.entry + queue.n - 1;
  unsigned next_idx = 0;
  TriSetup next;
  if (warp < singles) next_idx = (unsigned)__ldcg(one - warp), next = setup[next_idx];
  for (long long k = warp; k < singles; k += warps) {
    const TriSetup s = next;
    const unsigned idx = next_idx;
    if (k + warps < singles) next_idx = (unsigned)__ldcg(one - (k + warps)), next = setup[next_idx];
    raster_task<DEPTH>(s, idx, 0, box_width(s) * box_height(s), lane, (unsigned)T, W, view_px, img);
  }
}

// ---- resolve ---------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_raster_resolve(const float* __restrict__ verts,
                                                        const TriSetup* __restrict__ setup,
                                                        const unsigned long long* __restrict__ keys, int W, int H,
                                                        GbufDev g, int* __restrict__ ids, long long ids_pitch) {
  int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
  griddep_wait();  // launched early
  if (x >= W || y >= H) return;
  const unsigned long long key = __ldcg(keys + (size_t)y * W + x);
  float4* rt0 = (float4*)(const_cast<char*>(g.rt[0]) + (size_t)y * g.pitch[0]) + x;
  float4* rt1 = (float4*)(const_cast<char*>(g.rt[1]) + (size_t)y * g.pitch[1]) + x;
  float* dep = (float*)(const_cast<char*>(g.rt[3]) + (size_t)y * g.pitch[3]) + x;
  int* idp = ids ? (int*)((char*)ids + (size_t)y * ids_pitch) + x : nullptr;
  if (key == ~0ULL) {
    *rt0 = make_float4(0, 0, 0, 0);
    *rt1 = make_float4(0, 0, 0, 0);
    *dep = __int_as_float(0x7f800000);
    if (idp) *idp = -1;
    return;
  }
  const int t = (int)(key & 0xffffffffULL);
  const TriSetup s = setup[t];
  const long long px = 256LL * x + 128, py = 256LL * y + 128;
  // perspective-correct weights b_i / z_i normalised, from the exact edge functions
  float wa = __ll2float_rn(edge_fn(s.qab.z, s.qab.w, s.qc_xy.x, s.qc_xy.y, px, py)) * s.iz.x;
  float wb = __ll2float_rn(edge_fn(s.qc_xy.x, s.qc_xy.y, s.qab.x, s.qab.y, px, py)) * s.iz.y;
  float wc = __ll2float_rn(edge_fn(s.qab.x, s.qab.y, s.qab.z, s.qab.w, px, py)) * s.iz.z;
  const float inv = rcp_ftz(wa + wb + wc);
  wa *= inv;
  wb *= inv;
  wc *= inv;
  // vertex values 3 .. 10 (normal, albedo, metal, rough) read as three float4 of each 48-byte
  // record (16-byte aligned, checked on the host): normal.x is the w of the first, normal.yz and
  // albedo.rg fill the second, albedo.b, metal and rough lead the third
  const float4* A = (const float4*)(verts + 12 * (size_t)s.meta.y);
  const float4* B = (const float4*)(verts + 12 * (size_t)s.meta.z);
  const float4* C = (const float4*)(verts + 12 * (size_t)s.meta.w);
  float at[8];
  {
    const float4 a0 = __ldg(A), a1 = __ldg(A + 1), a2 = __ldg(A + 2);
    const float4 b0 = __ldg(B), b1 = __ldg(B + 1), b2 = __ldg(B + 2);
    const float4 c0 = __ldg(C), c1 = __ldg(C + 1), c2 = __ldg(C + 2);
    const float va[8] = {a0.w, a1.x, a1.y, a1.z, a1.w, a2.x, a2.y, a2.z};
    const float vb[8] = {b0.w, b1.x, b1.y, b1.z, b1.w, b2.x, b2.y, b2.z};
    const float vc[8] = {c0.w, c1.x, c1.y, c1.z, c1.w, c2.x, c2.y, c2.z};
#pragma unroll
    for (int q = 0; q < 8; ++q) at[q] = fmaf(wa, va[q], fmaf(wb, vb[q], wc * vc[q]));
  }
  float3 n = f3(at[0], at[1], at[2]);
  n = n * rsqrt_ftz(dot3(n, n));
  *rt0 = make_float4(at[3], at[4], at[5], at[6]);
  *rt1 = make_float4(n.x, n.y, n.z, at[7]);
  *dep = __uint_as_float((unsigned)(key >> 32));
  if (idp) *idp = t;
}

// The value of a shadow map texel that nothing covers.
__global__ void __launch_bounds__(256) k_fill_inf(float* __restrict__ out, long long n) {
  for (long long k = blockIdx.x * 256LL + threadIdx.x; k < n; k += gridDim.x * 256LL) out[k] = __int_as_float(0x7f800000);
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr int kCounters = 32;  // queue counters, two per group of views, reset together

struct RasterLayout {
  size_t count, keys, setup, entry, bytes;
};

// The workspace of `views` views of W x H pixels and T triangles each: the queue counters, the
// keys, 64 B of set-up and 8 B of queue entry per triangle.  `bytes` includes 8 B per 1024
// triangles that nothing uses, the size callers have always been told.
static RasterLayout raster_layout(long long T, int W, int H, int views = 1) {
  RasterLayout l;
  const long long n = T * views;
  const size_t count_bytes = align256(sizeof(long long) * (size_t)((n + 1023) / 1024 + 1));
  l.count = 0;  // followed by the keys: one memset resets both
  l.keys = sizeof(unsigned long long) * kCounters;
  l.setup = align256(l.keys + sizeof(unsigned long long) * (size_t)W * H * views);
  l.entry = align256(l.setup + sizeof(TriSetup) * (size_t)n);
  l.bytes = align256(sizeof(unsigned long long) * (size_t)W * H * views) + align256(sizeof(TriSetup) * (size_t)n) +
            align256(sizeof(long long) * (size_t)(n + 1)) + count_bytes;
  return l;
}

// The queue of n set-ups over images of `px` pixels: enough bits for n entries, and tasks long
// enough for the task count to fit the others (n * ceil(px / chunk) < 2^(64 - bits)).
static RasterQueue raster_queue(char* ws, size_t count, size_t entry, long long n, long long px) {
  RasterQueue q;
  q.count = (unsigned long long*)(ws + count);
  q.entry = (unsigned long long*)(ws + entry);
  q.n = n;
  q.bits = 1;
  while ((1ull << q.bits) <= (unsigned long long)n) ++q.bits;
  q.chunk = kChunkPx;
  while ((unsigned long long)n * (unsigned long long)((px + q.chunk - 1) / q.chunk) >= 1ull << (64 - q.bits)) q.chunk *= 2;
  return q;
}

}  // namespace epbr

using namespace epbr;

extern "C" epbr_status epbr_raster_workspace_size(int32_t num_triangles, int32_t width, int32_t height, size_t* bytes) {
  if (!bytes || num_triangles < 0 || width < 1 || height < 1 || width > (1 << 15) || height > (1 << 15))
    return fail(EPBR_ERR_INVALID_ARG, "raster: bytes NULL, num_triangles < 0 or size outside [1, 32768]");
  *bytes = raster_layout(num_triangles, width, height).bytes;
  return ok();
}

namespace epbr {

static epbr_status validate_mesh(const epbr_mesh* mesh, float near_depth) {
  if (mesh->num_vertices < 0 || mesh->num_triangles < 0 || mesh->num_vertices > (1 << 28) ||
      (mesh->num_triangles > 0 && (!mesh->vertices || !mesh->triangles)) || (uintptr_t)mesh->vertices % 16 ||
      (uintptr_t)mesh->triangles % 4)
    return fail(EPBR_ERR_INVALID_ARG, "raster: vertices / triangles NULL, misaligned or counts out of range");
  if (!(near_depth > 0.0f) || !std::isfinite(near_depth)) return fail(EPBR_ERR_INVALID_ARG, "raster: near must be > 0");
  return EPBR_OK;
}

static RasterCam make_raster_cam(const epbr_camera& camera, float near_depth) {
  RasterCam rc;
  CamDev cd = make_cam(camera);
  for (int i = 0; i < 9; ++i) rc.r[i] = cd.r[i];
  for (int i = 0; i < 3; ++i) rc.eye[i] = cd.eye[i];
  const int W = camera.width, H = camera.height;
  double t = std::tan(0.5 * (double)camera.fov_y);
  rc.ky = (float)(1.0 / t);
  rc.kx = (float)((double)H / ((double)W * t));
  rc.hw = (float)(0.5 * W);
  rc.hh = (float)(0.5 * H);
  rc.near = near_depth;
  rc.W = W;
  rc.H = H;
  return rc;
}

// Coverage of the mesh seen by `views` cameras of the same size: the nearest (depth, triangle) key
// of every pixel (DEPTH 0) or the maps' depths (DEPTH 1) in the views' images at `img`.
template <int DEPTH>
static cudaError_t raster_cover(const epbr_mesh* mesh, const RasterCams& rc, int views, TriSetup* setup,
                                const RasterQueue& q, void* img, cudaStream_t s) {
  const int T = mesh->num_triangles, W = rc.c[0].W;
  const long long view_px = (long long)W * rc.c[0].H;
  k_raster_tri<DEPTH><<<dim3((T + 255) / 256, views), 256, 0, s>>>(mesh->vertices, mesh->num_vertices, mesh->triangles, T,
                                                                    rc, setup, q, view_px, img);
  return launch_kernel(k_raster_large<DEPTH>, dim3(num_sms() * 8), dim3(256), 0, s, true, (const TriSetup*)setup, q, T, W,
                       view_px, img);
}

}  // namespace epbr

extern "C" epbr_status epbr_raster_gbuffer(const epbr_mesh* mesh, const epbr_camera* camera, float near_depth,
                                           const epbr_gbuffer* out, int32_t* ids, int64_t ids_pitch, void* workspace,
                                           size_t workspace_bytes, void* stream) {
  if (!mesh || !out) return fail(EPBR_ERR_INVALID_ARG, "raster: mesh or gbuffer is NULL");
  epbr_status st = validate_camera(camera, out);
  if (st) return st;
  if (out->format != EPBR_GBUFFER_FP32) return fail(EPBR_ERR_INVALID_ARG, "raster: the output G-buffer must be FP32");
  if ((st = validate_gbuffer(out, true))) return st;
  if ((st = validate_mesh(mesh, near_depth))) return st;
  if (ids && (ids_pitch < 4LL * out->width || ids_pitch % 4 || (uintptr_t)ids % 4))
    return fail(EPBR_ERR_INVALID_ARG, "raster: ids misaligned or pitch too small");
  const int W = out->width, H = out->height, T = mesh->num_triangles;
  RasterLayout l = raster_layout(T, W, H);
  if (!workspace || (uintptr_t)workspace % 256 || workspace_bytes < l.bytes)
    return fail(EPBR_ERR_INVALID_ARG, "raster: workspace NULL, not 256-byte aligned or below %zu bytes", l.bytes);
  char* ws = (char*)workspace;
  cudaStream_t s = (cudaStream_t)stream;
  RasterCams rc;
  rc.c[0] = make_raster_cam(*camera, near_depth);
  TriSetup* setup = (TriSetup*)(ws + l.setup);
  unsigned long long* keys = (unsigned long long*)(ws + l.keys);
  if (cudaMemsetAsync(ws + l.count, 0xff, l.keys + sizeof(unsigned long long) * (size_t)W * H, s) != cudaSuccess)
    return fail(EPBR_ERR_CUDA, "raster: memset failed");
  cudaError_t e = cudaSuccess;
  if (T > 0)
    e = raster_cover<0>(mesh, rc, 1, setup, raster_queue(ws, l.count, l.entry, T, (long long)W * H), keys, s);
  GbufDev gd = make_gbuf(*out);
  dim3 blk(32, 8), grd((W + 31) / 32, (H + 7) / 8);
  if (e == cudaSuccess)
    e = launch_kernel(k_raster_resolve, grd, blk, 0, s, true, mesh->vertices, (const TriSetup*)setup,
                      (const unsigned long long*)keys, W, H, gd, (int*)ids, (long long)ids_pitch);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(EPBR_ERR_CUDA, "raster: %s", cudaGetErrorString(e));
  }
  if ((st = check_launch("raster"))) return st;
  return ok();
}

extern "C" epbr_status epbr_shadow_maps_workspace_size(int32_t num_triangles, int32_t size, size_t* bytes) {
  if (!bytes || num_triangles < 0 || size < 1 || size > (1 << 15))
    return fail(EPBR_ERR_INVALID_ARG, "shadow_maps: bytes NULL, num_triangles < 0 or size outside [1, 32768]");
  *bytes = raster_layout(num_triangles, size, size, kMaxViews).bytes;
  return ok();
}

extern "C" epbr_status epbr_shadow_maps(const epbr_mesh* mesh, const epbr_camera* cameras, int32_t num_maps,
                                        float near_depth, float* maps, void* workspace, size_t workspace_bytes,
                                        void* stream) {
  if (!mesh || !cameras || num_maps < 0 || (num_maps > 0 && !maps) || (uintptr_t)maps % 4)
    return fail(EPBR_ERR_INVALID_ARG, "shadow_maps: mesh, cameras or maps NULL / misaligned, or num_maps < 0");
  if (num_maps == 0) return ok();
  epbr_status st = validate_mesh(mesh, near_depth);
  if (st) return st;
  const int S = cameras[0].width;
  for (int i = 0; i < num_maps; ++i) {
    const epbr_camera& c = cameras[i];
    if (c.width != S || c.height != S || S < 1 || S > (1 << 15) || !(c.fov_y > 0.0f && c.fov_y < 3.1f))
      return fail(EPBR_ERR_INVALID_ARG, "shadow_maps: camera %d must be square, of the first camera's size (%d), "
                                        "with a field of view in (0, 3.1) rad", i, S);
    for (int k = 0; k < 16; ++k)
      if (!std::isfinite(c.view_to_world[k])) return fail(EPBR_ERR_INVALID_ARG, "shadow_maps: camera %d not finite", i);
  }
  const long long T = mesh->num_triangles;
  if (T * kMaxViews >= (1LL << 31))
    return fail(EPBR_ERR_UNSUPPORTED, "shadow_maps: %lld triangles x %d views exceed 2^31 set-ups", T, kMaxViews);
  const RasterLayout full = raster_layout(T, S, S, kMaxViews);
  if (!workspace || (uintptr_t)workspace % 256 || workspace_bytes < full.bytes)
    return fail(EPBR_ERR_INVALID_ARG, "shadow_maps: workspace NULL, not 256-byte aligned or below %zu bytes",
                full.bytes);
  char* ws = (char*)workspace;
  cudaStream_t s = (cudaStream_t)stream;
  const long long px = (long long)S * S;
  k_fill_inf<<<num_sms() * 8, 256, 0, s>>>(maps, px * num_maps);
  // Lights per set of launches: as many as the workspace holds set-ups and queue entries for (the
  // maps are drawn in place, so its key images are not needed), at least kMaxViews.
  const size_t per_view = (sizeof(TriSetup) + sizeof(unsigned long long)) * (size_t)T;
  const size_t room = full.bytes - sizeof(unsigned long long) * kCounters - 512;
  const int group = T > 0 ? (int)std::min<size_t>({(size_t)kMaxGroup, std::max<size_t>(room / per_view, kMaxViews),
                                                    (size_t)(((1LL << 31) - 1) / T)}) : 1;  // set-up indices are ints
  cudaError_t e = cudaSuccess;
  for (int i0 = 0, k = 0; T > 0 && i0 < num_maps && e == cudaSuccess; i0 += group, ++k) {
    const int views = std::min(group, num_maps - i0);
    RasterCams rc;
    for (int v = 0; v < views; ++v) rc.c[v] = make_raster_cam(cameras[i0 + v], near_depth);
    if (k % (kCounters / 2) == 0 && cudaMemsetAsync(ws, 0xff, sizeof(unsigned long long) * kCounters, s) != cudaSuccess)
      return fail(EPBR_ERR_CUDA, "shadow_maps: memset failed");
    const size_t setup = 256, entry = setup + align256(sizeof(TriSetup) * (size_t)(T * views));
    e = raster_cover<1>(mesh, rc, views, (TriSetup*)(ws + setup),
                        raster_queue(ws, 2 * sizeof(unsigned long long) * (k % (kCounters / 2)), entry, T * views, px),
                        maps + (size_t)i0 * px, s);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(EPBR_ERR_CUDA, "shadow_maps: %s", cudaGetErrorString(e));
  }
  if ((st = check_launch("shadow_maps"))) return st;
  return ok();
}
