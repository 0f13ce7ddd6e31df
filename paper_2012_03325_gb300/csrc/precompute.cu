// Image-based lighting precompute (paper Sec. 3.1; split sum of Karis 2013):
//   k_brdf_lut          BRDF integration table (A, B), one warp per texel, Kahan + shuffles
//   k_irradiance_part   exact-quadrature irradiance, per-block partial sums over a slice of source
//                       row pieces: a row's hemisphere is one interval of columns, summed from
//                       sums of 64 and 8 texels and single texels at its ends (Kahan across pieces)
//   k_irradiance_texels the same for narrow environments, every output and texel (packed FP32x2 over
//                       output pairs, plain sums per staged tile, Kahan across tiles)
//   k_irradiance_final  one warp per output: lanes sum the block partials, a shuffle butterfly
//                       adds the lanes (fixed order: deterministic), then the ratio
//   k_prefilter         GGX-prefiltered levels 1..M-1, a block per segment of a row of a level: the
//                       row's sample geometry computed once (the sampling frame turns with the texel
//                       about the pole axis), each texel sums its samples at shifted columns
#include <cuda.h>  // CUcontext and CUresult for the context queries (fetched at run time)

#include <algorithm>
#include <type_traits>
#include <mutex>

#include "epbr_internal.cuh"

namespace epbr {

// Hammersley point k of N: (k / N, radical_inverse_2(k)).  For k < 2^24 the mirrored bits fit
// the float mantissa, so xi2 is exact.
__device__ __forceinline__ float hammersley_xi2(unsigned k) {
  return __uint2float_rn(__brev(k)) * 2.3283064365386963e-10f;
}

// GGX half vector in the frame (t, b, n): phi = 2 pi xi1, cos^2 = (1 - xi2) / d,
// sin^2 = alpha^2 xi2 / d with d = 1 + (alpha^2 - 1) xi2 (sin^2 taken directly, which avoids
// the cancellation of 1 - cos^2 near the lobe centre).
__device__ __forceinline__ float3 ggx_half(float xi1, float xi2, float a2, float3 t, float3 b, float3 n) {
  float inv = 1.0f / fmaf(a2 - 1.0f, xi2, 1.0f);
  float ct = sqrtf((1.0f - xi2) * inv);
  float st = sqrtf(a2 * xi2 * inv);
  float sp, cp;
  sincospif(2.0f * xi1, &sp, &cp);
  return t * (st * cp) + b * (st * sp) + n * ct;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A compensated sum of three channels.
struct Kahan3 {
  Kahan x, y, z;
  __device__ __forceinline__ void add(float3 v) { x.add(v.x), y.add(v.y), z.add(v.z); }
  __device__ __forceinline__ float3 value() const { return f3(x.s - x.c, y.s - y.c, z.s - z.c); }
};

// The kernels of a lighting set read only the environment and write their own outputs, so each is
// launched early and fills the SMs that the last blocks of the ones before leave.  One block of a
// kernel waits for the previous kernel at its end, so that none is complete before that one is, and
// the last kernel of a call does not let others begin early (a compose may read what the call wrote).
// Set of a 1024 x 512 environment (8 levels, 1024 samples), one after another 574 us, overlapped 536 us.
__device__ __forceinline__ void complete_in_order() {
  if (blockIdx.x == 0 && blockIdx.y == 0) griddep_wait();
}

// ------------------------------------------------------------------------------------------
// BRDF integration table
// ------------------------------------------------------------------------------------------
__global__ void k_brdf_lut(int S, int N, float2* __restrict__ lut, bool more) {
  if (more) griddep_launch_dependents();
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (warp >= S * S) return;  // not all warps of a block
  int i = warp % S, j = warp / S;
  float mu = (i + 0.5f) / S, r = (j + 0.5f) / S;
  float alpha = r * r, a2 = alpha * alpha, k = 0.5f * alpha;
  float3 v = f3(sqrtf(fmaf(-mu, mu, 1.0f)), 0.0f, mu);
  float nv = mu;
  float g1v = nv / fmaf(nv, 1.0f - k, k);
  Kahan A, B;
  const float3 t = f3(1, 0, 0), b = f3(0, 1, 0), n = f3(0, 0, 1);
  float invN = 1.0f / N;
  for (int s = lane; s < N; s += 32) {
    float3 h = ggx_half(s * invN, hammersley_xi2((unsigned)s), a2, t, b, n);
    float vh = dot3(v, h);
    float nl = fmaf(2.0f * vh, h.z, -v.z);
    if (nl > 0.0f) {
      float g = g1v * nl / fmaf(nl, 1.0f - k, k);
      float gvis = g * vh / (h.z * nv);
      float x = 1.0f - vh, x2 = x * x;
      float fc = x2 * x2 * x;
      A.add((1.0f - fc) * gvis);
      B.add(fc * gvis);
    }
  }
  float a = warp_sum(A.s - A.c), bb = warp_sum(B.s - B.c);
  if (lane == 0) lut[warp] = make_float2(a * invN, bb * invN);
  complete_in_order();
}

// ------------------------------------------------------------------------------------------
// Irradiance: sum_t L_t max(n.d_t, 0) Omega_t / sum_t max(n.d_t, 0) Omega_t
// ------------------------------------------------------------------------------------------
constexpr int kIrrThreads = 512;     // threads per block at most, an output each
constexpr int kIrrPiece = 2048;      // source columns staged per step
constexpr int kIrrGroup = 8, kIrrSeg = 64;  // columns per sum of the two levels
constexpr int kIrrTexelsPerBlock = 1024;
constexpr int kIrrMaxBlocks = 608;

int irr_blocks(int We, int He) {
  long long n = (long long)We * He;
  long long b = (n + kIrrTexelsPerBlock - 1) / kIrrTexelsPerBlock;
  return (int)std::min<long long>(std::max<long long>(b, 1), kIrrMaxBlocks);
}

size_t irr_workspace_bytes(int We, int He, int Wi, int Hi) {
  return (size_t)irr_blocks(We, He) * Wi * Hi * sizeof(float4);
}

// Unit direction of the centre of texel (i, j) of a W x H equirect map.
__device__ __forceinline__ float3 texel_dir(int i, int j, int W, int H) {
  float st, ct, sp, cp;
  sincospif((j + 0.5f) / H, &st, &ct);
  sincospif(2.0f * ((i + 0.5f) / W) - 1.0f, &sp, &cp);
  return f3(st * sp, ct, -st * cp);
}

// With the azimuth phi of source column x and of the output, n.d = A cos(phi_x - phi_i) + B, A and B
// constant along a source row, so that the hemisphere of n is one interval of the row's columns
// (none, some or all), and over any columns inside it
//   sum L (n.d) = A (cos phi_i sum L cos phi_x + sin phi_i sum L sin phi_x) + B sum L.
// Sums of these three over 8 and over 64 columns are formed once per row piece, so that an output
// needs about 30 terms per row instead of all its texels; the texels at the interval's ends are
// clamped one by one, as the definition has it.
struct IrrSums {
  float t[3], c[3], s[3];  // sums of L, L cos phi, L sin phi (three channels)
  float c1, s1, pad;       // sums of cos phi, sin phi
};

struct IrrAcc {
  float r = 0.0f, g = 0.0f, b = 0.0f, w = 0.0f;
};

__device__ __forceinline__ void irr_add(IrrAcc& a, const IrrSums& q, float ac, float as, float B, float n) {
  a.r += fmaf(ac, q.c[0], fmaf(as, q.s[0], B * q.t[0]));
  a.g += fmaf(ac, q.c[1], fmaf(as, q.s[1], B * q.t[1]));
  a.b += fmaf(ac, q.c[2], fmaf(as, q.s[2], B * q.t[2]));
  a.w += fmaf(ac, q.c1, fmaf(as, q.s1, B * n));
}

// Shared memory of a piece of n columns, one entry skipped per segment: the outputs of a warp, a
// segment apart on the usual maps, then read different banks.
__host__ __device__ inline int irr_at(int column) { return column + column / kIrrSeg; }
__host__ __device__ inline int irr_group_at(int g) { return g + g / (kIrrSeg / kIrrGroup); }
struct IrrShared {
  float4* texel;
  IrrSums* group;
  IrrSums* seg;
  float2* phi;  // cos, sin of the columns' azimuths
  size_t bytes;
};
__host__ __device__ inline IrrShared irr_shared(char* base, int n) {
  IrrShared s;
  size_t off = 0;
  s.texel = (float4*)base;
  off += sizeof(float4) * (irr_at(n - 1) + 1);
  s.group = (IrrSums*)(base + off);
  off += sizeof(IrrSums) * (irr_group_at(n / kIrrGroup) + 1);
  s.seg = (IrrSums*)(base + off);
  off += sizeof(IrrSums) * (n / kIrrSeg + 1);
  s.phi = (float2*)(base + off);
  s.bytes = off + sizeof(float2) * (irr_at(n - 1) + 1);
  return s;
}

// Bound by issue (the terms of every output and row): 39 us for a 2048 x 1024 environment, 319 us by
// k_irradiance_texels.
// Each block takes the row pieces of its slice, a thread one output per pass (blockIdx.y and its
// stride: the passes).  A piece's sums (L w and w, with the row's solid angle) are added to the
// slice totals with Kahan compensation.  ROUND: a piece is a whole row of whole segments, so the
// interval is walked round the row's end and every output of a row has the same count of terms.
template <bool ROUND>
__global__ void __launch_bounds__(kIrrThreads) k_irradiance_part(const float4* __restrict__ env, int We,
                                                                 int He, int Wi, int Hi,
                                                                 float4* __restrict__ part) {
  extern __shared__ __align__(16) char s_irr[];
  const IrrShared sh = irr_shared(s_irr, min(We, kIrrPiece));
  const int tid = threadIdx.x, threads = blockDim.x;
  const int per_row = (We + kIrrPiece - 1) / kIrrPiece;
  const long long pieces = (long long)He * per_row;
  const long long p0 = pieces * blockIdx.x / gridDim.x, p1 = pieces * (blockIdx.x + 1) / gridDim.x;
  const int nout = Wi * Hi;
  constexpr int kPer = kIrrSeg / kIrrGroup;
  // Omega of row y = (2 pi / W)(cos(pi y / H) - cos(pi (y + 1) / H))
  //               = (4 pi / W) sin(pi (y + 0.5) / H) sin(pi / (2 H))   (product form)
  const float row_k = 4.0f * kPi / We * sinpif(0.5f / He);
  for (int og = blockIdx.y * threads; og < nout; og += gridDim.y * threads) {
    const int o = og + tid, i = min(o, nout - 1) % Wi, j = min(o, nout - 1) / Wi;
    float st, ct, sp, cp;
    sincospif((j + 0.5f) / Hi, &st, &ct);
    sincospif(2.0f * ((i + 0.5f) / Wi) - 1.0f, &sp, &cp);
    const float X = (i + 0.5f) * ((float)We / (float)Wi) - 0.5f;  // the output's azimuth as a source column
    Kahan acc[4];
    int have = -1;  // the piece of a row whose azimuths are staged
    for (long long p = p0; p < p1; ++p) {
      const int y = (int)(p / per_row), c = (int)(p - (long long)y * per_row);
      const int c0 = c * kIrrPiece, n = min(kIrrPiece, We - c0);
      __syncthreads();
      for (int q = tid; q < n; q += threads) {
        sh.texel[irr_at(q)] = __ldg(env + (long long)y * We + c0 + q);
        if (have != c) {
          float sx, cx;
          sincospif(2.0f * ((c0 + q + 0.5f) / We) - 1.0f, &sx, &cx);
          sh.phi[irr_at(q)] = make_float2(cx, sx);
        }
      }
      have = c;
      __syncthreads();
      for (int g = tid; g < n / kIrrGroup; g += threads) {
        IrrSums q = {};
#pragma unroll
        for (int k = 0; k < kIrrGroup; ++k) {
          // the lanes of a warp start at different texels of their groups: fewer bank conflicts
          const int at = irr_at(g * kIrrGroup + ((k + tid) & (kIrrGroup - 1)));
          const float4 L = sh.texel[at];
          const float2 f = sh.phi[at];
          const float v[3] = {L.x, L.y, L.z};
#pragma unroll
          for (int h = 0; h < 3; ++h) {
            q.t[h] += v[h];
            q.c[h] = fmaf(v[h], f.x, q.c[h]);
            q.s[h] = fmaf(v[h], f.y, q.s[h]);
          }
          q.c1 += f.x;
          q.s1 += f.y;
        }
        sh.group[irr_group_at(g)] = q;
      }
      __syncthreads();
      constexpr int kWords = sizeof(IrrSums) / 4;
      for (int q = tid; q < n / kIrrSeg * kWords; q += threads) {
        const int g = q / kWords, f = q - g * kWords;
        float sum = 0.0f;
#pragma unroll
        for (int k = 0; k < kPer; ++k) sum += ((const float*)&sh.group[irr_group_at(g * kPer + k)])[f];
        ((float*)&sh.seg[g])[f] = sum;
      }
      __syncthreads();
      float sty, cty;
      sincospif((y + 0.5f) / He, &sty, &cty);
      const float omega = row_k * sty;
      const float A = st * sty, B = ct * cty, ac = A * cp, as = A * sp;
      if (!(B > -A)) continue;  // the row lies below the horizon
      // columns lo .. hi (modulo We) hold every texel with n.d > 0, at most a rounding beyond
      int lo = 0, hi = We - 1;
      const bool all = !(B < A);
      if (!all) {
        const float D = acosf(-B / A) * (We * kInv2Pi);
        lo = (int)ceilf(X - D) - 1;
        hi = min((int)floorf(X + D) + 1, lo + We - 1);  // once round: a gap of one column is lo itself
      }
      IrrAcc a;
      auto wrap = [We](int q, int period) { return ROUND && q >= period ? q - period : q; };
      // whole groups strictly inside lo .. hi (not the two columns at either end, whose texels are
      // clamped), whole segments where they fit; columns from .. to - 1 of the piece
      auto interval = [&](int x0, int x1, int i0, int i1) {
        const int g0 = (i0 + kIrrGroup - 1) / kIrrGroup, g1 = max(i1, 0) / kIrrGroup;
        const int s0 = (g0 + kPer - 1) / kPer, s1 = g1 / kPer;
        const bool groups = g0 < g1, segs = groups && s0 < s1;
        // single texels x0 .. e0 - 1 and b1 .. x1 - 1, groups g0 .. h0 - 1 and h1 .. g1 - 1
        const int e0 = groups ? g0 * kIrrGroup : x1, b1 = groups ? g1 * kIrrGroup : x1;
        const int h0 = segs ? s0 * kPer : g1, h1 = segs ? s1 * kPer : g1;
        const int nt = (e0 - x0) + (x1 - b1), ng = groups ? (h0 - g0) + (g1 - h1) : 0, nx = segs ? s1 - s0 : 0;
        for (int k = 0, q = x0; k < nt; ++k, ++q) {
          if (q == e0) q = b1;
          const int at = irr_at(wrap(q, We));
          const float2 f = sh.phi[at];
          const float4 L = sh.texel[at];
          const float w = fmaxf(fmaf(ac, f.x, fmaf(as, f.y, B)), 0.0f);
          a.r = fmaf(L.x, w, a.r);
          a.g = fmaf(L.y, w, a.g);
          a.b = fmaf(L.z, w, a.b);
          a.w += w;
        }
        for (int k = 0, q = g0; k < ng; ++k, ++q) {
          if (q == h0) q = h1;
          irr_add(a, sh.group[irr_group_at(wrap(q, We / kIrrGroup))], ac, as, B, (float)kIrrGroup);
        }
        for (int k = 0; k < nx; ++k) irr_add(a, sh.seg[wrap(s0 + k, We / kIrrSeg)], ac, as, B, (float)kIrrSeg);
      };
      if (ROUND) {
        if (lo < 0) lo += We, hi += We;
        interval(lo, hi + 1, all ? lo : lo + 2, all ? hi + 1 : hi - 1);
      } else {
#pragma unroll 1
        for (int turn = -1; turn <= 1; ++turn) {  // the interval's copies one turn apart
          const int l = lo + turn * We - c0, h = hi + turn * We - c0;
          const int x0 = max(l, 0), x1 = min(h, n - 1) + 1;
          if (x0 < x1) interval(x0, x1, !all && l > -2 ? l + 2 : 0, min(!all && h < n + 1 ? h - 1 : n, n));
        }
      }
      acc[0].add(a.r * omega);
      acc[1].add(a.g * omega);
      acc[2].add(a.b * omega);
      acc[3].add(a.w * omega);
    }
    if (o < nout)
      part[(size_t)blockIdx.x * nout + o] =
          make_float4(acc[0].s - acc[0].c, acc[1].s - acc[1].c, acc[2].s - acc[2].c, acc[3].s - acc[3].c);
  }
  complete_in_order();
}

// Rows of fewer columns than this, unless of whole segments.  32 x 16 outputs by texels / by intervals (us): 16 x 8
// environment 12 / 26, 40 x 20 31 / 66, 64 x 32 37 / 33 (whole segments), 96 x 50 36 / 45, 130 x 65 35 / 39, 250 x 125
// 37 / 27, 37 x 4001 38 / 193.
constexpr int kIrrNarrow = 192;
constexpr int kIrrTexThreads = 128;
constexpr int kIrrOutPerThread = 4;  // outputs per thread and pass (two packed pairs): 512 per pass
constexpr int kIrrTile = 256;        // source texels staged per step

// Narrow environments, whose rows have too few columns for sums of 8 and 64: each block sums over its slice
// of source texels, a thread owns kIrrOutPerThread outputs of a group of 512 (blockIdx.y and its stride) as
// two pairs whose arithmetic runs in packed FP32x2 instructions.
// A source texel is staged once per tile as d Omega (max(n.d, 0) Omega = max(n.(d Omega), 0) since
// Omega > 0) and L, every value duplicated into both halves of a pair: (dx, dx, dy, dy),
// (dz, dz, Lr, Lr), (Lg, Lg, Lb, Lb).  Per tile the four sums of each output (L w and w) are
// plain FP32; the tile's sums are then added to the slice totals with Kahan compensation.
__global__ void __launch_bounds__(kIrrTexThreads) k_irradiance_texels(const float4* __restrict__ env, int We,
                                                                 int He, int Wi, int Hi,
                                                                 float4* __restrict__ part) {
  __shared__ float4 s_src[kIrrTile][3];
  long long ntex = (long long)We * He;
  long long per = (ntex + gridDim.x - 1) / gridDim.x;
  long long t0 = per * blockIdx.x;
  long long t1 = t0 + per < ntex ? t0 + per : ntex;
  int nout = Wi * Hi;
  // Omega of row y = (2 pi / W)(cos(pi y / H) - cos(pi (y + 1) / H))
  //               = (4 pi / W) sin(pi (y + 0.5) / H) sin(pi / (2 H))   (product form)
  float row_k = 4.0f * kPi / We * sinpif(0.5f / He);
  for (int og = blockIdx.y * kIrrTexThreads * kIrrOutPerThread; og < nout;
       og += gridDim.y * kIrrTexThreads * kIrrOutPerThread) {
    // pair p holds outputs og + (2p + h) * kIrrTexThreads + tid, h = 0, 1; an absent output has n = 0
    float2 nx[2], ny[2], nz[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      float3 a, b;
      int oa = og + (2 * p) * kIrrTexThreads + threadIdx.x, ob = oa + kIrrTexThreads;
      a = oa < nout ? texel_dir(oa % Wi, oa / Wi, Wi, Hi) : f3(0, 0, 0);
      b = ob < nout ? texel_dir(ob % Wi, ob / Wi, Wi, Hi) : f3(0, 0, 0);
      nx[p] = make_float2(a.x, b.x), ny[p] = make_float2(a.y, b.y), nz[p] = make_float2(a.z, b.z);
    }
    Kahan acc[kIrrOutPerThread][4];
    for (long long base = t0; base < t1; base += kIrrTile) {
      int cnt = (int)(t1 - base < kIrrTile ? t1 - base : kIrrTile);
      __syncthreads();
      for (int q = threadIdx.x; q < cnt; q += kIrrTexThreads) {
        long long t = base + q;
        int x = (int)(t % We), y = (int)(t / We);
        float3 d = texel_dir(x, y, We, He) * (row_k * sinpif((y + 0.5f) / He));
        float4 L = __ldg(env + t);
        s_src[q][0] = make_float4(d.x, d.x, d.y, d.y);
        s_src[q][1] = make_float4(d.z, d.z, L.x, L.x);
        s_src[q][2] = make_float4(L.y, L.y, L.z, L.z);
      }
      __syncthreads();
      float2 sr[2], sg[2], sb[2], sw[2];
#pragma unroll
      for (int p = 0; p < 2; ++p) sr[p] = sg[p] = sb[p] = sw[p] = make_float2(0.0f, 0.0f);
#pragma unroll 4
      for (int q = 0; q < cnt; ++q) {
        const float4 u = s_src[q][0], v = s_src[q][1], z = s_src[q][2];
        const float2 dx = make_float2(u.x, u.y), dy = make_float2(u.z, u.w), dz = make_float2(v.x, v.y);
        const float2 Lr = make_float2(v.z, v.w), Lg = make_float2(z.x, z.y), Lb = make_float2(z.z, z.w);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          float2 w = __ffma2_rn(nx[p], dx, __ffma2_rn(ny[p], dy, __fmul2_rn(nz[p], dz)));
          w = make_float2(fmaxf(w.x, 0.0f), fmaxf(w.y, 0.0f));
          sr[p] = __ffma2_rn(Lr, w, sr[p]);
          sg[p] = __ffma2_rn(Lg, w, sg[p]);
          sb[p] = __ffma2_rn(Lb, w, sb[p]);
          sw[p] = __fadd2_rn(sw[p], w);
        }
      }
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        acc[2 * p][0].add(sr[p].x), acc[2 * p][1].add(sg[p].x), acc[2 * p][2].add(sb[p].x);
        acc[2 * p][3].add(sw[p].x);
        acc[2 * p + 1][0].add(sr[p].y), acc[2 * p + 1][1].add(sg[p].y), acc[2 * p + 1][2].add(sb[p].y);
        acc[2 * p + 1][3].add(sw[p].y);
      }
    }
#pragma unroll
    for (int r = 0; r < kIrrOutPerThread; ++r) {
      int o = og + r * kIrrTexThreads + threadIdx.x;
      if (o < nout)
        part[(size_t)blockIdx.x * nout + o] =
            make_float4(acc[r][0].s - acc[r][0].c, acc[r][1].s - acc[r][1].c,
                        acc[r][2].s - acc[r][2].c, acc[r][3].s - acc[r][3].c);
    }
  }
  complete_in_order();
}

// One warp per output texel: lane l sums the partials of blocks l, l + 32, ... (Kahan), then the
// lanes' sums are added by a butterfly of shuffles (a fixed order: deterministic).
__global__ void k_irradiance_final(const float4* __restrict__ part, int nblocks, int nout,
                                   float4* __restrict__ out) {
  const int o = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (o >= nout) return;  // warp-uniform
  Kahan s[4];
  for (int b = lane; b < nblocks; b += 32) {
    float4 p = __ldg(part + (size_t)b * nout + o);
    s[0].add(p.x);
    s[1].add(p.y);
    s[2].add(p.z);
    s[3].add(p.w);
  }
  const float r = warp_sum(s[0].s - s[0].c), g = warp_sum(s[1].s - s[1].c);
  const float bl = warp_sum(s[2].s - s[2].c), den = warp_sum(s[3].s - s[3].c);
  if (lane != 0) return;
  float inv = den > 0.0f ? 1.0f / den : 0.0f;  // no texel centre in the hemisphere: 0
  out[o] = make_float4(r * inv, g * inv, bl * inv, 1.0f);
}

// ------------------------------------------------------------------------------------------
// Prefiltered levels 1..M-1
// ------------------------------------------------------------------------------------------
struct ChainDev {
  int M;
  int W[EPBR_MAX_LEVELS], H[EPBR_MAX_LEVELS];
  float4* dst[EPBR_MAX_LEVELS];
};

// With n = v, a GGX half vector h with tangent-space components (sin t cos p, sin t sin p, cos t)
// gives l = 2 (n.h) h - n = T (2 h_z h_x) + B (2 h_z h_y) + n (2 h_z^2 - 1), n.l = 2 h_z^2 - 1:
// functions of the sample and the level only.  The frame (T, B, n) is built from the map's pole
// axis (T = y x n normalised, B = n x T), so it turns with n about that axis: the texels of one
// row of a level share every sample's polar angle, and their sample directions differ only by
// the row's azimuth step.  In the source map (level 0, W0 columns) texel i of a level-m row
// therefore reads each sample at the source coordinate of texel 0 moved right by i * W0 / Wm
// columns.  One block per (level, row): the block computes, once, every kept sample's source
// coordinate for texel 0 (the only equirect mapping in the kernel) and its bilinear weights,
// then every texel of the row sums its samples from the shifted coordinates.  Rows wider than
// kPrefilterSeg texels (shorter ones where there are few rows) are split into segments, one block each.
constexpr int kPrefilterMaxSamples = 2048;
constexpr int kPrefilterThreads = 256;
constexpr int kPrefilterTexels = 2;  // texels per thread: a block shades a segment of up to 512 texels of a row
constexpr int kPrefilterSeg = kPrefilterThreads * kPrefilterTexels;
// Twice the threads and segment, one block per SM, where level 1 has rows of 1024 to 2048 texels (columns shifted
// by whole texels) and the records of a row, now made once or twice, are many: 2048 x 1024, 256 / 512 threads (us): 8
// levels 256, 512, 1024, 2048 samples 544 / 558, 1054 / 1037, 2067 / 2004, 4562 / 3933; 3 levels 1024 samples
// 1623 / 1526; 2048 x 300 920 / 818; but 1024 x 512, 8 levels, 1024 samples 529 / 569 and 8192 x 256, 512
// samples 1181 / 1321.
constexpr int kPrefilterWideMin = 1024, kPrefilterWideMax = 2048, kPrefilterWideSamples = 512;
// Segments are halved down to kPrefilterMinSeg texels until a launch has kPrefilterFill blocks per SM (each
// block makes its row's records anew).  Prefilter (us) with the shortest segment 64, 128, 256 or 512 texels: 2048 x
// 64, 8 levels, 1024 samples 224, 252, 357, 315; 512 x 256, 6 levels, 512 samples 121, 103, 98, 98; 2048 x 1024
// 2083 with each.  With 2, 3, 4 or 8 blocks per SM: 1024 x 512, 8 levels, 1024 samples 524, 524, 566, 654; 750 x
// 375, 6 levels, 512 samples 384, 356, 356, 357.
constexpr int kPrefilterMinSeg = 128, kPrefilterFill = 3;

// Sample `sidx` of N for alpha^2 = a2 as (2 h_z h_x, 2 h_z h_y, n.l, -); kept iff n.l > 0.  Both
// compaction passes call this, so they agree on every decision.
__device__ __forceinline__ float4 prefilter_sample(int sidx, float a2, float invN) {
  float xi2 = hammersley_xi2((unsigned)sidx);
  float inv = 1.0f / fmaf(a2 - 1.0f, xi2, 1.0f);
  float ct = sqrtf((1.0f - xi2) * inv), st = sqrtf(a2 * xi2 * inv);
  float sp, cp;
  sincospif(2.0f * (sidx * invN), &sp, &cp);
  return make_float4(2.0f * ct * st * cp, 2.0f * ct * st * sp, fmaf(2.0f * ct, ct, -1.0f), 0.0f);
}

// Source coordinate of a sample direction l in the level-0 map: x = u W0 - 0.5, y = v H0 - 0.5.
__device__ __forceinline__ float2 prefilter_src_xy(float3 l, int W0, int H0) {
  float u, v;
  dir_to_uv(l, u, v);
  return make_float2(fmaf(u, (float)W0, -0.5f), fmaf(v, (float)H0, -0.5f));
}

// Shared memory of a block that prefilters a row: N float4 weights, N int2, N ushort sorted
// positions; the sort keys (N unsigned) occupy the weights' space until the records are written.
struct PrefilterShared {
  int base[kPrefilterMaxSamples / 32 + 1];
  float wsum[16];
};

// The samples of row j of level m as records in order of source row (a deterministic bitonic sort of
// (source row, sample) keys), by a whole block: `emit(position, sample (.z = n.l), source x, y for texel 0)`
// writes a record.  Returns the number of kept samples and their weight sum sum_k n.l_k (the same for every
// texel of the level).
template <int THREADS, typename Emit>
__device__ __forceinline__ int prefilter_records(PrefilterShared& sh, unsigned* s_key, unsigned short* s_pos, int m,
                                                 int M, int j, int W, int H, int W0, int H0, int N, float& wsum,
                                                 Emit emit) {
  const float r = (float)m / (float)(M - 1);
  const float a2 = r * r * r * r;
  const float invN = 1.0f / N;
  const int groups = (N + 31) / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // kept samples per group of 32, then an exclusive prefix over the groups (sample order)
  for (int gi = warp; gi < groups; gi += THREADS / 32) {
    int sidx = gi * 32 + lane;
    bool keep = sidx < N && prefilter_sample(sidx, a2, invN).z > 0.0f;
    unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) sh.base[gi] = __popc(bal);
  }
  __syncthreads();
  if (tid == 0) {
    int acc = 0;
    for (int gi = 0; gi < groups; ++gi) {
      int c = sh.base[gi];
      sh.base[gi] = acc;
      acc += c;
    }
    sh.base[groups] = acc;
  }
  __syncthreads();
  const int ns = sh.base[groups];
  // the frame of texel 0 of the row: n, T = y x n / |y x n| = (-cos phi0, 0, -sin phi0), B = n x T
  const float3 n = texel_dir(0, j, W, H);
  float sp0, cp0;
  sincospif(2.0f * (0.5f / W) - 1.0f, &sp0, &cp0);
  const float3 T = f3(-cp0, 0.0f, -sp0);
  const float3 B = cross3(n, T);
  // pass A: each kept sample's source row, as a sort key
  for (int gi = warp; gi < groups; gi += THREADS / 32) {
    int sidx = gi * 32 + lane;
    float4 e = sidx < N ? prefilter_sample(sidx, a2, invN) : make_float4(0, 0, 0, 0);
    bool keep = sidx < N && e.z > 0.0f;
    unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (keep) {
      const int q = sh.base[gi] + __popc(bal & ((1u << lane) - 1u));
      const float2 xy = prefilter_src_xy(T * e.x + B * e.y + n * e.z, W0, H0);
      const int iy = min(max((int)floorf(xy.y), 0), H0 - 1);
      s_key[q] = ((unsigned)iy << 16) | (unsigned)q;
    }
  }
  int P = 1;
  while (P < ns) P <<= 1;
  for (int q = ns + tid; q < P; q += THREADS) s_key[q] = 0xffffffffu;
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1) {
    for (int jj = k >> 1; jj > 0; jj >>= 1) {
      for (int q = tid; q < P; q += THREADS) {
        const int o = q ^ jj;
        if (o > q) {
          const unsigned a = s_key[q], b = s_key[o];
          if ((a > b) == ((q & k) == 0)) {
            s_key[q] = b;
            s_key[o] = a;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int q = tid; q < ns; q += THREADS) s_pos[s_key[q] & 0xffffu] = (unsigned short)q;
  __syncthreads();  // the keys are dead from here: their space takes the records
  // pass B: the records at their sorted positions; the weights summed in sample order
  float wpart = 0.0f;
  for (int gi = warp; gi < groups; gi += THREADS / 32) {
    int sidx = gi * 32 + lane;
    float4 e = sidx < N ? prefilter_sample(sidx, a2, invN) : make_float4(0, 0, 0, 0);
    bool keep = sidx < N && e.z > 0.0f;
    unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (keep) {
      const int q = sh.base[gi] + __popc(bal & ((1u << lane) - 1u));
      emit(s_pos[q], e, prefilter_src_xy(T * e.x + B * e.y + n * e.z, W0, H0));
      wpart += e.z;
    }
  }
  wpart = warp_sum(wpart);
  if (lane == 0) sh.wsum[warp] = wpart;
  __syncthreads();
  wsum = 0.0f;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) wsum += sh.wsum[w];
  return ns;
}

// Per kept sample, for texel 0 of the row, in order of source row: INT_SHIFT (W0 a multiple of
// Wm) stores the four bilinear weights times n.l and (column, row); otherwise the two row weights
// times n.l and the source x coordinate (the column fraction then varies along the row), and the
// row.  Samples are visited in order of their source row so that consecutive samples read the
// same two rows, which stay in L1.  A plain FP32 sum takes 64 samples, compensated sums take the
// plain ones and the shares.
template <bool INT_SHIFT, int THREADS>
__device__ __forceinline__ void prefilter_segment(const MapDev& src, const ChainDev& ch, int N, int seg) {
  extern __shared__ __align__(16) float4 s_pf[];
  __shared__ PrefilterShared sh;
  __shared__ float3 s_sum[THREADS * 2];  // the shares' sums
  float4* s_w = s_pf;
  int2* s_xy = (int2*)(s_pf + N);
  unsigned short* s_pos = (unsigned short*)(s_xy + N);
  const int m = blockIdx.y + 1;
  const int W = ch.W[m], H = ch.H[m];
  const int segs = (W + seg - 1) / seg;
  const int j = blockIdx.x / segs, i0 = (blockIdx.x - j * segs) * seg;
  if (j >= H) return;  // block-uniform
  const int W0 = src.W, H0 = src.H;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float wsum;
  const int ns = prefilter_records<THREADS>(
      sh, (unsigned*)s_pf, s_pos, m, ch.M, j, W, H, W0, H0, N, wsum,
      [&](int p, float4 e, float2 xy) {
        const float xf = floorf(xy.x), yf = floorf(xy.y);
        const float fx = xy.x - xf, fy = xy.y - yf;
        const float wt = e.z * (1.0f - fy), wb = e.z * fy;
        if (INT_SHIFT)
          s_w[p] = make_float4(wt * (1.0f - fx), wt * fx, wb * (1.0f - fx), wb * fx);
        else
          s_w[p] = make_float4(wt, wb, xy.x, 0.0f);
        s_xy[p] = make_int2((int)xf, (int)yf);
      });
  const float inv = 1.0f / wsum;
  const int step_i = W0 / W;  // INT_SHIFT: whole source columns per texel
  const float step_f = (float)W0 / (float)W;
  if (INT_SHIFT) {
    // Lanes by tap column: lane l of warp w serves output texels i = i0 + 64 w + 16 g + (l >> 1),
    // g = 0..3, with the tap column d = l & 1 (columns x0 + s i + d), so a warp's loads of one
    // row and group are 32 consecutive texels at level 1 (s = 2); the two lanes of a texel add
    // their sums at the end.
    // A segment of at most 256 texels leaves warps over: these take shares of the samples (`split`).
    const int cols = (min(W - i0, seg) + 63) / 64;  // warps side by side
    const int across = cols > 8 ? 16 : (cols > 4 ? 8 : (cols > 2 ? 4 : cols));
    const int split = warp / across, splits = THREADS / 32 / across;
    const int t = lane >> 1, dl = lane & 1;
    const int wbase = i0 + (warp - split * across) * 64;
    int col[4];
    bool ong[4];
    Kahan3 acc[4];
    float3 part[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int i = wbase + 16 * g + t;
      ong[g] = wbase + 16 * g < W;  // warp-uniform: whether group g has texels
      col[g] = min(i, W - 1) * step_i + dl;
      part[g] = f3(0, 0, 0);
    }
    // WHOLE: all samples in turn, the usual case, whose loop a stride known only at run time slows down (1000 x
    // 500, 3 levels, 128 samples: 121 us instead of 83)
    auto sum = [&](auto whole) {
      constexpr bool WHOLE = decltype(whole)::value;
      int since = 0;
#pragma unroll 2
      for (int q = WHOLE ? 0 : split; q < ns; q += WHOLE ? 1 : splits) {
        const float4 w = s_w[q];
        const int2 xy = s_xy[q];
        const int r0 = max(xy.y, 0) * W0, r1 = min(xy.y + 1, H0 - 1) * W0;
        const float wa = dl ? w.y : w.x, wb = dl ? w.w : w.z;  // this column's weights in rows r0, r1
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (!ong[g]) continue;
          int c = xy.x + col[g];  // in [-1, 2 W0 - 1)
          c = c < 0 ? c + W0 : (c >= W0 ? c - W0 : c);
          const float4 a = __ldg(src.texels + (r0 + c)), p = __ldg(src.texels + (r1 + c));
          part[g].x = fmaf(wa, a.x, fmaf(wb, p.x, part[g].x));
          part[g].y = fmaf(wa, a.y, fmaf(wb, p.y, part[g].y));
          part[g].z = fmaf(wa, a.z, fmaf(wb, p.z, part[g].z));
        }
        if (WHOLE ? (q & 63) == 63 : (++since & 63) == 0) {  // fold every 64 samples' plain sums into the running sums
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            acc[g].add(part[g]);
            part[g] = f3(0, 0, 0);
          }
        }
      }
    };
    if (splits == 1) {
      if (!ong[0]) return;  // warp-uniform, after the last barrier
      sum(std::true_type());
    } else if (ong[0]) {
      sum(std::false_type());
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      acc[g].add(part[g]);
      float3 v = acc[g].value();
      v.x += __shfl_xor_sync(0xffffffffu, v.x, 1);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, 1);
      v.z += __shfl_xor_sync(0xffffffffu, v.z, 1);
      part[g] = v;
      if (splits > 1 && dl == 0) s_sum[warp * 64 + 16 * g + t] = v;
    }
    if (splits > 1) __syncthreads();  // block-uniform
    if (split > 0) return;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int i = wbase + 16 * g + t;
      if (dl || !ong[g] || i >= W) continue;
      Kahan3 v;
      v.add(part[g]);
      for (int k = 1; k < splits; ++k) v.add(s_sum[(warp + k * across) * 64 + 16 * g + t]);
      const float3 o = v.value() * inv;
      ch.dst[m][(long long)j * W + i] = make_float4(o.x, o.y, o.z, 1.0f);
    }
    return;
  }
  // a thread per texel, or per texel and share of the samples where the segment has at most 128
  const int n = min(W - i0, seg);
  const int across = n > 128 ? THREADS : (n > 64 ? 128 : (n > 32 ? 64 : 32)), split = tid / across;
  const int splits = THREADS / across, me = tid - split * across;
  int ii[kPrefilterTexels];
  bool on[kPrefilterTexels];  // block-uniform: whether the segment has a texel group c
  Kahan3 acc[kPrefilterTexels];
  float3 part[kPrefilterTexels];
#pragma unroll
  for (int c = 0; c < kPrefilterTexels; ++c) {
    on[c] = c * THREADS < n;
    ii[c] = min(i0 + c * THREADS + me, W - 1);  // duplicates of the last texel are not stored
    part[c] = f3(0, 0, 0);
  }
  auto sum = [&](auto whole) {
    constexpr bool WHOLE = decltype(whole)::value;
    int since = 0;
#pragma unroll 2
    for (int q = WHOLE ? 0 : split; q < ns; q += WHOLE ? 1 : splits) {
      const float4 w = s_w[q];
      const int2 xy = s_xy[q];
      const int r0 = max(xy.y, 0) * W0, r1 = min(xy.y + 1, H0 - 1) * W0;
#pragma unroll
      for (int c = 0; c < kPrefilterTexels; ++c) {
        if (!on[c]) continue;
        const float x = fmaf((float)ii[c], step_f, w.z);
        const float xf = floorf(x), fx = x - xf;
        int x0 = (int)xf;
        const float4 wq = make_float4(w.x * (1.0f - fx), w.x * fx, w.y * (1.0f - fx), w.y * fx);
        x0 = x0 < 0 ? x0 + W0 : (x0 >= W0 ? x0 - W0 : x0);
        const int x1 = x0 + 1 == W0 ? 0 : x0 + 1;
        const float4 a = __ldg(src.texels + (r0 + x0)), b = __ldg(src.texels + (r0 + x1));
        const float4 p = __ldg(src.texels + (r1 + x0)), d = __ldg(src.texels + (r1 + x1));
        part[c].x = fmaf(wq.x, a.x, fmaf(wq.y, b.x, fmaf(wq.z, p.x, fmaf(wq.w, d.x, part[c].x))));
        part[c].y = fmaf(wq.x, a.y, fmaf(wq.y, b.y, fmaf(wq.z, p.y, fmaf(wq.w, d.y, part[c].y))));
        part[c].z = fmaf(wq.x, a.z, fmaf(wq.y, b.z, fmaf(wq.z, p.z, fmaf(wq.w, d.z, part[c].z))));
      }
      if (WHOLE ? (q & 63) == 63 : (++since & 63) == 0) {  // fold every 64 samples' plain sums into the running sums
#pragma unroll
        for (int c = 0; c < kPrefilterTexels; ++c) {
          acc[c].add(part[c]);
          part[c] = f3(0, 0, 0);
        }
      }
    }
  };
  if (splits == 1)
    sum(std::true_type());
  else
    sum(std::false_type());
  if (splits > 1) {  // block-uniform
    acc[0].add(part[0]);
    part[0] = f3(0, 0, 0);
    s_sum[tid] = acc[0].value();
    __syncthreads();
    if (split > 0) return;
  }
#pragma unroll
  for (int c = 0; c < kPrefilterTexels; ++c) {
    const int i = i0 + c * THREADS + me;
    if (on[c] && i < W) {
      Kahan3 v = acc[c];
      v.add(part[c]);
      for (int k = 1; k < splits; ++k) v.add(s_sum[me + k * across]);
      const float3 o = v.value() * inv;
      ch.dst[m][(long long)j * W + i] = make_float4(o.x, o.y, o.z, 1.0f);
    }
  }
}

// Bound by L1 (16 bytes per tap, of which 12 are used) and its latency: two blocks per SM with up to 128 registers,
// so that the loads of two samples are under way, take 2083 us for the levels of a 2048 x 1024 environment (8
// levels, 1024 samples), three blocks 2202 us; 1024 x 512, 3 levels, 128 samples 76 and 92 us.  Source rows
// staged in shared memory for levels 1 and 2 took 2020 us for the first and 229 us for the second: a row is
// staged for too few samples unless the lobe is narrow and the count high.
template <bool INT_SHIFT, int THREADS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS)
    k_prefilter(const __grid_constant__ MapDev src, const __grid_constant__ ChainDev ch, int N, int seg) {
  griddep_launch_dependents();
  prefilter_segment<INT_SHIFT, THREADS>(src, ch, N, seg);
  complete_in_order();
}

// Level 0.
__global__ void __launch_bounds__(256) k_copy_texels(const float4* src, float4* dst, long long n, bool more) {
  if (more) griddep_launch_dependents();
  for (long long k = blockIdx.x * 256LL + threadIdx.x; k < n; k += gridDim.x * 256LL) dst[k] = src[k];
  complete_in_order();
}

static epbr_status validate_ibl_for(const epbr_ibl* ibl, int We, int He) {
  if (!ibl) return fail(EPBR_ERR_INVALID_ARG, "ibl is NULL");
  if (ibl->num_levels < 1 || ibl->num_levels > EPBR_MAX_LEVELS)
    return fail(EPBR_ERR_INVALID_ARG, "ibl->num_levels %d invalid", ibl->num_levels);
  for (int m = 0; m < ibl->num_levels; ++m) {
    int w = std::max(1, We >> m), h = std::max(1, He >> m);
    if (!ibl->level[m] || ibl->level_width[m] != w || ibl->level_height[m] != h)
      return fail(EPBR_ERR_INVALID_ARG, "ibl level %d does not match the env (%dx%d expected)", m, w, h);
    if ((uintptr_t)ibl->level[m] % 16) return fail(EPBR_ERR_INVALID_ARG, "ibl level %d not 16-byte aligned", m);
  }
  return EPBR_OK;
}

}  // namespace epbr

using namespace epbr;

namespace epbr {

// Each step of a lighting set is checked, then launched; `early` says whether the kernel before it on
// the stream is another one of these, `more` whether one follows in the same call.
static epbr_status validate_lut(int S, int N, const float* lut) {
  if (S < 1 || S > 4096 || N < 1 || N > (1 << 24) || !lut)
    return fail(EPBR_ERR_INVALID_ARG, "brdf_lut: size %d / samples %d / pointer invalid", S, N);
  if ((uintptr_t)lut % 8) return fail(EPBR_ERR_INVALID_ARG, "brdf_lut: lut not 8-byte aligned");
  return EPBR_OK;
}

static epbr_status launched(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return check_launch(what);
  cudaGetLastError();
  return fail(EPBR_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// Raises kernel k's limit of dynamic shared memory to `most` bytes, the most that any call needs and
// never one call's own need: the limit belongs to the function, so a smaller value set by another
// thread between this thread's setting and its launch would refuse the launch.
template <typename K>
static epbr_status allow_shared(K* k, size_t most, const char* what) {
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess)
    return fail(EPBR_ERR_CUDA, "%s: shared-memory attribute: %s", what, cudaGetErrorString(cudaGetLastError()));
  return EPBR_OK;
}

static epbr_status launch_lut(int S, int N, float* lut, cudaStream_t s, bool early, bool more) {
  const long long threads = (long long)S * S * 32;
  return launched(launch_kernel(k_brdf_lut, dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, s, early, S, N, (float2*)lut,
                                more),
                  "k_brdf_lut");
}

}  // namespace epbr

extern "C" epbr_status epbr_brdf_lut(int32_t S, int32_t N, float* lut, void* stream) {
  epbr_status st = validate_lut(S, N, lut);
  if (st || (st = launch_lut(S, N, lut, (cudaStream_t)stream, false, false))) return st;
  return ok();
}

extern "C" epbr_status epbr_precompute_ibl_workspace_size(const epbr_ibl_params* p, int32_t We,
                                                          int32_t He, size_t* bytes) {
  if (!p || !bytes) return fail(EPBR_ERR_INVALID_ARG, "params or bytes is NULL");
  if (We < 1 || He < 1 || p->irr_width < 1 || p->irr_height < 1)
    return fail(EPBR_ERR_INVALID_ARG, "sizes must be positive");
  *bytes = irr_workspace_bytes(We, He, p->irr_width, p->irr_height);
  return ok();
}

namespace epbr {

// Partial sums into `ws` (at least irr_workspace_bytes), then the outputs.
static epbr_status launch_irradiance(const epbr_env* env, int Wi, int Hi, float4* ws, float4* out, cudaStream_t s,
                                     bool early) {
  const int We = env->width, He = env->height, nout = Wi * Hi;
  epbr_status st;
  int nb;
  const bool round = We <= kIrrPiece && We % kIrrSeg == 0;
  if (!round && We < kIrrNarrow) {
    nb = irr_blocks(We, He);
    const int groups = (nout + kIrrTexThreads * kIrrOutPerThread - 1) / (kIrrTexThreads * kIrrOutPerThread);
    const int gy = (int)std::min<long long>(groups, std::max<long long>(1, 8LL * num_sms() / nb));
    if ((st = launched(launch_kernel(k_irradiance_texels, dim3(nb, gy), dim3(kIrrTexThreads), 0, s, early,
                                     (const float4*)env->texels, We, He, Wi, Hi, ws),
                       "k_irradiance_texels")))
      return st;
  } else {
    // slices of whole row pieces, as even as the three blocks an SM holds allow
    const long long pieces = (long long)He * ((We + kIrrPiece - 1) / kIrrPiece), room = 3LL * num_sms();
    const long long each = (pieces + room - 1) / room;
    nb = (int)std::min<long long>(irr_blocks(We, He), (pieces + each - 1) / each);
    // few slices (a small environment): smaller blocks, several per slice
    const int threads = nb >= num_sms() ? kIrrThreads : 128, passes = (nout + threads - 1) / threads;
    const int gy = (int)std::min<long long>(std::min(passes, 65535), std::max<long long>(1, room / nb));
    const size_t smem = irr_shared(nullptr, std::min(We, kIrrPiece)).bytes;
    void (*k)(const float4*, int, int, int, int, float4*) = round ? k_irradiance_part<true> : k_irradiance_part<false>;
    if ((st = allow_shared(k, irr_shared(nullptr, kIrrPiece).bytes, "irradiance"))) return st;
    if ((st = launched(launch_kernel(k, dim3(nb, gy), dim3(threads), smem, s, early, (const float4*)env->texels, We, He,
                                     Wi, Hi, ws),
                       "k_irradiance_part")))
      return st;
  }
  k_irradiance_final<<<(unsigned)(((long long)nout * 32 + 255) / 256), 256, 0, s>>>(ws, nb, nout, out);
  return check_launch("k_irradiance_final");
}

}  // namespace epbr

namespace epbr {

static epbr_status validate_irradiance(const epbr_env* env, int Wi, int Hi, const float* out, const void* ws,
                                       size_t ws_bytes) {
  epbr_status st = validate_env(env);
  if (st) return st;
  if (Wi < 1 || Hi < 1 || Wi > 4096 || Hi > 4096 || !out)
    return fail(EPBR_ERR_INVALID_ARG, "irradiance: output %dx%d or pointer invalid", Wi, Hi);
  if ((uintptr_t)out % 16) return fail(EPBR_ERR_INVALID_ARG, "irradiance: out not 16-byte aligned");
  const size_t need = irr_workspace_bytes(env->width, env->height, Wi, Hi);
  if (!ws || ws_bytes < need || (uintptr_t)ws % 16)
    return fail(EPBR_ERR_NO_MEMORY, "irradiance: workspace needs %zu bytes (16-byte aligned), got %zu", need,
                ws ? ws_bytes : (size_t)0);
  return EPBR_OK;
}

}  // namespace epbr

extern "C" epbr_status epbr_irradiance(const epbr_env* env, int32_t Wi, int32_t Hi, float* out,
                                       void* ws, size_t ws_bytes, void* stream) {
  epbr_status st = validate_irradiance(env, Wi, Hi, out, ws, ws_bytes);
  if (st || (st = launch_irradiance(env, Wi, Hi, (float4*)ws, (float4*)out, (cudaStream_t)stream, false))) return st;
  return ok();
}

// ------------------------------------------------------------------------------------------
// Irradiance for callers that cannot allocate: the per-block partial sums go to a fixed,
// library-owned device array instead of caller workspace.
// ------------------------------------------------------------------------------------------
namespace epbr {

constexpr size_t kStaticScratchBytes = (size_t)8 << 20;  // 8 MiB: 32x16 outputs over 608 blocks need 4.75 MiB
static __device__ __align__(256) float4 g_irr_scratch[kStaticScratchBytes / sizeof(float4)];

constexpr int kMaxDevices = 64;

// The array's device address is per context: a caller may run its own driver context on a
// device instead of the primary one, and a device reset gives the device a new primary context
// (with the array loaded afresh).  The cache therefore keeps, per device, the unique id of the
// context the address was looked up in (cuCtxGetId, never reused within a process) and looks
// the address up again when the current context is another one.
struct ScratchSlot {
  unsigned long long ctx_id;
  void* addr;
};
static std::mutex g_scratch_mutex;
static ScratchSlot g_scratch_slot[kMaxDevices];

typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

template <typename Fn>
static Fn driver_fn(const char* name) {
  void* f = nullptr;
  cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
  if (cudaGetDriverEntryPointByVersion(name, &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    return nullptr;
  return (Fn)f;
}

// Unique id of the calling thread's current context (0 and false when there is none).
static bool current_ctx_id(unsigned long long* id) {
  static const CtxGetCurrentFn get_cur = driver_fn<CtxGetCurrentFn>("cuCtxGetCurrent");
  static const CtxGetIdFn get_id = driver_fn<CtxGetIdFn>("cuCtxGetId");
  CUcontext ctx = nullptr;
  if (!get_cur || !get_id || get_cur(&ctx) != CUDA_SUCCESS || !ctx) return false;
  return get_id(ctx, id) == CUDA_SUCCESS;
}

// Device address of g_irr_scratch in the current context.  In host code the name g_irr_scratch
// is only a host-side handle, so the address is asked from the runtime (with the device current)
// once per device and context and cached.
static epbr_status static_scratch(void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(EPBR_ERR_CUDA, "irradiance_noalloc: cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return fail(EPBR_ERR_UNSUPPORTED, "irradiance_noalloc: device %d", dev);
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  unsigned long long id = 0;
  bool have_id = current_ctx_id(&id);
  ScratchSlot& slot = g_scratch_slot[dev];
  if (!have_id || !slot.addr || slot.ctx_id != id) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_irr_scratch);  // also makes the primary context current if none is
    if (e != cudaSuccess || !p)
      return fail(EPBR_ERR_CUDA, "irradiance_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
    if (!have_id && !current_ctx_id(&id))
      return fail(EPBR_ERR_CUDA, "irradiance_noalloc: no current context after the symbol lookup");
    slot.ctx_id = id;
    slot.addr = p;
  }
  *out = slot.addr;
  return EPBR_OK;
}

}  // namespace epbr

extern "C" epbr_status epbr_irradiance_noalloc(const epbr_env* env, int32_t Wi, int32_t Hi, float* out,
                                               void* stream) {
  epbr_status st = validate_env(env);
  if (st) return st;
  if (Wi < 1 || Hi < 1 || Wi > 4096 || Hi > 4096 || !out)
    return fail(EPBR_ERR_INVALID_ARG, "irradiance_noalloc: output %dx%d or pointer invalid", Wi, Hi);
  if ((uintptr_t)out % 16) return fail(EPBR_ERR_INVALID_ARG, "irradiance_noalloc: out not 16-byte aligned");
  size_t need = irr_workspace_bytes(env->width, env->height, Wi, Hi);
  if (need > kStaticScratchBytes)
    return fail(EPBR_ERR_INVALID_ARG,
                "irradiance_noalloc: a %dx%d map over a %dx%d environment needs %zu bytes of scratch; the "
                "static scratch holds %zu (use epbr_irradiance with a workspace)",
                Wi, Hi, env->width, env->height, need, kStaticScratchBytes);
  void* ws = nullptr;
  if ((st = static_scratch(&ws))) return st;
  // Every partial the final pass reads is written by the first pass, so the scratch needs no
  // clearing between calls.
  if ((st = launch_irradiance(env, Wi, Hi, (float4*)ws, (float4*)out, (cudaStream_t)stream, false))) return st;
  return ok();
}

namespace epbr {

static epbr_status validate_prefilter(const epbr_env* env, int N, const epbr_ibl* ibl) {
  epbr_status st = validate_env(env);
  if (st) return st;
  if ((st = validate_ibl_for(ibl, env->width, env->height))) return st;
  if (N < 1 || N > kPrefilterMaxSamples)
    return fail(EPBR_ERR_INVALID_ARG, "prefilter: samples %d outside [1, %d]", N, kPrefilterMaxSamples);
  return EPBR_OK;
}

// The levels, then level 0.
static epbr_status launch_prefilter(const epbr_env* env, int N, const epbr_ibl* ibl, cudaStream_t s, bool more) {
  ChainDev ch;
  ch.M = ibl->num_levels;
  for (int m = 0; m < EPBR_MAX_LEVELS; ++m) {
    ch.W[m] = ibl->level_width[m];
    ch.H[m] = ibl->level_height[m];
    ch.dst[m] = (float4*)ibl->level[m];
  }
  const int W0 = env->width, H0 = env->height;
  MapDev src{(const float4*)env->texels, W0, H0};
  epbr_status st;
  bool early = false;
  // a block per segment of a row (level 1 has the most); whole-column shifts when every level's width
  // divides the source width
  if (ch.M > 1) {
    bool int_shift = true;
    for (int m = 1; m < ch.M; ++m) int_shift = int_shift && W0 % ch.W[m] == 0;
    const bool wide = int_shift && ch.W[1] >= kPrefilterWideMin && ch.W[1] <= kPrefilterWideMax && N >= kPrefilterWideSamples;
    int seg = wide ? 2 * kPrefilterSeg : kPrefilterSeg;
    unsigned most = 0;
    for (;; seg /= 2) {
      long long blocks = 0;
      most = 0;
      for (int m = 1; m < ch.M; ++m) {
        const unsigned b = (unsigned)(ch.H[m] * ((ch.W[m] + seg - 1) / seg));
        blocks += b;
        most = std::max(most, b);
      }
      if (seg <= kPrefilterMinSeg || blocks >= (long long)kPrefilterFill * num_sms()) break;
    }
    constexpr size_t kSampleBytes = sizeof(float4) + sizeof(int2) + sizeof(unsigned short);
    const size_t smem = (size_t)N * kSampleBytes;
    void (*k)(const MapDev, const ChainDev, int, int) = wide ? k_prefilter<true, 512> : (int_shift ? k_prefilter<true, 256> : k_prefilter<false, 256>);
    // for every count: without it the 48 KB limit also covers the kernel's static 6.3 KB
    if ((st = allow_shared(k, kPrefilterMaxSamples * kSampleBytes, "prefilter"))) return st;
    // a small shared-memory carve-out leaves most of the SM's 256 KB to L1, which holds the source rows the
    // resident blocks read (two rows of up to 16 KB per block); 40% (100 KB) holds two blocks of up to 1600
    // samples, 58% (132 KB) two of any count: levels of a 2048 x 1024 environment at 50% 2101 us, at 40% 2060,
    // at 25% (one block) 2321
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, !wide && N > 1600 ? 58 : 40);  // a hint; failure is harmless
    if ((st = launched(launch_kernel(k, dim3(most, (unsigned)(ch.M - 1)), dim3(wide ? 512 : 256), smem, s, early, src,
                                     ch, N, seg),
                       "k_prefilter")))
      return st;
    early = true;
  }
  return launched(launch_kernel(k_copy_texels, dim3(num_sms() * 4), dim3(256), 0, s, early, src.texels, ch.dst[0],
                                (long long)W0 * H0, more),
                  "k_copy_texels");
}

}  // namespace epbr

extern "C" epbr_status epbr_prefilter(const epbr_env* env, int32_t N, const epbr_ibl* ibl, void* stream) {
  epbr_status st = validate_prefilter(env, N, ibl);
  if (st || (st = launch_prefilter(env, N, ibl, (cudaStream_t)stream, false))) return st;
  return ok();
}

extern "C" epbr_status epbr_precompute_ibl(const epbr_env* env, const epbr_ibl_params* p, const epbr_ibl* ibl,
                                           void* ws, size_t ws_bytes, void* stream) {
  epbr_status st = validate_env(env);
  if (st) return st;
  if (!p) return fail(EPBR_ERR_INVALID_ARG, "params is NULL");
  if ((st = validate_ibl_for(ibl, env->width, env->height))) return st;
  if (ibl->num_levels != p->num_levels || ibl->lut_size != p->lut_size || ibl->irr_width != p->irr_width ||
      ibl->irr_height != p->irr_height || !ibl->lut || !ibl->irradiance)
    return fail(EPBR_ERR_INVALID_ARG, "ibl layout does not match params");
  if ((st = validate_lut(p->lut_size, p->lut_samples, ibl->lut))) return st;
  if ((st = validate_irradiance(env, p->irr_width, p->irr_height, ibl->irradiance, ws, ws_bytes))) return st;
  if ((st = validate_prefilter(env, p->prefilter_samples, ibl))) return st;
  cudaStream_t s = (cudaStream_t)stream;
  // the longest first, each of the others beginning as the blocks of those before run out
  if ((st = launch_prefilter(env, p->prefilter_samples, ibl, s, true))) return st;
  if ((st = launch_lut(p->lut_size, p->lut_samples, ibl->lut, s, true, true))) return st;
  if ((st = launch_irradiance(env, p->irr_width, p->irr_height, (float4*)ws, (float4*)ibl->irradiance, s, true))) return st;
  return ok();
}
