// Image-based lighting precompute (paper Sec. 3.1; split sum of Karis 2013):
//   k_brdf_lut          BRDF integration table (A, B), one warp per texel, Kahan + shuffles
//   k_irradiance_part   exact-quadrature irradiance, per-block partial sums over a slice of source
//                       row pieces: a row's hemisphere is one interval of columns, summed from
//                       sums of 64 and 8 texels and single texels at its ends (Kahan across pieces)
//   k_irradiance_final  one warp per output: lanes sum the block partials, a shuffle butterfly
//                       adds the lanes (fixed order: deterministic), then the ratio
//   k_prefilter_rows    GGX-prefiltered levels 1 and 2 of the usual maps, one block per row of a level:
//                       the row's sample geometry computed once (the sampling frame turns with the
//                       texel about the pole axis), each texel sums its samples at shifted columns of
//                       source rows staged in shared memory
//   k_prefilter         the other levels, source rows read through L1
#include <cuda.h>  // CUcontext and CUresult for the context queries (fetched at run time)

#include <algorithm>
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
// Set of a 2048 x 1024 environment, one after another 2143 us, overlapped 1986 us.
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

// Bound by issue (the terms of every output and row): 39 us for a 2048 x 1024 environment, 319 us
// when every output summed every source texel in packed FP32x2 arithmetic (62% of the FMA pipe).
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
  int first;  // the first level a launch writes
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
// Segments are halved down to kPrefilterMinSeg texels until a launch has kPrefilterFill blocks per SM (each
// block makes its row's records anew).  Lighting set of a 2048 x 1024 environment, levels 3 .. 7 here, the
// shortest segment 64, 128, 256 or 512 texels: 1998, 1986, 2365, 2366 us.
constexpr int kPrefilterMinSeg = 128, kPrefilterFill = 4;

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
// (source row + 1, sample) keys), by a block of THREADS threads.  `keyed(keys, ns)` sees the sorted
// keys, `emit(position, sample (.z = n.l), source x, y for texel 0)` writes a record.  Returns the
// number of kept samples and their weight sum sum_k n.l_k (the same for every texel of the level).
template <int THREADS, typename Keyed, typename Emit>
__device__ __forceinline__ int prefilter_records(PrefilterShared& sh, unsigned* s_key, unsigned short* s_pos, int m,
                                                 int M, int j, int W, int H, int W0, int H0, int N, float& wsum,
                                                 Keyed keyed, Emit emit) {
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
      const int iy = min(max((int)floorf(xy.y), -1), H0 - 1) + 1;
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
  keyed(s_key, ns);
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
// same two rows, which stay in L1.
template <bool INT_SHIFT>
__device__ __forceinline__ void prefilter_segment(const MapDev& src, const ChainDev& ch, int N, int seg) {
  extern __shared__ __align__(16) float4 s_pf[];
  __shared__ PrefilterShared sh;
  __shared__ float3 s_sum[kPrefilterThreads * 2];  // the shares' sums
  float4* s_w = s_pf;
  int2* s_xy = (int2*)(s_pf + N);
  unsigned short* s_pos = (unsigned short*)(s_xy + N);
  const int m = blockIdx.y + ch.first;
  const int W = ch.W[m], H = ch.H[m];
  const int segs = (W + seg - 1) / seg;
  const int j = blockIdx.x / segs, i0 = (blockIdx.x - j * segs) * seg;
  if (j >= H) return;  // block-uniform
  const int W0 = src.W, H0 = src.H;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float wsum;
  const int ns = prefilter_records<kPrefilterThreads>(
      sh, (unsigned*)s_pf, s_pos, m, ch.M, j, W, H, W0, H0, N, wsum, [](const unsigned*, int) {},
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
    const int across = cols > 4 ? 8 : (cols > 2 ? 4 : cols), split = warp / across, splits = 8 / across;
    const int t = lane >> 1, dl = lane & 1;
    const int wbase = i0 + (warp - split * across) * 64;
    int col[4];
    bool ong[4];
    float3 acc[4], part[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int i = wbase + 16 * g + t;
      ong[g] = wbase + 16 * g < W;  // warp-uniform: whether group g has texels
      col[g] = min(i, W - 1) * step_i + dl;
      acc[g] = part[g] = f3(0, 0, 0);
    }
    int since = 0;
#pragma unroll 2
    for (int q = split; q < (ong[0] ? ns : 0); q += splits) {
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
      if ((++since & 63) == 0) {  // fold every 64 samples' plain sums into the running sums
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          acc[g] = acc[g] + part[g];
          part[g] = f3(0, 0, 0);
        }
      }
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      float3 v = acc[g] + part[g];
      v.x += __shfl_xor_sync(0xffffffffu, v.x, 1);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, 1);
      v.z += __shfl_xor_sync(0xffffffffu, v.z, 1);
      acc[g] = v;
      if (splits > 1 && dl == 0) s_sum[warp * 64 + 16 * g + t] = v;
    }
    if (splits > 1) __syncthreads();  // block-uniform
    if (split > 0) return;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int i = wbase + 16 * g + t;
      if (dl || !ong[g] || i >= W) continue;
      Kahan3 v;
      v.add(acc[g]);
      for (int k = 1; k < splits; ++k) v.add(s_sum[(warp + k * across) * 64 + 16 * g + t]);
      const float3 o = v.value() * inv;
      ch.dst[m][(long long)j * W + i] = make_float4(o.x, o.y, o.z, 1.0f);
    }
    return;
  }
  // a thread per texel, or per texel and share of the samples where the segment has at most 128
  const int n = min(W - i0, seg);
  const int across = n > 128 ? 256 : (n > 64 ? 128 : (n > 32 ? 64 : 32)), split = tid / across;
  const int splits = kPrefilterThreads / across, me = tid - split * across;
  int ii[kPrefilterTexels];
  bool on[kPrefilterTexels];  // block-uniform: whether the segment has a texel group c
  float3 acc[kPrefilterTexels], part[kPrefilterTexels];
#pragma unroll
  for (int c = 0; c < kPrefilterTexels; ++c) {
    on[c] = c * kPrefilterThreads < n;
    ii[c] = min(i0 + c * kPrefilterThreads + me, W - 1);  // duplicates of the last texel are not stored
    acc[c] = part[c] = f3(0, 0, 0);
  }
  int since = 0;
#pragma unroll 2
  for (int q = split; q < ns; q += splits) {
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
    if ((++since & 63) == 0) {  // fold every 64 samples' plain sums into the running sums
#pragma unroll
      for (int c = 0; c < kPrefilterTexels; ++c) {
        acc[c] = acc[c] + part[c];
        part[c] = f3(0, 0, 0);
      }
    }
  }
  if (splits > 1) {  // block-uniform
    s_sum[tid] = acc[0] + part[0];
    __syncthreads();
    if (split > 0) return;
  }
#pragma unroll
  for (int c = 0; c < kPrefilterTexels; ++c) {
    const int i = i0 + c * kPrefilterThreads + me;
    if (on[c] && i < W) {
      Kahan3 v;
      v.add(acc[c] + part[c]);
      for (int k = 1; k < splits; ++k) v.add(s_sum[me + k * across]);
      const float3 o = v.value() * inv;
      ch.dst[m][(long long)j * W + i] = make_float4(o.x, o.y, o.z, 1.0f);
    }
  }
}

template <bool INT_SHIFT>
__global__ void __launch_bounds__(kPrefilterThreads)
    k_prefilter(const __grid_constant__ MapDev src, const __grid_constant__ ChainDev ch, int N, int seg) {
  griddep_launch_dependents();
  prefilter_segment<INT_SHIFT>(src, ch, N, seg);
  complete_in_order();
}

// Level 0.
__global__ void __launch_bounds__(256) k_copy_texels(const float4* src, float4* dst, long long n, bool more) {
  if (more) griddep_launch_dependents();
  for (long long k = blockIdx.x * 256LL + threadIdx.x; k < n; k += gridDim.x * 256LL) dst[k] = src[k];
  complete_in_order();
}

// Levels whose texels are a power of two of source columns apart: the block of a row stages every
// source row its samples touch, once, in shared memory as three channel planes of phases
// (column c = phase + phases * k at [phase][k]), so that a tap of all texels of the row is three
// conflict-free reads of consecutive words, 12 bytes per texel instead of the 16 of an L1 read whose
// lines are half, a quarter, ... used.  A thread owns two neighbouring texels (their columns are
// `step` apart, so a row is staged in 2 step phases and one index serves all four taps); threads left
// over take shares of the samples.  Bound by shared-memory bandwidth (two rows x two columns x 12
// bytes per texel and sample; ncu: 74% of the LSU data pipe, tail included): levels 1 .. 7 of a 2048 x
// 1024 environment at 1024 samples 2545 us with every level read through L1; with levels 1 and 2 here,
// 1800 us, and the others after them in the SMs that the last rows leave, the whole set takes 1986 us
// (2143 us with the others first: their blocks' shared memory leaves no room for the rows').
constexpr int kRowsThreads = 512, kRowsMaxW = 2048, kRowsMaxH = 2048;
constexpr int kRowsMinW = 128;  // texels per row of a level
// Above a step of 4 a source row is staged for too few texels: the lighting set of a 2048 x 1024
// environment takes 2316, 2145 and 2248 us with steps up to 2, 4 and 8.
constexpr int kRowsMaxStep = 4;
// A plain FP32 sum takes at most this many samples (four taps each), however many lie between two source
// rows (1052 of 2048 over a 2048 x 64 environment), before it is added to a compensated running sum: the
// rounding of the sums is then below that of 64 samples per tap column and plain running sums (k_prefilter),
// 3.5e-8 against 5.4e-8 rms for 1000 samples (both orders replayed on the host).  Lighting set of a 2048 x 1024 environment, sums of whole
// rows, plain, 1984 us; of at most 32 samples, plain, 2005; compensated 2028, and 2050 where every row goes
// through the loop of the long ones.
constexpr int kRowsFold = 32;
constexpr int kRowsPlane = kRowsMaxW + 32;     // words per channel: phases padded by 32 / phases words
constexpr int kRowsSlot = 3 * kRowsPlane;      // words per staged row; three of them: two in use, one being filled

// A sample as the taps read it: byte offset of k for texel 0, then byte offsets of the phases of the
// two tap columns of an even texel and of the odd texel after it (relative to k, so 4 more where a
// column belongs to the next k).
struct RowsTap {
  unsigned k;
  unsigned even, odd;  // first column | second column << 16
  unsigned pad;
};

__device__ __forceinline__ RowsTap rows_tap(int c, int step, int phases, int phase_words) {
  const int p = c & (phases - 1);
  auto at = [&](int d) { return (unsigned)(((p + d) & (phases - 1)) * phase_words + (p + d >= phases ? 1 : 0)) * 4u; };
  return RowsTap{(unsigned)(c / phases) * 4u, at(0) | (at(1) << 16), at(step) | (at(step + 1) << 16), 0u};
}

extern __shared__ __align__(16) float s_rows[];

// Adds samples from, from + stride, ... below to, between the rows in slots SLOT and SLOT + 1 (modulo
// 3), to the texel pair whose even texel is k4 / 4 pairs along the row of n4 / 4 pairs.
template <int SLOT>
__device__ __forceinline__ void prefilter_taps(float3 (&part)[2], const float4* s_w, const RowsTap* s_tap, int from,
                                               int to, int stride, unsigned k4, unsigned n4) {
  constexpr int kTop = SLOT * kRowsSlot, kBot = (SLOT + 1) % 3 * kRowsSlot;
  for (int q = from; q < to; q += stride) {
    const float4 w = s_w[q];
    const uint4 t = *(const uint4*)(s_tap + q);
    unsigned k = t.x + k4;
    k = min(k, k - n4);  // wrapped round the row
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const unsigned o = g ? t.z : t.y;
      const float* a = (const float*)((const char*)s_rows + (k + (o & 0xffffu)));
      const float* b = (const float*)((const char*)s_rows + (k + (o >> 16)));
      part[g].x = fmaf(w.x, a[kTop], fmaf(w.y, b[kTop], fmaf(w.z, a[kBot], fmaf(w.w, b[kBot], part[g].x))));
      part[g].y = fmaf(w.x, a[kTop + kRowsPlane], fmaf(w.y, b[kTop + kRowsPlane],
                  fmaf(w.z, a[kBot + kRowsPlane], fmaf(w.w, b[kBot + kRowsPlane], part[g].y))));
      part[g].z = fmaf(w.x, a[kTop + 2 * kRowsPlane], fmaf(w.y, b[kTop + 2 * kRowsPlane],
                  fmaf(w.z, a[kBot + 2 * kRowsPlane], fmaf(w.w, b[kBot + 2 * kRowsPlane], part[g].z))));
    }
  }
}

// s_list: the `rows` source rows that are read (r + 1, -1 and H0 the clamped edges), in ascending
// order, a sample's two rows next to each other.
__device__ __forceinline__ void prefilter_row(const float4* s_w, const RowsTap* s_tap, const unsigned short* s_start,
                                              const unsigned short* s_list, int rows, const MapDev& src,
                                              float4* __restrict__ dst, int W, int phases, int phase_words, float inv) {
  const int tid = threadIdx.x, W0 = src.W, H0 = src.H;
  const int pairs = W / 2, share = tid / pairs, shares = kRowsThreads / pairs, me = tid - share * pairs;
  constexpr int kLoads = kRowsMaxW / kRowsThreads;
  float4 v[kLoads];
  auto load = [&](int k0) {
    const float4* row = src.texels + (size_t)min(max((int)s_list[k0] - 1, 0), H0 - 1) * W0;
#pragma unroll
    for (int k = 0; k < kLoads; ++k)
      if (tid + k * kRowsThreads < W0) v[k] = __ldg(row + tid + k * kRowsThreads);
  };
  const int log2p = 31 - __clz(phases);
  auto store = [&](int slot) {
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int c = tid + k * kRowsThreads;
      if (c >= W0) continue;
      float* q = s_rows + slot * kRowsSlot + (c & (phases - 1)) * phase_words + (c >> log2p);
      q[0] = v[k].x, q[kRowsPlane] = v[k].y, q[2 * kRowsPlane] = v[k].z;
      if (c < phases) {  // each phase's first column once more after its last
        q += pairs;
        q[0] = v[k].x, q[kRowsPlane] = v[k].y, q[2 * kRowsPlane] = v[k].z;
      }
    }
  };
  Kahan3 acc[2];
  float3 part[2];
  part[0] = part[1] = f3(0, 0, 0);
  auto fold = [&]() {  // the plain sums into the running sums
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      acc[g].add(part[g]);
      part[g] = f3(0, 0, 0);
    }
  };
  load(0);
  store(0);
  load(1);
  store(1);
  __syncthreads();
  int since = 0;
  for (int k = 0, slot = 0; k + 1 < rows; ++k) {
    if (k + 2 < rows) load(k + 2);
    const int from = s_start[s_list[k]], to = s_start[s_list[k] + 1];  // the samples between rows k and k + 1
    if (since + (to - from) > kRowsFold) fold(), since = 0;
    since += to - from;
    if (share < shares) {
      auto taps = [&](int a, int b) {
        if (slot == 0) prefilter_taps<0>(part, s_w, s_tap, a + share, b, shares, 4u * me, 4u * pairs);
        if (slot == 1) prefilter_taps<1>(part, s_w, s_tap, a + share, b, shares, 4u * me, 4u * pairs);
        if (slot == 2) prefilter_taps<2>(part, s_w, s_tap, a + share, b, shares, 4u * me, 4u * pairs);
      };
      if (to - from <= kRowsFold) {
        taps(from, to);
      } else {
#pragma unroll 1
        for (int q = from; q < to; q += kRowsFold) {
          taps(q, min(to, q + kRowsFold));
          fold();
        }
      }
    }
    if (k + 2 < rows) store(slot == 0 ? 2 : slot - 1);  // the slot of row k - 1
    slot = slot == 2 ? 0 : slot + 1;
    __syncthreads();
  }
  fold();
  float3 sum[2] = {acc[0].value(), acc[1].value()};
  if (shares > 1) {  // block-uniform; the staged rows are dead
    float3* s_sum = (float3*)s_rows;
    s_sum[2 * tid] = sum[0];
    s_sum[2 * tid + 1] = sum[1];
    __syncthreads();
    if (share == 0) {
      for (int k = 1; k < shares; ++k) {
        acc[0].add(s_sum[2 * (tid + k * pairs)]);
        acc[1].add(s_sum[2 * (tid + k * pairs) + 1]);
      }
      sum[0] = acc[0].value(), sum[1] = acc[1].value();
    }
  }
  if (share > 0) return;
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const float3 o = sum[g] * inv;
    dst[2 * me + g] = make_float4(o.x, o.y, o.z, 1.0f);
  }
}

// Dynamic shared memory: the staged rows, N float4 weights (first the sort keys), N taps, N sorted
// positions, H0 + 3 first samples (of source row r at [r + 1]), the list of source rows.
size_t rows_shared_bytes(int N, int H0) {
  return 4 * (size_t)(3 * kRowsSlot) + (sizeof(float4) + sizeof(RowsTap) + 2) * (size_t)N + 4 * (size_t)(H0 + 3);
}

__global__ void __launch_bounds__(kRowsThreads, 2) k_prefilter_rows(MapDev src, ChainDev ch, int N) {
  __shared__ PrefilterShared rec;
  __shared__ int s_rows_n;
  const int m = blockIdx.y + ch.first, j = blockIdx.x, W = ch.W[m], H = ch.H[m], H0 = src.H, W0 = src.W;
  griddep_launch_dependents();
  if (j < H) {  // block-uniform
    float4* s_w = (float4*)(s_rows + 3 * kRowsSlot);
    RowsTap* s_tap = (RowsTap*)(s_w + N);
    unsigned short* s_pos = (unsigned short*)(s_tap + N);
    unsigned short* s_start = s_pos + N;
    unsigned short* s_list = s_start + H0 + 3;
    const int step = 1 << m, phases = 2 * step, phase_words = (W0 + 32) / phases;
    float wsum;
    prefilter_records<kRowsThreads>(
        rec, (unsigned*)s_w, s_pos, m, ch.M, j, W, H, W0, H0, N, wsum,
        [&](const unsigned* key, int n) {
          // start[k] = number of samples whose source row + 1 is below k
          for (int q = threadIdx.x; q <= n; q += kRowsThreads) {
            const int lo = q > 0 ? (int)(key[q - 1] >> 16) + 1 : 0, hi = q < n ? (int)(key[q] >> 16) : H0 + 2;
            for (int k = lo; k <= hi; ++k) s_start[k] = (unsigned short)q;
          }
        },
        [&](int p, float4 e, float2 xy) {
          const float xf = floorf(xy.x), yf = floorf(xy.y);
          const float fx = xy.x - xf, fy = xy.y - yf;
          const float wt = e.z * (1.0f - fy), wb = e.z * fy;
          s_w[p] = make_float4(wt * (1.0f - fx), wt * fx, wb * (1.0f - fx), wb * fx);
          const int c = (int)xf;
          s_tap[p] = rows_tap(c < 0 ? c + W0 : (c >= W0 ? c - W0 : c), step, phases, phase_words);
        });
    // the source rows with a sample (between them and the next) and the rows after these
    if (threadIdx.x < 32) {
      int n = 0;
      for (int r0 = 0; r0 < H0 + 2; r0 += 32) {
        const int r = r0 + threadIdx.x;  // source row + 1
        const bool need = r < H0 + 2 && s_start[r + 1] > s_start[max(r - 1, 0)];
        const unsigned bal = __ballot_sync(0xffffffffu, need);
        if (need) s_list[n + __popc(bal & ((1u << threadIdx.x) - 1u))] = (unsigned short)r;
        n += __popc(bal);
      }
      if (threadIdx.x == 0) s_rows_n = n;
    }
    __syncthreads();
    float4* dst = ch.dst[m] + (long long)j * W;
    prefilter_row(s_w, s_tap, s_start, s_list, s_rows_n, src, dst, W, phases, phase_words, 1.0f / wsum);
  }
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
  const bool round = We <= kIrrPiece && We % kIrrSeg == 0;
  // slices of whole row pieces, as even as the three blocks an SM holds allow
  const long long pieces = (long long)He * ((We + kIrrPiece - 1) / kIrrPiece), room = 3LL * num_sms();
  const long long each = (pieces + room - 1) / room;
  const int nb = (int)std::min<long long>(irr_blocks(We, He), (pieces + each - 1) / each);
  // few slices (a small environment): smaller blocks, several per slice
  const int threads = nb >= num_sms() ? kIrrThreads : 128, passes = (nout + threads - 1) / threads;
  const int gy = (int)std::min<long long>(std::min(passes, 65535), std::max<long long>(1, room / nb));
  const size_t smem = irr_shared(nullptr, std::min(We, kIrrPiece)).bytes;
  epbr_status st;
  void (*k)(const float4*, int, int, int, int, float4*) = round ? k_irradiance_part<true> : k_irradiance_part<false>;
  if ((st = allow_shared(k, irr_shared(nullptr, kIrrPiece).bytes, "irradiance"))) return st;
  if ((st = launched(launch_kernel(k, dim3(nb, gy), dim3(threads), smem, s, early, (const float4*)env->texels, We, He, Wi, Hi,
                                   ws),
                     "k_irradiance_part")))
    return st;
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
  // levels 1 .. rows by k_prefilter_rows: texels 2 or 4 source columns apart, texel pairs of whole warps
  int rows = 0;
  while (rows + 1 < ch.M && (2 << rows) <= kRowsMaxStep && W0 <= kRowsMaxW && H0 <= kRowsMaxH &&
         W0 % (64 * (2 << rows)) == 0 && W0 / (2 << rows) >= kRowsMinW)
    ++rows;
  if (rows > 0) {
    ch.first = 1;
    const size_t smem = rows_shared_bytes(N, H0);
    if ((st = allow_shared(k_prefilter_rows, rows_shared_bytes(kPrefilterMaxSamples, kRowsMaxH), "prefilter"))) return st;
    if ((st = launched(launch_kernel(k_prefilter_rows, dim3(ch.H[1], rows), dim3(kRowsThreads), smem, s, early, src, ch, N),
                       "k_prefilter_rows")))
      return st;
    early = true;
  }
  // the others a block per segment of a row (level rows + 1 has the most); whole-column shifts when
  // every level's width divides the source width
  ch.first = rows + 1;
  if (ch.first < ch.M) {
    bool int_shift = true;
    for (int m = ch.first; m < ch.M; ++m) int_shift = int_shift && W0 % ch.W[m] == 0;
    int seg = kPrefilterSeg;
    unsigned most = 0;
    for (;; seg /= 2) {
      long long blocks = 0;
      most = 0;
      for (int m = ch.first; m < ch.M; ++m) {
        const unsigned b = (unsigned)(ch.H[m] * ((ch.W[m] + seg - 1) / seg));
        blocks += b;
        most = std::max(most, b);
      }
      if (seg <= kPrefilterMinSeg || blocks >= (long long)kPrefilterFill * num_sms()) break;
    }
    constexpr size_t kSampleBytes = sizeof(float4) + sizeof(int2) + sizeof(unsigned short);
    const size_t smem = (size_t)N * kSampleBytes;
    void (*k)(const MapDev, const ChainDev, int, int) = int_shift ? k_prefilter<true> : k_prefilter<false>;
    // for every count: without it the 48 KB limit also covers the kernel's static 6.3 KB
    if ((st = allow_shared(k, kPrefilterMaxSamples * kSampleBytes, "prefilter"))) return st;
    // a small shared-memory carve-out leaves most of the SM's 256 KB to L1, which holds the source
    // rows the resident blocks read (two rows of up to 16 KB per block)
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 50);  // a hint; failure is harmless
    if ((st = launched(launch_kernel(k, dim3(most, (unsigned)(ch.M - ch.first)), dim3(kPrefilterThreads), smem, s, early, src,
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
