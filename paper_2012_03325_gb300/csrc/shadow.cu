// Shadow maps with 3x3 percentage-closer filtering for the point lights (Sec. 5.1; Williams
// 1978, Reeves et al. 1987), evaluated inside the compose's light loop.
//   k_shade_shadow  one pixel per thread in 32x4 or 32x8 blocks, lights and their shadow cameras staged
//                   in shared memory in chunks of 128; per light (longer lists two lights at a time in
//                   packed FP32x2 arithmetic, the same bits) the direct terms of Eq. 1 and,
//                   when the light reaches the pixel (n.l > 0), its PCF visibility: the fragment
//                   projected into the light's map and the 3x3 block of depths around its texel
//                   compared with z - b0 - b1 z.  Ambient, background and tone map as k_shade.
#include <cmath>

#include "shade_core.cuh"

namespace epbr {

constexpr int kShadowChunk = 128;
// Lists of at least this many lights go two lights at a time, shorter ones (and the diffuse-only mode) one,
// with more warps for the work per pixel: below, the wider kernel's gain per light does not make up for
// its 37% of the warps against 50%.  1080p, 512^2 maps, us one / two at a time: 1 light 67 / 74, 4 lights
// 90 / 94, 8 123 / 125, 12 154 / 155, 16 183 / 182, 24 244 / 242, 64 573 / 551; coloured 67 / 74, 90 / 96,
// 123 / 127, 154 / 158, 184 / 186, 248 / 248, 581 / 568.
constexpr int kShadowPairs = 16;

struct ShadowDev {
  const float* maps;
  const float4* cams;  // 4 float4 per light: rows 0..2 of world -> light view, (f, -, -, -)
  long long map_texels;  // S * S
  int S;
  float b0, b1;
};

// Lit share of the 3x3 block of map texels around the projection of P (a tap outside the map,
// or P behind the light, counts as lit).
__device__ __forceinline__ float shadow_visibility(const float4* cam, float3 P, const float* __restrict__ map, int S,
                                                   float b0, float b1) {
  float4 r0 = cam[0], r1 = cam[1], r2 = cam[2];
  float f = cam[3].x;
  float qx = fmaf(r0.x, P.x, fmaf(r0.y, P.y, fmaf(r0.z, P.z, r0.w)));
  float qy = fmaf(r1.x, P.x, fmaf(r1.y, P.y, fmaf(r1.z, P.z, r1.w)));
  float z = -fmaf(r2.x, P.x, fmaf(r2.y, P.y, fmaf(r2.z, P.z, r2.w)));
  if (!(z > 0.0f)) return 1.0f;
  float half = 0.5f * (float)S, k = f * rcp_ftz(z);
  float s = fmaf(qx * k, half, half), t = fmaf(-qy * k, half, half);
  if (!(fabsf(s) < 1e9f && fabsf(t) < 1e9f)) return 1.0f;  // far outside the frustum
  int i0 = __float2int_rd(s), j0 = __float2int_rd(t);
  float thr = fmaf(-b1, z, z) - b0;  // lit when d >= z - b1 z - b0
  // the whole block inside (1 <= i0, j0 < S - 1, one unsigned compare each; none for S <= 2): no
  // per-tap bounds
  const unsigned inner = (unsigned)max(S - 2, 0);
  if ((unsigned)(i0 - 1) < inner && (unsigned)(j0 - 1) < inner) {
    // the lit taps counted in FP32 (sums of 0 and 1, exact): a compare-and-set and an FP32 add per
    // tap instead of an integer select and add, fewer instructions for the integer pipe, the busier
    // one in this kernel; the offset within the map fits 32 bits (S <= 8192)
    const float* p0 = map + ((j0 - 1) * S + (i0 - 1));
    float lit = 0.0f;
#pragma unroll
    for (int dy = 0; dy < 3; ++dy, p0 += S)
      lit += ((__ldg(p0) >= thr) ? 1.0f : 0.0f) + ((__ldg(p0 + 1) >= thr) ? 1.0f : 0.0f) +
             ((__ldg(p0 + 2) >= thr) ? 1.0f : 0.0f);
    return lit * (1.0f / 9.0f);
  }
  int lit = 0;
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy) {
    int j = j0 + dy;
    bool jin = (unsigned)j < (unsigned)S;
    const float* row = map + (size_t)(jin ? j : 0) * S;
#pragma unroll
    for (int dx = -1; dx <= 1; ++dx) {
      int i = i0 + dx;
      bool in = jin && (unsigned)i < (unsigned)S;
      lit += in ? (__ldg(row + (in ? i : 0)) >= thr) : 1;
    }
  }
  return (float)lit * (1.0f / 9.0f);
}

// Two lights' shadow cameras, value by value next to each other for packed arithmetic on -P: rows 0
// (negated rotation), 1 and 2 (negated offset) of world -> light view, so that -P gives q.x, -q.y and
// z = -q.z with the products and sums of shadow_visibility, then f.
struct CamPair {
  float2 r[3][4];
  float2 f, pad;
};

// shadow_visibility of P for two lights; the taps of both are under way together where both blocks
// lie inside their maps.
__device__ __forceinline__ float2 shadow_visibility2(const CamPair& c, const float4* cams, const float3& P, float2 mPx,
                                                     float2 mPy, float2 mPz, const float* __restrict__ map0,
                                                     const float* __restrict__ map1, int S, float b0, float b1) {
  const float2 qx = pfma(c.r[0][0], mPx, pfma(c.r[0][1], mPy, pfma(c.r[0][2], mPz, c.r[0][3])));
  const float2 mqy = pfma(c.r[1][0], mPx, pfma(c.r[1][1], mPy, pfma(c.r[1][2], mPz, c.r[1][3])));
  const float2 z = pfma(c.r[2][0], mPx, pfma(c.r[2][1], mPy, pfma(c.r[2][2], mPz, c.r[2][3])));
  const float2 half = dup2(0.5f * (float)S), k = pmul(c.f, make_float2(rcp_ftz(z.x), rcp_ftz(z.y)));
  const float2 s = pfma(pmul(qx, k), half, half), t = pfma(pmul(mqy, k), half, half);
  const float2 thr = padd(pfma(dup2(-b1), z, z), dup2(-b0));
  // a coordinate beyond +-1e9 converts to a texel outside the map as well
  const int i0 = __float2int_rd(s.x), j0 = __float2int_rd(t.x), i1 = __float2int_rd(s.y), j1 = __float2int_rd(t.y);
  const unsigned inner = (unsigned)max(S - 2, 0);
  const bool in0 = z.x > 0.0f && (unsigned)i0 - 1u < inner && (unsigned)j0 - 1u < inner;
  const bool in1 = z.y > 0.0f && (unsigned)i1 - 1u < inner && (unsigned)j1 - 1u < inner;
  if (in0 && in1) {
    const float* p = map0 + ((j0 - 1) * S + (i0 - 1));
    const float* q = map1 + ((j1 - 1) * S + (i1 - 1));
    float d[2][9];
#pragma unroll
    for (int r = 0; r < 3; ++r, p += S, q += S)
#pragma unroll
      for (int x = 0; x < 3; ++x) d[0][3 * r + x] = __ldg(p + x), d[1][3 * r + x] = __ldg(q + x);
    float l0 = 0.0f, l1 = 0.0f;
#pragma unroll
    for (int x = 0; x < 9; ++x) {
      l0 += d[0][x] >= thr.x ? 1.0f : 0.0f;
      l1 += d[1][x] >= thr.y ? 1.0f : 0.0f;
    }
    return make_float2(l0 * (1.0f / 9.0f), l1 * (1.0f / 9.0f));
  }
  return make_float2(shadow_visibility(cams, P, map0, S, b0, b1), shadow_visibility(cams + 4, P, map1, S, b0, b1));
}

// PAIRS: 128 threads, six blocks per SM (80 registers); else 256 threads, four blocks (64 registers).  Bound by
// issue and the LSU data pipe.  Two lights at a time in 256 threads at 64 (spills), 80 and 96 registers took
// 552, 561 and 680 us against 547 us (1080p, 64 lights, 512^2 maps), the taps requested before the light terms
// 589 us at best.
template <int FMT, int HDR, bool LDR, bool PAIRS>
__global__ void __launch_bounds__(32 * (PAIRS ? 4 : 8), PAIRS ? 6 : 4)
    k_shade_shadow(GbufDev g, CamDev cam, const float4* __restrict__ lights, int NL, IblDev ibl, ShadeDev p,
                   ShadowDev sh, void* hdr, long long hdr_pitch, uint8_t* ldr, long long ldr_pitch) {
  __shared__ float4 s_lights[2 * kShadowChunk];
  __shared__ float4 s_cams[4 * kShadowChunk];
  __shared__ float4 s_pos[PAIRS ? kShadowChunk : 1];  // per light pair (x, x, y, y), (z, z, Ic, Ic)
  __shared__ __align__(16) CamPair s_pair[PAIRS ? kShadowChunk / 2 : 1];
  constexpr int kShadowBY = PAIRS ? 4 : 8, kShadowThreads = 32 * kShadowBY;
  const int tid = threadIdx.y * 32 + threadIdx.x;
  const int by = gridDim.y - 1 - blockIdx.y;  // costliest rows first, as k_shade
  const int x = blockIdx.x * 32 + threadIdx.x, y = by * kShadowBY + threadIdx.y;
  const bool inside = x < g.W && y < g.H;
  Px s;
  if (inside) s = px_setup<FMT>(g, cam, x, y);
  const bool active = inside && s.surface;
  const bool diffuse_only = (p.flags & EPBR_SHADE_DIFFUSE_ONLY) != 0;
  Direct d;
  if (active) d = px_direct_begin(s);
  for (int base = 0; base < NL; base += kShadowChunk) {
    const int cnt = min(kShadowChunk, NL - base);
    __syncthreads();  // the previous chunk has been read
    for (int q = tid; q < 4 * cnt; q += kShadowThreads) s_cams[q] = __ldg(sh.cams + 4 * (size_t)base + q);
    // a chunk of monochrome lights keeps one sum per kind (each channel's sum would be the same)
    const bool mono = __syncthreads_and(stage_lights(s_lights, lights, base, cnt, tid, kShadowThreads));
    if (PAIRS && !diffuse_only) {  // block-uniform
      for (int q = tid; q < cnt / 2; q += kShadowThreads) {
        const float4 a = s_lights[4 * q], b = s_lights[4 * q + 2];
        s_pos[2 * q] = make_float4(a.x, b.x, a.y, b.y);
        s_pos[2 * q + 1] = make_float4(a.z, b.z, a.w, b.w);
      }
      for (int q = tid; q < cnt / 2 * 4; q += kShadowThreads) {
        const int r = q & 3;
        const float4 a = s_cams[8 * (q >> 2) + r], b = s_cams[8 * (q >> 2) + 4 + r];
        CamPair& c = s_pair[q >> 2];
        if (r == 3) {
          c.f = make_float2(a.x, b.x);
        } else {
          const float rot = r == 0 ? -1.0f : 1.0f;  // sign changes only: exact
          c.r[r][0] = make_float2(rot * a.x, rot * b.x);
          c.r[r][1] = make_float2(rot * a.y, rot * b.y);
          c.r[r][2] = make_float2(rot * a.z, rot * b.z);
          c.r[r][3] = make_float2(-rot * a.w, -rot * b.w);
        }
      }
      __syncthreads();
    }
    if (!active) continue;
    if (!diffuse_only) {
      // every light's terms times its visibility, added by `add(light, a, b, bf)`
      const float* map = sh.maps + (size_t)base * sh.map_texels;
      auto each = [&](auto add) {
        int i = 0;
        if (PAIRS) {
          Geo2 g;
          g.nx = dup2(s.n.x), g.ny = dup2(s.n.y), g.nz = dup2(s.n.z);
          g.mnx = dup2(-s.n.x), g.mny = dup2(-s.n.y), g.mnz = dup2(-s.n.z);
          g.vx = dup2(s.v.x), g.vy = dup2(s.v.y), g.vz = dup2(s.v.z);
          g.nva = dup2(d.nva), g.alpha = dup2(d.alpha), g.k = dup2(d.k), g.omk = dup2(d.omk);
          const float2 mPx = dup2(-s.P.x), mPy = dup2(-s.P.y), mPz = dup2(-s.P.z);
          for (; i + 1 < cnt; i += 2, map += 2 * sh.map_texels) {  // two lights at a time
            const float4 u = s_pos[i], z = s_pos[i + 1];
            Terms2 t = light_terms2(g, padd(make_float2(u.x, u.y), mPx), padd(make_float2(u.z, u.w), mPy),
                                    padd(make_float2(z.x, z.y), mPz));
            // the visibility (1 or less, finite) leaves the zero terms of an unlit light as they are
            if (t.a.x > 0.0f || t.b.x > 0.0f || t.a.y > 0.0f || t.b.y > 0.0f) {
              const float2 v = shadow_visibility2(s_pair[i >> 1], s_cams + 4 * i, s.P, mPx, mPy, mPz, map,
                                                  map + sh.map_texels, sh.S, sh.b0, sh.b1);
              t.a = pmul(t.a, v);
              t.b = pmul(t.b, v);
              t.bf = pmul(t.bf, v);
            }
            add(i, z.z, t.a.x, t.b.x, t.bf.x);
            add(i + 1, z.w, t.a.y, t.b.y, t.bf.y);
          }
        }
        for (; i < cnt; ++i, map += sh.map_texels) {
          const float4 lp = s_lights[2 * i];
          LightTerms t = light_terms(s, d, lp);
          if (t.a > 0.0f || t.b > 0.0f) {
            const float v = shadow_visibility(s_cams + 4 * i, s.P, map, sh.S, sh.b0, sh.b1);
            t.a *= v;
            t.b *= v;
            t.bf *= v;
          }
          add(i, lp.w, t.a, t.b, t.bf);
        }
      };
      if (mono) {
        float sa = 0.0f, sb = 0.0f, sbf = 0.0f;
        each([&](int, float Ic, float a, float b, float bf) {
          sa = fmaf(Ic, a, sa);
          sb = fmaf(Ic, b, sb);
          sbf = fmaf(Ic, bf, sbf);
        });
        d.sa = d.sa + f3(sa, sa, sa);
        d.sb = d.sb + f3(sb, sb, sb);
        d.sbf = d.sbf + f3(sbf, sbf, sbf);
      } else {
        float3 sa = d.sa, sb = d.sb, sbf = d.sbf;
        each([&](int i, float, float a, float b, float bf) {
          const float3 lc = xyz(s_lights[2 * i + 1]);
          sa = sa + lc * a;
          sb = sb + lc * b;
          sbf = sbf + lc * bf;
        });
        d.sa = sa;
        d.sb = sb;
        d.sbf = sbf;
      }
      continue;
    }
    float3 sa = d.sa;
    for (int i = 0; i < cnt; ++i) {
      float4 lp = s_lights[2 * i], lc = s_lights[2 * i + 1];
      const float* map = sh.maps + (size_t)(base + i) * sh.map_texels;
      float3 L = xyz(lp) - s.P;
      float rs = rsqrt_ftz(fmaf(L.x, L.x, fmaf(L.y, L.y, fmaf(L.z, L.z, 1e-30f))));
      float w = rs * rs * fmaxf(dot3(s.n, L) * rs, 0.0f);
      if (w > 0.0f) w *= shadow_visibility(s_cams + 4 * i, s.P, map, sh.S, sh.b0, sh.b1);
      sa = sa + xyz(lc) * w;
    }
    d.sa = sa;
  }
  if (!inside) return;
  if (active && NL > 0) {
    if (diffuse_only)
      px_direct_diffuse_end(s, d);
    else
      px_direct_end(s, d);
  }
  // Launched early (EPBR_SHADE_EARLY_START), the kernel before this one on the stream may still be
  // running up to here: the AO it writes is read, and the outputs written, only after it ends.
  griddep_wait();
  const float ao = active ? ao_at(p, x, y) : 1.0f;
  float3 c = px_finish(s, ibl, p.flags, ao);
  if (hdr) store_hdr<HDR>(hdr, hdr_pitch, x, y, c);
  if (LDR) ((unsigned*)(ldr + (size_t)y * ldr_pitch))[x] = pack_rgba8(c, p.exposure, p.op);
}

template <int FMT, int HDR>
static cudaError_t launch_shadow(cudaStream_t st, const GbufDev& g, const CamDev& c, const float4* L, int NL,
                                 const IblDev& ibl, const ShadeDev& p, const ShadowDev& sh, void* hdr, long long hp,
                                 uint8_t* ldr, long long lp) {
  const bool early = (p.flags & EPBR_SHADE_EARLY_START) != 0;
  const bool pairs = NL >= kShadowPairs && !(p.flags & EPBR_SHADE_DIFFUSE_ONLY);
  const int by = pairs ? 4 : 8;
  auto k = pairs ? (ldr ? k_shade_shadow<FMT, HDR, true, true> : k_shade_shadow<FMT, HDR, false, true>)
                 : (ldr ? k_shade_shadow<FMT, HDR, true, false> : k_shade_shadow<FMT, HDR, false, false>);
  cudaError_t e = launch_kernel(k, dim3((g.W + 31) / 32, (g.H + by - 1) / by), dim3(32, by), 0, st, early, g, c, L, NL, ibl,
                                p, sh, hdr, hp, ldr, lp);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

epbr_status launch_shade_shadows(const GbufDev& g, const CamDev& c, int fmt, const float4* L, int NL,
                                 const IblDev& ibl, const ShadeDev& p, const epbr_shadows* shadows, void* hdr,
                                 int hdr_format, long long hp, uint8_t* ldr, long long lp, cudaStream_t st) {
  const epbr_shadows* s = shadows;
  if (!s || !s->maps || !s->cameras || (uintptr_t)s->maps % 4 || (uintptr_t)s->cameras % 16 || s->size < 1 ||
      s->size > 8192 || !(s->bias_const >= 0.0f) || !(s->bias_slope >= 0.0f) || !std::isfinite(s->bias_const) ||
      !std::isfinite(s->bias_slope))
    return fail(EPBR_ERR_INVALID_ARG, "shadows: maps / cameras NULL or misaligned, size outside [1, 8192] or "
                "negative / non-finite bias");
  ShadowDev sh{s->maps, (const float4*)s->cameras, (long long)s->size * s->size, s->size, s->bias_const,
               s->bias_slope};
  cudaError_t e;
  if (fmt == EPBR_GBUFFER_FP32) {
    if (hdr_format == EPBR_HDR_RGBA32F)
      e = launch_shadow<EPBR_GBUFFER_FP32, EPBR_HDR_RGBA32F>(st, g, c, L, NL, ibl, p, sh, hdr, hp, ldr, lp);
    else
      e = launch_shadow<EPBR_GBUFFER_FP32, EPBR_HDR_RGBA16F>(st, g, c, L, NL, ibl, p, sh, hdr, hp, ldr, lp);
  } else {
    if (hdr_format == EPBR_HDR_RGBA32F)
      e = launch_shadow<EPBR_GBUFFER_COMPACT, EPBR_HDR_RGBA32F>(st, g, c, L, NL, ibl, p, sh, hdr, hp, ldr, lp);
    else
      e = launch_shadow<EPBR_GBUFFER_COMPACT, EPBR_HDR_RGBA16F>(st, g, c, L, NL, ibl, p, sh, hdr, hp, ldr, lp);
  }
  if (e != cudaSuccess) return fail(EPBR_ERR_CUDA, "k_shade_shadow: %s", cudaGetErrorString(e));
  return check_launch("k_shade_shadow");
}

}  // namespace epbr
