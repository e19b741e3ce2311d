// Lookup kernels for 2D MIP-mapped textures, shared by the translation units that
// instantiate them for the plain (FP32 / FP16) and the DCT-compressed formats.
//
// One thread per query (grid-stride).  The stochastic kernels pick a level and one
// tap per axis by inverse CDF over |w| (sampling arrays, Section 2.2; separable
// sampling, Section 4.2), by positivization or by filter importance sampling, and
// fetch one texel (Eq. 3); the deterministic kernels sum every tap (Eq. 2, Eq. 9)
// over one level or two blended by frac(lod); the accumulate kernels repeat the
// stochastic form over many sample indices in float64 (validation only).
//
// Triplanar mapping (Section 5.2, "Triplanar mapping"): the query is a position p
// and a normal n; the three planes YZ, XZ, XY (uv = scale (p_y, p_z), scale (p_x, p_z),
// scale (p_x, p_y)) carry weights |n_x|, |n_y|, |n_z|.  Stochastically one plane is
// drawn with probability equal to its normalised weight (Eq. 3; inverse CDF in float32
// on word 2 of the query's stream 0) and its lookup is filtered stochastically; the
// deterministic form blends the three deterministic lookups.
#pragma once
#include "stf_launch.h"

namespace stf {

// Level choice: floor(lod + 1/2) (nearest) or floor(lod + u) (stochastic), lod
// clamped to [0, levels - 1].
__device__ __forceinline__ int level_stochastic(const Tex2DView& t, const LookupArgs& a,
                                                float lod, float u) {
  if (a.lod == nullptr || t.levels <= 1) return 0;
  const float lc = fminf(fmaxf(lod, 0.0f), (float)(t.levels - 1));
  const float s = __fadd_rn(lc, a.level_mode == STF_LEVEL_NEAREST ? 0.5f : u);
  return min((int)floorf(s), t.levels - 1);
}

template <int FMT, int C>
__device__ __forceinline__ void fetch_clamped(const Tex2DView& t, int L, int ix, int iy, float* v) {
  fetch2d<FMT, C>(t, L, min(max(ix, 0), t.level_w[L] - 1), min(max(iy, 0), t.level_h[L] - 1), v);
}

// One stochastic lookup at (uv, lod) with the variates r of caller query j.
template <int F, int FMT, int C, bool REUSE>
__device__ __forceinline__ void tex2d_stochastic_at(const Tex2DView& t, const LookupArgs& a,
                                                    float2 uv, float lod, int64_t j, uint32_t sample,
                                                    const uint4& r, float* v, int4& tap) {
  const int L = level_stochastic(t, a, lod, unit24(r.w));
  const int W = t.level_w[L], H = t.level_h[L];
  float x[2] = {__fsub_rn(__fmul_rn(uv.x, (float)W), 0.5f),
                __fsub_rn(__fmul_rn(uv.y, (float)H), 0.5f)};
  if (!(prepare_coords<2>(x) && isfinite(lod))) {
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = 0.0f;
    tap = make_int4(0, 0, 0, -1);
    return;
  }
  if constexpr (IsFis<F>::value) {
    int idx[2];
    pick_fis<F, 2>(x, a, j, sample, r, idx);
    tap = make_int4(idx[0], idx[1], 0, L);
    fetch_clamped<FMT, C>(t, L, idx[0], idx[1], v);
  } else if constexpr (F == STF_FILTER_CATMULL_ROM_POSITIVIZED) {
    const uint4 r1 = query_variates(a, j, sample, 1u);
    const float up[3] = {unit24(r.x), unit24(r.y), unit24(r.z)};
    const float un[3] = {unit24(r1.x), unit24(r1.y), unit24(r1.z)};
    int ip[2], in[2];
    float Wp, Wn;
    pick_positivized<2>(x, up, un, ip, in, Wp, Wn);
    tap = make_int4(ip[0], ip[1], 0, L);
    fetch_clamped<FMT, C>(t, L, ip[0], ip[1], v);
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] *= Wp;
    if (Wn > 0.0f) {
      float tn[C];
      fetch_clamped<FMT, C>(t, L, in[0], in[1], tn);
#pragma unroll
      for (int c = 0; c < C; ++c) v[c] = fmaf(-Wn, tn[c], v[c]);
    }
  } else {
    int idx[2];
    const float sigma = pick_taps_r<F, 2, REUSE>(x, r, idx);
    tap = make_int4(idx[0], idx[1], 0, L);
    fetch_clamped<FMT, C>(t, L, idx[0], idx[1], v);
    if constexpr (!Filter<F>::NONNEG) {
#pragma unroll
      for (int c = 0; c < C; ++c) v[c] *= sigma;
    }
  }
}

// One stochastic lookup of query i (caller's index j); I is int64_t, or uint32_t in the
// fast loop.
template <int F, int FMT, int C, bool REUSE, typename I>
__device__ __forceinline__ void tex2d_stochastic_one(const Tex2DView& t, const LookupArgs& a,
                                                     I i, I j, uint32_t sample,
                                                     float* v, int4& tap) {
  const float2 uv = reinterpret_cast<const float2*>(a.coords)[i];
  const float lod = a.lod ? a.lod[i] : 0.0f;
  const uint4 r = query_variates(a, j, sample);
  tex2d_stochastic_at<F, FMT, C, REUSE>(t, a, uv, lod, j, sample, r, v, tap);
}

// Deterministic filter at one level, weighted by `scale`, added to acc.
template <int F, int FMT, int C>
__device__ __forceinline__ void tex2d_det_level(const Tex2DView& t, int L, float2 uv, float scale,
                                                float width, float* acc) {
  using Fl = Filter<F>;
  const int W = t.level_w[L], H = t.level_h[L];
  float x[2] = {__fsub_rn(__fmul_rn(uv.x, (float)W), 0.5f),
                __fsub_rn(__fmul_rn(uv.y, (float)H), 0.5f)};
  if (!prepare_coords<2>(x)) return;
  if constexpr (F == STF_FILTER_FIS_GAUSSIAN) {
    const GaussAxis gx = gauss_axis(x[0], width), gy = gauss_axis(x[1], width);
    float ey0 = gauss_edge(gy, gy.lo);
    for (int iy = gy.lo; iy <= gy.hi; ++iy) {
      const float ey1 = gauss_edge(gy, iy + 1);
      const float wy = 0.5f * (ey1 - ey0) * scale;
      ey0 = ey1;
      const int cy = min(max(iy, 0), H - 1);
      float ex0 = gauss_edge(gx, gx.lo);
      for (int ix = gx.lo; ix <= gx.hi; ++ix) {
        const float ex1 = gauss_edge(gx, ix + 1);
        const float w = 0.5f * (ex1 - ex0) * wy;
        ex0 = ex1;
        float tv[C];
        fetch2d<FMT, C>(t, L, min(max(ix, 0), W - 1), cy, tv);
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = fmaf(w, tv[c], acc[c]);
      }
    }
  } else {
    float fx, fy;
    const int bx = axis_base(x[0], fx) + Fl::OFF0, by = axis_base(x[1], fy) + Fl::OFF0;
    float wx[Fl::T], wy[Fl::T];
    Fl::weights(fx, wx);
    Fl::weights(fy, wy);
    int cxs[Fl::T];
#pragma unroll
    for (int k = 0; k < Fl::T; ++k) cxs[k] = min(max(bx + k, 0), W - 1);
#pragma unroll
    for (int ky = 0; ky < Fl::T; ++ky) {
      const int cy = min(max(by + ky, 0), H - 1);
      const float wyk = wy[ky] * scale;
#pragma unroll
      for (int kx = 0; kx < Fl::T; ++kx) {
        float tv[C];
        fetch2d<FMT, C>(t, L, cxs[kx], cy, tv);
        const float w = wx[kx] * wyk;
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = fmaf(w, tv[c], acc[c]);
      }
    }
  }
}

// Deterministic lookup at (uv, lod) weighted by `scale`, added to acc: one level
// (nearest mode or no lod) or floor(lod) and the next blended by frac(lod).
template <int F, int FMT, int C>
__device__ __forceinline__ void tex2d_det_at(const Tex2DView& t, const LookupArgs& a, float2 uv,
                                             float lod, float scale, float* acc) {
  if (!isfinite(lod)) return;
  if (a.lod == nullptr || t.levels <= 1) {
    tex2d_det_level<F, FMT, C>(t, 0, uv, scale, a.width, acc);
    return;
  }
  const float lc = fminf(fmaxf(lod, 0.0f), (float)(t.levels - 1));
  if (a.level_mode == STF_LEVEL_NEAREST) {
    tex2d_det_level<F, FMT, C>(t, min((int)floorf(__fadd_rn(lc, 0.5f)), t.levels - 1), uv, scale,
                               a.width, acc);
  } else {
    const float fl = floorf(lc);
    const float frac = __fsub_rn(lc, fl);
    const int L0 = (int)fl, L1 = min(L0 + 1, t.levels - 1);
    tex2d_det_level<F, FMT, C>(t, L0, uv, scale * (1.0f - frac), a.width, acc);
    if (frac > 0.0f) tex2d_det_level<F, FMT, C>(t, L1, uv, scale * frac, a.width, acc);
  }
}

// Levels of a deterministic lookup and their weights: one level (nearest mode or no lod)
// or floor(lod) and the next blended by frac(lod); weights 0 for a lod that is not finite.
struct DetLevels {
  int L0, L1;
  float w0, w1;
};

__device__ __forceinline__ DetLevels det_levels(const Tex2DView& t, const LookupArgs& a, float lod) {
  DetLevels d = {0, 0, isfinite(lod) ? 1.0f : 0.0f, 0.0f};
  if (a.lod == nullptr || t.levels <= 1 || d.w0 == 0.0f) return d;
  const float lc = fminf(fmaxf(lod, 0.0f), (float)(t.levels - 1));
  if (a.level_mode == STF_LEVEL_NEAREST) {
    d.L0 = min((int)floorf(__fadd_rn(lc, 0.5f)), t.levels - 1);
  } else {
    const float fl = floorf(lc);
    d.w1 = __fsub_rn(lc, fl);
    d.w0 = 1.0f - d.w1;
    d.L0 = (int)fl;
    d.L1 = min(d.L0 + 1, t.levels - 1);
  }
  return d;
}

// ---------------------------------------------------------------- triplanar

struct Planes {
  float2 uv[3];
  float a[3];       // |n_x|, |n_y|, |n_z|
  bool ok;          // finite position and normal, non-zero normal
};

__device__ __forceinline__ Planes triplanar_planes(const LookupArgs& a, int64_t i) {
  Planes P;
  const float px = __ldg(a.coords + 3 * i), py = __ldg(a.coords + 3 * i + 1), pz = __ldg(a.coords + 3 * i + 2);
  const float nx = __ldg(a.normals + 3 * i), ny = __ldg(a.normals + 3 * i + 1), nz = __ldg(a.normals + 3 * i + 2);
  const float s = a.tri_scale;
  P.uv[0] = make_float2(__fmul_rn(py, s), __fmul_rn(pz, s));
  P.uv[1] = make_float2(__fmul_rn(px, s), __fmul_rn(pz, s));
  P.uv[2] = make_float2(__fmul_rn(px, s), __fmul_rn(py, s));
  P.a[0] = fabsf(nx);
  P.a[1] = fabsf(ny);
  P.a[2] = fabsf(nz);
  P.ok = finite3(px, py, pz) && finite3(nx, ny, nz) && (P.a[0] > 0.0f || P.a[1] > 0.0f || P.a[2] > 0.0f);
  return P;
}

// ---------------------------------------------------------------- DCT6, deterministic
//
// A DCT6 texel is linear in its block's coefficients and separable in x and y, so the
// weighted sum of a window's texels inside one block is one decode with the window's
// summed basis: sum_k w_k a(u) cos((2 x_k + 1) u pi / 16) per axis.  A window meets one
// or two blocks per axis (a bilinear one mostly one, of 64 one meets four), instead of
// T^2 decodes per level.  Each lane decodes the block of its window's first tap; the
// blocks beyond it differ from query to query, so a warp lists them in shared memory and
// decodes them 32 at a time: on the 4096^2 8-channel plane view, 17 such blocks for 32
// trilinear queries, in 3 decodes per lane in all instead of 8.  5.4 M queries: 225 us
// decoding every texel, 126 us (162 us with every block listed); bound by the ALU pipe
// (70%), mostly the decodes' shifts and conversions.
struct DctItems {
  static constexpr int MAX = 192;      // 32 queries x 2 levels x 3 further blocks
  // item: code word (64 bits), X0, X1 | X2, Y0, Y1, Y2; then channels 0..3 | 4..7 of its value
  float4 a[MAX], b[MAX];
};

struct __align__(8) DctLevel {
  int64_t off;
  int32_t w, h, blocks_w, pad;
};

// Window of one axis: block of its first tap, and the basis sums of the taps in that block
// and in the next (`two`: there are some).
template <int F>
struct DctAxis {
  float s[2][3];
  int block;
  bool two;
  __device__ __forceinline__ DctAxis(float x, int size, float c0, const float2* basis) {
    using Fl = Filter<F>;
    float f, w[Fl::T];
    const int first = axis_base(x, f) + Fl::OFF0;
    Fl::weights(f, w);
    block = min(max(first, 0), size - 1) >> 3;
    two = false;
#pragma unroll
    for (int b = 0; b < 2; ++b) s[b][0] = s[b][1] = s[b][2] = 0.0f;
#pragma unroll
    for (int k = 0; k < Fl::T; ++k) {
      const int c = min(max(first + k, 0), size - 1);
      const float2 q = basis[c & 7];
      const float v[3] = {w[k] * c0, w[k] * q.x, w[k] * q.y};
      two = (c >> 3) != block;         // the taps run on: once in the next block, always
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        s[0][u] += two ? 0.0f : v[u];
        s[1][u] += two ? v[u] : 0.0f;
      }
    }
  }
};

// Basis products of a block from the axes' sums.
__device__ __forceinline__ void dct_products(const float* X, const float* Y, float* b) {
  b[0] = X[0] * Y[0] * (8.0f / 127.0f);
  b[1] = X[1] * Y[0];
  b[2] = X[0] * Y[1];
  b[3] = X[2] * Y[0];
  b[4] = X[1] * Y[1];
  b[5] = X[0] * Y[2];
}

// Adds `scale` times the deterministic lookups at (uv, lod) of the warp's queries (those
// with `ok`) to acc.  Called by all 32 lanes.
template <int F, int C>
__device__ __forceinline__ void dct_det_warp(const Tex2DView& t, const LookupArgs& a, const DctLevel* levels, bool ok,
                                             float2 uv, float lod, float scale, const float2* basis, DctItems& items,
                                             float* acc) {
  const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
  const DetLevels d = det_levels(t, a, lod);
  const int L[2] = {d.L0, d.L1};
  const float part[2] = {d.w0, d.w1};
  uint32_t first[2] = {0, 0}, count[2] = {0, 0}, total = 0;
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    if (p == 1 && !__any_sync(0xffffffffu, ok && part[1] > 0.0f)) break;
    const DctLevel lv = levels[L[p]];
    float x[2] = {__fsub_rn(__fmul_rn(uv.x, (float)lv.w), 0.5f), __fsub_rn(__fmul_rn(uv.y, (float)lv.h), 0.5f)};
    const bool on = ok && part[p] > 0.0f && prepare_coords<2>(x);
    if (!on) x[0] = x[1] = 0.0f;
    DctAxis<F> ax(x[0], lv.w, t.dct_k[0], basis), ay(x[1], lv.h, t.dct_k[0], basis);
    const float sc = scale * part[p];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int u = 0; u < 3; ++u) ay.s[k][u] *= sc;
    const int64_t word = lv.off + ((int64_t)ay.block * lv.blocks_w + ax.block) * C;
    if (on) {
      uint32_t w[C];
      dct_codes<C>(t, word, w);
      float b[6], v[C];
      dct_products(ax.s[0], ay.s[0], b);
      dct_decode<C>(t, w, b, v);
#pragma unroll
      for (int c = 0; c < C; ++c) acc[c] += v[c];
    }
    const bool fx = on && ax.two, fy = on && ay.two;
    const uint32_t mx = __ballot_sync(0xffffffffu, fx), my = __ballot_sync(0xffffffffu, fy), mb = mx & my;
    first[p] = total + __popc(mx & below) + __popc(my & below) + __popc(mb & below);
    count[p] = (fx ? 1 : 0) + (fy ? 1 : 0) + (fx && fy ? 1 : 0);
    total += __popc(mx) + __popc(my) + __popc(mb);
    uint32_t s = first[p];
#pragma unroll
    for (int k = 1; k < 4; ++k) {
      const int bx = k & 1, by = k >> 1;
      if ((bx == 0 || fx) && (by == 0 || fy)) {
        const int64_t wk = word + (by ? (int64_t)lv.blocks_w * C : 0) + bx * C;
        items.a[s] = make_float4(__uint_as_float((uint32_t)wk), __uint_as_float((uint32_t)(wk >> 32)),
                                 ax.s[bx][0], ax.s[bx][1]);
        items.b[s] = make_float4(ax.s[bx][2], ay.s[by][0], ay.s[by][1], ay.s[by][2]);
        ++s;
      }
    }
  }
  if (total == 0) return;
  __syncwarp();
  for (uint32_t s = lane; s < total; s += 32) {
    const float4 p = items.a[s], q = items.b[s];
    const int64_t word = (int64_t)(((uint64_t)__float_as_uint(p.y) << 32) | __float_as_uint(p.x));
    const float X[3] = {p.z, p.w, q.x}, Y[3] = {q.y, q.z, q.w};
    uint32_t w[C];
    dct_codes<C>(t, word, w);
    float b[6], v[8] = {};
    dct_products(X, Y, b);
    dct_decode<C>(t, w, b, v);
    items.a[s] = make_float4(v[0], v[1], v[2], v[3]);
    if constexpr (C == 8) items.b[s] = make_float4(v[4], v[5], v[6], v[7]);
  }
  __syncwarp();
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    for (uint32_t s = first[p]; s < first[p] + count[p]; ++s) {
      const float4 v = items.a[s];
      acc[0] += v.x;
      if constexpr (C >= 2) acc[1] += v.y;
      if constexpr (C >= 4) {
        acc[2] += v.z;
        acc[3] += v.w;
      }
      if constexpr (C == 8) {
        const float4 u = items.b[s];
        acc[4] += u.x;
        acc[5] += u.y;
        acc[6] += u.z;
        acc[7] += u.w;
      }
    }
  }
  __syncwarp();          // the slots may be filled again
}

// Basis values by texel and the level table in shared memory (lanes index them apart).
__device__ __forceinline__ void stage_dct(const Tex2DView& t, float2* basis, DctLevel* levels) {
  const int k = threadIdx.x;
  if (k < 8) {
    float c0, c1, c2;
    dct_basis(t, k, c0, c1, c2);
    basis[k] = make_float2(c1, c2);
  }
  if (k < t.levels) levels[k] = {t.level_off[k], t.level_w[k], t.level_h[k], t.blocks_w[k], 0};
  __syncthreads();
}

// Deterministic lookups of a DCT6 texture, also over the planes of triplanar queries.
template <int F, int C, bool TRIPLANAR>
__global__ void __launch_bounds__(128) k_dct_deterministic(Tex2DView t, LookupArgs a) {
  __shared__ DctItems items[4];
  __shared__ float2 basis[8];
  __shared__ DctLevel levels[STF_MAX_LEVELS];
  stage_dct(t, basis, levels);
  DctItems& it = items[threadIdx.x >> 5];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  // (every lane of a warp runs the same iterations)
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; i0 < a.n; i0 += stride) {
    const int64_t i = i0 + lane;
    const bool live = i < a.n;
    float acc[C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = 0.0f;
    const float lod = live && a.lod ? a.lod[i] : 0.0f;
    if constexpr (TRIPLANAR) {
      const Planes P = triplanar_planes(a, live ? i : 0);
      const float S = __fadd_rn(__fadd_rn(P.a[0], P.a[1]), P.a[2]);
#pragma unroll 1
      for (int k = 0; k < 3; ++k) {
        const float w = k == 0 ? P.a[0] : k == 1 ? P.a[1] : P.a[2];
        const float2 uv = k == 0 ? P.uv[0] : k == 1 ? P.uv[1] : P.uv[2];
        dct_det_warp<F, C>(t, a, levels, live && P.ok && w > 0.0f, uv, lod, __fdiv_rn(w, S), basis, it, acc);
      }
    } else {
      const float2 uv = live ? reinterpret_cast<const float2*>(a.coords)[i] : make_float2(0.0f, 0.0f);
      dct_det_warp<F, C>(t, a, levels, live, uv, lod, 1.0f, basis, it, acc);
    }
    if (live) store_out<C>(a.out, i, acc);
  }
}

// Whether the deterministic form decodes blocks (dct_det_warp) rather than texels: all
// filters but the Gaussian, whose window can meet more than two blocks per axis.
template <int F, int FMT>
struct DctByBlock {
  static constexpr bool value = FMT == STF_FMT_DCT6 && F != STF_FILTER_FIS_GAUSSIAN;
};

template <int F, int FMT, int C, bool REUSE>
__global__ void __launch_bounds__(256) k_tex2d_stochastic(Tex2DView t, LookupArgs a) {
  if (fast_loop(a)) {
    const uint32_t n = (uint32_t)a.n, stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
      float v[C];
      int4 tap;
      tex2d_stochastic_one<F, FMT, C, REUSE>(t, a, i, i, a.sample_index, v, tap);
      store_out<C>(a.out, i, v);
    }
    return;
  }
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    float v[C];
    int4 tap;
    const int64_t j = query_slot(a, i);
    tex2d_stochastic_one<F, FMT, C, REUSE>(t, a, i, j, a.sample_index, v, tap);
    store_out<C>(a.out, j, v);
    if (a.taps) reinterpret_cast<int4*>(a.taps)[j] = tap;
  }
}

// ---------------------------------------------------------------- deterministic, scattered warps
//
// The cubic filters of plain textures.  With one thread per query, the 16 loads of a warp
// whose queries lie apart each read 32 lines, and the L1 data pipe bounds the filter (96%
// busy).  Such a warp runs its queries in four rounds of eight instead, four lanes to a
// query, one per tap column: the lanes read the four neighbouring texels of a row in one
// load, and their partial sums meet by halving exchanges.  Queries that are neighbours share
// lines between lanes already and keep one thread each, which sets up its weights once
// instead of four times.  4.2 M lookups of a 256^2 FP32 RGBA texture: 168 -> 104 us at random
// points, 58 -> 52 us in raster order (94 us by columns); half random and then in raster order
// 111 -> 77 us (101 us when a warp's first queries decided for all of its later ones).

// The window at raster position (x, y) of level L with its weights times `scale`.
template <int F, int FMT, int C>
struct CubicWindow {
  int L, W, H, bx, by;
  float wx[4], wy[4];
  __device__ __forceinline__ CubicWindow(const Tex2DView& t, int L_, float x, float y, float scale) : L(L_) {
    using Fl = Filter<F>;
    W = t.level_w[L];
    H = t.level_h[L];
    float fx, fy;
    bx = axis_base(x, fx) + Fl::OFF0;
    by = axis_base(y, fy) + Fl::OFF0;
    Fl::weights(fx, wx);
    Fl::weights(fy, wy);
#pragma unroll
    for (int k = 0; k < 4; ++k) wy[k] *= scale;
  }
  // Column k, added to acc.
  __device__ __forceinline__ void column(const Tex2DView& t, int k, float* acc) const {
    const float wk = k == 0 ? wx[0] : k == 1 ? wx[1] : k == 2 ? wx[2] : wx[3];
    const int cx = min(max(bx + k, 0), W - 1);
#pragma unroll
    for (int ky = 0; ky < 4; ++ky) {
      float tv[C];
      fetch2d<FMT, C>(t, L, cx, min(max(by + ky, 0), H - 1), tv);
      const float w = wk * wy[ky];
#pragma unroll
      for (int c = 0; c < C; ++c) acc[c] = fmaf(w, tv[c], acc[c]);
    }
  }
};

// One thread per query: the loop of the filters that do not gather by warp.
template <int F, int FMT, int C, typename I>
__device__ __forceinline__ void tex2d_det_loop(const Tex2DView& t, const LookupArgs& a) {
  const I n = (I)a.n, stride = (I)gridDim.x * blockDim.x;
  for (I i = (I)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const float2 uv = reinterpret_cast<const float2*>(a.coords)[i];
    const float lod = a.lod ? a.lod[i] : 0.0f;
    float acc[C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = 0.0f;
    tex2d_det_at<F, FMT, C>(t, a, uv, lod, 1.0f, acc);
    store_out<C>(a.out, i, acc);
  }
}

// A query's window positions: at level 0, or (LEVELS) at one or two levels with their
// weights.  A part that adds nothing has level -1.
template <bool LEVELS>
struct CubicParts {
  static constexpr int N = LEVELS ? 2 : 1;
  int L[N];
  float x[N], y[N], w[N];
  __device__ __forceinline__ CubicParts(const Tex2DView& t, const LookupArgs& a, float2 uv, float lod, bool live) {
    L[0] = live && isfinite(lod) ? 0 : -1;
    w[0] = 1.0f;
    if constexpr (LEVELS) {
      const DetLevels d = det_levels(t, a, lod);
      L[0] = live && d.w0 > 0.0f ? d.L0 : -1;
      L[1] = live && d.w1 > 0.0f ? d.L1 : -1;
      w[0] = d.w0;
      w[1] = d.w1;
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
      const int l = LEVELS ? max(L[p], 0) : 0;
      float q[2] = {__fsub_rn(__fmul_rn(uv.x, (float)t.level_w[l]), 0.5f),
                    __fsub_rn(__fmul_rn(uv.y, (float)t.level_h[l]), 0.5f)};
      if (!prepare_coords<2>(q)) L[p] = -1;
      x[p] = q[0];
      y[p] = q[1];
    }
  }
};

// At most kFastLoopMaxQueries queries.  Both ways of a warp's 32 queries sum a column's texels
// in the same order (of both levels), then columns 0 and 2, 1 and 3, and the two sums: a
// query's value does not depend on the queries beside it.
// (Four FP16 channels on six blocks an SM, 40 registers: raster order 56 -> 54 us.)
template <int F, int FMT, int C, bool LEVELS>
__global__ void __launch_bounds__(256, FMT == STF_FMT_F16 && C == 4 && !LEVELS ? 6 : 0) k_tex2d_cubic(Tex2DView t, LookupArgs a) {
  using Parts = CubicParts<LEVELS>;
  constexpr uint32_t full = 0xffffffffu;
  const uint32_t n = (uint32_t)a.n, stride = gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31, k = lane & 3;
  // (every lane of a warp runs the same iterations)
  for (uint32_t i0 = blockIdx.x * blockDim.x + threadIdx.x - lane; i0 < n; i0 += stride) {
    const uint32_t i = i0 + lane;
    const bool live = i < n;
    const float2 uv = live ? reinterpret_cast<const float2*>(a.coords)[i] : make_float2(0.0f, 0.0f);
    const float lod = live && a.lod ? a.lod[i] : 0.0f;
    const Parts q(t, a, uv, lod, live);
    // lanes whose neighbour's level-0 window is within a few texels of theirs
    const float x0 = uv.x * (float)t.level_w[0], y0 = uv.y * (float)t.level_h[0];
    const float dx = __shfl_xor_sync(full, x0, 1) - x0, dy = __shfl_xor_sync(full, y0, 1) - y0;
    if (__popc(__ballot_sync(full, fabsf(dx) < 5.0f && fabsf(dy) < 2.0f)) >= 16) {
      float v[4][C];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int c = 0; c < C; ++c) v[j][c] = 0.0f;
#pragma unroll
      for (int p = 0; p < Parts::N; ++p) {
        if (q.L[p] < 0) continue;
        const CubicWindow<F, FMT, C> w(t, LEVELS ? q.L[p] : 0, q.x[p], q.y[p], q.w[p]);
#pragma unroll
        for (int j = 0; j < 4; ++j) w.column(t, (j == 1 ? 2 : j == 2 ? 1 : j), v[(j == 1 ? 2 : j == 2 ? 1 : j)]);
      }
#pragma unroll
      for (int c = 0; c < C; ++c) v[0][c] = (v[0][c] + v[2][c]) + (v[1][c] + v[3][c]);
      if (!live) continue;
      store_out<C>(a.out, i, v[0]);
      continue;
    }
    const bool blend = LEVELS && __any_sync(full, q.L[Parts::N - 1] >= 0);
    float own[2] = {0.0f, 0.0f};                     // (C <= 2: the lane's own query)
#pragma unroll 1
    for (int r = 0; r < 4; ++r) {
      const int src = 8 * r + (lane >> 2);
      float v[C];
#pragma unroll
      for (int c = 0; c < C; ++c) v[c] = 0.0f;
#pragma unroll
      for (int p = 0; p < Parts::N; ++p) {
        if (p == 1 && !blend) break;
        const float x = __shfl_sync(full, q.x[p], src), y = __shfl_sync(full, q.y[p], src);
        const float sc = LEVELS ? __shfl_sync(full, q.w[p], src) : 1.0f;
        const int L = __shfl_sync(full, q.L[p], src);
        if (L >= 0) CubicWindow<F, FMT, C>(t, LEVELS ? L : 0, x, y, sc).column(t, k, v);
      }
      // sum over the four lanes; each exchange halves the channels a lane keeps
      int c0 = 0;
#pragma unroll
      for (int off = 2, kept = C; off >= 1; off /= 2) {
        const bool up = k & off;
        if (kept > 1) {
          kept /= 2;
#pragma unroll
          for (int c = 0; c < kept; ++c) {
            const float o = __shfl_xor_sync(full, up ? v[c] : v[c + kept], off);
            v[c] = (up ? v[c + kept] : v[c]) + o;
          }
          c0 += up ? kept : 0;
        } else {
          v[0] += __shfl_xor_sync(full, v[0], off);
        }
      }
      const uint32_t j = i0 + src;
      if constexpr (C <= 2) {
        // to the lane whose query it is, for one store of the warp's results in a row (stored
        // by round, 32 or 64 bytes at a time, results in host memory took a third longer)
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const float o = __shfl_sync(full, v[0], 4 * (lane & 7) + 2 * c);
          if (lane >> 3 == r) own[c] = o;
        }
      } else if (j < n) {
        float* o = a.out + (size_t)j * C + c0;
        if constexpr (C == 8) *reinterpret_cast<float2*>(o) = make_float2(v[0], v[1]);
        else *o = v[0];
      }
    }
    if (C <= 2 && live) store_out<(C <= 2 ? C : 1)>(a.out, i, own);
  }
}

// The other cubic lookups of at most kFastLoopMaxQueries: one thread per query.  (Eight
// channels take the 64-bit loop: the same time on device arrays, 890 us instead of 1070 for
// 2^22 lookups of arrays in host memory.)
template <int F, int FMT, int C>
__global__ void __launch_bounds__(256) k_tex2d_cubic_each(Tex2DView t, LookupArgs a) {
  tex2d_det_loop<F, FMT, C, uint32_t>(t, a);
}

// Whether warps with levels of detail may take their queries by columns: the second level's
// setup is paid four times as well.  Four FP32 channels gain (2^22 lookups at random levels
// 210 -> 193 us), eight FP16 channels lose (218 -> 234 us), and so do smaller texels.
template <int FMT, int C>
struct CubicLevels {
  static constexpr bool value = FMT == STF_FMT_F32 && C >= 4;
};

template <int F, int FMT, int C>
__global__ void __launch_bounds__(256) k_tex2d_deterministic(Tex2DView t, LookupArgs a) {
  tex2d_det_loop<F, FMT, C, int64_t>(t, a);
}

template <int F, int FMT, int C, bool REUSE>
__global__ void __launch_bounds__(256) k_tex2d_accumulate(Tex2DView t, LookupArgs a) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    double s[C], s2[C];
#pragma unroll
    for (int c = 0; c < C; ++c) s[c] = s2[c] = 0.0;
    for (int k = 0; k < a.n_samples; ++k) {
      float v[C];
      int4 tap;
      tex2d_stochastic_one<F, FMT, C, REUSE>(t, a, i, i, a.sample_index + (uint32_t)k, v, tap);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        s[c] += (double)v[c];
        s2[c] += (double)v[c] * (double)v[c];
      }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      a.sum[i * C + c] = s[c];
      a.sumsq[i * C + c] = s2[c];
    }
  }
}

template <int F, int FMT, int C>
__device__ __forceinline__ void triplanar_stochastic_one(const Tex2DView& t, const LookupArgs& a,
                                                         int64_t i, int64_t j, uint32_t sample,
                                                         float* v, int4& tap) {
  const Planes P = triplanar_planes(a, i);
  if (!P.ok) {
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = 0.0f;
    tap = make_int4(0, 0, 0, -1);
    return;
  }
  const uint4 r = query_variates(a, j, sample);
  const float c0 = P.a[0], c1 = __fadd_rn(P.a[0], P.a[1]), S = __fadd_rn(c1, P.a[2]);
  const float us = __fmul_rn(unit24(r.z), S);
  const int k = (us >= c0 ? 1 : 0) + (us >= c1 ? 1 : 0);
  const float lod = a.lod ? a.lod[i] : 0.0f;
  tex2d_stochastic_at<F, FMT, C, false>(t, a, P.uv[k], lod, j, sample, r, v, tap);
  if (tap.w >= 0) tap.z = k;
}

template <int F, int FMT, int C>
__global__ void __launch_bounds__(256) k_triplanar_stochastic(Tex2DView t, LookupArgs a) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    float v[C];
    int4 tap;
    triplanar_stochastic_one<F, FMT, C>(t, a, i, i, a.sample_index, v, tap);
    store_out<C>(a.out, i, v);
    if (a.taps) reinterpret_cast<int4*>(a.taps)[i] = tap;
  }
}

template <int F, int FMT, int C>
__global__ void __launch_bounds__(256) k_triplanar_deterministic(Tex2DView t, LookupArgs a) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    const Planes P = triplanar_planes(a, i);
    float acc[C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = 0.0f;
    if (P.ok) {
      const float S = __fadd_rn(__fadd_rn(P.a[0], P.a[1]), P.a[2]);
      const float lod = a.lod ? a.lod[i] : 0.0f;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (P.a[k] > 0.0f) tex2d_det_at<F, FMT, C>(t, a, P.uv[k], lod, __fdiv_rn(P.a[k], S), acc);
    }
    store_out<C>(a.out, i, acc);
  }
}

// ---------------------------------------------------------------- launchers

template <int F, int FMT, int C>
static cudaError_t run_tex2d(Op op, const Tex2DView& t, const LookupArgs& a, cudaStream_t s) {
  constexpr int D = deterministic_filter(F);
  const int threads = 256;
  const int blocks = grid_blocks(a.n, threads);
  if (a.normals) {                                    // triplanar queries
    if constexpr (F == STF_FILTER_CATMULL_ROM_POSITIVIZED) {
      return cudaErrorInvalidValue;                   // rejected by the argument checks
    } else {
      if (op == OP_STOCHASTIC) k_triplanar_stochastic<F, FMT, C><<<blocks, threads, 0, s>>>(t, a);
      else if (op == OP_DETERMINISTIC) {
        if constexpr (DctByBlock<D, FMT>::value) k_dct_deterministic<D, C, true><<<grid_blocks(a.n, 128), 128, 0, s>>>(t, a);
        else k_triplanar_deterministic<D, FMT, C><<<blocks, threads, 0, s>>>(t, a);
      } else return cudaErrorInvalidValue;              // no triplanar accumulation
      return cudaGetLastError();
    }
  }
  if (op == OP_STOCHASTIC) {
    if constexpr (UsesReuse<F>::value) {
      if (a.reuse) k_tex2d_stochastic<F, FMT, C, true><<<blocks, threads, 0, s>>>(t, a);
      else k_tex2d_stochastic<F, FMT, C, false><<<blocks, threads, 0, s>>>(t, a);
    } else {
      k_tex2d_stochastic<F, FMT, C, false><<<blocks, threads, 0, s>>>(t, a);
    }
  } else if (op == OP_DETERMINISTIC) {
    if constexpr (DctByBlock<D, FMT>::value) k_dct_deterministic<D, C, false><<<grid_blocks(a.n, 128), 128, 0, s>>>(t, a);
    else if constexpr (FMT != STF_FMT_DCT6 && (D == STF_FILTER_BSPLINE3 || D == STF_FILTER_CATMULL_ROM)) {
      for (int64_t i = 0; i < a.n; i += kFastLoopMaxQueries) {        // slices of 32-bit indices
        LookupArgs b = a;
        b.coords += 2 * i;
        if (b.lod) b.lod += i;
        b.out += C * i;
        b.n = a.n - i < kFastLoopMaxQueries ? a.n - i : kFastLoopMaxQueries;
        const int grid = grid_blocks(b.n, threads);
        if (a.lod == nullptr || t.levels <= 1) k_tex2d_cubic<D, FMT, C, false><<<grid, threads, 0, s>>>(t, b);
        else if constexpr (CubicLevels<FMT, C>::value) k_tex2d_cubic<D, FMT, C, true><<<grid, threads, 0, s>>>(t, b);
        else if constexpr (C == 8) k_tex2d_deterministic<D, FMT, C><<<grid, threads, 0, s>>>(t, b);
        else k_tex2d_cubic_each<D, FMT, C><<<grid, threads, 0, s>>>(t, b);
      }
    }
    else k_tex2d_deterministic<D, FMT, C><<<blocks, threads, 0, s>>>(t, a);
  } else {
    if constexpr (UsesReuse<F>::value) {
      if (a.reuse) k_tex2d_accumulate<F, FMT, C, true><<<blocks, threads, 0, s>>>(t, a);
      else k_tex2d_accumulate<F, FMT, C, false><<<blocks, threads, 0, s>>>(t, a);
    } else {
      k_tex2d_accumulate<F, FMT, C, false><<<blocks, threads, 0, s>>>(t, a);
    }
  }
  return cudaGetLastError();
}

template <int F, int FMT>
static cudaError_t run_tex2d_c(Op op, int c, const Tex2DView& t, const LookupArgs& a, cudaStream_t s) {
  switch (c) {
    case 1: return run_tex2d<F, FMT, 1>(op, t, a, s);
    case 2: return run_tex2d<F, FMT, 2>(op, t, a, s);
    case 4: return run_tex2d<F, FMT, 4>(op, t, a, s);
    case 8: return run_tex2d<F, FMT, 8>(op, t, a, s);
  }
  return cudaErrorInvalidValue;
}

// All filters for one storage format.
template <int FMT>
static cudaError_t launch_tex2d_format(Op op, int filter, int channels, const Tex2DView& t,
                                      const LookupArgs& a, cudaStream_t s) {
  switch (filter) {
    case STF_FILTER_LINEAR: return run_tex2d_c<STF_FILTER_LINEAR, FMT>(op, channels, t, a, s);
    case STF_FILTER_BSPLINE3: return run_tex2d_c<STF_FILTER_BSPLINE3, FMT>(op, channels, t, a, s);
    case STF_FILTER_CATMULL_ROM: return run_tex2d_c<STF_FILTER_CATMULL_ROM, FMT>(op, channels, t, a, s);
    case STF_FILTER_CATMULL_ROM_POSITIVIZED:
      return run_tex2d_c<STF_FILTER_CATMULL_ROM_POSITIVIZED, FMT>(op, channels, t, a, s);
    case STF_FILTER_FIS_LINEAR: return run_tex2d_c<STF_FILTER_FIS_LINEAR, FMT>(op, channels, t, a, s);
    case STF_FILTER_FIS_BSPLINE3: return run_tex2d_c<STF_FILTER_FIS_BSPLINE3, FMT>(op, channels, t, a, s);
    case STF_FILTER_FIS_GAUSSIAN: return run_tex2d_c<STF_FILTER_FIS_GAUSSIAN, FMT>(op, channels, t, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace stf
