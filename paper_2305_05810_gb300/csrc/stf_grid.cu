// Lookup kernels for dense 3D voxel grids, the 2D launcher's format dispatch (the 2D
// kernels are in stf_tex2d.cuh, one translation unit per storage format), and the
// create-time kernels of regular grids.
//
// One thread per query (grid-stride), or warps that queue the queries that need work (the
// fixed-window filters).  The stochastic kernels draw one tap per axis
// by inverse CDF over |w| (sampling arrays, Section 2.2; separable sampling,
// Section 4.2) and fetch a single texel (Eq. 3); the deterministic kernels sum all
// 2^d / 4^d taps (Eq. 2, Eq. 9); the accumulate kernels repeat the stochastic form
// over many sample indices and sum in float64 (validation only).
#include "stf_launch.h"

namespace stf {

// ---------------------------------------------------------------- dense 3D

// Voxel (ix, iy, iz), or the background outside the grid.  OFF32: the grid has at
// most 2^32 voxels, so the element offset is computed in 32 bits.
template <int FMT, bool OFF32 = false>
__device__ __forceinline__ float dense_fetch(const Dense3DView& g, int ix, int iy, int iz) {
  if ((unsigned)ix >= (unsigned)g.nx || (unsigned)iy >= (unsigned)g.ny ||
      (unsigned)iz >= (unsigned)g.nz)
    return g.background;
  int64_t e;
  if constexpr (OFF32)
    e = (uint32_t)(((uint32_t)iz * (uint32_t)g.ny + (uint32_t)iy) * (uint32_t)g.nx + (uint32_t)ix);
  else
    e = ((int64_t)iz * g.ny + iy) * g.nx + ix;
  if constexpr (FMT == STF_FMT_F16)
    return __half2float(__ldg(reinterpret_cast<const __half*>(g.texels) + e));
  else
    return __ldg(reinterpret_cast<const float*>(g.texels) + e);
}

// One stochastic lookup at coordinates x (caller's query index j).  J is int64_t, or
// uint32_t in the fast loops.  With a miss box (the fast loops, which write no tap
// output), a fixed-window filter whose window lies outside the grid returns the
// background without drawing.
template <int F, int FMT, bool REUSE, bool OFF32 = false, typename J>
__device__ __forceinline__ float dense_stochastic_at(const Dense3DView& g, const LookupArgs& a,
                                                     float* x, J j, uint32_t sample, int4& tap,
                                                     const MissBox* miss = nullptr) {
  if (!prepare_coords<3>(x)) {
    tap = make_int4(0, 0, 0, -1);
    return g.background;
  }
  if constexpr (FixedWindow<F>::value) {
    if (miss && misses(*miss, x)) return g.background;
  }
  const uint4 r = query_variates(a, j, sample);
  if constexpr (IsFis<F>::value) {
    int idx[3];
    pick_fis<F, 3>(x, a, j, sample, r, idx);
    tap = make_int4(idx[0], idx[1], idx[2], 0);
    return dense_fetch<FMT, OFF32>(g, idx[0], idx[1], idx[2]);
  } else if constexpr (F == STF_FILTER_CATMULL_ROM_POSITIVIZED) {
    const uint4 r1 = query_variates(a, j, sample, 1u);
    const float up[4] = {unit24(r.x), unit24(r.y), unit24(r.z), unit24(r.w)};
    const float un[4] = {unit24(r1.x), unit24(r1.y), unit24(r1.z), unit24(r1.w)};
    int ip[3], in[3];
    float Wp, Wn;
    pick_positivized<3>(x, up, un, ip, in, Wp, Wn);
    tap = make_int4(ip[0], ip[1], ip[2], 0);
    float t = Wp * dense_fetch<FMT, OFF32>(g, ip[0], ip[1], ip[2]);
    if (Wn > 0.0f) t = fmaf(-Wn, dense_fetch<FMT, OFF32>(g, in[0], in[1], in[2]), t);
    return t;
  } else {
    int idx[3];
    const float sigma = pick_taps_r<F, 3, REUSE>(x, r, idx);
    tap = make_int4(idx[0], idx[1], idx[2], 0);
    float t = dense_fetch<FMT, OFF32>(g, idx[0], idx[1], idx[2]);
    if constexpr (!Filter<F>::NONNEG) t *= sigma;
    return t;
  }
}

// One stochastic lookup of query i (caller's index j).  I is int64_t, or uint32_t in
// the fast loop (3 i + 2 < 2^32 there).
template <int F, int FMT, bool REUSE, bool OFF32 = false, typename I>
__device__ __forceinline__ float dense_stochastic_one(const Dense3DView& g, const LookupArgs& a,
                                                      I i, I j, uint32_t sample, int4& tap) {
  float x[3] = {__ldg(a.coords + 3 * i), __ldg(a.coords + 3 * i + 1), __ldg(a.coords + 3 * i + 2)};
  return dense_stochastic_at<F, FMT, REUSE, OFF32>(g, a, x, j, sample, tap);
}

// Stochastic lookups of the fixed-window filters (tent, B-spline and their FIS forms), of
// grids of at most 2^32 voxels and at most kFastLoopMaxQueries queries, without tap output
// or permutation.  A ray-march chunk holds from none to three quarters of live samples; the
// queue lets every draw run on full lanes.  33 M samples of a 256^3 FP16 grid, B-spline:
// 135 us with the live ones of each chunk packed on its own lanes (two or four draws a
// lane), 121 us by queue (95 M instead of 117 M warp instructions; the coordinates kept
// beside the indices instead of read again: 4 us; the next chunk loaded ahead on five
// blocks an SM instead of six: 3 us; two draws a lane: 3 us slower).
constexpr int kDenseQueueBlocks = 5;      // resident 256-thread blocks per SM
template <int F, int FMT, int PER>
__global__ void __launch_bounds__(256, kDenseQueueBlocks) k_dense_stochastic_queue(Dense3DView g, LookupArgs a) {
  using W = FixedWindow<F>;
  __shared__ LiveQueue<PER> queues[8];
  __shared__ LiveCall call;
  const int zero[3] = {0, 0, 0}, dims[3] = {g.nx, g.ny, g.nz};
  float sample[3];
  load_sample<PER>(a, sample);
  stage_live(live_box(zero, dims, W::LO, W::HI), sample, call);
  __syncthreads();
  if (PER == 4 && call.direct) {
    const MissBox mb = miss_box<F>(0, 0, 0, g.nx, g.ny, g.nz);
    quad_loop3_joint(a, [&](float (&x)[4][3], uint32_t i) {
      return joint_one_tap4<F>(a, x, i, mb, g.background,
                               [&](const int* t) { return dense_fetch<FMT, true>(g, t[0], t[1], t[2]); });
    }, [&](float x0, float x1, float x2, uint32_t j) {
      float x[3] = {x0, x1, x2};
      int4 tap;
      return dense_stochastic_at<F, FMT, false, true>(g, a, x, j, a.sample_index, tap, &mb);
    });
    return;
  }
  live_queue_loop<PER>(a, g.background, call.box, queues[threadIdx.x >> 5], [&](uint32_t i, float (&x)[3], bool ok) {
    const uint4 v = query_variates(a, i, a.sample_index);
    prepare_coords<3>(x);
    int t[3];
    draw_one_tap3<F>(a, x, i, v, t);
    if (ok) a.out[i] = dense_fetch<FMT, true>(g, t[0], t[1], t[2]);
  });
}

// Resident 256-thread blocks per SM: six (at most 40 registers a thread) for the tent
// and B-spline filters, 1.4% sooner than five without spills when ray marches took this
// kernel (now the other calls do: host memory, tap output, binned, one variate reused); five
// for Catmull-Rom and the Gaussian, which would spill at 40; four for
// the two-tap positivized Catmull-Rom (at 84 registers and three blocks it ran 17%
// slower).
template <int F>
constexpr int dense_stochastic_min_blocks() {
  return F == STF_FILTER_CATMULL_ROM_POSITIVIZED ? 4
         : (F == STF_FILTER_CATMULL_ROM || F == STF_FILTER_FIS_GAUSSIAN) ? 5 : 6;
}

template <int F, int FMT, bool REUSE>
__global__ void __launch_bounds__(256, dense_stochastic_min_blocks<F>()) k_dense_stochastic(Dense3DView g,
                                                                                         LookupArgs a) {
  const bool off32 = (uint64_t)g.nx * (uint64_t)g.ny * (uint64_t)g.nz <= (uint64_t(1) << 32);
  const MissBox mb = miss_box<F>(0, 0, 0, g.nx, g.ny, g.nz);
  if constexpr (JointOneTap<F, REUSE>::value) {
    if (off32 && quad_loop3_ok(a)) {
      quad_loop3_joint(a, [&](float (&x)[4][3], uint32_t i) {
        return joint_one_tap4<F>(a, x, i, mb, g.background,
                                 [&](const int* t) { return dense_fetch<FMT, true>(g, t[0], t[1], t[2]); });
      }, [&](float x0, float x1, float x2, uint32_t j) {
        float x[3] = {x0, x1, x2};
        int4 tap;
        return dense_stochastic_at<F, FMT, REUSE, true>(g, a, x, j, a.sample_index, tap, &mb);
      });
      return;
    }
  }
  if (off32 && quad_loop3_ok(a)) {
    quad_loop3(a, (uint32_t)a.n >> 2, [&](float x0, float x1, float x2, uint32_t j) {
      float x[3] = {x0, x1, x2};
      int4 tap;
      return dense_stochastic_at<F, FMT, REUSE, true>(g, a, x, j, a.sample_index, tap, &mb);
    });
    return;
  }
  if (fast_loop(a) && off32) {
    const uint32_t n = (uint32_t)a.n, stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
      float x[3] = {__ldg(a.coords + 3 * i), __ldg(a.coords + 3 * i + 1), __ldg(a.coords + 3 * i + 2)};
      int4 tap;
      a.out[i] = dense_stochastic_at<F, FMT, REUSE, true>(g, a, x, i, a.sample_index, tap, &mb);
    }
    return;
  }
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    int4 tap;
    const int64_t j = query_slot(a, i);
    a.out[j] = dense_stochastic_one<F, FMT, REUSE>(g, a, i, j, a.sample_index, tap);
    if (a.taps) reinterpret_cast<int4*>(a.taps)[j] = tap;
  }
}

// The T consecutive voxels e .. e + T - 1 of one grid row, from the aligned word that holds
// e plus, when the row runs over it, the start of the next one: 16 bytes (eight FP16
// voxels, and 8 bytes more for e mod 8 > 4; four FP32 voxels, and 16 bytes more for
// e mod 4 > 0) for rows of four, two voxels (and one more for odd e) for rows of two.  The
// texel allocation is padded by 16 bytes, so no load leaves it.  The L1 wavefronts of these
// loads bound the filters.  (Two aligned 8-byte words for FP16 rows of four, needed for 3
// of 4 rows, took 15% more of them at the same time.)
template <int FMT, int T>
__device__ __forceinline__ void dense_row(const void* texels, uint32_t e, float* v) {
  if constexpr (FMT == STF_FMT_F16 && T == 4) {
    const uint4* w = reinterpret_cast<const uint4*>(texels) + (e >> 3);
    const uint4 a = __ldg(w);
    uint2 b = make_uint2(0u, 0u);
    if ((e & 7) > 4) b = __ldg(reinterpret_cast<const uint2*>(w + 1));
    const bool by2 = e & 4, by1 = e & 2;
    const uint32_t y0 = by2 ? a.z : a.x, y1 = by2 ? a.w : a.y, y2 = by2 ? b.x : a.z, y3 = by2 ? b.y : a.w;
    const uint32_t x0 = by1 ? y1 : y0, x1 = by1 ? y2 : y1, x2 = by1 ? y3 : y2;
    const uint32_t sh = (e & 1) * 16;
    const uint32_t lo = __funnelshift_r(x0, x1, sh), hi = __funnelshift_r(x1, x2, sh);
    const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&lo));
    const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&hi));
    v[0] = f0.x; v[1] = f0.y; v[2] = f1.x; v[3] = f1.y;
  } else if constexpr (FMT == STF_FMT_F32 && T == 4) {
    const float4* w = reinterpret_cast<const float4*>(texels) + (e >> 2);
    const float4 a = __ldg(w);
    float4 b = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (e & 3) b = __ldg(w + 1);
    const bool by2 = e & 2, by1 = e & 1;
    const float y0 = by2 ? a.z : a.x, y1 = by2 ? a.w : a.y, y2 = by2 ? b.x : a.z, y3 = by2 ? b.y : a.w,
                y4 = by2 ? b.z : b.x;
    v[0] = by1 ? y1 : y0; v[1] = by1 ? y2 : y1; v[2] = by1 ? y3 : y2; v[3] = by1 ? y4 : y3;
  } else if constexpr (FMT == STF_FMT_F16) {
    static_assert(T == 2, "rows of two or four");
    const __half2 a = __ldg(reinterpret_cast<const __half2*>(texels) + (e >> 1));
    v[0] = __high2float(a);
    if (e & 1) {
      v[1] = __half2float(__ldg(reinterpret_cast<const __half*>(texels) + e + 1));
    } else {
      v[1] = v[0];
      v[0] = __low2float(a);
    }
  } else {
    static_assert(T == 2, "rows of two or four");
    const float2 a = __ldg(reinterpret_cast<const float2*>(texels) + (e >> 1));
    v[0] = a.y;
    if (e & 1) {
      v[1] = __ldg(reinterpret_cast<const float*>(texels) + e + 1);
    } else {
      v[1] = v[0];
      v[0] = a.x;
    }
  }
}

// Deterministic window at one query: base voxel, weights per axis.
template <int F>
struct DenseWindow {
  static constexpr int T = Filter<F>::T;
  int bx, by, bz;
  float wx[T], wy[T], wz[T];
  __device__ __forceinline__ explicit DenseWindow(const float* x) {
    float fx, fy, fz;
    bx = axis_base(x[0], fx) + Filter<F>::OFF0;
    by = axis_base(x[1], fy) + Filter<F>::OFF0;
    bz = axis_base(x[2], fz) + Filter<F>::OFF0;
    Filter<F>::weights(fx, wx);
    Filter<F>::weights(fy, wy);
    Filter<F>::weights(fz, wz);
  }
};

// The whole window inside a grid of at most 2^32 voxels: rows of T voxels along x, no
// bounds tests; each row's weighted sum, then the rows weighted by wy * wz.
template <int F, int FMT>
__device__ __forceinline__ float dense_inner_sum(const Dense3DView& g, const float* x) {
  constexpr int T = Filter<F>::T;
  const DenseWindow<F> w(x);
  const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny;
  const uint32_t e0 = ((uint32_t)w.bz * ny + (uint32_t)w.by) * nx + (uint32_t)w.bx;
  float acc = 0.0f;
#pragma unroll
  for (int kz = 0; kz < T; ++kz) {
#pragma unroll
    for (int ky = 0; ky < T; ++ky) {
      float v[T];
      dense_row<FMT, T>(g.texels, e0 + ((uint32_t)kz * ny + (uint32_t)ky) * nx, v);
      float r = w.wx[0] * v[0];
#pragma unroll
      for (int kx = 1; kx < T; ++kx) r = fmaf(w.wx[kx], v[kx], r);
      acc = fmaf(w.wy[ky] * w.wz[kz], r, acc);
    }
  }
  return acc;
}

// A window that straddles the grid's edge (or any window of a larger grid): every voxel
// checked.
template <int F, int FMT>
__device__ __forceinline__ float dense_edge_sum(const Dense3DView& g, const float* x) {
  constexpr int T = Filter<F>::T;
  const DenseWindow<F> w(x);
  float acc = 0.0f;
#pragma unroll
  for (int kz = 0; kz < T; ++kz) {
#pragma unroll
    for (int ky = 0; ky < T; ++ky) {
      const float wyz = w.wy[ky] * w.wz[kz];
#pragma unroll
      for (int kx = 0; kx < T; ++kx)
        acc = fmaf(w.wx[kx] * wyz, dense_fetch<FMT>(g, w.bx + kx, w.by + ky, w.bz + kz), acc);
    }
  }
  return acc;
}

// One warp's live queries, waiting until 32 of one kind can run side by side: windows
// inside the grid from the front, windows straddling its edge from the back.  At most
// 31 of each kind wait while a chunk of up to 128 is added.
struct DenseQueue {
  static constexpr int CAP = 192;
  uint32_t i[CAP];
  float x[3][CAP];
};

constexpr int kDenseDetBlocks = 3;   // resident 256-thread blocks per SM

// Deterministic lookups of at most kFastLoopMaxQueries queries.  Each warp walks chunks
// of 32 * PER queries, writes the background where the window misses the grid, and queues
// the others in shared memory; whenever 32 windows of one kind wait, they run on all 32
// lanes.  Ray-march samples mix misses, inner and edge windows in every warp: run in
// place, 10 of 32 lanes were active.  8.3 M samples of a 256^3 FP16 grid, tricubic:
// 323 us in place, 173 us queued (60 M instead of 184 M warp instructions), now bound by
// the L1 wavefronts of the row loads (84%).  The grid is the resident blocks only: with
// two waves of blocks, twice as many warps ended with partly filled queues (15% later).
template <int F, int FMT, int PER>
__global__ void __launch_bounds__(256, kDenseDetBlocks) k_dense_deterministic(Dense3DView g, LookupArgs a) {
  constexpr int T = Filter<F>::T, OFF0 = Filter<F>::OFF0;
  __shared__ DenseQueue queues[8];
  // a window entirely outside the grid on some axis reads only the background, and the
  // weights sum to one (partition of unity)
  __shared__ LiveBox live, inner;
  const bool off32 = (uint64_t)g.nx * (uint64_t)g.ny * (uint64_t)g.nz <= (uint64_t(1) << 32);
  if (threadIdx.x == 0) {
    const int zero[3] = {0, 0, 0}, dims[3] = {g.nx, g.ny, g.nz};
    live = live_box(zero, dims, OFF0, OFF0 + T - 1);
    inner = live_box(zero, dims, OFF0 + T - 1, OFF0);
  }
  __syncthreads();
  DenseQueue& q = queues[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
  const uint32_t n = (uint32_t)a.n;
  const bool aligned = (((uintptr_t)a.coords | (uintptr_t)a.out) & 15) == 0;
  uint32_t n_inner = 0, n_edge = 0;
  for (WarpChunks<32 * PER> w;; w.next()) {
    const bool more = w.row < n;                     // else: only what still waits
    const uint32_t i0 = w.first() + lane * PER;
    float x[PER][3];
    load_and_clear<PER>(a, g.background, aligned, i0, n, x);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const bool hit = live.has(x[k]), in = hit && off32 && inner.has(x[k]), edge = hit && !in;
      const uint32_t mi = __ballot_sync(0xffffffffu, in), me = __ballot_sync(0xffffffffu, edge);
      if (hit) {
        const uint32_t s = in ? n_inner + __popc(mi & below) : DenseQueue::CAP - 1 - n_edge - __popc(me & below);
        q.i[s] = i0 + k;
        q.x[0][s] = x[k][0]; q.x[1][s] = x[k][1]; q.x[2][s] = x[k][2];
      }
      n_inner += __popc(mi);
      n_edge += __popc(me);
    }
    __syncwarp();          // the queue and the background stores, before other lanes' results
    const uint32_t least = more ? 32 : 1;
    while (n_inner >= least) {
      const uint32_t count = min(n_inner, 32u), s = n_inner - count + lane;
      if (lane < count) {
        float xs[3] = {q.x[0][s], q.x[1][s], q.x[2][s]};
        prepare_coords<3>(xs);
        a.out[q.i[s]] = dense_inner_sum<F, FMT>(g, xs);
      }
      n_inner -= count;
    }
    while (n_edge >= least) {
      const uint32_t count = min(n_edge, 32u), s = DenseQueue::CAP - 1 - (n_edge - count + lane);
      if (lane < count) {
        float xs[3] = {q.x[0][s], q.x[1][s], q.x[2][s]};
        prepare_coords<3>(xs);
        a.out[q.i[s]] = dense_edge_sum<F, FMT>(g, xs);
      }
      n_edge -= count;
    }
    if (!more) break;
    __syncwarp();          // the slots just read may be filled again
  }
}

// One thread per query: the trilinear filter (eight scattered voxels of a 256^3 FP16 grid: 10 M
// hits 137 us in place, 164 us queued; 8.4 M ray-march samples 48 and 49 us; of 33 M, the most
// warps' worth, 197 and 182 us, before the live test 236), and arrays that are not in this
// device's memory, whose link bounds the call: a queued kernel writes results
// twice and reads coordinates from few warps (4 M hits with results in host memory, trilinear
// 96 us in place, 514 us queued; tricubic 258 and 590 us).
template <int F, int FMT>
__global__ void __launch_bounds__(256) k_dense_deterministic_each(Dense3DView g, LookupArgs a) {
  constexpr int T = Filter<F>::T, OFF0 = Filter<F>::OFF0;
  __shared__ LiveBox live, inner;
  const bool off32 = (uint64_t)g.nx * (uint64_t)g.ny * (uint64_t)g.nz <= (uint64_t(1) << 32);
  if (threadIdx.x == 0) {
    const int zero[3] = {0, 0, 0}, dims[3] = {g.nx, g.ny, g.nz};
    live = live_box(zero, dims, OFF0, OFF0 + T - 1);
    inner = live_box(zero, dims, OFF0 + T - 1, OFF0);
  }
  __syncthreads();
  const uint32_t n = (uint32_t)a.n, stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    float x[3] = {__ldg(a.coords + 3 * i), __ldg(a.coords + 3 * i + 1), __ldg(a.coords + 3 * i + 2)};
    float acc = g.background;
    if (live.has(x)) {
      const bool in = T == 4 && off32 && inner.has(x);
      prepare_coords<3>(x);
      acc = in ? dense_inner_sum<F, FMT>(g, x) : dense_edge_sum<F, FMT>(g, x);
    }
    a.out[i] = acc;
  }
}

// Deterministic form of the Gaussian FIS filter: one thread per query.
template <int FMT>
__global__ void __launch_bounds__(256) k_dense_gaussian(Dense3DView g, LookupArgs a) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    float x[3] = {__ldg(a.coords + 3 * i), __ldg(a.coords + 3 * i + 1), __ldg(a.coords + 3 * i + 2)};
    float acc = g.background;
    if (prepare_coords<3>(x))
      acc = gauss_window_sum3(x, a.width, [&](int ix, int iy, int iz) { return dense_fetch<FMT>(g, ix, iy, iz); });
    a.out[i] = acc;
  }
}

template <int F, int FMT, bool REUSE>
__global__ void __launch_bounds__(256) k_dense_accumulate(Dense3DView g, LookupArgs a) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    double s = 0.0, s2 = 0.0;
    for (int k = 0; k < a.n_samples; ++k) {
      int4 tap;
      const double v = dense_stochastic_one<F, FMT, REUSE>(g, a, i, i, a.sample_index + (uint32_t)k, tap);
      s += v;
      s2 += v * v;
    }
    a.sum[i] = s;
    a.sumsq[i] = s2;
  }
}

// ---------------------------------------------------------------- launchers

cudaError_t launch_tex2d(Op op, int filter, int fmt, int channels, const Tex2DView& t,
                         const LookupArgs& a, cudaStream_t s) {
  if (fmt == STF_FMT_F32) return launch_tex2d_f32(op, filter, channels, t, a, s);
  if (fmt == STF_FMT_F16) return launch_tex2d_f16(op, filter, channels, t, a, s);
  if (fmt == STF_FMT_DCT6) return launch_tex2d_dct(op, filter, channels, t, a, s);
  return cudaErrorInvalidValue;
}

template <int F, int FMT>
static cudaError_t run_dense(Op op, const Dense3DView& g, const LookupArgs& a, cudaStream_t s) {
  const int threads = 256;
  // the four-query loop needs a quarter of the threads
  const int64_t units = (op == OP_STOCHASTIC && quad_loop3_ok(a)) ? (a.n + 3) / 4 : a.n;
  const int blocks = grid_blocks(units, threads, op == OP_STOCHASTIC ? kStochasticWaves : 4);
  if (op == OP_STOCHASTIC) {
    if constexpr (FixedWindow<F>::value) {
      const bool off32 = (uint64_t)g.nx * (uint64_t)g.ny * (uint64_t)g.nz <= (uint64_t(1) << 32);
      // (results in host memory, which the queue writes twice: in place, 4 M hits 96 us, 495 queued)
      if (off32 && fast_loop(a) && !(UsesReuse<F>::value && a.reuse) && local_arrays(a)) {
        if (a.n >= kQueueChunkMin)
          k_dense_stochastic_queue<F, FMT, 4><<<queue_blocks((a.n + 3) / 4, threads, kDenseQueueBlocks), threads, 0, s>>>(g, a);
        else
          k_dense_stochastic_queue<F, FMT, 1><<<queue_blocks(a.n, threads, kDenseQueueBlocks), threads, 0, s>>>(g, a);
        return cudaGetLastError();
      }
    }
    if constexpr (UsesReuse<F>::value) {
      if (a.reuse) k_dense_stochastic<F, FMT, true><<<blocks, threads, 0, s>>>(g, a);
      else k_dense_stochastic<F, FMT, false><<<blocks, threads, 0, s>>>(g, a);
    } else {
      k_dense_stochastic<F, FMT, false><<<blocks, threads, 0, s>>>(g, a);
    }
  } else if (op == OP_DETERMINISTIC) {
    constexpr int D = deterministic_filter(F);
    if constexpr (D == STF_FILTER_FIS_GAUSSIAN) {
      k_dense_gaussian<FMT><<<blocks, threads, 0, s>>>(g, a);
    } else {
      // slices of 32-bit indices
      for (int64_t i = 0; i < a.n; i += kFastLoopMaxQueries) {
        LookupArgs b = a;
        b.coords += 3 * i;
        b.out += i;
        b.n = a.n - i < kFastLoopMaxQueries ? a.n - i : kFastLoopMaxQueries;
        if constexpr (Filter<D>::T == 4) {
          if (local_arrays(a)) {
            if (b.n >= kQueueChunkMin)
              k_dense_deterministic<D, FMT, 4><<<queue_blocks((b.n + 3) / 4, threads, kDenseDetBlocks), threads, 0, s>>>(g, b);
            else
              k_dense_deterministic<D, FMT, 1><<<queue_blocks(b.n, threads, kDenseDetBlocks), threads, 0, s>>>(g, b);
            continue;
          }
        }
        k_dense_deterministic_each<D, FMT><<<grid_blocks(b.n, threads), threads, 0, s>>>(g, b);
      }
    }
  } else {
    if constexpr (UsesReuse<F>::value) {
      if (a.reuse) k_dense_accumulate<F, FMT, true><<<blocks, threads, 0, s>>>(g, a);
      else k_dense_accumulate<F, FMT, false><<<blocks, threads, 0, s>>>(g, a);
    } else {
      k_dense_accumulate<F, FMT, false><<<blocks, threads, 0, s>>>(g, a);
    }
  }
  return cudaGetLastError();
}

template <int F>
static cudaError_t run_dense_f(Op op, int fmt, const Dense3DView& g, const LookupArgs& a,
                               cudaStream_t s) {
  if (fmt == STF_FMT_F32) return run_dense<F, STF_FMT_F32>(op, g, a, s);
  if (fmt == STF_FMT_F16) return run_dense<F, STF_FMT_F16>(op, g, a, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_dense3d(Op op, int filter, int fmt, const Dense3DView& g, const LookupArgs& a,
                           cudaStream_t s) {
  switch (filter) {
    case STF_FILTER_LINEAR: return run_dense_f<STF_FILTER_LINEAR>(op, fmt, g, a, s);
    case STF_FILTER_BSPLINE3: return run_dense_f<STF_FILTER_BSPLINE3>(op, fmt, g, a, s);
    case STF_FILTER_CATMULL_ROM: return run_dense_f<STF_FILTER_CATMULL_ROM>(op, fmt, g, a, s);
    case STF_FILTER_CATMULL_ROM_POSITIVIZED:
      return run_dense_f<STF_FILTER_CATMULL_ROM_POSITIVIZED>(op, fmt, g, a, s);
    case STF_FILTER_FIS_LINEAR: return run_dense_f<STF_FILTER_FIS_LINEAR>(op, fmt, g, a, s);
    case STF_FILTER_FIS_BSPLINE3: return run_dense_f<STF_FILTER_FIS_BSPLINE3>(op, fmt, g, a, s);
    case STF_FILTER_FIS_GAUSSIAN: return run_dense_f<STF_FILTER_FIS_GAUSSIAN>(op, fmt, g, a, s);
  }
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------- create-time kernels

__global__ void k_convert_f32(const float* __restrict__ src, void* __restrict__ dst, int fmt,
                              int64_t n) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const float v = src[i];
    if (fmt == STF_FMT_F16) reinterpret_cast<__half*>(dst)[i] = __float2half_rn(v);
    else reinterpret_cast<float*>(dst)[i] = v;
  }
}

cudaError_t launch_convert_f32(const float* src, void* dst, int fmt, int64_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_convert_f32<<<grid_blocks(n, 256), 256, 0, s>>>(src, dst, fmt, n);
  return cudaGetLastError();
}

// One level of a 2x2 box pyramid from the level above it (w x h x c floats):
// ((a + b) + (c + d)) / 4, or the mean of 2 where one dimension is already 1.
__global__ void k_box_mip(const float* __restrict__ src, float* __restrict__ dst, int w, int h,
                          int c) {
  const int w2 = max(1, w >> 1), h2 = max(1, h >> 1);
  const int64_t n = (int64_t)w2 * h2 * c;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const int ch = (int)(i % c);
    const int64_t p = i / c;
    const int x = (int)(p % w2), y = (int)(p / w2);
    const int x0 = (w > 1) ? 2 * x : x, x1 = (w > 1) ? 2 * x + 1 : x;
    const int y0 = (h > 1) ? 2 * y : y, y1 = (h > 1) ? 2 * y + 1 : y;
    const float a = src[((int64_t)y0 * w + x0) * c + ch], b = src[((int64_t)y0 * w + x1) * c + ch];
    const float d = src[((int64_t)y1 * w + x0) * c + ch], e = src[((int64_t)y1 * w + x1) * c + ch];
    dst[i] = __fmul_rn(__fadd_rn(__fadd_rn(a, b), __fadd_rn(d, e)), 0.25f);
  }
}

cudaError_t launch_box_mip(const float* src, float* dst, int w, int h, int c, cudaStream_t s) {
  const int64_t n = (int64_t)max(1, w >> 1) * max(1, h >> 1) * c;
  k_box_mip<<<grid_blocks(n, 256), 256, 0, s>>>(src, dst, w, h, c);
  return cudaGetLastError();
}

}  // namespace stf
