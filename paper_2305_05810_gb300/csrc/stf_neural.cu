// Neural textures: latent MIP levels decoded by an 8 -> 64 -> 64 -> 7 ReLU MLP on
// the tensor cores (binary16 operands, float32 accumulation).
//
// The paper motivates stochastic filtering for decoders that are expensive to run
// per texel, neural texture representations among them (Section 1; Section 5.2,
// "Texture compression"): the stochastic lookup picks one latent texel with the same
// inverse-CDF tap choice as a plain 2D texture and decodes it once; the
// deterministic lookup decodes every tap and filters the decoded values.
//
// The stochastic and the deterministic decode and the training (forward, backward and
// weight gradients) run on the fifth-generation tensor cores: tcgen05.mma on 128-row
// tiles, operands in shared memory, accumulators in tensor memory (see the tcgen05
// sections below).
#include <cstddef>
#include <math.h>

#include "stf_internal.h"
#include "stf_memory.h"
#include "stf_once.h"
#include "stf_round.h"

namespace stf {

namespace nn {

constexpr int P_W1 = 0, P_B1 = 512, P_W2 = 576, P_B2 = 4672, P_W3 = 4736, P_B3 = 5184;
constexpr int NPARAM = STF_NEURAL_PARAMS;
static_assert(NPARAM == 5191, "parameter count");

// binary16 weight images (halves): w1t[64][24] = W1^T (k >= 8 zero), w2t[64][72] = W2^T,
// w3t[8][72] = W3^T (row 7 zero); backward: w2r[64][72] = W2, w3r[64][8] = W3 (col 7
// zero), w1r[8][72] = W1.
constexpr int I_W1T = 0, I_W2T = 1536, I_W3T = 6144, I_W2R = 6720, I_W3R = 11328, I_W1R = 11840;
constexpr int IMG_ALL = 12416;
constexpr int NBIAS = 136;   // b1[64], b2[64], b3[8] (b3[7] = 0)

}  // namespace nn

// ---------------------------------------------------------------- binary16 pairs

__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ float2 unpack_h2(uint32_t w) {
  return __half22float2(*reinterpret_cast<const __half2*>(&w));
}

// ---------------------------------------------------------------- lookups


__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// Per-lane state of one 32-query chunk between tap choice and output.
struct NeuralPick {
  int64_t j;      // caller's query slot
  float sigma;    // estimator scale (Catmull-Rom)
  int mode;       // 0: no texel (background), 1: decode the latent, 2: stored fallback texel
};

// Tap choice for query i of the chunk; starts the 16-byte gather of the chosen texel
// (latent or fallback) into the lane's shared-memory row.  SLIM: the call has no
// binning permutation and no tap output, so the caller's index is i.
// uv and lod of query i (zeros past the end).
struct QueryCoords {
  float2 uv;
  float lod;
};
__device__ __forceinline__ QueryCoords load_coords(const LookupArgs& a, int64_t i) {
  QueryCoords q;
  q.uv = make_float2(0.0f, 0.0f);
  q.lod = 0.0f;
  if (i < a.n) {
    q.uv = reinterpret_cast<const float2*>(a.coords)[i];
    q.lod = a.lod ? a.lod[i] : 0.0f;
  }
  return q;
}

template <int F, bool SLIM = false>
__device__ __forceinline__ NeuralPick neural_pick(const NeuralDev& nd, const LookupArgs& a, int64_t i,
                                                  uint4* row, const QueryCoords* pre = nullptr) {
  NeuralPick pk;
  pk.j = 0;
  pk.sigma = 1.0f;
  pk.mode = 0;
  if (i >= a.n) return pk;
  pk.j = SLIM ? i : query_slot(a, i);
  const QueryCoords qc = pre ? *pre : load_coords(a, i);
  const float2 uv = qc.uv;
  const float lod = qc.lod;
  const uint4 r = query_variates(a, pk.j, a.sample_index);
  int L = 0;
  if (a.lod != nullptr && nd.nlev > 1) {
    const float lc = fminf(fmaxf(lod, 0.0f), (float)(nd.nlev - 1));
    L = min((int)floorf(__fadd_rn(lc, a.level_mode == STF_LEVEL_NEAREST ? 0.5f : unit24(r.w))), nd.nlev - 1);
  }
  const int w = nd.lvl_w[L], h = nd.lvl_h[L];
  float x[2] = {__fsub_rn(__fmul_rn(uv.x, (float)w), 0.5f), __fsub_rn(__fmul_rn(uv.y, (float)h), 0.5f)};
  const bool ok = prepare_coords<2>(x) && isfinite(lod);
  int idx[2] = {0, 0};
  if (ok) pk.sigma = pick_taps_r<F, 2, false>(x, r, idx);
  // (the tap goes out here: carried to the tile's end, two tiles' taps were eight registers)
  if (!SLIM && a.taps) reinterpret_cast<int4*>(a.taps)[pk.j] = ok ? make_int4(idx[0], idx[1], 0, L) : make_int4(0, 0, 0, -1);
  if (!ok) return pk;
  const int cx = min(max(idx[0], 0), w - 1), cy = min(max(idx[1], 0), h - 1);
  const __half* base = L < nd.nlat ? nd.lat16 : nd.fb16;
  cp_async16(row, base + (nd.lvl_off[L] + (int64_t)cy * w + cx) * 8);
  pk.mode = L < nd.nlat ? 1 : 2;
  return pk;
}

// ---------------------------------------------------------------- tcgen05 decode
//
// The stochastic decode on the fifth-generation tensor cores: for a tile of 128
// queries (one per thread) the chosen latent texels are gathered into a shared-memory
// A tile; one elected thread issues the three layers as tcgen05.mma (M = 128, binary16
// operands from shared memory, float32 accumulators in tensor memory); after each
// layer (its bias included) every thread loads its own accumulator row with tcgen05.ld,
// applies ReLU, rounds to binary16 and writes the next layer's A operand: layer 2's to a
// tile in shared memory, layer 3's to tensor memory.  Operand tiles
// use the no-swizzle K-major layout: 8-row x 16-byte core matrices, core matrices
// along K 128 bytes apart (LBO), 8-row groups K/8 * 128 bytes apart (SBO).

namespace tc {

constexpr int ROWS = 128;            // queries per tile = threads per group
constexpr int TMEM_COLS = 128;       // 64 columns per group: D1/D2 in 0..63, then layer 3's A in 0..31, D3 in 32..47
constexpr int A1_BYTES = ROWS * 16 * 2, A2_BYTES = ROWS * 64 * 2;
constexpr int B1_BYTES = 64 * 16 * 2, B2_BYTES = 64 * 64 * 2, B3_BYTES = 16 * 64 * 2;

// byte offset of element (r, k) in an R x K tile (K = 16 or 64)
__host__ __device__ constexpr int off(int r, int k, int K) {
  return (r >> 3) * (K / 8) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

// Descriptor of the K-major tile `bytes` after the shared-memory address whose field is
// `base` (base_of): next core matrix along K 128 bytes on (LBO), next 8-row group K/8 * 128
// (SBO), descriptor version, no swizzle.  The sum needs no masks or shifts where the MMAs
// are issued.
__device__ __forceinline__ uint32_t base_of(const void* p) { return ((uint32_t)__cvta_generic_to_shared(p) & 0x3FFFF) >> 4; }
__device__ __forceinline__ uint64_t desc_at(uint32_t base, uint32_t bytes, int K) {
  const uint32_t lo = base + (bytes >> 4) + ((128u >> 4) << 16), hi = (uint32_t)((K / 8) * 128) >> 4 | 1u << 14;
  return (uint64_t)hi << 32 | lo;
}

// The same with the 8-row-group stride set to 0: every group of 8 rows reads the same
// two core matrices, so one 8-row tile stands for a 128-row operand whose rows are
// all equal.
__device__ __forceinline__ uint64_t desc_rows_repeated(uint32_t base, uint32_t bytes) {
  return (uint64_t)(1u << 14) << 32 | (base + (bytes >> 4) + ((128u >> 4) << 16));
}

// kind::f16 instruction descriptor: F32 accumulate, F16 A and B, both K-major.
__host__ __device__ constexpr uint32_t idesc(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}

// The same with A in tensor memory: lane = row, each 32-bit column two consecutive k.
__device__ __forceinline__ void mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(id), "r"(acc));
}

__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
      (uint32_t)__cvta_generic_to_shared(bar)));
}

// Wait for phase `parity` of the mbarrier; false on timeout.  Each try_wait may suspend
// the thread for up to 20 us, waking it when the phase completes, so the waiting lane
// does not spin on the issue slots its warp shares with the computing warps; at most
// 2^16 tries (about 1.3 s).
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(bar);
  uint32_t done = 0;
  for (int it = 0; it < (1 << 16) && !done; ++it) {
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done) : "r"(a), "r"(parity), "r"(20000u));
  }
  return done != 0;
}

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r);

template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
}

template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
}

template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]));
}

// The forward weights as K-major no-swizzle B tiles (threads tid, tid + nt, ...):
// W1^T (64 x 16) with its bias split into binary16 (hi, lo) in k 8, 9; W2^T (64 x 64);
// W3^T (16 x 64, rows >= 7 zero); the b2 and b3 bias chunks (64 x 16, 16 x 16) with
// (hi, lo) in k 0, 1; and one 8-row group of ones in columns 0, 1.  A bias b enters the
// accumulator as b_hi + b_lo, b_hi = fp16(b), b_lo = fp16(b - b_hi): to about 2^-22 |b|.
__device__ __forceinline__ void stage_fwd_weights(const NeuralDev& nd, unsigned char* b1, unsigned char* b2,
                                                  unsigned char* b3, unsigned char* b2x, unsigned char* b3x,
                                                  unsigned char* ones, int tid, int nt) {
  const uint4* img = reinterpret_cast<const uint4*>(nd.wimg);
  auto split = [](float b) -> uint32_t {
    const __half hi = __float2half_rn(b);
    const __half lo = __float2half_rn(b - __half2float(hi));
    return (uint32_t)__half_as_ushort(hi) | ((uint32_t)__half_as_ushort(lo) << 16);
  };
  const uint4 z = make_uint4(0, 0, 0, 0);
  for (int n = tid; n < 64; n += nt) {
    *reinterpret_cast<uint4*>(b1 + off(n, 0, 16)) = __ldg(img + (nn::I_W1T + n * 24) / 8);
    *reinterpret_cast<uint4*>(b1 + off(n, 8, 16)) = make_uint4(split(__ldg(nd.bias + n)), 0, 0, 0);
    *reinterpret_cast<uint4*>(b2x + off(n, 0, 16)) = make_uint4(split(__ldg(nd.bias + 64 + n)), 0, 0, 0);
    *reinterpret_cast<uint4*>(b2x + off(n, 8, 16)) = z;
  }
  for (int n = tid; n < 16; n += nt) {
    const uint32_t b = n < 7 ? split(__ldg(nd.bias + 128 + n)) : 0u;
    *reinterpret_cast<uint4*>(b3x + off(n, 0, 16)) = make_uint4(b, 0, 0, 0);
    *reinterpret_cast<uint4*>(b3x + off(n, 8, 16)) = z;
  }
  for (int r = tid; r < 8; r += nt) {
    *reinterpret_cast<uint4*>(ones + off(r, 0, 16)) = make_uint4(0x3C003C00u, 0, 0, 0);
    *reinterpret_cast<uint4*>(ones + off(r, 8, 16)) = z;
  }
  for (int e = tid; e < 64 * 8; e += nt) {
    const int n = e >> 3, kc = e & 7;
    *reinterpret_cast<uint4*>(b2 + off(n, 8 * kc, 64)) = __ldg(img + (nn::I_W2T + n * 72 + 8 * kc) / 8);
  }
  for (int e = tid; e < 16 * 8; e += nt) {
    const int n = e >> 3, kc = e & 7;
    *reinterpret_cast<uint4*>(b3 + off(n, 8 * kc, 64)) = n < 8 ? __ldg(img + (nn::I_W3T + n * 72 + 8 * kc) / 8) : z;
  }
}

struct Group {                       // one tile in flight
  unsigned char a1[A1_BYTES];
  unsigned char a2[A2_BYTES];          // H1, then the staged output rows
  uint64_t bar;
  int32_t dead, pad;                   // a warp gave up: its rows of the staged ones are not there
};

struct Smem {
  unsigned char b1[B1_BYTES];          // W1^T in k 0..7, (b1_hi, b1_lo) in k 8, 9
  unsigned char b2[B2_BYTES];
  unsigned char b3[B3_BYTES];
  unsigned char b2x[64 * 16 * 2];      // (b2_hi, b2_lo) in k 0, 1
  unsigned char b3x[16 * 16 * 2];      // (b3_hi, b3_lo) in k 0, 1
  unsigned char ones[8 * 16 * 2];      // one 8-row group: 1 in columns 0, 1
  Group grp[2];
  uint32_t tmem;
};
// A2 doubles as the 16-byte-aligned staging area of the output rows
static_assert(offsetof(Smem, grp) % 16 == 0 && offsetof(Group, a2) % 16 == 0 && sizeof(Group) % 16 == 0,
              "A2 tiles are 16-byte aligned");

}  // namespace tc

// Hidden layer epilogue: D (64 float32 per row, tensor memory, bias included by the
// MMA) -> ReLU -> binary16 row of the next A tile, 16 columns per tensor-memory load:
// 32-column loads left the stochastic decode spilling at its 64-register cap and made
// it 26% slower.
__device__ __forceinline__ void tc_hidden(uint32_t taddr, unsigned char* a2, int row) {
#pragma unroll
  for (int half = 0; half < 4; ++half) {
    uint32_t r[16];
    tc::tmem_ld<16>(taddr + 16 * half, r);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = 8 * q + 2 * e;
        const float lo = __uint_as_float(r[c]);
        const float hi = __uint_as_float(r[c + 1]);
        // ReLU and round to binary16 in one instruction (the first source goes to the
        // upper half)
        asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(w[e]) : "f"(hi), "f"(lo));
      }
      *reinterpret_cast<uint4*>(a2 + tc::off(row, 16 * half + 8 * q, 64)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// The same for the last hidden layer, whose row goes back to tensor memory as layer 3's A
// operand: in place, 16 columns of D become 8 of A at or below them, so a tile still
// takes 64 columns (A in 0..31, D3 in 32..47).  Through shared memory the rows took 128 of
// a tile's 558 wavefronts to write and as much again for the MMA to read, in a decode that
// the shared-memory pipe bounded (68% busy; now 53%): 16.8 M stochastic lookups 425 us,
// 382 us this way.
__device__ __forceinline__ void tc_hidden_tmem(uint32_t taddr) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t r[16], w[8];
    tc::tmem_ld<16>(taddr + 16 * q, r);
#pragma unroll
    for (int e = 0; e < 8; ++e)
      asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(w[e]) : "f"(__uint_as_float(r[2 * e + 1])), "f"(__uint_as_float(r[2 * e])));
    tc::tmem_st8(taddr + 8 * q, w);
  }
  asm volatile("tcgen05.wait::st.sync.aligned;");
}

// One thread of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p != 0;
}

// RoundOf's hardware: the named barrier 1 + g of the group's 128 threads, and an mbarrier.
struct MmaGroup {
  using Bar = uint64_t*;
  static __device__ __forceinline__ void before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
  static __device__ __forceinline__ void after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
  static __device__ __forceinline__ void sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); }
  static __device__ __forceinline__ void arrive(int g) { asm volatile("bar.arrive %0, 128;" ::"r"(1 + g) : "memory"); }
  template <class Issue>
  static __device__ __forceinline__ void issue_and_commit(Issue issue, uint64_t* bar) {
    if (elect_one()) {
      issue();
      tc::commit(bar);
    }
    __syncwarp();
  }
  static __device__ __forceinline__ bool wait(uint64_t* bar, uint32_t parity) {
    return __all_sync(0xffffffffu, tc::wait_bar(bar, parity));
  }
};
using Round = RoundOf<MmaGroup>;

__device__ __forceinline__ void fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Layer 3 from the A operand in columns 0..31: D3 (128 x 16) in columns 32..47, bias included.
template <class S>
__device__ __forceinline__ void tc_layer3(uint32_t tmem, uint32_t sb) {
#pragma unroll
  for (int kk = 0; kk < 4; ++kk)
    tc::mma_ts(tmem + 32, tmem + 8 * kk, tc::desc_at(sb, offsetof(S, b3) + kk * 256, 64), tc::idesc(128, 16), kk);
  tc::mma(tmem + 32, tc::desc_rows_repeated(sb, offsetof(S, ones)), tc::desc_at(sb, offsetof(S, b3x), 16), tc::idesc(128, 16), 1);
}

// Layers 1 and 2 from A tiles at a1 and a2 (fields of their addresses): D in columns 0..63.
template <class S>
__device__ __forceinline__ void tc_layer1(uint32_t tmem, uint32_t sb, uint32_t a1) {
  tc::mma(tmem, tc::desc_at(a1, 0, 16), tc::desc_at(sb, offsetof(S, b1), 16), tc::idesc(128, 64), 0);
}
template <class S>
__device__ __forceinline__ void tc_layer2(uint32_t tmem, uint32_t sb, uint32_t a2, int K) {
#pragma unroll
  for (int kk = 0; kk < 4; ++kk)
    tc::mma(tmem, tc::desc_at(a2, kk * 256, K), tc::desc_at(sb, offsetof(S, b2) + kk * 256, 64), tc::idesc(128, 64), kk);
  tc::mma(tmem, tc::desc_rows_repeated(sb, offsetof(S, ones)), tc::desc_at(sb, offsetof(S, b2x), 16), tc::idesc(128, 64), 1);   // + b2
}

// Named barrier of one 128-thread group.
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); }

// Start of a decode CTA of two groups: the weights and the constant columns of the A
// tiles in shared memory, the mbarriers, tensor memory.  Returns the caller's group's first
// column.
__device__ __forceinline__ uint32_t decode_begin(tc::Smem& s, const NeuralDev& nd) {
  const int tid = threadIdx.x, g = tid >> 7, row = tid & 127;
  tc::stage_fwd_weights(nd, s.b1, s.b2, s.b3, s.b2x, s.b3x, s.ones, tid, 256);
  // columns 8..15 of A1: the ones that multiply W1's bias rows, then zeros (the
  // gathers write columns 0..7 only)
  *reinterpret_cast<uint4*>(s.grp[g].a1 + tc::off(row, 8, 16)) = make_uint4(0x3C003C00u, 0, 0, 0);
  if (row == 0) {
    s.grp[g].dead = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(&s.grp[g].bar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&s.tmem)), "n"(tc::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  return __shfl_sync(0xffffffffu, s.tmem + 64 * g, 0);
}

__device__ __forceinline__ void decode_end(tc::Smem& s, const NeuralDev& nd, int warp, const Round& round) {
  cp_async_wait<0>();
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (round.dead) atomicOr(nd.status, STF_DEV_MMA_TIMEOUT);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s.tmem), "n"(tc::TMEM_COLS));
}

// Two groups of 128 threads per CTA decode two tiles concurrently: each group owns an
// A1/A2 tile pair, 64 tensor-memory columns (D1, D2, then layer 3's A operand and D3), an
// mbarrier and a named barrier, and walks its own tile sequence;
// while one group waits on its MMAs or its gathers the other computes.  The weights
// are shared.  A group's A1 is refilled with the next tile's gather as soon as layer 1
// has consumed it, and the coordinates of the tile after that are loaded right then, a
// whole tile ahead of its tap choice (6% sooner than loading them at the choice).
//
// SLIM (calls without a binning permutation or tap output) compiles out the per-query
// caller index and tap, which leaves the registers the epilogues need at the
// 64-register cap of four CTAs per SM.
template <int F, bool SLIM>
__global__ void __launch_bounds__(256, 4) k_neural_stochastic_tc(NeuralDev nd, LookupArgs a) {
  extern __shared__ __align__(1024) unsigned char dyn[];
  tc::Smem& s = *reinterpret_cast<tc::Smem*>(dyn);
  const uint32_t tmem = decode_begin(s, nd);                      // this group's columns
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int g = warp >> 2, row = tid & 127;          // group, row of the group's tile
  tc::Group& G = s.grp[g];
  const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);  // this warp's lanes
  Round round{&G.bar, 0, g, (warp & 3) == 0, false};
  const uint32_t sb = tc::base_of(&s), a1 = tc::base_of(G.a1), a2 = tc::base_of(G.a2);
  const int64_t ntiles = (a.n + tc::ROWS - 1) / tc::ROWS;
  const int64_t step = 2 * (int64_t)gridDim.x;
  int64_t tile = 2 * (int64_t)blockIdx.x + g;
  uint4* arow = reinterpret_cast<uint4*>(G.a1 + tc::off(row, 0, 16));
  NeuralPick cur;
  if (tile < ntiles) cur = neural_pick<F, SLIM>(nd, a, tile * tc::ROWS + row, arow);
  cp_async_commit();
  // coordinates of the next tile, loaded a whole tile ahead of its tap choice
  QueryCoords qn = load_coords(a, (tile + step) * tc::ROWS + row);
  // barrier phases of a tile, and those still to come in it where a wait runs out
  const int phases = SLIM || a.perm == nullptr ? 4 : 3;
  int left = -1;
  for (; tile < ntiles; tile += step) {
    cp_async_wait<0>();
    uint4 fb = make_uint4(0, 0, 0, 0);
    if (cur.mode == 2) fb = *arow;                   // stored fallback texel (own row)
    fence_smem();
    left = phases - 1;
    if (!round([&] { tc_layer1<tc::Smem>(tmem, sb, a1); })) break;
    tc_hidden(trow, G.a2, row);
    fence_smem();
    round.start([&] { tc_layer2<tc::Smem>(tmem, sb, a2, 64); });
    // while layer 2 runs (A1 is free): the next tile's tap choices and gather
    const int64_t next = tile + step;
    NeuralPick nxt;
    if (next < ntiles) nxt = neural_pick<F, SLIM>(nd, a, next * tc::ROWS + row, arow, &qn);
    cp_async_commit();
    qn = load_coords(a, (next + step) * tc::ROWS + row);
    left = phases - 2;
    if (!round.finish()) break;
    tc_hidden_tmem(trow);
    left = phases - 3;
    if (!round([&] { tc_layer3<tc::Smem>(tmem, sb); })) break;
    left = -1;
    float v[8];
    {
      uint32_t r[8];
      tc::tmem_ld<8>(trow + 32, r);
#pragma unroll
      for (int k = 0; k < 7; ++k) v[k] = __uint_as_float(r[k]);
    }
    if (cur.mode == 2) {
      const uint32_t* tw = reinterpret_cast<const uint32_t*>(&fb);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 f = unpack_h2(tw[k]);
        v[2 * k] = f.x;
        v[2 * k + 1] = f.y;
      }
    } else if (cur.mode == 0) {
#pragma unroll
      for (int k = 0; k < 7; ++k) v[k] = 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] *= cur.sigma;
    if (SLIM || a.perm == nullptr) {
      // stage the tile's rows in A2 (free now) and store them coalesced
      float* stage = reinterpret_cast<float*>(G.a2);
#pragma unroll
      for (int k = 0; k < 7; ++k) stage[row * 7 + k] = v[k];
      group_sync(g);
      const int nrows = G.dead ? 0 : (int)min((int64_t)tc::ROWS, a.n - tile * tc::ROWS);
      float* dst = a.out + tile * tc::ROWS * 7;
      if (nrows == tc::ROWS && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
        // a full tile: 896 floats as 224 16-byte copies
        const float4* src4 = reinterpret_cast<const float4*>(stage);
        float4* dst4 = reinterpret_cast<float4*>(dst);
        for (int e = row; e < tc::ROWS * 7 / 4; e += 128) dst4[e] = src4[e];
      } else {
        for (int e = row; e < nrows * 7; e += 128) dst[e] = stage[e];
      }
    } else if (tile * tc::ROWS + row < a.n) {
#pragma unroll
      for (int k = 0; k < 7; ++k) a.out[cur.j * 7 + k] = v[k];
    }
    cur = nxt;
    // the next iteration's first group barrier orders these reads of A2 before the
    // next tile writes it
  }
  if (left >= 0) {
    G.dead = 1;
    round.give_up(left, phases, tile, ntiles, step);
  }
  decode_end(s, nd, warp, round);
}

// Deterministic decode on the tensor cores: every tap of the filter window (at one
// level, or at two blended by frac(lod)) is a row of a 128-row tile; a query takes R =
// parts x T^2 consecutive rows (parts = 2 when the level is blended, else 1), so a tile
// holds 128 / R queries.  Each thread gathers its tap's latent texel into the A tile
// (zeros for fallback levels and for taps of queries without a texture value), the
// three layers run as in the stochastic decode, and each row's output times its
// weight (the tap weights wx wy times the level weight) is summed over the query's R
// rows.  Fallback levels use the stored texel.
// One row of a deterministic tile: its weight and texel kind.  The texel (latent
// or stored fallback) is gathered into the row of the A tile by cp.async.
struct DetRow {
  float w;       // tap weight times level weight (0: the row adds nothing)
  int mode;      // 0: nothing, 1: decode the latent, 2: stored fallback texel
};

template <int F>
__device__ __forceinline__ DetRow det_row(const NeuralDev& nd, const LookupArgs& a, int64_t i, int p, int tx,
                                          int ty, uint4* arow, const QueryCoords* pre = nullptr) {
  using Fl = Filter<F>;
  DetRow d;
  d.w = 0.0f;
  d.mode = 0;
  if (i >= a.n) return d;
  const QueryCoords qc = pre ? *pre : load_coords(a, i);
  const float2 uv = qc.uv;
  const float lod = qc.lod;
  if (!(isfinite(lod) && isfinite(uv.x) && isfinite(uv.y))) return d;
  float lw = p == 0 ? 1.0f : 0.0f;
  int L = 0;
  if (a.lod != nullptr && nd.nlev > 1) {
    const float lc = fminf(fmaxf(lod, 0.0f), (float)(nd.nlev - 1));
    if (a.level_mode == STF_LEVEL_NEAREST) {
      L = min((int)floorf(__fadd_rn(lc, 0.5f)), nd.nlev - 1);
    } else {
      const float fl = floorf(lc), fr = __fsub_rn(lc, fl);
      L = p == 0 ? (int)fl : min((int)fl + 1, nd.nlev - 1);
      lw = p == 0 ? 1.0f - fr : fr;
    }
  }
  const int w = nd.lvl_w[L], h = nd.lvl_h[L];
  float x[2] = {__fsub_rn(__fmul_rn(uv.x, (float)w), 0.5f), __fsub_rn(__fmul_rn(uv.y, (float)h), 0.5f)};
  if (!(lw > 0.0f) || !prepare_coords<2>(x)) return d;
  float fx, fy;
  const int bx = axis_base(x[0], fx) + Fl::OFF0, by = axis_base(x[1], fy) + Fl::OFF0;
  float wx[Fl::T], wy[Fl::T];
  Fl::weights(fx, wx);
  Fl::weights(fy, wy);
  float wxs = wx[0], wys = wy[0];
#pragma unroll
  for (int k = 1; k < Fl::T; ++k) {
    if (tx == k) wxs = wx[k];
    if (ty == k) wys = wy[k];
  }
  d.w = wxs * wys * lw;
  const int cx = min(max(bx + tx, 0), w - 1), cy = min(max(by + ty, 0), h - 1);
  const __half* base = L < nd.nlat ? nd.lat16 : nd.fb16;
  cp_async16(arow, base + (nd.lvl_off[L] + (int64_t)cy * w + cx) * 8);
  d.mode = L < nd.nlat ? 1 : 2;
  return d;
}

// As in the stochastic decode, two groups of 128 threads per CTA and four CTAs per SM keep
// eight tiles in flight on one copy of the weights per pair (six one-group CTAs fitted:
// 307 us against 281 us for 4.2 M bilinear lookups).
template <int F>
__global__ void __launch_bounds__(256, 4) k_neural_deterministic_tc(NeuralDev nd, LookupArgs a) {
  using Fl = Filter<F>;
  extern __shared__ __align__(1024) unsigned char dyn[];
  tc::Smem& s = *reinterpret_cast<tc::Smem*>(dyn);
  const uint32_t tmem = decode_begin(s, nd);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int g = warp >> 2, row = tid & 127;
  tc::Group& G = s.grp[g];
  const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  uint4* arow = reinterpret_cast<uint4*>(G.a1 + tc::off(row, 0, 16));
  Round round{&G.bar, 0, g, (warp & 3) == 0, false};
  const uint32_t sb = tc::base_of(&s), a1 = tc::base_of(G.a1), a2 = tc::base_of(G.a2);
  constexpr int T2 = Fl::T * Fl::T;
  const int parts = (a.lod != nullptr && nd.nlev > 1 && a.level_mode != STF_LEVEL_NEAREST) ? 2 : 1;
  const int R = parts * T2;                    // rows per query: 4, 8, 16 or 32
  const int Q = 128 / R;                       // queries per tile
  const int qi = row / R, sub = row % R, p = sub / T2, tap = sub % T2;
  const int tx = tap % Fl::T, ty = tap / Fl::T;
  const int64_t ntiles = (a.n + Q - 1) / Q;
  const int64_t step = 2 * (int64_t)gridDim.x;
  int64_t tile = 2 * (int64_t)blockIdx.x + g;
  DetRow cur;
  if (tile < ntiles) cur = det_row<F>(nd, a, tile * Q + qi, p, tx, ty, arow);
  cp_async_commit();
  QueryCoords qn = load_coords(a, (tile + step) * Q + qi);        // a tile ahead
  int left = -1;                               // barrier phases still to come in the tile, where a wait runs out
  for (; tile < ntiles; tile += step) {
    cp_async_wait<0>();
    uint4 fb = make_uint4(0, 0, 0, 0);
    if (cur.mode == 2) fb = *arow;               // stored fallback texel (own row)
    if (cur.mode != 1) *arow = make_uint4(0, 0, 0, 0);
    fence_smem();
    left = 2;
    if (!round([&] { tc_layer1<tc::Smem>(tmem, sb, a1); })) break;
    tc_hidden(trow, G.a2, row);
    fence_smem();
    round.start([&] { tc_layer2<tc::Smem>(tmem, sb, a2, 64); });
    // while layer 2 runs (A1 is free): the next tile's taps and gather
    const int64_t next = tile + step;
    DetRow nxt;
    if (next < ntiles) nxt = det_row<F>(nd, a, next * Q + qi, p, tx, ty, arow, &qn);
    cp_async_commit();
    qn = load_coords(a, (next + step) * Q + qi);
    left = 1;
    if (!round.finish()) break;
    tc_hidden_tmem(trow);
    left = 0;
    if (!round([&] { tc_layer3<tc::Smem>(tmem, sb); })) break;
    left = -1;
    float v[8];
    {
      uint32_t r[8];
      tc::tmem_ld<8>(trow + 32, r);
#pragma unroll
      for (int k = 0; k < 7; ++k) v[k] = __uint_as_float(r[k]);
    }
    if (cur.mode == 2) {
      const uint32_t* tw = reinterpret_cast<const uint32_t*>(&fb);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 f = unpack_h2(tw[k]);
        v[2 * k] = f.x;
        v[2 * k + 1] = f.y;
      }
    }
    // Sum of the query's R rows, which are R consecutive lanes: each exchange halves the
    // channels a lane keeps (8, 4, 2, 1), further ones add single channels; a lane then
    // holds channels c and c + 1 (R = 4), or channel c (R >= 8).  Summed by one
    // thread from rows staged in shared memory, the stores' bank conflicts alone were 224
    // of a tile's 832 wavefronts.
    v[7] = 0.0f;
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = cur.mode ? cur.w * v[k] : 0.0f;
    const bool hi0 = tid & 1, hi1 = tid & 2, hi2 = tid & 4;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float o = __shfl_xor_sync(0xffffffffu, hi0 ? v[k] : v[k + 4], 1);
      v[k] = (hi0 ? v[k + 4] : v[k]) + o;
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float o = __shfl_xor_sync(0xffffffffu, hi1 ? v[k] : v[k + 2], 2);
      v[k] = (hi1 ? v[k + 2] : v[k]) + o;
    }
    int c = (hi0 ? 4 : 0) + (hi1 ? 2 : 0);
    if (R >= 8) {
      const float o = __shfl_xor_sync(0xffffffffu, hi2 ? v[0] : v[1], 4);
      v[0] = (hi2 ? v[1] : v[0]) + o;
      c += hi2 ? 1 : 0;
      if (R >= 16) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 8);
      if (R >= 32) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
    }
    const int64_t i = tile * Q + qi;
    if (i < a.n) {
      if (sub < 8 && c < 7) a.out[i * 7 + c] = v[0];
      if (R == 4 && c + 1 < 7) a.out[i * 7 + c + 1] = v[1];
    }
    cur = nxt;
  }
  if (left >= 0) round.give_up(left, 3, tile, ntiles, step);
  decode_end(s, nd, warp, round);
}

// ---------------------------------------------------------------- training

struct TrainArgs {
  const int64_t* ids;          // explicit texel ids (gradient check) or NULL
  const float* target_rows;    // explicit targets [B][7] or NULL
  const float* target_levels;  // targets [texel][7] (training)
  int64_t batch;
  float inv_batch;
  uint64_t seed;
  int64_t step;                // training step (permutation position and Adam t)
  float lr, beta1, beta2, eps;
  float* grads;                // parameter gradients, accumulated (16-byte aligned)
  float* loss;                 // accumulated sum of squared errors / batch
  float* dx_out;               // [B][8] latent gradients (gradient check) or NULL
  int train;                   // 1: Adam update of the latents in place
};

__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352dU;
  x ^= x >> 15;
  x *= 0x846ca68bU;
  x ^= x >> 16;
  return x;
}

// Seeded bijection of [0, n): a 4-round Feistel network on the smallest even-width
// power-of-two domain covering n, with cycle walking back into [0, n).
__device__ __forceinline__ int64_t permute_index(int64_t x, int64_t n, uint64_t seed) {
  int bits = 2;
  while ((1LL << bits) < n) bits += 2;
  const int h = bits / 2;
  const uint64_t mask = (1ull << h) - 1;
  uint64_t v = (uint64_t)x;
  for (int walk = 0; walk < 4096; ++walk) {
    uint64_t L = v >> h, R = v & mask;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint64_t f = mix32((uint32_t)R ^ (uint32_t)(seed >> (16 * r)) ^ (0x9E3779B9u * (r + 1))) & mask;
      const uint64_t nl = R;
      R = L ^ f;
      L = nl;
    }
    v = (L << h) | R;
    if ((int64_t)v < n) return (int64_t)v;
  }
  return x % n;   // unreachable in practice: cycles return to [0, n) within a few steps
}

// ---------------------------------------------------------------- tcgen05 training
//
// Forward and backward of the decoder and the parameter gradients for tiles of 128
// training texels on the fifth-generation tensor cores: six tcgen05.mma round trips per
// tile (M = 128, binary16 operands in shared memory, float32 accumulators in tensor
// memory), issued by one thread of a 128-thread group, each followed by an epilogue in
// which every thread reads its row:
//   1  H1 = ReLU(X W1 + b1)
//   2  H2 = ReLU(H1 W2 + b2)
//   3  Y = H2 W3 + b3, dY = 2 (Y - T) / B
//   4  dA2 = (dY W3^T) [H2 > 0]        and  [H1 | H2]^T dY    : dW3 in rows 64..127
//   5  dA1 = (dA2 W2^T) [H1 > 0]       and  [H1 | dA2]^T dA2  : dW2 in rows 0..63
//   6  dX = dA1 W1^T                   and  [dA1 | dA2]^T [X | 1] : dW1^T in rows 0..63,
//                                           db1 and db2 in the column of ones
// The gradients' reduction runs over the batch, the rows of the tiles: the tiles that are
// K-major operands of the layers are read as MN-major ones there, so nothing is
// transposed or written to memory.  dA2 and dA1 replace H2 and H1 in place once step 4
// and step 5 have read them.  The gradient accumulators stay in tensor memory over a
// group's tiles; the groups' sums meet in shared memory and one vector atomic add per
// four entries takes a CTA's to memory.  The biases enter the forward MMAs as an extra K
// chunk against columns of ones, as in the decode.
//
// A group takes 160 tensor-memory columns (64 for the layers, 96 for the gradients) and
// 40 KB of tiles: three groups fill an SM's 512 columns, and their waits overlap.  Per
// 65,536 texels (1024^2 texture): 33 us for the two passes and 54 us for a separate kernel that
// read the activations back and transposed them in shared memory, 30 us fused; bound by the
// latency of the six round trips and of the gathers.

namespace tct {

constexpr int GROUPS = 3;
constexpr int TMEM_COLS = 512;
constexpr int COLS = 160, C_W2 = 64, C_W3 = 128, C_W1 = 144;   // a group's columns: D, dW2, dW3, dW1

struct alignas(128) Group {
  unsigned char x[128 * 16 * 2];       // latents in k 0..7, ones in k 8, 9
  unsigned char dy[128 * 16 * 2];      // dY in k 0..6, zeros beyond
  unsigned char h[128 * 128 * 2];      // H1 in k 0..63, H2 in k 64..127; then dA1, dA2
  uint64_t bar;
  int abort, tiles;
};

struct Smem {
  unsigned char b1[tc::B1_BYTES];      // W1^T (64 x 16): k 0..7, biases (hi, lo) in k 8, 9
  unsigned char b2[tc::B2_BYTES];      // W2^T (64 x 64)
  unsigned char b3[tc::B3_BYTES];      // W3^T (16 x 64), rows >= 7 zero
  unsigned char b2x[64 * 16 * 2];      // (b2_hi, b2_lo) in k 0, 1
  unsigned char b3x[16 * 16 * 2];      // (b3_hi, b3_lo) in k 0, 1
  unsigned char ones[8 * 16 * 2];      // one 8-row group: 1 in columns 0, 1
  unsigned char r3[64 * 16 * 2];       // W3 (64 x 16): B of dY W3^T (k = output, < 7)
  unsigned char r2[64 * 64 * 2];       // W2 (64 x 64): B of dA2 W2^T
  unsigned char r1[16 * 64 * 2];       // W1 (16 x 64), rows >= 8 zero: B of dA1 W1^T
  Group grp[GROUPS];
  float sums[GROUPS * 4][8];           // per warp: db3, loss
  uint32_t tmem;
};
static_assert(offsetof(Smem, grp) % 128 == 0 && offsetof(Group, h) % 128 == 0, "tiles are 128-byte aligned");

// Descriptor of a tile stored with K columns of 16-bit values per row, read as an
// MN-major operand (no swizzle) from column c0: M or N runs along the columns (core
// matrices of 8 columns x 8 rows, 128 bytes apart), K along the rows (8-row groups
// K/8 * 128 bytes apart).  Rows 16 j .. 16 j + 15 start j * K/8 * 256 bytes further.
__device__ __forceinline__ uint64_t desc_mn(uint32_t base, int c0, int j, int K) {
  const uint32_t lo = base + (((c0 >> 3) * 128 + j * (K / 8) * 256) >> 4) +
                      ((uint32_t)(((K / 8) * 128) >> 4) << 16);       // next 8 rows
  const uint32_t hi = (128u >> 4) | 1u << 14;                         // next 8 columns; version
  return (uint64_t)hi << 32 | lo;
}

// Both operands MN-major.
__host__ __device__ constexpr uint32_t idesc_mn(int M, int N) { return tc::idesc(M, N) | (1u << 15) | (1u << 16); }

}  // namespace tct

// Forward hidden epilogue: D -> ReLU -> binary16 -> columns c0 .. c0 + 63 of the row.
__device__ __forceinline__ void tct_hidden(uint32_t taddr, unsigned char* h, int c0, int row) {
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    uint32_t r[32];
    tc::tmem_ld<32>(taddr + 32 * half, r);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = 8 * q + 2 * e;
        asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(w[e]) : "f"(__uint_as_float(r[c + 1])), "f"(__uint_as_float(r[c])));
      }
      *reinterpret_cast<uint4*>(h + tc::off(row, c0 + 32 * half + 8 * q, 128)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// Backward epilogue, in place: D (64 float32), kept where the activation in the row's
// columns c0 .. c0 + 63 is > 0 (the ReLU derivative), replaces it as binary16.
__device__ __forceinline__ void tct_masked(uint32_t taddr, unsigned char* h, int c0, int row) {
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    uint32_t r[32];
    tc::tmem_ld<32>(taddr + 32 * half, r);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint4* p = reinterpret_cast<uint4*>(h + tc::off(row, c0 + 32 * half + 8 * q, 128));
      const uint4 m = *p;
      const uint32_t mw[4] = {m.x, m.y, m.z, m.w};
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = 8 * q + 2 * e;
        const float2 a = unpack_h2(mw[e]);
        w[e] = pack_h2(a.x > 0.f ? __uint_as_float(r[c]) : 0.f, a.y > 0.f ? __uint_as_float(r[c + 1]) : 0.f);
      }
      *p = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// One texel of a training batch: its latents and target (zeros past the end).
struct TrainRow {
  int64_t id, epoch;
  float x[8], t[7];
  bool live;
  __device__ __forceinline__ void load(const NeuralDev& nd, const TrainArgs& ta, int64_t r) {
    live = r < ta.batch;
    id = epoch = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = 0.0f;
#pragma unroll
    for (int k = 0; k < 7; ++k) t[k] = 0.0f;
    if (!live) return;
    if (ta.ids) {
      id = ta.ids[r];
    } else {
      const int64_t gp = ta.step * ta.batch + r;
      epoch = gp / nd.n_lat_texels;
      id = permute_index(gp % nd.n_lat_texels, nd.n_lat_texels, ta.seed);
    }
    const float4 x0 = reinterpret_cast<const float4*>(nd.lat32 + id * 8)[0];
    const float4 x1 = reinterpret_cast<const float4*>(nd.lat32 + id * 8)[1];
    x[0] = x0.x; x[1] = x0.y; x[2] = x0.z; x[3] = x0.w;
    x[4] = x1.x; x[5] = x1.y; x[6] = x1.z; x[7] = x1.w;
    const float* tp = ta.target_rows ? ta.target_rows + r * 7 : ta.target_levels + id * 7;
#pragma unroll
    for (int k = 0; k < 7; ++k) t[k] = tp[k];
  }
};

// A tile's texels are gathered ahead of its turn: the first one's before the weights are
// staged, the next one's during the backward round trips (a batch's texels are distinct, so
// the latents' update in between does not touch them).
__global__ void __launch_bounds__(128 * tct::GROUPS, 1) k_neural_train_tc(NeuralDev nd, TrainArgs ta) {
  extern __shared__ __align__(1024) unsigned char dyn[];
  tct::Smem& s = *reinterpret_cast<tct::Smem*>(dyn);
  constexpr int NT = 128 * tct::GROUPS;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int g = warp >> 2, row = tid & 127;
  tct::Group& G = s.grp[g];
  const int64_t ntiles = (ta.batch + 127) / 128;
  const int64_t step = (int64_t)gridDim.x * tct::GROUPS;
  int64_t tile = blockIdx.x + (int64_t)gridDim.x * g;
  TrainRow cur;
  cur.load(nd, ta, tile * 128 + row);
  {
    const uint4* img = reinterpret_cast<const uint4*>(nd.wimg);
    const uint4 z = make_uint4(0, 0, 0, 0);
    tc::stage_fwd_weights(nd, s.b1, s.b2, s.b3, s.b2x, s.b3x, s.ones, tid, NT);
    for (int n = tid; n < 64; n += NT) {       // W3 rows (k = output) for dY W3^T
      *reinterpret_cast<uint4*>(s.r3 + tc::off(n, 0, 16)) = __ldg(img + (nn::I_W3R + n * 8) / 8);
      *reinterpret_cast<uint4*>(s.r3 + tc::off(n, 8, 16)) = z;
    }
    for (int e = tid; e < 64 * 8; e += NT) {   // W2 rows for dA2 W2^T
      const int n = e >> 3, kc = e & 7;
      *reinterpret_cast<uint4*>(s.r2 + tc::off(n, 8 * kc, 64)) = __ldg(img + (nn::I_W2R + n * 72 + 8 * kc) / 8);
    }
    for (int e = tid; e < 16 * 8; e += NT) {   // W1 rows (rows >= 8 zero) for dA1 W1^T
      const int n = e >> 3, kc = e & 7;
      *reinterpret_cast<uint4*>(s.r1 + tc::off(n, 8 * kc, 64)) =
          n < 8 ? __ldg(img + (nn::I_W1R + n * 72 + 8 * kc) / 8) : z;
    }
    *reinterpret_cast<uint4*>(G.x + tc::off(row, 8, 16)) = make_uint4(0x3C003C00u, 0, 0, 0);
    *reinterpret_cast<uint4*>(G.dy + tc::off(row, 8, 16)) = z;
  }
  if (row == 0) {
    G.abort = G.tiles = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(&G.bar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    // (the tiles' shared memory keeps a second CTA of this kernel off the SM)
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&s.tmem)), "n"(tct::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = s.tmem + tct::COLS * g;
  const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);   // this warp's lanes
  Round round{&G.bar, 0, g, (warp & 3) == 0, false};
  const uint32_t sb = tc::base_of(&s), gx = tc::base_of(G.x), gdy = tc::base_of(G.dy), gh = tc::base_of(G.h);
  using S = tct::Smem;
  float sums[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // db3, sum of squared errors
  uint32_t more = 0;                          // 0 for the group's first tile: accumulators start from zero
  int left = -1;                              // barrier phases still to come in the tile, where a wait runs out
  for (; tile < ntiles; tile += step) {
    const int64_t r = tile * 128 + row;
    const bool live = cur.live;
    const float* X = cur.x;
    *reinterpret_cast<uint4*>(G.x + tc::off(row, 0, 16)) =
        make_uint4(pack_h2(X[0], X[1]), pack_h2(X[2], X[3]), pack_h2(X[4], X[5]), pack_h2(X[6], X[7]));
    fence_smem();
    left = 5;
    if (!round([&] { tc_layer1<S>(tmem, sb, gx); })) break;
    tct_hidden(trow, G.h, 0, row);
    fence_smem();
    left = 4;
    if (!round([&] { tc_layer2<S>(tmem, sb, gh, 128); })) break;
    tct_hidden(trow, G.h, 64, row);
    fence_smem();
    left = 3;
    if (!round([&] {
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        tc::mma(tmem, tc::desc_at(gh, 1024 + kk * 256, 128), tc::desc_at(sb, offsetof(S, b3) + kk * 256, 64),
                tc::idesc(128, 16), kk);
      tc::mma(tmem, tc::desc_rows_repeated(sb, offsetof(S, ones)), tc::desc_at(sb, offsetof(S, b3x), 16),
              tc::idesc(128, 16), 1);
    })) break;
    {
      uint32_t y[8];
      tc::tmem_ld<8>(trow, y);
      float d[8];
#pragma unroll
      for (int k = 0; k < 7; ++k) {
        const float e = live ? __uint_as_float(y[k]) - cur.t[k] : 0.0f;
        sums[7] = fmaf(e, e, sums[7]);
        d[k] = 2.0f * ta.inv_batch * e;
      }
      d[7] = 0.0f;
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        w[k] = pack_h2(d[2 * k], d[2 * k + 1]);
        const float2 f = unpack_h2(w[k]);
        sums[2 * k] += f.x;
        if (k < 3) sums[2 * k + 1] += f.y;
      }
      *reinterpret_cast<uint4*>(G.dy + tc::off(row, 0, 16)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    TrainRow nxt;
    nxt.load(nd, ta, (tile + step) * 128 + row);
    fence_smem();
    left = 2;
    if (!round([&] {
      tc::mma(tmem, tc::desc_at(gdy, 0, 16), tc::desc_at(sb, offsetof(S, r3), 16), tc::idesc(128, 64), 0);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        tc::mma(tmem + tct::C_W3, tct::desc_mn(gh, 0, j, 128), tct::desc_mn(gdy, 0, j, 16), tct::idesc_mn(128, 16),
                more | j);
    })) break;
    tct_masked(trow, G.h, 64, row);
    fence_smem();
    left = 1;
    if (!round([&] {
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        tc::mma(tmem, tc::desc_at(gh, 1024 + kk * 256, 128), tc::desc_at(sb, offsetof(S, r2) + kk * 256, 64),
                tc::idesc(128, 64), kk);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        tc::mma(tmem + tct::C_W2, tct::desc_mn(gh, 0, j, 128), tct::desc_mn(gh, 64, j, 128), tct::idesc_mn(128, 64),
                more | j);
    })) break;
    tct_masked(trow, G.h, 0, row);
    fence_smem();
    left = 0;
    if (!round([&] {
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        tc::mma(tmem, tc::desc_at(gh, kk * 256, 128), tc::desc_at(sb, offsetof(S, r1) + kk * 256, 64),
                tc::idesc(128, 16), kk);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        tc::mma(tmem + tct::C_W1, tct::desc_mn(gh, 0, j, 128), tct::desc_mn(gx, 0, j, 16), tct::idesc_mn(128, 16),
                more | j);
    })) break;
    left = -1;
    more = 1;
    float dx[8];
    {
      uint32_t q[8];
      tc::tmem_ld<8>(trow, q);
#pragma unroll
      for (int k = 0; k < 8; ++k) dx[k] = __uint_as_float(q[k]);
    }
    if (live) {
      if (ta.dx_out) {
#pragma unroll
        for (int k = 0; k < 8; ++k) ta.dx_out[r * 8 + k] = dx[k];
      }
      if (ta.train) {
        // Adam on this latent row; its update count is its epoch + 1 (one visit per epoch)
        const float tt = (float)(cur.epoch + 1);
        const float c1 = 1.0f - powf(ta.beta1, tt), c2 = 1.0f - powf(ta.beta2, tt);
        float xn[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int64_t e = cur.id * 8 + k;
          const float mm = ta.beta1 * nd.m_lat[e] + (1.0f - ta.beta1) * dx[k];
          const float vv = ta.beta2 * nd.v_lat[e] + (1.0f - ta.beta2) * dx[k] * dx[k];
          nd.m_lat[e] = mm;
          nd.v_lat[e] = vv;
          xn[k] = X[k] - ta.lr * (mm / c1) / (sqrtf(vv / c2) + ta.eps);
          nd.lat32[e] = xn[k];
        }
        reinterpret_cast<uint4*>(const_cast<__half*>(nd.lat16))[cur.id] =
            make_uint4(pack_h2(xn[0], xn[1]), pack_h2(xn[2], xn[3]), pack_h2(xn[4], xn[5]),
                       pack_h2(xn[6], xn[7]));
      }
    }
    cur = nxt;
  }
  if (left >= 0) round.give_up(left, 6, tile, ntiles, step);
  // The groups' gradients: groups 1 and 2 leave their rows in their own tiles, [column]
  // [row], group 0 adds them to its own and takes them to memory.
#pragma unroll
  for (int k = 0; k < 8; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sums[k] += __shfl_xor_sync(0xffffffffu, sums[k], o);
    if (lane == 0) s.sums[warp][k] = sums[k];
  }
  if (row == 0) G.tiles = (int)more;
  if (round.dead) G.abort = 1;
  float* stage = reinterpret_cast<float*>(G.h);       // dW2 64 x 64, then dW3 or dW1 and db 9 x 128
  const bool upper = row >= 64;
  uint32_t v[32];
  if (g > 0 && more) {
#pragma unroll
    for (int cb = 0; cb < 2; ++cb) {
      tc::tmem_ld<32>(trow + tct::C_W2 + 32 * cb, v);
      if (!upper)
#pragma unroll
        for (int n = 0; n < 32; ++n) stage[(32 * cb + n) * 64 + row] = __uint_as_float(v[n]);
    }
    tc::tmem_ld<16>(trow + tct::C_W3, v);
    tc::tmem_ld<16>(trow + tct::C_W1, v + 16);
#pragma unroll
    for (int n = 0; n < 9; ++n) stage[4096 + n * 128 + row] = __uint_as_float(upper && n < 7 ? v[n] : v[16 + n]);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  bool aborted = false;
#pragma unroll
  for (int k = 0; k < tct::GROUPS; ++k) aborted = aborted || s.grp[k].abort;
  if (g == 0 && more && !aborted) {                    // (group 0 has a tile if any has)
    auto others = [&](int at) {
      float a = 0.0f;
#pragma unroll
      for (int k = 1; k < tct::GROUPS; ++k)
        if (s.grp[k].tiles) a += reinterpret_cast<const float*>(s.grp[k].h)[at];
      return a;
    };
#pragma unroll
    for (int cb = 0; cb < 2; ++cb) {
      tc::tmem_ld<32>(trow + tct::C_W2 + 32 * cb, v);
      if (!upper)
#pragma unroll
        for (int n = 0; n < 32; n += 4) {
          float q[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) q[e] = __uint_as_float(v[n + e]) + others((32 * cb + n + e) * 64 + row);
          atomicAdd(reinterpret_cast<float4*>(ta.grads + nn::P_W2 + row * 64 + 32 * cb + n),
                    make_float4(q[0], q[1], q[2], q[3]));
        }
    }
    tc::tmem_ld<16>(trow + tct::C_W3, v);
    tc::tmem_ld<16>(trow + tct::C_W1, v + 16);
#pragma unroll
    for (int n = 0; n < 9; ++n) {
      const float q = __uint_as_float(upper && n < 7 ? v[n] : v[16 + n]) + others(4096 + n * 128 + row);
      if (upper) {
        if (n < 7) atomicAdd(ta.grads + nn::P_W3 + (row - 64) * 7 + n, q);
        if (n == 8) atomicAdd(ta.grads + nn::P_B2 + row - 64, q);
      } else {
        atomicAdd(ta.grads + (n < 8 ? nn::P_W1 + n * 64 : nn::P_B1) + row, q);
      }
    }
  }
  if (tid < 8 && !aborted) {
    float a = 0.0f;
#pragma unroll
    for (int w = 0; w < 4 * tct::GROUPS; ++w) a += s.sums[w][tid];
    if (tid < 7) atomicAdd(ta.grads + nn::P_B3 + tid, a);
    else atomicAdd(ta.loss, a * ta.inv_batch);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && aborted) atomicOr(nd.status, STF_DEV_MMA_TIMEOUT);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s.tmem), "n"(tct::TMEM_COLS));
}

// Forward, backward and parameter gradients of a batch (ta.grads and ta.loss zero before).
static cudaError_t launch_train_tc(const NeuralDev& nd, const TrainArgs& ta, cudaStream_t s) {
  const int smem = (int)sizeof(tct::Smem);
  static OncePerDevice once;
  const cudaError_t e = once([&] {
    return cudaFuncSetAttribute(k_neural_train_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  });
  if (e != cudaSuccess) return e;
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t ntiles = (ta.batch + 127) / 128;
  const int grid = (int)(ntiles < (int64_t)sms ? ntiles : (int64_t)sms);
  k_neural_train_tc<<<grid, 128 * tct::GROUPS, smem, s>>>(nd, ta);
  return cudaGetLastError();
}

// Parameter k as the kernels use it: binary16 in the weight images, or float32 bias.  (The
// images' padding and the last bias stay zero from the texture's creation.)
__device__ __forceinline__ void store_param(int k, float p, __half* img, float* bias) {
  const __half v = __float2half_rn(p);
  if (k < nn::P_B1) {                                  // W1[c][h]
    const int c = k / 64, h = k % 64;
    img[nn::I_W1T + h * 24 + c] = v;
    img[nn::I_W1R + c * 72 + h] = v;
  } else if (k < nn::P_W2) {
    bias[k - nn::P_B1] = p;
  } else if (k < nn::P_B2) {                           // W2[i][o]
    const int i = (k - nn::P_W2) / 64, o = (k - nn::P_W2) % 64;
    img[nn::I_W2T + o * 72 + i] = v;
    img[nn::I_W2R + i * 72 + o] = v;
  } else if (k < nn::P_W3) {
    bias[64 + k - nn::P_B2] = p;
  } else if (k < nn::P_B3) {                           // W3[h][o]
    const int h = (k - nn::P_W3) / 7, o = (k - nn::P_W3) % 7;
    img[nn::I_W3T + o * 72 + h] = v;
    img[nn::I_W3R + h * 8 + o] = v;
  } else {
    bias[128 + k - nn::P_B3] = p;
  }
}

constexpr int kParamBlocks = (nn::NPARAM + 255) / 256;   // one thread per parameter

__global__ void __launch_bounds__(256) k_neural_images(const float* params, __half* img, float* bias) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k < nn::NPARAM) store_param(k, params[k], img, bias);
}

// Adam on the MLP parameters (step t >= 1), their binary16 images, and the batch's loss
// copied out; gradients and loss are zero again after it, for the next batch.  One thread
// per parameter: on one block, the update and the rebuilt images took half of a training
// step of 65,536 texels (71 us a step, 48 us now).
__global__ void __launch_bounds__(256) k_neural_adam(float* params, float* m, float* v, float* grads,
                                                     float t, float lr, float beta1, float beta2,
                                                     float eps, __half* img, float* bias,
                                                     float* loss, float* loss_out) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k < nn::NPARAM) {
    const float c1 = 1.0f - powf(beta1, t), c2 = 1.0f - powf(beta2, t);
    const float gk = grads[k];
    const float mm = beta1 * m[k] + (1.0f - beta1) * gk;
    const float vv = beta2 * v[k] + (1.0f - beta2) * gk * gk;
    m[k] = mm;
    v[k] = vv;
    const float p = params[k] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    params[k] = p;
    grads[k] = 0.0f;
    store_param(k, p, img, bias);
  }
  if (k == 0) {
    if (loss_out) *loss_out = *loss;
    *loss = 0.0f;
  }
}

// Float32 -> binary16 rows: dst[r][0..7] from src[r][0..cin-1] (zero beyond cin).
__global__ void k_rows_to_h8(const float* src, int cin, __half* dst, int64_t rows) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += stride) {
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = k < cin ? src[r * cin + k] : 0.0f;
    reinterpret_cast<uint4*>(dst)[r] = make_uint4(pack_h2(v[0], v[1]), pack_h2(v[2], v[3]),
                                                  pack_h2(v[4], v[5]), pack_h2(v[6], v[7]));
  }
}

// ---------------------------------------------------------------- launchers

// Launches a decode kernel over `tiles` tiles, two per CTA pass.
template <class Kernel>
static cudaError_t launch_decode(Kernel k, OncePerDevice& once, int64_t tiles, const NeuralDev& nd, const LookupArgs& a,
                                 cudaStream_t s) {
  // that much shared memory per CTA keeps at most 4 CTAs on an SM (228 KiB), so their
  // 4 x 128 tensor-memory columns fit in the SM's 512 and no allocation waits
  constexpr int smem = (int)sizeof(tc::Smem) + 1024;
  static_assert(smem >= 46 * 1024, "four CTAs on an SM at most");
  const cudaError_t e = once([&] { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); });
  if (e != cudaSuccess) return e;
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t pairs = (tiles + 1) / 2;
  const int grid = (int)(pairs < (int64_t)sms * 4 ? pairs : (int64_t)sms * 4);
  k<<<grid, 256, smem, s>>>(nd, a);
  return cudaGetLastError();
}

template <int F>
static cudaError_t run_neural(Op op, const NeuralDev& nd, const LookupArgs& a, cudaStream_t s) {
  static OncePerDevice once[3];
  const int64_t tiles = (a.n + tc::ROWS - 1) / tc::ROWS;
  if (op == OP_STOCHASTIC) {
    if (a.perm == nullptr && a.taps == nullptr)
      return launch_decode(k_neural_stochastic_tc<F, true>, once[0], tiles, nd, a, s);
    return launch_decode(k_neural_stochastic_tc<F, false>, once[1], tiles, nd, a, s);
  }
  if (op == OP_DETERMINISTIC) {
    const int parts = (a.lod != nullptr && nd.nlev > 1 && a.level_mode != STF_LEVEL_NEAREST) ? 2 : 1;
    const int q = tc::ROWS / (parts * Filter<F>::T * Filter<F>::T);
    return launch_decode(k_neural_deterministic_tc<F>, once[2], (a.n + q - 1) / q, nd, a, s);
  }
  return cudaErrorNotSupported;
}

cudaError_t launch_neural(Op op, int filter, const NeuralDev& nd, const LookupArgs& a, cudaStream_t s) {
  switch (filter) {
    case STF_FILTER_LINEAR: return run_neural<STF_FILTER_LINEAR>(op, nd, a, s);
    case STF_FILTER_BSPLINE3: return run_neural<STF_FILTER_BSPLINE3>(op, nd, a, s);
    case STF_FILTER_CATMULL_ROM: return run_neural<STF_FILTER_CATMULL_ROM>(op, nd, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace stf

// ---------------------------------------------------------------- host side

namespace stf {

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

stf_status build_neural(stf_texture_s* t, const stf_neural_desc* d, cudaStream_t s) {
  const int W = d->width, H = d->height;
  auto pow2 = [](int v) { return v > 0 && (v & (v - 1)) == 0; };
  if (!pow2(W) || !pow2(H)) return fail(STF_ERR_INVALID_ARGUMENT, "neural texture sizes must be powers of two");
  int maxlev = 1;
  while ((W >> maxlev) > 0 || (H >> maxlev) > 0) ++maxlev;
  if (d->latent_levels < 1 || d->latent_levels > 4)
    return fail(STF_ERR_INVALID_ARGUMENT, "latent_levels must be 1 .. 4");
  if (d->levels < d->latent_levels || d->levels > maxlev || d->levels > STF_MAX_LEVELS)
    return fail(STF_ERR_INVALID_ARGUMENT, "levels %d outside [latent_levels, %d]", d->levels, maxlev);
  if (!d->latents || !d->params) return fail(STF_ERR_INVALID_ARGUMENT, "latents or params is NULL");
  if (d->levels > d->latent_levels && !d->fallback)
    return fail(STF_ERR_INVALID_ARGUMENT, "fallback texels are NULL");
  NeuralDev& nd = t->neural;
  memset(&nd, 0, sizeof(nd));
  nd.nlat = d->latent_levels;
  nd.nlev = d->levels;
  int64_t n_lat = 0, n_fb = 0;
  for (int L = 0; L < d->levels; ++L) {
    nd.lvl_w[L] = (W >> L) > 0 ? (W >> L) : 1;
    nd.lvl_h[L] = (H >> L) > 0 ? (H >> L) : 1;
    const int64_t cnt = (int64_t)nd.lvl_w[L] * nd.lvl_h[L];
    if (L < nd.nlat) {
      nd.lvl_off[L] = n_lat;
      n_lat += cnt;
    } else {
      nd.lvl_off[L] = n_fb;
      n_fb += cnt;
    }
  }
  nd.n_lat_texels = n_lat;
  const size_t b_lat = al256(sizeof(float) * 8 * n_lat), b_lat16 = al256(2 * 8 * n_lat);
  const size_t b_fb16 = al256(2 * 8 * (n_fb > 0 ? n_fb : 1));
  const size_t b_p = al256(sizeof(float) * nn::NPARAM);
  const size_t b_img = al256(2 * nn::IMG_ALL), b_bias = al256(sizeof(float) * nn::NBIAS);
  const size_t total = 3 * b_lat + b_lat16 + b_fb16 + 4 * b_p + 256 + b_img + b_bias;
  cudaError_t e = dev_alloc(&t->d_neural, total);
  if (e != cudaSuccess) return fail_cuda(e, "neural texture allocation");
  t->bytes += (int64_t)total;
  char* p = (char*)t->d_neural;
  nd.lat32 = (float*)p;  p += b_lat;
  nd.m_lat = (float*)p;  p += b_lat;
  nd.v_lat = (float*)p;  p += b_lat;
  nd.lat16 = (const __half*)p; p += b_lat16;
  nd.fb16 = (const __half*)p;  p += b_fb16;
  t->n_params = (float*)p; p += b_p;
  t->n_m = (float*)p;      p += b_p;
  t->n_v = (float*)p;      p += b_p;
  t->n_grads = (float*)p;  p += b_p;
  t->n_loss = (float*)p;   p += 256;
  nd.wimg = (const __half*)p; p += b_img;
  nd.bias = (const float*)p;
  const cudaMemcpyKind kind = d->data_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  e = cudaMemcpyAsync(nd.lat32, d->latents, sizeof(float) * 8 * n_lat, kind, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(nd.m_lat, 0, 2 * b_lat, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(t->n_params, d->params, sizeof(float) * nn::NPARAM, kind, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->n_m, 0, 2 * b_p, s);
  if (e == cudaSuccess) {
    k_rows_to_h8<<<grid_blocks(n_lat, 256), 256, 0, s>>>(nd.lat32, 8, (__half*)nd.lat16, n_lat);
    e = cudaMemsetAsync((void*)nd.wimg, 0, b_img + b_bias, s);       // adjacent, with their padding
    if (e == cudaSuccess) {
      k_neural_images<<<kParamBlocks, 256, 0, s>>>(t->n_params, (__half*)nd.wimg, (float*)nd.bias);
      e = cudaGetLastError();
    }
  }
  float* tmp = nullptr;
  if (e == cudaSuccess && n_fb > 0) {
    e = dev_alloc((void**)&tmp, sizeof(float) * 7 * n_fb);
    if (e == cudaSuccess) e = cudaMemcpyAsync(tmp, d->fallback, sizeof(float) * 7 * n_fb, kind, s);
    if (e == cudaSuccess) {
      k_rows_to_h8<<<grid_blocks(n_fb, 256), 256, 0, s>>>(tmp, 7, (__half*)nd.fb16, n_fb);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(tmp);
  if (e != cudaSuccess) return fail_cuda(e, "neural texture upload");
  t->kind = STF_KIND_NEURAL2D;
  t->channels = STF_NEURAL_OUT;
  t->levels = d->levels;
  t->dims[0] = W;
  t->dims[1] = H;
  t->dims[2] = 1;
  t->n_step = 0;
  return STF_OK;
}

static stf_status neural_handle(stf_texture t) {
  if (!handle_ok(t)) return fail(STF_ERR_INVALID_HANDLE, "unknown texture handle");
  if (t->kind != STF_KIND_NEURAL2D) return fail(STF_ERR_UNSUPPORTED, "not a neural texture");
  return STF_OK;
}

}  // namespace stf

using namespace stf;

extern "C" stf_status stf_neural_gradients(stf_texture t, const int64_t* ids, int64_t batch,
                                           const float* target_rows, float* d_param_grads,
                                           float* d_latent_grads, float* d_loss, void* stream) {
  stf_status st = neural_handle(t);
  if (st != STF_OK) return st;
  if (batch < 1 || !ids || !target_rows) return fail(STF_ERR_INVALID_ARGUMENT, "need batch >= 1, ids and targets");
  cudaStream_t s = (cudaStream_t)stream;
  TrainArgs ta;
  memset(&ta, 0, sizeof(ta));
  ta.ids = ids;
  ta.target_rows = target_rows;
  ta.batch = batch;
  ta.inv_batch = 1.0f / (float)batch;
  // straight into the caller's arrays where they are this device's memory (the atomics cross
  // neither the host link nor to another device) and, for the vector atomics, 16-byte aligned
  const bool direct = (uintptr_t)d_param_grads % 16 == 0 && local_memory(d_param_grads);
  const bool direct_loss = local_memory(d_loss);
  ta.grads = direct ? d_param_grads : t->n_grads;
  ta.loss = direct_loss ? d_loss : t->n_loss;
  ta.dx_out = d_latent_grads;
  cudaError_t e = cudaMemsetAsync(ta.grads, 0, sizeof(float) * nn::NPARAM, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(ta.loss, 0, sizeof(float), s);
  if (e == cudaSuccess) e = launch_train_tc(t->neural, ta, s);
  if (e == cudaSuccess && d_param_grads && !direct)
    e = cudaMemcpyAsync(d_param_grads, t->n_grads, sizeof(float) * nn::NPARAM, cudaMemcpyDefault, s);
  if (e == cudaSuccess && d_loss && !direct_loss)
    e = cudaMemcpyAsync(d_loss, t->n_loss, sizeof(float), cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? STF_OK : fail_cuda(e, "neural gradients");
}

extern "C" stf_status stf_neural_train(stf_texture t, const float* d_target, const stf_train_config* cfg,
                                       int32_t steps, float* d_loss_per_step, void* stream) {
  stf_status st = neural_handle(t);
  if (st != STF_OK) return st;
  if (!cfg || !d_target) return fail(STF_ERR_INVALID_ARGUMENT, "config or target is NULL");
  if (cfg->batch < 1 || cfg->batch > t->neural.n_lat_texels)
    return fail(STF_ERR_INVALID_ARGUMENT, "batch must be in [1, %lld]", (long long)t->neural.n_lat_texels);
  if (!(cfg->lr_latent >= 0.f) || !(cfg->lr_params >= 0.f) || !(cfg->beta1 >= 0.f && cfg->beta1 < 1.f) ||
      !(cfg->beta2 >= 0.f && cfg->beta2 < 1.f) || !(cfg->eps > 0.f))
    return fail(STF_ERR_INVALID_ARGUMENT, "invalid optimizer settings");
  if (steps < 0) return fail(STF_ERR_INVALID_ARGUMENT, "steps < 0");
  if (steps == 0) return STF_OK;
  cudaStream_t s = (cudaStream_t)stream;
  // zero before the first batch; the parameter update leaves them zero for the next
  cudaError_t e = cudaMemsetAsync(t->n_grads, 0, sizeof(float) * nn::NPARAM, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->n_loss, 0, sizeof(float), s);
  for (int k = 0; k < steps && e == cudaSuccess; ++k) {
    TrainArgs ta;
    memset(&ta, 0, sizeof(ta));
    ta.target_levels = d_target;
    ta.batch = cfg->batch;
    ta.inv_batch = 1.0f / (float)cfg->batch;
    ta.seed = cfg->seed;
    ta.step = t->n_step;
    ta.lr = cfg->lr_latent;
    ta.beta1 = cfg->beta1;
    ta.beta2 = cfg->beta2;
    ta.eps = cfg->eps;
    ta.grads = t->n_grads;
    ta.loss = t->n_loss;
    ta.train = 1;
    e = launch_train_tc(t->neural, ta, s);
    if (e != cudaSuccess) break;
    k_neural_adam<<<kParamBlocks, 256, 0, s>>>(t->n_params, t->n_m, t->n_v, t->n_grads, (float)(t->n_step + 1),
                                    cfg->lr_params, cfg->beta1, cfg->beta2, cfg->eps,
                                    (__half*)t->neural.wimg, (float*)t->neural.bias, t->n_loss,
                                    d_loss_per_step ? d_loss_per_step + k : nullptr);
    e = cudaGetLastError();
    t->n_step += 1;
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? STF_OK : fail_cuda(e, "neural training");
}

extern "C" stf_status stf_neural_read(stf_texture t, float* d_params, float* d_latents, void* stream) {
  stf_status st = neural_handle(t);
  if (st != STF_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  if (d_params) e = cudaMemcpyAsync(d_params, t->n_params, sizeof(float) * nn::NPARAM, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && d_latents)
    e = cudaMemcpyAsync(d_latents, t->neural.lat32, sizeof(float) * 8 * t->neural.n_lat_texels,
                        cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? STF_OK : fail_cuda(e, "neural read");
}
