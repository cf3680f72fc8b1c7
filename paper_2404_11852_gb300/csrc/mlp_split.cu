// Feature Gathering + Feature Computation with FP32-class accuracy on the tensor cores (tcgen05,
// sm_103a): operands split into BF16 parts, products accumulated in FP32 in tensor memory.
//
//   NP = 3  v = hi + mid + lo (24 significant bits), the six products above 2^-24: FP32 accuracy
//   NP = 2  v = hi + lo (16 bits), three products (Henry, Tang and Heinecke, ARITH 2019)
//
// One persistent CTA per SM, a pipeline of roles over the CTA's tiles of 128 samples of one brick:
//   G   two groups of 4 warps (alternate tiles), a thread per sample: interpolates the features from
//       global memory, encodes the direction, splits the input row into operand x (shared memory)
//   M   one thread: issues every MMA.  Layer 1: D = x W1^T, both operands in shared memory.
//       Layer 2: D = h1 W2^T with h1 read from tensor memory, in two chunks of 64 hidden units
//   E1  8 warps, two threads per sample (half of the hidden units each): layer 1's accumulators ->
//       bias, ReLU, split -> h1 in tensor memory, chunk by chunk
//   E2  8 warps: layer 2's accumulators -> bias, ReLU, layer 3 in FP32, sigmoid -> (c, w) into the
//       sample's record
// Layer 1 of tile i + 1 is issued between the two chunks of layer 2 of tile i, and h1's chunk c of tile
// i + 1 is written as soon as chunk c of tile i has been read, so the tensor pipe runs on while E1 and
// E2 work.
// Order of the products: a tensor-core accumulation rounds its running sum towards zero, so the more
// steps are added to a sum of full size, the further it drifts.  The hi hi products come last, after all
// the small ones of both chunks: 8 steps at full size in layer 2 instead of 48.  The hi part of h1
// then outlives the others, hence its two buffers.
//
// What bounds it: with NP = 3 the MMAs, (48 + 128) / 16 K steps x 6 products of M = N = 128 at 64 clocks
// each, 4,224 clocks a tile of the ~5,000 measured.  With h1 in tensor memory layer 2 reads one operand
// from shared memory, half of what a tile of two shared operands needs.  With NP = 2 (2,112 clocks of
// MMAs, ~3,900 measured) the latency of G's and E1's instructions.
// Measured, gather + MLP: 62.5 M samples of a 256^3 x 12 FP16 grid, NP = 3, 52.5 ms on the CUDA cores
// before, 8.7 ms; 6.7 M samples of a 160^3 x 12 FP16 grid, NP = 2, 1.70 ms (one thread per sample for
// everything, two tiles in flight) before, 0.70 ms.  Steps on the way: E1 and E2 as one role 12.0 / 0.93
// ms; the MMAs issued with warp-uniform operands 13.4 -> 9.8; h1 in two chunks instead of four 10.4 -> 8.9.
// All waits are bounded; a role that runs into a timeout records it and leaves, and so do the others.
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace cicero {

namespace ms {

constexpr int kK1 = kMaxIn;                 // layer-1 K: the input row padded to 48
constexpr int kEpiWarps = 8, kGatWarps = 4;  // warps of E1 and of E2; warps of one of G's two groups
constexpr int kE2 = kEpiWarps, kG = 2 * kEpiWarps, kM = kG + 2 * kGatWarps;  // first warp of each role
constexpr int kThreads = 32 * (kM + 4);      // M's warpgroup has one working warp
// Registers per thread: 72 at launch (28 warps), then shared out by role (setmaxnreg):
// 256 (E1 + E2 + G) + 128 x 24 = 896 x 72.  HOLD: see k_mlp_split.
template <bool HOLD>
struct Regs {
  static constexpr int e1 = HOLD ? 88 : 72, e2 = HOLD ? 80 : 72, g = HOLD ? 72 : 96, m = 24;
  static_assert(kThreads == 896 && 256 * (e1 + e2 + g) + 128 * m <= kThreads * 72, "register shares");
};
template <int R>
__device__ __forceinline__ void set_regs() {
  if constexpr (R > 72) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R));
  if constexpr (R < 72) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R));
}
constexpr int kChunks = 2;                  // chunks of hidden units of layer 2's K
constexpr int kMeta = 4;                    // tiles of per-sample data in flight
constexpr int kXBytes = kTile * kK1 * 2;    // one part of the input operand
constexpr int kW1Bytes = kHidden * kK1 * 2, kW2Bytes = kHidden * kHidden * 2;

template <int NP>
struct Smem {
  static constexpr int w1 = 0;                               // [NP][128][48] bf16: row n, K = k: W1[n][k]
  static constexpr int w2 = w1 + NP * kW1Bytes;              // [NP][128][128]
  static constexpr int x = w2 + NP * kW2Bytes;               // [2][NP][128][48]: the input rows of two tiles
  static constexpr int b1 = x + 2 * NP * kXBytes;            // [128] f32
  static constexpr int l3 = b1 + kHidden * 4;                // per pair of hidden units: b2, w3 rows 0, 1, 2
  static constexpr int b3 = l3 + 4 * kHidden * 4;            // [4]
  static constexpr int z = b3 + 16;                          // [kMeta][128] float4: partial layer-3 sums
  static constexpr int meta = z + kMeta * kTile * 16;        // [kMeta][128] float4: record, weight, sorted place, ||x||^2
  static constexpr int bars = meta + kMeta * kTile * 16;
  static constexpr int bytes = bars + 8 * 32;
  // a backward's recompute: ||W1_n|| [128], ||W2_n|| [128], ||W1||_F, then [2][2][128]: partial ||h1||^2 of
  // two tiles, by half of the hidden units, the sign bit set where a decision is uncertain
  static constexpr int nrm = bytes;
  static constexpr int hs = nrm + (2 * kHidden + 4) * 4;
  static constexpr int bytes_bwd = hs + 2 * 2 * kTile * 4;
  static_assert(x % 16 == 0 && w2 % 16 == 0 && bars % 16 == 0 && bytes_bwd <= 227 * 1024, "layout");
};

struct Bars {  // one phase per use, in tile order
  uint64_t xfull[2];       // x of tile i written                          (4 G warps)
  uint64_t l1done[2];      // layer 1 of tile i done, x free               (commit)
  uint64_t afull[kChunks]; // chunk c of h1 written                        (8 E1 warps)
  uint64_t cdone[kChunks]; // chunk c of h1 but its hi part read           (commit)
  uint64_t l2done[2];      // layer 2 of tile i done                       (commit)
  uint64_t dfree[2];       // accumulator of tile i read                   (8 E2 warps)
  uint64_t zfull[kMeta];   // partial layer-3 sums of tile i written       (4 E2 warps)
  uint64_t mfull[kMeta];   // per-sample data of tile i written            (4 G warps)
  uint64_t hfull[2];       // partial ||h1||^2 of tile i written           (8 E1 warps, backward)
  uint64_t last;           // every MMA done                               (commit)
  uint32_t tmem;
  uint32_t odd;            // what the weights ask for (Odd)
  uint32_t marked;         // whether a sample is marked to be taken again
};
static_assert(sizeof(Bars) <= 8 * 32, "barrier block");

__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// after every lane's writes (and its fence): one arrival per warp
__device__ __forceinline__ void warp_arrive(uint64_t* bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) arrive(bar);
}
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, uint32_t* err) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, err));
}

// Columns 32 c + 16 h + j (c < 4, j < 16) of this thread's lane of the accumulator at d, into v[16 c + j].
__device__ __forceinline__ void load_half(uint32_t d, int h, float* v) {
  uint32_t r[64];
  const uint32_t a = d + 16u * (uint32_t)h;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%64];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%65];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47}, [%66];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%67];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]),
        "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]),
        "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]),
        "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]),
        "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(a), "r"(a + 32u), "r"(a + 64u), "r"(a + 96u)
      : "memory");
#pragma unroll
  for (int i = 0; i < 64; i++) v[i] = __uint_as_float(r[i]);
}

// Columns 32 c + 16 h + j (c = 2 g, 2 g + 1, j < 16) of this thread's lane of the accumulator at d.
__device__ __forceinline__ void load_quarter(uint32_t d, int h, int g, float* v) {
  uint32_t r[32];
  const uint32_t a = d + 16u * (uint32_t)h + 64u * (uint32_t)g;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(a), "r"(a + 32u)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// two packed FP32 operations
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 p, q, s;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tadd.rn.f32x2 s, p, q;\n\t"
      "mov.b64 {%0, %1}, s;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n\t.reg .b64 p, q, t, s;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tmov.b64 t, {%6, %7};\n\t"
      "fma.rn.f32x2 s, p, q, t;\n\tmov.b64 {%0, %1}, s;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

// (a, b) split into NP packed BF16 parts: each part rounds what the ones before it left.
template <int NP>
__device__ __forceinline__ void split2(float2 v, uint32_t p[NP]) {
#pragma unroll
  for (int k = 0; k < NP; k++) {
    p[k] = tc::pack_bf16(v.x, v.y);
    if (k + 1 < NP)  // v - part, exactly
      v = fma2(make_float2(__uint_as_float(p[k] << 16), __uint_as_float(p[k] & 0xffff0000u)),
               make_float2(-1.0f, -1.0f), v);
  }
}

// The NP operand rows (16 bytes each) of 8 consecutive K values of one row.
template <int NP>
__device__ __forceinline__ void split_row(const float* v, uint4 q[NP]) {
  uint32_t p[4][NP];
#pragma unroll
  for (int j = 0; j < 4; j++) split2<NP>(make_float2(v[2 * j], v[2 * j + 1]), p[j]);
#pragma unroll
  for (int k = 0; k < NP; k++) q[k] = make_uint4(p[0][k], p[1][k], p[2][k], p[3][k]);
}

// The products of one K step of 16 but the largest (hi hi): those of parts a + b < NP, smallest first.
template <int NP, typename MMA>
__device__ __forceinline__ void small_products(MMA mma) {
#pragma unroll
  for (int s = NP - 1; s > 0; s--)
#pragma unroll
    for (int a = 0; a <= s; a++) mma(a, s - a);
}

// Tensor memory: part k of h1 of tile i at h1_col (two buffers of the hi part), then the accumulators.
template <int NP>
struct Tmem {
  static constexpr uint32_t acc = 64 * (NP + 1);  // accumulator of tile i: + 128 (i & 1)
  static_assert(acc + 256 <= 512, "tensor memory");
};
__device__ __forceinline__ uint32_t h1_col(int k, uint32_t i) { return k == 0 ? 64u * (i & 1) : 64u * (uint32_t)(k + 1); }

// FP32 renders: an operand that is infinite, or that BF16 rounds to infinity, has NaN parts, and every unit of
// the sample would come out as NaN, 0 behind the ReLU, where the FP32 chain has infinities, zeros or finite
// values.  Such samples are marked in their record's colour and taken again by E2 (sample_f32) when it is done
// with the CTA's tiles.  E1 lets a NaN of its first unit through the ReLU (all units are NaNs then: an input
// that cannot be split), layer 2's sums carry it (or that of an h1 that cannot be split), and E2 carries it
// into the colour.  A NaN among the weights or biases of a unit marks nothing: the unit is 0 in both chains and
// is taken out of the operands (drop_nan_units).  One in layer 3's first row makes every first colour a NaN, as
// it should be, and no mark can be told from it (kOddBlind).
// A weight or a bias of layer 1 from kHuge on marks every sample.  One below kTiny has parts below BF16's smallest number and is off
// by up to 2^-134, too little to count beside operands below kHuge; with such weights G and E1 mark the
// samples of larger ones.
// A render without any of these pays a few instructions per thread and tile, the look at the weights and what the
// code below does to the roles' registers: 0.98 to 1.03 of the time without, over five FP32 calls from 85 us to 2.8
// ms (a mean of 1.00; 62.5 M samples 8.78 -> 8.85 ms).  (Flags from an earlier kernel and the samples taken again by
// one of its own: the same within 1%.)  A sample taken again costs an SM ~5,000 clocks.
constexpr float kHuge = 0x1p100f, kTiny = 0x1p-109f;
constexpr uint32_t kOddColour = 0x7FC0BABEu;  // a NaN that no arithmetic returns
enum Odd : uint32_t { kOddNan = 1, kOddAll = 2, kOddTiny = 4, kOddBlind = 8 };
__device__ __forceinline__ float relu_nan(float v) {
  float r;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(v));
  return r;
}
template <int N>
__device__ __forceinline__ bool any_huge(const float* v) {
  float m = 0.0f;
#pragma unroll
  for (int k = 0; k < N; k++) m = fmaxf(m, fabsf(v[k]));
  return m >= kHuge;
}

// What the parameters in shared memory ask for, by this thread's share of the weights' hi parts (pairs of BF16
// numbers; a NaN or an infinity shows there) and of the biases and layer 3.
template <int NP>
__device__ __forceinline__ uint32_t odd_parameters(const char* sm) {
  using S = Smem<NP>;
  uint32_t top = 0u, low = 0xFFFFFFFFu;  // per half: the largest magnitude, and the smallest but 0, minus 1
#pragma unroll
  for (int k = 0; k < (kW1Bytes + kW2Bytes + 16 * kThreads - 1) / (16 * kThreads); k++) {
    const int i = 16 * (threadIdx.x + k * kThreads);
    if (i >= kW1Bytes + kW2Bytes) break;
    const uint4 q = *(const uint4*)(sm + (i < kW1Bytes ? S::w1 + i : S::w2 - kW1Bytes + i));
    const uint32_t v[4] = {q.x & 0x7FFF7FFFu, q.y & 0x7FFF7FFFu, q.z & 0x7FFF7FFFu, q.w & 0x7FFF7FFFu};
#pragma unroll
    for (int u = 0; u < 4; u++) {
      top = __vmaxu2(top, v[u]);
      low = __vminu2(low, __vsub2(v[u], 0x00010001u));
    }
  }
  const uint32_t hi = max(top & 0xFFFFu, top >> 16), lo = min(low & 0xFFFFu, low >> 16);
  uint32_t f = (hi > 0x7F80u ? kOddNan : hi >= (__float_as_uint(kHuge) >> 16) ? kOddAll : 0u) |
               (lo < (__float_as_uint(kTiny) >> 16) - 1u ? kOddTiny : 0u);
  for (int i = threadIdx.x; i < 5 * kHidden; i += kThreads) {
    const float v = ((const float*)(sm + S::b1))[i];
    f |= (isnan(v) ? (i >= kHidden && (i & 6) == 2 ? kOddBlind : kOddNan) : 0u) |
         (i < kHidden && fabsf(v) >= kHuge ? kOddAll : 0u);
  }
  if (isnan(((const float*)(sm + S::b3))[0])) f |= kOddBlind;
  return f;
}

// Zeros in place of the weights and the bias of every unit that has a NaN among them (layer 3 is left alone).
template <int NP>
__device__ __noinline__ void drop_nan_units(char* sm, const MlpPtrs mlp) {
  using S = Smem<NP>;
  for (int r = threadIdx.x; r < 2 * kHidden; r += kThreads) {
    const int n = r % kHidden, in = r < kHidden ? mlp.in_dim : kHidden, K = r < kHidden ? kK1 : kHidden;
    const float* row = (r < kHidden ? mlp.w1 : mlp.w2) + (size_t)n * in;
    float* bias = r < kHidden ? (float*)(sm + S::b1) + n : (float*)(sm + S::l3) + 8 * (n >> 1) + (n & 1);
    bool drop = isnan(*bias);
    for (int k = 0; k < in; k++) drop |= isnan(row[k]);
    if (!drop) continue;
    *bias = 0.0f;
    for (int p = 0; p < NP; p++)
      for (int k = 0; k < K; k += 8)
        *(uint4*)(sm + (r < kHidden ? S::w1 + p * kW1Bytes : S::w2 + p * kW2Bytes) + tc::kmaj_off(n, k, K)) =
            make_uint4(0u, 0u, 0u, 0u);
  }
}

// Weights [rows][in] (FP32, global) into NP K-major operands of K columns (zeros from `in` on).
template <int NP>
__device__ __forceinline__ void load_weights(char* dst, int part_bytes, const float* w, int rows, int in, int K) {
  const int chunks = rows * (K / 8);
  const bool vec = (in & 3) == 0 && (reinterpret_cast<uintptr_t>(w) & 15u) == 0;
#pragma unroll 2
  for (int i = threadIdx.x; i < chunks; i += kThreads) {
    const int n = i / (K / 8), k0 = (i % (K / 8)) * 8;
    const float* src = w + (size_t)n * in + k0;
    float v[8];
    if (vec && k0 + 8 <= in) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(src)), b = __ldg(reinterpret_cast<const float4*>(src) + 1);
      v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
#pragma unroll
      for (int j = 0; j < 8; j++) v[j] = k0 + j < in ? __ldg(src + j) : 0.0f;
    }
    uint4 q[NP];
    split_row<NP>(v, q);
#pragma unroll
    for (int p = 0; p < NP; p++) *reinterpret_cast<uint4*>(dst + p * part_bytes + tc::kmaj_off(n, k0, K)) = q[p];
  }
}

__device__ __forceinline__ float4 ld4(const float* v) { return __ldg(reinterpret_cast<const float4*>(v)); }
__device__ __forceinline__ float4 ld4(const __half* v) {
  const uint2 a = __ldg(reinterpret_cast<const uint2*>(v));
  const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&a.x));
  const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&a.y));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

constexpr int kMaxC = 21;
// Trilinear features of voxel i0 at fractions f, from global memory, into out[0, C) (FP32; the rest of
// out untouched).  CC > 0: C = CC.
template <typename T, int CC>
__device__ __forceinline__ void gather(const GridGeo& g, const T* __restrict__ feat, const int i0[3], const float f[3],
                                       float* out) {
  const int C = CC ? CC : g.C;
  constexpr int N = CC ? CC : kMaxC;
  float wq[8];
  const T* v[4];  // the x-pairs of vertices: (y, z) = (0, 0), (1, 0), (0, 1), (1, 1)
#pragma unroll
  for (int q = 0; q < 8; q++)
    wq[q] = ((q & 1) ? f[0] : 1.f - f[0]) * (((q >> 1) & 1) ? f[1] : 1.f - f[1]) * ((q >> 2) ? f[2] : 1.f - f[2]);
#pragma unroll
  for (int r = 0; r < 4; r++)
    v[r] = feat + (((size_t)(i0[2] + (r >> 1)) * g.n[1] + (i0[1] + (r & 1))) * g.n[0] + i0[0]) * C;
  if (CC ? CC % 4 == 0 : (C & 3) == 0) {  // rows of the grid start on 16 bytes, vertices on 4 channels
#pragma unroll
    for (int c = 0; c + 4 <= N; c += 4)
      if (CC || c < C) {  // the eight corners' loads of four channels in flight together
        float4 a[8];
#pragma unroll
        for (int q = 0; q < 8; q++) a[q] = ld4(v[q >> 1] + (q & 1) * C + c);
#pragma unroll
        for (int q = 0; q < 8; q++) {
          out[c] = fmaf(wq[q], a[q].x, out[c]);
          out[c + 1] = fmaf(wq[q], a[q].y, out[c + 1]);
          out[c + 2] = fmaf(wq[q], a[q].z, out[c + 2]);
          out[c + 3] = fmaf(wq[q], a[q].w, out[c + 3]);
        }
      }
  } else {
#pragma unroll
    for (int c = 0; c < N; c++)
      if (c < C) {
#pragma unroll
        for (int q = 0; q < 8; q++) out[c] = fmaf(wq[q], ldf(v[q >> 1] + (q & 1) * C + c), out[c]);
      }
  }
}

// d, then sin/cos(2^k d) for k < NF (the recurrence of encode_dir), unrolled
template <int NF>
__device__ __forceinline__ void encode(const float d[3], float* x) {
  float s[3], c[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    x[a] = d[a];
    sincosf(d[a], &s[a], &c[a]);
  }
#pragma unroll
  for (int k = 0; k < NF; k++) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      x[3 + 6 * k + a] = s[a];
      x[3 + 6 * k + 3 + a] = c[a];
      const float s2 = 2.0f * s[a] * c[a];
      c[a] = 1.0f - 2.0f * s[a] * s[a];
      s[a] = s2;
    }
  }
}

// The colour of one sample from the FP32 chain on the CUDA cores, by a whole warp: for samples whose
// operands cannot be split.  Lane l holds inputs l and l + 32 and hidden units 4 l .. 4 l +
// 3; every unit's sum runs over its inputs in order, one FMA each.
__device__ __forceinline__ float3 sample_f32(const GridGeo& g, const MlpPtrs& mlp, const void* feat, int f16,
                                             const SrtRec* rec, bool w_finite) {
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  float x[2] = {0.0f, 0.0f};
  {
    const float4 pw = rec->pw, qd = rec->qd;
    const float p[3] = {pw.x, pw.y, pw.z};
    int i0[3];
    float f[3];
    const bool in = index_sample(g, p, i0, f);  // (a sample that this rejects has set the error word)
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const int k = lane + 32 * u;
      if (k < g.C) {
        if (!in) continue;
#pragma unroll 1
        for (int q = 0; q < 8; q++) {
          const float wq = ((q & 1) ? f[0] : 1.f - f[0]) * (((q >> 1) & 1) ? f[1] : 1.f - f[1]) *
                           ((q >> 2) ? f[2] : 1.f - f[2]);
          const size_t at = (((size_t)(i0[2] + (q >> 2)) * g.n[1] + (i0[1] + ((q >> 1) & 1))) * g.n[0] + i0[0] +
                             (q & 1)) * g.C + k;
          x[u] = fmaf(wq, f16 ? __half2float(((const __half*)feat)[at]) : ((const float*)feat)[at], x[u]);
        }
      } else if (k < mlp.in_dim) {  // d, then sin/cos(2^j d) as encode has them
        const int e = k - g.C, a = e % 3;
        const float d = a == 0 ? qd.y : (a == 1 ? qd.z : qd.w);
        float s, c;
        sincosf(d, &s, &c);
#pragma unroll 1
        for (int j = e < 3 ? 0 : (e - 3) / 6; j > 0; j--) {
          const float s2 = 2.0f * s * c;
          c = 1.0f - 2.0f * s * s;
          s = s2;
        }
        x[u] = e < 3 ? d : ((e / 3) & 1 ? s : c);
      }
    }
  }
  float h[4] = {0.f, 0.f, 0.f, 0.f}, z[4] = {0.f, 0.f, 0.f, 0.f};
  const bool none = __any_sync(full, isnan(x[0]) || isnan(x[1]));  // then all units of layer 1 are NaN, h1 0
  if (none) z[0] = z[1] = z[2] = z[3] = NAN;
#pragma unroll 1
  for (int k = 0; k < mlp.in_dim && !none; k++) {
    const float v = __shfl_sync(full, k < 32 ? x[0] : x[1], k & 31);
#pragma unroll
    for (int u = 0; u < 4; u++) z[u] = fmaf(v, mlp.w1[(4 * lane + u) * mlp.in_dim + k], z[u]);
  }
#pragma unroll
  for (int u = 0; u < 4; u++) {
    h[u] = fmaxf(z[u] + mlp.b1[4 * lane + u], 0.0f);
    z[u] = 0.0f;
  }
#pragma unroll 1
  for (int k4 = 0; k4 < kHidden / 4 && !(none && w_finite); k4++)  // (h1 = 0 otherwise)
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const float v = __shfl_sync(full, h[j], k4);
#pragma unroll
      for (int u = 0; u < 4; u++) z[u] = fmaf(v, mlp.w2[(4 * lane + u) * kHidden + 4 * k4 + j], z[u]);
    }
  float o[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int u = 0; u < 4; u++) {
    const float h2 = fmaxf(z[u] + mlp.b2[4 * lane + u], 0.0f);
#pragma unroll
    for (int c = 0; c < 3; c++) o[c] = fmaf(mlp.w3[c * kHidden + 4 * lane + u], h2, o[c]);
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) o[c] += __shfl_xor_sync(full, o[c], off);
    o[c] = sigmoid_f(o[c] + mlp.b3[c]);
  }
  return make_float3(o[0], o[1], o[2]);
}

// M: every MMA of the CTA's n tiles, by one warp: the control flow and the operands are the warp's, one
// elected lane issues.  (Issued from a thread of its own, each MMA's operands took a dozen instructions
// through per-thread registers: ~110 clocks an MMA beside 27 other warps, against the 64 it runs.)
template <int NP, bool HOLD>
__device__ __forceinline__ void issue_mmas(char* sm, Bars& B, uint32_t tmem, uint32_t n, uint32_t* err) {
  using namespace tc;
  using S = Smem<NP>;
  tmem = __shfl_sync(0xffffffffu, tmem, 0);
  n = __shfl_sync(0xffffffffu, n, 0);
  const uint32_t dcol = tmem + Tmem<NP>::acc;
  constexpr uint32_t hi1 = desc_hi(kK1 * 16), hi2 = desc_hi(kHidden * 16), id = idesc_bf16(kHidden);
  const uint32_t x = desc_lo(smem_u32(sm + S::x), 128u);
  const uint32_t w1 = desc_lo(smem_u32(sm + S::w1), 128u);
  const uint32_t w2 = desc_lo(smem_u32(sm + S::w2), 128u);
  const bool leader = elect_one();
  auto layer1 = [&](uint32_t i) -> bool {
    if (!warp_wait(&B.xfull[i & 1], (i >> 1) & 1, err)) return false;
    if (i >= 2 && !warp_wait(&B.dfree[i & 1], ((i >> 1) - 1) & 1, err)) return false;
    fence_after();
    const uint32_t d = dcol + 128u * (i & 1);
    const uint32_t xo = x + (i & 1) * (NP * kXBytes / 16);
    if (leader) {
#pragma unroll
      for (int s = 0; s < kK1 / 16; s++)
        small_products<NP>([&](int a, int b) {
          mma_u<hi1, hi1, id>(d, xo + (a * (kXBytes / 16) + 16 * s), w1 + (b * (kW1Bytes / 16) + 16 * s),
                              (s > 0 || a > 0 || b < NP - 1) ? 1u : 0u);
        });
#pragma unroll
      for (int s = 0; s < kK1 / 16; s++) mma_u<hi1, hi1, id>(d, xo + 16 * s, w1 + 16 * s, 1u);
      mma_commit(&B.l1done[i & 1]);
    }
    __syncwarp();
    return true;
  };
  bool alive = layer1(0);
  for (uint32_t i = 0; i < n && alive; i++) {
    const uint32_t d = dcol + 128u * (i & 1);
#pragma unroll
    for (int c = 0; c < kChunks; c++) {
      if (c == kChunks / 2 && i + 1 < n && !(alive = layer1(i + 1))) break;
      if ((HOLD || c == 0) && !(alive = warp_wait(&B.afull[HOLD ? c : kChunks - 1], i & 1, err))) break;
      fence_after();
      if (leader) {
#pragma unroll
        for (int s = c * (8 / kChunks); s < (c + 1) * (8 / kChunks); s++)
          small_products<NP>([&](int a, int b) {
            mma_u_ta<hi2, id>(d, tmem + h1_col(a, i) + 8u * s, w2 + (b * (kW2Bytes / 16) + 16 * s),
                              (s > 0 || a > 0 || b < NP - 1) ? 1u : 0u);
          });
        mma_commit(&B.cdone[c]);
        if (c == kChunks - 1) {
#pragma unroll
          for (int s = 0; s < kHidden / 16; s++) mma_u_ta<hi2, id>(d, tmem + h1_col(0, i) + 8u * s, w2 + 16 * s, 1u);
          mma_commit(&B.l2done[i & 1]);
        }
      }
      __syncwarp();
    }
  }
  if (leader) {
    mma_commit(&B.last);
    mbar_wait(&B.last, 0, err);  // nothing in flight when tensor memory is given back
  }
  __syncwarp();
}

// A ReLU decision of the recompute can differ from the FP32 MLP's where the pre-activation is within
// their errors of zero, and one flipped mask moves that sample's whole gradient through the unit.  Unit n
// of layer 1 is uncertain when |z1_n| <= eps ||W1_n|| ||x||, unit n of layer 2 when |z2_n| <= eps ||W2_n||
// (||h1|| + ||x|| ||W1||_F) (its own sum plus layer 1's errors carried through W2); samples with an
// uncertain unit are listed (their sorted index, in rec_key; count in hdr[4]) and taken again by k_fwd_fix.
// With three parts the dropped products are ~2^-24 of a term; what is left is rounding: the tensor core's
// ~8 truncations at full size and the FP32 chain's ~K roundings, each some 2^-24 of ||w o x|| ~ ||w||
// ||x|| / sqrt(K), a total of ~2^-24 ||w|| ||x||: eps = 2^-21 leaves a factor of 8.  0.5% of the samples
// of the 8192-ray workload are listed (8.6% with two parts and 2^-17).
constexpr float kEps = 4.76837158203125e-07f;  // 2^-21

// What is written besides (c, w): nothing (a render), the ReLU masks (a backward follows), or the masks
// and the weight gradients' operands x, h1 and h2 (WgStage: the first two BF16 parts).
enum class Out { Colour, Masks, Stage };

// row group g (8 rows) of the staged operand at offset op (R rows) of one sample, whose rows start at col
__device__ __forceinline__ void stage_put(char* col, int op, int R, int g, const uint4& hi, const uint4& lo) {
  *reinterpret_cast<uint4*>(col + op + 256 * g) = hi;
  *reinterpret_cast<uint4*>(col + op + 32 * R + 256 * g) = lo;
}
// HOLD: E1 takes all of its 64 accumulator columns into registers before it converts them, so that layer 2
// can overwrite them as soon as the first chunk of h1 is written.  Without it E1 (and E2) load 32 at a
// time, layer 2 waits for both chunks, and G has the registers for more loads in flight.
// A render holds (62.5 M samples, NP = 3: 8.7 ms against 10.1); a recompute, whose E1 and E2 also keep
// masks, norms and staging addresses, does not (2.06 M samples of an FP32 grid: 0.51 ms against 0.59,
// with the staging 0.74 against 0.96 on 1.8 M: the held columns spilled).
template <Out OUT>
__host__ __device__ constexpr bool hold() { return OUT == Out::Colour; }

// CC, NF: channels and frequencies as constants (12 and 4), or 0: known at run time only.
template <int NP, int CC, int NF, Out OUT>
__global__ void __launch_bounds__(kThreads, 1) k_mlp_split(GridGeo g, MlpPtrs mlp, RenderWs w, const void* feat_,
                                                           int f16) {
  using namespace tc;
  using S = Smem<NP>;
  constexpr bool HOLD = hold<OUT>(), ODD = NP == 3 && OUT == Out::Colour;
  using RG = Regs<HOLD>;
  extern __shared__ __align__(1024) char sm[];
  Bars& B = *(Bars*)(sm + S::bars);
  uint32_t* err = &w.hdr[0];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the weights, split; biases and layer 3 in FP32
  load_weights<NP>(sm + S::w1, kW1Bytes, mlp.w1, kHidden, mlp.in_dim, kK1);
  load_weights<NP>(sm + S::w2, kW2Bytes, mlp.w2, kHidden, kHidden, kHidden);
  float* b1s = (float*)(sm + S::b1);
  float* l3 = (float*)(sm + S::l3);
  float* b3s = (float*)(sm + S::b3);
  for (int i = threadIdx.x; i < kHidden; i += kThreads) {
    b1s[i] = mlp.b1[i];
    float* p = l3 + 8 * (i >> 1) + (i & 1);
    p[0] = mlp.b2[i];
    p[2] = mlp.w3[i];
    p[4] = mlp.w3[kHidden + i];
    p[6] = mlp.w3[2 * kHidden + i];
  }
  if (threadIdx.x < 4) b3s[threadIdx.x] = threadIdx.x < 3 ? mlp.b3[threadIdx.x] : 0.0f;
  float* nrm = (float*)(sm + S::nrm);
  if constexpr (OUT != Out::Colour) {  // a warp per row
    for (int r = wid; r < 2 * kHidden; r += kThreads / 32) {
      const int in = r < kHidden ? mlp.in_dim : kHidden;
      const float* row = r < kHidden ? mlp.w1 + r * in : mlp.w2 + (r - kHidden) * in;
      float q = 0.0f;
      for (int k = lane; k < in; k += 32) q = fmaf(row[k], row[k], q);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      if (lane == 0) nrm[r] = sqrtf(q);
    }
  }
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; b++) {
      mbar_init(&B.xfull[b], kGatWarps);
      mbar_init(&B.l1done[b], 1);
      mbar_init(&B.l2done[b], 1);
      mbar_init(&B.dfree[b], kEpiWarps);
      mbar_init(&B.hfull[b], kEpiWarps);
    }
    for (int c = 0; c < kChunks; c++) {
      mbar_init(&B.afull[c], kEpiWarps);
      mbar_init(&B.cdone[c], 1);
    }
    for (int k = 0; k < kMeta; k++) {
      mbar_init(&B.zfull[k], kEpiWarps / 2);
      mbar_init(&B.mfull[k], kGatWarps);
    }
    mbar_init(&B.last, 1);
    B.odd = B.marked = 0u;
    fence_mbar_init();
  }
  fence_proxy_async();
  if (wid == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&B.tmem)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  if constexpr (ODD) {
    const uint32_t f = odd_parameters<NP>(sm);
    if (f) atomicOr(&B.odd, f);
    __syncthreads();
    if (B.odd & kOddNan) {
      drop_nan_units<NP>(sm, mlp);
      fence_proxy_async();
      __syncthreads();
    }
  }
  if constexpr (OUT != Out::Colour) {
    if (wid == 0) {
      float q = 0.0f;
      for (int k = lane; k < kHidden; k += 32) q = fmaf(nrm[k], nrm[k], q);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      if (lane == 0) nrm[2 * kHidden] = sqrtf(q);
    }
    __syncthreads();
  }
  const uint32_t tmem = B.tmem;
  dependents_sync();  // the weights are in place by the time the previous kernel has ended
  const uint32_t dcol = tmem + Tmem<NP>::acc;  // accumulator of tile i: dcol + 128 (i & 1)

  const uint32_t n_tiles = w.hdr[1];
  const uint32_t per = (n_tiles + gridDim.x - 1) / gridDim.x;
  const uint32_t t0 = min(n_tiles, blockIdx.x * per), n = min(n_tiles, t0 + per) - t0;

  if (wid < kE2) {
    // ------------------------------------------------------------------ E1: layer 1 -> h1
    set_regs<RG::e1>();
    const int h = wid >> 2, m = (wid & 3) * 32 + lane;
    const uint32_t lanes = (uint32_t)((wid & 3) * 32) << 16;
    const float4* meta = (const float4*)(sm + S::meta);
    (void)m;
    (void)meta;
    bool alive = true;
    const bool tiny = ODD && (B.odd & kOddTiny);
    (void)tiny;
    for (uint32_t i = 0; i < n && alive; i++) {
      if (!(alive = warp_wait(&B.l1done[i & 1], (i >> 1) & 1, err))) break;
      uint32_t rid = 0xffffffffu, mw[2] = {0u, 0u}, unsure = 0u;
      float2 hh = make_float2(0.f, 0.f);  // ||h1||^2 of this half
      float tx = 0.0f;
      char* stg = nullptr;
      if constexpr (OUT != Out::Colour) {
        if (!(alive = warp_wait(&B.mfull[i % kMeta], (i / kMeta) & 1, err))) break;
        const float4 md = meta[(i % kMeta) * kTile + m];
        rid = __float_as_uint(md.x);
        tx = -kEps * sqrtf(md.w);
        if (OUT == Out::Stage) stg = w.stage + stage_col(__float_as_uint(md.z));
      }
      fence_after();
      float v[HOLD ? 64 : 32];
      if constexpr (HOLD) load_half(dcol + 128u * (i & 1) + lanes, h, v);
      if constexpr (ODD) {
        if (tiny && any_huge<64>(v)) v[0] = NAN;
      }
#pragma unroll
      for (int q4 = 0; q4 < 4; q4++) {  // 16 units at a time, 4 / kChunks of them per chunk
        if constexpr (!HOLD) {
          if (q4 % 2 == 0) load_quarter(dcol + 128u * (i & 1) + lanes, h, q4 / 2, v);
        }
        constexpr int kPer = 4 / kChunks;
        const int c = q4 / kPer;
        const float4* b4 = reinterpret_cast<const float4*>(b1s + 32 * q4 + 16 * h);
        uint32_t o[NP][8];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const float4 b = b4[q];
          const float* z = v + 16 * (HOLD ? q4 : q4 % 2) + 4 * q;
          const float2 u0 = add2(make_float2(z[0], z[1]), make_float2(b.x, b.y));
          const float2 u1 = add2(make_float2(z[2], z[3]), make_float2(b.z, b.w));
          float2 r0 = make_float2(fmaxf(u0.x, 0.0f), fmaxf(u0.y, 0.0f));
          if constexpr (ODD) {
            if (q4 == 0 && q == 0) r0.x = relu_nan(u0.x);
          }
          const float2 r1 = make_float2(fmaxf(u1.x, 0.0f), fmaxf(u1.y, 0.0f));
          if constexpr (OUT != Out::Colour) {
            mw[q4 & 1] |= ((u0.x > 0.0f ? 1u : 0u) | (u0.y > 0.0f ? 2u : 0u) | (u1.x > 0.0f ? 4u : 0u) |
                           (u1.y > 0.0f ? 8u : 0u)) << (8 * q + 4 * (q4 >> 1));
            const float4 nw = reinterpret_cast<const float4*>(nrm + 32 * q4 + 16 * h)[q];
            // (the sign of |z| - eps ||W_n|| ||x||: set where uncertain; a NaN decides like the FP32 MLP)
            unsure |= __float_as_uint(fmaf(tx, nw.x, fabsf(u0.x))) | __float_as_uint(fmaf(tx, nw.y, fabsf(u0.y)));
            unsure |= __float_as_uint(fmaf(tx, nw.z, fabsf(u1.x))) | __float_as_uint(fmaf(tx, nw.w, fabsf(u1.y)));
            hh = fma2(r0, r0, hh);
            hh = fma2(r1, r1, hh);
          }
          uint32_t p0[NP], p1[NP];
          split2<NP>(r0, p0);
          split2<NP>(r1, p1);
#pragma unroll
          for (int k = 0; k < NP; k++) {
            o[k][2 * q] = p0[k];
            o[k][2 * q + 1] = p1[k];
          }
        }
        if (OUT == Out::Stage && rid != 0xffffffffu) {
#pragma unroll
          for (int u = 0; u < 2; u++)
            stage_put(stg, WgStage::h1, kHidden, 4 * q4 + 2 * h + u,
                      make_uint4(o[0][4 * u], o[0][4 * u + 1], o[0][4 * u + 2], o[0][4 * u + 3]),
                      make_uint4(o[1][4 * u], o[1][4 * u + 1], o[1][4 * u + 2], o[1][4 * u + 3]));
        }
        // the hi part's other buffer is free (layer 2 of tile i - 2 was issued before layer 1 of tile i)
        tmem_st8(tmem + lanes + h1_col(0, i) + 16u * q4 + 8u * h, o[0]);
        if (i > 0 && q4 % kPer == 0) {  // the smaller parts of tile i - 1's chunk have been read
          if (!(alive = warp_wait(&B.cdone[c], (i - 1) & 1, err))) break;
          fence_after();
        }
#pragma unroll
        for (int k = 1; k < NP; k++) tmem_st8(tmem + lanes + h1_col(k, i) + 16u * q4 + 8u * h, o[k]);
        if (q4 % kPer == kPer - 1) {
          tmem_wait_st();
          fence_before();
          warp_arrive(&B.afull[c]);
        }
      }
      if constexpr (OUT != Out::Colour) {
        if (!alive) break;
        ((float*)(sm + S::hs))[((i & 1) * 2 + h) * kTile + m] =
            __uint_as_float(__float_as_uint(hh.x + hh.y) | (unsure & 0x80000000u));
        warp_arrive(&B.hfull[i & 1]);
        if (rid != 0xffffffffu)
          *reinterpret_cast<uint2*>(reinterpret_cast<char*>(w.rec_mask + 2 * (size_t)rid) + 8 * h) =
              make_uint2(mw[0], mw[1]);
      }
    }
  } else if (wid < kG) {
    // ------------------------------------------------------------------ E2: layer 2 -> layer 3 -> record
    set_regs<RG::e2>();
    const int h = (wid - kE2) >> 2, m = (wid & 3) * 32 + lane;
    const uint32_t lanes = (uint32_t)((wid & 3) * 32) << 16;
    float4* zbuf = (float4*)(sm + S::z);
    const float4* meta = (const float4*)(sm + S::meta);
    for (uint32_t t = 0; t < n; t++) {
      if (!warp_wait(&B.l2done[t & 1], (t >> 1) & 1, err)) break;
      if (!warp_wait(&B.mfull[t % kMeta], (t / kMeta) & 1, err)) break;
      fence_after();
      const float4 md = meta[(t % kMeta) * kTile + m];
      const uint32_t rid = __float_as_uint(md.x);
      uint32_t mw[2] = {0u, 0u}, sh[2][4], unsure = 0u;
      float th = 0.0f;
      if constexpr (OUT != Out::Colour) {
        if (!warp_wait(&B.hfull[t & 1], (t >> 1) & 1, err)) break;
        const float* hs = (const float*)(sm + S::hs) + (t & 1) * 2 * kTile + m;
        unsure = __float_as_uint(hs[0]) | __float_as_uint(hs[kTile]);
        th = -kEps * (sqrtf(fabsf(hs[0]) + fabsf(hs[kTile])) + sqrtf(md.w) * nrm[2 * kHidden]);
      }
      char* stg = OUT == Out::Stage ? w.stage + stage_col(__float_as_uint(md.z)) : nullptr;
      (void)mw;
      (void)sh;
      (void)stg;
      (void)th;
      float v[HOLD ? 64 : 32];
      if constexpr (HOLD) {  // all of it, to free the accumulator at once
        load_half(dcol + 128u * (t & 1) + lanes, h, v);
        fence_before();
        warp_arrive(&B.dfree[t & 1]);
      }
      float2 z0 = make_float2(0.f, 0.f), z1 = z0, z2 = z0;
      const float4* l4 = reinterpret_cast<const float4*>(l3) + 16 * h;  // two per pair of units
#pragma unroll
      for (int q = 0; q < 32; q++) {
        if constexpr (!HOLD) {
          if (q % 16 == 0) load_quarter(dcol + 128u * (t & 1) + lanes, h, q / 16, v);
          if (q == 16) {
            fence_before();
            warp_arrive(&B.dfree[t & 1]);
          }
        }
        if constexpr (ODD) {  // a NaN stays one, a number adds 0
          if (q == 0) z0.x = 0.0f * v[0];
        }
        const float4 a = l4[32 * (q / 8) + 2 * (q % 8)], b = l4[32 * (q / 8) + 2 * (q % 8) + 1];
        float2 u = add2(make_float2(v[2 * (HOLD ? q : q % 16)], v[2 * (HOLD ? q : q % 16) + 1]), make_float2(a.x, a.y));
        if constexpr (OUT != Out::Colour) {
          mw[(q >> 3) & 1] |= ((u.x > 0.0f ? 1u : 0u) | (u.y > 0.0f ? 2u : 0u)) <<
                              (8 * ((q & 7) >> 1) + 2 * (q & 1) + 4 * (q >> 4));
          const float2 nw = *reinterpret_cast<const float2*>(nrm + kHidden + 32 * (q / 8) + 16 * h + 2 * (q % 8));
          unsure |= __float_as_uint(fmaf(th, nw.x, fabsf(u.x))) | __float_as_uint(fmaf(th, nw.y, fabsf(u.y)));
        }
        u.x = fmaxf(u.x, 0.0f);
        u.y = fmaxf(u.y, 0.0f);
        z0 = fma2(make_float2(a.z, a.w), u, z0);
        z1 = fma2(make_float2(b.x, b.y), u, z1);
        z2 = fma2(make_float2(b.z, b.w), u, z2);
        if constexpr (OUT == Out::Stage) {
          uint32_t p[2];
          split2<2>(u, p);
          sh[0][q & 3] = p[0];
          sh[1][q & 3] = p[1];
          if ((q & 3) == 3 && rid != 0xffffffffu)  // 8 units complete
            stage_put(stg, WgStage::h2, kHidden, 4 * (q >> 3) + 2 * h + ((q >> 2) & 1),
                      make_uint4(sh[0][0], sh[0][1], sh[0][2], sh[0][3]), make_uint4(sh[1][0], sh[1][1], sh[1][2], sh[1][3]));
        }
      }
      if (OUT != Out::Colour && rid != 0xffffffffu)
        *reinterpret_cast<uint2*>(reinterpret_cast<char*>(w.rec_mask + 2 * (size_t)rid + 1) + 8 * h) =
            make_uint2(mw[0], mw[1]);
      float4* zp = &zbuf[(t % kMeta) * kTile + m];
      if (h) {
        *zp = make_float4(z0.x + z0.y, z1.x + z1.y, z2.x + z2.y, __uint_as_float(unsure));
        warp_arrive(&B.zfull[t % kMeta]);
      } else {
        if (!warp_wait(&B.zfull[t % kMeta], (t / kMeta) & 1, err)) break;
        const float4 o = *zp;
        if constexpr (OUT != Out::Colour) {  // list the uncertain samples (one atomic per warp)
          const bool fix = rid != 0xffffffffu && ((unsure | __float_as_uint(o.w)) >> 31);
          const uint32_t bal = __ballot_sync(0xffffffffu, fix);
          uint32_t base = 0;
          if (lane == 0 && bal) base = atomicAdd(&w.hdr[4], (uint32_t)__popc(bal));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (fix) w.rec_key[base + __popc(bal & ((1u << lane) - 1u))] = __float_as_uint(md.z);
        }
        if (rid != 0xffffffffu) {
          float4 c = make_float4(sigmoid_f(z0.x + z0.y + o.x + b3s[0]), sigmoid_f(z1.x + z1.y + o.y + b3s[1]),
                                 sigmoid_f(z2.x + z2.y + o.z + b3s[2]), md.y);
          if constexpr (ODD) {
            if (isnan(c.x)) {
              c.x = __uint_as_float(kOddColour);
              B.marked = 1u;
            }
          }
          w.rec_c[rid] = c;
        }
      }
    }
    if constexpr (ODD) {  // the marked samples again, a tile per warp at a time
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");  // every mark of E2's warps
      const bool all = B.odd & kOddAll;
      if (all || (B.marked && !(B.odd & kOddBlind))) {
        for (uint32_t i = wid - kE2; i < n; i += kEpiWarps) {
          const uint4 td = w.tile[t0 + i];
          for (uint32_t k = 0; k < (td.y & 0xFFu); k += 32) {
            uint32_t rid = 0xffffffffu;
            if (k + lane < (td.y & 0xFFu)) rid = __float_as_uint(w.srt[td.x + k + lane].qd.x);
            uint32_t todo = __ballot_sync(0xffffffffu, rid != 0xffffffffu && (all ||
                                                       __float_as_uint(w.rec_c[rid].x) == kOddColour));
            for (; todo; todo &= todo - 1u) {
              const int s = __ffs(todo) - 1;
              const float3 c = sample_f32(g, mlp, feat_, f16, w.srt + td.x + k + s,
                                         !(B.odd & (kOddAll | kOddNan)));
              if (lane == s) w.rec_c[rid] = make_float4(c.x, c.y, c.z, w.rec_c[rid].w);
            }
          }
        }
      }
    }
  } else if (wid < kM) {
    // ------------------------------------------------------------------ G: the input rows
    set_regs<RG::g>();
    const int m = (wid & 3) * 32 + lane;
    const uint32_t grp = (uint32_t)(wid - kG) / kGatWarps;  // takes tiles grp, grp + 2, ...
    const int C = CC ? CC : g.C, n_freq = NF ? NF : mlp.n_freq, Br = g.brick;
    float4* meta = (float4*)(sm + S::meta);
    const bool tiny = ODD && (B.odd & kOddTiny);
    (void)tiny;
    uint4 td = make_uint4(0u, 0u, 0u, 0u);
    float4 pw = make_float4(0.f, 0.f, 0.f, 0.f), qd = pw;
    auto fetch = [&](uint32_t i) {
      td = w.tile[t0 + i];
      if (m < (int)(td.y & 0xFFu)) {
        pw = w.srt[td.x + m].pw;
        qd = w.srt[td.x + m].qd;
      }
    };
    if (grp < n) fetch(grp);
    for (uint32_t i = grp; i < n; i += 2) {
      const bool valid = m < (int)(td.y & 0xFFu);
      float x[kK1];
#pragma unroll
      for (int k = 0; k < kK1; k++) x[k] = 0.0f;
      float d[3] = {0.f, 0.f, 0.f};
      float4 md = make_float4(__uint_as_float(0xffffffffu), 0.f, 0.f, 0.f);
      if (valid) {
        const float p[3] = {pw.x, pw.y, pw.z};
        d[0] = qd.y;
        d[1] = qd.z;
        d[2] = qd.w;
        md.x = qd.x;
        md.y = pw.w;
        md.z = __uint_as_float(td.x + m);  // its place in the sorted order
        const int bx = (int)(td.w & 0xFFFFu), by = (int)(td.w >> 16), bz = (int)((td.y >> 8) & 0x1FFFu);
        int i0[3];
        float f[3];
        const bool in = index_sample(g, p, i0, f);
        const int l[3] = {i0[0] - bx * Br, i0[1] - by * Br, i0[2] - bz * Br};
        if (!(in && l[0] >= 0 && l[0] < Br && l[1] >= 0 && l[1] < Br && l[2] >= 0 && l[2] < Br))
          set_err(err, kErrInternal);
        else if (f16)
          gather<__half, CC>(g, (const __half*)feat_, i0, f, x);
        else
          gather<float, CC>(g, (const float*)feat_, i0, f, x);
      }
      if (i + 2 < n) fetch(i + 2);
      if constexpr (ODD) {
        if (tiny && any_huge<CC ? CC : kMaxC>(x)) x[0] = INFINITY;
      }
      if (CC && NF && valid) encode<NF>(d, x + CC);
      if constexpr (OUT != Out::Colour) {  // ||x||^2 (the encoding's part below, if it is not in x yet)
#pragma unroll
        for (int k = 0; k < kK1; k++) md.w = fmaf(x[k], x[k], md.w);
      }
      // x's buffer: layer 1 of tile i - 2 has read it
      if (i >= 2 && !warp_wait(&B.l1done[i & 1], ((i >> 1) - 1) & 1, err)) break;
      char* xb = sm + S::x + (int)(i & 1) * NP * kXBytes;
#pragma unroll
      for (int k0 = 0; k0 < kK1; k0 += 8) {
        uint4 q[NP];
        split_row<NP>(x + k0, q);
#pragma unroll
        for (int p = 0; p < NP; p++) *reinterpret_cast<uint4*>(xb + p * kXBytes + kmaj_off(m, k0, kK1)) = q[p];
        if (OUT == Out::Stage && CC && NF && valid)
          stage_put(w.stage + stage_col(__float_as_uint(md.z)), WgStage::x, kMaxIn, k0 / 8, q[0], q[1]);
      }
      if (!(CC && NF) && valid) {
        // channels known at run time only: the encoding is written over columns C .. element by element
        constexpr int F = (kK1 - 4) / 6;  // most frequencies with one channel
        float e[3 + 6 * F + 1];
        e[3 + 6 * F] = 0.0f;
        encode<F>(d, e);
        const int ne = 3 + 6 * n_freq;
#pragma unroll
        for (int j = 0; j < 3 + 6 * F; j += 2) {
          uint32_t p[NP];
          split2<NP>(make_float2(e[j], e[j + 1]), p);
#pragma unroll
          for (int u = 0; u < 2; u++) {
            const int k = C + j + u;
            if (OUT != Out::Colour && j + u < ne) md.w = fmaf(e[j + u], e[j + u], md.w);
            if (j + u < ne)
#pragma unroll
              for (int a = 0; a < NP; a++)
                *reinterpret_cast<uint16_t*>(xb + a * kXBytes + kmaj_off(m, 0, kK1) + (k >> 3) * 128 + (k & 7) * 2) =
                    (uint16_t)(p[a] >> (16 * u));
          }
        }
      }
      if (OUT == Out::Stage && !(CC && NF) && valid) {  // the row as it now stands in shared memory
#pragma unroll
        for (int k0 = 0; k0 < kK1; k0 += 8)
          stage_put(w.stage + stage_col(__float_as_uint(md.z)), WgStage::x, kMaxIn, k0 / 8,
                    *reinterpret_cast<uint4*>(xb + kmaj_off(m, k0, kK1)),
                    *reinterpret_cast<uint4*>(xb + kXBytes + kmaj_off(m, k0, kK1)));
      }
      meta[(i % kMeta) * kTile + m] = md;
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        arrive(&B.xfull[i & 1]);
        arrive(&B.mfull[i % kMeta]);
      }
    }
  } else {
    // ------------------------------------------------------------------ M: the MMAs
    set_regs<RG::m>();
    if (wid == kM && n) issue_mmas<NP, HOLD>(sm, B, tmem, n, err);
  }
  fence_before();
  __syncthreads();
  if (wid == 0) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}
template <int NP, int CC, int NF, Out OUT>
static cicero_status launch(const cicero_grid* grid, const GridGeo& geo, const MlpPtrs& mlp, const RenderWs& ws,
                            cudaStream_t st) {
  auto kern = k_mlp_split<NP, CC, NF, OUT>;
  constexpr int smem = OUT == Out::Colour ? Smem<NP>::bytes : Smem<NP>::bytes_bwd;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_mlp_split)");
  {
    ProfScope ps(kStGatherMlp, st);
    launch_kernel(kern, num_sms(), kThreads, smem, st, geo, mlp, ws, grid->features, grid->dtype == CICERO_F16);
  }
  count_launches(1);
  e = cudaGetLastError();
  return e == cudaSuccess ? CICERO_OK : cuda_fail(e, "k_mlp_split");
}

template <int NP, Out OUT>
static cicero_status launch_channels(const cicero_grid* grid, const GridGeo& geo, const MlpPtrs& mlp,
                                     const RenderWs& ws, cudaStream_t st) {
  return geo.C == 12 && mlp.n_freq == 4 ? launch<NP, 12, 4, OUT>(grid, geo, mlp, ws, st)
                                        : launch<NP, 0, 0, OUT>(grid, geo, mlp, ws, st);
}

}  // namespace ms

cicero_status launch_mlp_split(const cicero_grid* grid, const GridGeo& geo, int parts, const MlpPtrs& mlp,
                               const RenderWs& ws, cudaStream_t st) {
  return parts == 3 ? ms::launch_channels<3, ms::Out::Colour>(grid, geo, mlp, ws, st)
                    : ms::launch_channels<2, ms::Out::Colour>(grid, geo, mlp, ws, st);
}

cicero_status launch_mlp_recompute(const cicero_grid* grid, const GridGeo& geo, const MlpPtrs& mlp, const RenderWs& ws,
                                   cudaStream_t st) {
  return ws.stage ? ms::launch_channels<3, ms::Out::Stage>(grid, geo, mlp, ws, st)
                  : ms::launch_channels<3, ms::Out::Masks>(grid, geo, mlp, ws, st);
}

}  // namespace cicero
