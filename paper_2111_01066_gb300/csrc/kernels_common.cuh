// Device-side descriptors and helpers shared by the kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace tnx {

// Programmatic dependent launch.  Every kernel of a plan or a pairwise
// contraction is launched with the stream-serialisation attribute: it may start
// once every CTA of the kernel before it has passed its own pdl_wait, sets itself
// up under that kernel's run, and waits here until that kernel has completed and
// its writes are visible (to ordinary loads: what another kernel of the chain
// writes is never read as read-only data).  Before pdl_wait a kernel touches only its arguments,
// tables written when the plan was built, and its own shared and tensor memory;
// every thread that touches anything else passes it, so a kernel's completion
// implies that of all kernels before it.  The next kernel is let go after the
// wait, not before it: no CTA is then resident while the kernel two before its
// own still runs.  Without the attribute (a launch outside such a chain) both
// instructions are no-ops.
// A chain of small kernels costs 4-6 us a link without it (launch, arguments,
// decode tables, then the work).
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Per-chunk parameters, read by the kernels from device memory at
// params[*counter] so that one captured launch sequence serves every chunk.
struct ChunkParam {
  uint64_t slice_base;   // first slice id of the chunk (aligned to 2^b)
  uint64_t valid_lo;     // slices [valid_lo, valid_hi) of the chunk are summed
  uint64_t valid_hi;
  uint64_t bitstring;    // closed output bits of the batch
  int64_t out_index;     // batch index into the output amplitudes
  double* out;           // the call's output amplitudes (complex128)
};

// Launch arguments of one gathered complex GEMM (one plan step or one
// tn_contract_pair call).  C[m, n] = sum_k A[m, k] B[k, n] for every batch
// instance; operand element offsets are sums of 2^position over set bits.
constexpr int KMAXR = 48;
constexpr int KMAXB = 16;
constexpr int KTB = 24;   // tile bits per operand tile
struct GemmArgs {
  const float2* A;
  const float2* B;
  float2* C;
  // instance i of a batch starts at i * istride + sum_j bit_j(i) 2^{bpos[j]}
  int64_t a_istride, b_istride, c_istride;
  int32_t n_inst;                  // batch instances (grid z)
  int32_t nb;                      // bits of the instance index deposited through *_bpos
  int32_t nm, nk, nn;              // log2 M, K, N
  int32_t tm, tk, tn;              // log2 of the tile extents actually used
  // tile decode in memory-position order: *_tsel[t] = index | (64 if a k bit)
  int32_t a_tbits, b_tbits;
  int8_t a_tpos[KTB], a_tsel[KTB];
  int8_t b_tpos[KTB], b_tsel[KTB];
  // all bit positions (tile bits first)
  int8_t a_mpos[KMAXR], a_kpos[KMAXR], b_kpos[KMAXR], b_npos[KMAXR], c_mpos[KMAXR], c_npos[KMAXR];
  int8_t a_bpos[KMAXB], b_bpos[KMAXB], c_bpos[KMAXB];
  // FP16 split with power-of-two scaling (NULL when unused): max |re|, |im| of
  // A and B (written by their producers) and C's maximum, which this GEMM
  // records for its consumer
  const float* amax_a;
  const float* amax_b;
  float* amax_c;
  // lanes (chunks run side by side, one arena each, see k_leaf_select): their bits
  // are the highest of the instance index; lane l records its maximum at
  // amax_c + l * amax_lane
  int32_t ls_lanes;                // log2 of the lanes (0: one)
  int32_t amax_lane;
};

static_assert(sizeof(GemmArgs) % 4 == 0, "GemmArgs is copied to shared memory in 4-byte words");

// Exponent s of the power-of-two scale 2^s that maps a tensor's largest
// component into [2^14, 2^15), inside the FP16 range (|s| <= 126; 0 when the
// maximum is zero, subnormal or not recorded).
__device__ __forceinline__ int fp16_scale_exp(const float* amax) {
  if (!amax) return 0;
  // past L1: the maxima share sectors with ones that running kernels raise
  const int be = (int)((__float_as_uint(__ldcg(amax)) >> 23) & 255u);
  if (be == 0 || be == 255) return 0;
  const int s = 14 - (be - 127);
  return s < -126 ? -126 : (s > 126 ? 126 : s);
}
// 2^e for |e| <= 126, exact
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }
// Warp-collective: raise *amax_c to the warp's largest m (m >= 0; non-negative
// floats order like their bit patterns).
__device__ __forceinline__ void amax_update(float* amax_c, float m) {
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned*>(amax_c), __float_as_uint(m));
}
__device__ __forceinline__ float cabs_max(float2 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }

// Sum over bits i < n <= N of bit_i(x) << pos[i], unrolled (no loop over the argument bank)
template <int N>
__device__ __forceinline__ int64_t deposit_lo(uint32_t x, const int8_t* pos, int n) {
  int64_t r = 0;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i < n && ((x >> i) & 1u)) r += (int64_t)1 << pos[i];
  return r;
}

// Sum over bits i >= from of bit_{i - from}(x) << pos[i], one bit per lane (the
// positions are distinct, so the sum is an OR); every lane of the warp calls it.
__device__ __forceinline__ int64_t warp_deposit(uint32_t x, const int8_t* pos, int from, int to) {
  const int lane = threadIdx.x & 31;
  uint64_t v = 0;
  if (from + lane < to && ((x >> lane) & 1u)) v = (uint64_t)1 << pos[from + lane];
  const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)v);
  const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32));
  return (int64_t)(((uint64_t)hi << 32) | lo);
}
__device__ __forceinline__ int64_t warp_inst_offset(uint32_t inst, int64_t istride, const int8_t* bpos, int nb) {
  return (int64_t)inst * istride + warp_deposit(inst, bpos, 0, nb);
}

}  // namespace tnx
