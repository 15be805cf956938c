// Small kernels of the slice loop: leaf select (slicing, main text section II),
// FP64 slice sum into the amplitudes, chunk advance, XEB reduction (Eq. (1))
// and the standalone index permutation (SI Eq. (2)).
#pragma once
#include "kernels_common.cuh"
#include "tn_internal.h"

namespace tnx {

// Materialise every leaf of the chunk: the sliced wires take the bits of the
// slice id, the closed output wires the bits of the batch's bitstring.  Lane
// blockIdx.y does so for the chunk params[counter + lane] in its own arena: the
// chunks of several lanes then run through the same launches, as further instances
// of every step, which is what chains of steps too small for the GPU wait for (a
// chunk of 11 steps of 2^11 multiply-adds or less takes 36 us of launches, nine of
// them side by side hardly more).  Also clears amax[z0, z1) of the lane (FP16 split:
// the maxima the coming steps record).
__global__ void __launch_bounds__(128) k_leaf_select(const float2* __restrict__ leaf_data,
                                                     const LeafDesc* __restrict__ leaves, int n_leaves,
                                                     float2* arena, const ChunkParam* params,
                                                     const unsigned* counter, int64_t lane_stride,
                                                     float* amax, int amax_lane, int z0, int z1) {
  const int lane = blockIdx.y;
  arena += lane * lane_stride;
  amax += (int64_t)lane * amax_lane;
  __shared__ LeafDesc d;
  static_assert(sizeof(LeafDesc) % 4 == 0, "LeafDesc is copied in 4-byte words");
  bool waited = false;
  ChunkParam p{};
  for (int li = blockIdx.x; li < n_leaves; li += gridDim.x) {
    __syncthreads();
    for (int w = threadIdx.x; w < (int)(sizeof(LeafDesc) / 4); w += blockDim.x)
      reinterpret_cast<uint32_t*>(&d)[w] = reinterpret_cast<const uint32_t*>(leaves + li)[w];
    __syncthreads();
    if (!waited) {
      pdl_wait();
      p = params[__ldcg(counter) + lane];
      for (int i = z0 + blockIdx.x * blockDim.x + threadIdx.x; i < z1; i += gridDim.x * blockDim.x) amax[i] = 0.f;
      waited = true;
    }
    const int rank = d.rank;
    const int64_t per = (int64_t)1 << rank;
    const int nbat = __popc(d.bmask);
    const int64_t total = per << nbat;
    // the bits every instance shares, and those that an instance's batch bits set
    int64_t fix0 = 0;
    for (int f = 0; f < d.nfixed; ++f) {
      const int idx = d.fixed_index[f];
      const uint64_t v = d.fixed_kind[f] == 0 ? ((p.slice_base >> idx) & 1) : ((p.bitstring >> idx) & 1);
      fix0 |= (int64_t)v << f;
    }
    for (int64_t e = threadIdx.x; e < total; e += blockDim.x) {
      const uint32_t inst = (uint32_t)(e >> rank);
      const int64_t i = e & (per - 1);
      int64_t fix = fix0;
      for (int t = 0; t < nbat; ++t)
        if ((inst >> t) & 1u)
          for (int f = 0; f < d.nfixed; ++f)
            if (d.fixed_kind[f] == 0 && d.fixed_index[f] == d.bslice[t]) fix |= (int64_t)1 << f;
      arena[d.dst_off + e] = leaf_data[d.src_off + fix * per + i];
    }
  }
  if (!waited) pdl_wait();
}

// Slice sum of a chunk (main text, section II: the sliced network is the sum of
// the smaller networks) in FP64, deterministic: block (x, g, lane) sums the slices of
// group g (slices g*per .. g*per+per-1 of the lane's chunk) for its amplitudes j into
// part[lane][g][j]; the last of the lane's blocks to arrive for the same amplitudes
// adds its groups, the last lane's block adds the lanes into out[batch][j], both in
// order, and the last block of all advances the chunk counter by the lanes.  Slices outside the call's range are
// skipped.  The tickets are zero between launches.
// MAXJ: amplitudes that a thread holds in registers, 1 where the grid has a thread
// for each: the registers of four, mostly unused, let two blocks on an SM (4096
// slices of 4096 amplitudes: 206-215 us, 157 with one).
template <int MAXJ>
__global__ void __launch_bounds__(256) k_root_sum(const float2* arena, const RootDesc r, int b,
                                                 int groups, double2* part,
                                                 const ChunkParam* params, unsigned* counter,
                                                 unsigned* tickets, int64_t lane_stride) {
  // the group's slices in rounds of 256: their instance offsets in the root
  // (or -1 outside the call's range) are found once per block, then every
  // thread adds its amplitudes over them with four independent FP64
  // accumulators (slice i of a round goes to accumulator i % 4), combined in a
  // fixed order.  256 threads, s_off has 256 entries: cnt <= 256 and its padding
  // to a multiple of 4 stays <= 256
  __shared__ int64_t s_off[256];
  __shared__ int s_last;
  pdl_wait();
  const int lane = blockIdx.z, lanes = gridDim.z;
  const unsigned first = __ldcg(counter);   // changes under a running kernel: past L1
  const ChunkParam p = params[first + lane];
  arena += lane * lane_stride;
  const int k = r.rank;
  const int64_t nout = (int64_t)1 << k;
  const uint32_t per = (1u << b) / (uint32_t)groups;
  const int g = blockIdx.y;
  const int nbat = __popc(r.bmask);
  const int64_t j0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t jstep = (int64_t)gridDim.x * blockDim.x;
  // every thread of the block takes part in the rounds (the barriers) the same
  // number of times, even where it has no amplitude: the pass count depends
  // on the grid only
  const int my_n = j0 < nout ? (int)((nout - 1 - j0) / jstep) + 1 : 0;
  const int64_t max_n = (nout + jstep - 1) / jstep;
  const int passes = (int)((max_n + MAXJ - 1) / MAXJ);
  double ar[MAXJ][4], ai[MAXJ][4];
  int64_t ri[MAXJ];
  for (int pass = 0; pass < passes; ++pass) {
    const int jj0 = pass * MAXJ;
    const int nj = my_n - jj0 < 0 ? 0 : (my_n - jj0 < MAXJ ? my_n - jj0 : MAXJ);
#pragma unroll
    for (int t = 0; t < MAXJ; ++t) {
      ri[t] = 0;
      if (t < nj) {
        const int64_t j = j0 + (int64_t)(jj0 + t) * jstep;
        for (int q = 0; q < k; ++q)
          if ((j >> q) & 1) ri[t] |= (int64_t)1 << r.pos_of_open[q];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) ar[t][u] = ai[t][u] = 0.0;
    }
    for (uint32_t s0 = (uint32_t)g * per; s0 < (uint32_t)(g + 1) * per; s0 += 256) {
      const uint32_t cnt = min(256u, (uint32_t)(g + 1) * per - s0);
      const uint32_t cnt4 = (cnt + 3u) & ~3u;   // padded with -1 (no slice) to whole quadruples
      __syncthreads();
      if (threadIdx.x < cnt4) {
        const uint32_t sl = s0 + threadIdx.x;
        const uint64_t sid = p.slice_base + sl;
        int64_t o = -1;
        if (threadIdx.x < cnt && sid >= p.valid_lo && sid < p.valid_hi) {
          uint32_t inst = 0;
          for (int t = 0; t < nbat; ++t) inst |= ((sl >> r.bslice[t]) & 1u) << t;
          o = r.off + ((int64_t)inst << k);
        }
        s_off[threadIdx.x] = o;
      }
      __syncthreads();
      // four slices per pass, one per accumulator: four independent loads in flight
      for (uint32_t i = 0; i < cnt4; i += 4) {
        int64_t o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) o[u] = s_off[i + u];
#pragma unroll
        for (int t = 0; t < MAXJ; ++t)
          if (t < nj) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (o[u] >= 0) {
                const float2 v = arena[o[u] + ri[t]];
                ar[t][u] += (double)v.x;
                ai[t][u] += (double)v.y;
              }
          }
      }
    }
#pragma unroll
    for (int t = 0; t < MAXJ; ++t)
      if (t < nj) {
        const int64_t j = j0 + (int64_t)(jj0 + t) * jstep;
        part[((int64_t)lane * groups + g) * nout + j] = make_double2((ar[t][0] + ar[t][1]) + (ar[t][2] + ar[t][3]),
                                                   (ai[t][0] + ai[t][1]) + (ai[t][2] + ai[t][3]));
      }
  }
  // the last block of the lane for these amplitudes sums its groups in order ...
  auto arrive_last = [&](unsigned* ticket, int of) {   // whether this block is the last of `of` at the ticket
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      s_last = atomicAdd(ticket, 1u) == (unsigned)of - 1u;
      if (s_last) *ticket = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last != 0;
  };
  if (!arrive_last(&tickets[1 + gridDim.x + blockIdx.x * lanes + lane], groups)) return;
  for (int64_t j = j0; j < nout; j += jstep) {
    double2* pj = part + (int64_t)lane * groups * nout + j;
    double sr = 0.0, si = 0.0;
    // eight loads in flight, added in group order
    for (int q0 = 0; q0 < groups; q0 += 8) {
      double2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = q0 + u < groups ? __ldcg(pj + (q0 + u) * nout) : make_double2(0.0, 0.0);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (q0 + u < groups) {
          sr += v[u].x;
          si += v[u].y;
        }
    }
    if (lanes > 1) {
      *pj = make_double2(sr, si);
    } else {
      double* o = p.out + 2 * (p.out_index * nout + j);
      o[0] += sr;
      o[1] += si;
    }
  }
  // ... and the last lane's adds the lanes in order, those of one batch onto one value
  if (lanes > 1) {
    if (!arrive_last(&tickets[1 + blockIdx.x], lanes)) return;
    for (int64_t j = j0; j < nout; j += jstep) {
      double* o = nullptr;
      double ar0 = 0.0, ai0 = 0.0;
      for (int l0 = 0; l0 < lanes; l0 += 8) {
        double2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          v[u] = l0 + u < lanes ? __ldcg(part + (int64_t)(l0 + u) * groups * nout + j) : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (l0 + u >= lanes) break;
          const ChunkParam& pl = params[first + l0 + u];
          if (pl.valid_lo >= pl.valid_hi) continue;   // a lane without slices only fills the launch
          double* ol = pl.out + 2 * (pl.out_index * nout + j);
          if (ol != o) {
            if (o) {
              o[0] = ar0;
              o[1] = ai0;
            }
            o = ol;
            ar0 = o[0];
            ai0 = o[1];
          }
          ar0 += v[u].x;
          ai0 += v[u].y;
        }
      }
      if (o) {
        o[0] = ar0;
        o[1] = ai0;
      }
    }
  }
  // all blocks have read the counter: each did before its arrival above
  if (threadIdx.x == 0 && atomicAdd(&tickets[0], 1u) == gridDim.x - 1u) {
    tickets[0] = 0u;
    *counter = first + (unsigned)lanes;
  }
}

// Largest |re|, |im| over n complex values, raised into *out (which the caller
// zeroes first): the FP16 split's scale of an operand without a producer.
__global__ void k_amax(const float2* __restrict__ x, int64_t n, float* out) {
  float m = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = fmaxf(m, cabs_max(x[i]));
  amax_update(out, m);   // blockDim is a multiple of 32
}

// Frugal rejection sampling (main text, section III): sample s walks its
// draws t, draw t proposing batch member cand[s][t] with uniform u[s][t]; the
// first draw with u * M < 2^n |a|^2 is the sample.  Every draw is tested in
// parallel and the smallest accepted t per sample kept.  The products are
// rounded separately (no fused multiply-add), as the decision's definition
// states them.  first[0] becomes 0 when a candidate is outside [0, count) (it is
// skipped), first[1 + s] is sample s's draw; all are ~0 before.
__global__ void k_frugal(const double2* __restrict__ a, int64_t count, int n_qubits, double m_bound,
                         const int64_t* __restrict__ cand, const double* __restrict__ u, int64_t n_draws,
                         int64_t n_samples, unsigned long long* first) {
  const int64_t total = n_draws * n_samples;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = cand[i];
    if (c < 0 || c >= count) {
      atomicExch(first, 0ull);
      continue;
    }
    const double2 v = a[c];
    const double p = __dadd_rn(__dmul_rn(v.x, v.x), __dmul_rn(v.y, v.y));
    if (__dmul_rn(u[i], m_bound) < ldexp(p, n_qubits))
      atomicMin(first + 1 + i / n_draws, (unsigned long long)(i % n_draws));
  }
}

// sum_i |a_i|^2 in FP64, deterministic: every block adds its share (thread t of
// the grid takes elements t, t + threads, ..., four loads in flight) into
// part[1 + block]; the last block to arrive (a ticket, zero between launches)
// adds the blocks' sums in a fixed order into part[0].  Bound by latency up to
// about 10^5 amplitudes and by HBM above: 10^6 amplitudes (16 MB) took 494 us on
// one block.  XEB_BLOCKS partial sums at most.
constexpr int XEB_BLOCKS = 1024, XEB_THREADS = 256;
__device__ __forceinline__ double block_sum_256(double s, double* red) {
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double r = 0.0;
  for (int w = 0; w < XEB_THREADS / 32; ++w) r += red[w];
  __syncthreads();
  return r;
}
__global__ void __launch_bounds__(XEB_THREADS) k_xeb_sum(const double2* __restrict__ a, int64_t n, double* part,
                                                         unsigned* ticket) {
  __shared__ double red[XEB_THREADS / 32];
  __shared__ int s_last;
  double s = 0.0;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < n; i0 += 4 * step) {
    double2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = i0 + u * step < n ? a[i0 + u * step] : make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      s = fma(v[u].x, v[u].x, s);
      s = fma(v[u].y, v[u].y, s);
    }
  }
  s = block_sum_256(s, red);
  if (gridDim.x == 1) {
    if (threadIdx.x == 0) part[0] = s;
    return;
  }
  if (threadIdx.x == 0) {
    part[1 + blockIdx.x] = s;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double t = 0.0;
  for (int q = threadIdx.x; q < (int)gridDim.x; q += blockDim.x) t += __ldcg(part + 1 + q);
  t = block_sum_256(t, red);
  if (threadIdx.x == 0) {
    part[0] = t;
    *ticket = 0u;
  }
}

constexpr int PERM_MAX_T = 12;   // tile bits at most
struct PermArgs {
  int8_t src_pos[KMAXR];  // output bit p <- input bit src_pos[p]
  // tiled variant: tile bit q in input order at input position t_in[q], tile bit
  // q in output order at output position t_out[q]; an element's shared-memory
  // slot is the XOR of wcol[q] over its set bits in input order, of rcol[q] over
  // those in output order
  int32_t nt;             // tile bits
  int8_t t_in[PERM_MAX_T], t_out[PERM_MAX_T];
  int16_t wcol[PERM_MAX_T], rcol[PERM_MAX_T];
  int32_t nr;             // remaining bits (at most 32), input order
  int8_t r_in[KMAXR], r_out[KMAXR];
};

// Standalone permutation: one thread per output element (coalesced writes,
// gathered reads); used for small ranks.
__global__ void k_permute_gather(const float2* __restrict__ in, float2* __restrict__ out, int rank,
                                 const PermArgs pa, int64_t total) {
  const int64_t mask = ((int64_t)1 << rank) - 1;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = idx & mask;
    int64_t src = 0;
    for (int p = 0; p < rank; ++p)
      if ((o >> p) & 1) src |= (int64_t)1 << pa.src_pos[p];
    out[idx] = __ldg(in + (idx - o) + src);
  }
}

// Tiled permutation (SI Eq. (2) as a standalone pass): a tile holds every
// combination of nt = 10 or 12 tile bits: the input's lowest bits and the input
// bits that feed the output's lowest positions, so reads and writes both run
// along memory in runs of 2^5 or 2^6 elements, in 16-byte pairs where both
// arrays are aligned to 16 bytes.  Threads write the tile into shared memory in
// input order and read it back in output order; the remaining nr bits select the
// tile.  A persistent block loads its next tile into registers before it writes
// the current one out.  HBM-bound: what counts is bytes in flight (32 KB a block
// of 4096 elements, loads of the next tile among them) and the lengths of the
// runs; a random permutation of 2^27 elements takes 338 us, 6.4 TB/s (557 us,
// 3.9 TB/s, with 8 KB tiles, 8-byte accesses and no load in flight across the
// write-back).
template <int NT>
__global__ void __launch_bounds__(256) k_permute_tiled(const float2* __restrict__ in, float2* __restrict__ out,
                                                       int rank, const __grid_constant__ PermArgs pa,
                                                       int64_t n_tiles, int vec) {
  constexpr int JB = NT - 9, NJ = 1 << JB;   // a thread has NJ pairs: bits 1-8 its index, 0 the pair, 9.. j
  __shared__ float2 tile[1 << NT];
  const int lane = threadIdx.x & 31;
  int64_t ioff = 0, ooff = 0;
  int ws = 0, rs = 0;
#pragma unroll
  for (int q = 1; q <= 8; ++q)
    if ((threadIdx.x >> (q - 1)) & 1) {
      ioff += (int64_t)1 << pa.t_in[q];
      ooff += (int64_t)1 << pa.t_out[q];
      ws ^= pa.wcol[q];
      rs ^= pa.rcol[q];
    }
  auto joff = [&](int j, const int8_t* pos) {
    int64_t v = 0;
#pragma unroll
    for (int q = 0; q < JB; ++q)
      if ((j >> q) & 1) v += (int64_t)1 << pos[9 + q];
    return v;
  };
  auto jcol = [&](int j, const int16_t* col) {
    int v = 0;
#pragma unroll
    for (int q = 0; q < JB; ++q)
      if ((j >> q) & 1) v ^= col[9 + q];
    return v;
  };
  // a tile's base in both arrays: one bit per lane, OR over the warp
  const int64_t rin = lane < pa.nr ? (int64_t)1 << pa.r_in[lane] : 0, rout = lane < pa.nr ? (int64_t)1 << pa.r_out[lane] : 0;
  auto base = [&](int64_t t, int64_t bit) {
    const uint64_t v = ((t >> lane) & 1) && lane < pa.nr ? (uint64_t)bit : 0;
    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)v), hi = __reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32));
    return ((t >> pa.nr) << rank) + (int64_t)(((uint64_t)hi << 32) | lo);
  };
  float4 v[NJ];
  auto load = [&](int64_t t) {
    const float2* p = in + base(t, rin) + ioff;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float2* q = p + joff(j, pa.t_in);
      if (vec) {
        v[j] = __ldcs(reinterpret_cast<const float4*>(q));
      } else {
        const float2 x = __ldcs(q), y = __ldcs(q + 1);
        v[j] = make_float4(x.x, x.y, y.x, y.y);
      }
    }
  };
  int64_t t = blockIdx.x;
  if (t < n_tiles) load(t);
  for (; t < n_tiles; t += gridDim.x) {
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int s0 = ws ^ jcol(j, pa.wcol);
      tile[s0] = make_float2(v[j].x, v[j].y);
      tile[s0 ^ pa.wcol[0]] = make_float2(v[j].z, v[j].w);
    }
    __syncthreads();
    if (t + gridDim.x < n_tiles) load(t + gridDim.x);
    float2* p = out + base(t, rout) + ooff;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int s0 = rs ^ jcol(j, pa.rcol);
      const float2 x = tile[s0], y = tile[s0 ^ pa.rcol[0]];
      float2* q = p + joff(j, pa.t_out);
      if (vec) {
        __stcs(reinterpret_cast<float4*>(q), make_float4(x.x, x.y, y.x, y.y));
      } else {
        __stcs(q, x);
        __stcs(q + 1, y);
      }
    }
    __syncthreads();
  }
}

}  // namespace tnx
