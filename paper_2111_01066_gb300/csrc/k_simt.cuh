// Complex GEMM on the CUDA cores (complex64, FP32 FMA): the plain FP32 path and
// the small steps of the tensor-core modes.
// Operands are gathered straight from their tensors' storage order, so the
// index permutation of SI Eq. (2) is folded into the loads (the paper's fused
// permutation-multiplication, SI figure S7a): each tile covers the lowest
// memory positions of its operand, so the gathers read contiguous runs.
#pragma once
#include "kernels_common.cuh"

namespace tnx {

// ------------------------------------------------------------------ packed FP32 pairs
// Two independent FP32 FMAs in one instruction (fma.rn.f32x2); each half rounds
// as fmaf does.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// ---- cluster helpers (split-K over the CTAs of a cluster)
__device__ __forceinline__ void simt_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t simt_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ float2 ld_peer_f2(const void* local, uint32_t rank) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
  uint32_t p;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(a), "r"(rank));
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(p));
  return v;
}

constexpr int SIMT_THREADS = 256;
constexpr int SIMT_MAX_SPLIT = 8;   // CTAs of one split-K cluster (the portable cluster size)

// A tiling: TM x TN outputs per CTA, TK of k per stage, RM x RN outputs per
// thread, KG groups of threads that each take 1/KG of a stage's k (their sums
// are added at the end), MINB CTAs per SM that the registers are kept to, two
// stages, filled one chunk ahead by asynchronous copies or (REGS) through registers.  Copies need no registers, which the small tilings'
// short loops want; they move 4 bytes at a time (the two planes of A), twice the L1
// requests of the register path's 16-byte loads, which is faster where a loop is
// long (2^17 x 256 x 256: 1198 us against 1310 with 128x64).  A is staged as two planes
// (re, im) whose consecutive rows make the packed pairs.
template <int TM_, int TN_, int TK_, int RM_, int RN_, int KG_, int MINB_, bool REGS_>
struct SimtCfg {
  static constexpr int TM = TM_, TN = TN_, TK = TK_, RM = RM_, RN = RN_, KG = KG_, MINB = MINB_;
  static constexpr bool REGS = REGS_;
  static constexpr int NTX = TM / RM, NTY = TN / RN;
  static_assert(NTX * NTY * KG == SIMT_THREADS, "one thread per RM x RN outputs and k group");
  static constexpr int RG = 4;                         // consecutive rows of a thread
  static_assert(RM % RG == 0, "whole runs of rows");
  static constexpr int AS = TM + 4;                    // plane row stride: k-fastest stores stay conflict-free
  static constexpr bool SPLIT = KG > 1;                // partial tiles: k groups, and CTAs of a split-K cluster
  struct Stage {
    float ar[TK][AS];
    float ai[TK][AS];
    float2 b[TK][TN + 1];
  };
};
template <class Cfg>
struct SimtSmem {
  union alignas(16) {
    typename Cfg::Stage st[2];
    // partial tiles of the k groups (column-major); the first one then takes their sum
    float2 part[Cfg::SPLIT ? Cfg::KG : 1][Cfg::SPLIT ? Cfg::TN : 1][Cfg::SPLIT ? Cfg::TM + 2 : 1];
  };
  int64_t offCm[Cfg::TM];
  int64_t offCn[Cfg::TN];
  // step of A's and B's k offset from chunk c to c + 1, by the number of
  // trailing one bits of c
  int64_t kdA[KMAXR];
  int64_t kdB[KMAXR];
};

using SimtBig = SimtCfg<128, 64, 8, 8, 4, 1, 2, true>;
using Simt64 = SimtCfg<64, 64, 8, 4, 4, 1, 3, true>;
using Simt128x16 = SimtCfg<128, 16, 16, 4, 2, 1, 3, false>;
using Simt256x4 = SimtCfg<256, 4, 8, 4, 1, 1, 4, false>;
using Simt32 = SimtCfg<32, 32, 32, 4, 4, 4, 2, false>;

// One thread's pairs of tile elements (2p, 2p + 1) of an operand: the elements
// of a tile are numbered by the tile bits in ascending memory position, so
// consecutive threads read consecutive addresses.
template <int NP>
struct PairMap {
  int64_t off[NP];   // memory offset of the pair's first element
  int32_t at[NP];    // its (k, row or column) packed as k << 16 | r; -1: no pair
  int64_t step;      // memory offset of the second from the first
  int32_t dat;       // the second's packed position less the first's; 0: no second
};
template <int NP>
__device__ __forceinline__ void pair_map(PairMap<NP>& m, int tbits, const int8_t* tpos, const int8_t* tsel) {
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    m.off[j] = 0;
    m.at[j] = 2 * ((int)threadIdx.x + j * SIMT_THREADS) < (1 << tbits) ? 0 : -1;
  }
  m.step = 0;
  m.dat = 0;
  if (tbits > 0) {
    m.step = (int64_t)1 << tpos[0];
    m.dat = (tsel[0] & 64) ? (1 << (16 + (tsel[0] & 63))) : (1 << tsel[0]);
  }
#pragma unroll 4
  for (int t = 1; t < tbits; ++t) {
    const int s = tsel[t];
    const int w = (s & 64) ? (1 << (16 + (s & 63))) : (1 << s);
    const int64_t o = (int64_t)1 << tpos[t];
#pragma unroll
    for (int j = 0; j < NP; ++j)
      if ((((int)threadIdx.x + j * SIMT_THREADS) >> (t - 1)) & 1) {
        m.off[j] += o;
        if (m.at[j] >= 0) m.at[j] += w;
      }
  }
}
// Asynchronous copies global -> shared of 4 and 8 bytes (no registers between)
__device__ __forceinline__ void cp_async_f1(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_f2(float2* dst, const float2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_groups() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Loads that stay where they are written: left to the compiler, the next chunk's
// loads moved down to their use, behind the products they should run under.
__device__ __forceinline__ float4 ldv4(const float2* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ldv2(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
template <int NP>
__device__ __forceinline__ void pair_load(float4 (&v)[NP], const PairMap<NP>& m, const float2* base, bool vec) {
#pragma unroll
  for (int j = 0; j < NP; ++j)
    if (m.at[j] >= 0) {
      const float2* p = base + m.off[j];
      if (vec) {
        v[j] = ldv4(p);
      } else {
        const float2 x = ldv2(p);
        const float2 y = m.dat ? ldv2(p + m.step) : make_float2(0.f, 0.f);
        v[j] = make_float4(x.x, x.y, y.x, y.y);
      }
    }
}

// One (m tile bx, n tile by) of a GEMM for instances bz, bz + gz, ... ; with
// split > 1 CTA `rank` of every `split` consecutive ones takes 1/split of the k
// chunks and the partial tiles are added over the cluster's shared memory in
// rank order (deterministic).  Every thread of the block calls it; g is in
// shared memory.  Rows and columns past the operand's extent hold whatever the
// stage buffers held: they only reach outputs that are not stored.
// Large GEMMs are bound by the FP32 pipe's issue slots: a product of two packed
// FMAs takes half the slots of four scalar ones, and 8 x 4 outputs per thread
// leave 24 register moves and 8 shared loads per 64 of them; 4096 x 1024 x 4096
// runs at 57 TFLOP/s (35 with scalar FMAs and 4 x 4 outputs), 2^17 x 256 x 256 at 57
// (34), of about 70.  Small ones are bound by latency: k offsets advance by one
// table entry per chunk (decoding all k bits per chunk took longer than the
// chunk's products), and one chunk with its set-up takes about 3 us in a chain of
// launches (12 before).
template <class Cfg>
__device__ __forceinline__ void simt_tile(const GemmArgs& g, int bx, int by, int bz, int gz, int split, int rank,
                                          SimtSmem<Cfg>& sm) {
  constexpr int TM = Cfg::TM, TN = Cfg::TN, TK = Cfg::TK, RM = Cfg::RM, RN = Cfg::RN;
  constexpr int NTX = Cfg::NTX, RG = Cfg::RG, RP = RM / 2;
  constexpr int AP = (TM * TK / 2 + SIMT_THREADS - 1) / SIMT_THREADS;
  constexpr int BP = (TN * TK / 2 + SIMT_THREADS - 1) / SIMT_THREADS;
  const int tid = threadIdx.x;
  // a warp covers 8 x 4 threads of the tile: it then reads 8 distinct 16-byte pieces
  // of A's planes and 4 of B per k, against 16 and 2 in rows of 16 (3-6% on large
  // GEMMs)
  const int kg = tid / (NTX * Cfg::NTY), w = (tid / 32) % (NTX * Cfg::NTY / 32);
  const int tx = (w % (NTX / 8)) * 8 + tid % 8, ty = (w / (NTX / 8)) * 4 + (tid % 32) / 8;
  const int TMv = 1 << g.tm, TKv = 1 << g.tk, TNv = 1 << g.tn;
  const int n_hi = g.nk - g.tk;
  const int kc_per = (1 << n_hi) / split, kc0 = rank * kc_per;

  // offsets of the tile's rows and columns in C, and the k chunk steps
  for (int r = tid; r < TM; r += SIMT_THREADS) sm.offCm[r] = r < TMv ? deposit_lo<8>((uint32_t)r, g.c_mpos, g.tm) : 0;
  if (tid < TN) sm.offCn[tid] = tid < TNv ? deposit_lo<6>((uint32_t)tid, g.c_npos, g.tn) : 0;
  {
    const int t = SIMT_THREADS - 1 - tid;   // other threads than the ones above where the tile is small
    if (t < n_hi) {
      int64_t a = (int64_t)1 << g.a_kpos[g.tk + t], b = (int64_t)1 << g.b_kpos[g.tk + t];
      for (int j = 0; j < t; ++j) {
        a -= (int64_t)1 << g.a_kpos[g.tk + j];
        b -= (int64_t)1 << g.b_kpos[g.tk + j];
      }
      sm.kdA[t] = a;
      sm.kdB[t] = b;
    }
  }
  PairMap<AP> ma;
  PairMap<BP> mb;
  pair_map(ma, g.a_tbits, g.a_tpos, g.a_tsel);
  pair_map(mb, g.b_tbits, g.b_tpos, g.b_tsel);
  const int64_t abase = warp_deposit((uint32_t)bx, g.a_mpos, g.tm, g.nm) + warp_deposit((uint32_t)kc0, g.a_kpos, g.tk, g.nk);
  const int64_t bbase = warp_deposit((uint32_t)by, g.b_npos, g.tn, g.nn) + warp_deposit((uint32_t)kc0, g.b_kpos, g.tk, g.nk);
  const int64_t cbase = warp_deposit((uint32_t)bx, g.c_mpos, g.tm, g.nm) + warp_deposit((uint32_t)by, g.c_npos, g.tn, g.nn);
  const float2 *A0, *B0;
  float2* C0;
  auto inst_bases = [&](int inst) {
    A0 = g.A + warp_inst_offset(inst, g.a_istride, g.a_bpos, g.nb) + abase;
    B0 = g.B + warp_inst_offset(inst, g.b_istride, g.b_bpos, g.nb) + bbase;
    C0 = g.C + warp_inst_offset(inst, g.c_istride, g.c_bpos, g.nb) + cbase;
  };
  inst_bases(bz);
  __syncthreads();
  pdl_wait();

  float am = 0.f;   // largest component written (for the FP16 split's scaling)
  // every CTA of a cluster goes through the same number of rounds (the cluster
  // barriers), also one without an instance left
  const int rounds = split > 1 ? (g.n_inst + gz - 1) / gz : 0x7fffffff;
  for (int it = 0, inst = bz; it < rounds; ++it, inst += gz) {
    if (bz >= gz || inst >= g.n_inst) {
      if (split == 1) break;
      simt_cluster_sync();
      simt_cluster_sync();
      continue;
    }
    if (it > 0) inst_bases(inst);
    const float2* A = A0;
    const float2* B = B0;
    float2* C = C0;
    f32x2 re[RP][RN], im[RP][RN];
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j) re[i][j] = im[i][j] = 0ull;
    auto issue = [&](typename Cfg::Stage& st) {
      auto put_a = [&](int at, const float2* p) {
        cp_async_f1(&st.ar[at >> 16][at & 0xffff], &p->x);
        cp_async_f1(&st.ai[at >> 16][at & 0xffff], &p->y);
      };
#pragma unroll
      for (int j = 0; j < AP; ++j)
        if (ma.at[j] >= 0) {
          put_a(ma.at[j], A + ma.off[j]);
          if (ma.dat) put_a(ma.at[j] + ma.dat, A + ma.off[j] + ma.step);
        }
#pragma unroll
      for (int j = 0; j < BP; ++j)
        if (mb.at[j] >= 0) {
          const int at = mb.at[j], a2 = at + mb.dat;
          cp_async_f2(&st.b[at >> 16][at & 0xffff], B + mb.off[j]);
          if (mb.dat) cp_async_f2(&st.b[a2 >> 16][a2 & 0xffff], B + mb.off[j] + mb.step);
        }
    };
    auto step = [&](const typename Cfg::Stage& st, int kk) {
      f32x2 ar[RP], ai[RP];
#pragma unroll
      for (int gq = 0; gq < RM / RG; ++gq) {
        const int r0 = (gq * NTX + tx) * RG;
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(&st.ar[kk][r0]);
        const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(&st.ai[kk][r0]);
        ar[2 * gq] = x.x;
        ar[2 * gq + 1] = x.y;
        ai[2 * gq] = y.x;
        ai[2 * gq + 1] = y.y;
      }
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        const float2 v = st.b[kk][ty + j * Cfg::NTY];
        const f32x2 br = pack2(v.x, v.x), bi = pack2(v.y, v.y), nb = pack2(-v.y, -v.y);
#pragma unroll
        for (int i = 0; i < RP; ++i) {
          re[i][j] = fma2(ar[i], br, re[i][j]);
          im[i][j] = fma2(ar[i], bi, im[i][j]);
        }
#pragma unroll
        for (int i = 0; i < RP; ++i) {
          re[i][j] = fma2(ai[i], nb, re[i][j]);
          im[i][j] = fma2(ai[i], br, im[i][j]);
        }
      }
    };
    if constexpr (Cfg::REGS) {
      static_assert(!Cfg::REGS || Cfg::KG == 1, "one k group");
      float4 la[AP], lb[BP];
      const bool va = g.a_tbits > 0 && g.a_tpos[0] == 0 && (reinterpret_cast<uintptr_t>(g.A) & 15) == 0;
      const bool vb = g.b_tbits > 0 && g.b_tpos[0] == 0 && (reinterpret_cast<uintptr_t>(g.B) & 15) == 0;
      auto load = [&]() {
        pair_load(la, ma, A, va);
        pair_load(lb, mb, B, vb);
      };
      auto put = [&](typename Cfg::Stage& st) {
        auto put_a = [&](int at, float x, float y) {
          st.ar[at >> 16][at & 0xffff] = x;
          st.ai[at >> 16][at & 0xffff] = y;
        };
#pragma unroll
        for (int j = 0; j < AP; ++j)
          if (ma.at[j] >= 0) {
            put_a(ma.at[j], la[j].x, la[j].y);
            if (ma.dat) put_a(ma.at[j] + ma.dat, la[j].z, la[j].w);
          }
#pragma unroll
        for (int j = 0; j < BP; ++j)
          if (mb.at[j] >= 0) {
            const int at = mb.at[j], a2 = at + mb.dat;
            st.b[at >> 16][at & 0xffff] = make_float2(lb[j].x, lb[j].y);
            if (mb.dat) st.b[a2 >> 16][a2 & 0xffff] = make_float2(lb[j].z, lb[j].w);
          }
      };
      load();
      put(sm.st[0]);
      __syncthreads();
      for (int c = 0; c < kc_per; ++c) {
        const bool more = c + 1 < kc_per;
        if (more) {
          const int t = __ffs(~(kc0 + c)) - 1;
          A += sm.kdA[t];
          B += sm.kdB[t];
          load();
        }
        const typename Cfg::Stage& st = sm.st[c & 1];
        if (TKv == TK) {
#pragma unroll 8
          for (int kk = 0; kk < TK; ++kk) step(st, kk);
        } else {
          for (int kk = 0; kk < TKv; ++kk) step(st, kk);
        }
        if (more) put(sm.st[(c + 1) & 1]);
        __syncthreads();
      }
    } else {
      // one chunk in flight ahead of the one being multiplied; a chunk's stage was last
      // read before the barrier that lets its copies be issued
      auto next = [&](int c) {   // chunk c's copies, as one group (empty past the end)
        if (c < kc_per) {
          if (c > 0) {
            const int t = __ffs(~(kc0 + c - 1)) - 1;   // trailing ones of the chunk before
            A += sm.kdA[t];
            B += sm.kdB[t];
          }
          issue(sm.st[c & 1]);
        }
        cp_async_commit_group();
      };
      next(0);
      for (int c = 0; c < kc_per; ++c) {
        cp_async_wait_groups<0>();
        __syncthreads();
        next(c + 1);
        const typename Cfg::Stage& st = sm.st[c & 1];
        if (TKv == TK) {
#pragma unroll 8
          for (int kk = 0; kk < TK / Cfg::KG; ++kk) step(st, kk * Cfg::KG + kg);
        } else {
          for (int kk = kg; kk < TKv; kk += Cfg::KG) step(st, kk);
        }
      }
    }
    __syncthreads();   // the stages are free for the partial tiles or the next instance
    if constexpr (!Cfg::SPLIT) {
      const bool vc = g.tm > 0 && g.c_mpos[0] == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        const int r = ((2 * i / RG) * NTX + tx) * RG + (2 * i) % RG;
        if (r < TMv) {
#pragma unroll
          for (int j = 0; j < RN; ++j) {
            const int cidx = ty + j * Cfg::NTY;
            if (cidx < TNv) {
              const float2 x = unpack2(re[i][j]), y = unpack2(im[i][j]);
              float2* p = C + sm.offCm[r] + sm.offCn[cidx];
              am = fmaxf(am, cabs_max(make_float2(x.x, y.x)));
              if (r + 1 < TMv) {
                am = fmaxf(am, cabs_max(make_float2(x.y, y.y)));
                if (vc && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
                  *reinterpret_cast<float4*>(p) = make_float4(x.x, y.x, x.y, y.y);
                } else {
                  *p = make_float2(x.x, y.x);
                  C[sm.offCm[r + 1] + sm.offCn[cidx]] = make_float2(x.y, y.y);
                }
              } else {
                *p = make_float2(x.x, y.x);
              }
            }
          }
        }
      }
    } else {
      // the k groups' partial tiles to shared memory, added in group order; with a split, each CTA then adds its
      // share of the tile's elements over the cluster, in rank order
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        const int r = ((2 * i / RG) * NTX + tx) * RG + (2 * i) % RG;
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          const float2 x = unpack2(re[i][j]), y = unpack2(im[i][j]);
          *reinterpret_cast<float4*>(&sm.part[kg][ty + j * Cfg::NTY][r]) = make_float4(x.x, y.x, x.y, y.y);
        }
      }
      __syncthreads();
      const int total = 1 << (g.tm + g.tn);
      for (int e = tid; e < total; e += SIMT_THREADS) {
        const int r = e & (TMv - 1), c = e >> g.tm;
        float2 acc = sm.part[0][c][r];
#pragma unroll
        for (int q = 1; q < Cfg::KG; ++q) {
          acc.x += sm.part[q][c][r].x;
          acc.y += sm.part[q][c][r].y;
        }
        if (split == 1) {
          C[sm.offCm[r] + sm.offCn[c]] = acc;
          am = fmaxf(am, cabs_max(acc));
        } else {
          sm.part[0][c][r] = acc;   // read by this thread alone so far
        }
      }
      if (split == 1) {
        __syncthreads();   // the next instance's stages overwrite the partial tiles
        continue;
      }
      simt_cluster_sync();
      const uint32_t me = simt_cluster_rank(), base = me - (uint32_t)rank;
      for (int e = rank * SIMT_THREADS + tid; e < total; e += split * SIMT_THREADS) {
        const int r = e & (TMv - 1), c = e >> g.tm;
        float2 v[SIMT_MAX_SPLIT];
#pragma unroll
        for (int q = 0; q < SIMT_MAX_SPLIT; ++q)
          if (q < split) v[q] = ld_peer_f2(&sm.part[0][c][r], base + q);
        float2 acc = v[0];
#pragma unroll
        for (int q = 1; q < SIMT_MAX_SPLIT; ++q)
          if (q < split) {
            acc.x += v[q].x;
            acc.y += v[q].y;
          }
        C[sm.offCm[r] + sm.offCn[c]] = acc;
        am = fmaxf(am, cabs_max(acc));
      }
      simt_cluster_sync();   // the peers have read this CTA's partial tile
    }
  }
  // every thread reaches here; with several lanes a block has one instance (bz; past
  // the last one in a block that only fills a cluster)
  if (g.amax_c && bz < gz) amax_update(g.amax_c + (int64_t)(bz >> (g.nb - g.ls_lanes)) * g.amax_lane, am);
}

__device__ __forceinline__ void copy_args(GemmArgs& dst, const GemmArgs* src) {
  constexpr int words = (int)(sizeof(GemmArgs) / 4);
  const uint32_t* s = reinterpret_cast<const uint32_t*>(src);
  uint32_t* d = reinterpret_cast<uint32_t*>(&dst);
  for (int w = threadIdx.x; w < words; w += blockDim.x) d[w] = s[w];
}

// One GEMM: grid (m tiles x split, n tiles, min(instances, 65535)); split > 1:
// clusters of `split` CTAs along x.
template <class Cfg>
__global__ void __launch_bounds__(SIMT_THREADS, Cfg::MINB) k_cgemm_simt(const __grid_constant__ GemmArgs g, int split) {
  __shared__ GemmArgs sg;
  __shared__ SimtSmem<Cfg> sm;
  copy_args(sg, &g);
  __syncthreads();
  simt_tile<Cfg>(sg, blockIdx.x / split, blockIdx.y, blockIdx.z, gridDim.z, split, blockIdx.x % split, sm);
}

// Several independent GEMMs in one launch (a group of small steps that
// neither read nor write what another of the group writes), on clusters of
// SIMT_MAX_SPLIT CTAs where one of them splits its k: block b runs block b - start[i] of GEMM i, where
// start[i] <= b < start[i + 1] (start[n] is the grid size; every start is a
// multiple of the cluster size, so a cluster has one GEMM), decoded as (split
// rank fastest, m tile, n tile, instance), with that GEMM's tiling[i] (0:
// 64x64, 1: 128x16, 2: 256x4, 3: 32x32; all use 256 threads) and split[i].
__global__ void __launch_bounds__(SIMT_THREADS, 2)
k_cgemm_simt_multi(const GemmArgs* __restrict__ gs, const int32_t* __restrict__ start,
                   const int8_t* __restrict__ tiling, const int8_t* __restrict__ splits, int32_t n) {
  __shared__ GemmArgs sg;
  __shared__ int s_i;
  __shared__ union {   // one tiling per block: their tiles share the space
    SimtSmem<Simt64> t0;
    SimtSmem<Simt128x16> t1;
    SimtSmem<Simt256x4> t2;
    SimtSmem<Simt32> t3;
  } sm;
  const int b = blockIdx.x;
  if (threadIdx.x < 32) {   // the last start at or before b
    int i = -1;
    for (int t = threadIdx.x; t < n; t += 32)
      if (start[t] <= b) i = t;
    i = __reduce_max_sync(0xffffffffu, i);
    if (threadIdx.x == 0) s_i = i;
  }
  __syncthreads();
  const int i = s_i;
  copy_args(sg, gs + i);
  __syncthreads();
  const int split = splits[i];
  const int gx = 1 << (sg.nm - sg.tm), gy = 1 << (sg.nn - sg.tn);
  const int gz = sg.n_inst < 65535 ? sg.n_inst : 65535;
  const int lb = b - start[i], rank = lb % split, lt = lb / split;
  const int bx = lt % gx, by = (lt / gx) % gy, bz = lt / (gx * gy);
  // blocks past the GEMM's last tile (bz >= gz) fill its last cluster: they run
  // no instance, only the barriers
  switch (tiling[i]) {   // block-uniform
    case 0:
      simt_tile<Simt64>(sg, bx, by, bz, gz, 1, 0, sm.t0);
      break;
    case 1:
      simt_tile<Simt128x16>(sg, bx, by, bz, gz, 1, 0, sm.t1);
      break;
    case 2:
      simt_tile<Simt256x4>(sg, bx, by, bz, gz, 1, 0, sm.t2);
      break;
    default:
      simt_tile<Simt32>(sg, bx, by, bz, gz, split, rank, sm.t3);
      break;
  }
}

}  // namespace tnx
