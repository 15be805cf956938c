// Device executor: the slice loop of a plan on one GPU, the XEB reduction, and
// the standalone kernel entry points of the C ABI.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <array>
#include <atomic>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <unordered_map>
#include <vector>

#include "k_misc.cuh"
#include "k_simt.cuh"
#include "k_tc.cuh"
#include "kernels_common.cuh"
#include "tn_internal.h"

namespace tnx {

#define CK(x)                                                                          \
  do {                                                                                 \
    cudaError_t e_ = (x);                                                              \
    if (e_ != cudaSuccess) fail(TN_ERR_CUDA, std::string(#x) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// ------------------------------------------------------------------ kernel table
enum KernelId {
  K_SIMT_64x64 = 0,   // TM 64, TN 64, TK 8
  K_SIMT_128x16 = 1,  // TM 128, TN 16, TK 16
  K_SIMT_256x4 = 2,   // TM 256, TN 4, TK 8
  K_TC_TF32 = 3,      // tcgen05 kind::tf32, tile 128 x (<=128 complex), k chunk 16
  K_TC_BF16X3 = 4,    // tcgen05 kind::f16 bf16 hi/lo split
  K_TC_TF32_3M = 5,   // the same with 3M products (three accumulators per tile)
  K_TC_BF16X3_3M = 6,
  K_TC_FP16X3 = 7,    // tcgen05 kind::f16 fp16 hi/lo split, operands scaled by powers of two
  K_TC_FP16X3_3M = 8,
  K_SIMT_128x64 = 9,  // TM 128, TN 64, TK 8
  K_SIMT_32x32 = 10,  // TM 32, TN 32, TK 32; split-K over a cluster's CTAs
  K_COUNT
};
struct KernelCfg {
  int tm, tn, tk;  // log2 tile extents
};
static const KernelCfg kCfg[K_COUNT] = {{6, 6, 3}, {7, 4, 4}, {8, 2, 3}, {7, 7, 4}, {7, 7, 4}, {7, 7, 4}, {7, 7, 4}, {7, 7, 4}, {7, 7, 4}, {7, 6, 3}, {5, 5, 5}};

static int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
  }
  return n;
}

static bool is_simt(int kid) { return kid >= 0 && kid < K_COUNT && !(kid >= K_TC_TF32 && kid <= K_TC_FP16X3_3M); }

// CUDA-core tiling of a step, from times on a GB300 (us a launch, log2 m, k, n):
//  * few outputs (at most two 32x32 tiles per SM): 32x32, whose k groups and
//    split-K clusters keep the SMs busy -- (7, 10, 6): 8.5 against 149 with 64x64;
//    (10, 6, 8): 7.8 against 11.5; with more tiles the larger ones win, (12, 4, 9): 32
//    against 11 with 128x64;
//  * n <= 4: 256x4, n <= 16: 128x16 -- (20, 3, 1): 45 with 256x4, 96 with 128x16;
//    (16, 5, 4): 15 with 128x16, 30 with 64x64;
//  * n = 32 with k >= 64: 32x32 -- (15, 8, 5): 70 against 108 with 64x64;
//  * otherwise 128x64 where its tiles fill the SMs -- (12, 10, 12): 2424 against
//    2705 with 64x64 -- and 64x64 where they do not.
static int pick_simt(const StepDesc& d, int64_t n_inst) {
  auto tiles = [&](int tm, int tn) {
    return ((int64_t)1 << (std::max(d.nm, tm) - tm)) * ((int64_t)1 << (std::max(d.nn, tn) - tn)) * n_inst;
  };
  const int64_t sms = sm_count();
  if (tiles(5, 5) <= 2 * sms || (d.nm < 5 && d.nn >= 5)) return K_SIMT_32x32;
  if (d.nn <= 2) return K_SIMT_256x4;
  if (d.nn <= 4) return K_SIMT_128x16;
  if (d.nn == 5 && d.nk >= 6) return K_SIMT_32x32;
  if (d.nn >= 6 && d.nm >= 7 && tiles(7, 6) >= 128) return K_SIMT_128x64;
  return K_SIMT_64x64;
}

// CTAs of a cluster that share a tile's k loop (1: no split): as many as leave
// each at least two k chunks and the grid within two CTAs per SM.  A cluster
// costs 2-4 us, a 32-k chunk of a lone CTA 1-1.5 (back to back (8, 8, 6) takes 11.5 us
// unsplit, 5.6 over 4 CTAs with 2 chunks each, 5.8 over 8; (7, 10, 6) 40, 12.7 and 8.5).
static int simt_split(const GemmArgs& g, int kid) {
  if (kid != K_SIMT_32x32) return 1;
  // of one lane: the same sums however many chunks run side by side
  const int64_t tiles = ((int64_t)1 << (g.nm - g.tm)) * ((int64_t)1 << (g.nn - g.tn)) * (g.n_inst >> g.ls_lanes);
  const int n_kc = 1 << (g.nk - g.tk);
  int sp = 1;
  while (sp < SIMT_MAX_SPLIT && sp * 4 <= n_kc && tiles * sp * 2 <= 2 * (int64_t)sm_count()) sp *= 2;
  return sp;
}

// Tile decode tables: the tile's bits in ascending memory position.
static GemmArgs make_args(const StepDesc& d, int kid, const float2* A, const float2* B, float2* C,
                          int32_t n_inst, int64_t a_istride = 0, int64_t b_istride = 0,
                          int64_t c_istride = 0, int tn_log = -1) {
  GemmArgs g;
  std::memset(&g, 0, sizeof(g));
  g.A = A;
  g.B = B;
  g.C = C;
  g.a_istride = a_istride;
  g.b_istride = b_istride;
  g.c_istride = c_istride;
  g.n_inst = n_inst;
  g.nb = d.nb;
  g.nm = d.nm;
  g.nk = d.nk;
  g.nn = d.nn;
  std::memcpy(g.a_bpos, d.a_bpos, KMAXB);
  std::memcpy(g.b_bpos, d.b_bpos, KMAXB);
  std::memcpy(g.c_bpos, d.c_bpos, KMAXB);
  const KernelCfg& k = kCfg[kid];
  g.tm = std::min(k.tm, d.nm);
  g.tk = std::min(k.tk, d.nk);
  g.tn = std::min(tn_log >= 0 ? tn_log : k.tn, d.nn);
  std::memcpy(g.a_mpos, d.a_mpos, KMAXR);
  std::memcpy(g.a_kpos, d.a_kpos, KMAXR);
  std::memcpy(g.b_kpos, d.b_kpos, KMAXR);
  std::memcpy(g.b_npos, d.b_npos, KMAXR);
  std::memcpy(g.c_mpos, d.c_mpos, KMAXR);
  std::memcpy(g.c_npos, d.c_npos, KMAXR);
  std::vector<std::pair<int, int>> ta, tb;  // (position, sel)
  for (int i = 0; i < g.tm; ++i) ta.push_back({d.a_mpos[i], i});
  for (int j = 0; j < g.tk; ++j) ta.push_back({d.a_kpos[j], j | 64});
  for (int j = 0; j < g.tk; ++j) tb.push_back({d.b_kpos[j], j | 64});
  for (int i = 0; i < g.tn; ++i) tb.push_back({d.b_npos[i], i});
  std::sort(ta.begin(), ta.end());
  std::sort(tb.begin(), tb.end());
  if ((int)ta.size() > KTB || (int)tb.size() > KTB) fail(TN_ERR_UNSUPPORTED, "tile too large");
  g.a_tbits = (int)ta.size();
  g.b_tbits = (int)tb.size();
  for (size_t t = 0; t < ta.size(); ++t) {
    g.a_tpos[t] = (int8_t)ta[t].first;
    g.a_tsel[t] = (int8_t)ta[t].second;
  }
  for (size_t t = 0; t < tb.size(); ++t) {
    g.b_tpos[t] = (int8_t)tb[t].first;
    g.b_tsel[t] = (int8_t)tb[t].second;
  }
  return g;
}

// Launch with programmatic dependent launch (the kernel calls pdl_wait), on
// clusters of `cluster` CTAs along x where that is above 1.
template <class... KArgs, class... Args>
static void klaunch(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t s, int cluster,
                    Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  CK(cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...));
}

template <class Cfg>
static void launch_simt_cfg(const GemmArgs& g, dim3 grid, int split, cudaStream_t s) {
  klaunch(k_cgemm_simt<Cfg>, grid, SIMT_THREADS, 0, s, split, g, split);
}
static void launch_simt(const GemmArgs& g, int kid, cudaStream_t s) {
  if (g.n_inst <= 0) return;
  const int split = simt_split(g, kid);
  const int64_t gx = ((int64_t)1 << (g.nm - g.tm)) * split;
  const int64_t gy = (int64_t)1 << (g.nn - g.tn);
  if (gx > 0x7fffffff || gy > 65535) fail(TN_ERR_UNSUPPORTED, "GEMM grid too large");
  dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)std::min<int32_t>(g.n_inst, 65535));
  switch (kid) {
    case K_SIMT_64x64:
      launch_simt_cfg<Simt64>(g, grid, 1, s);
      break;
    case K_SIMT_128x16:
      launch_simt_cfg<Simt128x16>(g, grid, 1, s);
      break;
    case K_SIMT_256x4:
      launch_simt_cfg<Simt256x4>(g, grid, 1, s);
      break;
    case K_SIMT_128x64:
      launch_simt_cfg<SimtBig>(g, grid, 1, s);
      break;
    case K_SIMT_32x32:
      launch_simt_cfg<Simt32>(g, grid, split, s);
      break;
    default:
      fail(TN_ERR_UNSUPPORTED, "kernel variant not built");
  }
}

// One step ready to launch: GEMM arguments, tensor-core tiling, B' workspace
// size, and the tensor map of A when its tiles are fetched by TMA.
struct StepLaunch {
  int kid = 0;
  GemmArgs g;
  TcArgs tc;
  CUtensorMap tma;   // 64-byte aligned by its own declaration
  int64_t ws_bytes = 0;
  int64_t split_off = 0;   // split-K partials inside the workspace
  int64_t c_total = 0;     // elements of C (all instances)
  int smem = 0;
  // B' images built ahead of the chunks (the step's B depends on no slice):
  // built by the prologue of class bimg_cls (0 once per plan, 2 once per
  // batch) into bimg_own; null: built with every launch in the workspace
  uint8_t* bimg_own = nullptr;
  int bimg_cls = -1;
  int64_t bimg_lane = 0;   // bytes from one lane's images to the next one's
};

static bool is_tc(int kid) { return kid >= K_TC_TF32 && kid <= K_TC_FP16X3_3M; }
static bool tc_is_3m(int kid) { return kid == K_TC_TF32_3M || kid == K_TC_BF16X3_3M || kid == K_TC_FP16X3_3M; }
struct TcGeom {   // the plane geometry of TcPl<MODE, CM> for a kernel id
  int planes, rows_per_col, a_slot, min_tn_c, esz;
};
static TcGeom tc_geom(int kid) {
  switch (kid) {
    case K_TC_TF32:
      return {TcPl<TC_TF32, 4>::PLANES, TcPl<TC_TF32, 4>::ROWS_PER_COL, TcPl<TC_TF32, 4>::A_SLOT,
              TcPl<TC_TF32, 4>::MIN_TN_C, 4};
    case K_TC_BF16X3:
      return {TcPl<TC_BF16X3, 4>::PLANES, TcPl<TC_BF16X3, 4>::ROWS_PER_COL, TcPl<TC_BF16X3, 4>::A_SLOT,
              TcPl<TC_BF16X3, 4>::MIN_TN_C, 2};
    case K_TC_TF32_3M:
      return {TcPl<TC_TF32, 3>::PLANES, TcPl<TC_TF32, 3>::ROWS_PER_COL, TcPl<TC_TF32, 3>::A_SLOT,
              TcPl<TC_TF32, 3>::MIN_TN_C, 4};
    case K_TC_BF16X3_3M:
      return {TcPl<TC_BF16X3, 3>::PLANES, TcPl<TC_BF16X3, 3>::ROWS_PER_COL, TcPl<TC_BF16X3, 3>::A_SLOT,
              TcPl<TC_BF16X3, 3>::MIN_TN_C, 2};
    case K_TC_FP16X3:
      return {TcPl<TC_FP16X3, 4>::PLANES, TcPl<TC_FP16X3, 4>::ROWS_PER_COL, TcPl<TC_FP16X3, 4>::A_SLOT,
              TcPl<TC_FP16X3, 4>::MIN_TN_C, 2};
    default:
      return {TcPl<TC_FP16X3, 3>::PLANES, TcPl<TC_FP16X3, 3>::ROWS_PER_COL, TcPl<TC_FP16X3, 3>::A_SLOT,
              TcPl<TC_FP16X3, 3>::MIN_TN_C, 2};
  }
}

static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  }
  return fn;
}

// A can be fetched by TMA when it is stored as [its k bits in order, then at
// least 128 rows of m bits in order]: a row-major matrix per dimension-2 index.
// a_bits = log2 of A's elements over one linear instance; n_lin = linear instances.
static void setup_tma(StepLaunch& L, int a_bits, int64_t n_lin) {
  const GemmArgs& g = L.g;
  TcArgs& t = L.tc;
  t.a_tma = 0;
  // tiles of 2^tm rows (tm <= 7; a 128-row MMA tile whose rows past 2^tm the epilogue drops)
  if (g.nk < 4 || g.tm < 3 || g.tm > 7 || (reinterpret_cast<uintptr_t>(g.A) & 15)) return;
  for (int j = 0; j < g.nk; ++j)
    if (g.a_kpos[j] != j) return;
  int nmw = 0;
  while (nmw < g.nm && g.a_mpos[nmw] == g.nk + nmw) ++nmw;
  if (nmw < g.tm) return;
  const int hi_shift = g.nk + nmw;
  if (a_bits < hi_shift) return;
  const uint64_t dim2 = ((uint64_t)1 << (a_bits - hi_shift)) * (uint64_t)n_lin;
  if (dim2 > ((uint64_t)1 << 31)) return;
  auto enc = tensor_map_encoder();
  if (!enc) return;
  cuuint64_t dims[3] = {(cuuint64_t)2 << g.nk, (cuuint64_t)1 << nmw, (cuuint64_t)dim2};
  cuuint64_t strides[2] = {((cuuint64_t)1 << g.nk) * 8, ((cuuint64_t)1 << hi_shift) * 8};
  cuuint32_t box[3] = {(cuuint32_t)TC_KP, (cuuint32_t)1u << g.tm, 1};
  cuuint32_t es[3] = {1, 1, 1};
  const CUresult r = enc(&L.tma, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float2*>(g.A), dims, strides, box,
                         es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return;
  t.a_tma = 1;
  t.a_box_bytes = (TC_KP * 4) << g.tm;
  t.nmw = nmw;
  t.hi_shift = hi_shift;
  t.c2_inst_mul = n_lin > 1 ? ((int64_t)1 << (a_bits - hi_shift)) : 0;
}

// How a tile's k chunks are divided: n_split work units (partial tiles through
// memory) of n_seg accumulators each (in TMEM, acc_cols * tn_c columns apiece).
// `need`: n_split * n_seg must reach it, so that no chain of 32-bit accumulation
// gets longer.  Of what fits, the least modeled time: the work units in waves, each
// its chunks and a write-back, plus the partial tiles' way through memory and the
// reduction's launch.  A chunk of 128 columns takes about 0.6 us, one of few
// columns the 0.37 in which an SM's share of HBM brings its 16 KB of A; the
// write-back 3.  (With partial tiles alone 2048 x 256 x 1024, whose 64 pairs already
// fill 76, wrote four of them: 36 us.)
struct TcSplit {
  int n_split, n_seg;
  double us;
};
static TcSplit tc_split(int64_t n_tiles, int64_t slots, int n_kc, int tn_c, int acc_cols, int64_t c_total,
                        int64_t cap_bytes, int need) {
  const double chunk_us = std::max(0.37, 0.15 + 0.45 * tn_c / 128.0), tile_us = 1.0 + 2.0 * tn_c / 128.0;
  TcSplit best = {0, 1, 0.0};
  for (int sp = 1; sp <= 32 && (sp == 1 || n_kc / sp >= 4); sp *= 2) {
    if (sp > 1 && ((n_tiles >= slots && sp > need) || (int64_t)sp * c_total * 8 > cap_bytes)) break;
    int sg = std::max(1, need / sp);
    if (sg > 1 && (acc_cols != 2 || sg * acc_cols * tn_c > TC_TMEM_COLS)) continue;   // 4M only, where they fit
    const double waves = (double)((n_tiles * sp + slots - 1) / slots);
    double us = waves * (n_kc / sp * chunk_us + tile_us);
    if (sp > 1) us += 3.0 + (2.0 * sp + 1.0) * (double)c_total * 8.0 / 5.5e6;
    if (best.n_split == 0 || us < best.us) best = {sp, sg, us};
  }
  return best;
}
// The parts that a tile's k is divided into at least: when the tiles of the
// default width (128 columns) cannot fill the SMs, as many as keep eight per SM at
// most and 4 chunks each.
static int tc_min_parts(int kid, int nm, int nk, int nn, int64_t n_inst, int64_t c_total, int64_t cap_bytes) {
  const KernelCfg& k = kCfg[kid];
  const int tm = std::min(k.tm, nm), tk = std::min(k.tk, nk), tn = std::min(k.tn, nn);
  const int64_t tiles = n_inst * ((int64_t)1 << (nm - tm)) * ((int64_t)1 << (nn - tn));
  const int n_kc = 1 << (nk - tk);
  int sp = 1;
  if (tiles < sm_count() && n_kc >= 8)
    while (sp < 32 && tiles * sp * 2 <= 8 * (int64_t)sm_count() && n_kc / (sp * 2) >= 4) sp *= 2;
  return (int64_t)sp * c_total * 8 <= cap_bytes ? sp : 1;
}

// epi_mode: -1 chooses the write-back by the coalesced run lengths, 0 forces
// direct per-column stores, 1 the staged order (where the tile allows it)
// b_slots: B' ring slots (<= 0: 4 for slots up to 16 KB, else 3; at most
// TC_MAX_B; the rest of the shared-memory budget goes to A slots)
// pair_mode: SM pairs (cta_group::2, two m tiles per work unit, half of B' per
// CTA) where the step allows them -- 4M products and at least two full 128-row
// m tiles: 1 uses them there, 0 never, -1 unless the step has at most 64 k and 256
// columns: there B' is a small part of the traffic and a pair's launch and
// barriers cost more than they save (16384 x 16 x 256: 13.0 us on single SMs, 14.4 on
// pairs; 2^18 x 64 x 128: 75 and 78; with 1024 columns or 128 k pairs win, 65536 x 64
// x 1024: 113 and 107, 2^21 x 128 x 128: 704 and 669)
static bool pair_ok(int kid, int nm, int tm) { return !tc_is_3m(kid) && tm == 7 && nm - tm >= 1; }
static bool pair_pays(int ls_kc, int ls_nt) { return ls_kc > 2 || ls_nt > 1; }

// Default tile width (log2 complex columns): 128, or 64 or 32 where the tiles are
// few and that takes less modeled time: narrower tiles spread over more SMs and
// leave room for more accumulators of a divided k (2048 x 256 x 1024: 36 us with 128
// columns and four partial results, 25 with 64 columns and four accumulators).
static int tc_tile(int kid, int nm, int nk, int nn, int64_t n_inst, int64_t c_total, int64_t cap_bytes, bool pairs) {
  const KernelCfg& k = kCfg[kid];
  const int tm = std::min(k.tm, nm), tk = std::min(k.tk, nk), widest = std::min(k.tn, nn);
  const int need = tc_min_parts(kid, nm, nk, nn, n_inst, c_total, cap_bytes);
  if (need == 1) return widest;
  int best = widest;
  double best_us = 0.0;
  for (int tn = widest; tn >= std::min(5, widest); --tn) {
    const int pair = pairs && pair_ok(kid, nm, tm) && pair_pays(nk - tk, nn - tn) ? 1 : 0;
    const int64_t units = n_inst * ((int64_t)1 << (nm - tm - pair)) * ((int64_t)1 << (nn - tn));
    const double us = tc_split(units, sm_count() / (1 + pair), 1 << (nk - tk), std::max(tc_geom(kid).min_tn_c, 1 << tn),
                               tc_is_3m(kid) ? 3 : 2, c_total, cap_bytes, need).us;
    if (tn == widest || us < best_us) {
      best = tn;
      best_us = us;
    }
  }
  return best;
}

static StepLaunch make_launch(const GemmArgs& g, int kid, int a_bits, int64_t n_lin, int64_t c_total = 0,
                              bool allow_split = false, int epi_mode = -1,
                              int64_t split_cap_bytes = (int64_t)256 << 20, int b_slots = 0, int pair_mode = -1) {
  StepLaunch L;
  L.kid = kid;
  L.g = g;
  std::memset(&L.tc, 0, sizeof(L.tc));
  std::memset(&L.tma, 0, sizeof(L.tma));
  if (!is_tc(kid)) return L;
  TcArgs& t = L.tc;
  t.g = g;
  t.tnb = g.tn;
  const TcGeom geo = tc_geom(kid);
  t.tn_c = std::max(geo.min_tn_c, 1 << g.tn);
  t.pair = (pair_mode != 0 && pair_ok(kid, g.nm, g.tm) && (pair_mode > 0 || pair_pays(g.nk - g.tk, g.nn - g.tn))) ? 1 : 0;
  t.n_mt = 1 << (g.nm - g.tm - t.pair);
  t.n_nt = 1 << (g.nn - g.tn);
  t.n_kc = 1 << (g.nk - g.tk);
  t.n_tiles = (int64_t)g.n_inst * t.n_mt * t.n_nt;
  const int b_plane = tc_plane_bytes(geo.rows_per_col * t.tn_c, geo.esz);
  const int npl = geo.planes;
  L.ws_bytes = (int64_t)g.n_inst * t.n_nt * t.n_kc * npl * b_plane;
  // few output tiles and a long k loop: the k chunks of a tile go to n_split work
  // units, whose partial tiles are added by k_split_reduce, and to n_seg
  // accumulators in each (tc_split)
  const int64_t unit_sms = 1 + t.pair, slots = std::max<int64_t>(1, sm_count() / unit_sms);
  t.n_split = 1;
  t.n_seg = 1;
  if (allow_split && c_total > 0) {
    const TcSplit c = tc_split(t.n_tiles, slots, t.n_kc, t.tn_c, tc_is_3m(kid) ? 3 : 2, c_total, split_cap_bytes,
                               tc_min_parts(kid, g.nm, g.nk, g.nn, g.n_inst, c_total, split_cap_bytes));
    t.n_split = c.n_split;
    t.n_seg = c.n_seg;
    if (t.n_split > 1) {
      t.c_part_stride = c_total;
      L.split_off = (L.ws_bytes + 255) / 256 * 256;
      L.ws_bytes = L.split_off + (int64_t)t.n_split * c_total * 8;
      L.c_total = c_total;
    }
  }
  t.ls_seg_len = __builtin_ctz((unsigned)(t.n_kc / (t.n_split * t.n_seg)));
  t.n_tiles *= t.n_split;
  t.ls_split = __builtin_ctz((unsigned)t.n_split);
  t.ls_nt = g.nn - g.tn;
  t.ls_mt = g.nm - g.tm - t.pair;
  // the n tiles of one A block back to back on the same SM (pair), so that the
  // block's later reads hit L2: when the A blocks in flight on all SMs fit half
  // of L2 (else they evict each other between reads, while in index order the
  // n tiles of a block run at the same time on neighbouring SMs) and there are
  // at least 8 blocks per SM (pair), so that the coarser units leave no long tail
  const int64_t units = t.pair ? sm_count() / 2 : sm_count();
  const double a_block_bytes = 8.0 * TC_M * (1 + t.pair) * std::ldexp(1.0, g.nk);
  t.nt_inner = (t.n_nt > 1 && (t.n_tiles >> t.ls_nt) >= 8 * units &&
                units * a_block_bytes <= 64.0 * (1 << 20))
                   ? 1
                   : 0;
  t.ls_kc = g.nk - g.tk;
  setup_tma(L, a_bits, n_lin);
  // epilogue write order: a warp's rows are m bits 0-4, a chunk's 16 columns n bits 0-3
  t.epi_ok = 0;
  if (g.tm >= 5 && g.tn >= 4) {
    std::vector<std::pair<int, int>> bits;
    for (int i = 0; i < 5; ++i) bits.push_back({g.c_mpos[i], i});
    for (int j = 0; j < 4; ++j) bits.push_back({g.c_npos[j], j | 64});
    std::sort(bits.begin(), bits.end());
    for (int t2 = 0; t2 < 9; ++t2) {
      t.epi_pos[t2] = (int8_t)bits[t2].first;
      t.epi_sel[t2] = (int8_t)bits[t2].second;
    }
    // direct per-column stores write runs of 2^run_d elements (C's lowest
    // positions hold row bits 0, 1, ... in order); the staged order writes runs
    // of 2^run_s (C's lowest positions among the block's 9 bits).  Runs of 4+
    // elements fill whole 32-byte sectors, so stage only below that
    int run_d = 0, run_s = 0;
    while (run_d < 5 && g.c_mpos[run_d] == run_d) ++run_d;
    while (run_s < 5 && bits[run_s].first == run_s) ++run_s;
    t.epi_ok = epi_mode >= 0 ? epi_mode : (run_s > run_d && run_d < 2 ? 1 : 0);
  }
  // rings: B' slots first (3, or 4 when small), the rest of the shared memory
  // to A slots: up to the 227 KB opt-in, less the barriers, the alignment slack
  // and the write-back staging (only when the staged order is used); a pair's
  // CTA holds half of every B' plane
  const int b_slot = npl * (t.pair ? b_plane / 2 : b_plane);
  const int epi_bytes = t.epi_ok ? TC_EPI_BYTES : 0;
  const int budget = TC_MAX_SMEM - 4096 - 1024 - epi_bytes;
  t.nbs = b_slots > 0 ? std::min(b_slots, TC_MAX_B) : (b_slot <= 16384 ? 4 : 3);
  t.na = std::min(TC_MAX_A, (budget - t.nbs * b_slot) / geo.a_slot);
  // A by tensor-map loads converted in place: the two converter groups take
  // alternate k chunks, and chunk q sits in A slot q % na.  An even na keeps
  // every slot with one group, which then waits for the slot's phases strictly
  // in order; with an odd na a group could wait for phase u of a slot before the
  // other group's phase u - 1 had landed, and a parity wait cannot tell the two
  // apart (it would pass on the stale phase and convert the wrong data).
  const bool converters = t.a_tma && (tc_is_3m(kid) || kid != K_TC_TF32);
  if (converters) t.na &= ~1;
  if (t.na < 2) fail(TN_ERR_UNSUPPORTED, "tensor-core rings do not fit shared memory");
  t.nbs = std::min(t.nbs, t.na);   // B' slots are released through the A slots' barriers
  // arrivals on an A slot: the TMA itself (TF32 4M), one converter group (TMA otherwise), all loaders
  t.fa_count = (t.a_tma && kid == K_TC_TF32) ? 1 : (t.a_tma ? TC_LOAD_THREADS / 2 : TC_LOAD_THREADS);
  // as many accumulator sets as fit the 512 TMEM columns (at most 8): narrow
  // tiles let the MMAs run several tiles ahead of the epilogue
  t.n_acc = std::max(1, std::min(TC_MAX_ACC, TC_TMEM_COLS / ((tc_is_3m(kid) ? 3 : 2) * t.tn_c * t.n_seg)));
  L.smem = std::max(t.na * geo.a_slot + t.nbs * b_slot + 4096 + epi_bytes + 1024, TC_MIN_SMEM);
  return L;
}

// SM pairs of a tensor-core kernel that can be resident at once (one pair per
// two SMs when the device fits them all), queried once per kernel and device
template <int MODE, bool PAIR>
static int pair_clusters() {
  static std::atomic<int> cached[64];
  int dev = 0;
  CK(cudaGetDevice(&dev));
  const int slot = dev < 64 ? dev : 63;
  int n = cached[slot].load(std::memory_order_acquire);
  if (n > 0) return n;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sm_count() / 2));
  cfg.blockDim = dim3(TC_THREADS);
  cfg.dynamicSmemBytes = TC_MAX_SMEM;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int q = 0;
  CK(cudaFuncSetAttribute(k_cgemm_tc<MODE, 4, PAIR, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_MAX_SMEM));
  if (cudaOccupancyMaxActiveClusters(&q, k_cgemm_tc<MODE, 4, PAIR, false>, &cfg) != cudaSuccess || q <= 0) {
    cudaGetLastError();
    q = sm_count() / 2;
  }
  n = std::min(q, sm_count() / 2);
  cached[slot].store(n, std::memory_order_release);
  return n;
}

// The B' images of a tensor-core step into t.bimg.
template <int MODE, int CM>
static void launch_prep(const TcArgs& t, cudaStream_t s) {
  const int ls_cols = __builtin_ctz((unsigned)t.tn_c);
  const int64_t threads = ((int64_t)t.g.n_inst * t.n_nt * t.n_kc) << (ls_cols + TcPrep<MODE, CM>::LS_KT);
  const int64_t grid = (threads + PREP_THREADS - 1) / PREP_THREADS;
  if (grid > 0x7fffffff) fail(TN_ERR_UNSUPPORTED, "B' image grid too large");
  klaunch(k_tc_prep_b<MODE, CM>, dim3((unsigned)grid), PREP_THREADS, 0, s, 1, t, ls_cols);
}
static void launch_prep_kid(const TcArgs& t, int kid, cudaStream_t s) {
  switch (kid) {
    case K_TC_TF32:
      launch_prep<TC_TF32, 4>(t, s);
      break;
    case K_TC_BF16X3:
      launch_prep<TC_BF16X3, 4>(t, s);
      break;
    case K_TC_TF32_3M:
      launch_prep<TC_TF32, 3>(t, s);
      break;
    case K_TC_BF16X3_3M:
      launch_prep<TC_BF16X3, 3>(t, s);
      break;
    case K_TC_FP16X3:
      launch_prep<TC_FP16X3, 4>(t, s);
      break;
    default:
      launch_prep<TC_FP16X3, 3>(t, s);
      break;
  }
}

template <int MODE, int CM, bool PAIR, bool SEG>
static void launch_tc_kernel(const TcArgs& t, const StepLaunch& L, int grid, cudaStream_t s) {
  // the shared-memory opt-in is a per-device function attribute: one bit per
  // device (ids < 64) records that it was set there; two threads racing on the
  // same bit both set the same value, which is harmless
  static std::atomic<uint64_t> attr_set{0};
  int dev = 0;
  CK(cudaGetDevice(&dev));
  const uint64_t bit = dev < 64 ? (1ULL << dev) : 0;
  if (!bit || !(attr_set.load(std::memory_order_acquire) & bit)) {
    CK(cudaFuncSetAttribute(k_cgemm_tc<MODE, CM, PAIR, SEG>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_MAX_SMEM));
    attr_set.fetch_or(bit, std::memory_order_acq_rel);
  }
  if constexpr (PAIR) {
    // clusters of two CTAs, each pair persistent over the work units
    const int clusters = (int)std::min<int64_t>(t.n_tiles, pair_clusters<MODE, PAIR>());
    klaunch(k_cgemm_tc<MODE, CM, PAIR, SEG>, dim3(2 * clusters), TC_THREADS, L.smem, s, 2, t, L.tma);
  } else {
    klaunch(k_cgemm_tc<MODE, CM, PAIR, SEG>, dim3(grid), TC_THREADS, L.smem, s, 1, t, L.tma);
  }
}
template <int MODE, int CM, bool PAIR>
static void launch_tc(const TcArgs& t, const StepLaunch& L, int grid, cudaStream_t s) {
  if (!L.bimg_own) launch_prep<MODE, CM>(t, s);   // else built ahead by a prologue
  if constexpr (CM == 4)
    if (t.n_seg > 1) {
      launch_tc_kernel<MODE, CM, PAIR, true>(t, L, grid, s);
      return;
    }
  launch_tc_kernel<MODE, CM, PAIR, false>(t, L, grid, s);
}

// clear_amax: the step's recorded maximum starts at zero here (in a chunk or a
// prologue the leaf select has cleared it)
static void launch_step(StepLaunch& L, uint8_t* ws, int32_t* err, cudaStream_t s, bool clear_amax) {
  if (L.g.amax_c && clear_amax) CK(cudaMemsetAsync(L.g.amax_c, 0, sizeof(float), s));   // the result's maximum, recorded anew
  if (!is_tc(L.kid)) {
    launch_simt(L.g, L.kid, s);
    return;
  }
  TcArgs t = L.tc;
  t.bimg = L.bimg_own ? L.bimg_own : ws;
  t.err = err;
  if (t.n_split > 1) t.c_part = reinterpret_cast<float2*>(ws + L.split_off);
  if (t.n_tiles <= 0) return;
  const int grid = (int)std::min<int64_t>(t.n_tiles, sm_count());
  switch (L.kid) {
    case K_TC_TF32:
      if (t.pair)
        launch_tc<TC_TF32, 4, true>(t, L, grid, s);
      else
        launch_tc<TC_TF32, 4, false>(t, L, grid, s);
      break;
    case K_TC_BF16X3:
      if (t.pair)
        launch_tc<TC_BF16X3, 4, true>(t, L, grid, s);
      else
        launch_tc<TC_BF16X3, 4, false>(t, L, grid, s);
      break;
    case K_TC_TF32_3M:
      launch_tc<TC_TF32, 3, false>(t, L, grid, s);
      break;
    case K_TC_BF16X3_3M:
      launch_tc<TC_BF16X3, 3, false>(t, L, grid, s);
      break;
    case K_TC_FP16X3:
      if (t.pair)
        launch_tc<TC_FP16X3, 4, true>(t, L, grid, s);
      else
        launch_tc<TC_FP16X3, 4, false>(t, L, grid, s);
      break;
    default:
      launch_tc<TC_FP16X3, 3, false>(t, L, grid, s);
      break;
  }
  if (t.n_split > 1) {
    const int rb = (int)std::min<int64_t>((L.c_total + 255) / 256, (int64_t)sm_count() * 8);
    klaunch(k_split_reduce, dim3(rb), 256, 0, s, 1, (const float2*)t.c_part, (int)t.n_split, t.c_part_stride, t.g.C,
            L.c_total, t.g.amax_c);
  }
}

// ------------------------------------------------------------------ plan device state
// groups of small independent steps (StepDesc::group): per group, the steps
// [first, end) and the launches that run them -- one multi-step launch for
// all its CUDA-core steps (each block with its step's tiling), single
// launches for its tensor-core steps; rebuilt whenever the kernels are
// chosen again
struct GroupRun {
  int first = 0, end = 0;
  std::vector<int> singles;                  // steps launched alone
  struct Multi {
    int blocks = 0, n = 0;
    int cluster = 1;                         // SIMT_MAX_SPLIT where a step's k is split
    // offsets in DeviceState::group_buf: n GemmArgs, n + 1 block offsets (int32), n
    // CUDA-core tilings (simt_multi_tiling), n split-K factors
    size_t args_at = 0, start_at = 0, tiling_at = 0, split_at = 0;
  };
  std::vector<Multi> multi;
};

// The launches of a plan for 2^ls lanes: CUDA-core steps with the lanes as further
// instances, tensor-core steps once per lane (lane l > 0 in more[step][l - 1]), so that
// a chunk's result does not depend on what runs beside it.
struct LaunchSet {
  int ls = 0;
  std::vector<StepLaunch> launches;
  std::vector<std::vector<StepLaunch>> more;   // [step][lane - 1], tensor-core steps only (empty: one lane)
  std::vector<GroupRun> groups;
  std::vector<int> group_at;                   // per step: its group run's index, or -1
  // the launch sequences as CUDA graphs, each captured at its second use (the
  // first runs eagerly): [0] a chunk per lane, [1] with the prologue of new
  // batches; every kernel reads its chunk parameters from device memory
  cudaGraphExec_t graph[2] = {nullptr, nullptr};
  bool graph_failed[2] = {false, false};
  bool eager_done[2] = {false, false};
};
constexpr int MAX_LS_LANES = 4;
constexpr size_t PARAMS_AT = 64;

struct DeviceState {
  int device = -1;
  float2* arena = nullptr;
  float2* leaf_data = nullptr;
  LeafDesc* leaf_desc = nullptr;
  unsigned* counter = nullptr;    // one buffer: the chunk counter, then (at PARAMS_AT) the chunks' parameters
  ChunkParam* params = nullptr;
  size_t params_cap = 0;
  int32_t* err = nullptr;
  uint8_t* ws = nullptr;
  int64_t ws_bytes = 0;           // capacity of ws
  double2* root_part = nullptr;   // [groups][2^k] partial slice sums
  unsigned* root_tickets = nullptr;   // arrivals of the slice sum's blocks (zero between launches)
  int root_blocks = 1;
  float* amax = nullptr;          // FP16X3: largest component of every node (leaves, then steps), per lane
  int amax_nodes = 0;
  int root_groups = 1;
  LaunchSet set[MAX_LS_LANES + 1];
  std::vector<StepLaunch>& launches = set[0].launches;
  uint8_t* group_buf = nullptr;   // the arrays of every set's multi-step launches
  int ls_lanes = 0;               // lanes that the arena has room for (log2)
  // rough times that a call's lanes are chosen by (set_lane_times)
  double chain_us = 0.0;          // a chunk's launches that its lanes share
  double pro_chain_us = 0.0;      // the same of a batch's prologue
  double pro_us[2] = {0.0, 0.0};  // one lane's part of the prologue: per plan, per batch
  bool tc_chunk = false;          // a chunk or its batch's prologue has tensor-core steps
  int64_t lane_stride = 0;        // elements between the lanes' arenas (a power of two where there are several)
  std::vector<uint8_t*> own_imgs;              // B' images built ahead of the chunks (StepLaunch::bimg_own)
  cudaEvent_t done = nullptr;
  bool have_done = false;
  // prologues: steps whose result depends on no slice run once per plan
  // (dependence flags 0) or once per batch bitstring (flags 2); their results
  // that later steps read sit in the arena's persistent pool, each lane's in its own
  int pro0_lanes = 0;             // lanes whose per-plan steps have run
  bool pro2_valid[1 << MAX_LS_LANES] = {false};
  uint64_t pro2_bits[1 << MAX_LS_LANES] = {0};
  void forget_prologues() {
    pro0_lanes = 0;
    for (bool& v : pro2_valid) v = false;
  }
};

static int tc_kernel(int precision, int cmult) {
  if (precision == TN_PREC_TF32) return cmult == 3 ? K_TC_TF32_3M : K_TC_TF32;
  if (precision == TN_PREC_FP16X3) return cmult == 3 ? K_TC_FP16X3_3M : K_TC_FP16X3;
  return cmult == 3 ? K_TC_BF16X3_3M : K_TC_BF16X3;
}
// Tensor-core kernels (4M or 3M products) for the steps with enough work in the
// TF32 / BF16X3 / FP16X3 modes, from 2^25 multiply-adds over all instances; the
// rest (and the FP32 mode) on the CUDA cores, which always form 4M products in
// FP32.  A tensor-core step has a B' image launch, a pipeline to fill and an
// accumulator to drain, about 7 us at least back to back (BF16x3): at 2^20 the CUDA
// cores take 4.3 us against 7.4, at 2^22 4-5 against 7-9, at 2^24 8-9 against 7-10 (16
// columns: 8-12 against 7-10), at 2^25 13.1 against 12.5 (16 columns: 21 against 12).
static int pick_kernel(int precision, int cmult, const StepDesc& d, int64_t n_inst) {
  if (precision == TN_PREC_FP32) return pick_simt(d, n_inst);
  const double macs = std::ldexp((double)n_inst, d.nm + d.nk + d.nn);
  if (macs < 33554432.0 || d.nm < 4) return pick_simt(d, n_inst);
  return tc_kernel(precision, cmult);
}

// Launch arguments of plan step d for kernel kid in one lane's arena; FP16X3 plans also
// get the maxima of the step's operands (to scale them) and of its result (to record).
static GemmArgs step_args(const DeviceState& ds, const StepDesc& d, int kid, int tn_log = -1, int lane = 0) {
  float2* arena = ds.arena + lane * ds.lane_stride;
  GemmArgs g = make_args(d, kid, arena + d.a_off, arena + d.b_off, arena + d.c_off, 1 << d.nb, 0, 0, 0, tn_log);
  if (ds.amax) {
    float* amax = ds.amax + (int64_t)lane * ds.amax_nodes;
    g.amax_a = amax + d.a_node;
    g.amax_b = amax + d.b_node;
    g.amax_c = amax + d.c_node;
  }
  return g;
}
// The same with the lanes 0 .. 2^ls - 1 as further instances, from the arguments of lane 0.
static GemmArgs lanes_args(const DeviceState& ds, GemmArgs g, int ls) {
  for (int t = 0; t < ls; ++t)
    g.a_bpos[g.nb + t] = g.b_bpos[g.nb + t] = g.c_bpos[g.nb + t] =
        (int8_t)(__builtin_ctzll((uint64_t)ds.lane_stride) + t);
  g.nb += ls;
  g.n_inst <<= ls;
  g.ls_lanes = ls;
  g.amax_lane = ds.amax ? ds.amax_nodes : 0;
  return g;
}

// The tiling index of k_cgemm_simt_multi for a kernel id, -1 for a tiling it does not have.
static int simt_multi_tiling(int kid) {
  return kid == K_SIMT_32x32 ? 3 : (kid >= K_SIMT_64x64 && kid <= K_SIMT_256x4 ? kid : -1);
}

static void launch_simt_multi(const DeviceState& ds, const GroupRun::Multi& m, cudaStream_t s) {
  const uint8_t* buf = ds.group_buf;
  klaunch(k_cgemm_simt_multi, dim3((unsigned)m.blocks), SIMT_THREADS, 0, s, m.cluster,
          reinterpret_cast<const GemmArgs*>(buf + m.args_at), reinterpret_cast<const int32_t*>(buf + m.start_at),
          reinterpret_cast<const int8_t*>(buf + m.tiling_at), reinterpret_cast<const int8_t*>(buf + m.split_at), (int32_t)m.n);
}

// Dependence flags of a node (bit 0: on the slice id, bit 1: on the closed
// output bits): a step's own flags; a leaf's from the wires its select fixes
// and the slice bits it carries as batch bits.
static int node_flags(const Plan& p, int node) {
  const int nl = (int)p.leaves.size();
  if (node >= nl) return p.steps[node - nl].dep_flags;
  const LeafDesc& lf = p.leaves[node];
  int f = lf.bmask ? 1 : 0;
  for (int t = 0; t < lf.nfixed; ++t) f |= lf.fixed_kind[t] == 0 ? 1 : 2;
  return f;
}

// B' images of per-chunk tensor-core steps whose B depends on no slice: one
// buffer each per lane, built by the prologue of B's class (once per plan, or once
// per batch bitstring) instead of with every chunk, for the lane's own arena: they
// are as valid as the results of that prologue in that lane, whichever launch set
// runs it and reads them.  Where the buffers cannot be had the step keeps building its
// images per launch.
static void setup_hoisted(Plan& p, DeviceState& ds) {
  for (uint8_t* b : ds.own_imgs) cudaFree(b);
  ds.own_imgs.clear();
  for (size_t i = 0; i < p.steps.size(); ++i) {
    StepLaunch& L = ds.launches[i];
    L.bimg_own = nullptr;
    L.bimg_cls = -1;
    L.bimg_lane = 0;
    const StepDesc& d = p.steps[i];
    if (!is_tc(L.kid) || !(d.dep_flags & 1)) continue;
    const int bf = node_flags(p, d.b_node);
    if (bf & 1) continue;
    const int64_t img = ((L.tc.n_split > 1 ? L.split_off : L.ws_bytes) + 255) / 256 * 256;
    uint8_t* buf = nullptr;
    if (img <= 0 || cudaMalloc(&buf, (size_t)img << ds.ls_lanes) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    ds.own_imgs.push_back(buf);
    L.bimg_own = buf;
    L.bimg_cls = bf;
    L.bimg_lane = img;
  }
}

// Group runs from the plan's step groups and the kernels chosen so far.  The arrays of
// their multi-step launches are appended to `host`, the image of group_buf, and addressed
// by their offsets in it.
static void build_groups(const Plan& p, LaunchSet& ds, std::vector<uint8_t>& host) {
  ds.groups.clear();
  ds.group_at.assign(p.steps.size(), -1);
  for (size_t i = 0; i < p.steps.size();) {
    const int gid = p.steps[i].group;
    size_t j = i + 1;
    if (gid >= 0)
      while (j < p.steps.size() && p.steps[j].group == gid) ++j;
    if (gid < 0 || j - i < 2) {
      i = j;
      continue;
    }
    GroupRun gr;
    gr.first = (int)i;
    gr.end = (int)j;
    std::vector<int> simt;
    for (size_t t = i; t < j; ++t) {
      if (simt_multi_tiling(ds.launches[t].kid) < 0) gr.singles.push_back((int)t);
      else simt.push_back((int)t);
    }
    if (simt.size() == 1) gr.singles.push_back(simt[0]);
    if (simt.size() >= 2) {
      GroupRun::Multi m;
      m.n = (int)simt.size();
      m.args_at = (host.size() + 255) / 256 * 256;
      m.start_at = (m.args_at + sizeof(GemmArgs) * simt.size() + 15) / 16 * 16;
      m.tiling_at = m.start_at + sizeof(int32_t) * (simt.size() + 1);
      m.split_at = m.tiling_at + simt.size();
      host.resize(m.split_at + simt.size(), 0);
      for (int t : simt)
        if (simt_split(ds.launches[t].g, ds.launches[t].kid) > 1) m.cluster = SIMT_MAX_SPLIT;
      int32_t blocks = 0;
      for (size_t q = 0; q < simt.size(); ++q) {
        const GemmArgs& g = ds.launches[simt[q]].g;
        const int kid = ds.launches[simt[q]].kid, split = simt_split(g, kid);
        std::memcpy(host.data() + m.args_at + q * sizeof(GemmArgs), &g, sizeof(GemmArgs));
        host[m.tiling_at + q] = (uint8_t)simt_multi_tiling(kid);
        host[m.split_at + q] = (uint8_t)split;
        // whole clusters: the kernel's blocks past the last tile only keep its barriers
        int64_t nb = ((int64_t)1 << (g.nm - g.tm)) * ((int64_t)1 << (g.nn - g.tn)) * split *
                     std::min<int64_t>(g.n_inst, 65535);
        nb = (nb + m.cluster - 1) / m.cluster * m.cluster;
        if (blocks + nb > 0x7fffffff) fail(TN_ERR_UNSUPPORTED, "step group grid too large");
        std::memcpy(host.data() + m.start_at + q * sizeof(int32_t), &blocks, sizeof(int32_t));
        blocks += (int32_t)nb;
      }
      std::memcpy(host.data() + m.start_at + simt.size() * sizeof(int32_t), &blocks, sizeof(int32_t));
      m.blocks = blocks;
      gr.multi.push_back(m);
    }
    for (size_t t = i; t < j; ++t) ds.group_at[t] = (int)ds.groups.size();
    ds.groups.push_back(gr);
    i = j;
  }
}

// Step d's launch with one kernel choice (as the autotuner builds its candidates).
static StepLaunch build_choice(const DeviceState& ds, const StepDesc& d, int kid, int tn_log, int epi, int bslots,
                               int pair, int lane = 0) {
  return make_launch(step_args(ds, d, kid, tn_log, lane), kid, 64 - __builtin_clzll((uint64_t)d.a_elems) - 1, 1,
                     d.c_elems, true, epi, (int64_t)256 << 20, bslots, pair);
}

// The launch sets of every number of lanes, built from the kernels chosen for one lane:
// all of them at once, so that no later call allocates or waits, whatever its number
// of chunks.
static void build_sets(Plan& p, DeviceState& ds) {
  std::vector<uint8_t> host;
  for (int ls = 0; ls <= ds.ls_lanes; ++ls) {
    LaunchSet& st = ds.set[ls];
    if (ls > 0) {
      st.ls = ls;
      st.launches.clear();
      st.launches.reserve(p.steps.size());
      st.more.assign(p.steps.size(), {});
      for (size_t i = 0; i < p.steps.size(); ++i) {
        const StepDesc& d = p.steps[i];
        const StepLaunch& one = ds.launches[i];
        if (is_tc(one.kid)) {
          st.launches.push_back(one);
          for (int l = 1; l < (1 << ls); ++l) {
            StepLaunch L = build_choice(ds, d, one.kid, one.g.tn, one.tc.epi_ok, one.tc.nbs, one.tc.pair, l);
            if (one.bimg_own) L.bimg_own = one.bimg_own + l * one.bimg_lane;
            L.bimg_cls = one.bimg_cls;
            st.more[i].push_back(L);
          }
        } else {
          st.launches.push_back(make_launch(lanes_args(ds, one.g, ls), one.kid, 0, 1));
        }
      }
    }
    build_groups(p, st, host);
  }
  if (ds.group_buf) CK(cudaFree(ds.group_buf));
  ds.group_buf = nullptr;
  if (host.empty()) return;
  CK(cudaMalloc(&ds.group_buf, host.size()));
  CK(cudaMemcpy(ds.group_buf, host.data(), host.size(), cudaMemcpyHostToDevice));
}

// Launches for the steps of a class in plan order: CUDA-core ones, which all lanes
// share, into *shared, kernels of tensor-core steps, which run once per lane, into *alone.
template <class Pred>
static void class_launches(const Plan& p, Pred in_class, int* shared, int* alone) {
  const LaunchSet& st = p.dev->set[0];
  *shared = *alone = 0;
  auto one = [&](int i) {
    const StepLaunch& L = st.launches[i];
    if (is_tc(L.kid)) *alone += (L.tc.n_split > 1 ? 3 : 2) - (L.bimg_own ? 1 : 0);
    else ++*shared;
  };
  for (size_t i = 0; i < p.steps.size(); ++i) {
    if (!in_class(p.steps[i].dep_flags)) continue;
    const int gi = st.group_at.empty() ? -1 : st.group_at[i];
    if (gi < 0) {
      one((int)i);
      continue;
    }
    const GroupRun& gr = st.groups[gi];
    *shared += (int)gr.multi.size();
    for (int t : gr.singles) one(t);
    i = (size_t)gr.end - 1;
  }
}

// Rough times of the parts that the choice of lanes trades: a launch of a chain of
// small steps takes about 3 us, a prologue's multiply-adds about 8 flops at 30
// TFLOP/s on the CUDA cores, and a tensor-core step 8 us at least.
static void set_lane_times(const Plan& p, DeviceState& ds) {
  int shared, alone;
  class_launches(p, [](int f) { return (f & 1) != 0; }, &shared, &alone);
  ds.chain_us = 3.0 * (2 + shared);
  class_launches(p, [](int f) { return f == 2; }, &shared, &alone);
  ds.pro_chain_us = 3.0 * shared;
  ds.tc_chunk = false;
  ds.pro_us[0] = ds.pro_us[1] = 0.0;
  for (size_t i = 0; i < p.steps.size(); ++i) {
    const StepDesc& d = p.steps[i];
    const bool tc = is_tc(ds.launches[i].kid);
    if (d.dep_flags != 0) ds.tc_chunk = ds.tc_chunk || tc;
    if (d.dep_flags & 1) continue;
    const double us = std::ldexp(8.0, d.nm + d.nk + d.nn + d.nb) / 1e6 / (tc ? 500.0 : 30.0) + (tc ? 8.0 : 0.0);
    ds.pro_us[d.dep_flags == 0 ? 0 : 1] += us;
  }
}

// Lanes of a call (log2) for `chunks` chunks of each of `batches` batches: the more,
// the fewer chains of launches, but a batch's prologue runs in min(lanes, chunks)
// arenas.  Measured (us; all lanes, and what this takes): 30 + 6 qubits of which only the
// 6 are sliced, prologue of 2^24.8 multiply-adds, 16 chunks of 2^11: 16 lanes 329, 8
// lanes 231; 36 + 6 qubits, 2^26.7, 4 chunks: 4 lanes 254, 2 lanes 227, and four such
// batches 821 with 8 lanes, 899 with 2.
static int lanes_of_call(const DeviceState& ds, size_t batches, size_t chunks) {
  const size_t total = batches * chunks;
  int best = 0;
  double best_us = 0.0;
  for (int ls = 0; ls <= ds.ls_lanes && (ls == 0 || ((size_t)1 << (ls - 1)) < total); ++ls) {
    const size_t n = (size_t)1 << ls, runs = (total + n - 1) / n;
    const double us = (double)runs * ds.chain_us + (double)std::min(runs, batches) * ds.pro_chain_us +
                      (double)(batches * std::min(n, chunks)) * ds.pro_us[1] +
                      (double)std::max(0, (int)n - ds.pro0_lanes) * ds.pro_us[0];
    if (ls == 0 || us <= best_us) {
      best = ls;
      best_us = us;
    }
  }
  return best;
}

static int ceil_log2(int64_t v) { return v <= 1 ? 0 : 64 - __builtin_clzll((uint64_t)(v - 1)); }

// Lanes of a plan (log2): as many as keep their arenas in 64 MB -- in L2, and of
// plans whose chunks are so small that they are launches and latency rather than
// work -- and under the caller's bound, at most 16.
static int lanes_of(const Plan& p) {
  const int64_t cap = std::min<int64_t>((int64_t)64 << 20, p.opts.max_arena_bytes > 0 ? p.opts.max_arena_bytes : INT64_MAX);
  const int64_t arena = (int64_t)sizeof(float2) << ceil_log2(std::max<int64_t>(p.arena_elems, 32));
  const int64_t part = (int64_t)sizeof(double2) * std::min(1 << p.log2_batch, 64) << p.root.rank;
  int nb = 0;
  for (const StepDesc& d : p.steps) nb = std::max(nb, d.nb);
  int ls = 0;
  while (ls < MAX_LS_LANES && (arena << (ls + 1)) <= cap && (part << (ls + 1)) <= cap && nb + ls + 1 < KMAXB) ++ls;
  return ls;
}

static void build_device_state(Plan& p, DeviceState* ds) {
  const size_t ab = std::max<size_t>(256, (size_t)p.arena_elems * sizeof(float2));
  ds->ls_lanes = lanes_of(p);
  if (ds->ls_lanes > 0) {   // several arenas; where they cannot be had, one
    ds->lane_stride = (int64_t)1 << ceil_log2(std::max<int64_t>(p.arena_elems, 32));
    if (cudaMalloc(&ds->arena, ((size_t)ds->lane_stride * sizeof(float2)) << ds->ls_lanes) != cudaSuccess) {
      cudaGetLastError();
      ds->arena = nullptr;
      ds->ls_lanes = 0;
      ds->lane_stride = 0;
    }
  }
  if (!ds->arena && cudaMalloc(&ds->arena, ab) != cudaSuccess) {
    cudaGetLastError();
    fail(TN_ERR_OOM, "arena allocation of " + std::to_string(ab) + " bytes failed");
  }
  const size_t lb = std::max<size_t>(16, p.leaf_data.size() * sizeof(float2));
  CK(cudaMalloc(&ds->leaf_data, lb));
  CK(cudaMemcpy(ds->leaf_data, p.leaf_data.data(), p.leaf_data.size() * sizeof(float2),
                cudaMemcpyHostToDevice));
  CK(cudaMalloc(&ds->leaf_desc, std::max<size_t>(1, p.leaves.size()) * sizeof(LeafDesc)));
  CK(cudaMemcpy(ds->leaf_desc, p.leaves.data(), p.leaves.size() * sizeof(LeafDesc),
                cudaMemcpyHostToDevice));
  CK(cudaMalloc(&ds->err, sizeof(int32_t)));
  CK(cudaMemset(ds->err, 0, sizeof(int32_t)));
  CK(cudaEventCreateWithFlags(&ds->done, cudaEventDisableTiming));
  if (p.opts.precision == TN_PREC_FP16X3) {
    // leaves' maxima are constants of the plan; the steps' are recorded per chunk
    const size_t nn = std::max<size_t>(p.leaves.size() + p.steps.size(), 1);
    ds->amax_nodes = (int)nn;
    CK(cudaMalloc(&ds->amax, (sizeof(float) * nn) << ds->ls_lanes));
    CK(cudaMemset(ds->amax, 0, (sizeof(float) * nn) << ds->ls_lanes));
    if (!p.leaf_amax.empty())
      for (int l = 0; l < (1 << ds->ls_lanes); ++l)
        CK(cudaMemcpy(ds->amax + l * nn, p.leaf_amax.data(), sizeof(float) * p.leaf_amax.size(),
                      cudaMemcpyHostToDevice));
  }
  // bounds of every operand inside the arena, checked once on the host
  const int64_t ae = p.arena_elems;
  auto in_arena = [&](int64_t off, int64_t size, int insts) {
    return off >= 0 && off + size * (int64_t)insts <= ae;
  };
  for (const LeafDesc& l : p.leaves)
    if (!in_arena(l.dst_off, (int64_t)1 << l.rank, 1 << __builtin_popcount(l.bmask)))
      fail(TN_ERR_PLAN, "internal: leaf outside the arena");
  for (const StepDesc& d : p.steps) {
    // every bit position must address inside the operand's own extent
    auto span_ok = [](const int8_t* pos, int n, int64_t elems) {
      for (int i = 0; i < n; ++i)
        if (pos[i] < 0 || ((int64_t)1 << pos[i]) >= elems) return false;
      return true;
    };
    const bool ok = in_arena(d.a_off, d.a_elems, 1) && in_arena(d.b_off, d.b_elems, 1) &&
                    in_arena(d.c_off, d.c_elems, 1) && span_ok(d.a_mpos, d.nm, d.a_elems) &&
                    span_ok(d.a_kpos, d.nk, d.a_elems) && span_ok(d.b_kpos, d.nk, d.b_elems) &&
                    span_ok(d.b_npos, d.nn, d.b_elems) && span_ok(d.c_mpos, d.nm, d.c_elems) &&
                    span_ok(d.c_npos, d.nn, d.c_elems) && span_ok(d.a_bpos, d.nb, d.a_elems) &&
                    span_ok(d.b_bpos, d.nb, d.b_elems) && span_ok(d.c_bpos, d.nb, d.c_elems) &&
                    ((int64_t)1 << (d.nm + d.nk + d.nb)) == d.a_elems &&
                    ((int64_t)1 << (d.nk + d.nn + d.nb)) == d.b_elems &&
                    ((int64_t)1 << (d.nm + d.nn + d.nb)) == d.c_elems;
    if (!ok) fail(TN_ERR_PLAN, "internal: step operand outside its extent");
    const int kid = pick_kernel(p.opts.precision, p.opts.complex_mult, d, (int64_t)1 << d.nb);
    const int tn = is_tc(kid) ? tc_tile(kid, d.nm, d.nk, d.nn, (int64_t)1 << d.nb, d.c_elems, (int64_t)256 << 20,
                                        p.opts.sm_pairs != 0)
                              : -1;
    ds->launches.push_back(make_launch(step_args(*ds, d, kid, tn), kid, 64 - __builtin_clzll((uint64_t)d.a_elems) - 1, 1,
                                       d.c_elems, true, -1, (int64_t)256 << 20, 0, p.opts.sm_pairs ? -1 : 0));
  }
  int64_t ws = 16;
  for (const StepLaunch& L : ds->launches) ws = std::max(ws, L.ws_bytes);
  if (cudaMalloc(&ds->ws, (size_t)ws) != cudaSuccess) {
    cudaGetLastError();
    fail(TN_ERR_OOM, "workspace allocation of " + std::to_string(ws) + " bytes failed");
  }
  ds->ws_bytes = ws;
  ds->root_groups = std::min(1 << p.log2_batch, 64);
  CK(cudaMalloc(&ds->root_part, (sizeof(double2) * (size_t)ds->root_groups << p.root.rank) << ds->ls_lanes));
  ds->root_blocks = (int)std::min<int64_t>((((int64_t)1 << p.root.rank) + 255) / 256, 4096);
  const size_t tickets = 1 + (size_t)ds->root_blocks * (1 + ((size_t)1 << ds->ls_lanes));
  CK(cudaMalloc(&ds->root_tickets, sizeof(unsigned) * tickets));
  CK(cudaMemset(ds->root_tickets, 0, sizeof(unsigned) * tickets));
  if (!in_arena(p.root.off, (int64_t)1 << p.root.rank, 1 << __builtin_popcount(p.root.bmask)))
    fail(TN_ERR_PLAN, "internal: root outside the arena");
  setup_hoisted(p, *ds);
  build_sets(p, *ds);
  set_lane_times(p, *ds);
}

// The plan's device state, built by its first call; one that could not be built whole
// is taken down again, so that a later call starts anew.
static void ensure_device(Plan& p) {
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (p.dev) {
    if (p.dev->device != dev) fail(TN_ERR_ARG, "plan was first used on another device");
    return;
  }
  p.dev = new DeviceState;
  p.dev->device = dev;
  try {
    build_device_state(p, p.dev);
  } catch (...) {
    destroy_device_state(&p);
    throw;
  }
}

static void drop_graphs(DeviceState& ds) {
  for (LaunchSet& st : ds.set)
    for (int w = 0; w < 2; ++w) {
      if (st.graph[w]) cudaGraphExecDestroy(st.graph[w]);
      st.graph[w] = nullptr;
      st.graph_failed[w] = false;
      st.eager_done[w] = false;
    }
}

void destroy_device_state(Plan* p) {
  if (!p || !p->dev) return;
  DeviceState* ds = p->dev;
  int cur = 0;
  cudaGetDevice(&cur);
  cudaSetDevice(ds->device);
  if (ds->have_done) cudaEventSynchronize(ds->done);
  cudaFree(ds->arena);
  cudaFree(ds->leaf_data);
  cudaFree(ds->leaf_desc);
  cudaFree(ds->counter);
  cudaFree(ds->err);
  cudaFree(ds->ws);
  cudaFree(ds->root_part);
  cudaFree(ds->root_tickets);
  cudaFree(ds->amax);
  cudaFree(ds->group_buf);
  for (uint8_t* b : ds->own_imgs) cudaFree(b);
  drop_graphs(*ds);
  if (ds->done) cudaEventDestroy(ds->done);
  cudaSetDevice(cur);
  delete ds;
  p->dev = nullptr;
}

// A workspace of at least `bytes` (synchronises the device).  Where it cannot be had
// the old one is, or else the plan starts anew with its next call; fails either way.
static void grow_workspace(Plan& p, int64_t bytes, const char* who) {
  DeviceState& ds = *p.dev;
  if (bytes <= ds.ws_bytes) return;
  drop_graphs(ds);   // captured with the old workspace's address
  CK(cudaFree(ds.ws));
  ds.ws = nullptr;
  if (cudaMalloc(&ds.ws, (size_t)bytes) == cudaSuccess) {
    ds.ws_bytes = bytes;
    return;
  }
  cudaGetLastError();
  ds.ws = nullptr;
  if (cudaMalloc(&ds.ws, (size_t)ds.ws_bytes) != cudaSuccess) {
    cudaGetLastError();
    destroy_device_state(&p);
  }
  fail(TN_ERR_OOM, std::string(who) + ": workspace allocation of " + std::to_string(bytes) + " bytes failed");
}

// The steps whose dependence flags satisfy `in_class`, in plan order; a group
// of independent small steps runs as its multi-step launches, then the rest of
// the group alone.
template <class Pred>
static void launch_class(Plan& p, cudaStream_t s, LaunchSet& st, Pred in_class) {
  DeviceState& ds = *p.dev;
  auto one = [&](int i) {
    launch_step(st.launches[i], ds.ws, ds.err, s, false);
    if (!st.more.empty())
      for (StepLaunch& lane : st.more[i]) launch_step(lane, ds.ws, ds.err, s, false);
  };
  for (size_t i = 0; i < p.steps.size(); ++i) {
    if (!in_class(p.steps[i].dep_flags)) continue;
    const int gi = st.group_at.empty() ? -1 : st.group_at[i];
    if (gi < 0) {
      one((int)i);
      continue;
    }
    const GroupRun& gr = st.groups[gi];
    for (const auto& m : gr.multi) launch_simt_multi(ds, m, s);
    for (int t : gr.singles) one(t);
    i = (size_t)gr.end - 1;
  }
}

// Leaf select with the current chunk's parameters.  FP16X3: it also clears the
// maxima that the steps of the coming classes record (classes: bit 0
// slice-dependent steps, bit 1 per-batch ones; 0 the per-plan ones); the
// execution order keeps each class's steps together.
static void launch_leaf_select(Plan& p, cudaStream_t s, int classes, int ls) {
  DeviceState& ds = *p.dev;
  const int nl = (int)p.leaves.size();
  int z0 = 0, z1 = 0;
  if (ds.amax) {
    for (int i = 0; i < (int)p.steps.size(); ++i) {
      const int f = p.steps[i].dep_flags;
      const bool in = classes == 0 ? f == 0 : ((f & 1) && (classes & 1)) || (f == 2 && (classes & 2));
      if (!in) continue;
      if (z1 == 0) z0 = nl + i;
      else if (z1 != nl + i) fail(TN_ERR_PLAN, "internal: steps of a class are not consecutive");
      z1 = nl + i + 1;
    }
  }
  klaunch(k_leaf_select, dim3((unsigned)std::max(1, std::min(nl, 4096)), 1u << ls), 128, 0, s, 1,
          (const float2*)ds.leaf_data, (const LeafDesc*)ds.leaf_desc, nl, ds.arena, (const ChunkParam*)ds.params, (const unsigned*)ds.counter,
          ds.lane_stride, ds.amax, ds.amax_nodes, z0, z1);
}

// Whether a class has anything to run: 0, steps that depend on neither the
// slice nor the bitstring; 2, on the bitstring only; and the B' images of later
// steps whose B that class completes.
static bool has_prologue(const Plan& p, int cls) {
  for (const StepDesc& d : p.steps)
    if (d.dep_flags == cls) return true;
  for (const StepLaunch& L : p.dev->launches)
    if (L.bimg_own && L.bimg_cls == cls) return true;
  return false;
}

// The steps and B' images of one prologue class, on the leaves already selected.
static void run_prologue(Plan& p, cudaStream_t s, LaunchSet& st, int cls) {
  DeviceState& ds = *p.dev;
  launch_class(p, s, st, [cls](int f) { return f == cls; });
  auto images = [&](const StepLaunch& L) {
    if (!L.bimg_own || L.bimg_cls != cls) return;
    TcArgs t = L.tc;
    t.bimg = L.bimg_own;
    t.err = ds.err;
    launch_prep_kid(t, L.kid, s);
  };
  for (size_t i = 0; i < st.launches.size(); ++i) {
    images(st.launches[i]);
    if (!st.more.empty())
      for (const StepLaunch& L : st.more[i]) images(L);
  }
}

// One chunk per lane; new_batch: with their batches' prologues, which work on the
// same leaf select (the arena gives no leaf away before its last reader, and the
// prologue's steps come before the chunk's in the order it was laid out for).
static void run_chunk(Plan& p, cudaStream_t s, LaunchSet& st, bool new_batch) {
  DeviceState& ds = *p.dev;
  launch_leaf_select(p, s, new_batch ? 3 : 1, st.ls);
  if (new_batch) run_prologue(p, s, st, 2);
  launch_class(p, s, st, [](int f) { return (f & 1) != 0; });   // slice-dependent steps
  const bool one = ((int64_t)1 << p.root.rank) <= (int64_t)ds.root_blocks * 256;   // amplitude per thread
  klaunch(one ? k_root_sum<1> : k_root_sum<4>, dim3((unsigned)ds.root_blocks, (unsigned)ds.root_groups, 1u << st.ls),
          256, 0, s, 1, (const float2*)ds.arena, p.root, p.log2_batch, ds.root_groups, ds.root_part,
          (const ChunkParam*)ds.params, ds.counter, ds.root_tickets, ds.lane_stride);
}

// Capture run_chunk once into a graph (on a private stream, thread-local
// capture mode).  Any failure leaves the plan on eager launches.
static void capture_chunk_graph(Plan& p, LaunchSet& st, bool new_batch) {
  const int w = new_batch ? 1 : 0;
  if (st.graph[w] || st.graph_failed[w]) return;
  cudaStream_t cs = nullptr;
  if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    st.graph_failed[w] = true;
    return;
  }
  cudaGraph_t graph = nullptr;
  bool ok = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
  if (ok) {
    try {
      run_chunk(p, cs, st, new_batch);
    } catch (const TnError&) {
      ok = false;
    }
    ok = (cudaStreamEndCapture(cs, &graph) == cudaSuccess) && ok;
  }
  if (ok) ok = cudaGraphInstantiate(&st.graph[w], graph, 0) == cudaSuccess;
  if (graph) cudaGraphDestroy(graph);
  cudaStreamDestroy(cs);
  if (!ok) {
    cudaGetLastError();
    st.graph[w] = nullptr;
    st.graph_failed[w] = true;
  }
}

}  // namespace tnx

using namespace tnx;

#define API_BEGIN \
  try {           \
    clear_error();
#define API_END                        \
  return TN_OK;                        \
  }                                    \
  catch (const TnError& e) {           \
    set_error(e.msg);                  \
    return e.code;                     \
  }                                    \
  catch (const std::bad_alloc&) {      \
    set_error("host allocation failed"); \
    return TN_ERR_OOM;                 \
  }

extern "C" tn_status tn_contract_slices(tn_plan_t* h, uint64_t first, uint64_t count,
                                        const uint64_t* bitstrings, int32_t n_batches, double* out,
                                        void* stream) {
  API_BEGIN
  if (!h || !bitstrings || !out) fail(TN_ERR_ARG, "tn_contract_slices: NULL argument");
  Plan& p = h->plan;
  if (p.sticky != TN_OK) fail(p.sticky, p.sticky_msg);
  if (n_batches < 1) fail(TN_ERR_ARG, "n_batches must be >= 1");
  const int S = (int)p.sliced.size();
  const uint64_t total = S >= 64 ? ~0ULL : (1ULL << S);
  if (first > total || count > total - first) fail(TN_ERR_ARG, "slice range beyond 2^S");
  if (count == 0) return TN_OK;
  cudaStream_t s = (cudaStream_t)stream;
  ensure_device(p);
  DeviceState& ds = *p.dev;
  const int b = p.log2_batch;
  const uint64_t step = 1ULL << b;
  uint64_t open_mask = 0;
  for (int q : p.open_qubits) open_mask |= 1ULL << q;
  std::vector<ChunkParam> prm;
  for (int i = 0; i < n_batches; ++i)
    for (uint64_t base = (first >> b) << b; base < first + count; base += step) {
      ChunkParam c;
      c.slice_base = base;
      c.valid_lo = std::max(first, base);
      c.valid_hi = std::min(first + count, base + step);
      c.bitstring = bitstrings[i] & ~open_mask;
      c.out_index = i;
      c.out = out;
      prm.push_back(c);
    }
  if (ds.have_done) CK(cudaStreamWaitEvent(s, ds.done, 0));
  // Runs of chunks side by side: as many as the call has lanes.  A rest that is no
  // power of two is filled up with copies of its last chunk that count no slices
  // where a chunk is little work and all its launches are shared by the lanes, else
  // it is divided into powers of two.
  struct Run {
    size_t at;
    int ls;
  };
  std::vector<Run> runs;
  std::vector<ChunkParam> lanes;
  const bool fill = p.stats.flops_chunk <= 5e8 && !ds.tc_chunk;
  const int ls_call = lanes_of_call(ds, (size_t)n_batches, prm.size() / (size_t)n_batches);
  for (size_t i = 0; i < prm.size();) {
    const size_t q = std::min(prm.size() - i, (size_t)1 << ls_call);
    int ls = 0;
    while (fill ? ((size_t)1 << ls) < q : ((size_t)2 << ls) <= q) ++ls;
    runs.push_back({lanes.size(), ls});
    for (size_t l = 0; l < ((size_t)1 << ls); ++l) {
      lanes.push_back(prm[std::min(i + l, prm.size() - 1)]);
      if (l >= q) lanes.back().valid_lo = lanes.back().valid_hi = 0;
    }
    i += std::min(q, (size_t)1 << ls);
  }
  if (lanes.size() > ds.params_cap) {
    if (ds.params) {
      CK(cudaStreamSynchronize(s));
      drop_graphs(ds);   // captured with the old buffer's address
      CK(cudaFree(ds.counter));
      ds.counter = nullptr;
      ds.params = nullptr;
    }
    ds.params_cap = 0;
    const size_t cap = std::max<size_t>(lanes.size(), 1024);
    CK(cudaMalloc(&ds.counter, PARAMS_AT + cap * sizeof(ChunkParam)));
    ds.params = reinterpret_cast<ChunkParam*>(reinterpret_cast<uint8_t*>(ds.counter) + PARAMS_AT);
    ds.params_cap = cap;
  }
  // the counter (zero) and the parameters in one copy
  std::vector<uint8_t> up(PARAMS_AT + lanes.size() * sizeof(ChunkParam), 0);
  std::memcpy(up.data() + PARAMS_AT, lanes.data(), lanes.size() * sizeof(ChunkParam));
  CK(cudaMemcpyAsync(ds.counter, up.data(), up.size(), cudaMemcpyHostToDevice, s));
  const bool pro0 = has_prologue(p, 0), pro2 = has_prologue(p, 2);
  for (const Run& r : runs) {
    const int n = 1 << r.ls;
    LaunchSet& st = ds.set[r.ls];
    if (ds.pro0_lanes < n) {
      if (pro0) {
        launch_leaf_select(p, s, 0, r.ls);
        run_prologue(p, s, st, 0);
      }
      ds.pro0_lanes = n;
    }
    bool new_batch = false;
    for (int l = 0; l < n && pro2; ++l)
      new_batch = new_batch || !ds.pro2_valid[l] || ds.pro2_bits[l] != lanes[r.at + l].bitstring;
    const int w = new_batch ? 1 : 0;
    if (!st.eager_done[w]) {
      run_chunk(p, s, st, new_batch);           // the first one runs eagerly (sets kernel attributes)
      st.eager_done[w] = true;
    } else {
      capture_chunk_graph(p, st, new_batch);
      if (st.graph[w])
        CK(cudaGraphLaunch(st.graph[w], s));
      else
        run_chunk(p, s, st, new_batch);
    }
    CK(cudaGetLastError());
    for (int l = 0; l < n && new_batch; ++l) {
      ds.pro2_valid[l] = true;
      ds.pro2_bits[l] = lanes[r.at + l].bitstring;
    }
    // one batch's prologue is kept, the last one's (for its further slices), however
    // many lanes there are: a batch that comes back is contracted again
    const uint64_t last = lanes[r.at + n - 1].bitstring;
    for (int l = 0; l < (1 << MAX_LS_LANES); ++l) ds.pro2_valid[l] = ds.pro2_valid[l] && ds.pro2_bits[l] == last;
  }
  CK(cudaEventRecord(ds.done, s));
  ds.have_done = true;
  API_END
}

extern "C" tn_status tn_plan_step_times(tn_plan_t* h, int32_t reps, double* ms_out, int32_t* kernel_out,
                                        void* stream) {
  API_BEGIN
  if (!h || !ms_out) fail(TN_ERR_ARG, "tn_plan_step_times: NULL argument");
  if (reps < 1) fail(TN_ERR_ARG, "tn_plan_step_times: reps must be >= 1");
  Plan& p = h->plan;
  if (!p.dev) fail(TN_ERR_ARG, "tn_plan_step_times: run tn_contract_slices first");
  cudaStream_t s = (cudaStream_t)stream;
  DeviceState& ds = *p.dev;
  if (ds.have_done) CK(cudaStreamWaitEvent(s, ds.done, 0));
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  for (size_t i = 0; i < p.steps.size(); ++i) {
    launch_step(ds.launches[i], ds.ws, ds.err, s, true);  // warm-up
    CK(cudaEventRecord(e0, s));
    for (int r = 0; r < reps; ++r) launch_step(ds.launches[i], ds.ws, ds.err, s, true);
    CK(cudaEventRecord(e1, s));
    CK(cudaEventSynchronize(e1));
    float ms = 0;
    CK(cudaEventElapsedTime(&ms, e0, e1));
    ms_out[i] = (double)ms / reps;
    if (kernel_out) kernel_out[i] = ds.launches[i].kid;
  }
  CK(cudaGetLastError());
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  ds.forget_prologues();   // the arena was overwritten: they run again
  API_END
}

// After the kernels of a plan changed: launch sets, graphs and prologues anew (a plan
// whose sets cannot be built starts anew with its next call).
static void kernels_changed(Plan& p, DeviceState& ds) {
  drop_graphs(ds);
  try {
    setup_hoisted(p, ds);
    build_sets(p, ds);
  } catch (...) {
    destroy_device_state(&p);
    throw;
  }
  set_lane_times(p, ds);
  ds.forget_prologues();   // the arena may have been overwritten: they run again
}

// Autotuner: for every step, time the candidate kernels in place (tensor-core
// tiles of 32, 64 or 128 complex columns in the TF32 / BF16X3 / FP16X3 modes,
// each with either write-back order, with the default or a deeper B' ring (4,
// 6 or 8 slots) and on one SM or an SM pair, and the CUDA-core tilings
// where the step is small or the mode is FP32) and keep the fastest.  The
// chunk graph is captured again on the next call.
extern "C" tn_status tn_plan_autotune(tn_plan_t* h, int32_t reps, void* stream) {
  API_BEGIN
  if (!h) fail(TN_ERR_ARG, "tn_plan_autotune: NULL plan");
  if (reps < 1) fail(TN_ERR_ARG, "tn_plan_autotune: reps must be >= 1");
  Plan& p = h->plan;
  if (!p.dev) fail(TN_ERR_ARG, "tn_plan_autotune: run tn_contract_slices first");
  DeviceState& ds = *p.dev;
  cudaStream_t s = (cudaStream_t)stream;
  if (ds.have_done) CK(cudaStreamWaitEvent(s, ds.done, 0));
  CK(cudaStreamSynchronize(s));
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  auto time_launch = [&](StepLaunch& L) -> double {
    if (L.ws_bytes > ds.ws_bytes) {
      CK(cudaStreamSynchronize(s));
      grow_workspace(p, L.ws_bytes, "tn_plan_autotune");
    }
    launch_step(L, ds.ws, ds.err, s, true);  // warm-up
    CK(cudaEventRecord(e0, s));
    for (int r = 0; r < reps; ++r) launch_step(L, ds.ws, ds.err, s, true);
    CK(cudaEventRecord(e1, s));
    CK(cudaEventSynchronize(e1));
    float ms = 0;
    CK(cudaEventElapsedTime(&ms, e0, e1));
    return (double)ms / reps;
  };
  for (size_t i = 0; i < p.steps.size(); ++i) {
    const StepDesc& d = p.steps[i];
    auto build = [&](int kid, int tn_log, int epi, int bslots, int pair) {
      return build_choice(ds, d, kid, tn_log, epi, bslots, pair);
    };
    StepLaunch cur = ds.launches[i];
    cur.bimg_own = nullptr;   // timed like the candidates: B' images built with the launch
    double best = time_launch(cur);
    // kernel, tile width (log2 complex columns), write-back, B' slots, SM pairs
    std::vector<std::array<int, 5>> cands;
    const bool tc_mode = p.opts.precision != TN_PREC_FP32;
    const int tc_kid = tc_kernel(p.opts.precision, p.opts.complex_mult);
    if (tc_mode && d.nm >= 4)
      for (int tn_log : {7, 6, 5})
        if (tn_log <= std::max(3, d.nn))
          for (int epi : {0, 1})
            for (int bs : {0, 4, 6, 8})
              for (int pair : {1, 0})
                if (pair == 0 || p.opts.sm_pairs) cands.push_back({tc_kid, tn_log, epi, bs, pair});
    // CUDA-core tilings: FP32 mode, tiny steps, and low arithmetic intensity
    // (complex flops per byte moved), where a tile's fixed cost on the tensor
    // cores outweighs its few products
    const double flops = 8.0 * std::ldexp(1.0, d.nm + d.nk + d.nn + d.nb);
    const double bytes = 8.0 * (double)(d.a_elems + d.b_elems + d.c_elems);
    if (!tc_mode || best < 0.05 || flops / bytes < 48.0)
      for (int k : {K_SIMT_64x64, K_SIMT_128x16, K_SIMT_256x4, K_SIMT_128x64, K_SIMT_32x32})
        cands.push_back({k, -1, 0, 0, 0});
    std::vector<std::array<int, 5>> seen;
    auto key = [](const StepLaunch& L) {
      return std::array<int, 5>{L.kid, L.g.tn, is_tc(L.kid) ? L.tc.epi_ok : 0, is_tc(L.kid) ? L.tc.nbs : 0,
                                is_tc(L.kid) ? L.tc.pair : 0};
    };
    seen.push_back(key(ds.launches[i]));
    for (auto [kid, tn_log, epi, bs, pair] : cands) {
      StepLaunch L;
      try {
        L = build(kid, tn_log, epi, bs, pair);
      } catch (const TnError&) {
        continue;   // this configuration does not fit: not a candidate
      }
      if (std::find(seen.begin(), seen.end(), key(L)) != seen.end()) continue;
      seen.push_back(key(L));
      const double t = time_launch(L);
      if (t < best * 0.97) {
        best = t;
        ds.launches[i] = L;
      }
    }
  }
  CK(cudaGetLastError());
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  kernels_changed(p, ds);
  API_END
}

extern "C" tn_status tn_plan_get_tuning(const tn_plan_t* h, int32_t* out, int32_t cap, int32_t* n_out) {
  API_BEGIN
  if (!h || !out || !n_out) fail(TN_ERR_ARG, "tn_plan_get_tuning: NULL argument");
  const Plan& p = h->plan;
  if (!p.dev) fail(TN_ERR_ARG, "tn_plan_get_tuning: run tn_contract_slices first");
  const int64_t need = (int64_t)p.steps.size() * TN_TUNING_INTS;
  if (cap < need) fail(TN_ERR_ARG, "tn_plan_get_tuning: cap below n_steps * TN_TUNING_INTS");
  for (size_t i = 0; i < p.steps.size(); ++i) {
    const StepLaunch& L = p.dev->launches[i];
    int32_t* o = out + i * TN_TUNING_INTS;
    const bool tc = is_tc(L.kid);
    o[0] = L.kid;
    o[1] = tc ? L.g.tn : -1;
    o[2] = tc ? L.tc.epi_ok : 0;
    o[3] = tc ? L.tc.nbs : 0;
    o[4] = tc ? L.tc.pair : 0;
  }
  *n_out = (int32_t)need;
  API_END
}

extern "C" tn_status tn_plan_set_tuning(tn_plan_t* h, const int32_t* in, int32_t n) {
  API_BEGIN
  if (!h || !in) fail(TN_ERR_ARG, "tn_plan_set_tuning: NULL argument");
  Plan& p = h->plan;
  if (!p.dev) fail(TN_ERR_ARG, "tn_plan_set_tuning: run tn_contract_slices first");
  if ((int64_t)n != (int64_t)p.steps.size() * TN_TUNING_INTS)
    fail(TN_ERR_ARG, "tn_plan_set_tuning: n is not n_steps * TN_TUNING_INTS");
  DeviceState& ds = *p.dev;
  std::vector<StepLaunch> next(p.steps.size());
  int64_t ws = ds.ws_bytes;
  for (size_t i = 0; i < p.steps.size(); ++i) {
    const int32_t* c = in + i * TN_TUNING_INTS;
    const int kid = c[0];
    const bool simt = is_simt(kid);
    if (!simt && !is_tc(kid)) fail(TN_ERR_ARG, "tn_plan_set_tuning: unknown kernel id");
    if (is_tc(kid) && (p.opts.precision == TN_PREC_FP32 || kid != tc_kernel(p.opts.precision, p.opts.complex_mult)))
      fail(TN_ERR_ARG, "tn_plan_set_tuning: tensor-core kernel of another precision or product");
    if (c[2] < 0 || c[2] > 1 || c[3] < 0 || c[3] > TC_MAX_B || c[4] < 0 || c[4] > 1 || c[1] < -1 || c[1] > 7)
      fail(TN_ERR_ARG, "tn_plan_set_tuning: choice out of range");
    try {
      next[i] = simt ? build_choice(ds, p.steps[i], kid, -1, 0, 0, 0)
                     : build_choice(ds, p.steps[i], kid, c[1], c[2], c[3], c[4] && p.opts.sm_pairs ? 1 : 0);
    } catch (const TnError& e) {
      fail(TN_ERR_ARG, std::string("tn_plan_set_tuning: step ") + std::to_string(i) + ": " + e.msg);
    }
    ws = std::max(ws, next[i].ws_bytes);
  }
  grow_workspace(p, ws, "tn_plan_set_tuning");
  ds.launches.swap(next);
  kernels_changed(p, ds);
  API_END
}

// Time a few chunks of every candidate (seed and memory weight per candidate, the
// rest from *opts) after an untimed warm-up, and keep the plan whose estimate for
// all 2^S slices is smallest.
static void select_among(const tn_network_t* net, const tn_plan_opts* opts, int32_t n_candidates,
                         const uint64_t* seeds, const double* weights, uint64_t bitstring, void* stream,
                         tn_plan_t** out, double* cand_seconds) {
  *out = nullptr;
  cudaStream_t s = (cudaStream_t)stream;
  tn_plan_t* best = nullptr;
  double best_t = 0.0;
  double* amps = nullptr;
  size_t amps_bytes = 0;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  for (int i = 0; i < n_candidates; ++i) {
    if (cand_seconds) cand_seconds[i] = -1.0;
    tn_plan_opts o = *opts;
    o.seed = seeds[i];
    o.mem_weight = weights[i];
    tn_plan_t* h = nullptr;
    if (tn_plan(net, &o, &h) != TN_OK || !h) continue;
    Plan& p = h->plan;
    const uint64_t chunk = 1ULL << p.log2_batch;
    const size_t need = sizeof(double) * 2 * ((size_t)1 << p.root.rank);
    if (need > amps_bytes) {
      if (amps) CK(cudaFree(amps));
      amps = nullptr;
      CK(cudaMalloc(&amps, need));
      amps_bytes = need;
    }
    double est = -1.0;
    // warm-up (device state, prologues, graph capture), then the fastest of three
    // timed calls of as many chunks as the plan runs side by side
    if (tn_contract_slices(h, 0, chunk, &bitstring, 1, amps, s) == TN_OK) {
      const int log2_timed = std::min((int)p.sliced.size(), p.log2_batch + p.dev->ls_lanes);
      const uint64_t timed = 1ULL << log2_timed;
      float best_ms = -1.f;
      tn_status st = timed > chunk ? tn_contract_slices(h, 0, timed, &bitstring, 1, amps, s) : TN_OK;
      for (int r = 0; r < 3 && st == TN_OK; ++r) {
        CK(cudaEventRecord(e0, s));
        st = tn_contract_slices(h, 0, timed, &bitstring, 1, amps, s);
        CK(cudaEventRecord(e1, s));
        CK(cudaEventSynchronize(e1));
        float ms = 0.f;
        CK(cudaEventElapsedTime(&ms, e0, e1));
        if (best_ms < 0.f || ms < best_ms) best_ms = ms;
      }
      if (st == TN_OK && tn_plan_sync(h, s) == TN_OK)
        est = (double)best_ms / 1e3 * std::ldexp(1.0, (int)p.sliced.size() - log2_timed);
    }
    CK(cudaStreamSynchronize(s));
    destroy_device_state(&p);
    cudaGetLastError();
    clear_error();
    if (cand_seconds) cand_seconds[i] = est;
    if (est >= 0.0 && (!best || est < best_t)) {
      if (best) tn_plan_destroy(best);
      best = h;
      best_t = est;
    } else {
      tn_plan_destroy(h);
    }
  }
  if (amps) cudaFree(amps);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!best) fail(TN_ERR_PLAN, "plan selection: no candidate plan could be built and run");
  best->plan.sticky = TN_OK;
  *out = best;
}

extern "C" tn_status tn_plan_select(const tn_network_t* net, const tn_plan_opts* opts, int32_t n_candidates,
                                    uint64_t bitstring, void* stream, tn_plan_t** out, double* cand_seconds) {
  API_BEGIN
  if (!net || !opts || !out) fail(TN_ERR_ARG, "tn_plan_select: NULL argument");
  if (n_candidates < 1 || n_candidates > 1024) fail(TN_ERR_ARG, "tn_plan_select: n_candidates must be in [1, 1024]");
  const double w0 = opts->mem_weight > 0.0 ? opts->mem_weight : 32.0;
  const double wmul[3] = {1.0, 0.25, 4.0};
  std::vector<uint64_t> seeds(n_candidates);
  std::vector<double> weights(n_candidates);
  for (int i = 0; i < n_candidates; ++i) {
    seeds[i] = opts->seed + (uint64_t)i;
    weights[i] = w0 * wmul[i % 3];
  }
  select_among(net, opts, n_candidates, seeds.data(), weights.data(), bitstring, stream, out, cand_seconds);
  API_END
}

extern "C" tn_status tn_plan_select_list(const tn_network_t* net, const tn_plan_opts* opts, int32_t n_candidates,
                                         const uint64_t* seeds, const double* mem_weights, uint64_t bitstring,
                                         void* stream, tn_plan_t** out, double* cand_seconds) {
  API_BEGIN
  if (!net || !opts || !out || !seeds || !mem_weights) fail(TN_ERR_ARG, "tn_plan_select_list: NULL argument");
  if (n_candidates < 1 || n_candidates > 1024)
    fail(TN_ERR_ARG, "tn_plan_select_list: n_candidates must be in [1, 1024]");
  for (int i = 0; i < n_candidates; ++i)
    if (!(mem_weights[i] <= 0.0 || (mem_weights[i] >= 1e-6 && mem_weights[i] <= 1e9)))
      fail(TN_ERR_ARG, "tn_plan_select_list: mem_weight must be <= 0 (default) or in [1e-6, 1e9]");
  select_among(net, opts, n_candidates, seeds, mem_weights, bitstring, stream, out, cand_seconds);
  API_END
}

extern "C" tn_status tn_plan_chunk_launches(const tn_plan_t* h, int32_t* launches) {
  API_BEGIN
  if (!h || !launches) fail(TN_ERR_ARG, "tn_plan_chunk_launches: NULL argument");
  const Plan& p = h->plan;
  if (!p.dev) fail(TN_ERR_ARG, "tn_plan_chunk_launches: call after the first tn_contract_slices");
  int shared, alone;
  class_launches(p, [](int f) { return (f & 1) != 0; }, &shared, &alone);
  *launches = 2 + shared + alone;
  API_END
}

extern "C" tn_status tn_plan_batch_launches(const tn_plan_t* h, int32_t* launches) {
  API_BEGIN
  if (!h || !launches) fail(TN_ERR_ARG, "tn_plan_batch_launches: NULL argument");
  const Plan& p = h->plan;
  if (!p.dev) fail(TN_ERR_ARG, "tn_plan_batch_launches: call after the first tn_contract_slices");
  int shared, alone;
  class_launches(p, [](int f) { return f == 2; }, &shared, &alone);
  int n = shared + alone;
  for (const StepLaunch& L : p.dev->launches) n += (L.bimg_own && L.bimg_cls == 2) ? 1 : 0;   // B' images
  *launches = n;   // on the leaf select of the batch's first chunk
  API_END
}

extern "C" tn_status tn_plan_sync(tn_plan_t* h, void* stream) {
  API_BEGIN
  if (!h) fail(TN_ERR_ARG, "tn_plan_sync: NULL plan");
  CK(cudaStreamSynchronize((cudaStream_t)stream));
  if (h->plan.dev && h->plan.sticky == TN_OK) {
    int32_t e = 0;
    CK(cudaMemcpy(&e, h->plan.dev->err, sizeof(e), cudaMemcpyDeviceToHost));
    if (e != 0) {
      h->plan.sticky = e;
      h->plan.sticky_msg = "a device kernel reported error " + std::to_string(e) +
                           " (bounded wait expired or device check failed)";
    }
  }
  if (h->plan.sticky != TN_OK) fail(h->plan.sticky, h->plan.sticky_msg);
  API_END
}

extern "C" void tn_plan_destroy(tn_plan_t* h) {
  if (!h) return;
  destroy_device_state(&h->plan);
  delete h;
}

// FP16X3 calls without a plan: the maxima of A and B by one reduction pass each
static void operand_maxima(const float2* a, int64_t na, const float2* b, int64_t nb, float* amax, cudaStream_t s) {
  CK(cudaMemsetAsync(amax, 0, 2 * sizeof(float), s));
  const int ga = (int)std::min<int64_t>((na + 255) / 256, (int64_t)sm_count() * 8);
  const int gb = (int)std::min<int64_t>((nb + 255) / 256, (int64_t)sm_count() * 8);
  k_amax<<<std::max(ga, 1), 256, 0, s>>>(a, na, amax);
  k_amax<<<std::max(gb, 1), 256, 0, s>>>(b, nb, amax + 1);
}

// Per-device scratch of the calls that have no plan: the XEB sum, the sampling
// results, the error word and the B' workspace of tn_contract_pair.
constexpr int64_t kHostWords = 8192;
struct Scratch {
  // held by tn_xeb and tn_frugal_sample from their launch to their result: the
  // buffers they share, and the ticket, then serve one call at a time
  std::mutex sync_calls;
  double* xeb = nullptr;          // XEB: the sum, then the blocks' partial sums
  unsigned* xeb_ticket = nullptr; // zero between launches
  bool xeb_ticket_zero = false;   // false while a launch's end has not been seen
  int32_t* err = nullptr;
  float* amax = nullptr;   // FP16X3 operand maxima of the last call (A, B)
  unsigned long long* first = nullptr;   // frugal sampling: ~0 unless a candidate was out of range, then the
                                         // first accepted draw per sample (~0: none)
  int64_t first_cap = 0;
  unsigned long long* host = nullptr;    // page-locked: results on their way to the caller
  uint8_t* ws = nullptr;
  int64_t ws_bytes = 0;
};
static std::mutex g_scratch_mu;
static std::unordered_map<int, Scratch> g_scratch;   // per device
static Scratch& scratch_for_device() {
  int dev = 0;
  CK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  Scratch& s = g_scratch[dev];
  if (!s.host) {   // the last of them: what an earlier, failed call allocated is kept
    if (!s.xeb_ticket) CK(cudaMalloc(&s.xeb_ticket, sizeof(unsigned)));
    if (!s.xeb) CK(cudaMalloc(&s.xeb, sizeof(double) * (1 + XEB_BLOCKS)));
    if (!s.err) {
      int32_t* err = nullptr;
      CK(cudaMalloc(&err, sizeof(int32_t)));
      CK(cudaMemset(err, 0, sizeof(int32_t)));
      s.err = err;
    }
    if (!s.amax) CK(cudaMalloc(&s.amax, 2 * sizeof(float)));
    CK(cudaMallocHost(&s.host, kHostWords * sizeof(unsigned long long)));
  }
  return s;
}

extern "C" tn_status tn_xeb(const double* amps, int64_t count, int32_t n_qubits, double* xeb_out,
                            void* stream) {
  API_BEGIN
  if (!amps || !xeb_out) fail(TN_ERR_ARG, "tn_xeb: NULL argument");
  if (count < 1) fail(TN_ERR_ARG, "tn_xeb: count must be >= 1");
  if (n_qubits < 0 || n_qubits > 1023) fail(TN_ERR_ARG, "tn_xeb: n_qubits out of range");
  Scratch& sc = scratch_for_device();
  std::lock_guard<std::mutex> one(sc.sync_calls);
  double* scratch = sc.xeb;
  cudaStream_t s = (cudaStream_t)stream;
  if (!sc.xeb_ticket_zero) CK(cudaMemsetAsync(sc.xeb_ticket, 0, sizeof(unsigned), s));
  sc.xeb_ticket_zero = false;
  // a block per 1024 amplitudes (four a thread), at most four blocks per SM
  const int64_t per = 4 * XEB_THREADS;
  const int blocks = (int)std::min<int64_t>((count + per - 1) / per, std::min<int64_t>(4 * sm_count(), XEB_BLOCKS));
  k_xeb_sum<<<blocks, XEB_THREADS, 0, s>>>(reinterpret_cast<const double2*>(amps), count, scratch, sc.xeb_ticket);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(sc.host, scratch, sizeof(double), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  sc.xeb_ticket_zero = true;
  double sum = 0;
  std::memcpy(&sum, sc.host, sizeof(double));
  *xeb_out = std::ldexp(sum / (double)count, n_qubits) - 1.0;
  API_END
}

extern "C" tn_status tn_frugal_sample(const double* amps, int64_t count, int32_t n_qubits, double m_bound,
                                     const int64_t* candidates, const double* uniforms, int64_t n_draws,
                                     int64_t n_samples, int64_t* first_out, void* stream) {
  API_BEGIN
  if (!amps || !candidates || !uniforms || !first_out) fail(TN_ERR_ARG, "tn_frugal_sample: NULL argument");
  if (count < 1 || n_draws < 1 || n_samples < 1) fail(TN_ERR_ARG, "tn_frugal_sample: empty batch, draws or samples");
  if (n_qubits < 0 || n_qubits > 1000) fail(TN_ERR_ARG, "tn_frugal_sample: n_qubits out of range");
  if (!(m_bound > 0.0) || !std::isfinite(m_bound)) fail(TN_ERR_ARG, "tn_frugal_sample: m_bound must be positive");
  if (n_draws > ((int64_t)1 << 40) / n_samples) fail(TN_ERR_ARG, "tn_frugal_sample: too many draws");
  Scratch& sc = scratch_for_device();
  std::lock_guard<std::mutex> one(sc.sync_calls);
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t words = n_samples + 1;
  if (words > sc.first_cap) {
    CK(cudaStreamSynchronize(s));
    if (sc.first) CK(cudaFree(sc.first));
    sc.first = nullptr;
    sc.first_cap = 0;
    CK(cudaMalloc(&sc.first, sizeof(unsigned long long) * (size_t)words));
    sc.first_cap = words;
  }
  CK(cudaMemsetAsync(sc.first, 0xff, sizeof(unsigned long long) * (size_t)words, s));
  const int64_t total = n_draws * n_samples;
  const int blocks = (int)std::min<int64_t>((total + 255) / 256, (int64_t)sm_count() * 16);
  k_frugal<<<blocks, 256, 0, s>>>(reinterpret_cast<const double2*>(amps), count, n_qubits, m_bound, candidates,
                                  uniforms, n_draws, n_samples, sc.first);
  CK(cudaGetLastError());
  std::vector<unsigned long long> many;   // more samples than the page-locked area holds
  unsigned long long* f = sc.host;
  if (words > kHostWords) {
    many.resize((size_t)words);
    f = many.data();
  }
  CK(cudaMemcpyAsync(f, sc.first, sizeof(unsigned long long) * (size_t)words, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (f[0] != ~0ULL) fail(TN_ERR_ARG, "tn_frugal_sample: a candidate index is outside [0, count)");
  std::memcpy(first_out, f + 1, sizeof(int64_t) * (size_t)n_samples);   // ~0 is -1: no accepted draw
  API_END
}

// Tile bits and shared-memory slots of the tiled permutation with nt tile bits.
static void permute_tile(PermArgs& pa, int rank, const int32_t* perm, int nt) {
  std::vector<int> out_of_in(rank);
  for (int p = 0; p < rank; ++p) out_of_in[perm[p]] = p;
  // alternately the next input position and the source of the next output
  // position, so that both runs grow alike
  std::vector<char> in_tile(rank, 0);
  for (int n = 0, ni = 0, no = 0; n < nt;) {
    while (ni < rank && in_tile[ni]) ++ni;
    if (ni < rank) {
      in_tile[ni] = 1;
      ++n;
    }
    while (no < rank && in_tile[perm[no]]) ++no;
    if (n < nt && no < rank) {
      in_tile[perm[no]] = 1;
      ++n;
    }
  }
  pa.nt = nt;
  pa.nr = 0;
  std::vector<int> in_order, out_order;   // input positions of the tile bits, in either order
  for (int i = 0; i < rank; ++i) {
    if (in_tile[i]) {
      in_order.push_back(i);
    } else {
      pa.r_in[pa.nr] = (int8_t)i;
      pa.r_out[pa.nr] = (int8_t)out_of_in[i];
      ++pa.nr;
    }
  }
  for (int p = 0; p < rank; ++p)
    if (in_tile[perm[p]]) out_order.push_back(perm[p]);
  std::vector<int> q_of_in(rank, -1);
  for (int q = 0; q < nt; ++q) q_of_in[in_order[q]] = q;
  // The slot of an element is (4-bit linear map of its bits, bits 4..) in input
  // order: 8-byte accesses are free of bank conflicts when the 16 elements of a
  // half warp, which differ in bits 1-4 of either order, differ in that map.  So
  // the columns of bits 0-3 (the slot stays a permutation), of input-order bits
  // 1-4 and of output-order bits 1-4 must each be independent.
  int col[PERM_MAX_T] = {1, 2, 4, 8};
  int oq[4];
  for (int i = 0; i < 4; ++i) oq[i] = q_of_in[out_order[i + 1]];
  auto independent = [](const std::vector<int>& v) {
    for (int m = 1; m < (1 << v.size()); ++m) {
      int x = 0;
      for (size_t i = 0; i < v.size(); ++i)
        if ((m >> i) & 1) x ^= v[i];
      if (x == 0) return false;
    }
    return true;
  };
  for (int c4 = 1; c4 < 16; c4 += 2) {   // odd: independent of the columns of bits 1-3
    col[4] = c4;
    std::vector<int> fixed;
    for (int i = 0; i < 4; ++i)
      if (oq[i] <= 4) fixed.push_back(col[oq[i]]);
    if (!independent(fixed)) continue;
    for (int i = 0; i < 4; ++i) {
      if (oq[i] <= 4) continue;
      for (int c = 1; c < 16; ++c) {
        fixed.push_back(c);
        if (independent(fixed)) {
          col[oq[i]] = c;
          break;
        }
        fixed.pop_back();
      }
    }
    break;
  }
  for (int q = 0; q < nt; ++q) {
    pa.t_in[q] = (int8_t)in_order[q];
    pa.wcol[q] = (int16_t)((q >= 4 ? 1 << q : 0) ^ col[q]);
  }
  for (int q = 0; q < nt; ++q) {
    pa.t_out[q] = (int8_t)out_of_in[out_order[q]];
    pa.rcol[q] = pa.wcol[q_of_in[out_order[q]]];
  }
}

extern "C" tn_status tn_permute(const float* in, float* out, int32_t rank, const int32_t* perm,
                                int64_t batch, void* stream) {
  API_BEGIN
  if (!in || !out || (!perm && rank > 0)) fail(TN_ERR_ARG, "tn_permute: NULL argument");
  if (rank < 0 || rank > 34) fail(TN_ERR_ARG, "tn_permute: rank must be in [0, 34]");
  if (batch < 0) fail(TN_ERR_ARG, "tn_permute: negative batch");
  PermArgs pa;
  std::memset(&pa, 0, sizeof(pa));
  std::vector<char> seen(rank, 0);
  for (int p = 0; p < rank; ++p) {
    if (perm[p] < 0 || perm[p] >= rank || seen[perm[p]]) fail(TN_ERR_ARG, "tn_permute: not a permutation");
    seen[perm[p]] = 1;
    pa.src_pos[p] = (int8_t)perm[p];
  }
  const int64_t total = batch << rank;
  if (total == 0) return TN_OK;
  if (rank < 10) {
    const int blocks = (int)std::min<int64_t>((total + 255) / 256, 152 * 64);
    k_permute_gather<<<blocks, 256, 0, (cudaStream_t)stream>>>(reinterpret_cast<const float2*>(in),
                                                               reinterpret_cast<float2*>(out), rank, pa, total);
  } else {
    // tiles of 2^12 elements where they give every SM at least four (5.4 TB/s at
    // rank 24, 6.0-6.4 from 26 on; 3.2 and 3.9 with 2^10), else 2^10 (rank 20: 2.5
    // TB/s, its 8 MB a few microseconds of latency)
    const int nt = rank >= 12 && (batch << (rank - 12)) >= 4 * (int64_t)sm_count() ? 12 : 10;
    permute_tile(pa, rank, perm, nt);
    const int64_t tiles = batch << pa.nr;
    // 16-byte pairs need both arrays aligned (an instance is 2^rank elements)
    const int vec = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const int blocks = (int)std::min<int64_t>(tiles, (int64_t)sm_count() * (nt == 12 ? 4 : 8));
    const float2* x = reinterpret_cast<const float2*>(in);
    float2* y = reinterpret_cast<float2*>(out);
    if (nt == 12)
      k_permute_tiled<12><<<blocks, 256, 0, (cudaStream_t)stream>>>(x, y, rank, pa, tiles, vec);
    else
      k_permute_tiled<10><<<blocks, 256, 0, (cudaStream_t)stream>>>(x, y, rank, pa, tiles, vec);
  }
  CK(cudaGetLastError());
  API_END
}

// Order of the m and n bits of a pairwise contraction (the tile takes the first
// ones; any order gives the same sums).  Operands in any order: rows alternate
// between C's lowest positions and A's, columns between C's and B's, so that a
// tile's reads and writes both run along memory.  A stored [contracted...,
// free...] keeps its rows in order, for its tensor-map loads.  In the wires'
// order of A and B C's stores were mostly single elements: 2^18 x 64 x 128 in random
// order, TF32, took 208 us (271 with the older gather), 82 with this.
static void order_pair_bits(StepDesc& d) {
  // op, cp: positions of the n bits in the operand and in C
  auto order = [](int n, int8_t* op, int8_t* cp) {
    int8_t at_op[64], at_c[64], o[MAXR], c[MAXR];   // bit at a position, -1 for none
    std::memset(at_op, -1, sizeof(at_op));
    std::memset(at_c, -1, sizeof(at_c));
    std::memcpy(o, op, sizeof(o));
    std::memcpy(c, cp, sizeof(c));
    for (int i = 0; i < n; ++i) {
      at_op[o[i]] = (int8_t)i;
      at_c[c[i]] = (int8_t)i;
    }
    uint64_t used = 0;
    for (int k = 0, pc = 0, po = 0; k < n;) {
      auto take = [&](const int8_t* at, int& pos) {   // the lowest bit of one side not taken yet
        while (pos < 64 && (at[pos] < 0 || ((used >> at[pos]) & 1))) ++pos;
        if (pos == 64 || k == n) return;
        const int i = at[pos];
        used |= 1ull << i;
        op[k] = o[i];
        cp[k] = c[i];
        ++k;
      };
      take(at_c, pc);
      take(at_op, po);
    }
  };
  bool k_first = true;
  for (int j = 0; j < d.nk; ++j) k_first = k_first && d.a_kpos[j] == j;
  if (!(k_first && d.nk >= 4)) order(d.nm, d.a_mpos, d.c_mpos);
  order(d.nn, d.b_npos, d.c_npos);
}

extern "C" tn_status tn_contract_pair(const float* a, const int32_t* aw, int32_t ar, const float* b,
                                      const int32_t* bw, int32_t br, float* c, const int32_t* cw,
                                      int32_t cr, int64_t batch, int32_t precision, int32_t cmult,
                                      void* stream) {
  API_BEGIN
  if (!a || !b || !c || (ar && !aw) || (br && !bw) || (cr && !cw)) fail(TN_ERR_ARG, "tn_contract_pair: NULL argument");
  if (ar < 0 || br < 0 || cr < 0 || ar > 34 || br > 34 || cr > 34) fail(TN_ERR_ARG, "tn_contract_pair: rank out of range");
  if (batch < 1 || batch > 65535) fail(TN_ERR_ARG, "tn_contract_pair: batch must be in [1, 65535]");
  if (precision < TN_PREC_FP32 || precision > TN_PREC_FP16X3) fail(TN_ERR_ARG, "unknown precision");
  if (cmult != 3 && cmult != 4) fail(TN_ERR_ARG, "complex_mult must be 3 or 4");
  if (cmult == 3 && precision == TN_PREC_FP32)
    fail(TN_ERR_UNSUPPORTED, "the FP32 CUDA-core path forms 4M products only; 3M needs TF32 or BF16X3");
  std::vector<int> A(aw, aw + ar), B(bw, bw + br), Cw(cw, cw + cr);
  auto has = [](const std::vector<int>& v, int w) { return std::find(v.begin(), v.end(), w) != v.end(); };
  for (size_t i = 0; i < A.size(); ++i)
    for (size_t j = i + 1; j < A.size(); ++j)
      if (A[i] == A[j]) fail(TN_ERR_ARG, "repeated wire in a_wires");
  for (size_t i = 0; i < B.size(); ++i)
    for (size_t j = i + 1; j < B.size(); ++j)
      if (B[i] == B[j]) fail(TN_ERR_ARG, "repeated wire in b_wires");
  StepDesc d;
  std::memset(&d, 0, sizeof(d));
  std::vector<int> mw, kw, nw;
  for (int w : A) (has(B, w) ? kw : mw).push_back(w);
  for (int w : B)
    if (!has(A, w)) nw.push_back(w);
  if (mw.size() + nw.size() != Cw.size()) fail(TN_ERR_ARG, "c_wires must be the uncontracted wires");
  for (int w : mw)
    if (!has(Cw, w)) fail(TN_ERR_ARG, "c_wires misses a wire of A");
  for (int w : nw)
    if (!has(Cw, w)) fail(TN_ERR_ARG, "c_wires misses a wire of B");
  auto pos = [](const std::vector<int>& v, int w) { return (int)(std::find(v.begin(), v.end(), w) - v.begin()); };
  d.nm = (int)mw.size();
  d.nk = (int)kw.size();
  d.nn = (int)nw.size();
  for (int i = 0; i < d.nm; ++i) {
    d.a_mpos[i] = (int8_t)pos(A, mw[i]);
    d.c_mpos[i] = (int8_t)pos(Cw, mw[i]);
  }
  for (int j = 0; j < d.nk; ++j) {
    d.a_kpos[j] = (int8_t)pos(A, kw[j]);
    d.b_kpos[j] = (int8_t)pos(B, kw[j]);
  }
  for (int i = 0; i < d.nn; ++i) {
    d.b_npos[i] = (int8_t)pos(B, nw[i]);
    d.c_npos[i] = (int8_t)pos(Cw, nw[i]);
  }
  d.a_elems = (int64_t)1 << ar;
  d.b_elems = (int64_t)1 << br;
  d.c_elems = (int64_t)1 << cr;
  order_pair_bits(d);
  d.nb = 0;
  const int kid = pick_kernel(precision, cmult, d, batch);
  GemmArgs g = make_args(d, kid, reinterpret_cast<const float2*>(a), reinterpret_cast<const float2*>(b),
                         reinterpret_cast<float2*>(c), (int32_t)batch, d.a_elems, d.b_elems, d.c_elems,
                         is_tc(kid) ? tc_tile(kid, d.nm, d.nk, d.nn, batch, batch * d.c_elems, (int64_t)256 << 20, true)
                                    : -1);
  Scratch& sc = scratch_for_device();
  if (precision == TN_PREC_FP16X3 && is_tc(kid)) {   // operand maxima for the FP16 scaling (one extra read)
    operand_maxima(reinterpret_cast<const float2*>(a), batch << ar, reinterpret_cast<const float2*>(b),
                   batch << br, sc.amax, (cudaStream_t)stream);
    g.amax_a = sc.amax;
    g.amax_b = sc.amax + 1;
  }
  StepLaunch L = make_launch(g, kid, ar, batch, batch * d.c_elems, true);
  if (L.ws_bytes > sc.ws_bytes) {
    CK(cudaStreamSynchronize((cudaStream_t)stream));
    if (sc.ws) CK(cudaFree(sc.ws));
    sc.ws = nullptr;
    CK(cudaMalloc(&sc.ws, (size_t)L.ws_bytes));
    sc.ws_bytes = L.ws_bytes;
  }
  launch_step(L, sc.ws, sc.err, (cudaStream_t)stream, true);
  CK(cudaGetLastError());
  API_END
}

extern "C" tn_status tn_selftest_bounded_wait(int32_t wait_ms, int32_t* device_status, void* stream) {
  API_BEGIN
  if (!device_status) fail(TN_ERR_ARG, "tn_selftest_bounded_wait: NULL argument");
  if (wait_ms < 1 || wait_ms > 5000) fail(TN_ERR_ARG, "tn_selftest_bounded_wait: wait_ms must be in [1, 5000]");
  Scratch& sc = scratch_for_device();
  cudaStream_t s = (cudaStream_t)stream;
  k_selftest_wait<<<1, 32, 0, s>>>(sc.err, (uint64_t)wait_ms * 1000000ull);
  CK(cudaGetLastError());
  int32_t e = 0;
  CK(cudaMemcpyAsync(&e, sc.err, sizeof(e), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  *device_status = e;   // the word stays set until tn_device_sync reads it
  API_END
}

// ---------------------------------------------------------------- no-allocation variant
// Some callers cannot call cudaMalloc at all: code running while a CUDA graph
// is being captured, allocation-free real-time or embedded hosts, and programs
// whose memory pool is owned by someone else.  tn_contract_pair_noalloc serves
// them with the same kernels as tn_contract_pair, taking its scratch (the
// device error word and the B' images of the tensor-core kernels) from this
// file-scope device array instead of allocating it.  Every GPU that loads the
// library holds the array until the process exits.
constexpr size_t kNoAllocScratchBytes = (size_t)32 << 20;   // 32 MiB
constexpr size_t kNoAllocErrBytes = 256;                     // error word, then the B' images
// log2 of the multiply-adds an instance has at least where scratch beyond the array is an error
constexpr int kNoAllocLog2Refused = 20;
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocScratchBytes];

static std::mutex g_noalloc_mu;
static std::unordered_map<int, void*> g_noalloc_addr;   // per device, found once with that device current

static void* noalloc_scratch_address() {
  int dev = 0;
  CK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  auto it = g_noalloc_addr.find(dev);
  if (it != g_noalloc_addr.end()) return it->second;
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess || !p)
    fail(TN_ERR_CUDA, std::string("cudaGetSymbolAddress of the scratch array: ") + cudaGetErrorString(e));
  g_noalloc_addr[dev] = p;
  return p;
}

extern "C" tn_status tn_contract_pair_noalloc(const float* a, const int32_t* aw, int32_t ar, const float* b,
                                              const int32_t* bw, int32_t br, float* c, const int32_t* cw,
                                              int32_t cr, int64_t batch, int32_t precision, int32_t cmult,
                                              void* stream) {
  API_BEGIN
  if (!a || !b || !c || (ar && !aw) || (br && !bw) || (cr && !cw))
    fail(TN_ERR_ARG, "tn_contract_pair_noalloc: NULL argument");
  if (ar < 0 || br < 0 || cr < 0 || ar > 34 || br > 34 || cr > 34)
    fail(TN_ERR_ARG, "tn_contract_pair_noalloc: rank out of range");
  if (batch < 1 || batch > 65535) fail(TN_ERR_ARG, "tn_contract_pair_noalloc: batch must be in [1, 65535]");
  if (precision < TN_PREC_FP32 || precision > TN_PREC_FP16X3) fail(TN_ERR_ARG, "unknown precision");
  if (cmult != 3 && cmult != 4) fail(TN_ERR_ARG, "complex_mult must be 3 or 4");
  if (cmult == 3 && precision == TN_PREC_FP32)
    fail(TN_ERR_UNSUPPORTED, "the FP32 CUDA-core path forms 4M products only; 3M needs TF32 or BF16X3");
  std::vector<int> A(aw, aw + ar), B(bw, bw + br), Cw(cw, cw + cr);
  auto has = [](const std::vector<int>& v, int w) { return std::find(v.begin(), v.end(), w) != v.end(); };
  auto dup = [](const std::vector<int>& v) {
    for (size_t i = 0; i < v.size(); ++i)
      for (size_t j = i + 1; j < v.size(); ++j)
        if (v[i] == v[j]) return true;
    return false;
  };
  if (dup(A) || dup(B) || dup(Cw)) fail(TN_ERR_ARG, "repeated wire in a wire list");
  StepDesc d;
  std::memset(&d, 0, sizeof(d));
  std::vector<int> mw, kw, nw;
  for (int w : A) (has(B, w) ? kw : mw).push_back(w);
  for (int w : B)
    if (!has(A, w)) nw.push_back(w);
  if (mw.size() + nw.size() != Cw.size()) fail(TN_ERR_ARG, "c_wires must be the uncontracted wires");
  for (int w : mw)
    if (!has(Cw, w)) fail(TN_ERR_ARG, "c_wires misses a wire of A");
  for (int w : nw)
    if (!has(Cw, w)) fail(TN_ERR_ARG, "c_wires misses a wire of B");
  auto pos = [](const std::vector<int>& v, int w) { return (int)(std::find(v.begin(), v.end(), w) - v.begin()); };
  d.nm = (int)mw.size();
  d.nk = (int)kw.size();
  d.nn = (int)nw.size();
  for (int i = 0; i < d.nm; ++i) {
    d.a_mpos[i] = (int8_t)pos(A, mw[i]);
    d.c_mpos[i] = (int8_t)pos(Cw, mw[i]);
  }
  for (int j = 0; j < d.nk; ++j) {
    d.a_kpos[j] = (int8_t)pos(A, kw[j]);
    d.b_kpos[j] = (int8_t)pos(B, kw[j]);
  }
  for (int i = 0; i < d.nn; ++i) {
    d.b_npos[i] = (int8_t)pos(B, nw[i]);
    d.c_npos[i] = (int8_t)pos(Cw, nw[i]);
  }
  d.a_elems = (int64_t)1 << ar;
  d.b_elems = (int64_t)1 << br;
  d.c_elems = (int64_t)1 << cr;
  order_pair_bits(d);
  int kid = pick_kernel(precision, cmult, d, batch);
  const int64_t cap = (int64_t)(kNoAllocScratchBytes - kNoAllocErrBytes);
  // bytes left for partial sums beside the B' images, whose size no tile width changes
  int64_t part_cap = cap;
  if (is_tc(kid)) {
    const GemmArgs gw = make_args(d, kid, reinterpret_cast<const float2*>(a), reinterpret_cast<const float2*>(b),
                                  reinterpret_cast<float2*>(c), (int32_t)batch, d.a_elems, d.b_elems, d.c_elems);
    part_cap = std::max<int64_t>(0, cap - (make_launch(gw, kid, ar, batch).ws_bytes + 255) / 256 * 256);
  }
  GemmArgs g = make_args(d, kid, reinterpret_cast<const float2*>(a), reinterpret_cast<const float2*>(b),
                         reinterpret_cast<float2*>(c), (int32_t)batch, d.a_elems, d.b_elems, d.c_elems,
                         is_tc(kid) ? tc_tile(kid, d.nm, d.nk, d.nn, batch, batch * d.c_elems, part_cap, true) : -1);
  uint8_t* base = static_cast<uint8_t*>(noalloc_scratch_address());
  int32_t* err = reinterpret_cast<int32_t*>(base);
  float* amax = reinterpret_cast<float*>(base + 16);   // FP16X3 operand maxima, inside the header
  cudaStream_t s = (cudaStream_t)stream;
  if (precision == TN_PREC_FP16X3 && is_tc(kid)) {
    g.amax_a = amax;
    g.amax_b = amax + 1;
  }
  // split-K as tn_contract_pair chooses it, among the choices whose partial sums
  // fit beside the B' images.  (Chosen against the whole array, 16 partial tiles of 12 x
  // 1024 x 2^14 x 8 did not fit where 8 do, and one pass over k instead took 383 us
  // with an error of 1.1e-4; 8 take 353 us with 1.5e-5.)
  StepLaunch L = make_launch(g, kid, ar, batch, batch * d.c_elems, true, -1, part_cap);
  if (L.ws_bytes > cap) L = make_launch(g, kid, ar, batch);
  // many small instances whose B' images do not fit together: the CUDA cores, which
  // need no scratch (4096 x (128 x 32 x 32): 64 MiB of images)
  if (is_tc(kid) && L.ws_bytes > cap && d.nm + d.nk + d.nn < kNoAllocLog2Refused) {
    kid = pick_simt(d, batch);
    g = make_args(d, kid, g.A, g.B, g.C, (int32_t)batch, d.a_elems, d.b_elems, d.c_elems);
    L = make_launch(g, kid, ar, batch);
  }
  // the documented limit is on the operands, not on the kernel that the step's
  // size selects: what the tensor-core path could not hold is refused from 2^20
  // multiply-adds an instance on (kNoAllocLog2Refused), also where the CUDA cores (no scratch) run it
  if (!is_tc(kid) && precision != TN_PREC_FP32 && d.nm + d.nk + d.nn >= kNoAllocLog2Refused && d.nm >= 4) {
    const int tk = tc_kernel(precision, cmult);
    const GemmArgs gt = make_args(d, tk, reinterpret_cast<const float2*>(a), reinterpret_cast<const float2*>(b),
                                  reinterpret_cast<float2*>(c), (int32_t)batch, d.a_elems, d.b_elems, d.c_elems);
    L.ws_bytes = make_launch(gt, tk, ar, batch).ws_bytes;
  }
  if (L.ws_bytes > cap)
    fail(TN_ERR_ARG, "tn_contract_pair_noalloc: this contraction needs " + std::to_string(L.ws_bytes) +
                         " bytes of scratch; the static array holds " + std::to_string(cap));
  // the error word is zero when the library loads and is cleared by
  // tn_device_sync; kernels only ever set it, so it is not cleared here
  if (g.amax_a)
    operand_maxima(reinterpret_cast<const float2*>(a), batch << ar, reinterpret_cast<const float2*>(b),
                   batch << br, amax, s);
  launch_step(L, base + kNoAllocErrBytes, err, s, true);
  CK(cudaGetLastError());
  API_END
}

// ---------------------------------------------------------------- device error word
// Calls without a plan (tn_contract_pair, tn_contract_pair_noalloc,
// tn_selftest_bounded_wait) leave device-side errors in a per-device word: the
// scratch area's word, and the first word of the static array of the
// no-allocation entry point.  This reads both, clears what was set, and
// allocates nothing: a word that was never created cannot hold an error.
extern "C" tn_status tn_device_sync(void* stream) {
  API_BEGIN
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0;
  CK(cudaGetDevice(&dev));
  int32_t* words[2] = {nullptr, nullptr};
  {
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    auto it = g_scratch.find(dev);
    if (it != g_scratch.end()) words[0] = it->second.err;
  }
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    auto it = g_noalloc_addr.find(dev);
    if (it != g_noalloc_addr.end()) words[1] = static_cast<int32_t*>(it->second);
  }
  int32_t val[2] = {0, 0};
  for (int i = 0; i < 2; ++i)
    if (words[i]) CK(cudaMemcpyAsync(&val[i], words[i], sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  int32_t e = 0;
  for (int i = 0; i < 2; ++i)
    if (val[i] != 0) {
      CK(cudaMemsetAsync(words[i], 0, sizeof(int32_t), s));
      if (e == 0) e = val[i];
    }
  if (e != 0) {
    CK(cudaStreamSynchronize(s));
    const tn_status code = (e == TN_ERR_TIMEOUT || e == TN_ERR_DEVICE || e == TN_ERR_ARG) ? e : TN_ERR_DEVICE;
    fail(code, "a device kernel of a call without a plan reported error " + std::to_string(e) +
                   (e == TN_ERR_TIMEOUT ? " (a bounded wait expired; its result is incomplete)" : ""));
  }
  API_END
}
