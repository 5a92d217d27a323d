// Recursive device-resident partition solve: Stage 1 on the input, the same
// method on the reduced interface system (Stage 2) until it fits one warp
// or the GPU's shared memory (the on-chip solve), then Stage 3
// back up the levels.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <type_traits>
#include <vector>

#include "onchip.cuh"
#include "tps_internal.h"
#include "window_kernels.cuh"

namespace tps {

size_t onchip_exchange_bytes() { return (size_t)4 * 2 * kOcMaxCtas * 8; }
int truncate_rows_max() { return kWinRowsMax; }
int truncate_warp_mb(int R, int h) {
  const int64_t e = (int64_t)R + 2 * (int64_t)h;
  if (R < 2 || h < 0 || e % 32) return 0;
  const int mb = (int)(e / 32);
  return (mb >= kWinBlockMin && mb <= kWinBlockMax) ? mb : 0;
}
size_t truncate_rel_bytes(int64_t n_max, int R, int h, int dtype) {
  const int mb = truncate_warp_mb(R, h);
  if (mb == 0 || n_max <= 0) return 0;
  const int64_t windows = (n_max + R - 1) / R;
  return (size_t)windows * win_rel_rows(mb) * 96 * elem_bytes_red(dtype);
}

// ------------------------------------------------------------------ on-chip solve
struct OcGeom {
  int mt;     // level-0 block rows (odd)
  int64_t p;  // level-0 blocks
  int B;      // level-0 blocks per CTA
  int G;      // CTAs
};

// Blocks of mt rows, B to a CTA; a one-row tail is merged into the block
// before it.  False: more than `ctas_max` CTAs, or more rows than one holds.
template <class Tin>
static bool oc_fits(int64_t n, int mt, int B, int ctas_max, OcGeom& g) {
  if (mt * B >= oc_rows_max<Tin>()) return false;
  int64_t p = (n + mt - 1) / mt;
  if (n - (p - 1) * mt == 1) --p;
  const int64_t G = (p + B - 1) / B;
  if (G > ctas_max) return false;
  g = {mt, p, B, (int)G};
  return true;
}

// One CTA where its longer blocks cost less than the grid barrier and the
// exchange, else the shortest odd block length whose CTAs fit.
template <class Ar, class Tin>
static bool oc_geometry(int64_t n, int ctas_max, OcGeom& g) {
  if (n <= kBaseMax || ctas_max < 1) return false;
  for (int mt = 3; mt <= kOcSoloRows<Ar>; mt += 2)
    if (oc_fits<Tin>(n, mt, kOcBlocks<Ar>, 1, g)) return true;
  for (int B = kOcBlocks<Ar>; B <= kOcThreads; B *= 2)
    for (int mt = 3; mt <= oc_block_rows_max<Tin>(B); mt += 2)
      if (oc_fits<Tin>(n, mt, B, ctas_max, g)) return true;
  return false;
}

// CTAs of k_onchip<Ar, Tin> that can be resident at once on the current
// device (at most kOcMaxCtas), found once per device; 0 if it cannot run.
// (Threads may race to fill an entry; they store the same value.)
template <class Ar, class Tin>
static int oc_ctas_max() {
  static std::atomic<int> cache[kMaxDevices];  // CTAs + 1; 0 = not known yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return 0;
  }
  const int known = cache[dev].load(std::memory_order_acquire);
  if (known > 0) return known - 1;
  int sms = 0, per = 0;
  const size_t smem = OcLayout<Ar, Tin>::kBytes;
  if (cudaFuncSetAttribute(k_onchip<Ar, Tin>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_onchip<Ar, Tin>, kOcThreads,
                                                    smem) != cudaSuccess) {
    cudaGetLastError();
    per = 0;
  }
  const int ctas = std::min(kOcMaxCtas, sms * per);
  cache[dev].store(ctas + 1, std::memory_order_release);
  return ctas;
}

// Solve the system on chip if it fits (used = true), else leave it.  xch:
// onchip_exchange_bytes() of device memory; bar: the barrier's two counters,
// the first zero between solves; test: 0, or to exercise the barrier one CTA
// more awaited than launched, in a cooperative launch (1: it times out) or a
// chained one (2: every CTA gives up and is done again), or every second CTA
// giving up (3); nested: this is another solve's Stage 2; report: see OcShared
// (own_status where given).
template <class Ar, class Tin>
static cudaError_t launch_onchip_raw(int64_t n, const Tin* a, const Tin* b, const Tin* c,
                                     const Tin* d, Tin* x, void* xch, unsigned* bar,
                                     int* status, int test, cudaStream_t s, bool& used,
                                     bool codes, bool nested, bool own_status = false,
                                     int32_t* report = nullptr) {
  used = false;
  OcGeom g;
  if (!oc_geometry<Ar, Tin>(n, oc_ctas_max<Ar, Tin>(), g)) return cudaSuccess;
  using T = typename Ar::T;
  const uintptr_t al = (uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d | (uintptr_t)x;
  const int vec16 = (al % 16) == 0;
  // Two chained launches, or a cooperative one and k_onchip_end: the pair starts
  // sooner, the cooperative launch is short of the look at who gave up.  Measured
  // back to back, us a solve, pair against cooperative: fp64 10007 rows 12.3 /
  // 14.3 and 65536 14.4 / 15.4, double-float 800000 19.2 / 20.5 and as Stage 2 of
  // 3000017 rows 59.9 / 61.5, fp32 1000003 11.2 / 12.3, but as Stage 2 of 256
  // fp32 systems 56.4 / 55.7: fp32 is cooperative there.
  const bool coop =
      test == 1 || (std::is_same<Ar, ArF32>::value && nested && g.G > 1 && test == 0);
  OcShared sh{bar, (unsigned)g.G + (test == 1 || test == 2 ? 1u : 0u), status, report,
              own_status ? 1 : 0, kFirst, test == 3};
  constexpr size_t smem = OcLayout<Ar, Tin>::kBytes;
  cudaError_t e;
  if (coop) {
    sh.mode = kCoop;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.G);
    cfg.blockDim = dim3((unsigned)g.B);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_onchip<Ar, Tin>, n, g.mt, g.p, g.G, a, b, c, d, x,
                           reinterpret_cast<T*>(xch), sh, vec16, codes ? 1 : 0);
    if (e == cudaSuccess) {
      e = launch_chained(k_onchip_end, 1, 1, 0, s, sh);
      if (e != cudaSuccess) cudaMemsetAsync(bar, 0, sizeof(unsigned), s);
    }
  } else {
    if (g.G == 1) sh.mode = kSolo;  // no barrier, nothing to finish
    auto go = [&](int ctas) {
      return launch_chained(k_onchip<Ar, Tin>, (unsigned)ctas, (unsigned)g.B, smem, s, n, g.mt,
                            g.p, g.G, a, b, c, d, x, reinterpret_cast<T*>(xch), sh, vec16,
                            codes ? 1 : 0);
    };
    e = go(g.G);
    if (e == cudaSuccess && g.G > 1) {
      sh.mode = kFinish;
      e = go(std::min(g.G, kOcFinishCtas));
      if (e != cudaSuccess) cudaMemsetAsync(bar, 0, sizeof(unsigned), s);
    }
  }
  if (e == cudaSuccess) used = true;
  return e;
}

// codes: this is level 0 of fp64 inputs in narrower arithmetic (level0_dmax).
template <class Ar, class Tin>
static cudaError_t launch_onchip(tps_plan_s* P, int64_t n, const Tin* a, const Tin* b,
                                 const Tin* c, const Tin* d, Tin* x, cudaStream_t s,
                                 bool& used, bool codes, bool nested) {
  used = false;
  if (P->desc.flags & TPS_NO_ONCHIP) return cudaSuccess;
  if (P->desc.flags & TPS_EXTERNAL_WORKSPACE) {  // the caller may have used it in between
    const cudaError_t e = cudaMemsetAsync(P->ws + 32, 0, 2 * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
  }
  return launch_onchip_raw<Ar, Tin>(n, a, b, c, d, x, P->ws + P->off_xch,
                                    reinterpret_cast<unsigned*>(P->ws + 32), P->d_status,
                                    P->test_onchip, s, used, codes, nested);
}

unsigned* level0_dmax(tps_plan_s* P) {
  const bool on = P->desc.dtype == TPS_F64_DF ||
                  (P->desc.dtype == TPS_MIXED_F32_F64 && !P->codes_off);
  return on ? reinterpret_cast<unsigned*>(P->ws + P->off_dmax) : nullptr;
}

cudaError_t dcode_check(tps_plan_s* P, int64_t count, cudaStream_t s) {
  unsigned* dmax = level0_dmax(P);
  if (!dmax) return cudaSuccess;
  return launch_chained(k_dcode_check, 1, 256, 0, s, dmax, count, P->d_status);
}

Level make_level(int64_t n, int m, int R) {
  // a block longer than the system ends with its last chunk (m identity rows
  // would be swept, one after the other)
  m = (int)std::min<int64_t>(m, (n + R - 1) / R * R);
  Level lv{};
  lv.n = n;
  lv.m = m;
  const int64_t p = (n + m - 1) / m;
  const int64_t last = n - (p - 1) * (int64_t)m;
  lv.p = p;
  lv.k_begin = 0;
  lv.k_end = p;
  lv.bnd = nullptr;
  lv.nbnd = 0;
  lv.llast = (int32_t)last;
  lv.ncap = m - 2 >= R ? (m - 2) / R : 0;  // checkpoint slots of a block
  return lv;
}

size_t build_levels(int64_t n, int m0, int mr, size_t top_elem, size_t red_elem, bool rel,
                    size_t base, std::vector<LevelPlan>& out) {
  out.clear();
  size_t off = base;
  int64_t N = n;
  size_t elem = top_elem;
  int m = m0;
  while (N > kBaseMax) {
    LevelPlan L{};
    L.R = chunk_rows(elem);
    L.lv = make_level(N, m, L.R);
    const int64_t nr = 2 * L.lv.p;
    for (int i = 0; i < 5; ++i) {
      L.off_red[i] = off;
      off = align_up(off + (size_t)nr * red_elem);
    }
    L.rel = rel;
    if (rel) {
      const size_t rows = (size_t)L.lv.p * (size_t)rel_cap(L.lv.m);
      L.off_rel[0] = off;
      off = align_up(off + 2 * rows * red_elem);
      L.off_rel[1] = off;
      off = align_up(off + rows * red_elem);
      L.off_rel[2] = off;
      off = align_up(off + (size_t)L.lv.p * sizeof(int));
    } else {
      const size_t nck = (size_t)L.lv.ncap * (size_t)L.lv.p;
      for (int i = 0; i < 3; ++i) {
        L.off_ck[i] = off;
        off = align_up(off + nck * red_elem);
      }
    }
    out.push_back(L);
    N = nr;
    elem = red_elem;
    m = mr;
  }
  return off;
}

size_t elem_bytes_io(int dtype) { return dtype == TPS_F32 ? 4 : 8; }
size_t elem_bytes_red(int dtype) {
  return (dtype == TPS_F32 || dtype == TPS_MIXED_F32_F64) ? 4 : 8;
}

// ------------------------------------------------------------------ launchers
// 16-byte copies need 16-byte aligned arrays and blocks that start on a
// 16-byte boundary (m a multiple of the 16-byte vector); otherwise the
// kernels copy element by element.
template <class Tin>
static bool vec16_ok(int m, const void* const* ptrs, int n) {
  constexpr int kVec = 16 / (int)sizeof(Tin);
  if (m % kVec) return false;
  for (int i = 0; i < n; ++i)
    if ((uintptr_t)ptrs[i] % 16) return false;
  return true;
}

// The dynamic shared-memory limit is a per-device attribute of a kernel:
// set it once per device (bit `dev` of `done`), from any host thread.
template <class K>
static cudaError_t set_smem(K kernel, size_t smem, std::atomic<uint64_t>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (uint64_t(1) << dev) : 0;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

// Stage 1 streams chunks of K rows (or a multiple) and writes a checkpoint
// every K rows, K being Stage 3's chunk length.
#ifndef TPS_STAGE1_MUL
#define TPS_STAGE1_MUL 1  // Stage-1 chunk rows = K * TPS_STAGE1_MUL / TPS_STAGE1_DIV
#endif
#ifndef TPS_STAGE1_DIV
#define TPS_STAGE1_DIV 1
#endif
// The workspace buffers of a level: reduced system (ra, rb, rc, rd, xr) and
// what Stage 1 leaves for Stage 3, relations or checkpoints.
template <class Tred>
struct LevelBufs {
  Tred* red[5];
  Tred* ck[3];
  RelIO rl;
  LevelBufs(tps_plan_s* P, const LevelPlan& L) {
    for (int i = 0; i < 5; ++i) red[i] = reinterpret_cast<Tred*>(P->ws + L.off_red[i]);
    for (int i = 0; i < 3; ++i)
      ck[i] = L.rel ? nullptr : reinterpret_cast<Tred*>(P->ws + L.off_ck[i]);
    rl = L.rel ? RelIO{P->ws + L.off_rel[0], P->ws + L.off_rel[1],
                       reinterpret_cast<int*>(P->ws + L.off_rel[2]), rel_cap(L.lv.m)}
               : RelIO{nullptr, nullptr, nullptr, 0};
  }
};

// kRef: a fused refinement step (RefineIO rf; fp64 arrays).
template <class Ar, class Tin, class Tred, int K, bool kRef = false>
static cudaError_t launch_stage1(const Level& lv, const Tin* a, const Tin* b, const Tin* c,
                                 const Tin* d, const LevelBufs<Tred>& B, int* status,
                                 cudaStream_t s, RefineIO rf = {}) {
  constexpr int W = kWarpsPerCta;
  constexpr int R = K * TPS_STAGE1_MUL / TPS_STAGE1_DIV;
  const size_t smem = stage1_smem_per_warp<Tin, R, kRef ? 5 : 4>() * W;
  const int64_t warps = (lv.k_end - lv.k_begin + 31) / 32;
  const unsigned grid = (unsigned)((warps + W - 1) / W);
  if (grid == 0) return cudaSuccess;
  const bool rel = B.rl.rel != nullptr;
  const void* ptrs[6] = {a, b, c, d, rf.x, rel ? nullptr : rf.r};
  auto go = [&](auto vec, auto rl) -> cudaError_t {
    static std::atomic<uint64_t> done{0};
    auto k = k_stage1<Ar, Tin, Tred, R, K, W, decltype(vec)::value, kRef, decltype(rl)::value>;
    const cudaError_t e = set_smem(k, smem, done);
    if (e != cudaSuccess) return e;
    return launch_chained(k, grid, 32 * W, smem, s, lv, a, b, c, d, B.red[0], B.red[1], B.red[2],
                          B.red[3], B.ck[0], B.ck[1], B.ck[2], status, rf, B.rl);
  };
  const bool vec = vec16_ok<Tin>(lv.m, ptrs, kRef ? 6 : 4);
  if (rel) return vec ? go(std::true_type{}, std::true_type{})
                      : go(std::false_type{}, std::true_type{});
  return vec ? go(std::true_type{}, std::false_type{}) : go(std::false_type{}, std::false_type{});
}

// d: the right-hand side (a refinement step without relations: the residual).
template <class Ar, class Tin, class Tred, int R, bool kRef = false>
static cudaError_t launch_stage3(const Level& lv, const Tin* a, const Tin* b, const Tin* c,
                                 const Tin* d, const LevelBufs<Tred>& B, Tin* x, int* status,
                                 cudaStream_t s, RefineIO rf = {}) {
  const int64_t warps = (lv.k_end - lv.k_begin + 31) / 32;
  if (warps == 0) return cudaSuccess;
  if (B.rl.rel) {  // from the relations: a, b, c, d are not read again
    const void* xp[1] = {x};
    auto go = [&](auto vec) -> cudaError_t {
      static std::atomic<uint64_t> done{0};
      auto k = k_back<Ar, Tin, Tred, R, decltype(vec)::value, kRef>;
      constexpr size_t bytes = BackTile<Ar, Tin, R, kRef>::kBytes;
      const cudaError_t e = set_smem(k, bytes, done);
      if (e != cudaSuccess) return e;
      return launch_chained(k, (unsigned)warps, 32, bytes, s, lv, B.red[4], x, status, B.rl, rf);
    };
    return vec16_ok<Tin>(lv.m, xp, 1) ? go(std::true_type{}) : go(std::false_type{});
  }
  constexpr int W = kWarpsPerCta;
  const size_t smem = Tile3<Tin, Tred, R, kRef ? 5 : 4>::kBytesPerWarp * W;
  const unsigned grid = (unsigned)((warps + W - 1) / W);
  const void* ptrs[5] = {a, b, c, d, x};
  auto go = [&](auto vec) -> cudaError_t {
    static std::atomic<uint64_t> done{0};
    auto k = k_stage3<Ar, Tin, Tred, R, W, decltype(vec)::value, kRef>;
    const cudaError_t e = set_smem(k, smem, done);
    if (e != cudaSuccess) return e;
    return launch_chained(k, grid, 32 * W, smem, s, lv, a, b, c, d, B.red[4], B.ck[0], B.ck[1],
                          B.ck[2], x, status, rf);
  };
  return vec16_ok<Tin>(lv.m, ptrs, 5) ? go(std::true_type{}) : go(std::false_type{});
}

template <class Ar, class Tin, class Tred>
static cudaError_t run_levels(tps_plan_s* P, const std::vector<LevelPlan>& levels, size_t idx,
                              int64_t n, const Tin* a, const Tin* b, const Tin* c, const Tin* d,
                              Tin* x, cudaStream_t s) {
  if (idx == levels.size()) {
    if (n <= 0) return cudaSuccess;
    return launch_chained(k_base<Ar, Tin, Tin>, 1, 32, 0, s, n, a, b, c, d, x, nullptr, 0,
                          P->d_status, nullptr);
  }
  bool used = false;
  cudaError_t eo = launch_onchip<Ar, Tin>(P, n, a, b, c, d, x, s, used, false, true);
  if (eo != cudaSuccess || used) {
    if (used) {
      P->last_onchip = 2;
      P->last_levels = (int32_t)idx;  // levels launched before the on-chip solve
    }
    return eo;
  }
  const LevelPlan& L = levels[idx];
  constexpr int R = kChunkRows<Tin>;
  const LevelBufs<Tred> B(P, L);
  cudaError_t e = launch_stage1<Ar, Tin, Tred, R>(L.lv, a, b, c, d, B, P->d_status, s);
  if (e != cudaSuccess) return e;
  e = run_levels<Ar, Tred, Tred>(P, levels, idx + 1, 2 * L.lv.p, B.red[0], B.red[1], B.red[2],
                                 B.red[3], B.red[4], s);
  if (e != cudaSuccess) return e;
  return launch_stage3<Ar, Tin, Tred, R>(L.lv, a, b, c, d, B, x, P->d_status, s);
}

// ------------------------------------------------------------------ kernel copies
// Grid-stride copy in 16-byte vectors (both pointers 16-byte aligned) or
// 4-byte words; consecutive threads move consecutive vectors, so every warp
// instruction covers 512 contiguous bytes of both sides.
__global__ void k_copy16(const float4* __restrict__ src, float4* __restrict__ dst, size_t n16,
                         const uint32_t* __restrict__ src_tail, uint32_t* __restrict__ dst_tail,
                         int tail_words) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n16; i += stride)
    dst[i] = src[i];
  if (blockIdx.x == 0 && (int)threadIdx.x < tail_words) dst_tail[threadIdx.x] = src_tail[threadIdx.x];
}
__global__ void k_copy4(const uint32_t* __restrict__ src, uint32_t* __restrict__ dst, size_t n4) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += stride)
    dst[i] = src[i];
}

cudaError_t kernel_copy(void* dst, const void* src, size_t bytes, cudaStream_t s) {
  if (bytes == 0) return cudaSuccess;
  if ((bytes | (uintptr_t)dst | (uintptr_t)src) % 4) return cudaErrorInvalidValue;
  constexpr int kThreads = 256;
  constexpr size_t kMaxBlocks = 152 * 4;  // four CTAs per SM saturate the host link
  if (((uintptr_t)dst | (uintptr_t)src) % 16 == 0) {
    const size_t n16 = bytes / 16;
    const int tail = (int)((bytes % 16) / 4);
    const size_t blocks = std::max<size_t>(1, std::min(kMaxBlocks, (n16 + kThreads - 1) / kThreads));
    k_copy16<<<(unsigned)blocks, kThreads, 0, s>>>(
        static_cast<const float4*>(src), static_cast<float4*>(dst), n16,
        reinterpret_cast<const uint32_t*>(static_cast<const unsigned char*>(src) + n16 * 16),
        reinterpret_cast<uint32_t*>(static_cast<unsigned char*>(dst) + n16 * 16), tail);
  } else {
    const size_t n4 = bytes / 4;
    const size_t blocks = std::max<size_t>(1, std::min(kMaxBlocks, (n4 + kThreads - 1) / kThreads));
    k_copy4<<<(unsigned)blocks, kThreads, 0, s>>>(static_cast<const uint32_t*>(src),
                                                  static_cast<uint32_t*>(dst), n4);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------ dtype dispatch
// Level-0 pieces, used by the device path (with optional stage events) and
// by the chunked host pipeline.
template <class F>
static cudaError_t dispatch(int dtype, F&& f) {
  switch (dtype) {
    case TPS_F64: return f(ArF64{}, (double*)nullptr, (double*)nullptr);
    case TPS_F64_DF: return f(ArDF{}, (double*)nullptr, (float2*)nullptr);
    case TPS_F32: return f(ArF32{}, (float*)nullptr, (float*)nullptr);
    case TPS_MIXED_F32_F64: return f(ArF32{}, (double*)nullptr, (float*)nullptr);
  }
  return cudaErrorInvalidValue;
}

cudaError_t stage1_range(tps_plan_s* P, const LevelPlan& L, int64_t kb, int64_t ke,
                         const void* a, const void* b, const void* c, const void* d,
                         cudaStream_t s) {
  return dispatch(P->desc.dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
    using Ar = decltype(ar);
    using Tin = std::remove_pointer_t<decltype(tin)>;
    using Tred = std::remove_pointer_t<decltype(tred)>;
    constexpr int R = kChunkRows<Tin>;
    Level lv = L.lv;
    lv.k_begin = kb;
    lv.k_end = ke;
    lv.dmax = level0_dmax(P);
    return launch_stage1<Ar, Tin, Tred, R>(lv, (const Tin*)a, (const Tin*)b, (const Tin*)c,
                                           (const Tin*)d, LevelBufs<Tred>(P, L), P->d_status, s);
  });
}

cudaError_t stage3_range(tps_plan_s* P, const LevelPlan& L, int64_t kb, int64_t ke,
                         const void* a, const void* b, const void* c, const void* d, void* x,
                         cudaStream_t s, bool judge) {
  return dispatch(P->desc.dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
    using Ar = decltype(ar);
    using Tin = std::remove_pointer_t<decltype(tin)>;
    using Tred = std::remove_pointer_t<decltype(tred)>;
    constexpr int R = kChunkRows<Tin>;
    Level lv = L.lv;
    lv.k_begin = kb;
    lv.k_end = ke;
    lv.dmax = judge ? level0_dmax(P) : nullptr;
    return launch_stage3<Ar, Tin, Tred, R>(lv, (const Tin*)a, (const Tin*)b, (const Tin*)c,
                                           (const Tin*)d, LevelBufs<Tred>(P, L), (Tin*)x,
                                           P->d_status, s);
  });
}

// One fused refinement step of the mixed solve on level 0 (fp64 arrays,
// fp32 elimination): Stage 1 on the residual of x (written to r), the
// reduced solve, Stage 3 adding the correction to x and raising max2.
cudaError_t refine_step(tps_plan_s* P, const std::vector<LevelPlan>& levels, const double* a,
                        const double* b, const double* c, const double* d, double* x, double* r,
                        unsigned long long* max2, cudaStream_t s) {
  using Ar = ArF32;
  using Tin = double;
  using Tred = float;
  constexpr int R = kChunkRows<Tin>;
  const LevelPlan& L = levels[0];
  const RefineIO rf{x, r, max2};
  const LevelBufs<Tred> B(P, L);
  Level lv = L.lv;
  lv.k_begin = 0;
  lv.k_end = lv.p;
  lv.dmax = nullptr;  // a residual's range codes are not judged
  cudaError_t e = cudaMemsetAsync(max2, 0, 2 * sizeof(unsigned long long), s);
  if (e == cudaSuccess)
    e = launch_stage1<Ar, Tin, Tred, R, true>(lv, a, b, c, d, B, P->d_status, s, rf);
  if (e == cudaSuccess) e = reduced_solve(P, levels, s);
  if (e == cudaSuccess)
    e = launch_stage3<Ar, Tin, Tred, R, true>(lv, a, b, c, r, B, x, P->d_status, s, rf);
  return e;
}

// Stage 2: the recursive solve of level 0's reduced system.
cudaError_t reduced_solve(tps_plan_s* P, const std::vector<LevelPlan>& levels, cudaStream_t s) {
  return dispatch(P->desc.dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
    using Ar = decltype(ar);
    using Tred = std::remove_pointer_t<decltype(tred)>;
    (void)tin;
    const LevelPlan& L = levels[0];
    Tred* red[5];
    for (int i = 0; i < 5; ++i) red[i] = reinterpret_cast<Tred*>(P->ws + L.off_red[i]);
    return run_levels<Ar, Tred, Tred>(P, levels, 1, 2 * L.lv.p, red[0], red[1], red[2], red[3],
                                      red[4], s);
  });
}

// The one-warp solve of a system of at most kBaseMax rows (bnd: first rows
// of packed systems 1.., or null).
cudaError_t base_solve(tps_plan_s* P, int64_t n, const void* a, const void* b, const void* c,
                       const void* d, void* x, cudaStream_t s, const int64_t* bnd,
                       int64_t nbnd) {
  return dispatch(P->desc.dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
    using Ar = decltype(ar);
    using Tin = std::remove_pointer_t<decltype(tin)>;
    (void)tred;
    return launch_chained(k_base<Ar, Tin, Tin>, 1, 32, 0, s, n, (const Tin*)a, (const Tin*)b,
                          (const Tin*)c, (const Tin*)d, (Tin*)x, bnd, nbnd, P->d_status,
                          level0_dmax(P));
  });
}

// TPS_GRAPH: Stage 2 (every level below the top, many small launches)
// touches only workspace buffers, so one captured graph serves every solve
// with the same level geometry; it is replayed as a single launch.
cudaError_t reduced_solve_graph(tps_plan_s* P, const std::vector<LevelPlan>& levels,
                                cudaStream_t s) {
  const Level& L0 = levels[0].lv;
  const int64_t key[12] = {2 * L0.p, (int64_t)levels.size(), P->m_reduced, (int64_t)P->ws,
                           P->desc.dtype, (int64_t)levels[0].off_red[0], levels[0].rel, 0, 0, 0, 0, 0};
  bool same = P->graph != nullptr;
  for (int i = 0; i < 12 && same; ++i) same = P->gkey[i] == key[i];
  if (!same) {
    if (P->graph) {
      cudaGraphExecDestroy(P->graph);
      P->graph = nullptr;
    }
    cudaError_t e = cudaSuccess;
    if (!P->cap_stream) e = cudaStreamCreateWithFlags(&P->cap_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(P->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    const cudaError_t ec = reduced_solve(P, levels, P->cap_stream);
    cudaGraph_t g = nullptr;
    e = cudaStreamEndCapture(P->cap_stream, &g);
    if (ec != cudaSuccess || e != cudaSuccess || !g) {
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      return ec != cudaSuccess ? ec : (e != cudaSuccess ? e : cudaErrorUnknown);
    }
    e = cudaGraphInstantiate(&P->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      P->graph = nullptr;
      return e;
    }
    for (int i = 0; i < 12; ++i) P->gkey[i] = key[i];
    P->graph_onchip = P->last_onchip;
    P->graph_levels = P->last_levels;
  }
  P->last_onchip = P->graph_onchip;
  P->last_levels = P->graph_levels;
  return cudaGraphLaunch(P->graph, s);
}

static tps_status run_solve_direct(tps_plan_s* P, int64_t n, const void* a, const void* b,
                                   const void* c, const void* d, void* x, cudaStream_t s,
                                   const std::vector<LevelPlan>& lv, cudaEvent_t* ev,
                                   const int64_t* bnd, int64_t nbnd);

// TPS_GRAPH without stage events: capture the whole solve on the plan's
// private stream the first time a geometry and set of pointers is seen,
// then replay it as one graph launch.  Everything the captured launches
// read from the host (sizes, pointers, the level plan) is in the key.
static tps_status run_solve_graph(tps_plan_s* P, int64_t n, const void* a, const void* b,
                                  const void* c, const void* d, void* x, cudaStream_t s,
                                  const std::vector<LevelPlan>& lv, const int64_t* bnd,
                                  int64_t nbnd) {
  const int64_t key[16] = {n, (int64_t)a, (int64_t)b, (int64_t)c, (int64_t)d, (int64_t)x,
                           (int64_t)bnd, nbnd, P->m, P->m_reduced, (int64_t)lv.size(),
                           (int64_t)P->ws, P->desc.dtype, (int64_t)P->desc.flags, P->rel, 0};
  bool same = P->solve_graph != nullptr;
  for (int i = 0; i < 16 && same; ++i) same = P->sgkey[i] == key[i];
  if (!same) {
    if (P->solve_graph) {
      cudaGraphExecDestroy(P->solve_graph);
      P->solve_graph = nullptr;
    }
    cudaError_t e = cudaSuccess;
    if (!P->cap_stream) e = cudaStreamCreateWithFlags(&P->cap_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(P->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return TPS_ERR_CUDA;
    const tps_status st = run_solve_direct(P, n, a, b, c, d, x, P->cap_stream, lv, nullptr, bnd,
                                           nbnd);
    cudaGraph_t g = nullptr;
    e = cudaStreamEndCapture(P->cap_stream, &g);
    if (st != TPS_OK || e != cudaSuccess || !g) {
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      return st != TPS_OK ? st : TPS_ERR_CUDA;
    }
    e = cudaGraphInstantiate(&P->solve_graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      P->solve_graph = nullptr;
      return TPS_ERR_CUDA;
    }
    for (int i = 0; i < 16; ++i) P->sgkey[i] = key[i];
    P->sg_onchip = P->last_onchip;
    P->sg_levels = P->last_levels;
  }
  P->last_onchip = P->sg_onchip;
  P->last_levels = P->sg_levels;
  return cudaGraphLaunch(P->solve_graph, s) == cudaSuccess ? TPS_OK : TPS_ERR_CUDA;
}

tps_status run_solve(tps_plan_s* P, int64_t n, const void* a, const void* b, const void* c,
                     const void* d, void* x, cudaStream_t s, const std::vector<LevelPlan>& lv,
                     cudaEvent_t* ev, const int64_t* bnd, int64_t nbnd) {
  if ((P->desc.flags & TPS_GRAPH) && !ev && P->desc.dtype != TPS_MIXED_F32_F64)
    return run_solve_graph(P, n, a, b, c, d, x, s, lv, bnd, nbnd);
  return run_solve_direct(P, n, a, b, c, d, x, s, lv, ev, bnd, nbnd);
}

static tps_status run_solve_direct(tps_plan_s* P, int64_t n, const void* a, const void* b,
                                   const void* c, const void* d, void* x, cudaStream_t s,
                                   const std::vector<LevelPlan>& lv, cudaEvent_t* ev,
                                   const int64_t* bnd, int64_t nbnd) {
  cudaError_t e = cudaSuccess;
  P->last_onchip = 0;
  if (ev) e = cudaEventRecord(ev[0], s);
  bool onchip = false;
  if (e == cudaSuccess && !lv.empty() && nbnd == 0) {  // the whole system on chip
    e = dispatch(P->desc.dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
      using Ar = decltype(ar);
      using Tin = std::remove_pointer_t<decltype(tin)>;
      (void)tred;
      return launch_onchip<Ar, Tin>(P, n, (const Tin*)a, (const Tin*)b, (const Tin*)c,
                                    (const Tin*)d, (Tin*)x, s, onchip,
                                    level0_dmax(P) != nullptr, false);
    });
    if (onchip) {
      P->last_onchip = 1;
      P->last_levels = 0;
    }
  }
  if (onchip) {
    for (int i = 1; i < 3 && e == cudaSuccess && ev; ++i) e = cudaEventRecord(ev[i], s);
  } else if (lv.empty()) {
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[1], s);
    if (e == cudaSuccess) e = base_solve(P, n, a, b, c, d, x, s, bnd, nbnd);
    if (e == cudaSuccess) e = dcode_check(P, nbnd + 1, s);
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[2], s);
  } else {
    if (e == cudaSuccess) e = stage1_range(P, lv[0], 0, lv[0].lv.p, a, b, c, d, s);
    const bool judge = lv[0].rel;  // k_back judges the range codes
    if (e == cudaSuccess && !judge) e = dcode_check(P, nbnd + 1, s);
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[1], s);
    // with stage events (TPS_TRACE) TPS_GRAPH captures Stage 2 alone; without
    // them the whole solve is one graph already (run_solve_graph)
    if (e == cudaSuccess)
      e = ((P->desc.flags & TPS_GRAPH) && ev) ? reduced_solve_graph(P, lv, s)
                                              : reduced_solve(P, lv, s);
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[2], s);
    if (e == cudaSuccess) e = stage3_range(P, lv[0], 0, lv[0].lv.p, a, b, c, d, x, s, judge);
  }
  if (e == cudaSuccess && ev) e = cudaEventRecord(ev[3], s);
  return e == cudaSuccess ? TPS_OK : TPS_ERR_CUDA;
}

// ------------------------------------------------------------------ windowed solve
template <class Ar, class Tin>
static cudaError_t launch_window(tps_plan_s* P, int64_t n, const Tin* a, const Tin* b,
                                 const Tin* c, const Tin* d, Tin* x, cudaStream_t s) {
  static std::atomic<uint64_t> done{0};  // the attribute allows the largest window
  cudaError_t e = set_smem(k_window<Ar, Tin>, WinLayout<Ar, Tin>::bytes(kWinRowsMax), done);
  if (e != cudaSuccess) return e;
  const int R = P->m, h = P->m_reduced;
  const size_t smem = WinLayout<Ar, Tin>::bytes(R + 2 * h);  // this window size
  const int64_t windows = (n + R - 1) / R;
  const uintptr_t al = (uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d | (uintptr_t)x;
  unsigned* bound = reinterpret_cast<unsigned*>(P->ws + 8);
  e = cudaMemsetAsync(bound, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  const float tol = (float)(P->desc.tol > 0.0 ? P->desc.tol : 1e-12);
  k_window<Ar, Tin><<<(unsigned)windows, kWinThreads, smem, s>>>(
      n, R, h, a, b, c, d, x, tol, bound, P->d_status, (al % 16) == 0, level0_dmax(P));
  return cudaGetLastError();
}

// One warp per window (k_wsolve): R + 2 h = 32 mb.
template <class Ar, class Tin, class Tred>
static cudaError_t launch_wsolve(tps_plan_s* P, int64_t n, int mb, const Tin* a, const Tin* b,
                                 const Tin* c, const Tin* d, Tin* x, cudaStream_t s) {
  using T = typename Ar::T;
  const int R = P->m, h = P->m_reduced;
  constexpr int kVec = 16 / (int)sizeof(Tin);
  const uintptr_t al = (uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d | (uintptr_t)x;
  const bool vec = (al % 16) == 0 && mb % kVec == 0 && R % kVec == 0 && h % kVec == 0;
  unsigned* bound = reinterpret_cast<unsigned*>(P->ws + 8);
  cudaError_t e = cudaMemsetAsync(bound, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  const float tol = (float)(P->desc.tol > 0.0 ? P->desc.tol : 1e-12);
  Tred* rel = reinterpret_cast<Tred*>(P->ws + P->off_rel);
  const unsigned windows = (unsigned)((n + R - 1) / R);
  constexpr size_t smem = WinSmem<Tin, Tred, T>::kBytes;
  if (vec)
    k_wsolve<Ar, Tin, Tred, true><<<windows, 32, smem, s>>>(n, R, h, mb, a, b, c, d, x, rel, tol,
                                                            bound, P->d_status, level0_dmax(P));
  else
    k_wsolve<Ar, Tin, Tred, false><<<windows, 32, smem, s>>>(n, R, h, mb, a, b, c, d, x, rel, tol,
                                                             bound, P->d_status, level0_dmax(P));
  return cudaGetLastError();
}

tps_status run_truncated(tps_plan_s* P, int64_t n, const void* a, const void* b, const void* c,
                         const void* d, void* x, cudaStream_t s) {
  P->last_onchip = 0;
  P->last_levels = 0;
  cudaError_t e = cudaSuccess;
  const int mb = truncate_warp_mb(P->m, P->m_reduced);
  if (n <= kBaseMax) {
    e = base_solve(P, n, a, b, c, d, x, s, nullptr, 0);
  } else if (mb > 0) {
    e = dispatch(P->desc.dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
      using Ar = decltype(ar);
      using Tin = std::remove_pointer_t<decltype(tin)>;
      using Tred = std::remove_pointer_t<decltype(tred)>;
      return launch_wsolve<Ar, Tin, Tred>(P, n, mb, (const Tin*)a, (const Tin*)b, (const Tin*)c,
                                          (const Tin*)d, (Tin*)x, s);
    });
  } else {
    e = dispatch(P->desc.dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
      using Ar = decltype(ar);
      using Tin = std::remove_pointer_t<decltype(tin)>;
      (void)tred;
      return launch_window<Ar, Tin>(P, n, (const Tin*)a, (const Tin*)b, (const Tin*)c,
                                    (const Tin*)d, (Tin*)x, s);
    });
  }
  if (e == cudaSuccess) e = dcode_check(P, 1, s);
  return e == cudaSuccess ? TPS_OK : TPS_ERR_CUDA;
}


bool onchip_fits(int dtype, int64_t n) {
  OcGeom g;
  bool fits = n <= kBaseMax;
  if (!fits)
    dispatch(dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
      using Ar = decltype(ar);
      using Tin = std::remove_pointer_t<decltype(tin)>;
      (void)tred;
      fits = oc_geometry<Ar, Tin>(n, oc_ctas_max<Ar, Tin>(), g);
      return cudaSuccess;
    });
  return fits;
}

cudaError_t onchip_solve(int dtype, int64_t n, const void* a, const void* b, const void* c,
                         const void* d, void* x, void* xch, unsigned* bar, int* status,
                         int32_t* report, int test, cudaStream_t s, bool& used) {
  return dispatch(dtype, [&](auto ar, auto* tin, auto* tred) -> cudaError_t {
    using Ar = decltype(ar);
    using Tin = std::remove_pointer_t<decltype(tin)>;
    (void)tred;
    return launch_onchip_raw<Ar, Tin>(n, (const Tin*)a, (const Tin*)b, (const Tin*)c,
                                      (const Tin*)d, (Tin*)x, xch, bar, status, test, s, used,
                                      dtype == TPS_F64_DF, false, true, report);
  });
}

}  // namespace tps
