// Single-pass, on-chip partition solve for systems that fit in the GPU's
// shared memory (the same method as the multi-launch path: Sec. 1 and
// Sec. 2.2 of the paper, blocks eliminated onto their first and last rows,
// a reduced interface system, per-block recovery), in one pass that reads a,
// b, c, d from HBM once and writes x once.
//
//   CTA c owns the consecutive level-0 blocks [c*B, (c+1)*B) of mt rows (one
//   block per thread; mt odd, so a thread's rows start on a different bank
//   than its neighbour's) and loads their rows into shared memory.
//   Stage 1: every thread eliminates its block; the relation
//   beta_j x_j = g_j - al_j f - c_j x_{j+1} of each interior row overwrites
//   that row in place; the block's two interface equations stay in
//   registers.  Neighbouring segments are merged in pairs (the inner l and f
//   eliminated), in the warp by shuffles and then across the warps (every
//   warp the same), until the CTA's own two equations are left; they go to
//   global memory, divided by their diagonals.
//   One grid barrier (bounded wait, see OcMode); a system that fits one CTA
//   has none.
//   Stage 2: every warp solves for its CTA's two values by parallel cyclic
//   reduction over the interface rows around them, which ends once their
//   couplings are 0; where they do not decay in time, the CTA
//   reduces all interface rows (redundantly, so no second barrier).
//   Stage 3: down the merges, then every block back-substitutes from its two
//   interface values through the stored relations, leaving x in the d slots,
//   which go out to global memory in 16-byte pieces.
//
// Bound: latency (load, Stage 1, merges, barrier, Stage 2, merges, Stage 3 in
// series), except for Stage 1 of the larger systems: instruction issue in
// double-float, the fp64 pipe in native fp64.  That pipe takes 64 clocks for
// an instruction of one warp (a dependent one or not), four warps in
// parallel on the four quarters of an SM; so native fp64 takes 2 or 4 warps a
// CTA, and the two equations of a merge are worked out side by side in two
// lanes (18 fp64 instructions instead of 25).
// Measured in clocks (double-float, 256 blocks / fp64, 64 blocks): merges
// up 3300 / 8600, down 1150 / 1450; in shared memory, one barrier a merge, 5000 / 14000
// and 3600 / 4200; by 8-row blocks level by level 8500 / 31000 and 3800 / 6100.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "partition_kernels.cuh"
#include "window_bound.cuh"

namespace tps {

constexpr int kOcThreads = 256;                 // most threads (level-0 blocks) per CTA
constexpr int kOcMaxCtas = 160;                 // interface rows <= 2 * this
constexpr unsigned kOcSpinLimit = 1u << 22;     // grid barrier: polls of ~100 ns each

template <class Tin>
constexpr int oc_mt_max() {  // largest level-0 block (odd)
  return sizeof(Tin) >= 8 ? 23 : 47;
}
// Blocks (threads) per CTA: the fp64 pipe is full with a warp per quarter of
// the SM, and fewer blocks mean fewer merges.  Doubled where the system
// needs it, up to kOcThreads.
template <class Ar>
constexpr int kOcBlocks = 256;
template <>
constexpr int kOcBlocks<ArF64> = 64;
// The longest block for which one CTA alone is taken: a row costs a block
// about 450 (double-float), 130 (fp32) or 850 clocks (fp64), the barrier and
// the exchange 3000 to 4000.
template <class Ar>
constexpr int kOcSoloRows = 9;
template <>
constexpr int kOcSoloRows<ArF32> = 23;
template <>
constexpr int kOcSoloRows<ArF64> = 7;
template <class Tin>
constexpr int oc_rows_max() {  // level-0 rows of one CTA (one merged one-row tail)
  return kOcThreads * oc_mt_max<Tin>() + 1;
}

// The longest (odd) block of a CTA of B blocks.  64 blocks (native fp64) use
// two quarters of the SM's fp64 pipe: kept while the rows are few.
template <class Tin>
constexpr int oc_block_rows_max(int B) {
  return B == 64 ? 7 : ((oc_rows_max<Tin>() - 1) / B - 1) / 2 * 2 + 1;
}

// An interface equation of a segment, from the end whose unknown y has its
// diagonal: w z + b y + i v = d, z the neighbouring segment's nearest unknown,
// v the unknown at the segment's other end.
template <class T>
struct EndEq {
  T w, b, i, d;
};

// Shared-memory layout: level-0 arrays (Tin), the warps' interface equations,
// the interface system twice (T); each part 16-byte aligned.
template <class Ar, class Tin>
struct OcLayout {
  using T = typename Ar::T;
  static constexpr size_t kL0 = ((size_t)oc_rows_max<Tin>() * sizeof(Tin) + 15) / 16 * 16;
  static constexpr size_t kEq = kOcThreads / 32 * 2 * sizeof(EndEq<T>);
  static constexpr size_t kPc = (size_t)2 * kOcMaxCtas * sizeof(T);
  static constexpr size_t kBytes = 4 * kL0 + kEq + 6 * kPc;
};

// Level-0 rows in shared memory (element type Tin); relations stored as T
// in the same 8- or 4-byte slots.
template <class Ar, class Tin>
struct AccL0 {
  using T = typename Ar::T;
  struct Raw {
    Tin v[4];
  };
  Tin* p[4];
  int r0;
  __device__ __forceinline__ Raw load(int r) const {
    return {{p[0][r0 + r], p[1][r0 + r], p[2][r0 + r], p[3][r0 + r]}};
  }
  // a row, scaled and range-checked like the multi-launch path's rows
  __device__ __forceinline__ static void row(const Raw& w, T& av, T& bv, T& cv, T& dv,
                                             RowChk& k) {
    Ar::template row<true>(w.v[0], w.v[1], w.v[2], w.v[3], av, bv, cv, dv, k);
  }
  __device__ __forceinline__ T rel(int k, int r) const {
    return *reinterpret_cast<const T*>(&p[k][r0 + r]);
  }
  __device__ __forceinline__ void set_rel(int k, int r, T v) const {
    *reinterpret_cast<T*>(&p[k][r0 + r]) = v;
  }
  __device__ __forceinline__ void set_x(int r, T v) const { Ar::to(p[3][r0 + r], v); }
};

// Stage 1 on one block of L >= 2 rows: the top-down sweep of k_stage1 (f kept
// symbolic, x_1 = P - Q f - S x_{j+1} carried for the first equation), every
// interior row's relation  beta_j x_j = g_j - al_j f - c_j x_{j+1}  written
// over its a (al), b (1 / beta), c (c) and d (g).  F, E: the block's first
// and last interface equations.  The next row's loads are issued before a
// row is worked on.  (The relations stay undivided: three products a row
// fewer here, one more in oc_bwd, and one rounding fewer in x.)
template <class Ar, class Acc>
__device__ __forceinline__ void oc_fwd(const Acc& A, int L, EndEq<typename Ar::T>& F,
                                       EndEq<typename Ar::T>& E, bool& bad, RowChk& chk) {
  using T = typename Ar::T;
  T a0, b0, c0, d0;
  typename Acc::Raw cur = A.load(0), nxt = A.load(1);
  A.row(cur, a0, b0, c0, d0, chk);
  T rbp = Ar::one(), cprev = Ar::zero(), g = Ar::zero(), al = Ar::neg(Ar::one());  // x_0 = f
  T P = Ar::zero(), Q = Ar::zero(), S = Ar::neg(Ar::one());                        // x_1 = x_1
#pragma unroll 1
  for (int j = 1; j < L; ++j) {
    cur = nxt;
    if (j + 1 < L) nxt = A.load(j + 1);
    T av, bv, cv, dv;
    A.row(cur, av, bv, cv, dv, chk);
    const T ratio = Ar::mul(av, rbp);
    const T beta = Ar::sub_mul_dom(bv, ratio, cprev);
    bad |= Ar::bad_pivot(beta);
    g = Ar::sub_mul(dv, ratio, g);
    al = Ar::neg(Ar::mul(ratio, al));
    if (j == L - 1) {
      E = {cv, beta, al, g};
      break;
    }
    const T rbeta = Ar::rcp(beta);
    const T tt = Ar::mul(S, rbeta);
    P = Ar::sub_mul(P, tt, g);
    Q = Ar::sub_mul(Q, tt, al);
    S = Ar::neg(Ar::mul(tt, cv));
    A.set_rel(0, j, al);
    A.set_rel(1, j, rbeta);
    A.set_rel(2, j, cv);
    A.set_rel(3, j, g);
    rbp = rbeta;
    cprev = cv;
  }
  F = {a0, Ar::sub_mul(b0, c0, Q), Ar::neg(Ar::mul(c0, S)), Ar::sub_mul(d0, c0, P)};
}

// Stage 3 on one block: x_0 = f, x_{L-1} = l, interior rows bottom-up from
// the stored relations; x goes to the d slots.
template <class Ar, class Acc>
__device__ __forceinline__ void oc_bwd(const Acc& A, int L, typename Ar::T f,
                                       typename Ar::T l) {
  using T = typename Ar::T;
  A.set_x(L - 1, l);
  T xn = l;
#pragma unroll 1
  for (int j = L - 2; j >= 1; --j) {
    const T al = A.rel(0, j), rb = A.rel(1, j), cv = A.rel(2, j), g = A.rel(3, j);
    xn = Ar::mul(Ar::sub_mul(Ar::sub_mul(g, al, f), cv, xn), rb);
    A.set_x(j, xn);
  }
  A.set_x(0, f);
}

__device__ __forceinline__ float shfl_v(float v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
__device__ __forceinline__ double shfl_v(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
__device__ __forceinline__ df64 shfl_v(df64 v, int src) {
  return {__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}
template <class T>
__device__ __forceinline__ EndEq<T> shfl_eq(const EndEq<T>& e, int src) {
  return {shfl_v(e.w, src), shfl_v(e.b, src), shfl_v(e.i, src), shfl_v(e.d, src)};
}

// One side of a merge of two neighbouring segments.  near: the equation of
// this segment's inner unknown y, far: of the other segment's (both couple to
// each other through w).  The far unknown is eliminated like a Thomas row
// (no product of two pivots is formed), which leaves
//   y = rel[0] - rel[1] x_own - rel[2] x_other
// in the two outer unknowns; `out`, this segment's outer equation, then
// couples to the other segment's outer unknown.
template <class Ar>
__device__ __forceinline__ void oc_merge(const EndEq<typename Ar::T>& near,
                                         const EndEq<typename Ar::T>& far,
                                         EndEq<typename Ar::T>& out, typename Ar::T (&rel)[3],
                                         bool& bad) {
  using T = typename Ar::T;
  const T k = Ar::mul(near.w, Ar::rcp(far.b));
  const T det = Ar::sub_mul_dom(near.b, k, far.w);
  bad |= Ar::bad_pivot(far.b) | Ar::bad_pivot(det);
  const T rd = Ar::rcp(det);
  rel[0] = Ar::quot(Ar::sub_mul(near.d, k, far.d), det, rd);
  rel[1] = Ar::mul(near.i, rd);
  rel[2] = Ar::neg(Ar::mul(Ar::mul(k, far.i), rd));
  out.b = Ar::sub_mul_dom(out.b, out.i, rel[1]);
  out.d = Ar::sub_mul(out.d, out.i, rel[0]);
  out.i = Ar::neg(Ar::mul(out.i, rel[2]));
}

// The merges of one CTA (nw warps, a power of two; one segment per thread).
// A segment of s lanes has its first equation in its first lane and its last
// one in its last; merging lanes [g, g + s) and [g + s, g + 2s) runs in the
// outer lanes g and g + 2s - 1, each working out its own side (the lanes
// between compute along on the same inner equations and are ignored).  Five
// levels in the warp, then the warps' equations go through shared memory and
// every warp merges them all in its first 2 nw lanes.
template <class Ar>
struct OcMerge {
  using T = typename Ar::T;
  static constexpr int kIn = 5, kAcross = 3;  // levels in a warp, across at most 8
  T rel[kIn + kAcross][3];
  EndEq<T> own;  // after up(): lane 0 the CTA's first equation, lane 2 nw - 1 its last

  __device__ __forceinline__ void level(int s, T (&r)[3], int lane, bool& bad) {
    const int g = lane & ~(2 * s - 1);
    const bool right = (lane & s) != 0;
    const EndEq<T> near = shfl_eq(own, right ? g + s : g + s - 1);
    const EndEq<T> far = shfl_eq(own, right ? g + s - 1 : g + s);
    oc_merge<Ar>(near, far, own, r, bad);
  }
  // F, E: the thread's block (identity rows where it has none); weq: 2 nw
  // equations of shared memory.  Needs every thread.
  __device__ __forceinline__ void up(const EndEq<T>& F, const EndEq<T>& E, EndEq<T>* weq, int nw,
                                     int tid, bool& bad) {
    const int lane = tid & 31;
    const bool right = (lane & 1) != 0;
    const EndEq<T> near = right ? F : E;
    own = right ? E : F;
    oc_merge<Ar>(near, shfl_eq(near, lane ^ 1), own, rel[0], bad);
#pragma unroll
    for (int j = 1; j < kIn; ++j) level(1 << j, rel[j], lane, bad);
    if (lane == 0) weq[2 * (tid >> 5)] = own;
    if (lane == 31) weq[2 * (tid >> 5) + 1] = own;
    __syncthreads();
    own = lane < 2 * nw ? weq[lane] : EndEq<T>{Ar::zero(), Ar::one(), Ar::zero(), Ar::zero()};
#pragma unroll
    for (int j = 0; j < kAcross; ++j)
      if ((1 << j) < nw) level(2 << j, rel[kIn + j], lane, bad);
  }
  __device__ __forceinline__ T expand(int s, const T (&r)[3], int lane, T xv) const {
    const int g = lane & ~(2 * s - 1), e = g + 2 * s - 1;
    const bool right = (lane & s) != 0;
    const T xx = shfl_v(xv, right ? g : e);
    const T y = Ar::sub_mul(Ar::sub_mul(r[0], r[1], xv), r[2], xx);
    const T t = shfl_v(y, right ? e : g);
    return (lane == g + s - 1 || lane == g + s) ? t : xv;
  }
  // The CTA's interface values xv (lane 0: the first, lane 2 nw - 1: the
  // last) down to the thread's block.
  __device__ __forceinline__ void down(T xv, int nw, int tid, T& f, T& l) const {
    const int lane = tid & 31, w = tid >> 5;
#pragma unroll
    for (int j = kAcross - 1; j >= 0; --j)
      if ((1 << j) < nw) xv = expand(2 << j, rel[kIn + j], lane, xv);
    const T fw = shfl_v(xv, 2 * w), lw = shfl_v(xv, 2 * w + 1);
    xv = lane == 31 ? lw : fw;
#pragma unroll
    for (int j = kIn - 1; j >= 1; --j) xv = expand(1 << j, rel[j], lane, xv);
    const T y = Ar::sub_mul(Ar::sub_mul(rel[0][0], rel[0][1], xv), rel[0][2],
                            shfl_v(xv, lane ^ 1));
    const bool right = (lane & 1) != 0;
    f = right ? y : xv;
    l = right ? xv : y;
  }
};

// One step of parallel cyclic reduction on rows x_i = p - u x_{i-s} - v x_{i+s}
// (m, q: the rows at -s and +s): x_i = p' - u' x_{i-2s} - v' x_{i+2s}.
template <class Ar>
__device__ __forceinline__ void oc_pcr(typename Ar::T& p, typename Ar::T& u, typename Ar::T& v,
                                       typename Ar::T pm, typename Ar::T um, typename Ar::T vm,
                                       typename Ar::T pq, typename Ar::T uq, typename Ar::T vq,
                                       bool& bad) {
  using T = typename Ar::T;
  const T det = Ar::sub_mul(Ar::sub_mul(Ar::one(), u, vm), v, uq);
  bad |= Ar::bad_pivot(det);
  const T r = Ar::rcp(det);
  p = Ar::mul(Ar::sub_mul(Ar::sub_mul(p, u, pm), v, pq), r);
  u = Ar::neg(Ar::mul(Ar::mul(u, um), r));
  v = Ar::neg(Ar::mul(Ar::mul(v, vq), r));
}
// The same where u, v, vm and uq are all below 2^-54: det is 1 (native fp64,
// where the strides until the couplings are 0 would take 11 slow instructions
// each: n = 10007 12.7 us, 13.1 with oc_pcr alone, and 12.0 when the couplings
// were dropped below 2^-160, which lost what came through them).
__device__ __forceinline__ void oc_pcr_small(double& p, double& u, double& v, double pm, double um,
                                             double pq, double vq) {
  p = ArF64::sub_mul(ArF64::sub_mul(p, u, pm), v, pq);
  u = ArF64::neg(ArF64::mul(u, um));
  v = ArF64::neg(ArF64::mul(v, vq));
}

// a value of 4 or 8 bytes that another CTA or kernel wrote, read from L2, past
// the (non-coherent) L1, where the program says (volatile: not ahead of a wait)
template <class T>
__device__ __forceinline__ T ld_l2(const T* p) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "element size");
  T r;
  if constexpr (sizeof(T) == 8) {
    unsigned long long v;
    asm volatile("ld.global.cg.u64 %0, [%1];\n" : "=l"(v) : "l"(p) : "memory");
    memcpy(&r, &v, 8);
  } else {
    unsigned v;
    asm volatile("ld.global.cg.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    memcpy(&r, &v, 4);
  }
  return r;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

// How a system of several CTAs is launched.  A cooperative launch keeps all
// CTAs resident for the barrier, but cannot be chained (launch_chained), which
// costs up to 3 us.  The other way is two chained launches: in kFirst a
// CTA that has waited long enough for the others (they may not all be
// resident: another stream's kernel holds SMs) leaves without its x; kFinish,
// kOcFinishCtas CTAs, returns at once if none did, else its CTAs share the rows
// of those that did and do them again, by when every interface equation is
// there.  No CTA waits for one that cannot run.  (launch_onchip_raw chooses.)
// Measured, us a solve with no CTA giving up / all of them (130 us of which is
// the wait), 1, 8 and 32 CTAs: fp64 10007 rows 11.8 / 568, 11.9 / 186, 11.9 / 145;
// double-float 800000 rows 18.9 / 2213, 18.8 / 399, 18.8 / 203.
constexpr int kOcFinishCtas = 32;
enum OcMode : int { kSolo = 0, kCoop = 1, kFirst = 2, kFinish = 3 };
constexpr unsigned kOcPatience = 512;  // kFirst: polls of about 0.3 us

// What the CTAs of one solve share.
struct OcShared {
  unsigned* bar;      // [0] arrivals at the barrier; 0 between solves: whatever they
                      // left there, the solve's last launch clears it (kFinish,
                      // k_onchip_end), so that no solve can spoil a later one;
                      // [1] kFinish's CTAs that are done, cleared by kFirst
  unsigned arrivals;  // what the barrier waits for: G (more only to exercise the timeout)
  int* status;
  int32_t* report;    // with own_status: the solve's tps_status, or null
  int own_status;     // the status word belongs to this solve: cleared at its end
  int mode;           // OcMode
  int leave;          // to exercise kFinish: every second CTA of kFirst does not wait
};

__device__ __forceinline__ void oc_report(const OcShared& sh) {
  if (sh.own_status) {
    const int w = atomicExch(sh.status, 0);
    if (sh.report) *sh.report = status_code(w);
  }
}
// After a cooperative launch: the barrier's counter and the solve's report.
static __global__ void k_onchip_end(OcShared sh) {
  chain_wait();
  *sh.bar = 0u;
  oc_report(sh);
}

// n rows, level-0 blocks of mt rows (p blocks, the last of length in
// [2, mt + 1]), blockDim.x of them per CTA (64, 128 or 256), G CTAs.  xch: 3 x 2G
// values of T (the interface equations), then 3 x G range codes and G flags
// (1: the CTA gave up; kFirst).  vec16: a, b, c, d, x 16-byte aligned.
// codes: judge the system's range (level 0 of fp64 inputs in narrower
// arithmetic).
template <class Ar, class Tin>
__global__ void __launch_bounds__(kOcThreads, 1)
    k_onchip(int64_t n, int mt, int64_t p, int G, const Tin* a, const Tin* b, const Tin* c,
             const Tin* d, Tin* __restrict__ x, typename Ar::T* xch, OcShared sh, int vec16,
             int codes) {
  using T = typename Ar::T;
  using Lay = OcLayout<Ar, Tin>;
  static_assert(sizeof(T) <= sizeof(Tin), "relations are stored in the input slots");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned code_s[2][3];  // this CTA's range codes; CTA 0: the system's
  __shared__ int ok_s;
  __shared__ bool gave_s[kOcMaxCtas];
  Tin* s0[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) s0[k] = reinterpret_cast<Tin*>(smem_raw + k * Lay::kL0);
  EndEq<T>* const weq = reinterpret_cast<EndEq<T>*>(smem_raw + 4 * Lay::kL0);
  T* const pc = reinterpret_cast<T*>(smem_raw + 4 * Lay::kL0 + Lay::kEq);
  const int tid = (int)threadIdx.x, B = (int)blockDim.x, nw = B >> 5, lane = tid & 31;
  const int M = 2 * G, last = 2 * nw - 1;
  unsigned* const xcode = reinterpret_cast<unsigned*>(xch + 3 * M);
  unsigned* const xgave = xcode + 3 * G;
  const Tin* const src[4] = {a, b, c, d};
  constexpr int V = 16 / (int)sizeof(Tin);
  const bool fin = sh.mode == kFinish;
  chain_wait();
  if (sh.mode == kFirst && blockIdx.x == 0 && tid == 0) sh.bar[1] = 0u;
  if (fin) {  // which CTAs gave up, read once for all threads
    if (blockIdx.x == 0 && tid == 0) sh.bar[0] = 0u;
    bool any = false;
    for (int i = tid; i < G; i += B) any |= gave_s[i] = ld_l2(xgave + i) != 0u;
    if (!__syncthreads_or(any)) {
      if (blockIdx.x == 0 && tid == 0) oc_report(sh);
      return;
    }
  }
  int turn = (int)blockIdx.x;  // kFinish: CTAs that gave up until this one's next
#pragma unroll 1
  for (int cta = fin ? 0 : (int)blockIdx.x; cta < (fin ? G : (int)blockIdx.x + 1); ++cta) {
    if (fin) {
      if (!gave_s[cta] || turn-- != 0) continue;
      turn = (int)gridDim.x - 1;
    }
    const int64_t kb = (int64_t)cta * B;
    const int64_t ke = kb + B < p ? kb + B : p;
    const int nb = (int)(ke - kb);
    const int64_t r0 = kb * mt;
    const int64_t r1 = ke == p ? n : ke * mt;
    const int rows = (int)(r1 - r0);

    // ---- load the CTA's rows (r0 * sizeof(Tin) is a multiple of 16)
    const int nv = vec16 ? rows / V : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      for (int i = tid; i < nv; i += B) cp_async<16>(s0[k] + i * V, src[k] + r0 + i * V);
      for (int i = nv * V + tid; i < rows; i += B)
        cp_async<sizeof(Tin)>(s0[k] + i, src[k] + r0 + i);
    }
    cp_async_commit();
    if (tid < 6) code_s[tid / 3][tid % 3] = 0u;
    cp_async_wait<0>();
    __syncthreads();
    // a[0] and c[n-1] are not part of the system
    if (tid == 0 && cta == 0) s0[0][0] = Tin{};
    if (tid == 0 && ke == p) s0[2][rows - 1] = Tin{};
    __syncthreads();

    // ---- Stage 1: one block per thread (past the last block: identity rows)
    bool bad = false;
    int L0len = 0;
    RowChk chk;
    EndEq<T> F{Ar::zero(), Ar::one(), Ar::zero(), Ar::zero()}, E = F;
    if (tid < nb) {
      const int64_t k = kb + tid;
      L0len = k == p - 1 ? (int)(n - k * mt) : mt;
      const AccL0<Ar, Tin> A{{s0[0], s0[1], s0[2], s0[3]}, (int)(k * mt - r0)};
      oc_fwd<Ar>(A, L0len, F, E, bad, chk);
    }
    // the rows' range: a, c, d too large or b invalid; the codes of the
    // system's range are collected per CTA and judged after the barrier
    if (codes) {
      const unsigned dc = __reduce_max_sync(0xffffffffu, chk.dcode());
      const unsigned ec = __reduce_max_sync(0xffffffffu, chk.ecode);
      const unsigned fc = __reduce_max_sync(0xffffffffu, chk.fcode());
      if ((tid & 31) == 0) {
        atomicMax(&code_s[0][0], dc);
        atomicMax(&code_s[0][1], ec);
        atomicMax(&code_s[0][2], fc);
      }
    }
    if (chk.range_bad()) atomicOr(sh.status, ST_RANGE);
    bad |= chk.b_bad();

    // ---- the CTA's own two interface equations, divided by their diagonals:
    // f = p - u l_prev - v l (lane 0),  l = p - u f - v f_next (lane 2 nw - 1)
    OcMerge<Ar> mg;
    mg.up(F, E, weq, nw, tid, bad);
    const T rown = Ar::rcp(mg.own.b);
    const T wn = Ar::mul(mg.own.w, rown), in = Ar::mul(mg.own.i, rown);
    T pv = Ar::mul(mg.own.d, rown), uv = lane == 0 ? wn : in, vv = lane == 0 ? in : wn;
    if (lane == 0 || lane == last) bad |= Ar::bad_pivot(mg.own.b);
    const bool publish = G > 1 && !fin;
    if (publish && (tid == 0 || tid == last)) {
      const int i = 2 * cta + (tid != 0);
      xch[i] = pv;
      xch[M + i] = uv;
      xch[2 * M + i] = vv;
    }
    if (codes && publish && tid == 0) {
#pragma unroll
      for (int q = 0; q < 3; ++q) xcode[q * G + cta] = code_s[0][q];
    }
    if (bad) atomicOr(sh.status, ST_BAD_PIVOT);
    if (tid < 32) __syncwarp();  // lane `last`'s stores before lane 0's release

    // ---- grid barrier; warp 0 wrote all that the other CTAs read
    if (publish) {
      if (tid == 0) {
        red_release_add(sh.bar, 1u);
        int ok = 1;
        unsigned it = 0;
        const unsigned limit = sh.mode == kFirst ? kOcPatience : kOcSpinLimit;
        while (ld_acquire_u32(sh.bar) < sh.arrivals || (sh.leave && (cta & 1))) {
          if (++it > limit) {
            ok = 0;
            if (sh.mode == kCoop) atomicOr(sh.status, ST_TIMEOUT);
            break;
          }
          if (sh.mode == kCoop && it > 64) __nanosleep(100);
        }
        xgave[cta] = ok ? 0u : 1u;
        ok_s = ok;
      }
      __syncthreads();
      if (!ok_s) return;
    }

    // ---- Stage 2.  Lane j takes interface row 2 cta - 15 + j, so the CTA's
    // own rows are lanes 15 and 16 and four strides (1, 2, 4, 8) reach no
    // further than the warp.  Every stride squares the couplings' order; between
    // CTAs of many rows these are 0 already or, underflown, after one or two
    // strides, and then further strides would change nothing.
    if (G > 1) {
      const int i = 2 * cta - 15 + lane;
      const bool in_sys = i >= 0 && i < M;
      pv = in_sys ? ld_l2(xch + i) : Ar::zero();
      uv = in_sys ? ld_l2(xch + M + i) : Ar::zero();
      vv = in_sys ? ld_l2(xch + 2 * M + i) : Ar::zero();
    } else {
      const int src = lane == 16 ? last : 0;
      const T p1 = shfl_v(pv, src), u1 = shfl_v(uv, src), v1 = shfl_v(vv, src);
      const bool own = lane == 15 || lane == 16;
      pv = own ? p1 : Ar::zero();
      uv = own ? u1 : Ar::zero();
      vv = own ? v1 : Ar::zero();
    }
    if (codes && cta == 0 && G > 1) {  // every CTA's codes are in
      for (int i = tid; i < G; i += B) {
#pragma unroll
        for (int q = 0; q < 3; ++q) atomicMax(&code_s[1][q], ld_l2(xcode + q * G + i));
      }
    }
    bool badr = false;
    auto settled = [&]() {
      const unsigned q = __ballot_sync(0xffffffffu, Ar::is_zero(uv) && Ar::is_zero(vv));
      return ((q >> 15) & 3u) == 3u;
    };
    bool done = settled();
#pragma unroll 1
    for (int s = 1; s <= 8 && !done; s <<= 1) {
      const T z = Ar::zero();
      const bool lo = lane >= s, hi = lane + s < 32;
      const T pm = shfl_v(pv, lane - s), um = shfl_v(uv, lane - s), vm = shfl_v(vv, lane - s);
      const T pq = shfl_v(pv, lane + s), uq = shfl_v(uv, lane + s), vq = shfl_v(vv, lane + s);
      bool small = false;
      if constexpr (std::is_same<Ar, ArF64>::value) {
        constexpr unsigned kSmall = (1023u - 54u) << 20;
        small = __all_sync(0xffffffffu, max(Ar::exponent(uv), Ar::exponent(vv)) < kSmall);
        if (small) oc_pcr_small(pv, uv, vv, lo ? pm : z, lo ? um : z, hi ? pq : z, hi ? vq : z);
      }
      if (!small)
        oc_pcr<Ar>(pv, uv, vv, lo ? pm : z, lo ? um : z, lo ? vm : z, hi ? pq : z, hi ? uq : z,
                   hi ? vq : z, badr);
      done = settled();
    }
    T fc = shfl_v(pv, 15), lc = shfl_v(pv, 16);
    // the same in every warp, of which each has read the rows by itself: made
    // so, since the barriers below need it even if another solve on the same
    // exchange rows (a misuse) changed them in between
    if (!(G > 1 ? __syncthreads_and(done) : done)) {  // not weakly coupled nearby
      T* cur = pc;
      T* nxt = pc + 3 * M;
      for (int i = tid; i < 3 * M; i += B) cur[i] = ld_l2(xch + i);
      __syncthreads();
      bool stop = false;
      for (int s = 1; s < M && !stop; s <<= 1) {
        bool quiet = true;
        for (int i = tid; i < M; i += B) {
          const T z = Ar::zero();
          const int im = i - s, iq = i + s;
          const bool lo = im >= 0, hi = iq < M;
          T pi = cur[i], ui = cur[M + i], vi = cur[2 * M + i];
          oc_pcr<Ar>(pi, ui, vi, lo ? cur[im] : z, lo ? cur[M + im] : z, lo ? cur[2 * M + im] : z,
                     hi ? cur[iq] : z, hi ? cur[M + iq] : z, hi ? cur[2 * M + iq] : z, badr);
          nxt[i] = pi;
          nxt[M + i] = ui;
          nxt[2 * M + i] = vi;
          quiet &= Ar::is_zero(ui) && Ar::is_zero(vi);
        }
        stop = __syncthreads_and(quiet);
        T* const t = cur;
        cur = nxt;
        nxt = t;
      }
      fc = cur[2 * cta];
      lc = cur[2 * cta + 1];
    }
    if (badr) atomicOr(sh.status, ST_BAD_PIVOT);

    // ---- Stage 3 down the merges, then the block
    T f, l;
    mg.down(lane == 0 ? fc : lc, nw, tid, f, l);
    if (tid < nb) {
      const int64_t k = kb + tid;
      const AccL0<Ar, Tin> A{{s0[0], s0[1], s0[2], s0[3]}, (int)(k * mt - r0)};
      oc_bwd<Ar>(A, L0len, f, l);
    }
    __syncthreads();

    // ---- x out of the d slots
    for (int i = tid; i < nv; i += B)
      *reinterpret_cast<float4*>(x + r0 + i * V) = *reinterpret_cast<const float4*>(s0[3] + i * V);
    for (int i = nv * V + tid; i < rows; i += B) x[r0 + i] = s0[3][i];
    bool oob = false;
    for (int i = tid; i < rows; i += B) oob |= Ar::out_bad(s0[3][i]);
    if (codes && cta == 0 && tid == 0) {
      const unsigned* q = code_s[G > 1 ? 1 : 0];
      oob |= range_codes_bad(q[0], q[1], q[2]);
    }
    if (oob) atomicOr(sh.status, ST_RANGE);
    if (fin) __syncthreads();  // the next CTA's rows take this one's place
  }
  if (sh.own_status && (fin || sh.mode == kSolo)) {
    __syncthreads();
    if (tid == 0) {
      __threadfence();  // this CTA's status bits before its count
      if (!fin || atomicAdd(sh.bar + 1, 1u) == gridDim.x - 1) oc_report(sh);
    }
  }
}

}  // namespace tps

namespace tps {

// ------------------------------------------------------------------ truncated decoupling
// Not the paper's method: an approximation for strongly dominant systems
// (TPS_TRUNCATE).  Window w keeps rows [wR, wR + R) and is solved, on chip
// in one CTA, as the tridiagonal system on the extended rows
// [wR - h, wR + R + h) (clipped to [0, n)) with the couplings that leave that
// range cut.  With q = max (|a| + |c|) / |b| over the window (cut couplings
// zero) the inverse of the window's matrix decays like q^|i-j|, so the kept
// rows differ from the exact solution by at most
//     (|a_cut| q^dl + |c_cut| q^dr) / ((1 - q) min |b|) * ||x||_inf,
// dl, dr the distances from the kept rows to the two cut ends.  Each window
// publishes that bound (maximum over windows, as the bits of a
// non-negative float) and flags ST_NO_CONVERGENCE where it exceeds `tol`.
constexpr int kWinThreads = 128;
constexpr int kWinRowsMax = 1792;              // extended rows of one window

// Shared memory of a window of at most `rows` extended rows: the warps'
// interface equations first, then four row arrays of `rows` elements.
template <class Ar, class Tin>
struct WinLayout {
  using T = typename Ar::T;
  static constexpr size_t kEq = kWinThreads / 32 * 2 * sizeof(EndEq<T>);
  __host__ __device__ static constexpr size_t l0(int rows) {
    return ((size_t)rows * sizeof(Tin) + 15) / 16 * 16;
  }
  __host__ __device__ static constexpr size_t bytes(int rows) { return kEq + 4 * l0(rows); }
};


// R, h even; one CTA per window.
template <class Ar, class Tin>
__global__ void __launch_bounds__(kWinThreads)
    k_window(int64_t n, int R, int h, const Tin* __restrict__ a, const Tin* __restrict__ b,
             const Tin* __restrict__ c, const Tin* __restrict__ d, Tin* __restrict__ x, float tol,
             unsigned* __restrict__ bound_max, int* __restrict__ status, int vec16,
             unsigned* __restrict__ dmax) {
  using T = typename Ar::T;
  using Lay = WinLayout<Ar, Tin>;
  static_assert(sizeof(T) <= sizeof(Tin), "relations are stored in the input slots");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Tin* s0[4];
  const size_t l0 = Lay::l0(R + 2 * h);
  EndEq<T>* const weq = reinterpret_cast<EndEq<T>*>(smem_raw);
#pragma unroll
  for (int k = 0; k < 4; ++k) s0[k] = reinterpret_cast<Tin*>(smem_raw + Lay::kEq + k * l0);
  __shared__ unsigned q_bits, bmin_key;
  __shared__ Tin cut_s[2];
  const int tid = (int)threadIdx.x;
  const int64_t k0 = (int64_t)blockIdx.x * R;
  const int64_t k1 = k0 + R < n ? k0 + R : n;
  const int64_t e0 = k0 - h > 0 ? k0 - h : 0;
  const int64_t e1 = k1 + h < n ? k1 + h : n;
  const int E = (int)(e1 - e0);

  // ---- load the extended rows (16-byte pieces only where the window start
  // is a whole number of pieces from the 16-byte aligned base)
  const Tin* const src[4] = {a, b, c, d};
  constexpr int V = 16 / (int)sizeof(Tin);
  const int nv = (vec16 && e0 % V == 0) ? E / V : 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    for (int i = tid; i < nv; i += kWinThreads) cp_async<16>(s0[k] + i * V, src[k] + e0 + i * V);
    for (int i = nv * V + tid; i < E; i += kWinThreads)
      cp_async<sizeof(Tin)>(s0[k] + i, src[k] + e0 + i);
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();  // every thread's copies have landed
  if (tid == 0) {
    cut_s[0] = e0 > 0 ? s0[0][0] : Tin{};  // the couplings being cut
    cut_s[1] = e1 < n ? s0[2][E - 1] : Tin{};
    q_bits = 0u;
    bmin_key = 0x7FFFFFFFu;
    s0[0][0] = Tin{};
    s0[2][E - 1] = Tin{};
  }
  __syncthreads();
  // ---- q and min |b| of the window (cut couplings zero): q per row from
  // the scaled row, rounded up; min |b| as the smallest magnitude key
  float qmax = 0.0f;
  unsigned bkey = 0x7FFFFFFFu;
  for (int i = tid; i < E; i += kWinThreads) {
    qmax = fmaxf(qmax, win_row_q(s0[0][i], s0[1][i], s0[2][i]));
    bkey = min(bkey, mag_key(s0[1][i]));
  }
  // truncated parts and fp32 rounding: widen q by a relative 2^-20 margin
  qmax = __fmul_ru(qmax, 1.0f + 9.5367431640625e-07f);
  atomicMax(&q_bits, __float_as_uint(qmax));
  atomicMin(&bmin_key, bkey);
  __syncthreads();  // every row read before Stage 1 overwrites a, b, c in place

  // ---- Stage 1: thread blocks of mt rows (odd) over the E rows, then merges
  int mt = (E + kWinThreads - 1) / kWinThreads;
  if (mt < 3) mt = 3;
  mt |= 1;
  int p = (E + mt - 1) / mt;
  if (p > 1 && E - (p - 1) * mt == 1) --p;  // merge a one-row tail
  bool bad = false;
  RowChk chk;
  const int myL = tid < p ? (tid == p - 1 ? E - tid * mt : mt) : 0;
  EndEq<T> F{Ar::zero(), Ar::one(), Ar::zero(), Ar::zero()}, E2 = F;
  if (tid < p) {
    const AccL0<Ar, Tin> A{{s0[0], s0[1], s0[2], s0[3]}, tid * mt};
    oc_fwd<Ar>(A, myL, F, E2, bad, chk);
  }
  // the rows' range (the system-wide |d / b| test runs after the launch)
  if (dmax) codes_raise_warp(dmax, 0, true, chk);
  if (chk.range_bad()) atomicOr(status, ST_RANGE);
  bad |= chk.b_bad();
  constexpr int kNw = kWinThreads / 32;
  OcMerge<Ar> mg;
  mg.up(F, E2, weq, kNw, tid, bad);
  // ---- the window's two interface equations, with nothing outside:
  // b1 f + i1 l = d1;  i2 f + b2 l = d2, eliminated as two Thomas rows (rows
  // of any scale, e.g. 2^-600, whose determinant would underflow)
  const EndEq<T> qf = shfl_eq(mg.own, 0), ql = shfl_eq(mg.own, 2 * kNw - 1);
  bad |= Ar::bad_pivot(qf.b);
  const T r1 = Ar::rcp(qf.b);
  const T g1 = Ar::mul(qf.i, r1), z1 = Ar::mul(qf.d, r1);
  const T b2p = Ar::sub_mul(ql.b, ql.i, g1);
  bad |= Ar::bad_pivot(b2p);
  const T lw = Ar::mul(Ar::sub_mul(ql.d, ql.i, z1), Ar::rcp(b2p));
  const T fw = Ar::sub_mul(z1, g1, lw);
  T fl, ll;
  mg.down((tid & 31) == 0 ? fw : lw, kNw, tid, fl, ll);
  if (tid < p) {
    const AccL0<Ar, Tin> A{{s0[0], s0[1], s0[2], s0[3]}, tid * mt};
    oc_bwd<Ar>(A, myL, fl, ll);
  }
  if (bad) atomicOr(status, ST_BAD_PIVOT);
  __syncthreads();

  // ---- the kept rows out (16-byte pieces where both the global row k0 and
  // the shared-memory row o are whole pieces from aligned bases)
  const int o = (int)(k0 - e0), K = (int)(k1 - k0);
  const int kv = (vec16 && k0 % V == 0 && o % V == 0) ? K / V : 0;
  for (int i = tid; i < kv; i += kWinThreads)
    *reinterpret_cast<float4*>(x + k0 + i * V) =
        *reinterpret_cast<const float4*>(s0[3] + o + i * V);
  for (int i = kv * V + tid; i < K; i += kWinThreads) x[k0 + i] = s0[3][o + i];
  bool oob = false;
  for (int i = tid; i < K; i += kWinThreads) oob |= Ar::out_bad(s0[3][o + i]);
  if (oob) atomicOr(status, ST_RANGE);

  // ---- the window's truncation bound
  if (tid == 0) {
    const float q = __uint_as_float(q_bits);
    // |a_cut| / min |b| and |c_cut| / min |b|, rounded up (scale-free, so a
    // system scaled anywhere in the input's range gets the same bound)
    float ra, rc;
    if constexpr (sizeof(Tin) == 8) {
      const double bmd = __hiloint2double((int)bmin_key, 0);
      ra = __double2float_ru(__ddiv_ru(fabs((double)cut_s[0]), bmd));
      rc = __double2float_ru(__ddiv_ru(fabs((double)cut_s[1]), bmd));
    } else {
      const float bmf = __uint_as_float(bmin_key);
      ra = __fdiv_ru(fabsf((float)cut_s[0]), bmf);
      rc = __fdiv_ru(fabsf((float)cut_s[1]), bmf);
    }
    float eps;
    if (ra == 0.0f && rc == 0.0f) {
      eps = 0.0f;  // nothing cut
    } else if (!(q < 1.0f) || !(ra < __int_as_float(0x7f800000)) ||
               !(rc < __int_as_float(0x7f800000))) {
      eps = __int_as_float(0x7f800000);
    } else {
      const float num = __fadd_ru(__fmul_ru(ra, powf(q, (float)o)),
                                  __fmul_ru(rc, powf(q, (float)(e1 - k1))));
      eps = __fdiv_ru(num, __fsub_rd(1.0f, q)) * (1.0f + 1e-5f);
    }
    atomicMax(bound_max, __float_as_uint(eps));
    if (!(eps <= tol)) atomicOr(status, ST_NO_CONVERGENCE);
  }
}

}  // namespace tps
