// Stage 1, Stage 3 and the small-system solve of the tridiagonal partition
// method (Sec. 1 and Sec. 2.2 of the paper: per-block elimination onto the
// interface unknowns, a reduced interface solve, per-block recovery).
//
// System: a[i] x[i-1] + b[i] x[i] + c[i] x[i+1] = d[i]; a[0], c[n-1] unused.
// Blocks: block k owns rows k*m .. k*m + m - 1.  The last block's rows past
// the system's end are taken as decoupled identity rows (b that of the last
// row, a = c = d = 0): the loads fill them in shared memory, the stores leave
// them out, and every lane sweeps m rows alike (a last block of its own length
// sent its whole warp through the row-by-row path: 20 us of 87 at n = 3e6).
// The first and last row of each block are its
// interface unknowns f_k and l_k; the reduced system in (f_0, l_0, f_1, ...)
// is tridiagonal: row 2k is block k's "first" equation in (l_{k-1}, f_k, l_k)
// and row 2k+1 its "last" equation in (f_k, l_k, f_{k+1}).
//
// GPU mapping.  One lane owns one block and sweeps it serially (the
// recurrences are first-order); a warp owns 32 consecutive blocks and a CTA
// W warps.  The warp streams its blocks through shared memory in chunks of R
// rows, double buffered: for each of a, b, c, d the warp copies the chunk's
// rows of its 32 blocks with cp.async in 16-byte pieces, consecutive lanes
// taking consecutive pieces of one block (64 contiguous bytes per block for
// fp64), so each copy instruction moves 512 coalesced bytes.  Per-lane piece
// offsets are computed once per kernel.  In shared memory each block's rows
// sit in a slot padded to R + 16/sizeof(element) elements, so the 128-bit
// loads with which a lane reads its own block hit distinct banks across a
// quarter-warp.  Where pointers are not 16-byte aligned (or m is not a
// multiple of the 16-byte vector) the same copies go element by element.
//
// Stage 1 is a single top-down sweep per block.  Writing the interior
// relation after row j as  beta_j x_j + c_j x_{j+1} = g_j - alpha_j f  (a
// forward elimination that keeps f symbolic), the last reduced equation is
// the relation after the block's last row, (alpha, beta, c, g) on
// (f_k, l_k, f_{k+1}).  The first reduced equation needs the first interior
// unknown as a function of f_k and l_k; instead of a second, bottom-up
// sweep, the sweep carries x_1 = P - Q f - S x_{j+1} along, which costs four
// multiply-adds per row and no extra reciprocal.
//
// Stage 3, the ordinary way (kRel, k_back): Stage 1 writes the normalised
// relation x_j = g_j - alpha_j f - c_j x_{j+1} of every interior row, lane by
// lane as it makes them, and Stage 3 back-substitutes from these.  In
// double-float and fp32 alpha and the chain for x_1 are left out once they are
// 0 (underflown: 50 to 80 rows into a block of an ordinary system); native
// fp64 leaves out the chain below 2^-60 and always writes alpha, which Stage 3
// reads only where it may be seen.
// Both sweeps are bound by memory: 49 and 25 bytes a row, at n = 2^25 in
// double-float 268 and 132 us, 91% and 95% of the copy rate (k_stage1 with
// checkpoints 215 us, k_stage3 218 us).  Native fp64 Stage 1 is bound by the
// fp64 pipe: 532 us (k_stage3's half of that work is gone: 490 -> 131 us).
//
// Without the workspace that takes (24 bytes a row), Stage 1 writes the
// relation only at every chunk boundary, as a checkpoint, and k_stage3 walks
// each block's chunks bottom-up: a chunk restarts the forward elimination
// from its checkpoint (with f now known), keeps the R pivots and right-hand
// sides in registers, and back-substitutes from the x of the row below it
// (l_k for the last chunk).  The chunk's x goes back through the
// shared-memory slots and out with the same coalesced piece mapping.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "arith.cuh"
#include "tps.h"

namespace tps {

// ------------------------------------------------------------------ geometry
struct Level {
  int64_t n;        // rows
  int64_t p;        // blocks
  int64_t k_begin;  // blocks this launch processes: [k_begin, k_end)
  int64_t k_end;
  const int64_t* bnd;  // batched systems: first rows of systems 1.., sorted (device)
  int64_t nbnd;        // number of such rows (0: one system)
  int32_t m;        // nominal block length
  int32_t llast;    // rows of block p-1 inside the system, in [1, m]
  int32_t ncap;     // checkpoint slots per block
  int32_t pad;
  // level 0 of fp64 inputs in narrower arithmetic: per system (nbnd + 1
  // of them) the kCodes range codes of its rows (RowChk), raised by Stage 1
  // with atomicMax; null elsewhere
  unsigned* dmax;
};

__device__ __forceinline__ int block_len(const Level& lv, int64_t k) {
  return k == lv.p - 1 ? lv.llast : lv.m;
}

// Systems packed back to back are solved as one system whose couplings are
// cut at every system boundary: a of a system's first row and c of its last
// row are taken as 0, whatever is stored there: they are overwritten in the
// chunk's shared-memory slots (cut_chunk).  A block may straddle
// boundaries; its recurrences then decouple exactly there.  Each lane keeps
// the boundaries that touch its block, bnd[first .. first+cnt).
struct Bounds {
  const int64_t* bnd;
  int64_t first;
  int cnt;
  // first index i with bnd[i] >= v
  __device__ __forceinline__ static int64_t lower(const int64_t* b, int64_t nb, int64_t v) {
    int64_t lo = 0, hi = nb;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (b[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
  }
  // boundaries o with start <= o <= start + len (a start row, or the row
  // after the block's last row)
  __device__ __forceinline__ void init(const Level& lv, int64_t start, int len, bool active) {
    bnd = lv.bnd;
    first = 0;
    cnt = 0;
    if (lv.nbnd == 0 || !active) return;
    first = lower(lv.bnd, lv.nbnd, start);
    cnt = (int)(lower(lv.bnd, lv.nbnd, start + len + 1) - first);
  }
};

// Every kernel of a solve is launched with programmatic stream serialization
// (launch_chained) and starts with this wait, so it is set up while the kernel
// before it in the stream still runs, and goes on once that one has completed
// and its writes are visible: the stream's order as ever, but a boundary
// between two kernels costs about 0.5 us where an ordinary one costs 1.5 us
// and is then rounded up to the next 2.048 us (measured back to back: 1 us of
// work a kernel takes 1.5 against 4.1 us, 5 us of work 5.4 against 8.2).
// The memory such a kernel reads may still change while it runs, which
// const __restrict__ on a parameter would deny: the compiler could then read it
// before the wait.  So its inputs are plain pointers.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Status bits written into the device status word.
enum : int { ST_BAD_PIVOT = 1, ST_NO_CONVERGENCE = 2, ST_TIMEOUT = 4, ST_RANGE = 8 };

// The tps_status of a status word (numeric values of tps.h).
__device__ __forceinline__ int32_t status_code(int w) {
  return (w & ST_BAD_PIVOT) ? TPS_ERR_ZERO_PIVOT
         : (w & ST_TIMEOUT) ? TPS_ERR_TIMEOUT
         : (w & ST_RANGE)   ? TPS_ERR_RANGE
                            : TPS_OK;
}

// Range codes of packed systems: three words per system (RowChk's dcode,
// ecode, fcode maxima).  Raise system `sys`'s codes to v (an atomic only
// where that would change a code; the entries are read from L2).
constexpr int kCodes = 3;
__device__ __forceinline__ void code_raise(unsigned* p, unsigned v) {
  if (v != 0u && __ldcg(p) < v) atomicMax(p, v);
}
__device__ __forceinline__ void codes_raise(unsigned* dmax, int64_t sys, unsigned dc,
                                            unsigned ec, unsigned fc) {
  unsigned* p = dmax + kCodes * sys;
  code_raise(p, dc);
  code_raise(p + 1, ec);
  code_raise(p + 2, fc);
}
// The warp's codes: one set of atomics per warp where every lane is in the
// same system (always for a single system), else per lane.
__device__ __forceinline__ void codes_raise_warp(unsigned* dmax, int64_t sys, bool active,
                                                 const RowChk& k) {
  const unsigned dc = active ? k.dcode() : 0u, ec = active ? k.ecode : 0u,
                 fc = active ? k.fcode() : 0u;
  const int64_t sys0 = __shfl_sync(0xffffffffu, sys, 0);
  if (__all_sync(0xffffffffu, !active || sys == sys0)) {
    const unsigned wd = __reduce_max_sync(0xffffffffu, dc);
    const unsigned we = __reduce_max_sync(0xffffffffu, ec);
    const unsigned wf = __reduce_max_sync(0xffffffffu, fc);
    if ((threadIdx.x & 31) == 0) codes_raise(dmax, sys0, wd, we, wf);
  } else if (active) {
    codes_raise(dmax, sys, dc, ec, fc);
  }
}

// After every row of the level-0 system has been loaded: flag ST_RANGE for
// each system i, i + step, .. < count whose codes are out of range
// (range_codes_bad), and clear the codes for the next solve.
__device__ __forceinline__ void judge_codes(unsigned* dmax, int64_t i, int64_t step,
                                            int64_t count, int* status) {
  bool bad = false;
  for (; i < count; i += step) {
    unsigned* p = dmax + kCodes * i;
    bad |= range_codes_bad(p[0], p[1], p[2]);
    p[0] = p[1] = p[2] = 0u;
  }
  if (bad) atomicOr(status, ST_RANGE);
}
// The same as a launch of its own, one CTA (k_back does it where it follows
// in the same stream: 2 to 3 us less a solve).
static __global__ void __launch_bounds__(256)
    k_dcode_check(unsigned* __restrict__ dmax, int64_t count, int* __restrict__ status) {
  chain_wait();
  judge_codes(dmax, threadIdx.x, blockDim.x, count, status);
}

// ------------------------------------------------------------------ cp.async
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem_dst, const void* gmem_src) {
  const uint32_t s = smem_u32(smem_dst);
  if constexpr (BYTES == 16) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem_src) : "memory");
  } else if constexpr (BYTES == 8) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem_src) : "memory");
  } else {
    static_assert(BYTES == 4, "cp.async size");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem_src) : "memory");
  }
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ------------------------------------------------------------------ warp tile
// NA arrays per buffer: a, b, c, d, and for a refinement step (RefineIO) the
// current x as a fifth.
template <class Tin, int R, int NA = 4>
struct Tile {
  static constexpr int kVec = 16 / (int)sizeof(Tin);  // elements per 16-byte piece
  static_assert(R % kVec == 0, "chunk rows must fill 16-byte pieces");
  static constexpr int kPieces = R / kVec;            // pieces per block and chunk
  static constexpr int kStride = R + kVec;            // padded block slot (16-byte multiple)
  static constexpr int kArr = 32 * kStride;           // one array of one buffer
  static constexpr int kBuf = NA * kArr;
  static constexpr size_t kBytesPerWarp = sizeof(Tin) * 2 * kBuf;
};

// Stage 3 also prefetches each chunk's checkpoint (three values per block)
// with the chunk: per buffer, 3 x 32 values after the warp's two buffers.
template <class Tin, class Tred, int R, int NA = 4>
struct Tile3 : Tile<Tin, R, NA> {
  static constexpr size_t kCkBytesPerBuf = 3 * 32 * sizeof(Tred);
  static constexpr size_t kBytesPerWarp = Tile<Tin, R, NA>::kBytesPerWarp + 2 * kCkBytesPerBuf;
};

// One correction step of mixed-precision iterative refinement, fused into
// the level-0 sweeps (kRef kernels; fp64 arrays).  Stage 1 forms the
// residual r = d - A x of the current iterate in fp64 while it streams the
// rows, eliminates with r as the right-hand side and writes r out; Stage 3,
// given r as its right-hand side, adds the correction delta to x in place
// and raises max2[0] = max |delta|, max2[1] = max |x + delta|, each as the
// bit pattern of a non-negative double (which orders like the value; a NaN
// ranks above +inf).
struct RefineIO {
  const double* x;          // Stage 1: the current iterate (read with its neighbours)
  double* r;                // Stage 1: the residual, written
  unsigned long long* max2; // Stage 3: the two maxima (zeroed before the launch)
};

// The relations of a level's interior rows, x_j = g_j - al_j f - c_j x_{j+1},
// written by Stage 1 and read by k_back in the order in which their lanes own
// them: row j of the nb (32, or the launch's last few) blocks of the warp that
// starts at block k0 is nb consecutive values from (k0 * cap + j * nb).
// na[k0] says how many chunks of the warp have an al that counts (k_stage1).
template <class T>
struct alignas(2 * sizeof(T)) RelRow {
  T c, g;
};
struct RelIO {
  void* rel;  // RelRow<T>
  void* al;   // T
  int* na;    // one per block, used at each warp's first
  int cap;    // rows per block: m, rounded up to 4 (16-byte chunk starts)
};
__host__ __device__ constexpr int rel_cap(int m) { return (m + 3) / 4 * 4; }

// Pieces of the current x a Stage-1 refinement chunk needs: its R rows and
// the next piece (the row below the chunk), i.e. kPieces + 1 pieces filling
// the block's padded slot; piece q = lane + 32 j (j <= kPieces) is piece
// q % (kPieces + 1) of block q / (kPieces + 1).
template <class Tin, int R>
struct XPieceMap {
  using TL = Tile<Tin, R>;
  static constexpr int kP = TL::kPieces + 1;
  int64_t goff[kP];
  int soff[kP];
  int row[kP];
  int len[kP];
  __device__ __forceinline__ void init(const Level& lv, int64_t k0, int nb, int lane) {
#pragma unroll
    for (int j = 0; j < kP; ++j) {
      const int q = lane + 32 * j;
      const int blk = q / kP;
      const int pc = q % kP;
      row[j] = pc * TL::kVec;
      len[j] = blk < nb ? block_len(lv, k0 + blk) : 0;
      goff[j] = (k0 + blk) * (int64_t)lv.m + row[j];
      soff[j] = blk * TL::kStride + row[j];
    }
  }
};

// 16 bytes of consecutive rows (one 128-bit shared access).
template <class Tin>
struct Vec16 {
  Tin v[16 / sizeof(Tin)];
};
template <class Tin>
__device__ __forceinline__ Vec16<Tin> lds16(const Tin* p) {
  Vec16<Tin> r;
  *reinterpret_cast<float4*>(&r) = *reinterpret_cast<const float4*>(p);
  return r;
}

// The pieces lane `lane` copies for every array: piece q = lane + 32 j
// (j < kPieces) is piece q % kPieces of block q / kPieces of the warp.
template <class Tin, int R>
struct PieceMap {
  using TL = Tile<Tin, R>;
  int64_t goff[TL::kPieces];  // element offset of the piece in the arrays (chunk 0)
  int soff[TL::kPieces];      // element offset in a buffer's array
  int row[TL::kPieces];       // first row of the piece within its block (chunk 0)
  int len[TL::kPieces];       // rows of the piece's block, 0 past the last block
  int m;                      // nominal block length (a last block may be shorter)
  __device__ __forceinline__ void init(const Level& lv, int64_t k0, int nb, int lane);
};

template <class Tin, int R>
__device__ __forceinline__ void PieceMap<Tin, R>::init(const Level& lv, int64_t k0, int nb,
                                                       int lane) {
  m = lv.m;
#pragma unroll
  for (int j = 0; j < TL::kPieces; ++j) {
    const int q = lane + 32 * j;
    const int blk = q / TL::kPieces;
    const int pc = q % TL::kPieces;
    row[j] = pc * TL::kVec;
    len[j] = blk < nb ? block_len(lv, k0 + blk) : 0;
    goff[j] = (k0 + blk) * (int64_t)lv.m + row[j];
    soff[j] = blk * TL::kStride + row[j];
  }
}

// Copy rows [row0, row0 + R) of the warp's blocks (clipped to each block's
// length) of src[0..n_arr) into the buffer's arrays.  kVec16: whole pieces
// go as one 16-byte copy (arrays 16-byte aligned, m a multiple of kVec);
// otherwise, and for a block's ragged last piece, element by element.  With
// n_arr = 4 (a, b, c, d) the rows past a short last block become identity
// rows of its last row's scale.
template <class Tin, int R, bool kVec16, class PM>
__device__ __forceinline__ void load_chunk(Tin* buf, const Tin* const* src, int n_arr,
                                           const PM& pm, int row0) {
  using TL = Tile<Tin, R>;
#pragma unroll
  for (int j = 0; j < TL::kPieces; ++j) {
    const int avail = pm.len[j] - (row0 + pm.row[j]);  // rows of this piece in its block
    const int64_t g = pm.goff[j] + row0;
    if (kVec16 && avail >= TL::kVec) {
      for (int t = 0; t < n_arr; ++t) cp_async<16>(buf + t * TL::kArr + pm.soff[j], src[t] + g);
    } else if (avail > 0 || (pm.len[j] > 0 && pm.len[j] < pm.m)) {
#pragma unroll
      for (int v = 0; v < TL::kVec; ++v) {
        if (v < avail) {
          for (int t = 0; t < n_arr; ++t)
            cp_async<sizeof(Tin)>(buf + t * TL::kArr + pm.soff[j] + v, src[t] + g + v);
        } else if (n_arr == 4 && pm.len[j] < pm.m) {
          Tin* const o = buf + pm.soff[j] + v;
          o[0] = o[2 * TL::kArr] = o[3 * TL::kArr] = Tin{};
          cp_async<sizeof(Tin)>(o + TL::kArr, src[1] + (g + avail - 1));
        }
      }
    }
  }
}

// The couplings that leave a system, zeroed in the lane's own slots t of the
// chunk at row0: a[0], c[n-1] (cut_chunk), and at a boundary `o` rows into
// the lane's block a of the row and c of the row above it (cut_boundary).
template <class Tin, int R, int kArr>
__device__ __forceinline__ void cut_chunk(Tin* t, const Level& lv, int64_t k, int row0) {
  if (k == 0 && row0 == 0) t[0] = Tin{};
  if (k == lv.p - 1) {
    const int r = lv.llast - 1 - row0;
    if (r >= 0 && r < R) t[2 * kArr + r] = Tin{};
  }
}
template <class Tin, int R, int kArr>
__device__ __forceinline__ void cut_boundary(Tin* t, int o, int row0) {
  if (o >= row0 && o < row0 + R) t[o - row0] = Tin{};
  if (o > row0 && o <= row0 + R) t[2 * kArr + o - 1 - row0] = Tin{};
}

// Write rows [row0, row0 + R) of the warp's blocks from the buffer's first
// array to x (same piece mapping as the loads).
template <class Tin, int R, bool kVec16>
__device__ __forceinline__ void store_chunk(Tin* __restrict__ x, const Tin* buf,
                                            const PieceMap<Tin, R>& pm, int row0) {
  using TL = Tile<Tin, R>;
#pragma unroll
  for (int j = 0; j < TL::kPieces; ++j) {
    const int avail = pm.len[j] - (row0 + pm.row[j]);
    const int64_t g = pm.goff[j] + row0;
    if (kVec16 && avail >= TL::kVec) {
      *reinterpret_cast<float4*>(x + g) = *reinterpret_cast<const float4*>(buf + pm.soff[j]);
    } else if (avail > 0) {
#pragma unroll
      for (int v = 0; v < TL::kVec; ++v)
        if (v < avail) x[g + v] = buf[pm.soff[j] + v];
    }
  }
}

// Rows [row0, row0 + R] of the current x for the warp's blocks: every row up
// to and including the one below the block (the next block's first row);
// 0 past the array's n rows.
template <class Tin, int R, bool kVec16>
__device__ __forceinline__ void load_xchunk(Tin* buf, const Tin* x, const XPieceMap<Tin, R>& xm,
                                            int row0, int64_t n) {
  using TL = Tile<Tin, R>;
#pragma unroll
  for (int j = 0; j < XPieceMap<Tin, R>::kP; ++j) {
    if (xm.len[j] == 0) continue;
    const int64_t g = xm.goff[j] + row0;
    const int64_t avail = min((int64_t)(xm.len[j] + 1 - (row0 + xm.row[j])), n - g);
    if (kVec16 && avail >= TL::kVec) {
      cp_async<16>(buf + xm.soff[j], x + g);
    } else {
#pragma unroll
      for (int v = 0; v < TL::kVec; ++v) {
        if (v < avail) cp_async<sizeof(Tin)>(buf + xm.soff[j] + v, x + g + v);
        else if (g + v >= n) buf[xm.soff[j] + v] = Tin{};
      }
    }
  }
}

// r = d - (a x_{i-1} + b x_i + c x_{i+1}) in fp64.  Where a or c is 0 (cut at
// a boundary) the x beside it, which may belong to another system, is left out:
// it must not reach this one as 0 * inf.
__device__ __forceinline__ double residual_row(double a, double b, double c, double d, double xm,
                                               double x0, double xp) {
  double r = fma(-b, x0, d);
  r = fma(-a, ArF64::is_zero(a) ? 0.0 : xm, r);
  return fma(-c, ArF64::is_zero(c) ? 0.0 : xp, r);
}
// |v|'s bit pattern from integer operations on the two halves (masking the
// sign of the 64-bit pattern is compiled as an fp64 absolute value, an
// instruction of the slow fp64 pipe: measured 2 of the 3 fp64 instructions
// per row of the refinement's Stage 3)
__device__ __forceinline__ unsigned long long abs_bits(double v) {
  const unsigned hi = (unsigned)__double2hiint(v) & 0x7FFFFFFFu;
  const unsigned lo = (unsigned)__double2loint(v);
  return ((unsigned long long)hi << 32) | lo;
}

// ------------------------------------------------------------------ Stage 1
// Chunk buffers per warp in Stage 1's copy pipeline (2: the next chunk is
// copied while one is processed).
#ifndef TPS_STAGE1_STAGES
#define TPS_STAGE1_STAGES 2
#endif
// kRel compiles its row body twice (with and without the chain), so it is
// unrolled by pairs of 16-byte row groups only: back to back at n = 2^25 in
// double-float four groups take 318 us (instruction fetch), two 289, one 292.
#ifndef TPS_REL_UNROLL
#define TPS_REL_UNROLL 2
#endif
constexpr int kRelUnroll = TPS_REL_UNROLL;
constexpr int kS1Stages = TPS_STAGE1_STAGES;
static_assert(kS1Stages >= 2 && kS1Stages <= 4, "Stage-1 pipeline depth");
// Shared memory of one Stage-1 warp (NA arrays per buffer).
template <class Tin, int R, int NA = 4>
constexpr size_t stage1_smem_per_warp() {
  return Tile<Tin, R, NA>::kBytesPerWarp / 2 * kS1Stages;
}

// R rows per chunk; a checkpoint every K rows (K the chunk length of
// Stage 3; one of R and K divides the other).  kRef: a refinement step
// (RefineIO), the right-hand side being the residual of rf.x.  kRel: every
// interior row's relation goes out (RelIO) for k_back, and no checkpoints.
template <class Ar, class Tin, class Tred, int R, int K, int W, bool kVec16, bool kRef = false,
          bool kRel = false>
__global__ void __launch_bounds__(W * 32)
    k_stage1(Level lv, const Tin* a, const Tin* b, const Tin* c, const Tin* d,
             Tred* __restrict__ ra, Tred* __restrict__ rb, Tred* __restrict__ rc,
             Tred* __restrict__ rd, Tred* __restrict__ ck_gam, Tred* __restrict__ ck_y,
             Tred* __restrict__ ck_v, int* __restrict__ status, RefineIO rf = {}, RelIO rl = {}) {
  using T = typename Ar::T;
  using TL = Tile<Tin, R, kRef ? 5 : 4>;
  constexpr bool kSkip = Ar::kSkipChain || kRel;  // decayed chains are skipped
  constexpr bool kRelF64 = Ar::kSkipChain && kRel;
  constexpr int V = TL::kVec;
  static_assert(!kRef || std::is_same<Tin, double>::value, "refinement steps are fp64");
  static_assert(R % K == 0 || K % R == 0, "chunk rows and checkpoint spacing must nest");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = W == 1 ? 0 : threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t k0 = lv.k_begin + ((int64_t)blockIdx.x * W + warp) * 32;
  if (k0 >= lv.k_end) return;
  const int nb = (int)(lv.k_end - k0 < 32 ? lv.k_end - k0 : 32);
  const int64_t k = k0 + lane;
  const bool active = lane < nb;
  const int L = lv.m;
  const int nch = (L + R - 1) / R;

  Tin* tile = reinterpret_cast<Tin*>(smem_raw) + warp * kS1Stages * TL::kBuf;
  const Tin* const srcs[4] = {a, b, c, d};
  PieceMap<Tin, R> pm;
  pm.init(lv, k0, nb, lane);
  XPieceMap<Tin, R> xpm;
  if constexpr (kRef) xpm.init(lv, k0, nb, lane);
  chain_wait();
  // chunk c goes to buffer c % kS1Stages, one commit group per chunk
  auto fetch = [&](int c) {
    if (c < nch) {
      Tin* buf = tile + (c % kS1Stages) * TL::kBuf;
      load_chunk<Tin, R, kVec16>(buf, srcs, 4, pm, c * R);
      if constexpr (kRef)
        load_xchunk<Tin, R, kVec16>(buf + 4 * TL::kArr, (const Tin*)rf.x, xpm, c * R, lv.n);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int c = 0; c < kS1Stages - 1; ++c) fetch(c);
  const int64_t start = k * (int64_t)lv.m;
  Bounds bd;
  bd.init(lv, start, active ? block_len(lv, k) : 0, active);
  int bj = 0;               // boundaries passed
  int bnext = 0x7FFFFFFF;   // the next one, in rows from the block's first
  if (bd.cnt > 0) bnext = (int)(bd.bnd[bd.first] - start);
  // refinement: x of the row above the current one (the previous block's
  // last row before the block's first row)
  Tin xup = Tin{};
  if constexpr (kRef) {
    if (active && start > 0) xup = rf.x[start - 1];
  }

  // virtual state before row 1 (relation x_0 = f): rbeta = 1, c_prev = 0,
  // g = 0, alpha = -1; first interior unknown x_1 = P - Q f - S x_1 with
  // P = Q = 0, S = -1.
  T rbp = Ar::one(), cprev = Ar::zero(), g = Ar::zero(), al = Ar::neg(Ar::one());
  T P = Ar::zero(), Q = Ar::zero(), S = Ar::neg(Ar::one());
  T a0 = Ar::zero(), b0 = Ar::one(), c0 = Ar::zero(), d0 = Ar::zero();
  T beta = Ar::one(), clast = Ar::zero();
  bool bad = false;
  // range of the rows (fp64 inputs in narrower arithmetic), and the packed
  // system the current row belongs to (for its |d / b| code)
  RowChk chk;
  int64_t sys = lv.nbnd > 0 && active ? bd.first : 0;

  // The first interior unknown's chain (P, Q, S) only adds terms scaled by
  // S, whose magnitude falls by |c / beta| < 1 every row of a strictly
  // diagonally dominant block.  In native fp64 (Ar::kSkipChain), once every
  // lane's |S| is below 2^-60 the rest of the chain is below rounding (of an f
  // no more than 2^60 times smaller than the x it hangs on) and the rows skip it
  // (kChain false); they check |c| <= |beta| instead, so S cannot grow back, and
  // a block where that fails reports a pivot failure (not dominant).
  // The last unknown's coupling to f, al, is never left out.  With kRel the
  // other policies skip too, S and al together, but only once both are 0 in
  // every lane (underflown, or cut off at a system boundary), from where on
  // every term with them is 0: nothing is lost by it.  na: the chunks in which
  // k_back has to read al.
  bool chain = true, nondom = false;
  int na = nch;
  unsigned alex = 0;  // native fp64: the chunk's largest exponent field of al
  // the last row's relation; before row 1, x_0 = f
  T cp = Ar::zero(), gp = Ar::zero(), alp = Ar::neg(Ar::one());

  // one interior row (1 <= row <= L-2).  The product chains alpha and S and
  // the accumulators P and Q are left unnormalised here and renormalised
  // once per chunk (renorm), which bounds their low parts to a few ulps.
  RelRow<T>* const rel = static_cast<RelRow<T>*>(rl.rel) + (kRel ? k0 * rl.cap : 0);
  T* const rel_al = static_cast<T*>(rl.al) + (kRel ? k0 * rl.cap : 0);
  // a row's pivot, right-hand side and coupling to f after the row above it
  auto eliminate = [&](const T av, const T bv, const T dv) {
    if constexpr (kRelF64) {
      beta = Ar::sub_mul_dom(bv, av, cp);
      g = Ar::sub_mul(dv, av, gp);
      al = Ar::mul_neg_nn(av, alp);
    } else {
      const T ratio = Ar::mul_nn(av, rbp);
      beta = Ar::sub_mul_dom(bv, ratio, cprev);
      g = Ar::sub_mul(dv, ratio, g);
      al = Ar::mul_neg_nn(ratio, al);
    }
  };
  auto interior = [&](const T av, const T bv, const T cv, const T dv, auto kChain, int row) {
    if constexpr (kRelF64) {  // in the relations' own terms: one product fewer
      eliminate(av, bv, dv);
      bad |= Ar::bad_pivot(beta);
      const T rbeta = Ar::rcp(beta);
      cp = Ar::mul(cv, rbeta);
      gp = Ar::mul(g, rbeta);
      alp = Ar::mul(al, rbeta);
      alex = max(alex, Ar::exponent(alp));
      const RelRow<T> w{cp, gp};
      if (active) {
        rel[row * nb + lane] = w;
        rel_al[row * nb + lane] = alp;
      }
      if constexpr (decltype(kChain)::value) {
        P = Ar::sub_mul_nn(P, S, gp);
        Q = Ar::sub_mul_nn(Q, S, alp);
        S = Ar::mul_neg_nn(S, cp);
      } else {
        nondom |= !Ar::mag_le(cv, beta);
      }
      return;
    }
    const T ratio = Ar::mul_nn(av, rbp);
    beta = Ar::sub_mul_dom(bv, ratio, cprev);
    g = Ar::sub_mul(dv, ratio, g);
    if constexpr (!kRel || decltype(kChain)::value) al = Ar::mul_neg_nn(ratio, al);
    bad |= Ar::bad_pivot(beta);
    const T rbeta = Ar::rcp(beta);
    if constexpr (kRel) {
      RelRow<T> w;
      if constexpr (sizeof(Tin) == 4) {  // bound by memory: round the quotients once
        w.c = Ar::quot(cv, beta, rbeta);
        w.g = Ar::quot(g, beta, rbeta);
      } else {
        w.c = Ar::mul(cv, rbeta);
        w.g = Ar::mul(g, rbeta);
      }
      if (active) rel[row * nb + lane] = w;
      if constexpr (decltype(kChain)::value) {
        const T aw = Ar::mul(Ar::norm(al), rbeta);
        if (active) rel_al[row * nb + lane] = aw;
        // not from w and aw, which would live longer and cost a tenth of Stage 1
        const T tt = Ar::mul_nn(S, rbeta);
        P = Ar::sub_mul_nn(P, tt, g);
        Q = Ar::sub_mul_nn(Q, tt, al);
        S = Ar::mul_neg_nn(tt, cv);
      }
    } else if constexpr (decltype(kChain)::value) {
      const T tt = Ar::mul_nn(S, rbeta);
      P = Ar::sub_mul_nn(P, tt, g);
      Q = Ar::sub_mul_nn(Q, tt, al);
      S = Ar::mul_neg_nn(tt, cv);
    } else {
      nondom |= !Ar::mag_le(cv, beta);
    }
    rbp = rbeta;
    cprev = cv;
  };
  auto renorm = [&]() {
    al = Ar::norm(al);
    S = Ar::norm(S);
    P = Ar::norm(P);
    Q = Ar::norm(Q);
  };
  // checkpoint after row `row` (a multiple of K minus one), when the next K
  // rows start with an interior row (Stage 3 restarts its chunk there)
  auto checkpoint = [&](int row) {
    if (!kRel && active && row + 1 <= L - 2) {
      const int64_t slot = (int64_t)((row + 1) / K - 1) * lv.p + k;
      Ar::to(ck_gam[slot], Ar::mul(cprev, rbp));
      Ar::to(ck_y[slot], Ar::mul(Ar::norm(g), rbp));
      Ar::to(ck_v[slot], Ar::mul(Ar::norm(al), rbp));
    }
  };

  for (int ch = 0; ch < nch; ++ch) {
    const int row0 = ch * R;
    fetch(ch + kS1Stages - 1);
    cp_async_wait<kS1Stages - 1>();
    __syncwarp();
    Tin* const tb = tile + (ch % kS1Stages) * TL::kBuf;
    Tin* const t = tb + lane * TL::kStride;
    cut_chunk<Tin, R, TL::kArr>(t, lv, k, row0);
    // system boundaries in the lane's rows: the couplings cut, and the codes
    // of its rows (which belong to two systems or more) taken row by row
    const bool split = lv.dmax && bnext < row0 + R;
    unsigned ecode = 0;
    int rdmax = 0;
    bool flushed = false;
    if (bnext <= row0 + R) {
      int r = 0;
      while (bnext <= row0 + R) {
        cut_boundary<Tin, R, TL::kArr>(t, bnext, row0);
        if (bnext == row0 + R) break;
        if (split) {
          for (; r < bnext - row0; ++r) {
            T av, bv, cv, dv;
            Ar::template row<true>(t[r], t[TL::kArr + r], t[2 * TL::kArr + r],
                                   t[3 * TL::kArr + r], av, bv, cv, dv, chk);
          }
          codes_raise(lv.dmax, sys, chk.dcode(), chk.ecode, chk.fcode());
          chk.reset_codes();
        }
        ++sys;
        bnext = ++bj < bd.cnt ? (int)(bd.bnd[bd.first + bj] - start) : 0x7FFFFFFF;
      }
      if (split) {
        for (; r < R && row0 + r < L; ++r) {
          T av, bv, cv, dv;
          Ar::template row<true>(t[r], t[TL::kArr + r], t[2 * TL::kArr + r], t[3 * TL::kArr + r],
                                 av, bv, cv, dv, chk);
        }
        ecode = chk.ecode;
        rdmax = chk.rdmax;
        flushed = chk.flushed;
      }
    }
    // one unrolled body (only row 0 and row R-1 test, warp-uniformly, whether
    // they are the block's f or l row), compiled with and without the first
    // unknown's chain; a last chunk that ends before its R rows (m not a
    // multiple of R) goes row by row
    const bool slow = row0 + R > L;
    auto fast_chunk = [&](auto kChain) {
      const bool first = ch == 0, last = row0 + R == L;
#pragma unroll (kRel ? kRelUnroll : R / V)
      for (int r = 0; r < R; r += V) {
        const Vec16<Tin> xa = lds16(t + r), xb = lds16(t + TL::kArr + r),
                         xc = lds16(t + 2 * TL::kArr + r), xd = lds16(t + 3 * TL::kArr + r);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int rr = r + v;
          Tin din = xd.v[v];
          if constexpr (kRef) {  // the residual of the current x
            const Tin x0 = t[4 * TL::kArr + rr], xdn = t[4 * TL::kArr + rr + 1];
            din = residual_row(xa.v[v], xb.v[v], xc.v[v], din, xup, x0, xdn);
            xup = x0;
            if constexpr (!kRel) t[3 * TL::kArr + rr] = din;
          }
          T av, bv, cv, dv;
          Ar::template row<true>(xa.v[v], xb.v[v], xc.v[v], din, av, bv, cv, dv, chk);
          if (v == 0 && rr == 0 && first) {  // the block's first row: f's equation
            a0 = av; b0 = bv; c0 = cv; d0 = dv;
          } else if (v == V - 1 && rr == R - 1 && last) {  // the block's last row
            eliminate(av, bv, dv);
            clast = cv;
          } else {
            interior(av, bv, cv, dv, kChain, row0 + rr);
            if constexpr (R > K) {  // chunk spans several checkpoint intervals
              if ((rr + 1) % K == 0 && rr + 1 < R) checkpoint(row0 + rr);
            }
          }
        }
      }
    };
    if (!slow) {
      if constexpr (kSkip) {
        if (chain) fast_chunk(std::true_type{});
        else fast_chunk(std::false_type{});
      } else {
        fast_chunk(std::true_type{});
      }
    } else {
#pragma unroll 1
      for (int r = 0; r < R; ++r) {
        const int row = row0 + r;
        if (row < L) {
          Tin din = t[3 * TL::kArr + r];
          if constexpr (kRef) {
            const Tin x0 = t[4 * TL::kArr + r], xdn = t[4 * TL::kArr + r + 1];
            din = residual_row(t[r], t[TL::kArr + r], t[2 * TL::kArr + r], din, xup, x0, xdn);
            xup = x0;
            t[3 * TL::kArr + r] = din;
          }
          T av, bv, cv, dv;
          Ar::template row<true>(t[r], t[TL::kArr + r], t[2 * TL::kArr + r], din, av, bv, cv, dv,
                                 chk);
          if (row == 0) {
            a0 = av; b0 = bv; c0 = cv; d0 = dv;
          } else if (row < L - 1) {
            if (!kSkip || chain) interior(av, bv, cv, dv, std::true_type{}, row);
            else interior(av, bv, cv, dv, std::false_type{}, row);
            if constexpr (R > K) {
              if ((row + 1) % K == 0 && r + 1 < R) checkpoint(row);
            }
          } else {
            eliminate(av, bv, dv);
            clast = cv;
          }
        }
      }
    }
    if (split) {  // the body took the chunk's rows together
      chk.ecode = ecode;
      chk.rdmax = rdmax;
      chk.flushed = flushed;
    }
    renorm();
    // the checkpoint at the chunk's end (row0 + R is a multiple of K when
    // K divides R, and every K / R chunks otherwise)
    if (((row0 + R) % K) == 0) checkpoint(row0 + R - 1);
    if constexpr (Ar::kSkipChain) {
      if (chain) {
        na = ch + 1;
        if (__all_sync(0xffffffffu, !active || Ar::chain_small(S))) {
          chain = false;
          // not even the decayed S: it belongs to the row below this chunk,
          // not to l, which may be another packed system's
          S = Ar::zero();
        }
      } else if (kRel && __any_sync(0xffffffffu, active && alex >= Ar::kLateExponent)) {
        na = ch + 1;
      }
      alex = 0;
    } else if constexpr (kRel) {
      if (chain && __all_sync(0xffffffffu, !active || (Ar::is_zero(S) && Ar::is_zero(al)))) {
        chain = false;
        na = ch + 1;
      }
    }
    if constexpr (kRef && !kRel) {  // the chunk's residual (in the d slots) out
      __syncwarp();
      store_chunk<Tin, R, kVec16>(rf.r, tb + 3 * TL::kArr, pm, row0);
    }
    __syncwarp();  // the buffer is refilled by the next iteration's copies
  }
  bad |= nondom;
  if constexpr (kRel) {
    if (lane == 0) rl.na[k0] = na;
  }
  if (active) {
    bad |= Ar::bad_pivot(beta);
    // first equation of block k, unknowns (l_{k-1}, f_k, l_k)
    Ar::to(ra[2 * k], a0);
    Ar::to(rb[2 * k], Ar::sub_mul(b0, c0, Q));
    Ar::to(rc[2 * k], Ar::neg(Ar::mul(c0, S)));
    Ar::to(rd[2 * k], Ar::sub_mul(d0, c0, P));
    // last equation of block k, unknowns (f_k, l_k, f_{k+1})
    Ar::to(ra[2 * k + 1], al);
    Ar::to(rb[2 * k + 1], beta);
    Ar::to(rc[2 * k + 1], clast);
    Ar::to(rd[2 * k + 1], g);
    if (bad || chk.b_bad()) atomicOr(status, ST_BAD_PIVOT);
    if (chk.range_bad()) atomicOr(status, ST_RANGE);
  }
  if (lv.dmax) codes_raise_warp(lv.dmax, sys, active, chk);
}

// ------------------------------------------------------------------ Stage 3
// kRef: a refinement step (RefineIO): d is the residual Stage 1 wrote, the
// result is added to x in place and the maxima go to rf.max2.
template <class Ar, class Tin, class Tred, int R, int W, bool kVec16, bool kRef = false>
__global__ void __launch_bounds__(W * 32)
    k_stage3(Level lv, const Tin* a, const Tin* b, const Tin* c, const Tin* d, const Tred* xred,
             const Tred* ck_gam, const Tred* ck_y, const Tred* ck_v, Tin* __restrict__ x,
             int* __restrict__ status, RefineIO rf = {}) {
  using T = typename Ar::T;
  using TL = Tile<Tin, R, kRef ? 5 : 4>;
  using TL3 = Tile3<Tin, Tred, R, kRef ? 5 : 4>;
  static_assert(!kRef || std::is_same<Tin, double>::value, "refinement steps are fp64");
  constexpr int V = TL::kVec;
  static_assert(sizeof(T) <= sizeof(Tin), "boundary chunks park T values in Tin slots");
  static_assert(sizeof(Tred) == 4 || sizeof(Tred) == 8, "checkpoint element size");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // CTAs run in the reverse of Stage 1's order: the rows Stage 1 read last
  // are the ones still in L2 (and the next solve's Stage 1 starts on the
  // rows this one read last)
  const int64_t k0 = lv.k_begin + ((int64_t)(gridDim.x - 1 - blockIdx.x) * W + warp) * 32;
  if (k0 >= lv.k_end) return;
  const int nb = (int)(lv.k_end - k0 < 32 ? lv.k_end - k0 : 32);
  const int64_t k = k0 + lane;
  const bool active = lane < nb;
  const int L = lv.m;
  const int len = active ? block_len(lv, k) : 0;  // rows inside the system
  const int nch = (L + R - 1) / R;

  unsigned char* wbase = smem_raw + warp * TL3::kBytesPerWarp;
  Tin* tile = reinterpret_cast<Tin*>(wbase);
  Tred* ckbuf = reinterpret_cast<Tred*>(wbase + TL::kBytesPerWarp);  // [buf][3][32]
  const Tin* const srcs[4] = {a, b, c, d};
  const Tin* const xsrc[1] = {x};  // refinement: the current iterate, a fifth array
  PieceMap<Tin, R> pm;
  pm.init(lv, k0, nb, lane);
  // the lane's checkpoint for chunk ch (written by Stage 1 after row ch*R-1)
  auto load_ck = [&](Tred* dst, int ch) {
    if (active && ch > 0 && ch * R <= L - 2) {
      const int64_t slot = (int64_t)(ch - 1) * lv.p + k;
      cp_async<sizeof(Tred)>(dst + lane, ck_gam + slot);
      cp_async<sizeof(Tred)>(dst + 32 + lane, ck_y + slot);
      cp_async<sizeof(Tred)>(dst + 64 + lane, ck_v + slot);
    }
  };
  chain_wait();
  load_chunk<Tin, R, kVec16>(tile, srcs, 4, pm, (nch - 1) * R);
  if constexpr (kRef) load_chunk<Tin, R, kVec16>(tile + 4 * TL::kArr, xsrc, 1, pm, (nch - 1) * R);
  load_ck(ckbuf, nch - 1);
  cp_async_commit();
  unsigned long long mdel = 0, mx = 0;  // refinement maxima (bit patterns)

  const int64_t start = k * (int64_t)lv.m;
  Bounds bd;
  bd.init(lv, start, len, active);
  T f = Ar::zero(), l = Ar::zero();
  if (active) {
    f = Ar::from(xred[2 * k]);
    l = Ar::from(xred[2 * k + 1]);
  }
  T xnext = l;  // x of the row below the chunk being processed
  bool bad = false, oob = false;
  RowChk nochk;  // the rows' range was checked by Stage 1

  // chunks bottom-up: ch = nch-1 .. 0; buffer parity follows the visiting order
  for (int it = 0; it < nch; ++it) {
    const int ch = nch - 1 - it;
    const int row0 = ch * R;
    if (ch > 0) {
      load_chunk<Tin, R, kVec16>(tile + ((it + 1) & 1) * TL::kBuf, srcs, 4, pm, row0 - R);
      if constexpr (kRef)
        load_chunk<Tin, R, kVec16>(tile + ((it + 1) & 1) * TL::kBuf + 4 * TL::kArr, xsrc, 1, pm,
                                   row0 - R);
      load_ck(ckbuf + ((it + 1) & 1) * 96, ch - 1);
    }
    cp_async_commit();
    cp_async_wait<1>();
    __syncwarp();
    Tin* tb = tile + (it & 1) * TL::kBuf;
    Tin* t = tb + lane * TL::kStride;

    // relation entering the chunk: x_{row0-1} = zp - gp * x_{row0}
    T zp = f, gp = Ar::zero();
    if (active && ch > 0 && row0 <= L - 2) {
      const Tred* ck = ckbuf + (it & 1) * 96;
      gp = Ar::from(ck[lane]);
      zp = Ar::sub_mul(Ar::from(ck[32 + lane]), Ar::from(ck[64 + lane]), f);
    }
    cut_chunk<Tin, R, TL::kArr>(t, lv, k, row0);
    for (int j = 0; j < bd.cnt; ++j)
      cut_boundary<Tin, R, TL::kArr>(t, (int)(bd.bnd[bd.first + j] - start), row0);
    if (row0 + R <= L) {
      // unrolled chunk: forward over the interior rows, back-substitution
      // from the row below; only row 0 (f) and row R-1 (l) test their role,
      // warp-uniformly
      const bool first = ch == 0, last = row0 + R == L;
      T Z[R], G[R];
      Tin xo[R];
#pragma unroll
      for (int r = 0; r < R; r += V) {
        const Vec16<Tin> xa = lds16(t + r), xb = lds16(t + TL::kArr + r),
                         xc = lds16(t + 2 * TL::kArr + r), xd = lds16(t + 3 * TL::kArr + r);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int rr = r + v;
          if ((rr == 0 && first) || (rr == R - 1 && last)) continue;
          T av, bv, cv, dv;
          Ar::template row<false>(xa.v[v], xb.v[v], xc.v[v], xd.v[v], av, bv, cv, dv, nochk);
          const T beta = Ar::sub_mul_dom(bv, av, gp);
          bad |= Ar::bad_pivot(beta);
          const T rbeta = Ar::rcp(beta);
          zp = Ar::mul_nn(Ar::sub_mul(dv, av, zp), rbeta);
          gp = Ar::mul_nn(cv, rbeta);
          Z[rr] = zp;
          G[rr] = gp;
        }
      }
      // back-substitution (x over the Z slots), then the output conversion
#pragma unroll
      for (int r = R - 1; r >= 0; --r) {
        if (r == R - 1 && last) {
          Z[r] = l;  // xnext is l already
        } else if (r == 0 && first) {
          Z[r] = f;
        } else {
          xnext = Ar::sub_mul(Z[r], G[r], xnext);
          Z[r] = xnext;
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        Ar::to(xo[r], Z[r]);
        oob |= Ar::out_bad(xo[r]);
        if constexpr (kRef) {  // x += delta
          const Tin xn = t[4 * TL::kArr + r] + xo[r];
          if (row0 + r < len) {
            mdel = max(mdel, abs_bits(xo[r]));
            mx = max(mx, abs_bits(xn));
          }
          xo[r] = xn;
        }
      }
#pragma unroll
      for (int r = 0; r < R; r += V) {
        Vec16<Tin> w;
#pragma unroll
        for (int v = 0; v < V; ++v) w.v[v] = xo[r + v];
        *reinterpret_cast<float4*>(t + r) = *reinterpret_cast<const float4*>(&w);
      }
    } else {
      // a last chunk that ends before its R rows: the same recurrences, row by
      // row, with the pivots and right-hand sides parked in the lane's b and c
      // slots
      T* zs = reinterpret_cast<T*>(t + TL::kArr);
      T* gs = reinterpret_cast<T*>(t + 2 * TL::kArr);
#pragma unroll 1
      for (int r = 0; r < R; ++r) {
        const int row = row0 + r;
        if (row >= 1 && row <= L - 2) {
          T av, bv, cv, dv;
          Ar::template row<false>(t[r], t[TL::kArr + r], t[2 * TL::kArr + r],
                                  t[3 * TL::kArr + r], av, bv, cv, dv, nochk);
          const T beta = Ar::sub_mul_dom(bv, av, gp);
          bad |= Ar::bad_pivot(beta);
          const T rbeta = Ar::rcp(beta);
          zp = Ar::mul_nn(Ar::sub_mul(dv, av, zp), rbeta);
          gp = Ar::mul_nn(cv, rbeta);
          zs[r] = zp;
          gs[r] = gp;
        }
      }
#pragma unroll 1
      for (int r = R - 1; r >= 0; --r) {
        const int row = row0 + r;
        if (row < L) {
          T xr;
          if (row == 0) {
            xr = f;
          } else if (row == L - 1) {
            xr = l;
          } else {
            xr = Ar::sub_mul(zs[r], gs[r], xnext);
            xnext = xr;
          }
          Ar::to(t[r], xr);
          oob |= Ar::out_bad(t[r]);
          if constexpr (kRef) {  // x += delta
            const Tin xn = t[4 * TL::kArr + r] + t[r];
            if (row < len) {
              mdel = max(mdel, abs_bits(t[r]));
              mx = max(mx, abs_bits(xn));
            }
            t[r] = xn;
          }
        }
      }
    }
    // the chunk's x is in the lanes' a slots (a is no longer needed): out
    __syncwarp();
    store_chunk<Tin, R, kVec16>(x, tb, pm, row0);
    __syncwarp();  // the buffer is refilled by the next iteration's copies
  }
  if (active && bad) atomicOr(status, ST_BAD_PIVOT);
  if (active && oob) atomicOr(status, ST_RANGE);
  if constexpr (kRef) {
    for (int o = 16; o > 0; o >>= 1) {
      mdel = max(mdel, __shfl_xor_sync(0xffffffffu, mdel, o));
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    // most warps see maxima already raised past theirs: read before the atomic
    if (lane == 0) {
      if (mdel > *(volatile unsigned long long*)&rf.max2[0]) atomicMax(&rf.max2[0], mdel);
      if (mx > *(volatile unsigned long long*)&rf.max2[1]) atomicMax(&rf.max2[1], mx);
    }
  }
}

// ------------------------------------------------------------------ Stage 3 from relations
// Back-substitution of every block from its two interface values through the
// relations Stage 1 wrote (kRel): one multiply-add a row where k_stage3
// repeats the elimination, and 24 bytes a row (2 values of a relation in, x
// out; fp32 12) where k_stage3 moves 40.  Bound by those bytes, so what
// counts is how many are on their way: a chunk's relations are one contiguous
// piece of memory, copied with cp.async kBackStages - 1 chunks ahead.
// Where lv.dmax is given, the range codes Stage 1 raised are judged on the way.
// kRef: the result is added to x in place and the maxima go to rf.max2.
#ifndef TPS_BACK_STAGES
#define TPS_BACK_STAGES 3
#endif
constexpr int kBackStages = TPS_BACK_STAGES;
template <class Ar, class Tin, int R, bool kRef>
struct BackTile {
  using T = typename Ar::T;
  static constexpr size_t kRows = (size_t)32 * R * sizeof(RelRow<T>);
  static constexpr size_t kAl = (size_t)32 * R * sizeof(T);
  static constexpr size_t kX = Tile<Tin, R, 1>::kArr * sizeof(Tin);
  static constexpr size_t kStage = kRows + kAl + (kRef ? kX : 0);
  static constexpr size_t kBytes = kBackStages * kStage + (kRef ? 0 : kX);
};
template <class Ar, class Tin, class Tred, int R, bool kVec16, bool kRef = false>
__global__ void __launch_bounds__(32)
    k_back(Level lv, const Tred* xred, Tin* __restrict__ x, int* __restrict__ status,
           RelIO rl, RefineIO rf) {
  using T = typename Ar::T;
  using TL = Tile<Tin, R, 1>;
  using BT = BackTile<Ar, Tin, R, kRef>;
  constexpr int V = TL::kVec;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x;
  // the reverse of Stage 1's order: its last relations are still in L2
  const int64_t k0 = lv.k_begin + (int64_t)(gridDim.x - 1 - blockIdx.x) * 32;
  const int nb = (int)(lv.k_end - k0 < 32 ? lv.k_end - k0 : 32);
  const int64_t k = k0 + lane;
  const bool active = lane < nb;
  const int L = lv.m;
  const int len = active ? block_len(lv, k) : 0;  // rows inside the system
  const int nch = (L + R - 1) / R;
  const RelRow<T>* const rel = static_cast<const RelRow<T>*>(rl.rel) + k0 * rl.cap;
  const T* const rel_al = static_cast<const T*>(rl.al) + k0 * rl.cap;
  PieceMap<Tin, R> pm;
  pm.init(lv, k0, nb, lane);
  chain_wait();
  int na = rl.na[k0];
  const Tin* const xsrc[1] = {x};
  auto rows_of = [&](int st) {
    return reinterpret_cast<RelRow<T>*>(smem_raw + st * BT::kStage);
  };
  auto al_of = [&](int st) {
    return reinterpret_cast<T*>(smem_raw + st * BT::kStage + BT::kRows);
  };
  auto x_of = [&](int st) {
    return reinterpret_cast<Tin*>(smem_raw + (kRef ? st * BT::kStage + BT::kRows + BT::kAl
                                                   : kBackStages * BT::kStage));
  };
  // `rows` rows (a multiple of 4) of nb elements each, in 16-byte pieces
  auto copy = [&](auto* dst, const auto* src, int rows) {
    constexpr int kSize = sizeof(*dst);
    unsigned char* const o = reinterpret_cast<unsigned char*>(dst) + 16 * lane;
    const unsigned char* const i = reinterpret_cast<const unsigned char*>(src) + 16 * lane;
    if (rows == R && nb == 32) {
#pragma unroll
      for (int j = 0; j < R * kSize / 16; ++j) cp_async<16>(o + 512 * j, i + 512 * j);
    } else {
      for (int j = 0; j < rows * nb * kSize - 16 * lane; j += 512) cp_async<16>(o + j, i + j);
    }
  };
  // chunk ch to stage st, one commit group (rows 0 and L - 1 have no relation:
  // what their slots hold is copied and not used)
  auto fetch = [&](int ch, int st) {
    if (ch >= 0) {
      const int row0 = ch * R, rows = min(R, rl.cap - row0);
      copy(rows_of(st), rel + row0 * nb, rows);
      if (ch < na) copy(al_of(st), rel_al + row0 * nb, rows);
      if constexpr (kRef) load_chunk<Tin, R, kVec16>(x_of(st), xsrc, 1, pm, row0);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < kBackStages - 1; ++i) fetch(nch - 1 - i, i);
  T f = Ar::zero(), l = Ar::zero();
  if (active) {
    f = Ar::from(xred[2 * k]);
    l = Ar::from(xred[2 * k + 1]);
  }
  T xn = l;
  bool oob = false, late = false;
  unsigned long long mdel = 0, mx = 0;  // refinement maxima (bit patterns)
  int st = 0;
  for (int ch = nch - 1; ch >= 0; --ch) {
    const int row0 = ch * R;
    fetch(ch - (kBackStages - 1), st == 0 ? kBackStages - 1 : st - 1);
    cp_async_wait<kBackStages - 1>();
    __syncwarp();  // other lanes' copies
    const RelRow<T>* const w = rows_of(st) + lane;
    const T* const wal = al_of(st) + lane;
    Tin* const tile = x_of(st);
    Tin* const t = tile + lane * TL::kStride;
    // x of rows row0 + r; where every lane's rows are interior the tests go
    auto chunk = [&](auto kMid, auto kAl) {
      Tin xo[V];
#pragma unroll
      for (int r = R - 1; r >= 0; --r) {
        const int row = row0 + r;
        T xr = Ar::zero();
        const bool in = row < len;
        if (decltype(kMid)::value || (row >= 1 && row < L - 1)) {
          const RelRow<T> e = w[r * nb];
          T g = e.g;
          if constexpr (decltype(kAl)::value) g = Ar::sub_mul(g, wal[r * nb], f);
          xn = Ar::sub_mul(g, e.c, xn);
          xr = xn;
          if constexpr (Ar::kSkipChain) {
            if constexpr (!decltype(kAl)::value) late |= in && Ar::late(xr, f);
          }
        } else if (row == 0) {
          xr = f;
        } else if (row == L - 1) {
          xr = l;
        }
        Tin xv;
        Ar::to(xv, xr);
        oob |= in && Ar::out_bad(xv);
        if constexpr (kRef) {  // x += delta
          const Tin xs = t[r] + xv;
          if (in) {
            mdel = max(mdel, abs_bits(xv));
            mx = max(mx, abs_bits(xs));
          }
          xv = xs;
        }
        xo[r % V] = xv;
        if (r % V == 0) {
          Vec16<Tin> o;
#pragma unroll
          for (int v = 0; v < V; ++v) o.v[v] = xo[v];
          *reinterpret_cast<float4*>(t + r) = *reinterpret_cast<const float4*>(&o);
        }
      }
    };
    const bool mid = ch >= 1 && row0 + R <= L - 1;
    if (mid && ch >= na) chunk(std::true_type{}, std::false_type{});
    else if (mid) chunk(std::true_type{}, std::true_type{});
    else if (ch >= na) chunk(std::false_type{}, std::false_type{});
    else chunk(std::false_type{}, std::true_type{});
    __syncwarp();
    store_chunk<Tin, R, kVec16>(x, tile, pm, row0);
    __syncwarp();  // the slots are refilled by a later chunk
    st = st == kBackStages - 1 ? 0 : st + 1;
    if constexpr (Ar::kSkipChain) {  // an x so small that f may be missed: again, with every al
      if (ch == na && __any_sync(0xffffffffu, late)) {
        cp_async_wait<0>();
        __syncwarp();
        na = nch;
        xn = l;
        st = 0;
#pragma unroll
        for (int i = 0; i < kBackStages - 1; ++i) fetch(nch - 1 - i, i);
        ch = nch;
      }
    }
  }
  if (oob) atomicOr(status, ST_RANGE);
  if (lv.dmax)
    judge_codes(lv.dmax, (int64_t)blockIdx.x * 32 + lane, (int64_t)gridDim.x * 32, lv.nbnd + 1,
                status);
  if constexpr (kRef) {
    for (int o = 16; o > 0; o >>= 1) {
      mdel = max(mdel, __shfl_xor_sync(0xffffffffu, mdel, o));
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    // most warps see maxima already raised past theirs: read before the atomic
    if (lane == 0) {
      if (mdel > *(volatile unsigned long long*)&rf.max2[0]) atomicMax(&rf.max2[0], mdel);
      if (mx > *(volatile unsigned long long*)&rf.max2[1]) atomicMax(&rf.max2[1], mx);
    }
  }
}

// ------------------------------------------------------------------ small systems
// One warp solves a system of n <= 64 rows by parallel cyclic reduction
// (Hockney 1965): at stride s every row eliminates its neighbours at
// distance s, after ceil(log2 n) steps each row is decoupled and
// x_i = d_i / b_i.  Rows outside [0, n) act as identity rows.
constexpr int kBaseMax = 64;

// dmax (level 0 of fp64 inputs in narrower arithmetic, else null): the
// per-system range codes, raised here; x is checked for range.
template <class Ar, class Tin, class Tout>
__global__ void __launch_bounds__(32)
    k_base(int64_t n, const Tin* a, const Tin* b, const Tin* c, const Tin* d,
           Tout* __restrict__ x, const int64_t* bnd, int64_t nbnd, int* __restrict__ status,
           unsigned* __restrict__ dmax) {
  using T = typename Ar::T;
  __shared__ T sa[kBaseMax], sb[kBaseMax], sc[kBaseMax], sd[kBaseMax];
  const int lane = threadIdx.x;
  const int nn = (int)n;
  bool bad = false, oob = false;
  chain_wait();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = lane + 32 * h;
    if (i < nn) {
      bool start = (i == 0), end = (i == nn - 1);
      int64_t sys = 0;
      for (int64_t j = 0; j < nbnd; ++j) {  // packed systems: cut the couplings
        start |= bnd[j] == i;
        end |= bnd[j] == i + 1;
        sys += bnd[j] <= i;
      }
      RowChk rc;
      Ar::template row<true>(start ? Tin{} : a[i], b[i], end ? Tin{} : c[i], d[i], sa[i], sb[i],
                             sc[i], sd[i], rc);
      oob |= rc.range_bad();
      bad |= rc.b_bad();
      if (dmax) codes_raise(dmax, sys, rc.dcode(), rc.ecode, rc.fcode());
    } else {
      sa[i] = Ar::zero(); sb[i] = Ar::one(); sc[i] = Ar::zero(); sd[i] = Ar::zero();
    }
  }
  __syncwarp();
  for (int s = 1; s < nn; s <<= 1) {
    T na[2], nbv[2], nc[2], nd[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = lane + 32 * h;
      const int im = i - s, ip = i + s;
      const T am = im >= 0 ? sa[im] : Ar::zero();
      const T bm = im >= 0 ? sb[im] : Ar::one();
      const T cm = im >= 0 ? sc[im] : Ar::zero();
      const T dm = im >= 0 ? sd[im] : Ar::zero();
      const T ap = ip < kBaseMax ? sa[ip] : Ar::zero();
      const T bp = ip < kBaseMax ? sb[ip] : Ar::one();
      const T cp = ip < kBaseMax ? sc[ip] : Ar::zero();
      const T dp = ip < kBaseMax ? sd[ip] : Ar::zero();
      bad |= Ar::bad_pivot(bm) | Ar::bad_pivot(bp);
      const T k1 = Ar::mul(sa[i], Ar::rcp(bm));
      const T k2 = Ar::mul(sc[i], Ar::rcp(bp));
      na[h] = Ar::neg(Ar::mul(am, k1));
      nc[h] = Ar::neg(Ar::mul(cp, k2));
      nbv[h] = Ar::sub_mul(Ar::sub_mul(sb[i], cm, k1), ap, k2);
      nd[h] = Ar::sub_mul(Ar::sub_mul(sd[i], dm, k1), dp, k2);
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = lane + 32 * h;
      sa[i] = na[h]; sb[i] = nbv[h]; sc[i] = nc[h]; sd[i] = nd[h];
    }
    __syncwarp();
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = lane + 32 * h;
    if (i < nn) {
      bad |= Ar::bad_pivot(sb[i]);
      Tout xv;
      Ar::to(xv, Ar::mul(sd[i], Ar::rcp(sb[i])));
      oob |= Ar::out_bad(xv);
      x[i] = xv;
    }
  }
  if (bad) atomicOr(status, ST_BAD_PIVOT);
  if (oob) atomicOr(status, ST_RANGE);
}

}  // namespace tps
