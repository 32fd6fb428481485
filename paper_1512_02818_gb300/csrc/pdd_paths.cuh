// pdd_paths.cuh -- the path kernels of the PDD Monte Carlo nodal stage
// (Bernal & Acebron, Algorithm 1 with the pathwise control variate of
// eq. F:xiControlVariate) and their launchers.  One translation unit per
// problem instantiates PathLaunch, so that they compile side by side.
//
// Execution model.  One path per lane.  The paths of all nodes form one flat
// path-major index space g = path * n_nodes + node (consecutive indices are
// different nodes, so the paths in flight at any moment spread their record
// atomics over all node records instead of queueing on one record's cache
// line); warps take batches of 32 indices from a global cursor (atomicAdd)
// and the lanes whose paths have finished take the next indices of their warp's
// batch at an iteration boundary (short paths: once enough lanes wait, see
// refill_min), so lanes stay busy whatever the spread of exit times (paths of
// one node range over ~12x the mean number of steps).  The grid is persistent
// (occupancy x SM count blocks), smaller where a launch has few paths per lane
// (target_warps); a launch with fewer paths than lanes gives each warp one
// smaller batch instead (spread_batch).  A finished path parks in its warp's
// exit ring in shared memory and is scored and recorded later, 32 at a time by
// the whole warp, into a per-block shared-memory copy of the records where that
// pays (use_cache), which the block adds into the global ones at the end.  Once
// the cursor is exhausted a warp with half its lanes idle takes batches of steps
// of the paths it still holds (see Drain).  Per-node sums are exact integers, so
// which lane, warp or block runs a path changes nothing in the results.
//
// One iteration takes a whole number of Philox blocks' worth of Euler steps (2D:
// two steps a block; 3D: four steps of three blocks), so no random word is wasted
// and every path's stream is the one fixed by its (seed, stream_tag, node, path)
// key.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <type_traits>

#include "pdd_device.cuh"
#include "pdd_internal.h"
#include "pdd_launch.h"

namespace pdd {

constexpr int kBlockThreads = 128;     // default block size (smaller blocks retire sooner as a launch drains)
constexpr int kMaxBlockThreads = 512;  // largest block size a launch may ask for
// Minimum resident blocks per SM requested from the compiler (register cap).
#ifndef PDD_MIN_BLOCKS_2D
#define PDD_MIN_BLOCKS_2D 1
#endif
#ifndef PDD_MIN_BLOCKS_3D
#define PDD_MIN_BLOCKS_3D 2  // 64 registers: twice the warps of the unconstrained 3D kernel
#endif
constexpr unsigned kFull = 0xFFFFFFFFu;
// Euler steps per iteration of the path kernels (between lane refills and
// exit parking): 4 in 2D (two Philox blocks; 8 for the plain estimator, see
// LongSteps2D) and 8 in 3D (six) halve the
// per-step share of the refill, ring and loop work against 2 and 4, but a
// lane whose path ends early in an iteration idles for the rest of it, which
// costs on short paths.  A launch takes the longer iterations when segments
// with time steps above kLongPathH (paths of under ~100 steps) hold at most
// kShortWorkShare of its expected path-steps (n_nodes x n_paths / h per
// segment).
constexpr double kLongPathH = 2e-3;
// The long 2D iteration: eight steps (four Philox blocks) for the plain
// estimator, whose step is short enough that the refill and ring bookkeeping
// still weigh (+3 % path-steps/s against four), and four with a control
// variate (eight measured no faster).
template <class T, int CV>
struct LongSteps2D {
  static constexpr int value = sizeof(T) == 4 ? (CV == 0 ? 8 : 4) : 2;
};
constexpr double kShortWorkShare = 0.05;
enum { kCvNone = 0, kCvGrid = 1, kCvExact = 2 };

// Per-lane path state.
template <class T>
struct PathState {
  T x[3];
  T Y, Z, Zc, XI, XIc;
  int k;
  uint32_t node, path, seg;
};

// Per-lane copy of the parameters of the segment the lane's path belongs to.
// With a single segment they are the same for every lane and never change.
// FP32 paths read the cell-coefficient table, FP64 paths the nodal table
// (whose multilinear interpolation they evaluate in FP64, as the oracle does).
#ifndef PDD_CELLS_2D
#define PDD_CELLS_2D 1
#endif
#ifndef PDD_CELLS_3D
#define PDD_CELLS_3D 1
#endif
template <class T, int D>
struct UseCells {
  static constexpr bool value =
      sizeof(T) == 4 && ((D == 2 && PDD_CELLS_2D) || (D == 3 && PDD_CELLS_3D));
};

template <class T>
struct LaneSeg {
  T h, sqh, thr0;
  const void* grad;  // the table this lane reads (cells or nodal); null: no grid
  int gn, max_steps;
};

template <class T, int D>
__device__ __forceinline__ void load_seg(const SegArgs& sg, LaneSeg<T>& ls) {
  if constexpr (sizeof(T) == 4) {
    ls.h = sg.h32;
    ls.sqh = sg.sqrt_h32;
    ls.thr0 = sg.thr32;
  } else {
    ls.h = sg.h;
    ls.sqh = sg.sqrt_h;
    ls.thr0 = sg.thr0;
  }
  ls.grad = sg.grad;
  if (UseCells<T, D>::value && sg.grad != nullptr)
    ls.grad = (const char*)sg.grad + cell_table_offset(sg.grid_n, D);
  ls.gn = sg.grid_n;
  ls.max_steps = sg.max_steps;
}

template <bool MULTI>
constexpr int kSegs = MULTI ? kMaxSegments : 1;  // length of a kernel's segment table

// Segment of path index g: the last one whose begin <= g.
template <class A>
__device__ __forceinline__ uint32_t segment_of(const A& a, unsigned long long g) {
  int lo = 0, hi = a.n_segs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.seg[mid].begin <= g) lo = mid;
    else hi = mid - 1;
  }
  return (uint32_t)lo;
}

// Start path g of the launch's flat index space.
template <class T, int D, bool MULTI, class A>
__device__ __forceinline__ void start_path(const A& a, unsigned long long g, uint32_t from,
                                           PathState<T>& s, LaneSeg<T>& ls) {
  uint32_t si = 0;
  if (MULTI) {
    si = from;
    while ((int)si + 1 < a.n_segs && a.seg[si + 1].begin <= g) ++si;
  }
  const SegArgs& sg = a.seg[si];
  const unsigned long long li = g - sg.begin;
  if (!PDD_IN_BOUNDS(a, si < (uint32_t)a.n_segs && g >= sg.begin && li < sg.total && g < a.total,
                     kErrBoundsIndex)) {
    // leave the lane on node 0, path 0 of segment 0 (in bounds); the call fails
    s.node = s.path = s.seg = 0;
    s.x[0] = s.x[1] = s.x[2] = T(0.5);
    s.Y = T(1);
    s.Z = s.Zc = s.XI = s.XIc = T(0);
    s.k = 0;
    if (MULTI) load_seg<T, D>(a.seg[0], ls);
    return;
  }
  if (sg.total <= 0xFFFFFFFFull) {  // 32-bit division when the index space allows
    const uint32_t gg = (uint32_t)li, nn = (uint32_t)sg.n_nodes;
    const uint32_t p = gg / nn;
    s.node = gg - p * nn;
    s.path = sg.path_off + p;
  } else {
    const unsigned long long p = li / sg.n_nodes;
    s.node = (uint32_t)(li - p * sg.n_nodes);
    s.path = sg.path_off + (uint32_t)p;
  }
  s.seg = si;
  if (!PDD_IN_BOUNDS(a, s.node < sg.n_nodes && s.path - sg.path_off < sg.n_paths,
                     kErrBoundsIndex))
    s.node = 0;
  s.x[0] = (T)__ldg(sg.cx + s.node);
  s.x[1] = (T)__ldg(sg.cy + s.node);
  s.x[2] = (D == 3) ? (T)__ldg(sg.cz + s.node) : T(0);
  s.Y = T(1);
  s.Z = s.Zc = s.XI = s.XIc = T(0);
  s.k = 0;
  if (MULTI) load_seg<T, D>(sg, ls);
}

#ifndef PDD_EXIT_CENTRED
#define PDD_EXIT_CENTRED 1
#endif
// Finish test of Algorithm 1: d(X_k) >= -c0 |sigma^T N| sqrt(h).
template <class P, class T, int D>
__device__ __forceinline__ bool outside(const T* x, T thr0) {
  T thr = thr0;
  if (P::kAniso || P::kIsoScaled) thr = mul_rn(thr, P::template exit_scale<T>(x[0], x[1], x[2]));
  if (sizeof(T) == 4 && PDD_EXIT_CENTRED) {
    // FP32: the distance to the unit box's faces is 1/2 - max_i |X_i - 1/2|,
    // one instruction fewer than the minimum over the 2D faces
    T e = fmaxf(fabsf(sub_rn(x[0], T(0.5))), fabsf(sub_rn(x[1], T(0.5))));
    if (D == 3) e = fmaxf(e, fabsf(sub_rn(x[2], T(0.5))));
    return e >= sub_rn(T(0.5), thr);
  }
  const T m = (D == 3) ? face_distance(x[0], x[1], x[2]) : face_distance(x[0], x[1]);
  return m <= thr;
}
template <class P, class T, int D>
__device__ __forceinline__ bool should_finish(const PathState<T>& s, T thr0) {
  return outside<P, T, D>(s.x, thr0);
}

// Philox block `blk` of the lane's path.
template <bool MULTI, class A>
__device__ __forceinline__ uint4 path_block(const A& a, uint32_t seg, uint32_t blk,
                                            uint32_t path, uint32_t node) {
  const SegArgs& sg = a.seg[MULTI ? seg : 0];
  uint2 key = make_uint2(sg.key0, sg.key1);
  if (MULTI) asm volatile("" : "+r"(key.x), "+r"(key.y));  // see drain()
  return philox4x32_10(make_uint4(blk, path, node, sg.seed_hi), key);
}

// Gradient of the control grid at x.
template <class T, int D, class A>
__device__ __forceinline__ void grid_gradient(const A& a, const LaneSeg<T>& ls,
                                              const T* x, T* gv) {
  unsigned* err = PDD_DEBUG_BOUNDS ? a.err : nullptr;
  if (D == 2) {
    if (UseCells<T, 2>::value)
      grid_cells_2d<T>((const float4*)ls.grad, ls.gn, x[0], x[1], gv[0], gv[1], err);
    else
      grid_grad_2d<T>((const float2*)ls.grad, ls.gn, x[0], x[1], gv[0], gv[1], err);
  } else {
    if (UseCells<T, 3>::value)
      grid_cells_3d<T>((const float4*)ls.grad, ls.gn, x[0], x[1], x[2], gv[0], gv[1], gv[2], err);
    else
      grid_grad_3d<T>((const float4*)ls.grad, ls.gn, x[0], x[1], x[2], gv[0], gv[1], gv[2], err);
  }
}

// sigma dW.
template <class P, class T, int D>
__device__ __forceinline__ void noise(const Coef<T>& o, const T* dW, T* sdW) {
  const T dW0 = dW[0], dW1 = dW[1];
  if (P::kAniso) {  // sigma = sqrt(a) [[1, 0], [1/2, sqrt(3)/2]]
    sdW[0] = mul_rn(o.sa, dW0);
    sdW[1] = mul_rn(o.sa, fma_rn(T(0.86602540378443864676), dW1, mul_rn(T(0.5), dW0)));
  } else if (P::kIsoScaled) {  // sigma = sa I
    sdW[0] = mul_rn(o.sa, dW0);
    sdW[1] = mul_rn(o.sa, dW1);
  } else {
    sdW[0] = dW0;
    sdW[1] = dW1;
  }
  sdW[2] = (D == 3) ? dW[2] : T(0);
}

// grad v . sigma dW, the integrand of the control variate without its -Y.
template <class T, int D>
__device__ __forceinline__ T cv_dot(const T* gv, const T* sdW) {
  T dot = fma_rn(gv[1], sdW[1], mul_rn(gv[0], sdW[0]));
  if (D == 3) dot = fma_rn(gv[2], sdW[2], dot);
  return dot;
}

// X_{k+1} = X_k + h b + sigma dW.  The drift's step is h b, or (h/2)(2 b) for
// problems whose eval returns 2 b (the same product: halving h is exact).
template <class P, class T, int D>
__device__ __forceinline__ void advance(T* x, T h, const Coef<T>& o, const T* sdW) {
  const T hb = P::kDriftHalf ? mul_rn(T(0.5), h) : h;
  x[0] = add_rn(x[0], fma_rn(hb, o.b0, sdW[0]));
  x[1] = add_rn(x[1], fma_rn(hb, o.b1, sdW[1]));
  if (D == 3) x[2] = add_rn(x[2], fma_rn(hb, o.b2, sdW[2]));
}

// One Euler-Maruyama step (eq. F:E_M) with the Feynman-Kac weights and the
// control variate, all right-hand sides at X_k.  dW holds sqrt(h) * normals.
// YRULE: the step honours the launch's Y rule (a.y_exp); without it the step
// uses the default Euler rule Y(1 - h c).  The single-segment build of the
// path kernels has YRULE = false and launches with the exponential rule go to
// the segment-table build: dropping the per-step choice made the
// single-segment build 2.4 % faster with the control variate, 5 % without.
template <class P, class T, int D, int CV, bool MULTI, bool YRULE = MULTI, class A>
__device__ __forceinline__ void euler_step(const A& a, PathState<T>& s,
                                           const LaneSeg<T>& ls, const T* dW) {
  const T h = ls.h;
  // with several segments a segment without a grid runs the plain estimator
  constexpr bool kCv = CV != kCvNone;
  const bool use_cv = kCv && (CV != kCvGrid || !MULTI || ls.grad != nullptr);
  // The cell-record gather depends only on X_k: it is issued before the
  // coefficients are evaluated, so its latency overlaps their arithmetic.
  T gv[3] = {T(0), T(0), T(0)};
  if (CV == kCvGrid && use_cv) grid_gradient<T, D>(a, ls, s.x, gv);
  Coef<T> o;
  P::template eval<T, CV == kCvExact>(s.x[0], s.x[1], s.x[2], o, a.f64);
  T sdW[3];
  noise<P, T, D>(o, dW, sdW);
  if (use_cv) {
    if (CV == kCvExact) {
      gv[0] = o.g0;
      gv[1] = o.g1;
      gv[2] = o.g2;
    }
    kahan_add(s.XI, s.XIc, -s.Y, cv_dot<T, D>(gv, sdW));
  }
  // h Y_k serves the Z increment and the Euler rule Y_k (1 - h c) = Y_k - (h Y_k) c
  const T hY = P::kUnitY ? T(0) : mul_rn(h, s.Y);
  if (!P::kUnitY) kahan_add(s.Z, s.Zc, -hY, o.f);
  advance<P, T, D>(s.x, h, o, sdW);
  if (!P::kUnitY)
    s.Y = (YRULE && a.y_exp) ? mul_rn(s.Y, m_exp(mul_rn(-h, o.c))) : fma_rn(-hY, o.c, s.Y);
  s.k += 1;
}

// Exact fixed-point accumulation of one path's (phi, psi = phi + xi, k) into a
// node record (global, or the block's shared-memory copy), and of k into the
// launch's step counter `steps` when there is one.
template <class T, class A>
__device__ __forceinline__ void accumulate(const A& a, unsigned long long* w,
                                           unsigned long long* steps, T phi, T psi, int k_steps,
                                           bool trunc) {
  long long qa, qb;
  const bool ok = to_fixed(phi, qa) & to_fixed(psi, qb);
  if (!ok) atomicOr(a.err, kErrOverflow);
  atomic_add_s64(w + 0, qa);
  atomic_add_prod(w + 2, qa, qa);
  atomic_add_s64(w + 4, qb);
  atomic_add_prod(w + 6, qb, qb);
  atomic_add_prod(w + 8, qa, qb);
  const unsigned long long k = (unsigned long long)k_steps;
  atomic_add_u128(w + 10, k, 0ull);
  atomic_add_u128(w + 12, k * k, 0ull);
  atomicAdd(w + 14, 1ull);
  if (trunc) {
    atomicAdd(w + 15, 1ull);
    atomicAdd(a.trunc_total, 1ull);
  }
  if (steps != nullptr) atomicAdd(steps, k);
}

// Block-level record cache.  When the launch's segments hold at most
// kCacheMaxNodes node records, every block keeps its own copy of them in
// shared memory: exits add into the copy with shared-memory atomics (exits of
// different nodes no longer meet on a few cache lines of L2), and once all
// warps of the block have finished the block adds its non-empty records into
// the global ones (128-bit adds with carry: the same exact sums).  Slot
// seg.cache_base + node holds the record of `node` of segment `seg`; the word
// after the last slot counts the block's exit indices for a.steps_total.
extern __shared__ unsigned long long s_cache[];
// Slot stride in 64-bit words: one word of padding per record, so the same
// word of consecutive slots falls in different shared-memory banks.
constexpr uint32_t kCacheStride = kAccWords + 1;

template <class A>
__device__ __forceinline__ void cache_init(const A& a) {
  if (a.cache_nodes == 0) return;
  const uint32_t words = a.cache_nodes * kCacheStride + 1;
  for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) s_cache[i] = 0ull;
  __syncthreads();
}

template <class A>
__device__ __forceinline__ void cache_flush(const A& a) {
  if (a.cache_nodes == 0) return;
  __syncthreads();
  const uint32_t pairs = a.cache_nodes * (kAccWords / 2);
  for (uint32_t i = threadIdx.x; i < pairs; i += blockDim.x) {
    const uint32_t slot = i / (kAccWords / 2), q = i % (kAccWords / 2);
    const unsigned long long* s = s_cache + (size_t)slot * kCacheStride;
    if (s[14] == 0ull) continue;  // no path of this node ended in this block
    int lo = 0, hi = a.n_segs - 1;  // last segment whose cache_base <= slot
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.seg[mid].cache_base <= slot) lo = mid;
      else hi = mid - 1;
    }
    const SegArgs& sg = a.seg[lo];
    if (!PDD_IN_BOUNDS(a, slot >= sg.cache_base && slot - sg.cache_base < sg.n_nodes,
                       kErrBoundsRecord))
      continue;
    unsigned long long* g = sg.acc + (size_t)(slot - sg.cache_base) * kAccWords;
    if (q < 7) {
      if ((s[2 * q] | s[2 * q + 1]) != 0ull) atomic_add_u128(g + 2 * q, s[2 * q], s[2 * q + 1]);
    } else {
      atomicAdd(g + 14, s[14]);
      if (s[15] != 0ull) atomicAdd(g + 15, s[15]);
    }
  }
  if (threadIdx.x == 0 && a.steps_total != nullptr) {
    const unsigned long long st = s_cache[(size_t)a.cache_nodes * kCacheStride];
    if (st != 0ull) atomicAdd(a.steps_total, st);
  }
}

// Add one path into the record of `node` of segment `sg` (cached or global).
template <class T, class A>
__device__ __forceinline__ void record_path(const A& a, const SegArgs& sg, uint32_t node,
                                            T phi, T psi, int k_steps, bool trunc) {
  if (!PDD_IN_BOUNDS(a, node < sg.n_nodes, kErrBoundsRecord)) return;
  if (a.cache_nodes != 0) {
    if (!PDD_IN_BOUNDS(a, sg.cache_base + node < a.cache_nodes, kErrBoundsRecord)) return;
    accumulate(a, s_cache + (size_t)(sg.cache_base + node) * kCacheStride,
               a.steps_total != nullptr ? s_cache + (size_t)a.cache_nodes * kCacheStride : nullptr,
               phi, psi, k_steps, trunc);
  } else {
    accumulate(a,
               sg.acc + (size_t)(blockIdx.x & a.copy_mask) * a.copy_words + (size_t)node * kAccWords,
               a.steps_total, phi, psi, k_steps, trunc);
  }
}

// Exit scoring: X_tau = Pi(X_k), phi = g(X_tau) Y + Z, and xi.
template <class P, class T, int D>
__device__ __forceinline__ void score_path(const PathState<T>& s, T& phi, T& xi) {
  T p[3] = {s.x[0], s.x[1], s.x[2]};
  project_box<T>(p, D);
  const T g = P::template g<T>(p[0], p[1], p[2]);
  phi = fma_rn(g, s.Y, sub_rn(s.Z, s.Zc));
  xi = sub_rn(s.XI, s.XIc);
}

// Exit scoring and the exact fixed-point accumulation into the node record.
template <class P, class T, int D, bool MULTI, class A>
__device__ __forceinline__ void finish_path(const A& a, const PathState<T>& s, bool trunc) {
  T phi, xi;
  score_path<P, T, D>(s, phi, xi);
  const SegArgs& sg = a.seg[MULTI ? s.seg : 0];
  record_path(a, sg, s.node, phi, phi + xi, s.k, trunc);
  if (sg.emit_phi != nullptr) {
    const size_t i = (size_t)s.node * sg.emit_stride + s.path;
    if (!PDD_IN_BOUNDS(a, i < sg.n_nodes * sg.emit_stride, kErrBoundsEmit)) return;
    sg.emit_phi[i] = (float)phi;
    sg.emit_xi[i] = (float)xi;
    sg.emit_steps[i] = s.k;
  }
}

// Refill idle lanes from the warp's batch once a.refill_min of them are idle;
// returns false when no lane of the warp has a path left to run.  All arguments
// except the lane state are warp-uniform; bseg is the segment of the batch's
// first path.
template <class T, int D, bool MULTI, class A>
__device__ __forceinline__ bool refill(const A& a, PathState<T>& s, LaneSeg<T>& ls,
                                       bool& active, unsigned long long& bnext,
                                       unsigned long long& bend, uint32_t& bseg,
                                       bool& exhausted) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt = (1u << lane) - 1u;
  unsigned idle = __ballot_sync(kFull, !active);
  if (__popc(idle) < a.refill_min) return true;
  while (idle != 0u && !exhausted) {
    if (bnext >= bend) {
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(a.cursor, a.warp_batch);
      base = __shfl_sync(kFull, base, 0);
      if (base >= a.total) {
        exhausted = true;
        break;
      }
      bnext = base;
      bend = min(base + a.warp_batch, a.total);
      if (MULTI) bseg = segment_of(a, base);
    }
    const unsigned avail = (unsigned)min(bend - bnext, 32ull);
    const unsigned rank = __popc(idle & lt);
    if (!active && rank < avail) {
      start_path<T, D, MULTI>(a, bnext + rank, bseg, s, ls);
      active = true;
    }
    bnext += min((unsigned)__popc(idle), avail);
    idle = __ballot_sync(kFull, !active);
  }
  return __ballot_sync(kFull, active) != 0u;
}

// Spread launches (see spread_batch): every warp has a batch of its own, and
// the cursor is past the last path when the warp asks it for more (and counts
// the warps).  A warp that finds the launch aborted takes no batch.
template <bool MULTI, class A>
__device__ __forceinline__ void spread_claim(const A& a, unsigned long long& bnext,
                                             unsigned long long& bend, uint32_t& bseg) {
  if (a.one_claim == 0) return;
  // (the shuffle tells the compiler that the batch is the warp's: without it
  // the kernels take 20 registers more)
  const unsigned warp = __shfl_sync(kFull, (blockIdx.x * blockDim.x + threadIdx.x) >> 5, 0);
  unsigned long long before = 0;
  if ((threadIdx.x & 31u) == 0u) before = atomicAdd(a.cursor, kSpreadClaim);
  const unsigned long long end = __any_sync(kFull, before >= kAborted) ? 0ull : a.total;
  bnext = min(warp * a.warp_batch, end);
  bend = min(bnext + a.warp_batch, end);
  if (MULTI) bseg = segment_of(a, bnext);
}

// Per-warp exit ring.  A lane whose path has ended parks the path's final
// state (X, Y, Z, xi, k, node, path, segment | truncated) in its warp's ring
// in shared memory and takes a new path at once; whenever 32 exits are
// parked, the whole warp scores and records them, one per lane.  Exit work
// (projection, g, fixed-point conversion, the record's 13 atomic adds) thus
// runs with all lanes busy instead of one lane at a time while the rest of
// the warp waits.  Rings follow the record cache in dynamic shared memory.
constexpr uint32_t kRing = 64;  // entries per warp (>= 2 x 32: a full batch plus one iteration)
// The ring is two halves of 32 entries, each with its own field arrays, so
// that the drain can park exits in the first half and work in the second.
template <class T, int D>
struct ExitRing {
  static constexpr uint32_t kHalf = 32 * ((D + 3) * sizeof(T) + 4 * sizeof(uint32_t));
  static constexpr size_t kBytes = 2 * kHalf;
  char* base;
  // fields of entry j, 32 apart: X_0 .. X_(D-1), Y, Z, xi
  __device__ __forceinline__ T* f(uint32_t j) const {
    return (T*)(base + (j >> 5) * kHalf) + (j & 31u);
  }
  // k, node, path, segment | truncated << 31
  __device__ __forceinline__ uint32_t* u(uint32_t j) const {
    return (uint32_t*)(base + (j >> 5) * kHalf + 32 * (D + 3) * sizeof(T)) + (j & 31u);
  }
};

__host__ __device__ __forceinline__ size_t cache_bytes(uint32_t cache_nodes) {
  if (cache_nodes == 0) return 0;
  return (((size_t)cache_nodes * (kAccWords + 1) + 1) * 8 + 15) / 16 * 16;
}

template <class T, int D, class A>
__device__ __forceinline__ ExitRing<T, D> ring_of_warp(const A& a) {
  return {(char*)s_cache + cache_bytes(a.cache_nodes) +
          (size_t)(threadIdx.x >> 5) * ExitRing<T, D>::kBytes};
}

template <class T, int D>
__device__ __forceinline__ void ring_put(const ExitRing<T, D>& r, uint32_t j,
                                         const PathState<T>& s, bool trunc) {
  T* f = r.f(j);
  uint32_t* u = r.u(j);
#pragma unroll
  for (int d = 0; d < D; ++d) f[d * 32] = s.x[d];
  f[D * 32] = s.Y;
  f[(D + 1) * 32] = s.Z - s.Zc;
  f[(D + 2) * 32] = s.XI - s.XIc;
  u[0] = (uint32_t)s.k;
  u[32] = s.node;
  u[64] = s.path;
  u[96] = s.seg | (trunc ? 0x80000000u : 0u);
}

// Score and record `count` (<= 32) parked exits starting at ring slot `first`.
template <class P, class T, int D, bool MULTI, class A>
__device__ __forceinline__ void ring_drain(const A& a, const ExitRing<T, D>& r,
                                           uint32_t first, uint32_t count) {
  __syncwarp();
  const uint32_t lane = threadIdx.x & 31u;
  if (lane < count) {
    const uint32_t j = (first + lane) & (kRing - 1);
    const T* f = r.f(j);
    const uint32_t* u = r.u(j);
    PathState<T> e;
    e.x[0] = e.x[1] = e.x[2] = T(0);
#pragma unroll
    for (int d = 0; d < D; ++d) e.x[d] = f[d * 32];
    e.Y = f[D * 32];
    e.Z = f[(D + 1) * 32];
    e.XI = f[(D + 2) * 32];
    e.Zc = e.XIc = T(0);
    e.k = (int)u[0];
    e.node = u[32];
    e.path = u[64];
    const uint32_t st = u[96];
    e.seg = st & 0x7FFFFFFFu;
    finish_path<P, T, D, MULTI>(a, e, (st >> 31) != 0u);
  }
  __syncwarp();
}

// Warp-uniform ring cursor: `head` counts parked exits, `held` those not yet
// drained.
struct RingCursor {
  uint32_t head = 0, held = 0;
};

// Moves the parked exits (fewer than 32, anywhere in the ring) to the first
// entries: NF words of type T and NU of 32 bits each.
template <int NF, int NU = 4, class Ring>
__device__ __forceinline__ void ring_move(const Ring& r, const RingCursor& c) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t from = (c.head - c.held + lane) & (kRing - 1);
  if (((c.head - c.held) & (kRing - 1)) == 0u) return;
  typename std::remove_pointer<decltype(r.f(0u))>::type f[NF];
  uint32_t u[NU];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < NF; ++i) f[i] = r.f(from)[32 * i];
#pragma unroll
  for (int i = 0; i < NU; ++i) u[i] = r.u(from)[32 * i];
  __syncwarp();
  if (lane < c.held) {
#pragma unroll
    for (int i = 0; i < NF; ++i) r.f(lane)[32 * i] = f[i];
#pragma unroll
    for (int i = 0; i < NU; ++i) r.u(lane)[32 * i] = u[i];
  }
  __syncwarp();
}

// Park the exits of this iteration (`done` lanes) and drain a full batch.
template <class P, class T, int D, bool MULTI, class A>
__device__ __forceinline__ void ring_exit(const A& a, const ExitRing<T, D>& r,
                                          RingCursor& c, const PathState<T>& s, bool done,
                                          bool trunc) {
  const unsigned m = __ballot_sync(kFull, done);
  if (m == 0u) return;
  // never more than kRing parked: fewer than 32 are held before this iteration
  if (!PDD_IN_BOUNDS(a, c.held + __popc(m) <= kRing, kErrBoundsRing)) return;
  if (done) {
    const unsigned lt = (1u << (threadIdx.x & 31u)) - 1u;
    ring_put<T, D>(r, (c.head + __popc(m & lt)) & (kRing - 1), s, trunc);
  }
  c.head += __popc(m);
  c.held += __popc(m);
  if (c.held >= 32u) {
    ring_drain<P, T, D, MULTI>(a, r, c.head - c.held, 32u);
    c.held -= 32u;
  }
}

template <class T, int D, class A>
__device__ __forceinline__ void init_lane(const A& a, PathState<T>& s, LaneSeg<T>& ls) {
  s.x[0] = s.x[1] = s.x[2] = T(0);
  s.Y = s.Z = s.Zc = s.XI = s.XIc = T(0);
  s.k = 0;
  s.node = s.path = s.seg = 0;
  load_seg<T, D>(a.seg[0], ls);
}

// Running lanes of a warp at which it goes over to the drain (see Drain): 6,
// 12, 16 and 20 in 2D took 3.38, 3.00, 2.88 and 3.05 ms on 256 nodes x 1,387
// paths with the control variate; a 3D batch needs four lanes per path.
#ifndef PDD_DRAIN_RUN_2D
#define PDD_DRAIN_RUN_2D 16
#endif
#ifndef PDD_DRAIN_RUN_3D
#define PDD_DRAIN_RUN_3D 8
#endif

// Position of the q-th (from 0) set bit of m, q < popc(m): the largest p
// with fewer than q + 1 set bits below it, by binary search.
__device__ __forceinline__ int nth_set_bit(unsigned m, int q) {
  int p = 0;
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1)
    if (__popc(m & ((1u << (p + w)) - 1u)) <= q) p += w;
  return p;
}

// The drain.  Once the launch's cursor is exhausted a warp only finishes the
// paths it holds, and as lanes retire the launch's time becomes the serial
// latency of its longest paths.  Of an Euler step only the position's own
// recurrence (the drift and the noise) has to wait for the previous step;
// the random numbers depend on the path's key alone, and the exit test, the
// coefficients c and f and the control variate on one position each.  When at
// most Drain::kMaxRun lanes of a warp still run a path, the warp takes S steps
// of its A paths at a time, in four passes over its scratch:
//   1. every lane draws a Philox block and its four scaled normals;
//   2. lane q < A advances path q by S positions, without testing for the
//      exit (what lies past it is not used), one multiply, one SFU call and
//      two additions deep per step;
//   3. every lane tests the exit at, and evaluates the coefficients and
//      grad v . sigma dW of, one or two (path, step) pairs;
//   4. lane q folds path q's steps up to its exit into Y, Z and xi, in order.
// Path q and its state move to lane q whenever paths have ended.  Every value
// comes from the operations of euler_step in their order, so a path's result
// does not depend on where it ran.
// What bounds it: alone, the chains of passes 2 and 4 (about 90 cycles a step
// plain, 105 with the control variate; drawing the random numbers on idle
// lanes and taking the whole step in order afterwards took 320 and 560);
// with all of a chip's warps in it, the issue slots, most of which go to the
// two chains' few lanes.  256 nodes x 1,387 paths at h = 1e-4: 2.95 -> 2.24 ms
// plain, 4.79 -> 2.96 ms with the control variate; 10 paths per node in 3D,
// 2.67 -> 1.40 ms (with fewer warps, and spread, 1.74, 2.65 and 0.46: see
// target_warps and spread_batch).
template <class T, int D>
struct Drain {
  static constexpr int kMaxRun = D == 2 ? PDD_DRAIN_RUN_2D : PDD_DRAIN_RUN_3D;
  // 2D: a lane's block makes two steps of one path (4 scratch words each)
  static constexpr int kLanes = ExitRing<T, D>::kHalf / (8 * sizeof(T)) < 32
                                    ? ExitRing<T, D>::kHalf / (8 * sizeof(T))
                                    : 32;
  // Philox blocks and steps per path with A running paths (3D: 3 blocks make
  // 4 steps, and a lane evaluates one step)
  __device__ static int blocks(int A) { return D == 2 ? kLanes / A : 3 * (8 / A); }
  __device__ static int steps(int A) { return D == 2 ? 2 * (kLanes / A) : 4 * (8 / A); }
};
static_assert(32 * 6 * sizeof(float) <= ExitRing<float, 3>::kHalf, "3D drain scratch");
static_assert(32 * 6 * sizeof(double) <= ExitRing<double, 3>::kHalf, "3D drain scratch");

// Scratch vectors of D words: 2D as one 2-word access, 3D A words apart.
template <class T, int D>
__device__ __forceinline__ void get_vec(const T* base, int step, int q, int A, T* v) {
  if (D == 2) {
    using V = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
    const V w = ((const V*)base)[step * A + q];
    v[0] = w.x;
    v[1] = w.y;
    v[2] = T(0);
  } else {
    const T* p = base + 3 * step * A + q;
    v[0] = p[0];
    v[1] = p[A];
    v[2] = p[2 * A];
  }
}
template <class T, int D>
__device__ __forceinline__ void put_vec(T* base, int step, int q, int A, T v0, T v1, T v2) {
  if (D == 2) {
    using V = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
    V w;
    w.x = v0;
    w.y = v1;
    ((V*)base)[step * A + q] = w;
  } else {
    T* p = base + 3 * step * A + q;
    p[0] = v0;
    p[A] = v1;
    p[2 * A] = v2;
  }
}

// Where a lane stands in a batch of A paths: it works for path q = lane mod A
// as number m = lane / A of the lanes `mine`, and lanes below A own a path.
struct BatchLane {
  int lane, A, q, m;
  unsigned mine;
  __device__ __forceinline__ explicit BatchLane(int paths)
      : lane((int)(threadIdx.x & 31u)), A(paths), q(lane % A), m(lane / A), mine(0u) {
    for (int l = q; l < 32; l += A) mine |= 1u << l;
  }
};

// Pass 1: Philox block blk of the lane's path into words 4m .. 4m + 3 of the
// path's normals.
template <class T, int D>
__device__ __forceinline__ void batch_normals(const BatchLane& b, uint32_t blk, uint32_t path,
                                              uint32_t node, uint32_t seed_hi, uint2 key, T sqh,
                                              T* nrm, const F64Tables* tb) {
  const uint4 w = philox4x32_10(make_uint4(blk, path, node, seed_hi), key);
  T n[4];
  box_muller(w.x, w.y, n[0], n[1], sqh, tb);
  box_muller(w.z, w.w, n[2], n[3], sqh, tb);
  if (D == 2) {
    put_vec<T, D>(nrm, 2 * b.m, b.q, b.A, n[0], n[1], T(0));
    put_vec<T, D>(nrm, 2 * b.m + 1, b.q, b.A, n[2], n[3], T(0));
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) nrm[(4 * b.m + c) * b.A + b.q] = n[c];
  }
}

// Increment of step i; PAIR: the sum of those of steps 2i and 2i + 1, rounded by
// itself here and in the ordinary iterations (there each is a product in the
// same function, with which a plain sum may be fused).
template <class T, int D, bool PAIR>
__device__ __forceinline__ void batch_noise(const T* nrm, int i, const BatchLane& b, T* dW) {
  get_vec<T, D>(nrm, PAIR ? 2 * i : i, b.q, b.A, dW);
  if (PAIR) {
    T e[3];
    get_vec<T, D>(nrm, 2 * i + 1, b.q, b.A, e);
#pragma unroll
    for (int d = 0; d < D; ++d) dW[d] = add_rn(dW[d], e[d]);
  }
}

// Passes 2 to 4 over up to S steps of every path that is `on`; returns the
// steps the lane's path takes and whether max_steps stopped it.  dots[(i A + q)
// dot_stride] takes grad v . sigma dW in 2D (3D keeps it beside c and f).
template <class P, class T, int D, int CV, bool PAIR, class A>
__device__ __forceinline__ int batch_steps(const A& a, const LaneSeg<T>& ls,
                                           PathState<T>& s, const T* nrm, T* pos, T* dots,
                                           int dot_stride, const BatchLane& b, int S, bool on,
                                           bool use_cv, bool y_exp, bool& trunc) {
  constexpr int kFold = 4;  // steps whose terms are read at once in pass 4
  // (path, step) pairs per lane: a 2D block makes two steps, one of a pair's sums
  constexpr int kItems = D == 2 && !PAIR ? 2 : 1;
  // 2. positions; the normals are read U steps ahead (U divides S)
  constexpr int U = PAIR ? 1 : 2;
  const bool own = b.lane < b.A && on;
  if (own) {
    T dW[U][3], next[U][3];
#pragma unroll
    for (int j = 0; j < U; ++j) batch_noise<T, D, PAIR>(nrm, j, b, dW[j]);
#pragma unroll 1
    for (int i = 0; i < S; i += U) {
      const int ahead = min(i + U, S - U);
#pragma unroll
      for (int j = 0; j < U; ++j) batch_noise<T, D, PAIR>(nrm, ahead + j, b, next[j]);
#pragma unroll
      for (int j = 0; j < U; ++j) {
        put_vec<T, D>(pos, i + j, b.q, b.A, s.x[0], s.x[1], s.x[2]);
        Coef<T> o;
        P::template eval<T, false>(s.x[0], s.x[1], s.x[2], o, a.f64);
        T sdW[3];
        noise<P, T, D>(o, dW[j], sdW);
        advance<P, T, D>(s.x, ls.h, o, sdW);
#pragma unroll
        for (int d = 0; d < D; ++d) dW[j][d] = next[j][d];
      }
    }
  }
  __syncwarp();
  // 3. exit tests, then coefficients of the steps before the exit
  unsigned f[kItems];
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = kItems * b.m + j;
    bool fin = false;
    if (i < S && on) {
      T x[3];
      get_vec<T, D>(pos, i, b.q, b.A, x);
      fin = outside<P, T, D>(x, ls.thr0);
    }
    f[j] = __ballot_sync(kFull, fin) & b.mine;
  }
  int n = on ? S : 0;
  const unsigned any = f[0] | f[kItems - 1];
  if (any != 0u) {
    const int l = __ffs(any) - 1;
    n = kItems * (l / b.A) + ((f[0] >> l) & 1u ? 0 : 1);
  }
  trunc = on && n >= ls.max_steps - s.k;
  if (trunc) n = ls.max_steps - s.k;
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = kItems * b.m + j;
    if (i < n) {
      T x[3];
      get_vec<T, D>(pos, i, b.q, b.A, x);
      T gv[3] = {T(0), T(0), T(0)}, dot = T(0);
      if (CV == kCvGrid && use_cv) grid_gradient<T, D>(a, ls, x, gv);
      Coef<T> o;
      P::template eval<T, CV == kCvExact>(x[0], x[1], x[2], o, a.f64);
      if (use_cv) {
        T dW[3], sdW[3];
        batch_noise<T, D, PAIR>(nrm, i, b, dW);
        noise<P, T, D>(o, dW, sdW);
        if (CV == kCvExact) {
          gv[0] = o.g0;
          gv[1] = o.g1;
          gv[2] = o.g2;
        }
        dot = cv_dot<T, D>(gv, sdW);
      }
      const T c = y_exp ? m_exp(mul_rn(-ls.h, o.c)) : o.c;
      put_vec<T, D>(pos, i, b.q, b.A, c, o.f, dot);
      if (D == 2 && use_cv) dots[(i * b.A + b.q) * dot_stride] = dot;
    }
  }
  __syncwarp();
  // 4. Y, Z and xi
  if (own) {
    auto fold = [&](const T* v) {
      if (use_cv) kahan_add(s.XI, s.XIc, -s.Y, v[2]);
      if (!P::kUnitY) {
        const T hY = mul_rn(ls.h, s.Y);
        kahan_add(s.Z, s.Zc, -hY, v[1]);
        s.Y = y_exp ? mul_rn(s.Y, v[0]) : fma_rn(-hY, v[0], s.Y);
      }
    };
    auto read = [&](int i, T* v) {
      get_vec<T, D>(pos, i, b.q, b.A, v);
      if (D == 2 && use_cv) v[2] = dots[(i * b.A + b.q) * dot_stride];
    };
    int i = 0;
#pragma unroll 1
    for (; i + kFold <= n; i += kFold) {
      T v[kFold][3];
#pragma unroll
      for (int j = 0; j < kFold; ++j) read(i + j, v[j]);
#pragma unroll
      for (int j = 0; j < kFold; ++j) fold(v[j]);
    }
#pragma unroll 1
    for (; i < n; ++i) {
      T v[3];
      read(i, v);
      fold(v);
    }
    if (n < S) get_vec<T, D>(pos, n, b.q, b.A, s.x);  // X at the exit
  }
  s.k += n;
  return n;
}

// The lane takes the path of lane `src` (position, sums and step).
template <class T, int D>
__device__ __forceinline__ void take_path(PathState<T>& s, int src) {
#pragma unroll
  for (int d = 0; d < D; ++d) s.x[d] = __shfl_sync(kFull, s.x[d], src);
  s.Y = __shfl_sync(kFull, s.Y, src);
  s.Z = __shfl_sync(kFull, s.Z, src);
  s.Zc = __shfl_sync(kFull, s.Zc, src);
  s.XI = __shfl_sync(kFull, s.XI, src);
  s.XIc = __shfl_sync(kFull, s.XIc, src);
  s.k = __shfl_sync(kFull, s.k, src);
}

template <class P, class T, int D, int CV, bool MULTI, class A>
__device__ __forceinline__ void drain(const A& a, const ExitRing<T, D> ring, RingCursor rc,
                                      PathState<T> s, LaneSeg<T> ls, bool active) {
  // the ring's first half parks the exits from here on, its second is scratch
  uint32_t held = rc.held;
  ring_move<D + 3>(ring, rc);
  T* const nrm = (T*)(ring.base + ExitRing<T, D>::kHalf);  // scaled normals, then grad v . sigma dW
  T* const pos = nrm + (D == 2 ? 4 * Drain<T, D>::kLanes : 96);  // X, then c, f (and the dot in 3D)
  unsigned runm = __ballot_sync(kFull, active);
  while (runm != 0u) {
    const BatchLane b(__popc(runm));
    const int src = nth_set_bit(runm, b.q);
    take_path<T, D>(s, src);
    s.node = __shfl_sync(kFull, s.node, src);
    s.path = __shfl_sync(kFull, s.path, src);
    if (MULTI) {
      s.seg = __shfl_sync(kFull, s.seg, src);
      load_seg<T, D>(a.seg[s.seg], ls);
    }
    const SegArgs& sg = a.seg[MULTI ? s.seg : 0];
    const uint32_t key0 = sg.key0, key1 = sg.key1, seed_hi = sg.seed_hi;
    const bool use_cv = CV != kCvNone && (CV != kCvGrid || !MULTI || ls.grad != nullptr);
    const int blocks = Drain<T, D>::blocks(b.A), S = Drain<T, D>::steps(b.A);
    unsigned endm = 0u;
    bool trunc = false;
    do {
      if (b.m < blocks) {
        const uint32_t blk0 = D == 2 ? (uint32_t)s.k >> 1 : 3u * ((uint32_t)s.k >> 2);
        // (the empty asm keeps the ten rounds' keys from living in registers
        // across the batches: 20 of them with per-lane keys)
        uint2 key = make_uint2(key0, key1);
        if (MULTI) asm volatile("" : "+r"(key.x), "+r"(key.y));
        batch_normals<T, D>(b, blk0 + (uint32_t)b.m, s.path, s.node, seed_hi, key, ls.sqh, nrm,
                            a.f64);
      }
      __syncwarp();
      const int n = batch_steps<P, T, D, CV, false>(a, ls, s, nrm, pos, nrm, 2, b, S, true, use_cv,
                                                    MULTI && a.y_exp, trunc);
      endm = __ballot_sync(kFull, b.lane < b.A && (trunc || n < S));
      __syncwarp();
    } while (endm == 0u);
    // park the exits
    const uint32_t ended = (uint32_t)__popc(endm);
    if (held + ended > 32u) {
      ring_drain<P, T, D, MULTI>(a, ring, 0u, held);
      held = 0;
    }
    if ((endm >> b.lane) & 1u)
      ring_put<T, D>(ring, held + (uint32_t)__popc(endm & ((1u << b.lane) - 1u)), s, trunc);
    held += ended;
    runm = ((1u << b.A) - 1u) & ~endm;
  }
  if (held > 0u) ring_drain<P, T, D, MULTI>(a, ring, 0u, held);
}

template <class P, class T, int CV, bool MULTI, int STEPS, class A>
__device__ __forceinline__ void run_2d(const A& a) {
  PathState<T> s;
  LaneSeg<T> ls;
  init_lane<T, 2>(a, s, ls);
  cache_init(a);
  const ExitRing<T, 2> ring = ring_of_warp<T, 2>(a);
  RingCursor rc;
  bool active = false, exhausted = false;
  unsigned long long bnext = 0, bend = 0;
  uint32_t bseg = 0;
  spread_claim<MULTI>(a, bnext, bend, bseg);
  while (refill<T, 2, MULTI>(a, s, ls, active, bnext, bend, bseg, exhausted)) {
    // warp-uniform: few paths left, on to the drain
    if (exhausted && __popc(__ballot_sync(kFull, active)) <= Drain<T, 2>::kMaxRun) break;
    bool fin = false, trunc = false;
    // A path that ends leaves the iteration: one divergent region per iteration
    // with one branch per test.  As a chain of steps that each ask whether the
    // path still runs (a region, its join and a flag per step and half-step) the
    // plain 256 x 20,000 launch took 16.9 ms, now 15.3; with the control variate
    // 256 x 100,000 107.7 and 102.  Unrolled, the segment-table build takes 94
    // registers instead of 76 (fixed-error run 3.24 and 3.00 ms).
    if (active) {
#pragma unroll (MULTI ? 1 : STEPS / 2)
      for (int half = 0; half < STEPS / 2; ++half) {
        T n[3];
        n[2] = T(0);
        if (should_finish<P, T, 2>(s, ls.thr0)) {
          fin = true;
          break;
        }
        const uint4 w = path_block<MULTI>(a, s.seg, (uint32_t)(s.k >> 1), s.path, s.node);
        box_muller(w.x, w.y, n[0], n[1], ls.sqh, a.f64);
        euler_step<P, T, 2, CV, MULTI>(a, s, ls, n);
        if (s.k >= ls.max_steps) {
          fin = trunc = true;
          break;
        }
        if (should_finish<P, T, 2>(s, ls.thr0)) {
          fin = true;
          break;
        }
        box_muller(w.z, w.w, n[0], n[1], ls.sqh, a.f64);
        euler_step<P, T, 2, CV, MULTI>(a, s, ls, n);
        if (s.k >= ls.max_steps) {
          fin = trunc = true;
          break;
        }
      }
    }
    ring_exit<P, T, 2, MULTI>(a, ring, rc, s, active && fin, trunc);
    if (fin) active = false;
  }
  drain<P, T, 2, CV, MULTI>(a, ring, rc, s, ls, active);
  cache_flush(a);
}

// The segment-table build keeps per-lane segment parameters in registers.  Its
// short iteration is held to 64 of them: short paths want the warps (130
// segments x 217 nodes x 4,942 paths of 10 to 100 steps: 48.4 ms at 72
// registers, 47.3 at 64).
template <class T, bool MULTI, int STEPS>
constexpr int kMinBlocks2D = MULTI && sizeof(T) == 4 && STEPS == 2 ? 2 : PDD_MIN_BLOCKS_2D;
template <class P, class T, int CV, bool MULTI, int STEPS>
__global__ void __launch_bounds__(kMaxBlockThreads, (kMinBlocks2D<T, MULTI, STEPS>))
    paths_2d(const __grid_constant__ PathArgsN<kSegs<MULTI>> a) {
  run_2d<P, T, CV, MULTI, STEPS>(a);
}

// The segment-table build with the long iteration (FP32).  Left to itself it
// takes 76 registers and one block of 512 threads an SM; asked for two such
// blocks it fits 64 by trading the whole loop's schedule for them; under a limit
// on the registers alone ptxas finds a schedule of 64 that is faster than both.
// 128 segments x 2 nodes x 48,000 paths at h = 1e-4 with the control variate:
// 81.7 ms, 65.6 and 61.0 (plain 43.4, 45.7 and 43.4); 8 segments x 32 nodes x
// 8,000 paths 14.2 ms and 11.3; 128 x 2 x 1,387, where the drain weighs, 3.03 and
// 3.10.  (Bounds of 1,024 threads, 57 registers: 61.0, 42.8, 11.2, 3.15.)
template <class P, int CV>
__global__ void __maxnreg__(72)
    paths_2d_table(const __grid_constant__ PathArgs a) {
  run_2d<P, float, CV, true, LongSteps2D<float, CV>::value>(a);
}

// The long-iteration kernel of a build.
template <class P, class T, int CV, bool MULTI>
constexpr auto long_kernel_2d() {
  if constexpr (MULTI && sizeof(T) == 4) return paths_2d_table<P, CV>;
  else return paths_2d<P, T, CV, MULTI, LongSteps2D<T, CV>::value>;
}

// 3D: steps 4j .. 4j+3 use normals 12j .. 12j+11, i.e. Philox blocks 3j,
// 3j+1, 3j+2 (words a0..a3, b0..b3, c0..c3):
//   step 0: a0 a1 a2   step 1: a3 b0 b1   step 2: b2 b3 c0   step 3: c1 c2 c3
// Blocks are drawn only when the path is still running.  STEPS / 4 such
// groups of four steps run per iteration (between lane refills).
template <class P, class T, int CV, bool MULTI, int STEPS>
__global__ void __launch_bounds__(kMaxBlockThreads, PDD_MIN_BLOCKS_3D)
    paths_3d(const __grid_constant__ PathArgsN<kSegs<MULTI>> a) {
  PathState<T> s;
  LaneSeg<T> ls;
  init_lane<T, 3>(a, s, ls);
  cache_init(a);
  const ExitRing<T, 3> ring = ring_of_warp<T, 3>(a);
  RingCursor rc;
  bool active = false, exhausted = false;
  unsigned long long bnext = 0, bend = 0;
  uint32_t bseg = 0;
  spread_claim<MULTI>(a, bnext, bend, bseg);
  while (refill<T, 3, MULTI>(a, s, ls, active, bnext, bend, bseg, exhausted)) {
    if (exhausted && __popc(__ballot_sync(kFull, active)) <= Drain<T, 3>::kMaxRun) break;
    bool fin = false, trunc = false;
    // as in paths_2d; 9,216 nodes x 2,000 paths at h = 1e-3: 4.99 -> 4.50 ms
    // plain (4.67 unrolled), 8.89 -> 8.56 ms with the control variate (8.70
    // not unrolled), whose bound is L1: two record loads of 32 distinct lines
    // each are 64 wavefronts of its data pipe a warp step, 80 % of the cycles
    if (active) {
#pragma unroll (CV == kCvNone ? 1 : STEPS / 4)
      for (int quad = 0; quad < STEPS / 4; ++quad) {
        T n[3], carry0, carry1;  // carry: normals left over from the previous block
        const uint32_t blk0 = 3u * ((uint32_t)s.k >> 2);
        // step 0
        if (should_finish<P, T, 3>(s, ls.thr0)) {
          fin = true;
          break;
        }
        uint4 w = path_block<MULTI>(a, s.seg, blk0, s.path, s.node);
        box_muller(w.x, w.y, n[0], n[1], ls.sqh, a.f64);
        box_muller(w.z, w.w, n[2], carry0, ls.sqh, a.f64);
        euler_step<P, T, 3, CV, MULTI>(a, s, ls, n);
        if (s.k >= ls.max_steps) {
          fin = trunc = true;
          break;
        }
        // step 1
        if (should_finish<P, T, 3>(s, ls.thr0)) {
          fin = true;
          break;
        }
        w = path_block<MULTI>(a, s.seg, blk0 + 1u, s.path, s.node);
        n[0] = carry0;
        box_muller(w.x, w.y, n[1], n[2], ls.sqh, a.f64);
        euler_step<P, T, 3, CV, MULTI>(a, s, ls, n);
        if (s.k >= ls.max_steps) {
          fin = trunc = true;
          break;
        }
        // step 2
        if (should_finish<P, T, 3>(s, ls.thr0)) {
          fin = true;
          break;
        }
        box_muller(w.z, w.w, n[0], n[1], ls.sqh, a.f64);
        w = path_block<MULTI>(a, s.seg, blk0 + 2u, s.path, s.node);
        box_muller(w.x, w.y, n[2], carry1, ls.sqh, a.f64);
        euler_step<P, T, 3, CV, MULTI>(a, s, ls, n);
        if (s.k >= ls.max_steps) {
          fin = trunc = true;
          break;
        }
        // step 3
        if (should_finish<P, T, 3>(s, ls.thr0)) {
          fin = true;
          break;
        }
        n[0] = carry1;
        box_muller(w.z, w.w, n[1], n[2], ls.sqh, a.f64);
        euler_step<P, T, 3, CV, MULTI>(a, s, ls, n);
        if (s.k >= ls.max_steps) {
          fin = trunc = true;
          break;
        }
      }
    }
    ring_exit<P, T, 3, MULTI>(a, ring, rc, s, active && fin, trunc);
    if (fin) active = false;
  }
  drain<P, T, 3, CV, MULTI>(a, ring, rc, s, ls, active);
  cache_flush(a);
}

// ---------------------------------------------------------------------------
// Multilevel coupling: per lane a fine path at h_f = h/2 on the path's own
// stream and a coarse path at h driven by the sums of pairs of fine
// increments, dW_c(m) = dW_f(2m) + dW_f(2m+1).  Iteration j draws the
// Philox blocks that feed kFine fine steps (2D: block j, normals 4j .. 4j+3,
// two fine steps; 3D: blocks 3j .. 3j+2, normals 12j .. 12j+11, four fine
// steps) and the kFine / 2 coarse steps those increments make.  Each path
// has its own exit test; when both have finished the lane adds
// (phi_f, phi_f + xi_f) to the fine records (seg[0].acc) and the differences
// (phi_f - phi_c, psi_f - psi_c) with the coarse exit index to the
// difference records (seg[1].acc).  seg[0] holds the fine step and the node /
// path layout (path_off included), seg[1] the coarse step; emit pointers of
// seg[0] / seg[1] receive fine / coarse per-path output.
// ---------------------------------------------------------------------------
template <int D>
struct CoupledShape {
  static constexpr int kBlocks = D == 2 ? 1 : 3;        // Philox blocks per iteration
  static constexpr int kNormals = 4 * kBlocks;
  static constexpr int kFine = kNormals / D;            // fine steps per iteration
  static constexpr int kCoarse = kFine / 2;
};

// What a finished pair leaves: the two scores of each path, both exit indices.
template <class T>
struct PairEnd {
  T phif, xif, phic, xic;
  int kf, kc;
  uint32_t node, path, trunc;  // truncated: bit 0 fine, bit 1 coarse
};

// Per-warp ring of finished pairs (the coupled counterpart of ExitRing),
// drained 32 pairs at a time into the fine and difference records.
template <class T>
struct PairRing {
  static constexpr uint32_t kHalf = 32 * (4 * sizeof(T) + 5 * sizeof(uint32_t));
  static constexpr size_t kBytes = 2 * kHalf;
  char* base;
  __device__ __forceinline__ T* f(uint32_t j) const {
    return (T*)(base + (j >> 5) * kHalf) + (j & 31u);
  }
  __device__ __forceinline__ uint32_t* u(uint32_t j) const {
    return (uint32_t*)(base + (j >> 5) * kHalf + 32 * 4 * sizeof(T)) + (j & 31u);
  }
  __device__ __forceinline__ void put(uint32_t j, const PairEnd<T>& e) const {
    T* v = f(j);
    uint32_t* w = u(j);
    v[0] = e.phif;
    v[32] = e.xif;
    v[64] = e.phic;
    v[96] = e.xic;
    w[0] = (uint32_t)e.kf;
    w[32] = (uint32_t)e.kc;
    w[64] = e.node;
    w[96] = e.path;
    w[128] = e.trunc;
  }
};

template <class T, class A>
__device__ __forceinline__ PairRing<T> pair_ring_of_warp(const A& a) {
  return {(char*)s_cache + cache_bytes(a.cache_nodes) +
          (size_t)(threadIdx.x >> 5) * PairRing<T>::kBytes};
}

template <class T, class A>
__device__ __forceinline__ void pair_drain(const A& a, const PairRing<T>& r,
                                           uint32_t first, uint32_t count) {
  __syncwarp();
  const uint32_t lane = threadIdx.x & 31u;
  if (lane < count) {
    const uint32_t j = (first + lane) & (kRing - 1);
    const T* v = r.f(j);
    const uint32_t* w = r.u(j);
    const T phif = v[0], xif = v[32], phic = v[64], xic = v[96];
    const int kf = (int)w[0], kc = (int)w[32];
    const uint32_t node = w[64], path = w[96], tr = w[128];
    const SegArgs& s0 = a.seg[0];
    const SegArgs& s1 = a.seg[1];
    record_path(a, s0, node, phif, phif + xif, kf, (tr & 1u) != 0u);
    record_path(a, s1, node, phif - phic, (phif + xif) - (phic + xic), kc, (tr & 2u) != 0u);
    if (s0.emit_phi != nullptr &&
        PDD_IN_BOUNDS(a, (size_t)node * s0.emit_stride + path < s0.n_nodes * s0.emit_stride,
                      kErrBoundsEmit)) {
      const size_t i = (size_t)node * s0.emit_stride + path;
      s0.emit_phi[i] = (float)phif;
      s0.emit_xi[i] = (float)xif;
      s0.emit_steps[i] = kf;
      s1.emit_phi[i] = (float)phic;
      s1.emit_xi[i] = (float)xic;
      s1.emit_steps[i] = kc;
    }
  }
  __syncwarp();
}

// Per-lane state of a pair.
template <class T>
struct PairState {
  PathState<T> f, c;  // fine and coarse path
  bool af, ac;        // still running
  bool tf, tc;        // truncated
  T phif, xif, phic, xic;
  uint32_t j;         // iterations of CoupledShape done
  __device__ __forceinline__ PairEnd<T> end() const {
    return {phif, xif, phic, xic, f.k, c.k, f.node, f.path, (tf ? 1u : 0u) | (tc ? 2u : 0u)};
  }
};

// The drain of a warp's last pairs (see Drain): a batch draws the fine path's
// normals once and takes S fine steps, then the S / 2 coarse ones that their
// sums make.  A pair whose one path has ended goes on with the other.
// 1,024 pairs at h = 1e-3 took 696 us plain and 935 us with the control variate
// in ordinary iterations of one lane per pair, a step of which is as deep as
// both paths' steps and the random numbers of a lane.
template <class T, int D>
struct PairDrain {
  // 2D scratch: 4 normals, X or c and f of two steps and their dots per lane
  static constexpr int kLanes = PairRing<T>::kHalf / (10 * sizeof(T)) < 32
                                    ? PairRing<T>::kHalf / (10 * sizeof(T))
                                    : 32;
  static constexpr int kMaxRun = D == 2 ? 14 : 8;
  __device__ static int blocks(int A) { return D == 2 ? kLanes / A : 3 * (8 / A); }
  __device__ static int steps(int A) { return D == 2 ? 2 * (kLanes / A) : 4 * (8 / A); }
};
static_assert(32 * 6 * sizeof(float) <= PairRing<float>::kHalf, "3D pair drain scratch");

template <class P, class T, int D, int CV, class A>
__device__ __forceinline__ void drain_pairs(const A& a, const PairRing<T> ring,
                                            RingCursor rc, PairState<T> s, const LaneSeg<T>& lf,
                                            const LaneSeg<T>& lc, bool active) {
  using S4 = CoupledShape<D>;
  using Shape = PairDrain<T, D>;
  uint32_t held = rc.held;
  ring_move<4, 5>(ring, rc);
  T* const nrm = (T*)(ring.base + PairRing<T>::kHalf);
  T* const pos = nrm + (D == 2 ? 4 * Shape::kLanes : 96);
  T* const dots = pos + 4 * Shape::kLanes;  // 2D
  const SegArgs& sg = a.seg[0];
  unsigned runm = __ballot_sync(kFull, active);
  while (runm != 0u) {
    const BatchLane b(__popc(runm));
    const int src = nth_set_bit(runm, b.q);
    take_path<T, D>(s.f, src);
    take_path<T, D>(s.c, src);
    s.f.node = __shfl_sync(kFull, s.f.node, src);
    s.f.path = __shfl_sync(kFull, s.f.path, src);
    s.j = __shfl_sync(kFull, s.j, src);
    s.phif = __shfl_sync(kFull, s.phif, src);
    s.xif = __shfl_sync(kFull, s.xif, src);
    s.phic = __shfl_sync(kFull, s.phic, src);
    s.xic = __shfl_sync(kFull, s.xic, src);
    const unsigned flags = __shfl_sync(kFull, (s.af ? 1u : 0u) | (s.ac ? 2u : 0u) |
                                                  (s.tf ? 4u : 0u) | (s.tc ? 8u : 0u), src);
    s.af = (flags & 1u) != 0u;
    s.ac = (flags & 2u) != 0u;
    s.tf = (flags & 4u) != 0u;
    s.tc = (flags & 8u) != 0u;
    const int blocks = Shape::blocks(b.A), S = Shape::steps(b.A);
    unsigned endm = 0u;
    do {
      if (b.m < blocks)
        batch_normals<T, D>(b, S4::kBlocks * s.j + (uint32_t)b.m, s.f.path, s.f.node, sg.seed_hi,
                            make_uint2(sg.key0, sg.key1), lf.sqh, nrm, a.f64);
      __syncwarp();
      bool trunc = false;
      int n = batch_steps<P, T, D, CV, false>(a, lf, s.f, nrm, pos, dots, 1, b, S, s.af,
                                              CV != kCvNone, a.y_exp != 0, trunc);
      if (s.af && (trunc || n < S)) {
        s.af = false;
        s.tf = trunc;
        score_path<P, T, D>(s.f, s.phif, s.xif);
      }
      __syncwarp();
      n = batch_steps<P, T, D, CV, true>(a, lc, s.c, nrm, pos, dots, 1, b, S / 2, s.ac,
                                         CV != kCvNone, a.y_exp != 0, trunc);
      if (s.ac && (trunc || n < S / 2)) {
        s.ac = false;
        s.tc = trunc;
        score_path<P, T, D>(s.c, s.phic, s.xic);
      }
      s.j += (uint32_t)(S / S4::kFine);
      endm = __ballot_sync(kFull, b.lane < b.A && !s.af && !s.ac);
      __syncwarp();
    } while (endm == 0u);
    const uint32_t ended = (uint32_t)__popc(endm);
    if (held + ended > 32u) {
      pair_drain<T>(a, ring, 0u, held);
      held = 0;
    }
    if ((endm >> b.lane) & 1u)
      ring.put(held + (uint32_t)__popc(endm & ((1u << b.lane) - 1u)), s.end());
    held += ended;
    runm = ((1u << b.A) - 1u) & ~endm;
  }
  if (held > 0u) pair_drain<T>(a, ring, 0u, held);
}

template <class P, class T, int CV, int D>
__global__ void __launch_bounds__(kMaxBlockThreads, 1) paths_coupled(
    const __grid_constant__ PathArgsN<2> a) {
  using S = CoupledShape<D>;
  const PairRing<T> ring = pair_ring_of_warp<T>(a);
  RingCursor rc;
  PairState<T> p;
  PathState<T>& f = p.f;
  PathState<T>& c = p.c;
  LaneSeg<T> lf, lc;
  init_lane<T, D>(a, f, lf);
  init_lane<T, D>(a, c, lc);
  load_seg<T, D>(a.seg[1], lc);
  p.af = p.ac = p.tf = p.tc = false;
  p.phif = p.xif = p.phic = p.xic = T(0);
  p.j = 0;
  cache_init(a);
  bool active = false, exhausted = false;  // active: the pair still has work
  unsigned long long bnext = 0, bend = 0;
  uint32_t bseg = 0;
  spread_claim<false>(a, bnext, bend, bseg);
  while (refill<T, D, false>(a, f, lf, active, bnext, bend, bseg, exhausted)) {
    if (active && f.k == 0 && !p.af && !p.ac) {  // refill has just started a new pair in f
      c = f;
      p.af = p.ac = true;
      p.tf = p.tc = false;
      p.j = 0;
    }
    if (exhausted && __popc(__ballot_sync(kFull, active)) <= PairDrain<T, D>::kMaxRun) break;
    if (active) {
      T n[S::kNormals];
#pragma unroll
      for (int b = 0; b < S::kBlocks; ++b) {
        const uint4 w = path_block<false>(a, 0, S::kBlocks * p.j + b, f.path, f.node);
        box_muller(w.x, w.y, n[4 * b], n[4 * b + 1], lf.sqh, a.f64);
        box_muller(w.z, w.w, n[4 * b + 2], n[4 * b + 3], lf.sqh, a.f64);
      }
      if (p.af) {
#pragma unroll
        for (int q = 0; q < S::kFine; ++q) {
          if (p.af) {
            if (should_finish<P, T, D>(f, lf.thr0)) {
              p.af = false;
            } else {
              T d[3] = {n[D * q], n[D * q + 1], D == 3 ? n[D * q + 2] : T(0)};
              euler_step<P, T, D, CV, false, true>(a, f, lf, d);
              if (f.k >= lf.max_steps) {
                p.af = false;
                p.tf = true;
              }
            }
          }
        }
        if (!p.af) score_path<P, T, D>(f, p.phif, p.xif);
      }
      if (p.ac) {
#pragma unroll
        for (int q = 0; q < S::kCoarse; ++q) {
          if (p.ac) {
            if (should_finish<P, T, D>(c, lc.thr0)) {
              p.ac = false;
            } else {
              const int o = 2 * D * q;  // fine steps 2q and 2q+1 of this iteration
              T d[3] = {add_rn(n[o], n[o + D]), add_rn(n[o + 1], n[o + D + 1]),
                        D == 3 ? add_rn(n[o + 2], n[o + D + 2]) : T(0)};
              euler_step<P, T, D, CV, false, true>(a, c, lc, d);
              if (c.k >= lc.max_steps) {
                p.ac = false;
                p.tc = true;
              }
            }
          }
        }
        if (!p.ac) score_path<P, T, D>(c, p.phic, p.xic);
      }
      p.j += 1;
    }
    // park finished pairs; drain 32 at a time with the whole warp
    const bool done = active && !p.af && !p.ac;
    const unsigned m = __ballot_sync(kFull, done);
    // never more than kRing parked: fewer than 32 are held before this iteration
    // (bounds-checked build: an over-full ring drops the pairs, never stalls)
    if (m != 0u && !PDD_IN_BOUNDS(a, rc.held + __popc(m) <= kRing, kErrBoundsRing)) {
      if (done) active = false;
    } else if (m != 0u) {
      if (done) {
        const unsigned lt = (1u << (threadIdx.x & 31u)) - 1u;
        ring.put((rc.head + __popc(m & lt)) & (kRing - 1), p.end());
        active = false;
      }
      rc.head += __popc(m);
      rc.held += __popc(m);
      if (rc.held >= 32u) {
        pair_drain<T>(a, ring, rc.head - rc.held, 32u);
        rc.held -= 32u;
      }
    }
  }
  drain_pairs<P, T, D, CV>(a, ring, rc, p, lf, lc, active);
  cache_flush(a);
}

// ---------------------------------------------------------------------------
// Launch dispatch.
// ---------------------------------------------------------------------------
// Whether a launch keeps its records in shared memory.  Finished paths cost
// about 10 ns each per record line in L2 (13 atomics on one line), so the cache
// pays when few records take many exits: 1.5e9 path-steps on 64 nodes take
// 5.8 ms with it and 9.6 ms without at 100 steps a path, 5.5 and 5.5 ms at
// 330; on 256 nodes 10 and 34 ms at 10 steps, 5.7 and 5.6 ms at 100.  But its
// copies take shared memory from L1, and with less than about 40 KB of L1 left
// the gathers of the control variate starve: 480 records in two blocks an SM
// (204 KB) run 2e9 path-steps in 13.7 ms against 9.5 ms without the cache, 448
// records (196 KB) 9.3 ms.  So:
//  - a spread launch, in 128-thread blocks with a copy each, caches up to 64
//    records (1 node x 18,000 10-step paths: 38 us with, 197 us without; 256
//    nodes: no difference);
//  - a kernel that lives by L1 (`l1`: a control grid, or the coupled kernels,
//    which have room for one such block only: 21.3 against 19.2 ms) caches more
//    than kCacheL1Bytes only when records x mean steps is under 2e4.
// The mean number of steps is taken as 0.1 / h, that of the unit box.
constexpr size_t kCacheL1Bytes = 97 * 1024;  // per block, rings included
static bool use_cache(const PathArgs& a, unsigned long long records, bool spread, bool l1,
                      size_t smem) {
  if (records == 0 || records > kCacheMaxNodes) return false;
  if (spread) return records <= 64;
  if (!l1 || smem <= kCacheL1Bytes) return true;
  double paths = 0.0, steps = 0.0;
  for (int i = 0; i < a.n_segs; ++i) {
    paths += (double)a.seg[i].total;
    steps += (double)a.seg[i].total * 0.1 / a.seg[i].h;
  }
  return (double)records * steps < 2e4 * paths;
}

// Shared-memory record slots of a launch: the segments' nodes in segment order.
template <class A>
static void place_records(A& b) {
  uint32_t base = 0;
  for (int i = 0; i < b.n_segs; ++i) {
    b.seg[i].cache_base = base;
    base += (uint32_t)b.seg[i].n_nodes;
  }
  b.cache_nodes = base;
}

// Default block size of launches with the record cache: large, so that many
// warps share one copy of the records, and two blocks to an SM where that
// costs few warps (up to 64 registers a thread: 512 threads, 72: 448, which
// measured 23.0 -> 16.6 ms on 512 nodes x 10-step paths against one block of
// 512; the coupled kernels, above 72, are faster with one).  A caller's choice
// of more threads, made for another kernel, is cut to it (31,744 nodes of the
// anisotropic problem, 69 registers: 75.3 ms with 512 threads, 62.3 with 448).
constexpr int kTwoBlocks72 = 448;
static int cache_block_threads(int regs) { return regs > 64 && regs <= 72 ? kTwoBlocks72 : 512; }

// Whether a launch takes the long iteration (see kLongPathH).
static bool long_iterations(const PathArgs& a) {
  double all = 0.0, shorter = 0.0;
  for (int i = 0; i < a.n_segs; ++i) {
    const double w = (double)a.seg[i].total / a.seg[i].h;
    all += w;
    if (!(a.seg[i].h <= kLongPathH)) shorter += w;
  }
  return shorter <= kShortWorkShare * all;
}

// Paths per lane a warp claims from the launch's cursor at once.  Automatic:
// 4 when the launch's paths are short (the segments with time steps of at
// most kLongPathH hold at most kShortWorkShare of its expected path-steps)
// and it has at least kAutoClaim x 32 paths for every warp that can be
// resident (64 per SM), else 1.  A claim of c paths per lane means one
// cursor atomic per 32 c paths: with ~10-step paths the cursor is hit at a
// rate where that matters (measured +4.5 % path-steps/s with c = 4 on
// 10-step paths; no change on 100-step paths), while with long paths the
// paths a warp still holds unstarted lengthen the end of the launch.
constexpr int kAutoClaim = 4;
static int resolve_claim(const PathArgs& a, int num_sms) {
  if (a.claim > 0) return a.claim;
  double all = 0.0, longer = 0.0;
  for (int i = 0; i < a.n_segs; ++i) {
    const double w = (double)a.seg[i].total / a.seg[i].h;
    all += w;
    if (a.seg[i].h <= kLongPathH) longer += w;
  }
  const unsigned long long enough =
      (unsigned long long)kAutoClaim * kWarpBatch * 64ull * (unsigned long long)num_sms;
  return (longer <= kShortWorkShare * all && a.total >= enough) ? kAutoClaim : 1;
}

// Paths per warp of a launch too small to fill the chip, 0 for the others.
// Such a launch is over when its longest path is, and a step of a warp's paths
// takes the less time the fewer paths the warp holds, as the other lanes then
// work for them (see Drain): 1,024 paths at h = 1e-4 take 830 us as 32 full
// warps and 330 us as 1,024 warps of one path.  More than about 2.5 warps per
// scheduler compete for its issue slots instead (5,120 paths: 435 us with 2
// per warp, 450 with 4, 532 with 8; 20,480 paths: 685 us with 8, 621 with 12,
// 703 with 16), and from 24 paths per warp on a full chip in ordinary
// iterations is as fast (102,400 paths: 1,376 us with 24, 1,485 with 32).
// Short paths end before the sharing pays: 100,000 of 10 steps take 37 us in
// full warps and 43 with 24 paths per warp (20,480: 31 us and 27 with 12).
// FP64 paths are bound by the SM's one FP64 pipe, which a warp's instruction
// holds as long for one lane as for 32: they get one warp per scheduler.
constexpr int kSpreadMax = 24;
template <class T>
static int spread_batch(const PathArgs& a, int num_sms) {
  const unsigned long long sms = (unsigned long long)num_sms;
  const unsigned long long want = sizeof(T) == 4 ? 10 * sms : 4 * sms;  // warps
  const unsigned long long each = (a.total + want - 1) / want;
  if (a.claim > 0) return 0;  // the caller chose the claim
  const bool longer = long_iterations(a);
  if (each <= (unsigned long long)(longer ? kSpreadMax : kSpreadMax / 2)) return (int)each;
  return sizeof(T) == 4 && longer && a.total <= kSpreadMax * 32ull * sms ? kSpreadMax : 0;
}

// Idle lanes at which a warp starts new paths.  Starting one costs the whole
// warp a path's set-up, so short paths, of which some lane ends at almost every
// iteration, are started a few at a time; a lane that waits loses steps, so
// long ones are not.  1.5e9 path-steps of the plain 2D problem with 1, 2, 3, 6
// and 8 lanes: 9.44, 9.38, 9.26, 8.98, 8.96 ms at 10 steps a path; 7.61, 7.31,
// 7.12, 6.99, 7.05 at 25; 5.11, 5.05, 5.05, 5.17, 5.30 at 100; 4.84, 4.79, 4.82,
// 4.99, 5.13 at 250; 5.22, 5.25, 5.29, 5.42, 5.62 at 1,000.  The lines are the
// same with the control variate and on the other problems.  FP64 paths: 1.
template <class T>
static int refill_min(const PathArgs& a) {
  double paths = 0.0, steps = 0.0;  // 0.1 / h steps a path, that of the unit box
  for (int i = 0; i < a.n_segs; ++i) {
    paths += (double)a.seg[i].total;
    steps += (double)a.seg[i].total * 0.1 / a.seg[i].h;
  }
  if (sizeof(T) == 8 || steps > 500.0 * paths) return 1;
  return steps > 150.0 * paths ? 2 : steps > 30.0 * paths ? 3 : 6;
}

// Warps per SM a launch asks for, 0 for all that fit.  With few paths per lane a
// launch's end weighs as much as its bulk, and the fewer warps share an SM's
// issue slots then the faster the longest paths go, while 24 (16 for the plain
// 2D step, which waits for no load) fill them as well as 28 or 32: 256 nodes x
// 1,000 paths at h = 1e-4 take 2.36 ms with 28 warps and 2.17 with 24 with the
// control variate, 1.70 with 28 and 1.46 with 16 plain; x 8,000 paths 9.50 and
// 9.67, 6.68 and 6.77.  Short paths finish so often that the plain step too
// wants 24 (x 2,000 paths at h = 1e-2: 70 us with 28, 72 with 24, 78 with 16).
// FP64 paths wait for the SM's one FP64 pipe, which six warps keep busy, four
// almost: 64 nodes x 1,000 paths at h = 1e-3 take 4.5 ms with 12 warps, 3.3 with
// 6 and with 4, x 16,000 paths 27.0, 26.2 and 28.1.
template <class T, int D, int CV>
static int target_warps(const PathArgs& a, int num_sms) {
  if (a.block_threads > 0 || a.max_blocks > 0) return 0;  // the caller chose the shape
  const auto few = [&](int warps) { return a.total <= 8ull * 32ull * warps * num_sms; };
  if (sizeof(T) == 8) return few(4) ? 4 : 6;
  if (D == 2 && CV == kCvNone && long_iterations(a) && few(16)) return 16;
  return few(24) ? 24 : 0;
}

// Persistent launch of `kern` over the flat index space of `a`: occupancy x
// SM count blocks (at most one warp per 32 paths), with the record cache
// when the launch's nodes fit it and `ring_per_warp` bytes of exit ring per
// warp.  `spread` > 0: that many paths per warp (see spread_batch), in blocks
// of 128 threads so that the warps cover the SMs evenly.  `warps`: see
// target_warps; `refill`: see refill_min; `l1`: see use_cache.  `occ_cache` is
// the kernel's own (static) state: its registers and the occupancy per block
// size without the cache, the same on every device that runs this code (it is
// compiled for one architecture).
template <int N>
static cudaError_t launch_persistent(void (*kern)(PathArgsN<N>), const PathArgs& a, int num_sms,
                                     cudaStream_t st, LaunchInfo* info, size_t ring_per_warp, int spread,
                                     int warps, int refill, bool l1, std::atomic<int>* occ_cache) {
  if (a.n_segs > N) return cudaErrorInvalidValue;
  PathArgsN<N> b;
  (PathHead&)b = a;
  b.refill_min = refill;
  for (int i = 0; i < a.n_segs; ++i) {
    b.seg[i] = a.seg[i];
    b.seg[i].h32 = (float)a.seg[i].h;
    b.seg[i].sqrt_h32 = (float)a.seg[i].sqrt_h;
    b.seg[i].thr32 = (float)a.seg[i].thr0;
  }
  b.warp_batch = spread > 0 ? (unsigned long long)spread
                            : kWarpBatch * (unsigned long long)resolve_claim(a, num_sms);
  unsigned long long records = 0;
  for (int i = 0; i < a.n_segs; ++i) records += a.seg[i].n_nodes;
  int threads = a.block_threads > 0 ? a.block_threads : kBlockThreads;
  if (threads % 32 != 0 || threads > kMaxBlockThreads) return cudaErrorInvalidValue;
  const bool sized = a.block_threads <= 0 && spread == 0 && records <= kCacheMaxNodes;
  if (sized || threads > kTwoBlocks72) {
    // occ_cache[0] keeps the kernel's register count (block sizes start at 32)
    int regs = occ_cache[0].load(std::memory_order_relaxed);
    if (regs == 0) {
      cudaFuncAttributes fa;
      cudaError_t e = cudaFuncGetAttributes(&fa, kern);
      if (e != cudaSuccess) return e;
      regs = fa.numRegs > 0 ? fa.numRegs : 1;
      occ_cache[0].store(regs, std::memory_order_relaxed);
    }
    const int most = cache_block_threads(regs);
    if (sized || threads > most) threads = most;
  }
  if (sized) {
    // a launch that does not fill the chip: as many warps on every SM
    unsigned long long per_sm =
        ((a.total + b.warp_batch - 1ull) / b.warp_batch + num_sms - 1) / num_sms;
    if (warps > 0 && per_sm > (unsigned long long)warps) per_sm = warps;
    const unsigned long long full = (unsigned long long)threads / 32;
    if (per_sm <= full) threads = 32 * (int)per_sm;
    else if (per_sm <= 2 * full) threads = 32 * (int)((per_sm + 1) / 2);
  }
  size_t cache = 0;
  b.cache_nodes = 0;
  if (use_cache(a, records, spread > 0, l1,
                cache_bytes((uint32_t)records) + (size_t)(threads / 32) * ring_per_warp)) {
    cache = cache_bytes((uint32_t)records);
    place_records(b);
  } else if (a.block_threads <= 0) {
    threads = kBlockThreads;
  }
  const size_t smem = cache + (size_t)(threads / 32) * ring_per_warp;
  if (smem > 48u * 1024u) {
    // for the current device alone, so at every such launch (0.2 us)
    const int lim = (int)(cache_bytes(kCacheMaxNodes) + (kMaxBlockThreads / 32) * ring_per_warp);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (e != cudaSuccess) return e;
  }
  int occ = 0;
  const int known = occ_cache[threads / 32].load(std::memory_order_relaxed);
  if (cache == 0 && known != 0) {
    occ = known;
  } else {
    int v = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, threads, smem);
    if (e != cudaSuccess) return e;
    occ = v > 0 ? v : 1;
    if (cache == 0) occ_cache[threads / 32].store(occ, std::memory_order_relaxed);
  }
  const unsigned long long warps_needed = (a.total + b.warp_batch - 1ull) / b.warp_batch;
  const unsigned long long blocks_needed =
      (warps_needed + (threads / 32) - 1) / (threads / 32);
  unsigned long long nb = (unsigned long long)occ * (unsigned long long)num_sms;
  if (spread > 0 && nb < blocks_needed) nb = blocks_needed;
  if (spread == 0 && warps > 0) {
    const unsigned long long most =
        (unsigned long long)num_sms * ((32 * warps + threads - 1) / threads);
    if (nb > most) nb = most;
  }
  if (a.max_blocks > 0 && nb > (unsigned long long)a.max_blocks) nb = a.max_blocks;
  if (nb > blocks_needed) nb = blocks_needed;
  if (nb < 1) nb = 1;
  b.one_claim = spread > 0 && nb == blocks_needed;  // the warps' single batches cover every path
  info->blocks = (int)nb;
  info->threads = threads;
  info->cached_records = b.cache_nodes;
  info->paths_per_warp = b.one_claim ? spread : 0;
  info->cursor_end = b.one_claim ? (nb * (threads / 32)) * kSpreadClaim : a.total;
  kern<<<(unsigned)nb, (unsigned)threads, smem, st>>>(b);
  return cudaGetLastError();
}


template <class P, class T, int CV, bool MULTI>
static cudaError_t launch_one(const PathArgs& a, int num_sms, cudaStream_t st, LaunchInfo* info) {
  // FP64 paths: the step dominates, they always take the short iteration
  const bool longer = sizeof(T) == 4 && (a.iter_mode == PDD_ITER_LONG ||
                                         (a.iter_mode == PDD_ITER_AUTO && long_iterations(a)));
  const int spread = spread_batch<T>(a, num_sms);
  const int warps = target_warps<T, P::kDim, CV>(a, num_sms);
  const int refill = refill_min<T>(a);
  if constexpr (P::kDim == 3) {
    if (longer) {
      static std::atomic<int> per_sm[kMaxBlockThreads / 32 + 1];
      return launch_persistent(paths_3d<P, T, CV, MULTI, sizeof(T) == 4 ? 8 : 4>, a, num_sms, st,
                               info, ExitRing<T, 3>::kBytes, spread, warps, refill,
                               CV == kCvGrid, per_sm);
    }
    static std::atomic<int> per_sm[kMaxBlockThreads / 32 + 1];
    return launch_persistent(paths_3d<P, T, CV, MULTI, 4>, a, num_sms, st, info,
                             ExitRing<T, 3>::kBytes, spread, warps, refill, CV == kCvGrid, per_sm);
  } else if (longer) {
    static std::atomic<int> per_sm[kMaxBlockThreads / 32 + 1];
    return launch_persistent(long_kernel_2d<P, T, CV, MULTI>(), a, num_sms, st, info,
                             ExitRing<T, 2>::kBytes, spread, warps, refill, CV == kCvGrid,
                             per_sm);
  } else {
    static std::atomic<int> per_sm[kMaxBlockThreads / 32 + 1];
    return launch_persistent(paths_2d<P, T, CV, MULTI, 2>, a, num_sms, st, info,
                             ExitRing<T, 2>::kBytes, spread, warps, refill, CV == kCvGrid, per_sm);
  }
}

template <class P, class T, int CV, bool MULTI>
static cudaError_t occupancy_one(int threads, int* occ) {
  if (threads % 32 != 0 || threads < 32 || threads > kMaxBlockThreads) return cudaErrorInvalidValue;
  void (*kern)(PathArgsN<kSegs<MULTI>>);
  if constexpr (P::kDim == 3)
    kern = paths_3d<P, T, CV, MULTI, sizeof(T) == 4 ? 8 : 4>;
  else
    kern = long_kernel_2d<P, T, CV, MULTI>();
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      occ, kern, threads, (size_t)(threads / 32) * ExitRing<T, P::kDim>::kBytes);
}

template <class P, class T, bool MULTI>
static cudaError_t occupancy_cv(int cv, int threads, int* occ) {
  switch (cv) {
    case kCvNone: return occupancy_one<P, T, kCvNone, MULTI>(threads, occ);
    case kCvGrid: return occupancy_one<P, T, kCvGrid, MULTI>(threads, occ);
    default: return occupancy_one<P, T, kCvExact, MULTI>(threads, occ);
  }
}

template <class P, class T, bool MULTI>
static cudaError_t launch_cv(int cv, const PathArgs& a, int sms, cudaStream_t st, LaunchInfo* info) {
  switch (cv) {
    case kCvNone: return launch_one<P, T, kCvNone, MULTI>(a, sms, st, info);
    case kCvGrid: return launch_one<P, T, kCvGrid, MULTI>(a, sms, st, info);
    default: return launch_one<P, T, kCvExact, MULTI>(a, sms, st, info);
  }
}

template <class P, class T, int CV, int D>
static cudaError_t launch_coupled_one(const PathArgs& a, int num_sms, cudaStream_t st,
                                      LaunchInfo* info) {
  static std::atomic<int> per_sm[kMaxBlockThreads / 32 + 1];
  return launch_persistent(paths_coupled<P, T, CV, D>, a, num_sms, st, info,
                           PairRing<T>::kBytes, spread_batch<T>(a, num_sms), 0, 1, true,
                           per_sm);
}

template <class P, class T, int D>
static cudaError_t launch_coupled_cv(int cv, const PathArgs& a, int sms, cudaStream_t st,
                                     LaunchInfo* info) {
  switch (cv) {
    case kCvNone: return launch_coupled_one<P, T, kCvNone, D>(a, sms, st, info);
    case kCvGrid: return launch_coupled_one<P, T, kCvGrid, D>(a, sms, st, info);
    default: return launch_coupled_one<P, T, kCvExact, D>(a, sms, st, info);
  }
}

// The kernels of problem P.  3D launches always run the segment-table build:
// on GB300 it measured 1.43x faster than the single-segment build on one
// segment (1.26e11 vs 8.8e10 path-steps/s; ncu showed the single-segment build
// stalled on the texture/MIO queues), so the latter is not instantiated.
template <class P>
cudaError_t PathLaunch<P>::paths(int precision, int cv, bool multi, const PathArgs& a, int num_sms,
                                 cudaStream_t st, LaunchInfo* info) {
  constexpr bool kTable = P::kDim == 3;
  if (precision == 1)
    return multi ? launch_cv<P, double, true>(cv, a, num_sms, st, info)
                 : launch_cv<P, double, kTable>(cv, a, num_sms, st, info);
  return multi ? launch_cv<P, float, true>(cv, a, num_sms, st, info)
               : launch_cv<P, float, kTable>(cv, a, num_sms, st, info);
}

template <class P>
cudaError_t PathLaunch<P>::occupancy(int precision, int cv, bool multi, int threads, int* occ) {
  constexpr bool kTable = P::kDim == 3;
  if (precision == 1)
    return multi ? occupancy_cv<P, double, true>(cv, threads, occ)
                 : occupancy_cv<P, double, kTable>(cv, threads, occ);
  return multi ? occupancy_cv<P, float, true>(cv, threads, occ)
               : occupancy_cv<P, float, kTable>(cv, threads, occ);
}

template <class P>
cudaError_t PathLaunch<P>::coupled(int cv, const PathArgs& a, int num_sms, cudaStream_t st,
                                   LaunchInfo* info) {
  return launch_coupled_cv<P, float, P::kDim>(cv, a, num_sms, st, info);
}

}  // namespace pdd
