// One-level space-time restricted additive Schwarz preconditioner (Sec. 3.2)
// with ILU(0) subdomain solves, all subdomains in one launch.
//
// Subdomains.  The node range of each axis and the level range 0..M are cut
// into nsub parts (part k of n holds floor(n/p) + (k < n mod p)); a box is the
// product of one part per axis (owned set), extended by `overlap` on every
// side and trimmed to the domain (extended set, Fig. 1).  The subdomain
// matrix M_ij is the principal submatrix of F_h on the extended set, i.e. the
// discretisation with homogeneous Dirichlet data on every cut face in space
// and time (Eq. 10-12).
//
// Storage.  A row of F_h is described by its row type (C, G or f) and a fixed
// list of slots (level offset dt, spatial offset, column component) -- the
// structural stencil of that block row, ordered as the columns are ordered
// (time slowest, then z, y, x, then component).  Every point of a box stores
// 108 + 56 + 162 = 326 slot values, no column indices; slots whose column is
// outside the box hold 0, which is the same as leaving them out of the
// pattern.
//
// Layout in HBM.  The points of each wavefront are stored in groups of 8 (fewer
// in boxes of a few points a wavefront: ras.cuh), one after the other; the values of a group form one block, the L-slots first,
// then the diagonals and U-slots, so the forward sweep streams the lower
// halves of the groups in order and the backward sweep the upper halves.  In
// FP32 and BF16 a half is ordered by the lanes of the solve (lane_place, ras.cuh),
// in FP64 by slot rank ([rank][points of a group]).
//
// Ordering and parallelism.  Points are processed in the natural
// (lexicographic) order of the box; with this stencil every lower-triangular
// dependency of point (x, y, z, t) lies on a wavefront w' < w where
// w = x + 2y + 4z + 8t, so all points of one wavefront are independent.  Within
// a point the rows go C, G, f.  A box is worked on by one CTA or a cluster: the
// factorisations have a barrier between wavefronts, the solve a counter of
// finished groups.
//
// ILU(0) (IKJ form, on the structural pattern):
//   for each row i in order, for each k < i in pattern(i) ascending:
//     a_ik /= u_kk;  a_ij -= a_ik u_kj  for j > k in pattern(i) and pattern(k).
// The (row slot, column slot) pairs of the inner update are fixed per row
// type and written out as straight-line code (ilu_rows.inc).  The diagonal
// slot of a factored row stores 1/u_kk, so both the factorisation and the
// backward sweep multiply instead of divide.
//
// Solve.  One CTA per box, or a cluster of 2 to 8 where few boxes leave SMs
// idle; a warp takes a group of points of the wavefront.  The local vector of
// each box has a ghost layer of zeros one point wide in every direction, so the
// triangular sweeps need no bounds tests: a slot whose column leaves the box
// reads 0 and has factor value 0.

#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include <cuda_bf16.h>

#include "internal.cuh"
#include "ras.cuh"

namespace {

// ---------------------------------------------------------------------------
// slot tables (host-built, copied to constant memory)
// ---------------------------------------------------------------------------
struct SlotTables {
  // per slot (0..325): packed offsets
  int8_t dt[kSlots], dz[kSlots], dy[kSlots], dx[kSlots], comp[kSlots];
  int base[3], count[3], diag[3];       // diag = absolute slot index of the diagonal
};

SlotTables build_tables() {
  SlotTables T;
  int s = 0;
  for (int c = 0; c < 3; ++c) {
    T.base[c] = s;
    const int dt_lo = (c == 1) ? 0 : -1;
    const int dt_hi = (c == 0) ? 0 : 1;
    for (int dt = dt_lo; dt <= dt_hi; ++dt)
      for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
          for (int dx = -1; dx <= 1; ++dx)
            for (int cc = 0; cc < 3; ++cc) {
              bool use;
              if (c == 0) use = (cc == 0 || cc == 2);
              else if (c == 1) use = (cc == 1) || (cc == 0 && dx == 0 && dy == 0 && dz == 0);
              else use = (cc == 1 || cc == 2);
              if (!use) continue;
              T.dt[s] = (int8_t)dt; T.dz[s] = (int8_t)dz; T.dy[s] = (int8_t)dy; T.dx[s] = (int8_t)dx;
              T.comp[s] = (int8_t)cc;
              if (dt == 0 && dz == 0 && dy == 0 && dx == 0 && cc == c) T.diag[c] = s;
              ++s;
            }
    T.count[c] = s - T.base[c];
  }
  return T;
}

const SlotTables& tables() {
  static const SlotTables T = build_tables();
  return T;
}

// Checksum of the slot list and group rank of every slot, as the
// generated factorisation code (factor32.cu, factor64.cu) assumes them.
#include "ilu_slots.inc"

// Slot ranges of the three row types (checked against the tables on the host).
constexpr int kCBase = 0, kCDiag = 80, kCEnd = 108;
constexpr int kGBase = 108, kGDiag = 122, kGEnd = 164;
constexpr int kFBase = 164, kFDiag = 245, kFEnd = 326;
constexpr int kLRanks = 175;        // L-slots of the three rows

// rank of slot s in a group: L-slots of C, G, f, then diag+U of C, G, f
int slot_rank(int s) {
  if (s < kCDiag) return s;
  if (s >= kGBase && s < kGDiag) return 80 + (s - kGBase);
  if (s >= kFBase && s < kFDiag) return 94 + (s - kFBase);
  if (s >= kCDiag && s < kCEnd) return kLRanks + (s - kCDiag);
  if (s >= kGDiag && s < kGEnd) return kLRanks + 28 + (s - kGDiag);
  return kLRanks + 70 + (s - kFDiag);
}

// Size classes of the solve's CTA, per stored type S: the first field of a
// shape (its names are fixed by the interface) and the warps it stands for.
template <typename S>
struct SizeClasses {   // FP32
  static constexpr int name[3] = {52, 36, 20}, warps[3] = {16, 8, 4};
};
template <>
struct SizeClasses<double> {
  static constexpr int name[3] = {34, 26, 18}, warps[3] = {16, 8, 4};
};
template <>
struct SizeClasses<__nv_bfloat16> {   // FP32 factors stored as BF16
  static constexpr int name[3] = {72, 40, 8}, warps[3] = {16, 8, 4};
};
constexpr int kLanes = 4;   // lanes per point of the subdomain solve
// arithmetic type of the solve for a storage type (BF16 factors: FP32)
template <typename S>
struct SolveArith {
  using type = S;
};
template <>
struct SolveArith<__nv_bfloat16> {
  using type = float;
};
// ---------------------------------------------------------------------------
// TMA bulk copies, mbarriers and counters (inline PTX)
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// asks for bytes (a multiple of 16, from a 16-byte boundary) in L2; nothing waits for them
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ int ld_acquire_cta(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void add_release_cta(int* p, int v) {
  asm volatile("red.release.cta.shared::cta.add.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
// the same across a cluster: a counter of CTA `rank`, given by its place in this CTA
__device__ __forceinline__ int ld_acquire_cluster(const int* p) {
  int v;
  asm volatile("ld.acquire.cluster.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void add_release_cluster(int* p, int v, int rank) {
  asm volatile(
      "{\n .reg .b32 a;\n mapa.shared::cluster.u32 a, %0, %2;\n red.release.cluster.shared::cluster.add.s32 [a], %1;\n}\n" ::"r"(
          smem_u32(p)),
      "r"(v), "r"(rank)
      : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded waits of a warp.  All 32 lanes call them and all get the same verdict, by a vote: lanes
// that went different ways would leave the others at the next full-warp shuffle for good.  The
// timer is read only every so many polls, so what arrives within the first polls is seen without
// its latency.
constexpr unsigned kAllLanes = 0xffffffffu;
// Phase `parity` of an mbarrier; gives up after limit_ns() nanoseconds of polling, records status 2
// in *failed and returns false.
template <typename Limit>
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, int* failed, Limit&& limit_ns) {
  unsigned long long t0 = 0;
  for (unsigned it = 0;; ++it) {
    if (__all_sync(kAllLanes, mbar_try_wait(bar, parity))) return true;
    if ((it & 63u) == 63u) {
      const unsigned long long t = global_ns();
      if (t0 == 0) {
        t0 = t;
      } else if (__any_sync(kAllLanes, t - t0 > limit_ns())) {
        atomicExch(failed, 2);
        return false;
      }
    }
  }
}
// At least n groups in the counter `finished`; false, with status 2 in *failed and give_up() called,
// when the limit ran out here, and false when *aborted says that it ran out in another warp.
// CLUSTER: the counter is written by other CTAs of the cluster too.
constexpr unsigned kPollNs = 20;   // a warp that polls without a pause takes issue slots from those at work
template <bool CLUSTER, typename Limit, typename GiveUp>
__device__ __forceinline__ bool count_wait(const int* finished, int n, const int* aborted, int* failed,
                                           Limit&& limit_ns, GiveUp&& give_up) {
  unsigned long long t0 = 0;
  for (unsigned it = 0; !__all_sync(kAllLanes, (CLUSTER ? ld_acquire_cluster(finished) : ld_acquire_cta(finished)) >= n);
       ++it) {
    __nanosleep(kPollNs);
    if ((it & 255u) == 255u) {
      const unsigned long long now = global_ns();
      if (t0 == 0) {
        t0 = now;
      } else if (__any_sync(kAllLanes, now - t0 > limit_ns())) {
        atomicExch(failed, 2);
        give_up();
        return false;
      }
      if (__any_sync(kAllLanes, *(const volatile int*)aborted != 0)) return false;
    }
  }
  return true;
}

// Self-test of the bounded wait (ras_selftest_wait): one warp waits for
// limit_ns on an mbarrier that expects one arrival, which nothing makes; the
// wait gives up, sets *status = 2 and the kernel returns.  No copy is issued,
// so nothing is in flight when the CTA exits.
__global__ void wait_selftest(int* status, unsigned long long limit_ns) {
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncwarp();
  mbar_wait(&bar, 0u, status, [=] { return limit_ns; });
}

// Self-test of the verdict (ras_selftest_lanes): the first warp waits, on an mbarrier (KIND 0) or a
// counter (1), half of its lanes for `limit_ns` and half for 100 times that; the second warp
// completes what it waits for after 3 limit_ns.  verdict: what each lane got.
template <int KIND>
__global__ void lane_selftest(int* status, unsigned long long limit_ns, int* verdict) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int finished, aborted;
  const int lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
    finished = aborted = 0;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    auto limit = [=] { return lane < 16 ? limit_ns : 100 * limit_ns; };
    const bool ok = KIND == 0 ? mbar_wait(&bar, 0u, status, limit)
                              : count_wait<false>(&finished, 1, &aborted, status, limit, [] {});
    verdict[lane] = ok;
  } else if (lane == 0) {
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < 3 * limit_ns) __nanosleep(1000);
    if (KIND == 0) mbar_expect_tx(&bar, 0);
    else add_release_cta(&finished, 1);
  }
}

// ---------------------------------------------------------------------------
// Subdomain solve z = sum_boxes (R^0)^T M^{-1} R^delta r: one CTA per box,
// 4 lanes per point, one group of 8 points per warp at a time.
//
// The box's padded local vector holds 4 values per point (C, G, f and a zero),
// so one 16-byte load fetches a neighbour's three unknowns.  Every L-slot of
// the three rows of a point reads one of 40 earlier stencil neighbours (27 at
// level n-1, 13 earlier ones at level n) and every U-slot one of 40 later
// ones (13 at level n, 27 at n+1), besides the point itself.  Lane l takes
// the neighbours q = l + 4 i (i < 10) of both sweeps, loads their values once
// and forms its parts of the C, G and f row sums; a shuffle reduction over the
// 4 lanes closes each sum.
//
// The factor values of a group (FP32, BF16) come by TMA bulk copy into the
// warp's own buffers in shared memory, asked for while the warp still works on
// the groups before.  (Loads through L1 into registers ahead of their use were
// measured slower, 2.30 against 2.16 ms at 32^3 x 64: the neighbours' loads wait
// behind them in L1's queue.  Chunks of 52 points with a CTA barrier each: 2.81.)  The warps of a box do not meet at
// wavefronts: a counter of finished groups in shared memory tells a warp when
// the wavefronts before its group's are done.  What does not depend on the
// last of them -- all neighbours but those one wavefront away -- is loaded and
// multiplied before that wait.
//
// A wait that runs out sets status 2, tells every CTA of the box, waits for the
// warp's copies in flight and leaves z unwritten.
// ---------------------------------------------------------------------------
constexpr size_t kSmemLimit = 227 * 1024;          // dynamic shared memory of one CTA
constexpr size_t kSolveReserve = 2048;   // what the shape interface sets aside beside the buffers it counts
constexpr int kMaxStages = 4;        // factor groups asked for ahead, the one in use included
constexpr int kNbr = 40;             // earlier (and later) stencil neighbours of a point
constexpr int kNbrPerLane = kNbr / kLanes;
constexpr int kVecWidth = 4;         // values per point in the local vectors

// the three unknowns of a local-vector point (4 values, 16- or 32-byte aligned)
__device__ __forceinline__ void ld3(const float* p, float& a, float& b, float& c) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a = v.x;
  b = v.y;
  c = v.z;
}
__device__ __forceinline__ void ld3(const double* p, double& a, double& b, double& c) {
  const double2 v0 = *reinterpret_cast<const double2*>(p);
  a = v0.x;
  b = v0.y;
  c = p[2];
}
__device__ __forceinline__ void st3(float* p, float a, float b, float c) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, 0.f);
}
__device__ __forceinline__ void st3(double* p, double a, double b, double c) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
  *reinterpret_cast<double2*>(p + 2) = make_double2(c, 0.0);
}

template <typename T>
__device__ __forceinline__ T lane_sum(T v) {
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One lane's factor values of a group.  Lower: l(i, 0..3) the C row's C and f
// columns and the f row's G and f columns of neighbour q = lane + 4 i, g(i) the
// G row's G column (q >= 27), own_c (lane 0), own_g (lane 1).  Upper: f(i, 0..1)
// the f row's G and f columns, g(i) the G row's G column, c(i, 0..1) the C row's
// C and f columns (q < 13), and what lanes 1 to 3 hold in place of c(3, .):
// lane 1 1/u of the f and G rows, lane 2 the G row's C column at level n+1
// (q = 26), lane 3 1/u of the C row and its own-point f column.
template <typename S, int G>
struct LaneFactors;

template <int G>
struct LaneFactors<float, G> {
  static constexpr bool kStaged = true;   // comes through shared memory
  float v[kLaneL];
  __device__ __forceinline__ void load(const float* F, bool upper, int lane) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float4 w = *reinterpret_cast<const float4*>(F + 4 * lane + 16 * G * k);
      v[4 * k] = w.x;
      v[4 * k + 1] = w.y;
      v[4 * k + 2] = w.z;
      v[4 * k + 3] = w.w;
    }
    if (upper) {
      const float2 w = *reinterpret_cast<const float2*>(F + 4 * G * 36 + 2 * lane);
      v[36] = w.x;
      v[37] = w.y;
    } else {
#pragma unroll
      for (int k = 9; k < 11; ++k) {
        const float4 w = *reinterpret_cast<const float4*>(F + 4 * lane + 16 * G * k);
        v[4 * k] = w.x;
        v[4 * k + 1] = w.y;
        v[4 * k + 2] = w.z;
        v[4 * k + 3] = w.w;
      }
    }
  }
  __device__ __forceinline__ float at(int i) const { return v[i]; }
};

template <int G>
struct LaneFactors<__nv_bfloat16, G> {
  static constexpr bool kStaged = true;
  unsigned v[kLaneL / 2];   // pairs: value 2 k in the low half
  __device__ __forceinline__ void load(const __nv_bfloat16* F, bool upper, int lane) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint4 w = *reinterpret_cast<const uint4*>(F + 8 * lane + 32 * G * k);
      v[4 * k] = w.x;
      v[4 * k + 1] = w.y;
      v[4 * k + 2] = w.z;
      v[4 * k + 3] = w.w;
    }
    if (upper) {
#pragma unroll
      for (int k = 0; k < 3; ++k) v[16 + k] = *reinterpret_cast<const unsigned*>(F + 4 * G * 32 + 6 * lane + 2 * k);
    } else {
      const uint4 w = *reinterpret_cast<const uint4*>(F + 8 * lane + 128 * G);
      v[16] = w.x;
      v[17] = w.y;
      v[18] = w.z;
      v[19] = w.w;
      const uint2 t = *reinterpret_cast<const uint2*>(F + 4 * G * 40 + 4 * lane);
      v[20] = t.x;
      v[21] = t.y;
    }
  }
  __device__ __forceinline__ float at(int i) const {
    return __uint_as_float(i % 2 ? v[i / 2] & 0xffff0000u : v[i / 2] << 16);
  }
};

// FP64: the values stay in global memory ([slot rank][G] groups) until they
// are used; a warp has its next group's brought to L2 while it works on one, by one bulk
// prefetch.  (Without it every wavefront waited for HBM: boxes of two or three groups a
// wavefront were slower than with chunks copied to shared memory.  us an apply, with / without /
// chunks: 64 boxes, 2.9 groups 813 / 970 / 835, 1.5 groups 574 / 707 / 621; 128 boxes, 2.7 groups
// 787 / 924 / 801; 64 boxes, 8.4 groups 2383 / 2628 / 4866; 32^3 x 64 9242 / 9840 / 12600.  Prefetches
// of the own group to L1 before the wait, alone or besides: 1 to 4 % slower than this.)
template <int G>
struct LaneFactors<double, G> {
  static constexpr bool kStaged = false;
  const double* p;
  __device__ __forceinline__ void load(const double* F, bool upper, int lane) {
    p = F + (upper ? kLRanks * G : 0) + lane / kLanes;
  }
  __device__ __forceinline__ double rank(int r) const { return __ldcs(p + r * G); }
};

// Most warps of a CTA (ras_setup_shape's largest size class).
constexpr int kSolveWarpsMax = 16;

// Lanes (bits) whose neighbour q = lane + 4 i lies one wavefront away (w - 1 in
// the forward sweep, w + 1 in the backward one).  With the wavefront weights
// (1, 2, 4, 8) these are, forward (level n-1: d = q; level n: d = q - 27),
// (1, 1, 1) at n-1 and (1, 1, -1), (1, -1, 0), (-1, 0, 0) at n: q = 26, 35, 38,
// 39; backward (level n: d = 14 + q; level n+1: d = q - 13) the mirror images,
// q = 0, 1, 4, 13.
__host__ __device__ constexpr int dep_lanes(bool upper, int i) {
  return upper ? (i == 0 ? 3 : i == 1 ? 1 : i == 3 ? 2 : 0) : (i == 6 ? 4 : i == 8 ? 8 : i == 9 ? 12 : 0);
}

// The ring of wavefronts (FP32, BF16 where it fits): the solved values of the last 16
// wavefronts, 4 values a point, wavefront w in slot w mod 16 at the places of its
// groups, and one point of zeros for columns outside the box.  No neighbour lies
// more than 15 wavefronts away.  A table holds the ring place of every neighbour (10
// of 16 bits a lane, sweep and group, 12 % more bytes than the FP32 values) and comes with
// the factor values.  Through L1 a group's 10 neighbour loads touch 16 to 24 lines
// each.  Measured, one apply: 32^3 x 64 FP32 2150 -> 2047 us, BF16 2038 -> 1857; coarse 16^3 x
// 32 FP32 211 -> 191; 40^3 x 39 BF16 1433 -> 1345; 192 uneven boxes 695 -> 597; 16 boxes 638 ->
// 650 (not used there).  What is left is the latency of a group's 600 instructions.
constexpr int kNbrBytes = 32 * kNbrPerLane * 2;
constexpr int kRingWaves = 16;
constexpr int kMaxRingPlaces = 65535 / kRingWaves - 1;   // places a wavefront, in 16 bits

// Bytes of a warp's factor buffer (the lower half of a group is the larger one).
template <typename S>
__host__ __device__ constexpr int solve_buffer(int group, bool ring) {
  return LaneFactors<S, kGroup>::kStaged ? 4 * group * kLaneL * (int)sizeof(S) + (ring ? kNbrBytes : 0) : 0;
}
constexpr int kSolveHeader = 1024;   // mbarriers (kMaxStages per warp), counter of finished groups, abort word

// S: type of the stored factor values; T: arithmetic and local-vector type.
// SMEM: the local vector in shared memory.  RING: the last wavefronts there.  G: points per group.
// CS: CTAs of a cluster that share a box: the groups go round the warps of all of them, the
// local vector stays in global memory (the L2 holds it), and each CTA has its own counter of
// the box's finished groups, to which every group adds.  The bits are those of one CTA.
// HOLD: the self-test's instance, in which waits of one CTA of a box run out (RasExtra).  (The limit and
// the hold as run-time arguments of the others cost 1 % through the registers they were given.)
template <typename S, bool SMEM, bool RING, int CS, bool HOLD = false, int G = kGroup>
__global__ void __launch_bounds__(32 * kSolveWarpsMax) ras_solve(
    const BoxDesc* __restrict__ boxes, const int* __restrict__ gptr, const S* __restrict__ F,
    typename SolveArith<S>::type* __restrict__ V, const double* __restrict__ r, double* __restrict__ z,
    const int2* __restrict__ gtab, const int2* __restrict__ otab, const int* __restrict__ vtab,
    const unsigned short* __restrict__ ntab, int wcap, int gptr_bytes, int nbuf, int* __restrict__ status,
    const int* gate, int gate_stride, RasExtra extra) {
  using T = typename SolveArith<S>::type;
  constexpr bool kStaged = LaneFactors<S, G>::kStaged;
  // the box's problem gate (one problem: gate_stride 0, every box reads gate[0])
  if (gate != nullptr && gate[boxes[blockIdx.x / CS].prob * gate_stride] == 0) return;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(smem);
  int* finished = reinterpret_cast<int*>(smem + 8 * kSolveWarpsMax * (kMaxStages - 1));   // groups done
  int* aborted = finished + 1;
  const BoxDesc bx = boxes[blockIdx.x / CS];
  const int P = (int)bx.P, nlev = bx.nlev;
  const S* Fb = F + bx.foff;
  const int* vt = vtab + G * bx.goff;
  const int px = bx.lx + 2, py = bx.ly + 2, pz = bx.lz + 2;
  const int sy = px, sz = px * py, st = px * py * pz;
  const int lane = threadIdx.x & 31, sub = lane & (kLanes - 1);
  const int flane = G == kGroup ? lane : min(lane, kLanes * G - 1);   // whose values the lane reads (idle ones: the last's)
  const int rank = CS == 1 ? 0 : blockIdx.x % CS, local_warp = threadIdx.x / 32;
  const int warp = local_warp * CS + rank, nwarp = blockDim.x / 32 * CS;   // of all CTAs of the box
  auto box_sync = [&]() {
    if constexpr (CS == 1) __syncthreads();
    else cluster_sync();
  };
  // shared memory: header, group pointers, the warps' factor buffers, the local vector
  unsigned char* bufs = smem + kSolveHeader + gptr_bytes;
  unsigned char* rest = bufs + (size_t)(blockDim.x / 32) * nbuf * solve_buffer<S>(G, RING);   // the ring or the local vector
  T* v = SMEM ? reinterpret_cast<T*>(rest) : V + bx.voff;
  T* ring = reinterpret_cast<T*>(rest);   // RING: [16][wcap] points and the zeros
  unsigned char* mine = bufs + (size_t)local_warp * nbuf * solve_buffer<S>(G, RING);
  unsigned long long* bar = bars + local_warp * (kMaxStages - 1);
  const int* gp = gptr + bx.loff;   // first group of every wavefront
  if (gptr_bytes) {
    int* copy = reinterpret_cast<int*>(smem + kSolveHeader);
    for (int i = threadIdx.x; i <= nlev; i += blockDim.x) copy[i] = gp[i];
    gp = copy;
  }
  if (kStaged && lane < nbuf) {
    // (2: an arrival that never comes)
    mbar_init(&bar[lane], HOLD && extra.hold == kHoldCopies && rank == extra.hold_cta ? 2 : 1);
    mbar_fence_init();
  }
  if (threadIdx.x == 0) {
    *finished = HOLD && extra.hold == kHoldCounter && rank == extra.hold_cta ? -1 : 0;   // -1: one group short for good
    *aborted = 0;
  }
  if (RING && threadIdx.x < kVecWidth) ring[kVecWidth * kRingWaves * wcap + threadIdx.x] = (T)0;
  if (SMEM)
    for (int i = threadIdx.x; i < kVecWidth * st * (bx.lt + 2); i += blockDim.x) v[i] = (T)0;
  __syncthreads();
  // The groups in the order of the sweeps: k < ng is group k of the forward
  // sweep, then they come back last to first; a warp takes every nwarp-th of
  // them, wherever the wavefronts end.  Step s < nlev is wavefront s of the
  // forward sweep, then the wavefronts come back as well.
  const int ng = gp[nlev];
  auto before = [&](int s) { return s < nlev ? gp[s] : 2 * ng - gp[2 * nlev - s]; };   // groups of steps < s
  auto group = [&](int k) { return k < ng ? k : 2 * ng - 1 - k; };
  auto issue = [&](int k, int t) {   // copy of group k, the warp's t-th, into its buffer
    if (kStaged && k < 2 * ng && lane == 0) {
      const bool up = k >= ng;
      const unsigned bytes = kLanes * G * (up ? kLaneU : kLaneL) * (unsigned)sizeof(S);
      unsigned char* to = mine + (t % nbuf) * solve_buffer<S>(G, RING);
      fence_proxy_async();
      mbar_expect_tx(&bar[t % nbuf], bytes + (RING ? kNbrBytes : 0));
      bulk_g2s(to, Fb + (long long)group(k) * group_vals(32, G) + (up ? kLanes * G * kLaneL : 0), bytes, &bar[t % nbuf]);
      if (RING)
        bulk_g2s(to + kLanes * G * kLaneL * sizeof(S), ntab + (2 * (bx.goff + group(k)) + (up ? 1 : 0)) * (kNbrBytes / 2),
                 kNbrBytes, &bar[t % nbuf]);
    }
  };
  for (int t = 0; t < nbuf; ++t) issue(warp + t * nwarp, t);
  // the points of the warp's next two groups: the neighbours' and the own point's addresses
  // come from them
  auto point = [&](int k) {
    int q = k < 2 * ng ? vt[G * group(k) + flane / kLanes] : 0;
    if (G < kGroup && lane >= kLanes * G && q >= 0) q = ~q;   // an idle lane: as in an empty place
    return q;
  };
  int vq = point(warp), vq2 = point(warp + nwarp);
  // R^delta r into the padded local vector (gtab: per box point, its global unknown index and
  // its padded offset); four points at a time, so that their loads overlap
  const int member = rank * blockDim.x + threadIdx.x, members = CS * blockDim.x;   // threads of the box
  for (int q0 = member; q0 < P; q0 += 4 * members) {
    int2 e[4];
    T a[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = q0 + k * members;
      e[k] = q < P ? gtab[bx.poff + q] : make_int2(-1, 0);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) a[k][c] = e[k].x >= 0 ? (T)r[e[k].x + c] : (T)0;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (e[k].x >= 0) st3(v + e[k].y, a[k][0], a[k][1], a[k][2]);
  }
  box_sync();

  auto abort_box = [&]() {   // in every CTA of the box: none may write its part of z
    if constexpr (CS == 1) atomicExch(aborted, 1);
    else
      for (int c = 0; c < CS; ++c) add_release_cluster(aborted, 1, c);
  };
  // waits until n groups are done; false when the limit ran out here or in another warp
  auto limit = [&]() { return HOLD && rank == extra.hold_cta ? extra.limit_ns : kWaitLimitNs; };
  auto wait_done = [&](int n) -> bool {
    return count_wait<(CS > 1)>(finished, n, aborted, status, limit, abort_box);
  };
  LaneFactors<S, G> fac;
  int off[kNbrPerLane];   // offsets of the lane's neighbours in the padded local vector
  int s = 0, t = 0;       // step of the warp's group, number of its groups so far
  int k = warp;
  T v0 = 0, v1 = 0, v2 = 0, a0 = 0, a1 = 0, a2 = 0;   // the own point's values, of this group and the next
  bool ahead = false;                                 // the next one's are loaded
  // one sweep: the warp's groups k < kend
  auto sweep = [&](int kend, auto upper_tag) -> int {
    constexpr bool kUpper = decltype(upper_tag)::value;
    for (; k < kend; k += nwarp, ++t) {
      while (k >= before(s + 1)) ++s;
      const bool act = vq >= 0;
      T* vp = v + (act ? vq : ~vq);
      vq = vq2;
      vq2 = point(k + 2 * nwarp);
      [[maybe_unused]] unsigned places[kNbrPerLane / 2];   // RING: the neighbours' places, two a word
      if (kStaged) {
        if (!mbar_wait(&bar[t % nbuf], (unsigned)(t / nbuf) & 1u, status, limit)) {
          abort_box();
          return 1;
        }
        const unsigned char* from = mine + (t % nbuf) * solve_buffer<S>(G, RING);
        fac.load(reinterpret_cast<const S*>(from), kUpper, flane);
        if constexpr (RING)
#pragma unroll
          for (int i = 0; i < kNbrPerLane / 2; ++i)
            places[i] = reinterpret_cast<const unsigned*>(from + kLanes * G * kLaneL * sizeof(S))[kNbrPerLane / 2 * lane + i];
        __syncwarp();
        issue(k + nbuf * nwarp, t + nbuf);
      } else {
        fac.load(Fb + (long long)group(k) * group_vals(64, G), kUpper, flane);
        if (const int kn = k + nwarp; lane == 0 && kn < 2 * ng) {   // the warp's next group
          const bool up = kn >= ng;
          bulk_prefetch_l2(Fb + (long long)group(kn) * group_vals(64, G) + (up ? kLRanks * G : 0),
                           (up ? kSlots - kLRanks : kLRanks) * G * (unsigned)sizeof(S));
        }
      }
      // neighbours two and more wavefronts away (at the first backward step the own point is one
      // of the last wavefront's)
      if (!wait_done(s == nlev ? ng : before(max(s - 1, 0)))) return 2;
      if (RING && ahead) {
        v0 = a0;
        v1 = a1;
        v2 = a2;
      } else {
        ld3(vp, v0, v1, v2);
      }
      if constexpr (RING) {   // the next own point's (in the backward sweep all forward values are there by now)
        ahead = k + nwarp < kend;
        if (ahead) ld3(v + (vq >= 0 ? vq : ~vq), a0, a1, a2);
      }
      T nc[kNbrPerLane], nG[kNbrPerLane], nf[kNbrPerLane];   // the neighbours' unknowns
      auto neighbour = [&](int i) {
        if constexpr (RING)
          ld3(ring + kVecWidth * (i % 2 ? places[i / 2] >> 16 : places[i / 2] & 0xffffu), nc[i], nG[i], nf[i]);
        else
          ld3(vp + off[i], nc[i], nG[i], nf[i]);
      };
#pragma unroll
      for (int i = 0; i < kNbrPerLane; ++i)
        if (!(dep_lanes(kUpper, i) >> sub & 1)) neighbour(i);
      T sc = 0, sg = 0, sf = 0;
      T rc = 0, rg = 0, rf = 0, cf = 0, own_c = 0, own_g = 0;
      if constexpr (sizeof(T) == 8) {
        if (!wait_done(before(s))) return 2;
#pragma unroll
        for (int i = 0; i < kNbrPerLane; ++i)
          if (dep_lanes(kUpper, i) >> sub & 1) neighbour(i);
        // one FMA per product into two chains per sum (the FP64 pipe is the limit)
        T sc1 = 0, sf1 = 0;
#pragma unroll
        for (int i = 0; i < kNbrPerLane; ++i) {
          const int q = sub + kLanes * i, d = q - 13;
          if constexpr (!kUpper) {
            sc = fma(fac.rank(2 * q), nc[i], sc);
            sc1 = fma(fac.rank(2 * q + 1), nf[i], sc1);
            sf = fma(fac.rank(94 + 2 * q), nG[i], sf);
            sf1 = fma(fac.rank(95 + 2 * q), nf[i], sf1);
            if (q >= 27) sg = fma(fac.rank(80 + q - 27), nG[i], sg);
          } else {
            sf = fma(fac.rank(71 + 2 * q), nG[i], sf);
            sf1 = fma(fac.rank(72 + 2 * q), nf[i], sf1);
            if (q < 13) {
              sc = fma(fac.rank(3 + 2 * q), nf[i], fma(fac.rank(2 + 2 * q), nc[i], sc));
              sg += fac.rank(29 + q) * nG[i];
            } else {
              sg += fac.rank(42 + d + (d >= 13 ? 1 : 0)) * nG[i];
              if (d == 13) sg += fac.rank(55) * nc[i];
            }
          }
        }
        if (!kUpper) sc += sc1;
        sf += sf1;
        if constexpr (!kUpper) {
          own_c = fac.rank(93);
          own_g = fac.rank(174);
        } else {
          rc = fac.rank(0);
          cf = fac.rank(1);
          rg = fac.rank(28);
          rf = fac.rank(70);
        }
      } else {
        // products of the neighbours that are there, then the others' and the sums in order
        T pc[kNbrPerLane], pf[kNbrPerLane];
        auto products = [&](int i) {
          if constexpr (!kUpper) {
            pc[i] = fac.at(4 * i) * nc[i] + fac.at(4 * i + 1) * nf[i];
            pf[i] = fac.at(4 * i + 2) * nG[i] + fac.at(4 * i + 3) * nf[i];
          } else {
            pf[i] = fac.at(2 * i) * nG[i] + fac.at(2 * i + 1) * nf[i];
            if (i < 4) pc[i] = fac.at(30 + 2 * i) * nc[i] + fac.at(31 + 2 * i) * nf[i];
          }
        };
#pragma unroll
        for (int i = 0; i < kNbrPerLane; ++i)
          if (!(dep_lanes(kUpper, i) >> sub & 1)) products(i);
        if constexpr (!kUpper) {
          own_c = fac.at(40);
          own_g = __shfl_down_sync(0xffffffffu, own_c, 1);
        } else {
          rf = __shfl_down_sync(0xffffffffu, fac.at(36), 1);
          rg = __shfl_down_sync(0xffffffffu, fac.at(37), 1);
          rc = __shfl_down_sync(0xffffffffu, fac.at(36), 3);
          cf = __shfl_down_sync(0xffffffffu, fac.at(37), 3);
        }
        if (!wait_done(before(s))) return 2;
#pragma unroll
        for (int i = 0; i < kNbrPerLane; ++i)
          if (dep_lanes(kUpper, i) >> sub & 1) neighbour(i);
#pragma unroll
        for (int i = 0; i < kNbrPerLane; ++i)
          if (dep_lanes(kUpper, i) >> sub & 1) products(i);
#pragma unroll
        for (int i = 0; i < kNbrPerLane; ++i) {
          sf += pf[i];
          if constexpr (!kUpper) {
            sc += pc[i];
            if (i >= 7 || (i == 6 && sub == 3)) sg += fac.at(34 + i) * nG[i];
          } else {
            if (i < 3 || (i == 3 && sub == 0)) sc += pc[i];
            sg += fac.at(20 + i) * nG[i];
            if (i == 6 && sub == 2) sg += fac.at(36) * nc[i];
          }
        }
      }
      sc = lane_sum(sc);
      sg = lane_sum(sg);
      sf = lane_sum(sf);
      auto place = [&]() {   // of the point in the ring
        const int w = s < nlev ? s : 2 * nlev - 1 - s;
        return kVecWidth * (w % kRingWaves * wcap + G * (group(k) - gp[w]) + lane / kLanes);
      };
      if (act && sub == 0) {
        if constexpr (!kUpper) {
          // own-point terms in C, G, f order: the G row's own-C and the f row's own-G slot
          const T yc = v0 - sc;
          const T yg = v1 - sg - own_c * yc;
          const T yf = v2 - sf - own_g * yg;
          st3(vp, yc, yg, yf);
          if (RING) st3(ring + place(), yc, yg, yf);
        } else {
          // the C row's own-point f column is applied after the f row is solved
          const T zf = (v2 - sf) * rf;
          const T zg = (v1 - sg) * rg;
          const T zc = (v0 - sc - cf * zf) * rc;
          st3(vp, zc, zg, zf);
          if (RING) st3(ring + place(), zc, zg, zf);
        }
      }
      __syncwarp();
      if constexpr (CS == 1) {
        if (lane == 0) add_release_cta(finished, 1);
      } else {
        if (lane < CS) add_release_cluster(finished, 1, lane);
      }
    }
    return 0;
  };
#pragma unroll
  for (int i = 0; i < kNbrPerLane; ++i) {   // earlier neighbour q: level n-1, d = q (q < 27); level n, d = q - 27
    const int q = sub + kLanes * i, d = q < 27 ? q : q - 27, dt = q < 27 ? -1 : 0;
    off[i] = kVecWidth * ((d % 3 - 1) + sy * ((d / 3) % 3 - 1) + sz * (d / 9 - 1) + st * dt);
  }
  int gave_up = sweep(ng, std::false_type{});   // forward, unit lower factor
  ahead = false;
  if (!gave_up) {
#pragma unroll
    for (int i = 0; i < kNbrPerLane; ++i) {   // later neighbour q: level n, d = 14 + q (q < 13); level n+1, d = q - 13
      const int q = sub + kLanes * i, d = q < 13 ? 14 + q : q - 13, dt = q < 13 ? 0 : 1;
      off[i] = kVecWidth * ((d % 3 - 1) + sy * ((d / 3) % 3 - 1) + sz * (d / 9 - 1) + st * dt);
    }
    gave_up = sweep(2 * ng, std::true_type{});   // backward, upper factor
  }
  if (kStaged && gave_up) {
    const int first = t + gave_up - 1;
    // a wait gave up (status 2 is set): nbuf copies may still be in flight into the warp's buffers;
    // wait for them, again with the limit
    for (int q = first; q < first + nbuf; ++q)
      if (warp + q * nwarp < 2 * ng && mbar_wait(&bar[q % nbuf], (unsigned)(q / nbuf) & 1u, status, limit) &&
          HOLD && lane == 0)
        atomicAdd(extra.drained, warp + q * nwarp + 1);
  }
  box_sync();             // (no CTA of the box ends while another may still count in its counter)
  if (*aborted) return;   // without writing z
  // scatter the owned part: (R^0)^T (otab: the owned points' global indices and offsets)
  for (int q0 = member; q0 < bx.nown; q0 += 4 * members) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = q0 + k * members;
      if (q >= bx.nown) break;
      const int2 e = otab[bx.ooff + q];
      T a0, a1, a2;
      ld3(v + e.y, a0, a1, a2);
      double d0 = (double)a0, d1 = (double)a1, d2 = (double)a2;
      if (extra.add != nullptr) {
        d0 += extra.add[e.x];
        d1 += extra.add[e.x + 1];
        d2 += extra.add[e.x + 2];
      }
      z[e.x] = d0;
      z[e.x + 1] = d1;
      z[e.x + 2] = d2;
      if (extra.z32 != nullptr) {
        extra.z32[e.x] = (float)d0;
        extra.z32[e.x + 1] = (float)d1;
        extra.z32[e.x + 2] = (float)d2;
      }
    }
  }
}

// Ring places of every neighbour of every group place (see kNbrBytes): one thread per lane and
// group.  inv: group place of every box point.
__global__ void place_points(const BoxDesc* __restrict__ boxes, const int* __restrict__ gptr,
                             const int* __restrict__ perm, int G, int* __restrict__ inv) {
  const BoxDesc bx = boxes[blockIdx.x];
  const int q = blockIdx.y * blockDim.x + threadIdx.x;
  if (q >= G * gptr[bx.loff + bx.nlev]) return;
  const int lex = perm[G * bx.goff + q];
  if (lex >= 0) inv[bx.poff + lex] = q;
}
__global__ void neighbour_places(const BoxDesc* __restrict__ boxes, const int* __restrict__ gptr,
                                 const int* __restrict__ perm, const int* __restrict__ inv, int G, int wcap,
                                 unsigned short* __restrict__ out) {
  const BoxDesc bx = boxes[blockIdx.x];
  const int* gp = gptr + bx.loff;
  const int g = blockIdx.y * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x % 32, sub = lane % kLanes;
  if (g >= gp[bx.nlev]) return;
  const int lex = lane / kLanes < G ? perm[G * (bx.goff + g) + lane / kLanes] : -1;
  const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
  const int kt = lex / (bx.lx * bx.ly * bx.lz);
  for (int up = 0; up < 2; ++up)
    for (int i = 0; i < kNbrPerLane; ++i) {
      const int q = sub + kLanes * i;
      const int d = up ? (q < 13 ? 14 + q : q - 13) : (q < 27 ? q : q - 27), dt = up ? (q < 13 ? 0 : 1) : (q < 27 ? -1 : 0);
      const int x = kx + d % 3 - 1, y = ky + d / 3 % 3 - 1, z = kz + d / 9 - 1, t = kt + dt;
      int place = kRingWaves * wcap;
      if (lex >= 0 && x >= 0 && x < bx.lx && y >= 0 && y < bx.ly && z >= 0 && z < bx.lz && t >= 0 && t < bx.lt) {
        const int w = x + 2 * y + 4 * z + 8 * t;
        place = w % kRingWaves * wcap + inv[bx.poff + x + bx.lx * (y + bx.ly * (z + bx.lz * t))] - G * gp[w];
      }
      out[((2 * (bx.goff + g) + up) * 32 + lane) * kNbrPerLane + i] = (unsigned short)place;
    }
}

// points of every wavefront of a box
std::vector<int> wavefronts(const int l[4]) {
  std::vector<int> h(1, 1);
  for (int a = 0; a < 4; ++a) {
    const int step = 1 << a;
    std::vector<int> n(h.size() + (size_t)step * (l[a] - 1), 0);
    for (size_t i = 0; i < n.size(); ++i) {   // n[i] = sum over k < l[a] of h[i - step k]
      n[i] = (i >= (size_t)step ? n[i - step] : 0) + (i < h.size() ? h[i] : 0);
      const size_t out = (size_t)step * l[a];
      if (i >= out && i - out < h.size()) n[i] -= h[i - out];
    }
    h.swap(n);
  }
  return h;
}

std::vector<std::pair<int, int>> parts(int n, int p) {
  std::vector<std::pair<int, int>> out;
  const int base = n / p, extra = n % p;
  int s = 0;
  for (int k = 0; k < p; ++k) {
    const int e = s + base + (k < extra ? 1 : 0);
    out.emplace_back(s, e);
    s = e;
  }
  return out;
}

// The wavefronts' group pointers (kept in shared memory up to kGptrLimit
// bytes, else read from global memory) and the local vector.
constexpr int kGptrLimit = 32 * 1024;
int gptr_smem(int nlev) {
  const int bytes = (nlev + 1 + 31) / 32 * 32 * (int)sizeof(int);
  return bytes <= kGptrLimit ? bytes : 0;
}

// dynamic shared memory of the solve without the ring and the local vector
template <typename S>
size_t solve_smem(int gptr_bytes, int warps, int nbuf, int group, bool ring) {
  return kSolveHeader + gptr_bytes + (size_t)warps * nbuf * solve_buffer<S>(group, ring);
}
size_t ring_smem(int wcap) { return ((size_t)kRingWaves * wcap + 1) * kVecWidth * sizeof(float); }

struct SolveShape {
  int ch, nstage, lanes;          // as the shape interface names them
  int warps, nbuf, gptr_bytes;    // as the kernel runs: a warp's buffers, group pointers in shared memory
  bool smem_vec, ring;
  int cluster;
};
// groups per wavefront from which the largest CTA is taken
constexpr int kFillGroups = 4;
// smallest cluster that shares a box (choose_cluster)
template <typename T>
constexpr int min_cluster() {
  return sizeof(T) == 8 ? 2 : 4;
}
template <typename T, bool HOLD = false>
const void* solve_kernel(int group, bool smem_vec, bool ring, int cluster) {
  constexpr int N = narrow_group(8 * sizeof(T));
  if (!HOLD && group != kGroup) {   // (boxes of narrow groups have too few of them for a cluster)
    if constexpr (LaneFactors<T, N>::kStaged)
      if (ring) return (const void*)ras_solve<T, false, true, 1, false, N>;
    return smem_vec ? (const void*)ras_solve<T, true, false, 1, false, N>
                    : (const void*)ras_solve<T, false, false, 1, false, N>;
  }
  if constexpr (LaneFactors<T, kGroup>::kStaged)
    if (ring) return (const void*)ras_solve<T, false, true, 1, HOLD>;
  if (smem_vec) return (const void*)ras_solve<T, true, false, 1, HOLD>;
  if constexpr (min_cluster<T>() == 2)
    if (cluster == 2) return (const void*)ras_solve<T, false, false, 2, HOLD>;
  return cluster == 8   ? (const void*)ras_solve<T, false, false, 8, HOLD>
         : cluster == 4 ? (const void*)ras_solve<T, false, false, 4, HOLD>
                        : (const void*)ras_solve<T, false, false, 1, HOLD>;
}
// CTAs (a cluster) per box where the boxes alone leave SMs idle: the most whose clusters all
// run at once and that have 2.5 groups of a wavefront each; FP32 and BF16, less bound by
// arithmetic, 4 or 8 only.  Counting in every CTA's counter and waiting for the
// other SMs costs more than fewer groups give.  Measured, FP64 (FP32) us a solve with 1, 2, 4, 8 CTAs a box:
//   16 boxes, 2.3 groups a wavefront:   593   709   643  1031   ( 112     -  210  345)
//   64 boxes, 5.4:                     1702  1642  2992  7151   ( 342, the ring)  (4: the wait for a second wave)
//   16 boxes, 9.3:                     2434  1991  1737  3143   ( 535     -  604 1117)
//   64 boxes, 8.4:                     2903  2385  4009  9522   ( 614, the ring)
//   16 boxes, 16.4:                    5026  3103  2251  3544   (1080     -  782 1229)
//   1 box, 25.2:                       5703  3803  2229  1759   (1306     -  732  592)
//   8 boxes, 125:                     56892 31839 17992  9836   (16045    - 6644 3675)
template <typename T>
kkt_status choose_cluster(int nbox, double groups, int warps, size_t smem, int* out) {
  *out = 1;
  for (int cs = 8; cs >= min_cluster<T>(); cs /= 2) {
    if (groups < 2.5 * cs) continue;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(nbox * cs);
    cfg.blockDim = dim3(32 * warps);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim = {(unsigned)cs, 1, 1};
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int fit = 0;
    KKT_TRY_CUDA(cudaOccupancyMaxActiveClusters(&fit, solve_kernel<T>(kGroup, false, false, cs), &cfg));
    if (nbox <= fit) {
      *out = cs;
      return KKT_OK;
    }
  }
  return KKT_OK;
}
// A requested shape (ras_setup_shape): 0 in a field leaves it to the chooser.
struct ShapeRequest {
  int ch = 0, nstage = 0, lanes = 0, place = 0;   // place: 1 shared-memory vector, 2 global-memory vector
};
// Picks the best shape allowed by `req`; KKT_ERR_ARG when none is.  Boxes whose
// wavefronts fill the largest CTA take it (one per SM, its L1 to itself); others
// take the shape with the fewest waves of CTAs over the SMs.  Measured with 16, 8 (two
// CTAs an SM) and 4 warps, FP32, before the ring below, 256 boxes of 32^3 x 64: fine boxes
// (11 groups a wavefront) 2.16, 2.46, 4.04 ms, coarse boxes (2.5 groups) 303, 221, 300 us;
// 192 uneven boxes (5.6 groups) 695, 1039, 1633 us.  FP64, one CTA a box: 64 boxes of 8.4
// groups 2.91, 3.46, 5.41 ms; 256 boxes of 32^3 x 64 9.31, 8.89, 11.15.  Then the local vectors in
// global memory, the fewest buffers, the largest CTA.  ras_autotune measures instead.
template <typename T>
kkt_status choose_solve_shape(int nbox, long long points, long long max_pad, int nlev, int group, double gpw, int wcap,
                              int nsm, const ShapeRequest& req, SolveShape* out) {
  if (req.lanes != 0 && req.lanes != kLanes) {
    set_error("ras_setup: the subdomain solve runs 4 lanes per point");
    return KKT_ERR_ARG;
  }
  for (int form = 0; form < 6; ++form)
    KKT_TRY_CUDA(cudaFuncSetAttribute(solve_kernel<T>(group, form == 1, form == 2, form > 2 ? 1 << (form - 2) : 1),
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit));
  SolveShape best{};
  long long best_key = -1;
  for (int ci = 0; ci < 3; ++ci)
    for (int ns = 2; ns <= kMaxStages; ++ns)
      for (int sv = 1; sv >= 0; --sv) {
        const int ch = SizeClasses<T>::name[ci], warps = SizeClasses<T>::warps[ci];
        if ((req.ch && req.ch != ch) || (req.nstage && req.nstage != ns) || (req.place == 1 && !sv) ||
            (req.place == 2 && sv))
          continue;
        const size_t vec = sv ? (size_t)max_pad * sizeof(typename SolveArith<T>::type) : 0;
        // the interface's limit: a vector in shared memory leaves room for ns lower blocks of ch points
        if (sv && vec + kSolveReserve + (size_t)ns * kLRanks * ch * sizeof(T) > kSmemLimit) continue;
        // The warps' buffers can take more than those blocks (16 warps x 3 x 5632 bytes against
        // 4 x 36,400).  Where they do not fit, there are fewer of them a warp, then the group
        // pointers stay in global memory, then there are fewer warps.
        // (fewer boxes than a quarter of the SMs: their vectors stay in L1 without the ring, measured 2 to 3 % faster)
        const bool can_ring = LaneFactors<T, kGroup>::kStaged && !sv && wcap <= kMaxRingPlaces && 4 * nbox >= nsm;
        int w = warps, nbuf = 0, gbytes = gptr_smem(nlev);
        bool ring = false;
        size_t sm = 0;
        auto fits = [&]() {
          for (nbuf = ns - 1; nbuf >= 1; --nbuf)
            for (int without = can_ring ? 0 : 1; without < 2; ++without) {
              ring = !without;
              sm = solve_smem<T>(gbytes, w, nbuf, group, ring) + (ring ? ring_smem(wcap) : vec);
              if (sm <= kSmemLimit) return true;
            }
          return false;
        };
        bool ok = fits();
        if (!ok) {
          gbytes = 0;
          while (!(ok = fits()) && w > 1) --w;
        }
        if (!ok) continue;
        int per_sm = 0;
        KKT_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, solve_kernel<T>(group, sv != 0, ring, 1), 32 * w, sm));
        if (per_sm < 1) continue;
        const long long waves = (nbox + (long long)nsm * per_sm - 1) / ((long long)nsm * per_sm);
        const bool filled = ci == 0 && points > (long long)nbox * nlev * kGroup * kFillGroups;
        const long long key = (filled ? 0 : waves) * 100000000LL + (sv ? 1000000 : 0) + (ns - 2) * 1000 + (100 - ch);
        if (best_key >= 0 && key >= best_key) continue;
        best_key = key;
        best = SolveShape{ch, ns, kLanes, w, nbuf, gbytes, sv != 0, ring, 1};
        if (ci < 2 || waves < 2 || (sizeof(T) == 4 && group == kGroup)) continue;
        // Boxes beyond what the SMs hold at a time, with hardly more than a group a wavefront: fewer warps
        // each, more boxes at a time.  A wave of CTAs of w warps with g groups a wavefront was measured
        // to take about 1 + 5 g / w.  us an apply with 1, 2, 3, 4 warps, FP64 (FP32; BF16):
        //   9537 lines of 17 points:         1012 1090 1481 1818   (221 240 277 306; 214 234 273 307)
        //   4913 lines of 33 levels:         1202 1270 1580 1976   (364 370 421 461; 341 359 415 455)
        //   4096 boxes of 2^4 points:         424  505  636  742   (106 112 124 136;  99 108 122 136)
        //   1296 boxes of 3^4 points:         472  615  539  701   (103 111  87 105; 101 105  83 102)
        //   4096 boxes of 3 or 4 a side:     1263 1508 1949 2295   (381 369 364 367; 297 291 307 326)
        //   256 boxes of 3 or 4 a side:       358  311  308  311   (171  93  68  58; 161  87  64  54)
        // The last are one wave in any case; the last but one are FP32's groups of 8, bound by their bytes.
        double cost = waves * (1 + 5 * gpw / w);
        for (int fewer = w - 1; fewer >= 1 && fewer >= gpw; --fewer) {
          const size_t less = solve_smem<T>(gbytes, fewer, nbuf, group, ring) + (ring ? ring_smem(wcap) : vec);
          KKT_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
              &per_sm, solve_kernel<T>(group, sv != 0, ring, 1), 32 * fewer, less));
          if (per_sm < 1) continue;
          const double c = (nbox + (long long)nsm * per_sm - 1) / ((long long)nsm * per_sm) * (1 + 5 * gpw / fewer);
          if (c < cost) {
            cost = c;
            best.warps = fewer;
          }
        }
      }
  if (best_key < 0) {
    set_error("ras_setup: no subdomain-solve shape fits the request (size class, groups ahead and vector "
              "placement must be a compiled combination that fits in shared memory)");
    return KKT_ERR_ARG;
  }
  if (group == kGroup && best.ch == SizeClasses<T>::name[0] && !best.smem_vec && !best.ring)
    KKT_TRY(choose_cluster<T>(nbox, (double)points / ((double)nbox * nlev * kGroup), best.warps,
                              solve_smem<T>(best.gptr_bytes, best.warps, best.nbuf, group, false), &best.cluster));
  *out = best;
  return KKT_OK;
}

}  // namespace

kkt_status ras_create(kkt_problem* const* probs, int nprob, const int nsub[4], int overlap, int local,
                      int factor_prec, const int* shape, ras_precond** out) {
  if (!probs || nprob < 1 || !nsub || !out) {
    set_error("ras_setup: null argument or no problem");
    return KKT_ERR_ARG;
  }
  *out = nullptr;
  for (int k = 0; k < nprob; ++k) {
    const kkt_problem* pk = probs[k];
    if (!pk) {
      set_error("ras_setup: null problem");
      return KKT_ERR_ARG;
    }
    const int dk[4] = {pk->nx, pk->ny, pk->nz, pk->L};
    for (int a = 0; a < 4; ++a)
      if (nsub[a] < 1 || nsub[a] > dk[a]) {
        set_error("ras_setup: each nsub must lie in [1, points along that axis]");
        return KKT_ERR_ARG;
      }
  }
  if (nprob > 1 && local != 0) {
    set_error("ras_setup_batch: the subdomains of several problems use ILU(0) local solves");
    return KKT_ERR_ARG;
  }
  kkt_problem* p = probs[0];
  if (overlap < 0 || local < 0 || local > 3 || (factor_prec != 64 && factor_prec != 32 && factor_prec != 16)) {
    set_error("ras_setup: overlap must be >= 0, local 0 (ILU(0)), 1 (exact LU), 2 (ILU(1)) or 3 (point-block "
              "ILU(0)), factor_prec 64, 32 or 16");
    return KKT_ERR_ARG;
  }
  if (local == 1 && factor_prec != 64) {
    set_error("ras_setup: the exact local LU is FP64 only (factor_prec 64)");
    return KKT_ERR_ARG;
  }
  if (local >= 2 && factor_prec == 16) {
    set_error("ras_setup: ILU(1) and point-block ILU(0) factor in FP64 or FP32 (factor_prec 64 or 32)");
    return KKT_ERR_ARG;
  }
  const SlotTables& T = tables();
  {
    long long h = 0;
    for (int i = 0; i < kSlots; ++i)
      h = (h * 131 + (i + 1) * (T.dt[i] + 2) * 7 + (T.dz[i] + 2) * 11 + (T.dy[i] + 2) * 13 + (T.dx[i] + 2) * 17 +
           T.comp[i] * 19) % 1000000007LL;
    if (h != kGenSlotChecksum || kGenRowSlots0 != T.count[0] || kGenRowSlots1 != T.count[1] ||
        kGenRowSlots2 != T.count[2]) {
      set_error("ras_setup: generated elimination code does not match the slot tables");
      return KKT_ERR_ARG;
    }
    for (int i = 0; i < kSlots; ++i)
      if (kGenRank[i] != slot_rank(i)) {
        set_error("ras_setup: generated elimination code does not match the group order");
        return KKT_ERR_ARG;
      }
  }
  if (T.base[0] != kCBase || T.diag[0] != kCDiag || T.base[1] != kGBase || T.diag[1] != kGDiag ||
      T.base[2] != kFBase || T.diag[2] != kFDiag || T.base[2] + T.count[2] != kFEnd) {
    set_error("ras_setup: internal slot table mismatch");
    return KKT_ERR_ARG;
  }

  ras_precond* m = new (std::nothrow) ras_precond();
  if (!m) return KKT_ERR_NOMEM;
  m->prob = p;
  m->probs.assign(probs, probs + nprob);
  m->vec_off.assign(1, 0);
  for (int k = 0; k < nprob; ++k) m->vec_off.push_back(m->vec_off.back() + probs[k]->n);
  m->n_total = m->vec_off.back();
  m->prec = factor_prec;
  m->local = local;
  // every box: its problem and the owned part of each axis (part k of n holds
  // floor(n/p) + (k < n mod p)); the extended box adds `overlap`, trimmed
  struct Geom {
    int prob;
    std::pair<int, int> own[4];
    long long points;
  };
  std::vector<Geom> geoms;
  for (int k = 0; k < nprob; ++k) {
    const kkt_problem* pk = probs[k];
    const int dk[4] = {pk->nx, pk->ny, pk->nz, pk->L};
    std::vector<std::pair<int, int>> prk[4];
    for (int a = 0; a < 4; ++a) prk[a] = parts(dk[a], nsub[a]);
    for (int it = 0; it < nsub[3]; ++it)
      for (int iz = 0; iz < nsub[2]; ++iz)
        for (int iy = 0; iy < nsub[1]; ++iy)
          for (int ix = 0; ix < nsub[0]; ++ix) {
            Geom g{k, {prk[0][ix], prk[1][iy], prk[2][iz], prk[3][it]}, 1};
            for (int a = 0; a < 4; ++a)
              g.points *= std::min(dk[a], g.own[a].second + overlap) - std::max(0, g.own[a].first - overlap);
            geoms.push_back(g);
          }
  }
  // the largest boxes first, so that the CTAs of a launch (one per box, started in list order)
  // finish as close together as they can
  std::stable_sort(geoms.begin(), geoms.end(), [](const Geom& a, const Geom& b) { return a.points > b.points; });
  {
    // largest padded local vector, most wavefronts, points of all boxes, groups of 8 and of the narrow
    // size, wavefronts with points, whether a box of groups of 8 has too many values for the FP64 factorisation's offsets
    long long pad = 0, points = 0, wide = 0, narrow = 0, fronts = 0;
    bool too_large = false;
    for (const Geom& g : geoms) {
      const kkt_problem* pk = probs[g.prob];
      const int dk[4] = {pk->nx, pk->ny, pk->nz, pk->L};
      long long v = kVecWidth;
      int nlev = 1, len[4];
      for (int a = 0; a < 4; ++a) {
        const int l = len[a] = std::min(dk[a], g.own[a].second + overlap) - std::max(0, g.own[a].first - overlap);
        v *= l + 2;
        nlev += (l - 1) << a;
      }
      if (local == 0) {
        long long groups = 0;
        for (int n : wavefronts(len)) {
          groups += (n + kGroup - 1) / kGroup;
          narrow += (n + narrow_group(factor_prec) - 1) / narrow_group(factor_prec);
          fronts += n > 0;
          m->wcap = std::max(m->wcap, (n + kGroup - 1) / kGroup * kGroup);   // places of the widest wavefront
        }
        wide += groups;
        too_large = too_large || (groups + 1) * group_vals(64, kGroup) > INT32_MAX;
      }
      pad = std::max(pad, v);
      points += g.points;
      m->max_nlev = std::max(m->max_nlev, nlev);
    }
    // Narrow groups where groups of 8 would be filled by less than a third, in FP32 a half (BF16 at a
    // half: 256 boxes of 3 or 4 nodes a side 43.5 -> 45.5 us an apply).  Factor values a point with groups
    // of 8 and narrow ones: boxes of one node in two or three axes, or of two nodes a side, FP64 2608 and
    // 652, FP32 2624 and 1312; 17 x 1 x 1 x 65 nodes FP64 1249 and 349, FP32 1256 and 628; 3 x 3 x 3 x 3
    // FP64 998 and 411, FP32 1004 and 567.
    if (local == 0 && (wide * kGroup > (factor_prec == 32 ? 2 : 3) * points || (factor_prec == 64 && too_large)))
      m->group = narrow_group(factor_prec);
    const double gpw = (double)(m->group == kGroup ? wide : narrow) / std::max(fronts, 1LL);   // groups a wavefront
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1) {
      cudaGetLastError();
      set_error("ras_setup: cannot query the current device");
      delete m;
      return KKT_ERR_CUDA;
    }
    const int nbox = (int)geoms.size();
    ShapeRequest req;
    if (shape) {
      req.ch = shape[0];
      req.nstage = shape[1];
      req.lanes = shape[2];
      req.place = shape[3];
    }
    SolveShape sh{};
    const kkt_status cs = factor_prec == 64   ? choose_solve_shape<double>(nbox, points, pad, m->max_nlev, m->group, gpw, m->wcap, nsm, req, &sh)
                          : factor_prec == 32 ? choose_solve_shape<float>(nbox, points, pad, m->max_nlev, m->group, gpw, m->wcap, nsm, req, &sh)
                                              : choose_solve_shape<__nv_bfloat16>(nbox, points, pad, m->max_nlev, m->group, gpw, m->wcap, nsm, req, &sh);
    if (cs != KKT_OK) {
      delete m;
      return cs;
    }
    m->ch = sh.ch;
    m->warps = sh.warps;
    m->nbuf = sh.nbuf;
    m->gptr_bytes = sh.gptr_bytes;
    m->smem_vec = sh.smem_vec;
    m->ring = sh.ring;
    m->cluster = sh.cluster;
    m->nstage = sh.nstage;
    m->lanes = sh.lanes;
  }
  std::vector<BoxDesc> boxes;
  std::vector<int> perm, gptr, ptab, vtab;
  std::vector<int2> gtab, otab;
  if (m->n_total >= INT32_MAX) {
    set_error("ras_setup: more than 2^31 unknowns are not supported");
    delete m;
    return KKT_ERR_ARG;
  }
  const int G = m->group, gvals = group_vals(factor_prec, G);
  long long foff = 0, voff = 0, poff = 0, ngroup = 0;
  for (const Geom& geo : geoms) {
    const kkt_problem* pk = probs[geo.prob];
    const long long gbase = m->vec_off[geo.prob];   // the problem's first unknown
    const int dims[4] = {pk->nx, pk->ny, pk->nz, pk->L};
    BoxDesc b{};
    b.prob = geo.prob;
    const std::pair<int, int>* own[4] = {&geo.own[0], &geo.own[1], &geo.own[2], &geo.own[3]};
    int lo[4], hi[4];
    for (int a = 0; a < 4; ++a) {
      lo[a] = std::max(0, own[a]->first - overlap);
      hi[a] = std::min(dims[a], own[a]->second + overlap);
    }
    b.x0 = lo[0]; b.y0 = lo[1]; b.z0 = lo[2]; b.t0 = lo[3];
    b.lx = hi[0] - lo[0]; b.ly = hi[1] - lo[1]; b.lz = hi[2] - lo[2]; b.lt = hi[3] - lo[3];
    b.ox0 = own[0]->first; b.ox1 = own[0]->second; b.oy0 = own[1]->first; b.oy1 = own[1]->second;
    b.oz0 = own[2]->first; b.oz1 = own[2]->second; b.ot0 = own[3]->first; b.ot1 = own[3]->second;
    b.P = (long long)b.lx * b.ly * b.lz * b.lt;
    b.nlev = (b.lx - 1) + 2 * (b.ly - 1) + 4 * (b.lz - 1) + 8 * (b.lt - 1) + 1;
    b.foff = foff;
    b.voff = voff;
    b.poff = poff;
    b.goff = ngroup;
    b.loff = (long long)gptr.size();
    poff += b.P;
    voff += (long long)kVecWidth * (b.lx + 2) * (b.ly + 2) * (b.lz + 2) * (b.lt + 2);
    if (b.P * kSlots > INT32_MAX) {
      set_error("ras_setup: a subdomain holds more than 2^31 factor values; use more subdomains");
      delete m;
      return KKT_ERR_ARG;
    }
    if (local == 0) {
      // groups of G points per wavefront: counting sort of the points (lexicographic within a wavefront)
      std::vector<int> fill(b.nlev + 1, 0);
      for (int kt = 0; kt < b.lt; ++kt)
        for (int kz = 0; kz < b.lz; ++kz)
          for (int ky = 0; ky < b.ly; ++ky)
            for (int kx = 0; kx < b.lx; ++kx) fill[kx + 2 * ky + 4 * kz + 8 * kt]++;
      int groups = 0;
      for (int w = 0; w < b.nlev; ++w) {
        gptr.push_back(groups);
        const int n = fill[w];
        fill[w] = G * groups;
        groups += (n + G - 1) / G;
      }
      gptr.push_back(groups);
      m->max_groups = std::max(m->max_groups, groups);
      ngroup += groups;
      // index tables: lexicographic index and padded offset of every group place, place in the
      // factors, global index and padded offset of every point, owned points
      const long long sy = b.lx + 2, sz = sy * (b.ly + 2), st = sz * (b.lz + 2);
      auto pad = [&](int kx, int ky, int kz, int kt) {
        return (int)(kVecWidth * ((kx + 1) + sy * (ky + 1) + sz * (kz + 1) + st * (kt + 1)));
      };
      auto glob = [&](int kx, int ky, int kz, int kt) {
        return (int)(gbase + 3 * ((long long)(b.t0 + kt) * pk->N + (b.x0 + kx) +
                                  (long long)pk->nx * ((b.y0 + ky) + (long long)pk->ny * (b.z0 + kz))));
      };
      const size_t q0 = perm.size(), p0 = gtab.size();
      perm.resize(q0 + (size_t)G * groups, -1);
      vtab.resize(q0 + (size_t)G * groups, ~pad(0, 0, 0, 0));
      gtab.resize(p0 + b.P);
      if (factor_prec == 64) ptab.resize(p0 + b.P);
      int lex = 0;
      for (int kt = 0; kt < b.lt; ++kt)
        for (int kz = 0; kz < b.lz; ++kz)
          for (int ky = 0; ky < b.ly; ++ky)
            for (int kx = 0; kx < b.lx; ++kx, ++lex) {
              const int q = fill[kx + 2 * ky + 4 * kz + 8 * kt]++;
              perm[q0 + q] = lex;
              vtab[q0 + q] = pad(kx, ky, kz, kt);
              gtab[p0 + lex] = make_int2(glob(kx, ky, kz, kt), vtab[q0 + q]);
              if (factor_prec == 64) ptab[p0 + lex] = q / G * gvals + q % G;
            }
      b.ooff = (long long)otab.size();
      for (int gt = b.ot0; gt < b.ot1; ++gt)
        for (int gz = b.oz0; gz < b.oz1; ++gz)
          for (int gy = b.oy0; gy < b.oy1; ++gy)
            for (int gx = b.ox0; gx < b.ox1; ++gx)
              otab.push_back(make_int2(glob(gx - b.x0, gy - b.y0, gz - b.z0, gt - b.t0),
                                       pad(gx - b.x0, gy - b.y0, gz - b.z0, gt - b.t0)));
      b.nown = (int)((long long)otab.size() - b.ooff);
      // FP64: the unit row of pivot points outside the box is one more group
      b.unit = (long long)groups * gvals;
      if (factor_prec == 64 && b.unit + gvals > INT32_MAX) {
        set_error("ras_setup: a subdomain holds more than 2^31 factor values; use more subdomains");
        delete m;
        return KKT_ERR_ARG;
      }
      foff += b.unit + (factor_prec == 64 ? gvals : 0);
    }
    if (local == 1) {
      // exact LU: band of the box matrix in natural point-block order
      const long long n_b = 3 * b.P;
      b.kl = 3 * (1 + b.lx + b.lx * b.ly + b.lx * b.ly * b.lz) + 2;
      if (b.kl > kMaxLuBand || n_b > kMaxLuUnknowns) {
        set_error("ras_setup: a subdomain is too large for the exact local LU (at most " +
                  std::to_string(kMaxLuUnknowns) + " unknowns and half-bandwidth " +
                  std::to_string(kMaxLuBand) + "); use ILU(0) or more subdomains");
        delete m;
        return KKT_ERR_ARG;
      }
      b.aoff = m->ab_count;
      m->ab_count += n_b * (3LL * b.kl + 1);
    }
    boxes.push_back(b);
  }
  m->nbox = (int)boxes.size();
  m->ngroup = ngroup;
  m->boxes_h = boxes;
  m->fcount = foff;
  m->vcount = voff;
  m->max_pad = 0;
  for (const BoxDesc& b : boxes)
    m->max_pad = std::max(m->max_pad, (long long)kVecWidth * (b.lx + 2) * (b.ly + 2) * (b.lz + 2) * (b.lt + 2));
  // bytes of a stored factor value and of a local-vector value
  const size_t esz = factor_prec == 64 ? sizeof(double) : (factor_prec == 32 ? sizeof(float) : 2);
  const size_t vsz = factor_prec == 64 ? sizeof(double) : sizeof(float);
  // every lane vector must start on a 16-byte boundary (group and box offsets are whole groups)
  static_assert(group_vals(32, kGroup) * 2 % 16 == 0 && group_vals(32, narrow_group(32)) * 2 % 16 == 0 &&
                kLanes * narrow_group(32) * kLaneL * 2 % 16 == 0, "16-byte lane vectors");
  auto fail = [&](kkt_status st, const char* what) {
    cudaGetLastError();
    set_error(std::string("ras_setup: ") + what);
    ras_destroy(m);
    return st;
  };
  auto bytes = [](size_t n, size_t size) { return std::max<size_t>(1, n) * size; };
  if (cudaMalloc(&m->boxes, boxes.size() * sizeof(BoxDesc)) != cudaSuccess ||
      cudaMalloc(&m->perm, bytes(perm.size(), sizeof(int))) != cudaSuccess ||
      cudaMalloc(&m->gptr, bytes(gptr.size(), sizeof(int))) != cudaSuccess ||
      cudaMalloc(&m->ptab, bytes(ptab.size(), sizeof(int))) != cudaSuccess ||
      cudaMalloc(&m->gtab, bytes(gtab.size(), sizeof(int2))) != cudaSuccess ||
      cudaMalloc(&m->otab, bytes(otab.size(), sizeof(int2))) != cudaSuccess ||
      cudaMalloc(&m->vtab, bytes(vtab.size(), sizeof(int))) != cudaSuccess ||
      cudaMalloc(&m->F, (local != 0 ? 16 : foff) * esz) != cudaSuccess ||
      cudaMalloc(&m->V, (local != 0 ? 16 : voff) * vsz) != cudaSuccess ||
      cudaMalloc(&m->status, sizeof(int)) != cudaSuccess ||
      cudaMalloc(&m->dprobs, m->probs.size() * sizeof(DevProblem)) != cudaSuccess)
    return fail(KKT_ERR_NOMEM, "device allocation failed");
  m->dprobs_h.resize(m->probs.size());
  if (local == 1) {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return fail(KKT_ERR_CUDA, "cudaMemGetInfo failed");
    const double need = (double)m->ab_count * sizeof(double);
    if (need > 0.8 * (double)free_b)
      return fail(KKT_ERR_NOMEM, ("the exact local LU needs " + std::to_string((long long)(need / 1e6)) +
                                  " MB of band storage; use ILU(0) or more subdomains").c_str());
    if (cudaMalloc(&m->AB, m->ab_count * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&m->ipiv, 3 * (size_t)poff * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&m->lu_ju, 2 * boxes.size() * sizeof(int)) != cudaSuccess)
      return fail(KKT_ERR_NOMEM, "device allocation failed (exact LU)");
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    m->lu_ctas = std::max(1, std::min(64, nsm / std::max(1, m->nbox)));   // one wave of 1024-thread CTAs
  }
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = cudaMemcpy(m->boxes, boxes.data(), boxes.size() * sizeof(BoxDesc), cudaMemcpyHostToDevice);
  auto copy = [&](void* dst, const void* src, size_t n) {
    if (e == cudaSuccess && n) e = cudaMemcpy(dst, src, n, cudaMemcpyHostToDevice);
  };
  copy(m->perm, perm.data(), perm.size() * sizeof(int));
  copy(m->gptr, gptr.data(), gptr.size() * sizeof(int));
  copy(m->ptab, ptab.data(), ptab.size() * sizeof(int));
  copy(m->gtab, gtab.data(), gtab.size() * sizeof(int2));
  copy(m->otab, otab.data(), otab.size() * sizeof(int2));
  copy(m->vtab, vtab.data(), vtab.size() * sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(m->F, 0, (local != 0 ? 16 : foff) * esz);
  if (e == cudaSuccess) e = cudaMemset(m->V, 0, (local != 0 ? 16 : voff) * vsz);
  if (e == cudaSuccess) e = cudaMemset(m->status, 0, sizeof(int));
  if (e != cudaSuccess) return fail(KKT_ERR_CUDA, cudaGetErrorString(e));
  if (local == 0 && m->ring) {
    // without room for the table (a quarter of what is free at most, so that a problem sized to the
    // memory still finds its Krylov vectors) the solve reads its neighbours from global memory
    int* inv = nullptr;
    const size_t tab = (size_t)ngroup * 2 * kNbrBytes, invb = (size_t)poff * sizeof(int);
    size_t free_b = 0, total_b = 0;
    m->ring = cudaMemGetInfo(&free_b, &total_b) == cudaSuccess && tab + invb <= free_b / 4 &&
              cudaMalloc(&inv, invb) == cudaSuccess && cudaMalloc(&m->ntab, tab) == cudaSuccess;
    if (m->ring) {
      place_points<<<dim3(m->nbox, (m->group * m->max_groups + 255) / 256), 256>>>(m->boxes, m->gptr, m->perm, m->group,
                                                                                   inv);
      neighbour_places<<<dim3(m->nbox, (m->max_groups + 7) / 8), 256>>>(m->boxes, m->gptr, m->perm, inv, m->group,
                                                                        m->wcap, m->ntab);
      KKT_COUNT(2);
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaDeviceSynchronize();
    } else {
      cudaGetLastError();
    }
    cudaFree(inv);
    if (e != cudaSuccess) return fail(KKT_ERR_CUDA, cudaGetErrorString(e));
  }
  kkt_status st = local >= 2 ? gp_create(m, local, factor_prec) : KKT_OK;
  if (st == KKT_OK && local == 0 && factor_prec != 64) st = ras_factor_prepare32(m);
  if (st == KKT_OK) st = ras_factor(m, nullptr);
  if (st != KKT_OK) {
    ras_destroy(m);
    return st;
  }
  *out = m;
  return KKT_OK;
}

namespace {

template <typename S>
kkt_status launch_solve(ras_precond* m, const double* r, double* z, typename SolveArith<S>::type* V,
                        cudaStream_t s, const int* gate = nullptr, int gate_stride = 0,
                        const RasExtra& extra = RasExtra()) {
  using T = typename SolveArith<S>::type;
  const int gbytes = m->gptr_bytes;
  // (the dynamic shared-memory limit of both instances is raised at set-up, in choose_solve_shape)
  const size_t smem = solve_smem<S>(gbytes, m->warps, m->nbuf, m->group, m->ring) +
                      (m->ring ? ring_smem(m->wcap) : m->smem_vec ? (size_t)m->max_pad * sizeof(T) : 0);
  const void* kernel = solve_kernel<S>(m->group, m->smem_vec, m->ring, m->cluster);
  if constexpr (std::is_same_v<S, float>)
    if (extra.hold != kHoldNone) kernel = solve_kernel<S, true>(m->group, m->smem_vec, m->ring, m->cluster);
  const BoxDesc* boxes = m->boxes;
  const S* F = (const S*)m->F;
  const int *gptr = m->gptr, *vtab = m->vtab;
  const int2 *gtab = m->gtab, *otab = m->otab;
  const unsigned short* ntab = m->ntab;
  int wcap = m->wcap, nbuf = m->nbuf;
  int* status = m->status;
  RasExtra ex = extra;
  void* args[] = {&boxes, &gptr, &F,    &V,      &r,    &z,      &gtab, &otab,        &vtab,
                  &ntab,  &wcap, (void*)&gbytes, &nbuf, &status, &gate, &gate_stride, &ex};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(m->nbox * m->cluster);
  cfg.blockDim = dim3(32 * m->warps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim = {(unsigned)m->cluster, 1, 1};
  cfg.attrs = &attr;
  cfg.numAttrs = m->cluster > 1 ? 1 : 0;
  KKT_TRY_CUDA(cudaLaunchKernelExC(&cfg, kernel, args));
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

}  // namespace

kkt_status ras_factor_enqueue(ras_precond* m, cudaStream_t s) {
  KKT_TRY_CUDA(cudaMemsetAsync(m->status, 0, sizeof(int), s));
  // the problems as the value gather reads them now (the regularisation may have changed)
  for (size_t k = 0; k < m->probs.size(); ++k) m->dprobs_h[k] = m->probs[k]->dev();
  KKT_TRY_CUDA(cudaMemcpyAsync(m->dprobs, m->dprobs_h.data(), m->dprobs_h.size() * sizeof(DevProblem),
                               cudaMemcpyHostToDevice, s));
  if (m->gp) KKT_TRY(gp_factor(m, s));
  else if (m->local == 1) KKT_TRY(ras_lu_factor(m, s));
  else if (m->prec == 64) KKT_TRY(ras_factor_launch64(m, s));
  else if (m->prec == 32) KKT_TRY(ras_factor_launch32(m, s));
  else KKT_TRY(ras_factor_launch16(m, s));
  return KKT_OK;
}

kkt_status ras_factor_status(ras_precond* m) {
  int st = 0;
  KKT_TRY_CUDA(cudaMemcpy(&st, m->status, sizeof(int), cudaMemcpyDeviceToHost));
  if (st != 0) {
    set_error("ras_setup: zero or non-finite pivot in a subdomain factorisation");
    return KKT_ERR_ZERO_PIVOT;
  }
  return KKT_OK;
}

kkt_status ras_factor(ras_precond* m, cudaStream_t s) {
  KKT_TRY(ras_factor_enqueue(m, s));
  KKT_TRY_CUDA(cudaStreamSynchronize(s));
  return ras_factor_status(m);
}

kkt_status ras_launch(ras_precond* m, const double* r, double* z, cudaStream_t s, const int* gate,
                      int gate_stride, const RasExtra& extra) {
  if (m->local == 0) {
    TimedScope timed(&m->timing, s);
    if (m->prec == 64) return launch_solve<double>(m, r, z, (double*)m->V, s, gate, gate_stride, extra);
    if (m->prec == 32) return launch_solve<float>(m, r, z, (float*)m->V, s, gate, gate_stride, extra);
    return launch_solve<__nv_bfloat16>(m, r, z, (float*)m->V, s, gate, gate_stride, extra);
  }
  {
    TimedScope timed(&m->timing, s);
    KKT_TRY(m->gp ? gp_solve(m, r, z, s, gate) : ras_lu_solve(m, r, z, s, gate));
  }
  if (extra.add) KKT_TRY(vec_axpby(z, 1.0, extra.add, 1.0, m->n_total, s, gate));
  if (extra.z32) KKT_TRY(launch_narrow(z, extra.z32, m->n_total, s, gate));
  return KKT_OK;
}

kkt_status ras_check(ras_precond* m) {
  int st = 0;
  KKT_TRY_CUDA(cudaMemcpy(&st, m->status, sizeof(int), cudaMemcpyDeviceToHost));
  if (st == 2) {
    set_error("ras_apply: a subdomain solve gave up waiting for a factor copy or an earlier wavefront");
    return KKT_ERR_CUDA;
  }
  return KKT_OK;
}

extern "C" kkt_status ras_setup(kkt_problem* p, const int nsub[4], int overlap, int local, int factor_prec,
                                ras_precond** out) {
  NvtxRange nvtx_("ras_setup");
  return ras_create(&p, 1, nsub, overlap, local, factor_prec, nullptr, out);
}

extern "C" kkt_status ras_setup_shape(kkt_problem* p, const int nsub[4], int overlap, int local, int factor_prec,
                                      const int shape[4], ras_precond** out) {
  if (!shape) {
    set_error("ras_setup_shape: null shape");
    return KKT_ERR_ARG;
  }
  if (shape[0] < 0 || shape[1] < 0 || (shape[1] != 0 && (shape[1] < 2 || shape[1] > kMaxStages)) ||
      (shape[2] != 0 && shape[2] != kLanes) || shape[3] < 0 || shape[3] > 2) {
    set_error("ras_setup_shape: shape = {size class >= 0, groups held 0 or 2..4, lanes 0 or 4, "
              "vector placement 0, 1 or 2}");
    return KKT_ERR_ARG;
  }
  return ras_create(&p, 1, nsub, overlap, local, factor_prec, shape, out);
}

extern "C" kkt_status ras_setup_batch(kkt_problem* const* probs, int nprob, const int nsub[4], int overlap,
                                      int factor_prec, const int shape[4], ras_precond** out) {
  if (shape && (shape[0] < 0 || shape[1] < 0 || (shape[1] != 0 && (shape[1] < 2 || shape[1] > kMaxStages)) ||
                (shape[2] != 0 && shape[2] != kLanes) || shape[3] < 0 || shape[3] > 2)) {
    set_error("ras_setup_batch: shape = {size class >= 0, groups held 0 or 2..4, lanes 0 or 4, "
              "vector placement 0, 1 or 2}");
    return KKT_ERR_ARG;
  }
  return ras_create(probs, nprob, nsub, overlap, 0, factor_prec, shape, out);
}

extern "C" kkt_status ras_apply(ras_precond* m, const double* r, double* z, void* stream) {
  NvtxRange nvtx_("ras_apply");
  if (!m || !r || !z) {
    set_error("ras_apply: null argument");
    return KKT_ERR_ARG;
  }
  if (spans_overlap(r, z, m->n_total)) {
    set_error("ras_apply: r and z must not overlap");
    return KKT_ERR_ARG;
  }
  return ras_launch(m, r, z, (cudaStream_t)stream);
}

extern "C" kkt_status ras_solve_shape(const ras_precond* m, int* chunk_points, int* stages, int* lanes,
                                      int* smem_vectors) {
  if (!m) {
    set_error("ras_solve_shape: null argument");
    return KKT_ERR_ARG;
  }
  if (chunk_points) *chunk_points = m->ch;
  if (stages) *stages = m->nstage;
  if (lanes) *lanes = m->lanes;
  if (smem_vectors) *smem_vectors = m->smem_vec ? 1 : 0;
  return KKT_OK;
}

extern "C" kkt_status ras_solve_form(const ras_precond* m, int* warps, int* buffers, int* cluster, int* ring) {
  if (!m) {
    set_error("ras_solve_form: null argument");
    return KKT_ERR_ARG;
  }
  if (warps) *warps = m->warps;
  if (buffers) *buffers = m->local == 0 && m->prec != 64 ? m->nbuf : 0;
  if (cluster) *cluster = m->cluster;
  if (ring) *ring = m->local == 0 && m->ring ? 1 : 0;
  return KKT_OK;
}

extern "C" kkt_status ras_status(ras_precond* m, int* code, void* stream) {
  if (!m || !code) {
    set_error("ras_status: null argument");
    return KKT_ERR_ARG;
  }
  const cudaStream_t s = (cudaStream_t)stream;
  int st = 0;
  KKT_TRY_CUDA(cudaMemcpyAsync(&st, m->status, sizeof(int), cudaMemcpyDeviceToHost, s));
  KKT_TRY_CUDA(cudaStreamSynchronize(s));
  *code = st;
  if (*code == 2) {
    set_error("ras_status: a subdomain solve gave up waiting for a factor copy or an earlier wavefront");
    return KKT_ERR_CUDA;
  }
  if (*code == 1) {
    set_error("ras_status: zero or non-finite pivot in a subdomain factorisation");
    return KKT_ERR_ZERO_PIVOT;
  }
  return KKT_OK;
}

extern "C" kkt_status ras_selftest_wait(ras_precond* m, double limit_ms, void* stream) {
  if (!m || !(limit_ms > 0.0) || limit_ms > 1000.0) {
    set_error("ras_selftest_wait: null handle or limit_ms outside (0, 1000]");
    return KKT_ERR_ARG;
  }
  wait_selftest<<<1, 32, 0, (cudaStream_t)stream>>>(m->status, (unsigned long long)(limit_ms * 1e6));
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

extern "C" kkt_status ras_selftest_solve(ras_precond* m, const double* r, double* z, double limit_ms, int hold, int cta,
                                         int* drained, void* stream) {
  if (!m || !r || !z || !(limit_ms > 0.0) || limit_ms > 1000.0 || hold < kHoldCounter || hold > kHoldCopies || cta < 0 ||
      m->local != 0 || m->prec != 32 || m->group != kGroup || cta >= m->cluster || spans_overlap(r, z, m->n_total)) {
    set_error("ras_selftest_solve: null argument, limit_ms outside (0, 1000], hold not 1 or 2, cta outside the cluster, "
              "r and z overlap, or not an ILU(0) preconditioner with FP32 factors in groups of 8");
    return KKT_ERR_ARG;
  }
  const cudaStream_t s = (cudaStream_t)stream;
  int* d = nullptr;
  KKT_TRY_CUDA(cudaMalloc(&d, sizeof(int)));
  RasExtra extra;
  extra.limit_ns = (unsigned long long)(limit_ms * 1e6);
  extra.hold = hold;
  extra.hold_cta = cta;
  extra.drained = d;
  cudaError_t e = cudaFuncSetAttribute(solve_kernel<float, true>(m->group, m->smem_vec, m->ring, m->cluster),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
  if (e == cudaSuccess) e = cudaMemsetAsync(d, 0, sizeof(int), s);
  const kkt_status st = e == cudaSuccess ? ras_launch(m, r, z, s, nullptr, 0, extra) : KKT_OK;
  int sum = 0;
  if (e == cudaSuccess && st == KKT_OK) e = cudaMemcpyAsync(&sum, d, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && st == KKT_OK) e = cudaStreamSynchronize(s);
  cudaFree(d);
  KKT_TRY_CUDA(e);
  if (drained) *drained = sum;
  return st;
}

extern "C" kkt_status ras_selftest_lanes(ras_precond* m, int kind, int verdict[32], void* stream) {
  if (!m || !verdict || kind < 0 || kind > 1) {
    set_error("ras_selftest_lanes: null argument or kind not 0 (mbarrier) / 1 (counter)");
    return KKT_ERR_ARG;
  }
  const cudaStream_t s = (cudaStream_t)stream;
  constexpr unsigned long long limit_ns = 5000000ull;
  int* d = nullptr;
  KKT_TRY_CUDA(cudaMalloc(&d, 32 * sizeof(int)));
  if (kind == 0) lane_selftest<0><<<1, 64, 0, s>>>(m->status, limit_ns, d);
  else lane_selftest<1><<<1, 64, 0, s>>>(m->status, limit_ns, d);
  KKT_COUNT(1);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(verdict, d, 32 * sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(d);
  KKT_TRY_CUDA(e);
  return KKT_OK;
}

extern "C" kkt_status ras_info(const ras_precond* m, int* nbox, long long* points, long long* factor_values,
                               int* value_bytes) {
  if (!m) {
    set_error("ras_info: null argument");
    return KKT_ERR_ARG;
  }
  long long pts = 0;
  for (const BoxDesc& b : m->boxes_h) pts += b.P;
  if (nbox) *nbox = m->nbox;
  if (points) *points = pts;
  if (factor_values) *factor_values = m->local == 1 ? m->ab_count : (m->gp ? gp_factor_count(m) : m->fcount);
  if (value_bytes) *value_bytes = m->prec == 64 ? 8 : (m->prec == 32 ? 4 : 2);
  return KKT_OK;
}

extern "C" kkt_status ras_refactor(ras_precond* m, void* stream) {
  NvtxRange nvtx_("ras_refactor");
  if (!m) {
    set_error("ras_refactor: null argument");
    return KKT_ERR_ARG;
  }
  return ras_factor(m, (cudaStream_t)stream);
}

extern "C" kkt_status ras_timing_read(ras_precond* m, int kernel, double* total_ms, long long* launches) {
  if (!m || (kernel != 0 && kernel != 1)) {
    set_error("ras_timing_read: null handle or kernel not 0 (solve) / 1 (factorisation)");
    return KKT_ERR_ARG;
  }
  TimingLog& log = kernel == 0 ? m->timing : m->factor_timing;
  log.drain();
  if (total_ms) *total_ms = log.total_ms;
  if (launches) *launches = log.count;
  return KKT_OK;
}

extern "C" kkt_status kkt_timing_reset(kkt_problem* p, ras_precond* m) {
  if (p) p->mv_timing.reset();
  if (m) {
    m->timing.reset();
    m->factor_timing.reset();
  }
  return KKT_OK;
}

extern "C" void ras_destroy(ras_precond* m) {
  if (!m) return;
  cudaFree(m->boxes);
  cudaFree(m->perm);
  cudaFree(m->gptr);
  cudaFree(m->ptab);
  cudaFree(m->gtab);
  cudaFree(m->otab);
  cudaFree(m->vtab);
  cudaFree(m->ntab);
  cudaFree(m->rec);
  cudaFree(m->AB);
  cudaFree(m->ipiv);
  cudaFree(m->lu_ju);
  cudaFree(m->F);
  cudaFree(m->V);
  cudaFree(m->status);
  cudaFree(m->dprobs);
  gp_destroy(m);
  delete m->bw;
  delete m;
}

// ---------------------------------------------------------------------------
// Allocation-free subdomain solve.  The padded local vectors the solve works
// in come from a fixed array compiled into the library instead of the handle.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kStaticScratchBytes = 32u << 20;   // 32 MiB per device
__device__ __align__(256) unsigned char g_ras_static_scratch[kStaticScratchBytes];

std::mutex g_static_mu;
void* g_static_ptr[64] = {};

// Device address of the static scratch on the current device, looked up once
// per device (the host-side symbol is only a stand-in for it).
kkt_status static_scratch(void** out) {
  int dev = 0;
  KKT_TRY_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("ras_apply_static: device ordinal out of range");
    return KKT_ERR_ARG;
  }
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* ptr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_ras_static_scratch);
    if (e != cudaSuccess || !ptr) {
      set_error(std::string("ras_apply_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      return KKT_ERR_CUDA;
    }
    g_static_ptr[dev] = ptr;
  }
  *out = g_static_ptr[dev];
  return KKT_OK;
}

}  // namespace

extern "C" kkt_status ras_apply_static(ras_precond* m, const double* r, double* z, void* stream) {
  if (!m || !r || !z) {
    set_error("ras_apply_static: null argument");
    return KKT_ERR_ARG;
  }
  if (spans_overlap(r, z, m->n_total)) {
    set_error("ras_apply_static: r and z must not overlap");
    return KKT_ERR_ARG;
  }
  if (m->local != 0) {
    set_error("ras_apply_static: only ILU(0) preconditioners have a static-scratch apply; use ras_apply");
    return KKT_ERR_ARG;
  }
  void* scratch = nullptr;
  KKT_TRY(static_scratch(&scratch));
  cudaStream_t s = (cudaStream_t)stream;
  // A solve that keeps the local vectors in shared memory never reads the
  // scratch: no size limit and nothing to clear.
  if (!m->smem_vec) {
    const size_t bytes = (size_t)m->vcount * (m->prec == 64 ? sizeof(double) : sizeof(float));
    if (bytes > kStaticScratchBytes) {
      set_error("ras_apply_static: the subdomain local vectors need " + std::to_string(bytes) +
                " bytes, more than the " + std::to_string(kStaticScratchBytes) +
                "-byte static scratch; use ras_apply");
      return KKT_ERR_ARG;
    }
    // the ghost layers of the local vectors must read zero; earlier calls (on
    // any handle) may have left other data at those positions
    KKT_TRY_CUDA(cudaMemsetAsync(scratch, 0, bytes, s));
  }
  if (m->prec == 64) return launch_solve<double>(m, r, z, (double*)scratch, s);
  if (m->prec == 32) return launch_solve<float>(m, r, z, (float*)scratch, s);
  return launch_solve<__nv_bfloat16>(m, r, z, (float*)scratch, s);
}

// ---------------------------------------------------------------------------
// Autotuner of the subdomain solve's shape: every compiled size class with
// 2 and 3 in the buffer field (local vectors placed as the chooser places them) is
// set up on the given problems and timed over `reps` applies with CUDA
// events; the fastest is returned and, with a cache file, remembered there
// under a key of the problems' sizes, the split, the precision and the
// device, one line per key ("key<TAB>size class, groups held, ms").
// ---------------------------------------------------------------------------
namespace {

std::string tune_key(kkt_problem* const* probs, int nprob, const int nsub[4], int overlap, int prec) {
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceProp prop{};
  cudaGetDeviceProperties(&prop, dev);
  std::string k = std::string(prop.name) + ";prec=" + std::to_string(prec) + ";ov=" + std::to_string(overlap) +
                  ";nsub=" + std::to_string(nsub[0]) + "," + std::to_string(nsub[1]) + "," + std::to_string(nsub[2]) +
                  "," + std::to_string(nsub[3]) + ";";
  for (int i = 0; i < nprob; ++i)
    k += std::to_string(probs[i]->nx) + "x" + std::to_string(probs[i]->ny) + "x" + std::to_string(probs[i]->nz) +
         "x" + std::to_string(probs[i]->L) + (i + 1 < nprob ? "," : "");
  for (char& c : k)
    if (c == '\t' || c == '\n') c = ' ';
  return k;
}

__global__ void fill_ones(double* x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    x[i] = 1.0;
}

}  // namespace

extern "C" kkt_status ras_autotune(kkt_problem* const* probs, int nprob, const int nsub[4], int overlap,
                                   int factor_prec, int reps, const char* cache_path, int shape_out[4],
                                   double* best_ms) {
  if (!probs || nprob < 1 || !nsub || !shape_out || reps < 1 ||
      (factor_prec != 64 && factor_prec != 32 && factor_prec != 16)) {
    set_error("ras_autotune: bad argument");
    return KKT_ERR_ARG;
  }
  const std::string key = tune_key(probs, nprob, nsub, overlap, factor_prec);
  if (cache_path) {
    if (FILE* f = std::fopen(cache_path, "r")) {
      char line[4096];
      while (std::fgets(line, sizeof(line), f)) {
        char* tab = std::strchr(line, '\t');
        if (!tab || std::string(line, tab) != key) continue;
        int ch = 0, ns = 0;
        double ms = 0.0;
        if (std::sscanf(tab + 1, "%d %d %lf", &ch, &ns, &ms) == 3) {
          std::fclose(f);
          shape_out[0] = ch;
          shape_out[1] = ns;
          shape_out[2] = kLanes;
          shape_out[3] = 0;
          if (best_ms) *best_ms = ms;
          return KKT_OK;
        }
      }
      std::fclose(f);
    }
  }
  const int* cands = factor_prec == 64   ? SizeClasses<double>::name
                     : factor_prec == 16 ? SizeClasses<__nv_bfloat16>::name
                                         : SizeClasses<float>::name;
  long long n = 0;
  for (int i = 0; i < nprob; ++i) n += probs[i]->n;
  double *r = nullptr, *z = nullptr;
  if (cudaMalloc(&r, n * sizeof(double)) != cudaSuccess || cudaMalloc(&z, n * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(r);
    set_error("ras_autotune: device allocation failed");
    return KKT_ERR_NOMEM;
  }
  fill_ones<<<1216, 256>>>(r, n);
  KKT_COUNT(1);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  double best = -1.0;
  int best_ch = 0, best_ns = 0;
  kkt_status err = KKT_OK;
  for (int ci = 0; ci < 3 && err == KKT_OK; ++ci)
    for (int ns = 2; ns <= 3 && err == KKT_OK; ++ns) {
      const int shape[4] = {cands[ci], ns, 0, 0};
      ras_precond* m = nullptr;
      const kkt_status st = ras_create(probs, nprob, nsub, overlap, 0, factor_prec, shape, &m);
      if (st == KKT_ERR_ARG) continue;   // this shape does not fit the device
      if (st != KKT_OK) {
        err = st;
        break;
      }
      kkt_status ls = ras_launch(m, r, z, nullptr);   // warm-up
      cudaEventRecord(e0, nullptr);
      for (int i = 0; i < reps && ls == KKT_OK; ++i) ls = ras_launch(m, r, z, nullptr);
      cudaEventRecord(e1, nullptr);
      float ms = 0.f;
      if (ls == KKT_OK && cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess) {
        const double per = ms / reps;
        if (best < 0 || per < best) {
          best = per;
          best_ch = cands[ci];
          best_ns = ns;
        }
      } else if (ls != KKT_OK) {
        err = ls;
      }
      ras_destroy(m);
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(r);
  cudaFree(z);
  if (err != KKT_OK) return err;
  if (best < 0) {
    set_error("ras_autotune: no shape of the subdomain solve fits these subdomains");
    return KKT_ERR_ARG;
  }
  shape_out[0] = best_ch;
  shape_out[1] = best_ns;
  shape_out[2] = kLanes;
  shape_out[3] = 0;
  if (best_ms) *best_ms = best;
  if (cache_path)
    if (FILE* f = std::fopen(cache_path, "a")) {
      std::fprintf(f, "%s\t%d %d %.6f\n", key.c_str(), best_ch, best_ns, best);
      std::fclose(f);
    }
  return KKT_OK;
}
