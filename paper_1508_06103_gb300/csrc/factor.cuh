// FP64 ILU(0) factorisation of all subdomain matrices (Sec. 3.2), in place on
// the [slot rank][G points] groups that the subdomain solve reads.  (FP32:
// factor32.cu.)
//
// Values.  gather_groups forms every slot value of every box point from the
// stencil coefficients (the principal submatrix of F_h on the extended box,
// Eq. 10-12; a slot whose column leaves the box holds 0) and writes it to the
// point's column of its group, row c_gen_rank[slot] (c_gen_rank_of by the
// slot's offsets).
//
// Elimination.  One CTA per box steps through the wavefronts
// w = x + 2y + 4z + 8t with a barrier between them; one thread takes one point
// of the wavefront and eliminates its C, G and f rows in turn with the
// straight-line code of ilu_rows.inc.  The thread first lists where the
// columns of its 41 possible pivot points are; a pivot point outside the box
// is sent to the box's unit row (1 at the three diagonal ranks, 0 elsewhere).
// The diagonal slot of a finished row holds 1/u_kk.  (One warp per point, as in
// FP32, would issue 2.5 times the FP64 instructions; the pipe has 2 lanes.)
#pragma once

#include "slotval.cuh"

namespace {

#include "ilu_rows.inc"

constexpr int kGatherThreads = 256;
// Threads per factor CTA, two CTAs per SM (all 256 boxes of the 4x4x4x4
// partition resident at once); the rows need the registers of 128 threads.
template <typename T>
constexpr int factor_threads = 128;

// offset of the column of group place q in the box's factor values
template <typename T, int G>
__device__ __forceinline__ int group_column(int q) {
  return q / G * group_vals(8 * sizeof(T), G) + q % G;
}

// One thread per point (wavefront order, so the threads of a group write
// consecutive addresses); all threads of a warp on the same slot.  Entries are
// formed in the factor precision, with the arithmetic of slot_value, but one
// spatial offset at a time: the point's B, S, S^T and K coefficients of that
// offset are loaded once and give all 12 slots that share it (C row: C and f
// columns at levels n-1, n; G row: G column at n, n+1; f row: G and f columns
// at n-1, n, n+1), plus the G row's two sensor slots at the centre.  Also
// writes each box's unit row.
template <typename T, int G>
__global__ void __launch_bounds__(kGatherThreads) gather_groups(const DevProblem* __restrict__ probs,
                                                                const BoxDesc* __restrict__ boxes,
                                                                const int* __restrict__ gptr,
                                                                const int* __restrict__ perm, T* __restrict__ F) {
  const BoxDesc bx = boxes[blockIdx.y];
  const DevProblem p = probs[bx.prob];
  T* Fb = F + bx.foff;
  if (blockIdx.x == 0)
    for (int s = threadIdx.x; s < kSlots; s += blockDim.x)
      Fb[bx.unit + c_gen_rank[s] * G] = (s == kDiagC || s == kDiagG || s == kDiagF) ? (T)1 : (T)0;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= G * gptr[bx.loff + bx.nlev]) return;
  const int lex = perm[G * bx.goff + q];
  if (lex < 0) return;
  const Coefs<T> cf = coefs<T>(p);
  const PointRow<T> pr = point_row<T>(p, bx, lex);
  T* dst = Fb + group_column<T, G>(q);
  const T tau = (T)p.tau, th = (T)p.theta, th1 = (T)(1.0 - p.theta), b1 = (T)p.beta1, b2 = (T)p.beta2;
  const T mt1 = tau / (T)6, lt1 = -(T)1 / tau;
  const bool idC = pr.n == 0 || pr.dirj, idG = pr.n == p.M || pr.dirj;   // identity rows
  const bool tm = pr.kt > 0, tp = pr.kt + 1 < bx.lt;                      // levels n-1, n+1 in the box
  const T z = (T)0;
  // slot (row type c, level offset dt, spatial offset d, column component cc)
#define PUT(c, dt, d, cc, v) dst[c_gen_rank_of[c][(dt) + 1][d][cc] * G] = (v)
#pragma unroll
  for (int d = 0; d < kStencil; ++d) {
    const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
    const int ax = pr.kx + dx, ay = pr.ky + dy, az = pr.kz + dz;
    const bool sp = ax >= 0 && ax < bx.lx && ay >= 0 && ay < bx.ly && az >= 0 && az < bx.lz;
    T Bv = z, Sv = z, STv = z, Kv = z;
    if (sp) {
      const size_t ci = (size_t)d * p.N + pr.j;
      Bv = cf.B[ci];
      Sv = cf.S[ci];
      STv = cf.ST[ci];
      Kv = p.reg ? Bv : cf.K[ci];   // beta2 term: K (H1-H1) or B (H1-L2)
    }
    constexpr int kCentre = 13;
    // C row
    PUT(0, 0, d, 0, !sp ? z : idC ? (d == kCentre ? (T)1 : z) : Bv + th * tau * Sv);
    PUT(0, 0, d, 2, !sp || idC ? z : -th * tau * Bv);
    PUT(0, -1, d, 0, !sp || !tm || idC ? z : -Bv + th1 * tau * Sv);
    PUT(0, -1, d, 2, !sp || !tm || idC ? z : -th1 * tau * Bv);
    // G row
    PUT(1, 0, d, 1, !sp ? z : idG ? (d == kCentre ? (T)1 : z) : Bv + th * tau * STv);
    PUT(1, 1, d, 1, !sp || !tp || idG ? z : -Bv + th1 * tau * STv);
    if (d == kCentre) {
      PUT(1, 0, d, 0, idG ? z : th1 * tau * pr.sj);
      PUT(1, 1, d, 0, !tp || idG ? z : th * tau * pr.sj);
    }
    // f row
    PUT(2, -1, d, 1, !sp || !tm ? z : -mt1 * Bv);
    PUT(2, -1, d, 2, !sp || !tm ? z : b1 * lt1 * Bv + b2 * mt1 * Kv);
    PUT(2, 0, d, 1, !sp ? z : -pr.mt0 * Bv);
    PUT(2, 0, d, 2, !sp ? z : b1 * pr.lt0 * Bv + b2 * pr.mt0 * Kv);
    PUT(2, 1, d, 1, !sp || !tp ? z : -mt1 * Bv);
    PUT(2, 1, d, 2, !sp || !tp ? z : b1 * lt1 * Bv + b2 * mt1 * Kv);
  }
#undef PUT
}

__device__ __forceinline__ void check_pivot(double d, int* status) {
  if (!(fabs(d) > 1e-300) || !isfinite(d)) atomicExch(status, 1);
}

template <typename T, int G>
__global__ void __launch_bounds__(factor_threads<T>, 2) ilu0_factor(const BoxDesc* __restrict__ boxes,
                                                                    const int* __restrict__ gptr,
                                                                    const int* __restrict__ perm,
                                                                    const int* __restrict__ ptab,
                                                                    T* __restrict__ F, int* __restrict__ status) {
  // per thread and pivot point: offset of its column in Fb
  constexpr int NS = factor_threads<T>;
  __shared__ int nbs[kGenNbrs * NS];
  const BoxDesc bx = boxes[blockIdx.x];
  T* Fb = F + bx.foff;
  const int* gp = gptr + bx.loff;
  const int* pm = perm + G * bx.goff;
  const int* pb = ptab + bx.poff;
  int* nb = nbs + threadIdx.x;
  const int unit = (int)bx.unit;
  for (int w = 0; w < bx.nlev; ++w) {
    const int q1 = G * gp[w + 1];
    for (int q = G * gp[w] + threadIdx.x; q < q1; q += blockDim.x) {
      const int lex = pm[q];
      if (lex < 0) continue;
      const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
      const int kt = lex / (bx.lx * bx.ly * bx.lz);
#pragma unroll 1
      for (int i = 0; i < kGenNbrs; ++i) {
        const int dt = c_gen_nbr[i][0], dz = c_gen_nbr[i][1], dy = c_gen_nbr[i][2], dx = c_gen_nbr[i][3];
        const int ax = kx + dx, ay = ky + dy, az = kz + dz, at = kt + dt;
        int e = unit;
        if (ax >= 0 && ax < bx.lx && ay >= 0 && ay < bx.ly && az >= 0 && az < bx.lz && at >= 0 && at < bx.lt)
          e = pb[ax + bx.lx * (ay + bx.ly * (az + bx.lz * at))];
        nb[i * NS] = e;
      }
      T* own = Fb + group_column<T, G>(q);
      // the G and f rows read the U parts of this point's C and G rows
      check_pivot((double)ilu_row0_64<T, NS, G>(own, Fb, nb), status);
      asm volatile("" ::: "memory");
      check_pivot((double)ilu_row1_64<T, NS, G>(own, Fb, nb), status);
      asm volatile("" ::: "memory");
      check_pivot((double)ilu_row2_64<T, NS, G>(own, Fb, nb), status);
    }
    __syncthreads();
  }
}

// gather, then factor, in place on F (groups of G points); both on stream s
template <typename T, int G>
kkt_status factor_launch(ras_precond* m, T* F, cudaStream_t s) {
  const dim3 g((unsigned)((G * (long long)m->max_groups + kGatherThreads - 1) / kGatherThreads), m->nbox);
  gather_groups<T, G><<<g, kGatherThreads, 0, s>>>(m->dprobs, m->boxes, m->gptr, m->perm, F);
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  {
    TimedScope timed(&m->factor_timing, s);
    ilu0_factor<T, G><<<m->nbox, factor_threads<T>, 0, s>>>(m->boxes, m->gptr, m->perm, m->ptab, F,
                                                      m->status);
  }
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

}  // namespace
