// Exact local solves of the one-level RAS: LU with partial pivoting of every
// subdomain matrix M_ij = R^delta F_h (R^delta)^T (Sec. 3.2, Eq. 10-12), FP64.
//
// Storage.  The unknowns of a box are numbered in its natural point-block
// order, u = 3 lex + c with lex = kx + lx (ky + ly (kz + lz kt)).  Every
// coupling of the KKT stencil then lies within kl = 3 (1 + lx + lx ly +
// lx ly lz) + 2 of the diagonal on either side, so the matrix is stored as a
// band, column-major with leading dimension ld = 3 kl + 1 (kl rows below the
// diagonal, kl above, and kl more for the fill that row interchanges bring
// into U): A(i, k) sits at A[(2 kl + i - k) + ld k].
//
// Factorisation (the column-by-column LU with partial pivoting of a band
// matrix): at step j the pivot is the first entry of largest magnitude in
// column j on or below the diagonal; rows j and p are interchanged in the
// columns j..ju (ju: the last column that fill can have reached), and the
// rank-1 update A(i, k) -= l_i u_k is applied below row j.  One launch per
// step covers all boxes; several CTAs share a box, each finds the pivot
// itself from column j and updates its own columns, and column j's own
// interchange and scaling by 1/pivot are written at the next step, when no
// CTA reads it any more.
//
// Solve.  One CTA per box: gather R^delta r, forward sweep with the row
// interchanges and the unit lower factor, backward sweep with U, scatter the
// owned part (R^0)^T; the box vector lives in shared memory.

#include <algorithm>
#include <cmath>

#include "slotval.cuh"

namespace {

constexpr int kLuThreads = 1024;
constexpr int kLuGather = 256;

__device__ __forceinline__ double* band_col(double* AB, const BoxDesc& bx, int k) {
  const int kl = bx.kl, ld = 3 * kl + 1;
  return AB + bx.aoff + (long long)ld * k + 2 * kl - k;   // [i] = A(i, k)
}

// the entries of every box matrix into its band (the band is zeroed before)
__global__ void __launch_bounds__(kLuGather) gather_band(DevProblem p, const BoxDesc* __restrict__ boxes,
                                                         double* __restrict__ AB) {
  const BoxDesc bx = boxes[blockIdx.y];
  const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (q >= bx.P) return;
  const int lex = (int)q;
  const Coefs<double> cf = coefs<double>(p);
  const PointRow<double> pr = point_row<double>(p, bx, lex);
  for (int s = 0; s < kSlots; ++s) {
    bool inb;
    const double v = slot_value<double>(p, bx, cf, pr, s, &inb);
    if (!inb) continue;
    const int c = s < kGenRowSlots0 ? 0 : (s < kGenRowSlots0 + kGenRowSlots1 ? 1 : 2);
    const int dt = c_gen_slot[s][0], dz = c_gen_slot[s][1], dy = c_gen_slot[s][2], dx = c_gen_slot[s][3];
    const int cc = c_gen_slot[s][4];
    const int lex2 = lex + dx + bx.lx * (dy + bx.ly * (dz + bx.lz * dt));
    const int i = 3 * lex + c, k = 3 * lex2 + cc;
    band_col(AB, bx, k)[i] = v;
  }
}

// One elimination step j for every box (grid: CTAs per box x boxes).  At
// j = n it only finishes column n - 1.
__global__ void __launch_bounds__(kLuThreads) lu_step(const BoxDesc* __restrict__ boxes, double* __restrict__ AB,
                                                      int* __restrict__ ipiv, int* __restrict__ ju2,
                                                      int* __restrict__ status, int j) {
  __shared__ double col[kMaxLuBand + 1];
  __shared__ double red_v[kLuThreads / 32];
  __shared__ int red_i[kLuThreads / 32];
  const BoxDesc bx = boxes[blockIdx.y];
  const int n = 3 * (int)bx.P, kl = bx.kl;
  int* ip = ipiv + 3 * bx.poff;
  // finish column j - 1: its interchange and its multipliers
  if (blockIdx.x == 0 && j >= 1 && j - 1 < n) {
    double* Ac = band_col(AB, bx, j - 1);
    const int jj = j - 1, p = ip[jj], km = min(kl, n - 1 - jj);
    const double a = Ac[jj], b = Ac[p];
    const double piv = b;
    const double rp = piv != 0.0 ? 1.0 / piv : 0.0;
    for (int t = 1 + threadIdx.x; t <= km; t += blockDim.x) {
      const double v = (jj + t == p) ? a : Ac[jj + t];
      Ac[jj + t] = v * rp;
    }
    __syncthreads();
    if (threadIdx.x == 0) Ac[jj] = piv;
  }
  if (j >= n) return;
  const double* Aj = band_col(AB, bx, j);
  const int km = min(kl, n - 1 - j);
  // pivot: first entry of largest magnitude on or below the diagonal
  double best = -1.0;
  int bi = 0;
  for (int t = threadIdx.x; t <= km; t += blockDim.x) {
    const double v = Aj[j + t];
    col[t] = v;
    if (fabs(v) > best) {
      best = fabs(v);
      bi = t;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > best || (ov == best && oi < bi)) {
      best = ov;
      bi = oi;
    }
  }
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nw = blockDim.x / 32;
  if (lane == 0) {
    red_v[warp] = best;
    red_i[warp] = bi;
  }
  __syncthreads();
  best = red_v[0];
  bi = red_i[0];
  for (int w = 1; w < nw; ++w)
    if (red_v[w] > best || (red_v[w] == best && red_i[w] < bi)) {
      best = red_v[w];
      bi = red_i[w];
    }
  const int jp = bi;
  const double piv = col[jp];
  const int ju_in = ju2[2 * blockIdx.y + (j & 1)];
  const int ju = max(ju_in, min(j + kl + jp, n - 1));
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ju2[2 * blockIdx.y + ((j + 1) & 1)] = ju;
    ip[j] = j + jp;
    if (!(piv != 0.0) || !isfinite(piv)) atomicExch(status, 1);
  }
  const double rp = piv != 0.0 ? 1.0 / piv : 0.0;
  // columns j+1..ju, one warp per column
  for (int k = j + 1 + blockIdx.x * nw + warp; k <= ju; k += gridDim.x * nw) {
    double* Ak = band_col(AB, bx, k);
    double u = Ak[j];
    if (jp != 0) {
      const double w = Ak[j + jp];
      if (lane == 0) {
        Ak[j + jp] = u;
        Ak[j] = w;
      }
      u = w;
    }
    __syncwarp();
    if (u != 0.0)
      for (int t = 1 + lane; t <= km; t += 32) {
        const double l = (t == jp ? col[0] : col[t]) * rp;
        Ak[j + t] -= l * u;
      }
  }
}

// z = sum over boxes (R^0)^T M_ij^{-1} R^delta r with the band LU factors.
//
// One CTA per box, one column a step, one barrier a step.  Row i belongs to
// thread i mod 1024: only it writes bvec[i].  What a step needs of other threads' rows
// -- the pivot row's value and, under an interchange, the value of row j -- their owners
// publish at the end of the step before, in slots that alternate.  A thread's
// entries of the next columns are loaded kLuAhead columns ahead into registers and
// the diagonals' reciprocals formed ahead, so a step's chain is two
// shared-memory reads, a few FMAs and the barrier.  (With the loads at their use and two
// barriers a column took 2.3 us.)  What is left is the FP64 pipe: 3 kl FMAs per
// column and box at 2 a clock.
constexpr int kLuAhead = 4;
constexpr int kLuFwd = (kMaxLuBand + kLuThreads - 1) / kLuThreads;       // rows per thread and column, L
constexpr int kLuBwd = (2 * kMaxLuBand + kLuThreads - 1) / kLuThreads;   // and U
static_assert((kLuThreads & (kLuThreads - 1)) == 0, "row owners by mask");

// v / d from r = 1 / d (rounded to nearest): the product and one correction by its exact residual,
// the last step of the division by Newton iteration of P. Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34 (1990).  The bits of the
// division, or one unit in the last place away where a value is subnormal; infinities, NaN and a
// reciprocal that overflows take the division itself.
__device__ __forceinline__ double quotient(double v, double d, double r) {
  const double q = v * r, e = fma(-d, q, v);
  return isfinite(e) ? fma(e, r, q) : v / d;
}

__global__ void quotient_selftest(const double* __restrict__ v, const double* __restrict__ d, double* __restrict__ q,
                                  long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) q[i] = quotient(v[i], d[i], 1.0 / d[i]);
}

// WIDE: a half-bandwidth above kLuThreads (more rows per thread)
template <bool WIDE>
__global__ void __launch_bounds__(kLuThreads) lu_solve(const BoxDesc* __restrict__ boxes,
                                                       const double* __restrict__ AB, const int* __restrict__ ipiv,
                                                       const double* __restrict__ r, double* __restrict__ z, int nx,
                                                       int ny, int N, const int* gate) {
  if (gated_off(gate)) return;
  constexpr int RF = WIDE ? kLuFwd : 1, RB = WIDE ? kLuBwd : 2;
  extern __shared__ __align__(16) double lu_sm[];
  double* pub = lu_sm;        // two alternating slots of {pivot row's value, row j's value} / {x_j}
  double* bvec = lu_sm + 4;
  const BoxDesc bx = boxes[blockIdx.x];
  const int n = 3 * (int)bx.P, kl = bx.kl, ld = 3 * kl + 1, t = threadIdx.x;
  const int* ip = ipiv + 3 * bx.poff;
  const double* A = AB + bx.aoff + 2 * kl;   // A(i, k) = A[(ld - 1) k + i]
  for (int u = t; u < n; u += kLuThreads) {
    const int lex = u / 3, c = u - 3 * lex;
    const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
    const int kt = lex / (bx.lx * bx.ly * bx.lz);
    const long long g =
        ((long long)(bx.t0 + kt) * N + (bx.x0 + kx) + (long long)nx * ((bx.y0 + ky) + (long long)ny * (bx.z0 + kz))) * 3;
    bvec[u] = r[g + c];
  }
  __syncthreads();
  const int mask = kLuThreads - 1;

  // forward: interchanges and the unit lower factor
  {
    double a[kLuAhead][RF];
    int piv[kLuAhead];
    auto load = [&](int j, double (&v)[RF], int& pj) {
      const double* Aj = A + (long long)(ld - 1) * j;
      const int i = j + 1 + ((t - j - 1) & mask), last = min(j + kl, n - 1);
#pragma unroll
      for (int q = 0; q < RF; ++q) v[q] = j < n - 1 && i + q * kLuThreads <= last ? Aj[i + q * kLuThreads] : 0.0;
      pj = j < n - 1 ? ip[j] : j;
    };
#pragma unroll
    for (int c = 0; c < kLuAhead; ++c) load(c, a[c], piv[c]);
    if (t == 0) {
      pub[0] = bvec[piv[0]];
      pub[1] = bvec[0];
    }
    __syncthreads();
    for (int j0 = 0; j0 < n - 1; j0 += kLuAhead) {
#pragma unroll
      for (int c = 0; c < kLuAhead; ++c) {
        const int j = j0 + c;
        if (j >= n - 1) break;
        const int p = piv[c];
        const double bj = pub[2 * (j & 1)], old = pub[2 * (j & 1) + 1];
        const int i = j + 1 + ((t - j - 1) & mask), last = min(j + kl, n - 1);
#pragma unroll
        for (int q = 0; q < RF; ++q) {
          const int ii = i + q * kLuThreads;
          if (ii <= last) bvec[ii] = fma(-a[c][q], bj, ii == p ? old : bvec[ii]);
        }
        if (t == (j & mask)) bvec[j] = bj;
        // the next column's pivot row and row, by their owners
        const int pn = piv[(c + 1) % kLuAhead];   // (loaded: kLuAhead > 1)
        if (j + 1 < n - 1) {
          if (t == (pn & mask)) pub[2 * ((j + 1) & 1)] = bvec[pn];
          if (t == ((j + 1) & mask)) pub[2 * ((j + 1) & 1) + 1] = bvec[j + 1];
        }
        load(j + kLuAhead, a[c], piv[c]);
        __syncthreads();
      }
    }
  }
  // backward: U has 2 kl superdiagonals
  {
    double a[kLuAhead][RB];
    auto load = [&](int j, double (&v)[RB]) {
      const double* Aj = A + (long long)(ld - 1) * j;
      const int i = j - 1 - ((j - 1 - t) & mask), first = max(0, j - 2 * kl);
#pragma unroll
      for (int q = 0; q < RB; ++q) v[q] = j > 0 && i - q * kLuThreads >= first ? Aj[i - q * kLuThreads] : 0.0;
    };
    // Diagonals and their reciprocals, a warp's 32 rows at a time: loaded two blocks of 32
    // columns before they are needed, divided one block before.
    const int warp = t / 32, warps = kLuThreads / 32;
    double ahead = 1.0, dg = 1.0, rd = 1.0;
    auto diag_load = [&](int blk) {
      if (blk >= 0 && blk % warps == warp) {
        const int row = 32 * blk + t % 32;
        ahead = row < n ? A[(long long)(ld - 1) * row + row] : 1.0;
      }
    };
    auto diag_divide = [&](int blk) {
      if (blk >= 0 && blk % warps == warp) {
        dg = ahead;
        rd = 1.0 / dg;
      }
    };
    const int top = (n - 1) / 32;
    diag_load(top);
    diag_divide(top);
    diag_load(top - 1);
#pragma unroll
    for (int c = 0; c < kLuAhead; ++c)
      if (n - 1 - c >= 0) load(n - 1 - c, a[c]);
    if (t == ((n - 1) & mask)) pub[2 * ((n - 1) & 1)] = quotient(bvec[n - 1], dg, rd);
    __syncthreads();
    for (int j0 = n - 1; j0 >= 0; j0 -= kLuAhead) {
#pragma unroll
      for (int c = 0; c < kLuAhead; ++c) {
        const int j = j0 - c;
        if (j < 0) break;
        if (j % 32 == 31 || j == n - 1) {   // a new block of columns: j / 32
          diag_divide(j / 32 - 1);
          diag_load(j / 32 - 2);
        }
        const double xj = pub[2 * (j & 1)];
        const int i = j - 1 - ((j - 1 - t) & mask), first = max(0, j - 2 * kl);
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          const int ii = i - q * kLuThreads;
          if (ii >= first) {
            const double v = fma(-a[c][q], xj, bvec[ii]);
            bvec[ii] = v;
            if (q == 0 && ii == j - 1) pub[2 * ((j - 1) & 1)] = quotient(v, dg, rd);
          }
        }
        if (t == (j & mask)) bvec[j] = xj;
        if (j - kLuAhead >= 0) load(j - kLuAhead, a[c]);
        __syncthreads();
      }
    }
  }
  // scatter the owned part
  const int ox = bx.ox1 - bx.ox0, oy = bx.oy1 - bx.oy0, oz = bx.oz1 - bx.oz0, ot = bx.ot1 - bx.ot0;
  const long long nown = (long long)ox * oy * oz * ot;
  for (long long q = threadIdx.x; q < nown; q += blockDim.x) {
    const int gx = bx.ox0 + (int)(q % ox), gy = bx.oy0 + (int)((q / ox) % oy);
    const int gz = bx.oz0 + (int)((q / ((long long)ox * oy)) % oz), gt = bx.ot0 + (int)(q / ((long long)ox * oy * oz));
    const int lex = (gx - bx.x0) + bx.lx * ((gy - bx.y0) + bx.ly * ((gz - bx.z0) + bx.lz * (gt - bx.t0)));
    const long long g = ((long long)gt * N + gx + (long long)nx * (gy + (long long)ny * gz)) * 3;
    z[g] = bvec[3 * lex];
    z[g + 1] = bvec[3 * lex + 1];
    z[g + 2] = bvec[3 * lex + 2];
  }
}

}  // namespace

kkt_status ras_lu_factor(ras_precond* m, cudaStream_t s) {
  const DevProblem dp = m->prob->dev();
  long long pmax = 0;
  int nmax = 0;
  for (const BoxDesc& b : m->boxes_h) {
    pmax = std::max(pmax, b.P);
    nmax = std::max(nmax, 3 * (int)b.P);
  }
  // the solve keeps a box's vector in shared memory (at most kMaxLuUnknowns values); the
  // limit is raised here, at set-up, so the solve's launch needs no attribute call
  KKT_TRY_CUDA(cudaFuncSetAttribute(lu_solve<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)((kMaxLuUnknowns + 4) * sizeof(double))));
  KKT_TRY_CUDA(cudaFuncSetAttribute(lu_solve<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)((kMaxLuUnknowns + 4) * sizeof(double))));
  KKT_TRY_CUDA(cudaMemsetAsync(m->AB, 0, m->ab_count * sizeof(double), s));
  KKT_TRY_CUDA(cudaMemsetAsync(m->lu_ju, 0, 2 * m->nbox * sizeof(int), s));
  const dim3 g((unsigned)((pmax + kLuGather - 1) / kLuGather), m->nbox);
  gather_band<<<g, kLuGather, 0, s>>>(dp, m->boxes, m->AB);
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  const dim3 sg(m->lu_ctas, m->nbox);
  for (int j = 0; j <= nmax; ++j) {
    lu_step<<<sg, kLuThreads, 0, s>>>(m->boxes, m->AB, m->ipiv, m->lu_ju, m->status, j);
    KKT_COUNT(1);
  }
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

kkt_status ras_lu_solve(ras_precond* m, const double* r, double* z, cudaStream_t s, const int* gate) {
  const kkt_problem* p = m->prob;
  int nmax = 0, klmax = 0;
  for (const BoxDesc& b : m->boxes_h) {
    nmax = std::max(nmax, 3 * (int)b.P);
    klmax = std::max(klmax, b.kl);
  }
  const size_t smem = ((size_t)nmax + 4) * sizeof(double);
  auto* kernel = klmax > kLuThreads ? lu_solve<true> : lu_solve<false>;   // L and U rows per thread: 2 and 4, or 1 and 2
  kernel<<<m->nbox, kLuThreads, smem, s>>>(m->boxes, m->AB, m->ipiv, r, z, p->nx, p->ny, p->N, gate);
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

extern "C" kkt_status lu_selftest_quotient(const double* v, const double* d, double* q, long long n, void* stream) {
  if (!v || !d || !q || n < 1 || n > (1LL << 30)) {
    set_error("lu_selftest_quotient: null argument or n outside [1, 2^30]");
    return KKT_ERR_ARG;
  }
  quotient_selftest<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(v, d, q, n);
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}
