// Subdomain solvers beyond ILU(0) (Sec. 4, Table 1; Sec. 3.2): ILU(1), the
// incomplete factorisation on the pattern grown by one level of fill, and the
// 3x3 point-block ILU(0), the incomplete factorisation on the pattern of whole
// point blocks (the point-block ordering of Sec. 3.2: C, G, f of a space-time
// point together).  Both run one pattern-driven elimination:
//
// Pattern.  Every row type c (C, G, f) has a list of slots (point offset
// (dt, dz, dy, dx), column component) in column order: the pattern of an
// interior point.  ILU(1): the level-1 pattern, found on the host by the
// symbolic elimination (levels of fill) on a box of 5^4 points around one
// point; block ILU(0): all components of the 81 points at offsets in
// {-1, 0, 1}^4.  A point near a box face or the domain boundary uses a subset:
// the per-point levels decide which slots it keeps.
//
// Values and levels.  Point-major per box, by the point's lexicographic index
// in the box (so a column's address is arithmetic on the point's, with no
// index lookup): slot s of point lex at F[foff + lex * S + s] (a warp takes
// one point, its lanes consecutive slots), its level of fill at LV[...] (0 for
// an entry of F_h's structural pattern, 255 for a slot the point does not
// have).  The local vectors of the solve are indexed the same way.
//
// Elimination (IKJ, rows in the natural point-block order, as the oracle's
// ILU0 on the same pattern).  For row (p, c): a symbolic pass over the L slots
// s in column order lowers the levels of the row's later slots through each
// pivot row's kept U entries (lev(s) + lev_piv(t) + 1); a numeric pass then
// divides by the pivot and updates every kept target.  The pairs (t, u) of a
// pivot slot t that lands on the row's slot u are tabulated on the host per
// (row type, L slot).  Schedule: wavefronts w = x + b y + b^2 z + b^3 t with
// b = R + 1 for the largest offset R of an L slot, so every L-slot column of
// a point lies on an earlier wavefront.
//
// Solve.  One CTA per box: gather R^delta r, forward and backward sweeps by
// wavefront over the same slot lists (a warp per point), scatter the owned
// points.  A slot's column comes from a table in shared memory (its offset in the
// box and the range of positions that have it), the box's vector sits there too
// where it fits; the point-block rows' values are loaded a point ahead and the
// three rows' columns together.

#include <algorithm>
#include <array>
#include <cstring>
#include <map>
#include <mutex>
#include <type_traits>
#include <vector>

#include "ras.cuh"
#include "slotval.cuh"

namespace {

constexpr int kGpMaxRow = 800;       // slots of one row type at most (ILU(1): 780 in the C row)

struct GpSlot {
  int dt, dz, dy, dx, cc;
};

bool slot_less(const GpSlot& a, const GpSlot& b) {
  if (a.dt != b.dt) return a.dt < b.dt;
  if (a.dz != b.dz) return a.dz < b.dz;
  if (a.dy != b.dy) return a.dy < b.dy;
  if (a.dx != b.dx) return a.dx < b.dx;
  return a.cc < b.cc;
}

// Structural columns of row c of an interior point (all sensor couplings
// present): C rows couple C and f at levels n-1, n; G rows G at n, n+1 and C
// at the node itself at n, n+1; f rows G and f at n-1, n, n+1 (Appendix).
std::vector<GpSlot> structural_row(int c) {
  std::vector<GpSlot> out;
  for (int dt = -1; dt <= 1; ++dt)
    for (int dz = -1; dz <= 1; ++dz)
      for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx) {
          if (c == 0 && dt <= 0) {
            out.push_back({dt, dz, dy, dx, 0});
            out.push_back({dt, dz, dy, dx, 2});
          } else if (c == 1 && dt >= 0) {
            out.push_back({dt, dz, dy, dx, 1});
            if (dz == 0 && dy == 0 && dx == 0) out.push_back({dt, 0, 0, 0, 0});
          } else if (c == 2) {
            out.push_back({dt, dz, dy, dx, 1});
            out.push_back({dt, dz, dy, dx, 2});
          }
        }
  std::sort(out.begin(), out.end(), slot_less);
  return out;
}

// Interior level-1 pattern per row type: the symbolic IKJ elimination with
// levels of fill on a box of 5^4 points (every level-1 path of the centre
// point's rows runs through points within distance 2), read at the centre.
std::array<std::vector<GpSlot>, 3> ilu1_interior_rows() {
  constexpr int E = 5, NP = E * E * E * E, NR = 3 * NP;
  auto col_of = [&](int x, int y, int z, int t, int c) { return 3 * (x + E * (y + E * (z + E * t))) + c; };
  std::vector<std::vector<std::pair<int, int>>> ulev(NR);   // kept upper entries (column, level)
  std::array<std::vector<GpSlot>, 3> rows;
  std::vector<int> lev(NR);
  const int centre = 2 + E * (2 + E * (2 + E * 2));
  for (int i = 0; i < NR; ++i) {
    const int pt = i / 3, c = i % 3;
    const int x = pt % E, y = (pt / E) % E, z = (pt / (E * E)) % E, t = pt / (E * E * E);
    std::fill(lev.begin(), lev.end(), 1 << 20);
    for (const GpSlot& s : structural_row(c)) {
      const int X = x + s.dx, Y = y + s.dy, Z = z + s.dz, T = t + s.dt;
      if (X < 0 || X >= E || Y < 0 || Y >= E || Z < 0 || Z >= E || T < 0 || T >= E) continue;
      lev[col_of(X, Y, Z, T, s.cc)] = 0;
    }
    for (int m = 0; m < i; ++m) {   // L entries in column order (fill joins before it is reached)
      if (lev[m] > 1) continue;
      for (const auto& e : ulev[m]) {
        const int nl = lev[m] + e.second + 1;
        if (nl <= 1 && nl < lev[e.first]) lev[e.first] = nl;
      }
    }
    for (int j = i + 1; j < NR; ++j)
      if (lev[j] <= 1) ulev[i].push_back({j, lev[j]});
    if (pt == centre)
      for (int j = 0; j < NR; ++j)
        if (lev[j] <= 1) {
          const int q = j / 3;
          rows[c].push_back({q / (E * E * E) - 2, (q / (E * E)) % E - 2, (q / E) % E - 2, q % E - 2, j % 3});
        }
  }
  for (auto& r : rows) std::sort(r.begin(), r.end(), slot_less);
  return rows;
}

std::array<std::vector<GpSlot>, 3> block_rows() {
  std::array<std::vector<GpSlot>, 3> rows;
  for (int c = 0; c < 3; ++c) {
    for (int dt = -1; dt <= 1; ++dt)
      for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
          for (int dx = -1; dx <= 1; ++dx)
            for (int cc = 0; cc < 3; ++cc) rows[c].push_back({dt, dz, dy, dx, cc});
    std::sort(rows[c].begin(), rows[c].end(), slot_less);
  }
  return rows;
}

std::array<std::vector<GpSlot>, 3> gp_rows(int local) {
  static std::array<std::vector<GpSlot>, 3> ilu1, blk;   // built once per process
  static bool have1 = false, haveb = false;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  if (local == 2) {
    if (!have1) {
      ilu1 = ilu1_interior_rows();
      have1 = true;
    }
    return ilu1;
  }
  if (!haveb) {
    blk = block_rows();
    haveb = true;
  }
  return blk;
}

}  // namespace

// Slots per row type of an interior point under the local solver `local`
// (0 ILU(0), 2 ILU(1), 3 point-block ILU(0)); host only.
extern "C" kkt_status ras_local_pattern(int local, int counts[3]) {
  if (!counts || (local != 0 && local != 2 && local != 3)) {
    set_error("ras_local_pattern: counts is null, or local is not 0, 2 or 3");
    return KKT_ERR_ARG;
  }
  if (local == 0) {
    for (int c = 0; c < 3; ++c) counts[c] = (int)structural_row(c).size();
    return KKT_OK;
  }
  const auto rows = gp_rows(local);
  for (int c = 0; c < 3; ++c) counts[c] = (int)rows[c].size();
  return KKT_OK;
}

// ---------------------------------------------------------------------------
// Device side
// ---------------------------------------------------------------------------

// Per-box storage of the pattern-driven factors.
struct GpBox {
  long long foff;   // values / levels: slot s of point lex (box-lexicographic) at foff + lex * S + s
  long long voff;   // local vector: 3 values per point
  long long poff;   // schedule array (perm: schedule position -> lexicographic index)
  long long loff;   // wavefront pointers
  int nlev;
  int P;
};

struct GpTables {
  const signed char* slot;   // [S][5]: dt, dz, dy, dx, column component
  const short* smap;         // [S]: the slot's index among the ILU(0) slots (its value), or -1
  const int* tptr;           // [S + 1]: update pairs of each L slot (global slot numbering)
  const int* tt;             // pivot-row slot (global index) of each pair
  const short* tu;           // target slot (row-local index) of each pair
  int base[3], cnt[3], diag[3];   // row types: first global slot, slots, row-local diagonal
  int S;                     // slots per point
  int K;                     // kept level of fill (ILU(1): 1, point-block ILU(0): 0)
};

struct GpFactor {
  int local = 2;
  int prec = 64;
  GpTables tab{};
  std::vector<GpBox> boxes_h;
  GpBox* boxes = nullptr;
  int* perm = nullptr;
  int* lptr = nullptr;
  signed char* slot = nullptr;
  short* smap = nullptr;
  int* tptr = nullptr;
  int* tt = nullptr;
  short* tu = nullptr;
  void* F = nullptr;
  unsigned char* LV = nullptr;
  void* V = nullptr;
  long long fcount = 0, vcount = 0;
  ~GpFactor() {
    cudaFree(boxes);
    cudaFree(perm);
    cudaFree(lptr);
    cudaFree(slot);
    cudaFree(smap);
    cudaFree(tptr);
    cudaFree(tt);
    cudaFree(tu);
    cudaFree(F);
    cudaFree(LV);
    cudaFree(V);
  }
};

namespace {

constexpr int kGpSmemLimit = 112 * 1024;   // two CTAs of the solve per SM
constexpr int kGpThreads = 192;        // factor CTA (row buffers: 6 warps x 800 slots fit 48 KB in FP64)

__device__ __forceinline__ int gp_row_of(const GpTables& tb, int s) {
  return s < tb.base[1] ? 0 : (s < tb.base[2] ? 1 : 2);
}

// Lexicographic box index of the column point of slot s, or -1 outside the box.
__device__ __forceinline__ int gp_col_lex(const BoxDesc& bx, const signed char* sl, int kx, int ky, int kz, int kt) {
  const int ax = kx + sl[3], ay = ky + sl[2], az = kz + sl[1], at = kt + sl[0];
  if (ax < 0 || ax >= bx.lx || ay < 0 || ay >= bx.ly || az < 0 || az >= bx.lz || at < 0 || at >= bx.lt) return -1;
  return ax + bx.lx * (ay + bx.ly * (az + bx.lz * at));
}

// Initial values (the principal submatrix of F_h on the box, Eq. 10-12) and
// levels (0: F_h's structural pattern; 255: not kept unless fill reaches it).
// One warp per point, its lanes over the slots (point-major storage).
template <typename T>
__global__ void gp_gather(const DevProblem* __restrict__ probs, const BoxDesc* __restrict__ boxes,
                          const GpBox* __restrict__ gb, const int* __restrict__ perm, GpTables tb, T* __restrict__ F,
                          unsigned char* __restrict__ LV) {
  const BoxDesc bx = boxes[blockIdx.y];
  const GpBox g = gb[blockIdx.y];
  const int q = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (q >= g.P) return;
  const DevProblem p = probs[bx.prob];
  const Coefs<T> cf = coefs<T>(p);
  const int lex = perm[g.poff + q];
  const PointRow<T> pr = point_row<T>(p, bx, lex);
  const bool idC = pr.n == 0 || pr.dirj, idG = pr.n == p.M || pr.dirj;
  const long long o = g.foff + (long long)lex * tb.S;
  for (int s = lane; s < tb.S; s += 32) {
    const signed char* sl = tb.slot + 5 * s;
    const int c = gp_row_of(tb, s);
    const bool inb = gp_col_lex(bx, sl, pr.kx, pr.ky, pr.kz, pr.kt) >= 0;
    const int ss = tb.smap[s];
    T v = (T)0;
    bool structural = false;
    if (inb && ss >= 0) {
      bool ib;
      v = slot_value<T>(p, bx, cf, pr, ss, &ib);
      const bool diag = s - tb.base[c] == tb.diag[c];
      structural = !((c == 0 && idC && !diag) || (c == 1 && idG && !diag) ||
                     (c == 1 && sl[4] == 0 && pr.sj == (T)0));
    }
    const bool keep0 = tb.K == 0 ? inb : structural;   // point-block: every in-box slot
    F[o + s] = v;
    LV[o + s] = keep0 ? 0 : 255;
  }
}

__device__ __forceinline__ void gp_check_pivot(double d, int* status) {
  if (!(fabs(d) > 1e-300) || !isfinite(d)) atomicExch(status, 1);
}

constexpr int kGpWarps = kGpThreads / 32;

// One CTA per box; wavefronts in order with a barrier between them; one warp
// per point, its C, G and f rows in turn (IKJ, see the file header).  The row
// (values and levels) sits in the warp's shared memory during its
// elimination; the L slots go in order, the update pairs of one L slot
// (distinct targets) are split over the lanes.
template <typename T>
__global__ void __launch_bounds__(kGpThreads) gp_factor(const BoxDesc* __restrict__ boxes,
                                                        const GpBox* __restrict__ gb, const int* __restrict__ perm,
                                                        const int* __restrict__ lptr,
                                                        GpTables tb, T* __restrict__ F, unsigned char* __restrict__ LV,
                                                        int* __restrict__ status) {
  __shared__ T rowv[kGpWarps][kGpMaxRow];
  __shared__ unsigned char rowl[kGpWarps][kGpMaxRow];
  const BoxDesc bx = boxes[blockIdx.x];
  const GpBox g = gb[blockIdx.x];
  const int lane = threadIdx.x & 31, wp = threadIdx.x / 32;
  T* rv = rowv[wp];
  unsigned char* rl = rowl[wp];
  const int K = tb.K;
  for (int w = 0; w < g.nlev; ++w) {
    const int l0 = lptr[g.loff + w], l1 = lptr[g.loff + w + 1];
    for (int q = l0 + wp; q < l1; q += kGpWarps) {
      const int lex = perm[g.poff + q];
      const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
      const int kt = lex / (bx.lx * bx.ly * bx.lz);
      T* own = F + g.foff + (long long)lex * tb.S;
      unsigned char* ownl = LV + g.foff + (long long)lex * tb.S;
      for (int c = 0; c < 3; ++c) {
        const int b = tb.base[c], nrow = tb.cnt[c], dg = tb.diag[c];
        for (int u = lane; u < nrow; u += 32) {
          rv[u] = own[b + u];
          rl[u] = ownl[b + u];
        }
        __syncwarp();
        if (K > 0) {   // symbolic pass: final levels of the row
          for (int s = 0; s < dg; ++s) {
            const int ls = rl[s];
            if (ls > K) continue;
            const int qp = gp_col_lex(bx, tb.slot + 5 * (b + s), kx, ky, kz, kt);
            const unsigned char* pl = LV + g.foff + (long long)qp * tb.S;
            for (int e = tb.tptr[b + s] + lane; e < tb.tptr[b + s + 1]; e += 32) {
              const int lp = pl[tb.tt[e]];
              const int nl = ls + lp + 1;
              const int u = tb.tu[e];
              if (lp <= K && nl <= K && nl < rl[u]) rl[u] = (unsigned char)nl;
            }
            __syncwarp();
          }
        }
        // numeric pass (a pivot's dropped entries hold 0, so every pair may update)
        for (int s = 0; s < dg; ++s) {
          if (rl[s] > K) continue;
          const int sc = tb.slot[5 * (b + s) + 4];
          const int qp = gp_col_lex(bx, tb.slot + 5 * (b + s), kx, ky, kz, kt);
          const T* pv = F + g.foff + (long long)qp * tb.S;
          const T l = rv[s] * pv[tb.base[sc] + tb.diag[sc]];
          for (int e = tb.tptr[b + s] + lane; e < tb.tptr[b + s + 1]; e += 32) {
            const int u = tb.tu[e];
            if (rl[u] <= K) rv[u] -= l * pv[tb.tt[e]];
          }
          __syncwarp();
          if (lane == 0) rv[s] = l;
        }
        __syncwarp();
        if (lane == 0) {
          const T d = rv[dg];
          gp_check_pivot((double)d, status);
          rv[dg] = (T)1 / d;
        }
        __syncwarp();
        for (int u = lane; u < nrow; u += 32) {
          own[b + u] = rv[u];
          ownl[b + u] = rl[u] <= K ? rl[u] : 255;
        }
        __syncwarp();
      }
    }
    __syncthreads();
  }
}

// z = sum over boxes (R^0)^T M^{-1} R^delta r with the pattern-driven factors:
// one CTA per box gathers its residual, sweeps forward and backward by
// wavefront, one warp per point and row, its lanes summing over the slots
// (slots whose column leaves the box are skipped; dropped entries hold 0),
// and writes its owned points.
//
// NIT: 32-slot steps of the longest row half.  BLOCK (the point-block pattern, 4
// steps): all three rows' values and columns are in registers at once, the values
// loaded a point ahead; a column of the point itself takes the value just solved.
// What bounds it is latency: a wavefront of 18 points (16^3 x 32, 4^4 boxes) is a
// round or two of the CTA's 12 warps.  Measured there, FP32: 5.47 -> 1.12 ms, FP64 7.09 -> 2.84, against
// index arithmetic per slot, rows one after the other, 8 warps; ILU(1) at 9^3 x 12, 3^4 boxes: 3.71 -> 1.10.
constexpr int kGpOwn = 1 << 22, kGpComp = 20;   // slot table: the point's own column, component (2 bits)
template <int NIT>
constexpr int gp_solve_threads() {
  return NIT <= 4 ? 384 : 256;
}

template <typename T, int NIT, bool SMEM>
__global__ void __launch_bounds__(gp_solve_threads<NIT>(), 2) gp_solve(
    const DevProblem* __restrict__ probs, const BoxDesc* __restrict__ boxes, const GpBox* __restrict__ gb,
    const int* __restrict__ perm, const int* __restrict__ lptr, GpTables tb, const T* __restrict__ F,
    T* __restrict__ V, const double* __restrict__ r, double* __restrict__ z, const int* gate) {
  if (gated_off(gate)) return;
  constexpr bool BLOCK = NIT <= 4;
  constexpr int nwarp = gp_solve_threads<NIT>() / 32;
  extern __shared__ __align__(16) unsigned char gp_sm[];
  int2* info = reinterpret_cast<int2*>(gp_sm);   // [S]: offset in the box's vector, positions that have the slot
  const BoxDesc bx = boxes[blockIdx.x];
  const GpBox g = gb[blockIdx.x];
  const int nx = probs[bx.prob].nx, ny = probs[bx.prob].ny, N = probs[bx.prob].N;
  T* Vb = SMEM ? reinterpret_cast<T*>(info + tb.S) : V + g.voff;
  const T* Fb = F + g.foff;
  const int* pm = perm + g.poff;
  const int* lp = lptr + g.loff;
  const int lane = threadIdx.x & 31, wp = threadIdx.x / 32;
  for (int s = threadIdx.x; s < tb.S; s += blockDim.x) {
    const signed char* sl = tb.slot + 5 * s;
    const int dt = sl[0], dz = sl[1], dy = sl[2], dx = sl[3], cc = sl[4];
    const bool own = dt == 0 && dz == 0 && dy == 0 && dx == 0;
    info[s] = make_int2(3 * (dx + bx.lx * (dy + bx.ly * (dz + bx.lz * dt))) + cc,
                        1 << (dx + 2) | 1 << (dy + 7) | 1 << (dz + 12) | 1 << (dt + 17) | cc << kGpComp | (own ? kGpOwn : 0));
  }
  auto global_point = [&](int lex) {
    const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
    const int kt = lex / (bx.lx * bx.ly * bx.lz);
    return (long long)(bx.t0 + kt) * N + (bx.x0 + kx) + (long long)nx * ((bx.y0 + ky) + (long long)ny * (bx.z0 + kz));
  };
  for (int lex = threadIdx.x; lex < g.P; lex += blockDim.x) {   // R^delta r
    const long long gi = 3 * global_point(lex);
    for (int c = 0; c < 3; ++c) Vb[3 * lex + c] = (T)r[gi + c];
  }
  __syncthreads();
  // offsets -2..2 that stay inside an axis of n at position k
  auto inside = [](int k, int n) {
    int m = 0;
#pragma unroll
    for (int d = -2; d <= 2; ++d) m |= (k + d >= 0 && k + d < n ? 1 : 0) << (d + 2);
    return m;
  };
  auto sweep = [&](auto pass_tag) {
    constexpr int pass = decltype(pass_tag)::value;   // 0 forward, 1 backward
    auto first = [&](int c) { return pass == 0 ? 0 : tb.diag[c] + 1; };
    auto count = [&](int c) { return pass == 0 ? tb.diag[c] : tb.cnt[c] - tb.diag[c] - 1; };
    T v[BLOCK ? 3 : 1][NIT];
    auto values = [&](int lex, int c, T (&o)[NIT]) {
      const T* Fp = Fb + (long long)lex * tb.S + tb.base[c] + first(c);
      const int n = count(c);
#pragma unroll
      for (int k = 0; k < NIT; ++k) o[k] = 32 * k + lane < n ? Fp[32 * k + lane] : (T)0;
    };
    // the warp's first point of a wavefront, its values loaded before the wavefront before ends
    auto wave = [&](int wi) { return pass == 0 ? wi : g.nlev - 1 - wi; };
    int q = lp[wave(0)] + wp, q1 = lp[wave(0) + 1], lex = q < q1 ? pm[q] : -1;
    if (BLOCK && lex >= 0)
#pragma unroll
      for (int c = 0; c < 3; ++c) values(lex, c, v[BLOCK ? c : 0]);
    for (int wi = 0; wi < g.nlev; ++wi) {
      const int wn = wave(min(wi + 1, g.nlev - 1)), qn = lp[wn] + wp, qn1 = wi + 1 < g.nlev ? lp[wn + 1] : 0;
      while (q < q1) {
        const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
        const int kt = lex / (bx.lx * bx.ly * bx.lz);
        const int here = inside(kx, bx.lx) | inside(ky, bx.ly) << 5 | inside(kz, bx.lz) << 10 | inside(kt, bx.lt) << 15;
        const T* Vp = Vb + 3 * lex;
        T x[BLOCK ? 3 : 1][NIT], sol[3] = {0, 0, 0}, old[3], inv[3];
        int own_k[3], own_c[3];   // the lane's slot of the point itself in row c: step (or -1) and component
        auto columns = [&](int c, T (&o)[NIT]) {
          const int n = count(c), b = tb.base[c] + first(c);
          own_k[c] = -1;
          own_c[c] = 0;
#pragma unroll
          for (int k = 0; k < NIT; ++k) {
            o[k] = (T)0;
            if (32 * k + lane < n) {
              const int2 e = info[b + 32 * k + lane];
              if (e.y & kGpOwn) {
                own_k[c] = k;
                own_c[c] = e.y >> kGpComp & 3;
              } else if ((e.y & here) == (e.y & 0xfffff)) {
                o[k] = Vp[e.x];
              }
            }
          }
        };
        const T* Fp = Fb + (long long)lex * tb.S;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          old[c] = Vp[c];
          inv[c] = pass == 1 ? Fp[tb.base[c] + tb.diag[c]] : (T)1;
        }
        if (BLOCK)
#pragma unroll
          for (int c = 0; c < 3; ++c) columns(c, x[BLOCK ? c : 0]);
        // the next point's index (and, point-block, its values, once this point's are used)
        int qx = q + nwarp, lexn = -1;
        if (qx < q1) lexn = pm[qx];
        else if (qn < qn1) lexn = pm[qn];
        auto row = [&](int c) {
          if (!BLOCK) {
            values(lex, c, v[0]);
            columns(c, x[0]);
          }
          T part = (T)0;
#pragma unroll
          for (int k = 0; k < NIT; ++k) {
            T xk = x[BLOCK ? c : 0][k];
            if (k == own_k[c]) xk = own_c[c] == 0 ? sol[0] : own_c[c] == 1 ? sol[1] : sol[2];
            part += v[BLOCK ? c : 0][k] * xk;
          }
          for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
          T acc = old[c] - part;
          if (pass == 1) acc *= inv[c];   // the stored 1 / u_ii
          sol[c] = acc;
        };
        if (pass == 0) {
          row(0);
          row(1);
          row(2);
        } else {
          row(2);
          row(1);
          row(0);
        }
        if (lane < 3) Vb[3 * lex + lane] = lane == 0 ? sol[0] : lane == 1 ? sol[1] : sol[2];
        if (BLOCK && lexn >= 0)
#pragma unroll
          for (int c = 0; c < 3; ++c) values(lexn, c, v[BLOCK ? c : 0]);
        q = qx;
        if (q < q1) lex = lexn;
      }
      __syncthreads();
      // (a warp without a point in this wavefront has not looked at the next one yet)
      if (wi + 1 < g.nlev) {
        const bool had = lp[wave(wi)] + wp < q1;
        q = qn;
        q1 = qn1;
        if (q < q1) {
          lex = pm[q];
          if (BLOCK && !had)
#pragma unroll
            for (int c = 0; c < 3; ++c) values(lex, c, v[BLOCK ? c : 0]);
        }
      }
    }
  };
  sweep(std::integral_constant<int, 0>{});
  sweep(std::integral_constant<int, 1>{});
  for (int lex = threadIdx.x; lex < g.P; lex += blockDim.x) {   // (R^0)^T: owned points only
    const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
    const int kt = lex / (bx.lx * bx.ly * bx.lz);
    const int x = bx.x0 + kx, y = bx.y0 + ky, zz = bx.z0 + kz, t = bx.t0 + kt;
    if (x < bx.ox0 || x >= bx.ox1 || y < bx.oy0 || y >= bx.oy1 || zz < bx.oz0 || zz >= bx.oz1 || t < bx.ot0 ||
        t >= bx.ot1)
      continue;
    const long long gi = 3 * global_point(lex);
    for (int c = 0; c < 3; ++c) z[gi + c] = (double)Vb[3 * lex + c];
  }
}

template <typename T>
kkt_status gp_factor_t(ras_precond* m, cudaStream_t s) {
  GpFactor* f = m->gp;
  int pmax = 0;
  for (const GpBox& b : f->boxes_h) pmax = std::max(pmax, b.P);
  gp_gather<T><<<dim3((pmax + 7) / 8, m->nbox), 256, 0, s>>>(m->dprobs, m->boxes, f->boxes, f->perm, f->tab,
                                                             (T*)f->F, f->LV);
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  {
    TimedScope timed(&m->factor_timing, s);
    gp_factor<T><<<m->nbox, kGpThreads, 0, s>>>(m->boxes, f->boxes, f->perm, f->lptr, f->tab, (T*)f->F,
                                                f->LV, m->status);
  }
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

}  // namespace

kkt_status gp_factor(ras_precond* m, cudaStream_t s) {
  return m->gp->prec == 64 ? gp_factor_t<double>(m, s) : gp_factor_t<float>(m, s);
}

namespace {

// shared memory of the solve: the slot table, and the largest box vector where two CTAs fit an SM with it
size_t gp_solve_smem(const GpFactor* f, bool* vec) {
  int pmax = 0;
  for (const GpBox& b : f->boxes_h) pmax = std::max(pmax, b.P);
  const size_t table = (size_t)f->tab.S * sizeof(int2);
  const size_t v = 3 * (size_t)pmax * (f->prec == 64 ? sizeof(double) : sizeof(float));
  *vec = table + v <= kGpSmemLimit;
  return table + (*vec ? v : 0);
}

template <typename T, int NIT>
kkt_status gp_solve_launch(ras_precond* m, const double* r, double* z, cudaStream_t s, const int* gate) {
  GpFactor* f = m->gp;
  bool vec = false;
  const size_t smem = gp_solve_smem(f, &vec);
  auto* kernel = vec ? gp_solve<T, NIT, true> : gp_solve<T, NIT, false>;
  kernel<<<m->nbox, gp_solve_threads<NIT>(), smem, s>>>(m->dprobs, m->boxes, f->boxes, f->perm, f->lptr, f->tab,
                                                        (const T*)f->F, (T*)f->V, r, z, gate);
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

template <typename T, int NIT>
kkt_status gp_solve_prepare() {   // raises the shared-memory limit, at set-up
  KKT_TRY_CUDA(cudaFuncSetAttribute(gp_solve<T, NIT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGpSmemLimit));
  KKT_TRY_CUDA(cudaFuncSetAttribute(gp_solve<T, NIT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGpSmemLimit));
  return KKT_OK;
}

}  // namespace

kkt_status gp_solve(ras_precond* m, const double* r, double* z, cudaStream_t s, const int* gate) {
  const bool block = m->gp->local == 3;
  if (m->gp->prec == 64)
    return block ? gp_solve_launch<double, 4>(m, r, z, s, gate) : gp_solve_launch<double, 14>(m, r, z, s, gate);
  return block ? gp_solve_launch<float, 4>(m, r, z, s, gate) : gp_solve_launch<float, 14>(m, r, z, s, gate);
}

void gp_destroy(ras_precond* m) {
  delete m->gp;
  m->gp = nullptr;
}

// Tables, schedule and storage of the pattern-driven factors of m's boxes.
kkt_status gp_create(ras_precond* m, int local, int prec) {
  GpFactor* f = new (std::nothrow) GpFactor();
  if (!f) return KKT_ERR_NOMEM;
  m->gp = f;
  f->local = local;
  f->prec = prec;
  const auto rows = gp_rows(local);
  GpTables& tb = f->tab;
  tb.K = local == 2 ? 1 : 0;
  std::vector<GpSlot> all;
  for (int c = 0; c < 3; ++c) {
    if ((int)rows[c].size() > kGpMaxRow) {
      set_error("ras_setup: internal error: a pattern row exceeds the kernel's level buffer");
      return KKT_ERR_ARG;
    }
    tb.base[c] = (int)all.size();
    tb.cnt[c] = (int)rows[c].size();
    tb.diag[c] = -1;
    for (int u = 0; u < tb.cnt[c]; ++u) {
      const GpSlot& sl = rows[c][u];
      if (sl.dt == 0 && sl.dz == 0 && sl.dy == 0 && sl.dx == 0 && sl.cc == c) tb.diag[c] = u;
      all.push_back(sl);
    }
    if (tb.diag[c] < 0) {
      set_error("ras_setup: internal error: a pattern row has no diagonal");
      return KKT_ERR_ARG;
    }
  }
  tb.S = (int)all.size();
  // the ILU(0) slot of each slot (its value comes from slot_value)
  signed char gen[kSlots][5];
  KKT_TRY_CUDA(cudaMemcpyFromSymbol(gen, c_gen_slot, sizeof(gen)));
  auto key = [](int c, int dt, int dz, int dy, int dx, int cc) {
    return ((((c * 3 + dt + 1) * 3 + dz + 1) * 3 + dy + 1) * 3 + dx + 1) * 3 + cc;
  };
  std::map<int, int> gen_of;
  for (int s = 0; s < kSlots; ++s) {
    const int c = s < kGenRowSlots0 ? 0 : (s < kGenRowSlots0 + kGenRowSlots1 ? 1 : 2);
    gen_of[key(c, gen[s][0], gen[s][1], gen[s][2], gen[s][3], gen[s][4])] = s;
  }
  std::vector<signed char> slot(5 * (size_t)tb.S);
  std::vector<short> smap(tb.S, -1);
  int R = 0;
  for (int c = 0; c < 3; ++c)
    for (int u = 0; u < tb.cnt[c]; ++u) {
      const GpSlot& sl = all[tb.base[c] + u];
      const int s = tb.base[c] + u;
      slot[5 * s] = (signed char)sl.dt;
      slot[5 * s + 1] = (signed char)sl.dz;
      slot[5 * s + 2] = (signed char)sl.dy;
      slot[5 * s + 3] = (signed char)sl.dx;
      slot[5 * s + 4] = (signed char)sl.cc;
      if (std::abs(sl.dt) <= 1 && std::abs(sl.dz) <= 1 && std::abs(sl.dy) <= 1 && std::abs(sl.dx) <= 1) {
        const auto it = gen_of.find(key(c, sl.dt, sl.dz, sl.dy, sl.dx, sl.cc));
        if (it != gen_of.end()) smap[s] = (short)it->second;
      }
      if (u < tb.diag[c])
        R = std::max({R, std::abs(sl.dt), std::abs(sl.dz), std::abs(sl.dy), std::abs(sl.dx)});
    }
  // update pairs: L slot s of row c (pivot row type cc_s at offset o_s) and U
  // slot t of the pivot row land on the row's slot u at o_s + o_t
  std::map<std::array<int, 6>, int> local_of;
  for (int c = 0; c < 3; ++c)
    for (int u = 0; u < tb.cnt[c]; ++u) {
      const GpSlot& sl = rows[c][u];
      local_of[{c, sl.dt, sl.dz, sl.dy, sl.dx, sl.cc}] = u;
    }
  std::vector<int> tptr(tb.S + 1, 0), tt;
  std::vector<short> tu;
  for (int c = 0; c < 3; ++c)
    for (int s = 0; s < tb.cnt[c]; ++s) {
      tptr[tb.base[c] + s] = (int)tt.size();
      if (s >= tb.diag[c]) continue;
      const GpSlot& a = rows[c][s];
      const int cs = a.cc;
      for (int t = tb.diag[cs] + 1; t < tb.cnt[cs]; ++t) {
        const GpSlot& b = rows[cs][t];
        const auto it = local_of.find({c, a.dt + b.dt, a.dz + b.dz, a.dy + b.dy, a.dx + b.dx, b.cc});
        if (it == local_of.end()) continue;
        if (it->second <= s) {
          set_error("ras_setup: internal error: an update lands left of its pivot slot");
          return KKT_ERR_ARG;
        }
        tt.push_back(tb.base[cs] + t);
        tu.push_back((short)it->second);
      }
    }
  tptr[tb.S] = (int)tt.size();
  // schedule: wavefronts x + b y + b^2 z + b^3 t, b = R + 1 (every L-slot column earlier)
  const int bw = R + 1;
  for (int c = 0; c < 3; ++c)
    for (int s = 0; s < tb.diag[c]; ++s) {
      const GpSlot& a = rows[c][s];
      if (a.dx + bw * (a.dy + bw * (a.dz + bw * a.dt)) >= 0 && !(a.dt == 0 && a.dz == 0 && a.dy == 0 && a.dx == 0)) {
        set_error("ras_setup: internal error: a pivot column is not on an earlier wavefront");
        return KKT_ERR_ARG;
      }
    }
  std::vector<int> perm, lptr;
  long long foff = 0, voff = 0;
  for (const BoxDesc& bx : m->boxes_h) {
    GpBox g{};
    g.P = (int)bx.P;
    g.foff = foff;
    g.voff = voff;
    g.poff = (long long)perm.size();
    g.loff = (long long)lptr.size();
    g.nlev = (bx.lx - 1) + bw * ((bx.ly - 1) + bw * ((bx.lz - 1) + bw * (bx.lt - 1))) + 1;
    std::vector<int> cnt(g.nlev + 1, 0);
    auto wof = [&](int lex) {
      const int kx = lex % bx.lx, ky = (lex / bx.lx) % bx.ly, kz = (lex / (bx.lx * bx.ly)) % bx.lz;
      const int kt = lex / (bx.lx * bx.ly * bx.lz);
      return kx + bw * (ky + bw * (kz + bw * kt));
    };
    for (int lex = 0; lex < g.P; ++lex) cnt[wof(lex) + 1]++;
    for (int w = 0; w < g.nlev; ++w) cnt[w + 1] += cnt[w];
    for (int w = 0; w <= g.nlev; ++w) lptr.push_back(cnt[w]);
    std::vector<int> pb(g.P);
    std::vector<int> fill(cnt.begin(), cnt.end() - 1);
    for (int lex = 0; lex < g.P; ++lex) {
      const int q = fill[wof(lex)]++;
      pb[q] = lex;
    }
    perm.insert(perm.end(), pb.begin(), pb.end());
    f->boxes_h.push_back(g);
    foff += (long long)tb.S * g.P;
    voff += 3LL * g.P;
  }
  f->fcount = foff;
  f->vcount = voff;
  const size_t esz = prec == 64 ? sizeof(double) : sizeof(float);
  auto up = [&](auto** dst, const auto& v) -> kkt_status {
    using E = typename std::remove_reference<decltype(v[0])>::type;
    if (cudaMalloc((void**)dst, std::max<size_t>(1, v.size()) * sizeof(E)) != cudaSuccess) {
      cudaGetLastError();
      set_error("ras_setup: device allocation failed (pattern tables)");
      return KKT_ERR_NOMEM;
    }
    if (!v.empty()) KKT_TRY_CUDA(cudaMemcpy(*dst, v.data(), v.size() * sizeof(E), cudaMemcpyHostToDevice));
    return KKT_OK;
  };
  KKT_TRY(up(&f->boxes, f->boxes_h));
  KKT_TRY(up(&f->perm, perm));
  KKT_TRY(up(&f->lptr, lptr));
  KKT_TRY(up(&f->slot, slot));
  KKT_TRY(up(&f->smap, smap));
  KKT_TRY(up(&f->tptr, tptr));
  KKT_TRY(up(&f->tt, tt));
  KKT_TRY(up(&f->tu, tu));
  if (cudaMalloc(&f->F, std::max<long long>(1, f->fcount) * esz) != cudaSuccess ||
      cudaMalloc(&f->LV, std::max<long long>(1, f->fcount)) != cudaSuccess ||
      cudaMalloc(&f->V, std::max<long long>(1, f->vcount) * esz) != cudaSuccess) {
    cudaGetLastError();
    set_error("ras_setup: device allocation failed (" + std::to_string(f->fcount) + " factor values)");
    return KKT_ERR_NOMEM;
  }
  for (int c = 0; c < 3; ++c)
    if (std::max(tb.diag[c], tb.cnt[c] - tb.diag[c] - 1) > 32 * (local == 3 ? 4 : 14)) {
      set_error("ras_setup: internal error: a pattern row exceeds the solve's steps");
      return KKT_ERR_ARG;
    }
  KKT_TRY((prec == 64 ? (local == 3 ? gp_solve_prepare<double, 4>() : gp_solve_prepare<double, 14>())
                      : (local == 3 ? gp_solve_prepare<float, 4>() : gp_solve_prepare<float, 14>())));
  tb.slot = f->slot;
  tb.smap = f->smap;
  tb.tptr = f->tptr;
  tb.tt = f->tt;
  tb.tu = f->tu;
  return KKT_OK;
}

long long gp_factor_count(const ras_precond* m) { return m->gp ? m->gp->fcount : 0; }
