// ILU(0) factorisation of all subdomain matrices in FP32 (Sec. 3.2), stored in
// FP32 or rounded to BF16, in the lane order of the subdomain solve.
//
// One warp eliminates one point's C, G and f rows; lane d (of 27) holds the
// rows' entries at spatial offset d = (dx+1) + 3 (dy+1) + 9 (dz+1): C row C and
// f columns at levels n-1, n; G row G column at n, n+1; f row G and f columns
// at n-1, n, n+1.  A pivot at spatial offset d1 updates the entry at d from its
// U entry at offset d - d1, so the lanes read consecutive values of the pivot's
// record and no index tables are needed.  The IKJ order is kept: pivots go in
// column order (level, spatial offset, component), and every entry receives its
// updates in that order, one FMA each.  The C and the f row do not depend on
// each other and run side by side, two chains of shuffles at a time.
//
// A pivot record holds what later rows read of a point, two float4 per offset:
//   {G row G(n), G(n+1), f row G(n), G(n+1)} and {f row f(n), f(n+1), C row C(n),
//   f(n)}, level-n entries up to the centre 0 (the C row's own-point f kept), and
//   the reciprocals of the three pivots.
// The pivot's lane forms all its multipliers before they are broadcast.
//
// What bounds it: L1's tag stage, about 16 cycles a pivot whatever the width of the
// loads (27 entries of 32 bytes at any 16-byte offset), besides the shuffles:
// 950 cycles a point and SM, with 8 or 12 warps.  One thread per point, which this
// replaced in FP32, had full lanes but far too few loads under way.  Measured,
// gather included, 32^3 x 64 (256 boxes): 50.7 -> 37.4 ms; 16^3 x 32, overlap 1: 10.3 ->
// 2.5; 64 boxes of 16,800 points: 19.7 -> 5.6; one box of 37,349 points: 24.5 -> 3.2.
// A record is last read 15 wavefronts after it was written, when its place is
// 16 wavefronts from being reused two levels later: two levels of records per
// box in work are enough (2.8 MB for 12^3 points a level).
//
// The matrix entries are formed in registers from the packed coefficients
// (432 bytes a point), so the factors are written once and never read.
#include <algorithm>
#include <type_traits>

#include <cuda_bf16.h>

#include "slotval.cuh"

namespace {

constexpr int kRecA = 0, kRecB = 108, kRecInv = 216, kRec = 220;   // floats
constexpr int kFacWarps = 12;   // one CTA per SM: the records under way take 168 registers
constexpr unsigned kAll27 = 0x7ffffffu;

using K0 = std::integral_constant<int, 0>;
using K1 = std::integral_constant<int, 1>;
using K2 = std::integral_constant<int, 2>;

struct Pivot {
  float4 a, b;   // G row G(n), G(n+1), f row G(n), G(n+1); f row f(n), f(n+1), C row C(n), f(n)
};

// Loads the record entries of pivot K mod 3 of a row (three spatial offsets along
// x) for this lane, where bit K of m (an entry at d - d1 exists) is set.  row:
// record of the row's middle offset, shifted by the lane's place.  CS > 1: other
// SMs write records, so L1 is bypassed.
template <int CS, int K>
__device__ __forceinline__ void load_pivot(Pivot& v, const float* row, unsigned m) {
#define KKT_LOAD_PIVOT(OP)                                                                                          \
  asm volatile(                                                                                                     \
      "{\n .reg .pred p;\n .reg .b32 t;\n and.b32 t, %9, %10;\n setp.ne.b32 p, t, 0;\n @p " OP                     \
      " {%0, %1, %2, %3}, [%8+%11];\n @p " OP " {%4, %5, %6, %7}, [%8+%12];\n}\n"                                   \
      : "=f"(v.a.x), "=f"(v.a.y), "=f"(v.a.z), "=f"(v.a.w), "=f"(v.b.x), "=f"(v.b.y), "=f"(v.b.z), "=f"(v.b.w)      \
      : "l"(row), "r"(m), "n"(1 << K), "n"(kOff + 4 * kRecA), "n"(kOff + 4 * kRecB))
  constexpr int kOff = 4 * ((K % 3 - 1) * kRec + 4 * (kCentre - K % 3));
  if constexpr (CS == 1)
    KKT_LOAD_PIVOT("ld.global.v4.f32");
  else
    KKT_LOAD_PIVOT("ld.global.cg.v4.f32");
#undef KKT_LOAD_PIVOT
}

// The updates by a pivot's rows where bit K of m is set, in column order: C row (C0,
// c0) by the C pivot, c0 (and c1: a pivot at level n-1) by the f pivot; f row (h0, h1) by
// the G and the f pivot, (f0, f1) by the f pivot.
template <int K>
__device__ __forceinline__ void update(float& C0, float& c0, float& c1, float lC, float lc, float& h0, float& h1,
                                       float& f0, float& f1, float lG, float lf, const Pivot& v, unsigned m) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b32 t;\n and.b32 t, %19, %20;\n setp.ne.b32 p, t, 0;\n"
      " @p fma.rn.f32 %0, %7, %17, %0;\n @p fma.rn.f32 %1, %7, %18, %1;\n"
      " @p fma.rn.f32 %3, %9, %11, %3;\n @p fma.rn.f32 %4, %9, %12, %4;\n"
      " @p fma.rn.f32 %5, %10, %15, %5;\n @p fma.rn.f32 %6, %10, %16, %6;\n"
      " @p fma.rn.f32 %1, %8, %15, %1;\n @p fma.rn.f32 %2, %8, %16, %2;\n"
      " @p fma.rn.f32 %3, %10, %13, %3;\n @p fma.rn.f32 %4, %10, %14, %4;\n}\n"
      : "+f"(C0), "+f"(c0), "+f"(c1), "+f"(h0), "+f"(h1), "+f"(f0), "+f"(f1)
      : "f"(-lC), "f"(-lc), "f"(-lG), "f"(-lf), "f"(v.a.x), "f"(v.a.y), "f"(v.a.z), "f"(v.a.w), "f"(v.b.x),
        "f"(v.b.y), "f"(v.b.z), "f"(v.b.w), "r"(m), "n"(1 << K));
}
// the same for a pivot at level n (the C row has no column at n+1), and the G row (g0, g1)
template <int K>
__device__ __forceinline__ void update_n(float& C0, float& c0, float lC, float lc, float& g0, float& g1, float lg,
                                         float& h0, float& h1, float& f0, float& f1, float lG, float lf,
                                         const Pivot& v, unsigned m) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b32 t;\n and.b32 t, %21, %22;\n setp.ne.b32 p, t, 0;\n"
      " @p fma.rn.f32 %0, %8, %19, %0;\n @p fma.rn.f32 %1, %8, %20, %1;\n"
      " @p fma.rn.f32 %4, %11, %13, %4;\n @p fma.rn.f32 %5, %11, %14, %5;\n"
      " @p fma.rn.f32 %2, %10, %13, %2;\n @p fma.rn.f32 %3, %10, %14, %3;\n"
      " @p fma.rn.f32 %6, %12, %17, %6;\n @p fma.rn.f32 %7, %12, %18, %7;\n"
      " @p fma.rn.f32 %1, %9, %17, %1;\n"
      " @p fma.rn.f32 %4, %12, %15, %4;\n @p fma.rn.f32 %5, %12, %16, %5;\n}\n"
      : "+f"(C0), "+f"(c0), "+f"(g0), "+f"(g1), "+f"(h0), "+f"(h1), "+f"(f0), "+f"(f1)
      : "f"(-lC), "f"(-lc), "f"(-lg), "f"(-lG), "f"(-lf), "f"(v.a.x), "f"(v.a.y), "f"(v.a.z), "f"(v.a.w),
        "f"(v.b.x), "f"(v.b.y), "f"(v.b.z), "f"(v.b.w), "r"(m), "n"(1 << K));
}

__device__ __forceinline__ float bcast(float v, int d) { return __shfl_sync(0xffffffffu, v, d); }

__device__ __forceinline__ void check_pivot(float d, int* status) {
  if (!(fabsf(d) > 0.f) || !isfinite(d)) atomicExch(status, 1);
}

// values of the solve's lane layout, streamed past L1
__device__ __forceinline__ void put4(float* p, float a, float b, float c, float d) {
  __stcs(reinterpret_cast<float4*>(p), make_float4(a, b, c, d));
}
__device__ __forceinline__ void put2(float* p, float a, float b) {
  __stcs(reinterpret_cast<float2*>(p), make_float2(a, b));
}
__device__ __forceinline__ void put1(float* p, float a) { __stcs(p, a); }
__device__ __forceinline__ void put4(__nv_bfloat16* p, float a, float b, float c, float d) {
  reinterpret_cast<__nv_bfloat162*>(p)[0] = __floats2bfloat162_rn(a, b);
  reinterpret_cast<__nv_bfloat162*>(p)[1] = __floats2bfloat162_rn(c, d);
}
__device__ __forceinline__ void put2(__nv_bfloat16* p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}
__device__ __forceinline__ void put1(__nv_bfloat16* p, float a) { *p = __float2bfloat16_rn(a); }

template <int CS>
__device__ __forceinline__ void box_sync() {
  if constexpr (CS == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// what a point's elimination needs besides the records; read a point ahead
struct Start {
  int lex;
  float4 coef;          // B, S, S^T, K at the lane's offset
  double sens;          // sensor count
  unsigned char dir;    // Dirichlet node
};

// a / b and a % b for 0 <= a < 2^23 with r = 1 / b
__device__ __forceinline__ int divide(int a, int b, float r, int& rem) {
  int q = __float2int_rd(((float)a + 0.5f) * r);
  rem = a - q * b;
  if (rem < 0) {
    --q;
    rem += b;
  } else if (rem >= b) {
    ++q;
    rem -= b;
  }
  return q;
}

// What the points of a box have in common, in shared memory: in registers it
// would crowd out the pivot records under way.
struct BoxConst {
  int x0, y0, z0, t0, lx, ly, lz, lt, sy, sz, nx, ny, M, reg;
  float rx, ry, rz;                          // 1 / lx, 1 / ly, 1 / lz
  float thtau, th1tau, mt1, mt_side, lt_side, b1, b2;   // (arithmetic of slotval.cuh in FP32)
  const float4* pack;
  const unsigned char* dirn;
  const double* sens;
};

// S: stored type.  CS: CTAs (a cluster) that share a box.  G: points per group.
template <typename S, int CS, int G>
__global__ void __launch_bounds__(32 * kFacWarps, 1) ilu0_factor32(
    const DevProblem* __restrict__ probs, const BoxDesc* __restrict__ boxes, int nbox, const int* __restrict__ gptr,
    const int* __restrict__ perm, S* __restrict__ F, float* __restrict__ recs, long long rec_floats,
    int* __restrict__ status) {
  const int lane = threadIdx.x & 31, d = min(lane, 26);
  const int ncl = gridDim.x / CS, cl = blockIdx.x / CS;
  const int wid = threadIdx.x / 32 * CS + blockIdx.x % CS, nw = kFacWarps * CS;
  float* rec = recs + cl * rec_floats;
  const int dx = d % 3 - 1, dy = d / 3 % 3 - 1, dz = d / 9 - 1;
  unsigned vm = 0;   // pivots d1 with an entry for this lane
  for (int d1 = 0; d1 < 27; ++d1)
    if (lane < 27 && abs(dx - d1 % 3 + 1) <= 1 && abs(dy - d1 / 3 % 3 + 1) <= 1 && abs(dz - d1 / 9 + 1) <= 1)
      vm |= 1u << d1;
  __shared__ BoxConst c;
  for (int b = cl; b < nbox; b += ncl) {
    const BoxDesc& bx = boxes[b];
    if (threadIdx.x == 0) {
      const DevProblem* pp = probs + bx.prob;
      c.x0 = bx.x0; c.y0 = bx.y0; c.z0 = bx.z0; c.t0 = bx.t0;
      c.lx = bx.lx; c.ly = bx.ly; c.lz = bx.lz; c.lt = bx.lt;
      c.sy = kRec * bx.lx;
      c.sz = c.sy * bx.ly;
      c.nx = pp->nx; c.ny = pp->ny; c.M = pp->M; c.reg = pp->reg;
      c.rx = 1.f / bx.lx; c.ry = 1.f / bx.ly; c.rz = 1.f / bx.lz;
      const float tau = (float)pp->tau;
      c.thtau = (float)pp->theta * tau;
      c.th1tau = (float)(1.0 - pp->theta) * tau;
      c.mt1 = tau / 6.f;
      c.mt_side = tau / 3.f;
      c.lt_side = 1.f / tau;
      c.b1 = (float)pp->beta1;
      c.b2 = (float)pp->beta2;
      c.pack = pp->pack32;
      c.dirn = pp->dir;
      c.sens = pp->sens;
    }
    const int nlev = bx.nlev;
    const int* gp = gptr + bx.loff;
    const int* pm = perm + G * bx.goff;
    S* Fb = F + bx.foff;
    __syncthreads();
    auto start = [&](int lex) {
      Start a;
      a.lex = lex;
      if (lex >= 0) {
        int x, y, z;
        divide(divide(divide(lex, c.lx, c.rx, x), c.ly, c.ry, y), c.lz, c.rz, z);
        const int j = c.x0 + x + c.nx * (c.y0 + y + c.ny * (c.z0 + z));
        a.coef = __ldg(c.pack + (size_t)j * kStencil + d);
        a.dir = __ldg(c.dirn + j);
        a.sens = __ldg(c.sens + j);
      }
      return a;
    };
    auto eliminate = [&](const Start& a, int idx) {
      asm volatile("" ::: "memory");   // read the box's constants here, do not keep them
      int x, y, z;
      const int t = divide(divide(divide(a.lex, c.lx, c.rx, x), c.ly, c.ry, y), c.lz, c.rz, z);
      const int n = c.t0 + t, M = c.M, sy = c.sy, sz = c.sz;
      const bool dir = a.dir != 0;
      const float sj = (float)a.sens;
      // pivots in the box
      unsigned bm = kAll27;
      if (x == 0) bm &= ~0x1249249u;
      if (x == c.lx - 1) bm &= ~0x4924924u;
      if (y == 0) bm &= ~0x01c0e07u;
      if (y == c.ly - 1) bm &= ~0x70381c0u;
      if (z == 0) bm &= ~0x00001ffu;
      if (z == c.lz - 1) bm &= ~0x7fc0000u;
      const bool sp = lane < 27 && (bm >> d & 1), tm = t > 0, tp = t + 1 < c.lt;
      const bool idC = n == 0 || dir, idG = n == M || dir;   // identity rows
      const long long slev = (long long)sz * c.lz, at = (long long)z * sz + y * sy + x * kRec;
      float* here = rec + (t & 1) * slev + at;
      const float* prev = rec + (~t & 1) * slev + at;
      // reciprocals of the pivots at the lane's own offset, levels n-1 and n
      float imC = 0, imG = 0, imF = 0, i0C = 0, i0G = 0, i0F = 0;
      const int own = (d % 3 - 1) * kRec + (d / 3 % 3 - 1) * sy + (d / 9 - 1) * sz;
      if (sp && tm) {
        const float4* q = reinterpret_cast<const float4*>(prev + own + kRecInv);
        const float4 v = CS == 1 ? *q : __ldcg(q);
        imC = v.x; imG = v.y; imF = v.z;
      }
      if (sp && d < 13) {
        const float4* q = reinterpret_cast<const float4*>(here + own + kRecInv);
        const float4 v = CS == 1 ? *q : __ldcg(q);
        i0C = v.x; i0G = v.y; i0F = v.z;
      }
      // the rows: C row C, f at levels m (n-1), 0 (n); G row G at 0, p (n+1) and its own-node C; f row G, f at m, 0, p
      const float Bv = a.coef.x, Sv = a.coef.y, STv = a.coef.z, Kv = c.reg ? Bv : a.coef.w;
      const float mt0 = (n > 0 ? c.mt_side : 0.f) + (n < M ? c.mt_side : 0.f);
      const float lt0 = (n > 0 ? c.lt_side : 0.f) + (n < M ? c.lt_side : 0.f);
      const bool centre = d == kCentre;
      const float thtau = c.thtau, th1tau = c.th1tau, mt1 = c.mt1, b1 = c.b1, b2 = c.b2, lt1 = -c.lt_side;
      float C0 = !sp ? 0.f : idC ? (centre ? 1.f : 0.f) : Bv + thtau * Sv;
      float c0 = !sp || idC ? 0.f : -thtau * Bv;
      float Cm = !sp || !tm || idC ? 0.f : -Bv + th1tau * Sv;
      float cm = !sp || !tm || idC ? 0.f : -th1tau * Bv;
      float G0 = !sp ? 0.f : idG ? (centre ? 1.f : 0.f) : Bv + thtau * STv;
      float Gp = !sp || !tp || idG ? 0.f : -Bv + th1tau * STv;
      const float gc0 = idG ? 0.f : th1tau * sj, gcp = !tp || idG ? 0.f : thtau * sj;
      float Hm = !sp || !tm ? 0.f : -mt1 * Bv;
      float fm = !sp || !tm ? 0.f : fmaf(b2 * mt1, Kv, b1 * lt1 * Bv);
      float H0 = !sp ? 0.f : -mt0 * Bv;
      float f0 = !sp ? 0.f : fmaf(b2 * mt0, Kv, b1 * lt0 * Bv);
      float Hp = !sp || !tp ? 0.f : -mt1 * Bv;
      float fp = !sp || !tp ? 0.f : fmaf(b2 * mt1, Kv, b1 * lt1 * Bv);

      // The records are read two rows of three offsets ahead of their use, through both levels
      // (loops, not straight-line code: unrolled, the compiler starts all 160 loads first and
      // spills them).  Bits of the masks: the 27 offsets of level n-1, then the 13 of level n.
      const unsigned m1 = tm ? vm & bm : 0u, m0 = vm & bm & 0x1fffu;
      unsigned mask = m1 | m0 << 27, mhi = m0 >> 5;
      const int next_row = sy - 12, next_plane = sz - 2 * sy - 12;   // to the record row d1 + 3 starts in
      const float* row = prev + 4 * lane - sz - sy;                  // row of the next load
      int loaded = 0;                                                // its number
      auto go_on = [&]() {
        ++loaded;
        row = loaded == 9 ? here + 4 * lane - sz - sy
                          : row + (loaded == 3 || loaded == 6 || loaded == 12 ? next_plane : next_row);
      };
      auto shift = [&]() {
        mask = __funnelshift_r(mask, mhi, 3);
        mhi >>= 3;
      };
      Pivot a0, a1, a2, e0, e1, e2;
      load_pivot<CS, 0>(a0, row, mask);
      load_pivot<CS, 1>(a1, row, mask);
      load_pivot<CS, 2>(a2, row, mask);
      go_on();
      load_pivot<CS, 3>(e0, row, mask);
      load_pivot<CS, 4>(e1, row, mask);
      load_pivot<CS, 5>(e2, row, mask);
      go_on();
      // One pivot of level n-1 and of level n; then its registers take the pivot six further on.
      // Every lane forms the multipliers as if it were the pivot's (in the lane at d1 the record's
      // centre is the pivot's own point), lane d1's are broadcast.
      auto step1 = [&](Pivot& v, int d1, auto kc) {
        constexpr int K = decltype(kc)::value;
        const float tC = Cm * imC, tc = fmaf(-tC, v.b.w, cm) * imF;
        const float lC = bcast(tC, d1), lG = bcast(Hm * imG, d1), lc = bcast(tc, d1), lf = bcast(fm * imF, d1);
        update<K>(Cm, cm, c0, lC, lc, Hm, H0, fm, f0, lG, lf, v, mask);
        load_pivot<CS, K + 6>(v, row, mask);
      };
      auto step0 = [&](Pivot& v, int d1, auto kc) {
        constexpr int K = decltype(kc)::value;
        const float tC = C0 * i0C, tc = fmaf(-tC, v.b.w, c0) * i0F;
        const float lC = bcast(tC, d1), lg = bcast(G0 * i0G, d1), lG = bcast(H0 * i0G, d1), lc = bcast(tc, d1),
                    lf = bcast(f0 * i0F, d1);
        update_n<K>(C0, c0, lC, lc, G0, Gp, lg, H0, Hp, f0, fp, lG, lf, v, mask);
        load_pivot<CS, K + 6>(v, row, mask);   // (no bits left after the last row)
      };
      auto row1 = [&](Pivot& u0, Pivot& u1, Pivot& u2, int d1) {
        step1(u0, d1, K0{});
        step1(u1, d1 + 1, K1{});
        step1(u2, d1 + 2, K2{});
        go_on();
        shift();
      };
      auto row0 = [&](Pivot& u0, Pivot& u1, Pivot& u2, int d1) {
        step0(u0, d1, K0{});
        step0(u1, d1 + 1, K1{});
        step0(u2, d1 + 2, K2{});
        go_on();
        shift();
      };
#pragma unroll 1
      for (int d1 = 0; d1 < 24; d1 += 6) {
        row1(a0, a1, a2, d1);
        row1(e0, e1, e2, d1 + 3);
      }
      row1(a0, a1, a2, 24);
#pragma unroll 1
      for (int d1 = 0; d1 < 12; d1 += 6) {
        row0(e0, e1, e2, d1);
        row0(a0, a1, a2, d1 + 3);
      }
      step0(e0, 12, K0{});
      // the point's own pivots: C scales the G row's C column, G eliminates the f row's G column
      const float pC = bcast(C0, kCentre), iC = 1.f / pC;
      const float pG = bcast(G0, kCentre), iG = 1.f / pG;
      const float lgc = gc0 * iC, lfg = bcast(H0, kCentre) * iG;
      if (d > kCentre) H0 = fmaf(-lfg, G0, H0);
      Hp = fmaf(-lfg, Gp, Hp);
      const float pF = bcast(f0, kCentre), iF = 1.f / pF;
      const float ownf = bcast(c0, kCentre);
      if (lane == 0) {
        check_pivot(pC, status);
        check_pivot(pG, status);
        check_pivot(pF, status);
      }
      const bool up = d > kCentre;
      if (lane < 27) {
        float4* o = reinterpret_cast<float4*>(here) + d;
        o[kRecA / 4] = make_float4(up ? G0 : 0.f, Gp, up ? H0 : 0.f, Hp);
        o[kRecB / 4] = make_float4(up ? f0 : 0.f, fp, up ? C0 : 0.f, d >= kCentre ? c0 : 0.f);
      } else if (lane == 27) {
        *reinterpret_cast<float4*>(here + kRecInv) = make_float4(iC, iG, iF, 0.f);
      }
      // the factors, in the lanes' order (LaneFactors, ras.cu); places formed here, not kept
      int d = lane;
      asm volatile("" : "+r"(d));
      S* g = Fb + (long long)(idx / G) * group_vals(32, G);
      const int pt = idx % G * 4;
      if (lane < 27) {
        put4(g + lane_place<S, G>(false, d & ~3, pt + (d & 3)), Cm * imC, cm * imF, Hm * imG, fm * imF);
        if (d < 13) {
          const int q = 27 + d;
          const float l = G0 * i0G;
          put4(g + lane_place<S, G>(false, q & ~3, pt + (q & 3)), C0 * i0C, c0 * i0F, H0 * i0G, f0 * i0F);
          put1(g + lane_place<S, G>(false, 34 + q / 4, pt + (q & 3)), l);
        } else if (d > 13) {
          const int q = d - 14, l = pt + (q & 3), i = q / 4;
          put2(g + lane_place<S, G>(true, 2 * i, l), H0, f0);
          put1(g + lane_place<S, G>(true, 20 + i, l), G0);
          put2(g + lane_place<S, G>(true, 30 + 2 * i, l), C0, c0);
        }
        const int q = d + 13, l = pt + (q & 3), i = q / 4;
        put2(g + lane_place<S, G>(true, 2 * i, l), Hp, fp);
        put1(g + lane_place<S, G>(true, 20 + i, l), Gp);
      } else if (lane == 27) {
        put1(g + lane_place<S, G>(false, 40, pt), lgc);
        put1(g + lane_place<S, G>(false, 40, pt + 1), lfg);
      } else if (lane == 28) {
        put2(g + lane_place<S, G>(true, 36, pt + 1), iF, iG);
      } else if (lane == 29) {
        put2(g + lane_place<S, G>(true, 36, pt + 2), gcp, 0.f);
      } else if (lane == 30) {
        put2(g + lane_place<S, G>(true, 36, pt + 3), iC, ownf);
      }
    };
    // Loaded ahead of their use: the wavefront pointers two wavefronts, the lexicographic index of
    // a place two points (a wavefront's first two from the start of the one before), the
    // coefficients one point.
    auto gp_at = [&](int w) { return gp[min(w, nlev)]; };
    auto lex_at = [&](int i, int end) { return i < G * end ? pm[i] : -1; };
    int g1 = gp[1], g2 = gp_at(2);
    int idx = G * gp[0] + wid;
    Start next = start(lex_at(idx, g1));
    int lex2 = lex_at(idx + nw, g1);
    for (int w = 0; w < nlev; ++w) {
      const int g3 = gp_at(w + 3), first = G * g1 + wid;
      const int lex3 = lex_at(first, g2), lex4 = lex_at(first + nw, g2);
      for (; idx < G * g1; idx += nw) {
        const Start cur = next;
        next = start(lex2);
        lex2 = lex_at(idx + 2 * nw, g1);
        if (cur.lex >= 0) eliminate(cur, idx);
      }
      idx = first;
      next = start(lex3);
      lex2 = lex4;
      box_sync<CS>();
      g1 = g2;
      g2 = g3;
    }
    __syncthreads();   // the constants are no longer read
  }
}

template <typename S>
const void* kernel_of(int cs, int group) {
  if (group != kGroup) return (const void*)ilu0_factor32<S, 1, narrow_group(32)>;
  return cs == 1   ? (const void*)ilu0_factor32<S, 1, kGroup>
         : cs == 2 ? (const void*)ilu0_factor32<S, 2, kGroup>
         : cs == 4 ? (const void*)ilu0_factor32<S, 4, kGroup>
                   : (const void*)ilu0_factor32<S, 8, kGroup>;
}

cudaLaunchConfig_t config_of(int cs, int ncl, cudaStream_t s, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(cs * ncl);
  c.blockDim = dim3(32 * kFacWarps);
  c.stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim = {(unsigned)cs, 1, 1};
  c.attrs = attr;
  c.numAttrs = 1;
  return c;
}

template <typename S>
kkt_status factor32_launch(ras_precond* m, S* F, cudaStream_t s) {
  cudaLaunchAttribute attr{};
  const cudaLaunchConfig_t cfg = config_of(m->fac_cluster, m->fac_nclusters, s, &attr);
  const DevProblem* probs = m->dprobs;
  const BoxDesc* boxes = m->boxes;
  int nbox = m->nbox;
  const int *gptr = m->gptr, *perm = m->perm;
  float* rec = m->rec;
  long long rf = m->rec_floats;
  int* status = m->status;
  void* args[] = {&probs, &boxes, &nbox, &gptr, &perm, &F, &rec, &rf, &status};
  {
    TimedScope timed(&m->factor_timing, s);
    KKT_TRY_CUDA(cudaLaunchKernelExC(&cfg, kernel_of<S>(m->fac_cluster, m->group), args));
  }
  KKT_COUNT(1);
  return KKT_OK;
}

}  // namespace

kkt_status ras_factor_launch32(ras_precond* m, cudaStream_t s) { return factor32_launch<float>(m, (float*)m->F, s); }

kkt_status ras_factor_launch16(ras_precond* m, cudaStream_t s) {
  return factor32_launch<__nv_bfloat16>(m, (__nv_bfloat16*)m->F, s);
}

// CTAs per box, clusters of the launch (each works through boxes of the list,
// largest first) and the pivot records, at set-up.
kkt_status ras_factor_prepare32(ras_precond* m) {
  long long rec = 0;
  for (const BoxDesc& b : m->boxes_h) rec = std::max(rec, 2LL * kRec * b.lx * b.ly * b.lz);
  m->rec_floats = rec;
  // CTAs per box: as many as have two points a warp in an average wavefront.  Fewer boxes at a
  // time also keep their records in L2 (3 MB each at 12^3 points a level).  Measured, ms with 1, 2,
  // 4, 8 CTAs: 119 points a wavefront, 256 boxes 47.7, 43.6, 37.4, 46.8; 74 points, 64 boxes 9.2, 5.6,
  // 5.8, 8.6; 90 points, 16 boxes 9.3, 5.4, 3.0, 3.5; 175 points, one box 18.9, 10.2, 5.6, 3.2; 20 points,
  // 256 boxes 2.5, 3.4, 5.2, 11.2.
  long long points = 0, waves = 0;
  for (const BoxDesc& b : m->boxes_h) {
    points += b.P;
    waves += b.nlev;
  }
  int cs = 1;
  while (m->group == kGroup && cs < 8 && 2 * cs * 21 * waves <= points) cs *= 2;
  m->fac_cluster = cs;
  cudaLaunchAttribute attr{};
  const cudaLaunchConfig_t cfg = config_of(cs, m->nbox, nullptr, &attr);
  int most = 0;
  KKT_TRY_CUDA(cudaOccupancyMaxActiveClusters(
      &most, m->prec == 16 ? kernel_of<__nv_bfloat16>(cs, m->group) : kernel_of<float>(cs, m->group), &cfg));
  m->fac_nclusters = std::max(1, std::min(most, m->nbox));
  // fewer boxes at a time where their records would take more than a quarter of the free memory, which
  // a problem sized to the memory needs for its Krylov vectors
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess)
    while (m->fac_nclusters > 1 && (size_t)m->fac_nclusters * rec * sizeof(float) > free_b / 4) m->fac_nclusters /= 2;
  for (;; m->fac_nclusters /= 2) {
    if (cudaMalloc(&m->rec, (size_t)m->fac_nclusters * rec * sizeof(float)) == cudaSuccess) return KKT_OK;
    cudaGetLastError();
    m->rec = nullptr;
    if (m->fac_nclusters == 1) {
      set_error("ras_setup: device allocation failed (pivot records)");
      return KKT_ERR_NOMEM;
    }
  }
}
