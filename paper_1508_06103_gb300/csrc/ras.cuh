// Internal declarations of the Schwarz preconditioner.
#pragma once

#include "internal.cuh"

// slots per point: C row 2*27*2 = 108, G row 2*(27+1) = 56, f row 3*27*2 = 162
constexpr int kSlots = 326;

// The points of a wavefront are stored in groups of G = 8 (the last one of a
// wavefront may be ragged): one warp of the subdomain solve takes one group.
// Where groups of 8 would be mostly empty (boxes of a few points a wavefront:
// lines, thin plates, a few nodes a side) G is narrow_group: the same kernels
// with some lanes idle, for a half or a quarter of the memory.
// Values per group: FP64 [slot rank][G] blocks; FP32 and BF16 44 lower and 38
// upper values for each of 4 G lanes (ras.cu), 326 slots x G points plus 2 G
// unused places.
constexpr int kGroup = 8;
__host__ __device__ constexpr int narrow_group(int prec) { return prec == 64 ? 2 : 4; }
constexpr int kLaneL = 44, kLaneU = 38;                        // values per lane of a group
__host__ __device__ constexpr int group_vals(int prec, int G) {
  return prec == 64 ? kSlots * G : 4 * G * (kLaneL + kLaneU);
}

// Where the solve's lanes keep their values (FP32 and BF16): place of value v
// of a lane within its group.  A lane's values form 16-byte vectors, vector k
// of the 4 G lanes side by side, so a warp reads up to 512 contiguous bytes at a
// time; the last vector is shorter where the count is no multiple.
template <typename S, int G>
__host__ __device__ __forceinline__ int lane_place(bool upper, int v, int lane) {
  constexpr int W = 16 / (int)sizeof(S), L = 4 * G;
  const int n = upper ? kLaneU : kLaneL, full = n / W * W, base = upper ? L * kLaneL : 0;
  return base + (v < full ? (v / W * L + lane) * W + v % W : full * L + lane * (n - full) + (v - full));
}

struct GpFactor;   // ILU(1) / point-block ILU(0) factors (iluk.cu)

// One subdomain box (extended set, owned set, storage offsets).
struct BoxDesc {
  int x0, y0, z0, t0;          // origin of the extended box (global node / level)
  int lx, ly, lz, lt;          // extended box extents
  int ox0, ox1, oy0, oy1, oz0, oz1, ot0, ot1;   // owned ranges (global, half open)
  int nlev;                    // wavefronts x + 2y + 4z + 8t
  long long P;                 // points of the extended box
  long long foff;              // offset of the box's factor groups (elements)
  long long unit;              // offset of the box's unit row within its factor values (elements)
  long long voff;              // offset of the box's padded local vector (elements)
  long long poff;              // offset into the per-point tables (lexicographic)
  long long goff;              // first group of the box
  long long loff;              // offset into the wavefront pointers
  int nown;                    // owned points
  long long ooff;              // offset into the owned-point table
  int kl;                      // exact LU: half-bandwidth of the box matrix
  int prob;                    // problem of the box (a preconditioner over several problems)
  long long aoff;              // exact LU: offset of the box's band (elements)
};

// exact LU: largest half-bandwidth and box size (the solve keeps a box's
// vector in shared memory)
constexpr int kMaxLuBand = 2048;
constexpr int kMaxLuUnknowns = 28672;

struct ras_precond {
  unsigned long long uid = next_handle_uid();
  kkt_problem* prob = nullptr;           // the (first) problem
  // problems of the boxes: one, or several solved together (ras_setup_batch); their
  // unknowns are concatenated in that order, problem k from vec_off[k]
  std::vector<kkt_problem*> probs;
  std::vector<long long> vec_off;        // nprob + 1 offsets
  long long n_total = 0;
  DevProblem* dprobs = nullptr;          // device copies of the problems' DevProblem
  std::vector<DevProblem> dprobs_h;
  int prec = 64;               // factor storage: 64, 32, or 16 (BF16; factorisation and solve in FP32)
  int nbox = 0;
  int ch = 0;                  // size class of the solve's CTA (ras_setup_shape)
  int warps = 0;               // warps of that CTA
  bool smem_vec = false;       // solve keeps the local vectors in shared memory
  int nstage = 2;              // factor groups a warp holds, the one in use included (ras_setup_shape)
  int nbuf = 1;                // buffers a warp has for them: one less, fewer where they do not fit
  int gptr_bytes = 0;          // wavefront pointers in the solve's shared memory (0: read from global memory)
  int lanes = 4;               // lanes per point in the solve
  int group = kGroup;          // points per group
  int cluster = 1;             // CTAs per box of the solve
  bool ring = false;           // solve keeps the last wavefronts in shared memory
  int wcap = 0;                // group places of the widest wavefront
  int max_nlev = 0;            // most wavefronts of a box
  long long ngroup = 0;        // groups of all boxes
  int max_groups = 0;          // most groups of a box
  long long fcount = 0;        // factor values
  long long max_pad = 0;       // largest padded local vector (elements)
  long long vcount = 0;        // elements of all padded local vectors (the solve's scratch)
  std::vector<BoxDesc> boxes_h;
  BoxDesc* boxes = nullptr;
  int* perm = nullptr;         // per group place: lexicographic local index, -1 in a ragged group's empty places
  int* gptr = nullptr;         // first group of each wavefront per box (nlev + 1 each)
  int2* gtab = nullptr;        // per point (lexicographic): {3 x global point index, padded offset}
  int2* otab = nullptr;        // per owned point: {3 x global point index, padded offset}
  int* vtab = nullptr;         // per group place: padded offset in the box's local vector; empty places hold
                               // the complement of an offset that can be read
  unsigned short* ntab = nullptr;   // ring: place of every neighbour per group, sweep and lane
  int* ptab = nullptr;         // per point (lexicographic): offset of its column in the box's factor values
  void* F = nullptr;           // factor values (FP64, FP32 or BF16, as the solve reads them)
  void* V = nullptr;           // padded local vectors
  int* status = nullptr;
  float* rec = nullptr;        // FP32 factorisation: pivot records of the boxes in work
  long long rec_floats = 0;    // per cluster
  int fac_cluster = 1;         // FP32 factorisation: CTAs per box, clusters of the launch
  int fac_nclusters = 0;
  int local = 0;               // 0: ILU(0) local solves, 1: exact banded LU (FP64)
  double* AB = nullptr;        // exact LU: band factors of all boxes
  long long ab_count = 0;
  int* ipiv = nullptr;         // exact LU: row interchanges (3 per box point)
  int* lu_ju = nullptr;        // exact LU: per box, last column reached by fill (two slots)
  int lu_ctas = 1;             // exact LU: CTAs per box in an elimination step
  TimingLog timing;            // subdomain-solve launches
  TimingLog factor_timing;     // ILU(0) factorisation launches
  BatchWork* bw = nullptr;     // gmres_solve_batch workspace (several problems)
  GpFactor* gp = nullptr;      // local 2 (ILU(1)) or 3 (point-block ILU(0))
};

// shape: NULL, or {size class, groups held, lanes per point, vector placement
// (1 shared, 2 global)} of the subdomain solve, 0 = chosen automatically.
// Several problems: every problem is split by nsub and all boxes form one list,
// largest first (so the CTAs of a launch finish together as far as they can).
kkt_status ras_create(kkt_problem* const* probs, int nprob, const int nsub[4], int overlap, int local,
                      int factor_prec, const int* shape, ras_precond** out);
// iluk.cu: the pattern-driven local solvers (local 2 and 3)
kkt_status gp_create(ras_precond* m, int local, int prec);
kkt_status gp_factor(ras_precond* m, cudaStream_t s);
kkt_status gp_solve(ras_precond* m, const double* r, double* z, cudaStream_t s, const int* gate);
void gp_destroy(ras_precond* m);
long long gp_factor_count(const ras_precond* m);
kkt_status ras_factor(ras_precond* m, cudaStream_t s);          // enqueue, synchronise, check
kkt_status ras_factor_enqueue(ras_precond* m, cudaStream_t s);  // enqueue only
kkt_status ras_factor_status(ras_precond* m);                   // after the stream completed
// gather and ILU(0) launches of factor32.cu / factor64.cu
kkt_status ras_factor_launch32(ras_precond* m, cudaStream_t s);
kkt_status ras_factor_launch64(ras_precond* m, cudaStream_t s);
kkt_status ras_factor_launch64_narrow(ras_precond* m, cudaStream_t s);   // groups of narrow_group points
kkt_status ras_factor_launch16(ras_precond* m, cudaStream_t s);   // FP32 factorisation, BF16 store
kkt_status ras_factor_prepare32(ras_precond* m);                  // launch shape and records of the two above
// exact banded LU (lu.cu)
kkt_status ras_lu_factor(ras_precond* m, cudaStream_t s);
kkt_status ras_lu_solve(ras_precond* m, const double* r, double* z, cudaStream_t s, const int* gate);
// the subdomain solve z = M^{-1} r on s; its kernel returns at once while *gate reads 0
// gate_stride: distance (ints) between the gates of consecutive problems; box b
// reads gate[prob(b) * gate_stride]
// z = M^{-1} r + add (where given); z32 (where given) also gets z rounded to FP32 (exact without add
// where the solve runs in FP32)
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s: copies and wavefronts take microseconds
struct RasExtra {
  const double* add = nullptr;
  float* z32 = nullptr;
  // ras_selftest_solve: makes waits of one CTA of every box run out (RasHold), after limit_ns there
  unsigned long long limit_ns = kWaitLimitNs;
  int hold = 0, hold_cta = 0;
  int* drained = nullptr;   // sum of the 1-based numbers of the groups whose copies were waited for on leaving
};
enum RasHold : int { kHoldNone = 0, kHoldCounter = 1, kHoldCopies = 2 };
kkt_status ras_launch(ras_precond* m, const double* r, double* z, cudaStream_t s, const int* gate = nullptr,
                      int gate_stride = 0, const RasExtra& extra = RasExtra());
kkt_status ras_check(ras_precond* m);
