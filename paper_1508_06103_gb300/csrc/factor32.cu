// Subdomain ILU(0) factorisation in FP32 (the mixed-precision form), and the
// BF16-stored variant: factored in FP32, then rounded to BF16 for the solve.
#include <algorithm>

#include <cuda_bf16.h>

#include "factor.cuh"

namespace {

// Rank (row of a [slot rank][8] group) of value v of lane l of a point, or -1.
__device__ __forceinline__ int lane_rank(bool upper, int v, int l) {
  if (!upper) {
    if (v < 40) {
      const int q = l + 4 * (v / 4), c = v % 4;
      return c < 2 ? 2 * q + c : 94 + 2 * q + c - 2;
    }
    const int q = l + 4 * (v - 34);
    return q >= 27 ? 80 + q - 27 : q == 24 ? 93 : q == 25 ? 174 : -1;
  }
  if (v < 20) return 175 + 71 + 2 * (l + 4 * (v / 2)) + v % 2;
  if (v < 30) {
    const int q = l + 4 * (v - 20), d = q - 13;
    return 175 + (q < 13 ? 29 + q : 42 + d + (d >= 13 ? 1 : 0));
  }
  const int q = l + 4 * ((v - 30) / 2), c = v % 2;
  if (q < 13) return 175 + 2 + 2 * q + c;
  if (q == 13) return 175 + (c == 0 ? 70 : 28);
  if (q == 14) return c == 0 ? 175 + 55 : -1;
  return 175 + c;
}

// groups [slot rank][8] of a -> the lane order of the solve in b (may be a itself), one warp per group
constexpr int kRepackWarps = 4;
template <typename S>
__global__ void __launch_bounds__(32 * kRepackWarps) repack(const BoxDesc* __restrict__ boxes,
                                                            const int* __restrict__ gptr, const float* a, S* b) {
  __shared__ float buf[kRepackWarps][kSlots * kGroup];
  const BoxDesc bx = boxes[blockIdx.y];
  const int lane = threadIdx.x % 32, g = blockIdx.x * kRepackWarps + threadIdx.x / 32;
  if (g >= gptr[bx.loff + bx.nlev]) return;
  float* t = buf[threadIdx.x / 32];
  const long long o = bx.foff + (long long)g * kGroupVals32;
  for (int i = lane; i < kSlots * kGroup; i += 32) t[i] = a[o + i];
  __syncwarp();
  for (int up = 0; up < 2; ++up)
    for (int v = 0; v < (up ? kLaneU : kLaneL); ++v) {
      const int r = lane_rank(up, v, lane % 4);
      b[o + lane_place<S>(up, v, lane)] = (S)(r >= 0 ? t[r * kGroup + lane / 4] : 0.f);
    }
}

template <typename S>
kkt_status repack_launch(ras_precond* m, const float* a, S* b, cudaStream_t s) {
  repack<S><<<dim3((m->max_groups + kRepackWarps - 1) / kRepackWarps, m->nbox), 32 * kRepackWarps, 0, s>>>(
      m->boxes, m->gptr, a, b);
  KKT_COUNT(1);
  KKT_TRY_CUDA(cudaGetLastError());
  return KKT_OK;
}

}  // namespace

kkt_status ras_factor_launch32(ras_precond* m, cudaStream_t s) {
  KKT_TRY(factor_launch<float>(m, (float*)m->F, s));
  return repack_launch<float>(m, (const float*)m->F, (float*)m->F, s);
}

kkt_status ras_factor_launch16(ras_precond* m, cudaStream_t s) {
  KKT_TRY(factor_launch<float>(m, (float*)m->Ffac, s));
  return repack_launch<__nv_bfloat16>(m, (const float*)m->Ffac, (__nv_bfloat16*)m->F, s);
}
