// mf_root.cuh -- building blocks shared by the evaluators (mf_eval.cu) and the
// vertex-grouped root solve (mf_roots.cu).
#pragma once
#include "mf_internal.cuh"

#define FULL 0xffffffffu

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Dimension of the work: a compile-time D below MF_MAXD is exact; D ==
// MF_MAXD serves every d <= MF_MAXD at run time.
template <int D>
__device__ __forceinline__ int dim_of(int rt) {
  return D < MF_MAXD ? D : rt;
}

// Support vector j's row for the root path, in one gather: the hi/lo
// coordinate pairs c[2k], c[2k + 1] (k < D) and, below 8 coordinates, alpha
// and the strong threshold from the row's padding (else from their arrays).
template <int D>
__device__ __forceinline__ void sv_row(const MfRbfDev &R, int j, float *c, float &al, float &s32) {
  constexpr int Q = D < 8 ? (2 * D + 2 + 3) / 4 : 4;
  const float4 *row = reinterpret_cast<const float4 *>(R.svhl + (int64_t)j * 16);
  float v[4 * Q];
#pragma unroll
  for (int q = 0; q < Q; q++) {
    const float4 t = __ldg(row + q);
    v[4 * q] = t.x;
    v[4 * q + 1] = t.y;
    v[4 * q + 2] = t.z;
    v[4 * q + 3] = t.w;
  }
#pragma unroll
  for (int k = 0; k < 2 * D && k < 4 * Q; k++) c[k] = v[k];
  if (D < 8) {
    al = v[D < 8 ? 2 * D : 0];
    s32 = v[D < 8 ? 2 * D + 1 : 0];
  } else {
    al = R.alpha32[j];
    s32 = R.strong32[j];
  }
}

// The root's FP64 step evaluates in FP64 only the terms that can exceed
// ROOT_TAU = 1e-8 (strong32 shifted by ln(ROOT_TAU / STRONG_TAU)); the band
// between STRONG_TAU and ROOT_TAU ("mid") joins the FP32 stage's list and is
// summed in FP32 with the weak terms in the FP64 step.
#define ROOT_TAU 1e-8f
#define ROOT_TAU_SHIFT 3.5065579f
// The mixed paths need |dt| <= 1e-6 only: their FP64 step takes the terms
// that can exceed 1e-5 (shift ln(1e-5 / STRONG_TAU)); the FP32 part may then
// move t by up to 1e-7 and the accepted Newton step leaves < 1e-7.
#define ROOT_TAU_FAST 1e-5f
#define ROOT_TAU_SHIFT_FAST 10.414313f

// Relative error bound of a cached weak term on an edge with |dir|^2 = dd32
// (every kept vector lies within sqrt(rs2) of a point of the segment;
// 1.1 covers this bound's own FP32 rounding).
__device__ __forceinline__ float root_rel_cached(const MfRbfDev &R, int d, float dd32, float rs2) {
  const float q = sqrtf(rs2) + 2.f * sqrtf(dd32);
  return 1.1f * ((float)d + 8.f) * 5.9604644775390625e-08f * (float)R.gamma * q * q +
         9.5367431640625e-07f + 2.f * 5.9604644775390625e-08f;
}

// The FP32 part of a root evaluation (mid and weak terms) errs by at most
// weak_rel * sum|terms|; with the dropped terms (drop_bound) that must stay
// below 1e-10 |g'| (t then moves by at most 1e-10), or below the vertex
// evaluation's own limit, whichever is larger.  Otherwise the point is
// evaluated again with every kept term in FP64.
// (The check runs in FP32: the 1.01 factor covers its roundings.)
__device__ __forceinline__ bool root_fp32_part_too_coarse(const MfRbfDev &R, float weak, float gp,
                                                          bool fast) {
  const float lim = fmaxf(R.weak_limit32, (fast ? 0.99e-7f : 0.99e-10f) * fabsf(gp) -
                                              (fast ? R.drop_bound32_fast : R.drop_bound32));
  return weak * (1.01f * R.weak_rel32) > lim;
}

// A root step handed to the lane-per-edge FP64 kernels (k_roots_terms,
// k_roots_finish): the edge (~0: none), the FP32 stage's t (where the FP64
// evaluation happens), the reused g' there and |g''|, the FP32 part of g at
// t (mid and weak terms, already checked against its error bound), and its
// strong entries: ns of them, in the 8-entry chunks from chunk ch on (records
// of the grouped stage carry [f(x1) >= 0] in ns's bit 31, and g'' signed).
struct __align__(16) RootRec {
  unsigned long long e;
  float t, gp, gpp, wf;
  uint32_t ch, ns;
};
#define DEFER_CHUNK 8

// The vertex-grouped FP32 stage of edges [e0, e0 + n) (mf_roots.cu): writes
// one record per edge with a list (B.cnt->n_defer of them) and queues the
// other edges in B.redo.
void mf_launch_roots_grouped(const MfFrame &F, const MfRbfDev &R, const MfTraceBufs &B, uint64_t e0,
                             uint64_t n, bool fast, int sms, cudaStream_t st);
