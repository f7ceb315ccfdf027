// mf_roots.cu -- the FP32 stage of the root solve (the "iterative algorithm"
// of Sec. VI), grouped by base vertex.
//
// The edges that leave one lattice vertex x1 see the same support vectors (the
// vertex's root-screen list) from the same point: u = x1 - s and |u|^2 are the
// same for all of them, only the direction differs.  So a warp takes one
// vertex at a time: it gathers the list's rows once and keeps u, -g2 |u|^2 and
// alpha in shared memory (g2 = gamma log2 e), then solves the vertex's edges,
// 32 / W of them at once with W lanes each.  Per edge and listed vector,
// Q = -2 g2 u . dir; at x(t) = x1 + t dir the exponent is
// P + t (Q - t g2 |dir|^2), so a Halley evaluation costs eight FP32 operations
// per term from registers, and its derivatives follow from the moments of Q.
// (A warp per edge screened the list anew for every edge, two gathered passes
// over it with most lanes idle after the screen.)  The chunk's edges are first
// bucketed by base vertex.  This stage and the redo on the d = 5 FP64 proof at
// lambda = 0.15 (1.32M edges, 0.24M vertices): 5.2 -> 3.2 ms; at lambda = 0.08
// (7.2M edges, 1.2M vertices): 28.1 -> 11.7 ms; d = 6 BF16: 2.9 -> 1.7 ms.
//
// What it hands over is one RootRec per edge: the converged FP32 t, g' and g''
// there, the FP32 sum of the terms below ROOT_TAU at t (checked against its
// error bound) and the list of the terms above it, which k_roots_terms sums in
// double-float and k_roots_finish turns into the final Newton step.  Edges it
// cannot settle (no list, cancellation in g', too coarse an FP32 part, full
// pools) go to the redo queue and are solved in full by the warp-per-edge
// kernel.
#include <algorithm>

#include "mf_root.cuh"

#define RG_WARPS 8
// Longest list of the three kernels.  Lists are as long as the screen's reach
// makes them (64 to 250 vectors on the 3- to 6-dimensional problems); each
// kernel holds a lane's share of the list in registers, so a shorter limit
// leaves room for more warps: 3 blocks per SM up to RG_SMALL, 2 up to RG_MID.
#define RG_SMALL 192
#define RG_MID 320
#define RG_BIG 512

// Scratch of one chunk, in the rows of the per-edge path that this one leaves
// unused (MfTraceBufs.ep32, at least 48 bytes per edge).
struct RgEdge {
  uint32_t vi, rank;  // base vertex (list index; ~0: none), place among its edges
};
struct __align__(16) RgItem {
  uint32_t e, mask;  // edge - e0; mask, bit 31: f(x1) >= 0
  float f0, f1;
};
struct RgGroup {
  uint32_t vi, off, n;
};
struct RgScratch {
  RgItem *item;
  RgGroup *group;  // short lists from the front, the longest from the back
  RgGroup *mid;
  RgEdge *edge;
};
__device__ __forceinline__ RgScratch rg_scratch(const MfTraceBufs &B) {
  RgScratch s;
  s.item = reinterpret_cast<RgItem *>(B.ep32);
  s.edge = reinterpret_cast<RgEdge *>(s.item + B.defer_cap);
  s.group = reinterpret_cast<RgGroup *>(s.edge + B.defer_cap);
  s.mid = s.group + B.defer_cap;
  return s;
}

__device__ __forceinline__ void rg_redo(const MfTraceBufs &B, uint64_t e) {
  const unsigned long long q = atomicAdd(&B.cnt->n_redo, 1ull);
  if (q < B.defer_cap) B.redo[q] = e;
}

// Edge -> base vertex, and its place among the vertex's edges of the chunk.
__global__ void __launch_bounds__(256) k_rg_count(MfFrame F, MfTraceBufs B, uint64_t e0, uint64_t n) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t e = e0 + i;
  int32_t y[MF_MAXD];
#pragma unroll
  for (int k = 0; k < MF_MAXD; k++) y[k] = k < F.d ? B.edge_y[e * F.d + k] : 0;
  const uint64_t slot = mf_table_find<2>(B.vtab_key, B.vtab_mask, mf_vertex_key(F, y));
  RgEdge g = {~0u, 0u};
  if (slot != ~0ull) {
    const uint32_t vi = B.vtab_idx[slot];
    const uint32_t nl = B.vlist_n[vi];
    if (nl != MF_NO_LIST && nl <= RG_BIG) {
      g.vi = vi;
      g.rank = atomicAdd(&B.vert_edges[vi], 1u);
    }
  }
  if (g.vi == ~0u) rg_redo(B, e);
  rg_scratch(B).edge[i] = g;
}

// A range of items for every vertex that has edges in the chunk (the ranges'
// order is of no matter), and its group.
__global__ void __launch_bounds__(256) k_rg_groups(MfTraceBufs B) {
  const RgScratch sc = rg_scratch(B);
  unsigned long long nv = B.cnt->n_vertices;
  if (nv > B.max_vertices) nv = B.max_vertices;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t v0 = blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); v0 < nv; v0 += stride) {
    const uint64_t v = v0 + lane;
    const uint32_t c = v < nv ? B.vert_edges[v] : 0u;
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    const uint32_t total = __shfl_sync(FULL, inc, 31);
    if (total == 0) continue;
    const uint32_t nl = c ? B.vlist_n[v] : 0u;
    const bool big = c && nl > RG_MID, mid = c && !big && nl > RG_SMALL, small = c && !big && !mid;
    const unsigned ms = __ballot_sync(FULL, small), mm = __ballot_sync(FULL, mid),
                   mb = __ballot_sync(FULL, big);
    unsigned long long base = 0, gs = 0, gm = 0, gb = 0;
    if (lane == 0) {
      base = atomicAdd(&B.cnt->n_defer, (unsigned long long)total);
      if (ms) gs = atomicAdd(&B.cnt->n_groups[0], (unsigned long long)__popc(ms));
      if (mm) gm = atomicAdd(&B.cnt->n_groups[1], (unsigned long long)__popc(mm));
      if (mb) gb = atomicAdd(&B.cnt->n_groups[2], (unsigned long long)__popc(mb));
    }
    base = __shfl_sync(FULL, base, 0);
    gs = __shfl_sync(FULL, gs, 0);
    gm = __shfl_sync(FULL, gm, 0);
    gb = __shfl_sync(FULL, gb, 0);
    if (c) {
      const uint32_t off = (uint32_t)base + inc - c;
      B.vert_edges[v] = off;
      RgGroup *at = small ? sc.group + gs + __popc(ms & lt)
                          : (mid ? sc.mid + gm + __popc(mm & lt)
                                 : sc.group + (B.defer_cap - 1 - (gb + __popc(mb & lt))));
      *at = {(uint32_t)v, off, c};
    }
  }
}

// Edges into their vertex's range, with what the solve needs of them.
__global__ void __launch_bounds__(256) k_rg_scatter(MfTraceBufs B, uint64_t e0, uint64_t n) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const RgScratch sc = rg_scratch(B);
  const RgEdge g = sc.edge[i];
  if (g.vi == ~0u) return;
  const double2 f = reinterpret_cast<const double2 *>(B.edge_f)[e0 + i];
  RgItem it;
  it.e = (uint32_t)i;
  it.mask = (B.edge_mask[e0 + i] & ((1u << MF_MAXD) - 1u)) | (f.x >= 0.0 ? 0x80000000u : 0u);
  it.f0 = (float)f.x;
  it.f1 = (float)f.y;
  sc.item[B.vert_edges[g.vi] + g.rank] = it;
}

// Sums of four values over each run of W lanes, every lane receiving all
// four: the lanes first split the values between halves, then quarters,
// before the plain butterfly.
template <int W>
__device__ __forceinline__ void sub_sum4(float &a, float &b, float &c, float &e) {
  const int lane = threadIdx.x & 31;
  const bool up = lane & (W / 2), odd = lane & (W / 4);
  const float r0 = __shfl_xor_sync(FULL, up ? a : c, W / 2);
  const float r1 = __shfl_xor_sync(FULL, up ? b : e, W / 2);
  const float x = (up ? c : a) + r0, y = (up ? e : b) + r1;
  float z = (odd ? y : x) + __shfl_xor_sync(FULL, odd ? x : y, W / 4);
#pragma unroll
  for (int o = W / 8; o; o >>= 1) z += __shfl_xor_sync(FULL, z, o);
  a = __shfl_sync(FULL, z, 0, W);
  b = __shfl_sync(FULL, z, W / 4, W);
  c = __shfl_sync(FULL, z, W / 2, W);
  e = __shfl_sync(FULL, z, 3 * W / 4, W);
}

// Per warp: u, P and alpha of the list (CAP entries each, D + 2 arrays), padded
// with zeros to the W K entries that the lanes hold.
struct RgCtx {
  const MfRbfDev &R;
  const MfTraceBufs &B;
  const float *lst;   // [D + 2][CAP] u_0 .. u_{D-1}, P = -g2 |u|^2, alpha
  const float *dirt;  // [2^d][D + 1] dir of each mask, |dir|^2
  const int32_t *src;
  int nl;
  uint64_t e0;
  const float *grad;  // sum over the list of alpha e^(-gamma |u|^2) u, at x1
  float g2, gm, b32, thr;
  bool fast;
};

// The edges of one vertex: items [off, off + n), 32 / W at a time, W lanes
// each holding K entries of the list, zeros past its end.
template <int D, int W, int K, int CAP>
__device__ __forceinline__ void rg_solve(const RgCtx &c, uint32_t off, uint32_t n,
                                         uint32_t &nterms) {
  constexpr int NSUB = 32 / W;
  const int lane = threadIdx.x & 31, sl = lane & (W - 1), q = lane / W;
  const RgScratch sc = rg_scratch(c.B);
  const float *lst = c.lst + sl;
  float P[K], al[K];
#pragma unroll
  for (int k = 0; k < K; k++) {
    P[k] = lst[D * CAP + k * W];
    al[k] = lst[(D + 1) * CAP + k * W];
  }
  for (uint32_t i0 = 0; i0 < n; i0 += NSUB) {
    const bool have = i0 + q < n;
    const uint32_t rec_at = off + (have ? i0 + q : i0);
    const RgItem it = sc.item[rec_at];
    const bool s1 = (it.mask >> 31) != 0;
    const float *dr = c.dirt + (it.mask & ((1u << MF_MAXD) - 1u)) * (D + 1);
    const float dd = dr[D], gdd = -c.g2 * dd;
    float Q[K];
#pragma unroll
    for (int k = 0; k < K; k++) {
      float bp = 0.f;
#pragma unroll
      for (int a = 0; a < D; a++) bp = fmaf(lst[a * CAP + k * W], dr[a], bp);
      Q[k] = -2.f * c.g2 * bp;
    }
    // with e = alpha 2^(P + t (Q + t gdd)) and m_i = sum e Q^i:
    //   sum e (u + t dir).dir = -m1 / (2 g2) + t |dir|^2 m0, and so on
    const float iq = -0.5f / c.g2;
    // FP32 Halley iteration (cubic: the evaluation yields g'' anyway),
    // bracketed, from the parabola through the end values with the slope that
    // the vertex's gradient gives at t = 0 (one evaluation per vertex, which
    // saves one of two per edge on a lattice fine enough: d = 5 at lambda =
    // 0.08 13.4 -> 11.7 ms, at 0.15 as before); else the linear interpolant
    float g0 = 0.f;
#pragma unroll
    for (int a = 0; a < D; a++) g0 = fmaf(dr[a], c.grad[a], g0);
    g0 *= -2.f * c.gm;
    const float q2 = (it.f1 - it.f0) - g0;
    const float r2 = g0 + copysignf(sqrtf(fmaxf(fmaf(g0, g0, -4.f * q2 * it.f0), 0.f)), g0);
    float t32 = __fdividef(-2.f * it.f0, r2);
    if (!(t32 > 0.f && t32 < 1.f)) t32 = __fdividef(-0.5f * r2, q2);
    if (!(t32 > 0.f && t32 < 1.f)) t32 = it.f0 / (it.f0 - it.f1);
    if (!(t32 > 0.f && t32 < 1.f)) t32 = 0.5f;
    float lo = 0.f, hi = 1.f, gpp = INFINITY;
    bool done = false;
    if (have && sl == 0) nterms += c.nl;  // the last evaluation
    for (int step_no = 0; step_no < 12; step_no++) {
      float m0 = 0.f, m1 = 0.f, m2 = 0.f, none = 0.f;
#pragma unroll
      for (int k = 0; k < K; k++) {
        const float e = al[k] * ex2_approx(fmaf(t32, fmaf(t32, gdd, Q[k]), P[k]));
        const float eq = e * Q[k];
        m0 += e;
        m1 += eq;
        m2 = fmaf(eq, Q[k], m2);
      }
      if (have && sl == 0 && !done) nterms += c.nl;
      sub_sum4<W>(m0, m1, m2, none);
      if (!done) {
        const float td = t32 * dd;
        const float sp = fmaf(td, m0, iq * m1);                               // sum e proj
        const float sq = fmaf(td, fmaf(td, m0, 2.f * iq * m1), iq * iq * m2);  // sum e proj^2
        const float g = m0 + c.b32, gp = -2.f * c.gm * sp;
        gpp = 4.f * c.gm * c.gm * sq - 2.f * c.gm * dd * m0;
        if ((g >= 0.f) == s1) lo = t32; else hi = t32;
        const float den = 2.f * gp * gp - g * gpp;
        const bool halley = den > 0.f;
        float tn = halley ? t32 - 2.f * g * gp / den : t32 - g / gp;
        const bool inside = tn > lo && tn < hi;
        if (!inside) tn = 0.5f * (lo + hi);
        const float step = fabsf(tn - t32);
        t32 = tn;
        // a Halley step of size s leaves an error of order s^3: below 4e-3
        // the FP32 noise floor (about 1e-6) is reached, and the last step
        // finishes
        done = step <= 2e-6f || (halley && inside && step <= 4e-3f);
      }
      if (__all_sync(FULL, done)) break;
    }
    // the terms at t: those that can exceed ROOT_TAU (with a margin of
    // e^-1/2, far above the FP32 error) to the strong list, the rest summed;
    // and g' there (m0 is -b up to the FP32 noise), trusted where its sum had
    // at most 4x cancellation: then good to ~1e-5, and a step of at most 1e-5
    // errs by far less than 1e-9 from it
    float wf = 0.f, wa = 0.f, m1 = 0.f, m1a = 0.f;
    unsigned strong = 0;  // bit k: entry k of this lane
#pragma unroll
    for (int k = 0; k < K; k++) {
      const float e = al[k] * ex2_approx(fmaf(t32, fmaf(t32, gdd, Q[k]), P[k])), ae = fabsf(e);
      const float eq = e * Q[k];
      const bool s = ae > c.thr;
      strong |= s ? 1u << k : 0u;
      wf += s ? 0.f : e;
      wa += s ? 0.f : ae;
      m1 += eq;
      m1a += fabsf(eq);
    }
    sub_sum4<W>(wf, wa, m1, m1a);
    const float gpf = -2.f * c.gm * fmaf(-t32 * dd, c.b32, iq * m1);
    const bool reuse = 2.f * c.gm * fabsf(iq) * m1a <= 4.f * fabsf(gpf) && gpf != 0.f && isfinite(gpf);
    const float kc =
        fmaxf(root_rel_cached(c.R, D < MF_MAXD ? D : c.R.d, dd, c.B.list_r2) / c.R.weak_rel32, 1.f);
    const bool ok = have && reuse && !root_fp32_part_too_coarse(c.R, wa * kc, gpf, c.fast);
    // places of the lanes' strong entries in the edge's list, lane by lane (a
    // ballot per entry took as many instructions as a Halley evaluation, in a
    // kernel whose first stall is the instruction fetch: 18.1 -> 13.4 ms for
    // the 7.2M edges of a d = 5 proof at lambda = 0.08)
    int at = __popc(strong);
    int ns = at;
#pragma unroll
    for (int o = 1; o < W; o <<= 1) {
      const int v = __shfl_up_sync(FULL, ns, o, W);
      if (sl >= o) ns += v;
    }
    at = ns - at;
    ns = __shfl_sync(FULL, ns, W - 1, W);
    // chunks of the strong list: one allocation for the edges of the round
    const uint32_t nch = ok ? (uint32_t)(ns + DEFER_CHUNK - 1) / DEFER_CHUNK : 0u;
    uint32_t my = 0, all = 0;
#pragma unroll
    for (int s = 0; s < NSUB; s++) {
      const uint32_t v = __shfl_sync(FULL, nch, s * W);
      if (s < q) my += v;
      all += v;
    }
    unsigned long long lat = 0;
    if (all) {
      if (lane == 0)
        lat = atomicAdd(&c.B.cnt->n_defer_list, (unsigned long long)all * DEFER_CHUNK);
      lat = __shfl_sync(FULL, lat, 0);
    }
    const uint64_t c0 = lat / DEFER_CHUNK + my, ncap = c.B.defer_list_cap / DEFER_CHUNK;
    const bool fits = c0 + nch <= ncap;
    if (ok)
      for (uint32_t h = sl; h < nch && c0 + h < ncap; h += W)
        c.B.defer_chunk[c0 + h] = fits ? rec_at : ~0u;
    const bool put = ok && fits;
    if (put) {
      int32_t *to = c.B.defer_list + c0 * DEFER_CHUNK;
      for (unsigned m = strong; m; m &= m - 1) to[at++] = c.src[(__ffs(m) - 1) * W + sl];
      for (uint32_t h = ns + sl; h < nch * DEFER_CHUNK; h += W) to[h] = -1;
    }
    if (have && sl == 0) {
      RootRec r;
      r.e = put ? c.e0 + it.e : ~0ull;
      r.t = t32;
      r.gp = gpf;
      r.gpp = gpp;
      r.wf = wf;
      r.ch = (uint32_t)c0;
      r.ns = (uint32_t)ns | (s1 ? 0x80000000u : 0u);
      reinterpret_cast<RootRec *>(c.B.defer_rec)[rec_at] = r;
      if (!put) rg_redo(c.B, c.e0 + it.e);
    }
  }
}

// Warp per group of size class CLS (0: lists up to RG_SMALL, 1: up to RG_MID,
// 2: up to RG_BIG).  Lanes per edge: fewer lanes share the sums' shuffles and
// the scalar steps between more edges, more lanes hold longer lists.
template <int CLS>
struct RgClass {
  static constexpr int CAP = CLS == 0 ? RG_SMALL : CLS == 1 ? RG_MID : RG_BIG;
  static constexpr int BLOCKS = CLS == 0 ? 3 : CLS == 1 ? 2 : 1;
};
template <int D, int CLS>
__global__ void __launch_bounds__(RG_WARPS * 32, RgClass<CLS>::BLOCKS) k_rg_solve(
    MfFrame F, MfRbfDev R, MfTraceBufs B, uint64_t e0, int fast) {
  extern __shared__ float rg_sh[];
  constexpr int CAP = RgClass<CLS>::CAP;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int d = dim_of<D>(F.d);
  float *dirt = rg_sh;                                      // [2^d][D + 1]
  float *lst = rg_sh + (1 << d) * (D + 1) + w * (D + 2) * CAP;  // [D + 2][CAP]
  // dir = lam (e(S) - c |S|) of every mask
  for (int m = threadIdx.x; m < (1 << d); m += blockDim.x) {
    const double cs = F.c * (double)__popc(m);
    float dd = 0.f;
    for (int k = 0; k < D; k++) {
      const float v = k < d ? (float)(F.lam * ((double)((m >> k) & 1) - cs)) : 0.f;
      dirt[m * (D + 1) + k] = v;
      dd = fmaf(v, v, dd);
    }
    dirt[m * (D + 1) + D] = dd;
  }
  __syncthreads();
  const RgScratch sc = rg_scratch(B);
  const uint64_t ng = B.cnt->n_groups[CLS];
  const uint64_t nwarps = (uint64_t)gridDim.x * RG_WARPS;
  // the lane's FP32 terms: at most 13 evaluations of 512 for each edge of the
  // warp's share of a chunk, far below 2^32
  uint32_t nterms = 0;
  for (uint64_t g = blockIdx.x * (uint64_t)RG_WARPS + w; g < ng; g += nwarps) {
    const RgGroup gr = CLS == 0 ? sc.group[g] : CLS == 1 ? sc.mid[g] : sc.group[B.defer_cap - 1 - g];
    const int nl = (int)B.vlist_n[gr.vi];
    const int32_t *src = B.vlist + B.vlist_off[gr.vi];
    // x1 (FP32 hi/lo): lane k < d computes axis k in mf_vertex_x's order
    float hi = 0.f, lo = 0.f;
    {
      const int ko = lane < d ? lane : 0;
      long long sy = 0;
      int32_t yo = 0;
#pragma unroll
      for (int k = 0; k < D; k++) {
        if (k < d) {
          const int32_t v = B.vert_y[(uint64_t)gr.vi * d + k];
          sy += v;
          if (k == ko) yo = v;
        }
      }
      const double x = __dadd_rn(
          __dmul_rn(F.lam, __dsub_rn((double)yo, __dmul_rn(F.c, (double)sy))), F.o[ko]);
      hi = (float)x;
      lo = (float)(x - (double)hi);
    }
    float xh[D], xl[D];
#pragma unroll
    for (int k = 0; k < D; k++) {
      xh[k] = k < d ? __shfl_sync(FULL, hi, k) : 0.f;
      xl[k] = k < d ? __shfl_sync(FULL, lo, k) : 0.f;
    }
    __syncwarp();  // the previous group's list has been read
    const float g2 = (float)(R.gamma * 1.4426950408889634);
    // W K of the instantiation that takes the list
    const int held = CLS == 2 ? RG_BIG : CLS == 1 ? (nl <= 256 ? 256 : RG_MID)
                                                  : (nl <= 64 ? 64 : nl <= 128 ? 128 : RG_SMALL);
    float gs[(D + 3) & ~3];
#pragma unroll
    for (int k = 0; k < ((D + 3) & ~3); k++) gs[k] = 0.f;
    for (int i = lane; i < held; i += 32) {
      float cc[2 * D], u[D], al = 0.f, s32, A = 0.f;
      const bool in = i < nl;
      if (in) sv_row<D>(R, src[i], cc, al, s32);
#pragma unroll
      for (int k = 0; k < D; k++) {
        u[k] = in && k < d ? (xh[k] - cc[2 * k]) + (xl[k] - cc[2 * k + 1]) : 0.f;
        lst[k * CAP + i] = u[k];
        A = fmaf(u[k], u[k], A);
      }
      lst[D * CAP + i] = -g2 * A;
      lst[(D + 1) * CAP + i] = al;
      const float e = al * ex2_approx(-g2 * A);
#pragma unroll
      for (int k = 0; k < D; k++) gs[k] = fmaf(e, u[k], gs[k]);
    }
#pragma unroll
    for (int k = 0; k < D; k += 4) sub_sum4<32>(gs[k], gs[k + 1], gs[k + 2], gs[k + 3]);
    __syncwarp();
    const RgCtx c = {R,  B,  lst, dirt, src, nl, e0, gs, g2, (float)R.gamma, (float)R.b,
                     (fast ? ROOT_TAU_FAST : ROOT_TAU) * 0.60653066f, fast != 0};
    if (CLS == 2) {
      rg_solve<D, 32, RG_BIG / 32, CAP>(c, gr.off, gr.n, nterms);
    } else if (CLS == 1) {
      if (held == 256) rg_solve<D, 16, 16, CAP>(c, gr.off, gr.n, nterms);
      else rg_solve<D, 16, RG_MID / 16, CAP>(c, gr.off, gr.n, nterms);
    } else {
      if (held == 64) rg_solve<D, 8, 8, CAP>(c, gr.off, gr.n, nterms);
      else if (held == 128) rg_solve<D, 16, 8, CAP>(c, gr.off, gr.n, nterms);
      else rg_solve<D, 16, RG_SMALL / 16, CAP>(c, gr.off, gr.n, nterms);
    }
  }
  const unsigned long long all = mf_warp_sum_ull(nterms);
  if (lane == 0 && all) atomicAdd(&B.cnt->root_terms_weak, all);
}

template <int D, int CLS>
static void launch_class(const MfFrame &F, const MfRbfDev &R, const MfTraceBufs &B, uint64_t e0,
                         bool fast, int sms, cudaStream_t st) {
  const int bytes = ((1 << F.d) * (D + 1) + RG_WARPS * (D + 2) * RgClass<CLS>::CAP) * 4;
  cudaFuncSetAttribute(k_rg_solve<D, CLS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  k_rg_solve<D, CLS><<<sms * RgClass<CLS>::BLOCKS, RG_WARPS * 32, bytes, st>>>(F, R, B, e0, fast ? 1 : 0);
}

template <int D>
static void launch_solve(const MfFrame &F, const MfRbfDev &R, const MfTraceBufs &B, uint64_t e0,
                         bool fast, int sms, cudaStream_t st) {
  launch_class<D, 0>(F, R, B, e0, fast, sms, st);
  if (R.n > RG_SMALL) launch_class<D, 1>(F, R, B, e0, fast, sms, st);
  if (R.n > RG_MID) launch_class<D, 2>(F, R, B, e0, fast, sms, st);
}

void mf_launch_roots_grouped(const MfFrame &F, const MfRbfDev &R, const MfTraceBufs &B, uint64_t e0,
                             uint64_t n, bool fast, int sms, cudaStream_t st) {
  const unsigned nb = (unsigned)((n + 255) / 256);
  cudaMemsetAsync(B.vert_edges, 0, B.max_vertices * 4, st);
  k_rg_count<<<nb, 256, 0, st>>>(F, B, e0, n);
  k_rg_groups<<<sms * 8, 256, 0, st>>>(B);
  k_rg_scatter<<<nb, 256, 0, st>>>(B, e0, n);
  switch (F.d) {
#define MF_CASE(DD) \
  case DD: launch_solve<DD>(F, R, B, e0, fast, sms, st); break;
    MF_CASE(2) MF_CASE(3) MF_CASE(4) MF_CASE(5) MF_CASE(6) MF_CASE(7)
#undef MF_CASE
    default: launch_solve<MF_MAXD>(F, R, B, e0, fast, sms, st);
  }
}
