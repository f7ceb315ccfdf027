// mf_sort.cu -- the sorted output order of mf_trace (MF_SORT_OUTPUT): edges
// by their 64-bit edge key, cells by (vertex key of z, pi), and the cell ->
// edge CSR carried over to both new orders.
//
// The sort is a stable least-significant-digit radix sort of (key, payload)
// pairs with digits of up to 8 bits; a first pass finds the bits where the
// keys differ, and the digits cover the span of those bits evenly.  Per pass,
// a block owns a tile of 4096 keys:
//   k_sort_hist     digit histogram of the tile (digit-major over the tiles,
//                   so one exclusive scan gives every (digit, tile) its
//                   output offset);
//   k_sort_scatter  reads the tile once, ranks the keys of one digit among
//                   themselves with __match_any_sync (each warp its contiguous
//                   512-key part in order, earlier warps and tiles first:
//                   stable), orders the tile by digit in shared memory and
//                   writes it out in runs of consecutive addresses.
// Bound by memory: 8 + 24 bytes per key and pass.  Scattered writes of a key at
// a time moved a 32-byte sector for each; in runs, the passes of a d = 5 proof
// at lambda = 0.08 take 4.3 ms instead of 6.9.
#include <algorithm>
#include <cstring>
#include <utility>
#include <vector>

#include "mf_internal.cuh"
#include "mf_ctx.h"

#define SORT_THREADS 256
#define SORT_ITEMS 16
#define SORT_TILE (SORT_THREADS * SORT_ITEMS)
#define SORT_SEG (SORT_TILE / (SORT_THREADS / 32))  // keys per warp: 512

__global__ void k_sort_bits(const unsigned long long *keys, int64_t n, unsigned long long *and_or) {
  unsigned long long a = ~0ull, o = 0ull;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    a &= keys[i];
    o |= keys[i];
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    a &= __shfl_xor_sync(0xffffffffu, a, s);
    o |= __shfl_xor_sync(0xffffffffu, o, s);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAnd(&and_or[0], a);
    atomicOr(&and_or[1], o);
  }
}

__global__ void __launch_bounds__(SORT_THREADS) k_sort_hist(const unsigned long long *keys, int64_t n,
                                                            int shift, uint32_t dmask, int64_t *hist,
                                                            int64_t nb) {
  __shared__ int cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = blockIdx.x * (int64_t)SORT_TILE;
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; i++) {
    const int64_t k = base + i * SORT_THREADS + threadIdx.x;
    if (k < n) atomicAdd(&cnt[(uint32_t)(keys[k] >> shift) & dmask], 1);
  }
  __syncthreads();
  if (threadIdx.x <= dmask) hist[(int64_t)threadIdx.x * nb + blockIdx.x] = cnt[threadIdx.x];
}

__global__ void __launch_bounds__(SORT_THREADS, 3) k_sort_scatter(const unsigned long long *keys,
                                                               const uint32_t *vals, int64_t n,
                                                               int shift, uint32_t dmask,
                                                               const int64_t *offs, int64_t nb,
                                                               unsigned long long *keys_out,
                                                               uint32_t *vals_out) {
  constexpr int W = SORT_THREADS / 32;
  __shared__ unsigned long long skey[SORT_TILE];  // the tile by digit; then its payloads
  __shared__ uint16_t cnt[W][256];  // keys of each digit in each warp's part, then their start
  // output position of the tile's place 0, per digit (n < 2^32: the sum with
  // the place is right modulo 2^32)
  __shared__ uint32_t gofs[256];
  __shared__ int wsum[W];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  for (int i = threadIdx.x; i < W * 256; i += SORT_THREADS) (&cnt[0][0])[i] = 0;
  __syncthreads();
  const int64_t tile = blockIdx.x * (int64_t)SORT_TILE, seg = tile + (int64_t)w * SORT_SEG;
  unsigned long long key[SORT_ITEMS];
  uint16_t rank[SORT_ITEMS];
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; i++) {
    const int64_t k = seg + i * 32 + lane;
    key[i] = k < n ? keys[k] : 0ull;
  }
  // 1. the place of each key among the warp's keys of its digit
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; i++) {
    const bool have = seg + i * 32 + lane < n;
    const uint32_t dg = have ? (uint32_t)(key[i] >> shift) & dmask : 256u + lane;
    const unsigned peers = __match_any_sync(0xffffffffu, dg);
    const uint32_t before = have ? cnt[w][dg] : 0u;
    rank[i] = (uint16_t)(before + __popc(peers & lt));
    __syncwarp();
    if (have && (peers & lt) == 0) cnt[w][dg] = (uint16_t)(before + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  // 2. where the digits, and in them the warps, start in the tile
  {
    const uint32_t dg = threadIdx.x;  // SORT_THREADS == 256 digits
    int total = 0;
#pragma unroll
    for (int q = 0; q < W; q++) {
      const int c = cnt[q][dg];
      cnt[q][dg] = (uint16_t)total;
      total += c;
    }
    int inc = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    int start = inc - total;
    for (int q = 0; q < w; q++) start += wsum[q];
#pragma unroll
    for (int q = 0; q < W; q++) cnt[q][dg] = (uint16_t)(cnt[q][dg] + start);
    if (dg <= dmask) gofs[dg] = (uint32_t)offs[(int64_t)dg * nb + blockIdx.x] - (uint32_t)start;
  }
  __syncthreads();
  // 3. the tile by digit, and out
  const int m = (int)(n - tile < SORT_TILE ? n - tile : SORT_TILE);
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; i++) {
    if (seg + i * 32 + lane < n) {
      rank[i] = (uint16_t)(rank[i] + cnt[w][(uint32_t)(key[i] >> shift) & dmask]);
      skey[rank[i]] = key[i];
    }
  }
  __syncthreads();
  uint32_t at[SORT_ITEMS];
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; i++) {
    const int p = i * SORT_THREADS + threadIdx.x;
    if (p < m) {
      const unsigned long long k = skey[p];
      at[i] = gofs[(uint32_t)(k >> shift) & dmask] + (uint32_t)p;
      keys_out[at[i]] = k;
    }
  }
  __syncthreads();
  uint32_t *sval = reinterpret_cast<uint32_t *>(skey);
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; i++) {
    const int64_t k = seg + i * 32 + lane;
    if (k < n) sval[rank[i]] = vals[k];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; i++) {
    const int p = i * SORT_THREADS + threadIdx.x;
    if (p < m) vals_out[at[i]] = sval[p];
  }
}

// Stable sort of n (key, payload) pairs; the result is in keys / vals.
// tmp_k, tmp_v: n each; hist: 256 * ceil(n / SORT_TILE) + 1 int64; scan:
// scratch of mf_exclusive_scan for that many entries; ao: 2 words.
static int radix_sort(mf_ctx *ctx, unsigned long long *keys, uint32_t *vals,
                      unsigned long long *tmp_k, uint32_t *tmp_v, int64_t n, int64_t *hist,
                      int64_t *scan, unsigned long long *ao, cudaStream_t st) {
  if (n <= 1) return MF_OK;
  const unsigned long long init[2] = {~0ull, 0ull};
  unsigned long long h[2];
  cudaMemcpyAsync(ao, init, sizeof(init), cudaMemcpyHostToDevice, st);
  k_sort_bits<<<ctx->sms * 4, 256, 0, st>>>(keys, n, ao);
  cudaMemcpyAsync(h, ao, sizeof(h), cudaMemcpyDeviceToHost, st);
  int rc = mf_cuda_check(ctx, cudaStreamSynchronize(st), "sort bits");
  if (rc) return rc;
  const unsigned long long diff = h[0] ^ h[1];
  const int64_t nb = (n + SORT_TILE - 1) / SORT_TILE;
  unsigned long long *ka = keys, *kb = tmp_k;
  uint32_t *va = vals, *vb = tmp_v;
  // digits of equal width over the span of the bits that differ
  int lo = 0, hi = 64;
  while (lo < 64 && !((diff >> lo) & 1ull)) lo++;
  while (hi > lo && !((diff >> (hi - 1)) & 1ull)) hi--;
  const int passes = (hi - lo + 7) / 8, width = passes ? (hi - lo + passes - 1) / passes : 0;
  for (int shift = lo; shift < hi; shift += width) {
    const int bits = std::min(width, hi - shift);
    const uint32_t dmask = (1u << bits) - 1u;
    if (!((diff >> shift) & (unsigned long long)dmask)) continue;
    k_sort_hist<<<(unsigned)nb, SORT_THREADS, 0, st>>>(ka, n, shift, dmask, hist, nb);
    mf_exclusive_scan(hist, hist, ((int64_t)dmask + 1) * nb, scan, st);
    k_sort_scatter<<<(unsigned)nb, SORT_THREADS, 0, st>>>(ka, va, n, shift, dmask, hist, nb, kb, vb);
    std::swap(ka, kb);
    std::swap(va, vb);
  }
  if (ka != keys) {
    cudaMemcpyAsync(keys, ka, (size_t)n * 8, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(vals, va, (size_t)n * 4, cudaMemcpyDeviceToDevice, st);
  }
  return mf_cuda_check(ctx, cudaGetLastError(), "radix sort");
}

__global__ void k_edge_keys(MfFrame F, MfTraceBufs B, uint64_t n, unsigned long long *keys,
                            uint32_t *vals) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  int32_t y[MF_MAXD];
#pragma unroll
  for (int k = 0; k < MF_MAXD; k++) y[k] = k < F.d ? B.edge_y[i * F.d + k] : 0;
  keys[i] = mf_edge_key(F, y, B.edge_mask[i]);
  vals[i] = (uint32_t)i;
}

// cell keys in one word: the vertex key of z above the lexicographic rank of
// pi (fewer bits than its base-8 digits, in the same order), where both fit:
// fewer passes than two sorts, and no gather of the keys between them.
__global__ void k_cell_keys(MfFrame F, MfTraceBufs B, uint64_t n, int rank_bits,
                            unsigned long long *keys, uint32_t *vals) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int d = F.d;
  int32_t z[MF_MAXD];
#pragma unroll
  for (int k = 0; k < MF_MAXD; k++) z[k] = k < d ? B.cell_y[i * d + k] : 0;
  uint32_t rank = 0, left = (1u << d) - 1u;  // elements not used yet
  for (int k = 0; k < d; k++) {
    const uint32_t p = B.cell_perm[i * d + k];
    rank = rank * (uint32_t)(d - k) + (uint32_t)__popc(left & ((1u << p) - 1u));
    left &= ~(1u << p);
  }
  keys[i] = (mf_vertex_key(F, z) << rank_bits) | rank;
  vals[i] = (uint32_t)i;
}

// else two sorts: lo = pi as base-8 digits (pi_0 most significant), then hi =
// the vertex key of z for the cells in the order of the first sort
__global__ void k_cell_keys_lo(MfFrame F, MfTraceBufs B, uint64_t n, unsigned long long *keys,
                               uint32_t *vals) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned long long code = 0;
  for (int k = 0; k < F.d; k++) code = (code << 3) | B.cell_perm[i * F.d + k];
  keys[i] = code;
  vals[i] = (uint32_t)i;
}

__global__ void k_cell_keys_hi(MfFrame F, MfTraceBufs B, uint64_t n, const uint32_t *vals,
                               unsigned long long *keys) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  int32_t z[MF_MAXD];
  const uint64_t c = vals[i];
#pragma unroll
  for (int k = 0; k < MF_MAXD; k++) z[k] = k < F.d ? B.cell_y[c * F.d + k] : 0;
  keys[i] = mf_vertex_key(F, z);
}

__global__ void k_inverse(const uint32_t *perm, uint64_t n, uint32_t *inv) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i < n) inv[perm[i]] = (uint32_t)i;
}

// Sorted copies into the caller's buffers.
__global__ void k_gather_edges(int d, MfTraceBufs B, const uint32_t *perm, uint64_t n, bool roots,
                               int32_t *ey, uint32_t *em, double *ef, double *et, double *ep) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t o = perm[i];
  for (int k = 0; k < d; k++) {
    if (ey) ey[i * d + k] = B.edge_y[o * d + k];
    if (ep && roots) ep[i * d + k] = B.edge_pt[o * d + k];
  }
  if (em) em[i] = B.edge_mask[o];
  if (ef) {
    ef[2 * i] = B.edge_f[2 * o];
    ef[2 * i + 1] = B.edge_f[2 * o + 1];
  }
  if (et && roots) et[i] = B.edge_t[o];
}

__global__ void k_gather_cells(int d, MfTraceBufs B, const uint32_t *perm, uint64_t n, int32_t *cy,
                               uint8_t *cp, int64_t *len) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t o = perm[i];
  for (int k = 0; k < d; k++) {
    if (cy) cy[i * d + k] = B.cell_y[o * d + k];
    if (cp) cp[i * d + k] = B.cell_perm[o * d + k];
  }
  if (len) len[i] = B.cell_off[o + 1] - B.cell_off[o];
}

// The rows in the cells' new order with the edges' new indices.  A warp takes 32
// cells, whose output is one contiguous range: lane per entry, so that the
// stores are whole lines and the loads whole rows (a thread per cell stored
// 8 bytes at a time, a row apart from its neighbours: 2.5 -> 2.0 ms for a d = 5
// proof at lambda = 0.08, 1.26 -> 0.95 ms for a d = 6 proof).
__global__ void __launch_bounds__(256) k_gather_csr(MfTraceBufs B, const uint32_t *perm,
                                                    const uint32_t *inv_e, uint64_t n,
                                                    const int64_t *new_off, int64_t *idx) {
  __shared__ uint32_t s_end[8][32];
  __shared__ int64_t s_src[8][32];  // source of the row's entries, less its start in the warp's range
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t c0 = (blockIdx.x * (uint64_t)8 + w) * 32, i = c0 + lane;
  if (c0 >= n) return;  // whole warp
  uint32_t len = 0;
  int64_t a = 0;
  if (i < n) {
    const uint64_t o = perm[i];
    a = B.cell_off[o];
    len = (uint32_t)(B.cell_off[o + 1] - a);
  }
  uint32_t inc = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  s_end[w][lane] = inc;
  s_src[w][lane] = a - (int64_t)(inc - len);
  const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
  __syncwarp();
  const int64_t out = new_off[c0];
  for (uint32_t q = lane; q < total; q += 32) {
    int o = 0;  // the first row that ends after q
#pragma unroll
    for (int step = 16; step; step >>= 1)
      if (s_end[w][o + step - 1] <= q) o += step;
    const int64_t e = B.cell_idx[s_src[w][o] + q];
    idx[out + q] = e >= 0 ? (int64_t)inv_e[e] : -1;
  }
}

// Computes the sorted orders of the trace in L (edge and cell permutations,
// new -> old, and the edges' inverse) into the context's sort slot.
int mf_sort_trace(mf_ctx *ctx, MfTraceState &L, cudaStream_t st) {
  const uint64_t E = (uint64_t)L.n_edges, C = (uint64_t)L.n_cells;
  if (E >= (1ull << 32) || C >= (1ull << 32))
    return mf_set_error(ctx, MF_ERR_INVALID, "sorted output needs fewer than 2^32 edges and cells");
  const uint64_t N = std::max<uint64_t>(std::max<uint64_t>(E, C), 2);
  const int64_t nb = (int64_t)((N + SORT_TILE - 1) / SORT_TILE);
  auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t hist_n = (size_t)256 * nb + 1;
  const size_t bytes = al(E * 4 + 8) * 2 + al(C * 4 + 8) + al(N * 8) * 2 + al(N * 4) +
                       al(hist_n * 8) + al((hist_n / 4096 + 2) * 8) + 256;
  char *p = (char *)mf_ctx_buffer(ctx, MF_SLOT_SORT, bytes);
  if (!p) return MF_ERR_OOM;
  uint32_t *perm_e = (uint32_t *)p; p += al(E * 4 + 8);
  uint32_t *inv_e = (uint32_t *)p; p += al(E * 4 + 8);
  uint32_t *perm_c = (uint32_t *)p; p += al(C * 4 + 8);
  unsigned long long *keys = (unsigned long long *)p; p += al(N * 8);
  unsigned long long *tk = (unsigned long long *)p; p += al(N * 8);
  uint32_t *tv = (uint32_t *)p; p += al(N * 4);
  int64_t *hist = (int64_t *)p; p += al(hist_n * 8);
  int64_t *scan = (int64_t *)p; p += al((hist_n / 4096 + 2) * 8);
  unsigned long long *ao = (unsigned long long *)p;
  int rc;
  if (E) {
    k_edge_keys<<<(unsigned)((E + 255) / 256), 256, 0, st>>>(L.F, L.B, E, keys, perm_e);
    if ((rc = radix_sort(ctx, keys, perm_e, tk, tv, (int64_t)E, hist, scan, ao, st))) return rc;
    k_inverse<<<(unsigned)((E + 255) / 256), 256, 0, st>>>(perm_e, E, inv_e);
  }
  // bits of the cells' vertex keys (a few lattice steps around the box, which
  // the packing covers) and of the rank of pi
  int rank_bits = 0, key_bits = 0;
  {
    unsigned long long f = 1;
    for (int k = 2; k <= L.F.d; k++) f *= (unsigned long long)k;
    while ((1ull << rank_bits) < f) rank_bits++;
    const unsigned __int128 top = (unsigned __int128)L.F.sstride * (uint32_t)L.F.kspan_s;
    while (key_bits < 64 && ((unsigned __int128)1 << key_bits) < top) key_bits++;
  }
  if (C && key_bits + rank_bits <= 64) {
    k_cell_keys<<<(unsigned)((C + 255) / 256), 256, 0, st>>>(L.F, L.B, C, rank_bits, keys, perm_c);
    if ((rc = radix_sort(ctx, keys, perm_c, tk, tv, (int64_t)C, hist, scan, ao, st))) return rc;
  } else if (C) {
    k_cell_keys_lo<<<(unsigned)((C + 255) / 256), 256, 0, st>>>(L.F, L.B, C, keys, perm_c);
    if ((rc = radix_sort(ctx, keys, perm_c, tk, tv, (int64_t)C, hist, scan, ao, st))) return rc;
    k_cell_keys_hi<<<(unsigned)((C + 255) / 256), 256, 0, st>>>(L.F, L.B, C, perm_c, keys);
    if ((rc = radix_sort(ctx, keys, perm_c, tk, tv, (int64_t)C, hist, scan, ao, st))) return rc;
  }
  L.perm_e = perm_e;
  L.inv_e = inv_e;
  L.perm_c = perm_c;
  L.sort_scan = scan;
  return mf_cuda_check(ctx, cudaGetLastError(), "sorted output");
}

// The copy-out of mf_trace in the sorted order (the caller checked the
// capacities).
int mf_copy_out_sorted(mf_ctx *ctx, const MfTraceState &L, mf_trace_out *out, cudaStream_t st) {
  const int d = L.F.d;
  const uint64_t E = (uint64_t)L.n_edges, C = (uint64_t)L.n_cells;
  const bool roots = (L.flags & MF_WANT_ROOTS) != 0;
  if (E && (out->edge_y || out->edge_mask || out->edge_f || out->edge_t || out->points))
    k_gather_edges<<<(unsigned)((E + 255) / 256), 256, 0, st>>>(
        d, L.B, L.perm_e, E, roots, out->edge_y, out->edge_mask, out->edge_f, out->edge_t,
        out->points);
  if ((L.flags & MF_WANT_CELLS) && (out->cell_y || out->cell_perm || out->cell_edge_off)) {
    if (C) {
      k_gather_cells<<<(unsigned)((C + 255) / 256), 256, 0, st>>>(
          d, L.B, L.perm_c, C, out->cell_y, out->cell_perm, out->cell_edge_off);
      if (out->cell_edge_off) {
        mf_exclusive_scan(out->cell_edge_off, out->cell_edge_off, (int64_t)C, L.sort_scan, st);
        if (out->cell_edge_idx)
          k_gather_csr<<<(unsigned)((C + 255) / 256), 256, 0, st>>>(
              L.B, L.perm_c, L.inv_e, C, out->cell_edge_off, out->cell_edge_idx);
      }
    } else if (out->cell_edge_off) {
      cudaMemsetAsync(out->cell_edge_off, 0, 8, st);
    }
  }
  return mf_cuda_check(ctx, cudaGetLastError(), "sorted copy");
}
