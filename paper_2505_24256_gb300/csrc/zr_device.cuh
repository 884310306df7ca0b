// zr_device.cuh -- device helpers shared by the step kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "zr_arith.cuh"
#include "zr_kernels.cuh"

namespace zr {

constexpr uint64_t kEmptySlot = ~0ull;

// Open-addressing node table (the distinctness check of the anchor values).
__device__ __forceinline__ uint64_t hash64(uint64_t x) {
  x ^= x >> 31;
  x *= 0x9E3779B97F4A7C15ull;
  return x ^ (x >> 29);
}

// Insert x into the open-addressing table; flags a duplicate.  Every probe
// sequence ends: the table has at least 2T slots and each thread inserts one key.
__device__ __forceinline__ void node_insert(uint64_t x, uint64_t* htab, uint64_t hmask, uint32_t* status) {
  uint64_t idx = hash64(x) & hmask;
  for (uint64_t probe = 0; probe <= hmask; probe++) {
    unsigned long long prev = atomicCAS((unsigned long long*)&htab[idx], (unsigned long long)kEmptySlot,
                                        (unsigned long long)x);
    if (prev == kEmptySlot) return;
    if (prev == x) { atomicOr(status, ST_DUP_NODE); return; }
    idx = (idx + 1) & hmask;
  }
  atomicOr(status, ST_HASH_FULL);
}

// Dot products of the product tree: a full 128-bit product per term.
__device__ __forceinline__ uint64_t conv_coef(const uint64_t* in, int po, int a, int b, int n, const Mod& M) {
  Acc8 acc = {0, 0, 0, 0, 0, 0, 0, 0};
  int ilo = n - b > 0 ? n - b : 0, ihi = n < a ? n : a;
  for (int i = ilo; i <= ihi; i++) {
    uint64_t Ai = (i < a) ? in[po + i] : 1;
    int jj = n - i;
    uint64_t Bj = (jj < b) ? in[po + a + jj] : 1;
    mac8(acc, lo32(Ai), hi32(Ai), lo32(Bj), hi32(Bj));
  }
  return acc8_value(acc, M);
}

// Inverse of d for every lane of a warp; lanes with d = 0 get 0.  Each lane runs
// its own inversion: the longest of 32 takes about a quarter more steps than one
// (Montgomery's trick, one inversion for the warp, put ten modular products of
// prefix and suffix scans and three more in front of and behind it).
__device__ __forceinline__ uint64_t warp_batch_inverse(uint64_t d, const Mod& M) { return inv_mod(d, M); }

// ---- Newton interpolation on shared nodes (Introduction, the Newton formula) -----
//
// Every term of a step is interpolated on the same S nodes x_0..x_{S-1}, so
// the map from the S values to the S monomial coefficients is one S x S
// matrix W shared by all terms.  Column s of W is the interpolant of the unit
// vector e_s (which Newton's formula and Lagrange's give alike): the
// coefficients of prod_{t != s} (z - x_t) / (x_s - x_t).  Applying W to a
// term's values is S^2 independent multiply-accumulates with one reduction per
// coefficient, instead of a chain of S^2 dependent modular products.

constexpr int kNewtonMax = 64;   // largest point count

// W[e S + s] for the nodes xs_g (S <= 32 NR) by one warp: P = prod_t (z - x_t), a
// factor at a time with the coefficients in the lanes; then lane s divides P by z -
// x_s, takes the quotient's value at x_s along the way and scales by its inverse.
// Equal nodes set ST_DUP_SAMPLE in *status (null: not reported; W is then
// meaningless).  About 3 S chain steps and one inversion: 0.012 ms at S = 21,
// where all S^2 pairs of the divided differences and of the nested expansion,
// level by level in a block of 1024 threads, took 0.047 ms (2 S barriers and an
// inversion per pair).
template <int NR>
__device__ inline void newton_matrix_warp(int S, const uint64_t* __restrict__ xs_g, uint64_t* W, uint32_t* status,
                                          const Mod& M) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  uint64_t x[NR], xq[NR], c[NR], q[NR], u[NR];
#pragma unroll
  for (int r = 0; r < NR; r++) {
    const int s = lane + 32 * r;
    x[r] = s < S ? canon(xs_g[s], M) : 0;
    xq[r] = shoup_pre(x[r], M);
    c[r] = s == 0 ? 1 : 0;
    q[r] = 1;
    u[r] = 0;
  }
  auto at = [&](const uint64_t(&v)[NR], int i) {
    const uint64_t lo = __shfl_sync(FULL, v[0], i & 31), hi = __shfl_sync(FULL, v[NR - 1], i & 31);
    return i < 32 ? lo : hi;
  };
  for (int t = 0; t < S; t++) {
    const uint64_t xt = at(x, t), xqt = at(xq, t);
    uint64_t below = 0;                          // coefficient 32 r - 1, for lane 0
#pragma unroll
    for (int r = 0; r < NR; r++) {
      uint64_t up = __shfl_up_sync(FULL, c[r], 1);
      const uint64_t top = __shfl_sync(FULL, c[r], 31);
      if (lane == 0) up = below;
      below = top;
      c[r] = sub_mod(up, canon(shoup_lazy(c[r], xt, xqt, M), M), M);
    }
  }
  for (int e = S - 1; e >= 0; e--) {
    const uint64_t pe = at(c, e);
#pragma unroll
    for (int r = 0; r < NR; r++) {
      const int s = lane + 32 * r;
      u[r] = add_mod(canon(shoup_lazy(u[r], x[r], xq[r], M), M), q[r], M);
      if (s < S) W[e * S + s] = q[r];
      q[r] = add_mod(canon(shoup_lazy(q[r], x[r], xq[r], M), M), pe, M);
    }
  }
#pragma unroll
  for (int r = 0; r < NR; r++) {
    const int s = lane + 32 * r;
    if (s >= S) continue;
    if (u[r] == 0 && status) atomicOr(status, ST_DUP_SAMPLE);
    const uint64_t inv = inv_mod(u[r], M), iq = shoup_pre(inv, M);
    for (int e = 0; e < S; e++) W[e * S + s] = canon(shoup_lazy(W[e * S + s], inv, iq, M), M);
  }
}
__device__ __forceinline__ void newton_matrix(int S, const uint64_t* __restrict__ xs_g, uint64_t* W, uint32_t* status,
                                              const Mod& M) {
  if (S == 1) {                                  // (the inverse of 1 takes as long as any)
    if ((threadIdx.x & 31) == 0) W[0] = 1;
    return;
  }
  if (S <= 32) newton_matrix_warp<1>(S, xs_g, W, status, M);
  else newton_matrix_warp<2>(S, xs_g, W, status, M);
}

// out[e * ld] = scale * sum_s W[e][s] val[s * stride] for e < S (W and val in
// shared memory, val canonical); returns how many of them are nonzero.
__device__ inline int newton_apply(int S, const uint64_t* W, const uint64_t* val, int stride, uint64_t scale,
                                   uint64_t* out, int64_t ld, const Mod& M, int e_first = 0, int e_step = 1) {
  int cnt = 0;
  if (e_step != 1) {
    // the outputs e_first, e_first + e_step, ... only
    for (int e = e_first; e < S; e += e_step) {
      Acc8 acc = {0, 0, 0, 0, 0, 0, 0, 0};
      const uint64_t* w = W + (int64_t)e * S;
      for (int s = 0; s < S; s++) {
        const uint64_t x = val[s * stride], y = w[s];
        mac8(acc, lo32(x), hi32(x), lo32(y), hi32(y));
      }
      const uint64_t g = mul_mod(acc8_value(acc, M), scale, M);
      out[(int64_t)e * ld] = g;
      cnt += g != 0;
    }
    return cnt;
  }
  for (int e0 = 0; e0 < S; e0 += 4) {
    Acc8 acc[4];
#pragma unroll
    for (int q = 0; q < 4; q++) acc[q] = Acc8{0, 0, 0, 0, 0, 0, 0, 0};
    const uint64_t* w0 = W + (e0 + 0 < S ? e0 + 0 : S - 1) * S;
    const uint64_t* w1 = W + (e0 + 1 < S ? e0 + 1 : S - 1) * S;
    const uint64_t* w2 = W + (e0 + 2 < S ? e0 + 2 : S - 1) * S;
    const uint64_t* w3 = W + (e0 + 3 < S ? e0 + 3 : S - 1) * S;
    for (int s = 0; s < S; s++) {
      const uint64_t x = val[s * stride];
      const uint32_t x0 = lo32(x), x1 = hi32(x);
      uint64_t w = w0[s];
      mac8(acc[0], x0, x1, lo32(w), hi32(w));
      w = w1[s];
      mac8(acc[1], x0, x1, lo32(w), hi32(w));
      w = w2[s];
      mac8(acc[2], x0, x1, lo32(w), hi32(w));
      w = w3[s];
      mac8(acc[3], x0, x1, lo32(w), hi32(w));
    }
#pragma unroll
    for (int q = 0; q < 4; q++)
      if (e0 + q < S) {
        const uint64_t g = mul_mod(acc8_value(acc[q], M), scale, M);
        out[(int64_t)(e0 + q) * ld] = g;
        cnt += g != 0;
      }
  }
  return cnt;
}

// Exclusive scan over a CTA (blockDim.x a multiple of 32, at most 1024);
// sh holds 33 words; every thread of the CTA must call it.
__device__ __forceinline__ int64_t block_exclusive_scan(int64_t x, int64_t* sh, int64_t& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int64_t incl = x;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    int64_t t = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += t;
  }
  if (lane == 31) sh[w] = incl;
  __syncthreads();
  if (w == 0) {
    const int64_t s = lane < nw ? sh[lane] : 0;
    int64_t si = s;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      int64_t t = __shfl_up_sync(0xffffffffu, si, off);
      if (lane >= off) si += t;
    }
    sh[lane] = si - s;          // exclusive prefix of warp totals
    if (lane == 31) sh[32] = si;
  }
  __syncthreads();
  total = sh[32];
  const int64_t r = incl - x + sh[w];
  __syncthreads();              // sh may be reused right after
  return r;
}

// Segment of a flattened index: the largest i < n with pre[i] <= x.
__device__ __forceinline__ int seg_of(const int64_t* __restrict__ pre, int n, int64_t x) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(pre + mid) <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

}  // namespace zr
