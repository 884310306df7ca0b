// zr_balance.cu -- the balanced Zippel step for rational functions (Sec. 1,
// Sec. 2.2, the balancing identity) and its univariate rational
// reconstruction (Thiele, Eq. thiele).
//
// For probe i the black box gives f(y^(i+off), c_s) for the Sf samples c_s.
// One warp per probe runs Thiele interpolation in the new variable:
//   inverse differences phi_l(x_t) = (x_t - x_{l-1}) / (phi_{l-1}(x_t) - b_{l-1}),
//   b_l = phi_l(x_l), stopped at the first level whose tail is constant on the
//   remaining samples, then the convergent P_L/Q_L of
//   b_0 + (x - x_0)/(b_1 + (x - x_1)/(b_2 + ...)) expanded to coefficients and
//   scaled so that Q(c_0) = 1: n_i = P/Q(c_0), d_i = Q/Q(c_0).
// All of it runs on fractions, so that the only inversion of a probe is the
// final scale (the probes of a block share it).
// The balancing factor is the previous
// denominator skeleton at the probe, D'(y^(i+off)) = C D(y^i, c_0); with
// d_i(c_0) = 1 it turns the reduced pair into
//   bN[s][i] = D'(y^i) n_i(c_s) = C N(y^i, c_s),   bD[s][i] = D'(y^i) d_i(c_s) = C D(y^i, c_s),
// the probes of one Zippel step for N and one for D with a common scale C.
// (The paper takes the ratio from the numerator skeleton; the denominator
// gives the same factor C/h_i and cannot vanish away from poles.)
#include <cuda_runtime.h>

#include "zr_device.cuh"
#include "zr_internal.h"

namespace zr {

static inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

// Lane t (and t + 32 with NR = 2 registers, up to 64 samples) holds sample t:
// phi_l(x_t) = (gn / gd) N_t / D_t with one scale gn / gd for the whole level,
//   D'_t = N_t D_b - N_b D_t   (zero exactly when phi_l(x_t) = b_l),
//   N'_t = (x_t - x_l) D_t,    gn' / gd' = D_b gd / gn,
// (N_b, D_b) the pair of lane l.  With B_l = gn N_b, E_l = gd D_b, b_l = B_l /
// E_l, the convergents multiplied by s_l = E_0 .. E_l satisfy
//   P_l = B_l P_{l-1} + E_l E_{l-1} (x - x_{l-1}) P_{l-2},
// and Q_l likewise, from (s_{-1} = 1) P_{-1} = 1, Q_{-1} = 0, P_0 = B_0,
// Q_0 = E_0.  deg P_l, Q_l <= (l + 1) / 2 and L <= n - 2, so the coefficients
// fit 16 lanes each for n <= 32 (P in the low, Q in the high half of the
// warp) and 32 lanes each for n <= 64 (one register each).
//
// The kernel is bound by the multiply pipe (about n^2 / 2 fractions updated
// with three products each, n^2 / 2 coefficients with three).  The five
// calls of a reconstruction with up to 5000 probes of 32 samples take 0.27 ms
// (0.093 ms the largest, 0.04 ms the latency of one probe); with one thread
// per probe, its tables in memory and a 63-bit power per level they took 3.9 ms
// (40 blocks), and a division N / D before them another 0.23 ms.
constexpr int kThieleWarps = 8;

// x a + y b mod p
__device__ __forceinline__ uint64_t dot2(uint64_t x, uint64_t a, uint64_t y, uint64_t b, const Mod& M) {
  uint64_t h0, l0, h1, l1;
  mul128(x, a, h0, l0);
  mul128(y, b, h1, l1);
  const uint64_t l = l0 + l1;
  uint64_t h = h0 + h1 + (l < l0);           // h0, h1 < p / 2: at most p
  if (h >= M.p) h -= M.p;
  return reduce128(h, l, M);
}

template <int NR>
__global__ void __launch_bounds__(32 * kThieleWarps)
    k_thiele_balance(int64_t Tmax, int n, const uint64_t* __restrict__ xs, const uint64_t* __restrict__ fvals,
                     const uint64_t* __restrict__ fdens, int64_t ldf, const uint64_t* __restrict__ dprev, int dN,
                     int dD, int64_t TN, int64_t TD, Mod M, uint64_t* __restrict__ bN, int64_t ldN,
                     uint64_t* __restrict__ bD, int64_t ldD, uint32_t* status) {
  __shared__ uint64_t q0s[32];
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * kThieleWarps + warp;
  if (threadIdx.x < 32) q0s[threadIdx.x] = 0;
  __syncthreads();
  uint64_t x[NR], N[NR], D[NR], pv[NR], qv[NR];
  bool ok = i < Tmax, pole = false;
#pragma unroll
  for (int r = 0; r < NR; r++) {
    const int t = lane + 32 * r;
    x[r] = t < n ? xs[t] : 0;
    N[r] = ok && t < n ? canon(fvals[(int64_t)t * ldf + i], M) : 0;
    D[r] = ok && t < n && fdens ? fdens[(int64_t)t * ldf + i] : 1;
    pole |= D[r] == 0;
    pv[r] = qv[r] = 0;
  }
  if (__any_sync(FULL, pole)) {
    if (lane == 0) atomicOr(status, ST_POLE);
    ok = false;
  }
  if (ok) {
    // sample l's value from its lane
    auto at = [&](const uint64_t(&v)[NR], int l) {
      uint64_t r = __shfl_sync(FULL, v[0], l & 31);
      if (NR == 2) {
        const uint64_t hi = __shfl_sync(FULL, v[NR - 1], l & 31);
        if (l >= 32) r = hi;
      }
      return r;
    };
    uint64_t gn = 1, gd = 1;
    uint64_t nb = at(N, 0), db = at(D, 0);
    // coefficients, two levels back (c2) and one back (c1): NR = 1: P[lane]
    // and Q[lane - 16] in one register; NR = 2: P[lane] and Q[lane]
    uint64_t c2[NR], c1[NR];
    const int e = NR == 1 ? (lane & 15) : lane;
#pragma unroll
    for (int r = 0; r < NR; r++) {
      const bool isQ = NR == 1 ? lane >= 16 : r == 1;
      c2[r] = (!isQ && e == 0) ? 1 : 0;
      c1[r] = e == 0 ? (isQ ? db : nb) : 0;
    }
    uint64_t eprev = db;                         // E_{l-1}
    int L = -1;
    for (int l = 1; l < n; l++) {
      uint64_t dn[NR];
      bool any = false, all = true;
      const uint64_t nbm = nb ? M.p - nb : 0;
#pragma unroll
      for (int r = 0; r < NR; r++) {
        const int t = lane + 32 * r;
        dn[r] = dot2(N[r], db, nbm, D[r], M);
        const unsigned in = __ballot_sync(FULL, t >= l && t < n);
        const unsigned eq = __ballot_sync(FULL, dn[r] == 0) & in;
        any |= eq != 0;
        all &= eq == in;
      }
      if (all) { L = l - 1; break; }
      if (any) { if (lane == 0) atomicOr(status, ST_THIELE); ok = false; break; }
      const uint64_t xl = at(x, l - 1);
#pragma unroll
      for (int r = 0; r < NR; r++) {
        N[r] = mul_mod(sub_mod(x[r], xl, M), D[r], M);
        D[r] = dn[r];
      }
      const uint64_t g = mul_mod(db, gd, M);
      gd = gn;
      gn = g;
      nb = at(N, l);
      db = at(D, l);
      // B_l in the even lanes, E_l in the odd ones: one product for both
      const uint64_t be = mul_mod(lane & 1 ? gd : gn, lane & 1 ? db : nb, M);
      const uint64_t B = __shfl_sync(FULL, be, 0), E = __shfl_sync(FULL, be, 1);
      const uint64_t c = mul_mod(E, eprev, M);
      eprev = E;
#pragma unroll
      for (int r = 0; r < NR; r++) {
        uint64_t lo = __shfl_up_sync(FULL, c2[r], 1);
        if (e == 0) lo = 0;
        const uint64_t u = sub_mod(lo, mul_mod(xl, c2[r], M), M);   // coefficient e of (x - x_{l-1}) c2
        c2[r] = c1[r];
        c1[r] = dot2(B, c1[r], c, u, M);
      }
    }
    if (ok && L < 0) {
      if (lane == 0) atomicOr(status, ST_DEGREE);
      ok = false;
    }
    if (ok) {
      // the degrees, and P, Q at the samples t = lane (+ 32): Horner's rule,
      // a Shoup product by x_t per coefficient
      int degp, degq;
      if (NR == 1) {
        const unsigned nz = __ballot_sync(FULL, c1[0] != 0);
        degp = 31 - __clz(nz & 0xffffu);
        degq = 31 - __clz(nz >> 16);
      } else {
        degp = 31 - __clz(__ballot_sync(FULL, c1[0] != 0));
        degq = 31 - __clz(__ballot_sync(FULL, c1[NR - 1] != 0));
      }
      uint64_t xq[NR];
#pragma unroll
      for (int r = 0; r < NR; r++) xq[r] = shoup_pre(x[r], M);
      const int deg = degp > degq ? degp : degq;
      for (int k = deg; k >= 0; k--) {
        const uint64_t pk = __shfl_sync(FULL, c1[0], k);
        const uint64_t qk = __shfl_sync(FULL, c1[NR - 1], NR == 1 ? 16 + k : k);
#pragma unroll
        for (int r = 0; r < NR; r++) {
          pv[r] = add_mod(canon(shoup_lazy(pv[r], x[r], xq[r], M), M), pk, M);
          qv[r] = add_mod(canon(shoup_lazy(qv[r], x[r], xq[r], M), M), qk, M);
        }
      }
      const uint64_t q0 = __shfl_sync(FULL, qv[0], 0);   // Q(c_0)
      if (q0 == 0) {
        if (lane == 0) atomicOr(status, ST_POLE);
        ok = false;
      } else if (degp > dN || degq > dD) {
        if (lane == 0) atomicOr(status, ST_DEGREE);
        ok = false;
      } else if (lane == 0) {
        q0s[warp] = q0;
      }
    }
  }
  __syncthreads();
  if (warp == 0) q0s[lane] = warp_batch_inverse(q0s[lane], M);
  __syncthreads();
  if (!ok) return;
  const uint64_t s = mul_mod(q0s[warp], canon(dprev[i], M), M);
#pragma unroll
  for (int r = 0; r < NR; r++) {
    const int t = lane + 32 * r;
    if (i < TN && t <= dN) bN[(int64_t)t * ldN + i] = mul_mod(s, pv[r], M);
    if (i < TD && t <= dD) bD[(int64_t)t * ldD + i] = mul_mod(s, qv[r], M);
  }
}

// Multiply n coefficients by c (used for the final normalisation).
__global__ void k_scale(int64_t n, uint64_t* __restrict__ a, const uint64_t* __restrict__ c, Mod M) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = mul_mod(a[i], *c, M);
}
__global__ void k_inv1(const uint64_t* __restrict__ a, uint64_t* __restrict__ out, Mod M, uint32_t* status) {
  const uint64_t x = *a;
  if (x == 0) atomicOr(status, ST_ZERO_DEN);
  *out = inv_mod(x, M);
}
void launch_normalise(int64_t n1, uint64_t* a1, int64_t n2, uint64_t* a2, const uint64_t* pivot, uint64_t* tmp,
                      const Mod& M, uint32_t* status, cudaStream_t st) {
  { k_inv1<<<1, 1, 0, st>>>(pivot, tmp, M, status); note_launch(); }
  if (n1 > 0) { k_scale<<<cdiv(n1, 256), 256, 0, st>>>(n1, a1, tmp, M); note_launch(); }
  if (n2 > 0) { k_scale<<<cdiv(n2, 256), 256, 0, st>>>(n2, a2, tmp, M); note_launch(); }
}

// Enqueues the per-probe Thiele + balancing of the values fvals / fdens
// (fdens null: fvals), n <= 64 samples.  A zero of fdens sets ST_POLE.
void launch_thiele_balance(int64_t Tmax, int n, const uint64_t* xs, const uint64_t* fvals, const uint64_t* fdens,
                           int64_t ldf, const uint64_t* dprev, int dN, int dD, int64_t TN, int64_t TD, const Mod& M,
                           uint64_t* bN, int64_t ldN, uint64_t* bD, int64_t ldD, uint32_t* status, cudaStream_t st) {
  if (Tmax <= 0) return;
  const unsigned grid = cdiv(Tmax, kThieleWarps);
  if (n <= 32)
    k_thiele_balance<1><<<grid, 32 * kThieleWarps, 0, st>>>(Tmax, n, xs, fvals, fdens, ldf, dprev, dN, dD, TN, TD, M,
                                                            bN, ldN, bD, ldD, status);
  else
    k_thiele_balance<2><<<grid, 32 * kThieleWarps, 0, st>>>(Tmax, n, xs, fvals, fdens, ldf, dprev, dN, dD, TN, TD, M,
                                                            bN, ldN, bD, ldD, status);
  note_launch();
}

}  // namespace zr
