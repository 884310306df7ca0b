// zr_eval.cu -- sparse black-box evaluator (Sec. 2.2, balanced coefficient
// preparation: base values raised to powers and substituted into the
// polynomial; one value per thread, terms split over threads, partial sums
// added).
//
// The Zippel probes of f for new variable k are the values
//     out[s][i] = f(y^(i+off), c_s, z_{k+1..})
//               = sum_t w_{t,s} u_t^(i+off),
//     u_t = prod_{m<k} y_m^{e_{t,m}},  w_{t,s} = coef_t c_s^{e_{t,k}} prod_{m>k} z_m^{e_{t,m}}.
// Terms with equal u are merged first (their w are added), which turns the
// evaluation into a transposed Vandermonde product over the G distinct u.
// The kernel (k_eval_ring) tiles it: a CTA owns 32 consecutive i and walks a
// range of groups in chunks of 32; for each chunk a producer warp fills the
// power table X[t][g] = u_g^(I0+off+t) in shared memory (the paper's power
// table, Sec. 2.2: a starting power, then one multiply by u_g per entry) and
// consumer warps accumulate sum_g w_{g,s} X[t][g] for their columns with the
// deferred multiply-accumulate.
#include <cuda_runtime.h>

#include <cmath>

#include <algorithm>

#include "zr_internal.h"
#include "zr_launch.cuh"
#include "zr_ring.cuh"

namespace zr {

static inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }
static constexpr uint64_t kEmpty = ~0ull;

__device__ __forceinline__ uint64_t ehash(uint64_t x) {
  x ^= x >> 31;
  x *= 0x9E3779B97F4A7C15ull;
  return x ^ (x >> 29);
}

// ---- groups --------------------------------------------------------------------
//
// Terms with equal anchor value are numbered and listed in five short launches
// (each bound by its latency, 2.5 to 4 us; numbering the groups by scans over
// the hash slots and the group sizes took fourteen): the inserting thread of a
// hash slot takes the group's number from a counter, the sizes take places in
// the list from another.  The numbering and the places vary from run to run;
// the sums over a group's terms and over the groups are exact, so the probes
// do not.

// The scratch's initial state and the power tables: blocks below `rows` write
// base[r]^e, e < 256, of row r (the k anchors, the nv rest values, the S
// samples); the others empty the hash table and zero the counts.
__global__ void k_eval_init(const uint64_t* __restrict__ y, int k, const uint64_t* __restrict__ z, int nz,
                            const uint64_t* __restrict__ cs, int S, Mod M, uint64_t* __restrict__ tabY,
                            uint64_t* __restrict__ tabZ, uint64_t* __restrict__ tabC, uint64_t* __restrict__ htab,
                            uint64_t H, int32_t* __restrict__ cnt, int64_t Tn, int64_t* __restrict__ Gdev,
                            int64_t* __restrict__ total) {
  pdl_enter();
  const int rows = k + nz + S;
  if (blockIdx.x < rows) {
    int r = blockIdx.x;
    const uint64_t* b = y;
    uint64_t* tab = tabY;
    if (r >= k + nz) r -= k + nz, b = cs, tab = tabC;
    else if (r >= k) r -= k, b = z, tab = tabZ;
    tab[(int64_t)r * kPowTab + threadIdx.x] = pow_mod(canon(b[r], M), (uint64_t)threadIdx.x, M);
    return;
  }
  const uint64_t n = (uint64_t)(gridDim.x - rows) * blockDim.x;
  const uint64_t at = (uint64_t)(blockIdx.x - rows) * blockDim.x + threadIdx.x;
  for (uint64_t i = at; i < H; i += n) htab[i] = kEmpty;
  for (uint64_t i = at; i < (uint64_t)Tn; i += n) cnt[i] = 0;
  if (at == 0) *Gdev = 0, *total = 0;
}

// per term: its anchor value u_t, its weight without the new variable,
// a_t = coef_t prod_{m>k} z_m^{e_{t,m}}, and its hash slot; the thread that
// fills a slot numbers the group
__global__ void __launch_bounds__(256) k_eval_terms(int64_t Tf, int nv, const uint8_t* __restrict__ exps, const uint64_t* __restrict__ coef,
                             int k, const uint64_t* __restrict__ tabY, const uint64_t* __restrict__ tabZ, Mod M,
                             uint64_t* __restrict__ a, uint64_t* htab, uint64_t hmask, int32_t* __restrict__ gid,
                             uint64_t* __restrict__ U, int64_t* Gdev, uint32_t* __restrict__ slot, uint32_t* status) {
  pdl_enter();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint64_t uu = 1, found = ~0ull;
  bool won = false;
  if (t < Tf) {
    const uint8_t* e = exps + t * nv;
    for (int m = 0; m < k; m++) uu = mul_mod(uu, tabY[m * kPowTab + e[m]], M);
    uint64_t c = coef[t];
    if (c >= M.p) c -= M.p;
    for (int m = k + 1; m < nv; m++) c = mul_mod(c, tabZ[m * kPowTab + e[m]], M);
    a[t] = c;
    // insert the key; equal keys share a slot
    uint64_t idx = ehash(uu) & hmask;
    for (uint64_t probe = 0; probe <= hmask; probe++) {
      unsigned long long prev = atomicCAS((unsigned long long*)&htab[idx], (unsigned long long)kEmpty,
                                          (unsigned long long)uu);
      won = prev == kEmpty;
      if (won || prev == uu) {
        found = idx;
        break;
      }
      idx = (idx + 1) & hmask;
    }
    slot[t] = (uint32_t)found;
    if (found == ~0ull) atomicOr(status, ST_HASH_FULL);
  }
  // a block's new groups take their numbers with one addition (one per warp
  // took 0.6 ms for the 2^20 groups of 9.4 million terms)
  __shared__ int warp_new[8];
  __shared__ unsigned long long first;
  const unsigned winners = __ballot_sync(0xffffffffu, won);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) warp_new[warp] = __popc(winners);
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < 8; w++) {
    if (w < warp) before += warp_new[w];
    total += warp_new[w];
  }
  if (threadIdx.x == 0 && total) first = atomicAdd((unsigned long long*)Gdev, (unsigned long long)total);
  __syncthreads();
  if (won) {
    const int32_t g = (int32_t)(first + before + __popc(winners & ((1u << lane) - 1)));
    gid[found] = g;
    U[g] = uu;
  }
}

// tg[t] = the term's group (over its hash slot), tp[t] = its place in the
// group, cnt[g] = the group's size.
__global__ void k_eval_count(int64_t Tf, const int32_t* __restrict__ gid, int32_t* __restrict__ cnt,
                             int32_t* __restrict__ tg, int32_t* __restrict__ tp) {
  pdl_enter();
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= Tf) return;
  const uint32_t slot = (uint32_t)tg[t];
  const int g = slot == ~0u ? -1 : gid[slot];
  tg[t] = g;
  if (g >= 0) tp[t] = atomicAdd(&cnt[g], 1);
}
// each group's first place in the list: the sizes of a warp's groups added up
// by shuffles, one atomic per warp
__global__ void k_eval_start(const int64_t* __restrict__ Gdev, const int32_t* __restrict__ cnt, int64_t* total,
                             int64_t* __restrict__ start) {
  pdl_enter();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, G = *Gdev;
  const int lane = threadIdx.x & 31;
  if (g - lane >= G) return;
  const int64_t n = g < G ? cnt[g] : 0;
  int64_t incl = n;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int64_t x = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += x;
  }
  int64_t base = 0;
  if (lane == 31) base = (int64_t)atomicAdd((unsigned long long*)total, (unsigned long long)incl);
  base = __shfl_sync(0xffffffffu, base, 31);
  if (g < G) start[g] = base + incl - n;
}
__global__ void k_eval_scatter(int64_t Tf, const int32_t* __restrict__ tg, const int32_t* __restrict__ tp,
                               const int64_t* __restrict__ start, int64_t* __restrict__ order) {
  pdl_enter();
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= Tf || tg[t] < 0) return;
  order[start[tg[t]] + tp[t]] = t;
}

// The merged weights W[g][s] = sum over group g's terms of a_t c_s^{e_{t,k}},
// s < S <= 256, handed to store(g, j, value) for the row entries j < rw,
// column(j) the entry's column s (negative: padding, zero).
//
// Many or short groups: a thread per entry.  Few long ones (n >= 8 terms on
// average, at most 80 n groups: the early variables of a reconstruction): a
// block per group, its terms staged 256 at a time, a warp every eighth of them,
// lanes the columns; a thread per entry then runs through hundreds of dependent
// gathers.  A block's round takes about as long as 20 of those, and 1216 blocks
// run at a time.  Whole calls, block against thread per entry, S = 1 .. 21: 32
// terms in 1200 groups 59 against 70 us, in 10000 136 against 110; 255 in 1200
// 100 against 158, in 16000 600 against 590; 64 in 62500 840 against 610.
constexpr int kWeightThreads = 256;
template <class Column, class Store>
__device__ __forceinline__ void group_weights(int64_t G, int64_t Tf, int S, int rw, const int64_t* __restrict__ start,
                                              const int32_t* __restrict__ cnt, const int64_t* __restrict__ order,
                                              const uint64_t* __restrict__ a, const uint8_t* __restrict__ exps, int nv,
                                              int k, const uint64_t* __restrict__ tabC, const Mod& M, Column column,
                                              Store store) {
  if (G * 8 <= Tf && G * G <= 80 * Tf) {
    __shared__ uint64_t sa[kWeightThreads], vals[256], red[kWeightThreads / 32][32];
    __shared__ uint8_t se[kWeightThreads];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t g = blockIdx.x; g < G; g += gridDim.x) {
      const int64_t r0 = start[g], n = cnt[g];
      for (int s0 = 0; s0 < S; s0 += 32) {
        const int s = s0 + lane;
        const uint64_t* cs = tabC + (int64_t)s * kPowTab;
        Acc8 acc{0, 0, 0, 0, 0, 0, 0, 0};
        for (int64_t x0 = 0; x0 < n; x0 += kWeightThreads) {
          const int m = n - x0 < kWeightThreads ? (int)(n - x0) : kWeightThreads;
          __syncthreads();
          if ((int)threadIdx.x < m) {
            const int64_t t = order[r0 + x0 + threadIdx.x];
            sa[threadIdx.x] = a[t];
            se[threadIdx.x] = exps[t * nv + k];
          }
          __syncthreads();
          if (s < S) {
#pragma unroll 4
            for (int x = warp; x < m; x += kWeightThreads / 32) {
              const uint64_t at = sa[x], w = cs[se[x]];
              mac8(acc, lo32(at), hi32(at), lo32(w), hi32(w));
            }
          }
        }
        red[warp][lane] = acc8_value(acc, M);
        __syncthreads();
        if (warp == 0 && s < S) {
          uint64_t r = 0;
#pragma unroll
          for (int w = 0; w < kWeightThreads / 32; w++) r = add_mod(r, red[w][lane], M);
          vals[s] = r;
        }
      }
      __syncthreads();
      for (int j = threadIdx.x; j < rw; j += kWeightThreads) {
        const int s = column(j);
        store(g, j, s < 0 ? 0 : vals[s]);
      }
      __syncthreads();
    }
    return;
  }
  const int64_t stride = (int64_t)gridDim.x * kWeightThreads;
  for (int64_t idx = (int64_t)blockIdx.x * kWeightThreads + threadIdx.x; idx < G * rw; idx += stride) {
    const int64_t g = idx / rw;
    const int j = (int)(idx - g * rw), s = column(j);
    uint64_t r = 0;
    if (s >= 0) {
      Acc8 acc{0, 0, 0, 0, 0, 0, 0, 0};
      const uint64_t* cs = tabC + (int64_t)s * kPowTab;
      const int64_t r0 = start[g], n = cnt[g];
      for (int64_t x = 0; x < n; x++) {
        const int64_t t = order[r0 + x];
        const uint64_t at = a[t], w = cs[exps[t * nv + k]];
        mac8(acc, lo32(at), hi32(at), lo32(w), hi32(w));
      }
      r = acc8_value(acc, M);
    }
    store(g, j, r);
  }
}

// Blocks of the kernels above for at most G groups of Tf terms: a thread per
// entry of rw a group, or a block per group where that is the choice (at most
// Tf / 8 groups), eight blocks an SM at most (both ways stride the grid).
// Sized by the entries alone, a block walked up to 256 groups in sequence: 0.12
// ms of a probe set of 16384 groups of 16 terms at S = 1.
static unsigned weight_blocks(const zr_ctx* ctx, int64_t G, int64_t Tf, int rw) {
  const int64_t want = std::max<int64_t>(cdiv(G * rw, kWeightThreads), std::min(G, Tf / 8));
  return (unsigned)std::min<int64_t>(want, 8ll * (ctx->sms ? ctx->sms : 152));
}

// Where the weights of the matrix-vector kernel live: column block b
// (columns s0[b] .. s0[b] + 63) holds, per group, its row of bw[b] words laid
// out as the kernel stages it ([consumer][column], pairs padded with zero).
struct RingLayout {
  int nb;
  int cg[4], cgp[4], bw[4];
  int64_t off[4];   // word offset of block b (G bw[b'] words per block before it)
};

// finalize, for the G groups counted on the device (G <= Tn, the stride of
// the tables): the merged weights as residues in the ring layout, zero in
// the padding; the squares table UP[a][g] = u_g^(2^a), a < nsq, with its
// Shoup quotients UPq; the quotients Uq[g] of u_g.
__global__ void __launch_bounds__(kWeightThreads)
    k_eval_finalize(const int64_t* __restrict__ Gdev, int64_t Tn, int S, const int64_t* __restrict__ start,
                    const int32_t* __restrict__ cnt, const int64_t* __restrict__ order, const uint64_t* __restrict__ a,
                    const uint8_t* __restrict__ exps, int nv, int k, const uint64_t* __restrict__ tabC,
                    const uint64_t* __restrict__ U, Mod M, RingLayout L, int rw, int nsq, uint64_t* __restrict__ Wr,
                    uint64_t* __restrict__ UP, uint64_t* __restrict__ UPq, uint64_t* __restrict__ Uq) {
  pdl_enter();
  const int64_t G = *Gdev;
  // entry j of a group's rows: block b, consumer q, column c
  auto place = [&](int j, int& b) {
    b = 0;
    while (j >= L.bw[b]) j -= L.bw[b++];
    return j;
  };
  auto column = [&](int j) {
    int b;
    j = place(j, b);
    const int q = j / L.cgp[b], c = j - q * L.cgp[b], s = 64 * b + q * L.cg[b] + c;
    return c < L.cg[b] && s < S ? s : -1;
  };
  group_weights(G, Tn, S, rw, start, cnt, order, a, exps, nv, k, tabC, M, column, [&](int64_t g, int j, uint64_t r) {
    int b;
    j = place(j, b);
    Wr[L.off[b] + g * L.bw[b] + j] = r;
  });
  // a grid-stride loop: the launch is sized for the SMs, the work for G
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < G; idx += stride) {
    uint64_t x = U[idx];
    for (int e = 0; e < nsq; e++) {
      const uint64_t xq = shoup_pre(x, M);
      if (e == 0) Uq[idx] = xq;
      UP[e * Tn + idx] = x;
      UPq[e * Tn + idx] = xq;
      x = mul_mod(x, x, M);
    }
  }
}

// The matrix-vector product out[s][i] = sum_g W[g][s] u_g^(i+off),
// warp-specialised like the solve.  A CTA owns a tile of 32 consecutive i and
// a range of groups, walked in chunks of 32 through a ring of shared-memory
// stages:
//   warp 0 (producer)     lane = group: stages the chunk's weights with
//                         cp.async and fills the power table
//                         X[t][g] = u_g^(I0+off+t), t < 32, starting from
//                         u_g^(I0+off) (a product of squares u_g^(2^a) over
//                         the set bits of the exponent) and running a Shoup
//                         multiply by u_g along t (the paper's power table,
//                         Sec. 2.2, one row per group);
//   warps 1.. (consumers) lane = i: CG columns each, acc_s += X[i][g] W[g][s]
//                         in 160-bit accumulators, reduced once.
// Every power is computed once and read by all consumer warps.  Columns
// beyond 64 run as further launches over the next column block.
template <int CG, int G>
struct EvalRingCfg {
  static constexpr int TI = 32;               // i per CTA: one per consumer lane
  static constexpr int GC = 32;               // groups per chunk: one per producer lane
  static constexpr int NST = 4;               // ring stages
  static constexpr int XP = GC + 1;           // padded row of X: the consumers read it across rows
  static constexpr int CGP = (CG + 1) & ~1;   // a consumer's columns, padded to pairs
  static constexpr int BW = G * CGP;          // staged weight row width
  static constexpr int NT = 32 * (1 + G);
  static constexpr int REG = CG <= 2 ? 72 : (CG <= 3 ? 80 : (CG <= 4 ? 104 : (CG <= 6 ? 136 : 168)));
  static constexpr int FIT = 65536 / (NT * REG);
  static constexpr int MINB = FIT < 1 ? 1 : (FIT > 6 ? 6 : FIT);
  static constexpr size_t XB = sizeof(uint64_t) * NST * TI * XP;
  static constexpr size_t WB = sizeof(uint64_t) * NST * GC * BW;
  static constexpr size_t SMEM = XB + WB + sizeof(uint64_t) * 2 * NST;
};

template <int CG, int G>
__global__ void __launch_bounds__(EvalRingCfg<CG, G>::NT, EvalRingCfg<CG, G>::MINB)
    k_eval_ring(int64_t T, int S, int s0, int offset, const int64_t* __restrict__ Gdev, int64_t NG, int gsplit,
                const uint64_t* __restrict__ UP,
                const uint64_t* __restrict__ UPq, const uint64_t* __restrict__ U, const uint64_t* __restrict__ Uq,
                const uint64_t* __restrict__ Wb, Mod M, uint64_t* __restrict__ out, int64_t ldo,
                uint64_t* __restrict__ partial, uint32_t* __restrict__ status) {
  using C = EvalRingCfg<CG, G>;
  extern __shared__ __align__(16) unsigned char smraw[];
  uint64_t(*xs)[C::TI][C::XP] = reinterpret_cast<uint64_t(*)[C::TI][C::XP]>(smraw);
  uint64_t(*ws)[C::GC][C::BW] = reinterpret_cast<uint64_t(*)[C::GC][C::BW]>(smraw + C::XB);
  uint64_t* full = reinterpret_cast<uint64_t*>(smraw + C::XB + C::WB);
  uint64_t* empty = full + C::NST;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int SC = (S - s0) < G * CG ? S - s0 : G * CG;   // columns of this launch
  pdl_enter();
  if (tid == 0)
    for (int st = 0; st < C::NST; st++) {
      mbar_init(&full[st], 32);
      mbar_init(&empty[st], G);
    }
  __syncthreads();
  const int64_t I0 = (int64_t)blockIdx.x * C::TI;
  const int split = blockIdx.y;
  const int64_t G_ = *Gdev;   // groups; NG (>= G_) is the stride of the squares table
  const int64_t glo = G_ * split / gsplit, ghi = G_ * (split + 1) / gsplit;
  const int nch = (int)((ghi - glo + C::GC - 1) / C::GC);

  if (warp == 0) {
    // ---- producer warp
    const uint32_t emask = (uint32_t)(I0 + offset);   // the exponent E < 2^32 of t = 0
    for (int c = 0; c < nch; c++) {
      const int st = c % C::NST;
      const uint32_t ph = (c / C::NST) & 1;
      if (c >= C::NST && !mbar_wait(&empty[st], ph ^ 1)) {
        atomicOr(status, ST_TIMEOUT);
        cp_async_wait<0>();
        return;
      }
      const int64_t gc = glo + (int64_t)c * C::GC;
      const int gn = (ghi - gc) < C::GC ? (int)(ghi - gc) : C::GC;
      // weights of the chunk: gn consecutive rows, already in the staged layout
      {
        const uint64_t* src = Wb + gc * C::BW;
        uint64_t* dst = &ws[st][0][0];
        const int n16 = gn * C::BW / 2;
        for (int q = lane; q < n16; q += 32) cp_async16(dst + 2 * q, src + 2 * q);
      }
      cp_async_commit();
      if (lane < gn) {
        const int64_t gg = gc + lane;
        const uint64_t u = __ldg(U + gg), uq = __ldg(Uq + gg);
        const uint64_t u16 = __ldg(UP + 4 * NG + gg), u16q = __ldg(UPq + 4 * NG + gg);
        // u_g^E: a Shoup product of the squares of E's set bits, their loads
        // issued eight at a time
        uint64_t x = 1;
        for (uint32_t m = emask; m;) {
          uint64_t f[8], fq[8];
          bool have[8];
#pragma unroll
          for (int q = 0; q < 8; q++) {
            have[q] = m != 0;
            const int a = have[q] ? __ffs(m) - 1 : 0;
            m &= m - 1;
            f[q] = have[q] ? __ldg(UP + (int64_t)a * NG + gg) : 0;
            fq[q] = have[q] ? __ldg(UPq + (int64_t)a * NG + gg) : 0;
          }
#pragma unroll
          for (int q = 0; q < 8; q++)
            if (have[q]) x = shoup_lazy(x, f[q], fq[q], M);
        }
        x = canon(x, M);
        // two interleaved chains, t < 16 and t >= 16, one Shoup multiply by u per step
        uint64_t xb = canon(shoup_lazy(x, u16, u16q, M), M);
#pragma unroll 4
        for (int t = 0; t < C::TI / 2; t++) {
          xs[st][t][lane] = x;
          xs[st][t + C::TI / 2][lane] = xb;
          x = canon(shoup_lazy(x, u, uq, M), M);
          xb = canon(shoup_lazy(xb, u, uq, M), M);
        }
      }
      cp_async_wait<0>();
      mbar_arrive(&full[st]);
    }
    return;
  }
  // ---- consumer w: columns s0 + w CG .. s0 + w CG + CG - 1
  const int w = warp - 1;
  Acc8 acc[CG];
#pragma unroll
  for (int q = 0; q < CG; q++) acc[q] = Acc8{0, 0, 0, 0, 0, 0, 0, 0};
  for (int c = 0; c < nch; c++) {
    const int st = c % C::NST;
    const uint32_t ph = (c / C::NST) & 1;
    if (!mbar_wait(&full[st], ph)) {
      atomicOr(status, ST_TIMEOUT);
      return;
    }
    const int64_t gc = glo + (int64_t)c * C::GC;
    const int gn = (ghi - gc) < C::GC ? (int)(ghi - gc) : C::GC;
    const uint64_t* xrow = xs[st][lane];
    if (gn == C::GC) {
#pragma unroll
      for (int g = 0; g < C::GC; g++) {
        const uint64_t x = xrow[g];
        const uint32_t x0 = lo32(x), x1 = hi32(x);
        const uint64_t* row = &ws[st][g][w * C::CGP];
#pragma unroll
        for (int q = 0; q + 1 < CG; q += 2) {
          const uint4 v = *reinterpret_cast<const uint4*>(row + q);
          mac8(acc[q], x0, x1, v.x, v.y);
          mac8(acc[q + 1], x0, x1, v.z, v.w);
        }
        if (CG & 1) {
          const uint2 v = *reinterpret_cast<const uint2*>(row + CG - 1);
          mac8(acc[CG - 1], x0, x1, v.x, v.y);
        }
      }
    } else {
#pragma unroll 1
      for (int g = 0; g < gn; g++) {
        const uint64_t x = xrow[g];
        const uint32_t x0 = lo32(x), x1 = hi32(x);
        const uint64_t* row = &ws[st][g][w * C::CGP];
#pragma unroll
        for (int q = 0; q + 1 < CG; q += 2) {
          const uint4 v = *reinterpret_cast<const uint4*>(row + q);
          mac8(acc[q], x0, x1, v.x, v.y);
          mac8(acc[q + 1], x0, x1, v.z, v.w);
        }
        if (CG & 1) {
          const uint2 v = *reinterpret_cast<const uint2*>(row + CG - 1);
          mac8(acc[CG - 1], x0, x1, v.x, v.y);
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[st]);
  }
  const int64_t i = I0 + lane;
  if (i >= T) return;
#pragma unroll
  for (int q = 0; q < CG; q++) {
    const int sidx = s0 + w * CG + q;
    if (w * CG + q >= SC) continue;
    const uint64_t r = acc8_value(acc[q], M);
    if (gsplit == 1) out[(int64_t)sidx * ldo + i] = r;
    else partial[((int64_t)split * S + sidx) * T + i] = r;
  }
}

// out = sum of the group splits' partial sums (with Gdev: of the splits the
// tensor-core kernel used)
__global__ void k_eval_combine(int64_t T, int S, int gsplit, const int64_t* __restrict__ Gdev,
                               const uint64_t* __restrict__ partial, Mod M, uint64_t* __restrict__ out, int64_t ldo) {
  pdl_enter();
  if (Gdev) gsplit = eval_tc_splits(gsplit, *Gdev);
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= T * S) return;
  int s = (int)(idx / T);
  int64_t i = idx - (int64_t)s * T;
  uint64_t r = 0;
  for (int q0 = 0; q0 < gsplit; q0 += 8) {   // eight loads in flight
    uint64_t x[8];
#pragma unroll
    for (int q = 0; q < 8; q++) x[q] = q0 + q < gsplit ? partial[((int64_t)(q0 + q) * S + s) * T + i] : 0;
#pragma unroll
    for (int q = 0; q < 8; q++) r = add_mod(r, x[q], M);
  }
  out[(int64_t)s * ldo + i] = r;
}

template <int CG, int G>
static int ring_occupancy_t() {
  using C = EvalRingCfg<CG, G>;
  static DeviceValue occ;
  return occ.get([] {
    cudaFuncSetAttribute(k_eval_ring<CG, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_eval_ring<CG, G>, C::NT, C::SMEM) != cudaSuccess || n < 1)
      n = 1;
    return n;
  });
}

// A grid that leaves slots of the GPU empty has to be spread over the SMs: as a
// programmatic dependent launch its CTAs come in while the kernel before it
// drains, several to the first SMs that have room (250000 groups, T = 64, S = 4
// / 21: 1213 / 1603 us against 593 / 745).  Short ranges of groups are launched
// early all the same, 3 us less of 50 to 60 (at most 2^17 terms times columns;
// the sides cross between 2^14 and 2^17, the later the more terms a group has).
constexpr int64_t kRingSpread = 1 << 17;
template <int CG, int G>
static void launch_ring_t(int sms, int64_t T, int S, int s0, int offset, const int64_t* Gdev, int64_t NG, int gsplit,
                          const uint64_t* UP,
                          const uint64_t* UPq, const uint64_t* U, const uint64_t* Uq, const uint64_t* Wb,
                          const Mod& M, uint64_t* out, int64_t ldo, uint64_t* partial, uint32_t* status,
                          cudaStream_t st) {
  using C = EvalRingCfg<CG, G>;
  const int occ = ring_occupancy_t<CG, G>();   // also sets the shared-memory attribute
  const int SC = S - s0 < G * CG ? S - s0 : G * CG;   // columns of this launch
  dim3 grid(cdiv(T, C::TI), gsplit);
  if ((int64_t)grid.x * gsplit < (int64_t)sms * occ && NG * SC > kRingSpread)
    k_eval_ring<CG, G><<<grid, C::NT, C::SMEM, st>>>(T, S, s0, offset, Gdev, NG, gsplit, UP, UPq, U, Uq, Wb, M, out,
                                                     ldo, partial, status);
  else
    launch_k(k_eval_ring<CG, G>, grid, dim3(C::NT), C::SMEM, st, T, S, s0, offset, Gdev, NG, gsplit, UP, UPq, U, Uq, Wb,
             M, out, ldo, partial, status);
  note_launch();
}

// The instances: columns per consumer and consumer warps for a block of
// SC <= 64 columns (at most 8 consumers).
using RingLaunch = void (*)(int, int64_t, int, int, int, const int64_t*, int64_t, int, const uint64_t*, const uint64_t*,
                            const uint64_t*,
                            const uint64_t*, const uint64_t*, const Mod&, uint64_t*, int64_t, uint64_t*, uint32_t*,
                            cudaStream_t);
struct RingInst {
  int cg, g;
  RingLaunch launch;
  int (*occupancy)();
};
#define ZR_RING(CGV, GV) {CGV, GV, launch_ring_t<CGV, GV>, ring_occupancy_t<CGV, GV>}
static const RingInst kRing[] = {ZR_RING(1, 1), ZR_RING(2, 1), ZR_RING(3, 1), ZR_RING(3, 2), ZR_RING(3, 3),
                                 ZR_RING(3, 4), ZR_RING(3, 5), ZR_RING(3, 6), ZR_RING(3, 7), ZR_RING(3, 8),
                                 ZR_RING(4, 7), ZR_RING(4, 8), ZR_RING(6, 6), ZR_RING(6, 7), ZR_RING(6, 8),
                                 ZR_RING(8, 7), ZR_RING(8, 8)};
#undef ZR_RING

static const RingInst* ring_inst(int SC) {
  const int cg = SC <= 2 ? SC : (SC <= 24 ? 3 : (SC <= 32 ? 4 : (SC <= 48 ? 6 : 8)));
  const int g = (SC + cg - 1) / cg;
  for (const RingInst& r : kRing)
    if (r.cg == cg && r.g == g) return &r;
  return nullptr;
}

// The weight layout for S columns over G groups (blocks of 64 columns).
static RingLayout ring_layout(int S, int64_t G) {
  RingLayout L{};
  int64_t off = 0;
  for (int s0 = 0; s0 < S; s0 += 64) {
    const RingInst* r = ring_inst(S - s0 < 64 ? S - s0 : 64);
    const int b = L.nb++;
    L.cg[b] = r->cg;
    L.cgp[b] = (r->cg + 1) & ~1;
    L.bw[b] = r->g * L.cgp[b];
    L.off[b] = off;
    off += G * L.bw[b];
  }
  return L;
}
static int64_t ring_words(int S, int64_t G) {
  const RingLayout L = ring_layout(S, G);
  return L.off[L.nb - 1] + G * L.bw[L.nb - 1];
}

static void launch_ring(const zr_ctx* ctx, int64_t T, int S, int offset, const int64_t* Gdev, int64_t NG, int gsplit, const uint64_t* UP,
                        const uint64_t* UPq, const uint64_t* U, const uint64_t* Uq, const uint64_t* Wr,
                        const RingLayout& L, const Mod& M, uint64_t* out, int64_t ldo, uint64_t* partial,
                        uint32_t* status, cudaStream_t st) {
  for (int b = 0; b < L.nb; b++) {
    const int s0 = 64 * b;
    const RingInst* r = ring_inst(S - s0 < 64 ? S - s0 : 64);
    r->launch(ctx->sms ? ctx->sms : 152, T, S, s0, offset, Gdev, NG, gsplit, UP, UPq, U, Uq, Wr + L.off[b], M, out, ldo, partial, status, st);
  }
}

// Group splits: the smallest count that gives at least two waves of CTAs
// with the last one at least 97% full (else the best fill up to 32 splits),
// keeping 64 or more groups per split.
static int eval_gsplit(const zr_ctx* ctx, int64_t T, int S, int64_t Tf) {
  const int64_t ctas = (int64_t)cdiv(T, 32);
  const int64_t slots = (int64_t)(ctx && ctx->sms ? ctx->sms : 152) * ring_inst(S < 64 ? S : 64)->occupancy();
  if (ctas >= 8 * slots) return 1;
  int best = 1;
  double best_fill = 0;
  for (int gs = 1; gs <= 32; gs++) {
    if (gs > 1 && Tf / gs < 64) break;
    const double waves = (double)(ctas * gs) / (double)slots;
    const double fill = waves / std::ceil(waves);
    if (waves >= 2 && fill >= 0.97) return gs;
    if (fill > best_fill + 1e-9) {
      best = gs;
      best_fill = fill;
    }
  }
  return best;
}

// Workspace bytes the evaluator needs for (f, S, T).
size_t probes_ws_need(const zr_ctx* ctx, const zr_poly* f, int k, int S, int64_t T);

zr_status probes_impl(zr_ctx* ctx, const zr_poly* f, int k, const uint64_t* y, int S, const uint64_t* samples,
                      const uint64_t* z, int64_t T, int offset, uint64_t* out, int64_t ldo, uint32_t* status,
                      cudaStream_t st, int lane) {
  if (lane < 0 || lane >= zr_ctx::kProbeLanes) {
    zr_status r = ensure_ws(ctx, probes_ws_need(ctx, f, k, S, T), st);
    if (r) return r;
    return probes_enqueue(ctx, f, k, y, S, samples, z, T, offset, out, ldo, status, ctx->ws, st);
  }
  // the lane's own scratch, grown (rarely) after its stream's queued work
  const size_t need = probes_ws_need(ctx, f, k, S, T);
  if (ctx->pl_cap[lane] < need) {
    cudaError_t e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && ctx->pl_ws[lane]) e = cudaFree(ctx->pl_ws[lane]);
    ctx->pl_ws[lane] = nullptr;
    ctx->pl_cap[lane] = 0;
    if (e == cudaSuccess) e = cudaMalloc(&ctx->pl_ws[lane], need + need / 4);
    if (e != cudaSuccess) {
      ctx->pl_ws[lane] = nullptr;
      return cuda_err(ctx, e, "probe lane workspace");
    }
    ctx->pl_cap[lane] = need + need / 4;
  }
  return probes_enqueue(ctx, f, k, y, S, samples, z, T, offset, out, ldo, status, ctx->pl_ws[lane], st,
                        &ctx->pl_fws[lane], &ctx->pl_fcap[lane]);
}

// The evaluator's scratch, carved the same way for sizing and for use.
struct EvalWs {
  uint64_t *tabY, *tabZ, *tabC, *a, *htab, *U, *Wp, *UP, *UPq, *Uq, *partial;
  int64_t *start, *order, *Gdev, *total;
  int32_t *gid, *cnt, *tg, *tp;
  EvalTcWs tc;
};
// The three ways to the same probes: the integer ring kernel, the tensor
// cores, the transposed tree.
enum EvalMethod { EVAL_RING, EVAL_TC, EVAL_TREE };
static EvalMethod eval_method(const zr_ctx* ctx, int64_t T, int64_t Tf, int S) {
  if (use_fast_probes(ctx, T, Tf, S)) return EVAL_TREE;
  return use_tc_probes(T, Tf, S) ? EVAL_TC : EVAL_RING;
}
static EvalWs carve_eval(Carver& cv, const zr_ctx* ctx, int64_t Tf, int nv, int k, int S, int64_t T, int gsplit,
                         EvalMethod method) {
  EvalWs w;
  const bool fast = method == EVAL_TREE;   // the transposed tree has its own workspace
  const int64_t Tn = Tf > 0 ? Tf : 1;
  const uint64_t H = hash_slots(Tn);
  w.tabY = cv.take<uint64_t>((size_t)(k > 0 ? k : 1) * kPowTab);
  w.tabZ = cv.take<uint64_t>((size_t)nv * kPowTab);
  w.tabC = cv.take<uint64_t>((size_t)S * kPowTab);
  w.a = cv.take<uint64_t>(Tn);
  w.htab = cv.take<uint64_t>(H);
  w.gid = cv.take<int32_t>(H);
  w.U = cv.take<uint64_t>(Tn);
  w.cnt = cv.take<int32_t>(Tn);
  w.tg = cv.take<int32_t>(Tn);
  w.tp = cv.take<int32_t>(Tn);
  w.start = cv.take<int64_t>(Tn);
  w.order = cv.take<int64_t>(Tn);
  if (method == EVAL_TC) w.tc = carve_eval_tc(cv, ctx, Tn, S, T);
  // the ring kernel's tables, kept when the tree may fall back to it
  const bool ring = method == EVAL_RING || (fast && (Tn > kFastMaxT || fast_probes_by_groups(ctx, T, Tf, S)));
  const int64_t Tr = ring ? Tn : 1;
  w.Wp = cv.take<uint64_t>((size_t)ring_words(S, Tr));
  w.UP = cv.take<uint64_t>((size_t)Tr * 32);
  w.UPq = cv.take<uint64_t>((size_t)Tr * 32);
  w.Uq = cv.take<uint64_t>(Tr);
  w.partial = cv.take<uint64_t>(Tr > 1 && gsplit > 1 ? (size_t)gsplit * S * (T > 0 ? T : 1) : 1);
  w.Gdev = cv.take<int64_t>(1);
  w.total = cv.take<int64_t>(1);
  return w;
}

// The merged weights in plain layout, W[s ld + g] (ld = 0: G), for the
// transposed tree and the tensor cores, times u_g when the probes start at
// the first power (offset 1); with Wq also the Shoup quotients.
__global__ void __launch_bounds__(kWeightThreads)
    k_eval_weights(const int64_t* __restrict__ Gdev, int64_t ld, int64_t Tf, int S, const int64_t* __restrict__ start, const int32_t* __restrict__ cnt,
                   const int64_t* __restrict__ order, const uint64_t* __restrict__ a, const uint8_t* __restrict__ exps,
                   int nv, int k, const uint64_t* __restrict__ tabC, const uint64_t* __restrict__ U, int offset, Mod M,
                   uint64_t* __restrict__ W, uint64_t* __restrict__ Wq) {
  pdl_enter();
  const int64_t G = *Gdev;
  if (ld == 0) ld = G;
  group_weights(G, Tf, S, S, start, cnt, order, a, exps, nv, k, tabC, M, [](int j) { return j; },
                [&](int64_t g, int s, uint64_t r) {
                  if (offset) r = mul_mod(r, U[g], M);
                  W[(int64_t)s * ld + g] = r;
                  if (Wq) Wq[(int64_t)s * ld + g] = shoup_pre(r, M);
                });
}

// The evaluation itself, with its scratch at `base` (capacity checked by the caller).
zr_status probes_enqueue(zr_ctx* ctx, const zr_poly* f, int k, const uint64_t* y, int S, const uint64_t* samples,
                         const uint64_t* z, int64_t T, int offset, uint64_t* out, int64_t ldo, uint32_t* status,
                         char* base, cudaStream_t st, char** fws, size_t* fcap) {
  if (!fws || !fcap) {
    fws = &ctx->fprobe_ws;
    fcap = &ctx->fprobe_cap;
  }
  const Mod& M = ctx->M;
  const int64_t Tf = f->T;
  const int nv = f->nv;
  const uint64_t H = hash_slots(Tf > 0 ? Tf : 1);
  const int gsplit = eval_gsplit(ctx, T, S, Tf);
  const EvalMethod method = eval_method(ctx, T, Tf, S);
  const bool fast = method == EVAL_TREE;
  Carver cv(base);
  const EvalWs w = carve_eval(cv, ctx, Tf, nv, k, S, T, gsplit, method);

  if (T <= 0) return ZR_OK;
  if (Tf == 0) {
    for (int s = 0; s < S; s++) cudaMemsetAsync(out + (int64_t)s * ldo, 0, sizeof(uint64_t) * T, st);
    return cuda_err(ctx, cudaGetLastError(), "zr_zippel_probes");
  }
  const int64_t Tn = Tf;
  const int nz = z && nv > k + 1 ? nv : 0;
  {
    const int64_t cap = 8ll * (ctx->sms ? ctx->sms : 152);
    const unsigned fill = (unsigned)std::min<int64_t>(cdiv((int64_t)H, kPowTab), cap);
    launch_k(k_eval_init, dim3(k + nz + S + fill), dim3(kPowTab), 0, st, y, k, z, nz, samples, S, M, w.tabY, w.tabZ,
             w.tabC, w.htab, H, w.cnt, Tn, w.Gdev, w.total);
  }
  // groups: the distinct u, numbered as their hash slots fill; then the terms
  // of each group, by a counting sort
  launch_k(k_eval_terms, dim3(cdiv(Tf, 256)), dim3(256), 0, st, Tf, nv, f->exps, f->coef, k, w.tabY, w.tabZ, M, w.a,
           w.htab, H - 1, w.gid, w.U, w.Gdev, (uint32_t*)w.tg, status);
  launch_k(k_eval_count, dim3(cdiv(Tf, 256)), dim3(256), 0, st, Tf, w.gid, w.cnt, w.tg, w.tp);
  launch_k(k_eval_start, dim3(cdiv(Tn, 256)), dim3(256), 0, st, w.Gdev, w.cnt, w.total, w.start);
  launch_k(k_eval_scatter, dim3(cdiv(Tf, 256)), dim3(256), 0, st, Tf, w.tg, w.tp, w.start, w.order);
  note_launches(5);
  // the transposed tree: its sizes follow the group count, read here (the
  // matrix-vector kernel below when there are more than kFastMaxT groups, or
  // too few of them for the tree)
  int64_t G = 0;
  if (fast) {
    cudaError_t e = cudaMemcpyAsync(&G, w.Gdev, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_err(ctx, e, "zr_zippel_probes: group count");
    if (G < 1 || G > Tn) return set_err(ctx, ZR_ERR_CUDA, "zr_zippel_probes: group count out of range");
  }
  if (fast && G <= kFastMaxT && (!fast_probes_by_groups(ctx, T, Tf, S) || use_fast_probes_groups(T, G, S))) {
    cudaError_t e = cudaSuccess;
    const size_t wbytes = (((size_t)S * G * sizeof(uint64_t)) + 255) & ~(size_t)255;
    const size_t need = wbytes + fast_probes_ws_need(G, T, S);
    if (*fcap < need) {
      if (*fws) cudaFree(*fws);
      *fws = nullptr;
      *fcap = 0;
      e = cudaMalloc(fws, need + need / 4);
      if (e != cudaSuccess) {
        *fws = nullptr;
        return cuda_err(ctx, e, "zr_zippel_probes: fast workspace");
      }
      *fcap = need + need / 4;
    }
    uint64_t* W = reinterpret_cast<uint64_t*>(*fws);
    {
      launch_k(k_eval_weights, dim3(weight_blocks(ctx, G, Tn, S)), dim3(kWeightThreads), 0, st, w.Gdev, (int64_t)0,
               Tf, S, w.start, w.cnt, w.order, w.a, f->exps, nv, k, w.tabC, w.U, offset, M, W, (uint64_t*)nullptr);
      note_launch();
    }
    return fast_probes_enqueue(ctx, G, w.U, W, G, S, T, out, ldo, *fws + wbytes, st);
  }
  // the group count stays on the device: the kernels read it, sized for Tf groups
  if (method == EVAL_TC) {
    launch_k(k_eval_weights, dim3(weight_blocks(ctx, Tn, Tn, S)), dim3(kWeightThreads), 0, st, w.Gdev,
             eval_tc_ld(Tn), Tf, S, w.start, w.cnt, w.order, w.a, f->exps, nv, k, w.tabC, w.U, offset, M, w.tc.W, w.tc.Wq);
    note_launch();
    const int64_t slab = eval_tc_slab(Tn, T);
    for (int64_t t0 = 0; t0 < T; t0 += slab) {
      const int64_t Ts = std::min(slab, T - t0);
      launch_eval_tc(ctx, w.tc, w.Gdev, Tn, w.U, S, t0, Ts, out, ldo, status, st);
      if (w.tc.gsplit > 1) {
        launch_k(k_eval_combine, dim3(cdiv(Ts * S, 256)), dim3(256), 0, st, Ts, S, w.tc.gsplit, w.Gdev, w.tc.partial, M,
                 out + t0, ldo);
        note_launch();
      }
    }
    return cuda_err(ctx, cudaGetLastError(), "zr_zippel_probes");
  }
  const RingLayout L = ring_layout(S, Tn);
  int rw = 0;
  for (int b = 0; b < L.nb; b++) rw += L.bw[b];
  {
    // squares up to the largest exponent's top bit, and u^16 for the kernel's
    // second chain
    int nsq = 5;
    while (nsq < 32 && (T + offset) >> nsq) nsq++;
    launch_k(k_eval_finalize, dim3(weight_blocks(ctx, Tn, Tn, rw)), dim3(kWeightThreads), 0, st, w.Gdev, Tn, S,
             w.start, w.cnt, w.order, w.a, f->exps, nv, k, w.tabC, w.U, M, L, rw, nsq, w.Wp, w.UP, w.UPq, w.Uq);
    note_launch();
  }
  launch_ring(ctx, T, S, offset, w.Gdev, Tn, gsplit, w.UP, w.UPq, w.U, w.Uq, w.Wp, L, M, out, ldo, w.partial, status, st);
  if (gsplit > 1) {
    launch_k(k_eval_combine, dim3(cdiv(T * S, 256)), dim3(256), 0, st, T, S, gsplit, (const int64_t*)nullptr, w.partial, M,
             out, ldo);
    note_launch();
  }
  return cuda_err(ctx, cudaGetLastError(), "zr_zippel_probes");
}

size_t probes_ws_need(const zr_ctx* ctx, const zr_poly* f, int k, int S, int64_t T) {
  Carver cv(nullptr);
  carve_eval(cv, ctx, f->T, f->nv, k, S, T, eval_gsplit(ctx, T, S, f->T), eval_method(ctx, T, f->T, S));
  return cv.off;
}

// ---------------------------------------------------------------------------
// f at arbitrary points: a cluster of CTAs per point, terms split over the
// CTAs and threads, partial sums reduced with shuffles (Sec. 2.2's warp sum,
// full-warp mask), then over the cluster through distributed shared memory.
// The point's powers x_m^e, e < 16, and x_m^(16 e) sit in shared memory (the
// power table of Sec. 2.2), so that a term takes at most two products per
// variable.  For the 5000 and 3000 terms and 32 points of a reconstruction's
// step 0 one CTA per point with a power per term and variable took 0.16 ms;
// this takes 0.02 ms (latency of the tables and one or two rounds of terms).
// ---------------------------------------------------------------------------
constexpr int kEvalPtThreads = 256;
constexpr int64_t kEvalPtMany = 1216;
__global__ void __launch_bounds__(kEvalPtThreads)
    k_eval_points(int64_t Tf, int nv, int cl, const uint8_t* __restrict__ exps, const uint64_t* __restrict__ coef,
                  const uint64_t* __restrict__ pts, Mod M, uint64_t* __restrict__ out) {
  __shared__ uint64_t tab[kMaxVars][32];         // [m][e]: x^e, [m][16 + e]: x^(16 e)
  __shared__ uint64_t red[kEvalPtThreads / 32];
  __shared__ uint64_t part[8];                   // the cluster's partial sums (CTA 0's copy is used)
  pdl_enter();
  const int64_t pt = blockIdx.x / cl;
  const int rank = (int)(blockIdx.x - pt * cl);
  // every CTA of the cluster has started before another writes to its memory
  if (cl > 1) asm volatile("barrier.cluster.arrive;" ::: "memory");
  for (int i = threadIdx.x; i < 32 * nv; i += kEvalPtThreads) {
    const int m = i >> 5, e = i & 31;
    tab[m][e] = pow_mod(canon(pts[pt * nv + m], M), e < 16 ? e : (uint64_t)(e - 16) * 16, M);
  }
  __syncthreads();
  uint64_t sum = 0;
  for (int64_t t = (int64_t)rank * kEvalPtThreads + threadIdx.x; t < Tf; t += (int64_t)cl * kEvalPtThreads) {
    uint64_t c = canon(coef[t], M);
    for (int m = 0; m < nv; m++) {
      const int e = exps[t * nv + m];
      c = mul_mod(c, tab[m][e & 15], M);
      if (e >> 4) c = mul_mod(c, tab[m][16 + (e >> 4)], M);
    }
    sum = add_mod(sum, c, M);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum = add_mod(sum, __shfl_down_sync(0xffffffffu, sum, off), M);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (cl > 1) asm volatile("barrier.cluster.wait;" ::: "memory");
  if (threadIdx.x == 0) {
    uint64_t s = 0;
    for (int q = 0; q < kEvalPtThreads / 32; q++) s = add_mod(s, red[q], M);
    if (cl == 1) {
      out[pt] = s;
    } else {
      // into CTA 0's shared memory
      uint32_t at;
      const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&part[rank]);
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(mine), "r"(0));
      asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(at), "l"(s) : "memory");
    }
  }
  if (cl == 1) return;
  asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
  if (rank == 0 && threadIdx.x == 0) {
    uint64_t s = 0;
    for (int q = 0; q < cl; q++) s = add_mod(s, part[q], M);
    out[pt] = s;
  }
}

// Many points of a function of at most 32 terms: a warp per point, lane = term,
// a power per variable, which bounds it: 10^6 points in five variables 2.4 ms
// for one term, 4.2 for 16.  A CTA per point spends its time on the table (32 nv
// powers), 7.7 to 8.2 ms.
__global__ void __launch_bounds__(kEvalPtThreads)
    k_eval_points_few(int64_t Tf, int nv, int64_t npts, const uint8_t* __restrict__ exps,
                      const uint64_t* __restrict__ coef, const uint64_t* __restrict__ pts, Mod M,
                      uint64_t* __restrict__ out) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t pt = ((int64_t)blockIdx.x * kEvalPtThreads + threadIdx.x) >> 5;
  if (pt >= npts) return;
  uint64_t c = 0;
  if (lane < Tf) {
    c = canon(coef[lane], M);
    for (int m = 0; m < nv; m++) c = mul_mod(c, pow_mod(canon(pts[pt * nv + m], M), exps[lane * nv + m], M), M);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) c = add_mod(c, __shfl_down_sync(0xffffffffu, c, off), M);
  if (lane == 0) out[pt] = c;
}

// The probe points of a Zippel step: thread i computes y_m^(i+off) once per
// variable and writes it into the S points of probe i.
__global__ void k_probe_points(int64_t T, int S, int nv, int k, int offset, const uint64_t* __restrict__ y,
                               const uint64_t* __restrict__ cs, const uint64_t* __restrict__ z, Mod M,
                               uint64_t* __restrict__ pts) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T) return;
  for (int m = 0; m < nv; m++) {
    if (m == k) {
      for (int s = 0; s < S; s++) pts[((int64_t)s * T + i) * nv + m] = canon(cs[s], M);
    } else {
      const uint64_t val = m < k ? pow_mod(canon(y[m], M), (uint64_t)(i + offset), M) : canon(z[m], M);
      for (int s = 0; s < S; s++) pts[((int64_t)s * T + i) * nv + m] = val;
    }
  }
}

void launch_probe_points(int64_t T, int S, int nv, int k, int offset, const uint64_t* y, const uint64_t* cs,
                         const uint64_t* z, const Mod& M, uint64_t* pts, cudaStream_t st) {
  if (T > 0 && S > 0) { k_probe_points<<<cdiv(T, 128), 128, 0, st>>>(T, S, nv, k, offset, y, cs, z, M, pts); note_launch(); }
}

void launch_eval_points(const zr_poly* f, int64_t npts, const uint64_t* pts, const Mod& M, uint64_t* out,
                        cudaStream_t st) {
  if (npts <= 0) return;
  // up to about 1200 points run at once, and the table's powers are spread over
  // a CTA there: 300 points of 16 terms in five variables 26 us, a power per
  // term 29
  if (f->T <= 32 && npts > kEvalPtMany) {
    launch_k(k_eval_points_few, dim3(cdiv(npts, kEvalPtThreads / 32)), dim3(kEvalPtThreads), 0, st, f->T, (int)f->nv,
             npts, f->exps, f->coef, pts, M, out);
    note_launch();
    return;
  }
  // CTAs per point: up to eight while the points alone do not fill the GPU
  // (about two CTAs per SM) and a CTA keeps a term per thread
  int cl = 1;
  while (cl < 8 && npts * cl < 256 && (int64_t)cl * kEvalPtThreads < f->T) cl *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(npts * cl));
  cfg.blockDim = dim3(kEvalPtThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cl;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cl > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, k_eval_points, f->T, (int)f->nv, cl, f->exps, f->coef, pts, M, out);
  note_launch();
}

}  // namespace zr

using namespace zr;

extern "C" zr_status zr_zippel_probes(zr_ctx* ctx, const zr_poly* f, int32_t k, const uint64_t* y, int32_t S,
                                      const uint64_t* samples, const uint64_t* z, int64_t T, int32_t offset,
                                      uint64_t* out, int64_t ldo, void* stream) {
  if (!ctx) return ZR_ERR_INVALID_ARG;
  if (!f || f->nv < 1 || f->nv > kMaxVars || k < 0 || k >= f->nv || S < 1 || S > 256 || T < 0 || ldo < T ||
      f->T < 0 || (offset != 0 && offset != 1))
    return set_err(ctx, ZR_ERR_INVALID_ARG, "zr_zippel_probes: arguments out of range");
  if ((f->T > 0 && (!f->exps || !f->coef)) || !samples || (k > 0 && !y) || (T > 0 && !out) ||
      (k < f->nv - 1 && !z))
    return set_err(ctx, ZR_ERR_INVALID_ARG, "zr_zippel_probes: null pointer");
  if (T >= (1ll << 32)) return set_err(ctx, ZR_ERR_INVALID_ARG, "zr_zippel_probes: T must be below 2^32");
  cudaStream_t st = (cudaStream_t)stream;
  cudaMemsetAsync(ctx->d_status_call, 0, sizeof(uint32_t), st);
  zr_status r = probes_impl(ctx, f, k, y, S, samples, z, T, offset, out, ldo, ctx->d_status_call, st);
  if (r) return r;
  cudaError_t e = cudaMemcpyAsync(ctx->h_status + 1, ctx->d_status_call, sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_err(ctx, e, "zr_zippel_probes");
  return status_from_flags(ctx, ctx->h_status[1]);
}

extern "C" zr_status zr_probe_plan(const zr_ctx* ctx, int64_t T, int64_t Tf, int32_t S, int32_t* method,
                                   int32_t* splits) {
  if (!ctx || T < 1 || Tf < 1 || S < 1 || S > 256) return ZR_ERR_INVALID_ARG;
  const EvalMethod m = eval_method(ctx, T, Tf, S);
  Carver cv(nullptr);
  if (method) *method = m;
  if (splits)
    *splits = m == EVAL_TREE ? 0 : m == EVAL_TC ? carve_eval_tc(cv, ctx, Tf, S, T).gsplit : eval_gsplit(ctx, T, S, Tf);
  return ZR_OK;
}

extern "C" zr_status zr_eval_points(zr_ctx* ctx, const zr_poly* f, int64_t npts, const uint64_t* pts, uint64_t* out,
                                    void* stream) {
  if (!ctx) return ZR_ERR_INVALID_ARG;
  if (!f || f->nv < 1 || f->nv > kMaxVars || f->T < 0 || npts < 0 || (npts > 0 && (!pts || !out)) ||
      (f->T > 0 && (!f->exps || !f->coef)))
    return set_err(ctx, ZR_ERR_INVALID_ARG, "zr_eval_points: arguments out of range");
  cudaStream_t st = (cudaStream_t)stream;
  launch_eval_points(f, npts, pts, ctx->M, out, st);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return cuda_err(ctx, e, "zr_eval_points");
}

extern "C" zr_status zr_probe_points(zr_ctx* ctx, int32_t nv, int32_t k, const uint64_t* y, int32_t S,
                                     const uint64_t* samples, const uint64_t* z, int64_t T, int32_t offset,
                                     uint64_t* pts, void* stream) {
  if (!ctx) return ZR_ERR_INVALID_ARG;
  if (nv < 1 || nv > kMaxVars || k < 0 || k >= nv || S < 1 || T < 0 || (offset != 0 && offset != 1) ||
      (T > 0 && (!pts || !samples || (k > 0 && !y) || (k + 1 < nv && !z))))
    return set_err(ctx, ZR_ERR_INVALID_ARG, "zr_probe_points: arguments out of range");
  launch_probe_points(T, S, nv, k, offset, y, samples, z, ctx->M, pts, (cudaStream_t)stream);
  return cuda_err(ctx, cudaGetLastError(), "zr_probe_points");
}
