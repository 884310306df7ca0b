// zr_small.cu -- small steps and systems in one launch.
//
// A Zippel step (or Vandermonde system) of at most 256 unknowns is too small for
// its ten launches to be anything but latency (0.10 ms of kernels at T = 200, S
// = 11, each of 5 to 24 us).  Here a cluster of up to eight CTAs takes the whole
// entry, 32 roots a CTA, by the same method (Sec. 2.2: Horner quotients, deferred
// dot products, one inverse per root, Newton in the new variable):
//   every CTA    the anchor values of all T terms and the master polynomial by
//                the product tree (short enough to repeat, so that nothing is
//                exchanged);
//   warps 0-15   lane = root, warp = k-block: the block's Horner value, the
//                carry from the blocks above, the quotients q_k with their Horner
//                value; then a warp per right-hand side and part of k: the dot
//                products;
//   warp 16      lane = sample: the values -> monomials matrix of Newton's
//                interpolation, beside all that;
//   then         the sums over the blocks, one inverse, Newton, and the compaction
//                (the CTAs' counts through distributed shared memory).
// Equal nodes make a denominator q_j(v_j) = prod (v_j - v_i) vanish, so they need
// no table.  (Step T = 200, S = 11: 0.088 ms a call against 0.152; 64 steps of T =
// 20 .. 66: 0.28 against 0.74 ms, most of that on the host.)
#include <cuda_runtime.h>

#include <algorithm>

#include "zr_device.cuh"
#include "zr_internal.h"
#include "zr_launch.cuh"
#include "zr_ring.cuh"

namespace zr {

namespace {

constexpr int kSmRoots = 32;                     // roots of a CTA: a lane each
constexpr int kSmWarps = 16;                     // k-blocks
constexpr int kSmThreads = 32 * (kSmWarps + 1);

struct SmallSmem {
  // word offsets of the dynamic shared memory
  int v, tree, tab, b, q, part, num, W, total;
};
// parts of k a dot product is split into: two or three items a warp
__host__ __device__ inline int small_parts(int S) { return S >= 2 * kSmWarps ? 1 : (2 * kSmWarps + S - 1) / S; }
__host__ __device__ inline SmallSmem small_smem(int T, int S, int Sn, int k) {
  SmallSmem o;
  int at = 0;
  o.v = at;
  at += T;
  o.tree = at;
  at += 2 * T;
  o.tab = at;
  at += 32 * k;
  o.b = at;
  at += S * T;
  o.q = at;                                      // the quotients, later the coefficients
  at += (T > Sn ? T : Sn) * kSmRoots;
  o.part = at;
  at += small_parts(S) * S * kSmRoots;
  o.num = at;
  at += Sn * kSmRoots;
  o.W = at;
  at += Sn * Sn;
  o.total = at;
  return o;
}

constexpr int kSmMain = 32 * kSmWarps;
__device__ __forceinline__ void main_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kSmMain) : "memory"); }

// Coefficient n of (A + z^a)(B + z^b), below z^(a+b), A at in[0..a), B at
// in[a..a+b): half h of the products by each of two neighbouring lanes, in two
// sums (a chain of multiply-adds takes 50 cycles a product).
__device__ __forceinline__ uint64_t conv_half(const uint64_t* in, int a, int b, int n, int h, const Mod& M) {
  const int lo = max(0, n - b + 1), hi = min(a - 1, n) + 1, mid = lo + (max(hi - lo, 0) >> 1);
  const int i0 = h ? mid : lo, i1 = h ? hi : mid;
  Acc8 s0 = {0, 0, 0, 0, 0, 0, 0, 0}, s1 = {0, 0, 0, 0, 0, 0, 0, 0};
  const uint64_t* B = in + a + n;
  int i = i0;
#pragma unroll 2
  for (; i + 1 < i1; i += 2) {
    const uint64_t x = in[i], y = B[-i], z = in[i + 1], w = B[-i - 1];
    mac8(s0, lo32(x), hi32(x), lo32(y), hi32(y));
    mac8(s1, lo32(z), hi32(z), lo32(w), hi32(w));
  }
  if (i < i1) {
    const uint64_t x = in[i], y = B[-i];
    mac8(s0, lo32(x), hi32(x), lo32(y), hi32(y));
  }
  acc8_add(s0, s1);
  uint64_t r = acc8_value(s0, M);
  if (h == 0 && n >= a) r = add_mod(r, in[n], M);            // z^a times B_{n-a}
  if (h == 1 && n >= b) r = add_mod(r, in[n - b], M);        // z^b times A_{n-b}
  return r;
}

__global__ void __launch_bounds__(kSmThreads, 1)
    k_small(const BDesc* __restrict__ Ds, const int64_t* __restrict__ idx, int cl, Mod M) {
  pdl_enter();
  extern __shared__ uint64_t ssm[];
  __shared__ uint64_t sq[kMaxVars][8], rs[kSmWarps][kSmRoots], us[kSmWarps][kSmRoots], invs[kSmRoots];
  __shared__ uint32_t nz[32], masks[kSmRoots];
  __shared__ int offs[kSmRoots], tot[8];
  asm volatile("barrier.cluster.arrive;" ::: "memory");   // waited for before another CTA's memory is written
  const int ent = blockIdx.x / cl, rank = blockIdx.x - ent * cl;
  const BDesc& D = Ds[idx[ent]];
  const int T = (int)D.T, S = D.S, Sn = D.Sn, k = D.mode == 0 ? D.k : 0, s1 = Sn - S;
  const SmallSmem o = small_smem(T, S, Sn, k);
  uint64_t *vs = ssm + o.v, *tree = ssm + o.tree, *tab = ssm + o.tab, *bs = ssm + o.b, *qs = ssm + o.q,
           *part = ssm + o.part, *num = ssm + o.num, *W = ssm + o.W;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j0 = rank * kSmRoots, j = j0 + lane;
  const bool live = j < T, any = j0 < T;         // CTAs past the entry's roots only count
  const unsigned FULL = 0xffffffffu;
  const int BK = (T + kSmWarps - 1) / kSmWarps, wl = (T - 1) / BK;   // the last block that holds anything
  const int kp = small_parts(S);

  if (warp == kSmWarps) {
    if (D.mode == 0 && any) newton_matrix_warp<1>(Sn, D.xs, W, rank == 0 ? D.status : nullptr, M);
  } else if (any) {
    // the right-hand sides, on their way while the nodes are made
    for (int s = 0; s < S; s++)
      if (tid < T) cp_async8(bs + s * T + tid, D.b + (int64_t)s * D.ldb + tid);
    cp_async_commit();
    // anchor powers: x^(2^b), then x^e and x^(16 e), e < 16, from them
    if (tid < k) {
      uint64_t x = D.y[tid];
      for (int b = 0; b < 8; b++) {
        sq[tid][b] = x;
        x = mul_mod(x, x, M);
      }
    }
    main_sync();
    for (int i = tid; i < 32 * k; i += kSmMain) {
      const uint64_t* b = sq[i >> 5] + ((i >> 2) & 4);
      uint64_t x = i & 1 ? b[0] : 1;
#pragma unroll
      for (int q = 1; q < 4; q++)
        if ((i >> q) & 1) x = mul_mod(x, b[q], M);
      tab[i] = x;
    }
    main_sync();
    if (tid < T) {
      uint64_t x;
      if (D.mode == 0) {
        const uint8_t* e = D.exps + (int64_t)tid * D.nv;
        x = 1;
        for (int m = 0; m < k; m++) {
          const int a = e[m];
          x = mul_mod(x, tab[32 * m + (a & 15)], M);
          if (a >> 4) x = mul_mod(x, tab[32 * m + 16 + (a >> 4)], M);
        }
      } else {
        x = D.v[tid];
        if (x >= M.p) {
          atomicOr(D.status, ST_DUP_NODE);
          x = 0;
        }
      }
      if (D.offset == 1 && x == 0) atomicOr(D.status, ST_ZERO_NODE);
      vs[tid] = x;
    }
    main_sync();
    // M's coefficients below its leading 1: blocks of 32 roots, a factor at a
    // time with the coefficients in a warp's lanes (half the time of the tree's
    // first five levels), then pairs, two lanes a coefficient
    if (32 * warp < T) {
      const uint64_t x = tid < T ? vs[tid] : 0, xq = shoup_pre(x, M);
      uint64_t c = lane == 0 ? 1 : 0;
      for (int t = 0; t < min(32, T - 32 * warp); t++) {
        uint64_t up = __shfl_up_sync(FULL, c, 1);
        if (lane == 0) up = 0;
        const uint64_t xt = __shfl_sync(FULL, x, t), xqt = __shfl_sync(FULL, xq, t);
        c = sub_mod(up, canon(shoup_lazy(c, xt, xqt, M), M), M);
      }
      if (tid < T) tree[tid] = c;
    }
    main_sync();
    int in = o.tree, out = o.tree + T;
    for (int size = 32; size < T; size *= 2) {
      const int n = tid >> 1, h = tid & 1, po = n & ~(2 * size - 1);
      uint64_t x = 0;
      const bool pair = n < T && T - po > size;
      if (pair) x = conv_half(ssm + in + po, size, min(size, T - po - size), n - po, h, M);
      x = add_mod(x, __shfl_xor_sync(FULL, x, 1), M);
      if (n < T && h == 0) ssm[out + n] = pair ? x : ssm[in + n];
      main_sync();
      const int t = in;
      in = out;
      out = t;
    }
    const uint64_t* m = ssm + in;
    // k-blocks [klo, khi): the block's Horner value (the last one's includes m_T
    // = 1), the carry from the blocks above, the quotients
    const uint64_t v = live ? vs[j] : 0, vq = shoup_pre(v, M);
    const uint64_t vBK = pow_mod(v, (uint64_t)BK, M), vBKq = shoup_pre(vBK, M);
    const int klo = min(warp * BK, T), khi = min(klo + BK, T);
    uint64_t r = warp == wl ? 1 : 0;
    for (int i = khi - 1; i >= klo; i--) r = canon(shoup_lazy(r, v, vq, M), M) + m[i];
    rs[warp][lane] = canon(r, M);
    main_sync();
    uint64_t q = warp == wl ? 1 : 0, u = 0;
    for (int w = wl; w > warp; w--) q = add_mod(canon(shoup_lazy(q, vBK, vBKq, M), M), rs[w][lane], M);
    uint64_t* qw = qs + klo * kSmRoots + lane;
    for (int i = khi - 1; i >= klo; i--) {
      const uint64_t qc = canon(q, M);
      qw[(i - klo) * kSmRoots] = qc;
      u = canon(shoup_lazy(u, v, vq, M), M) + qc;
      q = canon(shoup_lazy(qc, v, vq, M), M) + m[i];
    }
    us[warp][lane] = canon(u, M);
    cp_async_wait<0>();
    main_sync();
    // dot products: a warp takes right-hand side s and the p-th of kp parts of k
    for (int it = warp; it < S * kp; it += kSmWarps) {
      const int p = it / S, s = it - p * S;
      const int k0 = T * p / kp, k1 = T * (p + 1) / kp;
      Acc8 a0 = {0, 0, 0, 0, 0, 0, 0, 0}, a1 = {0, 0, 0, 0, 0, 0, 0, 0};
      const uint64_t *x = qs + lane, *w = bs + s * T;
      int i = k0;
#pragma unroll 2
      for (; i + 1 < k1; i += 2) {
        const uint64_t x0 = x[i * kSmRoots], x1 = x[(i + 1) * kSmRoots], w0 = w[i], w1 = w[i + 1];
        mac8(a0, lo32(x0), hi32(x0), lo32(w0), hi32(w0));
        mac8(a1, lo32(x1), hi32(x1), lo32(w1), hi32(w1));
      }
      if (i < k1) {
        const uint64_t x0 = x[i * kSmRoots], w0 = w[i];
        mac8(a0, lo32(x0), hi32(x0), lo32(w0), hi32(w0));
      }
      acc8_add(a0, a1);
      part[it * kSmRoots + lane] = acc8_value(a0, M);
    }
    main_sync();
    if (warp == 0) {
      uint64_t den = 0;
      for (int w = wl; w >= 0; w--) den = add_mod(canon(shoup_lazy(den, vBK, vBKq, M), M), us[w][lane], M);
      if (D.offset == 1) den = mul_mod(den, v, M);
      if (live && den == 0) atomicOr(D.status, ST_ZERO_DEN);
      invs[lane] = warp_batch_inverse(live ? den : 1, M);
    } else {
      for (int s = warp - 1; s < S; s += kSmWarps - 1) {
        uint64_t x = 0;
        for (int p = 0; p < kp; p++) x = add_mod(x, part[(p * S + s) * kSmRoots + lane], M);
        num[(s + s1) * kSmRoots + lane] = x;
      }
    }
  }
  __syncthreads();
  // every CTA has read all the nodes: a system's solution may lie over them
  // (the arrival at the top is an early one: a barrier of its own)
  if (D.mode != 0)
    asm volatile("barrier.cluster.wait;\n\tbarrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
  if (any && warp < kSmWarps) {
    const uint64_t inv = invs[lane];
    if (D.mode != 0) {
      for (int s = warp; s < S; s += kSmWarps)
        if (live) D.c[(int64_t)s * D.ldc + j] = mul_mod(num[s * kSmRoots + lane], inv, M);
    } else {
      if (s1) {
        // the given solution at sample 0, the solved ones scaled by the inverse
        for (int s = warp; s < Sn; s += kSmWarps) {
          uint64_t* x = num + s * kSmRoots + lane;
          *x = s == 0 ? (live ? D.c0[j] : 0) : mul_mod(*x, inv, M);
        }
        main_sync();
      }
      // the monomial coefficients, into the dot products' place
      for (int e = warp; e < Sn; e += kSmWarps) {
        Acc8 acc = {0, 0, 0, 0, 0, 0, 0, 0};
        const uint64_t* w = W + e * Sn;
        for (int s = 0; s < Sn; s++) {
          const uint64_t x = num[s * kSmRoots + lane], y = w[s];
          mac8(acc, lo32(x), hi32(x), lo32(y), hi32(y));
        }
        uint64_t g = acc8_value(acc, M);
        if (!s1) g = mul_mod(g, inv, M);
        qs[e * kSmRoots + lane] = g;
        const unsigned set = __ballot_sync(FULL, live && g != 0);
        if (lane == 0) nz[e] = set;
      }
      main_sync();
      if (warp == 0) {
        uint32_t mask = 0;
        for (int e = 0; e < Sn; e++) mask |= ((nz[e] >> lane) & 1u) << e;
        const int cnt = __popc(mask);
        int incl = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int x = __shfl_up_sync(FULL, incl, off);
          if (lane >= off) incl += x;
        }
        masks[lane] = mask;
        offs[lane] = incl - cnt;
        if (lane == 31) invs[0] = (uint64_t)incl;    // the inverses are no longer needed
      }
    }
  }
  if (D.mode != 0) return;
  __syncthreads();
  // every CTA's count into every CTA of the cluster
  asm volatile("barrier.cluster.wait;" ::: "memory");
  if (tid < cl) {
    uint32_t at;
    const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&tot[rank]);
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(mine), "r"(tid));
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(any ? (int)invs[0] : 0) : "memory");
  }
  asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
  int64_t base = 0, all = 0;
  for (int r = 0; r < cl; r++) {
    if (r < rank) base += tot[r];
    all += tot[r];
  }
  if (rank == 0 && tid == 0) *D.out_count = all;
  if (any && warp < kSmWarps) {
    const uint32_t mask = masks[lane];
    const int nv = D.nv;
    for (int e = warp; e < Sn; e += kSmWarps) {
      if (!((mask >> e) & 1u)) continue;
      const int64_t pos = base + offs[lane] + __popc(mask & ((1u << e) - 1));
      if (pos >= D.out_cap) continue;
      const uint8_t* src = D.exps + (int64_t)j * nv;
      uint8_t* dst = D.out_exps + pos * nv;
      for (int m = 0; m < nv; m++) dst[m] = m < k ? src[m] : 0;
      dst[k] = (uint8_t)e;
      D.out_coef[pos] = qs[e * kSmRoots + lane];
    }
  }
}

constexpr size_t kSmMaxSmem = 208 * 1024;   // beside 13 KB of static arrays

// whether this device runs clusters of eight with the largest shared memory
bool small_supported() {
  static DeviceValue ok;
  return ok.get([] {
           if (cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmMaxSmem) !=
               cudaSuccess) {
             (void)cudaGetLastError();
             return 2;
           }
           cudaLaunchConfig_t cfg = {};
           cfg.gridDim = dim3(8);
           cfg.blockDim = dim3(kSmThreads);
           cfg.dynamicSmemBytes = kSmMaxSmem;
           cudaLaunchAttribute attr[1];
           attr[0].id = cudaLaunchAttributeClusterDimension;
           attr[0].val.clusterDim.x = 8;
           attr[0].val.clusterDim.y = 1;
           attr[0].val.clusterDim.z = 1;
           cfg.attrs = attr;
           cfg.numAttrs = 1;
           int clusters = 0;
           if (cudaOccupancyMaxActiveClusters(&clusters, k_small, &cfg) != cudaSuccess) {
             (void)cudaGetLastError();
             return 2;
           }
           return clusters > 0 ? 1 : 2;
         }) == 1;
}

}  // namespace

// Up to 256 unknowns (eight CTAs), 32 samples (a lane each in Newton's matrix)
// and what fits the shared memory.
bool small_entry(int64_t T, int S, int Sn, int k) {
  if (T < 1 || T > 8 * kSmRoots || S < 1 || Sn > 32) return false;
  return 8 * (size_t)small_smem((int)T, S, Sn, k).total <= kSmMaxSmem && small_supported();
}

cudaError_t launch_small(const BDesc* Ds, const int64_t* idx, int n, int64_t Tmax, size_t words, const Mod& M,
                         cudaStream_t st) {
  const int cl = (int)((Tmax + kSmRoots - 1) / kSmRoots);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n * cl));
  cfg.blockDim = dim3(kSmThreads);
  cfg.dynamicSmemBytes = 8 * words;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_small, Ds, idx, cl, M);
  note_launch();
  return e;
}

int small_resident(int64_t Tmax, size_t words) {
  const int cl = (int)((Tmax + kSmRoots - 1) / kSmRoots);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cl);
  cfg.blockDim = dim3(kSmThreads);
  cfg.dynamicSmemBytes = 8 * words;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k_small, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 1;
  }
  return clusters > 0 ? clusters : 1;
}

size_t small_words(int64_t T, int S, int Sn, int k) { return (size_t)small_smem((int)T, S, Sn, k).total; }

}  // namespace zr
