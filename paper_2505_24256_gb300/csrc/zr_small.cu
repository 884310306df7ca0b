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
//   warps 0-7    lane = root, warp = k-block: the block's Horner value, the
//                carry from the blocks above, the quotients q_k with their Horner
//                value, then the block's part of every dot product;
//   warp 8       lane = sample: the values -> monomials matrix of Newton's
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
constexpr int kSmWarps = 8;                      // k-blocks
constexpr int kSmThreads = 32 * (kSmWarps + 1);

struct SmallSmem {
  // word offsets of the dynamic shared memory
  int v, tree, tab, b, q, part, num, W, total;
};
__host__ __device__ inline SmallSmem small_smem(int T, int S, int Sn, int k) {
  SmallSmem o;
  const int BK = (T + kSmWarps - 1) / kSmWarps;
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
  at += (kSmWarps * BK > Sn ? kSmWarps * BK : Sn) * kSmRoots;
  o.part = at;
  at += kSmWarps * S * kSmRoots;
  o.num = at;
  at += Sn * kSmRoots;
  o.W = at;
  at += Sn * Sn;
  o.total = at;
  return o;
}

__device__ __forceinline__ void main_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

__global__ void __launch_bounds__(kSmThreads, 1)
    k_small(const BDesc* __restrict__ Ds, const int64_t* __restrict__ idx, int cl, Mod M) {
  pdl_enter();
  extern __shared__ uint64_t ssm[];
  __shared__ uint64_t rs[kSmWarps][kSmRoots], us[kSmWarps][kSmRoots], invs[kSmRoots];
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

  if (warp == kSmWarps) {
    if (D.mode == 0 && any) {
      // W[e][s] = coefficient e of prod_{t != s} (z - x_t) / (x_s - x_t):
      // P = prod (z - x_t), lane e its coefficient; then lane s divides by z - x_s
      const uint64_t x = lane < Sn ? D.xs[lane] : 0, xq = shoup_pre(x, M);
      uint64_t c = lane == 0 ? 1 : 0;
      for (int t = 0; t < Sn; t++) {
        uint64_t up = __shfl_up_sync(FULL, c, 1);
        if (lane == 0) up = 0;
        c = sub_mod(up, mul_mod(__shfl_sync(FULL, x, t), c, M), M);
      }
      uint64_t q = 1, u = 0;
      for (int e = Sn - 1; e >= 0; e--) {
        u = add_mod(canon(shoup_lazy(u, x, xq, M), M), q, M);
        if (lane < Sn) W[e * Sn + lane] = q;
        q = add_mod(canon(shoup_lazy(q, x, xq, M), M), __shfl_sync(FULL, c, e), M);
      }
      if (lane < Sn && u == 0 && rank == 0) atomicOr(D.status, ST_DUP_SAMPLE);
      const uint64_t inv = warp_batch_inverse(lane < Sn ? u : 1, M);
      if (lane < Sn)
        for (int e = 0; e < Sn; e++) W[e * Sn + lane] = mul_mod(W[e * Sn + lane], inv, M);
    }
  } else if (any) {
    // the right-hand sides, on their way while the nodes are made
    for (int i = tid; i < S * T; i += 256) {
      const int s = i / T;
      cp_async8(bs + i, D.b + (int64_t)s * D.ldb + (i - s * T));
    }
    cp_async_commit();
    // anchor values
    for (int i = tid; i < 32 * k; i += 256) {
      const int m = i >> 5, e = i & 31;
      tab[i] = pow_mod(D.y[m], e < 16 ? e : (uint64_t)(e - 16) * 16, M);
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
      tree[tid] = x ? M.p - x : 0;               // z - v_j
    }
    main_sync();
    // M's coefficients below its leading 1
    uint64_t *in = tree, *out = tree + T;
    for (int size = 1; size < T; size *= 2) {
      if (tid < T) {
        const int po = tid & ~(2 * size - 1);
        out[tid] = T - po <= size ? in[tid] : conv_coef(in, po, size, min(size, T - po - size), tid - po, M);
      }
      main_sync();
      uint64_t* t = in;
      in = out;
      out = t;
    }
    const uint64_t* m = in;
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
    uint64_t* qw = qs + warp * BK * kSmRoots + lane;
    for (int i = khi - 1; i >= klo; i--) {
      const uint64_t qc = canon(q, M);
      qw[(i - klo) * kSmRoots] = qc;
      u = canon(shoup_lazy(u, v, vq, M), M) + qc;
      q = canon(shoup_lazy(qc, v, vq, M), M) + m[i];
    }
    us[warp][lane] = canon(u, M);
    cp_async_wait<0>();
    main_sync();
    // the block's part of the dot products, four right-hand sides at a time
    for (int s0 = 0; s0 < S; s0 += 4) {
      Acc8 acc[4];
      const uint64_t* row[4];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        acc[c] = Acc8{0, 0, 0, 0, 0, 0, 0, 0};
        row[c] = bs + min(s0 + c, S - 1) * T;
      }
#pragma unroll 4
      for (int i = klo; i < khi; i++) {
        const uint64_t x = qw[(i - klo) * kSmRoots];
#pragma unroll
        for (int c = 0; c < 4; c++) {
          const uint64_t w = row[c][i];
          mac8(acc[c], lo32(x), hi32(x), lo32(w), hi32(w));
        }
      }
#pragma unroll
      for (int c = 0; c < 4; c++)
        if (s0 + c < S) part[(warp * S + s0 + c) * kSmRoots + lane] = acc8_value(acc[c], M);
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
        for (int w = 0; w <= wl; w++) x = add_mod(x, part[(w * S + s) * kSmRoots + lane], M);
        num[(s + s1) * kSmRoots + lane] = x;
      }
    }
  }
  __syncthreads();
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
  if (D.mode != 0) {
    asm volatile("barrier.cluster.wait;" ::: "memory");
    return;
  }
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

constexpr size_t kSmMaxSmem = 216 * 1024;

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

size_t small_words(int64_t T, int S, int Sn, int k) { return (size_t)small_smem((int)T, S, Sn, k).total; }

}  // namespace zr
