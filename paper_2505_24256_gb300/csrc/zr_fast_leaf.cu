// zr_fast_leaf.cu -- the leaves of the O(T log^2 T) solve on the tensor cores.
//
// At a block P of L = 2^ll roots (zr_fast.cu) the values are
//     val_r(j) = <q^P_j, X_P^(r)>,   q_{j,d-1} = 1, q_{j,k-1} = p_k + v_j q_{j,k}
// for the block's d roots v_j and the R rows: a product of the d x d matrix of
// the q's, which one Shoup step per entry makes, with the d x R expansions, in
// digits (zr_tc.cuh).
#include <cuda_runtime.h>

#include "zr_internal.h"
#include "zr_launch.cuh"
#include "zr_tc.cuh"

namespace zr {

namespace {

constexpr int kLfStep = 16;                          // k per k-step
constexpr int kLfNC = 16;                            // columns of a CTA
constexpr uint32_t kLfPlane = kTcRows * 16;          // a digit plane of eight k of A
constexpr uint32_t kLfASlab = kTcLimbs * kLfPlane;
constexpr uint32_t kLfBSlab = kTcLimbs * kLfNC * 16;
constexpr uint32_t kLfStage = 2 * (kLfASlab + kLfBSlab);
constexpr int kLfStages = 3;
constexpr int kLfChunkSteps = kTcChunk / kLfStep;
constexpr int kLfAhead = 2;                          // k-steps of the next chunk made before a chunk is drained
constexpr int kLfThreads = 6 * 32;                   // 4 chain and drain warps, B's digits, the MMAs
constexpr size_t kLfSmem = kLfStages * (size_t)kLfStage + 128;
constexpr uint32_t kLfTmem = 256;

// A CTA takes 128 roots of one block and up to 16 rows.  The k-steps run from k
// = d - 1 down through a ring of three stages:
//   warps 0-3   lane = root: sixteen steps of the chain, their digits into the
//               stage; 128 k behind, the sums out of the tensor memory;
//   warp 4      the digits of the rows' expansions, and their sums;
//   warp 5      the MMAs.
// Two CTAs share an SM (110 KB of shared memory and 256 columns of tensor
// memory each), so that one drains or waits while the other's chains run.  The
// chain bounds it (about 40 instructions a step, sixteen for an entry's digits,
// each step waiting for the one before).  The blocks of 128 roots on the integer
// pipe, a thread per root that ran its chain again for every four rows, took
// 0.040 ms at T = 10^4, S = 21 and 1.31 ms at T = 2^20, S = 9; this kernel takes
// 0.048 and 1.32 ms for blocks of 256 (0.18 ms at T = 125000, S = 9), which saves
// the descent's level of 2^8 (0.040 and 1.6 ms).
__global__ void __launch_bounds__(kLfThreads, 2)
    k_leaf_tc(const uint64_t* __restrict__ coef, const uint64_t* __restrict__ X, int R, int cols, int ll, int64_t T,
              int64_t Tp, const uint64_t* __restrict__ v, const uint64_t* __restrict__ vp, Mod M, TcMod K,
              uint64_t* __restrict__ part, int64_t ldp, uint64_t* __restrict__ den, uint32_t* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char lsm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(lsm + kLfStages * kLfStage);
  uint64_t *empty = full + kLfStages, *tfull = empty + kLfStages, *tempty = tfull + 1, *done = tempty + 1,
           *summed = done + 1;
  uint32_t* slot = reinterpret_cast<uint32_t*>(summed + 1);
  __shared__ uint64_t sums[kLfNC];                   // 0x8080..80 times each row's sum

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_enter();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kLfStages; s++) {
      mbar_init(&full[s], 5);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, 4);
    mbar_init(done, 1);
    mbar_init(summed, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 5) tc_alloc(slot, kLfTmem);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  const int64_t j0 = (int64_t)blockIdx.x * kTcRows, base = j0 >> ll << ll;
  const int d = (int)((T - base) < (1ll << ll) ? (T - base) : (1ll << ll));
  const int r0 = blockIdx.y * cols, rn = R - r0 < cols ? R - r0 : cols;
  const int n = (d + kLfStep - 1) / kLfStep, chunks = (n + kLfChunkSteps - 1) / kLfChunkSteps;

  if (warp < 4) {
    const int64_t j = j0 + 32 * warp + lane;
    const bool live = j < T;
    const uint64_t vj = live ? v[j] : 0, vq = live ? vp[j] : 0;
    const uint32_t addr = tmem + ((uint32_t)warp << 21);
    TcAcc acc[kLfNC];
#pragma unroll
    for (int c = 0; c < kLfNC; c++) acc[c] = TcAcc{{0, 0, 0, 0, 0, 0}};
    bool ok = true;
    int drained = 0;
    auto drain = [&]() {
      if (!tc_wait(tfull, drained & 1)) {
        atomicOr(status, ST_TIMEOUT);
        ok = false;
        return;
      }
      drained++;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < kLfNC; c += 4)
        if (c < rn) tc_add_chunk<kLfNC>(addr + c, acc + c);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty);
    };
    // Eight steps of the chain, x[i] = q_k for k = k0 - i, below 2 p (which
    // Shoup's product takes as it is).  The bytes of x are the digits of
    // x - 0x8080..80: the value is that constant times the row's sum short.
    const uint64_t* pb = coef + base;
    uint64_t q = 1;
    auto chain = [&](int k0, uint64_t(&x)[8]) {
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const int k = k0 - i;
        const uint64_t pk = k >= 0 ? __ldg(pb + k) : 0;
        x[i] = q;
        q = canon(shoup_lazy(q, vj, vq, M), M) + pk;
      }
    };
    // the digits of eight k while the chain makes the next eight
    uint64_t x[8], y[8];
    chain(d - 1, x);
    for (int s = 0; ok && s < n; s++) {
      const int st = s % kLfStages;
      uint4* dst = reinterpret_cast<uint4*>(lsm + st * kLfStage) + 32 * warp + lane;
      if (s >= kLfStages && !tc_wait(&empty[st], ((s / kLfStages) & 1) ^ 1)) {
        atomicOr(status, ST_TIMEOUT);
        ok = false;
        break;
      }
      uint4 dg[kTcLimbs];
      chain(d - 1 - (s * kLfStep + 8), y);
      tc_bytes(x, dg);
#pragma unroll
      for (int i = 0; i < kTcLimbs; i++) dst[i * kTcRows] = dg[i];
      chain(d - 1 - (s * kLfStep + 16), x);
      tc_bytes(y, dg);
#pragma unroll
      for (int i = 0; i < kTcLimbs; i++) dst[(kTcLimbs + i) * kTcRows] = dg[i];
      tc_fence_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[st]);
      if (s + 1 >= kLfChunkSteps + kLfAhead && (s + 1 - kLfAhead) % kLfChunkSteps == 0) drain();
    }
    while (ok && drained < chunks) drain();
    if (ok && !tc_wait(summed, 0)) {
      atomicOr(status, ST_TIMEOUT);
      ok = false;
    }
    if (ok && live) {
#pragma unroll
      for (int c = 0; c < kLfNC; c++) {
        const int r = r0 + c;
        if (c >= rn) continue;
        const uint64_t val = add_mod(tc_value(acc[c], K, M), sums[c], M);
        if (r < R - 1) part[(int64_t)r * ldp + j] = val;
        else den[j] = val;
      }
    }
  } else if (warp == 4) {
    // lane = (eight k of the k-step, row)
    const int c = lane & 15, slab = lane >> 4;
    const uint64_t* x0 = X + (int64_t)(r0 + c) * Tp + base;
    uint64_t x[8];
    auto load = [&](int s) {
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const int k = d - 1 - (s * kLfStep + slab * 8 + i);
        x[i] = c < rn && k >= 0 ? __ldg(x0 + k) : 0;
      }
    };
    load(0);
    uint64_t sum = 0;
    for (int s = 0; s < n; s++) {
      const int st = s % kLfStages;
      uint4 dg[kTcLimbs];
#pragma unroll
      for (int i = 0; i < 8; i++) sum = add_mod(sum, x[i], M);
      tc_digits(x, M.p, dg);
      load(s + 1);
      if (s >= kLfStages && !tc_wait(&empty[st], ((s / kLfStages) & 1) ^ 1)) {
        atomicOr(status, ST_TIMEOUT);
        break;
      }
      uint4* dst = reinterpret_cast<uint4*>(lsm + st * kLfStage + 2 * kLfASlab + slab * kLfBSlab) + c;
#pragma unroll
      for (int i = 0; i < kTcLimbs; i++) dst[i * kLfNC] = dg[i];
      tc_fence_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[st]);
    }
    sum = add_mod(sum, __shfl_down_sync(0xffffffffu, sum, 16), M);
    if (lane < kLfNC) sums[lane] = mul_mod(sum, kTcBias % M.p, M);
    __syncwarp();
    if (lane == 0) mbar_arrive(summed);
  } else {
    const bool leader = tc_elect();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    for (int s = 0; s < n; s++) {
      const int st = s % kLfStages, c = s / kLfChunkSteps;
      const bool first = s % kLfChunkSteps == 0, last = s % kLfChunkSteps == kLfChunkSteps - 1 || s == n - 1;
      if ((first && c > 0 && !tc_wait(tempty, (c - 1) & 1)) || !tc_wait(&full[st], (s / kLfStages) & 1)) {
        if (leader) atomicOr(status, ST_TIMEOUT);
        break;
      }
      tc_fence_after();
      if (leader) {
        const uint32_t a = smem_addr(lsm) + st * kLfStage;
        tc_kstep<kLfNC>(tm, a, kLfPlane, kLfASlab, a + 2 * kLfASlab, kLfBSlab, first);
        tc_commit(&empty[st]);
        if (last) tc_commit(tfull);
      }
      __syncwarp();
    }
    // the MMAs issued have completed before the tensor memory goes back
    if (leader) tc_commit(done);
    mbar_wait(done, 0);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  __syncwarp();
  if (warp == 5) tc_dealloc(tmem, kLfTmem);
}

}  // namespace

TcMod tc_mod(const Mod& M) {
  auto pow2 = [&](int e) {
    unsigned __int128 r = 1;
    for (int i = 0; i < e; i++) r = r * 2 % M.p;
    return (uint64_t)r;
  };
  return TcMod{pow2(96), pow2(154)};
}

// The values of all T roots in blocks of 2^ll: rows r < R - 1 of X (stride Tp)
// to part[r ldp + j], row R - 1 to den[j]; coef: the block polynomials.
void launch_leaf_tc(const uint64_t* coef, const uint64_t* X, int R, int ll, int64_t T, int64_t Tp, const uint64_t* v,
                    const uint64_t* vp, const Mod& M, uint64_t* part, int64_t ldp, uint64_t* den, uint32_t* status,
                    cudaStream_t st) {
  static DeviceOnce attr;
  attr.run([] { cudaFuncSetAttribute(k_leaf_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLfSmem); });
  const int groups = (R + kLfNC - 1) / kLfNC, cols = (R + groups - 1) / groups;
  launch_k(k_leaf_tc, dim3((unsigned)((T + kTcRows - 1) / kTcRows), groups), dim3(kLfThreads), kLfSmem, st, coef, X, R,
           cols, ll, T, Tp, v, vp, M, tc_mod(M), part, ldp, den, status);
  note_launch();
}

}  // namespace zr
