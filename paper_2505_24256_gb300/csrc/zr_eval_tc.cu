// zr_eval_tc.cu -- the evaluator's matrix-vector product on the tensor cores.
//
//     out[s][i] = sum_g W[g][s] u_g^(i + off),  i < T,
// (zr_eval.cu) with i = 128 a + b is the product of
//     A[b][g] = u_g^b            (128 rows, shared by every column) and
//     B[g][(a, s)] = W[g][s] u_g^off u_g^(128 a)
// over k = g: S T G residue products as a GEMM, in digits (zr_tc.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "zr_internal.h"
#include "zr_launch.cuh"
#include "zr_tc.cuh"

namespace zr {

static inline unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

// A k-step is 16 groups, two slabs of eight.  A's digits are laid out once in
// global memory as the tensor core reads them, per slab [digit][row b][8 g],
// so that a k-step's 32 KB arrive by one bulk copy; the giant steps
// u_g^(128 a) go to giant[a ld + g].
constexpr int kEtcStep = 16;
constexpr uint32_t kEtcPlane = kTcRows * 16;                  // a digit plane of a slab
constexpr uint32_t kEtcSlab = kTcLimbs * kEtcPlane;
constexpr uint32_t kEtcABytes = 2 * kEtcSlab;                 // a k-step's A
constexpr int kEtcNC = 32;                                    // columns of a unit
constexpr uint32_t kEtcBSlab = kTcLimbs * kEtcNC * 16;
constexpr uint32_t kEtcBBytes = 2 * kEtcBSlab;
constexpr int kEtcStages = 5;
constexpr int kEtcChunkSteps = kTcChunk / kEtcStep;
// warps: 8 drain the tensor memory (a lane quadrant and half the columns
// each), one copies A, one issues the MMAs, four make B's digits
constexpr int kEtcDrain = 8, kEtcConv = 4;
constexpr int kEtcThreads = 32 * (kEtcDrain + 2 + kEtcConv);
constexpr size_t kEtcSmem = kEtcStages * (size_t)(kEtcABytes + kEtcBBytes) + 1024;

// Groups g >= G of the last k-step are zero (digits of 0).
__global__ void __launch_bounds__(kTcRows) k_etc_pack(const uint64_t* __restrict__ U, const int64_t* __restrict__ Gdev,
                                                      int A, int64_t ld, Mod M, uint4* __restrict__ pack,
                                                      uint64_t* __restrict__ giant) {
  pdl_enter();
  __shared__ uint64_t sq[12][8], lo[16][8], hi[8][8];         // u^(2^j), u^e, u^(16 h)
  const int64_t G = *Gdev, g0 = (int64_t)blockIdx.x * 8;
  if (g0 >= (G + kEtcStep - 1) / kEtcStep * kEtcStep) return;
  const int t = threadIdx.x, q = t & 7, e = t >> 3;
  const bool in = g0 + q < G;
  if (t < 8) {
    uint64_t x = in ? U[g0 + q] : 0;
    for (int j = 0; j < 12; j++) {
      sq[j][q] = x;
      x = mul_mod(x, x, M);
    }
  }
  __syncthreads();
  // u^(e 2^j0) from the squares
  auto power = [&](int e, int j0) {
    uint64_t x = 1;
    for (int j = j0; e; j++, e >>= 1)
      if (e & 1) x = x == 1 ? sq[j][q] : mul_mod(x, sq[j][q], M);
    return x;
  };
  lo[e][q] = in ? power(e, 0) : 0;
  if (e < 8) hi[e][q] = power(e, 4);
  if (in && e < A) {
    // sixteen chains along the giant steps
    uint64_t x = power(e, 7);
    const uint64_t w = sq[11][q], wq = shoup_pre(w, M);
    for (int a = e; a < A; a += 16) {
      giant[(int64_t)a * ld + g0 + q] = x;
      x = canon(shoup_lazy(x, w, wq, M), M);
    }
  }
  __syncthreads();
  uint64_t x[8];
#pragma unroll
  for (int k = 0; k < 8; k++) x[k] = mul_mod(lo[t & 15][k], hi[t >> 4][k], M);
  uint4 d[kTcLimbs];
  tc_digits(x, M.p, d);
  uint4* dst = pack + (int64_t)blockIdx.x * (kEtcSlab / 16) + t;
#pragma unroll
  for (int i = 0; i < kTcLimbs; i++) dst[i * kTcRows] = d[i];
}

// The giant steps of the next slab of rows (kEtcSlabRows): times u_g^stride,
// the exponent of a whole slab.  A thread takes one group and kEtcNextRows rows.
constexpr int kEtcNextRows = 16;
__global__ void __launch_bounds__(256) k_etc_next(const uint64_t* __restrict__ U, const int64_t* __restrict__ Gdev,
                                                  int A, int64_t ld, int64_t stride, Mod M,
                                                  uint64_t* __restrict__ giant) {
  pdl_enter();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= *Gdev) return;
  const uint64_t w = pow_mod(U[g], (uint64_t)stride, M), wq = shoup_pre(w, M);
  const int a0 = blockIdx.y * kEtcNextRows;
  for (int a = a0; a < A && a < a0 + kEtcNextRows; a++) {
    uint64_t* x = giant + (int64_t)a * ld + g;
    *x = canon(shoup_lazy(*x, w, wq, M), M);
  }
}

// A work unit is 32 columns (a, s) (column index a S + s) and the k-steps of
// one split; units of one split are neighbours, so that the CTAs at work read
// the same part of A.  One persistent CTA per SM walks them through a ring of
// five stages that runs on from unit to unit: bulk copies of A, digits of B
// made by four warps (two k-steps in turn) and the MMAs of zr_tc.cuh.
//
// The shared memory bounds the MMAs: a k-step reads A's 32 KB once and B's 8 KB
// for each of A's digits, and 40 KB come in, about 1060 clocks at 128 bytes
// against the tensor core's 1024.  (Two halves of 16 columns with tensor memory
// of their own would hide the drains, but read A for each: 1440 clocks a
// k-step, measured slower in all, 0.31 against 0.26 ms at T = 10^4, S = 21.)
//
// Every wait is bounded; on a timeout the roles leave their loops, the copies
// in flight are waited for and the tensor memory is given back.
__global__ void __launch_bounds__(kEtcThreads, 1)
    k_eval_tc(int64_t T, int S, const int64_t* __restrict__ Gdev, int A, int64_t ld, int tiles, int gsplit,
              const unsigned char* __restrict__ pack, const uint64_t* __restrict__ giant,
              const uint64_t* __restrict__ W, const uint64_t* __restrict__ Wq, Mod M, TcMod K, uint64_t* __restrict__ out, int64_t ldo,
              uint64_t* __restrict__ partial, uint32_t* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char esm[];
  unsigned char* As = esm;
  unsigned char* Bs = esm + kEtcStages * kEtcABytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(esm + kEtcStages * (kEtcABytes + kEtcBBytes));
  uint64_t *fullA = bars, *fullB = bars + kEtcStages, *empty = bars + 2 * kEtcStages, *tfull = bars + 3 * kEtcStages,
           *tempty = tfull + 1;
  uint64_t* done = tempty + 1;
  uint32_t* slot = reinterpret_cast<uint32_t*>(done + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_enter();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kEtcStages; s++) {
      mbar_init(&fullA[s], 1);
      mbar_init(&fullB[s], 2);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, kEtcDrain);
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == kEtcDrain + 1) tc_alloc(slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  const int64_t G = *Gdev;
  const int64_t steps = (G + kEtcStep - 1) / kEtcStep;
  const int gs = eval_tc_splits(gsplit, G), units = tiles * gs;
  // unit u: its first column, first k-step and k-steps
  auto unit = [&](int u, int& col0, int& split, int64_t& klo, int& n) {
    split = u / tiles;
    col0 = (u - split * tiles) * kEtcNC;
    klo = steps * split / gs;
    n = (int)(steps * (split + 1) / gs - klo);
  };
  int col0, split, n;
  int64_t klo;
  int t = 0;                       // k-steps through the ring so far

  if (warp < kEtcDrain) {
    // ---- tensor memory -> integer sums -> residues
    const int half = warp >> 2, b = 32 * (warp & 3) + lane;
    const uint32_t addr = tmem + ((uint32_t)(warp & 3) << 21) + half * 16;
    bool ok = true;
    uint32_t ph = 0;
    for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
      unit(u, col0, split, klo, n);
      TcAcc acc[16];
#pragma unroll
      for (int c = 0; c < 16; c++) acc[c] = TcAcc{{0, 0, 0, 0, 0, 0}};
      for (int k = 0; k < n; k += kEtcChunkSteps, ph ^= 1) {
        if (!tc_wait(tfull, ph)) {
          atomicOr(status, ST_TIMEOUT);
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < 16; c += 4) tc_add_chunk<kEtcNC>(addr + c, acc + c);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
        if ((k / kEtcChunkSteps) % kTcCarryChunks == kTcCarryChunks - 1) {
#pragma unroll
          for (int c = 0; c < 16; c++) tc_carry(acc[c]);
        }
      }
      if (!ok) break;
      int a = (col0 + half * 16) / S, s = col0 + half * 16 - a * S;
#pragma unroll
      for (int c = 0; c < 16; c++) {
        const int64_t i = (int64_t)a * kTcRows + b;
        if (a < A && i < T) {
          const uint64_t r = tc_value(acc[c], K, M);
          if (gsplit == 1) out[(int64_t)s * ldo + i] = r;
          else partial[((int64_t)split * S + s) * T + i] = r;
        }
        if (++s == S) s = 0, a++;
      }
    }
  } else if (warp == kEtcDrain) {
    // ---- A: one bulk copy per k-step
    if (lane == 0) {
      bool ok = true;
      for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
        unit(u, col0, split, klo, n);
        for (int k = 0; k < n; k++, t++) {
          const int st = t % kEtcStages;
          if (t >= kEtcStages && !mbar_wait(&empty[st], ((t / kEtcStages) & 1) ^ 1)) {
            atomicOr(status, ST_TIMEOUT);
            ok = false;
            break;
          }
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&fullA[st])),
                       "r"(kEtcABytes)
                       : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                  smem_addr(As + st * kEtcABytes)),
              "l"(pack + (klo + k) * (int64_t)kEtcABytes), "r"(kEtcABytes), "r"(smem_addr(&fullA[st]))
              : "memory");
        }
      }
      // the copies in flight land before the CTA may leave
      for (int w = t > kEtcStages ? t - kEtcStages : 0; w < t; w++)
        mbar_wait(&fullA[w % kEtcStages], (w / kEtcStages) & 1);
    }
  } else if (warp == kEtcDrain + 1) {
    // ---- MMAs: the whole warp runs the loop, so that the descriptors stay in
    // uniform registers; one lane issues
    const bool leader = tc_elect();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    uint32_t ch = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
      unit(u, col0, split, klo, n);
      for (int k = 0; k < n; k++, t++) {
        const int st = t % kEtcStages;
        const bool first = k % kEtcChunkSteps == 0, last = k % kEtcChunkSteps == kEtcChunkSteps - 1 || k == n - 1;
        const uint32_t ph = (t / kEtcStages) & 1;
        if ((first && ch > 0 && !tc_wait(tempty, (ch - 1) & 1)) || !tc_wait(&fullA[st], ph) ||
            !tc_wait(&fullB[st], ph)) {
          if (leader) atomicOr(status, ST_TIMEOUT);
          ok = false;
          break;
        }
        tc_fence_after();
        if (leader) {
          tc_kstep<kEtcNC>(tm, smem_addr(As) + st * kEtcABytes, kEtcPlane, kEtcSlab, smem_addr(Bs) + st * kEtcBBytes,
                           kEtcBSlab, first);
          tc_commit(&empty[st]);
          if (last) tc_commit(tfull);
        }
        __syncwarp();
        ch += last;
      }
    }
    // the MMAs issued have completed before the tensor memory goes back
    if (leader) tc_commit(done);
    mbar_wait(done, 0);
  } else {
    // ---- B: warp (slab, k-steps t = set mod 2), lane = column
    const int cw = warp - (kEtcDrain + 2), slab = cw & 1, set = cw >> 1;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
      unit(u, col0, split, klo, n);
      const int col = col0 + lane, a = col / S, s = col - a * S;
      const bool live = a < A;
      const uint64_t *wr = W + (int64_t)s * ld, *qr = Wq + (int64_t)s * ld, *gr = giant + (int64_t)a * ld;
      // eight groups of the weights, their Shoup quotients and the giant steps
      // (rows 128-byte aligned: ld a multiple of 16)
      ulonglong2 w[4], wq[4], v[4];
      auto load = [&](int k) {
        const int64_t g = (klo + k) * kEtcStep + slab * 8;
        const bool in = live && k < n;
#pragma unroll
        for (int q = 0; q < 4; q++) {
          w[q] = in ? __ldg(reinterpret_cast<const ulonglong2*>(wr + g) + q) : make_ulonglong2(0, 0);
          wq[q] = in ? __ldg(reinterpret_cast<const ulonglong2*>(qr + g) + q) : make_ulonglong2(0, 0);
          v[q] = in ? __ldg(reinterpret_cast<const ulonglong2*>(gr + g) + q) : make_ulonglong2(0, 0);
        }
      };
      const int k0 = (set + t) & 1;               // this set's first k-step of the unit
      load(k0);
      for (int k = k0; k < n; k += 2) {
        const int tt = t + k, st = tt % kEtcStages;
        const int64_t g = (klo + k) * kEtcStep + slab * 8;
        uint64_t x[8];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          x[2 * q] = g + 2 * q < G ? canon(shoup_lazy(v[q].x, w[q].x, wq[q].x, M), M) : 0;
          x[2 * q + 1] = g + 2 * q + 1 < G ? canon(shoup_lazy(v[q].y, w[q].y, wq[q].y, M), M) : 0;
        }
        load(k + 2);
        uint4 d[kTcLimbs];
        tc_digits(x, M.p, d);
        if (tt >= kEtcStages && !tc_wait(&empty[st], ((tt / kEtcStages) & 1) ^ 1)) {
          atomicOr(status, ST_TIMEOUT);
          ok = false;
          break;
        }
        uint4* dst = reinterpret_cast<uint4*>(Bs + st * kEtcBBytes + slab * kEtcBSlab) + lane;
#pragma unroll
        for (int j = 0; j < kTcLimbs; j++) dst[j * kEtcNC] = d[j];
        tc_fence_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&fullB[st]);
      }
      t += n;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  __syncwarp();
  if (warp == kEtcDrain + 1) tc_dealloc(tmem, 512);
}

// Scratch: the packed digits, the giant steps, the weights, the partial sums
// of the k splits.  The giant steps, a row of ld words per 128 probes, are held
// for one slab of probes at a time (256 MB at most, 2^15 rows: 16384 probes or
// more, since ld <= 2^18), so that the scratch does not grow with T; the next
// slab's come from this one's by a product each, one for 128 S of its products.
constexpr int64_t kEtcGiantWords = 1ll << 25, kEtcSlabRows = 1ll << 15;
static int etc_a(int64_t T) { return (int)((T + kTcRows - 1) / kTcRows); }
int64_t eval_tc_ld(int64_t Tn) { return (Tn + kEtcStep - 1) / kEtcStep * kEtcStep; }
int64_t eval_tc_slab(int64_t Tn, int64_t T) {
  const int64_t rows = std::min(kEtcSlabRows, std::max<int64_t>(1, kEtcGiantWords / eval_tc_ld(Tn)));
  return std::min(T, rows * kTcRows);
}

// k splits: the count with the shortest longest CTA, in k-steps' time: a unit
// costs its k-steps, three more for every chunk of eight (the drain) and eight
// for its start and end.
static int etc_split(const zr_ctx* ctx, int64_t T, int S, int64_t Tn) {
  const int64_t tiles = cdiv((int64_t)etc_a(T) * S, kEtcNC), steps = eval_tc_ld(Tn) / kEtcStep;
  const int64_t sms = ctx && ctx->sms ? ctx->sms : 152;
  int best = 1;
  int64_t cost = 0;
  for (int gs = 1; gs <= 64 && (gs == 1 || steps / gs >= 4); gs++) {
    const int64_t per = (steps + gs - 1) / gs;
    const int64_t c = (tiles * gs + sms - 1) / sms * (per + 3 * ((per + 7) / 8) + 8) + gs / 4;
    if (gs == 1 || c < cost) best = gs, cost = c;
  }
  return best;
}

EvalTcWs carve_eval_tc(Carver& cv, const zr_ctx* ctx, int64_t Tn, int S, int64_t T) {
  EvalTcWs w;
  const int64_t ld = eval_tc_ld(Tn);
  T = eval_tc_slab(Tn, T);
  w.gsplit = etc_split(ctx, T, S, Tn);
  w.W = cv.take<uint64_t>((size_t)S * ld);
  w.Wq = cv.take<uint64_t>((size_t)S * ld);
  w.giant = cv.take<uint64_t>((size_t)etc_a(T) * ld);
  w.pack = cv.take<unsigned char>((size_t)(ld / 8) * kEtcSlab);
  w.partial = cv.take<uint64_t>(w.gsplit > 1 ? (size_t)w.gsplit * S * T : 1);
  return w;
}

void launch_eval_tc(zr_ctx* ctx, const EvalTcWs& w, const int64_t* Gdev, int64_t Tn, const uint64_t* U, int S, int64_t t0,
                    int64_t T, uint64_t* out, int64_t ldo, uint32_t* status, cudaStream_t st) {
  static DeviceOnce attr;
  attr.run([] { cudaFuncSetAttribute(k_eval_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEtcSmem); });
  const Mod& M = ctx->M;
  const int64_t ld = eval_tc_ld(Tn);
  const int A = etc_a(T);
  const TcMod K = tc_mod(M);
  if (t0 == 0)
    launch_k(k_etc_pack, dim3((unsigned)(ld / 8)), dim3(kTcRows), 0, st, U, Gdev, A, ld, M, (uint4*)w.pack, w.giant);
  else
    launch_k(k_etc_next, dim3(cdiv(ld, 256), cdiv(A, kEtcNextRows)), dim3(256), 0, st, U, Gdev, A, ld,
             eval_tc_slab(Tn, t0), M, w.giant);
  const int tiles = (int)cdiv((int64_t)A * S, kEtcNC), sms = ctx->sms ? ctx->sms : 152;
  launch_k(k_eval_tc, dim3((unsigned)std::min(tiles * w.gsplit, sms)), dim3(kEtcThreads), kEtcSmem, st, T, S, Gdev, A,
           ld, tiles, w.gsplit, (const unsigned char*)w.pack, (const uint64_t*)w.giant, (const uint64_t*)w.W,
           (const uint64_t*)w.Wq, M, K, out + t0, ldo, w.partial, status);
  note_launches(2);
}

}  // namespace zr
