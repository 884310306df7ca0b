// zr_tc.cuh -- exact products of 63-bit residues on the tensor cores.
//
// A residue x, taken centred (|x| <= p / 2 < 2^62), is written in eight
// balanced base-256 digits, x = sum_i d_i 256^i with -128 <= d_i <= 127 (or
// any 64-bit word y as y - 0x8080..80, the constant corrected later); every
// digit is exact in bf16 (eight significand bits).  A sum over k <= 128 of
// products x_k y_k has the antidiagonal sums
//     D_m = sum_k sum_{i+j=m} d_i(x_k) d_j(y_k),   m = 0 .. 14,
// of at most 8 * 128 products below 2^14: |D_m| <= 2^24, so every partial sum
// is an integer that an fp32 accumulator holds exactly, in any order.  With
// the eight digit planes of y side by side along N (B, N = 8 NC) and D_m in
// the columns m NC .. m NC + NC - 1 of the accumulator, digit i of x is one
// MMA whose accumulator starts i NC columns to the right: eight MMAs of N =
// 8 NC per 16 k give all fifteen sums of 128 x NC outputs.  Every 128 k the
// sums leave the tensor memory and join multi-word integers (TcAcc).
//
// Per SM that is 64 residue products per clock at the tensor core's bf16 rate
// against 7.2 on the integer pipe (eight 32-bit multiply-adds each).
//
// Operands lie in shared memory in the K-major layout without swizzle: core
// matrices of 8 rows x 16 bytes, rows 16 bytes apart, so that the digits of
// eight consecutive k of a row are one 16-byte store (kTcSbo apart per 8 rows).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "zr_arith.cuh"
#include "zr_ring.cuh"

namespace zr {

constexpr int kTcLimbs = 8;
constexpr int kTcDiags = 2 * kTcLimbs - 1;
constexpr int kTcRows = 128;        // rows of a tile: the tensor memory's lanes
constexpr int kTcChunk = 128;       // k summed in the tensor memory at a time (the bound above)

// Digits of eight words y (consecutive k of one row): out[i] holds byte i less
// 128 of all eight as bf16, the digits of y - 0x8080..80.  A byte b becomes b -
// 128 through the bf16 numbers 128 + (b & 127) and 128 or 256 (ulp 1 in [128,
// 256)).
constexpr uint64_t kTcBias = 0x8080808080808080ull;
__device__ __forceinline__ void tc_bytes(const uint64_t (&y)[8], uint4 (&out)[kTcLimbs]) {
#pragma unroll
  for (int i = 0; i < kTcLimbs; i++) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint32_t a = i < 4 ? lo32(y[2 * q]) : hi32(y[2 * q]), b = i < 4 ? lo32(y[2 * q + 1]) : hi32(y[2 * q + 1]);
      const uint32_t two = __byte_perm(a, b, 0x4400u + 0x1111u * (i & 3));   // bytes i, i of a; i, i of b
      const uint32_t u = (two & 0x007f007fu) | 0x43004300u, v = (~two & 0x00800080u) | 0x43004300u;
      __nv_bfloat162 du, dv;
      memcpy(&du, &u, 4);
      memcpy(&dv, &v, 4);
      const __nv_bfloat162 d = __hsub2(du, dv);
      memcpy(&w[q], &d, 4);
    }
    out[i] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}
// Digits of eight residues, centred: at most 65 in magnitude for the top one.
__device__ __forceinline__ void tc_digits(const uint64_t (&x)[8], uint64_t p, uint4 (&out)[kTcLimbs]) {
  const uint64_t half = p >> 1;
  uint64_t y[8];
#pragma unroll
  for (int k = 0; k < 8; k++) y[k] = (x[k] > half ? x[k] - p : x[k]) + kTcBias;
  tc_bytes(y, out);
}

// ---- tcgen05 ---------------------------------------------------------------------

__device__ __forceinline__ void tc_alloc(uint32_t* slot, uint32_t cols) {   // one whole warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(uint32_t tmem, uint32_t cols) {   // the same warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
// generic-proxy writes to shared memory before the tensor core reads them
__device__ __forceinline__ void tc_fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// A bounded wait of a whole warp: its lanes go on, or give up, together (the
// instructions behind it are the warp's).
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}
// one lane of a converged warp
__device__ __forceinline__ bool tc_elect() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r;
}
// arrives on `bar` when the MMAs issued so far by this thread have completed
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}
// Descriptor of a K-major operand without swizzle at shared address `addr`:
// lbo bytes between core matrices along k, sbo bytes along the rows.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)((lbo >> 4) & 0x3fffu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3fffu) << 32) | (1ull << 46);
}
// bf16 x bf16 -> fp32, both K-major, M = 128
__device__ __forceinline__ constexpr uint32_t tc_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTcRows >> 4) << 24);
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
// One 16-deep k-step: digit planes of A a_plane bytes apart, B's planes
// together (NC rows each), core matrices a_lbo and b_lbo bytes apart along k.
// first: the chunk's first k-step, whose MMAs overwrite the columns nothing
// has written yet.
template <int NC>
__device__ __forceinline__ void tc_kstep(uint32_t tmem, uint32_t a, uint32_t a_plane, uint32_t a_lbo, uint32_t b,
                                         uint32_t b_lbo, bool first) {
  const uint64_t bd = tc_desc(b, b_lbo, 128);
  if (!first) {
#pragma unroll
    for (int i = 0; i < kTcLimbs; i++)
      tc_mma(tmem + i * NC, tc_desc(a + i * a_plane, a_lbo, 128), bd, tc_idesc(kTcLimbs * NC), true);
    return;
  }
  tc_mma(tmem, tc_desc(a, a_lbo, 128), bd, tc_idesc(kTcLimbs * NC), false);
  const uint64_t btop = tc_desc(b + (kTcLimbs - 1) * NC * 16, b_lbo, 128);
#pragma unroll
  for (int i = 1; i < kTcLimbs; i++) {
    const uint64_t ad = tc_desc(a + i * a_plane, a_lbo, 128);
    tc_mma(tmem + i * NC, ad, bd, tc_idesc((kTcLimbs - 1) * NC), true);
    tc_mma(tmem + (i + kTcLimbs - 1) * NC, ad, btop, tc_idesc(NC), false);
  }
}
// four consecutive columns of this lane (the warp's quadrant is in `addr`)
__device__ __forceinline__ void tc_ld4(uint32_t addr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr));
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---- sums of chunks -----------------------------------------------------------------

// A signed integer sum_g w[g] 2^(24 g); every added chunk changes a word by
// less than 2^23.1, so that tc_carry is due after at most 200 chunks.
struct TcAcc {
  int32_t w[6];
};
constexpr int kTcCarryChunks = 128;
__device__ __forceinline__ void tc_carry(TcAcc& a) {
#pragma unroll
  for (int g = 0; g < 5; g++) {
    const int32_t c = a.w[g] >> 24;
    a.w[g] -= c << 24;
    a.w[g + 1] += c;
  }
}
// The chunk sums D_0 .. D_14 of four columns (addr + m NC + c) added into acc.
//
// Sum by sum the excess over a balanced digit is carried on, D_m = 256 q + r,
// q = round(D_m / 256) added to D_{m+1}, all exact: one operand at least is
// centred, its top digits at most 65 in magnitude, so |D_m| <= 128 (7 * 2^14 +
// 128 * 65) < 2^24 - 2^17 leaves room for the carry, and q + 3 * 2^22 rounds
// to an integer.  Three digits make a 24-bit word, one conversion to integer each:
// conversions run at 16 lanes per SM and clock, and fifteen of them with
// 64-bit additions took 4430 clocks per 128 x 32 outputs, this 3300.
template <int NC>
__device__ __forceinline__ void tc_add_chunk(uint32_t addr, TcAcc* acc) {
  constexpr float kMagic = 12582912.0f;            // 3 * 2^22
  float carry[4] = {0, 0, 0, 0};
#pragma unroll
  for (int g = 0; g < 5; g++) {
    uint32_t v[3][4];
#pragma unroll
    for (int m = 0; m < 3; m++) tc_ld4(addr + (3 * g + m) * NC, v[m]);
    tc_wait_ld();
#pragma unroll
    for (int c = 0; c < 4; c++) {
      float r[3];
#pragma unroll
      for (int m = 0; m < 3; m++) {
        const float d = __fadd_rn(__uint_as_float(v[m][c]), carry[c]);
        carry[c] = __fsub_rn(__fmaf_rn(d, 1.0f / 256.0f, kMagic), kMagic);
        r[m] = __fmaf_rn(carry[c], -256.0f, d);
      }
      acc[c].w[g] += __float2int_rn(__fmaf_rn(r[2], 65536.0f, __fmaf_rn(r[1], 256.0f, r[0])));
      if (g == 4) acc[c].w[5] += __float2int_rn(carry[c]);
    }
  }
}
// The residue of a sum of magnitude below 2^150, carried: the words below the
// top one are then in [0, 2^24), so that the low 96 bits are nonnegative and
// their high word is below 2^32 < p, as reduce128 wants it for every prime.
// c96 = 2^96 mod p, bias = 2^154 mod p (the offset that makes the top part
// positive).
struct TcMod {
  uint64_t c96, bias;
};
TcMod tc_mod(const Mod& M);   // host
__device__ __forceinline__ uint64_t tc_value(TcAcc a, const TcMod& K, const Mod& M) {
  tc_carry(a);
  const int64_t x0 = (int64_t)a.w[0] + ((int64_t)a.w[1] << 24), x1 = (int64_t)a.w[2] + ((int64_t)a.w[3] << 24),
                x2 = (int64_t)a.w[4] + ((int64_t)a.w[5] << 24);
  const unsigned __int128 lo = (unsigned __int128)(uint64_t)x0 + ((unsigned __int128)(uint64_t)x1 << 48);
  const uint64_t r0 = reduce128((uint64_t)(lo >> 64), (uint64_t)lo, M);
  const uint64_t r2 = mul_mod(reduce128(0, (uint64_t)(x2 + (1ll << 58)), M), K.c96, M);
  return sub_mod(add_mod(r0, r2, M), K.bias, M);
}

}  // namespace zr
