// digits.cuh -- exact products on the 5th-generation tensor cores: an array
// element is written as a fixed-point integer relative to its column's
// largest magnitude and cut into signed 8-bit digits, which binary16 holds
// exactly; a tcgen05 kind::f16 product of two digit planes accumulated over
// at most 128 rows stays below 2^24, so its binary32 accumulator is exact.
// The products of equal weight ("level" s + t of digits s and t) share an
// accumulator, and the levels are combined in 64-bit integers.  This is the
// error-free splitting of Ozaki, Ogita, Oishi and Rump ("Error-free
// transformations of matrix multiplication", 2012) with integer digits.
//
//   binary64: 62 bits below the column's largest power of two, 8 digits;
//             elements within 2^9 of the column maximum are exact.
//   binary32: 38 bits, 5 digits.
//
// Layout of a digit plane in shared memory: K-major, no swizzle, core
// matrices of 8 rows x 8 binary16 (128 contiguous bytes), kStK = 32 elements
// of K per pipeline stage: core (a, b) at a * kPlaneSbo + b * 128.
#pragma once
#include "kernels.h"
#include "tc05.cuh"

namespace pylom {

constexpr int kStK = 32;                     // K elements per stage
constexpr int kPlaneSbo = (kStK / 8) * 128;  // bytes between 8-row groups
constexpr int kPlaneA = 128 * kStK * 2;      // 8 KB: 128 rows
constexpr int kPlaneB = 64 * kStK * 2;       // 4 KB: 64 rows
constexpr int kStagesPerSum = 4;             // stages accumulated before the sums are read: 128 elements of K
constexpr int kSlots = 8;                    // accumulators (levels) of 64 columns in tensor memory

template <typename TY> struct Dig;
template <> struct Dig<double> {
  static constexpr int S = 8;          // digits
  static constexpr int NST = 2;        // pipeline stages
  static constexpr int HALVES = 2;     // level ranges of the Gram kernel: 0..7 and 8..14
  static constexpr int LBM = 7;        // lowest level of the modes kernel
};
template <> struct Dig<float> {
  static constexpr int S = 5;
  static constexpr int NST = 3;
  static constexpr int HALVES = 1;     // levels 1..8 (level 0 lies 2^-60 below the top one)
  static constexpr int LBM = 1;
};
// lowest level of range `half` of the Gram kernel
template <typename TY> __host__ __device__ constexpr int gram_base(int half) { return sizeof(TY) == 8 ? 8 * half : 1; }
// y = v 2^(E - kFixBias): the fixed-point value v of an element of a column with exponent field E
template <typename TY> __host__ __device__ constexpr int fix_bias() { return sizeof(TY) == 8 ? 1084 : 164; }

// biased exponent field of |y| (at least 1, so subnormals share the lowest one)
__device__ __forceinline__ int exp_field(double y) {
  const int e = (__double2hiint(y) >> 20) & 0x7ff;
  return e > 1 ? e : 1;
}
__device__ __forceinline__ int exp_field(float y) {
  const int e = (__float_as_int(y) >> 23) & 0xff;
  return e > 1 ? e : 1;
}
// fixed-point value of y in a column whose largest exponent field is E: |v| < 2^62 (binary64), < 2^38 (binary32)
__device__ __forceinline__ int64_t to_fixed(double y, int E) {
  const uint32_t hi = (uint32_t)__double2hiint(y), lo = (uint32_t)__double2loint(y);
  const int e = (hi >> 20) & 0x7ff;
  const uint32_t mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  uint64_t m = (((uint64_t)mh << 32) | lo) << 9;
  const int sh = E - (e > 1 ? e : 1);
  m = sh < 63 ? m >> sh : 0;
  const int64_t sg = -(int64_t)(hi >> 31);
  return ((int64_t)m ^ sg) - sg;
}
__device__ __forceinline__ int64_t to_fixed(float y, int E) {
  const uint32_t b = (uint32_t)__float_as_int(y);
  const int e = (b >> 23) & 0xff;
  uint64_t m = (uint64_t)((b & 0x7fffffu) | (e ? 0x800000u : 0u)) << 14;
  const int sh = E - (e > 1 ? e : 1);
  m = sh < 63 ? m >> sh : 0;
  const int64_t sg = -(int64_t)(b >> 31);
  return ((int64_t)m ^ sg) - sg;
}

// Signed digits of v: v + B with 0x80 in every byte, byte k minus 128 is
// digit k in [-128, 127] (the top one in [-64, 64]).
__device__ __forceinline__ uint64_t bias_digits(int64_t v) { return (uint64_t)v + 0x8080808080808080ull; }
// digit k of two biased values as a binary16 pair: 1024 + byte by bit
// pattern, minus 1152
__device__ __forceinline__ uint32_t digit_pair(uint32_t wa, uint32_t wb, uint32_t sel) {
  const uint32_t x = (__byte_perm(wa, wb, sel) & 0x00ff00ffu) | 0x64006400u;
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0x64806480u));
  return r;
}
// all digits of eight values, digit s as one 16-byte store at dst + s * plane
template <int S>
__device__ __forceinline__ void store_digits(const uint64_t (&w)[8], unsigned char* dst, int plane) {
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const uint32_t sel = (uint32_t)((s & 3) | ((4 + (s & 3)) << 8));
    uint32_t d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t a = s < 4 ? (uint32_t)w[2 * i] : (uint32_t)(w[2 * i] >> 32);
      const uint32_t b = s < 4 ? (uint32_t)w[2 * i + 1] : (uint32_t)(w[2 * i + 1] >> 32);
      // bytes: [a.k, a.0, b.k, b.0]; the odd ones are masked off
      d[i] = digit_pair(a, b, (sel & 0xfu) | ((sel >> 8) & 0xfu) << 8);
    }
    *(uint4*)(dst + s * plane) = make_uint4(d[0], d[1], d[2], d[3]);
  }
}

// instruction descriptor of kind::f16: D binary32, A and B binary16, K-major
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t da, uint64_t db, uint32_t idesc, bool acc) {
  const uint32_t a = acc ? 1u : 0u;
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               :: "r"(dtmem), "l"(da), "l"(db), "r"(idesc), "r"(a));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tc05::smem_u32(mbar)) : "memory");
}

// One thread: all digit products of one stage with level LB <= s + t < LB + 8
// into the eight accumulators of 64 columns; `first`: the stage starts new
// sums.  Descriptors advance 256 bytes per K = 16 step.
template <int S, int LB>
__device__ __forceinline__ void issue_stage(uint32_t tmem, uint64_t dA, uint64_t dB, int planeB, bool first) {
  constexpr uint32_t id = idesc_f16(128, 64);
#pragma unroll
  for (int sl = 0; sl < kSlots; ++sl) {
    const int l = LB + sl;
    bool acc = !first;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int t = l - s;
      if (t < 0 || t >= S) continue;
#pragma unroll
      for (int ks = 0; ks < kStK / 16; ++ks) {
        mma_f16(tmem + sl * 64, dA + (uint64_t)((s * kPlaneA + ks * 256) >> 4),
                dB + (uint64_t)((t * planeB + ks * 256) >> 4), id, acc);
        acc = true;
      }
    }
  }
}

// 16 columns of one accumulator, no wait
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr));
}

// Adds the eight accumulators (exact integers) of this thread's row and 16
// columns into acc0 (levels 0..3 of the range) and acc1 (levels 4..7).
__device__ __forceinline__ void drain_slots(uint32_t taddr, int nslots, int64_t (&acc0)[16], int64_t (&acc1)[16]) {
#pragma unroll
  for (int sl = 0; sl < kSlots; ++sl) {
    if (sl >= nslots) break;
    uint32_t r[16];
    tmem_ld16_nowait(taddr + sl * 64, r);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int64_t p = (int64_t)__float2int_rn(__uint_as_float(r[c])) * (1 << (8 * (sl & 3)));
      if (sl < 4) acc0[c] += p;
      else acc1[c] += p;
    }
  }
}

// waits that first look once, without reading the clock
__device__ __forceinline__ bool mbar_wait_fast(uint64_t* mbar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
               "selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(done) : "r"(tc05::smem_u32(mbar)), "r"(parity) : "memory");
  return done ? true : tc05::mbar_wait(mbar, parity);
}

}  // namespace pylom
