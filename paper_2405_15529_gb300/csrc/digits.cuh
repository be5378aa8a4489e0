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
// Rows that are small in every column would keep few of those bits, so a row
// has a shift (row_scale_kernel, gram.cu): how far its largest element lies
// below its column's power of two.  The product Y C takes rows times 2^shift;
// a sum over rows takes every row at its columns' scale.
//
// Layout of a digit plane in shared memory: K-major, no swizzle, core
// matrices of 8 rows x 8 binary16 (128 contiguous bytes), kStK = 16 elements
// of K per pipeline stage: core (a, b) at a * kPlaneSbo + b * 128.
#pragma once
#include "kernels.h"
#include "tc05.cuh"

namespace pylom {

constexpr int kStK = 16;                     // K elements per stage
constexpr int kPlaneSbo = (kStK / 8) * 128;  // bytes between 8-row groups
constexpr int kPlaneA = 128 * kStK * 2;      // 4 KB: 128 rows
constexpr int kStagesPerSum = 8;             // stages accumulated before the sums are read: 128 elements of K
constexpr int kSlots = 8;                    // accumulators (levels) in tensor memory
// Two shapes of the kernels, by groups of eight warps in a block.
//   G = 2: one block an SM, output tiles of 128 x 64.  An element of the left
//          factor is cut for 64 columns; the groups fill alternate stages.
//   G = 1: two blocks an SM, tiles of 128 x 32, half of the tensor memory each:
//          while one block's warps read its accumulators or write its tile, the
//          MMAs of the other run.
// Long sums want the first (Gram matrix of 1,048,576 x 256: binary64 6.4 ms
// against 8.9, binary32 3.1 against 4.0), short ones the second (131072 x 1056
// in SPOD bins of 64 columns: Gram matrices 3.8 against 2.75 ms, modes 2.9
// against 1.6).
template <int G>
struct Shape {
  static constexpr int THREADS = 256 * G;     // 128 registers a thread: 64 hold the integer sums
  static constexpr int BLOCKS = 3 - G;        // per SM
  static constexpr int TILE = 32 * G;         // rows of the right factor, columns of an output tile
  static constexpr int PLANEB = TILE * kStK * 2;
  static constexpr int TMEM = kSlots * TILE;  // columns of tensor memory
};
constexpr int kRaw = 4;                      // stages of Y on their way in the Gram kernel
template <typename TY> struct Dig;
template <> struct Dig<double> {
  static constexpr int S = 8;          // digits
  template <int G> static constexpr int NST = 2;                  // pipeline stages
  template <int G> static constexpr int AHEAD = G == 1 ? 2 : 3;   // slots of a thread's ring in a product
  static constexpr int HALVES = 2;     // level ranges of the Gram kernel: 0..7 and 8..14
  static constexpr int LBM = 7;        // lowest level of the modes kernel
};
template <> struct Dig<float> {
  static constexpr int S = 5;
  template <int G> static constexpr int NST = G == 1 ? 3 : 4;
  template <int G> static constexpr int AHEAD = 4;
  static constexpr int HALVES = 1;     // levels 1..8 (level 0 lies 2^-60 below the top one)
  static constexpr int LBM = 1;
};
// lowest level of range `half` of the Gram kernel
template <typename TY> __host__ __device__ constexpr int gram_base(int half) { return sizeof(TY) == 8 ? 8 * half : 1; }
// y = v 2^(E - kFixBias): the fixed-point value v of an element of a column with exponent field E
template <typename TY> __host__ __device__ constexpr int fix_bias() { return sizeof(TY) == 8 ? 1084 : 164; }

// Exponent field that a column's scale is taken from, of one element: the
// biased exponent, from a floor on (elements below it count as zero in
// binary64; in binary32 the floor keeps the scale finite and loses nothing).
// (A row's shift can take the scale of a column that lies below 2^-100
// further down; what such a column has in that row counts for less.)
constexpr int kMinField64 = 64, kMinField32 = 8;
// That of infinities and NaN: such a column has no scale, and what is made of it is NaN.
constexpr int kMaxField64 = 2047, kMaxField32 = 255;
template <typename T> __host__ __device__ constexpr int max_field() { return sizeof(T) == 8 ? kMaxField64 : kMaxField32; }
__device__ __forceinline__ double quiet_nan() { return __longlong_as_double(0x7ff8000000000000ll); }
__device__ __forceinline__ int exp_field(double y) {
  const int e = (__double2hiint(y) >> 20) & 0x7ff;
  return e > kMinField64 ? e : kMinField64;
}
__device__ __forceinline__ int exp_field(float y) {
  const int e = (__float_as_int(y) >> 23) & 0xff;
  return e > kMinField32 ? e : kMinField32;
}

// Fixed-point value of y in a column whose largest exponent field is E, with
// 0x80 added to every byte: |v| < 2^62, and byte k minus 128 is the signed
// digit k in [-128, 127] (the top one in [-64, 64]).  An element of exponent
// field 0 (zero, subnormal) is shifted out.
constexpr uint32_t kDigitBias = 0x80808080u;
__device__ __forceinline__ uint2 biased_fixed(double y, int E) {
  const uint32_t hi = (uint32_t)__double2hiint(y), lo = (uint32_t)__double2loint(y);
  // E - e: the mantissa bits cannot borrow from the exponent's
  const uint32_t sh = min((((uint32_t)E << 20 | 0xfffffu) - (hi & 0x7fffffffu)) >> 20, 63u);
  uint32_t m1 = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 9), m0 = lo << 9;
  const bool far = sh >= 32;
  m0 = far ? m1 : m0;
  m1 = far ? 0u : m1;
  m0 = __funnelshift_r(m0, m1, sh);          // by sh mod 32
  m1 >>= (sh & 31);
  const uint32_t sg = (uint32_t)((int32_t)hi >> 31);       // 0 or all ones
  // (m ^ sg) - sg + bias
  uint2 w;
  asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
      : "=r"(w.x), "=r"(w.y)
      : "r"(m0 ^ sg), "r"(m1 ^ sg), "r"(kDigitBias - sg), "r"(kDigitBias));
  return w;
}
constexpr uint64_t kDigitBias64 = ((uint64_t)kDigitBias << 32) | kDigitBias;
__device__ __forceinline__ uint2 bias_digits(int64_t v) {
  const uint64_t w = (uint64_t)v + kDigitBias64;
  return make_uint2((uint32_t)w, (uint32_t)(w >> 32));
}
// the value that a biased word stands for, of a column with exponent field E
__device__ __forceinline__ double from_fixed(uint2 w, int E) {
  const int64_t v = (int64_t)((((uint64_t)w.y << 32) | w.x) - kDigitBias64);
  return scalbn((double)v, E - fix_bias<double>());
}
// the word of the same value with its last `s` bits shifted out (rounded down)
__device__ __forceinline__ uint2 shift_word(uint2 w, uint32_t s) {
  return bias_digits((int64_t)((((uint64_t)w.y << 32) | w.x) - kDigitBias64) >> (s < 63u ? s : 63u));
}
// shift i of eight packed ones
__device__ __forceinline__ uint32_t packed_shift(const uint4& s, int i) {
  return (((const uint32_t*)&s)[i >> 1] >> (16 * (i & 1))) & 0xffffu;
}
__device__ __forceinline__ int64_t to_fixed(double y, int E) {
  const uint2 w = biased_fixed(y, E);
  return (int64_t)((((uint64_t)w.y << 32) | w.x) - kDigitBias64);
}

// All digits of eight values, digit s as one 16-byte store at dst + s * plane
// (and, dst2 given, at dst2 + s * plane2).
// A digit of two values becomes a binary16 pair by its bit pattern (1024 +
// byte: 0x64 above the byte) minus 1152.
__device__ __forceinline__ uint32_t sub_1152(uint32_t x) {
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0x64806480u));
  return r;
}
template <int S>
__device__ __forceinline__ void store_digits(const uint2 (&w)[8], unsigned char* dst, int plane,
                                             unsigned char* dst2 = nullptr, int plane2 = 0) {
#pragma unroll
  for (int s = 0; s < S; s += 2) {
    uint32_t d0[4], d1[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t a = s < 4 ? w[2 * i].x : w[2 * i].y, b = s < 4 ? w[2 * i + 1].x : w[2 * i + 1].y;
      const uint32_t x = __byte_perm(a, b, (s & 2) ? 0x7632 : 0x5410);   // [a.s, a.s+1, b.s, b.s+1]
      d0[i] = sub_1152(__byte_perm(x, 0x64646464u, 0x4240));
      if (s + 1 < S) d1[i] = sub_1152(__byte_perm(x, 0x64646464u, 0x4341));
    }
    *(uint4*)(dst + s * plane) = make_uint4(d0[0], d0[1], d0[2], d0[3]);
    if (s + 1 < S) *(uint4*)(dst + (s + 1) * plane) = make_uint4(d1[0], d1[1], d1[2], d1[3]);
    if (dst2) {
      *(uint4*)(dst2 + s * plane2) = make_uint4(d0[0], d0[1], d0[2], d0[3]);
      if (s + 1 < S) *(uint4*)(dst2 + (s + 1) * plane2) = make_uint4(d1[0], d1[1], d1[2], d1[3]);
    }
  }
}

// What Y holds when the products run: binary32 as it is; binary64 as
// biased fixed-point words (row_scale_kernel).  A word costs 6 byte selections and
// 4 subtractions, a binary64 value 18 more operations of the half-rate
// integer pipe, and the Gram kernel cuts every element about nine times (at
// 256 columns); one pass over Y in place pays for that.
template <typename TY> struct Cell { typedef TY type; };
template <> struct Cell<double> { typedef uint2 type; };
template <typename C> __device__ __forceinline__ C zero_cell();
template <> __device__ __forceinline__ float zero_cell<float>() { return 0.f; }
template <> __device__ __forceinline__ uint2 zero_cell<uint2>() { return make_uint2(kDigitBias, kDigitBias); }

// Eight elements of one column (scale E), or each of its own, as digits in a stage.
__device__ __forceinline__ void put_digits(const uint2 (&w)[8], int, unsigned char* dst, int plane,
                                           unsigned char* dst2, int plane2) {
  store_digits<Dig<double>::S>(w, dst, plane, dst2, plane2);
}
__device__ __forceinline__ void put_digits(const uint2 (&w)[8], const int (&)[8], unsigned char* dst, int plane) {
  store_digits<Dig<double>::S>(w, dst, plane);
}
// Binary32: digits by rounding, top down, in binary32 itself (d = rint(r),
// r <- 256 (r - d), every step exact): three operations a digit on the
// full-rate pipe instead of a 64-bit shift and byte selection on the
// half-rate one.  The top digit is rint(y 2^(132 - E)), at most 64.
__device__ __forceinline__ void put_digits(const float (&y)[8], const int (&E)[8], unsigned char* dst, int plane,
                                           unsigned char* dst2 = nullptr, int plane2 = 0) {
  constexpr int S = Dig<float>::S;
  constexpr float kRound = 12582912.f;   // 1.5 2^23: adding it rounds to an integer
  float r[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) r[i] = y[i] * __int_as_float(min(132 - E[i] + 127, 254) << 23);   // (see kMinField32)
#pragma unroll
  for (int s = S - 1; s >= 0; --s) {
    float d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float t = s == S - 1 ? __fadd_rn(r[i], kRound) : __fmaf_rn(r[i], 256.f, kRound);
      d[i] = __fsub_rn(t, kRound);
      r[i] = s == S - 1 ? __fsub_rn(r[i], d[i]) : __fmaf_rn(r[i], 256.f, -d[i]);
    }
    uint32_t p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(p[i]) : "f"(d[2 * i + 1]), "f"(d[2 * i]));
    *(uint4*)(dst + s * plane) = make_uint4(p[0], p[1], p[2], p[3]);
    if (dst2) *(uint4*)(dst2 + s * plane2) = make_uint4(p[0], p[1], p[2], p[3]);
  }
}
__device__ __forceinline__ void put_digits(const float (&y)[8], int E, unsigned char* dst, int plane,
                                           unsigned char* dst2, int plane2) {
  const int e[8] = {E, E, E, E, E, E, E, E};
  put_digits(y, e, dst, plane, dst2, plane2);
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

// One thread: all digit products of a stage with levels LB .. LB + 7 (s + t,
// up to S - 1 each).  The right factor's planes follow one another with the
// stride of their row groups, so planes t .. t + n - 1 are one operand of 64 n
// rows (of 32 n with G = 1), and their products with plane s go to the n accumulators of the levels
// s + t .., which are neighbours too: one MMA of up to 256 columns.  (An MMA
// reads its left factor from shared memory again: of 64 columns each, the 72
// of a binary64 stage took 4500 clocks, eight warps issuing; the 28 wide ones
// do 2300 clocks of multiplications.)  `first`: the stage starts new sums.
template <int S, int LB, int G>
__device__ __forceinline__ void issue_stage(uint32_t tmem, uint64_t dA, uint64_t dB, bool first) {
  constexpr int T = Shape<G>::TILE, kPlaneB = Shape<G>::PLANEB;
  static_assert(kPlaneB == T / 8 * kPlaneSbo && kStK == 16, "planes of the right factor follow one another; one K step");
#pragma unroll
  for (int i = 0; i < S; ++i) {
    // the first products of a sum touch every level once, and overwrite it:
    // plane 0 (LB = 0) or S - 1 alone, or (S = 5) planes 0 and 4 between them
    const int s = S == 8 ? (LB == 0 ? i : S - 1 - i) : i == 0 ? 0 : i == 1 ? S - 1 : i - 1;
    const int ta = LB > s ? LB - s : 0, tb = LB + 7 - s < S - 1 ? LB + 7 - s : S - 1;
#pragma unroll
    for (int t = ta; t <= tb;) {
      const bool lone = S == 5 && i == 1 && t == 0;     // level 4 of plane 4: plane 0 has been there
      const int n = lone ? 1 : tb - t + 1 < 8 / G ? tb - t + 1 : 8 / G;
      const bool fresh = i == 0 || (S == 5 && i == 1 && t > 0);
      mma_f16(tmem + (s + t - LB) * T, dA + (uint64_t)((s * kPlaneA) >> 4), dB + (uint64_t)((t * kPlaneB) >> 4),
              idesc_f16(128, T * n), !(fresh && first));
      t += n;
    }
  }
}

// 8 columns of one accumulator, no wait
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// Adds the eight accumulators (exact integers) of this thread's row and 16
// columns into acc0 (levels 0..3 of the range) and acc1 (levels 4..7).  The
// next eight columns are on their way while eight are added; a value costs a
// conversion and one 32 x 32 + 64-bit multiply-add (as shift and 64-bit
// addition it was four operations of the half-rate integer pipe).
template <int G>
__device__ __forceinline__ void drain_slots(uint32_t taddr, int nslots, int64_t (&acc0)[16], int64_t (&acc1)[16]) {
  uint32_t r[2][8];
  tmem_ld8_nowait(taddr, r[0]);
#pragma unroll
  for (int q = 0; q < 2 * kSlots; ++q) {
    const int sl = q >> 1, c0 = (q & 1) * 8;
    if (sl >= nslots) break;
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[q & 1][0]), "+r"(r[q & 1][1]), "+r"(r[q & 1][2]), "+r"(r[q & 1][3]), "+r"(r[q & 1][4]),
                   "+r"(r[q & 1][5]), "+r"(r[q & 1][6]), "+r"(r[q & 1][7])
                 :
                 : "memory");
    if (q + 1 < 2 * kSlots) tmem_ld8_nowait(taddr + ((q + 1) >> 1) * Shape<G>::TILE + ((q + 1) & 1) * 8, r[(q + 1) & 1]);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      int64_t& a = sl < 4 ? acc0[c0 + c] : acc1[c0 + c];
      asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a) : "r"(__float2int_rn(__uint_as_float(r[q & 1][c]))), "r"(1 << (8 * (sl & 3))));
    }
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// (acc1 2^32 + acc0) 2^pk, rounded to nearest, by integer operations: the
// conversions of 64-bit integers are binary64 operations, of which this part
// does two a clock.  (Bits below 2^-64 of the value are cut off.)
struct Normal {
  uint64_t m;      // leading bit at 63, or 0
  int ex;          // |value| = m 2^ex
  bool neg;
};
__device__ __forceinline__ Normal normalise(int64_t acc0, int64_t acc1, int pk) {
  const int64_t hi = acc1 + (acc0 >> 32);
  const uint32_t lo = (uint32_t)acc0;
  Normal v;
  v.neg = hi < 0;
  const uint64_t h = v.neg ? ~(uint64_t)hi + (lo == 0) : (uint64_t)hi;
  const uint32_t l = v.neg ? 0u - lo : lo;
  // the upper 64 of the 96 bits, or all that there is
  const uint64_t top = h ? h : (uint64_t)l;
  const int n = __clzll((long long)top);
  const uint64_t below = h ? (uint64_t)l << 32 : 0;
  v.m = n ? (n < 64 ? (top << n) | (below >> (64 - n)) : 0) : top;
  v.ex = pk - n + (h ? 32 : 0);
  return v;
}
__device__ __forceinline__ double from_sums(int64_t acc0, int64_t acc1, int pk, double) {
  const Normal v = normalise(acc0, acc1, pk);
  if (v.m == 0) return 0.0;
  const uint64_t r = (v.m >> 11) + ((v.m >> 10) & 1);        // 53 bits, or 2^53
  const uint64_t sign = (uint64_t)v.neg << 63;
  const int e = v.ex + 11 + 52 + 1023;
  if (e >= 1 && e <= 2045) return __longlong_as_double((long long)(sign | (((uint64_t)(e - 1) << 52) + r)));
  return scalbn(__longlong_as_double((long long)(sign | (((uint64_t)(1023 + 52 - 1) << 52) + r))), v.ex + 11);
}
__device__ __forceinline__ float from_sums(int64_t acc0, int64_t acc1, int pk, float) {
  const Normal v = normalise(acc0, acc1, pk);
  if (v.m == 0) return 0.f;
  const uint32_t r = (uint32_t)(v.m >> 40) + ((uint32_t)(v.m >> 39) & 1u);
  const uint32_t sign = (uint32_t)v.neg << 31;
  const int e = v.ex + 40 + 23 + 127;
  if (e >= 1 && e <= 253) return __uint_as_float(sign | (((uint32_t)(e - 1) << 23) + r));
  return scalbnf(__uint_as_float(sign | (((uint32_t)(127 + 23 - 1) << 23) + r)), v.ex + 40);
}

template <int BYTES>
__device__ __forceinline__ void async_copy(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" :: "r"(tc05::smem_u32(dst)), "l"(src), "n"(BYTES) : "memory");
}

// waits that first look once, without reading the clock
__device__ __forceinline__ bool mbar_wait_fast(uint64_t* mbar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
               "selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(done) : "r"(tc05::smem_u32(mbar)), "r"(parity) : "memory");
  return done ? true : tc05::mbar_wait(mbar, parity);
}

// ---------------------------------------------------------------------------
// the two pipelines
// ---------------------------------------------------------------------------
template <int NST, int G>
struct DigitBarriers {
  uint64_t full[NST], empty[NST], dfull, dempty, issued, fin;
  uint32_t tmem;
  // all threads; `extra`: arrivals on a full barrier besides one per warp of a group
  __device__ __forceinline__ void open(int extra) {
    if (threadIdx.x == 0) {
      for (int b = 0; b < NST; ++b) {
        tc05::mbar_init(full + b, 8 + extra);
        tc05::mbar_init(empty + b, 1);
      }
      tc05::mbar_init(&dfull, G);
      tc05::mbar_init(&issued, 1);
      tc05::mbar_init(&dempty, 8 * G);
      tc05::mbar_init(&fin, 8 * G);
    }
    if (threadIdx.x < 32) tc05::tmem_alloc(&tmem, Shape<G>::TMEM);
    tc05::fence_before();
    __syncthreads();
    tc05::fence_after();
  }
  // all threads: nothing of this block is in flight when it gives its memory back
  __device__ __forceinline__ void close(bool ok, WsHeader* hdr) {
    if ((threadIdx.x & 31) == 0) tc05::commit(&fin);
    if (threadIdx.x == 0 && !mbar_wait_fast(&fin, 0)) ok = false;
    if (!ok) raise_status(hdr, PYLOM_ERR_TIMEOUT);
    tc05::fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tc05::tmem_dealloc(tmem, Shape<G>::TMEM);
  }
};

// Both pipelines: the stages alternate between two groups of eight warps.  A
// group fills its stage (fills wait on loads and on the integer pipe) and one
// thread issues the stage's MMAs when its eight warps are through; the other
// group fills meanwhile.  The MMAs of successive stages go to the same
// accumulators from two threads: a thread issues after the other has issued
// (an mbarrier and the fences around it keep the order), not after those MMAs
// are complete, which left the tensor cores idle for about 1000 clocks a
// stage.  At the end of a sum all sixteen warps read the accumulators; the
// group that fills the next sum's first stage does so before it reads.
//
// A commit covers the MMAs of its own thread, so with two groups the last two
// stages of a sum commit to `dfull` (two arrivals; a sum of one stage commits
// twice).
//
// Deadlock freedom: a group waits for (1) the MMAs of an earlier stage to be
// issued or complete, (2) the reads of an earlier sum by the other group,
// which reads before it fills unless it opens the sum itself, (3) the MMAs of
// the sum it reads, issued once (2) holds for the sums before.  All are
// earlier in the order of stages, and every wait is bounded.
// (Counters are 32-bit and stage numbers advance without divisions.)
template <int NST>
struct StageSlot {      // buffer and phase parity of a stage number
  int b;
  uint32_t par;
  __device__ __forceinline__ void advance(int n) {
    b += n;
    if (b >= NST) {
      b -= NST;
      par ^= 1u;
    }
  }
};

// Issuing stage j (buffer and phase `cur`): the first warp of the group that
// filled it.  `commits`: arrivals on dfull (1 for the last two stages of a
// sum, 2 for the only one, else 0); ahead(): what can start once the stage is
// filled.
template <int NST, int G, class Ahead, class Issue>
__device__ __forceinline__ bool issue_turn(DigitBarriers<NST, G>& bar, const StageSlot<NST>& cur, int j, int sum, bool first,
                                           int commits, uint32_t sa, Ahead ahead, Issue issue) {
  if ((threadIdx.x & 255) >= 32) return true;
  bool ok = true;
  if ((threadIdx.x & 31) == 0) {
    ok = mbar_wait_fast(bar.full + cur.b, cur.par);
    if (ok) ahead();
    if (G > 1 && ok && j > 0) ok = mbar_wait_fast(&bar.issued, (uint32_t)((j - 1) & 1));
    if (ok && first && sum > 0) ok = mbar_wait_fast(&bar.dempty, (uint32_t)((sum - 1) & 1));
    if (ok) {
      tc05::fence_after();
      issue(bar.tmem, sa, first);
      tc05::commit(bar.empty + cur.b);
      for (int c = 0; c < commits; ++c) tc05::commit(&bar.dfull);
      if (G > 1) {
        tc05::fence_before();
        mbar_arrive(&bar.issued);
      }
    }
  }
  return __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
}

template <int NST, int G>
__device__ __forceinline__ bool drain_turn(DigitBarriers<NST, G>& bar, int& drained, int nslots, int64_t (&acc0)[16],
                                           int64_t (&acc1)[16]) {
  const int warp = threadIdx.x >> 5;
  if (!__all_sync(0xffffffffu, mbar_wait_fast(&bar.dfull, (uint32_t)(drained & 1)))) return false;
  tc05::fence_after();
  drain_slots<G>(bar.tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 16, nslots, acc0, acc1);
  tc05::fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(&bar.dempty);
  ++drained;
  return true;
}

// Sums over a range of rows: `nstage` stages of kStK rows, read out every
// kStagesPerSum of them.  fetch(j) brings this thread's part of stage j into
// registers and fill(stage) writes its digits; issue(tensor memory, stage
// address, first) issues the MMAs; flush(acc0, acc1) hands on the 64-bit sums
// of this thread's row and 16 columns.  RAW = 0: fetch loads from global
// memory, a turn ahead.  RAW > 0 (even): it reads a ring of RAW stages in
// shared memory, which copy(j) (one thread, asynchronous) fills RAW stages
// ahead; settle(j) waits for the copies up to stage j, after a timeout.
template <int NST, int RAW, int G, class Copy, class Settle, class Fetch, class Fill, class Issue, class Flush>
__device__ __forceinline__ void gram_pipeline(DigitBarriers<NST, G>& bar, unsigned char* gsm, int stage_bytes, int nstage,
                                              int nslots, WsHeader* hdr, Copy copy, Settle settle, Fetch fetch, Fill fill,
                                              Issue issue, Flush flush) {
  const int lane = threadIdx.x & 31, group = G == 1 ? 0 : threadIdx.x >> 8;
  bar.open(0);
  const uint32_t base = tc05::smem_u32(gsm);
  bool ok = true;
  int64_t acc0[16], acc1[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc0[c] = acc1[c] = 0;
  int drained = 0, copied = group - G;
  auto ahead = [&](int j) {
    if (RAW > 0 && j < nstage) {
      copy(j);
      copied = j;
    }
  };
  if ((threadIdx.x & 255) == 0)
    for (int j = group; j < RAW; j += G) ahead(j);
  StageSlot<NST> cur{group, 0u};
  if (RAW == 0 && group < nstage) fetch(group);
  for (int j = group; j < nstage; j += G) {
    const int sum = j / kStagesPerSum, js = j % kStagesPerSum;
    if (js != 0 && drained < sum) {
      ok = drain_turn(bar, drained, nslots, acc0, acc1);
      if (!ok) break;
    }
    if (RAW > 0) {
      ok = fetch(j);
      if (!ok) break;
    }
    if (j >= NST) {
      ok = __all_sync(0xffffffffu, mbar_wait_fast(bar.empty + cur.b, cur.par ^ 1u));
      if (!ok) break;
    }
    fill(gsm + cur.b * stage_bytes);
    tc05::fence_smem_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar.full + cur.b);
    if (RAW == 0 && j + G < nstage) fetch(j + G);
    if (js == 0 && drained < sum) {
      ok = drain_turn(bar, drained, nslots, acc0, acc1);
      if (!ok) break;
    }
    // (64-bit sums of at most 2^20 rows)
    if (drained > 0 && (drained & 8191) == 0 && js < G) flush(acc0, acc1);
    ok = issue_turn(bar, cur, j, sum, js == 0, js >= kStagesPerSum - G, base + cur.b * stage_bytes,
                    [&] { ahead(j + RAW); }, issue);
    if (!ok) break;
    cur.advance(G);
  }
  while (ok && drained * kStagesPerSum < nstage) ok = drain_turn(bar, drained, nslots, acc0, acc1);
  if (ok) flush(acc0, acc1);
  else if (RAW > 0 && (threadIdx.x & 255) == 0) settle(copied);
  bar.close(ok, hdr);
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               :: "r"(tc05::smem_u32(dst)), "l"((uint64_t)__cvta_generic_to_global(src)), "r"(bytes),
                  "r"(tc05::smem_u32(mbar))
               : "memory");
}

// Products of `mine` output tiles of 128 rows x 32 G columns, K = `stages`
// stages of kStK elements each, as one sequence of stages: load(tile, js,
// slot) starts copies of this thread's part of the left factor into its slot
// of a ring of AHEAD (cp.async: the latency of memory spans several stages, and
// a thread that reads what it copied itself needs no barrier), fill(tile, js,
// slot, stage) writes its digits, the right factor's planes come by
// a bulk copy from bsrc(tile, js), store(tile, acc0, acc1) writes this
// thread's row and 16 columns.  `tile` counts 0 .. mine - 1.  LB: lowest
// level that is kept.
template <int S, int NST, int LB, int AHEAD, int G, class Load, class Fill, class Src, class Store>
__device__ __forceinline__ void product_pipeline(DigitBarriers<NST, G>& bar, unsigned char* gsm, int mine, int stages,
                                                 WsHeader* hdr, Load load, Fill fill, Src bsrc, Store store) {
  constexpr int kPlaneB = Shape<G>::PLANEB, kStage = S * (kPlaneA + kPlaneB);
  const int tid = threadIdx.x, lane = tid & 31, group = G == 1 ? 0 : tid >> 8;
  bar.open(1);
  const uint32_t base = tc05::smem_u32(gsm);
  const int sums = (stages + kStagesPerSum - 1) / kStagesPerSum;
  bool ok = true;
  int64_t acc0[16], acc1[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc0[c] = acc1[c] = 0;
  int drained = 0, dr_tile = 0, dr_sum = 0;
  // reads the sums before `upto`; the tile that the last of them completes is
  // written out by write_tile once the next MMAs are on their way
  bool whole = false;
  auto write_tile = [&] {
    if (!whole) return;
    store(dr_tile, acc0, acc1);
#pragma unroll
    for (int c = 0; c < 16; ++c) acc0[c] = acc1[c] = 0;
    ++dr_tile;
    whole = false;
  };
  auto read_upto = [&](int upto) {
    while (ok && drained < upto) {
      write_tile();
      ok = drain_turn(bar, drained, kSlots, acc0, acc1);
      if (ok && ++dr_sum == sums) {
        whole = true;
        dr_sum = 0;
      }
    }
  };
  auto issue = [&](uint32_t tmem, uint32_t sa, bool first) {
    issue_stage<S, LB, G>(tmem, tc05::desc(sa, 128, kPlaneSbo), tc05::desc(sa + S * kPlaneA, 128, kPlaneSbo), first);
  };
  StageSlot<NST> cur{group, 0u};
  int tile = 0, js = group, j = group;
  auto next = [&](int& t, int& q) {       // wraps the stage number
    if (G == 1) {
      if (q == stages) {
        q = 0;
        ++t;
      }
      return;
    }
    while (q >= stages) {
      q -= stages;
      ++t;
    }
  };
  next(tile, js);
  int ltile = tile, ljs = js, slot = 0;
  auto start = [&](int at) {
    if (ltile < mine) load(ltile, ljs, at);
    asm volatile("cp.async.commit_group;" ::: "memory");
    ljs += G;
    next(ltile, ljs);
  };
#pragma unroll
  for (int q = 0; q < AHEAD - 1; ++q) start(q);
  for (; tile < mine; j += G) {
    asm volatile("cp.async.wait_group %0;" :: "n"(AHEAD - 2) : "memory");
    const int sum = tile * sums + js / kStagesPerSum;
    const bool first = js % kStagesPerSum == 0;
    if (!first) read_upto(sum);
    if (ok && j >= NST) ok = __all_sync(0xffffffffu, mbar_wait_fast(bar.empty + cur.b, cur.par ^ 1u));
    if (!ok) break;
    unsigned char* st = gsm + cur.b * kStage;
    if ((tid & 255) == 0) {
      tc05::mbar_arrive_expect_tx(bar.full + cur.b, S * kPlaneB);
      bulk_load(st + S * kPlaneA, bsrc(tile, js), S * kPlaneB, bar.full + cur.b);
    }
    fill(tile, js, slot, st);
    tc05::fence_smem_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar.full + cur.b);
    start(slot == 0 ? AHEAD - 1 : slot - 1);
    slot = slot == AHEAD - 1 ? 0 : slot + 1;
    if (first) read_upto(sum);
    if (!ok) break;
    // stages of this sum from this one on
    const int in_sum = js % kStagesPerSum, rest = stages - js, left = rest < kStagesPerSum - in_sum ? rest : kStagesPerSum - in_sum;
    const int commits = left > G ? 0 : G == 2 && left == 1 && first ? 2 : 1;
    ok = issue_turn(bar, cur, j, sum, first, commits, base + cur.b * kStage, [] {}, issue);
    if (!ok) break;
    write_tile();
    js += G;
    next(tile, js);
    cur.advance(G);
  }
  read_upto(mine * sums);
  if (ok) write_tile();
  asm volatile("cp.async.wait_all;" ::: "memory");
  // bulk copies of stages that were never consumed (after a timeout) land
  // before the block ends
  if (!ok && tid == 0)
    for (int b = 0; b < NST; ++b) tc05::mbar_wait(bar.full + b, 0, 1000000ull);
  bar.close(ok, hdr);
}

// one integer sum into the global groups: the low 32 bits to group g, the
// carry to group g + 1 (so no group can overflow)
__device__ __forceinline__ void add_group(unsigned long long* G, int64_t MM, int64_t at, int g, int64_t v) {
  if (v == 0) return;
  atomicAdd(G + g * MM + at, (unsigned long long)(v & 0xffffffffll));
  atomicAdd(G + (g + 1) * MM + at, (unsigned long long)(v >> 32));
}

}  // namespace pylom
