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

// ---------------------------------------------------------------------------
// the two pipelines (512 threads, one block per SM)
// ---------------------------------------------------------------------------
constexpr int kDigThreads = 512;   // 128 registers a thread: 64 hold the integer sums

template <int NST>
struct DigitBarriers {
  uint64_t full[NST], empty[NST], dfull, dempty, fin;
  uint32_t tmem;
  // all threads; `extra`: arrivals on a full barrier besides one per warp
  __device__ __forceinline__ void open(int extra) {
    if (threadIdx.x == 0) {
      for (int b = 0; b < NST; ++b) {
        tc05::mbar_init(full + b, kDigThreads / 32 + extra);
        tc05::mbar_init(empty + b, 1);
      }
      tc05::mbar_init(&dfull, 1);
      tc05::mbar_init(&dempty, kDigThreads / 32);
      tc05::mbar_init(&fin, 1);
    }
    if (threadIdx.x < 32) tc05::tmem_alloc(&tmem, 512);
    tc05::fence_before();
    __syncthreads();
    tc05::fence_after();
  }
  // all threads: nothing of this block is in flight when it gives its memory back
  __device__ __forceinline__ void close(bool ok, WsHeader* hdr) {
    if (threadIdx.x == kDigThreads - 32) {
      tc05::commit(&fin);
      if (!mbar_wait_fast(&fin, 0)) ok = false;
    }
    if (!ok) raise_status(hdr, PYLOM_ERR_TIMEOUT);
    tc05::fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tc05::tmem_dealloc(tmem, 512);
  }
};

// Sums over a range of rows: `nstage` stages of kStK rows, read out every
// kStagesPerSum of them.  fill(j, stage) writes this thread's part of stage
// j; issue(stage address, first) issues its MMAs (one thread); flush(acc0,
// acc1) hands on the 64-bit sums of this thread's row and 16 columns.  The
// accumulators are read only after the next NST stages have been filled, so
// the warps work while the last MMAs of a sum run.
template <int NST, class Fill, class Issue, class Flush>
__device__ __forceinline__ void gram_pipeline(DigitBarriers<NST>& bar, unsigned char* gsm, int stage_bytes, int64_t nstage,
                                              int nslots, WsHeader* hdr, Fill fill, Issue issue, Flush flush) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bar.open(0);
  const uint32_t tmem = bar.tmem;
  const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 16;
  bool ok = true;
  int64_t acc0[16], acc1[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc0[c] = acc1[c] = 0;
  int64_t issued = 0, drained = 0;
  for (int64_t j = 0; j <= nstage; ++j) {
    const int b = (int)(j % NST);
    if (j < nstage) {
      if (j >= NST) {
        ok = __all_sync(0xffffffffu, mbar_wait_fast(bar.empty + b, (uint32_t)((j / NST - 1) & 1)));
        if (!ok) break;
      }
      fill(j, gsm + b * stage_bytes);
      tc05::fence_smem_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar.full + b);
    }
    // the sums of the 128 rows before, once the stages ahead are filled
    const bool due = (j % kStagesPerSum == NST - 1 && j >= kStagesPerSum && j < nstage) ||
                     (j == nstage && nstage > 0);
    if (due) {
      ok = __all_sync(0xffffffffu, mbar_wait_fast(&bar.dfull, (uint32_t)(drained & 1)));
      if (!ok) break;
      tc05::fence_after();
      drain_slots(taddr, nslots, acc0, acc1);
      tc05::fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar.dempty);
      ++drained;
      if ((drained & 8191) == 0) flush(acc0, acc1);
    }
    // MMAs of the stages that are filled; those of a new sum wait until the
    // last one has been read
    const bool held = j >= kStagesPerSum && j % kStagesPerSum < NST - 1;
    if (warp == kDigThreads / 32 - 1 && lane == 0 && j < nstage && !held) {
      for (; issued <= j && ok; ++issued) {
        const int ib = (int)(issued % NST);
        const int64_t sum = issued / kStagesPerSum;
        const bool first = issued % kStagesPerSum == 0;
        ok = mbar_wait_fast(bar.full + ib, (uint32_t)((issued / NST) & 1));
        if (ok && first && sum > 0) ok = mbar_wait_fast(&bar.dempty, (uint32_t)((sum - 1) & 1));
        if (!ok) break;
        tc05::fence_after();
        issue(tmem, tc05::smem_u32(gsm) + ib * stage_bytes, first);
        tc05::commit(bar.empty + ib);
        if (issued % kStagesPerSum == kStagesPerSum - 1) tc05::commit(&bar.dfull);
      }
    }
    ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
    if (!ok) break;
  }
  if (ok) flush(acc0, acc1);
  bar.close(ok, hdr);
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               :: "r"(tc05::smem_u32(dst)), "l"((uint64_t)__cvta_generic_to_global(src)), "r"(bytes),
                  "r"(tc05::smem_u32(mbar))
               : "memory");
}

// Products of `mine` output tiles of 128 rows x 64 columns, K = `stages`
// stages of kStK elements each, as one sequence of stages: fill(tile, js,
// stage) writes the left factor's digits, the right factor's planes come by
// a bulk copy from bsrc(tile, js), store(tile, acc0, acc1) writes this
// thread's row and 16 columns.  `tile` counts 0 .. mine - 1.  LB: lowest
// level that is kept.
template <int S, int NST, int LB, class Fill, class Src, class Store>
__device__ __forceinline__ void product_pipeline(DigitBarriers<NST>& bar, unsigned char* gsm, int64_t mine, int64_t stages,
                                                 WsHeader* hdr, Fill fill, Src bsrc, Store store) {
  constexpr int kStage = S * (kPlaneA + kPlaneB);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  bar.open(1);
  const uint32_t tmem = bar.tmem;
  const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * 16;
  const int64_t sums = (stages + kStagesPerSum - 1) / kStagesPerSum;
  const int64_t total = mine * stages, nsum = mine * sums;
  bool ok = true;
  int64_t acc0[16], acc1[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc0[c] = acc1[c] = 0;
  int64_t issued = 0, issued_sum = 0, drained = 0;
  int64_t tile = 0, js = 0, begun = 0;   // the stage being filled; sums whose first stage has been filled
  int ahead = 0;                         // stages filled of the current sum
  int64_t is_js = 0, dr_tile = 0, dr_sum = 0;
  for (int64_t j = 0; j <= total; ++j) {
    const int b = (int)(j % NST);
    if (j < total) {
      if (j >= NST) {
        ok = __all_sync(0xffffffffu, mbar_wait_fast(bar.empty + b, (uint32_t)((j / NST - 1) & 1)));
        if (!ok) break;
      }
      unsigned char* st = gsm + b * kStage;
      if (tid == 0) {
        tc05::mbar_arrive_expect_tx(bar.full + b, S * kPlaneB);
        bulk_load(st + S * kPlaneA, bsrc(tile, js), S * kPlaneB, bar.full + b);
      }
      fill(tile, js, st);
      tc05::fence_smem_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar.full + b);
      if (js % kStagesPerSum == 0) {
        ++begun;
        ahead = 0;
      }
      ++ahead;
      if (++js == stages) {
        js = 0;
        ++tile;
      }
    }
    // read the sums that are complete: all of them at the end; before that,
    // the one before the sum being filled, as soon as NST stages (or the
    // whole sum) are filled ahead of it
    const bool whole = j < total && (js == 0 || js % kStagesPerSum == 0);
    const int64_t upto = j == total ? nsum : (ahead >= NST || whole) ? begun - 1 : drained;
    while (drained < upto) {
      ok = __all_sync(0xffffffffu, mbar_wait_fast(&bar.dfull, (uint32_t)(drained & 1)));
      if (!ok) break;
      tc05::fence_after();
      drain_slots(taddr, kSlots, acc0, acc1);
      tc05::fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar.dempty);
      ++drained;
      if (++dr_sum == sums) {
        store(dr_tile, acc0, acc1);
#pragma unroll
        for (int c = 0; c < 16; ++c) acc0[c] = acc1[c] = 0;
        dr_sum = 0;
        ++dr_tile;
      }
    }
    if (!ok) break;
    // MMAs of filled stages, up to the first sum whose accumulators are still unread
    if (warp == kDigThreads / 32 - 1) {
      if (lane == 0) {
        while (issued <= j && issued < total) {
          const bool first = is_js % kStagesPerSum == 0;
          if (first && issued_sum > drained) break;      // this warp has not read the sum before
          const int ib = (int)(issued % NST);
          ok = mbar_wait_fast(bar.full + ib, (uint32_t)((issued / NST) & 1));
          if (ok && first && issued_sum > 0) ok = mbar_wait_fast(&bar.dempty, (uint32_t)((issued_sum - 1) & 1));
          if (!ok) break;
          if (first) ++issued_sum;
          tc05::fence_after();
          const uint32_t sa = tc05::smem_u32(gsm) + ib * kStage;
          issue_stage<S, LB>(tmem, tc05::desc(sa, 128, kPlaneSbo), tc05::desc(sa + S * kPlaneA, 128, kPlaneSbo),
                             kPlaneB, first);
          tc05::commit(bar.empty + ib);
          ++issued;
          if (++is_js == stages) is_js = 0;
          if (is_js % kStagesPerSum == 0) tc05::commit(&bar.dfull);
        }
      }
      ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
      if (!ok) break;
    }
  }
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
