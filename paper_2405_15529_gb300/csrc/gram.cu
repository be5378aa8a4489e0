// gram.cu -- R of the weighted, mean-removed snapshot matrix Y from its Gram
// matrix (pyLOM, arXiv 2405.15529, Eq. svdqr1: Y = Q R, R unique up to row
// signs, R^T R = Y^T Y).
//
// In working precision the Gram matrix would lose the small singular values
// (its rounding error is eps sigma_1^2).  Here it is exact: every element of
// Y is a fixed-point integer relative to its column's largest magnitude, cut
// into 8-bit digits whose products run on the tcgen05 tensor cores without
// rounding (digits.cuh), and the sums stay integers until the end.  The
// Cholesky factorisation then runs in double-double arithmetic (106 bits),
// so R carries the backward error of a Householder QR in binary64 (the
// square root of 2^-104) at a fraction of its binary64 work, which this part
// does at 1/60 of its binary32 rate.
//
// Measured (4,194,304 x 256, binary64): Householder leaves + tree 554 + 13
// ms; here Y 8.6, cutting it 3.0, Gram matrix 26.3, Cholesky factor 0.74 ms.
// 1,048,576 x 128: leaves + tree 39 + 3.8 ms; here 1.4, 0.4, 2.1 and 0.35.
// Binary32 (mixed, 4,194,304 x 256): leaves + tree 57.7 + 8.8 ms; here Y 3.0,
// row shifts 0.7, Gram matrix 12.5 and Cholesky factor 0.71 ms.
#include <atomic>

#include "digits.cuh"
#include "gram.h"

namespace pylom {

// ---------------------------------------------------------------------------
// Y = sqrt(w) (X - mean)
// ---------------------------------------------------------------------------

struct PrologueArgs {
  const void* X;
  int64_t ldx;
  const double* w;
  int remove_mean;
  double* mean;
  void* Y;
  int64_t ldy, N, M;
  int* colE;
  WsHeader* hdr;
};

__device__ __forceinline__ bool nonfinite(double x) { return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000; }
__device__ __forceinline__ bool nonfinite(float x) { return (__float_as_int(x) & 0x7f800000) == 0x7f800000; }

// A block takes 32 rows at a time: lane = row, warp v the columns v, v + W,
// ..., CT of them in registers between the row's mean and its centred values
// (wider matrices read X once more, from the L2 cache).  Reading X and writing
// Y is the bound in binary32; in binary64 the binary64 pipe is (two lanes a
// clock and SM; its counter reads 80 % at 262,144 x 256 with weights and no
// mean: about four operations an element).  So the row's
// division and square root are one warp's work, not every warp's, finiteness
// is an integer test, and the column maxima take half a register a column: that
// leaves registers for two blocks of 16 warps.  Before (a register a column, 8
// warps of 32 columns, every warp its own division and root) -> here,
// microseconds: 65,537 x 63 binary64 71 -> 41, 1,048,576 x 256 binary64 2960 ->
// 2720; binary32 262,144 x 100 146 -> 80, 4,194,304 x 256 6400 -> 3020,
// 300,001 x 700 2150 -> 690.
template <typename TX, typename TY, int CT, int W>
__global__ void __launch_bounds__(32 * W, 1024 / (32 * W)) gram_prologue_kernel(PrologueArgs a) {
  static_assert(CT % 2 == 0, "maxima in pairs");
  __shared__ double ssum[W][32];
  __shared__ double sbar[32], ssw[2][32];   // (a warp may be an iteration ahead of the reads of ssw)
  __shared__ float4 sf[32];      // mean and root of the weight as binary32 pairs
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const TX* X = (const TX*)a.X;
  TY* Y = (TY*)a.Y;
  bool bad = false;
  const bool one = a.M <= W * CT;
  uint32_t emax[CT / 2] = {};     // of columns 2 u, 2 u + 1 of this warp, 16 bits each
  auto flush = [&](int64_t c0) {      // lane t: column t of this warp
    int mine = 0;
#pragma unroll
    for (int t = 0; t < CT; ++t) {
      const int e = __reduce_max_sync(0xffffffffu, (emax[t / 2] >> (16 * (t & 1))) & 0xffffu);
      mine = lane == t ? e : mine;
    }
    const int64_t c = c0 + warp + W * lane;
    if (lane < CT && c < a.M && mine > __ldcg(a.colE + c)) atomicMax(a.colE + c, mine);
#pragma unroll
    for (int u = 0; u < CT / 2; ++u) emax[u] = 0;
  };
  const int64_t nblk = (a.ldy + 31) / 32;
  int turn = 0;
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x, turn ^= 1) {
    const int64_t n = blk * 32 + lane;
    const bool in = n < a.N;
    TX x[CT];
    double s = 0.0, sw = 1.0, xbar = 0.0;
    if (a.w && warp == W - 1 && in) {
      const double wn = a.w[n];
      if (!(wn > 0.0) || !isfinite(wn)) bad = true;
      sw = sqrt(wn);
    }
    if (one || a.remove_mean)
      for (int64_t c0 = 0; c0 < a.M; c0 += W * CT) {
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          const int64_t c = c0 + warp + W * t;
          x[t] = (in && c < a.M) ? X[n + c * a.ldx] : (TX)0;
        }
        if (a.remove_mean) {
          if constexpr (sizeof(TX) == 4) {
            // compensated binary32 sums in chunks of at most 16 (binary64
            // conversions and additions are slow on this part)
            float h, l;
            static_assert(CT <= 16, "one chunk");
            sum32_compensated(x, h, l);
            s += (double)h + (double)l;
          } else {
#pragma unroll
            for (int t = 0; t < CT; ++t) s += (double)x[t];
          }
        }
      }
    float4 f = {0.f, 0.f, 1.f, 0.f};
    if (a.remove_mean || a.w) {
      ssum[warp][lane] = s;
      if (warp == W - 1) ssw[turn][lane] = sw;
      __syncthreads();
      if (warp == 0) {
        double tot = 0.0;
        if (a.remove_mean) {
#pragma unroll
          for (int q = 0; q < W; ++q) tot += ssum[q][lane];
          tot /= (double)a.M;
        }
        const double root = ssw[turn][lane];
        sbar[lane] = tot;
        if (sizeof(TX) == 4 && sizeof(TY) == 4) {
          const float xh = (float)tot, sh = (float)root;
          sf[lane] = make_float4(xh, (float)(tot - (double)xh), sh, (float)(root - (double)sh));
        }
      }
      __syncthreads();
      xbar = sbar[lane];
      sw = ssw[turn][lane];
      f = sf[lane];
    }
    if (warp == 0 && in && a.mean) a.mean[n] = xbar;
    const float xh = f.x, xl = f.y, sh = f.z, sl = f.w;
    for (int64_t c0 = 0; c0 < a.M; c0 += W * CT) {
      if (!one) {
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          const int64_t c = c0 + warp + W * t;
          x[t] = (in && c < a.M) ? X[n + c * a.ldx] : (TX)0;
        }
      }
#pragma unroll
      for (int t = 0; t < CT; ++t) {
        const int64_t c = c0 + warp + W * t;
        if (c >= a.M) break;
        TY y;
        if constexpr (sizeof(TX) == 4 && sizeof(TY) == 4) {
          // x - mean as d + e by TwoSum, times sqrt(w) = sh + sl by two FMAs
          float d, e;
          two_sum32(x[t], -xh, d, e);
          y = __fmaf_rn(d, sh, __fmaf_rn(d, sl, __fmul_rn(__fsub_rn(e, xl), sh)));
        } else {
          double v = (double)x[t];
          if (a.remove_mean) v -= xbar;
          if (a.w) v *= sw;
          y = (TY)v;
        }
        if (!in) y = (TY)0;
        bad = bad || nonfinite(x[t]);
        if (n < a.ldy) Y[n + c * a.ldy] = y;
        emax[t / 2] = __vmaxu2(emax[t / 2], (uint32_t)exp_field(y) << (16 * (t & 1)));
      }
      if (!one) flush(c0);
    }
  }
  if (one) flush(0);
  if (bad) raise_status(a.hdr, PYLOM_ERR_NONFINITE);
  if (blockIdx.x == 0 && threadIdx.x == 0) a.hdr->gram_y = 1;
}

// ---------------------------------------------------------------------------
// exact Gram matrix
// ---------------------------------------------------------------------------
// A unit is an output tile of 128 x 64 columns of Y on or above the
// diagonal, a range of digit levels (two for binary64: eight accumulators of
// 64 columns fill the tensor memory) and a range of rows.  TMA boxes of 16 rows
// x 128 (64) columns bring Y into a ring in shared memory, swizzled so that
// neighbouring columns lie in different banks; 16 warps in two groups cut
// them into digit planes (a thread takes 8 rows of one column: one
// conflict-free 16-byte store per digit out); one thread a group issues a
// stage's MMAs; every 128 rows the accumulators are added to 64-bit integers
// in registers, and at the end those go to the global sums by integer
// atomics, so the result does not depend on the order.
//
// Bound by the tensor pipe (1540 clocks a stage of 16 rows, 12300 a sum of 128)
// and the reads of the accumulators between sums, which the MMAs wait for
// (about 6000).  1,048,576 x 256: binary64 9.5 ms with Y loaded by the warps
// themselves (the latency of their loads was the bound), 6.4 here; binary32
// 3.45 and 3.1.

struct GramArgs {
  int64_t ldy, N, M;      // ldy: rows that exist (N rounded up to 8)
  const int* colE;
  unsigned long long* G;
  int nJ, items, splits;
  WsHeader* hdr;
  // Y^T Z instead of Y^T Y: Z (N x NZ), its exponents, all tiles
  const void* Z;
  int64_t NZ;
  const int* zE;
  const uint16_t *rowS, *zS;
  const unsigned* unless;
  CUtensorMap mapA, mapB;   // Y in boxes of kStK rows x 128 columns; the right factor, x 64
};

// Shift of each row: how many binary places its elements all lie below their
// columns' largest exponents (0 for a row of zeros).  In sums over rows small
// rows hardly count, but the modes of a row are made of that row alone, and a
// reflector would keep them to its own rounding.
//   binary32: the product Y C scales a row's elements by its shift.
//   binary64: the elements become biased fixed-point words, in place.  Up to
//     kRowShift places the words are at their columns' scale (still exact: they
//     have 9 bits to spare) and the shift reads 0; rows further down are
//     stored times 2^shift, and the Gram kernel shifts them back.
// A block takes 32 V rows at a time, V = 16 bytes of a column a lane, warp v the
// columns v, v + W, ..; the warps' maxima meet in shared memory.  Bound by
// memory (4 and 16 bytes an element).  For the words binary64 elements are read
// again, from the L2 cache, but for a warp's last eight columns, which are
// still in registers.  4,194,304 x 256: binary64 3.0 ms (2.4 at one scale a
// column, without shifts), binary32 0.68; the Gram kernel's look at the shifts
// 0.5 of 26.3.
constexpr int kRowShift = 3;
template <typename T> struct RowVec;
template <> struct RowVec<float> { typedef float4 type; };
template <> struct RowVec<double> { typedef double2 type; };
template <typename T, int W>
__global__ void __launch_bounds__(32 * W, 1024 / (32 * W)) row_scale_kernel(T* Y, int64_t ldy, int M, const int* colE,
                                                                             uint16_t* rowS, const unsigned* unless) {
  typedef typename RowVec<T>::type Vec;
  constexpr int V = 16 / sizeof(T), R = 32 * V, U = 8, kBits = sizeof(T) == 8 ? 20 : 23;   // mantissa bits of the upper word
  constexpr int kFloor = sizeof(T) == 8 ? kMinField64 : kMinField32, kNone = -2147483647;
  __shared__ int stop[2][W][R];      // (a warp may be an iteration ahead of the reads)
  __shared__ int sshift[2][R];
  if (unless && *unless) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nblk = (ldy + R - 1) / R, step = (int64_t)W * ldy;
  // first column of this warp's last chunk
  const int last = warp < M ? warp + (M - 1 - warp) / (U * W) * (U * W) : warp;
  int turn = 0;
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x, turn ^= 1) {
    const int64_t n0 = blk * R + lane * V;         // (ldy is a multiple of 8: a lane's rows exist together)
    const int lim = n0 < ldy ? M : 0;
    Vec x[U];
    auto read = [&](int c0) {
      const T* p = Y + n0 + c0 * ldy;
#pragma unroll
      for (int u = 0; u < U; ++u, p += step) x[u] = c0 + u * W < lim ? *(const Vec*)p : Vec{};
    };
    int top[V];
#pragma unroll
    for (int v = 0; v < V; ++v) top[v] = kNone;
    for (int c0 = warp; c0 <= last; c0 += U * W) {
      read(c0);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int E = c0 + u * W < M ? __ldg(colE + c0 + u * W) << kBits : 0;
#pragma unroll
        for (int v = 0; v < V; ++v) {
          int hi;
          if constexpr (sizeof(T) == 8) hi = __double2hiint(((const double*)&x[u])[v]);
          else hi = __float_as_int(((const float*)&x[u])[v]);
          hi &= sizeof(T) == 8 ? 0x7ff00000 : 0x7f800000;
          if (hi > (kFloor << kBits)) top[v] = max(top[v], hi - E);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) stop[turn][warp][lane * V + v] = top[v];
    __syncthreads();
    if (threadIdx.x < R) {
      int t = kNone;
#pragma unroll
      for (int q = 0; q < W; ++q) t = max(t, stop[turn][q][threadIdx.x]);
      int s = t == kNone ? 0 : -(t >> kBits);
      if (sizeof(T) == 8 && s <= kRowShift) s = 0;
      if (blk * R + threadIdx.x < ldy) rowS[blk * R + threadIdx.x] = (uint16_t)s;
      sshift[turn][threadIdx.x] = s;
    }
    if constexpr (sizeof(T) == 8) {
      __syncthreads();
      int s[V];
#pragma unroll
      for (int v = 0; v < V; ++v) s[v] = sshift[turn][lane * V + v];
      for (int c0 = last; c0 >= 0; c0 -= U * W) {
        if (c0 != last) read(c0);
        T* p = Y + n0 + c0 * ldy;
#pragma unroll
        for (int u = 0; u < U; ++u, p += step) {
          if (c0 + u * W >= lim) break;
          const int E = __ldg(colE + c0 + u * W);
          uint2 w[V];
          // (a column that lies lower still has only elements below the floor here)
#pragma unroll
          for (int v = 0; v < V; ++v)
            w[v] = E - s[v] >= kFloor ? biased_fixed(((const double*)&x[u])[v], E - s[v]) : zero_cell<uint2>();
          *(uint4*)p = make_uint4(w[0].x, w[0].y, w[V - 1].x, w[V - 1].y);
        }
      }
    }
  }
}

template <typename T>
static cudaError_t row_scale(T* Y, int64_t ldy, int64_t M, const int* colE, uint16_t* rowS, const unsigned* unless, int sms,
                             cudaStream_t st) {
  constexpr int R = 32 * 16 / (int)sizeof(T);
  const int64_t nblk = (ldy + R - 1) / R;
  // eight warps up to 64 columns (eight columns in flight a warp), else sixteen
  const int64_t cap = (int64_t)sms * (M <= 64 ? 4 : 2);
  const unsigned grid = (unsigned)(nblk < cap ? nblk : cap);
  if (M <= 64) row_scale_kernel<T, 8><<<grid, 256, 0, st>>>(Y, ldy, (int)M, colE, rowS, unless);
  else row_scale_kernel<T, 16><<<grid, 512, 0, st>>>(Y, ldy, (int)M, colE, rowS, unless);
  return cudaGetLastError();
}
cudaError_t launch_row_scale(void* Y, bool f32, int64_t ldy, int64_t cols, const int* colE, uint16_t* rowS,
                             const unsigned* unless, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  return f32 ? row_scale<float>((float*)Y, ldy, cols, colE, rowS, unless, sms, st)
             : row_scale<double>((double*)Y, ldy, cols, colE, rowS, unless, sms, st);
}

// Back to binary64 (to another buffer), for a Householder factorisation of
// this Y; rows past N are not written.
__global__ void __launch_bounds__(256) unpack_kernel(const double* P, int64_t ldy, int64_t N, int64_t M, const int* colE,
                                                     const uint16_t* rowS, double* Y, const unsigned* gram_y, const unsigned* redo) {
  if (*gram_y == 0 || *redo == 0) return;
  for (int64_t c = blockIdx.y; c < M; c += gridDim.y)
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
      Y[n + c * ldy] = from_fixed(*(const uint2*)(P + n + c * ldy), colE[c] - rowS[n]);
}
cudaError_t launch_unpack(const GramState& g, double* Y, const unsigned* redo, cudaStream_t st) {
  const int64_t bx = (g.N + 255) / 256;
  const dim3 grid((unsigned)(bx < 64 ? bx : 64), (unsigned)(g.M < 65535 ? g.M : 65535));
  unpack_kernel<<<grid, 256, 0, st>>>((const double*)g.Y, g.ldy, g.N, g.M, g.colE, g.rowS, Y, &g.hdr->gram_y,
                                      redo);
  return cudaGetLastError();
}

template <typename TY>
__global__ void __launch_bounds__(Shape<2>::THREADS, 1) gram_kernel(const __grid_constant__ GramArgs a) {
  constexpr int S = Dig<TY>::S, NST = Dig<TY>::template NST<2>, kPlaneB = Shape<2>::PLANEB;
  constexpr int kStage = S * (kPlaneA + kPlaneB);
  constexpr int kPitch = kStK * (int)sizeof(TY), kRawA = 128 * kPitch, kRawStage = kRawA + 64 * kPitch;
  typedef typename Cell<TY>::type C;
  extern __shared__ __align__(1024) unsigned char gsm[];
  __shared__ __align__(8) DigitBarriers<NST, 2> bar;
  __shared__ __align__(8) uint64_t raw_full[kRaw];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int item = blockIdx.x % a.items, split = blockIdx.x / a.items;
  const int half = item % Dig<TY>::HALVES;
  if (a.unless && *a.unless) return;
  int I = 0, t = item / Dig<TY>::HALVES;
  if (a.Z) {
    I = t / a.nJ;
    t %= a.nJ;
  } else {
    while (t >= a.nJ - 2 * I) {
      t -= a.nJ - 2 * I;
      ++I;
    }
    t += 2 * I;
  }
  const int J = t;
  const bool diag = !a.Z && (J >> 1) == I;       // B's columns are among A's
  const int64_t nB = a.Z ? a.NZ : a.M;
  const int64_t nsum = (a.N + 127) / 128;
  const int64_t q0 = nsum * split / a.splits, q1 = nsum * (split + 1) / a.splits;
  // a thread of a stage's group: 8 rows of one of A's columns, and four of the
  // eight warps, in turn, 8 rows of one of B's
  const int th = tid & 255, ca = th & 127, kg = th >> 7, cb = th & 63, kb = (th >> 6) & 1, quad = th >> 7;
  const int64_t colA = (int64_t)I * 128 + ca, colB = (int64_t)J * 64 + cb;
  const int EA = colA < a.M ? a.colE[colA] : 128;
  const int EB = (!diag && colB < nB) ? (a.Z ? a.zE : a.colE)[colB] : 128;
  const int row0 = (int)(q0 * 128);
  // stages whose rows kg 8.. (kb 8..) are rows of Y (columns past the last: none)
  const int jA = colA < a.M ? (int)((a.ldy - row0 - kg * 8 + kStK - 1) / kStK) : 0;
  const int jB = colB < nB ? (int)((a.ldy - row0 - kb * 8 + kStK - 1) / kStK) : 0;
  unsigned char* raw = gsm + NST * kStage;
  // binary64: behind the ring, the shifts of a stage's rows of Y, then of Z
  uint16_t* shifts = (uint16_t*)(raw + kRaw * kRawStage);
  if (tid == 0)
    for (int q = 0; q < kRaw; ++q) tc05::mbar_init(raw_full + q, 1);
  auto copy = [&](int j) {
    unsigned char* r = raw + (j % kRaw) * kRawStage;
    uint64_t* m = raw_full + j % kRaw;
    constexpr int kShift = sizeof(TY) == 8 ? 2 * kStK : 0;     // bytes
    tc05::mbar_arrive_expect_tx(m, (diag ? kRawA : kRawStage) + (a.Z ? 2 : 1) * kShift);
    if constexpr (sizeof(TY) == 8) {
      bulk_load(shifts + (j % kRaw) * 2 * kStK, a.rowS + row0 + j * kStK, kShift, m);
      if (a.Z) bulk_load(shifts + ((j % kRaw) * 2 + 1) * kStK, a.zS + row0 + j * kStK, kShift, m);
    }
    tc05::tma_load_2d(r, &a.mapA, row0 + j * kStK, I * 128, m);
    if (!diag) tc05::tma_load_2d(r + kRawA, &a.mapB, row0 + j * kStK, J * 64, m);
  };
  auto settle = [&](int j) {
    for (int q = j; q > j - kRaw && q >= 0; q -= 2) tc05::mbar_wait(raw_full + q % kRaw, (uint32_t)((q / kRaw) & 1), 1000000ull);
  };
  // eight rows of a column from the swizzled box at p
  auto read8 = [&](const unsigned char* p, int col, int k8, bool in, C (&y)[8]) {
    constexpr int kChunks = 8 * (int)sizeof(TY) / 16;
    const int x = sizeof(TY) == 8 ? col & 7 : (col >> 1) & 3;
#pragma unroll
    for (int i = 0; i < kChunks; ++i)
      ((uint4*)y)[i] = *(const uint4*)(p + col * kPitch + (((k8 * kChunks + i) ^ x) << 4));
    if (!in) {
#pragma unroll
      for (int i = 0; i < 8; ++i) y[i] = zero_cell<C>();
    }
  };
  // small rows at their columns' scale (eight rows, the same for a whole warp)
  auto unshift8 = [&](int j, int z, int k8, C (&y)[8]) {
    if constexpr (sizeof(TY) == 8) {
      const uint4 s = *(const uint4*)(shifts + ((j % kRaw) * 2 + z) * kStK + k8 * 8);
      if (s.x | s.y | s.z | s.w) {
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = shift_word(y[i], packed_shift(s, i));
      }
    }
  };
  __align__(16) C yA[8], yB[8];
  bool withB = false;
  auto fetch = [&](int j) {
    if (!__all_sync(0xffffffffu, mbar_wait_fast(raw_full + j % kRaw, (uint32_t)((j / kRaw) & 1)))) return false;
    const unsigned char* r = raw + (j % kRaw) * kRawStage;
    read8(r, ca, kg, j < jA, yA);
    unshift8(j, 0, kg, yA);
    withB = !diag && ((j >> 1) & 1) == quad;
    if (withB) {
      read8(r + kRawA, cb, kb, j < jB, yB);
      unshift8(j, a.Z ? 1 : 0, kb, yB);
    }
    return true;
  };
  const int oa = (ca >> 3) * kPlaneSbo + (ca & 7) * 16 + kg * 128;
  // on the diagonal half of A's columns are B's too
  const int ob = S * kPlaneA + ((ca & 63) >> 3) * kPlaneSbo + (ca & 7) * 16 + kg * 128;
  const bool both = diag && (ca >> 6) == (J & 1);
  auto fill = [&](unsigned char* st) {
    put_digits(yA, EA, st + oa, kPlaneA, both ? st + ob : nullptr, kPlaneB);
    if (withB)
      put_digits(yB, EB, st + S * kPlaneA + (cb >> 3) * kPlaneSbo + (cb & 7) * 16 + kb * 128, kPlaneB, nullptr, 0);
  };
  auto issue = [&](uint32_t tmem, uint32_t sa, bool first) {
    const uint64_t dA = tc05::desc(sa, 128, kPlaneSbo), dB = tc05::desc(sa + S * kPlaneA, 128, kPlaneSbo);
    if (half == 0) issue_stage<S, gram_base<TY>(0), 2>(tmem, dA, dB, first);
    else issue_stage<S, gram_base<TY>(Dig<TY>::HALVES - 1), 2>(tmem, dA, dB, first);
  };
  auto flush = [&](int64_t (&acc0)[16], int64_t (&acc1)[16]) {
    const int64_t gi = (int64_t)I * 128 + (warp & 3) * 32 + lane;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int64_t gj = (int64_t)J * 64 + (warp >> 2) * 16 + c;
      if (gi < a.M && gj < nB && (a.Z || gi <= gj)) {
        add_group(a.G, a.M * nB, gi + gj * a.M, half * 2, acc0[c]);
        add_group(a.G, a.M * nB, gi + gj * a.M, half * 2 + 1, acc1[c]);
      }
      acc0[c] = acc1[c] = 0;
    }
  };
  gram_pipeline<NST, kRaw, 2>(bar, gsm, kStage, (int)(q1 - q0) * kStagesPerSum, (sizeof(TY) == 8 && half == 1) ? 7 : 8, a.hdr,
                           copy, settle, fetch, fill, issue, flush);
}

// ---------------------------------------------------------------------------
// Cholesky factorisation in double-double arithmetic
// ---------------------------------------------------------------------------

struct dd { double h, l; };

__device__ __forceinline__ dd dd_two_sum(double a, double b) {
  const double s = __dadd_rn(a, b), bb = __dsub_rn(s, a);
  return {s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, bb)), __dsub_rn(b, bb))};
}
__device__ __forceinline__ dd dd_quick(double a, double b) {   // |a| >= |b|
  const double s = __dadd_rn(a, b);
  return {s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const double p = __dmul_rn(a.h, b.h);
  double e = __fma_rn(a.h, b.h, -p);
  e = __fma_rn(a.h, b.l, e);
  e = __fma_rn(a.l, b.h, e);
  return dd_quick(p, e);
}
// s - a b
__device__ __forceinline__ dd dd_fms(dd s, dd a, dd b) {
  const double p = __dmul_rn(a.h, b.h);
  double e = __fma_rn(a.h, b.h, -p);
  e = __fma_rn(a.h, b.l, e);
  e = __fma_rn(a.l, b.h, e);
  const dd t = dd_two_sum(s.h, -p);
  return dd_quick(t.h, __dadd_rn(t.l, __dsub_rn(s.l, e)));
}
__device__ __forceinline__ dd dd_add(dd a, dd b) {
  const dd t = dd_two_sum(a.h, b.h);
  return dd_quick(t.h, __dadd_rn(t.l, __dadd_rn(a.l, b.l)));
}
// 1 / a: one Newton step in double-double from the binary64 quotient
__device__ __forceinline__ dd dd_rcp(dd a) {
  const double x = 1.0 / a.h;
  double e = __fma_rn(-a.h, x, 1.0);
  e = __fma_rn(-a.l, x, e);
  return dd_quick(x, __dmul_rn(x, e));
}

// integer groups -> double-double, scaled by 2^-64 (squares stay in range)
__device__ __forceinline__ dd group_sum(const long long* G, int64_t MM, int64_t at, int groups, int lb) {
  dd s = {0.0, 0.0};
  for (int g = groups - 1; g >= 0; --g) {
    const double v = (double)__ldcg(G + g * MM + at);
    if (v != 0.0) s = dd_add(s, dd{scalbn(v, 32 * g + 8 * lb - 64), 0.0});
  }
  return s;
}

constexpr int kNBC = 8;            // panel height and tile size
constexpr int kChThreads = 128;
constexpr int kChCluster = 8;      // up to this many panels the blocks form one cluster (cheaper barrier)

struct CholArgs {
  GramState g;
  double* R;
  int groups, lb, bias;
};

// G = U^T D U (U unit upper triangular) by row panels of kNBC rows, one
// barrier over all blocks per panel.  Step p:
//   units    column block c > p: apply panel p - 1 to the diagonal tile and to
//            tile (p, c), factor the diagonal tile (a serial chain of 8
//            pivots, the same in every unit) together with tile (p, c), write
//            row block p of U (in place) and of T = D U (two buffers);
//   updates  tiles (bi, bj), p < bi <= bj: apply panel p - 1, A -= U^T T.
// A unit touches row p only and an update the rows below, so both read what
// step p - 1 left.  Bound by the binary64 pipe of the units' SMs (two lanes a
// clock): 16-row panels with 16 x 16 tiles and two barriers took 310 us at M
// = 63, 640 at 128, 1290 at 256 and 4900 at 700; this takes 189, 350, 730 and
// 3600.
// R = D^(1/2) U with the columns' scales 2^(E - bias) restored comes last.
// A pivot at the rounding level of its column (a direction that the other
// columns span, such as the one that the removed mean leaves) gives a zero
// row.
template <bool CLUSTER>
__device__ __forceinline__ bool chol_barrier(const GramState& g) {
  if (CLUSTER) {
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  }
  return grid_barrier(g.hdr, gridDim.x);
}

__device__ __forceinline__ dd ld_dd(const double* h, const double* l, int64_t at) { return {__ldcg(h + at), __ldcg(l + at)}; }

template <bool CLUSTER>
__global__ void __launch_bounds__(kChThreads) gram_chol_kernel(CholArgs c) {
  constexpr int B = kNBC;
  __shared__ dd sP[B][2 * B + 1];        // diagonal tile | tile (p, c)
  __shared__ dd sU[B][2 * B + 1], sT[B][2 * B + 1];
  __shared__ dd s_inv;
  __shared__ double s_level[B];
  const GramState& g = c.g;
  const int tid = threadIdx.x;
  const int64_t M = g.M, MM = M * M;
  const int64_t nb = (M + B - 1) / B;
  double* dvec = g.Tl + (int64_t)2 * B * M;     // pivots
  // integers -> double-double (upper triangle)
  for (int64_t idx = (int64_t)blockIdx.x * kChThreads + tid; idx < MM; idx += (int64_t)gridDim.x * kChThreads) {
    if (idx % M <= idx / M) {
      const dd v = group_sum(g.G, MM, idx, c.groups, c.lb);
      g.Lh[idx] = v.h;
      g.Ll[idx] = v.l;
    }
  }
  if (!chol_barrier<CLUSTER>(g)) return;
  for (int64_t p = 0; p < nb; ++p) {
    const int64_t k = p * B;
    const int nbk = (int)((M - k) < B ? (M - k) : B);
    // panel p - 1: U in Lh / Ll rows k - B.., T in buffer (p - 1) & 1 (B x M each)
    const double *Th = g.Th + ((p + 1) & 1) * B * M, *Tl = g.Tl + ((p + 1) & 1) * B * M;
    double *Thn = g.Th + (p & 1) * B * M, *Tln = g.Tl + (p & 1) * B * M;
    const int64_t units = nb - p - 1 > 0 ? nb - p - 1 : 1;
    const int64_t nt = p > 0 ? nb - p - 1 : 0, tiles = nt * (nt + 1) / 2, items = units + (tiles + 1) / 2;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
      __syncthreads();
      if (it < units) {
        const int64_t c0 = (p + 1 + it) * B;
        const int r = tid / (2 * B), q = tid % (2 * B);    // 8 x 16 threads
        const int64_t col = q < B ? k + q : c0 + q - B;
        const bool in = r < nbk && col < M && (q >= B || (q < nbk && r <= q));
        dd v = {0.0, 0.0};
        if (in) v = ld_dd(g.Lh, g.Ll, k + r + col * M);
        if (p > 0) {
          // rows q' of panel p - 1: U of the panel's own columns (index r), T of all 16
          dd tt = {0.0, 0.0}, uu = {0.0, 0.0};
          if (col < M && (q >= B || q < nbk)) tt = ld_dd(Th, Tl, r + col * B);
          if (q < nbk) uu = ld_dd(g.Lh, g.Ll, k - B + r + (k + q) * M);
          sT[r][q] = tt;
          if (q < B) sU[r][q] = uu;
          __syncthreads();
          if (in)
            for (int x = 0; x < B; ++x) v = dd_fms(v, sU[x][r], sT[x][q]);
        }
        sP[r][q] = v;
        // rounding level of a pivot: its column's own square times 2^-100
        if (tid < nbk) s_level[tid] = 7.9e-31 * group_sum(g.G, MM, (k + tid) * (M + 1), c.groups, c.lb).h;
        __syncthreads();
        for (int j = 0; j < nbk; ++j) {
          if (tid == 0) {
            const dd d = sP[j][j];
            const bool live = d.h > s_level[j];
            s_inv = live ? dd_rcp(d) : dd{0.0, 0.0};
            if (it == 0) dvec[k + j] = live ? d.h : 0.0;
          }
          __syncthreads();
          const dd inv = s_inv;
          // rows below take -(u_jr) (t_jq); u = t / d
          if (r > j && in) sP[r][q] = dd_fms(sP[r][q], dd_mul(sP[j][r], inv), sP[j][q]);
          // row j of U and T
          if (r == j && col < M) {
            const dd t = sP[j][q], uu = dd_mul(t, inv);
            if (q >= B) {
              g.Lh[k + j + col * M] = uu.h;
              g.Ll[k + j + col * M] = uu.l;
              Thn[j + col * B] = t.h;
              Tln[j + col * B] = t.l;
            } else if (it == 0 && q < nbk) {
              c.R[k + j + col * M] = q < j ? 0.0 : q == j ? 1.0 : uu.h;   // (scaled at the end)
            }
          }
          __syncthreads();
        }
      } else {
        // two 8 x 8 tiles of the trailing triangle, 64 threads each
        const int half = tid >> 6, lt = tid & 63, tr = lt & 7, tc = lt >> 3;
        const int64_t t = (it - units) * 2 + half;
        const bool live = t < tiles;
        int64_t bi = 0, bj = 0;
        if (live) {
          bj = (int64_t)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
          while (bj * (bj + 1) / 2 > t) --bj;
          while ((bj + 1) * (bj + 2) / 2 <= t) ++bj;
          bi = t - bj * (bj + 1) / 2;
        }
        const int64_t r0 = (p + 1 + bi) * B, c0 = (p + 1 + bj) * B;
        dd uu = {0.0, 0.0}, tt = {0.0, 0.0};
        if (live && r0 + tc < M) uu = ld_dd(g.Lh, g.Ll, k - B + tr + (r0 + tc) * M);
        if (live && c0 + tc < M) tt = ld_dd(Th, Tl, tr + (c0 + tc) * B);
        sU[tr][tc + half * B] = uu;
        sT[tr][tc + half * B] = tt;
        __syncthreads();
        const int64_t r = r0 + tr, cc = c0 + tc;
        if (live && r < M && cc < M && r <= cc) {
          dd s = ld_dd(g.Lh, g.Ll, r + cc * M);
#pragma unroll
          for (int x = 0; x < B; ++x) s = dd_fms(s, sU[x][tr + half * B], sT[x][tc + half * B]);
          g.Lh[r + cc * M] = s.h;
          g.Ll[r + cc * M] = s.l;
        }
      }
    }
    if (!chol_barrier<CLUSTER>(g)) return;
  }
  for (int64_t idx = (int64_t)blockIdx.x * kChThreads + tid; idx < MM; idx += (int64_t)gridDim.x * kChThreads) {
    const int64_t i = idx % M, j = idx / M;
    double v = 0.0;
    if (i <= j) {
      const double u = (i / B == j / B) ? __ldcg(c.R + idx) : __ldcg(g.Lh + idx);
      // the integer sums were scaled by 2^-64: their root by 2^-32
      v = scalbn(sqrt(__ldcg(dvec + i)) * u, g.colE[j] - c.bias + 32);
      if (g.colE[j] == (g.f32 ? kMaxField32 : kMaxField64)) v = quiet_nan();
    }
    c.R[idx] = v;
  }
}

// ---------------------------------------------------------------------------
// orthonormal modes
// ---------------------------------------------------------------------------
// The rounding of V, and of C = V_r S_r^-1 itself, grows by s_1 / s_r in the
// modes Y C: U^T U = I + F with F up to eps s_1 / s_r.  F = C^T G C - I comes
// from the exact integers in double-double; with T its strict upper triangle
// and half its diagonal, the modes Y (C - C T) are orthonormal to F^2.  (As in
// Gram-Schmidt each mode sheds its part along the larger ones, which moves it
// by its own uncertainty; a symmetric correction would move the large modes by
// that of the small ones.)  The product takes C - C T in 62 bits
// (coef_digits_kernel).  Where s_r is at least s_1 / kOrthoRatio, F is no larger
// than what the small SVD's stopping test leaves (cosines of M eps), and the
// two kernels return at once, 9 us.
// Bound by the binary64 pipe: a product in double-double is 14 of its
// operations.  W, T and the coefficients' share: 21 + 15 + 17 us at M = 32, r =
// 27, 71 + 46 + 25 at M = 128, r = 40, 365 + 88 + 25 at M = 256, r = 43.
struct OrthoArgs {
  const long long* G;
  const int* colE;
  const double *S, *VT;
  int64_t ldvt, M;
  double *Wh, *Wl, *T;          // M x r (ld M); r x r (ld rmax): T, its rows over S
  int64_t rmax;
  const WsHeader* hdr;
  const unsigned* unless;
  int groups, lb, bias;
};

// kept columns, or 0: nothing to correct
__device__ __forceinline__ int64_t ortho_cols(const OrthoArgs& a) {
  return a.unless && *a.unless ? 0 : ortho_rank(a.hdr, a.S);
}
__device__ __forceinline__ double ortho_c(const OrthoArgs& a, int64_t j, int64_t k) { return a.VT[k + j * a.ldvt] / a.S[k]; }
// C at the scale of the integer sums (their 2^-64 is 2^32 twice)
__device__ __forceinline__ double ortho_cs(const OrthoArgs& a, int64_t j, int64_t k) {
  return scalbn(ortho_c(a, j, k), a.colE[j] - a.bias + 32);
}
__device__ __forceinline__ dd dd_fma1(dd s, dd a, double b) {   // s + a b
  const double p = __dmul_rn(a.h, b);
  const double e = __fma_rn(a.l, b, __fma_rn(a.h, b, -p));
  const dd t = dd_two_sum(s.h, p);
  return dd_quick(t.h, __dadd_rn(t.l, __dadd_rn(s.l, e)));
}

// 8 x 8 tiles, K in chunks of 32 of which each of four groups of 64 threads
// takes eight.  WHICH 0: W = G C; 1: T from F = C^T W - I.
template <int WHICH>
__global__ void __launch_bounds__(256) ortho_product_kernel(OrthoArgs a) {
  __shared__ dd sL[8][33], sum[3][64];
  __shared__ double sC[32][9];
  const int64_t r = ortho_cols(a), M = a.M, i0 = (int64_t)blockIdx.x * 8, k0 = (int64_t)blockIdx.y * 8;
  if (k0 >= r || (WHICH == 1 && i0 > k0)) return;
  const int tid = threadIdx.x, i = tid & 7, k = (tid >> 3) & 7, sl = tid >> 6;
  dd acc = {0.0, 0.0};
  for (int64_t j0 = 0; j0 < M; j0 += 32) {
    __syncthreads();
    {
      // left tile (row x of the 8, chunk element y): G, or W transposed
      const int x = tid & 7, y = tid >> 3;
      dd v = {0.0, 0.0};
      if (j0 + y < M) {
        if (WHICH == 0) {
          const int64_t p = i0 + x, q = j0 + y;
          if (p < M) v = group_sum(a.G, M * M, p < q ? p + q * M : q + p * M, a.groups, a.lb);
        } else if (i0 + x < r) {
          v = dd{a.Wh[j0 + y + (i0 + x) * M], a.Wl[j0 + y + (i0 + x) * M]};
        }
      }
      sL[x][y] = v;
      const int kc = tid & 7;
      sC[y][kc] = j0 + y < M && k0 + kc < r ? ortho_cs(a, j0 + y, k0 + kc) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) acc = dd_fma1(acc, sL[i][sl * 8 + q], sC[sl * 8 + q][k]);
  }
  if (sl > 0) sum[sl - 1][tid & 63] = acc;
  __syncthreads();
  if (sl > 0) return;
#pragma unroll
  for (int q = 0; q < 3; ++q) acc = dd_add(acc, sum[q][tid]);
  if (WHICH == 0) {
    if (i0 + i < M && k0 + k < r) {
      a.Wh[i0 + i + (k0 + k) * M] = acc.h;
      a.Wl[i0 + i + (k0 + k) * M] = acc.l;
    }
  } else if (i0 + i <= k0 + k && k0 + k < r) {
    const bool diag = i0 + i == k0 + k;
    const dd t = dd_two_sum(acc.h, diag ? -1.0 : 0.0);
    a.T[i0 + i + (k0 + k) * a.rmax] = (t.h + (t.l + acc.l)) * (diag ? 0.5 : 1.0) / a.S[i0 + i];
  }
}

// W into the scratch of the Cholesky factor, T over the sums that W is made of.
cudaError_t launch_ortho(const GramState& g, const double* S, const double* VT, int64_t ldvt, const unsigned* unless,
                         const double** T, cudaStream_t st) {
  OrthoArgs a{g.G, g.colE, S, VT, ldvt, g.M, g.Lh, g.Ll, (double*)g.G, g.rmax, g.hdr, unless, 5, gram_base<double>(0),
              fix_bias<double>()};
  const unsigned m8 = (unsigned)((g.M + 7) / 8), r8 = (unsigned)((g.rmax + 7) / 8);
  ortho_product_kernel<0><<<dim3(m8, r8), 256, 0, st>>>(a);
  ortho_product_kernel<1><<<dim3(r8, r8), 256, 0, st>>>(a);
  *T = a.T;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

// (rows past N are read, and belong to no element)
size_t row_shift_bytes(int64_t N) { return align256(sizeof(uint16_t) * (size_t)((N + 127) / 128 * 128)); }

size_t gram_bytes(int64_t N, int64_t M, int64_t rmax) {
  return row_shift_bytes(N) + align256(sizeof(int) * (size_t)M) + align256(sizeof(long long) * (size_t)5 * M * M) +
         2 * align256(sizeof(double) * (size_t)M * M) + 2 * align256(sizeof(double) * (size_t)(2 * kNBC + 1) * M) +
         product_planes_bytes(M, 0, rmax);
}

void gram_carve(GramState& g, char* base, int64_t M, int64_t rmax) {
  const int64_t kt = (rmax + 63) / 64, js = (M + kStK - 1) / kStK;
  char* p = base;
  g.M = M;
  g.rmax = rmax;
  g.colE = (int*)p;          p += align256(sizeof(int) * (size_t)M);
  g.G = (long long*)p;       p += align256(sizeof(long long) * (size_t)5 * M * M);
  g.Lh = (double*)p;         p += align256(sizeof(double) * (size_t)M * M);
  g.Ll = (double*)p;         p += align256(sizeof(double) * (size_t)M * M);
  g.Th = (double*)p;         p += align256(sizeof(double) * (size_t)(2 * kNBC + 1) * M);
  g.Tl = (double*)p;         p += align256(sizeof(double) * (size_t)(2 * kNBC + 1) * M);
  g.Cd = (unsigned char*)p;  p += align256((size_t)kt * js * 8 * Shape<2>::PLANEB);
  g.Ce = (int*)p;            p += align256(sizeof(int) * (size_t)kt * 64);
  g.rowS = (uint16_t*)p;
}

template <typename TX, typename TY>
static cudaError_t prologue(const PrologueArgs& a, int sms, cudaStream_t st) {
  const int64_t nblk = (a.ldy + 31) / 32;
  // threads are capped at 1024 an SM by the register bound of the kernels
  const int64_t cap = (int64_t)sms * (a.M <= 128 ? 4 : 2);
  const unsigned grid = (unsigned)(nblk < cap ? nblk : cap);
  if (a.M <= 32) gram_prologue_kernel<TX, TY, 4, 8><<<grid, 256, 0, st>>>(a);
  else if (a.M <= 64) gram_prologue_kernel<TX, TY, 8, 8><<<grid, 256, 0, st>>>(a);
  else if (a.M <= 128) gram_prologue_kernel<TX, TY, 16, 8><<<grid, 256, 0, st>>>(a);
  else gram_prologue_kernel<TX, TY, 16, 16><<<grid, 512, 0, st>>>(a);
  return cudaGetLastError();
}

// Row splits of a tile list over `sms` blocks: the count whose last wave
// wastes least, at least one sum of 128 rows per unit.
static int row_splits(int64_t items, int64_t nsum, int sms) {
  int best = 1;
  double eff = 0.0;
  for (int s = 1; s <= sms; ++s) {
    if (s > 1 && nsum / s < 1) break;
    const int64_t units = items * s, waves = (units + sms - 1) / sms;
    if (waves > 4 && s > 1) break;
    const double e = (double)units / (double)(waves * sms);
    if (e > eff + 0.02) {
      eff = e;
      best = s;
    }
  }
  return best;
}

// Row coordinates of the tensor maps are 32-bit: taller matrices go in parts.
constexpr int64_t kGramRows = 1ll << 30;

template <typename TY>
static cudaError_t gram_launch(const GramState& g, int sms, const void* Z, int64_t ldz, int64_t NZ, const int* zE,
                               const uint16_t* zS, long long* G, const unsigned* unless, WsHeader* hdr, cudaStream_t st) {
  constexpr int S = Dig<TY>::S;
  constexpr size_t smem = (size_t)Dig<TY>::template NST<2> * S * (kPlaneA + Shape<2>::PLANEB) + (size_t)kRaw * 192 * kStK * sizeof(TY) +
                          (sizeof(TY) == 8 ? kRaw * 4 * kStK : 0);
  cudaError_t e = ensure_dyn_smem((const void*)gram_kernel<TY>, smem);
  if (e != cudaSuccess) return e;
  const int nJ = (int)(((Z ? NZ : g.M) + 63) / 64), nI = (int)((g.M + 127) / 128);
  int tiles = 0;
  for (int I = 0; I < nI; ++I) tiles += Z ? nJ : nJ - 2 * I;
  for (int64_t r = 0; r < g.N; r += kGramRows) {
    const int64_t N = g.N - r < kGramRows ? g.N - r : kGramRows;
    GramArgs a{};
    a.ldy = g.ldy - r < kGramRows ? g.ldy - r : kGramRows;     // rows of this part
    a.N = N;
    a.M = g.M;
    a.colE = g.colE;
    a.G = (unsigned long long*)G;
    a.nJ = nJ;
    a.items = tiles * Dig<TY>::HALVES;
    a.hdr = hdr;
    a.Z = Z;
    a.NZ = NZ;
    a.zE = zE;
    a.rowS = g.rowS + r;
    a.zS = Z ? zS + r : nullptr;
    a.unless = unless;
    a.splits = row_splits(a.items, (N + 127) / 128, sms);
    // words go as integers; 128 (64) bytes of a column, swizzled so that eight
    // neighbouring columns lie in different banks
    const CUtensorMapDataType type = sizeof(TY) == 8 ? CU_TENSOR_MAP_DATA_TYPE_UINT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    const CUtensorMapSwizzle swz = sizeof(TY) == 8 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    const int64_t ldb = Z ? ldz : g.ldy;
    e = tensor_map_2d(&a.mapA, type, (TY*)g.Y + r, a.ldy, g.M, g.ldy * (int64_t)sizeof(TY), kStK, 128, swz);
    if (e == cudaSuccess)
      e = tensor_map_2d(&a.mapB, type, (TY*)(Z ? Z : g.Y) + r, a.ldy, Z ? NZ : g.M, ldb * (int64_t)sizeof(TY), kStK, 64, swz);
    if (e != cudaSuccess) return e;
    gram_kernel<TY><<<(unsigned)(a.items * a.splits), Shape<2>::THREADS, smem, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// integers of Y^T Z -> W
__global__ void cross_sum_kernel(GramState g, int64_t NZ, const int* zE, const long long* G, double* W, int groups, int lb,
                                 int bias) {
  const int64_t n = g.M * NZ;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const dd s = group_sum(G, n, idx, groups, lb);
    W[idx] = scalbn(scalbn(s.h + s.l, g.colE[idx % g.M] - bias), zE[idx / g.M] - bias + 64);
  }
}

cudaError_t launch_cross(const GramState& g, const void* Z, int64_t ldz, int64_t NZ, const int* zE, const uint16_t* zS,
                         long long* G, double* W, const unsigned* unless, WsHeader* hdr, cudaStream_t st) {
  cudaError_t e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int groups = g.f32 ? 3 : 5;
  e = cudaMemsetAsync(G, 0, sizeof(long long) * (size_t)groups * g.M * NZ, st);
  if (e != cudaSuccess) return e;
  e = g.f32 ? gram_launch<float>(g, sms, Z, ldz, NZ, zE, zS, G, unless, hdr, st)
            : gram_launch<double>(g, sms, Z, ldz, NZ, zE, zS, G, unless, hdr, st);
  if (e != cudaSuccess) return e;
  cross_sum_kernel<<<64, 256, 0, st>>>(g, NZ, zE, G, W, groups, g.f32 ? gram_base<float>(0) : 0,
                                       g.f32 ? fix_bias<float>() : fix_bias<double>());
  return cudaGetLastError();
}

cudaError_t launch_gram_r(const GramState& g, const void* X, int64_t ldx, int xtype, const double* w,
                          int remove_mean, double* mean, double* R, cudaStream_t st, cudaEvent_t mid) {
  cudaError_t e;
  int dev = 0, sms = 0, per = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int groups = g.f32 ? 3 : 5;
  // colE and G are neighbours: one clear
  const size_t clear = align256(sizeof(int) * (size_t)g.M) + sizeof(long long) * (size_t)groups * g.M * g.M;
  if ((e = cudaMemsetAsync(g.colE, 0, clear, st)) != cudaSuccess) return e;
  PrologueArgs pa{X, ldx, w, remove_mean, mean, g.Y, g.ldy, g.N, g.M, g.colE, g.hdr};
  if (g.f32) e = xtype == PYLOM_F32 ? prologue<float, float>(pa, sms, st) : prologue<double, float>(pa, sms, st);
  else e = xtype == PYLOM_F32 ? prologue<float, double>(pa, sms, st) : prologue<double, double>(pa, sms, st);
  if (e != cudaSuccess) return e;
  if ((e = launch_row_scale(g.Y, g.f32, g.ldy, g.M, g.colE, g.rowS, nullptr, st)) != cudaSuccess) return e;
  e = g.f32 ? gram_launch<float>(g, sms, nullptr, 0, 0, nullptr, nullptr, g.G, nullptr, g.hdr, st)
            : gram_launch<double>(g, sms, nullptr, 0, 0, nullptr, nullptr, g.G, nullptr, g.hdr, st);
  if (e != cudaSuccess) return e;
  if (mid && (e = cudaEventRecord(mid, st)) != cudaSuccess) return e;
  CholArgs c{g, R, groups, g.f32 ? gram_base<float>(0) : gram_base<double>(0),
             g.f32 ? fix_bias<float>() : fix_bias<double>()};
  const int64_t nb = (g.M + kNBC - 1) / kNBC;
  if (nb <= kChCluster) {
    cudaLaunchConfig_t cfg = {};
    const unsigned n = nb <= 2 ? 1u : (unsigned)kChCluster;
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(kChThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gram_chol_kernel<true>, c);
  }
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, gram_chol_kernel<false>, kChThreads, 0);
  if (e != cudaSuccess) return e;
  if (per < 1) return cudaErrorCooperativeLaunchTooLarge;
  int64_t grid = nb + nb * (nb - 1) / 4;
  if (grid > sms) grid = sms;
  void* args[] = {&c};
  return cudaLaunchCooperativeKernel((const void*)gram_chol_kernel<false>, dim3((unsigned)grid), dim3(kChThreads), args,
                                     0, st);
}

}  // namespace pylom
