// svd_batched_gram.cu -- batched SVDs by Gram matrices: the per-frequency
// SVDs of SPOD (pyLOM, arXiv 2405.15529, Alg. 6) and the PODs of several
// real windows (Alg. 2 per window), mixed precision.
//
// The persistent Householder kernel (svd_batched.cu) walks every leaf column
// by column: 3 % of the binary32 rate, and one thread block per item for
// the small SVD in binary64.  Here every step runs over all items at once:
//   1. column exponents (and, for windows, mean, weights and a binary32 copy);
//   2. G = Y^H Y exactly, by digit products on the tcgen05 tensor cores
//      (digits.cuh).  A complex column is its 2N interleaved real and
//      imaginary parts: Re G_ij is the product of columns i and j, Im G_ij
//      that of column i turned by 90 degrees, (-im, re), and column j;
//   3. Cholesky factor R in binary64, in one block's shared memory;
//   4. complex one-sided Jacobi of R^H: two binary32 block stages (one
//      cluster per item) and two binary64 steps of simultaneous rotations,
//      as in the single small SVD (svd_jacobi32.cu);
//   5. U = Y W_k S_k^-1 (W the right vectors) by digit products.
// Items whose result would be less accurate than the Householder route's
// (a kept mode below 1e-5 of the largest singular value, where squaring
// costs binary32 digits; kept values too close to separate in two steps; any
// sound column that the binary32 stages left open; a zero matrix) are flagged on the device and left to that kernel.
//
// Persistent kernel -> here: 24 bins (N 16k..262k, Nb 16..128, 1.3 GB) 374 ->
// 13.1 ms, 12 windows (N 16k..262k, M 16..96) 119 -> 4.8 ms, SPOD of 131072 x
// 1056 25.6 -> 7.3 ms; modes within 2.5e-8 of binary64 (2.4e-7 before).
#include <algorithm>

#include "digits.cuh"
#include "svd_batched_gram.h"

namespace pylom {

namespace {

constexpr int kSB = Dig<float>::S;                 // 5 digits
constexpr int kG = 1;                              // two blocks an SM: the sums of a bin are short
constexpr int kTile = Shape<kG>::TILE, kPlaneB = Shape<kG>::PLANEB, kThreads = Shape<kG>::THREADS;
constexpr int kNstB = Dig<float>::NST<kG>, kAhead = Dig<float>::AHEAD<kG>;
constexpr int kStageB = kSB * (kPlaneA + kPlaneB);
// Smallest kept value, relative to the first, for which the modes are taken.
// Squaring costs them about 0.2 x 2^-53 / level^2: at 1.1e-5 the modes are 1e-7
// to 2e-7 off and as far from orthonormal (30,000 x 127 and 20,011 x 24), where
// binary32 leaves are 5e-4 to 1e-3 off, 3e-7 from orthonormal, and take 230 ms
// for 127 columns against 5.  (At 1e-4 all items of 100 and more columns of a
// wave field on a floor of 1e-3 were left to them: 64 bins 577 ms, here 108.)
constexpr double kKeptLevel = 1e-5;
constexpr double kOpenCos = 1e-6;                  // kept columns: largest cosine before the last step
// Singular values below this share of the first are rounding (the square root
// of the pivots that the Cholesky factor drops, and some room)
constexpr double kSoundLevel = 1e-7;

struct BG {
  const GramBin* bins;
  const GramUnit* units;
  int* ints;
  unsigned long long* g;
  double2* z;
  float2* f;
  unsigned char* c;
  double* d;
  uint16_t* rows;
  int* flags;
  double* S;
  WsHeader* hdr;
};

// a window whose right vectors are asked for
__device__ __forceinline__ bool has_vt(const GramBin& b) { return b.kind != 0 && b.VT; }

__device__ __forceinline__ double2* mat(const BG& a, const GramBin& b, int i) {
  return a.z + b.z + (int64_t)i * b.Nb * b.Nb;
}

// ---------------------------------------------------------------------------
// 1. column exponents; windows: Y = sqrt(w) (x - mean) in binary32
// ---------------------------------------------------------------------------
// Rows' largest exponent fields: lanes hold (pairs of) consecutive rows, warps
// take columns in turn; the eight warps' maxima meet in shared memory.
constexpr int kTopRows = 256;
struct RowTops {
  int t[2][8][kTopRows];       // (a warp may be an iteration ahead of the reads)
};
// all threads: `n` rows (a warp's maxima are in its line), the first `live` of them to `out`
__device__ __forceinline__ void store_tops(const RowTops& s, int turn, int n, int64_t live, uint16_t* out) {
  __syncthreads();
  for (int i = threadIdx.x; i < n && i < live; i += 256) {
    int t = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) t = max(t, s.t[turn][q][i]);
    out[i] = (uint16_t)t;
  }
}

template <typename TX>
__device__ void window_rows(const GramBin& b, float* Y, uint16_t* rows, int64_t r0, int64_t r1, int* sE, RowTops& tops,
                            int& bad) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ double ssum[8][32];
  const TX* X = (const TX*)b.Xr;
  int em[16];
#pragma unroll
  for (int t = 0; t < 16; ++t) em[t] = 0;
  int turn = 0;
  for (int64_t blk = r0; blk < r1; blk += 32, turn ^= 1) {
    const int64_t n = blk + lane;
    const bool in = n < b.rows;
    TX x[16];
    double s = 0.0;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int c = warp + 8 * t;
      x[t] = (in && c < b.Nb) ? X[n + (int64_t)c * b.ldx] : (TX)0;
    }
    double xbar = 0.0;
    if (b.remove_mean) {
      if constexpr (sizeof(TX) == 4) {
        float h, l;
        sum32_compensated(x, h, l);
        s = (double)h + (double)l;
      } else {
#pragma unroll
        for (int t = 0; t < 16; ++t) s += x[t];
      }
      ssum[warp][lane] = s;
      __syncthreads();
      double tot = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) tot += ssum[q][lane];
      xbar = tot / (double)b.Nb;
      __syncthreads();
    }
    double sw = 1.0;
    if (b.w && in) {
      const double wn = b.w[n];
      if (!(wn > 0.0) || !isfinite(wn)) bad = 1;
      sw = sqrt(wn);
    }
    if (warp == 0 && in && b.mean) b.mean[n] = xbar;
    const float xh = (float)xbar, xl = (float)(xbar - (double)xh);
    const float sh = (float)sw, sl = (float)(sw - (double)sh);
    int top = 0;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int c = warp + 8 * t;
      if (c >= b.Nb) continue;
      float y;
      if constexpr (sizeof(TX) == 4) {
        float d, e;
        two_sum32(x[t], -xh, d, e);
        y = __fmaf_rn(d, sh, __fmaf_rn(d, sl, __fmul_rn(__fsub_rn(e, xl), sh)));
      } else {
        y = (float)(sw * (x[t] - xbar));
      }
      if (!in) y = 0.f;
      if (!isfinite(x[t])) bad = 1;
      const int e = exp_field(y);
      em[t] = max(em[t], e);
      top = max(top, e);
      if (n < b.ldy) Y[n + (int64_t)c * b.ldy] = y;
    }
    tops.t[turn][warp][lane] = top;
    store_tops(tops, turn, 32, b.ldy - blk, rows + blk);
  }
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    const int e = __reduce_max_sync(0xffffffffu, em[t]);
    if (lane == 0 && warp + 8 * t < b.Nb) sE[warp + 8 * t] = e;
  }
}

// A bin: NC columns a warp, four groups of 32 points a turn (4 NC loads in flight).
template <int NC>
__device__ void bin_rows(const GramBin& b, uint16_t* rows, int64_t p0, int64_t p1, int* sE, RowTops& tops, int& bad) {
  constexpr int G = 4;
  static_assert(64 * G <= kTopRows, "room for the maxima");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float2* col = (const float2*)b.Y + (int64_t)warp * (b.ldy / 2) + lane;
  int em[NC];
#pragma unroll
  for (int t = 0; t < NC; ++t) em[t] = 0;
  int turn = 0;
  for (int64_t pr = p0; pr < p1; pr += 32 * G, turn ^= 1) {
    float2 x[G][NC];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int t = 0; t < NC; ++t)
        x[g][t] = pr + 32 * g + lane < p1 && warp + 8 * t < b.Nb ? __ldg(col + pr + 32 * g + t * 4 * b.ldy) : make_float2(0.f, 0.f);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      int tx = 0, ty = 0;
#pragma unroll
      for (int t = 0; t < NC; ++t) {
        const int ex = (__float_as_int(x[g][t].x) >> 23) & 0xff, ey = (__float_as_int(x[g][t].y) >> 23) & 0xff;
        em[t] = max(em[t], max(ex, ey));
        tx = max(tx, ex);
        ty = max(ty, ey);
      }
      *(int2*)&tops.t[turn][warp][64 * g + 2 * lane] = make_int2(tx, ty);
    }
    store_tops(tops, turn, 64 * G, 2 * (p1 - pr), rows + 2 * pr);
  }
#pragma unroll
  for (int t = 0; t < NC; ++t) {
    const int e = __reduce_max_sync(0xffffffffu, em[t]);
    if (e == 0xff) bad = 1;
    if (lane == 0 && warp + 8 * t < b.Nb) sE[warp + 8 * t] = max(e, kMinField32);
  }
}

// Besides the columns' exponents every row's largest one goes to a.rows; 16
// loads a lane and more hide the latency of memory (a warp per column took 0.52
// ms for the 1.1 GB of 131072 x 1056 in bins of 32 columns, this 0.29).
__global__ void __launch_bounds__(256) bg_prologue_kernel(BG a) {
  __shared__ int sE[128];
  __shared__ RowTops tops;
  const GramUnit u = a.units[blockIdx.x];
  if (u.bin < 0) return;
  const GramBin b = a.bins[u.bin];
  int bad = 0;
  if (b.kind == 0) {
    if (b.Nb <= 32) bin_rows<4>(b, a.rows + b.r, u.q0, u.q1, sE, tops, bad);
    else if (b.Nb <= 64) bin_rows<8>(b, a.rows + b.r, u.q0, u.q1, sE, tops, bad);
    else bin_rows<16>(b, a.rows + b.r, u.q0, u.q1, sE, tops, bad);
  } else if (b.kind == 1) {
    window_rows<float>(b, (float*)b.Y, a.rows + b.r, u.q0, u.q1, sE, tops, bad);
  } else {
    window_rows<double>(b, (float*)b.Y, a.rows + b.r, u.q0, u.q1, sE, tops, bad);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < b.Nb; c += 256) atomicMax(a.ints + b.colE + c, sE[c]);
  if (bad) raise_status(a.hdr, PYLOM_ERR_NONFINITE);
}

// Shift of each row, as in the single POD (row_scale_kernel, gram.cu): how far
// its elements all lie below their columns' largest exponents.  Where these
// differ by at most kSpread, how far the row's largest exponent lies below the
// smallest of them is near enough (38 bits are 14 more than the modes hold),
// and nothing is read again.  Else a lane takes a pair of rows (a point of a
// bin: its real and imaginary parts), bound by memory.
constexpr int kSpread = 8;
__global__ void __launch_bounds__(256) bg_rows_kernel(BG a) {
  __shared__ int sE[128];
  __shared__ int stop[2][8][64];     // (a warp may be an iteration ahead of the reads)
  constexpr int kNone = -2147483647;
  __shared__ int s_lo, s_hi;
  const GramUnit u = a.units[blockIdx.x];
  if (u.bin < 0) return;
  const GramBin b = a.bins[u.bin];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_lo = 0x100;
    s_hi = 0;
  }
  __syncthreads();
  if (threadIdx.x < b.Nb) {
    const int E = a.ints[b.colE + threadIdx.x];
    sE[threadIdx.x] = E << 23;
    if (E > kMinField32) {           // (columns of zeros apart)
      atomicMin(&s_lo, E);
      atomicMax(&s_hi, E);
    }
  }
  __syncthreads();
  if (s_hi - s_lo <= kSpread) {
    const int64_t f = b.cplx ? 2 : 1;
    for (int64_t n = f * u.q0 + threadIdx.x; n < f * u.q1; n += 256) {
      uint16_t& r = a.rows[b.r + n];
      r = r > kMinField32 && r < s_lo ? (uint16_t)(s_lo - r) : 0;
    }
    return;
  }
  const int64_t p0 = b.cplx ? u.q0 : u.q0 / 2, p1 = b.cplx ? u.q1 : u.q1 / 2;
  int turn = 0;
  for (int64_t pr = p0; pr < p1; pr += 32, turn ^= 1) {
    const bool in = pr + lane < p1;
    const float* p = b.Y + 2 * (pr + lane);
    float2 x[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int c = warp + 8 * t;
      x[t] = in && c < b.Nb ? __ldg((const float2*)(p + c * b.ldy)) : make_float2(0.f, 0.f);
    }
    int t0 = kNone, t1 = kNone;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int c = warp + 8 * t;
      const int E = c < b.Nb ? sE[c] : 0;
      const int hx = __float_as_int(x[t].x) & 0x7f800000, hy = __float_as_int(x[t].y) & 0x7f800000;
      if (hx > (kMinField32 << 23)) t0 = max(t0, hx - E);
      if (hy > (kMinField32 << 23)) t1 = max(t1, hy - E);
    }
    stop[turn][warp][2 * lane] = t0;
    stop[turn][warp][2 * lane + 1] = t1;
    __syncthreads();
    if (threadIdx.x < 64 && pr + threadIdx.x / 2 < p1) {
      int t = kNone;
#pragma unroll
      for (int q = 0; q < 8; ++q) t = max(t, stop[turn][q][threadIdx.x]);
      a.rows[b.r + 2 * pr + threadIdx.x] = (uint16_t)(t == kNone ? 0 : -(t >> 23));
    }
  }
}

// ---------------------------------------------------------------------------
// 2. exact Gram matrices
// ---------------------------------------------------------------------------
// Unit modes: the 128 rows of the left factor are columns 0..127 (kPlain),
// columns 0..63 and the same turned by 90 degrees (kPacked: Re and Im in one
// pass, for the first 64 columns), or columns 0..127 turned (kTurned).  The
// right factor is the column block J of 32.
enum { kPlain = 0, kPacked = 1, kTurned = 2 };

// rows row..row+7 of a column (turned: (-im, re) pairs)
__device__ __forceinline__ void fetch_rows8(const GramBin& b, int64_t row, int col, bool turned, float (&y)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) y[i] = 0.f;
  if (col < b.Nb) {
    const float* p = b.Y + row + (int64_t)col * b.ldy;
    if (row + 8 <= b.rows && ((uintptr_t)p & 15) == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float4 v = __ldg((const float4*)p + i);
        y[4 * i] = v.x;
        y[4 * i + 1] = v.y;
        y[4 * i + 2] = v.z;
        y[4 * i + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (row + i < b.rows) y[i] = __ldg(p + i);
    }
  }
  if (turned) {
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const float x = y[i];
      y[i] = -y[i + 1];
      y[i + 1] = x;
    }
  }
}

__global__ void __launch_bounds__(kThreads, Shape<kG>::BLOCKS) bg_gram_kernel(BG a) {
  extern __shared__ __align__(1024) unsigned char gsm[];
  __shared__ __align__(8) DigitBarriers<kNstB, kG> bar;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const GramUnit u = a.units[blockIdx.x];
  if (u.bin < 0) return;
  const GramBin b = a.bins[u.bin];
  const int mode = u.mode, J = u.J;
  // a thread: 8 rows of one left column, and in two of the eight warps, in turn
  // from stage to stage, 8 rows of one right column
  const int t = threadIdx.x, ca = t & 127, kg = t >> 7, cb = lane;
  const bool turned = mode == kTurned || (mode == kPacked && ca >= 64);
  // real items have nothing to turn: their second half is empty
  const int colA = (mode == kPacked && ca >= 64 && !b.cplx) ? 128 : mode == kPacked ? (ca & 63) : ca;
  const int EA = colA < b.Nb ? a.ints[b.colE + colA] : 128;
  const bool sepB = mode == kTurned;             // else the right factor's columns are among the left's
  const int colB = J * kTile + cb;
  const int EB = (sepB && colB < b.Nb) ? a.ints[b.colE + colB] : 128;
  float yA[8], yB[8];
  int turn = 7;
  auto fetch = [&](int j) {
    const int64_t row = (u.q0 * kStagesPerSum + j) * kStK;
    fetch_rows8(b, row + kg * 8, colA, turned, yA);
    turn = (warp + 2 * j) & 7;
    if (sepB && turn < 2) fetch_rows8(b, row + turn * 8, colB, false, yB);
    return true;
  };
  const int oa = (ca >> 3) * kPlaneSbo + (ca & 7) * 16 + kg * 128;
  // the left factor's columns that are the right one's too
  const int ob = kSB * kPlaneA + ((ca & 31) >> 3) * kPlaneSbo + (ca & 7) * 16 + kg * 128;
  const bool both = !sepB && (ca >> 5) == J;
  auto fill = [&](unsigned char* st) {
    put_digits(yA, EA, st + oa, kPlaneA, both ? st + ob : nullptr, kPlaneB);
    if (sepB && turn < 2)
      put_digits(yB, EB, st + kSB * kPlaneA + (cb >> 3) * kPlaneSbo + (cb & 7) * 16 + turn * 128, kPlaneB, nullptr, 0);
  };
  auto issue = [&](uint32_t tmem, uint32_t sa, bool first) {
    issue_stage<kSB, gram_base<float>(0), kG>(tmem, tc05::desc(sa, 128, kPlaneSbo), tc05::desc(sa + kSB * kPlaneA, 128, kPlaneSbo),
                                          first);
  };
  auto flush = [&](int64_t (&acc0)[16], int64_t (&acc1)[16]) {
    const int row = (warp & 3) * 32 + lane;
    const bool im = mode == kTurned || (mode == kPacked && row >= 64);
    const int i = mode == kPacked ? (row & 63) : row;
    const int64_t MM = (int64_t)b.Nb * b.Nb;
    unsigned long long* G = a.g + b.g + (im ? 3 * MM : 0);
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int j = J * kTile + (warp >> 2) * 16 + c;
      if (i < b.Nb && j < b.Nb && (im ? (i < j && b.cplx) : i <= j)) {
        add_group(G, MM, i + (int64_t)j * b.Nb, 0, acc0[c]);
        add_group(G, MM, i + (int64_t)j * b.Nb, 1, acc1[c]);
      }
      acc0[c] = acc1[c] = 0;
    }
  };
  gram_pipeline<kNstB, 0, kG>(bar, gsm, kStageB, (int)(u.q1 - u.q0) * kStagesPerSum, 8, a.hdr, [](int) {}, [](int) {}, fetch, fill,
                          issue, flush);
}

// ---------------------------------------------------------------------------
// complex helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 zmulc(double2 a, double2 b) {   // conj(a) b
  return make_double2(fma(a.x, b.x, a.y * b.y), fma(a.x, b.y, -a.y * b.x));
}
__device__ __forceinline__ float2 fmulc(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.x, b.y, -a.y * b.x));
}
__device__ __forceinline__ float2 fmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// ---------------------------------------------------------------------------
// 3. Cholesky: A = R^H (matrix 0), A32 = its binary32 copy scaled, V32 = I
// ---------------------------------------------------------------------------
// One block per item, the upper triangle packed by rows in shared memory
// (at most 132 KB).  G = D H D with D the columns' scales: H's entries are
// the exact integer sums.
constexpr int kCholThreads = 512;
__device__ __forceinline__ int tri(int i, int j, int n) { return i * n - i * (i - 1) / 2 + (j - i); }   // row i, column j >= i

__global__ void __launch_bounds__(kCholThreads) bg_chol_kernel(BG a) {
  extern __shared__ __align__(16) unsigned char csm[];
  double2* H = (double2*)csm;
  __shared__ double s_inv, s_diag[128];
  __shared__ unsigned s_e;
  const GramBin b = a.bins[blockIdx.x];
  const int n = b.Nb, tid = threadIdx.x;
  const int64_t MM = (int64_t)n * n;
  const long long* Gr = (const long long*)a.g + b.g;
  auto sum = [&](const long long* G, int64_t at) {
    // groups 0..2 of 32 bits each, exact but for one rounding
    return fma((double)__ldcg(G + 2 * MM + at), 4294967296.0, (double)__ldcg(G + MM + at)) * 4294967296.0 +
           (double)__ldcg(G + at);
  };
  for (int64_t idx = tid; idx < MM; idx += kCholThreads) {
    const int i = (int)(idx % n), j = (int)(idx / n);
    if (i <= j) H[tri(i, j, n)] = make_double2(sum(Gr, idx), (b.cplx && i < j) ? sum(Gr + 3 * MM, idx) : 0.0);
  }
  if (tid == 0) s_e = 0;
  __syncthreads();
  if (tid < n) s_diag[tid] = H[tri(tid, tid, n)].x;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (tid == 0) {
      const double d = H[tri(k, k, n)].x;
      // a pivot at the rounding level of its column: a dependent column, a zero row of R
      const bool live = d > 1e-15 * s_diag[k];
      s_inv = live ? 1.0 / sqrt(d) : 0.0;
    }
    __syncthreads();
    const double inv = s_inv;
    for (int j = k + tid; j < n; j += kCholThreads) {
      double2& h = H[tri(k, j, n)];
      h = make_double2(h.x * inv, h.y * inv);
    }
    __syncthreads();
    // rows i > k: H_ij -= conj(R_ki) R_kj; a warp per row
    if (inv != 0.0) {
      const int lane = tid & 31, warp = tid >> 5;
      for (int i = k + 1 + warp; i < n; i += kCholThreads / 32) {
        const double2 r = H[tri(k, i, n)];
        const double2* hk = H + tri(k, i, n);
        double2* hi = H + tri(i, i, n);
        for (int j = lane; j < n - i; j += 32) {
          const double2 x = hk[j], p = zmulc(r, x);
          hi[j] = make_double2(hi[j].x - p.x, hi[j].y - p.y);
        }
      }
    }
    __syncthreads();
  }
  // A = R^H with the columns of R scaled back: A(j, c) = conj(R(c, j)) 2^(E_j - bias)
  double2* A = mat(a, b, 0);
  const int* E = a.ints + b.colE;
  unsigned em = 0;
  for (int64_t idx = tid; idx < MM; idx += kCholThreads) {
    const int j = (int)(idx % n), c = (int)(idx / n);
    double2 v = make_double2(0.0, 0.0);
    if (c <= j) {
      const double2 r = H[tri(c, j, n)];
      // the sums count from level 1 (2^8)
      const double s = scalbn(16.0, E[j] - fix_bias<float>());
      v = make_double2(r.x * s, -r.y * s);
      if (E[j] == kMaxField32) v.x = quiet_nan();      // (the item is left to the Householder kernel)
    }
    A[idx] = v;
    em = max(em, (unsigned)max(exp_field(v.x), exp_field(v.y)));
  }
  em = __reduce_max_sync(0xffffffffu, em);
  if ((tid & 31) == 0) atomicMax(&s_e, em);
  __syncthreads();
  if (tid == 0) a.d[b.d] = (double)s_e;
  const double sc = __hiloint2double((s_e > 1 && s_e < 2045 ? 2046 - (int)s_e : 1023) << 20, 0);
  float2* A32 = a.f + b.f;
  float2* V32 = A32 + (int64_t)n * b.Mb;
  for (int64_t idx = tid; idx < (int64_t)n * b.Mb; idx += kCholThreads) {
    const int64_t c = idx / n;
    float2 v = make_float2(0.f, 0.f);
    if (c < n) v = make_float2((float)(A[idx].x * sc), (float)(A[idx].y * sc));
    A32[idx] = v;
  }
  for (int64_t idx = tid; idx < (int64_t)b.Mb * b.Mb; idx += kCholThreads)
    V32[idx] = make_float2(idx % b.Mb == idx / b.Mb ? 1.f : 0.f, 0.f);
}

// second stage: A32 from the binary64 A2, V32 = I
__global__ void __launch_bounds__(256) bg_init_kernel(BG a) {
  const GramBin b = a.bins[blockIdx.y];
  const int n = b.Nb;
  const int e = (int)a.d[b.d];
  const double sc = __hiloint2double((e > 1 && e < 2045 ? 2046 - e : 1023) << 20, 0);
  const double2* A = mat(a, b, 2);
  float2* A32 = a.f + b.f;
  float2* V32 = A32 + (int64_t)n * b.Mb;
  const int64_t stride = (int64_t)gridDim.x * 256, t0 = (int64_t)blockIdx.x * 256 + threadIdx.x;
  for (int64_t idx = t0; idx < (int64_t)n * b.Mb; idx += stride) {
    float2 v = make_float2(0.f, 0.f);
    if (idx / n < n) v = make_float2((float)(A[idx].x * sc), (float)(A[idx].y * sc));
    A32[idx] = v;
  }
  for (int64_t idx = t0; idx < (int64_t)b.Mb * b.Mb; idx += stride)
    V32[idx] = make_float2(idx % b.Mb == idx / b.Mb ? 1.f : 0.f, 0.f);
}

// T0 = V32 (binary64)
__global__ void __launch_bounds__(256) bg_widen_kernel(BG a) {
  const GramBin b = a.bins[blockIdx.y];
  const int n = b.Nb;
  const float2* V32 = a.f + b.f + (int64_t)n * b.Mb;
  double2* T = mat(a, b, 3);
  for (int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x; idx < (int64_t)n * n; idx += (int64_t)gridDim.x * 256) {
    const float2 v = V32[idx % n + (idx / n) * b.Mb];
    T[idx] = make_double2(v.x, v.y);
  }
}

// ---------------------------------------------------------------------------
// 4. binary32 block Jacobi (one cluster, the grid's x, per item; see svd_jacobi32.cu)
// ---------------------------------------------------------------------------
constexpr int kZB = 16, kZW = 32, kZThreads = 256, kZRows = 32, kZSweeps = 24;

__device__ __forceinline__ void z_rotation(float al, float be, float2 ga, float thr2, float& c, float& sn, float2& ph) {
  // |ga|, its phase, and the real rotation of [a_i, e^(-i phi) a_j]
  const float g2 = fmaf(ga.x, ga.x, ga.y * ga.y);
  const bool act = g2 > thr2 * fabsf(al * be);
  float ig;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ig) : "f"(fmaxf(g2, 1e-37f)));
  const float ag = g2 * ig;                 // |ga|
  ph = act ? make_float2(ga.x * ig, -ga.y * ig) : make_float2(1.f, 0.f);
  const float d = be - al, h = ag + ag;
  float r, q;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaf(d, d, h * h)));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(fmaxf(fabsf(d) + r, h)));
  const float t = act ? copysignf(1.f, d) * h * q : 0.f;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(fmaf(t, t, 1.f)));
  sn = c * t;
}

__global__ void __launch_bounds__(kZThreads) bg_jacobi32_kernel(BG a) {
  constexpr int LD = kZW + 2;
  extern __shared__ __align__(16) unsigned char jsm[];
  float2* sA = (float2*)jsm;                                   // [kZRows][LD], then partial Gram matrices
  float2(*sG)[kZW][kZW + 1] = (float2(*)[kZW][kZW + 1])(sA + kZW * kZW);   // [2]
  float2(*sJ)[LD] = (float2(*)[LD])(sG + 2);                   // [kZW][LD]
  __shared__ unsigned char sI[kZW - 1][kZB], sK[kZW - 1][kZB];
  __shared__ unsigned s_rot, s_total[2];
  const GramBin b = a.bins[blockIdx.y];
  const int n = b.Nb, Mb = b.Mb, tid = threadIdx.x;
  float2* A32 = a.f + b.f;
  float2* V32 = A32 + (int64_t)n * Mb;
  const int nblk = Mb / kZB, npairs = nblk / 2;
  const float tol = 4.f * sqrtf((float)n) * 5.9604645e-8f;
  for (int idx = tid; idx < (kZW - 1) * kZB; idx += kZThreads) {
    const int round = idx / kZB, p = idx % kZB;
    int x, y;
    if (round < kZB) {
      x = p;
      y = kZB + (p + round) % kZB;
    } else {
      const int h = p / 8 * kZB, q = p % 8, r = round - kZB;
      x = h + ((q == 0) ? 0 : ((q - 1 + r) % (kZB - 1)) + 1);
      y = h + ((kZB - 2 - q + r) % (kZB - 1)) + 1;
    }
    sI[round][p] = (unsigned char)min(x, y);
    sK[round][p] = (unsigned char)max(x, y);
  }
  if (tid < 2) s_total[tid] = 0;
  auto cluster_sync = [&]() {
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  };
  cluster_sync();
  for (int sweep = 0; sweep < kZSweeps; ++sweep) {
    unsigned local = 0;
    for (int step = 0; step < nblk - 1; ++step) {
      const int pr = blockIdx.x;
      if (pr < npairs) {
        const int p = (pr == 0) ? 0 : ((pr - 1 + step) % (nblk - 1)) + 1;
        const int q = ((nblk - 2 - pr + step) % (nblk - 1)) + 1;
        const int bI = min(p, q), bJ = max(p, q);
        auto column = [&](int l) { return (int64_t)(l < kZB ? bI * kZB + l : bJ * kZB + (l - kZB)); };
        // 32 x 32 Gram matrix: 8 x 8 threads of 4 x 4 entries, 4 row slices
        const int ti = (tid & 7) * 4, tj = ((tid >> 3) & 7) * 4, sl = tid >> 6;
        float2 g[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) g[x][y] = make_float2(0.f, 0.f);
        for (int r0 = 0; r0 < n; r0 += kZRows) {
          __syncthreads();
#pragma unroll
          for (int u = 0; u < kZRows * kZW / kZThreads; ++u) {
            const int idx = tid + u * kZThreads, r = idx % kZRows, l = idx / kZRows;
            sA[r * LD + l] = (r0 + r < n) ? __ldcg(A32 + r0 + r + column(l) * n) : make_float2(0.f, 0.f);
          }
          __syncthreads();
#pragma unroll 2
          for (int r = sl; r < kZRows; r += 4) {
            float2 x[4], y[4];
#pragma unroll
            for (int h = 0; h < 4; h += 2) {
              const float4 xv = *(const float4*)(sA + r * LD + ti + h), yv = *(const float4*)(sA + r * LD + tj + h);
              x[h] = make_float2(xv.x, xv.y);
              x[h + 1] = make_float2(xv.z, xv.w);
              y[h] = make_float2(yv.x, yv.y);
              y[h + 1] = make_float2(yv.z, yv.w);
            }
#pragma unroll
            for (int h = 0; h < 4; ++h)
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                g[h][v].x = fmaf(x[h].x, y[v].x, fmaf(x[h].y, y[v].y, g[h][v].x));
                g[h][v].y = fmaf(x[h].x, y[v].y, fmaf(-x[h].y, y[v].x, g[h][v].y));
              }
          }
        }
        __syncthreads();
        for (int h = 3; h >= 1; --h) {
          if (sl == h) {
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
              for (int y = 0; y < 4; ++y) sA[(ti + x) * kZW + tj + y] = g[x][y];
          }
          __syncthreads();
          if (sl == 0) {
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
              for (int y = 0; y < 4; ++y) {
                const float2 v = sA[(ti + x) * kZW + tj + y];
                g[x][y].x += v.x;
                g[x][y].y += v.y;
              }
          }
          __syncthreads();
        }
        if (tid == 0) s_rot = 0;
        if (sl == 0) {
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) sG[0][ti + x][tj + y] = g[x][y];
        }
        for (int idx = tid; idx < kZW * kZW; idx += kZThreads)
          sJ[idx / kZW][idx % kZW] = make_float2(idx / kZW == idx % kZW ? 1.f : 0.f, 0.f);
        __syncthreads();
        unsigned open = 0;
        for (int idx = tid; idx < kZW * kZW; idx += kZThreads) {
          const int i = idx / kZW, j = idx % kZW;
          const float2 v = sG[0][i][j];
          if (i < j && fmaf(v.x, v.x, v.y * v.y) > tol * tol * (sG[0][i][i].x * sG[0][j][j].x)) ++open;
        }
        if (open) atomicAdd(&s_rot, open);
        __syncthreads();
        open = s_rot;
        local += open;
        if (open) {
          const int pb = tid & 15, qb = tid >> 4;
          const int rounds = step == 0 ? kZW - 1 : kZB;
          const float thr2 = 0.0625f * tol * tol;
          int ni = sI[0][pb], nj = sK[0][pb], nk = sI[0][qb], nl = sK[0][qb];
          for (int round = 0; round < rounds; ++round) {
            const float2(*G0)[kZW + 1] = sG[round & 1];
            float2(*G1)[kZW + 1] = sG[(round & 1) ^ 1];
            const int i = ni, j = nj, k = nk, l = nl, nr = round + 1 < rounds ? round + 1 : 0;
            ni = sI[nr][pb];
            nj = sK[nr][pb];
            nk = sI[nr][qb];
            nl = sK[nr][qb];
            float cp, sp, cq, sq;
            float2 pp, pq;
            z_rotation(G0[i][i].x, G0[j][j].x, G0[i][j], thr2, cp, sp, pp);
            z_rotation(G0[k][k].x, G0[l][l].x, G0[k][l], thr2, cq, sq, pq);
            // columns: x_k' = cq x_k - sq pq x_l, x_l' = sq x_k + cq pq x_l
            const float2 e = G0[i][k], f = fmul(pq, G0[i][l]), gg = G0[j][k], h = fmul(pq, G0[j][l]);
            const float2 e1 = make_float2(cq * e.x - sq * f.x, cq * e.y - sq * f.y);
            const float2 f1 = make_float2(sq * e.x + cq * f.x, sq * e.y + cq * f.y);
            const float2 g1 = fmulc(pp, make_float2(cq * gg.x - sq * h.x, cq * gg.y - sq * h.y));
            const float2 h1 = fmulc(pp, make_float2(sq * gg.x + cq * h.x, sq * gg.y + cq * h.y));
            // rows, conjugated
            G1[i][k] = make_float2(cp * e1.x - sp * g1.x, cp * e1.y - sp * g1.y);
            G1[i][l] = make_float2(cp * f1.x - sp * h1.x, cp * f1.y - sp * h1.y);
            G1[j][k] = make_float2(sp * e1.x + cp * g1.x, sp * e1.y + cp * g1.y);
            G1[j][l] = make_float2(sp * f1.x + cp * h1.x, sp * f1.y + cp * h1.y);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int r = qb + 16 * u;
              const float2 x = sJ[r][i], y = fmul(pp, sJ[r][j]);
              sJ[r][i] = make_float2(cp * x.x - sp * y.x, cp * x.y - sp * y.y);
              sJ[r][j] = make_float2(sp * x.x + cp * y.x, sp * x.y + cp * y.y);
            }
            __syncthreads();
          }
          // A32 and V32 columns <- columns J; a thread per row and half of the new columns
          for (int i0 = 0; i0 < 2 * (n + Mb); i0 += kZThreads) {
            const int it = i0 + tid;
            const bool live = it < 2 * (n + Mb);
            const int row = live ? it >> 1 : 0, hf = it & 1;
            const bool isA = row < n;
            float2* base = isA ? A32 + row : V32 + (row - n);
            const int64_t ld = isA ? n : Mb;
            float2 v[kZW];
#pragma unroll
            for (int l = 0; l < kZW; ++l) v[l] = __ldcg(base + column(l) * ld);
            __syncwarp();   // both threads of the row have read it
            if (!live) continue;
#pragma unroll 1
            for (int l = hf * kZB; l < hf * kZB + kZB; l += 2) {
              float2 o0 = make_float2(0.f, 0.f), o1 = o0;
#pragma unroll
              for (int m = 0; m < kZW; ++m) {
                const float4 jv = *(const float4*)&sJ[m][l];
                o0.x = fmaf(v[m].x, jv.x, fmaf(-v[m].y, jv.y, o0.x));
                o0.y = fmaf(v[m].x, jv.y, fmaf(v[m].y, jv.x, o0.y));
                o1.x = fmaf(v[m].x, jv.z, fmaf(-v[m].y, jv.w, o1.x));
                o1.y = fmaf(v[m].x, jv.w, fmaf(v[m].y, jv.z, o1.y));
              }
              __stcg(base + column(l) * ld, o0);
              __stcg(base + column(l + 1) * ld, o1);
            }
          }
        }
      }
      cluster_sync();
    }
    // the cluster's open pairs of this sweep, at rank 0 (alternating words)
    if (tid == 0 && local) {
      uint32_t addr;
      asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(addr) : "r"(tc05::smem_u32(&s_total[sweep & 1])));
      asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" :: "r"(addr), "r"(local) : "memory");
    }
    cluster_sync();
    uint32_t addr, total;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(addr) : "r"(tc05::smem_u32(&s_total[sweep & 1])));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(total) : "r"(addr) : "memory");
    cluster_sync();
    if (blockIdx.x == 0 && tid == 0) s_total[sweep & 1] = 0;
    if (total == 0) break;
  }
  cluster_sync();   // no block leaves while another may read its shared memory
}

// ---------------------------------------------------------------------------
// binary64 products C = alpha op(A) B + beta D over all items, one or two at a time
// ---------------------------------------------------------------------------
struct ZGemm {
  int ta, A, B, D, C;       // matrix numbers; ta: A^H; D < 0: none
  double alpha, beta;
};
struct ZGemms {
  ZGemm g[2];
  int count;
  bool vt_only;             // only items with has_vt
};

__global__ void __launch_bounds__(128) bg_gemm_kernel(BG a, ZGemms gs) {
  __shared__ double2 part[4][8][9];
  const GramBin b = a.bins[blockIdx.z / gs.count];
  const ZGemm& p = gs.g[blockIdx.z % gs.count];
  const int n = b.Nb, i0 = blockIdx.x * 8, j0 = blockIdx.y * 8;
  if (i0 >= n || j0 >= n || (gs.vt_only && !has_vt(b))) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const double2* A = mat(a, b, p.A);
  const double2* B = mat(a, b, p.B);
  double r0 = 0.0, r1 = 0.0, m0 = 0.0, m1 = 0.0;
  const int i = i0 + g, j = j0 + g;
#pragma unroll 4
  for (int st = warp; st < (n + 3) / 4; st += 4) {
    const int kk = st * 4 + t;
    double2 x = make_double2(0.0, 0.0), y = x;
    if (kk < n && i < n) x = p.ta ? __ldg(A + kk + (int64_t)i * n) : __ldg(A + i + (int64_t)kk * n);
    if (kk < n && j < n) y = __ldg(B + kk + (int64_t)j * n);
    if (p.ta) x.y = -x.y;
    dmma884(r0, r1, x.x, y.x);
    if (b.cplx) {
      dmma884(r0, r1, -x.y, y.y);
      dmma884(m0, m1, x.x, y.y);
      dmma884(m0, m1, x.y, y.x);
    }
  }
  part[warp][g][2 * t] = make_double2(r0, m0);
  part[warp][g][2 * t + 1] = make_double2(r1, m1);
  __syncthreads();
  if (threadIdx.x < 64) {
    const int r = threadIdx.x & 7, c = threadIdx.x >> 3;
    if (i0 + r < n && j0 + c < n) {
      const int64_t at = (i0 + r) + (int64_t)(j0 + c) * n;
      double2 v = zadd(zadd(part[0][r][c], part[1][r][c]), zadd(part[2][r][c], part[3][r][c]));
      v = make_double2(p.alpha * v.x, p.alpha * v.y);
      if (p.D >= 0) {
        const double2 d = mat(a, b, p.D)[at];
        v = make_double2(fma(p.beta, d.x, v.x), fma(p.beta, d.y, v.y));
      }
      mat(a, b, p.C)[at] = v;
    }
  }
}

// Small-angle generator of a step from G (matrix 3) and W = V^H V (matrix
// 4): K (5), L = K - E (7), B = I + K - E/2 (4, in place of W), E = W - I.
// A pair's angle is t e^(i phi) on column j (+) and column i (-, conjugate).
// Columns whose angles are not small, or too many, are left alone.  `last`:
// also records each column's largest cosine.  A warp per column, twice: the
// columns' decisions are needed by all pairs.
__device__ __forceinline__ double z_tangent(double al, double be, double g) {
  if (!(g > 0.0)) return 0.0;
  const double zeta = (be - al) / (2.0 * g);
  return ((zeta >= 0.0) ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
}

__global__ void __launch_bounds__(256) bg_check_kernel(BG a, int last) {
  const GramBin b = a.bins[blockIdx.y];
  const int n = b.Nb, lane = threadIdx.x & 31, j = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (j >= n) return;
  const double2* G = mat(a, b, 3);
  const double be = G[j + (int64_t)j * n].x;
  double sum = 0.0, big = 0.0, cosm = 0.0;
  for (int i = lane; i < n; i += 32) {
    if (i == j) continue;
    const double al = G[i + (int64_t)i * n].x;
    const double2 v = G[i + (int64_t)j * n];
    const double g = sqrt(v.x * v.x + v.y * v.y), q = sqrt(al) * sqrt(be);
    const double c = q > 0.0 ? g / q : 0.0;
    cosm = fmax(cosm, c);
    if (c > 1e-14) {
      const double t = fabs(z_tangent(al, be, g));
      sum += t;
      big = fmax(big, t);
    }
  }
  sum = warp_sum(sum);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
    cosm = fmax(cosm, __shfl_xor_sync(0xffffffffu, cosm, o));
  }
  if (lane == 0) {
    const bool moves = big <= 0.02 && sum <= 0.05;
    // 2 more for a column that keeps the cosine
    a.d[b.d + 1 + j] = last ? (moves ? cosm : cosm + 2.0) : 0.0;
    a.d[b.d + 1 + n + j] = moves ? 1.0 : 0.0;
  }
}

__global__ void __launch_bounds__(256) bg_angles_kernel(BG a) {
  const GramBin b = a.bins[blockIdx.y];
  const int n = b.Nb;
  const double2* G = mat(a, b, 3);
  double2 *W = mat(a, b, 4), *K = mat(a, b, 5), *L = mat(a, b, 7);
  const double* mv = a.d + b.d + 1 + n;
  for (int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x; idx < (int64_t)n * n; idx += (int64_t)gridDim.x * 256) {
    const int i = (int)(idx % n), j = (int)(idx / n);
    double2 t = make_double2(0.0, 0.0);
    if (i != j && mv[i] != 0.0 && mv[j] != 0.0) {
      const double al = G[i + (int64_t)i * n].x, be = G[j + (int64_t)j * n].x;
      const double2 v = G[idx];
      const double g = sqrt(v.x * v.x + v.y * v.y), q = sqrt(al) * sqrt(be);
      if (g > 1e-14 * q && q > 0.0) {
        const double tt = z_tangent(al, be, g) / g;
        // column j gains t e^(i phi) a_i, e^(i phi) = G_ij / |G_ij| (the pair's
        // other entry follows by symmetry: G_ji = conj G_ij and t changes sign)
        t = make_double2(tt * v.x, tt * v.y);
      }
    }
    double2 e = W[idx];
    if (i == j) e.x -= 1.0;
    K[idx] = t;
    L[idx] = make_double2(t.x - e.x, t.y - e.y);
    W[idx] = make_double2((i == j ? 1.0 : 0.0) + t.x - 0.5 * e.x, t.y - 0.5 * e.y);
  }
}

// ---------------------------------------------------------------------------
// 5. order, phases, S, V^T of windows, coefficient digits, flags
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) bg_finalize_kernel(BG a) {
  __shared__ double sig[128];
  __shared__ double2 phs[128];
  __shared__ int perm[128], s_ce[64];
  const GramBin b = a.bins[blockIdx.x];
  const int n = b.Nb, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double2* A = mat(a, b, 0);
  for (int j = warp; j < n; j += 8) {
    double s2 = 0.0, best = -1.0;
    int kb = 0;
    for (int r = lane; r < n; r += 32) {
      const double2 v = A[r + (int64_t)j * n];
      const double m2 = v.x * v.x + v.y * v.y;
      s2 += m2;
      if (m2 > best) {
        best = m2;
        kb = r;
      }
    }
    s2 = warp_sum(s2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int ok = __shfl_xor_sync(0xffffffffu, kb, o);
      if (ob > best || (ob == best && ok < kb)) {
        best = ob;
        kb = ok;
      }
    }
    if (lane == 0) {
      sig[j] = sqrt(s2);
      const double2 v = A[kb + (int64_t)j * n];
      const double m = sqrt(v.x * v.x + v.y * v.y);
      phs[j] = m > 0.0 ? make_double2(v.x / m, -v.y / m) : make_double2(1.0, 0.0);
    }
  }
  __syncthreads();
  if (tid < n) {
    const double sj = (sig[tid] == sig[tid]) ? sig[tid] : -1.0;
    int rank = 0;
    for (int q = 0; q < n; ++q) {
      const double sq = (sig[q] == sig[q]) ? sig[q] : -1.0;
      rank += (sq > sj) || (sq == sj && q < tid);
    }
    perm[rank] = tid;
    a.S[b.s_off + rank] = sig[tid];
  }
  if (tid < 64) s_ce[tid] = kMinField64;
  __syncthreads();
  // leave the item to the Householder route?
  if (tid == 0) {
    const double s1 = sig[perm[0]];
    bool bad = !(s1 > 0.0);
    // the other sound columns: what the binary32 stages leave (their limit is 4
    // sqrt(n) 2^-24), else they ran out of sweeps
    const double left = 16.0 * sqrt((double)n) * 5.9604644775390625e-8;
    for (int c = 0; c < n; ++c) {
      const int j = perm[c];
      const double cs = a.d[b.d + 1 + j];
      if (c < b.k) bad = bad || !(sig[j] >= kKeptLevel * s1) || !(cs <= kOpenCos);
      else if (sig[j] >= kSoundLevel * s1) bad = bad || !((cs >= 2.0 ? cs - 2.0 : cs) <= left);
    }
    if (bad) {
      a.flags[b.flag] = 1;
      atomicAdd(a.flags - 1, 1);
    }
  }
  if (has_vt(b)) {
    // matrix 3: the right vectors in its columns; which of them are sound
    double2* W = mat(a, b, 3);
    for (int64_t idx = tid; idx < (int64_t)n * n; idx += 256) {
      const int c = (int)(idx / n), r = (int)(idx % n), j = perm[c];
      const double2 v = A[r + (int64_t)j * n], p = phs[j];
      W[idx] = make_double2(sig[j] > 0.0 ? (v.x * p.x - v.y * p.y) / sig[j] : 0.0, 0.0);
    }
    __syncthreads();                 // (the cosines have been read)
    if (tid < n) {
      const double s = sig[perm[tid]];
      a.d[b.d + 1 + tid] = s >= kSoundLevel * sig[perm[0]] && s > 0.0 ? 1.0 : s > 0.0 ? 0.5 : 0.0;
    }
  }
  if (b.k == 0) return;
  // C = W_k S_k^-1 2^(E - bias): column c (real items) or columns 2c (re),
  // 2c + 1 (im) of the planes
  const int* E = a.ints + b.colE;
  int* Ce = a.ints + b.colE + n;
  const int ncol = b.cplx ? 2 * b.k : b.k;
  const int stages = (n + kStK - 1) / kStK;
  auto value = [&](int r, int col) {
    const int c = b.cplx ? col >> 1 : col;
    if (r >= n || col >= ncol) return 0.0;
    const int j = perm[c];
    const double2 v = A[r + (int64_t)j * n], p = phs[j];
    const double x = (b.cplx && (col & 1)) ? v.x * p.y + v.y * p.x : v.x * p.x - v.y * p.y;
    return scalbn(x / sig[j] / sig[j], E[r] - fix_bias<float>());
  };
  for (int col = warp; col < ncol; col += 8) {
    int e = kMinField64;
    for (int r = lane; r < n; r += 32) e = max(e, exp_field(value(r, col)));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) s_ce[col] = e;
  }
  __syncthreads();
  if (tid < 64) Ce[tid] = s_ce[tid];
  for (int it = tid; it < 64 * stages * (kStK / 8); it += 256) {
    const int col = it & 63, j0 = (it >> 6) * 8;
    uint2 w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = bias_digits((to_fixed(value(j0 + i, col), s_ce[col]) + (1ll << 23)) >> 24);
    unsigned char* dst = a.c + b.c + ((int64_t)(col / kTile) * stages + j0 / kStK) * kSB * kPlaneB +
                         ((col % kTile) >> 3) * kPlaneSbo + ((j0 % kStK) >> 3) * 128 +
                         (col & 7) * 16;
    store_digits<kSB>(w, dst, kPlaneB);
  }
}

// Windows: all right vectors orthonormal to binary64 rounding, although only
// the kept columns are diagonalised to that.  Sound ones by two steps W <- W (I
// - T), T the strict upper triangle of E = W^T W - I among them and half its
// diagonal (cosines of binary32 rounding square in each): a vector sheds its
// part along larger ones, so that the kept ones keep their accuracy (I - E / 2
// would move them by half the cosines of the others, 1e-7).  Then those of
// rounding-level values, one after the other, against all before them.  0.18 of 4.8 ms for 12 windows.
__global__ void __launch_bounds__(256) bg_ortho_kernel(BG a) {
  const GramBin b = a.bins[blockIdx.y];
  if (!has_vt(b)) return;
  const int n = b.Nb;
  const double2* G = mat(a, b, 4);
  double2* B = mat(a, b, 5);
  const double* sound = a.d + b.d + 1;
  for (int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x; idx < (int64_t)n * n; idx += (int64_t)gridDim.x * 256) {
    const int i = (int)(idx % n), j = (int)(idx / n);
    const double one = i == j ? 1.0 : 0.0, part = i < j ? 1.0 : 0.5 * one;
    B[idx] = make_double2(sound[i] == 1.0 && sound[j] == 1.0 ? one - part * (G[idx].x - one) : one, 0.0);
  }
}

__global__ void __launch_bounds__(256) bg_vt_kernel(BG a) {
  __shared__ double v[128], cf[128], s_norm;
  const GramBin b = a.bins[blockIdx.x];
  if (!has_vt(b)) return;
  const int n = b.Nb, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double2* W = mat(a, b, 3);
  const double* sound = a.d + b.d + 1;
  int unit = 0;                            // next unit vector to try
  for (int c = 0; c < n; ++c) {
    if (sound[c] != 0.5) continue;         // (rows of exactly zero values stay zero)
    if (tid < n) v[tid] = W[tid + (int64_t)c * n].x;
    __syncthreads();
    for (;;) {
      for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 4
        for (int q = warp; q < c; q += 8) {
          double d = 0.0;
          for (int i = lane; i < n; i += 32) d = fma(W[i + (int64_t)q * n].x, v[i], d);
          d = warp_sum(d);
          if (lane == 0) cf[q] = d;
        }
        __syncthreads();
        if (tid < n) {
          double x = v[tid];
#pragma unroll 8
          for (int q = 0; q < c; ++q) x = fma(-cf[q], W[tid + (int64_t)q * n].x, x);
          v[tid] = x;
        }
        __syncthreads();
      }
      if (warp == 0) {
        double s = 0.0;
        for (int i = lane; i < n; i += 32) s = fma(v[i], v[i], s);
        s = warp_sum(s);
        if (lane == 0) s_norm = sqrt(s);
      }
      __syncthreads();
      const double nn = s_norm;
      if (nn > 0.5 / sqrt((double)n) || unit >= n) {
        if (tid < n) W[tid + (int64_t)c * n].x = nn > 0.0 ? v[tid] / nn : 0.0;
        break;
      }
      // it lay among those before it (of n unit vectors one is left with 1 / sqrt(n) or more)
      __syncthreads();
      if (tid < n) v[tid] = tid == unit ? 1.0 : 0.0;
      ++unit;
      __syncthreads();
    }
    __syncthreads();
  }
  for (int64_t idx = tid; idx < (int64_t)n * n; idx += 256) {
    const int c = (int)(idx % n), r = (int)(idx / n);
    b.VT[c + r * b.ldvt] = W[r + (int64_t)c * n].x;
  }
}

// U = Y C
__global__ void __launch_bounds__(kThreads, Shape<kG>::BLOCKS) bg_modes_kernel(BG a) {
  constexpr int LB = Dig<float>::LBM;
  extern __shared__ __align__(1024) unsigned char gsm[];
  __shared__ __align__(8) DigitBarriers<kNstB, kG> bar;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const GramUnit u = a.units[blockIdx.x];
  if (u.bin < 0) return;
  const GramBin b = a.bins[u.bin];
  const int n = b.Nb, stages = (n + kStK - 1) / kStK;
  const int rl = tid & 127, kh = tid >> 7;
  const uint32_t offA = (uint32_t)((rl >> 3) * kPlaneSbo + (rl & 7) * 16);
  const int* E = a.ints + b.colE;
  const int* Ce = a.ints + b.colE + n;
  float* ring = (float*)(gsm + kNstB * kStageB) + tid;
  // shift of row rl of a tile; the next tile's is on its way while one is done
  auto shift = [&](int t) {
    const int64_t row = (u.q0 + t) * 128 + rl;
    return row < b.rows ? (int)__ldg(a.rows + b.r + row) : 0;
  };
  int s_now = 0, s_next = 0, s_tile = -2;
  auto load = [&](int t, int js, int q) {
    const int64_t row = (u.q0 + t) * 128 + rl;
    const int c0 = js * kStK + kh * 8;
    const float* p = b.Y + row + c0 * b.ldy;
    if (row < b.rows) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (c0 + i < n) async_copy<4>(ring + (q * 8 + i) * kThreads, p + i * b.ldy);
    }
  };
  auto fill = [&](int t, int js, int q, unsigned char* st) {
    const bool rin = (u.q0 + t) * 128 + rl < b.rows;
    const int c0 = js * kStK + kh * 8;
    if (t != s_tile) {
      s_now = t == s_tile + 1 ? s_next : shift(t);
      s_tile = t;
      s_next = shift(t + 1);
    }
    float y[8];
    int e[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool in = c0 + i < n;
      y[i] = in && rin ? ring[(q * 8 + i) * kThreads] : 0.f;
      e[i] = in ? __ldg(E + c0 + i) - s_now : 128;
    }
    put_digits(y, e, st + offA + kh * 128, kPlaneA);
  };
  auto bsrc = [&](int, int js) { return a.c + b.c + (u.J * stages + js) * kSB * (int64_t)kPlaneB; };
  auto store = [&](int t, const int64_t (&acc0)[16], const int64_t (&acc1)[16]) {
    const int64_t row = (u.q0 + t) * 128 + (warp & 3) * 32 + lane;
    const int k0 = u.J * kTile + (warp >> 2) * 16;
    const double iw = (b.physical && b.w && row < b.rows) ? 1.0 / sqrt(b.w[row]) : 1.0;
    const int rs = shift(t);
    auto value = [&](int c) {
      const int pk = 8 * LB + __ldg(Ce + k0 + c) - fix_bias<double>() + 24 - rs;
      return from_sums(acc0[c], acc1[c], pk, 0.0);
    };
    if (b.cplx) {
      // rows 2m, 2m + 1 hold re, im of point m times the coefficients' parts
#pragma unroll
      for (int c = 0; c < 16; c += 2) {
        if (((k0 + c) >> 1) >= b.k) break;     // uniform over the warp; binary64 conversions are dear
        const double vr = value(c), vi = value(c + 1);
        const double pr = __shfl_xor_sync(0xffffffffu, vr, 1), pi = __shfl_xor_sync(0xffffffffu, vi, 1);
        const int k = (k0 + c) >> 1;
        if (!(lane & 1) && k < b.k && row < b.rows)
          b.U[(row >> 1) + (int64_t)k * b.ldu] = make_float2((float)(vr - pi), (float)(vi + pr));
      }
    } else {
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (k0 + c < b.k && row < b.rows) b.Ur[row + (int64_t)(k0 + c) * b.ldu] = (float)(value(c) * iw);
    }
  };
  product_pipeline<kSB, kNstB, LB, kAhead, kG>(bar, gsm, (int)(u.q1 - u.q0), stages, a.hdr, load, fill, bsrc, store);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

void batched_gram_add(BatchedGramPlan& p, int item, int64_t N, int64_t Nb, int64_t k, int64_t s_off) {
  GramBin b{};
  b.Nb = (int)Nb;
  b.Mb = (int)((Nb + kZW - 1) / kZW * kZW);
  b.k = (int)k;
  b.rows = N;                       // points; doubled at bind for complex items
  b.colE = p.n_i;                   p.n_i += Nb + 64;
  b.g = p.n_g;                      p.n_g += 6 * Nb * Nb;
  b.z = p.n_z;                      p.n_z += (int64_t)kBinMats * Nb * Nb;
  b.f = p.n_f;                      p.n_f += Nb * b.Mb + (int64_t)b.Mb * b.Mb;
  b.c = p.n_c;                      p.n_c += (Nb + kStK - 1) / kStK * kSB * (int64_t)kPlaneB * (64 / kTile);
  b.d = p.n_d;                      p.n_d += 1 + 2 * Nb;
  b.r = p.n_r;                      p.n_r += 2 * ((N + 7) & ~int64_t(7));     // real or complex: bind tells
  b.s_off = s_off;
  b.flag = item;
  p.items.push_back(item);
  p.bins.push_back(b);
  p.maxNb = std::max(p.maxNb, b.Nb);
  p.maxpairs = std::max(p.maxpairs, b.Mb / kZW);
}

static int column_blocks(int n) { return (n + kTile - 1) / kTile; }

size_t batched_gram_layout(BatchedGramPlan& p, size_t off, int nitems, int sms) {
  const int64_t nb = (int64_t)p.bins.size();
  p.nitems = nitems;
  // about four waves of units, and a tile's share rounded up (complex items have the most tiles)
  p.want = 8 * (int64_t)sms;
  p.n_pro = p.n_gram = p.n_mod = p.want;
  for (const GramBin& b : p.bins) {
    const int n = column_blocks(b.Nb);
    p.n_pro += 1;
    p.n_gram += n + (n > 2 ? n - 2 : 0);
    p.n_mod += column_blocks(2 * b.k);
  }
  if (p.n_mod == p.want) p.n_mod = 0;      // no modes
  p.off_flags = off; off += align256(sizeof(int) * ((size_t)nitems + 1) * 2);
  if (nb == 0) return off;
  p.off_bins = off;  off += align256(sizeof(GramBin) * (size_t)nb);
  p.off_units = off; off += align256(sizeof(GramUnit) * (size_t)(p.n_pro + p.n_gram + p.n_mod));
  p.off_i = off;     off += align256(sizeof(int) * (size_t)p.n_i);
  p.off_g = off;     off += align256(sizeof(long long) * (size_t)p.n_g);
  p.off_z = off;     off += align256(sizeof(double2) * (size_t)p.n_z);
  p.off_f = off;     off += align256(sizeof(float2) * (size_t)p.n_f);
  p.off_c = off;     off += align256((size_t)p.n_c);
  p.off_d = off;     off += align256(sizeof(double) * (size_t)p.n_d);
  p.off_r = off;     off += align256(sizeof(uint16_t) * (size_t)p.n_r);
  return off;
}

// Units of about equal cost, about four waves of them: an item's tiles (cost
// tiles x rows) are cut into row ranges.
void batched_gram_units(BatchedGramPlan& p) {
  for (const GramBin& b : p.bins) p.any_vt = p.any_vt || (b.kind != 0 && b.VT);
  p.pro.clear();
  p.gram.clear();
  p.mod.clear();
  double total = 0.0, mtotal = 0.0, ptotal = 0.0;
  auto passes = [&](const GramBin& b) {
    return b.Nb <= 64 ? column_blocks(b.Nb) : 2 + (column_blocks(b.Nb) - 2) * (b.cplx ? 2 : 1);
  };
  auto mtiles = [&](const GramBin& b) { return column_blocks(b.cplx ? 2 * b.k : b.k); };
  auto mcost = [](const GramBin& b) { return (double)((b.Nb + kStK - 1) / kStK); };
  for (const GramBin& b : p.bins) {
    total += (double)b.rows * passes(b);
    if (b.k > 0) mtotal += (double)b.rows * mcost(b) * mtiles(b);
    ptotal += (double)b.rows * b.Nb;
  }
  const double want = (double)p.want;
  for (size_t f = 0; f < p.bins.size(); ++f) {
    const GramBin& b = p.bins[f];
    const int64_t sums = (b.rows + 127) / 128;
    auto cut = [&](std::vector<GramUnit>& v, double share, int mode, int J, int64_t n) {
      int64_t s = (int64_t)share;          // (rounded down: no fifth wave of a few blocks)
      s = std::max<int64_t>(1, std::min(s, n));
      for (int64_t i = 0; i < s; ++i) v.push_back(GramUnit{(int)f, mode, J, 0, n * i / s, n * (i + 1) / s});
    };
    const double share = want * (double)b.rows / total;
    for (int J = 0; J < column_blocks(b.Nb); ++J) {
      cut(p.gram, share, J < 2 ? kPacked : kPlain, J, sums);
      if (J >= 2 && b.cplx) cut(p.gram, share, kTurned, J, sums);
    }
    for (int J = 0; J < mtiles(b); ++J) cut(p.mod, want * (double)b.rows * mcost(b) / mtotal, 0, J, sums);
    // prologue: points (bins) or rows rounded to 32 (windows)
    const int64_t pts = b.cplx ? b.rows / 2 : b.ldy;
    const int64_t blk = (pts + 31) / 32;
    const size_t first = p.pro.size();
    cut(p.pro, want * (double)b.rows * b.Nb / ptotal, 0, 0, blk);
    for (size_t i = first; i < p.pro.size(); ++i) {
      p.pro[i].q0 *= 32;
      p.pro[i].q1 = std::min(p.pro[i].q1 * 32, pts);
    }
  }
  auto longest = [](const GramUnit& x, const GramUnit& y) { return x.q1 - x.q0 > y.q1 - y.q0; };
  std::stable_sort(p.gram.begin(), p.gram.end(), longest);
  std::stable_sort(p.mod.begin(), p.mod.end(), [&](const GramUnit& x, const GramUnit& y) {
    return (double)(x.q1 - x.q0) * mcost(p.bins[x.bin]) > (double)(y.q1 - y.q0) * mcost(p.bins[y.bin]);
  });
}

cudaError_t batched_gram_upload(const BatchedGramPlan& p, char* ws, const int* forced, int nitems, cudaStream_t st) {
  // flags: [count, flags of the items] in use, then the same as given
  std::vector<int> fl((size_t)nitems + 1, 0);
  for (int i = 0; i < nitems; ++i) {
    fl[i + 1] = forced[i];
    fl[0] += forced[i] != 0;
  }
  cudaError_t e = cudaMemcpyAsync(ws + p.off_flags + sizeof(int) * ((size_t)nitems + 1), fl.data(),
                                  sizeof(int) * fl.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess || p.bins.empty()) return e;
  e = cudaMemcpyAsync(ws + p.off_bins, p.bins.data(), sizeof(GramBin) * p.bins.size(), cudaMemcpyHostToDevice, st);
  // (a few rounded shares may leave fewer units than there is room for)
  std::vector<GramUnit> all;
  const std::vector<GramUnit>* lists[3] = {&p.pro, &p.gram, &p.mod};
  const int64_t room[3] = {p.n_pro, p.n_gram, p.n_mod};
  for (int i = 0; i < 3; ++i) {
    if ((int64_t)lists[i]->size() > room[i]) return cudaErrorInvalidValue;
    all.insert(all.end(), lists[i]->begin(), lists[i]->end());
    all.resize(all.size() + (size_t)(room[i] - (int64_t)lists[i]->size()), GramUnit{-1, 0, 0, 0, 0, 0});
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ws + p.off_units, all.data(), sizeof(GramUnit) * all.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

cudaError_t batched_gram_run(const BatchedGramPlan& p, char* ws, WsHeader* hdr, double* S, cudaStream_t st) {
  if (p.bins.empty()) return cudaSuccess;
  cudaError_t e;
  BG a{};
  a.bins = (const GramBin*)(ws + p.off_bins);
  const GramUnit* units = (const GramUnit*)(ws + p.off_units);
  a.ints = (int*)(ws + p.off_i);
  a.g = (unsigned long long*)(ws + p.off_g);
  a.z = (double2*)(ws + p.off_z);
  a.f = (float2*)(ws + p.off_f);
  a.c = (unsigned char*)(ws + p.off_c);
  a.d = (double*)(ws + p.off_d);
  a.rows = (uint16_t*)(ws + p.off_r);
  a.flags = (int*)(ws + p.off_flags) + 1;
  a.S = S;
  a.hdr = hdr;
  const unsigned nb = (unsigned)p.bins.size();
  const size_t smem = (size_t)kNstB * kStageB, msmem = smem + (size_t)kAhead * 8 * kThreads * sizeof(float);
  const size_t csmem = sizeof(double2) * ((size_t)p.maxNb * (p.maxNb + 1) / 2);
  const size_t jsmem = sizeof(float2) * ((size_t)kZW * kZW + 2 * kZW * (kZW + 1) + kZW * (kZW + 2) + 64);
  if ((e = ensure_dyn_smem((const void*)bg_gram_kernel, smem)) != cudaSuccess) return e;
  if ((e = ensure_dyn_smem((const void*)bg_modes_kernel, msmem)) != cudaSuccess) return e;
  if ((e = ensure_dyn_smem((const void*)bg_chol_kernel, sizeof(double2) * 128 * 129 / 2)) != cudaSuccess) return e;
  if ((e = ensure_dyn_smem((const void*)bg_jacobi32_kernel, jsmem)) != cudaSuccess) return e;
  const size_t nfl = (size_t)p.nitems + 1;
  e = cudaMemcpyAsync(a.flags - 1, a.flags - 1 + nfl, sizeof(int) * nfl, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  // column exponents and integer sums are neighbours: one clear
  e = cudaMemsetAsync(a.ints, 0, (size_t)((char*)a.z - (char*)a.ints), st);
  if (e != cudaSuccess) return e;
  BG au = a;
  au.units = units;
  bg_prologue_kernel<<<(unsigned)p.n_pro, 256, 0, st>>>(au);
  if (p.n_mod) bg_rows_kernel<<<(unsigned)p.n_pro, 256, 0, st>>>(au);
  au.units = units + p.n_pro;
  bg_gram_kernel<<<(unsigned)p.n_gram, kThreads, smem, st>>>(au);
  bg_chol_kernel<<<nb, kCholThreads, csmem, st>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const unsigned tiles = (unsigned)((p.maxNb + 7) / 8), el = (unsigned)std::max(1, p.maxNb * p.maxNb / 2048);
  enum { A = 0, V = 1, A2 = 2, T0 = 3, T1 = 4, T2 = 5, T3 = 6, T4 = 7 };
  // items count in the grid's y, or twice in its z, which end at 65,535
  constexpr unsigned kItems = 32767;
  for (unsigned f0 = 0; f0 < nb; f0 += kItems) {
    const unsigned ni = std::min(kItems, nb - f0);
    BG ac = a;
    ac.bins += f0;
    auto stage = [&]() {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)p.maxpairs, ni);
      cfg.blockDim = dim3(kZThreads);
      cfg.dynamicSmemBytes = jsmem;
      cfg.stream = st;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)p.maxpairs;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      return cudaLaunchKernelEx(&cfg, bg_jacobi32_kernel, ac);
    };
    auto gemm = [&](const ZGemm& x, bool vt_only = false) {
      bg_gemm_kernel<<<dim3(tiles, tiles, ni), 128, 0, st>>>(ac, ZGemms{{x, x}, 1, vt_only});
    };
    auto gemm2 = [&](const ZGemm& x, const ZGemm& y) {
      bg_gemm_kernel<<<dim3(tiles, tiles, 2 * ni), 128, 0, st>>>(ac, ZGemms{{x, y}, 2, false});
    };
    if ((e = stage()) != cudaSuccess) return e;
    bg_widen_kernel<<<dim3(el, ni), 256, 0, st>>>(ac);
    gemm(ZGemm{1, T0, T0, -1, T1, 1.0, 0.0});                 // V^H V
    gemm(ZGemm{0, T0, T1, T0, T3, -0.5, 1.5});                // V <- 1.5 V - 0.5 V V^H V
    gemm(ZGemm{0, A, T3, -1, A2, 1.0, 0.0});                  // A = R^H V
    bg_init_kernel<<<dim3(el, ni), 256, 0, st>>>(ac);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = stage()) != cudaSuccess) return e;
    bg_widen_kernel<<<dim3(el, ni), 256, 0, st>>>(ac);
    gemm2(ZGemm{0, T3, T0, -1, V, 1.0, 0.0}, ZGemm{0, A2, T0, -1, A, 1.0, 0.0});
    for (int it = 0; it < 2; ++it) {
      const int Ai = it ? A2 : A, Vi = it ? T3 : V, Ao = it ? A : A2, Vo = it ? V : T3;
      gemm2(ZGemm{1, Ai, Ai, -1, T0, 1.0, 0.0}, ZGemm{1, Vi, Vi, -1, T1, 1.0, 0.0});
      bg_check_kernel<<<dim3((unsigned)((p.maxNb + 7) / 8), ni), 256, 0, st>>>(ac, it);
      bg_angles_kernel<<<dim3(el, ni), 256, 0, st>>>(ac);
      gemm(ZGemm{0, T4, T2, T1, T0, 0.5, 1.0});               // Q
      gemm2(ZGemm{0, Ai, T0, -1, Ao, 1.0, 0.0}, ZGemm{0, Vi, T0, -1, Vo, 1.0, 0.0});
    }
    bg_finalize_kernel<<<ni, 256, 0, st>>>(ac);
    if (p.any_vt) {
      for (int it = 0; it < 2; ++it) {
        gemm(ZGemm{1, it ? T3 : T0, it ? T3 : T0, -1, T1, 1.0, 0.0}, true);      // W^T W
        bg_ortho_kernel<<<dim3(el, ni), 256, 0, st>>>(ac);
        gemm(ZGemm{0, it ? T3 : T0, T2, -1, it ? T0 : T3, 1.0, 0.0}, true);
      }
      bg_vt_kernel<<<ni, 256, 0, st>>>(ac);
    }
  }
  if (p.n_mod) {
    au.units = units + p.n_pro + p.n_gram;
    bg_modes_kernel<<<(unsigned)p.n_mod, kThreads, msmem, st>>>(au);
  }
  return cudaGetLastError();
}

}  // namespace pylom
