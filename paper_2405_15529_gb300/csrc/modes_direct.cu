// modes_direct.cu -- U = Y C for a tall Y (N x M, the weighted centred
// snapshot matrix) and a small C (M x r): the modes U = Y V_r S_r^-1 of the
// Gram route, which equal Q U_r (Eq. svdqr3 of pyLOM, arXiv 2405.15529), and
// the DMD modes.  Both factors are cut into digits (digits.cuh) and
// multiplied without rounding on the tcgen05 tensor cores; digit products
// below the level of a binary64 (binary32) rounding of the sum are left out.
// Measured (4,194,304 x 256, r = 43): top-down pass + reflectors 7.3 + 209 ms
// in binary64, 5.2 + 16.7 ms mixed; here 8.4 and 7.5 ms.
//
// A block takes tiles of 128 rows x 64 columns of U.  16 warps cut 32
// columns of the tile's rows of Y into digit planes per stage (a thread
// takes 8 columns of one row: coalesced loads, one conflict-free 16-byte
// store per digit), a bulk copy brings the stage's planes of C, which a
// small kernel has laid out in shared-memory order, and one thread issues
// the MMAs; every 128 columns of Y the accumulators go to 64-bit integers in
// registers, and at the tile's end those become U.
#include "digits.cuh"
#include "gram.h"

namespace pylom {

// Digit planes of C' = diag(2^(E_j - bias)) C, one block per column of C;
// planes of column tile kt and stage js at ((kt * stages + js) * S) kPlaneB
// bytes.  C null: C = V_r S_r^-1.
template <typename TY>
__global__ void __launch_bounds__(128) coef_digits_kernel(GramState g, const double* C, const double* S,
                                                         const double* VT, int64_t ldvt) {
  constexpr int SD = Dig<TY>::S;
  __shared__ int s_e;
  const int64_t k = blockIdx.x, r = g.hdr->r, M = g.M;
  if (k >= (r + 63) / 64 * 64) return;
  const int64_t stages = (M + kStK - 1) / kStK;
  if (threadIdx.x == 0) s_e = kMinField64;
  __syncthreads();
  const double sk = (!C && k < r) ? S[k] : 1.0;
  auto value = [&](int64_t j) {
    if (j >= M || k >= r) return 0.0;
    const double c = C ? C[j + k * M] : VT[k + j * ldvt] / sk;
    return scalbn(c, g.colE[j] - fix_bias<TY>());
  };
  int e = kMinField64;
  for (int64_t j = threadIdx.x; j < M; j += blockDim.x) {
    const int ej = exp_field(value(j));
    e = ej > e ? ej : e;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_e, e);
  __syncthreads();
  e = s_e;
  if (threadIdx.x == 0) g.Ce[k] = e;
  for (int64_t j0 = (int64_t)threadIdx.x * 8; j0 < stages * kStK; j0 += (int64_t)blockDim.x * 8) {
    uint2 w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      int64_t v = to_fixed(value(j0 + i), e);
      // binary32 Y: the coefficients keep 38 of the 62 bits (rounded)
      if (SD == 5) v = (v + (1ll << 23)) >> 24;
      w[i] = bias_digits(v);
    }
    const int64_t js = j0 / kStK;
    unsigned char* dst = g.Cd + (((k / 64) * stages + js) * SD) * (int64_t)kPlaneB + ((k & 63) >> 3) * kPlaneSbo +
                         ((j0 % kStK) >> 3) * 128 + (k & 7) * 16;
    store_digits<SD>(w, dst, kPlaneB);
  }
}

template <typename TY>
__global__ void __launch_bounds__(kDigThreads, 1) modes_direct_kernel(GramState g, const double* S0, const double* w,
                                                                     int physical, TY* U, int64_t ldu,
                                                                     int64_t* r_out) {
  constexpr int S = Dig<TY>::S, NST = Dig<TY>::NST, LB = Dig<TY>::LBM;
  extern __shared__ __align__(1024) unsigned char gsm[];
  __shared__ __align__(8) DigitBarriers<NST> bar;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t N = g.N, M = g.M, r = g.hdr->r;
  // a zero matrix keeps all modes (there is no energy to share): unit vectors
  const bool zero = S0 && S0[0] == 0.0;
  if (blockIdx.x == 0 && tid == 0 && r_out) *r_out = r;
  const int64_t ktiles = (r + 63) / 64, tiles = (N + 127) / 128 * ktiles;
  const int stages = (int)((M + kStK - 1) / kStK), m32 = (int)M;
  const uint32_t kt32 = (uint32_t)ktiles;
  const TY* Y = (const TY*)g.Y;
  const int rl = tid & 127, kh = (tid >> 7) & 1; // row of the tile, half of the stage's columns
  const uint32_t offA = (uint32_t)((rl >> 3) * kPlaneSbo + (rl & 7) * 16);
  const int mine = blockIdx.x < tiles ? (int)((tiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
  auto fill = [&](int t, int js, unsigned char* st) {
    const uint32_t tile = blockIdx.x + t * gridDim.x;
    const int64_t row = (int64_t)(tile / kt32) * 128 + rl;
    const bool rin = row < N;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int kg = 2 * kh + h;
      const int c0 = js * kStK + kg * 8;
      const TY* p = Y + row + c0 * g.ldy;
      TY y[8];
      int E[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const bool in = c0 + i < m32;
        y[i] = (in && rin) ? __ldg(p + i * g.ldy) : (TY)0;
        E[i] = in ? __ldg(g.colE + c0 + i) : 128;
      }
      put_digits(y, E, st + offA + kg * 128, kPlaneA);
    }
  };
  auto bsrc = [&](int t, int js) {
    const uint32_t tile = blockIdx.x + t * gridDim.x;
    return g.Cd + ((int64_t)(tile % kt32) * stages + js) * (S * kPlaneB);
  };
  auto store = [&](int t, const int64_t (&acc0)[16], const int64_t (&acc1)[16]) {
    // the tile's rows of U: lanes hold consecutive rows
    const uint32_t tile = blockIdx.x + t * gridDim.x;
    const int64_t row = (int64_t)(tile / kt32) * 128 + (warp & 3) * 32 + lane;
    const int k0 = (int)(tile % kt32) * 64 + (warp >> 2) * 16;
    const double iw = (physical && w && row < N) ? 1.0 / sqrt(w[row]) : 1.0;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int k = k0 + c;
      if (k >= r) break;     // uniform over the warp
      if (row < N) {
        const int pk = 8 * LB + __ldg(g.Ce + k) - fix_bias<double>() + (S == 5 ? 24 : 0);
        double v = __fma_rn((double)acc1[c], 4294967296.0, (double)acc0[c]);
        v = (pk > -900 && pk < 900) ? v * __hiloint2double((pk + 1023) << 20, 0) : scalbn(v, pk);
        if (zero) v = row == k ? 1.0 : 0.0;
        if (physical && w) v *= iw;
        U[row + k * ldu] = (TY)v;
      }
    }
  };
  product_pipeline<S, NST, LB>(bar, gsm, mine, stages, g.hdr, fill, bsrc, store);
}

template <typename TY>
static cudaError_t run(const GramState& g, const double* C, const double* S, const double* VT, int64_t ldvt,
                       const double* w, int physical, void* U, int64_t ldu, int64_t* r_out, int sms,
                       cudaStream_t st, cudaEvent_t mid) {
  constexpr size_t smem = (size_t)Dig<TY>::NST * Dig<TY>::S * (kPlaneA + kPlaneB);
  cudaError_t e = ensure_dyn_smem((const void*)modes_direct_kernel<TY>, smem);
  if (e != cudaSuccess) return e;
  const int64_t kt = (g.rmax + 63) / 64;
  coef_digits_kernel<TY><<<(unsigned)(kt * 64), 128, 0, st>>>(g, C, S, VT, ldvt);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (mid && (e = cudaEventRecord(mid, st)) != cudaSuccess) return e;
  int64_t grid = (g.N + 127) / 128 * kt;
  if (grid > sms) grid = sms;
  modes_direct_kernel<TY><<<(unsigned)grid, kDigThreads, smem, st>>>(g, C ? nullptr : S, w, physical, (TY*)U, ldu, r_out);
  return cudaGetLastError();
}

cudaError_t launch_modes_direct(const GramState& g, const double* C, const double* S, const double* VT, int64_t ldvt,
                                const double* w, int physical, void* U, int64_t ldu, int64_t* r_out,
                                cudaStream_t st, cudaEvent_t mid) {
  cudaError_t e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  return g.f32 ? run<float>(g, C, S, VT, ldvt, w, physical, U, ldu, r_out, sms, st, mid)
               : run<double>(g, C, S, VT, ldvt, w, physical, U, ldu, r_out, sms, st, mid);
}

}  // namespace pylom
