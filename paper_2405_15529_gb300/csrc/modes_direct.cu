// modes_direct.cu -- U = Y C for a tall Y (N x M, the weighted centred
// snapshot matrix) and a small C (M x r): the modes U = Y V_r S_r^-1 of the
// Gram route, which equal Q U_r (Eq. svdqr3 of pyLOM, arXiv 2405.15529), and
// the DMD modes.  Both factors are cut into digits (digits.cuh) and
// multiplied without rounding on the tcgen05 tensor cores; digit products
// below the level of a binary64 (binary32) rounding of the sum are left out.
// Measured (4,194,304 x 256, r = 43): top-down pass + reflectors 7.3 + 209 ms
// in binary64, 5.2 + 16.7 ms mixed; here 11.3 and 7.8 ms.
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

constexpr int kMdThreads = 512;

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
  if (threadIdx.x == 0) s_e = 1;
  __syncthreads();
  const double sk = (!C && k < r) ? S[k] : 1.0;
  auto value = [&](int64_t j) {
    if (j >= M || k >= r) return 0.0;
    const double c = C ? C[j + k * M] : VT[k + j * ldvt] / sk;
    return scalbn(c, g.colE[j] - fix_bias<TY>());
  };
  int e = 1;
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
    uint64_t w[8];
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

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               :: "r"(tc05::smem_u32(dst)), "l"((uint64_t)__cvta_generic_to_global(src)), "r"(bytes),
                  "r"(tc05::smem_u32(mbar))
               : "memory");
}

template <typename TY>
__global__ void __launch_bounds__(kMdThreads, 1) modes_direct_kernel(GramState g, const double* S0, const double* w,
                                                                    int physical, TY* U, int64_t ldu, int64_t* r_out) {
  constexpr int S = Dig<TY>::S, NST = Dig<TY>::NST, LB = Dig<TY>::LBM;
  constexpr int kStage = S * (kPlaneA + kPlaneB);
  extern __shared__ __align__(1024) unsigned char gsm[];
  __shared__ __align__(8) uint64_t full[NST], empty[NST], dfull, dempty, fin;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t N = g.N, M = g.M, r = g.hdr->r;
  // a zero matrix keeps all modes (there is no energy to share): unit vectors
  const bool zero = S0 && S0[0] == 0.0;
  if (blockIdx.x == 0 && tid == 0 && r_out) *r_out = r;
  const int64_t ktiles = (r + 63) / 64, tiles = (N + 127) / 128 * ktiles;
  const int64_t stages = (M + kStK - 1) / kStK, sums = (stages + kStagesPerSum - 1) / kStagesPerSum;
  if (tid == 0) {
    for (int b = 0; b < NST; ++b) {
      tc05::mbar_init(full + b, kMdThreads / 32 + 1);
      tc05::mbar_init(empty + b, 1);
    }
    tc05::mbar_init(&dfull, 1);
    tc05::mbar_init(&dempty, kMdThreads / 32);
    tc05::mbar_init(&fin, 1);
  }
  if (warp == 0) tc05::tmem_alloc(&tmem_base, 512);
  tc05::fence_before();
  __syncthreads();
  tc05::fence_after();
  const uint32_t tmem = tmem_base;
  bool ok = true;
  const TY* Y = (const TY*)g.Y;
  const int rl = tid & 127, kg = tid >> 7;       // row of the tile, group of 8 columns of the stage
  const uint32_t offA = (uint32_t)((rl >> 3) * kPlaneSbo + kg * 128 + (rl & 7) * 16);
  const int qd = warp & 3, cp = warp >> 2;
  const uint32_t taddr = tmem + ((uint32_t)(qd * 32) << 16) + cp * 16;
  const int64_t mine = blockIdx.x < tiles ? (tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  // this block's stages as one sequence: tile by tile, sum by sum
  const int64_t total = mine * stages, nsum = mine * sums;
  int64_t acc0[16], acc1[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) acc0[c] = acc1[c] = 0;
  int64_t issued = 0, issued_sum = 0, drained = 0;
  // position of the stage being filled: tile, stage within the tile
  int64_t tile = blockIdx.x, js = 0, begun = 0;    // begun: sums whose first stage has been filled
  int ahead = 0;                                   // stages filled of sums that have not been drained up to
  int64_t is_js = 0;
  int64_t dr_tile = blockIdx.x, dr_sum = 0;
  for (int64_t j = 0; j <= total; ++j) {
    const int b = (int)(j % NST);
    bool opens = false;
    if (j < total) {
      if (j >= NST) {
        ok = __all_sync(0xffffffffu, mbar_wait_fast(empty + b, (uint32_t)((j / NST - 1) & 1)));
        if (!ok) break;
      }
      unsigned char* st = gsm + b * kStage;
      if (tid == 0) {
        tc05::mbar_arrive_expect_tx(full + b, S * kPlaneB);
        bulk_load(st + S * kPlaneA, g.Cd + (((tile % ktiles) * stages + js) * S) * (int64_t)kPlaneB, S * kPlaneB,
                  full + b);
      }
      const int64_t row = tile / ktiles * 128 + rl, c0 = js * kStK + kg * 8;
      uint64_t wv[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int64_t c = c0 + i;
        const bool in = c < M && row < N;
        const TY y = in ? __ldg(Y + row + c * g.ldy) : (TY)0;
        const int E = c < M ? __ldg(g.colE + c) : 1;
        wv[i] = bias_digits(to_fixed(y, E));
      }
      store_digits<S>(wv, st + offA, kPlaneA);
      tc05::fence_smem_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(full + b);
      opens = js % kStagesPerSum == 0;
      if (opens) {
        ++begun;
        ahead = 0;
      }
      ++ahead;
      if (++js == stages) {
        js = 0;
        tile += gridDim.x;
      }
    }
    // read the sums that are complete: all of them at the end; before that,
    // the one before the sum being filled, as soon as NST stages (or the
    // whole sum) are filled ahead of it
    const bool whole = j < total && (js == 0 || js % kStagesPerSum == 0);
    int64_t upto = j == total ? nsum : (ahead >= NST || whole) ? begun - 1 : drained;
    while (drained < upto) {
      ok = __all_sync(0xffffffffu, mbar_wait_fast(&dfull, (uint32_t)(drained & 1)));
      if (!ok) break;
      tc05::fence_after();
      drain_slots(taddr, kSlots, acc0, acc1);
      tc05::fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&dempty);
      ++drained;
      if (++dr_sum == sums) {
        // the tile's rows of U: lanes hold consecutive rows
        const int64_t row = dr_tile / ktiles * 128 + qd * 32 + lane;
        const int64_t k0 = dr_tile % ktiles * 64 + cp * 16;
        const double iw = (physical && w && row < N) ? 1.0 / sqrt(w[row]) : 1.0;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int64_t k = k0 + c;
          if (k < r && row < N) {
            const int pk = 8 * LB + __ldg(g.Ce + k) - fix_bias<double>() + (S == 5 ? 24 : 0);
            double v = __fma_rn((double)acc1[c], 4294967296.0, (double)acc0[c]);
            v = (pk > -900 && pk < 900) ? v * __hiloint2double((pk + 1023) << 20, 0) : scalbn(v, pk);
            if (zero) v = row == k ? 1.0 : 0.0;
            if (physical && w) v *= iw;
            U[row + k * ldu] = (TY)v;
          }
          acc0[c] = acc1[c] = 0;
        }
        dr_sum = 0;
        dr_tile += gridDim.x;
      }
    }
    if (!ok) break;
    // MMAs of filled stages, up to the first sum whose accumulators are still unread
    if (warp == kMdThreads / 32 - 1) {
      if (lane == 0) {
        while (issued <= j && issued < total) {
          const bool first = is_js % kStagesPerSum == 0;
          if (first && issued_sum > drained) break;      // this warp has not read the sum before
          const int ib = (int)(issued % NST);
          ok = mbar_wait_fast(full + ib, (uint32_t)((issued / NST) & 1));
          if (ok && first && issued_sum > 0) ok = mbar_wait_fast(&dempty, (uint32_t)((issued_sum - 1) & 1));
          if (!ok) break;
          if (first) ++issued_sum;
          tc05::fence_after();
          const uint32_t sa = tc05::smem_u32(gsm) + ib * kStage;
          issue_stage<S, LB>(tmem, tc05::desc(sa, 128, kPlaneSbo), tc05::desc(sa + S * kPlaneA, 128, kPlaneSbo),
                             kPlaneB, first);
          tc05::commit(empty + ib);
          ++issued;
          if (++is_js == stages) is_js = 0;
          if (is_js % kStagesPerSum == 0) tc05::commit(&dfull);
        }
      }
      ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
      if (!ok) break;
    }
  }
  if (warp == kMdThreads / 32 - 1 && lane == 0) {
    tc05::commit(&fin);
    if (!mbar_wait_fast(&fin, 0)) ok = false;
  }
  // bulk copies of stages that were never consumed (after a timeout) land
  // before the block ends
  if (!ok && tid == 0)
    for (int b = 0; b < NST; ++b) tc05::mbar_wait(full + b, 0, 1000000ull);
  if (!ok) raise_status(g.hdr, PYLOM_ERR_TIMEOUT);
  tc05::fence_before();
  __syncthreads();
  if (warp == 0) tc05::tmem_dealloc(tmem, 512);
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
  modes_direct_kernel<TY><<<(unsigned)grid, kMdThreads, smem, st>>>(g, C ? nullptr : S, w, physical, (TY*)U, ldu, r_out);
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
