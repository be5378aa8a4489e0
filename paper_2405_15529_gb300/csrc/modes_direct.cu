// modes_direct.cu -- U = Y C for a tall Y (N x M, the weighted centred
// snapshot matrix) and a small C (M x r): the modes U = Y V_r S_r^-1 of the
// Gram route, which equal Q U_r (Eq. svdqr3 of pyLOM, arXiv 2405.15529), and
// the DMD modes.  Both factors are cut into digits (digits.cuh) and
// multiplied without rounding on the tcgen05 tensor cores; digit products
// below the level of a binary64 (binary32) rounding of the sum are left out.
// Measured (4,194,304 x 256, r = 43): top-down pass + reflectors 7.3 + 209 ms
// in binary64, 5.2 + 16.7 ms mixed; here 7.4 and 5.9 ms.
//
// A block takes tiles of 128 rows x 64 (32) columns of U (digits.cuh: two
// shapes).  The warps cut 16 columns of the tile's rows of Y into digit planes
// per stage (a thread takes 8 columns of one row: coalesced copies into its own
// ring in shared memory, one conflict-free 16-byte store per digit), a bulk
// copy brings the stage's planes of C, which a small kernel has laid out in
// shared-memory order, and one thread issues the MMAs; every 128 columns of Y
// the accumulators go to 64-bit integers in registers, and at the tile's end
// those become U, after the next tile's first MMAs have been issued.  The sums
// are made binary64 (binary32) by integer operations: 262,144 x 100 mixed 287
// us with binary64 ones, 234 with both changes.
#include "digits.cuh"
#include "gram.h"

namespace pylom {

__device__ __forceinline__ int64_t product_cols(const ProductArgs& p) { return p.cols >= 0 ? p.cols : (int64_t)p.hdr->r; }
// stages of the two left factors: each starts a stage of its own
__host__ __device__ __forceinline__ int product_stages(int64_t n) { return (int)((n + kStK - 1) / kStK); }

// Digit planes of the coefficients times their rows' scales 2^(E - bias),
// one block per column; planes of column tile kt and stage js at
// ((kt * stages + js) * S) kPlaneB bytes.
template <typename TY, int G>
__global__ void __launch_bounds__(128) coef_digits_kernel(ProductArgs p) {
  constexpr int SD = Dig<TY>::S, T = Shape<G>::TILE, kPlaneB = Shape<G>::PLANEB;
  __shared__ int s_e;
  if (p.unless && *p.unless) return;
  const int64_t k = blockIdx.x, r = product_cols(p);
  if (k >= (r + T - 1) / T * T) return;
  const int s1 = product_stages(p.M), stages = s1 + product_stages(p.NZ);
  if (threadIdx.x == 0) s_e = kMinField64;
  __syncthreads();
  const double sk = (!p.C && k < r) ? p.S[k] : 1.0;
  const double* tri = p.T && k < r && ortho_rank(p.hdr, p.S) ? p.T + k * p.cols_max : nullptr;
  auto value = [&](int64_t j) {
    if (k >= r) return 0.0;
    if (j < (int64_t)s1 * kStK) {
      if (j >= p.M) return 0.0;
      if (p.colE[j] == max_field<TY>()) return quiet_nan();
      return scalbn(p.C ? p.C[j + k * p.ldc] : p.VT[k + j * p.ldvt] / sk, p.colE[j] - fix_bias<TY>());
    }
    j -= (int64_t)s1 * kStK;
    if (j >= p.NZ) return 0.0;
    if (p.zE[j] == max_field<TY>()) return quiet_nan();
    return scalbn(p.D[j + k * p.ldd], p.zE[j] - fix_bias<TY>());
  };
  int e = kMinField64;
  for (int64_t j = threadIdx.x; j < (int64_t)stages * kStK; j += blockDim.x) {
    const int ej = exp_field(value(j));
    e = ej > e ? ej : e;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_e, e);
  __syncthreads();
  e = s_e;
  if (threadIdx.x == 0) p.Ce[k] = e;
  for (int64_t j0 = (int64_t)threadIdx.x * 8; j0 < (int64_t)stages * kStK; j0 += (int64_t)blockDim.x * 8) {
    uint2 w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      int64_t v = to_fixed(value(j0 + i), e);
      const int64_t j = j0 + i;
      if (tri && j < p.M) {
        double d = 0.0;
        for (int64_t c = 0; c <= k; ++c) d = fma(-p.VT[c + j * p.ldvt], tri[c], d);
        v += to_fixed(scalbn(d, p.colE[j] - fix_bias<TY>()), e);
      }
      // binary32 left factors: the coefficients keep 38 of the 62 bits (rounded)
      if (SD == 5) v = (v + (1ll << 23)) >> 24;
      w[i] = bias_digits(v);
    }
    unsigned char* dst = p.Cd + (((k / T) * stages + j0 / kStK) * SD) * (int64_t)kPlaneB + ((k % T) >> 3) * kPlaneSbo +
                         ((j0 % kStK) >> 3) * 128 + (k & 7) * 16;
    store_digits<SD>(w, dst, kPlaneB);
  }
}

template <typename TY, int G>
__global__ void __launch_bounds__(Shape<G>::THREADS, Shape<G>::BLOCKS) modes_direct_kernel(ProductArgs p, const double* S0, const double* w,
                                                                     int physical, TY* U, int64_t ldu,
                                                                     int64_t* r_out, WsHeader* hdr) {
  constexpr int S = Dig<TY>::S, NST = Dig<TY>::template NST<G>, LB = Dig<TY>::LBM, AHEAD = Dig<TY>::template AHEAD<G>;
  constexpr int T = Shape<G>::TILE, kPlaneB = Shape<G>::PLANEB;
  typedef typename Cell<TY>::type Cl;
  extern __shared__ __align__(1024) unsigned char gsm[];
  __shared__ __align__(8) DigitBarriers<NST, G> bar;
  if (p.unless && *p.unless) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t N = p.N, r = product_cols(p);
  // a zero matrix keeps all modes (there is no energy to share): unit vectors
  const bool zero = S0 && S0[0] == 0.0;
  if (blockIdx.x == 0 && tid == 0 && r_out) *r_out = r;
  const int64_t ktiles = (r + T - 1) / T, tiles = (N + 127) / 128 * ktiles;
  const int s1 = product_stages(p.M), stages = s1 + product_stages(p.NZ);
  const uint32_t kt32 = (uint32_t)ktiles;
  const int rl = tid & 127, kh = (tid >> 7) & 1; // row of the tile, half of the stage's columns
  const uint32_t offA = (uint32_t)((rl >> 3) * kPlaneSbo + (rl & 7) * 16);
  const int mine = blockIdx.x < tiles ? (int)((tiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
  // element i of this thread in slot q of its ring: ring[(q 8 + i) 256]
  Cl* ring = (Cl*)(gsm + NST * S * (kPlaneA + kPlaneB)) + (tid >> 8) * (AHEAD * 8 * 256) + (tid & 255);
  // shift of this thread's row of tile t: of Y, and of Z in the upper half
  auto shifts = [&](int t) {
    const int64_t row = (int64_t)((blockIdx.x + t * gridDim.x) / kt32) * 128 + rl;
    if (row >= N) return 0u;
    const uint32_t a = __ldg(p.rowS + row);
    return p.Z ? a | (uint32_t)__ldg(p.zS + row) << 16 : a | a << 16;
  };
  auto joint = [&](uint32_t s) { return (int)min(s & 0xffffu, s >> 16); };
  uint32_t s_now = 0, s_next = 0;
  int s_tile = -2;
  auto load = [&](int t, int js, int q) {
    const uint32_t tile = blockIdx.x + t * gridDim.x;
    const int64_t row = (int64_t)(tile / kt32) * 128 + rl;
    const bool second = js >= s1;
    const int64_t ld = second ? p.ldz : p.ldy;
    const int c0 = (second ? js - s1 : js) * kStK + kh * 8, m32 = (int)(second ? p.NZ : p.M);
    const Cl* src = (const Cl*)(second ? p.Z : p.Y) + row + c0 * ld;
    if (row < N) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (c0 + i < m32) async_copy<(int)sizeof(Cl)>(ring + (q * 8 + i) * 256, src + i * ld);
    }
  };
  auto fill = [&](int t, int js, int q, unsigned char* st) {
    const uint32_t tile = blockIdx.x + t * gridDim.x;
    const bool rin = (int64_t)(tile / kt32) * 128 + rl < N, second = js >= s1;
    const int* ex = second ? p.zE : p.colE;
    const int c0 = (second ? js - s1 : js) * kStK + kh * 8, m32 = (int)(second ? p.NZ : p.M);
    // the shifts of the next tile's row are on their way while this one is done
    if ((S == 5 || p.Z) && t != s_tile) {
      s_now = t == s_tile + 1 ? s_next : shifts(t);
      s_tile = t;
      if (t + 1 < mine) s_next = shifts(t + 1);
    }
    Cl y[8];
    int E[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool in = c0 + i < m32;
      y[i] = in && rin ? ring[(q * 8 + i) * 256] : zero_cell<Cl>();
      E[i] = (S == 5 && in) ? __ldg(ex + c0 + i) - joint(s_now) : 128;     // (words carry their scale)
    }
    if constexpr (S == 8) {
      // words of Y and of Z at the scale that both have room for
      const uint32_t d = (second ? s_now >> 16 : s_now & 0xffffu) - joint(s_now);
      if (__any_sync(0xffffffffu, d != 0)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = shift_word(y[i], d);
      }
    }
    put_digits(y, E, st + offA + kh * 128, kPlaneA);
  };
  auto bsrc = [&](int t, int js) {
    const uint32_t tile = blockIdx.x + t * gridDim.x;
    return p.Cd + ((int64_t)(tile % kt32) * stages + js) * (S * kPlaneB);
  };
  auto store = [&](int t, const int64_t (&acc0)[16], const int64_t (&acc1)[16]) {
    // the tile's rows of U: lanes hold consecutive rows
    const uint32_t tile = blockIdx.x + t * gridDim.x;
    const int64_t row = (int64_t)(tile / kt32) * 128 + (warp & 3) * 32 + lane;
    const int k0 = (int)(tile % kt32) * T + (warp >> 2) * 16;
    const double iw = (physical && w && row < N) ? 1.0 / sqrt(w[row]) : 1.0;
    if (k0 >= r) return;
    const int rs = joint(shifts(t));
    const int ce = lane < 16 && k0 + lane < r ? __ldg(p.Ce + k0 + lane) : 0;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int k = k0 + c;
      const int cc = __shfl_sync(0xffffffffu, ce, c);
      const int pk = 8 * LB + cc - fix_bias<double>() + (S == 5 ? 24 : 0) - rs;
      if (k < r && row < N) {
        TY v;
        if (zero) v = (TY)(row == k ? iw : 0.0);
        else if (cc == kMaxField64) v = (TY)quiet_nan();      // a coefficient, or a column of Y, is not finite
        else if (physical && w) v = (TY)(from_sums(acc0[c], acc1[c], pk, 0.0) * iw);
        else v = from_sums(acc0[c], acc1[c], pk, (TY)0);
        U[row + k * ldu] = v;
      }
    }
  };
  product_pipeline<S, NST, LB, AHEAD, G>(bar, gsm, mine, stages, hdr, load, fill, bsrc, store);
}

// Smallest kept value, relative to the largest, for which Y V_r S_r^-1 is
// taken: its rounding grows by sigma_1 / sigma_r.
constexpr double kKeptLevel64 = 1e-4, kKeptLevel32 = 1e-5;

__global__ void gram_check_kernel(WsHeader* hdr, const double* S, double level) {
  const long long r = hdr->r;
  if (r >= 1 && S[0] > 0.0 && !(S[r - 1] >= level * S[0])) {
    hdr->gram_redo = 1;
    hdr->gram_y = 0;
  }
}

cudaError_t launch_gram_check(const GramState& g, const double* S, cudaStream_t st) {
  gram_check_kernel<<<1, 1, 0, st>>>(g.hdr, S, g.f32 ? kKeptLevel32 : kKeptLevel64);
  return cudaGetLastError();
}

template <typename TY, int G>
static cudaError_t run_shape(const ProductArgs& p, const double* S0, const double* w, int physical, void* U, int64_t ldu,
                             int64_t* r_out, WsHeader* hdr, cudaStream_t st, cudaEvent_t mid) {
  constexpr int T = Shape<G>::TILE, threads = Shape<G>::THREADS;
  constexpr size_t smem = (size_t)Dig<TY>::template NST<G> * Dig<TY>::S * (kPlaneA + Shape<G>::PLANEB) +
                          (size_t)Dig<TY>::template AHEAD<G> * 8 * threads * sizeof(TY);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = ensure_dyn_smem((const void*)modes_direct_kernel<TY, G>, smem)) != cudaSuccess) return e;
  const int64_t kt = (p.cols_max + T - 1) / T;
  coef_digits_kernel<TY, G><<<(unsigned)(kt * T), 128, 0, st>>>(p);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (mid && (e = cudaEventRecord(mid, st)) != cudaSuccess) return e;
  int64_t grid = (p.N + 127) / 128 * kt;
  if (grid > Shape<G>::BLOCKS * sms) grid = Shape<G>::BLOCKS * sms;
  modes_direct_kernel<TY, G><<<(unsigned)grid, threads, smem, st>>>(p, S0, w, physical, (TY*)U, ldu, r_out, hdr);
  return cudaGetLastError();
}

// Short sums (up to 64 columns of Y) in two blocks an SM: 65,537 x 63, r = 42
// 40 us against 70; 262,144 x 100 mixed 336 against 234, 1,048,576 x 128
// 1360 against 1040.
template <typename TY>
static cudaError_t run(const ProductArgs& p, const double* S0, const double* w, int physical, void* U, int64_t ldu,
                       int64_t* r_out, WsHeader* hdr, cudaStream_t st, cudaEvent_t mid) {
  return p.M + p.NZ <= 64 ? run_shape<TY, 1>(p, S0, w, physical, U, ldu, r_out, hdr, st, mid)
                          : run_shape<TY, 2>(p, S0, w, physical, U, ldu, r_out, hdr, st, mid);
}

size_t product_planes_bytes(int64_t M, int64_t NZ, int64_t cols) {
  const int64_t kt = (cols + 63) / 64;       // (64 columns hold two tiles of the narrower shape)
  return align256((size_t)kt * (product_stages(M) + product_stages(NZ)) * 8 * Shape<2>::PLANEB) +
         align256(sizeof(int) * (size_t)kt * 64);
}

cudaError_t launch_product(const ProductArgs& p, bool f32, void* U, int64_t ldu, WsHeader* hdr, cudaStream_t st) {
  return f32 ? run<float>(p, nullptr, nullptr, 0, U, ldu, nullptr, hdr, st, nullptr)
             : run<double>(p, nullptr, nullptr, 0, U, ldu, nullptr, hdr, st, nullptr);
}

cudaError_t launch_modes_direct(const GramState& g, const double* C, const double* S, const double* VT, int64_t ldvt,
                                const double* w, int physical, void* U, int64_t ldu, int64_t* r_out,
                                const unsigned* unless, cudaStream_t st, cudaEvent_t mid) {
  ProductArgs p{};
  p.unless = unless;
  p.Y = g.Y;
  p.ldy = g.ldy;
  p.N = g.N;
  p.M = g.M;
  p.colE = g.colE;
  p.rowS = g.rowS;
  p.C = C;
  p.ldc = g.M;
  p.S = S;
  p.VT = VT;
  p.ldvt = ldvt;
  p.cols = -1;
  p.cols_max = g.rmax;
  p.Cd = g.Cd;
  p.Ce = g.Ce;
  p.hdr = g.hdr;
  const double* S0 = C ? nullptr : S;
  if (!C && !g.f32) {
    const cudaError_t e = launch_ortho(g, S, VT, ldvt, unless, &p.T, st);
    if (e != cudaSuccess) return e;
  }
  return g.f32 ? run<float>(p, S0, w, physical, U, ldu, r_out, g.hdr, st, mid)
               : run<double>(p, S0, w, physical, U, ldu, r_out, g.hdr, st, mid);
}

}  // namespace pylom
