// frame.cu -- U_R for the Q of a Householder TSQR behind the Gram route (POD
// of pyLOM, arXiv 2405.15529, Eqs. svdqr1-svdqr3).
//
// A call that the device takes from the Gram route to the Householder route
// has S and V already, from the Cholesky factor of the exact Gram matrix.  The
// Householder R of the same Y belongs to another Q: the two differ by row
// signs where the columns are independent, by more where one depends on
// earlier ones (a zero snapshot, one written twice).  So U_R comes from R V =
// U_R S with this R: the orthogonal factor of a QR of R V, whose columns are
// orthogonal to rounding and fall in norm.  It is u_i to eps s_1 / s_i, and an
// orthonormal completion where s_i is zero.  (A second SVD, of this R, was 50
// launches that return at once when nothing falls back, 150 us a call; this
// is two.)
#include "kernels.h"

namespace pylom {

// B = R V / s_1 (scaled: squares stay in range)
__global__ void __launch_bounds__(256) frame_product_kernel(TsqrState s, const double* VT, int64_t ldvt, const double* S, double* B) {
  if (passed_over(s) || already_factored(s)) return;
  const int64_t M = s.M;
  const double sc = S[0] > 0.0 ? 1.0 / S[0] : 1.0;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < M * M;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % M, j = idx / M;
    double a = 0.0;
    for (int64_t k = i; k < M; ++k) a = fma(s.Rs[i + k * M], VT[j + k * ldvt], a);
    B[idx] = a * sc;
  }
}

// Householder QR of B (M x M), one column and one grid barrier a step: every
// block forms the column's reflector, a warp a later column applies it.  F:
// reflectors (unit diagonal not stored), tau.  Then a warp a column of Q.
// Bound by the latency of a step's barrier and column (about 5 us a column); only calls that fall back come here.
constexpr int kFrameThreads = 256;
__global__ void __launch_bounds__(kFrameThreads) frame_kernel(TsqrState s, const double* UR, double* B, double* F,
                                                                 double* tau, double* Q) {
  extern __shared__ double v[];          // M
  __shared__ double sred[kFrameThreads / 32], sout[1];
  const int64_t M = s.M;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t warp = ((int64_t)blockIdx.x * kFrameThreads + tid) >> 5, nwarps = (int64_t)gridDim.x * kFrameThreads / 32;
  if (passed_over(s)) return;
  if (already_factored(s)) {
    for (int64_t idx = (int64_t)blockIdx.x * kFrameThreads + tid; idx < M * M; idx += (int64_t)gridDim.x * kFrameThreads)
      Q[idx] = UR[idx];
    return;
  }
  for (int64_t j = 0; j < M; ++j) {
    double a[1] = {0.0};
    for (int64_t i = j + tid; i < M; i += kFrameThreads) {
      const double x = ldcg(B + i + j * M);
      v[i] = x;
      if (i > j) a[0] = fma(x, x, a[0]);
    }
    block_sum<1>(a, sred, sout);
    const double sigma = sout[0], alpha = v[j];
    const bool act = sigma > 0.0;
    const double nrm = sqrt(fma(alpha, alpha, sigma)), beta = !act ? alpha : alpha >= 0.0 ? -nrm : nrm;
    const double t = act ? (beta - alpha) / beta : 0.0;
    __syncthreads();
    for (int64_t i = j + tid; i < M; i += kFrameThreads) {
      v[i] = i == j ? 1.0 : act ? v[i] / (alpha - beta) : 0.0;
      if (blockIdx.x == 0) F[i + j * M] = i == j ? beta : v[i];
    }
    if (blockIdx.x == 0 && tid == 0) tau[j] = t;
    __syncthreads();
    if (act)
      for (int64_t k = warp; k < M; k += nwarps) {
        if (k <= j) continue;
        double d = 0.0;
        for (int64_t i = j + lane; i < M; i += 32) d = fma(v[i], ldcg(B + i + k * M), d);
        d = warp_sum(d) * t;
        for (int64_t i = j + lane; i < M; i += 32) __stcg(B + i + k * M, ldcg(B + i + k * M) - d * v[i]);
      }
    if (!grid_barrier(s.hdr, gridDim.x)) return;
  }
  // column c: H_0 .. H_c e_c, signed so that the R factor's diagonal is not negative
  for (int64_t c = warp; c < M; c += nwarps) {
    double* q = Q + c * M;               // (a lane reads only what it wrote)
    const double one = ldcg(F + c + c * M) < 0.0 ? -1.0 : 1.0;
    for (int64_t i = lane; i < M; i += 32) q[i] = i == c ? one : 0.0;
    for (int64_t j = c; j >= 0; --j) {
      const double t = ldcg(tau + j);
      if (t == 0.0) continue;
      double d = 0.0;
      for (int64_t i = lane; i < M; i += 32)
        if (i >= j) d = fma(i == j ? 1.0 : ldcg(F + i + j * M), q[i], d);
      d = warp_sum(d) * t;
      for (int64_t i = lane; i < M; i += 32)
        if (i >= j) q[i] -= d * (i == j ? 1.0 : ldcg(F + i + j * M));
    }
  }
}

size_t frame_doubles(int64_t M) { return (size_t)(2 * M * M + M); }

cudaError_t launch_frame(const TsqrState& s, const double* S, const double* VT, int64_t ldvt, const double* UR,
                         double* scratch, double* Q, cudaStream_t st) {
  double *B = scratch, *F = B + s.M * s.M, *tau = F + s.M * s.M;
  int dev = 0, sms = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const size_t smem = sizeof(double) * (size_t)s.M;      // at most 32 KB
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, frame_kernel, kFrameThreads, smem);
  if (e != cudaSuccess) return e;
  if (per < 1) return cudaErrorCooperativeLaunchTooLarge;
  frame_product_kernel<<<s.M <= 64 ? 16 : 304, 256, 0, st>>>(s, VT, ldvt, S, B);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int64_t want = (s.M + kFrameThreads / 32 - 1) / (kFrameThreads / 32);
  TsqrState fs = s;
  void* args[] = {&fs, &UR, &B, &F, &tau, &Q};
  return cudaLaunchCooperativeKernel((const void*)frame_kernel, dim3((unsigned)(want < sms ? want : sms)),
                                     dim3(kFrameThreads), args, smem, st);
}

}  // namespace pylom
