// pod_backward_gram.cu -- the adjoint of the POD path (pod_backward.cu) for a
// forward that left Y unfactored: no reflectors, two products with Y.
//
// With Y = U S V^T, W = Y^T dU (so that u_i^T dU_j = v_i^T W_j / s_i) and
// r kept modes, the cotangent of Y is
//   dY = Y V K V^T + dU S_r^-1 V_r^T,
//   K_ij = F_ij (v_i^T W_j / s_j [j < r] - v_j^T W_i / s_i [i < r]) + F_ij (G2_ij - G2_ji)   (i != j),
//   K_ii = (dS_i - v_i^T W_i / s_i^2 [i < r] s_i / s_i) / s_i,
//   F_ij = 1 / (s_j^2 - s_i^2), G2 = V^T dV,
// which is pod_backward.cu's formula with u_i = Y v_i / s_i put in: the
// projection of dU on the left-out modes (i >= r) and the rest of space join
// in one term, and the factors s_i of the left-out modes cancel, so small and
// zero singular values among them do no harm.  Only the kept s_j, and those
// s_i whose own cotangent dS_i is not zero, are inverted; where one of them
// is too small (or the forward factored Y) the device leaves the call to the
// Householder form behind it.
//
// W and the product run on the tensor cores by digits (gram.cu,
// modes_direct.cu), without rounding; the M x M algebra is binary64.
//
// Measured (262,144 x 64 binary64, r = 20, one training step): 21.7 ms with
// leaves, tree, top-down and bottom-up passes, 2.9 ms here.
#include "digits.cuh"
#include "gram.h"

namespace pylom {

constexpr double kInvertLevel = 1e-4;

// redo = 1: the Householder form has to do this call
__global__ void bg_route_kernel(const WsHeader* fwd, WsHeader* hdr, const double* S, const double* dS, int64_t M,
                                int64_t r, double level) {
  bool bad = false;
  for (int64_t i = threadIdx.x; i < M; i += blockDim.x) {
    const bool inverted = i < r || (dS && dS[i] != 0.0);
    bad = bad || (inverted && !(S[i] >= level * S[0] && S[i] > 0.0));
  }
  if (threadIdx.x == 0) bad = bad || fwd->gram_y == 0;
  if (__syncthreads_or(bad) && threadIdx.x == 0) hdr->gram_redo = 1;
}

// Z = W^(-1/2) dU (physical modes) or dU, padding rows zero, and its column exponents
template <typename TY>
__global__ void __launch_bounds__(256) bg_load_kernel(const double* dU, int64_t lddu, const double* w, int physical, TY* Z,
                                                     int64_t ldz, int64_t N, int* zE, const unsigned* unless) {
  if (*unless) return;
  const int64_t c = blockIdx.y;
  int e = 0;
  for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < ldz; n += (int64_t)gridDim.x * blockDim.x) {
    double v = 0.0;
    if (n < N) {
      v = dU[n + c * lddu];
      if (physical && w) v /= sqrt(w[n]);
    }
    const TY z = (TY)v;
    Z[n + c * ldz] = z;
    const int ez = exp_field(z);
    e = ez > e ? ez : e;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0 && e > 0) atomicMax(zE + c, e);
}

// K from A1 = V^T W (M x r, ld M) and A2 = V^T dV (M x M, nullable)
__global__ void bg_core_kernel(const double* A1, const double* A2, const double* S, const double* dS, double* K,
                               int64_t M, int64_t r, const unsigned* unless) {
  if (*unless) return;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < M * M;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % M, j = idx / M;
    const double si = S[i], sj = S[j];
    double k = 0.0;
    if (i == j) {
      if (dS && dS[i] != 0.0) k = dS[i] / si;
      if (i < r) k -= A1[i + i * M] / si / si / si;
    } else {
      const double den = (sj - si) * (sj + si);
      if (den != 0.0) {
        if (j < r) k += A1[i + j * M] / sj;
        if (i < r) k -= A1[j + i * M] / si;
        if (A2) k += A2[i + j * M] - A2[j + i * M];
        k /= den;
      } else if (j < r) {
        k = -A1[i + j * M] / (si * si) / sj;   // equal values: no coupling, the projection stays
      }
    }
    K[idx] = k;
  }
}

struct BgLayout {
  void* Z;         // N x r (ld y_ld(N)), the working type
  int* zE;         // r
  uint16_t* zS;    // N: shifts of the rows of Z
  long long* G;    // 5 M r
  double *W, *A1, *A2, *K, *T, *C, *D;
  unsigned char* Cd;
  int* Ce;
};

static size_t planes_only(int64_t M, int64_t r) {
  return product_planes_bytes(M, r, M) - align256(sizeof(int) * (size_t)((M + 63) / 64) * 64);
}

size_t pod_backward_gram_bytes(int64_t N, int64_t M, int64_t r) {
  const int64_t r1 = r > 0 ? r : 1;
  return align256(sizeof(int) * (size_t)r1) + row_shift_bytes(N) +
         align256(sizeof(long long) * (size_t)5 * M * r1) + 3 * align256(sizeof(double) * (size_t)M * r1) +
         4 * align256(sizeof(double) * (size_t)M * M) + product_planes_bytes(M, r, M);
}

static BgLayout carve(char* p, void* Z, int64_t N, int64_t M, int64_t r) {
  const int64_t r1 = r > 0 ? r : 1;
  BgLayout L;
  const size_t mr = align256(sizeof(double) * (size_t)M * r1), mm = align256(sizeof(double) * (size_t)M * M);
  L.Z = Z;
  L.zE = (int*)p;          p += align256(sizeof(int) * (size_t)r1);
  L.zS = (uint16_t*)p;     p += row_shift_bytes(N);
  L.G = (long long*)p;     p += align256(sizeof(long long) * (size_t)5 * M * r1);
  L.W = (double*)p;        p += mr;
  L.A1 = (double*)p;       p += mr;
  L.D = (double*)p;        p += mr;
  L.A2 = (double*)p;       p += mm;
  L.K = (double*)p;        p += mm;
  L.T = (double*)p;        p += mm;
  L.C = (double*)p;        p += mm;
  L.Cd = (unsigned char*)p; p += planes_only(M, r);
  L.Ce = (int*)p;
  return L;
}

// dY (N x M, ld N, binary64 or binary32 as the forward's Y) where hdr->gram_redo stays 0.
cudaError_t launch_pod_backward_gram(const GramState& f, WsHeader* hdr, const double* S, const double* VT, int64_t ldvt,
                                     const double* dU, int64_t lddu, const double* dS, const double* dVT,
                                     int64_t lddvt, const double* w, int physical, int64_t r, void* Z, void* dY, char* base,
                                     cudaStream_t st) {
  const int64_t N = f.N, M = f.M;
  BgLayout L = carve(base, Z, N, M, r);
  const unsigned* redo = &hdr->gram_redo;
  if (!dU) r = 0;
  bg_route_kernel<<<1, 256, 0, st>>>(f.hdr, hdr, S, dS, M, r, f.f32 ? 0.1 * kInvertLevel : kInvertLevel);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ProductArgs p{};
  if (r > 0) {
    if ((e = cudaMemsetAsync(L.zE, 0, sizeof(int) * (size_t)r, st)) != cudaSuccess) return e;
    const int64_t ldz = y_ld(N);
    const dim3 grid((unsigned)(ldz > (1 << 18) ? 64 : (ldz + 4095) / 4096), (unsigned)r);
    if (f.f32) bg_load_kernel<float><<<grid, 256, 0, st>>>(dU, lddu, w, physical, (float*)L.Z, ldz, N, L.zE, redo);
    else bg_load_kernel<double><<<grid, 256, 0, st>>>(dU, lddu, w, physical, (double*)L.Z, ldz, N, L.zE, redo);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_row_scale(L.Z, f.f32, ldz, r, L.zE, L.zS, redo, st)) != cudaSuccess) return e;
    if ((e = launch_cross(f, L.Z, ldz, r, L.zE, L.zS, L.G, L.W, redo, hdr, st)) != cudaSuccess) return e;
    e = launch_bw_gemm(0, 0, M, r, M, 1.0, VT, ldvt, L.W, M, 0.0, L.A1, M, redo, st);            // V^T W
    if (e != cudaSuccess) return e;
    if ((e = launch_bw_scale_rows(VT, ldvt, S, L.D, r, M, redo, st)) != cudaSuccess) return e;    // S_r^-1 V_r^T
    p.Z = L.Z;
    p.ldz = ldz;
    p.NZ = r;
    p.zE = L.zE;
    p.zS = L.zS;
    p.D = L.D;
    p.ldd = r;
  }
  if (dVT && (e = launch_bw_gemm(0, 1, M, M, M, 1.0, VT, ldvt, dVT, lddvt, 0.0, L.A2, M, redo, st)) != cudaSuccess)
    return e;
  bg_core_kernel<<<256, 256, 0, st>>>(L.A1, dVT ? L.A2 : nullptr, S, dS, L.K, M, r, redo);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = launch_bw_gemm(0, 0, M, M, M, 1.0, L.K, M, VT, ldvt, 0.0, L.T, M, redo, st);
  if (e == cudaSuccess) e = launch_bw_gemm(1, 0, M, M, M, 1.0, VT, ldvt, L.T, M, 0.0, L.C, M, redo, st);
  if (e != cudaSuccess) return e;
  p.Y = f.Y;
  p.ldy = f.ldy;
  p.N = N;
  p.M = M;
  p.colE = f.colE;
  p.rowS = f.rowS;
  p.C = L.C;
  p.ldc = M;
  p.cols = p.cols_max = M;
  p.Cd = L.Cd;
  p.Ce = L.Ce;
  p.unless = redo;
  p.hdr = hdr;
  return launch_product(p, f.f32, dY, N, hdr, st);
}

}  // namespace pylom
