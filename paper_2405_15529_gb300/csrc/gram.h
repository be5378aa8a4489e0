// gram.h -- the Gram route of the POD: R from an exact Gram matrix, modes by
// a direct product (gram.cu, modes_direct.cu).
#pragma once
#include <cuda.h>

#include "kernels.h"

namespace pylom {

// tsqr_mixed.cu: tensor map of a column-major matrix in boxes of box_rows x box_cols; what a box has past it reads zeros
cudaError_t tensor_map_2d(CUtensorMap* map, CUtensorMapDataType type, void* base, int64_t rows, int64_t cols,
                          int64_t ld_bytes, int box_rows, int box_cols, CUtensorMapSwizzle swizzle);

struct GramState {
  WsHeader* hdr;
  int64_t N, M, ldy;      // ldy: rows of Y rounded up to 8, the padding rows hold zeros
  void* Y;                // N x M weighted centred matrix: binary32, or binary64 cut to fixed point (row_scale_kernel)
  bool f32;
  int* colE;              // M: largest exponent field of each column
  uint16_t* rowS;         // N, rounded up to 128: shift of each row (row_scale_kernel)
  long long* G;           // 5 x M x M: integer sums, group g weighs 2^(32 g)
  double* Lh;             // M x M double-double triangle (high parts)
  double* Ll;             // (low parts)
  double* Th;             // two row panels before division (high parts), kNBC x M each
  double* Tl;             // (low parts), then M pivots
  unsigned char* Cd;      // digit planes of the modes product's coefficients
  int* Ce;                // exponent field of each coefficient column
  int64_t rmax;
};

// U = [Y Z] [C; D]: a second left factor Z (N x NZ, nullable) beside g.Y, the
// coefficients given as doubles (C: M x cols, D: NZ x cols) or, C null, V_r
// S_r^-1 from VT and S.  cols < 0: hdr->r columns.  Cd, Ce: digit planes and
// exponents of the coefficients (product_planes_bytes).
struct ProductArgs {
  const void* Y;
  int64_t ldy, N, M;
  const int* colE;
  const uint16_t* rowS;
  const void* Z;
  int64_t ldz, NZ;
  const int* zE;
  const uint16_t* zS;
  const double *C, *D, *S, *VT;
  const double* T;          // nullable: C - V T instead of C where ortho_rank is not 0 (cols x cols, upper, ld cols_max)
  int64_t ldc, ldd, ldvt;
  int64_t cols, cols_max;
  unsigned char* Cd;
  int* Ce;
  const unsigned* unless;   // nullable: nothing to do when *unless is not 0
  const WsHeader* hdr;
};

#ifdef __CUDACC__
// Kept modes whose coefficients are corrected (launch_ortho): all or, where the
// smallest kept value is near the largest, none.
constexpr double kOrthoRatio = 16.0;
__device__ __forceinline__ int64_t ortho_rank(const WsHeader* hdr, const double* S) {
  const int64_t r = hdr->r;
  return r > 0 && S[r - 1] > 0.0 && !(S[r - 1] * kOrthoRatio >= S[0]) ? r : 0;
}
#endif
// The triangle T with which the modes Y (C - V T), C = V_r S_r^-1, are
// orthonormal to binary64 rounding (binary64 Y); uses the integer sums up.
cudaError_t launch_ortho(const GramState& g, const double* S, const double* VT, int64_t ldvt, const unsigned* unless,
                         const double** T, cudaStream_t st);

size_t row_shift_bytes(int64_t N);
size_t gram_bytes(int64_t N, int64_t M, int64_t rmax);
void gram_carve(GramState& g, char* base, int64_t M, int64_t rmax);

// Y = sqrt(w) (X - mean), the column exponents and the means; then the exact
// Gram matrix, its Cholesky factor in double-double arithmetic and R (M x M,
// upper triangular, zeros below, ld M).
cudaError_t launch_gram_r(const GramState& g, const void* X, int64_t ldx, int xtype, const double* w,
                          int remove_mean, double* mean, double* R, cudaStream_t st, cudaEvent_t mid);

// U (N x r) = Y C: C (M x rmax, ld M) given, or (C null) V_r S_r^-1 from VT and S.
// r is read from hdr->r.  U is binary64, or binary32 for a binary32 Y.  unless
// (nullable): nothing is done when *unless is not 0.
cudaError_t launch_modes_direct(const GramState& g, const double* C, const double* S, const double* VT, int64_t ldvt,
                                const double* w, int physical, void* U, int64_t ldu, int64_t* r_out,
                                const unsigned* unless, cudaStream_t st, cudaEvent_t mid);

// Shifts of the rows of Y (rows of zeros up to ldy); binary64 columns -> fixed-point
// words in place.  And Y of a forward back to binary64 where *redo is set.
cudaError_t launch_row_scale(void* Y, bool f32, int64_t ldy, int64_t cols, const int* colE, uint16_t* rowS,
                             const unsigned* unless, cudaStream_t st);
cudaError_t launch_unpack(const GramState& g, double* Y, const unsigned* redo, cudaStream_t st);
// W = Y^T Z (M x NZ, ld M) from the same integer products; Z as Y.  G: 5 M NZ integers.
cudaError_t launch_cross(const GramState& g, const void* Z, int64_t ldz, int64_t NZ, const int* zE, const uint16_t* zS,
                         long long* G, double* W, const unsigned* unless, WsHeader* hdr, cudaStream_t st);
// The product above into U (binary32 if f32, else binary64; ld ldu).
size_t product_planes_bytes(int64_t M, int64_t NZ, int64_t cols);
cudaError_t launch_product(const ProductArgs& p, bool f32, void* U, int64_t ldu, WsHeader* hdr, cudaStream_t st);

// The adjoint without reflectors (pod_backward_gram.cu); `f` the forward's
// state.  hdr->gram_redo = 1 afterwards: nothing was done.
size_t pod_backward_gram_bytes(int64_t N, int64_t M, int64_t r);
// Z: room for y_ld(N) max(r, 1) doubles.
cudaError_t launch_pod_backward_gram(const GramState& f, WsHeader* hdr, const double* S, const double* VT, int64_t ldvt,
                                     const double* dU, int64_t lddu, const double* dS, const double* dVT,
                                     int64_t lddvt, const double* w, int physical, int64_t r, void* Z, void* dY, char* base,
                                     cudaStream_t st);
// pod_backward.cu: C = alpha op(A) op(B) + beta C, and C = diag(1 / S) VT (rows of them), unless *unless
cudaError_t launch_bw_gemm(int ta, int tb, int64_t m, int64_t n, int64_t k, double alpha, const double* A, int64_t lda,
                           const double* B, int64_t ldb, double beta, double* C, int64_t ldc, const unsigned* unless,
                           cudaStream_t st);
cudaError_t launch_bw_scale_rows(const double* VT, int64_t ldvt, const double* S, double* C, int64_t rows, int64_t M,
                                 const unsigned* unless, cudaStream_t st);
// pod_backward.cu: dX = W^(1/2) dY, minus row means, where *redo is 0
cudaError_t launch_bw_finalize_gram(const void* dY, bool f32, const double* w, int remove_mean, void* dX, int64_t lddx,
                                    int dxtype, int64_t N, int64_t M, const unsigned* redo, cudaStream_t st);

// Whether the kept values are large enough for the direct product (hdr->r,
// S known): else hdr->gram_redo = 1 and hdr->gram_y = 0, and the Householder
// route on `ts` (ts.run_if = &hdr->gram_redo) gives the modes.
cudaError_t launch_gram_check(const GramState& g, const double* S, cudaStream_t st);

}  // namespace pylom
