// gram.h -- the Gram route of the POD: R from an exact Gram matrix, modes by
// a direct product (gram.cu, modes_direct.cu).
#pragma once
#include "kernels.h"

namespace pylom {

struct GramState {
  WsHeader* hdr;
  int64_t N, M, ldy;      // ldy: rows of Y rounded up to 8, the padding rows hold zeros
  void* Y;                // N x M weighted centred matrix, binary64 or binary32
  bool f32;
  int* colE;              // M: largest exponent field of each column
  long long* G;           // 5 x M x M: integer sums, group g weighs 2^(32 g)
  double* Lh;             // M x M double-double triangle (high parts)
  double* Ll;             // (low parts)
  double* Th;             // kNBC x M: current row panel before division (high)
  double* Tl;
  unsigned char* Cd;      // digit planes of the modes product's coefficients
  int* Ce;                // exponent field of each coefficient column
  int64_t rmax;
};

size_t gram_bytes(int64_t M, int64_t rmax);
void gram_carve(GramState& g, char* base, int64_t M, int64_t rmax);

// Y = sqrt(w) (X - mean), the column exponents and the means; then the exact
// Gram matrix, its Cholesky factor in double-double arithmetic and R (M x M,
// upper triangular, zeros below, ld M).
cudaError_t launch_gram_r(const GramState& g, const void* X, int64_t ldx, int xtype, const double* w,
                          int remove_mean, double* mean, double* R, cudaStream_t st, cudaEvent_t mid);

// U (N x r) = Y C: C (M x rmax, ld M) given, or (C null) V_r S_r^-1 from VT and S.
// r is read from hdr->r.  U is binary64, or binary32 for a binary32 Y.
cudaError_t launch_modes_direct(const GramState& g, const double* C, const double* S, const double* VT, int64_t ldvt,
                                const double* w, int physical, void* U, int64_t ldu, int64_t* r_out,
                                cudaStream_t st, cudaEvent_t mid);

}  // namespace pylom
