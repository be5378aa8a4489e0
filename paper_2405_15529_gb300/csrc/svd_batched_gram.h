// svd_batched_gram.h -- the Gram route of the batched SVDs (mixed precision):
// its tables in the plan's workspace and its launch sequence.
#pragma once
#include <vector>

#include "kernels.h"

namespace pylom {

// One item (a complex64 bin or a real window) of the Gram route.
struct GramBin {
  const float* Y;        // real matrix, rows x Nb: a bin's X with re / im interleaved, or a window's binary32 copy
  int64_t rows, ldy;
  int Nb, Mb, k, cplx;   // Mb: Nb rounded up to 32
  int64_t colE;          // ints: Nb exponent fields, then 64 of the coefficients
  int64_t g;             // long long: 3 Nb^2 (Re), 3 Nb^2 (Im)
  int64_t z;             // double2: kBinMats matrices Nb x Nb
  int64_t f;             // float2: A32 (Nb x Mb), V32 (Mb x Mb)
  int64_t c;             // bytes: digit planes of the coefficients
  int64_t r;             // uint16: shifts of the rows (twice the points)
  int64_t d;             // doubles: Nb (norms) + Nb (angle flags)
  int64_t s_off;         // offset in the packed S
  int flag;              // index in the flag array (the item's number in the plan)
  // outputs
  float2* U;             // bins
  float* Ur;             // windows
  int64_t ldu;
  double* VT;
  int64_t ldvt;
  // windows: input
  const void* Xr;
  int64_t ldx;
  int kind, remove_mean, physical, pad_;
  const double* w;
  double* mean;
};
constexpr int kBinMats = 8;   // A, V, A2, T0, T1, T2, T3, T4

// A piece of an item's work: kind of tile, its column block, a row range (bin < 0: none).
struct GramUnit {
  int bin, mode, J, pad_;
  int64_t q0, q1;
};

struct BatchedGramPlan {
  std::vector<int> items;          // item numbers of the plan that take this route
  std::vector<GramBin> bins;       // offsets by the plan, pointers by bind
  std::vector<GramUnit> pro, gram, mod;   // prologue, Gram and modes units
  int nitems = 0, maxNb = 0, maxpairs = 0;
  bool any_vt = false;             // some bind has asked for a window's right vectors
  // A plan may be bound to several workspaces, to bins in one and windows in
  // another: run launches what holds for all of them.  Units wanted, and the
  // lengths of the three lists (filled up with empty units).
  int64_t want = 0, n_pro = 0, n_gram = 0, n_mod = 0;
  size_t off_bins = 0, off_units = 0, off_i = 0, off_g = 0, off_z = 0, off_f = 0, off_c = 0, off_d = 0, off_r = 0, off_flags = 0;
  int64_t n_i = 0, n_g = 0, n_z = 0, n_f = 0, n_c = 0, n_d = 0, n_r = 0;
};

// Adds an item (N x Nb, kmodes modes) and, at the end, the sections to the workspace.
void batched_gram_add(BatchedGramPlan& p, int item, int64_t N, int64_t Nb, int64_t k, int64_t s_off);
size_t batched_gram_layout(BatchedGramPlan& p, size_t off, int nitems, int sms);
// Row units once the items' row counts are known (after bind).
void batched_gram_units(BatchedGramPlan& p);
cudaError_t batched_gram_upload(const BatchedGramPlan& p, char* ws, const int* forced, int nitems, cudaStream_t st);
// Runs the route; afterwards flags[i] != 0 marks the items that the
// Householder route has to do (given at upload, or found to need it).
cudaError_t batched_gram_run(const BatchedGramPlan& p, char* ws, WsHeader* hdr, double* S, cudaStream_t st);

}  // namespace pylom
