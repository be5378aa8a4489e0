// svd_jacobi32.cu -- preconditioning of the small SVD (Eq. svdqr2 of pyLOM,
// arXiv 2405.15529) so that the binary64 one-sided Jacobi of svd_jacobi.cu
// has (nearly) nothing left to rotate.
//
// A binary64 Jacobi sweep is M - 1 grid barriers and 5.5 M^3 binary64
// instructions, of which this part issues two per clock and SM; ten or more
// sweeps made the small SVD the largest part of every POD below a few
// hundred thousand rows.  Here:
//   1. binary32 block one-sided Jacobi on A32 = fl32(R^T) (blocks of 16
//      columns; a step's 32 columns are orthogonalised through their 32 x 32
//      Gram matrix in shared memory, then the accumulated rotation is
//      applied), giving V32; V = V32 made orthogonal (one Newton-Schulz
//      step) and A = R^T V in binary64;
//   2. the same again on fl32(A): each column now has its own binary32
//      scale, so columns of small singular value, which fl32(R^T) buried
//      under the rounding of the large ones, become orthogonal too;
//   3. two, four or six binary64 steps of simultaneous rotations: with
//      G = A^T A, E = V^T V - I and K_ij the Jacobi angle of pair (i, j)
//      (antisymmetric), Q = I + K + K^2/2 - E/2 and A <- A Q, V <- V Q: all
//      cosines square (Davies and Modi, "A direct method for completing
//      eigenproblem solutions on a parallel computer", 1986).  Two columns
//      whose angle is not small (double singular values) get their exact
//      rotation first, and K is formed in the rotated basis.
// Matrix products run on all SMs.  The binary64 sweeps then start from
// (A, V); when every pair already meets their stopping test they return at
// once, else they finish the job: the result is the binary64 SVD either way.
//
// Bound by the latency of the binary32 rounds (a round of 16 rotations is a
// chain of three approximate operations and one block barrier, about 300 ns;
// 7 to 10 sweeps) and, above M = 256, by the binary64 products.  Whole small
// SVD of a field with a decaying spectrum on a floor, ten binary64 sweeps ->
// here: M = 32 2.1 -> 0.25 ms, 64 4.2 -> 0.45, 128 9.6 -> 1.0; with the
// earlier preconditioning (8-column blocks, three binary64 sweeps after it)
// M = 256 13.3 -> 3.5, 700 114 -> 36 ms; singular values within 1.5e-15
// S_max (2e-14 before: fewer rotations).  At M = 700 the binary32 stages take
// 21 ms (23.8 before the next row tile was fetched during the products) and
// the products 14.5 (17.8 before symmetric ones computed half their tiles).
#include "kernels.h"

namespace pylom {

constexpr int kJB = 16;                // columns per block
constexpr int kJW = 2 * kJB;           // columns of a step
constexpr int kJ32Threads = 256;
constexpr int kJRows = 64;             // rows of the staged tile
constexpr int kJ32MaxSweeps = 24;
constexpr int kJClusterMax = 8;        // up to 8 blocks run as one cluster (cheaper barrier)
// words of s.rot32: rotations of each sweep of the two stages, then
constexpr int kJSteps = 6;                       // binary64 steps of simultaneous rotations
constexpr int kJManyColumns = 128;               // from here on all of them
constexpr int kJOpen = 2 * kJ32MaxSweeps;        // kJSteps + 1 words: pairs not converged at each check; then: entries of V^T V off
constexpr int kJWords = kJOpen + kJSteps + 2;

// A32 = A (M x Mp), binary32, zero padding columns; V32 = I.  First A = R^T,
// scaled (R given).
__global__ void jacobi32_init_kernel(SvdState s, double* A, const double* R, int64_t ldr) {
  const int64_t M = s.M, Mb = s.Mb;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const double sc = svd_scale(s);
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < M * Mb; idx += stride) {
    const int64_t i = idx % M, j = idx / M;
    double x = 0.0;
    if (j < M) {
      if (R) A[idx] = sc * R[j + i * ldr];
      x = A[idx];
    }
    s.A32[idx] = (float)x;
  }
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < Mb * Mb; idx += stride)
    s.V32[idx] = (idx % Mb == idx / Mb) ? 1.f : 0.f;
}

// Jacobi rotation of a pair with squared norms al, be and dot product ga
// (identity where |ga| is below the level thr2 of its squared cosine): no
// branches and three approximate operations, since the chain of rounds is
// latency bound (700 ns a round with IEEE square roots behind a branch).
// t = sign(d) 2 ga / (|d| + sqrt(d^2 + 4 ga^2)), d = be - al
__device__ __forceinline__ void rotation(float al, float be, float ga, float thr2, float& c, float& sn) {
  const float d = be - al, g2 = ga + ga;
  float r, q;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaf(d, d, g2 * g2)));
  const float den = fmaxf(fabsf(d) + r, fabsf(g2));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(den));
  const bool act = ga * ga > thr2 * fabsf(al * be);
  const float t = act ? copysignf(1.f, d) * g2 * q : 0.f;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(fmaf(t, t, 1.f)));
  sn = c * t;
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// One binary32 stage.  Blocks follow a round-robin order, a pair of column
// blocks per thread block and step; steps end with a barrier over all
// blocks (of the cluster, or of the grid in a cooperative launch).
template <bool CLUSTER>
__global__ void __launch_bounds__(kJ32Threads) jacobi32_block_kernel(SvdState s, int stage) {
  constexpr int LD = kJW + 4;
  __shared__ __align__(16) float sA[kJRows * LD];
  __shared__ float sG[2][kJW][kJW + 1];
  __shared__ __align__(16) float sJ[kJW][LD];
  __shared__ unsigned char sI[kJW - 1][kJB], sK[kJW - 1][kJB];
  __shared__ unsigned s_rot;
  const int64_t M = s.M, Mb = s.Mb;
  const int tid = threadIdx.x;
  const int64_t nblk = Mb / kJB, npairs = nblk / 2;
  const float tol = 4.f * sqrtf((float)M) * 5.9604645e-8f;   // the rounding level of a dot product
  unsigned* rot = s.rot32 + stage * kJ32MaxSweeps;
  for (int idx = tid; idx < (kJW - 1) * kJB; idx += kJ32Threads) {
    const int round = idx / kJB, p = idx % kJB;
    int a, b;
    if (round < kJB) {                 // across the blocks
      a = p;
      b = kJB + (p + round) % kJB;
    } else {                           // within them: two round-robins of 16 columns
      const int h = p / 8 * kJB, q = p % 8, r = round - kJB;
      a = h + ((q == 0) ? 0 : ((q - 1 + r) % (kJB - 1)) + 1);
      b = h + ((kJB - 2 - q + r) % (kJB - 1)) + 1;
    }
    sI[round][p] = (unsigned char)(a < b ? a : b);
    sK[round][p] = (unsigned char)(a < b ? b : a);
  }
  for (int sweep = 0; sweep < kJ32MaxSweeps; ++sweep) {
    unsigned local_rot = 0;
    const int64_t steps = nblk > 2 ? nblk - 1 : 1;
    for (int64_t step = 0; step < steps; ++step) {
      for (int64_t pr = blockIdx.x; pr < npairs; pr += gridDim.x) {
        const int64_t p = (pr == 0) ? 0 : ((pr - 1 + step) % (nblk - 1)) + 1;
        const int64_t q = ((nblk - 2 - pr + step) % (nblk - 1)) + 1;
        const int64_t bI = p < q ? p : q, bJ = p < q ? q : p;
        auto column = [&](int l) { return (l < kJB ? bI * kJB + l : bJ * kJB + (l - kJB)); };
        // 32 x 32 Gram matrix: 8 x 8 threads of 4 x 4 entries, 4 row slices
        const int ti = (tid & 7) * 4, tj = ((tid >> 3) & 7) * 4, sl = tid >> 6;
        float g[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) g[a][b] = 0.f;
        // (the next row tile is on its way while this one is multiplied)
        constexpr int kLoads = kJRows * kJW / kJ32Threads;
        const int lr = tid % kJRows, lc = tid / kJRows;
        const float* src[kLoads];
        float nx[kLoads];
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
          src[u] = s.A32 + lr + column(lc + u * (kJ32Threads / kJRows)) * M;
          nx[u] = lr < M ? __ldcg(src[u]) : 0.f;
        }
        for (int64_t r0 = 0; r0 < M; r0 += kJRows) {
          __syncthreads();
#pragma unroll
          for (int u = 0; u < kLoads; ++u) sA[lr * LD + lc + u * (kJ32Threads / kJRows)] = nx[u];
          __syncthreads();
#pragma unroll
          for (int u = 0; u < kLoads; ++u) nx[u] = r0 + kJRows + lr < M ? __ldcg(src[u] + r0 + kJRows) : 0.f;
#pragma unroll 4
          for (int r = sl; r < kJRows; r += 4) {
            const float4 x = *(const float4*)(sA + r * LD + ti), y = *(const float4*)(sA + r * LD + tj);
            const float xa[4] = {x.x, x.y, x.z, x.w}, ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
              for (int b = 0; b < 4; ++b) g[a][b] = fmaf(xa[a], ya[b], g[a][b]);
          }
        }
        __syncthreads();
        float* part = sA;
        static_assert(kJW * kJW <= kJRows * LD, "a slice's Gram matrix fits the row tile");
        for (int h = 3; h >= 1; --h) {
          // slices 3, 2, 1 hand their sums to slice 0 in a fixed order
          if (sl == h) {
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
              for (int b = 0; b < 4; ++b) part[(ti + a) * kJW + tj + b] = g[a][b];
          }
          __syncthreads();
          if (sl == 0) {
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
              for (int b = 0; b < 4; ++b) g[a][b] += part[(ti + a) * kJW + tj + b];
          }
          __syncthreads();
        }
        if (tid == 0) s_rot = 0;
        if (sl == 0) {
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) sG[0][ti + a][tj + b] = g[a][b];
        }
        for (int idx = tid; idx < kJW * kJW; idx += kJ32Threads) sJ[idx / kJW][idx % kJW] = idx / kJW == idx % kJW;
        __syncthreads();
        // pairs of this step that are not orthogonal yet
        {
          unsigned n = 0;
          for (int idx = tid; idx < kJW * kJW; idx += kJ32Threads) {
            const int i = idx / kJW, j = idx % kJW;
            if (i < j && sG[0][i][j] * sG[0][i][j] > tol * tol * (sG[0][i][i] * sG[0][j][j])) ++n;
          }
          if (n) atomicAdd(&s_rot, n);
        }
        __syncthreads();
        const unsigned open = s_rot;
        local_rot += open;
        if (open == 0) continue;
        // two-sided rotations on the Gram matrix: the 16 disjoint pairs of a
        // round at once, a thread per 2 x 2 block, each thread forming the
        // two rotations of its block itself (one barrier a round, the matrix
        // double-buffered).  Rounds 0..15 pair the columns of block I with
        // those of block J; the pairs within the blocks (rounds 16..30)
        // follow in the first step of a sweep only.
        const int pb = tid & 15, qb = tid >> 4;
        const int rounds = step == 0 ? kJW - 1 : kJB;
        const float thr2 = 0.0625f * tol * tol;
        int ni = sI[0][pb], nj = sK[0][pb], nk = sI[0][qb], nl = sK[0][qb];
        for (int round = 0; round < rounds; ++round) {
          const float(*G0)[kJW + 1] = sG[round & 1];
          float(*G1)[kJW + 1] = sG[(round & 1) ^ 1];
          const int i = ni, j = nj, k = nk, l = nl;
          const int nr = round + 1 < rounds ? round + 1 : 0;
          ni = sI[nr][pb];
          nj = sK[nr][pb];
          nk = sI[nr][qb];
          nl = sK[nr][qb];
          float cp, sp, cq, sq;
          rotation(G0[i][i], G0[j][j], G0[i][j], thr2, cp, sp);
          rotation(G0[k][k], G0[l][l], G0[k][l], thr2, cq, sq);
          const float a = G0[i][k], b = G0[i][l], c = G0[j][k], d = G0[j][l];
          // rows: [c -s; s c] on (i, j), columns the same on (k, l)
          const float a1 = cp * a - sp * c, c1 = sp * a + cp * c, b1 = cp * b - sp * d, d1 = sp * b + cp * d;
          G1[i][k] = cq * a1 - sq * b1;
          G1[i][l] = sq * a1 + cq * b1;
          G1[j][k] = cq * c1 - sq * d1;
          G1[j][l] = sq * c1 + cq * d1;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int r = qb + 16 * u;      // J's columns i, j of pair pb
            const float x = sJ[r][i], y = sJ[r][j];
            sJ[r][i] = cp * x - sp * y;
            sJ[r][j] = sp * x + cp * y;
          }
          __syncthreads();
        }
        // A32 and V32 columns <- columns J (a thread per row)
        float nv[kJW];
        auto fetch = [&](int64_t row) {
          const float* base = row < M ? s.A32 + row : s.V32 + (row - M);
          const int64_t ld = row < M ? M : Mb;
          if (row < M + Mb) {
#pragma unroll
            for (int l = 0; l < kJW; ++l) nv[l] = __ldcg(base + column(l) * ld);
          }
        };
        fetch(tid);
        for (int64_t row = tid; row < M + Mb; row += kJ32Threads) {
          float* base = row < M ? s.A32 + row : s.V32 + (row - M);
          const int64_t ld = row < M ? M : Mb;
          float v[kJW];
#pragma unroll
          for (int l = 0; l < kJW; ++l) v[l] = nv[l];
          fetch(row + kJ32Threads);
#pragma unroll 1
          for (int l = 0; l < kJW; l += 4) {
            float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int m = 0; m < kJW; ++m) {
              const float4 jv = *(const float4*)&sJ[m][l];
              o[0] = fmaf(v[m], jv.x, o[0]);
              o[1] = fmaf(v[m], jv.y, o[1]);
              o[2] = fmaf(v[m], jv.z, o[2]);
              o[3] = fmaf(v[m], jv.w, o[3]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) __stcg(base + column(l + u) * ld, o[u]);
          }
        }
      }
      __syncthreads();
      if (CLUSTER) cluster_barrier();
      else if (!grid_barrier(s.hdr, gridDim.x)) return;
    }
    if (tid == 0 && local_rot) atomicAdd(rot + sweep, local_rot);
    if (CLUSTER) {
      __threadfence();
      __syncthreads();
      cluster_barrier();
    } else if (!grid_barrier(s.hdr, gridDim.x)) {
      return;
    }
    if (ld_acquire_u32(rot + sweep) == 0) break;
  }
}

// V (Mp x Mp, binary64) = the leading Mp x Mp block of V32.
__global__ void jacobi32_widen_kernel(SvdState s, double* V) {
  const int64_t Mp = s.Mp, Mb = s.Mb;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < Mp * Mp;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % Mp, j = idx / Mp;
    V[idx] = (double)s.V32[i + j * Mb];
  }
}

// C = alpha op(A) B + beta D, binary64 on the FP64 tensor pipe, for the
// small products between the stages (one or two of them in a launch): T x T
// tiles, the K range split over the four warps of a block and summed in a
// fixed order.  `skip` (nullable): nothing to do when *skip is 0.
struct SmallGemm {
  int ta;
  int64_t m, n, k;
  const double* A;
  int64_t lda;
  const double* B;
  int64_t ldb;
  double alpha, beta;
  const double* D;   // ld m
  double* C;         // ld m
  int sym;           // op(A) B is symmetric: tiles on and above the diagonal, and their mirror images
};
struct SmallGemms {
  SmallGemm g[2];
  const unsigned* skip;
};

template <int T>
__global__ void __launch_bounds__(128) small_gemm_kernel(SmallGemms gs) {
  constexpr int U = T / 8;
  __shared__ double part[4][T][T + 1];
  if (gs.skip && *gs.skip == 0) return;
  const SmallGemm& p = gs.g[blockIdx.z];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int64_t i0 = (int64_t)blockIdx.x * T, j0 = (int64_t)blockIdx.y * T;
  if (i0 >= p.m || j0 >= p.n || (p.sym && i0 > j0)) return;
  double acc[U][U][2];
#pragma unroll
  for (int a = 0; a < U; ++a)
#pragma unroll
    for (int b = 0; b < U; ++b) acc[a][b][0] = acc[a][b][1] = 0.0;
  const int64_t nst = (p.k + 3) / 4;
#pragma unroll 4
  for (int64_t st = warp; st < nst; st += 4) {
    const int64_t kk = st * 4 + t;
    double av[U], bv[U];
#pragma unroll
    for (int a = 0; a < U; ++a) {
      const int64_t i = i0 + 8 * a + g, j = j0 + 8 * a + g;
      av[a] = (kk < p.k && i < p.m) ? (p.ta ? __ldg(p.A + kk + i * p.lda) : __ldg(p.A + i + kk * p.lda)) : 0.0;
      bv[a] = (kk < p.k && j < p.n) ? __ldg(p.B + kk + j * p.ldb) : 0.0;
    }
#pragma unroll
    for (int a = 0; a < U; ++a)
#pragma unroll
      for (int b = 0; b < U; ++b) dmma884(acc[a][b][0], acc[a][b][1], av[a], bv[b]);
  }
#pragma unroll
  for (int a = 0; a < U; ++a)
#pragma unroll
    for (int b = 0; b < U; ++b) {
      part[warp][8 * a + g][8 * b + 2 * t] = acc[a][b][0];
      part[warp][8 * a + g][8 * b + 2 * t + 1] = acc[a][b][1];
    }
  __syncthreads();
  for (int idx = threadIdx.x; idx < T * T; idx += 128) {
    const int r = idx % T, c = idx / T;
    const int64_t i = i0 + r, j = j0 + c;
    if (i < p.m && j < p.n) {
      const double v = (part[0][r][c] + part[1][r][c]) + (part[2][r][c] + part[3][r][c]);
      const double x = p.alpha * v + (p.D ? p.beta * p.D[i + j * p.m] : 0.0);
      p.C[i + j * p.m] = x;
      if (p.sym && i0 != j0) p.C[j + i * p.m] = x;
    }
  }
}

static cudaError_t small_gemms(const SmallGemms& gs, int count, cudaStream_t st) {
  int64_t m = gs.g[0].m, n = gs.g[0].n;
  for (int i = 1; i < count; ++i) {
    m = gs.g[i].m > m ? gs.g[i].m : m;
    n = gs.g[i].n > n ? gs.g[i].n : n;
  }
  // 8 x 8 tiles while 16 x 16 ones would leave most SMs idle
  if (m * n * count <= 2 * 144 * 144) {
    const dim3 grid((unsigned)((m + 7) / 8), (unsigned)((n + 7) / 8), (unsigned)count);
    small_gemm_kernel<8><<<grid, 128, 0, st>>>(gs);
  } else {
    const dim3 grid((unsigned)((m + 15) / 16), (unsigned)((n + 15) / 16), (unsigned)count);
    small_gemm_kernel<16><<<grid, 128, 0, st>>>(gs);
  }
  return cudaGetLastError();
}

// Jacobi angle of the pair (i, j) of A's columns from G = A^T A as its
// tangent t: column j gains +t a_i, column i gains -t a_j (antisymmetric).
__device__ __forceinline__ double pair_tangent(double al, double be, double ga) {
  if (ga == 0.0) return 0.0;
  const double zeta = (be - al) / (2.0 * ga);
  return ((zeta >= 0.0) ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
}

// Whether the pair takes part in a step as a small angle t: pairs that are
// converged do only where that is harmless (their angle is noise).
constexpr double kSmallAngle = 0.02;
__device__ __forceinline__ bool small_angle(bool open, double t, double M) {
  return open ? fabs(t) <= kSmallAngle : fabs(t) * M <= 1e-3;
}

// Check `c` on G: counts the pairs that the binary64 sweeps would rotate
// (open[c]), and leaves for each column the partner of its largest angle if
// that is not small (big[j], else -1) and the sum of its small ones.
// With W = V^T V given, entries away from the identity by more than wtol
// are counted in bad.  A warp per column.
__global__ void jacobi_check_kernel(SvdState s, const double* G, const double* W, double wtol, unsigned* bad, int c,
                                    const unsigned* skip) {
  if (skip && *skip == 0) return;
  const int64_t Mp = s.Mp;
  const int lane = threadIdx.x & 31;
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (j >= Mp) return;
  const double tol = (double)s.M * 1.1102230246251565e-16;
  const double be = G[j + j * Mp];
  unsigned n = 0, nw = 0;
  double best = kSmallAngle, sum = 0.0;
  int bi = -1;
  for (int64_t i = lane; i < Mp; i += 32) {
    if (W) nw += !(fabs(W[i + j * Mp] - (i == j ? 1.0 : 0.0)) <= wtol);
    if (i == j) continue;
    const double al = G[i + i * Mp], ga = G[i + j * Mp];
    const bool open = jacobi_open(al, be, ga, tol);
    n += open && i < j;
    const double t = fabs(pair_tangent(al, be, ga));
    if (open && t > best) {
      best = t;
      bi = (int)i;
    } else if (small_angle(open, t, (double)s.M)) {
      sum += t;
    }
  }
  sum = warp_sum(sum);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (oi >= 0 && (bi < 0 || ob > best || (ob == best && oi < bi))) {
      best = ob;
      bi = oi;
    }
  }
  n = __reduce_add_sync(0xffffffffu, n);
  nw = __reduce_add_sync(0xffffffffu, nw);
  if (lane == 0) {
    s.big[j] = bi;
    s.angle_sum[j] = sum;
    if (n) atomicAdd(s.rot32 + kJOpen + c, n);
    if (nw) atomicAdd(bad, nw);
  }
}

// Two columns that are each other's largest angle get their exact rotation
// (close singular values: the angle is anything up to 45 degrees): P is the
// product of these disjoint rotations.  In the rotated basis, G' = P^T G P and
// W' = P^T W P, K = the antisymmetric small angles, L = K - E and B = I + K -
// E / 2 with E = W' - I, so that B + L K / 2 = (I - E / 2)(I + K + K^2 / 2) up
// to E K^2; PL = P L and PB = P B go out, and Q = PB + PL K / 2.  A column
// whose small angles sum to more than `limit` takes none (a crowd of close
// singular values, where they are no small rotation together).
__global__ void jacobi_angles_kernel(SvdState s, const double* G, const double* W, double* K, double* PL,
                                     double* PB, double limit, const unsigned* skip) {
  if (skip && *skip == 0) return;
  const int64_t Mp = s.Mp;
  const double tol = (double)s.M * 1.1102230246251565e-16;
  struct Col {
    int64_t at, b;     // itself, its partner (or itself)
    double c, s, d;    // a' = c a + s a_b; its square
    bool act;
  };
  auto column = [&](int64_t i) {
    Col r{i, i, 1.0, 0.0, G[i + i * Mp], s.angle_sum[i] <= limit};
    const int64_t b = s.big[i];
    if (b >= 0 && s.big[b] == i) {
      const int64_t lo = i < b ? i : b, hi = i < b ? b : i;
      const double ga = G[lo + hi * Mp];
      double t = pair_tangent(G[lo + lo * Mp], G[hi + hi * Mp], ga);
      if (i == hi) t = -t;
      r.b = b;
      r.c = 1.0 / sqrt(1.0 + t * t);
      r.s = -t * r.c;
      r.d -= t * ga;
      r.act = s.angle_sum[i] + s.angle_sum[b] <= limit;
    }
    return r;
  };
  auto rotated = [&](const double* X, const Col& p, const Col& q) {
    double x = X[p.at + q.at * Mp];
    if (p.b != p.at || q.b != q.at)
      x = p.c * (q.c * x + q.s * X[p.at + q.b * Mp]) +
          p.s * (q.c * X[p.b + q.at * Mp] + q.s * X[p.b + q.b * Mp]);
    return x;
  };
  auto angle = [&](const Col& p, const Col& q) {
    if (p.at == q.at || p.b == q.at || !p.act || !q.act) return 0.0;
    const double ga = rotated(G, p, q), t = pair_tangent(p.d, q.d, ga);
    return small_angle(jacobi_open(p.d, q.d, ga, tol), t, (double)s.M) ? t : 0.0;
  };
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < Mp * Mp;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const Col p = column(idx % Mp), q = column(idx / Mp);
    const double one = p.at == q.at ? 1.0 : 0.0, t = angle(p, q), E = rotated(W, p, q) - one;
    double l = t - E, b = one + t - 0.5 * E;
    K[idx] = t;
    if (p.b != p.at) {
      const Col p2 = column(p.b);
      const double one2 = p2.at == q.at ? 1.0 : 0.0, t2 = angle(p2, q), E2 = rotated(W, p2, q) - one2;
      l = p.c * l - p.s * (t2 - E2);
      b = p.c * b - p.s * (one2 + t2 - 0.5 * E2);
    }
    PL[idx] = l;
    PB[idx] = b;
  }
}

__global__ void jacobi_restart_kernel(SvdState s, const double* R, int64_t ldr, const unsigned* bad, unsigned* open) {
  if (*bad == 0) return;
  const int64_t M = s.M, Mp = s.Mp, na = M * Mp, nv = Mp * Mp;
  const double sc = svd_scale(s);
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < na + nv;
       idx += (int64_t)gridDim.x * blockDim.x) {
    if (idx < na) {
      const int64_t i = idx % M, j = idx / M;
      s.A[idx] = (j < M) ? sc * R[j + i * ldr] : 0.0;
    } else {
      const int64_t v = idx - na;
      s.V[v] = (v % Mp == v / Mp) ? 1.0 : 0.0;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *open = 1;
}

size_t jacobi32_extra_bytes(int64_t M) {
  if (M < kJac32MinM) return 0;
  const int64_t Mp = M + (M & 1);
  const int64_t Mb = (M + kJW - 1) / kJW * kJW;
  return 2 * align256(sizeof(float) * (size_t)Mb * Mb) +
         5 * align256(sizeof(double) * (size_t)Mp * Mp) + align256(sizeof(unsigned) * kJWords) +
         align256(sizeof(double) * (size_t)M * Mp) + align256(sizeof(int) * (size_t)Mp) +
         align256(sizeof(double) * (size_t)Mp);
}

void jacobi32_carve(SvdState& s, char* p) {
  const int64_t M = s.M, Mp = s.Mp;
  const size_t sq = align256(sizeof(double) * (size_t)Mp * Mp);
  s.Mb = (M + kJW - 1) / kJW * kJW;
  s.A32 = (float*)p;    p += align256(sizeof(float) * (size_t)s.Mb * s.Mb);
  s.V32 = (float*)p;    p += align256(sizeof(float) * (size_t)s.Mb * s.Mb);
  for (int i = 0; i < 5; ++i) { s.T[i] = (double*)p; p += sq; }
  s.rot32 = (unsigned*)p; p += align256(sizeof(unsigned) * kJWords);
  s.A2 = (double*)p;    p += align256(sizeof(double) * (size_t)M * Mp);
  s.big = (int*)p;      p += align256(sizeof(int) * (size_t)Mp);
  s.angle_sum = (double*)p;
}

static cudaError_t stage32(const SvdState& s, int stage, cudaStream_t st) {
  cudaError_t e;
  const int64_t npairs = s.Mb / kJW;
  SvdState a = s;
  if (npairs <= kJClusterMax) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)npairs);
    cfg.blockDim = dim3(kJ32Threads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)npairs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, jacobi32_block_kernel<true>, a, stage);
  }
  int dev = 0, sms = 0, per = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, jacobi32_block_kernel<false>, kJ32Threads, 0);
  if (e != cudaSuccess) return e;
  if (per < 1) return cudaErrorCooperativeLaunchTooLarge;
  int64_t grid = npairs;
  if (grid > sms) grid = sms;
  void* args[] = {&a, &stage};
  return cudaLaunchCooperativeKernel((const void*)jacobi32_block_kernel<false>, dim3((unsigned)grid),
                                     dim3(kJ32Threads), args, 0, st);
}

// Leaves s.A = R^T V and s.V = V (orthogonal), the starting point of the
// binary64 sweeps; **open_pairs (device) is 0 when nothing is left for them.
cudaError_t launch_jacobi32_precondition(const SvdState& s, const double* R, int64_t ldr, const unsigned** open_pairs,
                                         cudaStream_t st) {
  const int64_t M = s.M, Mp = s.Mp;
  const int gr = M <= 64 ? 16 : M <= 256 ? 128 : 304;
  cudaError_t e = cudaMemsetAsync(s.rot32, 0, sizeof(unsigned) * kJWords, st);
  if (e != cudaSuccess) return e;
  double *T0 = s.T[0], *T1 = s.T[1], *T2 = s.T[2], *T3 = s.T[3], *T4 = s.T[4];
  double* T5 = (double*)s.A32;   // (A32 and V32 are done with when the steps begin)
  unsigned* open = s.rot32 + kJOpen;
  const double wtol = (double)M * 1.1102230246251565e-16 > 1e-14 ? (double)M * 1.1102230246251565e-16 : 1e-14;
  // a product whose left factor op(A) has `m` rows and K = `k` (B then has
  // leading dimension k, C and D m)
  auto mm = [&](int ta, int64_t m, int64_t k, double alpha, const double* A, int64_t lda, const double* B,
                double beta, const double* D, double* C) {
    return SmallGemm{ta, m, Mp, k, A, lda, B, k, alpha, beta, D, C, ta && A == B};
  };
  auto one = [&](const SmallGemm& g, const unsigned* skip = nullptr) {
    if (e == cudaSuccess) e = small_gemms(SmallGemms{{g, g}, skip}, 1, st);
  };
  auto two = [&](const SmallGemm& g, const SmallGemm& h, const unsigned* skip = nullptr) {
    if (e == cudaSuccess) e = small_gemms(SmallGemms{{g, h}, skip}, 2, st);
  };
  jacobi32_init_kernel<<<gr, 256, 0, st>>>(s, s.A, R, ldr);
  if ((e = cudaGetLastError()) != cudaSuccess || (e = stage32(s, 0, st)) != cudaSuccess) return e;
  jacobi32_widen_kernel<<<gr, 256, 0, st>>>(s, T0);
  e = cudaGetLastError();
  one(mm(1, Mp, Mp, 1.0, T0, Mp, T0, 0.0, nullptr, T1));                             // V^T V
  one(mm(0, Mp, Mp, -0.5, T0, Mp, T1, 1.5, T0, T3));                                 // V <- 1.5 V - 0.5 V V^T V
  one(SmallGemm{0, M, Mp, M, s.A, M, T3, Mp, 1.0, 0.0, nullptr, s.A2});              // A = R^T V (rows of V past M meet no row of R)
  if (e != cudaSuccess) return e;
  jacobi32_init_kernel<<<gr, 256, 0, st>>>(s, s.A2, nullptr, 0);
  if ((e = cudaGetLastError()) != cudaSuccess || (e = stage32(s, 1, st)) != cudaSuccess) return e;
  jacobi32_widen_kernel<<<gr, 256, 0, st>>>(s, T0);
  e = cudaGetLastError();
  two(mm(0, Mp, Mp, 1.0, T3, Mp, T0, 0.0, nullptr, s.V), mm(0, M, Mp, 1.0, s.A2, M, T0, 0.0, nullptr, s.A));
  // steps of simultaneous rotations in pairs, (A, V) -> (A2, T3) -> (A, V);
  // each pair begins with a look at G and, from the second on, ends all if
  // no pair is open.  V's departure from orthogonality, 1e-6 at first, is
  // squared by a step, which adds a^4 / 4 for angles that sum to a: the last
  // steps take small angles only.  The first takes up to 0.3: of 700 columns
  // whose 300 smallest singular values lie within 20 % of each other most
  // have angles above 0.05 together, and were left to the sweeps (42 ms).
  constexpr double kLimit[kJSteps] = {0.3, 0.1, 0.1, 0.02, 0.01, 2e-4};
  // (fewer columns hold no such crowd: the last two steps' ten empty launches
  // cost 65,537 x 63 25 of 1,100 us)
  const int steps = M >= kJManyColumns ? kJSteps : 4;
  const unsigned gc = (unsigned)((Mp * 32 + 255) / 256);
  for (int it = 0; it < steps; ++it) {
    const bool fwd = (it & 1) == 0;
    const double *Ai = fwd ? s.A : s.A2, *Vi = fwd ? s.V : T3;
    double *Ao = fwd ? s.A2 : s.A, *Vo = fwd ? T3 : s.V;
    // whether this pair of steps runs, and whether the one before did
    const unsigned* skip = it < 2 ? nullptr : open + (it & ~1);
    const unsigned* look = fwd ? (it < 4 ? nullptr : open + it - 2) : skip;
    two(mm(1, Mp, M, 1.0, Ai, M, Ai, 0.0, nullptr, T0), mm(1, Mp, Mp, 1.0, Vi, Mp, Vi, 0.0, nullptr, T1), look);
    if (e != cudaSuccess) return e;
    jacobi_check_kernel<<<gc, 256, 0, st>>>(s, T0, it >= 2 && fwd ? T1 : nullptr, wtol, open + it, it, look);
    jacobi_angles_kernel<<<gr, 256, 0, st>>>(s, T0, T1, T2, T4, T5, kLimit[it < 2 ? it : it + kJSteps - steps], skip);
    e = cudaGetLastError();
    one(mm(0, Mp, Mp, 0.5, T4, Mp, T2, 1.0, T5, T0), skip);                          // Q
    two(mm(0, M, Mp, 1.0, Ai, M, T0, 0.0, nullptr, Ao), mm(0, Mp, Mp, 1.0, Vi, Mp, T0, 0.0, nullptr, Vo), skip);
  }
  // (after fewer steps the last look stands)
  const unsigned* look = open + steps - 2;
  two(mm(1, Mp, M, 1.0, s.A, M, s.A, 0.0, nullptr, T0), mm(1, Mp, Mp, 1.0, s.V, Mp, s.V, 0.0, nullptr, T1), look);
  if (e != cudaSuccess) return e;
  jacobi_check_kernel<<<gc, 256, 0, st>>>(s, T0, T1, wtol, open + kJSteps + 1, steps, look);
  // a V that is not orthogonal after all: the binary64 sweeps start from R^T
  jacobi_restart_kernel<<<gr, 256, 0, st>>>(s, R, ldr, open + kJSteps + 1, open + steps);
  *open_pairs = open + steps;
  return cudaGetLastError();
}

}  // namespace pylom
