// Fine-grid Q1 FEM for large grids (the level-1 solves of the two-level
// Monte Carlo estimator, Remark in Sec. 4.1.1, Eq. MCmean2level): the
// standard Q1 system on the (nf-1)^2 interior nodes, zero Dirichlet data,
// load f h^2 per node, for a batch of samples, by conjugate gradients in
// FP64 preconditioned with one geometric multigrid V-cycle in FP32.
//
// Multigrid: levels nf_0 = nf, nf_{l+1} = nf_l / 2 down to nf_L <= 16;
// prolongation P (coarse node (I, J) at fine node (2I, 2J)) bilinear, or,
// when the batch's coefficient contrast exceeds kMgOdContrast, with the
// other fine nodes' weights from the fine stencil (mgf_interp_kernel);
// restriction P^T, Galerkin coarse operators A_{l+1} = P^T A_l P (9-point
// stencils again), damped Jacobi smoothing (two sweeps before
// and after the coarse correction: a symmetric V-cycle, so the
// preconditioner is symmetric positive definite and plain CG applies), and
// Chebyshev steps on the coarsest grid.  Stencils are stored per level and
// sample in FP32, over the full (nf_l+1)^2 node grid, in symmetric form: five couplings per node (centre, east, north,
// north-east, north-west), the other four read from the neighbours, so
// every level's operator is exactly symmetric (boundary nodes carry zero
// stencils and stay zero).
//
// CG: x, r, p, Ap in FP64; the matrix-vector product applies the fine
// 9-point stencil in FP64, formed from a once per solve and stored in
// symmetric form (five entries per node, nine FMAs per product); the
// per-sample dot products are block sums with one atomic per block; the
// step lengths are computed on the device.  The host checks convergence
// (max over samples of |r| / |f|) every few iterations.
#include <cmath>
#include <cstring>
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace stomsfem {

constexpr int kMgMaxLevels = 12;
// Damping of the two sweeps before and after the coarse correction.  On the
// bilinear levels the high-frequency eigenvalues of D^-1 A lie in [0.75, 1.5]
// (Q1 stencil, constant coefficient): the two sweeps are the Chebyshev pair
// of [0.8, 1.6] (largest factor on the former 0.09; 0.16 with 0.8 twice).  It
// converges, and the cycle stays definite, for eigenvalues below 2.4.  A
// bilinear level is the Q1 discretisation of its own elements with the fine
// coefficient inside, so its largest eigenvalue is at most that of one element's
// D^-1 A: 1.5 for a constant coefficient, and with a contrast of 1e3 (above it
// the other transfers run) 2.386, the maximum over all coefficients of 2^2 ..
// 64^2 fine cells an element (alternating between the vector and the bang-bang
// coefficient that is best for it; the hot cells then fill an element's corner;
// without a bound on the contrast it tends to 3).  The pair of [0.75, 1.75] would
// converge up to 2.5 and took one CG iteration more on smooth media (constant 9
// for 8, lognormal of contrast 900 18 for 17).  The operator-dependent levels
// keep 0.8 (see mgf_divisor_kernel).
constexpr float kMgOmega = 0.8f;
template <bool OD>
__device__ __forceinline__ float mg_omega(int sweep) {
  return OD ? kMgOmega : (sweep == 0 ? 1.0903f : 0.6744f);
}
// The coarsest grid (at most 16 elements per side): Chebyshev iteration in
// D^-1 A on [0.02, 2.5] (the smoothest mode of a 16^2 grid has 0.029, and the
// sweeps converge up to 2.5): 24 steps leave at most 0.03 of any mode in the
// interval, where 60 Jacobi sweeps left 0.25 of the smoothest.
constexpr int kMgCoarseSteps = 24;
constexpr float kMgCoarseLo = 0.02f, kMgCoarseHi = 2.5f;
constexpr int kMgSmall = 32;  // the level above the coarsest has at most this many elements per side; the two run in one kernel
constexpr int kMgThreads = 256;
// Coefficient contrast (max a / min a over the batch) above which the
// transfers between levels use the operator-dependent prolongation; below
// it the bilinear one, which converges as fast there (the same 12 CG
// iterations on the lognormal 1024^2 medium of contrast 100) and moves
// fewer bytes per cycle.
constexpr double kMgOdContrast = 1e3;

struct MgLevel {
  int nf;          // elements per side
  int N;           // (nf + 1)^2 nodes
  float* st;       // [S][st_stride(N)]: (centre, east, north, north-east)[N], north-west[N]
  float* u;        // [S][N]
  float* u2;       // [S][N] (Jacobi ping-pong)
  float* f;        // [S][N]
  float* P;        // [S][4][N]: prolongation weights from the next coarser level (per node type)
  float* dv;       // [S][N]: Jacobi divisor (see mgf_divisor_kernel)
};

__device__ __forceinline__ bool interior(int i, int j, int nf) { return i > 0 && j > 0 && i < nf && j < nf; }

// Stencils of every level in symmetric form: couplings m = 0..4 of a node
// are its centre, east, north, north-east and north-west ones; the west,
// south, south-west and south-east couplings are the east, north, north-east
// and north-west ones of the neighbour there (zero at the boundary nodes,
// whose values stay zero in every multigrid vector).  The first four lie
// side by side (one 16-byte load), the north-west ones follow.
__host__ __device__ __forceinline__ size_t st_stride(size_t N) { return (5 * N + 3) & ~size_t(3); }
__device__ __forceinline__ size_t st_at(int m, size_t N, long v) {
  return m < 4 ? 4 * (size_t)v + m : 4 * N + (size_t)v;
}
// Entry k = (dj + 1) * 3 + (di + 1) of the 9-point stencil of node v:
__device__ __forceinline__ int st_arr(int k) {  // coupling m holding entry k
  return k == 4 ? 0 : (k == 5 || k == 3) ? 1 : (k == 7 || k == 1) ? 2 : (k == 8 || k == 0) ? 3 : 4;
}
__device__ __forceinline__ long st_node(int k, long v, int W) {  // node whose coupling it is
  const int di = k % 3 - 1, dj = k / 3 - 1;
  return (dj < 0 || (dj == 0 && di < 0)) ? v + dj * W + di : v;
}
__device__ __forceinline__ float st_entry(const float* __restrict__ st, size_t N, int k, long v, int W) {
  return st[st_at(st_arr(k), N, st_node(k, v, W))];
}

// Level-0 stencil from a, FP32 for the preconditioner (symmetric form
// above); and the FP64 operator of the CG in symmetric form,
// st64[k][node] for k = centre, east, north, north-east, north-west (the
// west, south, south-west and south-east entries of a node are the east,
// north, north-east and north-west entries of its neighbours there; zero
// at the boundary nodes, whose values are zero in every CG vector).
// shift: the FP32 stencils are those of 2^shift a (a preconditioner may be
// scaled by any constant), which keeps their entries and the entries'
// reciprocals in range whatever the unit of the coefficient; 0 unless needed.
__device__ __forceinline__ float narrow_shifted(double v, int shift) {
  const int hi = __double2hiint(v);
  return narrow((hi & 0x7ff00000) ? __hiloint2double(hi + (int)((unsigned)shift << 20), __double2loint(v)) : v);
}
__global__ void mgf_fine_stencil_kernel(int nf, int shift, const double* __restrict__ a, float* __restrict__ st,
                                        double* __restrict__ st64) {
  const int s = blockIdx.y;
  const int W = nf + 1, N = W * W;
  const double* as = a + (size_t)s * nf * nf;
  float* ss = st + (size_t)s * st_stride(N);
  double* s64 = st64 + (size_t)s * 5 * N;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x) {
    const int i = v % W, j = v / W;
    double d[5] = {0, 0, 0, 0, 0};
    if (interior(i, j, nf)) {
      const double* p = as + (size_t)(j - 1) * nf + i - 1;
      const double aSW = p[0], aSE = p[1], aNE = p[nf + 1], aNW = p[nf];
      // products with 1/6 and 1/3, not quotients: an FP64 division is a
      // long instruction sequence on the FP64 pipe
      constexpr double k6 = 1.0 / 6.0, k3 = 1.0 / 3.0;
      const double north = aNW + aNE;
      d[0] = (4.0 * k6) * ((aSW + aSE) + north);
      d[1] = -(aSE + aNE) * k6;
      d[2] = -north * k6;
      d[3] = -aNE * k3;
      d[4] = -aNW * k3;
    }
    *reinterpret_cast<float4*>(ss + 4 * (size_t)v) =
        make_float4(narrow_shifted(d[0], shift), narrow_shifted(d[1], shift), narrow_shifted(d[2], shift),
                    narrow_shifted(d[3], shift));
    ss[4 * (size_t)N + v] = narrow_shifted(d[4], shift);
#pragma unroll
    for (int k = 0; k < 5; ++k) s64[(size_t)k * N + v] = d[k];
  }
}

// The 9-point stencil of interior node v (entries k = (dj + 1) * 3 + di + 1).
__device__ __forceinline__ void stencil9(const float* __restrict__ st, size_t N, long v, int W, float a[9]) {
#pragma unroll
  for (int k = 0; k < 9; ++k) a[k] = st_entry(st, N, k, v, W);
}

// The Jacobi divisor of a node from its nine entries (mgf_divisor_kernel).
__device__ __forceinline__ float jacobi_divisor(const float a[9]) {
  const float l1 = fabsf(a[0]) + fabsf(a[1]) + fabsf(a[2]) + fabsf(a[3]) + fabsf(a[5]) + fabsf(a[6]) +
                   fabsf(a[7]) + fabsf(a[8]);
  return fmaxf(a[4], 0.5f * (a[4] + l1));
}

// Operator-dependent prolongation (the black-box interpolation of Dendy,
// J. Comput. Phys. 48, 1982, for 9-point stencils): a fine node between
// two coarse nodes of a row takes weights from its stencil collapsed onto
// that row (columns summed: w_W = -a_W / a_C, w_E = -a_E / a_C), one between
// two coarse nodes of a column from the stencil collapsed onto the column;
// a cell-centre node solves its own equation with its four edge neighbours
// interpolated so.  Where the stencil sums to zero the weights sum to one;
// next to the Dirichlet boundary the couplings to boundary nodes (zero in
// the symmetric form) drop out.  Across jumps of the coefficient the
// weights follow the operator, which keeps the coarse-grid correction
// effective where bilinear interpolation is not.
// (A collapsed centre that is not positive, which a coarse Galerkin
// operator can in principle give, takes the bilinear weights instead.)
__device__ __forceinline__ void interp_row(const float a[9], float& wW, float& wE) {
  const float c = a[1] + a[4] + a[7];
  wW = c > 0.f ? -(a[0] + a[3] + a[6]) / c : 0.5f;
  wE = c > 0.f ? -(a[2] + a[5] + a[8]) / c : 0.5f;
}
__device__ __forceinline__ void interp_col(const float a[9], float& wS, float& wN) {
  const float c = a[3] + a[4] + a[5];
  wS = c > 0.f ? -(a[0] + a[1] + a[2]) / c : 0.5f;
  wN = c > 0.f ? -(a[6] + a[7] + a[8]) / c : 0.5f;
}

// Weights P[m][node] of every fine node: between coarse nodes of a row
// (x odd, y even) m = 0, 1 for the west and east ones; of a column (x even,
// y odd) m = 0, 1 for the south and north ones; a cell centre (both odd)
// m = 0..3 for its south-west, south-east, north-east and north-west
// corners; zero elsewhere (coarse-grid nodes take their coarse value).
__global__ void mgf_interp_kernel(int nff, const float* __restrict__ stf, float* __restrict__ P) {
  const int s = blockIdx.y;
  const int W = nff + 1;
  const size_t N = (size_t)W * W;
  const float* sf = stf + (size_t)s * st_stride(N);
  float* ps = P + (size_t)s * 4 * N;
  for (long v = blockIdx.x * (long)blockDim.x + threadIdx.x; v < (long)N; v += (long)gridDim.x * blockDim.x) {
    const int x = (int)(v % W), y = (int)(v / W);
    float w[4] = {0.f, 0.f, 0.f, 0.f};
    if (interior(x, y, nff) && ((x | y) & 1)) {
      float a[9];
      stencil9(sf, N, v, W, a);
      if ((x & 1) && !(y & 1)) {
        interp_row(a, w[0], w[1]);
      } else if (!(x & 1) && (y & 1)) {
        interp_col(a, w[0], w[1]);
      } else {
        // edge neighbours: south and north between coarse nodes of a row,
        // west and east between coarse nodes of a column
        float sW = 0.f, sE = 0.f, nW = 0.f, nE = 0.f, wS = 0.f, wN = 0.f, eS = 0.f, eN = 0.f, b[9];
        if (y - 1 > 0) { stencil9(sf, N, v - W, W, b); interp_row(b, sW, sE); }
        if (y + 1 < nff) { stencil9(sf, N, v + W, W, b); interp_row(b, nW, nE); }
        if (x - 1 > 0) { stencil9(sf, N, v - 1, W, b); interp_col(b, wS, wN); }
        if (x + 1 < nff) { stencil9(sf, N, v + 1, W, b); interp_col(b, eS, eN); }
        const float c = a[4];
        if (c > 0.f) {
          w[0] = -(a[0] + a[1] * sW + a[3] * wS) / c;  // south-west corner
          w[1] = -(a[2] + a[1] * sE + a[5] * eS) / c;  // south-east
          w[2] = -(a[8] + a[7] * nE + a[5] * eN) / c;  // north-east
          w[3] = -(a[6] + a[7] * nW + a[3] * wN) / c;  // north-west
        } else {
          w[0] = w[1] = w[2] = w[3] = 0.25f;
        }
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) ps[(size_t)m * N + v] = w[m];
  }
}

// Weight of fine node (gx, gy) in the operator-dependent prolongation of
// coarse node (I, J).
__device__ __forceinline__ float pweight(const float* __restrict__ ps, size_t N, int W, int gx, int gy, int I, int J) {
  const int dx = gx - 2 * I, dy = gy - 2 * J;
  if (dx < -1 || dx > 1 || dy < -1 || dy > 1) return 0.f;
  const size_t g = (size_t)gy * W + gx;
  const bool ox = gx & 1, oy = gy & 1;
  if (!ox && !oy) return (dx == 0 && dy == 0) ? 1.f : 0.f;
  if (ox && !oy) return dy != 0 ? 0.f : ps[(dx > 0 ? 0 : 1) * N + g];
  if (!ox && oy) return dx != 0 ? 0.f : ps[(dy > 0 ? 0 : 1) * N + g];
  const int m = dy > 0 ? (dx > 0 ? 0 : 1) : (dx < 0 ? 2 : 3);
  return ps[(size_t)m * N + g];
}

// Galerkin coarse stencils A_c = P^T A_f P at the interior coarse nodes,
// bilinear P.  Every weight is a constant once the loops are unrolled: the
// nine fine nodes of the coarse node's hat, their nine couplings, and the
// coarse nodes whose hats cover the coupled fine node; only the five stored
// couplings are formed.
// 1024^2, 8 samples, all levels: 508 -> 165 us.
__global__ void __launch_bounds__(kMgThreads) mgf_rap_bilinear_kernel(int nff, const float* __restrict__ stf,
                                                                      float* __restrict__ stc) {
  const int s = blockIdx.y;
  const int nfc = nff / 2, Wf = nff + 1, Wc = nfc + 1;
  const size_t Nf = (size_t)Wf * Wf, Nc = (size_t)Wc * Wc;
  const float* sf = stf + (size_t)s * st_stride(Nf);
  float* sc = stc + (size_t)s * st_stride(Nc);
  // (I, J) offsets of the stored couplings: centre, east, north, north-east, north-west
  constexpr int cI[5] = {0, 1, 0, 1, -1}, cJ[5] = {0, 0, 1, 1, 1};
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < (int)Nc; v += gridDim.x * blockDim.x) {
    const int I = v % Wc, J = v / Wc;
    float out[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    if (interior(I, J, nfc)) {
#pragma unroll
      for (int dj = -1; dj <= 1; ++dj)
#pragma unroll
        for (int di = -1; di <= 1; ++di) {
          const float wf = (di ? 0.5f : 1.f) * (dj ? 0.5f : 1.f);
          const long fv = (long)(2 * J + dj) * Wf + 2 * I + di;
#pragma unroll
          for (int ej = -1; ej <= 1; ++ej)
#pragma unroll
            for (int ei = -1; ei <= 1; ++ei) {
              const int k = (ej + 1) * 3 + ei + 1;
              const float afv = st_entry(sf, Nf, k, fv, Wf);
#pragma unroll
              for (int m = 0; m < 5; ++m) {
                const int tx = di + ei - 2 * cI[m], ty = dj + ej - 2 * cJ[m];
                const float px = tx == 0 ? 1.f : (tx == 1 || tx == -1) ? 0.5f : 0.f;
                const float py = ty == 0 ? 1.f : (ty == 1 || ty == -1) ? 0.5f : 0.f;
                if (px * py != 0.f) out[m] = fmaf(wf * px * py, afv, out[m]);
              }
            }
        }
#pragma unroll
      for (int m = 1; m < 5; ++m)
        if (!interior(I + cI[m], J + cJ[m], nfc)) out[m] = 0.f;
    }
#pragma unroll
    for (int m = 0; m < 5; ++m) sc[st_at(m, Nc, v)] = out[m];
  }
}

// The same with the operator-dependent P.
__global__ void mgf_rap_kernel(int nff, const float* __restrict__ stf, const float* __restrict__ P,
                               float* __restrict__ stc) {
  const int s = blockIdx.y;
  const int nfc = nff / 2;
  const int Wf = nff + 1;
  const int Nf = Wf * Wf, Nc = (nfc + 1) * (nfc + 1);
  const float* sf = stf + (size_t)s * st_stride(Nf);
  const float* ps = P + (size_t)s * 4 * Nf;
  float* sc = stc + (size_t)s * st_stride(Nc);
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < Nc; v += gridDim.x * blockDim.x) {
    const int I = v % (nfc + 1), J = v / (nfc + 1);
    float out[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (interior(I, J, nfc)) {
      for (int dj = -1; dj <= 1; ++dj)
        for (int di = -1; di <= 1; ++di) {
          const int fx = 2 * I + di, fy = 2 * J + dj;  // fine node in the support of coarse (I, J)
          const float wf = pweight(ps, Nf, Wf, fx, fy, I, J);
          if (wf == 0.f) continue;
          const int fv = fy * Wf + fx;
          for (int ej = -1; ej <= 1; ++ej)
            for (int ei = -1; ei <= 1; ++ei) {
              const int k = (ej + 1) * 3 + ei + 1;
              const float afv = st_entry(sf, Nf, k, fv, Wf);
              if (afv == 0.f) continue;
              const int gx = fx + ei, gy = fy + ej;  // neighbour fine node
              // the coarse nodes whose prolongation covers (gx, gy): one,
              // two or four by the node's type, with their weights
              int pI[4], pJ[4], np = 0;
              float pw[4];
              const size_t gv = (size_t)gy * Wf + gx;
              const int I0 = gx >> 1, J0 = gy >> 1;
              if (!(gx & 1) && !(gy & 1)) {
                pI[0] = I0; pJ[0] = J0; pw[0] = 1.f; np = 1;
              } else if (!(gy & 1)) {
                pI[0] = I0; pJ[0] = J0; pw[0] = ps[gv];
                pI[1] = I0 + 1; pJ[1] = J0; pw[1] = ps[(size_t)Nf + gv]; np = 2;
              } else if (!(gx & 1)) {
                pI[0] = I0; pJ[0] = J0; pw[0] = ps[gv];
                pI[1] = I0; pJ[1] = J0 + 1; pw[1] = ps[(size_t)Nf + gv]; np = 2;
              } else {
                pI[0] = I0; pJ[0] = J0; pw[0] = ps[gv];
                pI[1] = I0 + 1; pJ[1] = J0; pw[1] = ps[(size_t)Nf + gv];
                pI[2] = I0 + 1; pJ[2] = J0 + 1; pw[2] = ps[(size_t)2 * Nf + gv];
                pI[3] = I0; pJ[3] = J0 + 1; pw[3] = ps[(size_t)3 * Nf + gv]; np = 4;
              }
              for (int q = 0; q < np; ++q) {
                const int cI = pI[q] - I, cJ = pJ[q] - J;
                if (cI < -1 || cI > 1 || cJ < -1 || cJ > 1 || !interior(pI[q], pJ[q], nfc) || pw[q] == 0.f) continue;
                out[(cJ + 1) * 3 + cI + 1] += wf * afv * pw[q];
              }
            }
        }
    }
    sc[st_at(0, Nc, v)] = out[4];
    sc[st_at(1, Nc, v)] = out[5];
    sc[st_at(2, Nc, v)] = out[7];
    sc[st_at(3, Nc, v)] = out[8];
    sc[st_at(4, Nc, v)] = out[6];
  }
}

// Jacobi divisor of each interior node: its diagonal entry, or half the
// sum of the diagonal and the off-diagonal magnitudes where those exceed
// the diagonal.  With omega = 0.8 the damped sweep then converges on every
// level with a symmetric positive definite operator (the l1-Jacobi bound:
// the divisors are at least (a_ii + sum |a_ij|) / 1.6), so the V-cycle stays
// symmetric positive definite whatever the Galerkin coarse operators look
// like; on the fine level, an M-matrix, it is the diagonal itself.
__global__ void mgf_divisor_kernel(int nf, const float* __restrict__ st, float* __restrict__ dv) {
  const int s = blockIdx.y;
  const int W = nf + 1;
  const size_t N = (size_t)W * W;
  const float* ss = st + (size_t)s * st_stride(N);
  for (long v = blockIdx.x * (long)blockDim.x + threadIdx.x; v < (long)N; v += (long)gridDim.x * blockDim.x) {
    float d = 1.f;
    if (interior((int)(v % W), (int)(v / W), nf)) {
      float a[9];
      stencil9(ss, N, v, W, a);
      d = jacobi_divisor(a);
    }
    dv[(size_t)s * N + v] = d;
  }
}

// Block sum of v into acc[s] (one atomic per block).
__device__ __forceinline__ void block_sum_to(double v, double* acc) {
  __shared__ double part[32];
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) part[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = l < (int)(blockDim.x >> 5) ? part[l] : 0.0;
    t = warp_sum(t);
    if (l == 0) atomicAdd(acc, t);
  }
  __syncthreads();
}

// ---- the V-cycle's passes over a level, two fused kernels
//
// Smoothing sweeps, residual and transfers read the same five coupling
// arrays; as kernels of their own (two sweeps, residual, restriction going
// down; prolongation and two sweeps going up) they moved 152 bytes per node,
// five times the 28 that the arrays and vectors of one direction hold, and
// from 256^2 down a level's eight launches cost more than its work.  Here a
// warp marches up a strip of 32 columns, one row per step, with the stages
// one row behind each other: sweep 1 on row t, sweep 2 on row t - 1, the
// residual on row t - 2, the restriction on row t - 3.  The rows a stage
// needs of the one before it stay in registers, the neighbouring columns
// come from the neighbouring lanes, and each array entry is loaded once.
// The stages narrow the strip by one lane on either side each (26 of 32
// lanes write going down, 28 going up); a segment of rows starts three (two)
// rows early.  In shared-memory tiles (64 x 32 nodes, the first version) the
// same passes took 390 instructions per 32 nodes for index arithmetic and 18
// coupling loads, and ten turns of latency per phase on the small levels.
// 1024^2, 8 samples: the whole solve, with the leaner CG and set-up, 12.0 ->
// 6.84 ms; the finest level's passes 69 us down and 138 us up.
constexpr int kMgWarps = 4;
constexpr int kMgBlocks = 5;  // of the downward kernel, blocks an SM holds at least (96 registers a thread
                              // and a spill of six words; the upward one spills more there: 196 against 138 us
                              // on the finest level)

// One strip and row segment of a level for the calling warp.
struct MgMarch {
  int x, y0, y1;
  bool in;  // an interior column
};
__device__ __forceinline__ bool mg_march(int nf, int useful, int halo, int rows, MgMarch& m) {
  const int W = nf + 1, strips = (W + useful - 1) / useful;
  const int w = blockIdx.x * kMgWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int seg = w / strips;
  m.x = (w - seg * strips) * useful - halo + lane;
  m.y0 = seg * rows;
  m.y1 = min(m.y0 + rows, W);
  m.in = m.x > 0 && m.x < nf;
  return m.y0 < W;
}

__device__ __forceinline__ float lane_west(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float lane_east(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// A row of a vector with its two neighbouring columns.
struct MgTri {
  float w, c, e;
  __device__ __forceinline__ void set(float v) {
    c = v;
    w = lane_west(v);
    e = lane_east(v);
  }
};

// The couplings and right-hand side of one row; zero (centre 1) outside the
// interior.  q: the node.
struct MgCoef {
  float c, e, n, ne, nw, f;
  __device__ __forceinline__ void none() {
    c = 1.f;
    e = n = ne = nw = f = 0.f;
  }
};

// Rows in flight.  A warp's marches are bound by the latency of its rows (16
// warps an SM at about 100 registers): each lane copies its own entries of
// the row kMgAhead steps ahead into its own places of a ring in shared
// memory, which costs no registers and needs no barrier.
constexpr int kMgRing = 8, kMgAhead = kMgRing - 1;
struct MgRing {
  float4 st[kMgRing][32];
  float nw[kMgRing][32], f[kMgRing][32];
};
struct MgRingUp : MgRing {
  float u[kMgRing][32];
  double r[kMgRing][32];
};
template <int BYTES>
__device__ __forceinline__ void mg_cp(void* dst, const void* src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void mg_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void mg_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kMgAhead - 1) : "memory"); }
__device__ __forceinline__ void mg_fetch(MgRing& g, int slot, int lane, const float* st, const float* nws, const float* f,
                                         int q) {
  mg_cp<16>(&g.st[slot][lane], reinterpret_cast<const float4*>(st) + q);
  mg_cp<4>(&g.nw[slot][lane], nws + q);
  mg_cp<4>(&g.f[slot][lane], f + q);
}
__device__ __forceinline__ void mg_take(const MgRing& g, int slot, int lane, bool in, MgCoef& k) {
  k.none();
  if (in) {
    const float4 v = g.st[slot][lane];
    k.c = v.x;
    k.e = v.y;
    k.n = v.z;
    k.ne = v.w;
    k.nw = g.nw[slot][lane];
    k.f = g.f[slot][lane];
  }
}

// A 9-point stencil in place (its own row's entries and the row below's).
struct MgStencil {
  float a[9];
  __device__ __forceinline__ void set(const MgCoef& k, const MgCoef& below) {
    a[4] = k.c;
    a[5] = k.e;
    a[3] = lane_west(k.e);
    a[7] = k.n;
    a[1] = below.n;
    a[8] = k.ne;
    a[0] = lane_west(below.ne);
    a[6] = k.nw;
    a[2] = lane_east(below.nw);
  }
  __device__ __forceinline__ float apply(const MgTri& s, const MgTri& m, const MgTri& n) const {
    float t = 0.f;
    t = fmaf(a[0], s.w, t);
    t = fmaf(a[1], s.c, t);
    t = fmaf(a[2], s.e, t);
    t = fmaf(a[3], m.w, t);
    t = fmaf(a[4], m.c, t);
    t = fmaf(a[5], m.e, t);
    t = fmaf(a[6], n.w, t);
    t = fmaf(a[7], n.c, t);
    t = fmaf(a[8], n.e, t);
    return t;
  }
};

// Going down: u = two damped Jacobi sweeps from zero on A u = f, and fc =
// P^T (f - A u) at the next level's nodes.  OD: operator-dependent transfers,
// whose coarse operators need not be diagonally dominant: the sweeps divide
// by the divisor of mgf_divisor_kernel; with the bilinear transfers by the
// diagonal entry, as the bound on their eigenvalues allows (mg_omega).  rows: even.
template <bool OD>
__global__ void __launch_bounds__(kMgWarps * 32, kMgBlocks) mgf_down_kernel(int nf, int rows, const float* __restrict__ st,
                                                                 const float* __restrict__ dv,
                                                                 const float* __restrict__ P,
                                                                 const float* __restrict__ f, float* __restrict__ u,
                                                                 float* __restrict__ fc) {
  MgMarch m;
  if (!mg_march(nf, 26, 3, rows, m)) return;
  const int s = blockIdx.y, lane = threadIdx.x & 31;
  const int W = nf + 1, nfc = nf / 2, Wc = nfc + 1;
  const size_t N = (size_t)W * W;
  st += (size_t)s * st_stride(N);
  f += (size_t)s * N;
  u += (size_t)s * N;
  fc += (size_t)s * Wc * Wc;
  const float* nws = st + 4 * N;
  const float* ds = dv + (size_t)s * N;
  const float* ps = P + (size_t)s * 4 * N;
  const bool mine = lane >= 3 && lane < 29 && m.x < W;
  auto inside = [&](int y) { return m.in && y > 0 && y < nf; };
  __shared__ MgRing rings[kMgWarps];
  MgRing& ring = rings[threadIdx.x >> 5];
  MgCoef k0, k1, k2;          // rows t, t - 1, t - 2
  float r0, r1 = 0.f;         // reciprocal divisors of rows t, t - 1
  float dn = 1.f, dq = 1.f;   // divisors of rows t, t + 1 (OD)
  MgStencil sa, sb;           // rows t - 1, t - 2
  MgTri a0, a1{0.f, 0.f, 0.f}, a2{0.f, 0.f, 0.f};  // sweep 1: rows t, t - 1, t - 2
  MgTri b1, b2{0.f, 0.f, 0.f}, b3{0.f, 0.f, 0.f};  // sweep 2: rows t - 1, t - 2, t - 3
  MgTri c2, c3{0.f, 0.f, 0.f}, c4{0.f, 0.f, 0.f};  // residual: rows t - 2, t - 3, t - 4
  int t = m.y0 - 3;
  int q = t * W + m.x;  // node of row t
  k1.none();
  k2.none();
  sb.set(k1, k2);
#pragma unroll
  for (int k = 0; k < kMgAhead; ++k) {
    if (inside(t + k)) mg_fetch(ring, k, lane, st, nws, f, q + k * W);
    mg_commit();
  }
  if (OD) {
    if (inside(t)) dn = ds[q];
    if (inside(t + 1)) dq = ds[q + W];
  }
  int slot = 0;
#pragma unroll 2
  for (; t < m.y1 + 3; ++t, q += W, slot = (slot + 1) & (kMgRing - 1)) {
    mg_wait();
    mg_take(ring, slot, lane, inside(t), k0);
    r0 = __fdividef(1.f, OD ? dn : k0.c);
    if (t + kMgAhead < m.y1 + 3 && inside(t + kMgAhead))
      mg_fetch(ring, (slot + kMgAhead) & (kMgRing - 1), lane, st, nws, f, q + kMgAhead * W);
    mg_commit();
    if (OD) {
      dn = dq;
      dq = inside(t + 2) ? ds[q + 2 * W] : 1.f;
    }
    a0.set(mg_omega<OD>(0) * k0.f * r0);
    sa.set(k1, k2);
    const float v = inside(t - 1) ? a1.c + mg_omega<OD>(1) * (k1.f - sa.apply(a2, a1, a0)) * r1 : 0.f;
    if (mine && t - 1 >= m.y0 && t - 1 < m.y1) u[q - W] = v;
    b1.set(v);
    c2.set(inside(t - 2) ? k2.f - sb.apply(b3, b2, b1) : 0.f);
    const int y = t - 3;
    if (y >= m.y0 && y < m.y1 && !(y & 1) && mine && !(m.x & 1)) {
      const int I = m.x >> 1, J = y >> 1;
      float w = 0.f;
      if (interior(I, J, nfc)) {
        if constexpr (OD) {
          const MgTri* c[3] = {&c4, &c3, &c2};
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy) {
            w = fmaf(pweight(ps, N, W, m.x - 1, y + dy, I, J), c[dy + 1]->w, w);
            w = fmaf(pweight(ps, N, W, m.x, y + dy, I, J), c[dy + 1]->c, w);
            w = fmaf(pweight(ps, N, W, m.x + 1, y + dy, I, J), c[dy + 1]->e, w);
          }
        } else {
          w = c3.c + 0.5f * (c3.w + c3.e + c4.c + c2.c) + 0.25f * (c4.w + c4.e + c2.w + c2.e);
        }
      }
      fc[(size_t)J * Wc + I] = w;
    }
    a2 = a1;
    a1 = a0;
    b3 = b2;
    b2 = b1;
    c4 = c3;
    c3 = c2;
    sb = sa;
    k2 = k1;
    k1 = k0;
    r1 = r0;
  }
}

// (P u_c) at the interior fine node (x, y), operator-dependent P.
__device__ __forceinline__ float prolong_od(const float* __restrict__ ps, size_t Nf, int Wf, const float* __restrict__ u,
                                            int Wc, int x, int y) {
  const int I0 = x >> 1, J0 = y >> 1;
  const size_t v = (size_t)y * Wf + x;
  if (!(x & 1) && !(y & 1)) return u[J0 * Wc + I0];
  if (!(y & 1))  // between coarse nodes I0, I0 + 1 of row J0
    return ps[v] * u[J0 * Wc + I0] + ps[Nf + v] * u[J0 * Wc + I0 + 1];
  if (!(x & 1))  // between coarse nodes J0, J0 + 1 of column I0
    return ps[v] * u[J0 * Wc + I0] + ps[Nf + v] * u[(J0 + 1) * Wc + I0];
  // cell centre: corners SW, SE, NE, NW
  return ps[v] * u[J0 * Wc + I0] + ps[Nf + v] * u[J0 * Wc + I0 + 1] + ps[2 * Nf + v] * u[(J0 + 1) * Wc + I0 + 1] +
         ps[3 * Nf + v] * u[(J0 + 1) * Wc + I0];
}

// Going up: uo = two damped Jacobi sweeps on A u = f from ui + P uc.  r
// (the finest level, else NULL): the sample's r . uo is added to rz[s].
template <bool OD>
__global__ void __launch_bounds__(kMgWarps * 32) mgf_up_kernel(int nf, int rows, const float* __restrict__ st,
                                                               const float* __restrict__ dv,
                                                               const float* __restrict__ P,
                                                               const float* __restrict__ f,
                                                               const float* __restrict__ uc,
                                                               const float* __restrict__ ui, float* __restrict__ uo,
                                                               const double* __restrict__ r, double* __restrict__ rz) {
  MgMarch m;
  const bool run = mg_march(nf, 28, 2, rows, m);
  const int s = blockIdx.y, lane = threadIdx.x & 31;
  double acc = 0.0;
  if (run) {
    const int W = nf + 1, Wc = nf / 2 + 1;
    const size_t N = (size_t)W * W;
    st += (size_t)s * st_stride(N);
    f += (size_t)s * N;
    ui += (size_t)s * N;
    uo += (size_t)s * N;
    uc += (size_t)s * Wc * Wc;
    const float* nws = st + 4 * N;
    const float* ds = dv + (size_t)s * N;
    const float* ps = P + (size_t)s * 4 * N;
    const double* rs = r ? r + (size_t)s * N : nullptr;
    const bool mine = lane >= 2 && lane < 30 && m.x < W;
    auto inside = [&](int y) { return m.in && y > 0 && y < nf; };
    // bilinear: the coarse values beside column x, summed over the two
    // columns, of the coarse rows floor(y / 2) (ha) and the next (hb)
    const int I0 = m.x >> 1, I1 = (m.x + 1) >> 1;
    auto coarse = [&](int J) {
      return m.in && J > 0 && J < nf / 2 ? uc[J * Wc + I0] + uc[J * Wc + I1] : 0.f;
    };
    __shared__ MgRingUp rings[kMgWarps];
    MgRingUp& ring = rings[threadIdx.x >> 5];
    MgCoef k0, k1, k2;             // rows t, t - 1, t - 2
    float r0, r1 = 0.f, r2 = 0.f;  // reciprocal divisors of rows t, t - 1, t - 2
    float dn = 1.f, dq = 1.f;      // rows t, t + 1
    MgStencil sa, sb;              // rows t - 1, t - 2
    MgTri a0, a1{0.f, 0.f, 0.f}, a2{0.f, 0.f, 0.f};  // the starting values: rows t, t - 1, t - 2
    MgTri b1, b2{0.f, 0.f, 0.f}, b3{0.f, 0.f, 0.f};  // sweep 1: rows t - 1, t - 2, t - 3
    int t = m.y0 - 2;  // even
    int q = t * W + m.x;
    k1.none();
    k2.none();
    sb.set(k1, k2);
    auto fetch = [&](int y, int slot, int node) {
      if (inside(y)) {
        mg_fetch(ring, slot, lane, st, nws, f, node);
        mg_cp<4>(&ring.u[slot][lane], ui + node);
        if (rs) mg_cp<8>(&ring.r[slot][lane], rs + node);
      }
    };
#pragma unroll
    for (int k = 0; k < kMgAhead; ++k) {
      fetch(t + k, k, q + k * W);
      mg_commit();
    }
    int slot = 0;
    float ha = 0.f, hb = 0.f, hc = 0.f;  // coarse rows t / 2, t / 2 + 1, t / 2 + 2
    if constexpr (OD) {
      if (inside(t)) dn = ds[q];
      if (inside(t + 1)) dq = ds[q + W];
    } else {
      ha = coarse(t >> 1);
      hb = coarse((t >> 1) + 1);
    }
    double ra = 0.0, rb = 0.0;  // r of rows t - 1, t - 2
#pragma unroll 2
    for (; t < m.y1 + 2; ++t, q += W, slot = (slot + 1) & (kMgRing - 1)) {
      mg_wait();
      mg_take(ring, slot, lane, inside(t), k0);
      const float un = inside(t) ? ring.u[slot][lane] : 0.f;
      const double rt = rs && mine && inside(t) && t >= m.y0 && t < m.y1 ? ring.r[slot][lane] : 0.0;
      if (t + kMgAhead < m.y1 + 2) fetch(t + kMgAhead, (slot + kMgAhead) & (kMgRing - 1), q + kMgAhead * W);
      mg_commit();
      r0 = __fdividef(1.f, OD ? dn : k0.c);
      float v0 = 0.f;
      if constexpr (OD) {
        if (inside(t)) v0 = un + prolong_od(ps, N, W, uc, Wc, m.x, t);
        dn = dq;
        dq = inside(t + 2) ? ds[q + 2 * W] : 1.f;
      } else {
        if (t & 1) {
          v0 = un + 0.25f * (ha + hb);
          ha = hb;
          hb = hc;
        } else {
          v0 = un + 0.5f * ha;
          hc = coarse((t >> 1) + 2);
        }
        if (!inside(t)) v0 = 0.f;
      }
      a0.set(v0);
      sa.set(k1, k2);
      b1.set(inside(t - 1) ? a1.c + mg_omega<OD>(0) * (k1.f - sa.apply(a2, a1, a0)) * r1 : 0.f);
      const float v = inside(t - 2) ? b2.c + mg_omega<OD>(1) * (k2.f - sb.apply(b3, b2, b1)) * r2 : 0.f;
      if (mine && t - 2 >= m.y0 && t - 2 < m.y1) uo[q - 2 * W] = v;
      if (rs) acc = fma(rb, widen(v), acc);
      rb = ra;
      ra = rt;
      a2 = a1;
      a1 = a0;
      b3 = b2;
      b2 = b1;
      sb = sa;
      k2 = k1;
      k1 = k0;
      r2 = r1;
      r1 = r0;
    }
  }
  if (r) block_sum_to(acc, rz + s);
}

// ---- the last two levels of one sample in one CTA: the coarsest (at most 16
// elements per side) and the one above it (at most 32).  A thread holds one
// interior node of each (at most 961 and 225) with its couplings in registers;
// the vectors live in shared memory.  As marches and a kernel for the coarsest
// grid, three launches of 10 to 13 us; with the level of 64 and loops over the
// nodes in here too, 40 us.
struct MgSmallArgs {
  int nf;  // the upper level
  const float *st, *P;
  int nfc;  // the coarsest level
  const float* stc;
  const float* f;  // right-hand side on the upper level [S][N]
  float* out;      // solution there [S][N]
};
constexpr int kMgSmallThreads = 992;  // 31 warps: 31^2 interior nodes

template <bool OD>
__device__ __forceinline__ float mg_divisor(const float a[9]) {
  return OD ? jacobi_divisor(a) : a[4];
}
__device__ __forceinline__ float apply9s(const float a[9], const float* u, int W) {
  float t = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) t = fmaf(a[k], u[(k / 3 - 1) * W + k % 3 - 1], t);
  return t;
}

template <bool OD>
__global__ void __launch_bounds__(kMgSmallThreads) mgf_small_kernel(MgSmallArgs A) {
  constexpr int NF = (kMgSmall + 1) * (kMgSmall + 1), NC = 17 * 17;
  __shared__ float U[NF], V[NF], Uc[2][NC];
  const int s = blockIdx.x, tid = threadIdx.x;
  // the upper level's node (x, y) and the coarsest's (I, J)
  const int W = A.nf + 1, N = W * W, Wc = A.nfc + 1, Nc = Wc * Wc;
  const int mx = A.nf - 1, mc = A.nfc - 1;
  const int x = tid % mx + 1, y = tid / mx + 1, v = y * W + x;
  const int I = tid % mc + 1, J = tid / mc + 1, vc = J * Wc + I;
  const bool in = tid < mx * mx, inc = tid < mc * mc;
  for (int q = tid; q < NF; q += kMgSmallThreads) U[q] = V[q] = 0.f;
  for (int q = tid; q < NC; q += kMgSmallThreads) Uc[0][q] = Uc[1][q] = 0.f;
  float a[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, c[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  float fv = 0.f, fc = 0.f, rd = 0.f, rc = 0.f;
  if (in) {
    stencil9(A.st + (size_t)s * st_stride(N), N, v, W, a);
    fv = A.f[(size_t)s * N + v];
    rd = 1.f / mg_divisor<OD>(a);
  }
  if (inc) {
    stencil9(A.stc + (size_t)s * st_stride(Nc), Nc, vc, Wc, c);
    rc = 1.f / jacobi_divisor(c);
  }
  const float* ps = A.P + (size_t)s * 4 * N;
  __syncthreads();
  // two sweeps from zero, the residual and its restriction
  float u = mg_omega<OD>(0) * fv * rd;
  if (in) V[v] = u;
  __syncthreads();
  if (in) {
    u += mg_omega<OD>(1) * (fv - apply9s(a, V + v, W)) * rd;
    U[v] = u;
  }
  __syncthreads();
  if (in) V[v] = fv - apply9s(a, U + v, W);
  __syncthreads();
  if (inc) {
    const float* q = V + 2 * J * W + 2 * I;
    if constexpr (OD) {
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx)
          fc = fmaf(pweight(ps, N, W, 2 * I + dx, 2 * J + dy, I, J), q[dy * W + dx], fc);
    } else {
      fc = q[0] + 0.5f * (q[-1] + q[1] + q[-W] + q[W]) + 0.25f * (q[-W - 1] + q[-W + 1] + q[W - 1] + q[W + 1]);
    }
  }
  // the coarsest grid: Chebyshev steps from zero
  constexpr float theta = 0.5f * (kMgCoarseHi + kMgCoarseLo), delta = 0.5f * (kMgCoarseHi - kMgCoarseLo);
  constexpr float sigma = theta / delta;
  float d = fc * rc / theta, uc = d, rho = 1.f / sigma;
  if (inc) Uc[0][vc] = uc;
  __syncthreads();
  for (int k = 1; k < kMgCoarseSteps; ++k) {
    const float next = 1.f / (2.f * sigma - rho);
    if (inc) {
      d = next * rho * d + 2.f * next / delta * rc * (fc - apply9s(c, Uc[(k - 1) & 1] + vc, Wc));
      uc += d;
      Uc[k & 1][vc] = uc;
    }
    rho = next;
    __syncthreads();
  }
  // prolongation and two sweeps
  if (in) {
    const float* q = Uc[(kMgCoarseSteps - 1) & 1];
    if constexpr (OD) {
      u += prolong_od(ps, N, W, q, Wc, x, y);
    } else {
      const int I0 = x >> 1, J0 = y >> 1, I1 = (x + 1) >> 1, J1 = (y + 1) >> 1;
      u += 0.25f * (q[J0 * Wc + I0] + q[J0 * Wc + I1] + q[J1 * Wc + I0] + q[J1 * Wc + I1]);
    }
    U[v] = u;
  }
  __syncthreads();
  if (in) {
    u += mg_omega<OD>(0) * (fv - apply9s(a, U + v, W)) * rd;
    V[v] = u;  // (the residual in V was last read before the barriers of the Chebyshev steps)
  }
  __syncthreads();
  if (in) U[v] = u + mg_omega<OD>(1) * (fv - apply9s(a, V + v, W)) * rd;
  __syncthreads();
  for (int q = tid; q < N; q += kMgSmallThreads) A.out[(size_t)s * N + q] = U[q];
}

// mm[0] = bit pattern of max a, mm[1] = that of min a over the positive
// entries of a (the patterns of positive doubles order like their values;
// mm[0] starts at zero, mm[1] at the pattern 0x7F7F7F7F7F7F7F7F, a positive
// double of about 1.4e306).
__global__ void mgf_range_kernel(long long n, const double* __restrict__ a, unsigned long long* __restrict__ mm) {
  unsigned long long hi = 0, lo = 0x7F7F7F7F7F7F7F7Full;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(a[i]);
    if (b - 1 < 0x7ff0000000000000ull) {  // positive and not NaN
      hi = max(hi, b);
      lo = min(lo, b);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(mm, hi);
    atomicMin(mm + 1, lo);
  }
}

// ---------------------------------------------------------------- CG (FP64)

// Scalars of the iteration, per sample: r . z and p . Ap of this and the
// next iteration (two slots each, by the iteration's parity), r . r, b . b,
// and which samples have converged.  Each kernel clears the sums that the
// next ones add to (blocks x = y = 0 of a sample, values nothing reads then).
struct CgScal {
  double* v;  // [6][S]: r . z (two slots), p . Ap (two slots), r . r, b . b
  int32_t* done;
  int S;
  __device__ __forceinline__ double& rz(int slot, int s) const { return v[(size_t)slot * S + s]; }
  __device__ __forceinline__ double& pAp(int slot, int s) const { return v[(size_t)(2 + slot) * S + s]; }
  __device__ __forceinline__ double& rr(int s) const { return v[(size_t)4 * S + s]; }
};

// (A p)_v from the FP64 symmetric form: q points at p's value (pitch pw).
__device__ __forceinline__ double apply9d(const double* __restrict__ C, size_t N, long v, int W, const double* q, int pw) {
  const double *E = C + N, *Nn = C + 2 * N, *NE = C + 3 * N, *NW = C + 4 * N;
  double t = C[v] * q[0];
  t = fma(E[v], q[1], t);
  t = fma(E[v - 1], q[-1], t);
  t = fma(Nn[v], q[pw], t);
  t = fma(Nn[v - W], q[-pw], t);
  t = fma(NE[v], q[pw + 1], t);
  t = fma(NE[v - W - 1], q[-pw - 1], t);
  t = fma(NW[v], q[pw - 1], t);
  t = fma(NW[v - W + 1], q[-pw + 1], t);
  return t;
}

// p = z + beta p, beta = rz_new / rz_old (p = z on the first step, where p
// is not read: the workspace holds whatever it held before).  (In one kernel
// with the product A p, through a tile of p with its halo, the two took 255
// us where they take 28 and 165 apart, 1024^2, 8 samples: both are bound by
// the FP64 pipe, and the halo adds to it.)
__global__ void __launch_bounds__(kMgThreads) cg_direction_kernel(int nf, const float* __restrict__ z, CgScal c, int cur,
                                                                  int first, double* __restrict__ p) {
  const int s = blockIdx.y;
  const int N = (nf + 1) * (nf + 1);
  const double rn = c.rz(cur, s), ro = c.rz(cur ^ 1, s);
  const bool done = c.done[s] != 0;
  const double beta = (first || done || !(ro != 0.0)) ? 0.0 : rn / ro;
  if (blockIdx.x == 0 && threadIdx.x == 0) c.rr(s) = 0.0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x) {
    const size_t q = (size_t)s * N + v;
    p[q] = done ? 0.0 : first ? widen(z[q]) : fma(beta, p[q], widen(z[q]));
  }
}
__global__ void __launch_bounds__(kMgThreads) cg_matvec_kernel(int nf, const double* __restrict__ st64, CgScal c, int cur,
                                                               const double* __restrict__ p, double* __restrict__ Ap) {
  const int s = blockIdx.y;
  const int W = nf + 1, N = W * W;
  const double* C = st64 + (size_t)s * 5 * N;
  const double* ps = p + (size_t)s * N;
  double acc = 0.0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x) {
    const int i = v % W, j = v / W;
    double t = 0.0;
    if (interior(i, j, nf)) {
      t = apply9d(C, N, v, W, ps + v, W);
      acc += ps[v] * t;
    }
    Ap[(size_t)s * N + v] = t;
  }
  block_sum_to(acc, &c.pAp(cur, s));
}

// x += alpha p, r -= alpha Ap with alpha = rz / pAp (0 once converged or
// degenerate); rr[s] += r . r; the FP32 copy of r for the preconditioner.
// Clears the next iteration's r . z and p . Ap.
__global__ void __launch_bounds__(kMgThreads) cg_update_kernel(int nf, CgScal c, int cur, const double* __restrict__ p,
                                                               const double* __restrict__ Ap, double* __restrict__ x,
                                                               double* __restrict__ r, float* __restrict__ r32) {
  const int s = blockIdx.y;
  const int N = (nf + 1) * (nf + 1);
  const double pap = c.pAp(cur, s);
  const double al = (c.done[s] || !(pap > 0.0)) ? 0.0 : c.rz(cur, s) / pap;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    c.rz(cur ^ 1, s) = 0.0;
    c.pAp(cur ^ 1, s) = 0.0;
  }
  double acc = 0.0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x) {
    const size_t q = (size_t)s * N + v;
    x[q] += al * p[q];
    const double rv = r[q] - al * Ap[q];
    r[q] = rv;
    r32[q] = narrow(rv);
    acc += rv * rv;
  }
  block_sum_to(acc, &c.rr(s));
}

// r = b (f h^2 at the interior nodes), x = 0, |b|^2 per sample.
__global__ void __launch_bounds__(kMgThreads) cg_init_kernel(int nf, double fh2, double* __restrict__ x,
                                                             double* __restrict__ r, float* __restrict__ r32,
                                                             double* __restrict__ bb) {
  const int s = blockIdx.y;
  const int W = nf + 1, N = W * W;
  double acc = 0.0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x) {
    const int i = v % W, j = v / W;
    const double b = interior(i, j, nf) ? fh2 : 0.0;
    x[(size_t)s * N + v] = 0.0;
    r[(size_t)s * N + v] = b;
    r32[(size_t)s * N + v] = (float)b;
    acc += b * b;
  }
  block_sum_to(acc, bb + s);
}

}  // namespace stomsfem

using namespace stomsfem;

namespace {

// Level sizes: nf_0 = nf halved while even and above 16.
int mg_levels(int nf, int* nfs) {
  int L = 0;
  nfs[L++] = nf;
  while (nfs[L - 1] > 16 && nfs[L - 1] % 2 == 0 && L < kMgMaxLevels) {
    nfs[L] = nfs[L - 1] / 2;
    ++L;
  }
  return L;
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }
size_t range_offset(int S) { return (sizeof(double) * 6 * S + sizeof(int32_t) * S + 7) & ~size_t(7); }
size_t scal_bytes(int S) { return range_offset(S) + 2 * sizeof(unsigned long long); }

// Workspace layout of a batch of S samples.
size_t mg_layout(int nf, int S, MgLevel* lv, int* L, unsigned char* base, double** vec, double** scal) {
  int nfs[kMgMaxLevels];
  *L = mg_levels(nf, nfs);
  size_t o = 0;
  for (int l = 0; l < *L; ++l) {
    const size_t N = (size_t)(nfs[l] + 1) * (nfs[l] + 1);
    lv[l].nf = nfs[l];
    lv[l].N = (int)N;
    lv[l].st = reinterpret_cast<float*>(base + o);
    o += al256(sizeof(float) * st_stride(N) * S);
    lv[l].u = reinterpret_cast<float*>(base + o);
    o += al256(sizeof(float) * N * S);
    lv[l].u2 = reinterpret_cast<float*>(base + o);
    o += al256(sizeof(float) * N * S);
    lv[l].f = reinterpret_cast<float*>(base + o);
    o += al256(sizeof(float) * N * S);
    lv[l].P = reinterpret_cast<float*>(base + o);  // unused on the coarsest level
    o += l + 1 < *L ? al256(sizeof(float) * 4 * N * S) : 0;
    lv[l].dv = reinterpret_cast<float*>(base + o);
    o += al256(sizeof(float) * N * S);
  }
  const size_t N0 = (size_t)(nf + 1) * (nf + 1);
  for (int k = 0; k < 4; ++k) {  // r, p, Ap (x is the caller's u), then the FP64 stencil [S][5][N0]
    vec[k] = reinterpret_cast<double*>(base + o);
    o += al256(sizeof(double) * N0 * S * (k == 3 ? 5 : 1));
  }
  *scal = reinterpret_cast<double*>(base + o);  // alpha, pAp, rz, rz_old, rr, bb [S] doubles, done [S] int,
                                                // then the coefficient range (2 x 8 bytes, 8-aligned)
  o += al256(scal_bytes(S));
  return o;
}

dim3 grid2(int N, int S) {
  const int sms = device_sm_count() > 0 ? device_sm_count() : 152;
  long long bx = (N + kMgThreads - 1) / kMgThreads;
  const long long cap = ((long long)sms * 8 + S - 1) / S;
  if (bx > cap) bx = cap;
  if (bx < 1) bx = 1;
  return dim3((unsigned)bx, (unsigned)S);
}

// Rows per segment of a level's marches: the longest that still gives the
// chip twelve warps per SM (a segment repeats up to six rows of its
// neighbours; below that many warps the loads' latency shows), 8 at least.
int mg_rows(int nf, int S) {
  const int sms = device_sm_count() > 0 ? device_sm_count() : 152;
  int rows = 64;
  while (rows > 8 && (long long)((nf + 28) / 28) * ((nf + rows) / rows) * S < 12LL * sms) rows >>= 1;
  return rows;
}
dim3 mg_grid(int nf, int S, int useful, int rows) {
  const long long warps = (long long)((nf + useful) / useful) * ((nf + rows) / rows);
  return dim3((unsigned)((warps + kMgWarps - 1) / kMgWarps), (unsigned)S);
}

// z = V-cycle(r) on level l (f of level l holds the right-hand side; the
// result in u2 of level l); on the finest level rz[s] += r . z.  The level
// above the coarsest has at most kMgSmall elements per side and is not the
// finest (fine_mg_supported).
template <bool OD>
int vcycle(MgLevel* lv, int L, int l, int S, const double* r, double* rz, cudaStream_t st) {
  MgLevel& c = lv[l];
  if (l == L - 2) {
    const MgLevel& last = lv[L - 1];
    MgSmallArgs A;
    A.nf = c.nf;
    A.st = c.st;
    A.P = c.P;
    A.nfc = last.nf;
    A.stc = last.st;
    A.f = c.f;
    A.out = c.u2;
    mgf_small_kernel<OD><<<S, kMgSmallThreads, 0, st>>>(A);
    return check_cuda(cudaGetLastError(), "small levels");
  }
  const int rows = mg_rows(c.nf, S);
  MgLevel& n = lv[l + 1];
  mgf_down_kernel<OD><<<mg_grid(c.nf, S, 26, rows), kMgWarps * 32, 0, st>>>(c.nf, rows, c.st, c.dv, c.P, c.f, c.u, n.f);
  int rc = vcycle<OD>(lv, L, l + 1, S, nullptr, nullptr, st);
  if (rc) return rc;
  mgf_up_kernel<OD><<<mg_grid(c.nf, S, 28, rows), kMgWarps * 32, 0, st>>>(
      c.nf, rows, c.st, c.dv, c.P, c.f, n.u2, c.u, c.u2, r, rz);
  return check_cuda(cudaGetLastError(), "v-cycle");
}

}  // namespace

namespace stomsfem {

// (room to move the start to a 16-byte boundary)
size_t fine_mg_workspace_bytes(int nf, int S) {
  MgLevel lv[kMgMaxLevels];
  int L;
  double* vec[4];
  double* scal;
  return mg_layout(nf, S, lv, &L, nullptr, vec, &scal) + 16;
}

bool fine_mg_supported(int nf) {
  int nfs[kMgMaxLevels];
  const int L = mg_levels(nf, nfs);
  return nf > kMgSmall && nfs[L - 1] <= 16;  // (three levels at least)
}

// u [S][(nf+1)^2] (boundary 0) solves the Q1 system of each sample to
// |r| <= rtol |b|; returns the largest relative residual in *res and the
// iterations in *iters.  Synchronises the stream.
int fine_mg_solve(int nf, double f, const double* a, int S, double* u, void* workspace, size_t workspace_bytes,
                  double rtol, int max_iters, cudaStream_t st, double* res, int* iters) {
  MgLevel lv[kMgMaxLevels];
  int L;
  double* vec[4];
  double* scal;
  // the stencils are stored and copied 16 bytes at a time
  const size_t shift = (0 - reinterpret_cast<uintptr_t>(workspace)) & 15;
  const size_t need = shift + mg_layout(nf, S, lv, &L, static_cast<unsigned char*>(workspace) + shift, vec, &scal);
  if (workspace_bytes < need)
    return set_error(STOMSFEM_ENOMEM, "fine FEM workspace %zu < %zu bytes", workspace_bytes, need);
  double *r = vec[0], *p = vec[1], *Ap = vec[2], *st64 = vec[3];
  const CgScal sc{scal, reinterpret_cast<int32_t*>(scal + 6 * (size_t)S), S};
  double *rr = scal + 4 * (size_t)S, *bb = scal + 5 * (size_t)S;
  const int N0 = lv[0].N;
  const dim3 g0 = grid2(N0, S);
  unsigned long long* range = reinterpret_cast<unsigned long long*>(reinterpret_cast<unsigned char*>(scal) +
                                                                   range_offset(S));
  STOMSFEM_TRY_CUDA(cudaMemsetAsync(scal, 0, scal_bytes(S), st));
  STOMSFEM_TRY_CUDA(cudaMemsetAsync(range + 1, 0x7F, sizeof(unsigned long long), st));
  const int sms = device_sm_count() > 0 ? device_sm_count() : 152;
  mgf_range_kernel<<<sms * 4, kMgThreads, 0, st>>>((long long)S * nf * nf, a, range);
  const double h = 1.0 / nf;
  cg_init_kernel<<<g0, kMgThreads, 0, st>>>(nf, f * h * h, u, r, lv[0].f, bb);
  std::vector<double> hb(S), hr(S);
  std::vector<int32_t> hd(S, 0);
  unsigned long long hrange[2] = {0, 0};
  STOMSFEM_TRY_CUDA(cudaMemcpyAsync(hb.data(), bb, sizeof(double) * S, cudaMemcpyDeviceToHost, st));
  STOMSFEM_TRY_CUDA(cudaMemcpyAsync(hrange, range, sizeof(hrange), cudaMemcpyDeviceToHost, st));
  STOMSFEM_TRY_CUDA(cudaStreamSynchronize(st));
  double amax, amin;
  std::memcpy(&amax, &hrange[0], sizeof(double));
  std::memcpy(&amin, &hrange[1], sizeof(double));
  const bool od = amax > kMgOdContrast * amin;
  int exponent = 0;  // of the FP32 hierarchy's unit
  if (std::isfinite(amax) && (amax > 0x1p100 || amin < 0x1p-100))
    exponent = -(std::ilogb(amax) + std::ilogb(amin)) / 2;
  // multigrid set-up: stencils of every level
  mgf_fine_stencil_kernel<<<g0, kMgThreads, 0, st>>>(nf, exponent, a, lv[0].st, st64);
  for (int l = 0; l + 1 < L; ++l) {
    if (od) {
      mgf_interp_kernel<<<grid2(lv[l].N, S), kMgThreads, 0, st>>>(lv[l].nf, lv[l].st, lv[l].P);
      mgf_rap_kernel<<<grid2(lv[l + 1].N, S), kMgThreads, 0, st>>>(lv[l].nf, lv[l].st, lv[l].P, lv[l + 1].st);
    } else {
      mgf_rap_bilinear_kernel<<<grid2(lv[l + 1].N, S), kMgThreads, 0, st>>>(lv[l].nf, lv[l].st, lv[l + 1].st);
    }
  }
  // (the bilinear sweeps divide by the diagonal entry)
  for (int l = 0; l < L && od; ++l)
    mgf_divisor_kernel<<<grid2(lv[l].N, S), kMgThreads, 0, st>>>(lv[l].nf, lv[l].st, lv[l].dv);
  STOMSFEM_TRY_CUDA(cudaGetLastError());
  // z = M r, rz[cur] += r . z
  auto cycle = [&](int cur) {
    return od ? vcycle<true>(lv, L, 0, S, r, scal + (size_t)cur * S, st) : vcycle<false>(lv, L, 0, S, r, scal + (size_t)cur * S, st);
  };
  const float* z = lv[0].u2;
  int rc = cycle(0);
  if (rc) return rc;
  double worst = 1.0;
  // the next iteration whose residual the host reads: the fourth, then where
  // the reduction so far predicts the end, within four iterations
  int it = 0, check = 4;
  for (it = 1; it <= max_iters; ++it) {
    const int cur = (it - 1) & 1;  // slot of this iteration's scalars
    cg_direction_kernel<<<g0, kMgThreads, 0, st>>>(nf, z, sc, cur, it == 1, p);
    cg_matvec_kernel<<<g0, kMgThreads, 0, st>>>(nf, st64, sc, cur, p, Ap);
    cg_update_kernel<<<g0, kMgThreads, 0, st>>>(nf, sc, cur, p, Ap, u, r, lv[0].f);
    STOMSFEM_TRY_CUDA(cudaGetLastError());
    if (it == check || it == max_iters) {
      STOMSFEM_TRY_CUDA(cudaMemcpyAsync(hr.data(), rr, sizeof(double) * S, cudaMemcpyDeviceToHost, st));
      STOMSFEM_TRY_CUDA(cudaStreamSynchronize(st));
      worst = 0.0;
      bool all = true, finite = true;
      for (int s = 0; s < S; ++s) {
        const double rel = hb[s] > 0.0 ? std::sqrt(hr[s] / hb[s]) : 0.0;
        if (!std::isfinite(rel)) finite = false;
        if (rel <= rtol) hd[s] = 1;
        if (!hd[s]) all = false;
        worst = std::max(worst, rel);
      }
      if (!finite)
        return set_error(STOMSFEM_ENOTSPD, "fine FEM CG: non-finite residual after %d iterations", it);
      if (all) break;
      const double rate = std::log(worst) / it, left = rate < 0.0 ? (std::log(rtol) - std::log(worst)) / rate : 4.0;
      check = it + (left < 4.0 ? std::max(1, (int)left) : 4);
      STOMSFEM_TRY_CUDA(cudaMemcpyAsync(sc.done, hd.data(), sizeof(int32_t) * S, cudaMemcpyHostToDevice, st));
    }
    rc = cycle(cur ^ 1);
    if (rc) return rc;
  }
  if (res) *res = worst;
  if (iters) *iters = it > max_iters ? max_iters : it;
  if (!(worst <= rtol))
    return set_error(STOMSFEM_ENOTSPD, "fine FEM CG: relative residual %.3e after %d iterations", worst, max_iters);
  return STOMSFEM_OK;
}

}  // namespace stomsfem
