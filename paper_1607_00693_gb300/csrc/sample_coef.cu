// Coefficient sampling a(x, xi) at fine-element centroids (Sec. 2.1.3).
//
// The bumps are Gaussians on a tensor lattice, so
//   z(x, y) = sum_bx gx_bx(x) * U_bx(y),   U_bx(y) = sum_by xi[by][bx] gy_by(y),
// with gx_bx(x) = exp(-(x - cx_bx)^2 / w^2) (and gy likewise).  A block
// handles strips of R element rows of up to kCoefCols columns: gy of the
// strip and then U are built in shared memory, each thread keeps gx of its
// column in registers and sweeps its rows of the strip, so the work per
// element is at most nbx FMAs plus the final exponential (the table-driven FP64
// exp of fexp.cuh).
//
// The FP64 kernel is bound by the FP64 pipe.  gx and gy depend on the place
// only, so a block takes the samples of one place one after the other and
// makes them once; and the blocks are as many as fit the chip, with equal
// shares of the (place, sample) pairs (as a grid of strips, 6.7 blocks an SM
// left it idle a fifth of the time, and gx cost 1.8 of 28 operations an
// element).  Bumps further than kCoefReach widths from a warp's columns are
// left out, four at a time: exp(-7.5^2) = 3.7e-25, so with amplitudes below
// kCoefAmp (of the exponent, or of the mean level of an affine field) what they
// add stays below 3e-17, less than the rounding there; a strip with a larger
// one, or with one that is not finite, sums them all.  On the 1024^2 workload
// (16 bumps a row, spacing one width) 12 of 16 products remain, with 32 bumps of
// 3/4 of the spacing 15 of 32.  Where a batch gives fewer than four pairs a
// block the strips get shorter.  A block's width follows the grid's (see the rule at the launch),
// narrow ones split the rows among their warps and share gx through shared
// memory, and the strips are of equal height.
// 32 samples of the 1024^2 grid: 2.25 -> 1.65 ms; 60 samples of 513^2 1.31 ->
// 1.05 ms (1.43 with 256 columns in every block and strips of 64 rows); 64
// samples of 32^2 with 32^2 narrow bumps 161 -> 89 us (187 without shared gx).
#include <cmath>

#include "common.cuh"
#include "fexp.cuh"

namespace stomsfem {

constexpr int kMaxBumps = 64;  // per lattice side
constexpr int kCoefThreads = 128;
constexpr size_t kCoefSmem = 48 * 1024;
constexpr double kCoefReach = 7.5;  // in widths
constexpr double kCoefAmp = 1e6;
constexpr int kCoefCols = 256;      // threads per block, and its columns at most (FP64; or half of them)

__host__ __device__ inline int coef_rows(int nbx, int nby) {
  int R = 128;
  while (R > 8 && (size_t)(64 + (size_t)(nbx + nby) * R) * sizeof(double) > kCoefSmem) R >>= 1;
  return R;
}

// clog / (1 + e): the FP32 reciprocal r of d = 1 + e, one cubic step r (1 + g
// + g^2) with g = 1 - d r (|g| below 2^-22, so g^3 below 2^-66), and one
// residual correction of the quotient; the FP64 division where d leaves the
// FP32 range.
__device__ __forceinline__ double sigmoid_scaled(double clog, double e) {
  const double d = 1.0 + e;
  // d >= 1 (or NaN): exponents 0 .. 90
  if ((unsigned)__double2hiint(d) - (1023u << 20) > (90u << 20)) return clog / d;
  const double r0 = (double)__frcp_rn((float)d);
  const double g = fma(-d, r0, 1.0);
  const double r = fma(r0, fma(g, g, g), r0);
  const double q = clog * r;
  return fma(fma(-d, q, clog), r, q);
}

template <int NBX, int COLS>
__global__ void __launch_bounds__(COLS, (NBX <= 32 ? 512 : 256) / COLS)
sample_coef_kernel(int nf, int kind, int nbx, int nby, int R, int nstrip, int kw, int share, int S, int per_block,
                   unsigned extra, double w, double amp, double scale, double clog, double gain,
                   const double* __restrict__ xi, double* __restrict__ a) {
  extern __shared__ double csm[];
  double* tab = csm;                     // [64] 2^(j/64)
  double* gy = csm + 64;                 // [nby][R]
  double* U = gy + (size_t)nby * R;      // [nbx][R]
  double* gxs = U + (size_t)nbx * R;     // share: [nbx][32 kw]
  const int tid = threadIdx.x;
  const double h = 1.0 / nf;
  const double iw2 = 1.0 / (w * w);
  // the warps split into row groups of kw warps (32 kw columns); those left
  // over only help with the tables
  const int cols = 32 * kw, nrg = COLS / cols, rg = tid / cols, col = tid - rg * cols;
  exp_table_fill(tab);
  // this block's (place, sample) pairs, the samples fastest: from npair b / grid
  // on, with npair = per_block grid + extra (32-bit divisions: 64-bit ones run on
  // the FP64 pipe, 2 us of a small call's 20)
  auto first = [&](unsigned b) { return (long long)per_block * b + extra * b / gridDim.x; };
  const long long u0 = first(blockIdx.x);
  const int npair = (int)(first(blockIdx.x + 1) - u0);
  int t = u0 <= 0x7fffffffll ? (int)((unsigned)u0 / (unsigned)S) : (int)(u0 / S), s = (int)(u0 - (long long)t * S);
  int place = -1, ey0 = 0, rows = 0, ex = 0;
  unsigned near = 0;    // groups of four bumps within reach of the warp's 32 columns
  unsigned have = 0;    // those that gx holds
  double gx[NBX];
  for (int k = 0; k < npair; ++k, t += s + 1 == S ? 1 : 0, s = s + 1 == S ? 0 : s + 1) {
    __syncthreads();  // (the table; gy and U of the pair before are no longer read)
    if (t != place) {
      place = t;
      const int strip = t % nstrip, col0 = t / nstrip * cols;
      ey0 = strip * R;
      rows = min(R, nf - ey0);
      ex = col0 + col;
      for (int q = tid; q < nby * rows; q += COLS) {
        const int by = q / rows, r = q % rows;
        const double dy = (ey0 + r + 0.5) * h - (by + 0.5) / nby;
        gy[by * R + r] = fexp(-dy * dy * iw2, tab);
      }
      if (share)
        for (int q = tid; q < nbx * cols; q += COLS) {
          const int bx = q / cols;
          const double dx = (col0 + (q - bx * cols) + 0.5) * h - (bx + 0.5) / nbx;
          gxs[q] = fexp(-dx * dx * iw2, tab);
        }
      const int e0 = ex & ~31;
      const float lo = (float)((e0 + 0.5) * h - kCoefReach * w), hi = (float)((e0 + 31.5) * h + kCoefReach * w);
      near = have = 0;
#pragma unroll
      for (int g = 0; g < NBX / 4; ++g)
        if ((4 * g + 3.5f) / nbx >= lo && (4 * g + 0.5f) / nbx <= hi) near |= 1u << g;
    }
    __syncthreads();
    const double* xs = xi + (size_t)s * nbx * nby;
    int beyond = 0;
    for (int q = tid; q < nbx * rows; q += COLS) {
      const int bx = q / rows, r = q % rows;
      double acc = 0.0;
      for (int by = 0; by < nby; ++by) acc = fma(__ldg(xs + by * nbx + bx), gy[by * R + r], acc);
      U[bx * R + r] = acc;
      if (!(fabs(acc) <= amp)) beyond = 1;
    }
    // (a flag in shared memory would be static: the host gives the dynamic part
    // all of the 48 KB that a launch may have without opting in for more)
    const bool large = __syncthreads_or(beyond);
    if (ex >= nf || rg >= nrg) continue;  // (every thread comes back to the barriers above)
    const unsigned use = large ? 0xffffffffu : near;
    if (use & ~have) {
      have = use;
#pragma unroll
      for (int bx = 0; bx < NBX; ++bx) {
        gx[bx] = 0.0;
        if (bx < nbx && (use >> (bx / 4) & 1)) {
          if (share) {
            gx[bx] = gxs[bx * cols + col];
          } else {
            const double dx = (ex + 0.5) * h - (bx + 0.5) / nbx;
            gx[bx] = fexp(-dx * dx * iw2, tab);
          }
        }
      }
    }
    double* arow = a + ((size_t)s * nf + ey0 + rg) * nf + ex;
    const size_t astep = (size_t)nrg * nf;
    for (int r = rg; r < rows; r += nrg, arow += astep) {
      double z = 0.0;
#pragma unroll
      for (int g = 0; g < NBX / 4; ++g)
        if (use >> g & 1) {
#pragma unroll
          for (int bx = 4 * g; bx < 4 * g + 4; ++bx)
            if (bx < nbx) z = fma(gx[bx], U[bx * R + r], z);
        }
      double v;
      if (kind == STOMSFEM_FIELD_EXP)
        v = fexp(scale * z, tab);
      else if (kind == STOMSFEM_FIELD_AFFINE)
        v = fma(scale, z, gain);
      else
        v = fexp(sigmoid_scaled(clog, fexp(-gain * z, tab)), tab);
      *arow = v;
    }
  }
}

// The same sum in FP32 arithmetic (expf, FP32 bump tables and sums; the
// stored values are FP64): for the FP32 upscaling form, whose cell matrices
// are FP32 anyway.  Relative error of a about |scale z| times a few 1e-7.
template <int NBX>
__global__ void __launch_bounds__(kCoefThreads)
sample_coef_f32_kernel(int nf, int kind, int nbx, int nby, int R, float w, float scale, float clog,
                       float gain, const double* __restrict__ xi, double* __restrict__ a) {
  extern __shared__ float fsm[];
  float* gy = fsm;                      // [nby][R]
  float* U = gy + (size_t)nby * R;      // [nbx][R]
  const int s = blockIdx.y;
  const int ey0 = blockIdx.x * R;
  const int rows = min(R, nf - ey0);
  const float h = 1.0f / (float)nf;
  const float iw2 = 1.0f / (w * w);
  const double* xs = xi + (size_t)s * nbx * nby;
  for (int q = threadIdx.x; q < nby * rows; q += blockDim.x) {
    const int by = q / rows, r = q % rows;
    const float dy = ((float)(ey0 + r) + 0.5f) * h - ((float)by + 0.5f) / (float)nby;
    gy[by * R + r] = expf(-dy * dy * iw2);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nbx * rows; q += blockDim.x) {
    const int bx = q / rows, r = q % rows;
    float acc = 0.f;
    for (int by = 0; by < nby; ++by) acc = fmaf((float)__ldg(xs + by * nbx + bx), gy[by * R + r], acc);
    U[bx * R + r] = acc;
  }
  __syncthreads();
  for (int ex = threadIdx.x; ex < nf; ex += blockDim.x) {
    const float x = ((float)ex + 0.5f) * h;
    float gx[NBX];
#pragma unroll
    for (int bx = 0; bx < NBX; ++bx) {
      const float dx = x - ((float)bx + 0.5f) / (float)nbx;
      gx[bx] = bx < nbx ? expf(-dx * dx * iw2) : 0.f;
    }
    double* arow = a + ((size_t)s * nf + ey0) * nf + ex;
    for (int r = 0; r < rows; ++r) {
      float z = 0.f;
#pragma unroll
      for (int bx = 0; bx < NBX; ++bx)
        if (bx < nbx) z = fmaf(gx[bx], U[bx * R + r], z);
      const float v = kind == STOMSFEM_FIELD_EXP      ? expf(scale * z)
                      : kind == STOMSFEM_FIELD_AFFINE ? fmaf(scale, z, gain)
                                                      : expf(clog / (1.0f + expf(-gain * z)));
      arow[(size_t)r * nf] = (double)v;
    }
  }
}

}  // namespace stomsfem

using namespace stomsfem;

static int sample_coef_impl(const stomsfem_grid* grid, const stomsfem_field* field, const double* xi,
                            int32_t S, int32_t precision, double* a, stomsfem_stream_t stream) {
  if (!grid || !field) return set_error(STOMSFEM_EINVAL, "grid/field is NULL");
  if (grid->nf <= 0 || S < 0) return set_error(STOMSFEM_EINVAL, "bad nf or S");
  if (precision != STOMSFEM_FP64 && precision != STOMSFEM_FP32)
    return set_error(STOMSFEM_EINVAL, "sampling precision must be STOMSFEM_FP64 or STOMSFEM_FP32");
  if (field->kind != STOMSFEM_FIELD_EXP && field->kind != STOMSFEM_FIELD_EXP_SIGMOID &&
      field->kind != STOMSFEM_FIELD_AFFINE)
    return set_error(STOMSFEM_EINVAL, "unknown field kind %d", field->kind);
  if (field->nbx <= 0 || field->nby <= 0 || field->nbx > kMaxBumps || field->nby > kMaxBumps)
    return set_error(STOMSFEM_EINVAL, "bump lattice %dx%d outside 1..%d per side", field->nbx,
                     field->nby, kMaxBumps);
  if (!(field->width > 0.0)) return set_error(STOMSFEM_EINVAL, "width must be > 0");
  if (S == 0) return STOMSFEM_OK;
  if (!xi || !a) return set_error(STOMSFEM_EINVAL, "xi and a must be device pointers");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int nbx = field->nbx;
  const int R = coef_rows(field->nbx, field->nby);
  const size_t smem = (size_t)(field->nbx + field->nby) * R * sizeof(float);
  const size_t K = (size_t)field->nbx * field->nby;
  const int sms = device_sm_count() > 0 ? device_sm_count() : 152;
  if (precision == STOMSFEM_FP64) {
    struct Shape {
      int cols, kw, R, nstrip, share;
      long long npair, blocks;
      size_t bytes;
    };
    auto shape = [&](int cols) {  // with blocks of `cols` threads
      Shape h;
      h.cols = cols;
      // columns of a block, 32 kw: the kw of the least work, in FP64 warp
      // instructions per row and sample (an element takes about 14 and one for each
      // bump within reach, U nbx nby / 32); 256 columns for every grid left a
      // third of the lanes of 513 past its edge
      int nchunk = 1;
      double least = 0.0;
      for (int k = cols / 32; k >= 1; --k) {
        const int n = (grid->nf + 32 * k - 1) / (32 * k);
        const double cost = n * (k * (14.0 + nbx) + nbx * field->nby / 32.0);
        if (k == cols / 32 || cost < least) {
          least = cost;
          h.kw = k;
          nchunk = n;
        }
      }
      auto pairs = [&](int r) { return (long long)((grid->nf + r - 1) / r) * nchunk * S; };
      h.blocks = (nbx <= 32 ? 512LL : 256LL) / cols * sms;  // as many as are resident
      h.R = R < 64 ? R : 64;
      while (h.R > 8 && pairs(h.R) < 4 * h.blocks) h.R >>= 1;
      // strips of equal height (77 rows as 39 + 38, not 64 + 13: the blocks' shares
      // count pairs)
      h.nstrip = (grid->nf + h.R - 1) / h.R;
      h.npair = pairs(h.R);
      h.R = (grid->nf + h.nstrip - 1) / h.nstrip;
      // row groups share the bump values of their columns where these fit
      const size_t own = (64 + (size_t)(nbx + field->nby) * h.R) * sizeof(double);
      const size_t shared_gx = (size_t)nbx * 32 * h.kw * sizeof(double);
      h.share = h.kw <= cols / 64 && own + shared_gx <= kCoefSmem;
      h.bytes = own + (h.share ? shared_gx : 0);
      return h;
    };
    // Blocks of 128 threads for more than 32 bumps a row (255 registers a thread:
    // two blocks an SM, where one of 256 threads has no other to cover its
    // barriers) and where there is at most one pair for every block of 256 (the
    // pairs then run on twice as many).  256 against 128 threads, us: 20 samples
    // of 128^2 with 64^2 bumps 338, 240; 100 of 16^2 with 33 x 8 bumps 130, 72; 200
    // of 8^2 with 16^2 bumps 41.9, 31.3; 150 of 16^2 42.3, 31.3.
    Shape h = shape(kCoefCols);
    if (nbx > 32 || h.npair <= h.blocks) h = shape(kCoefCols / 2);
    const unsigned grd = (unsigned)(h.npair < h.blocks ? h.npair : h.blocks);
    // the largest amplitude with which far bumps are left out: what they add
    // stays below the rounding of the exponent, or of an affine field's mean
    // level (whose field may be sampled with the mean zero: every bump counts then)
    const double gain_z = field->kind == STOMSFEM_FIELD_EXP_SIGMOID ? 0.25 * std::fabs(field->contrast_log * field->gain)
                                                                    : std::fabs(field->scale);
    const double amp = field->kind == STOMSFEM_FIELD_AFFINE ? kCoefAmp * std::fabs(field->gain) / gain_z
                                                            : (gain_z > 1.0 ? kCoefAmp / gain_z : kCoefAmp);
#define LAUNCH(N, C)                                                                                               \
  sample_coef_kernel<N, C><<<grd, C, h.bytes, st>>>(grid->nf, field->kind, nbx, field->nby, h.R, h.nstrip, h.kw,   \
                                                    h.share, S, (int)(h.npair / grd), (unsigned)(h.npair % grd),   \
                                                    field->width, amp, field->scale, field->contrast_log,          \
                                                    field->gain, xi, a)
#define LAUNCH2(N)                          \
  do {                                      \
    if (h.cols == kCoefCols)                \
      LAUNCH(N, kCoefCols);                 \
    else                                    \
      LAUNCH(N, kCoefCols / 2);             \
  } while (0)
    if (nbx <= 4) LAUNCH2(4);
    else if (nbx <= 8) LAUNCH2(8);
    else if (nbx <= 16) LAUNCH2(16);
    else if (nbx <= 32) LAUNCH2(32);
    else LAUNCH(64, kCoefCols / 2);
#undef LAUNCH2
#undef LAUNCH
    STOMSFEM_TRY_CUDA(cudaGetLastError());
    return STOMSFEM_OK;
  }
  // the sample index runs over gridDim.y (at most 65535 per launch)
  for (int s0 = 0; s0 < S; s0 += 65535) {
    const int Sc = S - s0 < 65535 ? S - s0 : 65535;
    dim3 grd((grid->nf + R - 1) / R, Sc);
    const double* xs = xi + (size_t)s0 * K;
    double* as = a + (size_t)s0 * grid->nf * grid->nf;
#define LAUNCH(N)                                                                                         \
  sample_coef_f32_kernel<N><<<grd, kCoefThreads, smem, st>>>(grid->nf, field->kind, nbx, field->nby, R,   \
                                                             (float)field->width, (float)field->scale,    \
                                                             (float)field->contrast_log, (float)field->gain, xs, as)
    if (nbx <= 4) LAUNCH(4);
    else if (nbx <= 8) LAUNCH(8);
    else if (nbx <= 16) LAUNCH(16);
    else if (nbx <= 32) LAUNCH(32);
    else LAUNCH(64);
#undef LAUNCH
    STOMSFEM_TRY_CUDA(cudaGetLastError());
  }
  return STOMSFEM_OK;
}

extern "C" int stomsfem_sample_coef(const stomsfem_grid* grid, const stomsfem_field* field,
                                    const double* xi, int32_t S, double* a,
                                    stomsfem_stream_t stream) {
  return sample_coef_impl(grid, field, xi, S, STOMSFEM_FP64, a, stream);
}

extern "C" int stomsfem_sample_coef_precision(const stomsfem_grid* grid, const stomsfem_field* field,
                                              const double* xi, int32_t S, int32_t precision, double* a,
                                              stomsfem_stream_t stream) {
  return sample_coef_impl(grid, field, xi, S, precision, a, stream);
}
