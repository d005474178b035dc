// Banded SPD solver for 9-point-stencil matrices, one system per CTA of four
// warps, FP64, one right-hand side: the coarse systems, the same with mixed
// boundary data, and the small fine-grid systems.
//
// Right-looking banded L D L^T in column blocks of 8.  Per block
//   1. warp 0 factorises the panel in registers: lanes 0..7 hold the rows of
//      the diagonal block, lane 8 the right-hand side as one more row (its
//      multipliers are the forward solution already divided by D), and every
//      lane one row (RS = 1, half bandwidths up to 32) or two below it; the
//      multipliers l and the unscaled columns c = l d go to shared memory,
//      l also to global scratch;
//   2. all warps update the trailing window, W -= l c^T, in 1 x 2 tiles,
//      while the last warp clears the retired ring rows and writes the next
//      8 rows, whose values it loaded one block earlier.
// The back substitution is warp 0's, with the factor blocks copied back two
// blocks ahead.  Rows past the end are identity rows, so every block is full.
//
// What bounds it is the FP64 pipe (one warp instruction per 16 clocks of an
// SM, whatever its lanes do), so the split is made for full lanes and few
// FP64 instructions: a right-hand side that rides along as a row costs none
// in the panel, 1 / d takes three (see recip), 1 x 2 tiles fill 272 of 288
// lanes of a 32-row triangle's rounds where 4 x 4 tiles in whole rounds of a
// warp fill 36 of 64, and their two loads per two FMAs cost nothing here
// (shared memory serves a tile's operands in a tenth of its FMAs' time).  Four warps
// per system, not one, because the batches are small: 512 systems leave an
// SM three or four, and one warp alone reaches a quarter of the pipe.
// 512 coarse systems of 32^2 cells with moments: 2.79 ms with a warp per
// sample and column blocks of 16, 1.45 ms here.
//
// Systems of at most 16 unknowns: tiny_solve, 16 lanes each (below).
//
// Row generator interface (Gen): typename Raw; load(r, Raw&); template
// make<double, 1>(r, raw, e, rhs) as in band_block.cuh; mx.
#pragma once
#include "band_block.cuh"
#include "common.cuh"

namespace stomsfem {

constexpr int kCtaThreads = 128;
constexpr int kCtaPerSm = 4;  // CTAs an SM holds at least (128 registers a thread)
constexpr int kCtaNB = 8;
constexpr int kCtaStages = 3;  // factor blocks of the back substitution in flight or in use

// Shared memory of one system: window rows of even pitch P >= b + 1 (lanes
// one row apart then read entries an odd number of doubles apart), the two
// panels [8][PB], the right-hand sides of the window rows.  The back
// substitution's staging and its ring of solutions reuse the window.
struct CtaBand {
  double *W, *Lp, *Cp, *rh;
  int RW, P, PB, LP;  // LP: pitch of a stored factor block's columns
};

__host__ __device__ inline int cta_ring_rows(int b) { return (kCtaNB + b + kCtaNB - 1) / kCtaNB * kCtaNB; }
__host__ __device__ inline int cta_lp(int b) { return (kCtaNB + b + 1) & ~1; }
__host__ __device__ inline int cta_wnd_elems(int b) {
  const int w = cta_ring_rows(b) * ((b + 2) & ~1), s = kCtaStages * kCtaNB * cta_lp(b) + cta_ring_rows(b);
  return w > s ? w : s;
}
__host__ __device__ inline size_t cta_smem_bytes(int b) {
  return sizeof(double) * (size_t)(((cta_wnd_elems(b) + 1) & ~1) + 2 * kCtaNB * ((b + 2) & ~1) + cta_ring_rows(b));
}
__device__ inline CtaBand make_cta_band(unsigned char* smem, int b) {
  CtaBand s;
  s.RW = cta_ring_rows(b);
  s.P = (b + 2) & ~1;
  s.PB = (b + 2) & ~1;
  s.LP = cta_lp(b);
  s.W = reinterpret_cast<double*>(smem);
  s.Lp = s.W + ((cta_wnd_elems(b) + 1) & ~1);
  s.Cp = s.Lp + kCtaNB * s.PB;
  s.rh = s.Cp + kCtaNB * s.PB;
  return s;
}

// 1 / d: the FP32 reciprocal (relative error below 2^-22) with one cubic
// step r (1 + e + e^2), e = 1 - d r, whose error e^3 is below 2^-66; the
// conversions work on the bits (band_block.cuh).  Outside the FP32 range the
// FP64 division.
__device__ __forceinline__ double recip(double d) {
  if (!in_f32_range(d)) return 1.0 / d;
  const double r = exact_f64(__frcp_rn(near_f32(d)));
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

__device__ __forceinline__ double shfl_d(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// Row r of the system into ring slot `slot` (cleared before); r >= n: the
// identity.
template <class Gen>
__device__ __forceinline__ void cta_put_row(const Gen& gen, const CtaBand& s, int r, int n, int b, int slot,
                                            const typename Gen::Raw& raw) {
  double* row = s.W + slot * s.P;
  if (r >= n) {
    row[0] = 1.0;
    s.rh[slot] = 0.0;
    return;
  }
  double e[5], rh[1];
  gen.template make<double, 1>(r, raw, e, rh);
  const int mx = gen.mx;
  row[0] += e[0];
  if (r >= 1 && 1 <= b) row[1] += e[1];
  if (mx - 1 >= 0 && r >= mx - 1 && mx - 1 <= b) row[mx - 1] += e[2];
  if (r >= mx && mx <= b) row[mx] += e[3];
  if (r >= mx + 1 && mx + 1 <= b) row[mx + 1] += e[4];
  s.rh[slot] = rh[0];
}

// Solves the system into x[n] (global); Lg: ceil(n / 8) * 8 * LP doubles of
// global scratch.  Every thread of the CTA calls it.  Returns false when a
// pivot was not positive (x then holds no solution).
template <int RS, class Gen>
__device__ bool cta_band_solve(const Gen& gen, int n, int b, const CtaBand& s, double* __restrict__ Lg,
                               double* __restrict__ x) {
  constexpr int NB = kCtaNB;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int RW = s.RW, P = s.P, PB = s.PB, LP = s.LP;
  const int nkb = (n + NB - 1) / NB;
  const bool filler = warp == kCtaThreads / 32 - 1;
  bool ok = true;  // warp 0's
  for (int q = tid; q < RW * P; q += kCtaThreads) s.W[q] = 0.0;
  __syncthreads();
  for (int r = tid; r < NB + b; r += kCtaThreads) {
    typename Gen::Raw raw;
    if (r < n) gen.load(r, raw);
    cta_put_row(gen, s, r, n, b, r, raw);
  }
  typename Gen::Raw next;  // of row K + NB + b + lane (lanes 0..7 of the filling warp)
  if (filler && lane < NB && NB + b + lane < n) gen.load(NB + b + lane, next);
  __syncthreads();
  const int ntiles = ((b >> 1) + 1) * ((b >> 1) + (b & 1));
  int kslot = 0;
  for (int kb = 0; kb < nkb; ++kb, kslot = ring(kslot + NB, RW)) {
    const int K = kb * NB;
    if (warp == 0) {
      // ---- panel
      double dg[NB], a[RS][NB], y[RS];
#pragma unroll
      for (int p = 0; p < NB; ++p) {
        dg[p] = lane < NB && lane >= p && lane - p <= b ? s.W[(kslot + lane) * P + lane - p]
                                                        : (lane == NB ? s.rh[kslot + p] : 0.0);
      }
      int slot[RS];
#pragma unroll
      for (int q = 0; q < RS; ++q) {
        const int i = lane + 32 * q;
        slot[q] = ring(kslot + NB + min(i, b - 1), RW);
        y[q] = s.rh[slot[q]];
#pragma unroll
        for (int p = 0; p < NB; ++p)
          a[q][p] = i < b && NB + i - p <= b ? s.W[slot[q] * P + NB + i - p] : 0.0;
      }
      double* Lb = Lg + (size_t)kb * NB * LP;
#pragma unroll
      for (int J = 0; J < NB; ++J) {
        double d = shfl_d(dg[J], J);
        const long long bits = __double_as_longlong(d);  // positive and not NaN, by the bit pattern
        if (bits <= 0 || bits > 0x7ff0000000000000ll) {
          ok = false;
          d = 1.0;
        }
        const double r = recip(d);
        const double lg = dg[J] * r, yJ = shfl_d(dg[J], NB);
        if (lane > J && lane < NB) Lb[J * LP + lane] = lg;
        if (lane == NB && K + J < n) x[K + J] = lg;
        double l[RS];
#pragma unroll
        for (int q = 0; q < RS; ++q) {
          const int i = lane + 32 * q;
          l[q] = a[q][J] * r;
          y[q] = fma(-l[q], yJ, y[q]);
          if (i < b) {
            Lb[J * LP + NB + i] = l[q];
            s.Lp[J * PB + i] = l[q];
            s.Cp[J * PB + i] = a[q][J];
          }
        }
#pragma unroll
        for (int p = J + 1; p < NB; ++p) {
          const double c = shfl_d(dg[J], p);
          dg[p] = fma(-lg, c, dg[p]);
#pragma unroll
          for (int q = 0; q < RS; ++q) a[q][p] = fma(-l[q], c, a[q][p]);
        }
      }
#pragma unroll
      for (int q = 0; q < RS; ++q)
        if (lane + 32 * q < b) s.rh[slot[q]] = y[q];
    }
    __syncthreads();
    // ---- trailing update: rows and columns K + NB .. K + NB + b - 1
    // in 1 x 2 tiles: rows 2 R and 2 R + 1 have R + 1 pairs of columns each,
    // R (R + 1) tiles before them
    for (int t = tid; t < ntiles; t += kCtaThreads) {
      int R = (int)((sqrtf(4.0f * t + 1.0f) - 1.0f) * 0.5f);
      if ((R + 1) * (R + 2) <= t) ++R;
      if (R * (R + 1) > t) --R;
      const int rem = t - R * (R + 1), odd = rem > R, i = 2 * R + odd, j = 2 * (rem - odd * (R + 1));
      double* w = s.W + ring(kslot + NB + i, RW) * P + (i - j);  // (i, j); (i, j + 1) at -1
      const bool two = j + 1 <= i;
      double v0 = w[0], v1 = two ? w[-1] : 0.0;
#pragma unroll
      for (int p = 0; p < NB; ++p) {
        const double l = -s.Lp[p * PB + i];
        const double2 c2 = *reinterpret_cast<const double2*>(s.Cp + p * PB + j);
        v0 = fma(l, c2.x, v0);
        v1 = fma(l, c2.y, v1);
      }
      w[0] = v0;
      if (two) w[-1] = v1;
    }
    // ---- the retired rows' slots take rows K + NB + b ..  (RW = NB + b
    // rounded up: slots past K + NB + b - 1 stay free until then)
    if (filler) {
      const int r0 = K + NB + b, fslot = ring(kslot + NB + b, RW);
      // rows r0 .. r0 + 7 lie in slots fslot ..: the retired ones and, before
      // them, the free ones, all clear or retired by now
      for (int q = lane; q < NB * P; q += 32) {
        const int k = q / P;
        s.W[ring(fslot + k, RW) * P + q - k * P] = 0.0;
      }
      __syncwarp();
      if (lane < NB) cta_put_row(gen, s, r0 + lane, n, b, ring(fslot + lane, RW), next);
      if (lane < NB && r0 + NB + lane < n) gen.load(r0 + NB + lane, next);
    }
    __syncthreads();
  }
  ok = __syncthreads_and(ok);
  if (warp == 0) {
    // ---- back substitution: x_p = z_p - sum_{i > p} l_ip x_i
    double* stg = s.W;
    double* xr = s.W + kCtaStages * NB * LP;  // ring of solution rows, zero past the end
    for (int q = lane; q < RW; q += 32) xr[q] = 0.0;
    const int chunks = NB * LP / 2;
    auto stage = [&](int kb) {
      if (kb >= 0) {
        const double* src = Lg + (size_t)kb * NB * LP;
        double* dst = stg + (kb % kCtaStages) * NB * LP;
        for (int v = lane; v < chunks; v += 32) cp_async16(dst + 2 * v, src + 2 * v);
      }
      cp_async_commit();
    };
    stage(nkb - 1);
    stage(nkb - 2);
    const int pl = lane >> 2;  // this lane's column
    double zn = (nkb - 1) * NB + pl < n ? x[(nkb - 1) * NB + pl] : 0.0;
    int ks = ((nkb - 1) * NB) % RW;
    for (int kb = nkb - 1; kb >= 0; --kb, ks = ks >= NB ? ks - NB : ks - NB + RW) {
      const int K = kb * NB;
      stage(kb - 2);
      cp_async_wait<kCtaStages - 1>();
      __syncwarp();
      const double* L = stg + (kb % kCtaStages) * NB * LP;
      const double z = zn;
      if (kb > 0) zn = x[K - NB + pl];
      double acc[NB];
#pragma unroll
      for (int q = 0; q < RS; ++q) {
        const int i = lane + 32 * q;
        const bool in = i < b;
        const double xi = in ? xr[ring(ks + NB + i, RW)] : 0.0;
#pragma unroll
        for (int p = 0; p < NB; ++p) {
          const double li = in ? L[p * LP + NB + i] : 0.0;
          acc[p] = q == 0 ? li * xi : fma(li, xi, acc[p]);
        }
      }
      // sums over the lanes, halving the columns a lane carries
#pragma unroll
      for (int h = 4, m = 16; h >= 1; h >>= 1, m >>= 1) {
        const bool upper = lane & m;
#pragma unroll
        for (int k = 0; k < h; ++k) {
          const double send = upper ? acc[k] : acc[k + h], keep = upper ? acc[k + h] : acc[k];
          acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
      }
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
      double t = z - acc[0];
#pragma unroll
      for (int q = NB - 1; q > 0; --q) {
        const double xq = shfl_d(t, 4 * q);
        if (pl < q) t = fma(-L[pl * LP + q], xq, t);
      }
      if ((lane & 3) == 0) {
        xr[ks + pl] = t;
        if (K + pl < n) x[K + pl] = t;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  return ok;
}

// ---- systems of at most 16 unknowns, 16 lanes each
//
// A CTA for a system of 1, 4 or 9 unknowns spends its time in barriers and its
// lanes on identity rows.  Here lane r holds row r of the dense lower triangle in
// registers, the factor l d l^T goes column by column with shuffles inside the
// 16 lanes, and l into shared memory (pitch 17) for the back substitution; eight
// systems a CTA, no barrier between warps and no global scratch.  Coarse systems
// of 4^2 cells, 20,000: 555 -> 91 us (345 with a warp each and column blocks of 16),
// one 19.0 -> 12.0; of 2^2 cells 311 -> 43 (86), with mixed boundary data 570 -> 103
// (363).
constexpr int kTinyMax = 16;
constexpr int kTinySystems = kCtaThreads / kTinyMax;  // per CTA

// Returns (in every lane of the system) false when a pivot was not positive; x:
// the solution of this lane's row.
template <class Gen>
__device__ __forceinline__ bool tiny_solve(const Gen& gen, int n, double (*L)[kTinyMax + 1], double& x) {
  const int r = threadIdx.x % kTinyMax, mx = gen.mx;
  double e[5] = {1.0, 0.0, 0.0, 0.0, 0.0}, y[1] = {0.0};  // rows past the end: the identity
  if (r < n) {
    typename Gen::Raw raw;
    gen.load(r, raw);
    gen.template make<double, 1>(r, raw, e, y);
  }
  double a[kTinyMax], inv = 1.0;
#pragma unroll
  for (int j = 0; j < kTinyMax; ++j) {
    const int d = r - j;  // (d <= r: the entries of a row that do not exist are never met)
    a[j] = d == 0 ? e[0] : 0.0;
    if (d == 1) a[j] += e[1];
    if (d >= 0 && d == mx - 1) a[j] += e[2];
    if (d > 0 && d == mx) a[j] += e[3];
    if (d == mx + 1) a[j] += e[4];
  }
  bool ok = true;
#pragma unroll
  for (int J = 0; J < kTinyMax; ++J) {
    if (J < n) {
      double d = __shfl_sync(0xffffffffu, a[J], J, kTinyMax);
      const long long bits = __double_as_longlong(d);  // positive and not NaN, by the bit pattern
      if (bits <= 0 || bits > 0x7ff0000000000000ll) {
        ok = false;
        d = 1.0;
      }
      const double rd = recip(d), l = a[J] * rd, yJ = __shfl_sync(0xffffffffu, y[0], J, kTinyMax);
      if (r == J) inv = rd;
      if (r > J) y[0] = fma(-l, yJ, y[0]);
#pragma unroll
      for (int p = J + 1; p < kTinyMax; ++p)
        if (p < n) a[p] = fma(-l, __shfl_sync(0xffffffffu, a[J], p, kTinyMax), a[p]);
      L[r][J] = l;
    }
  }
  __syncwarp();
  double z = y[0] * inv;
  for (int J = n - 1; J > 0; --J) {
    const double xJ = __shfl_sync(0xffffffffu, z, J, kTinyMax);
    if (r < J) z = fma(-L[J][r], xJ, z);
  }
  x = z;
  return ok;
}

}  // namespace stomsfem
