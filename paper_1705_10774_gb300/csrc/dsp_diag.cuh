// dsp_diag.cuh -- the diagnostics reduction shared by dsp_diagnostics and
// dsp_diagnostics_noalloc: per-patch FP64 Neumaier-compensated volume
// integrals of rho, m, E and of the face fields (the low face of every cell,
// so each face of a periodic tiling counts once), max |sum_d Delta_d b| over
// cells and max |b| over those faces; then the patches combined in patch
// order.  Both orders are fixed, so the result is deterministic.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace dsp {

constexpr int DIAG_NT = 256;  // threads of a per-patch diagnostics block
constexpr int DIAG_PER = 10;  // values per patch: 8 integrals, max |div b|, max |b|

struct NSum {
  double s, c;
};
__host__ __device__ __forceinline__ void nadd(NSum &a, double x) {
  const double t = a.s + x;
  if (fabs(a.s) >= fabs(x)) a.c += (a.s - t) + x;
  else a.c += (x - t) + a.s;
  a.s = t;
}

#ifdef __CUDACC__
// The FP64 value of an FP32 one by integer operations (exact; a conversion
// takes an FP64-pipe slot); zero, subnormal, infinite and NaN by conversion.
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const int b = __float_as_int(x), m = b & 0x7fffffff;
  if ((unsigned)(m - 0x00800000) >= 0x7f000000u) return (double)x;
  return __hiloint2double((b & (int)0x80000000) | ((m >> 3) + (896 << 20)), b << 29);
}
// |x| as an ordered integer
__device__ __forceinline__ long long diag_mag(double x) {
  return ((long long)(__double2hiint(x) & 0x7fffffff) << 32) | (unsigned)__double2loint(x);
}
// nadd with the magnitudes compared as integers: four FP64 operations
__device__ __forceinline__ void nadd_dev(NSum &a, double x) {
  const double t = a.s + x;
  const bool big = diag_mag(a.s) >= diag_mag(x);
  const double u = big ? a.s : x, v = big ? x : a.s;
  a.c += (u - t) + v;
  a.s = t;
}
// the larger of two magnitudes, a NaN never (as fmax)
__device__ __forceinline__ long long diag_max(long long m, double x) {
  const long long i = diag_mag(x);
  return i > m && i <= 0x7ff0000000000000ll ? i : m;
}

// The threads' sums and maxima of one block combined in a fixed order: lanes,
// then warps; DIAG_PER values to out.
__device__ __forceinline__ void diag_block(NSum acc[8], long long mdiv, long long mb, double *out) {
  __shared__ double sh[DIAG_NT / 32][DIAG_PER + 8];
  auto merge = [&](NSum &a, double s, double e) {
    nadd_dev(a, s);
    a.c += e;
  };
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const double s = __shfl_down_sync(0xffffffffu, acc[q].s, o), e = __shfl_down_sync(0xffffffffu, acc[q].c, o);
      merge(acc[q], s, e);
    }
    mdiv = max(mdiv, __shfl_down_sync(0xffffffffu, mdiv, o));
    mb = max(mb, __shfl_down_sync(0xffffffffu, mb, o));
  }
  if (lane == 0) {
    for (int q = 0; q < 8; q++) {
      sh[wid][2 * q] = acc[q].s;
      sh[wid][2 * q + 1] = acc[q].c;
    }
    sh[wid][16] = __longlong_as_double(mdiv);
    sh[wid][17] = __longlong_as_double(mb);
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    NSum tot = {0.0, 0.0};
    for (int w = 0; w < DIAG_NT / 32; w++) merge(tot, sh[w][2 * threadIdx.x], sh[w][2 * threadIdx.x + 1]);
    out[threadIdx.x] = tot.s + tot.c;
  } else if (threadIdx.x < 10) {
    double m = 0.0;
    for (int w = 0; w < DIAG_NT / 32; w++) m = fmax(m, sh[w][threadIdx.x + 8]);
    out[threadIdx.x] = m;
  }
}

// One block of DIAG_NT threads reduces part `part` of `parts` of one patch:
// interior U[5][nz][ny][nx], faces bx[nz][ny][nx+1], by[nz][ny+1][nx],
// bz[nz+1][ny][nx], cell volume dV; DIAG_PER values to out.  Thread-strided
// compensated sums, combined by a tree in a fixed order (one thread adding
// the 256 partials in turn took 0.8 ms, a chain of dependent FP64 operations
// of 64 clocks each; the tree takes 13 levels).
template <typename T>
__device__ void diag_patch(const T *u, const T *fx, const T *fy, const T *fz, int nx, int ny, int nz, double dV,
                           double *out, int part, int parts) {
  const long long nc = (long long)nx * ny * nz;
  NSum acc[8];
  for (int q = 0; q < 8; q++) acc[q].s = acc[q].c = 0.0;
  long long mdiv = 0, mb = 0;
  for (long long id = (long long)part * DIAG_NT + threadIdx.x; id < nc; id += (long long)parts * DIAG_NT) {
    const int row = (int)(id / nx), k = row / ny;
#pragma unroll
    for (int q = 0; q < 5; q++) nadd_dev(acc[q], widen(u[q * nc + id]) * dV);
    const double bxl = widen(fx[id + row]), bxr = widen(fx[id + row + 1]);
    const T *const y = fy + id + (long long)k * nx;
    const double byl = widen(y[0]), byr = widen(y[nx]);
    const double bzl = widen(fz[id]), bzr = widen(fz[id + (long long)nx * ny]);
    nadd_dev(acc[5], bxl * dV);
    nadd_dev(acc[6], byl * dV);
    nadd_dev(acc[7], bzl * dV);
    mdiv = diag_max(mdiv, (bxr - bxl) + (byr - byl) + (bzr - bzl));
    mb = diag_max(diag_max(diag_max(mb, bxl), byl), bzl);
  }
  diag_block(acc, mdiv, mb, out);
}

// Blocks that share each of np patches: pieces of at least 1024 cells, a few
// blocks per SM in all (so that one large patch is spread over the GPU), at
// most `records` partial results.  A function of the sizes alone: the order of
// the sums, and so the result, is the same every time.
inline int diag_parts(long long cells, int np, long long records) {
  long long m = cells / 1024;
  if (m > 1824 / np) m = 1824 / np;
  if (m > records / np) m = records / np;
  return m < 1 ? 1 : (int)m;
}
#endif

// The patches' DIAG_PER values combined in patch order (compensated sums of
// the integrals, maxima of the rest) into out[DIAG_PER].
__host__ __device__ inline void diag_combine(const double *part, int np, double *out) {
  NSum s[8];
  for (int q = 0; q < 8; q++) s[q].s = s[q].c = 0.0;
  double md = 0.0, mb = 0.0;
  for (int P = 0; P < np; P++) {
    for (int q = 0; q < 8; q++) nadd(s[q], part[(long long)P * DIAG_PER + q]);
    md = fmax(md, part[(long long)P * DIAG_PER + 8]);
    mb = fmax(mb, part[(long long)P * DIAG_PER + 9]);
  }
  for (int q = 0; q < 8; q++) out[q] = s[q].s + s[q].c;
  out[8] = md;
  out[9] = mb;
}

}  // namespace dsp
