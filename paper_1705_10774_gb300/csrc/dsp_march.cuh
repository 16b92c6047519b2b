// dsp_march.cuh -- the update of one tile by threads that own columns.
//
// A tile is TX x TY columns of cells and a run of tz planes.  One thread
// owns one column of the tile or of the one-cell halo around it and marches
// it through the planes; a column's own data along z (its cells' primitive
// state, slopes, upper z-face state, z-flux, carried corners, old speeds and
// EMFs) never leaves the thread, and shared memory carries only what a
// neighbouring column needs.  Per plane p, three barriers:
//   1  the conservative and constrained-transport update of plane p-1
//      (whose EMFs the last barrier published); primitives of plane p+1 from
//      the values loaded one plane earlier (the high faces from the columns
//      at +x and +y), the loads of plane p+2 started; MC slopes and the
//      Hancock predictor of plane p; the face states and edge corners that
//      the columns at +x and +y will read
//   2  primitives of plane p+1 published, those of the ring around the halo
//      computed; the fluxes and speeds of the faces on the column's low side
//      (x, y, and z at p-1/2); the new cells' signal speeds
//   3  edge EMFs on the column's low edges (x and y at p-1/2, z in plane p),
//      the in-plane flux divergence, the loads of the old values to update,
//      the faces of plane p+2 published
// The first three iterations only fill this pipeline.
// What bounds it: in FP64 the FP64 pipe (an FP64 warp instruction takes its
// slot whatever its active lanes), so whole warps hold tile columns, and the
// halo's columns are dealt so that those with fluxes share one warp and those
// with speeds alone another; in FP32 the issue slots, so a thread's positions
// are fixed for the whole tile and every shared address is one base plus a
// constant.
#pragma once
#include <cuda_runtime.h>

#include "dsp_dispatch.cuh"
#include "dsp_fast.cuh"
#include "dsp_internal.h"
#include "dsp_physics.cuh"

namespace dsp {

// A value the compiler keeps in a register instead of recomputing it from
// the kernel's parameters at each use (an FP64-to-FP32 conversion of a
// parameter takes a slot of the FP64 pipe each time).
__device__ __forceinline__ void keep(float &x) { asm volatile("" : "+f"(x)); }
__device__ __forceinline__ void keep(double &x) { asm volatile("" : "+d"(x)); }

// Shared-memory layout: every exchanged quantity is a plane over the radius-2
// padded tile.  FP32 tiles 16 or 24 wide put several rows in one warp: their
// row pitch shifts successive rows to other banks, and two quantities share a
// row's space.
template <typename T, int TX, int TY>
struct March {
  static constexpr int ROWS = TY + 4;
  static constexpr bool PAIR = sizeof(T) == 4 && TX % 32 != 0;
  static constexpr int PITCH = !PAIR ? TX + 4 : TX == 16 ? 48 : TX == 8 ? 40 : 2 * (TX + 4);
  static constexpr int PLANE = ROWS * PITCH;
  __host__ __device__ static constexpr int q(int k) { return PAIR ? (k >> 1) * PLANE + (k & 1) * (PITCH / 2) : k * PLANE; }
  static constexpr int QW = 0;     // [8] primitive states of the next plane
  static constexpr int QXR = 8;    // [8] state at the cell's upper x-face
  static constexpr int QYR = 16;   // [8] at its upper y-face
  static constexpr int QXP = 24;   // [3] corner (+y,+z) of x-edges [E, B_y, B_z]
  static constexpr int QYP = 27;   // [3] corner (+z,+x) of y-edges [E, B_z, B_x]
  static constexpr int PSTEP = 6;  // and both again for planes of the other parity
  static constexpr int QXM = 36;   // [3] corner (+y,-z)
  static constexpr int QYM = 39;   // [3] corner (-z,+x)
  static constexpr int QZC = 42;   // [3 corners (+,+) (-,+) (+,-)][E, B_x, B_y] of z-edges
  static constexpr int QFX = 51;   // [5] x-face fluxes
  static constexpr int QFY = 56;   // [5] y-face fluxes
  static constexpr int QSX = 61;   // [2] x-face speeds
  static constexpr int QSY = 63;   // [2]
  static constexpr int QSZ = 65;   // [2]
  static constexpr int QE = 67;    // [3] x-, y- and z-edge EMFs
  static constexpr int QNB = 70;   // [2] new x- and y-faces
  static constexpr int QB = 72;    // [2] x- and y-faces of the plane to come
  static constexpr int QU = 74;    // [5] the cell just updated (its own thread's)
  static constexpr int NQ = 79 + 1;
  static constexpr int total = (PAIR ? NQ / 2 : NQ) * PLANE;
  // threads: the tile's columns, the halo columns with fluxes (right column,
  // top row), then the other halo columns (bottom row, left column, corners);
  // the ring around the halo (primitives only) is dealt to the halo's threads
  static constexpr int NTILE = TX * TY;
  static constexpr int HB0 = NTILE + (TX + TY + 31) / 32 * 32;
  static constexpr int NEED = HB0 + TX + TY + 4;
  static constexpr int NRING = 2 * (TX + 2) + 2 * (TY + 2);
};

template <typename T, int TX, int TY, int NT, bool CONC, int RS>
__device__ __forceinline__ void march_tile(const DevCtx &c, const int P, const double dt, const int tile,
                                           const int zlo, const int zrun, T *sm, TileShared<T, NT> &S) {
  using M = March<T, TX, TY>;
  static_assert(M::NTILE % 32 == 0, "whole warps of tile columns");
  static_assert(NT >= M::NEED && NT - M::NTILE >= M::NRING, "a thread per column");
  constexpr int PITCH = M::PITCH;
  const T **srcA = S.srcA;
  const int tid = threadIdx.x;
  const PatchGeo &gp = c.geo[P];
  const int nx = gp.n[0], ny = gp.n[1], nz = gp.n[2];
  const int lox = gp.lo[0], loy = gp.lo[1], loz = gp.lo[2];
  const long long nc = (long long)nx * ny * nz;
  const long long ofx = 5 * nc, ofy = ofx + (long long)(nx + 1) * ny * nz, ofz = ofy + (long long)nx * (ny + 1) * nz;
  T gamma = (T)c.gamma, igm1 = (T)(1.0 / (c.gamma - 1.0)), gm1 = gamma - T(1);
  const T half = T(0.5);
  const int lev = gp.level;
  const double dxl = ldexp(c.dx, -lev);
  T hdt = (T)(0.5 * dt / dxl), dtdx = (T)(dt / dxl);
  const float gamma32 = (float)c.gamma;
  keep(gamma);
  keep(igm1);
  keep(gm1);
  keep(hdt);
  keep(dtdx);
  const int tix = tile % gp.nt[0], tiy = (tile / gp.nt[0]) % gp.nt[1], tiz = tile / (gp.nt[0] * gp.nt[1]);
  const int x0 = tix * TX, y0 = tiy * TY, z0 = tiz * gp.tz + zlo;
  const int zend = min(tiz * gp.tz + gp.tz, nz);  // of the whole z run
  const int tx = min(TX, nx - x0), ty = min(TY, ny - y0), tz = min(zrun, zend - z0);
  if (tz <= 0) return;
  const int Lp = newest<CONC>(c, P);
  const double tP = slot_time<CONC>(c, (long long)P * c.ns + Lp);
  const T *const own = (const T *)c.slab + (long long)Lp * c.slot_stride + gp.off;
  T *const dst = (T *)c.slab + (long long)((Lp + 1) % c.ns) * c.slot_stride + gp.off;
  const int *const bsz = c.bsz[lev];
  const float *const binv = c.binv[lev];
  const int bx0 = floordiv(lox + x0 - 2, bsz[0]), by0 = floordiv(loy + y0 - 2, bsz[1]),
            bz0 = floordiv(loz + z0 - 2, bsz[2]);
  const int nbx = floordiv(lox + x0 + tx + 2, bsz[0]) - bx0 + 1;
  const int nby = floordiv(loy + y0 + ty + 2, bsz[1]) - by0 + 1;
  const int nbz = floordiv(loz + z0 + tz + 2, bsz[2]) - bz0 + 1;
  owner_table<T, NT, CONC>(c, P, lev, tP, bx0, by0, bz0, nbx, nby, nbz, S);
  if (tid == 0) {
    S.fallback = 0;
    S.floors = 0;
    S.least = 0;
  }
  __syncthreads();

  // Bounds-checked build: every global address of the update is tested
  // against the slab of slices and the cross-level guard buffers; an address
  // outside both records DSP_ERR_BOUNDS and the access is redirected to the
  // slab's first element (a load) or dropped (a store), so the run ends with
  // that status and nothing faults.
#ifdef DSP_BOUNDS_CHECK
  auto src = [&](const T *a) -> const T * {
    const T *s0 = (const T *)c.slab, *g0 = (const T *)c.gbuf;
    if ((a >= s0 && a < s0 + c.slot_stride * c.ns) || (g0 && a >= g0 && a < g0 + c.gbuf_len)) return a;
    set_error(c, DSP_ERR_BOUNDS, P, -1);
    return s0;
  };
  auto put_global = [&](T *a, T v) {
    const T *s0 = (const T *)c.slab;
    if ((const T *)a >= s0 && (const T *)a < s0 + c.slot_stride * c.ns) *a = v;
    else set_error(c, DSP_ERR_BOUNDS, P, -1);
  };
#else
  auto src = [&](const T *a) -> const T * { return a; };
  auto put_global = [&](T *a, T v) { *a = v; };
#endif

  // ---- the thread's column (i, j) of the tile or its halo
  int i = 0, j = 0;
  bool h1 = false;
  if (tid < M::NTILE) {
    i = tid % TX;
    j = tid / TX;
    h1 = i < tx && j < ty;
  } else if (tid < M::HB0) {
    const int r = tid - M::NTILE;
    if (r < ty) {
      i = tx;
      j = r;
      h1 = true;
    } else if (r < ty + tx) {
      i = r - ty;
      j = ty;
      h1 = true;
    }
  } else {
    const int r = tid - M::HB0;
    h1 = r < tx + ty + 4;
    if (r < tx) {
      i = r;
      j = -1;
    } else if (r < tx + ty) {
      i = -1;
      j = r - tx;
    } else {
      i = (r - tx - ty) & 1 ? tx : -1;
      j = (r - tx - ty) & 2 ? ty : -1;
    }
  }
  if (!h1) i = j = 0;
  const int x = x0 + i, y = y0 + j;
  // what the column has: x-, y-, z-faces on its low side (full: with their
  // flux, else the speeds alone), low edges, a cell to update
  const bool incol = h1 && i >= 0 && i < tx && j >= 0 && j < ty;
  const bool xf = h1 && i >= 0, yf = h1 && j >= 0;
  const bool xfull = xf && j >= 0 && j < ty, yfull = yf && i >= 0 && i < tx;
  const bool zf = h1 && ((i >= 0 && i < tx) || (j >= 0 && j < ty));
  const bool ez_ = h1 && i >= 0 && j >= 0, ex_ = ez_ && i < tx, ey_ = ez_ && j < ty;
  const bool ownxy = x >= 0 && x < nx && y >= 0 && y < ny;
  T *const s0p = sm + (j + 2) * PITCH + (i + 2);
  // a column of the ring around the halo (primitives only)
  int ri = 0, rj = 0;
  bool ring = false;
  {
    const int r = tid - M::NTILE;
    if (r >= 0 && r < 2 * (tx + 2)) {
      ri = r % (tx + 2) - 1;
      rj = r / (tx + 2) ? ty + 1 : -2;
      ring = true;
    } else if (r >= 0 && r < 2 * (tx + 2) + 2 * (ty + 2)) {
      const int k = r - 2 * (tx + 2);
      ri = k / (ty + 2) ? tx + 1 : -2;
      rj = k % (ty + 2) - 1;
      ring = true;
    }
  }
  const int rx = x0 + ri, ry = y0 + rj;
  const bool rown = rx >= 0 && rx < nx && ry >= 0 && ry < ny;
  T *const r0p = sm + (rj + 2) * PITCH + (ri + 2);

  // ---- loads.  Table entry of the level cell (gx, gy, gz) of the padded
  // tile (floor of a small integer quotient through a rounded-up float
  // product: exact for level extents far below 2^20 cells).
  auto entry = [&](int gx, int gy, int gz) -> int {
    const int ex = __float2int_rd(((float)gx + 0.5f) * binv[0]) - bx0;
    const int ey = __float2int_rd(((float)gy + 0.5f) * binv[1]) - by0;
    const int ez = __float2int_rd(((float)gz + 0.5f) * binv[2]) - bz0;
    return (ez * nby + ey) * nbx + ex;
  };
  auto fetch = [&](const T *p, int e) -> T {
    T a = *src(p);
    const int bl = S.blend[e];
    if (bl) {
      const T b = *src(p + (long long)(((bl >> 2) & 63) - 16) * c.slot_stride);
      if ((bl & 3) == 2) {
        a = a + S.wgt[0][e] * (b - a);
      } else {
        const T cc = *src(p + (long long)(((bl >> 8) & 63) - 16) * c.slot_stride);
        a = (S.wgt[0][e] * a + S.wgt[1][e] * b) + S.wgt[2][e] * cc;
      }
    }
    return a;
  };
  // the face along ax on the low side of patch cell (xx, yy, zz): the
  // patch's own where it lies on one of its interior cells, else that of the
  // patch that owns the cell
  auto face = [&](int ax, int xx, int yy, int zz) -> T {
    const int mx0 = nx + (ax == 0), my0 = ny + (ax == 1), mz0 = nz + (ax == 2);
    if (xx >= 0 && xx < mx0 && yy >= 0 && yy < my0 && zz >= 0 && zz < mz0)
      return *src(own + (ax == 0 ? ofx : ax == 1 ? ofy : ofz) + ((long long)zz * my0 + yy) * mx0 + xx);
    const int gx = lox + xx, gy = loy + yy, gz = loz + zz;
    const int e = entry(gx, gy, gz);
    const int mx = S.n[0][e], my = S.n[1][e], mz = S.n[2][e];
    const int lx = gx - S.lo[0][e], ly = gy - S.lo[1][e], lz = gz - S.lo[2][e];
    const long long m = (long long)mx * my * mz;
    long long o = 5 * m;
    if (ax >= 1) o += (long long)(mx + 1) * my * mz;
    if (ax == 2) o += (long long)mx * (my + 1) * mz;
    const int fx = mx + (ax == 0), fy = my + (ax == 1);
    return fetch(srcA[e] + o + ((long long)lz * fy + ly) * fx + lx, e);
  };
  // the five conserved values of patch cell (xx, yy, q), its low x- and
  // y-faces and its high z-face
  auto load_cell = [&](int xx, int yy, bool inxy, int q, T u[5], T &fx, T &fy, T &fz) {
    if (inxy && q >= 0 && q < nz) {
      const long long o = ((long long)q * ny + yy) * nx + xx;
      const T *const a = own + o;
#pragma unroll
      for (int k = 0; k < 5; k++) u[k] = *src(a + k * nc);
      fx = *src(a + ofx + ((long long)q * ny + yy));
      fy = *src(a + ofy + (long long)q * nx);
      fz = *src(a + ofz + (long long)nx * ny);
      return;
    }
    const int gx = lox + xx, gy = loy + yy, gz = loz + q;
    const int e = entry(gx, gy, gz);
    const int mx = S.n[0][e], my = S.n[1][e], mz = S.n[2][e];
    const int lx = gx - S.lo[0][e], ly = gy - S.lo[1][e], lz = gz - S.lo[2][e];
    const long long m = (long long)mx * my * mz;
    const long long row = (long long)lz * my + ly;
    const T *const a = srcA[e] + row * mx + lx;
#pragma unroll
    for (int k = 0; k < 5; k++) u[k] = fetch(a + k * m, e);
    const bool zin = q >= 0 && q < nz;
    if (zin && xx == nx && yy >= 0 && yy < ny) fx = *src(own + ofx + ((long long)q * ny + yy) * (nx + 1) + nx);
    else fx = fetch(a + 5 * m + row, e);
    if (zin && yy == ny && xx >= 0 && xx < nx) fy = *src(own + ofy + ((long long)q * (ny + 1) + ny) * nx + xx);
    else fy = fetch(a + 5 * m + (long long)(mx + 1) * my * mz + (long long)lz * mx, e);
    fz = face(2, xx, yy, q + 1);
  };
  auto prim_of = [&](const T u[5], T fxl, T fxh, T fyl, T fyh, T fzl, T fzh, T W[8], int *floored) {
    if constexpr (kFast) fast::prim(u[0], u[1], u[2], u[3], u[4], fxl, fxh, fyl, fyh, fzl, fzh, gm1, W, floored);
    else prim(u[0], u[1], u[2], u[3], u[4], fxl, fxh, fyl, fyh, fzl, fzh, gamma, W, floored);
  };
  // a cell state plus or minus half a slope (held as the half slope in the
  // fast forms)
  auto up = [&](T w, T d) -> T { return kFast ? w + d : w + half * d; };
  auto dn = [&](T w, T d) -> T { return kFast ? w - d : w - half * d; };

  // raw values of the next plane and the z-face below it
  T ru[5], rfx = T(0), rfy = T(0), rfz = T(0), fzl = T(0);
  T fd[3], zdl[8];  // plane p's normal-field differences, W(p) - W(p-1)

  T smax_t = T(0);
  T zp[8];                                   // state at the upper z-face of plane p-1
  T fzp[5], du[5];                           // z-flux at p-3/2, in-plane divergence of p-1
  T sxp[2], syp[2];                          // x- and y-face speeds of plane p-1
  T cxo[3], cyo[3];                          // corners (-y,+z) and (+z,-x) of plane p-1
  T exp_ = T(0), eyp_ = T(0);                // x- and y-edge EMFs at p-3/2
  T dey = T(0), dex = T(0);                  // E_z(j+1) - E_z and E_z(i+1) - E_z of plane p-1
  T nfzl = T(0), nfzh = T(0);  // new z-faces of the cell just updated
  const int nt_ = tz + 1;

  // signal speed of the cell just updated (plane q); needs the neighbours' new faces
  auto signal_new = [&](int q) {
    T Wn[8];
    int floored = 0;
    T un[5];
#pragma unroll
    for (int k = 0; k < 5; k++) un[k] = s0p[M::q(M::QU + k)];
    prim_of(un, s0p[M::q(M::QNB)], s0p[M::q(M::QNB) + 1], s0p[M::q(M::QNB + 1)], s0p[M::q(M::QNB + 1) + PITCH], nfzl,
            nfzh, Wn, &floored);
    if (floored) atomicAdd(&S.floors, 1);
    if (!(Wn[RHO] > T(0)) || !(Wn[PR] > T(0)))
      set_error(c, DSP_ERR_UNPHYSICAL, P, ((long long)q * ny + y) * nx + x);
    if constexpr (kFast) smax_t = tmax(smax_t, fast::signal_sum(Wn, gamma));
    else smax_t = tmax(smax_t, signal_sum(Wn, gamma));
  };

  for (int it = -3; it <= nt_ + 1; it++) {
    const int p = z0 - 1 + it;
    const int par = it & 1;

    const bool flux = it > 0 && it < nt_;  // planes whose in-plane fluxes are needed
    T fx[5], fy[5], fz[5], sx[2], sy[2], sz[2];
    // a face between its low cell's state L and the column's own state R, in
    // the frame of its axis; F in lab order
    auto face_of = [&](auto dd, const T *L8, const T *R8, bool full, T F[5], T s2[2]) {
      constexpr int d = decltype(dd)::value;
      constexpr int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
      constexpr int cmp[8] = {RHO, VX + d, VX + t1, VX + t2, PR, BX + d, BX + t1, BX + t2};
      T WL[8], WR[8], Fn[5];
#pragma unroll
      for (int k = 0; k < 8; k++) {
        WL[k] = L8[cmp[k]];
        WR[k] = R8[cmp[k]];
      }
      if (full) {
        if constexpr (kFast && RS == 0) fast::hll(WL, WR, gamma, igm1, Fn, s2[0], s2[1]);
        else face_flux<T, 0, RS>(WL, WR, gamma, igm1, Fn, s2[0], s2[1]);
        F[0] = Fn[0];
        F[1 + d] = Fn[1];
        F[1 + t1] = Fn[2];
        F[1 + t2] = Fn[3];
        F[4] = Fn[4];
      } else {
        if constexpr (kFast && RS == 0) fast::speeds(WL, WR, gamma, s2[0], s2[1]);
        else hll_speeds<T, 0>(WL, WR, gamma, s2[0], s2[1]);
      }
    };
    // ---- 1: primitives of plane p+1, loads of plane p+2
    T xr[8], yr[8];  // states at the low x- and y-faces' high side
    T cx0[3], cxn[3], cy0[3], cyn[3], cz0[3];
    T wn[8];
    if (h1 && it <= nt_) {
      T fn[3], w0[8];
      if (it >= -2) {
        const T fxh = s0p[M::q(M::QB) + 1], fyh = s0p[M::q(M::QB + 1) + PITCH];
        prim_of(ru, rfx, fxh, rfy, fyh, fzl, rfz, wn, nullptr);
        fn[0] = fxh - rfx;
        fn[1] = fyh - rfy;
        fn[2] = rfz - fzl;
        fzl = rfz;
      }
      if (it >= -1) {
#pragma unroll
        for (int k = 0; k < 8; k++) w0[k] = s0p[M::q(M::QW + k)];
      }
      // slopes and predictor of plane p
      T dX[8], dY[8], dZ[8], ws[8];
      if (it >= 0) {
#pragma unroll
        for (int k = 0; k < 8; k++) {
          const T *const q = s0p + M::q(M::QW + k);
          const T w = w0[k];
          const T zdr = wn[k] - w;
          if constexpr (kFast) {
            dX[k] = k == BX ? half * fd[0] : fast::mc_half(w - q[-1], q[1] - w);
            dY[k] = k == BY ? half * fd[1] : fast::mc_half(w - q[-PITCH], q[PITCH] - w);
            dZ[k] = k == BZ ? half * fd[2] : fast::mc_half(zdl[k], zdr);
          } else {
            dX[k] = k == BX ? fd[0] : mc(w - q[-1], q[1] - w);
            dY[k] = k == BY ? fd[1] : mc(w - q[-PITCH], q[PITCH] - w);
            dZ[k] = k == BZ ? fd[2] : mc(zdl[k], zdr);
          }
          zdl[k] = zdr;
        }
        if constexpr (kFast) fast::predict(w0, dX, dY, dZ, gamma, dtdx, ws);
        else predict(w0, dX, dY, dZ, gamma, hdt, ws);
        // every face state positive: the state less its largest half slope is
        const T dr = fmax_mag(fmax_mag(dX[RHO], dY[RHO]), dZ[RHO]), dp = fmax_mag(fmax_mag(dX[PR], dY[PR]), dZ[PR]);
        if (!tpos(dn(ws[RHO], dr)) || !tpos(dn(ws[PR], dp))) {
          // counted as 16 x 8 tiles and whole z runs meet the cell (the halo
          // cells of each with it), whatever the tile and its part
          const bool zc = (p >= z0 || zlo == 0) && (p < z0 + tz || z0 + tz == zend);
          const int cx = min(max(x, 0), nx - 1), cy = min(max(y, 0), ny - 1);
          if (zc && cx >= x0 && cx < x0 + tx && cy >= y0 && cy < y0 + ty) {
            const int kx = 1 + (x > 0 && x % 16 == 0 && x < nx) + (x >= 0 && x % 16 == 15 && x < nx - 1);
            const int ky = 1 + (y > 0 && y % 8 == 0 && y < ny) + (y >= 0 && y % 8 == 7 && y < ny - 1);
            atomicAdd(&S.fallback, kx * ky);
          }
#pragma unroll
          for (int k = 0; k < 8; k++) { dX[k] = T(0); dY[k] = T(0); dZ[k] = T(0); ws[k] = w0[k]; }
        }
        // face states
        T XR[8], YR[8], ZR[8], ZU[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
          XR[k] = up(ws[k], dX[k]);
          YR[k] = up(ws[k], dY[k]);
          ZU[k] = up(ws[k], dZ[k]);
          xr[k] = dn(ws[k], dX[k]);
          yr[k] = dn(ws[k], dY[k]);
          ZR[k] = dn(ws[k], dZ[k]);
          if constexpr (sizeof(T) == 8) {  // held, not added up again for each corner
            keep(XR[k]);
            keep(YR[k]);
            keep(ZU[k]);
            keep(xr[k]);
            keep(yr[k]);
            keep(ZR[k]);
          }
          s0p[M::q(M::QXR + k)] = XR[k];
          s0p[M::q(M::QYR + k)] = YR[k];
        }
        // corners: a face state of the edge's a axis extrapolated along b
        auto corner = [&](const T *Wa, const T *db, bool bp, int va, int vb, int ba, int bb, T o[3]) {
          auto at = [&](int k) -> T { return bp ? up(Wa[k], db[k]) : dn(Wa[k], db[k]); };
          const T a = at(ba), b = at(bb);
          if constexpr (kFast) o[0] = fast::fm(-at(va), b, at(vb) * a);
          else o[0] = at(vb) * a - at(va) * b;
          o[1] = a;
          o[2] = b;
        };
        auto put3 = [&](int k0, const T o[3], T *const b) {
#pragma unroll
          for (int k = 0; k < 3; k++) b[M::q(k0 + k)] = o[k];
        };
        T *const bp_ = s0p + par * M::q(M::PSTEP);
        T o[3];
        // z-edges: a = x, b = y
        corner(XR, dY, true, VX, VY, BX, BY, o);
        put3(M::QZC, o, s0p);
        corner(xr, dY, true, VX, VY, BX, BY, o);
        put3(M::QZC + 3, o, s0p);
        corner(XR, dY, false, VX, VY, BX, BY, o);
        put3(M::QZC + 6, o, s0p);
        corner(xr, dY, false, VX, VY, BX, BY, cz0);
        // x-edges: a = y, b = z
        corner(YR, dZ, false, VY, VZ, BY, BZ, o);
        put3(M::QXM, o, s0p);
        corner(YR, dZ, true, VY, VZ, BY, BZ, o);
        put3(M::QXP, o, bp_);
        corner(yr, dZ, true, VY, VZ, BY, BZ, cxn);
        corner(yr, dZ, false, VY, VZ, BY, BZ, cx0);
        // y-edges: a = z, b = x
        corner(ZR, dX, true, VZ, VX, BZ, BX, o);
        put3(M::QYM, o, s0p);
        corner(ZU, dX, true, VZ, VX, BZ, BX, o);
        put3(M::QYP, o, bp_);
        corner(ZU, dX, false, VZ, VX, BZ, BX, cyn);
        corner(ZR, dX, false, VZ, VX, BZ, BX, cy0);
        // the z-face at p-1/2 needs this column alone
        if (it > 0 && zf) {
          face_of(std::integral_constant<int, 2>{}, zp, ZR, incol, fz, sz);
          s0p[M::q(M::QSZ)] = sz[0];
          s0p[M::q(M::QSZ + 1)] = sz[1];
        }
#pragma unroll
        for (int k = 0; k < 8; k++) zp[k] = ZU[k];
      } else if (it == -1) {
#pragma unroll
        for (int k = 0; k < 8; k++) zdl[k] = wn[k] - w0[k];
      }
#pragma unroll
      for (int k = 0; k < 3; k++) fd[k] = fn[k];
    }
    __syncthreads();

    // ---- 2: the next plane's primitives
    if (h1 && it >= -2 && it <= nt_) {
#pragma unroll
      for (int k = 0; k < 8; k++) s0p[M::q(M::QW + k)] = wn[k];
    }
    // the new cells' signal speeds (plane p-2).  Only their maximum counts:
    // FP64 bounds each in FP32 and evaluates, after the next barrier, those
    // that may exceed the largest lower bound so far
    float above = 0.f;
    if (it >= 3) {
      if constexpr (sizeof(T) == 4) {
        if (incol) signal_new(p - 2);
      } else if (tid < M::NTILE) {
        float below = 0.f;
        if (incol) {
          T un[5];
#pragma unroll
          for (int k = 0; k < 5; k++) un[k] = s0p[M::q(M::QU + k)];
          fast::signal_bounds(un, s0p[M::q(M::QNB)], s0p[M::q(M::QNB) + 1], s0p[M::q(M::QNB + 1)],
                              s0p[M::q(M::QNB + 1) + PITCH], nfzl, nfzh, gamma32, above, below);
        }
        const int most = __reduce_max_sync(0xffffffffu, __float_as_int(fmaxf(below, 0.f)));
        if ((tid & 31) == 0 && most > S.least) atomicMax(&S.least, most);
      }
    }
    // fluxes and speeds of the low faces
    if (it >= 0 && it <= nt_ && xf) {
      T L8[8];
#pragma unroll
      for (int k = 0; k < 8; k++) L8[k] = s0p[M::q(M::QXR + k) - 1];
      face_of(std::integral_constant<int, 0>{}, L8, xr, xfull && flux, fx, sx);
      s0p[M::q(M::QSX)] = sx[0];
      s0p[M::q(M::QSX + 1)] = sx[1];
      if (xfull && flux) {
#pragma unroll
        for (int k = 0; k < 5; k++) s0p[M::q(M::QFX + k)] = fx[k];
      }
    }
    if (it >= 0 && it <= nt_ && yf) {
      T L8[8];
#pragma unroll
      for (int k = 0; k < 8; k++) L8[k] = s0p[M::q(M::QYR + k) - PITCH];
      face_of(std::integral_constant<int, 1>{}, L8, yr, yfull && flux, fy, sy);
      s0p[M::q(M::QSY)] = sy[0];
      s0p[M::q(M::QSY + 1)] = sy[1];
      if (yfull && flux) {
#pragma unroll
        for (int k = 0; k < 5; k++) s0p[M::q(M::QFY + k)] = fy[k];
      }
    }
    // loads of plane p+2, of plane p+1 of the ring and of the old values to
    // update: used after the next barrier
    T ou[5], obx = T(0), oby = T(0), obz = T(0), dun[5];
    const bool upd = it >= 2 && it <= nt_;
    const long long orow = (long long)(p - 1) * ny + y;
    if (upd) {
      if (incol) {
#pragma unroll
        for (int k = 0; k < 5; k++) ou[k] = *src(own + k * nc + orow * nx + x);
      }
      if (xfull) obx = *src(own + ofx + orow * (nx + 1) + x);
      if (yfull) oby = *src(own + ofy + (orow + (p - 1)) * nx + x);
    }
    if (it > 0 && it <= nt_ && incol) obz = *src(own + ofz + (orow + ny) * nx + x);
    T qu[5], qf[6];
    T bxe = T(0), bye = T(0);  // the ring's low faces that the halo's columns take as their high ones
    if (h1 && it <= tz) {
      if (it == -3) fzl = face(2, x, y, p + 2);
      load_cell(x, y, ownxy, p + 2, ru, rfx, rfy, rfz);
    }
    if (ring) {
      if (it >= -2 && it <= tz) {
        load_cell(rx, ry, rown, p + 1, qu, qf[0], qf[2], qf[5]);
        qf[1] = face(0, rx + 1, ry, p + 1);
        qf[3] = face(1, rx, ry + 1, p + 1);
        qf[4] = face(2, rx, ry, p + 1);
      }
      if (it <= tz && ri == tx + 1) bxe = face(0, rx, ry, p + 2);
      if (it <= tz && rj == ty + 1) bye = face(1, rx, ry, p + 2);
    }
    __syncthreads();

    // ---- 3: edge EMFs and in-plane divergence
    if constexpr (sizeof(T) == 8) {
      if (it >= 3 && incol && !(above < __int_as_float(S.least))) signal_new(p - 2);
    }
    auto emf_of = [&](T ell, T erl, T elr, T err, T all, T arl, T alr, T arr, T bll, T brl, T blr, T brr, T apa, T ama,
                      T apb, T amb) -> T {
      if constexpr (kFast)
        return fast::emf(ell, erl, elr, err, all, arl, alr, arr, bll, brl, blr, brr, apa, ama, apb, amb);
      else return emf(ell, erl, elr, err, all, arl, alr, arr, bll, brl, blr, brr, apa, ama, apb, amb);
    };
    T exn = T(0), eyn = T(0), ezn = T(0);
    if (it > 0 && it <= nt_) {
      if (ex_) {
        // LL and LR from the column at -y, RL and RR this column's
        const T *const m = s0p - PITCH;
        const T *const pl = m + (par ^ 1) * M::q(M::PSTEP);
        const T apa = pmax0(syp[1], sy[1]), ama = nmax0(syp[0], sy[0]);
        const T apb = pmax0(m[M::q(M::QSZ + 1)], sz[1]), amb = nmax0(m[M::q(M::QSZ)], sz[0]);
        exn = emf_of(pl[M::q(M::QXP)], cxo[0], m[M::q(M::QXM)], cx0[0], pl[M::q(M::QXP + 1)], cxo[1],
                     m[M::q(M::QXM + 1)], cx0[1], pl[M::q(M::QXP + 2)], cxo[2], m[M::q(M::QXM + 2)], cx0[2], apa, ama,
                     apb, amb);
        s0p[M::q(M::QE)] = exn;
      }
      if (ey_) {
        // LL and RL from the column at -x, LR and RR this column's
        const T *const m = s0p - 1;
        const T *const pl = m + (par ^ 1) * M::q(M::PSTEP);
        const T apa = pmax0(m[M::q(M::QSZ + 1)], sz[1]), ama = nmax0(m[M::q(M::QSZ)], sz[0]);
        const T apb = pmax0(sxp[1], sx[1]), amb = nmax0(sxp[0], sx[0]);
        eyn = emf_of(pl[M::q(M::QYP)], m[M::q(M::QYM)], cyo[0], cy0[0], pl[M::q(M::QYP + 1)], m[M::q(M::QYM + 1)],
                     cyo[1], cy0[1], pl[M::q(M::QYP + 2)], m[M::q(M::QYM + 2)], cyo[2], cy0[2], apa, ama, apb, amb);
        s0p[M::q(M::QE + 1)] = eyn;
      }
      if (ez_ && flux) {
        const T *const ll = s0p - PITCH - 1, *const rl = s0p - PITCH, *const lr = s0p - 1;
        const T apa = pmax0(rl[M::q(M::QSX + 1)], sx[1]), ama = nmax0(rl[M::q(M::QSX)], sx[0]);
        const T apb = pmax0(lr[M::q(M::QSY + 1)], sy[1]), amb = nmax0(lr[M::q(M::QSY)], sy[0]);
        ezn = emf_of(ll[M::q(M::QZC)], rl[M::q(M::QZC + 3)], lr[M::q(M::QZC + 6)], cz0[0], ll[M::q(M::QZC + 1)],
                     rl[M::q(M::QZC + 4)], lr[M::q(M::QZC + 7)], cz0[1], ll[M::q(M::QZC + 2)], rl[M::q(M::QZC + 5)],
                     lr[M::q(M::QZC + 8)], cz0[2], apa, ama, apb, amb);
        s0p[M::q(M::QE + 2)] = ezn;
      }
      if (incol && flux) {
#pragma unroll
        for (int k = 0; k < 5; k++)
          dun[k] = (s0p[M::q(M::QFX + k) + 1] - fx[k]) + (s0p[M::q(M::QFY + k) + PITCH] - fy[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 3; k++) {
      cxo[k] = cxn[k];
      cyo[k] = cyn[k];
    }
#pragma unroll
    for (int k = 0; k < 2; k++) {
      sxp[k] = sx[k];
      syp[k] = sy[k];
    }
    if (it <= tz) {
      if (h1) {
        s0p[M::q(M::QB)] = rfx;
        s0p[M::q(M::QB + 1)] = rfy;
      }
      if (ring) {
        if (it >= -2) {
          T W[8];
          prim_of(qu, qf[0], qf[1], qf[2], qf[3], qf[4], qf[5], W, nullptr);
#pragma unroll
          for (int k = 0; k < 8; k++) r0p[M::q(M::QW + k)] = W[k];
        }
        if (ri == tx + 1) r0p[M::q(M::QB)] = bxe;
        if (rj == ty + 1) r0p[M::q(M::QB + 1)] = bye;
      }
    }
    __syncthreads();

    // ---- the update of plane p-1 and of the z-faces at p-1/2
    auto less = [&](T a, T r) -> T { return kFast ? fast::fm(-dtdx, r, a) : a - dtdx * r; };
    if (upd) {
      if (xfull) {
        const T nfx = less(obx, dey - (eyn - eyp_));
        s0p[M::q(M::QNB)] = nfx;
        put_global(dst + ofx + orow * (nx + 1) + x, nfx);
      }
      if (yfull) {
        const T nfy = less(oby, (exn - exp_) - dex);
        s0p[M::q(M::QNB + 1)] = nfy;
        put_global(dst + ofy + (orow + (p - 1)) * nx + x, nfy);
      }
    }
    if (it > 0 && it <= nt_ && incol) {
      nfzl = nfzh;
      nfzh = less(obz, (s0p[M::q(M::QE + 1) + 1] - eyn) - (s0p[M::q(M::QE) + PITCH] - exn));
      put_global(dst + ofz + (orow + ny) * nx + x, nfzh);
      if (upd) {
#pragma unroll
        for (int k = 0; k < 5; k++) {
          const T un = less(ou[k], du[k] + (fz[k] - fzp[k]));
          s0p[M::q(M::QU + k)] = un;
          put_global(dst + k * nc + orow * nx + x, un);
        }
      }
    }
    if (flux) {
      if (xfull) dey = s0p[M::q(M::QE + 2) + PITCH] - ezn;
      if (yfull) dex = s0p[M::q(M::QE + 2) + 1] - ezn;
    }
    exp_ = exn;
    eyp_ = eyn;
#pragma unroll
    for (int k = 0; k < 5; k++) {
      fzp[k] = fz[k];
      du[k] = dun[k];
    }
  }
  // signal speed of the new slice: block max, then the patch max
  double v = (double)smax_t;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((tid & 31) == 0) S.red[tid >> 5] = v;
  __syncthreads();
  if (tid < 32) {
    double u = tid < NT / 32 ? S.red[tid] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) u = fmax(u, __shfl_xor_sync(0xffffffffu, u, o));
    if (tid == 0) {
      atomicMax(&c.smax_new[P], (unsigned long long)__double_as_longlong(u));
      if (S.fallback) atomicAdd((unsigned long long *)&c.cnt[CNT_FALLBACKS], (unsigned long long)S.fallback);
      if (S.floors) atomicAdd((unsigned long long *)&c.cnt[CNT_FLOORS], (unsigned long long)S.floors);
    }
  }
  __syncthreads();
}

}  // namespace dsp
