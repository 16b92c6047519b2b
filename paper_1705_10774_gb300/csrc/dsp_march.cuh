// dsp_march.cuh -- the update of one tile by threads that own columns.
//
// A tile is TX x TY columns of cells and a run of tz planes.  One thread
// owns one column of the tile or of the one-cell halo around it and marches
// it through the planes; a column's own data along z (its cells' primitive
// state, slopes, upper z-face state, z-flux, carried corners, old speeds and
// EMFs) never leaves the thread, and shared memory carries only what a
// neighbouring column needs.  Per plane p, three barriers:
//   1  the z-face flux at p-1/2; the conservative and constrained-transport
//      update of plane p-1 (whose EMFs the last barrier published); primitives
//      of plane p+1 from the values loaded one plane earlier (the high faces
//      from the columns at +x and +y); MC slopes and the Hancock predictor of
//      plane p; the face states and edge corners that the columns at +x and
//      +y will read
//   2  primitives of plane p+1 published; the fluxes and speeds of the faces
//      on the column's low side (x, y); the new cells' signal speeds; at its
//      end the loads of plane p+2, of the ring around the halo in plane p+1
//      and of the old values to update are started
//   3  edge EMFs on the column's low edges (x and y at p-1/2, z in plane p),
//      the in-plane flux divergence; the loads have arrived: values between
//      two times blended, the ring's primitives and the faces of plane p+2
//      published
// The first three iterations only fill this pipeline.
// What bounds it: in FP64 the FP64 pipe (an FP64 warp instruction takes its
// slot whatever its active lanes, one per 19 clocks of an SM), so whole warps
// hold tile columns, and the halo's columns are dealt so that those with
// fluxes share one warp and those with speeds alone another; in FP32 the issue
// slots and the latency of a column's chains, so a thread's positions are
// fixed for the whole tile and every shared address is one base plus a
// constant.  Measured, 256^3 in 32^3 patches, a sweep: FP64 with FMA 50.7 ms
// for the block marching phase by phase over shared planes, 36.4 so (76 % of
// the FP64 pipe's slots, where 84 % can be had; 930 FP64 operations a cell
// instead of 1530; 79 GB/s of algorithmic traffic); without FMA 78.3 and 68.1;
// FP32 4.33 and 2.53 (84 instead of 166 warp instructions a cell, 47 % of the
// issue slots, 567 GB/s).
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
  static constexpr int QU = 72;    // [5] the cell just updated, and its old values (its own thread's)
  // FP32: raw values of the plane to come [rho, m, E, x-, y-face below, z-face
  // above], copied here asynchronously, the old faces of the update and, where
  // two blocks need not share an SM, the state at the upper z-face of the
  // previous plane; FP64 holds these in registers and publishes the two faces
  static constexpr bool SL = sizeof(T) == 4;
  static constexpr int QRAW = 78;  // [8]
  static constexpr int QOF = 86;   // [3]
  static constexpr int QZP = 90;   // [8]
  static constexpr bool SZP = SL && !PAIR;
  static constexpr int QB = SL ? QRAW + 5 : 77;  // [2] x- and y-faces of the plane to come
  static constexpr int NQ1 = !SL ? 80 : SZP ? 98 : 90;
  // tiles that have an SM to themselves: the second slice's values of a column
  // blended in time, copied like the first's (the bounds-checked build: in its
  // one FP32 tile, so that these copies' addresses are tested too)
#ifdef DSP_BOUNDS_CHECK
  static constexpr bool DB = SL;
#else
  static constexpr bool DB = SL && (PAIR ? NQ1 / 2 : NQ1) * PLANE * sizeof(T) > 110000;
#endif
  static constexpr int QRB = NQ1;  // [8] (a ring column's: its places from QXR + 11 on)
  static constexpr int NQ = NQ1 + (DB ? 8 : 0);
  static constexpr int total = (PAIR ? NQ / 2 : NQ) * PLANE;
  // threads: the tile's columns, the halo columns with fluxes (right column,
  // top row), then the other halo columns (bottom row, left column, corners);
  // the ring around the halo (primitives only) is dealt to the halo's threads
  static constexpr int NTILE = TX * TY;
  // (from the next warp on, unless packing them saves a warp)
  static constexpr int NHA = TX + TY, NHB = TX + TY + 4, RND = (NHA + 31) / 32 * 32;
  static constexpr int HB0 = NTILE + ((RND + NHB + 31) / 32 > (NHA + NHB + 31) / 32 ? NHA : RND);
  static constexpr int NEED = HB0 + NHB;
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
  const int my_blend = owner_table<T, NT, CONC>(c, P, lev, tP, bx0, by0, bz0, nbx, nby, nbz, S);
  if (tid == 0) {
    S.fallback = 0;
    S.floors = 0;
    S.least = 0;
  }
  const int any_blend = __syncthreads_or(my_blend);  // some neighbour is not at the patch's time

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
  // a warp with any flux computes fluxes in all its faces' lanes at once
  const bool xw = __any_sync(0xffffffffu, xfull), yw = __any_sync(0xffffffffu, yfull);
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
  const int edge_ax = !ring ? -1 : ri == tx + 1 ? 0 : rj == ty + 1 ? 1 : -1;
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
  // a table entry's value: from one slice (bl = 0), or blended from two or three
  auto value = [&](const T *p, int bl, int e) -> T {
    T a = *src(p);
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
  // where a value lives: its address in a slice, blend code and table entry
  struct Loc {
    const T *p;
    int bl, e;
  };
  auto get = [&](const Loc &l) -> T { return value(l.p, l.bl, l.e); };
  // Table entries of a column, its +x and its +y neighbour in the lowest layer
  // of map blocks (a byte each); the layer of a plane.
  const int nbxy = nbx * nby;
  auto layer = [&](int z) -> int { return (__float2int_rd(((float)(loz + z) + 0.5f) * binv[2]) - bz0) * nbxy; };
  auto entries = [&](int xx, int yy) -> int {
    return entry(lox + xx, loy + yy, bz0 * bsz[2]) | entry(lox + xx + 1, loy + yy, bz0 * bsz[2]) << 8 |
           entry(lox + xx, loy + yy + 1, bz0 * bsz[2]) << 16;
  };
  // a patch seen from patch cell (xx, yy, zz): the patch itself, or the one of
  // table entry e (chosen by selects: the halo's warps mix both)
  struct View {
    const T *A;
    int mx, my, mz, lx, ly, lz, bl, e;
  };
  auto view = [&](bool mine, int e, int xx, int yy, int zz) -> View {
    const int4 n = S.nb[e], l = S.lo4[e];
    View v;
    v.A = mine ? own : srcA[e];
    v.mx = mine ? nx : n.x;
    v.my = mine ? ny : n.y;
    v.mz = mine ? nz : n.z;
    v.lx = mine ? xx : lox + xx - l.x;
    v.ly = mine ? yy : loy + yy - l.y;
    v.lz = mine ? zz : loz + zz - l.z;
    v.bl = mine ? 0 : n.w;
    v.e = e;
    return v;
  };
  // the face along ax on the low side of the view's cell
  auto face_at = [&](int ax, const View &v) -> Loc {
    const long long m = (long long)v.mx * v.my * v.mz;
    long long o = 5 * m;
    if (ax >= 1) o += (long long)(v.mx + 1) * v.my * v.mz;
    if (ax == 2) o += (long long)v.mx * (v.my + 1) * v.mz;
    return {v.A + o + ((long long)v.lz * (v.my + (ax == 1)) + v.ly) * (v.mx + (ax == 0)) + v.lx, v.bl, v.e};
  };
  // whether the face along ax on the low side of patch cell (xx, yy, zz) is
  // the patch's own: it lies on one of its interior cells
  auto own_face = [&](int ax, int xx, int yy, int zz) -> bool {
    return xx >= 0 && xx < nx + (ax == 0) && yy >= 0 && yy < ny + (ax == 1) && zz >= 0 && zz < nz + (ax == 2);
  };
  // that face: the patch's own, else that of the patch that owns the cell (ent:
  // the column's table entry in the lowest layer)
  auto face = [&](int ax, int ent, int xx, int yy, int zz) -> Loc {
    return face_at(ax, view(own_face(ax, xx, yy, zz), ent + layer(zz), xx, yy, zz));
  };
  // Hands to `to` (value number, place) the five conserved values of patch
  // cell (xx, yy, q), its low x- and y-faces (5, 6) and its high z-face (7);
  // for a ring column (RING) also its high x- and y-faces and its low z-face.
  // Straight-line code: with a branch for every own or foreign value, and a
  // lookup and a blend test for each, the halo's warps took 4800 clocks a
  // plane here where the tile's took 1350, and every warp waited for them
  // (3700 now; 256^3 in FP32: 2.87 -> 2.67 ms a sweep).  Addresses kept and
  // stepped from plane to plane, in shared or in local memory, took longer.
  auto load_cell = [&](auto rr, int ents, int xx, int yy, bool inxy, int q, auto to) {
    constexpr bool RING = decltype(rr)::value;
    const bool zin = q >= 0 && q < nz;
    if (__all_sync(__activemask(), inxy && zin)) {
      const long long o = ((long long)q * ny + yy) * nx + xx;
      const T *const a = own + o;
#pragma unroll
      for (int k = 0; k < 5; k++) to(k, Loc{a + k * nc, 0, 0});
      const T *const ax = a + ofx + ((long long)q * ny + yy), *const ay = a + ofy + (long long)q * nx, *const az = a + ofz;
      to(5, Loc{ax, 0, 0});
      to(6, Loc{ay, 0, 0});
      to(7, Loc{az + (long long)nx * ny, 0, 0});
      if constexpr (RING) {
        to(8, Loc{ax + 1, 0, 0});
        to(9, Loc{ay + nx, 0, 0});
        to(10, Loc{az, 0, 0});
      }
      return;
    }
    const int ent = (ents & 255), e = ent + layer(q);
    const View v = view(inxy && zin, e, xx, yy, q);
    const long long m = (long long)v.mx * v.my * v.mz;
    const T *const a = v.A + ((long long)v.lz * v.my + v.ly) * v.mx + v.lx;
#pragma unroll
    for (int k = 0; k < 5; k++) to(k, Loc{a + k * m, v.bl, e});
    to(5, face_at(0, view(own_face(0, xx, yy, q), e, xx, yy, q)));
    to(6, face_at(1, view(own_face(1, xx, yy, q), e, xx, yy, q)));
    to(7, face(2, ent, xx, yy, q + 1));
    if constexpr (RING) {
      to(8, face(0, ents >> 8 & 255, xx + 1, yy, q));
      to(9, face(1, ents >> 16, xx, yy + 1, q));
      to(10, face(2, ent, xx, yy, q));
    }
  };
  // The values of load_cell into shared memory, place(k): plain copies are
  // asynchronous (no register is held, and no branch taken, while they are in
  // flight).  Values blended from two slices: both are copied, the second to
  // second(k), and the thread blends them once they have arrived (bits of the
  // result: which values; entry e of value k in byte k < 7 or 10: 0, 7: 1, 8:
  // 2, 9: 3 of `es`); waiting for each in turn took a third of a pass of
  // local steps on 256^3 (51.0 ms, now 35.2).  Without room for that, and with
  // three slices, they are loaded here.  The ready queue copies too: the
  // slices a tile reads were published before its ticket, and none of them is
  // overwritten while the patch is behind (216 patches of 32^3 with local
  // steps: 25.5 ms with plain loads, one waiting for the other, now 13.1).
  auto stage = [&](auto rr, int ents, int xx, int yy, bool inxy, int q, auto place, auto second, int &es) -> int {
    int mask = 0;
    if (!any_blend) {
      load_cell(rr, ents, xx, yy, inxy, q, [&](int k, const Loc &l) { cp_async_elem(place(k), src(l.p)); });
    } else {
      int late = 0;
      es = 0;
      load_cell(rr, ents, xx, yy, inxy, q, [&](int k, const Loc &l) {
        const bool two = M::DB && (l.bl & 3) == 2;
        cp_async_if(place(k), src(l.p), l.bl == 0 || two);
        if constexpr (M::DB) {
          cp_async_if(second(k), src(l.p + (long long)(two ? (l.bl >> 2 & 63) - 16 : 0) * c.slot_stride), two);
          mask |= two ? 1 << k : 0;
          if (k == 0 || (k >= 7 && k < 10)) es |= l.e << (k == 0 ? 0 : 8 * (k - 6));
        }
        late |= l.bl != 0 && !two;
      });
      if (__any_sync(__activemask(), late))
        load_cell(rr, ents, xx, yy, inxy, q, [&](int k, const Loc &l) {
          if (l.bl && !(M::DB && (l.bl & 3) == 2)) *place(k) = get(l);
        });
    }
    return mask;
  };
  auto blend = [&](auto nk, int mask, int es, auto place, auto second) {
    if constexpr (M::DB) {
      constexpr int NK = decltype(nk)::value;
      if (mask) {
#pragma unroll
        for (int k = 0; k < NK; k++) {
          const T a = *place(k), w = S.wgt[0][es >> (k >= 7 && k < 10 ? 8 * (k - 6) : 0) & 255];
          if (mask >> k & 1) *place(k) = a + w * (*second(k) - a);
        }
      }
    }
  };
  auto copy_to = [&](T *d, const Loc &l) {
    if (l.bl == 0) cp_async_elem(d, src(l.p));
    else *d = get(l);
  };
  auto prim_of = [&](const T u[5], T fxl, T fxh, T fyl, T fyh, T fzl, T fzh, T W[8], int *floored) {
    if constexpr (kFast) fast::prim(u[0], u[1], u[2], u[3], u[4], fxl, fxh, fyl, fyh, fzl, fzh, gm1, W, floored);
    else prim(u[0], u[1], u[2], u[3], u[4], fxl, fxh, fyl, fyh, fzl, fzh, gamma, W, floored);
  };
  // a cell state plus or minus half a slope (held as the half slope in the
  // fast forms)
  auto up = [&](T w, T d) -> T { return kFast ? w + d : w + half * d; };
  auto dn = [&](T w, T d) -> T { return kFast ? w - d : w - half * d; };

  const int ents = entries(x, y), rents = ring ? entries(rx, ry) : 0;

  // places of the column's and the ring column's values (a ring column's in
  // planes that only the halo's columns use)
  auto raw_at = [&](int k) { return s0p + M::q(M::QRAW + k); };
  auto raw2_at = [&](int k) { return s0p + M::q(M::QRB + k); };
  auto ring_at = [&](int k) { return r0p + M::q(M::QXR + k); };
  auto ring2_at = [&](int k) { return r0p + M::q(M::QXR + 11 + k); };

  // raw values of the next plane and the z-face below it
  T raw[8];  // FP64 only
  T fzl = T(0);
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
        if constexpr (M::SL) {
#pragma unroll
          for (int k = 0; k < 8; k++) raw[k] = s0p[M::q(M::QRAW + k)];
        }
        prim_of(raw, raw[5], fxh, raw[6], fyh, fzl, raw[7], wn, nullptr);
        fn[0] = fxh - raw[5];
        fn[1] = fyh - raw[6];
        fn[2] = raw[7] - fzl;
        fzl = raw[7];
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
        T o[3], U_[8], ZR[8];
        // x-face states, z-edges (a = x, b = y)
#pragma unroll
        for (int k = 0; k < 8; k++) {
          U_[k] = up(ws[k], dX[k]);
          xr[k] = dn(ws[k], dX[k]);
          s0p[M::q(M::QXR + k)] = U_[k];
        }
        corner(U_, dY, true, VX, VY, BX, BY, o);
        put3(M::QZC, o, s0p);
        corner(xr, dY, true, VX, VY, BX, BY, o);
        put3(M::QZC + 3, o, s0p);
        corner(U_, dY, false, VX, VY, BX, BY, o);
        put3(M::QZC + 6, o, s0p);
        corner(xr, dY, false, VX, VY, BX, BY, cz0);
        // y-face states, x-edges (a = y, b = z)
#pragma unroll
        for (int k = 0; k < 8; k++) {
          U_[k] = up(ws[k], dY[k]);
          yr[k] = dn(ws[k], dY[k]);
          s0p[M::q(M::QYR + k)] = U_[k];
        }
        corner(U_, dZ, false, VY, VZ, BY, BZ, o);
        put3(M::QXM, o, s0p);
        corner(U_, dZ, true, VY, VZ, BY, BZ, o);
        put3(M::QXP, o, bp_);
        corner(yr, dZ, true, VY, VZ, BY, BZ, cxn);
        corner(yr, dZ, false, VY, VZ, BY, BZ, cx0);
        // z-face states, y-edges (a = z, b = x)
#pragma unroll
        for (int k = 0; k < 8; k++) {
          U_[k] = up(ws[k], dZ[k]);
          ZR[k] = dn(ws[k], dZ[k]);
        }
        corner(ZR, dX, true, VZ, VX, BZ, BX, o);
        put3(M::QYM, o, s0p);
        corner(U_, dX, true, VZ, VX, BZ, BX, o);
        put3(M::QYP, o, bp_);
        corner(U_, dX, false, VZ, VX, BZ, BX, cyn);
        corner(ZR, dX, false, VZ, VX, BZ, BX, cy0);
        // the z-face at p-1/2 needs this column alone
        if (it > 0 && zf) {
          if constexpr (M::SZP) {
#pragma unroll
            for (int k = 0; k < 8; k++) zp[k] = s0p[M::q(M::QZP + k)];
          }
          face_of(std::integral_constant<int, 2>{}, zp, ZR, incol, fz, sz);
          s0p[M::q(M::QSZ)] = sz[0];
          s0p[M::q(M::QSZ + 1)] = sz[1];
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
          if constexpr (M::SZP) s0p[M::q(M::QZP + k)] = U_[k];
          else zp[k] = U_[k];
        }
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
                              s0p[M::q(M::QNB + 1) + PITCH], nfzl, nfzh, c.gamma32, c.gm132, above, below);
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
      face_of(std::integral_constant<int, 0>{}, L8, xr, xw && flux, fx, sx);
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
      face_of(std::integral_constant<int, 1>{}, L8, yr, yw && flux, fy, sy);
      s0p[M::q(M::QSY)] = sy[0];
      s0p[M::q(M::QSY + 1)] = sy[1];
      if (yfull && flux) {
#pragma unroll
        for (int k = 0; k < 5; k++) s0p[M::q(M::QFY + k)] = fy[k];
      }
    }
    // loads of plane p+2, of plane p+1 of the ring and of the old values to
    // update: used after the next barrier.  (FP32: they overwrite the updated
    // cell that signal_new has just read.)
    if constexpr (M::SL) cp_async_after_reads();
    const bool upd = it >= 2 && it <= nt_;
    const long long orow = (long long)(p - 1) * ny + y;
    int hm = 0, rm = 0, hes = 0, res = 0, ee = -1;  // blended values on their way
    T dun[5];
    T ou[5], of[3], ring_raw[11], edge = T(0);  // FP64 only
    if (upd) {
      if (incol) {
        const T *const a = own + orow * nx + x;
#pragma unroll
        for (int k = 0; k < 5; k++) {
          if constexpr (M::SL) copy_to(s0p + M::q(M::QU + k), Loc{a + k * nc, 0, 0});
          else ou[k] = *src(a + k * nc);
        }
      }
      if (xfull) {
        const T *const a = own + ofx + orow * (nx + 1) + x;
        if constexpr (M::SL) copy_to(s0p + M::q(M::QOF), Loc{a, 0, 0});
        else of[0] = *src(a);
      }
      if (yfull) {
        const T *const a = own + ofy + (orow + (p - 1)) * nx + x;
        if constexpr (M::SL) copy_to(s0p + M::q(M::QOF + 1), Loc{a, 0, 0});
        else of[1] = *src(a);
      }
    }
    if (it > 0 && it <= nt_ && incol) {
      const T *const a = own + ofz + (orow + ny) * nx + x;
      if constexpr (M::SL) copy_to(s0p + M::q(M::QOF + 2), Loc{a, 0, 0});
      else of[2] = *src(a);
    }
    if (h1 && it <= tz) {
      if (it == -3) fzl = get(face(2, ents & 255, x, y, p + 2));
      if constexpr (M::SL)
        hm = stage(std::false_type{}, ents, x, y, ownxy, p + 2, raw_at, raw2_at, hes);
      else
        load_cell(std::false_type{}, ents, x, y, ownxy, p + 2, [&](int k, const Loc &l) { raw[k] = get(l); });
    }
    if (ring) {
      // (FP32: at the ring's places in planes that only the halo's columns use)
      if (it >= -2 && it <= tz) {
        if constexpr (M::SL)
          rm = stage(std::true_type{}, rents, rx, ry, rown, p + 1, ring_at, ring2_at, res);
        else
          load_cell(std::true_type{}, rents, rx, ry, rown, p + 1, [&](int k, const Loc &l) { ring_raw[k] = get(l); });
      }
      // the low face that a halo column takes as its high one
      if (it <= tz && edge_ax >= 0) {
        const Loc l = face(edge_ax, rents & 255, rx, ry, p + 2);
        if constexpr (M::SL) {
          T *const d = r0p + (edge_ax == 0 ? M::q(M::QB) : M::q(M::QB + 1));
          if (M::DB && (l.bl & 3) == 2) {
            cp_async_elem(d, src(l.p));
            cp_async_elem(r0p + M::q(M::QRB), src(l.p + (long long)((l.bl >> 2 & 63) - 16) * c.slot_stride));
            ee = l.e;
          } else {
            copy_to(d, l);
          }
        } else {
          edge = get(l);
        }
      }
    }
    if constexpr (M::SL) cp_async_commit();
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
    if (it >= 0 && it <= nt_) {  // the column's own speeds, from where phase 2 put them
#pragma unroll
      for (int k = 0; k < 2; k++) {
        sx[k] = s0p[M::q(M::QSX + k)];
        sy[k] = s0p[M::q(M::QSY + k)];
        sz[k] = s0p[M::q(M::QSZ + k)];
      }
    }
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
          dun[k] = (s0p[M::q(M::QFX + k) + 1] - s0p[M::q(M::QFX + k)]) +
                   (s0p[M::q(M::QFY + k) + PITCH] - s0p[M::q(M::QFY + k)]);
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
    if constexpr (M::SL) cp_async_wait<0>();
    if (it <= tz) {
      if (h1) blend(std::integral_constant<int, 8>{}, hm, hes, raw_at, raw2_at);
      if (ring) blend(std::integral_constant<int, 11>{}, rm, res, ring_at, ring2_at);
      if (M::DB && ee >= 0) {
        T *const d = r0p + (edge_ax == 0 ? M::q(M::QB) : M::q(M::QB + 1));
        *d = *d + S.wgt[0][ee] * (r0p[M::q(M::QRB)] - *d);
      }
    }
    if (it <= tz) {
      if constexpr (!M::SL) {
        if (h1) {
          s0p[M::q(M::QB)] = raw[5];
          s0p[M::q(M::QB + 1)] = raw[6];
        }
        if (edge_ax == 0) r0p[M::q(M::QB)] = edge;
        if (edge_ax == 1) r0p[M::q(M::QB + 1)] = edge;
      }
      if (ring && it >= -2) {
        T W[8];
        if constexpr (M::SL) {
#pragma unroll
          for (int k = 0; k < 11; k++) ring_raw[k] = r0p[M::q(M::QXR + k)];
        }
        prim_of(ring_raw, ring_raw[5], ring_raw[8], ring_raw[6], ring_raw[9], ring_raw[10], ring_raw[7], W, nullptr);
#pragma unroll
        for (int k = 0; k < 8; k++) r0p[M::q(M::QW + k)] = W[k];
      }
    }
    __syncthreads();

    // ---- the update of plane p-1 and of the z-faces at p-1/2
    auto less = [&](T a, T r) -> T { return kFast ? fast::fm(-dtdx, r, a) : a - dtdx * r; };
    if constexpr (M::SL) {  // copied by this thread
#pragma unroll
      for (int k = 0; k < 3; k++) of[k] = s0p[M::q(M::QOF + k)];
    }
    if (upd) {
      if (xfull) {
        const T nfx = less(of[0], dey - (eyn - eyp_));
        s0p[M::q(M::QNB)] = nfx;
        put_global(dst + ofx + orow * (nx + 1) + x, nfx);
      }
      if (yfull) {
        const T nfy = less(of[1], (exn - exp_) - dex);
        s0p[M::q(M::QNB + 1)] = nfy;
        put_global(dst + ofy + (orow + (p - 1)) * nx + x, nfy);
      }
    }
    if (it > 0 && it <= nt_ && incol) {
      nfzl = nfzh;
      nfzh = less(of[2], (s0p[M::q(M::QE + 1) + 1] - eyn) - (s0p[M::q(M::QE) + PITCH] - exn));
      put_global(dst + ofz + (orow + ny) * nx + x, nfzh);
      if (upd) {
#pragma unroll
        for (int k = 0; k < 5; k++) {
          const T un = less(M::SL ? s0p[M::q(M::QU + k)] : ou[k], du[k] + (fz[k] - fzp[k]));
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
