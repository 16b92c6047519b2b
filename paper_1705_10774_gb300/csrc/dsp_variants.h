// dsp_variants.h -- the compiled variants of the update kernel.
//
// Each row is compiled from dsp_variant.cu into its own object (the build
// reads this list): id, element type, tile TX x TY, threads per block,
// minimum resident blocks per SM, precision code of dsp_params (0 FP64
// without FMA, 1 FP32, 2 FP64 with FMA), Riemann solver of the face fluxes
// (0 HLL, 1 HLLD), non-ideal terms (1: the Ohmic and ambipolar EMFs).
// Ideal MHD has a thread per column of the tile and its halo, so the tile
// sets the block; wide tiles have less halo per cell (512^3 cells in 32^3
// patches, a sweep: FP64 with FMA 282 ms for 16 x 12, 323 for 16 x 8, 382 for
// 8 x 8; FP32 20.5 ms for 32 x 8, 22.2 for 16 x 16, 25.8 for two blocks of
// 16 x 8, 32.1 for one, 38.4 for 24 x 8, which 32^3 does not fit), small ones fit
// small patches.  The registers of a column (255 in FP64, 168 in FP32) set how
// many warps an SM holds.  The non-ideal tiles hold four planes of faces in
// shared memory, so the FP64 rows use a smaller one.  All variants of one
// precision, solver and physics compute bit-identical results; they differ
// only in how the work is spread over threads, so dsp_autotune may pick any of
// them.  The bounds-checked build (DSP_BOUNDS_CHECK) compiles the three rows
// of DSP_VARIANT_LIST_CHECKED only.
#pragma once

#define DSP_VARIANT_LIST_ALL(X)        \
  X(0, double, 16, 8, 192, 1, 0, 0, 0)    \
  X(2, double, 16, 8, 192, 1, 2, 0, 0)    \
  X(5, float, 16, 8, 192, 2, 1, 0, 0)     \
  X(6, float, 16, 8, 192, 1, 1, 0, 0)     \
  X(7, float, 32, 8, 352, 1, 1, 0, 0)     \
  X(8, float, 16, 16, 352, 1, 1, 0, 0)    \
  X(9, double, 16, 8, 192, 1, 0, 1, 0)    \
  X(10, double, 16, 8, 192, 1, 2, 1, 0)   \
  X(11, float, 16, 8, 192, 2, 1, 1, 0)  \
  X(12, double, 16, 4, 128, 1, 0, 0, 1) \
  X(13, double, 16, 4, 128, 1, 2, 0, 1) \
  X(14, float, 16, 8, 256, 1, 1, 0, 1) \
  X(15, double, 16, 4, 256, 1, 2, 0, 1) \
  X(16, float, 16, 4, 128, 2, 1, 0, 1) \
  X(17, double, 16, 4, 256, 1, 0, 0, 1) \
  X(18, double, 16, 4, 256, 1, 0, 1, 1) \
  X(19, double, 16, 4, 256, 1, 2, 1, 1) \
  X(20, float, 16, 8, 256, 1, 1, 1, 1)   \
  X(21, float, 24, 8, 288, 1, 1, 0, 0) \
  X(22, float, 32, 8, 352, 1, 1, 1, 0) \
  X(23, double, 8, 8, 128, 2, 0, 0, 0) \
  X(24, double, 8, 8, 128, 2, 2, 0, 0) \
  X(25, double, 16, 12, 256, 1, 2, 0, 0)

// Ids that callers may hold and whose form is another row's: the 16 x 8 tiles
// of FP64 with more threads than the tile and its halo have columns (384 and
// 512; the phase-by-phase kernel dealt its work to them).  A request for one
// gets the row's kernel under the requested id.
#define DSP_VARIANT_ALIASES(A) A(1, 0) A(3, 2) A(4, 2)

#define DSP_VARIANT_LIST_CHECKED(X)    \
  X(0, double, 16, 8, 192, 1, 0, 0, 0)    \
  X(2, double, 16, 8, 192, 1, 2, 0, 0)    \
  X(5, float, 16, 8, 192, 2, 1, 0, 0)

#ifdef DSP_BOUNDS_CHECK
#define DSP_VARIANT_LIST(X) DSP_VARIANT_LIST_CHECKED(X)
#else
#define DSP_VARIANT_LIST(X) DSP_VARIANT_LIST_ALL(X)
#endif
