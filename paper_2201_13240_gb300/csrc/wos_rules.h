// wos_rules.h -- which form of a kernel a call takes: rules on sizes, types and fields, apart from
// CUDA so that the host check library can be asked for them too.
#pragma once

#if defined(__CUDACC_RTC__)
#include "wos_math.cuh"  // fixed-width integer types of runtime compilation
#else
#include <stdint.h>
#endif

#if defined(__CUDACC__)
#define WOS_RULE __host__ __device__ constexpr
#else
#define WOS_RULE constexpr
#endif

namespace wos {

// A walk kernel's per-point sums: in FP64 as they come, or FP32 differences from the point's first walk.
// `gathers`: ended walks wait for each other and are finished `lanes` at a time.  Where six or eight
// are, two FP64 additions a walk cost less than the shift (a batch 46.2 -> 45.3 ms, the 2D square 4.48
// -> 4.37; at four the 3D cube 109.8 -> 110.2 ms), and the shifted FP32 sums lose digits when a point's
// first walk is an outlier of a heavy-tailed estimate.  Window and mesh walks end one by one, whatever
// the number of lanes that their problem's other kernels gather: FP32.
WOS_RULE bool sums_in_fp64(bool grad, bool gathers, int lanes) { return grad || (gathers && lanes >= 6); }

// The item of a lane's walk, for the per-walk outputs: carried (two registers), or found again from its
// point and walk id where eight lanes are gathered, that is where the fields need the registers (B-spline
// fields 7.57 -> 7.43 ms; the 3D cube 109.7 -> 111.2).
WOS_RULE bool finds_item_again(bool gathers, int lanes) { return gathers && lanes >= 8; }

// Largest launch (walks) that takes the per-walk buffers of a small solve (16 MB per context): about
// ten walks for each lane of the chip; a larger launch keeps every lane busy by itself (1.67e6
// walks: 1.02 ms either way).
constexpr uint64_t kSpreadItems = 1ull << 20;

// The rounding that a gradient walk's kernel names in the Green's-function norm (green_q3's FORM): the one
// that kernels of its kind have always had, so that their walks stay the same.  Compiled kernels of
// closed-form fields: 2; generic ones, and compiled ones with B-spline fields: 1.
WOS_RULE int gradient_form(bool compiled, bool bspline) { return compiled && !bspline ? 2 : 1; }

// Form of a walk kernel: its walks' sums are formed in the kernel, left to walk_sum_kernel, or either, by the
// number of walks in the launch.  As a choice at a walk's end it costs large solves up to 5 % (2D B-spline
// annulus, 4.2e6 walks, 4.30 -> 4.51 ms; noise cube at five blocks 8.94 -> 9.05 ms), so of the generic kernels
// large solves run the first form (4.35 ms).  Small solves with per-point counts, and small batches, run the
// second: 2 to 11 % faster than the third.  Small solves of equal counts keep the third: they wait for a lone
// walk's steps, and those are the faster in it (4096 x 256 windows 20.6 ms against 21.3, the 2D square's 32^2 x
// 256 walks 522 us against 530).  Windows wait for their longest walk at any size, and have that form alone
// (1.1e6 walks 18.5 ms against 18.7).  Compiled kernels hold the choice: a second kernel would add half to
// their compilation (0.1 to 0.8 s), and it costs nothing but in 3D windows (1.20 -> 1.22 ms).
enum SpreadForm { SPREAD_NEVER = 0, SPREAD_ALWAYS = 1, SPREAD_BY_SIZE = 2 };

// The register cap of the generic FP32 value kernel for a launch of `walks` walks: variant 0, five blocks
// per SM; 1, eight; 2, four.  3D B-spline fields keep 64 taps' weights and indices: four blocks (a noise cube,
// 4096 points x 256 walks: 4 / 5 / 6 / 8 blocks 4.21 / 4.70 / 5.38 / 5.94 ms; in 2D 4.77 / 4.51 / 4.46 /
// 4.81).  Closed-form fields keep little and wait on the interpreter's chains: eight, where there are
// walks enough to fill them (2D square 8.4e6 walks 6.24 / 5.58 / 5.27 / 5.07 ms, 3D cube 4.2e6 walks 8.77 /
// 7.91 / 7.46 / 7.21; a solve of 2.6e5 walks 441 / 437 / 450 / 495 us).
WOS_RULE int value_variant(int dim, bool bspline, uint64_t walks) {
  return bspline ? (dim == 3 ? 2 : 0) : (walks > kSpreadItems ? 1 : 0);
}

// The most walks of a launch whose total is `total`, or known on the device only (per-point counts: ~0).  Of
// those, the small solves' launch serves at most kSpreadItems walks and the other one more.
WOS_RULE uint64_t walks_of_launch(uint64_t total, bool small_launch) {
  return small_launch && total > kSpreadItems ? kSpreadItems : total;
}

// Resident blocks per SM (the register cap) of the FP32 next-flight kernels.  Few walks wait for the longest
// ones, so the four blocks that spill least are the fastest; many fill the chip, and more blocks hide its
// instruction fetches.  Blocks 4 / 5 / 6, ms, 3D cube with 0 and 8 terms: 2.0e5 walks 1.99 / 2.11 / 2.15 and 3.26 /
// 3.53 / 3.89, 3.9e5 walks 2.79 / 2.78 / 2.44 and 4.57 / 4.49 / 4.30 (six blocks round the series otherwise: other
// walks), 2.1e6 walks 8.57 / 8.33 / 7.68 and 14.8 / 14.3 / 14.7.  Noise cube (B-spline fields), 0 and 8 terms: 2.0e5
// walks 2.74 / 3.54 / 4.11 and 5.77 / 6.61 / 7.13, 2.1e6 walks 13.1 / 14.3 / 15.8 and 28.1 / 27.1 / 27.6; in
// 2D (annulus, 0 terms) 0.94 / 0.99 / 1.17 and 4.21 / 4.02 / 4.06.  Mesh, 20,480 triangles, 4 / 5:
// 1.3e5 walks 20.7 / 23.1 and 23.8 / 25.7, 5.2e5 walks 38.9 / 40.7 and 43.9 / 48.2, 1.05e6 walks 68.0 / 65.2 and 76.9 /
// 75.0, 4.2e6 walks 240 / 225 and 270 / 260.  nf_few_walks: the most walks that count as few.
WOS_RULE uint64_t nf_few_walks(bool mesh, bool bspline) {
  return mesh ? 3ull << 18 : (bspline ? 1ull << 20 : 1ull << 18);
}
WOS_RULE int nf_blocks(int dim, bool mesh, bool series, bool bspline, uint64_t walks) {
  if (walks <= nf_few_walks(mesh, bspline)) return 4;
  if (mesh || series) return 5;
  return bspline && dim == 3 ? 4 : 6;
}

// Whether wos_solve_host's results leave through a page-locked buffer, with one wait for the stream
// (a copy into a caller's pageable array waits by itself).  Larger results spend more on the second copy
// than on the waits: 8 walks per point of the 3D cube, copies per array / staged, us: 1,000 points 209 / 183,
// 5,003 239 / 222, 10,000 270 / 263, 16,384 325 / 327, 30,000 380 / 403, 65,536 522 / 599.
WOS_RULE bool host_staged(int64_t npts) { return npts <= 12288; }

// The per-CTA copy of an alpha grid in shared memory that an adjoint launch adds up in: strides of its rows
// and planes, and its size (nodes 0: no copy, the gradients go to global memory; grids above 8192 nodes).
struct AdjointCopy {
  int s1, s2, nodes;
};
// resident blocks per SM of an adjoint kernel with so many bytes of shared memory; its registers allow four
WOS_RULE int adjoint_blocks(int64_t bytes) {
  if (bytes > 200 * 1024) return 0;
  const int64_t n = 228 * 1024 / (bytes + 1024);  // an SM's shared memory, with what the system keeps of it
  return n < 4 ? (int)n : 4;
}
// `other`: the block's further bytes (problem, staged scatters).  The 32 taps that a warp adds at once are 4 x 4 x
// 2 neighbours: with a row stride of 4 (mod 8) and in 3D a plane stride of 16 (mod 32) they lie in 32
// different banks (16^3 controls 17.3 -> 14.2 ms together with the warp-wide scatter).  Where the padding
// for that costs a resident block, rows and planes are padded by one, which keeps the worst strides away.
WOS_RULE AdjointCopy adjoint_copy(int dim, int64_t res0, int64_t res1, int64_t res2, int64_t other, int real_bytes) {
  const int64_t planes = dim == 3 ? res2 : 1;
  if (res0 * res1 * planes > 8192) return AdjointCopy{0, 0, 0};
  const int64_t p1 = res0 + (12 - res0 % 8) % 8, rows = p1 * res1;
  const int64_t p2 = dim == 3 ? rows + (48 - rows % 32) % 32 : rows;
  const int64_t c1 = res0 + 1, c2 = c1 * res1 + 1;
  const int padded = adjoint_blocks(other + p2 * planes * real_bytes);
  const int close = adjoint_blocks(other + c2 * planes * real_bytes);
  if (padded > 0 && padded >= close) return AdjointCopy{(int)p1, (int)p2, (int)(p2 * planes)};
  return close > 0 ? AdjointCopy{(int)c1, (int)c2, (int)(c2 * planes)} : AdjointCopy{0, 0, 0};
}

}  // namespace wos
