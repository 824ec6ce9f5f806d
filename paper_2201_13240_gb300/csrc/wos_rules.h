// wos_rules.h -- which form of a kernel a call takes: rules on sizes, types and fields, apart from
// CUDA so that the host check library can be asked for them too.
#pragma once

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

}  // namespace wos
