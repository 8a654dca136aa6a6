// Entry points of the per-order compute launchers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#define GMP_KIND_FORWARD 0
#define GMP_KIND_VJP 1
#define GMP_KIND_JACOBIAN 2
#define GMP_KIND_BACKWARD 3
#define GMP_KIND_BACKWARD_VIRIAL 4  // backward + per-structure strain derivative

namespace gmpk {
struct KParams;
}

// Launch shape of a compute kernel (chosen by the autotuner or defaults).
struct GmpShape {
  int tile;   // forward tile: 16 pairs (two lanes per pair) or 32
  int warps;  // warps per CTA, 0 = the CTA size with the most resident warps
};

// The untuned forward tile of highest order L, ns padded sigmas and n_el
// elements of kmax Gaussians.  In a tile of 32 (orders up to 4, 8 or 16 sigmas) a
// lane takes the radial factors of two neighboring pairs, so that a table load
// serves both when they are of one element, as the lists are sorted by; the kernel
// is bound by shared-memory wavefronts.  It keeps at most 20 instead of 28 warps per
// SM; larger tables take more of that away, and with more elements fewer pairs
// agree.  Forward kernel, GB300, us, tile 16 -> 32, crystals of 4,096 / 32,768
// atoms (183 pairs a center) and 2,500 small structures (10 elements, 74 pairs):
//   8 sigmas, orders 0-2   47 -> 43 / 275 -> 253   775 -> 679
//             orders 0-3   55 -> 45 / 333 -> 274   938 -> 737
//             orders 0-4   53 -> 52 / 319 -> 299 with 3 elements, 53 -> 56 /
//                          324 -> 320 with 6, 54 -> 58 / 330 -> 349 with 10;  856 -> 868
//             orders 0-1   38 -> 40                546 -> 607
//  16 sigmas, orders 0-2   59 -> 58 / 384 -> 360  1060 -> 953
//             orders 0-3   72 -> 77               1313 -> 1350
//             orders 0-4   86 -> 92               1608 -> 2129
// and a crystal of 16,384 atoms (77 pairs a center) with elements x Gaussians:
//   8 sigmas, orders 0-2   20 x 4 74 -> 69, 10 x 8 89 -> 87, 6 x 16 119 -> 121, 40 x 8 95 -> 106
//             orders 0-3   20 x 4 86 -> 76, 10 x 8 109 -> 98, 10 x 16 158 -> 158, 40 x 8 115 -> 123
//             orders 0-4   1 x 16 134 -> 128, 3 x 8 96 -> 99, 3 x 32 222 -> 241, 40 x 16 231 -> 350
//  16 sigmas, orders 0-2   10 x 4 95 -> 93, 3 x 8 117 -> 115, 6 x 8 125 -> 127, 20 x 4 100 -> 105
constexpr int gmp_forward_tile(int L, int ns, int n_el, int kmax) {
  const int most = ns == 8 ? (L == 2 || L == 3 ? 80 : L == 4 && n_el <= 4 ? 20 : 0) : ns == 16 && L == 2 ? 40 : 0;
  return (int64_t)n_el * kmax <= most ? 32 : 16;
}

// The launch worked out for a request (shape and number of centers' class):
// kept by the handle, so that a call repeats neither the attribute nor the
// occupancy queries (several microseconds a launch).
struct GmpLaunchPlan {
  const void* fn = nullptr;   // null: nothing worked out yet
  int req_warps = 0, warps = 0, per_sm = 0;
  size_t smem = 0;
};

#define GMP_DECLARE_LAUNCHER(LV)                                                                \
  cudaError_t gmp_launch_compute_L##LV(int kind, int ns, const gmpk::KParams& K, GmpShape shape,  \
                                      GmpLaunchPlan* plan, cudaStream_t st, int sm_count, int64_t* launches);
GMP_DECLARE_LAUNCHER(0)
GMP_DECLARE_LAUNCHER(1)
GMP_DECLARE_LAUNCHER(2)
GMP_DECLARE_LAUNCHER(3)
GMP_DECLARE_LAUNCHER(4)
GMP_DECLARE_LAUNCHER(5)
GMP_DECLARE_LAUNCHER(6)
