// Launchers for one highest order L (included by gmp_inst_L<L>.cu so the
// seven orders compile in parallel).
#pragma once

#include "gmp_jacobian.cuh"
#include "gmp_kernels.cuh"
#include "gmp_launch.h"

#include <algorithm>

namespace gmpk {

template <int L, int NS, int TILE>
size_t smem_bytes(const GmpPass& P, int warps, bool pad = true) {
  return sizeof(float) * (table_floats(P.n_el, L, NS, P.kmax, pad) +
                          (size_t)warps * Shape<L, NS, TILE>::WARP_FLOATS);
}

// Whether k_jacobian_r (orders up to kJacRegOrders) is faster than k_jacobian
// beside these tables: it stages 2.6 times as much a warp, and with fewer than 6
// of its warps per SM that costs more than its fewer instructions spare.
// Jacobian kernel, 3,072 centers of 79 pairs, us, k_jacobian -> k_jacobian_r (GB300;
// elements x Gaussians, warps that fit beside the tables):
//   orders 0-4, 16 sigmas   12 x 16 (6) 387 -> 224, 24 x 8 (6) 242 -> 184,
//                           24 x 16 (1) 596 -> 962, 48 x 8 (1) 494 -> 802
//   orders 0-3              8 sigmas 48 x 16 (3) 151 -> 189, 16 sigmas 12 x 16 (9)
//                           381 -> 165, 48 x 8 (2) 234 -> 348
//   orders 0-2, 16 sigmas   24 x 8 (12) 155 -> 131, 48 x 8 (5) 178 -> 230
//   orders 0-2, 4 sigmas    6 x 8 44 -> 42, 12 x 8 45 -> 46, 24 x 16 56 -> 64
template <int L, int NS>
bool jacobian_r_pays(const GmpPass& P, size_t max_smem) {
  if (L == 2 && NS == 4 && P.n_el > 6) return false;
  return sizeof(float) * (table_floats(P.n_el, L, NS, P.kmax) + 6 * (size_t)JacShape<L, NS>::WARP_FLOATS) <= max_smem;
}

// shape.tile: 16 or 32 pairs per forward tile; shape.warps: warps per CTA
// (0 = the size with the most resident warps).
template <int L, int NS>
cudaError_t launch(int kind, const KParams& K, GmpShape shape, GmpLaunchPlan* plan, cudaStream_t st, int sm_count,
                   int64_t* launches) {
  constexpr size_t kMaxSmem = 227 * 1024;
  // a tile of 32 pairs gives way to one of 16 where not even one warp of it fits
  // beside the tables
  const int tile = kind == GMP_KIND_FORWARD && shape.tile == 32 && smem_bytes<L, NS, 32>(K.pass, 1) <= kMaxSmem ? 32 : 16;
  size_t jac_r_floats = 0;  // per warp of k_jacobian_r (0: not used)
  void (*fn)(KParams) = kind == GMP_KIND_FORWARD    ? (tile == 32 ? k_forward<L, NS, 32> : k_forward<L, NS, 16>)
                        : kind == GMP_KIND_VJP      ? k_vjp<L, NS>
                        : kind == GMP_KIND_BACKWARD
                            ? (K.pass.mixed_sign ? k_backward<L, NS, false, true> : k_backward<L, NS, false, false>)
                        : kind == GMP_KIND_BACKWARD_VIRIAL
                            ? (K.pass.mixed_sign ? k_backward<L, NS, true, true> : k_backward<L, NS, true, false>)
                            : k_jacobian<L, NS>;
  if constexpr (L <= kJacRegOrders) {
    if (kind == GMP_KIND_JACOBIAN && jacobian_r_pays<L, NS>(K.pass, kMaxSmem)) {
      fn = k_jacobian_r<L, NS>;
      jac_r_floats = JacShape<L, NS>::WARP_FLOATS;
    }
  }
  auto smem_of = [&](int w) -> size_t {
    if (jac_r_floats) return sizeof(float) * (table_floats(K.pass.n_el, L, NS, K.pass.kmax) + (size_t)w * jac_r_floats);
    if (kind == GMP_KIND_BACKWARD || kind == GMP_KIND_BACKWARD_VIRIAL) {
      const bool vir = kind == GMP_KIND_BACKWARD_VIRIAL;
      return sizeof(float) * (table_floats(K.pass.n_el, L, NS, K.pass.kmax, vir ? back_pad<L, true>() : back_pad<L, false>()) +
                              (size_t)w * back_warp_floats<L, NS>(vir));
    }
    const bool pad = kind != GMP_KIND_JACOBIAN;  // the general Jacobian kernel: unpadded table
    return tile == 32 ? smem_bytes<L, NS, 32>(K.pass, w) : smem_bytes<L, NS, 16>(K.pass, w, pad);
  };
  const int64_t n = K.N - K.center0;
  // fewer centers than a CTA of the usual size on every SM would take: as
  // many warps as spread them over the SMs (64 centers: 64 CTAs of one warp
  // instead of 4 of 16)
  const int spread = n < 16 * (int64_t)sm_count ? (int)std::max<int64_t>(1, (n + sm_count - 1) / sm_count) : 0;
  const int want = shape.warps > 0 && (spread == 0 || shape.warps < spread) ? shape.warps : spread;
  if (plan->fn != (const void*)fn || plan->req_warps != want) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return e;
    // always the same limit, so that no handle's launch depends on which one
    // set it last
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    if (e != cudaSuccess) return e;
    int warps = fa.maxThreadsPerBlock / 32;
    if (warps > 20) warps = 20;
    if (want > 0 && want < warps) warps = want;
    while (warps > 1 && smem_of(warps) > kMaxSmem) --warps;
    if (want <= 0) {
      // untuned: the CTA size with the most resident warps, of equals the
      // smallest with at least 4 (registers and the tables' share of the
      // shared memory decide: the forward kernel at orders 0-4 x 8 sigmas keeps
      // 28 warps in CTAs of 7 and 16 in one of 16, 3.40 against 4.03 ms on
      // 10,000 structures; 4096 Jacobian centers took 177 us in 12-warp CTAs
      // and 167 in as many warps of 4-warp ones)
      int best_w = warps, best_res = 0;
      for (int w = warps; w >= 1; --w) {
        if (smem_of(w) > kMaxSmem) continue;
        int ps = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, fn, w * 32, smem_of(w));
        if (e != cudaSuccess) return e;
        if (ps * w > best_res || (ps * w == best_res && w >= 4)) { best_res = ps * w; best_w = w; }
      }
      warps = best_w;
    }
    if (smem_of(warps) > kMaxSmem) return cudaErrorInvalidConfiguration;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, warps * 32, smem_of(warps));
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    *plan = GmpLaunchPlan{(const void*)fn, want, warps, per_sm, smem_of(warps)};
  }
  const int warps = plan->warps, per_sm = plan->per_sm;
  const size_t smem = plan->smem;
  int64_t blocks = (int64_t)sm_count * per_sm;
  const int64_t need = (n + warps - 1) / warps;
  if (blocks > need) blocks = need;
  if (blocks < 1) blocks = 1;
  ++*launches;
  return gmp_launch_next(fn, (unsigned)blocks, warps * 32, smem, st, K);
}

}  // namespace gmpk

#define GMP_DEFINE_LAUNCHER(LV)                                                                      \
  cudaError_t gmp_launch_compute_L##LV(int kind, int ns, const gmpk::KParams& K, GmpShape shape,      \
                                      GmpLaunchPlan* plan, cudaStream_t st, int sm_count, int64_t* launches) {             \
    switch (ns) {                                                                                    \
      case 4: return gmpk::launch<LV, 4>(kind, K, shape, plan, st, sm_count, launches);                    \
      case 8: return gmpk::launch<LV, 8>(kind, K, shape, plan, st, sm_count, launches);                    \
      case 16: return gmpk::launch<LV, 16>(kind, K, shape, plan, st, sm_count, launches);                  \
      default: return cudaErrorInvalidValue;                                                         \
    }                                                                                                \
  }
