// Double-float recomputation of features that FP32 cannot resolve.
//
// A feature f_{l,s} = sum_c w_c mu_c^2 whose value is tiny compared with the
// cancellation-free scale of its moments (near-symmetric environments make
// l >= 1 moments cancel) loses relative accuracy in FP32 in proportion to
// sqrt(scale / f).  The forward kernels queue such (center, order, two
// sigmas) entries; this kernel recomputes each of them in double-float
// arithmetic (pairs of FP32 words, about 2^-44 relative per operation), which
// FP32 hardware runs far faster than FP64: the displacement from the
// double-float split of the positions (the atoms, or the reference points of
// gmp_featurize_points), the radial factor with a double-float exponential,
// the angular part, and the invariant.  When a derivative kernel follows,
// the recomputed moments also replace the FP32 moments it reads: the adjoints
// of a cancelling moment group would otherwise carry its FP32 rounding, which
// is relative to the group's cancellation-free scale rather than to the
// moments themselves.
//
// The angular part takes the 2l+1 real solid harmonics of the one order l
// (powers of x + iy times polynomials in z and r^2: about 50 double-float
// operations at order 6) instead of raising the MCSH components through
// every order below (173 operations, all of them needed for the top one).
// The invariant is the same sum of squares in either basis (the addition
// theorem, checked in exact arithmetic by gen_mcsh.py), and the components'
// moments follow from the harmonics' by a constant matrix, once per entry.
#include "gmp_internal.cuh"
#include "mcsh_gen.cuh"

namespace {

// values of a warp's lanes reduced at once: the next power of two >= 2l+1
__host__ __device__ constexpr int log2_values(int l) {
  int b = 0;
  while ((1 << b) < 2 * l + 1) ++b;
  return b;
}

__device__ __forceinline__ gmp_f2 shfl_xor(gmp_f2 v, int d) {
  return gmp_f2{__shfl_xor_sync(0xffffffffu, v.hi, d), __shfl_xor_sync(0xffffffffu, v.lo, d)};
}

// Warp sums of v[0 .. 2^B-1]: halving exchanges leave the sum of value j in
// the lanes j << (5 - B) .. ((j + 1) << (5 - B)) - 1 (each step sends one half
// of the values and keeps the other), then plain butterflies.
template <int B>
__device__ __forceinline__ gmp_f2 reduce_scatter(gmp_f2 (&v)[1 << B], int lane) {
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const int d = 16 >> b, n = (1 << B) >> (b + 1);
    const bool up = lane & d;
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const gmp_f2 send = up ? v[j] : v[j + n];
      const gmp_f2 keep = up ? v[j + n] : v[j];
      v[j] = gmp_df_add(keep, shfl_xor(send, d));
    }
  }
#pragma unroll
  for (int d = 16 >> B; d; d >>= 1) v[0] = gmp_df_add(v[0], shfl_xor(v[0], d));
  return v[0];
}

// One entry of order L by a warp: the moments of the two sigmas sig, sig + 1
// (those in mask) over the center's pairs (lane-strided), the features, and
// with mu_out the moments.  Sums keep (hi, lo) with the errors of the hi sums
// and the terms' low words added to lo.
template <int L>
__device__ __forceinline__ void refine_entry(int lane, const GmpRefine& A, const float2* exp_tab, int64_t i, int col,
                                             unsigned mask) {
  constexpr int B = log2_values(L), NV = 1 << B;
  const int sig = A.col_info[col] & 0xffff;
  const GmpStruct& st = A.structs[A.center_struct[i]];
  const float4 xhi = A.center_xh[i], xli = A.center_xl[i];
  const int64_t p0 = A.nbr_beg[i], p1 = A.nbr_end[i];
  gmp_f2 mu[2][NV];
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int k = 0; k < NV; ++k) mu[g][k] = gmp_f2{0.0f, 0.0f};
  for (int64_t p = p0 + lane; p < p1; p += 32) {
    const GmpPair pr = A.pairs[p];
    // the next pair's atom, whose position is fetched while this one is computed
    const int jn = p + 32 < p1 ? A.pairs[p + 32].j : pr.j;
    int nn[3];
    gmp_unpack_shift(pr.shift, nn);
    gmp_f2 d[3], r2, H[2 * L + 1];
    gmp_df_disp(xhi, xli, A.atom_xh[pr.j], A.atom_xl[pr.j], st, nn, d, r2);
    asm volatile("prefetch.global.L1 [%0];" ::"l"(A.atom_xh + jn));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(A.atom_xl + jn));
    gmp_solid_df<L>(d[0], d[1], d[2], r2, H);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      if (!(mask & (1u << g))) continue;  // warp-uniform
      // radial factor: sum_q A_{q,L} exp(-b_q r^2); table entry (b, A_0 .. A_6) as double-floats
      const float2* te = reinterpret_cast<const float2*>(A.ktab) +
                         ((size_t)pr.e * A.nsig_total + sig + g) * A.kmax * 8;  // [element][sigma][primitive]
      gmp_f2 R{0.0f, 0.0f};
      for (int q = 0; q < A.kmax; ++q) {
        const float2 b = __ldg(te + 8 * q), a = __ldg(te + 8 * q + 1 + L);
        const gmp_f2 E = gmp_df_exp_neg(gmp_df_mul_u(gmp_f2{b.x, b.y}, r2), exp_tab);
        const gmp_f2 t = gmp_two_prod(a.x, E.hi);
        const gmp_f2 s = gmp_two_sum(R.hi, t.hi);
        R.hi = s.hi;
        R.lo = __fadd_rn(R.lo, __fadd_rn(s.lo, __fmaf_rn(a.x, E.lo, __fmaf_rn(a.y, E.hi, t.lo))));
      }
      R = gmp_fast_two_sum(R.hi, R.lo);
#pragma unroll
      for (int k = 0; k <= 2 * L; ++k) {
        const gmp_f2 t = gmp_two_prod(R.hi, H[k].hi);
        const gmp_f2 s = gmp_two_sum(mu[g][k].hi, t.hi);
        mu[g][k].hi = s.hi;
        mu[g][k].lo = __fadd_rn(mu[g][k].lo, __fadd_rn(s.lo, __fmaf_rn(R.hi, H[k].lo, __fmaf_rn(R.lo, H[k].hi, t.lo))));
      }
    }
  }
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    if (!(mask & (1u << g))) continue;
    const gmp_f2 M = reduce_scatter<B>(mu[g], lane);  // of value j = lane >> (5 - B)
    const int j = lane >> (5 - B);
    const float2 n = j <= 2 * L ? gmp_solid_norm[L][j] : make_float2(0.0f, 0.0f);
    gmp_f2 f = gmp_df_mul(gmp_df_mul(gmp_f2{n.x, n.y}, M), M);
#pragma unroll
    for (int d = 16; d > (16 >> B); d >>= 1) f = gmp_df_add(f, shfl_xor(f, d));
    if (lane == 0) A.features[i * A.F + col + g] = f.hi + f.lo;
    const int sp = sig + g - A.mu_sig0;
    if (A.mu_out && sp >= 0 && sp < A.mu_nsig) {
      // lane k: component k as a combination of the harmonics
      const int k = lane <= 2 * L ? lane : 0;
      gmp_f2 m{0.0f, 0.0f};
#pragma unroll
      for (int t = 0; t < GMP_SOLID_NZ; ++t) {
        const int src = gmp_solid_row[L][k][t] << (5 - B);
        const float2 c = gmp_solid_coef[L][k][t];
        const gmp_f2 v{__shfl_sync(0xffffffffu, M.hi, src), __shfl_sync(0xffffffffu, M.lo, src)};
        m = gmp_df_add(m, gmp_df_mul(gmp_f2{c.x, c.y}, v));
      }
      if (lane <= 2 * L) A.mu_out[(i * A.mu_nsig + sp) * (int64_t)A.mu_nind + L * L + lane] = m.hi + m.lo;
    }
  }
}

// (count: lane l holds the entries of order l)
template <int L>
__device__ __forceinline__ void refine_order(int lane, const GmpRefine& A, const float2* exp_tab, int64_t warp,
                                             int64_t nw, int64_t count, int64_t& done) {
  const int64_t n = __shfl_sync(0xffffffffu, count, L);
  if (n > 0) {
    const unsigned long long* queue = A.queue + A.qidx[L] * A.cap;
    int64_t v = (warp - done) % nw;
    if (v < 0) v += nw;
    for (; v < n; v += nw) {
      const unsigned long long e = queue[v];
      refine_entry<L>(lane, A, exp_tab, (int64_t)(e >> 32), (int)((e >> 16) & 0xffffu), (unsigned)(e & 3u));
    }
    done += n;
  }
  if constexpr (L > 0) refine_order<L - 1>(lane, A, exp_tab, warp, nw, count, done);
}

// A warp per entry, the entries of all orders numbered through, the largest
// order first: the warps that are left over by one order start on the next,
// and at one time most warps run the same order's code (its instructions are
// what a warp mostly waits for at orders 4-6).  One launch for all orders:
// a typical batch flags a few thousand features per order, one round of
// warps each, and a launch per order paid that round's latency five times.
// Measured on a GB300 with the solid harmonics, the cheaper exponential and sums
// left unnormalised (before: one launch per order, raising recurrences): perfect
// FCC crystal of 32,768 atoms, orders 0-6 x 16 sigmas, 2565 -> 589 us; 4,096-atom
// alloy crystal, orders 0-4 x 8 sigmas, 82 -> 24 us; alloy slab of 262,144 atoms
// 482 -> 104 us.  Bound by the double-float instructions themselves (issue 77%) at
// 16 warps per SM (128 registers).
__global__ void __launch_bounds__(256, 2) k_refine(const GmpRefine A) {
  __shared__ float2 exp_tab[64];
  if (threadIdx.x < 64) exp_tab[threadIdx.x] = A.exp_tab[threadIdx.x];
  const int lane = gmp_after_predecessor(threadIdx.x) & 31;
  int64_t count = 0;
#pragma unroll
  for (int l = 0; l < 7; ++l)
    if (lane == l && A.qidx[l] >= 0) count = (int64_t)min(A.count[A.qidx[l]], (unsigned long long)A.cap);
  __syncthreads();
  int64_t done = 0;
  refine_order<6>(lane, A, exp_tab, ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                  ((int64_t)gridDim.x * blockDim.x) >> 5, count, done);
}

}  // namespace

cudaError_t gmp_launch_refine(const GmpRefine& A, int sm_count, int* per_sm, cudaStream_t stream, int64_t* launches) {
  bool any = false;  // orders >= 0 requested
  for (int l = 0; l < 7; ++l) any = any || A.qidx[l] >= 0;
  if (A.n_centers <= 0 || !any) return cudaSuccess;
  // as many CTAs as can be resident: the warps take fixed strides of the
  // flagged entries, so a second partial wave would leave most of each SM
  // idle while it runs
  if (*per_sm < 1) {
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_refine, 256, 0);
    if (e != cudaSuccess) return e;
    if (*per_sm < 1) *per_sm = 1;
  }
  ++*launches;
  return gmp_launch_next(k_refine, (unsigned)(sm_count * *per_sm), 256, 0, stream, A);
}
