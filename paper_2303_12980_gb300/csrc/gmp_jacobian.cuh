// Jacobian rows for orders up to 4 (k_jacobian in gmp_kernels.cuh takes the
// higher ones, whose coefficients below do not fit the registers, and tables
// that leave room for few warps' rows below: jacobian_r_pays).
//
// For center i, order l and sigma s, with P = sum_k lam_k S_k(d) and lam = d f /
// d mu, a pair contributes d f / d d = 2 d (-beta R_{l+1}) P + R_l grad P.  The
// gradient of a harmonic polynomial of order l is one of order l - 1: grad_v P =
// sum_k' M_{v,k'} S_k' with M formed once per center from lam
// (gmp_mcsh_grad_coef_order_<l>), so a pair costs 2l+1 + 3 (2l-1) multiply-adds
// per order and sigma, no order L+1 and no division by r^2.
//
// The center's rows (distinct neighbor atoms; the list is sorted by atom) are
// split evenly among the 32 / NS groups of a warp.  A group's lanes first stage
// its next NS pairs, lane = pair: MCSH values, radial factors of every sigma
// (four per table load, exponent offset 2^S per center and sigma) and the
// density's derivative go to the pair's shared-memory row.  Then the group
// walks those pairs with one lane per sigma, lam and M in registers, and writes
// each finished row.  Against every sigma lane evaluating the MCSH values of its
// pair and 4 contractions per order through order L+1: 192 -> 113 warp
// instructions a pair, 219 -> 167 us on 4096 centers (759,118 rows of 40
// features, 364 MB: 54 us at the copy rate; GB300).  Bound by instruction issue
// (49% at 12 warps per SM, 166 registers) and the latency of its loads.  Rows of group g start g * NS (radial) or 4 g floats
// later than their index says, so that the groups' reads fall on different
// banks.
#pragma once

#include "gmp_kernels.cuh"

namespace gmpk {

constexpr int kJacRegOrders = 4;  // highest order whose lam and M (25 + 48) are held in registers

template <int l>
__device__ __forceinline__ void grad_coef_order(const float* lam, float* Mx, float* My, float* Mz) {
  if constexpr (l == 1) gmp_mcsh_grad_coef_order_1(lam, Mx, My, Mz);
  else if constexpr (l == 2) gmp_mcsh_grad_coef_order_2(lam, Mx, My, Mz);
  else if constexpr (l == 3) gmp_mcsh_grad_coef_order_3(lam, Mx, My, Mz);
  else if constexpr (l == 4) gmp_mcsh_grad_coef_order_4(lam, Mx, My, Mz);
}

template <int L, int NS>
struct JacShape {
  static constexpr int G = 32 / NS;                    // groups of a warp
  static constexpr int NIND = (L + 1) * (L + 1);
  static constexpr int NINDP = Shape<L, NS>::NINDP;
  static constexpr int SSTR = odd4(NIND);              // S row
  static constexpr int RSTR = odd4((L + 2) * NS);      // R row [order][sigma]
  static constexpr int S_FLOATS = 32 * SSTR + 4 * G;
  static constexpr int D_FLOATS = 32 * 4 + 4 * G;      // d, density derivative
  static constexpr int R_FLOATS = 32 * RSTR + NS * G;
  static constexpr int WARP_FLOATS = S_FLOATS + D_FLOATS + R_FLOATS + NS * NINDP + 16;
  static_assert(NS * NIND <= R_FLOATS, "the moments must fit the radial rows");
};

template <int L, int NS>
__global__ void __launch_bounds__(384) k_jacobian_r(KParams K) {
  using SH = JacShape<L, NS>;
  constexpr int RB = gmp_rad_block(L);
  extern __shared__ __align__(16) float smem[];
  const GmpPass& P = K.pass;
  float* s_rad = smem;
  float* s_dens = s_rad + (size_t)P.n_el * rad_elem_stride(L, NS, P.kmax);
  float* s_warp = s_dens + (size_t)P.n_el * dens_elem_stride(P.kmax);
  load_tables<L>(P, NS, s_rad, s_dens);
  __syncthreads();
  gmp_after_predecessor(0);  // (the tables belong to the handle)
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int g = lane / NS, s = lane % NS;  // group and, in it, the staged pair or the sigma
  const bool s_ok = s < P.nsig;
  const bool dens_lane = P.want_density && s == 0;
  const float nb2 = 2.0f * P.nbeta[s];
  float* Sr = s_warp + (size_t)wib * SH::WARP_FLOATS;
  float* Dr = Sr + SH::S_FLOATS;
  float* Rr = Dr + SH::D_FLOATS;
  float* Lam = Rr + SH::R_FLOATS;
  float* Sh = Lam + NS * SH::NINDP;  // exponent offset per sigma
  int col[L + 1];                    // feature column of order l, -1: not requested
#pragma unroll
  for (int l = 0; l <= L; ++l) {
    col[l] = -1;
    for (int o = 0; o < P.n_ord; ++o)
      if (P.ord_l[o] == l) col[l] = P.ord_col[o];
  }
  for (int64_t i = next_center(K); i < K.N; i = next_center(K)) {
    const int64_t p0 = K.nbr_beg[i], p1 = K.nbr_end[i];
    if (p1 > K.pair_cap) continue;  // over capacity: flagged by the fill pass
    const float* mrow = K.mu_out + i * (int64_t)P.nsig * SH::NIND;
    float* Mu = Rr;  // until the first pairs are staged
    for (int t = lane; t < NS * SH::NIND; t += 32) Mu[t] = (t < P.nsig * SH::NIND) ? mrow[t] : 0.0f;
    __syncwarp();
    adjoints<L, NS>(P, Mu, nullptr, Lam);  // per feature: lam = d f / d mu
    float lam[SH::NIND], M[3][L > 0 ? L * L : 1];
    float lm = 0.0f;
#pragma unroll
    for (int k = 0; k < SH::NIND; ++k) {
      lam[k] = Lam[s * SH::NINDP + k];
      lm = fmaxf(lm, fabsf(lam[k]));
    }
    static_for<L>([&](auto ll) { grad_coef_order<decltype(ll)::value + 1>(lam, M[0], M[1], M[2]); });
    // exponent offset of this lane's sigma, as k_jacobian chooses it: the
    // largest S (at most 90, at least 32) that keeps the scaled intermediates
    // below 2^126
    const int le = ((__float_as_int(lm) >> 23) & 255) - 126;                    // > log2(lm)
    const int lb = max(0, ((__float_as_int(-P.nbeta[s]) >> 23) & 255) - 126);  // >= log2(beta)
    const int Si = max(32, min(90, 94 - le - lb - P.jac_exp[s]));
    const float unshift = __int_as_float((127 - Si) << 23);
    if (lane < NS) Sh[s] = (float)Si;
    const int64_t r0 = K.jac_off[i - K.center0];
    const int R = (int)(K.jac_off[i - K.center0 + 1] - r0);
    // the center's own row: the rank of atom i among its neighbor atoms
    int64_t lo = p0, hi = p1;
    while (lo < hi) {
      const int64_t mid = lo + ((hi - lo) >> 1);
      if (K.pairs[mid].j < (int32_t)i) lo = mid + 1;
      else hi = mid;
    }
    // (the self pair, j = i with no shift, is always in the list)
    const int r_self = (lo < p1 && K.pairs[lo].j == (int32_t)i) ? K.jac_row[lo] : -1;
    // this group's rows [ra, rb) and their pairs [pa, pb)
    const int ra = (int)((int64_t)R * g / SH::G), rb = (int)((int64_t)R * (g + 1) / SH::G);
    const int64_t pa = first_pair_of_row(K.jac_row, p0, p1, ra);
    const int64_t pb = first_pair_of_row(K.jac_row, pa, p1, rb);
    const int n = (int)(pb - pa);
    const int n_max = __reduce_max_sync(0xffffffffu, n);
    float acc[L + 1][3], self[L + 1][3], dacc[3] = {0.0f, 0.0f, 0.0f}, dself[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int l = 0; l <= L; ++l)
#pragma unroll
      for (int v = 0; v < 3; ++v) acc[l][v] = self[l][v] = 0.0f;
    int cur = -1;  // row being accumulated
    auto write_row = [&](int64_t row, const float (&a)[L + 1][3], const float* d) {
      float* base = K.jac + row * P.F * 3;
      if (s_ok) {
#pragma unroll
        for (int l = 0; l <= L; ++l)
          if (col[l] >= 0) {
            float* dst = base + (col[l] + s) * 3;
            dst[0] = a[l][0] * unshift;
            dst[1] = a[l][1] * unshift;
            dst[2] = a[l][2] * unshift;
          }
      }
      if (dens_lane) {
        float* dst = base + P.dens_col * 3;
        dst[0] = d[0] * GMP_EXP_UNSHIFT;
        dst[1] = d[1] * GMP_EXP_UNSHIFT;
        dst[2] = d[2] * GMP_EXP_UNSHIFT;
      }
    };
    // a finished row is written (the own row below, from the sum of the
    // others) and taken off the own row
    auto flush = [&]() {
      if (cur >= 0 && cur != r_self) {
        write_row(r0 + cur, acc, dacc);
#pragma unroll
        for (int l = 0; l <= L; ++l)
#pragma unroll
          for (int v = 0; v < 3; ++v) self[l][v] -= acc[l][v];
#pragma unroll
        for (int v = 0; v < 3; ++v) dself[v] -= dacc[v];
      }
    };
    for (int t = 0; t < n_max; t += NS) {
      __syncwarp();  // the last rows (and the moments) have been read
      int row_id = -1;
      if (t + s < n) {  // stage pair pa + t + s
        const int64_t p = pa + t + s;
        float dx, dy, dz, r2h, r2l;
        int e, j;
        load_pair(K.pairs, p, dx, dy, dz, r2h, r2l, e, j);
        if (t + s + NS < n) prefetch_pair(K.pairs + p + NS);
        row_id = K.jac_row[p];
        float S[SH::NIND];
        GmpMcsh<L>::eval(dx, dy, dz, mcsh_r2(dx, dy, dz), S);
        float* srow = Sr + lane * SH::SSTR + 4 * g;
#pragma unroll
        for (int c = 0; c < (SH::NIND + 3) / 4; ++c)
          *reinterpret_cast<float4*>(srow + 4 * c) =
              make_float4(S[4 * c], 4 * c + 1 < SH::NIND ? S[4 * c + 1 < SH::NIND ? 4 * c + 1 : 0] : 0.0f,
                          4 * c + 2 < SH::NIND ? S[4 * c + 2 < SH::NIND ? 4 * c + 2 : 0] : 0.0f,
                          4 * c + 3 < SH::NIND ? S[4 * c + 3 < SH::NIND ? 4 * c + 3 : 0] : 0.0f);
        float drho = 0.0f;
        if (P.want_density) density_term(s_dens + (size_t)e * dens_elem_stride(P.kmax), P.kmax, r2h, r2l, &drho);
        *reinterpret_cast<float4*>(Dr + 4 * (lane + g)) = make_float4(dx, dy, dz, 2.0f * drho);
        // radial factors, orders 0 .. L+1, scaled by 2^S (double-float exponent
        // argument: a row of one neighbor averages no other terms)
        const float* tab_e = s_rad + (size_t)e * rad_elem_stride(L, NS, P.kmax);
        float* rrow = Rr + lane * SH::RSTR + NS * g;
        const float2 nr2h = make_float2(-r2h, -r2h), r2h2 = make_float2(r2h, r2h), r2l2 = make_float2(r2l, r2l);
#pragma unroll 1
        for (int sg = 0; sg < NS / 4; ++sg) {
          const float4 S4 = *reinterpret_cast<const float4*>(Sh + 4 * sg);
          float2 Rp[2][L + 2];
#pragma unroll
          for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int l = 0; l < L + 2; ++l) Rp[u][l] = make_float2(0.0f, 0.0f);
#pragma unroll 1
          for (int q = 0; q < P.kmax; ++q) {
            const float4* blk = reinterpret_cast<const float4*>(tab_e) + sg * rad_sg_stride(L, P.kmax) + q * RB;
            const float4 bh = blk[0], bl = blk[1];
            const float2 E0 = gmp_exp_neg2_shifted(make_float2(bh.x, bh.y), make_float2(bl.x, bl.y), nr2h, r2h2, r2l2,
                                                   make_float2(S4.x, S4.y));
            const float2 E1 = gmp_exp_neg2_shifted(make_float2(bh.z, bh.w), make_float2(bl.z, bl.w), nr2h, r2h2, r2l2,
                                                   make_float2(S4.z, S4.w));
#pragma unroll
            for (int l = 0; l < L + 2; ++l) {
              const float4 a = blk[2 + l];
              Rp[0][l] = gmp_fma2(make_float2(a.x, a.y), E0, Rp[0][l]);
              Rp[1][l] = gmp_fma2(make_float2(a.z, a.w), E1, Rp[1][l]);
            }
          }
#pragma unroll
          for (int l = 0; l < L + 2; ++l)
            *reinterpret_cast<float4*>(rrow + l * NS + 4 * sg) =
                make_float4(Rp[0][l].x, Rp[0][l].y, Rp[1][l].x, Rp[1][l].y);
        }
        if (t + s == 0 || K.jac_row[p - 1] != row_id) K.jac_j[r0 + row_id] = j;
      }
      __syncwarp();
      const int m = min(NS, n_max - t);
#pragma unroll 1
      for (int u = 0; u < m; ++u) {
        const int row = __shfl_sync(0xffffffffu, row_id, g * NS + u);
        if (row < 0) continue;  // past this group's pairs
        const int pr = g * NS + u;
        const float* srow = Sr + pr * SH::SSTR + 4 * g;
        const float4 d = *reinterpret_cast<const float4*>(Dr + 4 * (pr + g));
        const float* rrow = Rr + pr * SH::RSTR + NS * g + s;
        float S[(SH::NIND + 3) / 4 * 4];
#pragma unroll
        for (int c = 0; c < (SH::NIND + 3) / 4; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(srow + 4 * c);
          S[4 * c] = v.x; S[4 * c + 1] = v.y; S[4 * c + 2] = v.z; S[4 * c + 3] = v.w;
        }
        float Rn = rrow[0], a[L + 1][3];
#pragma unroll
        for (int l = 0; l <= L; ++l) {
          const float Rl = Rn;
          Rn = rrow[(l + 1) * NS];
          a[l][0] = a[l][1] = a[l][2] = 0.0f;
          if (col[l] < 0) continue;
          float Pl = 0.0f;
#pragma unroll
          for (int k = l * l; k < (l + 1) * (l + 1); ++k) Pl = __fmaf_rn(lam[k], S[k], Pl);
          const float c = __fmul_rn(__fmul_rn(nb2, Rn), Pl);  // dR_l/dr^2 = -beta R_{l+1}
          const float dv[3] = {d.x, d.y, d.z};
#pragma unroll
          for (int v = 0; v < 3; ++v) {
            float W = 0.0f;
            if (l > 0)
#pragma unroll
              for (int k = (l > 0 ? l - 1 : 0) * (l - 1); k < l * l; ++k) W = __fmaf_rn(M[v][k], S[k], W);
            a[l][v] = __fmaf_rn(dv[v], c, __fmul_rn(Rl, W));
          }
        }
        const float da[3] = {__fmul_rn(d.w, d.x), __fmul_rn(d.w, d.y), __fmul_rn(d.w, d.z)};
        if (row != cur) {  // the first pair of a row
          flush();
          cur = row;
#pragma unroll
          for (int l = 0; l <= L; ++l)
#pragma unroll
            for (int v = 0; v < 3; ++v) acc[l][v] = a[l][v];
          dacc[0] = da[0]; dacc[1] = da[1]; dacc[2] = da[2];
        } else {
#pragma unroll
          for (int l = 0; l <= L; ++l)
#pragma unroll
            for (int v = 0; v < 3; ++v) acc[l][v] += a[l][v];
          dacc[0] += da[0]; dacc[1] += da[1]; dacc[2] += da[2];
        }
      }
    }
    flush();
    // own row: the groups' sums of minus the other atoms' rows
#pragma unroll
    for (int l = 0; l <= L; ++l)
#pragma unroll
      for (int v = 0; v < 3; ++v)
#pragma unroll
        for (int k = NS; k < 32; k <<= 1) self[l][v] += __shfl_xor_sync(0xffffffffu, self[l][v], k);
#pragma unroll
    for (int v = 0; v < 3; ++v)
#pragma unroll
      for (int k = NS; k < 32; k <<= 1) dself[v] += __shfl_xor_sync(0xffffffffu, dself[v], k);
    if (g == 0 && r_self >= 0) write_row(r0 + r_self, self, dself);
    __syncwarp();
  }
}

}  // namespace gmpk
