// Generated by gen_mcsh.py -- do not edit.  MCSH angular probes (independent
// components a <= 1 of each order), their gradients, and the per-order
// rotation invariant with its adjoint.  See gen_mcsh.py for the derivation.
#pragma once
#define GMP_MCSH_LMAX 6

__device__ __forceinline__ void gmp_mcsh_indep_0(float x, float y, float z, float r2, float* __restrict__ S) {
  S[0] = 1.0f;
}
__device__ __forceinline__ void gmp_mcsh_indep_1(float x, float y, float z, float r2, float* __restrict__ S) {
  S[0] = 1.0f;
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
}
__device__ __forceinline__ void gmp_mcsh_indep_2(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_3 = __fmul_rn(3.0f, z);
  S[0] = 1.0f;
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
  S[4] = __fmaf_rn(r2_m1, S[0], __fmul_rn(y_3, S[1]));
  S[5] = __fmaf_rn(z_2, S[1], __fmul_rn(y, S[2]));
  S[6] = __fmaf_rn(r2_m1, S[0], __fmul_rn(z_3, S[2]));
  S[7] = __fmaf_rn(y_2, S[3], __fmul_rn(x, S[1]));
  S[8] = __fmaf_rn(z_2, S[3], __fmul_rn(x, S[2]));
}
__device__ __forceinline__ void gmp_mcsh_indep_3(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_3 = __fmul_rn(3.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_5 = __fmul_rn(5.0f, z);
  S[0] = 1.0f;
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
  S[4] = __fmaf_rn(r2_m1, S[0], __fmul_rn(y_3, S[1]));
  S[5] = __fmaf_rn(z_2, S[1], __fmul_rn(y, S[2]));
  S[6] = __fmaf_rn(r2_m1, S[0], __fmul_rn(z_3, S[2]));
  S[7] = __fmaf_rn(y_2, S[3], __fmul_rn(x, S[1]));
  S[8] = __fmaf_rn(z_2, S[3], __fmul_rn(x, S[2]));
  S[9] = __fmaf_rn(r2_m4, S[1], __fmul_rn(y_5, S[4]));
  S[10] = __fmaf_rn(r2_m1, S[2], __fmaf_rn(z_2, S[4], __fmul_rn(y_3, S[5])));
  S[11] = __fmaf_rn(r2_m2, S[1], __fmaf_rn(z_4, S[5], __fmul_rn(y, S[6])));
  S[12] = __fmaf_rn(r2_m4, S[2], __fmul_rn(z_5, S[6]));
  S[13] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(y_4, S[7], __fmul_rn(x, S[4])));
  S[14] = __fmaf_rn(z_2, S[7], __fmaf_rn(y_2, S[8], __fmul_rn(x, S[5])));
  S[15] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(z_4, S[8], __fmul_rn(x, S[6])));
}
__device__ __forceinline__ void gmp_mcsh_indep_4(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_3 = __fmul_rn(3.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_5 = __fmul_rn(5.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_7 = __fmul_rn(7.0f, z);
  S[0] = 1.0f;
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
  S[4] = __fmaf_rn(r2_m1, S[0], __fmul_rn(y_3, S[1]));
  S[5] = __fmaf_rn(z_2, S[1], __fmul_rn(y, S[2]));
  S[6] = __fmaf_rn(r2_m1, S[0], __fmul_rn(z_3, S[2]));
  S[7] = __fmaf_rn(y_2, S[3], __fmul_rn(x, S[1]));
  S[8] = __fmaf_rn(z_2, S[3], __fmul_rn(x, S[2]));
  S[9] = __fmaf_rn(r2_m4, S[1], __fmul_rn(y_5, S[4]));
  S[10] = __fmaf_rn(r2_m1, S[2], __fmaf_rn(z_2, S[4], __fmul_rn(y_3, S[5])));
  S[11] = __fmaf_rn(r2_m2, S[1], __fmaf_rn(z_4, S[5], __fmul_rn(y, S[6])));
  S[12] = __fmaf_rn(r2_m4, S[2], __fmul_rn(z_5, S[6]));
  S[13] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(y_4, S[7], __fmul_rn(x, S[4])));
  S[14] = __fmaf_rn(z_2, S[7], __fmaf_rn(y_2, S[8], __fmul_rn(x, S[5])));
  S[15] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(z_4, S[8], __fmul_rn(x, S[6])));
  S[16] = __fmaf_rn(r2_m9, S[4], __fmul_rn(y_7, S[9]));
  S[17] = __fmaf_rn(r2_m4, S[5], __fmaf_rn(z_2, S[9], __fmul_rn(y_5, S[10])));
  S[18] = __fmaf_rn(r2_m2, S[4], __fmaf_rn(r2_m1, S[6], __fmaf_rn(z_4, S[10], __fmul_rn(y_3, S[11]))));
  S[19] = __fmaf_rn(r2_m6, S[5], __fmaf_rn(z_6, S[11], __fmul_rn(y, S[12])));
  S[20] = __fmaf_rn(r2_m9, S[6], __fmul_rn(z_7, S[12]));
  S[21] = __fmaf_rn(r2_m6, S[7], __fmaf_rn(y_6, S[13], __fmul_rn(x, S[9])));
  S[22] = __fmaf_rn(r2_m2, S[8], __fmaf_rn(z_2, S[13], __fmaf_rn(y_4, S[14], __fmul_rn(x, S[10]))));
  S[23] = __fmaf_rn(r2_m2, S[7], __fmaf_rn(z_4, S[14], __fmaf_rn(y_2, S[15], __fmul_rn(x, S[11]))));
  S[24] = __fmaf_rn(r2_m6, S[8], __fmaf_rn(z_6, S[15], __fmul_rn(x, S[12])));
}
__device__ __forceinline__ void gmp_mcsh_indep_5(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m12 = __fmul_rn(-12.0f, r2);
  const float r2_m16 = __fmul_rn(-16.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float y_8 = __fmul_rn(8.0f, y);
  const float y_9 = __fmul_rn(9.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_3 = __fmul_rn(3.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_5 = __fmul_rn(5.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_7 = __fmul_rn(7.0f, z);
  const float z_8 = __fmul_rn(8.0f, z);
  const float z_9 = __fmul_rn(9.0f, z);
  S[0] = 1.0f;
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
  S[4] = __fmaf_rn(r2_m1, S[0], __fmul_rn(y_3, S[1]));
  S[5] = __fmaf_rn(z_2, S[1], __fmul_rn(y, S[2]));
  S[6] = __fmaf_rn(r2_m1, S[0], __fmul_rn(z_3, S[2]));
  S[7] = __fmaf_rn(y_2, S[3], __fmul_rn(x, S[1]));
  S[8] = __fmaf_rn(z_2, S[3], __fmul_rn(x, S[2]));
  S[9] = __fmaf_rn(r2_m4, S[1], __fmul_rn(y_5, S[4]));
  S[10] = __fmaf_rn(r2_m1, S[2], __fmaf_rn(z_2, S[4], __fmul_rn(y_3, S[5])));
  S[11] = __fmaf_rn(r2_m2, S[1], __fmaf_rn(z_4, S[5], __fmul_rn(y, S[6])));
  S[12] = __fmaf_rn(r2_m4, S[2], __fmul_rn(z_5, S[6]));
  S[13] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(y_4, S[7], __fmul_rn(x, S[4])));
  S[14] = __fmaf_rn(z_2, S[7], __fmaf_rn(y_2, S[8], __fmul_rn(x, S[5])));
  S[15] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(z_4, S[8], __fmul_rn(x, S[6])));
  S[16] = __fmaf_rn(r2_m9, S[4], __fmul_rn(y_7, S[9]));
  S[17] = __fmaf_rn(r2_m4, S[5], __fmaf_rn(z_2, S[9], __fmul_rn(y_5, S[10])));
  S[18] = __fmaf_rn(r2_m2, S[4], __fmaf_rn(r2_m1, S[6], __fmaf_rn(z_4, S[10], __fmul_rn(y_3, S[11]))));
  S[19] = __fmaf_rn(r2_m6, S[5], __fmaf_rn(z_6, S[11], __fmul_rn(y, S[12])));
  S[20] = __fmaf_rn(r2_m9, S[6], __fmul_rn(z_7, S[12]));
  S[21] = __fmaf_rn(r2_m6, S[7], __fmaf_rn(y_6, S[13], __fmul_rn(x, S[9])));
  S[22] = __fmaf_rn(r2_m2, S[8], __fmaf_rn(z_2, S[13], __fmaf_rn(y_4, S[14], __fmul_rn(x, S[10]))));
  S[23] = __fmaf_rn(r2_m2, S[7], __fmaf_rn(z_4, S[14], __fmaf_rn(y_2, S[15], __fmul_rn(x, S[11]))));
  S[24] = __fmaf_rn(r2_m6, S[8], __fmaf_rn(z_6, S[15], __fmul_rn(x, S[12])));
  S[25] = __fmaf_rn(r2_m16, S[9], __fmul_rn(y_9, S[16]));
  S[26] = __fmaf_rn(r2_m9, S[10], __fmaf_rn(z_2, S[16], __fmul_rn(y_7, S[17])));
  S[27] = __fmaf_rn(r2_m2, S[9], __fmaf_rn(r2_m4, S[11], __fmaf_rn(z_4, S[17], __fmul_rn(y_5, S[18]))));
  S[28] = __fmaf_rn(r2_m6, S[10], __fmaf_rn(r2_m1, S[12], __fmaf_rn(z_6, S[18], __fmul_rn(y_3, S[19]))));
  S[29] = __fmaf_rn(r2_m12, S[11], __fmaf_rn(z_8, S[19], __fmul_rn(y, S[20])));
  S[30] = __fmaf_rn(r2_m16, S[12], __fmul_rn(z_9, S[20]));
  S[31] = __fmaf_rn(r2_m12, S[13], __fmaf_rn(y_8, S[21], __fmul_rn(x, S[16])));
  S[32] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_2, S[21], __fmaf_rn(y_6, S[22], __fmul_rn(x, S[17]))));
  S[33] = __fmaf_rn(r2_m2, S[13], __fmaf_rn(r2_m2, S[15], __fmaf_rn(z_4, S[22], __fmaf_rn(y_4, S[23], __fmul_rn(x, S[18])))));
  S[34] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_6, S[23], __fmaf_rn(y_2, S[24], __fmul_rn(x, S[19]))));
  S[35] = __fmaf_rn(r2_m12, S[15], __fmaf_rn(z_8, S[24], __fmul_rn(x, S[20])));
}
__device__ __forceinline__ void gmp_mcsh_indep_6(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m12 = __fmul_rn(-12.0f, r2);
  const float r2_m16 = __fmul_rn(-16.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m20 = __fmul_rn(-20.0f, r2);
  const float r2_m25 = __fmul_rn(-25.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_10 = __fmul_rn(10.0f, y);
  const float y_11 = __fmul_rn(11.0f, y);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float y_8 = __fmul_rn(8.0f, y);
  const float y_9 = __fmul_rn(9.0f, y);
  const float z_10 = __fmul_rn(10.0f, z);
  const float z_11 = __fmul_rn(11.0f, z);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_3 = __fmul_rn(3.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_5 = __fmul_rn(5.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_7 = __fmul_rn(7.0f, z);
  const float z_8 = __fmul_rn(8.0f, z);
  const float z_9 = __fmul_rn(9.0f, z);
  S[0] = 1.0f;
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
  S[4] = __fmaf_rn(r2_m1, S[0], __fmul_rn(y_3, S[1]));
  S[5] = __fmaf_rn(z_2, S[1], __fmul_rn(y, S[2]));
  S[6] = __fmaf_rn(r2_m1, S[0], __fmul_rn(z_3, S[2]));
  S[7] = __fmaf_rn(y_2, S[3], __fmul_rn(x, S[1]));
  S[8] = __fmaf_rn(z_2, S[3], __fmul_rn(x, S[2]));
  S[9] = __fmaf_rn(r2_m4, S[1], __fmul_rn(y_5, S[4]));
  S[10] = __fmaf_rn(r2_m1, S[2], __fmaf_rn(z_2, S[4], __fmul_rn(y_3, S[5])));
  S[11] = __fmaf_rn(r2_m2, S[1], __fmaf_rn(z_4, S[5], __fmul_rn(y, S[6])));
  S[12] = __fmaf_rn(r2_m4, S[2], __fmul_rn(z_5, S[6]));
  S[13] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(y_4, S[7], __fmul_rn(x, S[4])));
  S[14] = __fmaf_rn(z_2, S[7], __fmaf_rn(y_2, S[8], __fmul_rn(x, S[5])));
  S[15] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(z_4, S[8], __fmul_rn(x, S[6])));
  S[16] = __fmaf_rn(r2_m9, S[4], __fmul_rn(y_7, S[9]));
  S[17] = __fmaf_rn(r2_m4, S[5], __fmaf_rn(z_2, S[9], __fmul_rn(y_5, S[10])));
  S[18] = __fmaf_rn(r2_m2, S[4], __fmaf_rn(r2_m1, S[6], __fmaf_rn(z_4, S[10], __fmul_rn(y_3, S[11]))));
  S[19] = __fmaf_rn(r2_m6, S[5], __fmaf_rn(z_6, S[11], __fmul_rn(y, S[12])));
  S[20] = __fmaf_rn(r2_m9, S[6], __fmul_rn(z_7, S[12]));
  S[21] = __fmaf_rn(r2_m6, S[7], __fmaf_rn(y_6, S[13], __fmul_rn(x, S[9])));
  S[22] = __fmaf_rn(r2_m2, S[8], __fmaf_rn(z_2, S[13], __fmaf_rn(y_4, S[14], __fmul_rn(x, S[10]))));
  S[23] = __fmaf_rn(r2_m2, S[7], __fmaf_rn(z_4, S[14], __fmaf_rn(y_2, S[15], __fmul_rn(x, S[11]))));
  S[24] = __fmaf_rn(r2_m6, S[8], __fmaf_rn(z_6, S[15], __fmul_rn(x, S[12])));
  S[25] = __fmaf_rn(r2_m16, S[9], __fmul_rn(y_9, S[16]));
  S[26] = __fmaf_rn(r2_m9, S[10], __fmaf_rn(z_2, S[16], __fmul_rn(y_7, S[17])));
  S[27] = __fmaf_rn(r2_m2, S[9], __fmaf_rn(r2_m4, S[11], __fmaf_rn(z_4, S[17], __fmul_rn(y_5, S[18]))));
  S[28] = __fmaf_rn(r2_m6, S[10], __fmaf_rn(r2_m1, S[12], __fmaf_rn(z_6, S[18], __fmul_rn(y_3, S[19]))));
  S[29] = __fmaf_rn(r2_m12, S[11], __fmaf_rn(z_8, S[19], __fmul_rn(y, S[20])));
  S[30] = __fmaf_rn(r2_m16, S[12], __fmul_rn(z_9, S[20]));
  S[31] = __fmaf_rn(r2_m12, S[13], __fmaf_rn(y_8, S[21], __fmul_rn(x, S[16])));
  S[32] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_2, S[21], __fmaf_rn(y_6, S[22], __fmul_rn(x, S[17]))));
  S[33] = __fmaf_rn(r2_m2, S[13], __fmaf_rn(r2_m2, S[15], __fmaf_rn(z_4, S[22], __fmaf_rn(y_4, S[23], __fmul_rn(x, S[18])))));
  S[34] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_6, S[23], __fmaf_rn(y_2, S[24], __fmul_rn(x, S[19]))));
  S[35] = __fmaf_rn(r2_m12, S[15], __fmaf_rn(z_8, S[24], __fmul_rn(x, S[20])));
  S[36] = __fmaf_rn(r2_m25, S[16], __fmul_rn(y_11, S[25]));
  S[37] = __fmaf_rn(r2_m16, S[17], __fmaf_rn(z_2, S[25], __fmul_rn(y_9, S[26])));
  S[38] = __fmaf_rn(r2_m2, S[16], __fmaf_rn(r2_m9, S[18], __fmaf_rn(z_4, S[26], __fmul_rn(y_7, S[27]))));
  S[39] = __fmaf_rn(r2_m6, S[17], __fmaf_rn(r2_m4, S[19], __fmaf_rn(z_6, S[27], __fmul_rn(y_5, S[28]))));
  S[40] = __fmaf_rn(r2_m12, S[18], __fmaf_rn(r2_m1, S[20], __fmaf_rn(z_8, S[28], __fmul_rn(y_3, S[29]))));
  S[41] = __fmaf_rn(r2_m20, S[19], __fmaf_rn(z_10, S[29], __fmul_rn(y, S[30])));
  S[42] = __fmaf_rn(r2_m25, S[20], __fmul_rn(z_11, S[30]));
  S[43] = __fmaf_rn(r2_m20, S[21], __fmaf_rn(y_10, S[31], __fmul_rn(x, S[25])));
  S[44] = __fmaf_rn(r2_m12, S[22], __fmaf_rn(z_2, S[31], __fmaf_rn(y_8, S[32], __fmul_rn(x, S[26]))));
  S[45] = __fmaf_rn(r2_m2, S[21], __fmaf_rn(r2_m6, S[23], __fmaf_rn(z_4, S[32], __fmaf_rn(y_6, S[33], __fmul_rn(x, S[27])))));
  S[46] = __fmaf_rn(r2_m6, S[22], __fmaf_rn(r2_m2, S[24], __fmaf_rn(z_6, S[33], __fmaf_rn(y_4, S[34], __fmul_rn(x, S[28])))));
  S[47] = __fmaf_rn(r2_m12, S[23], __fmaf_rn(z_8, S[34], __fmaf_rn(y_2, S[35], __fmul_rn(x, S[29]))));
  S[48] = __fmaf_rn(r2_m20, S[24], __fmaf_rn(z_10, S[35], __fmul_rn(x, S[30])));
}
__device__ __forceinline__ void gmp_mcsh_indep_7(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m12 = __fmul_rn(-12.0f, r2);
  const float r2_m16 = __fmul_rn(-16.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m20 = __fmul_rn(-20.0f, r2);
  const float r2_m25 = __fmul_rn(-25.0f, r2);
  const float r2_m30 = __fmul_rn(-30.0f, r2);
  const float r2_m36 = __fmul_rn(-36.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_10 = __fmul_rn(10.0f, y);
  const float y_11 = __fmul_rn(11.0f, y);
  const float y_12 = __fmul_rn(12.0f, y);
  const float y_13 = __fmul_rn(13.0f, y);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float y_8 = __fmul_rn(8.0f, y);
  const float y_9 = __fmul_rn(9.0f, y);
  const float z_10 = __fmul_rn(10.0f, z);
  const float z_11 = __fmul_rn(11.0f, z);
  const float z_12 = __fmul_rn(12.0f, z);
  const float z_13 = __fmul_rn(13.0f, z);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_3 = __fmul_rn(3.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_5 = __fmul_rn(5.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_7 = __fmul_rn(7.0f, z);
  const float z_8 = __fmul_rn(8.0f, z);
  const float z_9 = __fmul_rn(9.0f, z);
  S[0] = 1.0f;
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
  S[4] = __fmaf_rn(r2_m1, S[0], __fmul_rn(y_3, S[1]));
  S[5] = __fmaf_rn(z_2, S[1], __fmul_rn(y, S[2]));
  S[6] = __fmaf_rn(r2_m1, S[0], __fmul_rn(z_3, S[2]));
  S[7] = __fmaf_rn(y_2, S[3], __fmul_rn(x, S[1]));
  S[8] = __fmaf_rn(z_2, S[3], __fmul_rn(x, S[2]));
  S[9] = __fmaf_rn(r2_m4, S[1], __fmul_rn(y_5, S[4]));
  S[10] = __fmaf_rn(r2_m1, S[2], __fmaf_rn(z_2, S[4], __fmul_rn(y_3, S[5])));
  S[11] = __fmaf_rn(r2_m2, S[1], __fmaf_rn(z_4, S[5], __fmul_rn(y, S[6])));
  S[12] = __fmaf_rn(r2_m4, S[2], __fmul_rn(z_5, S[6]));
  S[13] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(y_4, S[7], __fmul_rn(x, S[4])));
  S[14] = __fmaf_rn(z_2, S[7], __fmaf_rn(y_2, S[8], __fmul_rn(x, S[5])));
  S[15] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(z_4, S[8], __fmul_rn(x, S[6])));
  S[16] = __fmaf_rn(r2_m9, S[4], __fmul_rn(y_7, S[9]));
  S[17] = __fmaf_rn(r2_m4, S[5], __fmaf_rn(z_2, S[9], __fmul_rn(y_5, S[10])));
  S[18] = __fmaf_rn(r2_m2, S[4], __fmaf_rn(r2_m1, S[6], __fmaf_rn(z_4, S[10], __fmul_rn(y_3, S[11]))));
  S[19] = __fmaf_rn(r2_m6, S[5], __fmaf_rn(z_6, S[11], __fmul_rn(y, S[12])));
  S[20] = __fmaf_rn(r2_m9, S[6], __fmul_rn(z_7, S[12]));
  S[21] = __fmaf_rn(r2_m6, S[7], __fmaf_rn(y_6, S[13], __fmul_rn(x, S[9])));
  S[22] = __fmaf_rn(r2_m2, S[8], __fmaf_rn(z_2, S[13], __fmaf_rn(y_4, S[14], __fmul_rn(x, S[10]))));
  S[23] = __fmaf_rn(r2_m2, S[7], __fmaf_rn(z_4, S[14], __fmaf_rn(y_2, S[15], __fmul_rn(x, S[11]))));
  S[24] = __fmaf_rn(r2_m6, S[8], __fmaf_rn(z_6, S[15], __fmul_rn(x, S[12])));
  S[25] = __fmaf_rn(r2_m16, S[9], __fmul_rn(y_9, S[16]));
  S[26] = __fmaf_rn(r2_m9, S[10], __fmaf_rn(z_2, S[16], __fmul_rn(y_7, S[17])));
  S[27] = __fmaf_rn(r2_m2, S[9], __fmaf_rn(r2_m4, S[11], __fmaf_rn(z_4, S[17], __fmul_rn(y_5, S[18]))));
  S[28] = __fmaf_rn(r2_m6, S[10], __fmaf_rn(r2_m1, S[12], __fmaf_rn(z_6, S[18], __fmul_rn(y_3, S[19]))));
  S[29] = __fmaf_rn(r2_m12, S[11], __fmaf_rn(z_8, S[19], __fmul_rn(y, S[20])));
  S[30] = __fmaf_rn(r2_m16, S[12], __fmul_rn(z_9, S[20]));
  S[31] = __fmaf_rn(r2_m12, S[13], __fmaf_rn(y_8, S[21], __fmul_rn(x, S[16])));
  S[32] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_2, S[21], __fmaf_rn(y_6, S[22], __fmul_rn(x, S[17]))));
  S[33] = __fmaf_rn(r2_m2, S[13], __fmaf_rn(r2_m2, S[15], __fmaf_rn(z_4, S[22], __fmaf_rn(y_4, S[23], __fmul_rn(x, S[18])))));
  S[34] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_6, S[23], __fmaf_rn(y_2, S[24], __fmul_rn(x, S[19]))));
  S[35] = __fmaf_rn(r2_m12, S[15], __fmaf_rn(z_8, S[24], __fmul_rn(x, S[20])));
  S[36] = __fmaf_rn(r2_m25, S[16], __fmul_rn(y_11, S[25]));
  S[37] = __fmaf_rn(r2_m16, S[17], __fmaf_rn(z_2, S[25], __fmul_rn(y_9, S[26])));
  S[38] = __fmaf_rn(r2_m2, S[16], __fmaf_rn(r2_m9, S[18], __fmaf_rn(z_4, S[26], __fmul_rn(y_7, S[27]))));
  S[39] = __fmaf_rn(r2_m6, S[17], __fmaf_rn(r2_m4, S[19], __fmaf_rn(z_6, S[27], __fmul_rn(y_5, S[28]))));
  S[40] = __fmaf_rn(r2_m12, S[18], __fmaf_rn(r2_m1, S[20], __fmaf_rn(z_8, S[28], __fmul_rn(y_3, S[29]))));
  S[41] = __fmaf_rn(r2_m20, S[19], __fmaf_rn(z_10, S[29], __fmul_rn(y, S[30])));
  S[42] = __fmaf_rn(r2_m25, S[20], __fmul_rn(z_11, S[30]));
  S[43] = __fmaf_rn(r2_m20, S[21], __fmaf_rn(y_10, S[31], __fmul_rn(x, S[25])));
  S[44] = __fmaf_rn(r2_m12, S[22], __fmaf_rn(z_2, S[31], __fmaf_rn(y_8, S[32], __fmul_rn(x, S[26]))));
  S[45] = __fmaf_rn(r2_m2, S[21], __fmaf_rn(r2_m6, S[23], __fmaf_rn(z_4, S[32], __fmaf_rn(y_6, S[33], __fmul_rn(x, S[27])))));
  S[46] = __fmaf_rn(r2_m6, S[22], __fmaf_rn(r2_m2, S[24], __fmaf_rn(z_6, S[33], __fmaf_rn(y_4, S[34], __fmul_rn(x, S[28])))));
  S[47] = __fmaf_rn(r2_m12, S[23], __fmaf_rn(z_8, S[34], __fmaf_rn(y_2, S[35], __fmul_rn(x, S[29]))));
  S[48] = __fmaf_rn(r2_m20, S[24], __fmaf_rn(z_10, S[35], __fmul_rn(x, S[30])));
  S[49] = __fmaf_rn(r2_m36, S[25], __fmul_rn(y_13, S[36]));
  S[50] = __fmaf_rn(r2_m25, S[26], __fmaf_rn(z_2, S[36], __fmul_rn(y_11, S[37])));
  S[51] = __fmaf_rn(r2_m2, S[25], __fmaf_rn(r2_m16, S[27], __fmaf_rn(z_4, S[37], __fmul_rn(y_9, S[38]))));
  S[52] = __fmaf_rn(r2_m6, S[26], __fmaf_rn(r2_m9, S[28], __fmaf_rn(z_6, S[38], __fmul_rn(y_7, S[39]))));
  S[53] = __fmaf_rn(r2_m12, S[27], __fmaf_rn(r2_m4, S[29], __fmaf_rn(z_8, S[39], __fmul_rn(y_5, S[40]))));
  S[54] = __fmaf_rn(r2_m20, S[28], __fmaf_rn(r2_m1, S[30], __fmaf_rn(z_10, S[40], __fmul_rn(y_3, S[41]))));
  S[55] = __fmaf_rn(r2_m30, S[29], __fmaf_rn(z_12, S[41], __fmul_rn(y, S[42])));
  S[56] = __fmaf_rn(r2_m36, S[30], __fmul_rn(z_13, S[42]));
  S[57] = __fmaf_rn(r2_m30, S[31], __fmaf_rn(y_12, S[43], __fmul_rn(x, S[36])));
  S[58] = __fmaf_rn(r2_m20, S[32], __fmaf_rn(z_2, S[43], __fmaf_rn(y_10, S[44], __fmul_rn(x, S[37]))));
  S[59] = __fmaf_rn(r2_m2, S[31], __fmaf_rn(r2_m12, S[33], __fmaf_rn(z_4, S[44], __fmaf_rn(y_8, S[45], __fmul_rn(x, S[38])))));
  S[60] = __fmaf_rn(r2_m6, S[32], __fmaf_rn(r2_m6, S[34], __fmaf_rn(z_6, S[45], __fmaf_rn(y_6, S[46], __fmul_rn(x, S[39])))));
  S[61] = __fmaf_rn(r2_m12, S[33], __fmaf_rn(r2_m2, S[35], __fmaf_rn(z_8, S[46], __fmaf_rn(y_4, S[47], __fmul_rn(x, S[40])))));
  S[62] = __fmaf_rn(r2_m20, S[34], __fmaf_rn(z_10, S[47], __fmaf_rn(y_2, S[48], __fmul_rn(x, S[41]))));
  S[63] = __fmaf_rn(r2_m30, S[35], __fmaf_rn(z_12, S[48], __fmul_rn(x, S[42])));
}
__device__ __forceinline__ void gmp_mcsh_top_1(float x, float y, float z, float r2, float* __restrict__ S) {
  S[1] = __fmul_rn(y, S[0]);
  S[2] = __fmul_rn(z, S[0]);
  S[3] = __fmul_rn(x, S[0]);
}
__device__ __forceinline__ void gmp_mcsh_top_2(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_3 = __fmul_rn(3.0f, z);
  S[4] = __fmaf_rn(r2_m1, S[0], __fmul_rn(y_3, S[1]));
  S[5] = __fmaf_rn(z_2, S[1], __fmul_rn(y, S[2]));
  S[6] = __fmaf_rn(r2_m1, S[0], __fmul_rn(z_3, S[2]));
  S[7] = __fmaf_rn(y_2, S[3], __fmul_rn(x, S[1]));
  S[8] = __fmaf_rn(z_2, S[3], __fmul_rn(x, S[2]));
}
__device__ __forceinline__ void gmp_mcsh_top_3(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_5 = __fmul_rn(5.0f, z);
  S[9] = __fmaf_rn(r2_m4, S[1], __fmul_rn(y_5, S[4]));
  S[10] = __fmaf_rn(r2_m1, S[2], __fmaf_rn(z_2, S[4], __fmul_rn(y_3, S[5])));
  S[11] = __fmaf_rn(r2_m2, S[1], __fmaf_rn(z_4, S[5], __fmul_rn(y, S[6])));
  S[12] = __fmaf_rn(r2_m4, S[2], __fmul_rn(z_5, S[6]));
  S[13] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(y_4, S[7], __fmul_rn(x, S[4])));
  S[14] = __fmaf_rn(z_2, S[7], __fmaf_rn(y_2, S[8], __fmul_rn(x, S[5])));
  S[15] = __fmaf_rn(r2_m2, S[3], __fmaf_rn(z_4, S[8], __fmul_rn(x, S[6])));
}
__device__ __forceinline__ void gmp_mcsh_top_4(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_7 = __fmul_rn(7.0f, z);
  S[16] = __fmaf_rn(r2_m9, S[4], __fmul_rn(y_7, S[9]));
  S[17] = __fmaf_rn(r2_m4, S[5], __fmaf_rn(z_2, S[9], __fmul_rn(y_5, S[10])));
  S[18] = __fmaf_rn(r2_m2, S[4], __fmaf_rn(r2_m1, S[6], __fmaf_rn(z_4, S[10], __fmul_rn(y_3, S[11]))));
  S[19] = __fmaf_rn(r2_m6, S[5], __fmaf_rn(z_6, S[11], __fmul_rn(y, S[12])));
  S[20] = __fmaf_rn(r2_m9, S[6], __fmul_rn(z_7, S[12]));
  S[21] = __fmaf_rn(r2_m6, S[7], __fmaf_rn(y_6, S[13], __fmul_rn(x, S[9])));
  S[22] = __fmaf_rn(r2_m2, S[8], __fmaf_rn(z_2, S[13], __fmaf_rn(y_4, S[14], __fmul_rn(x, S[10]))));
  S[23] = __fmaf_rn(r2_m2, S[7], __fmaf_rn(z_4, S[14], __fmaf_rn(y_2, S[15], __fmul_rn(x, S[11]))));
  S[24] = __fmaf_rn(r2_m6, S[8], __fmaf_rn(z_6, S[15], __fmul_rn(x, S[12])));
}
__device__ __forceinline__ void gmp_mcsh_top_5(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m12 = __fmul_rn(-12.0f, r2);
  const float r2_m16 = __fmul_rn(-16.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float y_8 = __fmul_rn(8.0f, y);
  const float y_9 = __fmul_rn(9.0f, y);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_8 = __fmul_rn(8.0f, z);
  const float z_9 = __fmul_rn(9.0f, z);
  S[25] = __fmaf_rn(r2_m16, S[9], __fmul_rn(y_9, S[16]));
  S[26] = __fmaf_rn(r2_m9, S[10], __fmaf_rn(z_2, S[16], __fmul_rn(y_7, S[17])));
  S[27] = __fmaf_rn(r2_m2, S[9], __fmaf_rn(r2_m4, S[11], __fmaf_rn(z_4, S[17], __fmul_rn(y_5, S[18]))));
  S[28] = __fmaf_rn(r2_m6, S[10], __fmaf_rn(r2_m1, S[12], __fmaf_rn(z_6, S[18], __fmul_rn(y_3, S[19]))));
  S[29] = __fmaf_rn(r2_m12, S[11], __fmaf_rn(z_8, S[19], __fmul_rn(y, S[20])));
  S[30] = __fmaf_rn(r2_m16, S[12], __fmul_rn(z_9, S[20]));
  S[31] = __fmaf_rn(r2_m12, S[13], __fmaf_rn(y_8, S[21], __fmul_rn(x, S[16])));
  S[32] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_2, S[21], __fmaf_rn(y_6, S[22], __fmul_rn(x, S[17]))));
  S[33] = __fmaf_rn(r2_m2, S[13], __fmaf_rn(r2_m2, S[15], __fmaf_rn(z_4, S[22], __fmaf_rn(y_4, S[23], __fmul_rn(x, S[18])))));
  S[34] = __fmaf_rn(r2_m6, S[14], __fmaf_rn(z_6, S[23], __fmaf_rn(y_2, S[24], __fmul_rn(x, S[19]))));
  S[35] = __fmaf_rn(r2_m12, S[15], __fmaf_rn(z_8, S[24], __fmul_rn(x, S[20])));
}
__device__ __forceinline__ void gmp_mcsh_top_6(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m12 = __fmul_rn(-12.0f, r2);
  const float r2_m16 = __fmul_rn(-16.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m20 = __fmul_rn(-20.0f, r2);
  const float r2_m25 = __fmul_rn(-25.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_10 = __fmul_rn(10.0f, y);
  const float y_11 = __fmul_rn(11.0f, y);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float y_8 = __fmul_rn(8.0f, y);
  const float y_9 = __fmul_rn(9.0f, y);
  const float z_10 = __fmul_rn(10.0f, z);
  const float z_11 = __fmul_rn(11.0f, z);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_8 = __fmul_rn(8.0f, z);
  S[36] = __fmaf_rn(r2_m25, S[16], __fmul_rn(y_11, S[25]));
  S[37] = __fmaf_rn(r2_m16, S[17], __fmaf_rn(z_2, S[25], __fmul_rn(y_9, S[26])));
  S[38] = __fmaf_rn(r2_m2, S[16], __fmaf_rn(r2_m9, S[18], __fmaf_rn(z_4, S[26], __fmul_rn(y_7, S[27]))));
  S[39] = __fmaf_rn(r2_m6, S[17], __fmaf_rn(r2_m4, S[19], __fmaf_rn(z_6, S[27], __fmul_rn(y_5, S[28]))));
  S[40] = __fmaf_rn(r2_m12, S[18], __fmaf_rn(r2_m1, S[20], __fmaf_rn(z_8, S[28], __fmul_rn(y_3, S[29]))));
  S[41] = __fmaf_rn(r2_m20, S[19], __fmaf_rn(z_10, S[29], __fmul_rn(y, S[30])));
  S[42] = __fmaf_rn(r2_m25, S[20], __fmul_rn(z_11, S[30]));
  S[43] = __fmaf_rn(r2_m20, S[21], __fmaf_rn(y_10, S[31], __fmul_rn(x, S[25])));
  S[44] = __fmaf_rn(r2_m12, S[22], __fmaf_rn(z_2, S[31], __fmaf_rn(y_8, S[32], __fmul_rn(x, S[26]))));
  S[45] = __fmaf_rn(r2_m2, S[21], __fmaf_rn(r2_m6, S[23], __fmaf_rn(z_4, S[32], __fmaf_rn(y_6, S[33], __fmul_rn(x, S[27])))));
  S[46] = __fmaf_rn(r2_m6, S[22], __fmaf_rn(r2_m2, S[24], __fmaf_rn(z_6, S[33], __fmaf_rn(y_4, S[34], __fmul_rn(x, S[28])))));
  S[47] = __fmaf_rn(r2_m12, S[23], __fmaf_rn(z_8, S[34], __fmaf_rn(y_2, S[35], __fmul_rn(x, S[29]))));
  S[48] = __fmaf_rn(r2_m20, S[24], __fmaf_rn(z_10, S[35], __fmul_rn(x, S[30])));
}
__device__ __forceinline__ void gmp_mcsh_top_7(float x, float y, float z, float r2, float* __restrict__ S) {
  const float r2_m1 = __fmul_rn(-1.0f, r2);
  const float r2_m12 = __fmul_rn(-12.0f, r2);
  const float r2_m16 = __fmul_rn(-16.0f, r2);
  const float r2_m2 = __fmul_rn(-2.0f, r2);
  const float r2_m20 = __fmul_rn(-20.0f, r2);
  const float r2_m25 = __fmul_rn(-25.0f, r2);
  const float r2_m30 = __fmul_rn(-30.0f, r2);
  const float r2_m36 = __fmul_rn(-36.0f, r2);
  const float r2_m4 = __fmul_rn(-4.0f, r2);
  const float r2_m6 = __fmul_rn(-6.0f, r2);
  const float r2_m9 = __fmul_rn(-9.0f, r2);
  const float y_10 = __fmul_rn(10.0f, y);
  const float y_11 = __fmul_rn(11.0f, y);
  const float y_12 = __fmul_rn(12.0f, y);
  const float y_13 = __fmul_rn(13.0f, y);
  const float y_2 = __fmul_rn(2.0f, y);
  const float y_3 = __fmul_rn(3.0f, y);
  const float y_4 = __fmul_rn(4.0f, y);
  const float y_5 = __fmul_rn(5.0f, y);
  const float y_6 = __fmul_rn(6.0f, y);
  const float y_7 = __fmul_rn(7.0f, y);
  const float y_8 = __fmul_rn(8.0f, y);
  const float y_9 = __fmul_rn(9.0f, y);
  const float z_10 = __fmul_rn(10.0f, z);
  const float z_12 = __fmul_rn(12.0f, z);
  const float z_13 = __fmul_rn(13.0f, z);
  const float z_2 = __fmul_rn(2.0f, z);
  const float z_4 = __fmul_rn(4.0f, z);
  const float z_6 = __fmul_rn(6.0f, z);
  const float z_8 = __fmul_rn(8.0f, z);
  S[49] = __fmaf_rn(r2_m36, S[25], __fmul_rn(y_13, S[36]));
  S[50] = __fmaf_rn(r2_m25, S[26], __fmaf_rn(z_2, S[36], __fmul_rn(y_11, S[37])));
  S[51] = __fmaf_rn(r2_m2, S[25], __fmaf_rn(r2_m16, S[27], __fmaf_rn(z_4, S[37], __fmul_rn(y_9, S[38]))));
  S[52] = __fmaf_rn(r2_m6, S[26], __fmaf_rn(r2_m9, S[28], __fmaf_rn(z_6, S[38], __fmul_rn(y_7, S[39]))));
  S[53] = __fmaf_rn(r2_m12, S[27], __fmaf_rn(r2_m4, S[29], __fmaf_rn(z_8, S[39], __fmul_rn(y_5, S[40]))));
  S[54] = __fmaf_rn(r2_m20, S[28], __fmaf_rn(r2_m1, S[30], __fmaf_rn(z_10, S[40], __fmul_rn(y_3, S[41]))));
  S[55] = __fmaf_rn(r2_m30, S[29], __fmaf_rn(z_12, S[41], __fmul_rn(y, S[42])));
  S[56] = __fmaf_rn(r2_m36, S[30], __fmul_rn(z_13, S[42]));
  S[57] = __fmaf_rn(r2_m30, S[31], __fmaf_rn(y_12, S[43], __fmul_rn(x, S[36])));
  S[58] = __fmaf_rn(r2_m20, S[32], __fmaf_rn(z_2, S[43], __fmaf_rn(y_10, S[44], __fmul_rn(x, S[37]))));
  S[59] = __fmaf_rn(r2_m2, S[31], __fmaf_rn(r2_m12, S[33], __fmaf_rn(z_4, S[44], __fmaf_rn(y_8, S[45], __fmul_rn(x, S[38])))));
  S[60] = __fmaf_rn(r2_m6, S[32], __fmaf_rn(r2_m6, S[34], __fmaf_rn(z_6, S[45], __fmaf_rn(y_6, S[46], __fmul_rn(x, S[39])))));
  S[61] = __fmaf_rn(r2_m12, S[33], __fmaf_rn(r2_m2, S[35], __fmaf_rn(z_8, S[46], __fmaf_rn(y_4, S[47], __fmul_rn(x, S[40])))));
  S[62] = __fmaf_rn(r2_m20, S[34], __fmaf_rn(z_10, S[47], __fmaf_rn(y_2, S[48], __fmul_rn(x, S[41]))));
  S[63] = __fmaf_rn(r2_m30, S[35], __fmaf_rn(z_12, S[48], __fmul_rn(x, S[42])));
}
__device__ __forceinline__ void gmp_solid_df_0(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* __restrict__ H) {
  H[0] = gmp_f2{1.0f, 0.0f};
}
__device__ __forceinline__ void gmp_solid_df_1(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* __restrict__ H) {
  gmp_f2 a = x, b = y;
  H[0] = z;
  H[1] = a; H[2] = b;
}
__device__ __forceinline__ void gmp_solid_df_2(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* __restrict__ H) {
  const gmp_f2 z2 = gmp_df_mul(z, z);
  gmp_f2 a = x, b = y;
  H[0] = gmp_df_add_sloppy(gmp_df_mul_fu(z2, 3.0f), gmp_df_mul_fu(r2, -1.0f));
  { const gmp_f2 q = z; H[1] = gmp_df_mul_u(q, a); H[2] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  H[3] = a; H[4] = b;
}
__device__ __forceinline__ void gmp_solid_df_3(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* __restrict__ H) {
  const gmp_f2 z2 = gmp_df_mul(z, z);
  gmp_f2 a = x, b = y;
  H[0] = gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 5.0f), gmp_df_mul_fu(r2, -3.0f)), z);
  { const gmp_f2 q = gmp_df_add_sloppy(gmp_df_mul_fu(z2, 5.0f), gmp_df_mul_fu(r2, -1.0f)); H[1] = gmp_df_mul_u(q, a); H[2] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = z; H[3] = gmp_df_mul_u(q, a); H[4] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  H[5] = a; H[6] = b;
}
__device__ __forceinline__ void gmp_solid_df_4(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* __restrict__ H) {
  const gmp_f2 z2 = gmp_df_mul(z, z);
  const gmp_f2 r2_2 = gmp_df_mul(r2, r2);
  gmp_f2 a = x, b = y;
  H[0] = gmp_df_add_sloppy(gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 35.0f), gmp_df_mul_fu(r2, -30.0f)), z2), gmp_df_mul_fu(r2_2, 3.0f));
  { const gmp_f2 q = gmp_df_mul(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 7.0f), gmp_df_mul_fu(r2, -3.0f)), z); H[1] = gmp_df_mul_u(q, a); H[2] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = gmp_df_add_sloppy(gmp_df_mul_fu(z2, 7.0f), gmp_df_mul_fu(r2, -1.0f)); H[3] = gmp_df_mul_u(q, a); H[4] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = z; H[5] = gmp_df_mul_u(q, a); H[6] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  H[7] = a; H[8] = b;
}
__device__ __forceinline__ void gmp_solid_df_5(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* __restrict__ H) {
  const gmp_f2 z2 = gmp_df_mul(z, z);
  const gmp_f2 r2_2 = gmp_df_mul(r2, r2);
  gmp_f2 a = x, b = y;
  H[0] = gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 63.0f), gmp_df_mul_fu(r2, -70.0f)), z2), gmp_df_mul_fu(r2_2, 15.0f)), z);
  { const gmp_f2 q = gmp_df_add_sloppy(gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 21.0f), gmp_df_mul_fu(r2, -14.0f)), z2), r2_2); H[1] = gmp_df_mul_u(q, a); H[2] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = gmp_df_mul(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 3.0f), gmp_df_mul_fu(r2, -1.0f)), z); H[3] = gmp_df_mul_u(q, a); H[4] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = gmp_df_add_sloppy(gmp_df_mul_fu(z2, 9.0f), gmp_df_mul_fu(r2, -1.0f)); H[5] = gmp_df_mul_u(q, a); H[6] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = z; H[7] = gmp_df_mul_u(q, a); H[8] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  H[9] = a; H[10] = b;
}
__device__ __forceinline__ void gmp_solid_df_6(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* __restrict__ H) {
  const gmp_f2 z2 = gmp_df_mul(z, z);
  const gmp_f2 r2_2 = gmp_df_mul(r2, r2);
  const gmp_f2 r2_3 = gmp_df_mul(r2, r2_2);
  gmp_f2 a = x, b = y;
  H[0] = gmp_df_add_sloppy(gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 231.0f), gmp_df_mul_fu(r2, -315.0f)), z2), gmp_df_mul_fu(r2_2, 105.0f)), z2), gmp_df_mul_fu(r2_3, -5.0f));
  { const gmp_f2 q = gmp_df_mul(gmp_df_add_sloppy(gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 33.0f), gmp_df_mul_fu(r2, -30.0f)), z2), gmp_df_mul_fu(r2_2, 5.0f)), z); H[1] = gmp_df_mul_u(q, a); H[2] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = gmp_df_add_sloppy(gmp_df_mul_u(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 33.0f), gmp_df_mul_fu(r2, -18.0f)), z2), r2_2); H[3] = gmp_df_mul_u(q, a); H[4] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = gmp_df_mul(gmp_df_add_sloppy(gmp_df_mul_fu(z2, 11.0f), gmp_df_mul_fu(r2, -3.0f)), z); H[5] = gmp_df_mul_u(q, a); H[6] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = gmp_df_add_sloppy(gmp_df_mul_fu(z2, 11.0f), gmp_df_mul_fu(r2, -1.0f)); H[7] = gmp_df_mul_u(q, a); H[8] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  { const gmp_f2 q = z; H[9] = gmp_df_mul_u(q, a); H[10] = gmp_df_mul_u(q, b); }
  { const gmp_f2 t = gmp_df_add_sloppy(gmp_df_mul_u(x, a), gmp_df_neg(gmp_df_mul_u(y, b)));
    b = gmp_df_add_sloppy(gmp_df_mul_u(x, b), gmp_df_mul_u(y, a));
    a = t; }
  H[11] = a; H[12] = b;
}
#define GMP_SOLID_NZ 4
static __device__ const float2 gmp_solid_norm[7][13] = {
  {{1.0f, 0.0f}},
  {{1.0f, 0.0f}, {1.0f, 0.0f}, {1.0f, 0.0f}},
  {{1.5f, 0.0f}, {18.0f, 0.0f}, {18.0f, 0.0f}, {4.5f, 0.0f}, {4.5f, 0.0f}},
  {{22.5f, 0.0f}, {33.75f, 0.0f}, {33.75f, 0.0f}, {337.5f, 0.0f}, {337.5f, 0.0f}, {56.25f, 0.0f}, {56.25f, 0.0f}},
  {{39.375f, 0.0f}, {1575.0f, 0.0f}, {1575.0f, 0.0f}, {787.5f, 0.0f}, {787.5f, 0.0f}, {11025.0f, 0.0f}, {11025.0f, 0.0f}, {1378.125f, 0.0f}, {1378.125f, 0.0f}},
  {{1771.875f, 0.0f}, {26578.125f, 0.0f}, {26578.125f, 0.0f}, {744187.5f, 0.0f}, {744187.5f, 0.0f}, {31007.8125f, 0.0f}, {31007.8125f, 0.0f}, {558140.625f, 0.0f}, {558140.625f, 0.0f}, {55814.0625f, 0.0f}, {55814.0625f, 0.0f}},
  {{29235.9375f, 0.0f}, {2455818.75f, 0.0f}, {2455818.75f, 0.0f}, {1534886.75f, -0.03125f}, {1534886.75f, -0.03125f}, {6139547.0f, -0.125f}, {6139547.0f, -0.125f}, {1841864.0f, 0.0625f}, {1841864.0f, 0.0625f}, {40521008.0f, 1.375f}, {40521008.0f, 1.375f}, {3376750.75f, 0.03125f}, {3376750.75f, 0.03125f}},
};
static __device__ const signed char gmp_solid_row[7][13][4] = {
  {{0, 0, 0, 0}},
  {{2, 0, 0, 0}, {0, 0, 0, 0}, {1, 0, 0, 0}},
  {{0, 3, 0, 0}, {2, 0, 0, 0}, {0, 0, 0, 0}, {4, 0, 0, 0}, {1, 0, 0, 0}},
  {{2, 6, 0, 0}, {0, 3, 0, 0}, {2, 0, 0, 0}, {0, 0, 0, 0}, {1, 5, 0, 0}, {4, 0, 0, 0}, {1, 0, 0, 0}},
  {{0, 3, 7, 0}, {2, 6, 0, 0}, {0, 3, 0, 0}, {2, 0, 0, 0}, {0, 0, 0, 0}, {4, 8, 0, 0}, {1, 5, 0, 0}, {4, 0, 0, 0}, {1, 0, 0, 0}},
  {{2, 6, 10, 0}, {0, 3, 7, 0}, {2, 6, 0, 0}, {0, 3, 0, 0}, {2, 0, 0, 0}, {0, 0, 0, 0}, {1, 5, 9, 0}, {4, 8, 0, 0}, {1, 5, 0, 0}, {4, 0, 0, 0}, {1, 0, 0, 0}},
  {{0, 3, 7, 11}, {2, 6, 10, 0}, {0, 3, 7, 0}, {2, 6, 0, 0}, {0, 3, 0, 0}, {2, 0, 0, 0}, {0, 0, 0, 0}, {4, 8, 12, 0}, {1, 5, 9, 0}, {4, 8, 0, 0}, {1, 5, 0, 0}, {4, 0, 0, 0}, {1, 0, 0, 0}},
};
static __device__ const float2 gmp_solid_coef[7][13][4] = {
  {{{1.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}},
  {{{1.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{1.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{1.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}},
  {{{-0.5f, 0.0f}, {-1.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{3.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{1.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{1.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{3.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}},
  {{{-2.25f, 0.0f}, {-3.75f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-1.5f, 0.0f}, {-7.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{3.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{3.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-0.75f, 0.0f}, {-3.75f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{7.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{3.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}},
  {{{1.125f, 0.0f}, {7.5f, 0.0f}, {13.125f, 0.0f}, {0.0f, 0.0f}}, {{-11.25f, 0.0f}, {-26.25f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-1.5f, 0.0f}, {-7.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{15.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{3.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-3.75f, 0.0f}, {-13.125f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-3.75f, 0.0f}, {-26.25f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{7.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{15.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}},
  {{{28.125f, 0.0f}, {32.8125f, 0.0f}, {59.0625f, 0.0f}, {0.0f, 0.0f}}, {{5.625f, 0.0f}, {157.5f, 0.0f}, {118.125f, 0.0f}, {0.0f, 0.0f}}, {{-33.75f, 0.0f}, {-26.25f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-7.5f, 0.0f}, {-157.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{45.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{15.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{5.625f, 0.0f}, {19.6875f, 0.0f}, {59.0625f, 0.0f}, {0.0f, 0.0f}}, {{-78.75f, 0.0f}, {-118.125f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-11.25f, 0.0f}, {-26.25f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{157.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{45.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}},
  {{{-14.0625f, 0.0f}, {-147.65625f, 0.0f}, {-177.1875f, 0.0f}, {-324.84375f, 0.0f}}, {{196.875f, 0.0f}, {295.3125f, 0.0f}, {649.6875f, 0.0f}, {0.0f, 0.0f}}, {{16.875f, 0.0f}, {157.5f, 0.0f}, {118.125f, 0.0f}, {0.0f, 0.0f}}, {{-236.25f, 0.0f}, {-236.25f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-22.5f, 0.0f}, {-157.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{315.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{45.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{49.21875f, 0.0f}, {118.125f, 0.0f}, {324.84375f, 0.0f}, {0.0f, 0.0f}}, {{39.375f, 0.0f}, {177.1875f, 0.0f}, {649.6875f, 0.0f}, {0.0f, 0.0f}}, {{-78.75f, 0.0f}, {-118.125f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{-78.75f, 0.0f}, {-236.25f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{157.5f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, {{315.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}},
};
__device__ __forceinline__ float gmp_mcsh_invariant_0(const float* __restrict__ mu) {
  float f = 0.0f;
  { const float m = mu[0]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  return f;
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint_0(const float* __restrict__ mu, float g, float* __restrict__ lam) {
  lam[0] = 0.0f;
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[0]));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
  }
}
__device__ __forceinline__ float gmp_mcsh_invariant_1(const float* __restrict__ mu) {
  float f = 0.0f;
  { const float m = mu[2]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[0]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[1]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  return f;
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint_1(const float* __restrict__ mu, float g, float* __restrict__ lam) {
  lam[0] = 0.0f;
  lam[1] = 0.0f;
  lam[2] = 0.0f;
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[2]));
    lam[2] = __fmaf_rn(1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[0]));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[1]));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
  }
}
__device__ __forceinline__ float gmp_mcsh_invariant_2(const float* __restrict__ mu) {
  float f = 0.0f;
  { const float m = __fmaf_rn(-1.0f, mu[2], -mu[0]); f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[3]; f = __fmaf_rn(__fmul_rn(2.0f, m), m, f); }
  { const float m = mu[4]; f = __fmaf_rn(__fmul_rn(2.0f, m), m, f); }
  { const float m = mu[0]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[1]; f = __fmaf_rn(__fmul_rn(2.0f, m), m, f); }
  { const float m = mu[2]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  return f;
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint_2(const float* __restrict__ mu, float g, float* __restrict__ lam) {
  lam[0] = 0.0f;
  lam[1] = 0.0f;
  lam[2] = 0.0f;
  lam[3] = 0.0f;
  lam[4] = 0.0f;
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[2], -mu[0])));
    lam[0] = __fmaf_rn(-1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(4.0f, __fmul_rn(g, mu[3]));
    lam[3] = __fmaf_rn(1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(4.0f, __fmul_rn(g, mu[4]));
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[0]));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
  }
  { const float m = __fmul_rn(4.0f, __fmul_rn(g, mu[1]));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[2]));
    lam[2] = __fmaf_rn(1.0f, m, lam[2]);
  }
}
__device__ __forceinline__ float gmp_mcsh_invariant_3(const float* __restrict__ mu) {
  float f = 0.0f;
  { const float m = __fmaf_rn(-1.0f, mu[6], -mu[4]); f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[2], -mu[0]); f = __fmaf_rn(__fmul_rn(3.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[3], -mu[1]); f = __fmaf_rn(__fmul_rn(3.0f, m), m, f); }
  { const float m = mu[4]; f = __fmaf_rn(__fmul_rn(3.0f, m), m, f); }
  { const float m = mu[5]; f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = mu[6]; f = __fmaf_rn(__fmul_rn(3.0f, m), m, f); }
  { const float m = mu[0]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[1]; f = __fmaf_rn(__fmul_rn(3.0f, m), m, f); }
  { const float m = mu[2]; f = __fmaf_rn(__fmul_rn(3.0f, m), m, f); }
  { const float m = mu[3]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  return f;
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint_3(const float* __restrict__ mu, float g, float* __restrict__ lam) {
  lam[0] = 0.0f;
  lam[1] = 0.0f;
  lam[2] = 0.0f;
  lam[3] = 0.0f;
  lam[4] = 0.0f;
  lam[5] = 0.0f;
  lam[6] = 0.0f;
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[6], -mu[4])));
    lam[4] = __fmaf_rn(-1.0f, m, lam[4]);
    lam[6] = __fmaf_rn(-1.0f, m, lam[6]);
  }
  { const float m = __fmul_rn(6.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[2], -mu[0])));
    lam[0] = __fmaf_rn(-1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(6.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[3], -mu[1])));
    lam[1] = __fmaf_rn(-1.0f, m, lam[1]);
    lam[3] = __fmaf_rn(-1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(6.0f, __fmul_rn(g, mu[4]));
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, mu[5]));
    lam[5] = __fmaf_rn(1.0f, m, lam[5]);
  }
  { const float m = __fmul_rn(6.0f, __fmul_rn(g, mu[6]));
    lam[6] = __fmaf_rn(1.0f, m, lam[6]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[0]));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
  }
  { const float m = __fmul_rn(6.0f, __fmul_rn(g, mu[1]));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
  }
  { const float m = __fmul_rn(6.0f, __fmul_rn(g, mu[2]));
    lam[2] = __fmaf_rn(1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[3]));
    lam[3] = __fmaf_rn(1.0f, m, lam[3]);
  }
}
__device__ __forceinline__ float gmp_mcsh_invariant_4(const float* __restrict__ mu) {
  float f = 0.0f;
  { const float m = __fmaf_rn(1.0f, mu[4], __fmaf_rn(2.0f, mu[2], mu[0])); f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[7], -mu[5]); f = __fmaf_rn(__fmul_rn(4.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[8], -mu[6]); f = __fmaf_rn(__fmul_rn(4.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[2], -mu[0]); f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[3], -mu[1]); f = __fmaf_rn(__fmul_rn(12.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[4], -mu[2]); f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = mu[5]; f = __fmaf_rn(__fmul_rn(4.0f, m), m, f); }
  { const float m = mu[6]; f = __fmaf_rn(__fmul_rn(12.0f, m), m, f); }
  { const float m = mu[7]; f = __fmaf_rn(__fmul_rn(12.0f, m), m, f); }
  { const float m = mu[8]; f = __fmaf_rn(__fmul_rn(4.0f, m), m, f); }
  { const float m = mu[0]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[1]; f = __fmaf_rn(__fmul_rn(4.0f, m), m, f); }
  { const float m = mu[2]; f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = mu[3]; f = __fmaf_rn(__fmul_rn(4.0f, m), m, f); }
  { const float m = mu[4]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  return f;
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint_4(const float* __restrict__ mu, float g, float* __restrict__ lam) {
  lam[0] = 0.0f;
  lam[1] = 0.0f;
  lam[2] = 0.0f;
  lam[3] = 0.0f;
  lam[4] = 0.0f;
  lam[5] = 0.0f;
  lam[6] = 0.0f;
  lam[7] = 0.0f;
  lam[8] = 0.0f;
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[4], __fmaf_rn(2.0f, mu[2], mu[0]))));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(2.0f, m, lam[2]);
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(8.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[7], -mu[5])));
    lam[5] = __fmaf_rn(-1.0f, m, lam[5]);
    lam[7] = __fmaf_rn(-1.0f, m, lam[7]);
  }
  { const float m = __fmul_rn(8.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[8], -mu[6])));
    lam[6] = __fmaf_rn(-1.0f, m, lam[6]);
    lam[8] = __fmaf_rn(-1.0f, m, lam[8]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[2], -mu[0])));
    lam[0] = __fmaf_rn(-1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(24.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[3], -mu[1])));
    lam[1] = __fmaf_rn(-1.0f, m, lam[1]);
    lam[3] = __fmaf_rn(-1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[4], -mu[2])));
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
    lam[4] = __fmaf_rn(-1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(8.0f, __fmul_rn(g, mu[5]));
    lam[5] = __fmaf_rn(1.0f, m, lam[5]);
  }
  { const float m = __fmul_rn(24.0f, __fmul_rn(g, mu[6]));
    lam[6] = __fmaf_rn(1.0f, m, lam[6]);
  }
  { const float m = __fmul_rn(24.0f, __fmul_rn(g, mu[7]));
    lam[7] = __fmaf_rn(1.0f, m, lam[7]);
  }
  { const float m = __fmul_rn(8.0f, __fmul_rn(g, mu[8]));
    lam[8] = __fmaf_rn(1.0f, m, lam[8]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[0]));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
  }
  { const float m = __fmul_rn(8.0f, __fmul_rn(g, mu[1]));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, mu[2]));
    lam[2] = __fmaf_rn(1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(8.0f, __fmul_rn(g, mu[3]));
    lam[3] = __fmaf_rn(1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[4]));
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
}
__device__ __forceinline__ float gmp_mcsh_invariant_5(const float* __restrict__ mu) {
  float f = 0.0f;
  { const float m = __fmaf_rn(1.0f, mu[10], __fmaf_rn(2.0f, mu[8], mu[6])); f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = __fmaf_rn(1.0f, mu[4], __fmaf_rn(2.0f, mu[2], mu[0])); f = __fmaf_rn(__fmul_rn(5.0f, m), m, f); }
  { const float m = __fmaf_rn(1.0f, mu[5], __fmaf_rn(2.0f, mu[3], mu[1])); f = __fmaf_rn(__fmul_rn(5.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[8], -mu[6]); f = __fmaf_rn(__fmul_rn(10.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[9], -mu[7]); f = __fmaf_rn(__fmul_rn(20.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[10], -mu[8]); f = __fmaf_rn(__fmul_rn(10.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[2], -mu[0]); f = __fmaf_rn(__fmul_rn(10.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[3], -mu[1]); f = __fmaf_rn(__fmul_rn(30.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[4], -mu[2]); f = __fmaf_rn(__fmul_rn(30.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[5], -mu[3]); f = __fmaf_rn(__fmul_rn(10.0f, m), m, f); }
  { const float m = mu[6]; f = __fmaf_rn(__fmul_rn(5.0f, m), m, f); }
  { const float m = mu[7]; f = __fmaf_rn(__fmul_rn(20.0f, m), m, f); }
  { const float m = mu[8]; f = __fmaf_rn(__fmul_rn(30.0f, m), m, f); }
  { const float m = mu[9]; f = __fmaf_rn(__fmul_rn(20.0f, m), m, f); }
  { const float m = mu[10]; f = __fmaf_rn(__fmul_rn(5.0f, m), m, f); }
  { const float m = mu[0]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[1]; f = __fmaf_rn(__fmul_rn(5.0f, m), m, f); }
  { const float m = mu[2]; f = __fmaf_rn(__fmul_rn(10.0f, m), m, f); }
  { const float m = mu[3]; f = __fmaf_rn(__fmul_rn(10.0f, m), m, f); }
  { const float m = mu[4]; f = __fmaf_rn(__fmul_rn(5.0f, m), m, f); }
  { const float m = mu[5]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  return f;
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint_5(const float* __restrict__ mu, float g, float* __restrict__ lam) {
  lam[0] = 0.0f;
  lam[1] = 0.0f;
  lam[2] = 0.0f;
  lam[3] = 0.0f;
  lam[4] = 0.0f;
  lam[5] = 0.0f;
  lam[6] = 0.0f;
  lam[7] = 0.0f;
  lam[8] = 0.0f;
  lam[9] = 0.0f;
  lam[10] = 0.0f;
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[10], __fmaf_rn(2.0f, mu[8], mu[6]))));
    lam[6] = __fmaf_rn(1.0f, m, lam[6]);
    lam[8] = __fmaf_rn(2.0f, m, lam[8]);
    lam[10] = __fmaf_rn(1.0f, m, lam[10]);
  }
  { const float m = __fmul_rn(10.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[4], __fmaf_rn(2.0f, mu[2], mu[0]))));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(2.0f, m, lam[2]);
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(10.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[5], __fmaf_rn(2.0f, mu[3], mu[1]))));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
    lam[3] = __fmaf_rn(2.0f, m, lam[3]);
    lam[5] = __fmaf_rn(1.0f, m, lam[5]);
  }
  { const float m = __fmul_rn(20.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[8], -mu[6])));
    lam[6] = __fmaf_rn(-1.0f, m, lam[6]);
    lam[8] = __fmaf_rn(-1.0f, m, lam[8]);
  }
  { const float m = __fmul_rn(40.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[9], -mu[7])));
    lam[7] = __fmaf_rn(-1.0f, m, lam[7]);
    lam[9] = __fmaf_rn(-1.0f, m, lam[9]);
  }
  { const float m = __fmul_rn(20.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[10], -mu[8])));
    lam[8] = __fmaf_rn(-1.0f, m, lam[8]);
    lam[10] = __fmaf_rn(-1.0f, m, lam[10]);
  }
  { const float m = __fmul_rn(20.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[2], -mu[0])));
    lam[0] = __fmaf_rn(-1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(60.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[3], -mu[1])));
    lam[1] = __fmaf_rn(-1.0f, m, lam[1]);
    lam[3] = __fmaf_rn(-1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(60.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[4], -mu[2])));
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
    lam[4] = __fmaf_rn(-1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(20.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[5], -mu[3])));
    lam[3] = __fmaf_rn(-1.0f, m, lam[3]);
    lam[5] = __fmaf_rn(-1.0f, m, lam[5]);
  }
  { const float m = __fmul_rn(10.0f, __fmul_rn(g, mu[6]));
    lam[6] = __fmaf_rn(1.0f, m, lam[6]);
  }
  { const float m = __fmul_rn(40.0f, __fmul_rn(g, mu[7]));
    lam[7] = __fmaf_rn(1.0f, m, lam[7]);
  }
  { const float m = __fmul_rn(60.0f, __fmul_rn(g, mu[8]));
    lam[8] = __fmaf_rn(1.0f, m, lam[8]);
  }
  { const float m = __fmul_rn(40.0f, __fmul_rn(g, mu[9]));
    lam[9] = __fmaf_rn(1.0f, m, lam[9]);
  }
  { const float m = __fmul_rn(10.0f, __fmul_rn(g, mu[10]));
    lam[10] = __fmaf_rn(1.0f, m, lam[10]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[0]));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
  }
  { const float m = __fmul_rn(10.0f, __fmul_rn(g, mu[1]));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
  }
  { const float m = __fmul_rn(20.0f, __fmul_rn(g, mu[2]));
    lam[2] = __fmaf_rn(1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(20.0f, __fmul_rn(g, mu[3]));
    lam[3] = __fmaf_rn(1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(10.0f, __fmul_rn(g, mu[4]));
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[5]));
    lam[5] = __fmaf_rn(1.0f, m, lam[5]);
  }
}
__device__ __forceinline__ float gmp_mcsh_invariant_6(const float* __restrict__ mu) {
  float f = 0.0f;
  { const float m = __fmaf_rn(-1.0f, mu[6], __fmaf_rn(-3.0f, mu[4], __fmaf_rn(-3.0f, mu[2], -mu[0]))); f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = __fmaf_rn(1.0f, mu[11], __fmaf_rn(2.0f, mu[9], mu[7])); f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = __fmaf_rn(1.0f, mu[12], __fmaf_rn(2.0f, mu[10], mu[8])); f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = __fmaf_rn(1.0f, mu[4], __fmaf_rn(2.0f, mu[2], mu[0])); f = __fmaf_rn(__fmul_rn(15.0f, m), m, f); }
  { const float m = __fmaf_rn(1.0f, mu[5], __fmaf_rn(2.0f, mu[3], mu[1])); f = __fmaf_rn(__fmul_rn(30.0f, m), m, f); }
  { const float m = __fmaf_rn(1.0f, mu[6], __fmaf_rn(2.0f, mu[4], mu[2])); f = __fmaf_rn(__fmul_rn(15.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[9], -mu[7]); f = __fmaf_rn(__fmul_rn(20.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[10], -mu[8]); f = __fmaf_rn(__fmul_rn(60.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[11], -mu[9]); f = __fmaf_rn(__fmul_rn(60.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[12], -mu[10]); f = __fmaf_rn(__fmul_rn(20.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[2], -mu[0]); f = __fmaf_rn(__fmul_rn(15.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[3], -mu[1]); f = __fmaf_rn(__fmul_rn(60.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[4], -mu[2]); f = __fmaf_rn(__fmul_rn(90.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[5], -mu[3]); f = __fmaf_rn(__fmul_rn(60.0f, m), m, f); }
  { const float m = __fmaf_rn(-1.0f, mu[6], -mu[4]); f = __fmaf_rn(__fmul_rn(15.0f, m), m, f); }
  { const float m = mu[7]; f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = mu[8]; f = __fmaf_rn(__fmul_rn(30.0f, m), m, f); }
  { const float m = mu[9]; f = __fmaf_rn(__fmul_rn(60.0f, m), m, f); }
  { const float m = mu[10]; f = __fmaf_rn(__fmul_rn(60.0f, m), m, f); }
  { const float m = mu[11]; f = __fmaf_rn(__fmul_rn(30.0f, m), m, f); }
  { const float m = mu[12]; f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = mu[0]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  { const float m = mu[1]; f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = mu[2]; f = __fmaf_rn(__fmul_rn(15.0f, m), m, f); }
  { const float m = mu[3]; f = __fmaf_rn(__fmul_rn(20.0f, m), m, f); }
  { const float m = mu[4]; f = __fmaf_rn(__fmul_rn(15.0f, m), m, f); }
  { const float m = mu[5]; f = __fmaf_rn(__fmul_rn(6.0f, m), m, f); }
  { const float m = mu[6]; f = __fmaf_rn(__fmul_rn(1.0f, m), m, f); }
  return f;
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint_6(const float* __restrict__ mu, float g, float* __restrict__ lam) {
  lam[0] = 0.0f;
  lam[1] = 0.0f;
  lam[2] = 0.0f;
  lam[3] = 0.0f;
  lam[4] = 0.0f;
  lam[5] = 0.0f;
  lam[6] = 0.0f;
  lam[7] = 0.0f;
  lam[8] = 0.0f;
  lam[9] = 0.0f;
  lam[10] = 0.0f;
  lam[11] = 0.0f;
  lam[12] = 0.0f;
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[6], __fmaf_rn(-3.0f, mu[4], __fmaf_rn(-3.0f, mu[2], -mu[0])))));
    lam[0] = __fmaf_rn(-1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(-3.0f, m, lam[2]);
    lam[4] = __fmaf_rn(-3.0f, m, lam[4]);
    lam[6] = __fmaf_rn(-1.0f, m, lam[6]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[11], __fmaf_rn(2.0f, mu[9], mu[7]))));
    lam[7] = __fmaf_rn(1.0f, m, lam[7]);
    lam[9] = __fmaf_rn(2.0f, m, lam[9]);
    lam[11] = __fmaf_rn(1.0f, m, lam[11]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[12], __fmaf_rn(2.0f, mu[10], mu[8]))));
    lam[8] = __fmaf_rn(1.0f, m, lam[8]);
    lam[10] = __fmaf_rn(2.0f, m, lam[10]);
    lam[12] = __fmaf_rn(1.0f, m, lam[12]);
  }
  { const float m = __fmul_rn(30.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[4], __fmaf_rn(2.0f, mu[2], mu[0]))));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(2.0f, m, lam[2]);
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(60.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[5], __fmaf_rn(2.0f, mu[3], mu[1]))));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
    lam[3] = __fmaf_rn(2.0f, m, lam[3]);
    lam[5] = __fmaf_rn(1.0f, m, lam[5]);
  }
  { const float m = __fmul_rn(30.0f, __fmul_rn(g, __fmaf_rn(1.0f, mu[6], __fmaf_rn(2.0f, mu[4], mu[2]))));
    lam[2] = __fmaf_rn(1.0f, m, lam[2]);
    lam[4] = __fmaf_rn(2.0f, m, lam[4]);
    lam[6] = __fmaf_rn(1.0f, m, lam[6]);
  }
  { const float m = __fmul_rn(40.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[9], -mu[7])));
    lam[7] = __fmaf_rn(-1.0f, m, lam[7]);
    lam[9] = __fmaf_rn(-1.0f, m, lam[9]);
  }
  { const float m = __fmul_rn(120.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[10], -mu[8])));
    lam[8] = __fmaf_rn(-1.0f, m, lam[8]);
    lam[10] = __fmaf_rn(-1.0f, m, lam[10]);
  }
  { const float m = __fmul_rn(120.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[11], -mu[9])));
    lam[9] = __fmaf_rn(-1.0f, m, lam[9]);
    lam[11] = __fmaf_rn(-1.0f, m, lam[11]);
  }
  { const float m = __fmul_rn(40.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[12], -mu[10])));
    lam[10] = __fmaf_rn(-1.0f, m, lam[10]);
    lam[12] = __fmaf_rn(-1.0f, m, lam[12]);
  }
  { const float m = __fmul_rn(30.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[2], -mu[0])));
    lam[0] = __fmaf_rn(-1.0f, m, lam[0]);
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(120.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[3], -mu[1])));
    lam[1] = __fmaf_rn(-1.0f, m, lam[1]);
    lam[3] = __fmaf_rn(-1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(180.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[4], -mu[2])));
    lam[2] = __fmaf_rn(-1.0f, m, lam[2]);
    lam[4] = __fmaf_rn(-1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(120.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[5], -mu[3])));
    lam[3] = __fmaf_rn(-1.0f, m, lam[3]);
    lam[5] = __fmaf_rn(-1.0f, m, lam[5]);
  }
  { const float m = __fmul_rn(30.0f, __fmul_rn(g, __fmaf_rn(-1.0f, mu[6], -mu[4])));
    lam[4] = __fmaf_rn(-1.0f, m, lam[4]);
    lam[6] = __fmaf_rn(-1.0f, m, lam[6]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, mu[7]));
    lam[7] = __fmaf_rn(1.0f, m, lam[7]);
  }
  { const float m = __fmul_rn(60.0f, __fmul_rn(g, mu[8]));
    lam[8] = __fmaf_rn(1.0f, m, lam[8]);
  }
  { const float m = __fmul_rn(120.0f, __fmul_rn(g, mu[9]));
    lam[9] = __fmaf_rn(1.0f, m, lam[9]);
  }
  { const float m = __fmul_rn(120.0f, __fmul_rn(g, mu[10]));
    lam[10] = __fmaf_rn(1.0f, m, lam[10]);
  }
  { const float m = __fmul_rn(60.0f, __fmul_rn(g, mu[11]));
    lam[11] = __fmaf_rn(1.0f, m, lam[11]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, mu[12]));
    lam[12] = __fmaf_rn(1.0f, m, lam[12]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[0]));
    lam[0] = __fmaf_rn(1.0f, m, lam[0]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, mu[1]));
    lam[1] = __fmaf_rn(1.0f, m, lam[1]);
  }
  { const float m = __fmul_rn(30.0f, __fmul_rn(g, mu[2]));
    lam[2] = __fmaf_rn(1.0f, m, lam[2]);
  }
  { const float m = __fmul_rn(40.0f, __fmul_rn(g, mu[3]));
    lam[3] = __fmaf_rn(1.0f, m, lam[3]);
  }
  { const float m = __fmul_rn(30.0f, __fmul_rn(g, mu[4]));
    lam[4] = __fmaf_rn(1.0f, m, lam[4]);
  }
  { const float m = __fmul_rn(12.0f, __fmul_rn(g, mu[5]));
    lam[5] = __fmaf_rn(1.0f, m, lam[5]);
  }
  { const float m = __fmul_rn(2.0f, __fmul_rn(g, mu[6]));
    lam[6] = __fmaf_rn(1.0f, m, lam[6]);
  }
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_0(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_1(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  vx = __fmaf_rn(lam[1], S1[7], vx);
  vy = __fmaf_rn(lam[1], S1[4], vy);
  vz = __fmaf_rn(lam[1], S1[5], vz);
  vx = __fmaf_rn(lam[2], S1[8], vx);
  vy = __fmaf_rn(lam[2], S1[5], vy);
  vz = __fmaf_rn(lam[2], S1[6], vz);
  vx = __fmaf_rn(lam[3], __fsub_rn(-S1[4], S1[6]), vx);
  vy = __fmaf_rn(lam[3], S1[7], vy);
  vz = __fmaf_rn(lam[3], S1[8], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_2(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  vx = __fmaf_rn(lam[1], S1[7], vx);
  vy = __fmaf_rn(lam[1], S1[4], vy);
  vz = __fmaf_rn(lam[1], S1[5], vz);
  vx = __fmaf_rn(lam[2], S1[8], vx);
  vy = __fmaf_rn(lam[2], S1[5], vy);
  vz = __fmaf_rn(lam[2], S1[6], vz);
  vx = __fmaf_rn(lam[3], __fsub_rn(-S1[4], S1[6]), vx);
  vy = __fmaf_rn(lam[3], S1[7], vy);
  vz = __fmaf_rn(lam[3], S1[8], vz);
  vx = __fmaf_rn(lam[4], S1[13], vx);
  vy = __fmaf_rn(lam[4], S1[9], vy);
  vz = __fmaf_rn(lam[4], S1[10], vz);
  vx = __fmaf_rn(lam[5], S1[14], vx);
  vy = __fmaf_rn(lam[5], S1[10], vy);
  vz = __fmaf_rn(lam[5], S1[11], vz);
  vx = __fmaf_rn(lam[6], S1[15], vx);
  vy = __fmaf_rn(lam[6], S1[11], vy);
  vz = __fmaf_rn(lam[6], S1[12], vz);
  vx = __fmaf_rn(lam[7], __fsub_rn(-S1[9], S1[11]), vx);
  vy = __fmaf_rn(lam[7], S1[13], vy);
  vz = __fmaf_rn(lam[7], S1[14], vz);
  vx = __fmaf_rn(lam[8], __fsub_rn(-S1[10], S1[12]), vx);
  vy = __fmaf_rn(lam[8], S1[14], vy);
  vz = __fmaf_rn(lam[8], S1[15], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_3(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  vx = __fmaf_rn(lam[1], S1[7], vx);
  vy = __fmaf_rn(lam[1], S1[4], vy);
  vz = __fmaf_rn(lam[1], S1[5], vz);
  vx = __fmaf_rn(lam[2], S1[8], vx);
  vy = __fmaf_rn(lam[2], S1[5], vy);
  vz = __fmaf_rn(lam[2], S1[6], vz);
  vx = __fmaf_rn(lam[3], __fsub_rn(-S1[4], S1[6]), vx);
  vy = __fmaf_rn(lam[3], S1[7], vy);
  vz = __fmaf_rn(lam[3], S1[8], vz);
  vx = __fmaf_rn(lam[4], S1[13], vx);
  vy = __fmaf_rn(lam[4], S1[9], vy);
  vz = __fmaf_rn(lam[4], S1[10], vz);
  vx = __fmaf_rn(lam[5], S1[14], vx);
  vy = __fmaf_rn(lam[5], S1[10], vy);
  vz = __fmaf_rn(lam[5], S1[11], vz);
  vx = __fmaf_rn(lam[6], S1[15], vx);
  vy = __fmaf_rn(lam[6], S1[11], vy);
  vz = __fmaf_rn(lam[6], S1[12], vz);
  vx = __fmaf_rn(lam[7], __fsub_rn(-S1[9], S1[11]), vx);
  vy = __fmaf_rn(lam[7], S1[13], vy);
  vz = __fmaf_rn(lam[7], S1[14], vz);
  vx = __fmaf_rn(lam[8], __fsub_rn(-S1[10], S1[12]), vx);
  vy = __fmaf_rn(lam[8], S1[14], vy);
  vz = __fmaf_rn(lam[8], S1[15], vz);
  vx = __fmaf_rn(lam[9], S1[21], vx);
  vy = __fmaf_rn(lam[9], S1[16], vy);
  vz = __fmaf_rn(lam[9], S1[17], vz);
  vx = __fmaf_rn(lam[10], S1[22], vx);
  vy = __fmaf_rn(lam[10], S1[17], vy);
  vz = __fmaf_rn(lam[10], S1[18], vz);
  vx = __fmaf_rn(lam[11], S1[23], vx);
  vy = __fmaf_rn(lam[11], S1[18], vy);
  vz = __fmaf_rn(lam[11], S1[19], vz);
  vx = __fmaf_rn(lam[12], S1[24], vx);
  vy = __fmaf_rn(lam[12], S1[19], vy);
  vz = __fmaf_rn(lam[12], S1[20], vz);
  vx = __fmaf_rn(lam[13], __fsub_rn(-S1[16], S1[18]), vx);
  vy = __fmaf_rn(lam[13], S1[21], vy);
  vz = __fmaf_rn(lam[13], S1[22], vz);
  vx = __fmaf_rn(lam[14], __fsub_rn(-S1[17], S1[19]), vx);
  vy = __fmaf_rn(lam[14], S1[22], vy);
  vz = __fmaf_rn(lam[14], S1[23], vz);
  vx = __fmaf_rn(lam[15], __fsub_rn(-S1[18], S1[20]), vx);
  vy = __fmaf_rn(lam[15], S1[23], vy);
  vz = __fmaf_rn(lam[15], S1[24], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_4(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  vx = __fmaf_rn(lam[1], S1[7], vx);
  vy = __fmaf_rn(lam[1], S1[4], vy);
  vz = __fmaf_rn(lam[1], S1[5], vz);
  vx = __fmaf_rn(lam[2], S1[8], vx);
  vy = __fmaf_rn(lam[2], S1[5], vy);
  vz = __fmaf_rn(lam[2], S1[6], vz);
  vx = __fmaf_rn(lam[3], __fsub_rn(-S1[4], S1[6]), vx);
  vy = __fmaf_rn(lam[3], S1[7], vy);
  vz = __fmaf_rn(lam[3], S1[8], vz);
  vx = __fmaf_rn(lam[4], S1[13], vx);
  vy = __fmaf_rn(lam[4], S1[9], vy);
  vz = __fmaf_rn(lam[4], S1[10], vz);
  vx = __fmaf_rn(lam[5], S1[14], vx);
  vy = __fmaf_rn(lam[5], S1[10], vy);
  vz = __fmaf_rn(lam[5], S1[11], vz);
  vx = __fmaf_rn(lam[6], S1[15], vx);
  vy = __fmaf_rn(lam[6], S1[11], vy);
  vz = __fmaf_rn(lam[6], S1[12], vz);
  vx = __fmaf_rn(lam[7], __fsub_rn(-S1[9], S1[11]), vx);
  vy = __fmaf_rn(lam[7], S1[13], vy);
  vz = __fmaf_rn(lam[7], S1[14], vz);
  vx = __fmaf_rn(lam[8], __fsub_rn(-S1[10], S1[12]), vx);
  vy = __fmaf_rn(lam[8], S1[14], vy);
  vz = __fmaf_rn(lam[8], S1[15], vz);
  vx = __fmaf_rn(lam[9], S1[21], vx);
  vy = __fmaf_rn(lam[9], S1[16], vy);
  vz = __fmaf_rn(lam[9], S1[17], vz);
  vx = __fmaf_rn(lam[10], S1[22], vx);
  vy = __fmaf_rn(lam[10], S1[17], vy);
  vz = __fmaf_rn(lam[10], S1[18], vz);
  vx = __fmaf_rn(lam[11], S1[23], vx);
  vy = __fmaf_rn(lam[11], S1[18], vy);
  vz = __fmaf_rn(lam[11], S1[19], vz);
  vx = __fmaf_rn(lam[12], S1[24], vx);
  vy = __fmaf_rn(lam[12], S1[19], vy);
  vz = __fmaf_rn(lam[12], S1[20], vz);
  vx = __fmaf_rn(lam[13], __fsub_rn(-S1[16], S1[18]), vx);
  vy = __fmaf_rn(lam[13], S1[21], vy);
  vz = __fmaf_rn(lam[13], S1[22], vz);
  vx = __fmaf_rn(lam[14], __fsub_rn(-S1[17], S1[19]), vx);
  vy = __fmaf_rn(lam[14], S1[22], vy);
  vz = __fmaf_rn(lam[14], S1[23], vz);
  vx = __fmaf_rn(lam[15], __fsub_rn(-S1[18], S1[20]), vx);
  vy = __fmaf_rn(lam[15], S1[23], vy);
  vz = __fmaf_rn(lam[15], S1[24], vz);
  vx = __fmaf_rn(lam[16], S1[31], vx);
  vy = __fmaf_rn(lam[16], S1[25], vy);
  vz = __fmaf_rn(lam[16], S1[26], vz);
  vx = __fmaf_rn(lam[17], S1[32], vx);
  vy = __fmaf_rn(lam[17], S1[26], vy);
  vz = __fmaf_rn(lam[17], S1[27], vz);
  vx = __fmaf_rn(lam[18], S1[33], vx);
  vy = __fmaf_rn(lam[18], S1[27], vy);
  vz = __fmaf_rn(lam[18], S1[28], vz);
  vx = __fmaf_rn(lam[19], S1[34], vx);
  vy = __fmaf_rn(lam[19], S1[28], vy);
  vz = __fmaf_rn(lam[19], S1[29], vz);
  vx = __fmaf_rn(lam[20], S1[35], vx);
  vy = __fmaf_rn(lam[20], S1[29], vy);
  vz = __fmaf_rn(lam[20], S1[30], vz);
  vx = __fmaf_rn(lam[21], __fsub_rn(-S1[25], S1[27]), vx);
  vy = __fmaf_rn(lam[21], S1[31], vy);
  vz = __fmaf_rn(lam[21], S1[32], vz);
  vx = __fmaf_rn(lam[22], __fsub_rn(-S1[26], S1[28]), vx);
  vy = __fmaf_rn(lam[22], S1[32], vy);
  vz = __fmaf_rn(lam[22], S1[33], vz);
  vx = __fmaf_rn(lam[23], __fsub_rn(-S1[27], S1[29]), vx);
  vy = __fmaf_rn(lam[23], S1[33], vy);
  vz = __fmaf_rn(lam[23], S1[34], vz);
  vx = __fmaf_rn(lam[24], __fsub_rn(-S1[28], S1[30]), vx);
  vy = __fmaf_rn(lam[24], S1[34], vy);
  vz = __fmaf_rn(lam[24], S1[35], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_5(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  vx = __fmaf_rn(lam[1], S1[7], vx);
  vy = __fmaf_rn(lam[1], S1[4], vy);
  vz = __fmaf_rn(lam[1], S1[5], vz);
  vx = __fmaf_rn(lam[2], S1[8], vx);
  vy = __fmaf_rn(lam[2], S1[5], vy);
  vz = __fmaf_rn(lam[2], S1[6], vz);
  vx = __fmaf_rn(lam[3], __fsub_rn(-S1[4], S1[6]), vx);
  vy = __fmaf_rn(lam[3], S1[7], vy);
  vz = __fmaf_rn(lam[3], S1[8], vz);
  vx = __fmaf_rn(lam[4], S1[13], vx);
  vy = __fmaf_rn(lam[4], S1[9], vy);
  vz = __fmaf_rn(lam[4], S1[10], vz);
  vx = __fmaf_rn(lam[5], S1[14], vx);
  vy = __fmaf_rn(lam[5], S1[10], vy);
  vz = __fmaf_rn(lam[5], S1[11], vz);
  vx = __fmaf_rn(lam[6], S1[15], vx);
  vy = __fmaf_rn(lam[6], S1[11], vy);
  vz = __fmaf_rn(lam[6], S1[12], vz);
  vx = __fmaf_rn(lam[7], __fsub_rn(-S1[9], S1[11]), vx);
  vy = __fmaf_rn(lam[7], S1[13], vy);
  vz = __fmaf_rn(lam[7], S1[14], vz);
  vx = __fmaf_rn(lam[8], __fsub_rn(-S1[10], S1[12]), vx);
  vy = __fmaf_rn(lam[8], S1[14], vy);
  vz = __fmaf_rn(lam[8], S1[15], vz);
  vx = __fmaf_rn(lam[9], S1[21], vx);
  vy = __fmaf_rn(lam[9], S1[16], vy);
  vz = __fmaf_rn(lam[9], S1[17], vz);
  vx = __fmaf_rn(lam[10], S1[22], vx);
  vy = __fmaf_rn(lam[10], S1[17], vy);
  vz = __fmaf_rn(lam[10], S1[18], vz);
  vx = __fmaf_rn(lam[11], S1[23], vx);
  vy = __fmaf_rn(lam[11], S1[18], vy);
  vz = __fmaf_rn(lam[11], S1[19], vz);
  vx = __fmaf_rn(lam[12], S1[24], vx);
  vy = __fmaf_rn(lam[12], S1[19], vy);
  vz = __fmaf_rn(lam[12], S1[20], vz);
  vx = __fmaf_rn(lam[13], __fsub_rn(-S1[16], S1[18]), vx);
  vy = __fmaf_rn(lam[13], S1[21], vy);
  vz = __fmaf_rn(lam[13], S1[22], vz);
  vx = __fmaf_rn(lam[14], __fsub_rn(-S1[17], S1[19]), vx);
  vy = __fmaf_rn(lam[14], S1[22], vy);
  vz = __fmaf_rn(lam[14], S1[23], vz);
  vx = __fmaf_rn(lam[15], __fsub_rn(-S1[18], S1[20]), vx);
  vy = __fmaf_rn(lam[15], S1[23], vy);
  vz = __fmaf_rn(lam[15], S1[24], vz);
  vx = __fmaf_rn(lam[16], S1[31], vx);
  vy = __fmaf_rn(lam[16], S1[25], vy);
  vz = __fmaf_rn(lam[16], S1[26], vz);
  vx = __fmaf_rn(lam[17], S1[32], vx);
  vy = __fmaf_rn(lam[17], S1[26], vy);
  vz = __fmaf_rn(lam[17], S1[27], vz);
  vx = __fmaf_rn(lam[18], S1[33], vx);
  vy = __fmaf_rn(lam[18], S1[27], vy);
  vz = __fmaf_rn(lam[18], S1[28], vz);
  vx = __fmaf_rn(lam[19], S1[34], vx);
  vy = __fmaf_rn(lam[19], S1[28], vy);
  vz = __fmaf_rn(lam[19], S1[29], vz);
  vx = __fmaf_rn(lam[20], S1[35], vx);
  vy = __fmaf_rn(lam[20], S1[29], vy);
  vz = __fmaf_rn(lam[20], S1[30], vz);
  vx = __fmaf_rn(lam[21], __fsub_rn(-S1[25], S1[27]), vx);
  vy = __fmaf_rn(lam[21], S1[31], vy);
  vz = __fmaf_rn(lam[21], S1[32], vz);
  vx = __fmaf_rn(lam[22], __fsub_rn(-S1[26], S1[28]), vx);
  vy = __fmaf_rn(lam[22], S1[32], vy);
  vz = __fmaf_rn(lam[22], S1[33], vz);
  vx = __fmaf_rn(lam[23], __fsub_rn(-S1[27], S1[29]), vx);
  vy = __fmaf_rn(lam[23], S1[33], vy);
  vz = __fmaf_rn(lam[23], S1[34], vz);
  vx = __fmaf_rn(lam[24], __fsub_rn(-S1[28], S1[30]), vx);
  vy = __fmaf_rn(lam[24], S1[34], vy);
  vz = __fmaf_rn(lam[24], S1[35], vz);
  vx = __fmaf_rn(lam[25], S1[43], vx);
  vy = __fmaf_rn(lam[25], S1[36], vy);
  vz = __fmaf_rn(lam[25], S1[37], vz);
  vx = __fmaf_rn(lam[26], S1[44], vx);
  vy = __fmaf_rn(lam[26], S1[37], vy);
  vz = __fmaf_rn(lam[26], S1[38], vz);
  vx = __fmaf_rn(lam[27], S1[45], vx);
  vy = __fmaf_rn(lam[27], S1[38], vy);
  vz = __fmaf_rn(lam[27], S1[39], vz);
  vx = __fmaf_rn(lam[28], S1[46], vx);
  vy = __fmaf_rn(lam[28], S1[39], vy);
  vz = __fmaf_rn(lam[28], S1[40], vz);
  vx = __fmaf_rn(lam[29], S1[47], vx);
  vy = __fmaf_rn(lam[29], S1[40], vy);
  vz = __fmaf_rn(lam[29], S1[41], vz);
  vx = __fmaf_rn(lam[30], S1[48], vx);
  vy = __fmaf_rn(lam[30], S1[41], vy);
  vz = __fmaf_rn(lam[30], S1[42], vz);
  vx = __fmaf_rn(lam[31], __fsub_rn(-S1[36], S1[38]), vx);
  vy = __fmaf_rn(lam[31], S1[43], vy);
  vz = __fmaf_rn(lam[31], S1[44], vz);
  vx = __fmaf_rn(lam[32], __fsub_rn(-S1[37], S1[39]), vx);
  vy = __fmaf_rn(lam[32], S1[44], vy);
  vz = __fmaf_rn(lam[32], S1[45], vz);
  vx = __fmaf_rn(lam[33], __fsub_rn(-S1[38], S1[40]), vx);
  vy = __fmaf_rn(lam[33], S1[45], vy);
  vz = __fmaf_rn(lam[33], S1[46], vz);
  vx = __fmaf_rn(lam[34], __fsub_rn(-S1[39], S1[41]), vx);
  vy = __fmaf_rn(lam[34], S1[46], vy);
  vz = __fmaf_rn(lam[34], S1[47], vz);
  vx = __fmaf_rn(lam[35], __fsub_rn(-S1[40], S1[42]), vx);
  vy = __fmaf_rn(lam[35], S1[47], vy);
  vz = __fmaf_rn(lam[35], S1[48], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_6(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  vx = __fmaf_rn(lam[1], S1[7], vx);
  vy = __fmaf_rn(lam[1], S1[4], vy);
  vz = __fmaf_rn(lam[1], S1[5], vz);
  vx = __fmaf_rn(lam[2], S1[8], vx);
  vy = __fmaf_rn(lam[2], S1[5], vy);
  vz = __fmaf_rn(lam[2], S1[6], vz);
  vx = __fmaf_rn(lam[3], __fsub_rn(-S1[4], S1[6]), vx);
  vy = __fmaf_rn(lam[3], S1[7], vy);
  vz = __fmaf_rn(lam[3], S1[8], vz);
  vx = __fmaf_rn(lam[4], S1[13], vx);
  vy = __fmaf_rn(lam[4], S1[9], vy);
  vz = __fmaf_rn(lam[4], S1[10], vz);
  vx = __fmaf_rn(lam[5], S1[14], vx);
  vy = __fmaf_rn(lam[5], S1[10], vy);
  vz = __fmaf_rn(lam[5], S1[11], vz);
  vx = __fmaf_rn(lam[6], S1[15], vx);
  vy = __fmaf_rn(lam[6], S1[11], vy);
  vz = __fmaf_rn(lam[6], S1[12], vz);
  vx = __fmaf_rn(lam[7], __fsub_rn(-S1[9], S1[11]), vx);
  vy = __fmaf_rn(lam[7], S1[13], vy);
  vz = __fmaf_rn(lam[7], S1[14], vz);
  vx = __fmaf_rn(lam[8], __fsub_rn(-S1[10], S1[12]), vx);
  vy = __fmaf_rn(lam[8], S1[14], vy);
  vz = __fmaf_rn(lam[8], S1[15], vz);
  vx = __fmaf_rn(lam[9], S1[21], vx);
  vy = __fmaf_rn(lam[9], S1[16], vy);
  vz = __fmaf_rn(lam[9], S1[17], vz);
  vx = __fmaf_rn(lam[10], S1[22], vx);
  vy = __fmaf_rn(lam[10], S1[17], vy);
  vz = __fmaf_rn(lam[10], S1[18], vz);
  vx = __fmaf_rn(lam[11], S1[23], vx);
  vy = __fmaf_rn(lam[11], S1[18], vy);
  vz = __fmaf_rn(lam[11], S1[19], vz);
  vx = __fmaf_rn(lam[12], S1[24], vx);
  vy = __fmaf_rn(lam[12], S1[19], vy);
  vz = __fmaf_rn(lam[12], S1[20], vz);
  vx = __fmaf_rn(lam[13], __fsub_rn(-S1[16], S1[18]), vx);
  vy = __fmaf_rn(lam[13], S1[21], vy);
  vz = __fmaf_rn(lam[13], S1[22], vz);
  vx = __fmaf_rn(lam[14], __fsub_rn(-S1[17], S1[19]), vx);
  vy = __fmaf_rn(lam[14], S1[22], vy);
  vz = __fmaf_rn(lam[14], S1[23], vz);
  vx = __fmaf_rn(lam[15], __fsub_rn(-S1[18], S1[20]), vx);
  vy = __fmaf_rn(lam[15], S1[23], vy);
  vz = __fmaf_rn(lam[15], S1[24], vz);
  vx = __fmaf_rn(lam[16], S1[31], vx);
  vy = __fmaf_rn(lam[16], S1[25], vy);
  vz = __fmaf_rn(lam[16], S1[26], vz);
  vx = __fmaf_rn(lam[17], S1[32], vx);
  vy = __fmaf_rn(lam[17], S1[26], vy);
  vz = __fmaf_rn(lam[17], S1[27], vz);
  vx = __fmaf_rn(lam[18], S1[33], vx);
  vy = __fmaf_rn(lam[18], S1[27], vy);
  vz = __fmaf_rn(lam[18], S1[28], vz);
  vx = __fmaf_rn(lam[19], S1[34], vx);
  vy = __fmaf_rn(lam[19], S1[28], vy);
  vz = __fmaf_rn(lam[19], S1[29], vz);
  vx = __fmaf_rn(lam[20], S1[35], vx);
  vy = __fmaf_rn(lam[20], S1[29], vy);
  vz = __fmaf_rn(lam[20], S1[30], vz);
  vx = __fmaf_rn(lam[21], __fsub_rn(-S1[25], S1[27]), vx);
  vy = __fmaf_rn(lam[21], S1[31], vy);
  vz = __fmaf_rn(lam[21], S1[32], vz);
  vx = __fmaf_rn(lam[22], __fsub_rn(-S1[26], S1[28]), vx);
  vy = __fmaf_rn(lam[22], S1[32], vy);
  vz = __fmaf_rn(lam[22], S1[33], vz);
  vx = __fmaf_rn(lam[23], __fsub_rn(-S1[27], S1[29]), vx);
  vy = __fmaf_rn(lam[23], S1[33], vy);
  vz = __fmaf_rn(lam[23], S1[34], vz);
  vx = __fmaf_rn(lam[24], __fsub_rn(-S1[28], S1[30]), vx);
  vy = __fmaf_rn(lam[24], S1[34], vy);
  vz = __fmaf_rn(lam[24], S1[35], vz);
  vx = __fmaf_rn(lam[25], S1[43], vx);
  vy = __fmaf_rn(lam[25], S1[36], vy);
  vz = __fmaf_rn(lam[25], S1[37], vz);
  vx = __fmaf_rn(lam[26], S1[44], vx);
  vy = __fmaf_rn(lam[26], S1[37], vy);
  vz = __fmaf_rn(lam[26], S1[38], vz);
  vx = __fmaf_rn(lam[27], S1[45], vx);
  vy = __fmaf_rn(lam[27], S1[38], vy);
  vz = __fmaf_rn(lam[27], S1[39], vz);
  vx = __fmaf_rn(lam[28], S1[46], vx);
  vy = __fmaf_rn(lam[28], S1[39], vy);
  vz = __fmaf_rn(lam[28], S1[40], vz);
  vx = __fmaf_rn(lam[29], S1[47], vx);
  vy = __fmaf_rn(lam[29], S1[40], vy);
  vz = __fmaf_rn(lam[29], S1[41], vz);
  vx = __fmaf_rn(lam[30], S1[48], vx);
  vy = __fmaf_rn(lam[30], S1[41], vy);
  vz = __fmaf_rn(lam[30], S1[42], vz);
  vx = __fmaf_rn(lam[31], __fsub_rn(-S1[36], S1[38]), vx);
  vy = __fmaf_rn(lam[31], S1[43], vy);
  vz = __fmaf_rn(lam[31], S1[44], vz);
  vx = __fmaf_rn(lam[32], __fsub_rn(-S1[37], S1[39]), vx);
  vy = __fmaf_rn(lam[32], S1[44], vy);
  vz = __fmaf_rn(lam[32], S1[45], vz);
  vx = __fmaf_rn(lam[33], __fsub_rn(-S1[38], S1[40]), vx);
  vy = __fmaf_rn(lam[33], S1[45], vy);
  vz = __fmaf_rn(lam[33], S1[46], vz);
  vx = __fmaf_rn(lam[34], __fsub_rn(-S1[39], S1[41]), vx);
  vy = __fmaf_rn(lam[34], S1[46], vy);
  vz = __fmaf_rn(lam[34], S1[47], vz);
  vx = __fmaf_rn(lam[35], __fsub_rn(-S1[40], S1[42]), vx);
  vy = __fmaf_rn(lam[35], S1[47], vy);
  vz = __fmaf_rn(lam[35], S1[48], vz);
  vx = __fmaf_rn(lam[36], S1[57], vx);
  vy = __fmaf_rn(lam[36], S1[49], vy);
  vz = __fmaf_rn(lam[36], S1[50], vz);
  vx = __fmaf_rn(lam[37], S1[58], vx);
  vy = __fmaf_rn(lam[37], S1[50], vy);
  vz = __fmaf_rn(lam[37], S1[51], vz);
  vx = __fmaf_rn(lam[38], S1[59], vx);
  vy = __fmaf_rn(lam[38], S1[51], vy);
  vz = __fmaf_rn(lam[38], S1[52], vz);
  vx = __fmaf_rn(lam[39], S1[60], vx);
  vy = __fmaf_rn(lam[39], S1[52], vy);
  vz = __fmaf_rn(lam[39], S1[53], vz);
  vx = __fmaf_rn(lam[40], S1[61], vx);
  vy = __fmaf_rn(lam[40], S1[53], vy);
  vz = __fmaf_rn(lam[40], S1[54], vz);
  vx = __fmaf_rn(lam[41], S1[62], vx);
  vy = __fmaf_rn(lam[41], S1[54], vy);
  vz = __fmaf_rn(lam[41], S1[55], vz);
  vx = __fmaf_rn(lam[42], S1[63], vx);
  vy = __fmaf_rn(lam[42], S1[55], vy);
  vz = __fmaf_rn(lam[42], S1[56], vz);
  vx = __fmaf_rn(lam[43], __fsub_rn(-S1[49], S1[51]), vx);
  vy = __fmaf_rn(lam[43], S1[57], vy);
  vz = __fmaf_rn(lam[43], S1[58], vz);
  vx = __fmaf_rn(lam[44], __fsub_rn(-S1[50], S1[52]), vx);
  vy = __fmaf_rn(lam[44], S1[58], vy);
  vz = __fmaf_rn(lam[44], S1[59], vz);
  vx = __fmaf_rn(lam[45], __fsub_rn(-S1[51], S1[53]), vx);
  vy = __fmaf_rn(lam[45], S1[59], vy);
  vz = __fmaf_rn(lam[45], S1[60], vz);
  vx = __fmaf_rn(lam[46], __fsub_rn(-S1[52], S1[54]), vx);
  vy = __fmaf_rn(lam[46], S1[60], vy);
  vz = __fmaf_rn(lam[46], S1[61], vz);
  vx = __fmaf_rn(lam[47], __fsub_rn(-S1[53], S1[55]), vx);
  vy = __fmaf_rn(lam[47], S1[61], vy);
  vz = __fmaf_rn(lam[47], S1[62], vz);
  vx = __fmaf_rn(lam[48], __fsub_rn(-S1[54], S1[56]), vx);
  vy = __fmaf_rn(lam[48], S1[62], vy);
  vz = __fmaf_rn(lam[48], S1[63], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order_0(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[0], S1[3], vx);
  vy = __fmaf_rn(lam[0], S1[1], vy);
  vz = __fmaf_rn(lam[0], S1[2], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order_1(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[1], S1[7], vx);
  vy = __fmaf_rn(lam[1], S1[4], vy);
  vz = __fmaf_rn(lam[1], S1[5], vz);
  vx = __fmaf_rn(lam[2], S1[8], vx);
  vy = __fmaf_rn(lam[2], S1[5], vy);
  vz = __fmaf_rn(lam[2], S1[6], vz);
  vx = __fmaf_rn(lam[3], __fsub_rn(-S1[4], S1[6]), vx);
  vy = __fmaf_rn(lam[3], S1[7], vy);
  vz = __fmaf_rn(lam[3], S1[8], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order_2(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[4], S1[13], vx);
  vy = __fmaf_rn(lam[4], S1[9], vy);
  vz = __fmaf_rn(lam[4], S1[10], vz);
  vx = __fmaf_rn(lam[5], S1[14], vx);
  vy = __fmaf_rn(lam[5], S1[10], vy);
  vz = __fmaf_rn(lam[5], S1[11], vz);
  vx = __fmaf_rn(lam[6], S1[15], vx);
  vy = __fmaf_rn(lam[6], S1[11], vy);
  vz = __fmaf_rn(lam[6], S1[12], vz);
  vx = __fmaf_rn(lam[7], __fsub_rn(-S1[9], S1[11]), vx);
  vy = __fmaf_rn(lam[7], S1[13], vy);
  vz = __fmaf_rn(lam[7], S1[14], vz);
  vx = __fmaf_rn(lam[8], __fsub_rn(-S1[10], S1[12]), vx);
  vy = __fmaf_rn(lam[8], S1[14], vy);
  vz = __fmaf_rn(lam[8], S1[15], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order_3(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[9], S1[21], vx);
  vy = __fmaf_rn(lam[9], S1[16], vy);
  vz = __fmaf_rn(lam[9], S1[17], vz);
  vx = __fmaf_rn(lam[10], S1[22], vx);
  vy = __fmaf_rn(lam[10], S1[17], vy);
  vz = __fmaf_rn(lam[10], S1[18], vz);
  vx = __fmaf_rn(lam[11], S1[23], vx);
  vy = __fmaf_rn(lam[11], S1[18], vy);
  vz = __fmaf_rn(lam[11], S1[19], vz);
  vx = __fmaf_rn(lam[12], S1[24], vx);
  vy = __fmaf_rn(lam[12], S1[19], vy);
  vz = __fmaf_rn(lam[12], S1[20], vz);
  vx = __fmaf_rn(lam[13], __fsub_rn(-S1[16], S1[18]), vx);
  vy = __fmaf_rn(lam[13], S1[21], vy);
  vz = __fmaf_rn(lam[13], S1[22], vz);
  vx = __fmaf_rn(lam[14], __fsub_rn(-S1[17], S1[19]), vx);
  vy = __fmaf_rn(lam[14], S1[22], vy);
  vz = __fmaf_rn(lam[14], S1[23], vz);
  vx = __fmaf_rn(lam[15], __fsub_rn(-S1[18], S1[20]), vx);
  vy = __fmaf_rn(lam[15], S1[23], vy);
  vz = __fmaf_rn(lam[15], S1[24], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order_4(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[16], S1[31], vx);
  vy = __fmaf_rn(lam[16], S1[25], vy);
  vz = __fmaf_rn(lam[16], S1[26], vz);
  vx = __fmaf_rn(lam[17], S1[32], vx);
  vy = __fmaf_rn(lam[17], S1[26], vy);
  vz = __fmaf_rn(lam[17], S1[27], vz);
  vx = __fmaf_rn(lam[18], S1[33], vx);
  vy = __fmaf_rn(lam[18], S1[27], vy);
  vz = __fmaf_rn(lam[18], S1[28], vz);
  vx = __fmaf_rn(lam[19], S1[34], vx);
  vy = __fmaf_rn(lam[19], S1[28], vy);
  vz = __fmaf_rn(lam[19], S1[29], vz);
  vx = __fmaf_rn(lam[20], S1[35], vx);
  vy = __fmaf_rn(lam[20], S1[29], vy);
  vz = __fmaf_rn(lam[20], S1[30], vz);
  vx = __fmaf_rn(lam[21], __fsub_rn(-S1[25], S1[27]), vx);
  vy = __fmaf_rn(lam[21], S1[31], vy);
  vz = __fmaf_rn(lam[21], S1[32], vz);
  vx = __fmaf_rn(lam[22], __fsub_rn(-S1[26], S1[28]), vx);
  vy = __fmaf_rn(lam[22], S1[32], vy);
  vz = __fmaf_rn(lam[22], S1[33], vz);
  vx = __fmaf_rn(lam[23], __fsub_rn(-S1[27], S1[29]), vx);
  vy = __fmaf_rn(lam[23], S1[33], vy);
  vz = __fmaf_rn(lam[23], S1[34], vz);
  vx = __fmaf_rn(lam[24], __fsub_rn(-S1[28], S1[30]), vx);
  vy = __fmaf_rn(lam[24], S1[34], vy);
  vz = __fmaf_rn(lam[24], S1[35], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order_5(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[25], S1[43], vx);
  vy = __fmaf_rn(lam[25], S1[36], vy);
  vz = __fmaf_rn(lam[25], S1[37], vz);
  vx = __fmaf_rn(lam[26], S1[44], vx);
  vy = __fmaf_rn(lam[26], S1[37], vy);
  vz = __fmaf_rn(lam[26], S1[38], vz);
  vx = __fmaf_rn(lam[27], S1[45], vx);
  vy = __fmaf_rn(lam[27], S1[38], vy);
  vz = __fmaf_rn(lam[27], S1[39], vz);
  vx = __fmaf_rn(lam[28], S1[46], vx);
  vy = __fmaf_rn(lam[28], S1[39], vy);
  vz = __fmaf_rn(lam[28], S1[40], vz);
  vx = __fmaf_rn(lam[29], S1[47], vx);
  vy = __fmaf_rn(lam[29], S1[40], vy);
  vz = __fmaf_rn(lam[29], S1[41], vz);
  vx = __fmaf_rn(lam[30], S1[48], vx);
  vy = __fmaf_rn(lam[30], S1[41], vy);
  vz = __fmaf_rn(lam[30], S1[42], vz);
  vx = __fmaf_rn(lam[31], __fsub_rn(-S1[36], S1[38]), vx);
  vy = __fmaf_rn(lam[31], S1[43], vy);
  vz = __fmaf_rn(lam[31], S1[44], vz);
  vx = __fmaf_rn(lam[32], __fsub_rn(-S1[37], S1[39]), vx);
  vy = __fmaf_rn(lam[32], S1[44], vy);
  vz = __fmaf_rn(lam[32], S1[45], vz);
  vx = __fmaf_rn(lam[33], __fsub_rn(-S1[38], S1[40]), vx);
  vy = __fmaf_rn(lam[33], S1[45], vy);
  vz = __fmaf_rn(lam[33], S1[46], vz);
  vx = __fmaf_rn(lam[34], __fsub_rn(-S1[39], S1[41]), vx);
  vy = __fmaf_rn(lam[34], S1[46], vy);
  vz = __fmaf_rn(lam[34], S1[47], vz);
  vx = __fmaf_rn(lam[35], __fsub_rn(-S1[40], S1[42]), vx);
  vy = __fmaf_rn(lam[35], S1[47], vy);
  vz = __fmaf_rn(lam[35], S1[48], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order_6(const float* __restrict__ lam, const float* __restrict__ S1, float* __restrict__ V) {
  float vx = 0.0f, vy = 0.0f, vz = 0.0f;
  vx = __fmaf_rn(lam[36], S1[57], vx);
  vy = __fmaf_rn(lam[36], S1[49], vy);
  vz = __fmaf_rn(lam[36], S1[50], vz);
  vx = __fmaf_rn(lam[37], S1[58], vx);
  vy = __fmaf_rn(lam[37], S1[50], vy);
  vz = __fmaf_rn(lam[37], S1[51], vz);
  vx = __fmaf_rn(lam[38], S1[59], vx);
  vy = __fmaf_rn(lam[38], S1[51], vy);
  vz = __fmaf_rn(lam[38], S1[52], vz);
  vx = __fmaf_rn(lam[39], S1[60], vx);
  vy = __fmaf_rn(lam[39], S1[52], vy);
  vz = __fmaf_rn(lam[39], S1[53], vz);
  vx = __fmaf_rn(lam[40], S1[61], vx);
  vy = __fmaf_rn(lam[40], S1[53], vy);
  vz = __fmaf_rn(lam[40], S1[54], vz);
  vx = __fmaf_rn(lam[41], S1[62], vx);
  vy = __fmaf_rn(lam[41], S1[54], vy);
  vz = __fmaf_rn(lam[41], S1[55], vz);
  vx = __fmaf_rn(lam[42], S1[63], vx);
  vy = __fmaf_rn(lam[42], S1[55], vy);
  vz = __fmaf_rn(lam[42], S1[56], vz);
  vx = __fmaf_rn(lam[43], __fsub_rn(-S1[49], S1[51]), vx);
  vy = __fmaf_rn(lam[43], S1[57], vy);
  vz = __fmaf_rn(lam[43], S1[58], vz);
  vx = __fmaf_rn(lam[44], __fsub_rn(-S1[50], S1[52]), vx);
  vy = __fmaf_rn(lam[44], S1[58], vy);
  vz = __fmaf_rn(lam[44], S1[59], vz);
  vx = __fmaf_rn(lam[45], __fsub_rn(-S1[51], S1[53]), vx);
  vy = __fmaf_rn(lam[45], S1[59], vy);
  vz = __fmaf_rn(lam[45], S1[60], vz);
  vx = __fmaf_rn(lam[46], __fsub_rn(-S1[52], S1[54]), vx);
  vy = __fmaf_rn(lam[46], S1[60], vy);
  vz = __fmaf_rn(lam[46], S1[61], vz);
  vx = __fmaf_rn(lam[47], __fsub_rn(-S1[53], S1[55]), vx);
  vy = __fmaf_rn(lam[47], S1[61], vy);
  vz = __fmaf_rn(lam[47], S1[62], vz);
  vx = __fmaf_rn(lam[48], __fsub_rn(-S1[54], S1[56]), vx);
  vy = __fmaf_rn(lam[48], S1[62], vy);
  vz = __fmaf_rn(lam[48], S1[63], vz);
  V[0] = vx; V[1] = vy; V[2] = vz;
}
__device__ __forceinline__ void gmp_mcsh_grad_coef_order_1(const float* __restrict__ lam, float* __restrict__ Mx, float* __restrict__ My, float* __restrict__ Mz) {
  Mx[0] = __fmul_rn(1.0f, lam[3]);
  My[0] = __fmul_rn(1.0f, lam[1]);
  Mz[0] = __fmul_rn(1.0f, lam[2]);
}
__device__ __forceinline__ void gmp_mcsh_grad_coef_order_2(const float* __restrict__ lam, float* __restrict__ Mx, float* __restrict__ My, float* __restrict__ Mz) {
  Mx[1] = __fmul_rn(3.0f, lam[7]);
  Mx[2] = __fmul_rn(3.0f, lam[8]);
  Mx[3] = __fmaf_rn(-2.0f, lam[6], __fmul_rn(-2.0f, lam[4]));
  My[1] = __fmaf_rn(-2.0f, lam[6], __fmul_rn(4.0f, lam[4]));
  My[2] = __fmul_rn(3.0f, lam[5]);
  My[3] = __fmul_rn(3.0f, lam[7]);
  Mz[1] = __fmul_rn(3.0f, lam[5]);
  Mz[2] = __fmaf_rn(4.0f, lam[6], __fmul_rn(-2.0f, lam[4]));
  Mz[3] = __fmul_rn(3.0f, lam[8]);
}
__device__ __forceinline__ void gmp_mcsh_grad_coef_order_3(const float* __restrict__ lam, float* __restrict__ Mx, float* __restrict__ My, float* __restrict__ Mz) {
  Mx[4] = __fmaf_rn(2.0f, lam[15], __fmul_rn(7.0f, lam[13]));
  Mx[5] = __fmul_rn(5.0f, lam[14]);
  Mx[6] = __fmaf_rn(7.0f, lam[15], __fmul_rn(2.0f, lam[13]));
  Mx[7] = __fmaf_rn(-2.0f, lam[11], __fmul_rn(-6.0f, lam[9]));
  Mx[8] = __fmaf_rn(-6.0f, lam[12], __fmul_rn(-2.0f, lam[10]));
  My[4] = __fmaf_rn(-2.0f, lam[11], __fmul_rn(9.0f, lam[9]));
  My[5] = __fmaf_rn(-6.0f, lam[12], __fmul_rn(8.0f, lam[10]));
  My[6] = __fmul_rn(5.0f, lam[11]);
  My[7] = __fmaf_rn(-2.0f, lam[15], __fmul_rn(8.0f, lam[13]));
  My[8] = __fmul_rn(5.0f, lam[14]);
  Mz[4] = __fmul_rn(5.0f, lam[10]);
  Mz[5] = __fmaf_rn(8.0f, lam[11], __fmul_rn(-6.0f, lam[9]));
  Mz[6] = __fmaf_rn(9.0f, lam[12], __fmul_rn(-2.0f, lam[10]));
  Mz[7] = __fmul_rn(5.0f, lam[14]);
  Mz[8] = __fmaf_rn(8.0f, lam[15], __fmul_rn(-2.0f, lam[13]));
}
__device__ __forceinline__ void gmp_mcsh_grad_coef_order_4(const float* __restrict__ lam, float* __restrict__ Mx, float* __restrict__ My, float* __restrict__ Mz) {
  Mx[9] = __fmaf_rn(2.0f, lam[23], __fmul_rn(13.0f, lam[21]));
  Mx[10] = __fmaf_rn(6.0f, lam[24], __fmul_rn(9.0f, lam[22]));
  Mx[11] = __fmaf_rn(9.0f, lam[23], __fmul_rn(6.0f, lam[21]));
  Mx[12] = __fmaf_rn(13.0f, lam[24], __fmul_rn(2.0f, lam[22]));
  Mx[13] = __fmaf_rn(-2.0f, lam[18], __fmul_rn(-12.0f, lam[16]));
  Mx[14] = __fmaf_rn(-6.0f, lam[19], __fmul_rn(-6.0f, lam[17]));
  Mx[15] = __fmaf_rn(-12.0f, lam[20], __fmul_rn(-2.0f, lam[18]));
  My[9] = __fmaf_rn(-2.0f, lam[18], __fmul_rn(16.0f, lam[16]));
  My[10] = __fmaf_rn(-6.0f, lam[19], __fmul_rn(15.0f, lam[17]));
  My[11] = __fmaf_rn(-12.0f, lam[20], __fmul_rn(12.0f, lam[18]));
  My[12] = __fmul_rn(7.0f, lam[19]);
  My[13] = __fmaf_rn(-2.0f, lam[23], __fmul_rn(15.0f, lam[21]));
  My[14] = __fmaf_rn(-6.0f, lam[24], __fmul_rn(12.0f, lam[22]));
  My[15] = __fmul_rn(7.0f, lam[23]);
  Mz[9] = __fmul_rn(7.0f, lam[17]);
  Mz[10] = __fmaf_rn(12.0f, lam[18], __fmul_rn(-12.0f, lam[16]));
  Mz[11] = __fmaf_rn(15.0f, lam[19], __fmul_rn(-6.0f, lam[17]));
  Mz[12] = __fmaf_rn(16.0f, lam[20], __fmul_rn(-2.0f, lam[18]));
  Mz[13] = __fmul_rn(7.0f, lam[22]);
  Mz[14] = __fmaf_rn(12.0f, lam[23], __fmul_rn(-6.0f, lam[21]));
  Mz[15] = __fmaf_rn(15.0f, lam[24], __fmul_rn(-2.0f, lam[22]));
}

template <int L> struct GmpMcsh;
template <> struct GmpMcsh<0> {
  static constexpr int kInd = 1;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_0(x, y, z, r2, S); }
  static __device__ __forceinline__ void shift_contract(const float* lam, const float* S1, float* V) { gmp_mcsh_shift_contract_0(lam, S1, V); }
};
template <> struct GmpMcsh<1> {
  static constexpr int kInd = 4;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_1(x, y, z, r2, S); }
  static __device__ __forceinline__ void eval_top(float x, float y, float z, float r2, float* S) { gmp_mcsh_top_1(x, y, z, r2, S); }
  static __device__ __forceinline__ void shift_contract(const float* lam, const float* S1, float* V) { gmp_mcsh_shift_contract_1(lam, S1, V); }
};
template <> struct GmpMcsh<2> {
  static constexpr int kInd = 9;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_2(x, y, z, r2, S); }
  static __device__ __forceinline__ void eval_top(float x, float y, float z, float r2, float* S) { gmp_mcsh_top_2(x, y, z, r2, S); }
  static __device__ __forceinline__ void shift_contract(const float* lam, const float* S1, float* V) { gmp_mcsh_shift_contract_2(lam, S1, V); }
};
template <> struct GmpMcsh<3> {
  static constexpr int kInd = 16;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_3(x, y, z, r2, S); }
  static __device__ __forceinline__ void eval_top(float x, float y, float z, float r2, float* S) { gmp_mcsh_top_3(x, y, z, r2, S); }
  static __device__ __forceinline__ void shift_contract(const float* lam, const float* S1, float* V) { gmp_mcsh_shift_contract_3(lam, S1, V); }
};
template <> struct GmpMcsh<4> {
  static constexpr int kInd = 25;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_4(x, y, z, r2, S); }
  static __device__ __forceinline__ void eval_top(float x, float y, float z, float r2, float* S) { gmp_mcsh_top_4(x, y, z, r2, S); }
  static __device__ __forceinline__ void shift_contract(const float* lam, const float* S1, float* V) { gmp_mcsh_shift_contract_4(lam, S1, V); }
};
template <> struct GmpMcsh<5> {
  static constexpr int kInd = 36;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_5(x, y, z, r2, S); }
  static __device__ __forceinline__ void eval_top(float x, float y, float z, float r2, float* S) { gmp_mcsh_top_5(x, y, z, r2, S); }
  static __device__ __forceinline__ void shift_contract(const float* lam, const float* S1, float* V) { gmp_mcsh_shift_contract_5(lam, S1, V); }
};
template <> struct GmpMcsh<6> {
  static constexpr int kInd = 49;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_6(x, y, z, r2, S); }
  static __device__ __forceinline__ void eval_top(float x, float y, float z, float r2, float* S) { gmp_mcsh_top_6(x, y, z, r2, S); }
  static __device__ __forceinline__ void shift_contract(const float* lam, const float* S1, float* V) { gmp_mcsh_shift_contract_6(lam, S1, V); }
};
template <> struct GmpMcsh<7> {
  static constexpr int kInd = 64;
  static __device__ __forceinline__ void eval(float x, float y, float z, float r2, float* S) { gmp_mcsh_indep_7(x, y, z, r2, S); }
  static __device__ __forceinline__ void eval_top(float x, float y, float z, float r2, float* S) { gmp_mcsh_top_7(x, y, z, r2, S); }
};

__device__ __forceinline__ float gmp_mcsh_invariant(int l, const float* mu) {
  switch (l) {
    case 0: return gmp_mcsh_invariant_0(mu);
    case 1: return gmp_mcsh_invariant_1(mu);
    case 2: return gmp_mcsh_invariant_2(mu);
    case 3: return gmp_mcsh_invariant_3(mu);
    case 4: return gmp_mcsh_invariant_4(mu);
    case 5: return gmp_mcsh_invariant_5(mu);
    case 6: return gmp_mcsh_invariant_6(mu);
    default: return 0.0f;
  }
}
// solid harmonics of order l in double-float arithmetic
template <int l>
__device__ __forceinline__ void gmp_solid_df(gmp_f2 x, gmp_f2 y, gmp_f2 z, gmp_f2 r2, gmp_f2* H) {
  if constexpr (l == 0) gmp_solid_df_0(x, y, z, r2, H);
  if constexpr (l == 1) gmp_solid_df_1(x, y, z, r2, H);
  if constexpr (l == 2) gmp_solid_df_2(x, y, z, r2, H);
  if constexpr (l == 3) gmp_solid_df_3(x, y, z, r2, H);
  if constexpr (l == 4) gmp_solid_df_4(x, y, z, r2, H);
  if constexpr (l == 5) gmp_solid_df_5(x, y, z, r2, H);
  if constexpr (l == 6) gmp_solid_df_6(x, y, z, r2, H);
}
__device__ __forceinline__ void gmp_mcsh_shift_contract_order(int l, const float* lam, const float* S1, float* V) {
  switch (l) {
    case 0: gmp_mcsh_shift_contract_order_0(lam, S1, V); break;
    case 1: gmp_mcsh_shift_contract_order_1(lam, S1, V); break;
    case 2: gmp_mcsh_shift_contract_order_2(lam, S1, V); break;
    case 3: gmp_mcsh_shift_contract_order_3(lam, S1, V); break;
    case 4: gmp_mcsh_shift_contract_order_4(lam, S1, V); break;
    case 5: gmp_mcsh_shift_contract_order_5(lam, S1, V); break;
    case 6: gmp_mcsh_shift_contract_order_6(lam, S1, V); break;
    default: V[0] = V[1] = V[2] = 0.0f; break;
  }
}
__device__ __forceinline__ void gmp_mcsh_invariant_adjoint(int l, const float* mu, float g, float* lam) {
  switch (l) {
    case 0: gmp_mcsh_invariant_adjoint_0(mu, g, lam); break;
    case 1: gmp_mcsh_invariant_adjoint_1(mu, g, lam); break;
    case 2: gmp_mcsh_invariant_adjoint_2(mu, g, lam); break;
    case 3: gmp_mcsh_invariant_adjoint_3(mu, g, lam); break;
    case 4: gmp_mcsh_invariant_adjoint_4(mu, g, lam); break;
    case 5: gmp_mcsh_invariant_adjoint_5(mu, g, lam); break;
    case 6: gmp_mcsh_invariant_adjoint_6(mu, g, lam); break;
    default: break;
  }
}
