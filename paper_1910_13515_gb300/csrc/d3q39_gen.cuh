// d3q39_gen.cuh -- GENERATED by gen_d3q39.py; do not edit.
#pragma once

namespace lbm39 {
namespace gen {

// Rounded products that are never contracted into a fused multiply-add.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

// e_i = sum_k l_k phi_k(xi_i) for every velocity (exponent of Eq. discrete-equilibrium),
// in the type of l (double; float for the single-precision start of a solve).
template <class T>
__device__ __forceinline__ void exponents(const T (&l)[13], T (&e)[39]) {
  const T c0_0 = l[0];
  e[0] = c0_0;
  const T c1_0 = l[0] + l[6];
  const T c1_z = l[3] + l[12];
  const T t1_0_0 = c1_0 + c1_z;
  const T t1_0_1 = c1_0 - c1_z;
  e[5] = t1_0_0;
  e[6] = t1_0_1;
  const T c2_0 = fma(T(4), l[6], l[0]);
  const T c2_z = fma(T(8), l[12], mul_rn(T(2), l[3]));
  const T t2_0_0 = c2_0 + c2_z;
  const T t2_0_1 = c2_0 - c2_z;
  e[19] = t2_0_0;
  e[20] = t2_0_1;
  const T c3_0 = fma(T(9), l[6], l[0]);
  const T c3_z = fma(T(27), l[12], mul_rn(T(3), l[3]));
  const T t3_0_0 = c3_0 + c3_z;
  const T t3_0_1 = c3_0 - c3_z;
  e[37] = t3_0_0;
  e[38] = t3_0_1;
  const T c4_0 = l[0] + l[5];
  const T c4_y = l[2] + l[11];
  const T t4_0_0 = c4_0 + c4_y;
  const T t4_0_1 = c4_0 - c4_y;
  e[3] = t4_0_0;
  e[4] = t4_0_1;
  const T c5_0 = fma(T(4), l[5], l[0]);
  const T c5_y = fma(T(8), l[11], mul_rn(T(2), l[2]));
  const T t5_0_0 = c5_0 + c5_y;
  const T t5_0_1 = c5_0 - c5_y;
  e[17] = t5_0_0;
  e[18] = t5_0_1;
  const T c6_0 = fma(T(4), l[6], fma(T(4), l[5], l[0]));
  const T c6_y = fma(T(16), l[11], mul_rn(T(2), l[2]));
  const T c6_z = fma(T(16), l[12], mul_rn(T(2), l[3]));
  const T c6_yz = mul_rn(T(4), l[9]);
  const T t6_0_0 = c6_0 + c6_y;
  const T t6_0_1 = c6_0 - c6_y;
  const T t6_0_2 = c6_z + c6_yz;
  const T t6_0_3 = c6_z - c6_yz;
  const T t6_1_0 = t6_0_0 + t6_0_2;
  const T t6_1_1 = t6_0_0 - t6_0_2;
  const T t6_1_2 = t6_0_1 + t6_0_3;
  const T t6_1_3 = t6_0_1 - t6_0_3;
  e[29] = t6_1_0;
  e[31] = t6_1_1;
  e[32] = t6_1_2;
  e[30] = t6_1_3;
  const T c7_0 = fma(T(9), l[5], l[0]);
  const T c7_y = fma(T(27), l[11], mul_rn(T(3), l[2]));
  const T t7_0_0 = c7_0 + c7_y;
  const T t7_0_1 = c7_0 - c7_y;
  e[35] = t7_0_0;
  e[36] = t7_0_1;
  const T c8_0 = l[0] + l[4];
  const T c8_x = l[1] + l[10];
  const T t8_0_0 = c8_0 + c8_x;
  const T t8_0_1 = c8_0 - c8_x;
  e[1] = t8_0_0;
  e[2] = t8_0_1;
  const T c9_0 = l[0] + l[4] + l[5] + l[6];
  const T c9_x = fma(T(3), l[10], l[1]);
  const T c9_y = fma(T(3), l[11], l[2]);
  const T c9_z = fma(T(3), l[12], l[3]);
  const T c9_xy = l[7];
  const T c9_xz = l[8];
  const T c9_yz = l[9];
  const T t9_0_0 = c9_0 + c9_x;
  const T t9_0_1 = c9_0 - c9_x;
  const T t9_0_2 = c9_y + c9_xy;
  const T t9_0_3 = c9_y - c9_xy;
  const T t9_0_4 = c9_z + c9_xz;
  const T t9_0_5 = c9_z - c9_xz;
  const T t9_1_0 = t9_0_0 + t9_0_2;
  const T t9_1_1 = t9_0_0 - t9_0_2;
  const T t9_1_2 = t9_0_1 + t9_0_3;
  const T t9_1_3 = t9_0_1 - t9_0_3;
  const T t9_1_4 = t9_0_4 + c9_yz;
  const T t9_1_5 = t9_0_4 - c9_yz;
  const T t9_1_6 = t9_0_5 + c9_yz;
  const T t9_1_7 = t9_0_5 - c9_yz;
  const T t9_2_0 = t9_1_0 + t9_1_4;
  const T t9_2_1 = t9_1_0 - t9_1_4;
  const T t9_2_2 = t9_1_1 + t9_1_5;
  const T t9_2_3 = t9_1_1 - t9_1_5;
  const T t9_2_4 = t9_1_2 + t9_1_6;
  const T t9_2_5 = t9_1_2 - t9_1_6;
  const T t9_2_6 = t9_1_3 + t9_1_7;
  const T t9_2_7 = t9_1_3 - t9_1_7;
  e[7] = t9_2_0;
  e[9] = t9_2_1;
  e[11] = t9_2_2;
  e[14] = t9_2_3;
  e[13] = t9_2_4;
  e[12] = t9_2_5;
  e[10] = t9_2_6;
  e[8] = t9_2_7;
  const T c10_0 = fma(T(4), l[4], l[0]);
  const T c10_x = fma(T(8), l[10], mul_rn(T(2), l[1]));
  const T t10_0_0 = c10_0 + c10_x;
  const T t10_0_1 = c10_0 - c10_x;
  e[15] = t10_0_0;
  e[16] = t10_0_1;
  const T c11_0 = fma(T(4), l[6], fma(T(4), l[4], l[0]));
  const T c11_x = fma(T(16), l[10], mul_rn(T(2), l[1]));
  const T c11_z = fma(T(16), l[12], mul_rn(T(2), l[3]));
  const T c11_xz = mul_rn(T(4), l[8]);
  const T t11_0_0 = c11_0 + c11_x;
  const T t11_0_1 = c11_0 - c11_x;
  const T t11_0_2 = c11_z + c11_xz;
  const T t11_0_3 = c11_z - c11_xz;
  const T t11_1_0 = t11_0_0 + t11_0_2;
  const T t11_1_1 = t11_0_0 - t11_0_2;
  const T t11_1_2 = t11_0_1 + t11_0_3;
  const T t11_1_3 = t11_0_1 - t11_0_3;
  e[25] = t11_1_0;
  e[27] = t11_1_1;
  e[28] = t11_1_2;
  e[26] = t11_1_3;
  const T c12_0 = fma(T(4), l[5], fma(T(4), l[4], l[0]));
  const T c12_x = fma(T(16), l[10], mul_rn(T(2), l[1]));
  const T c12_y = fma(T(16), l[11], mul_rn(T(2), l[2]));
  const T c12_xy = mul_rn(T(4), l[7]);
  const T t12_0_0 = c12_0 + c12_x;
  const T t12_0_1 = c12_0 - c12_x;
  const T t12_0_2 = c12_y + c12_xy;
  const T t12_0_3 = c12_y - c12_xy;
  const T t12_1_0 = t12_0_0 + t12_0_2;
  const T t12_1_1 = t12_0_0 - t12_0_2;
  const T t12_1_2 = t12_0_1 + t12_0_3;
  const T t12_1_3 = t12_0_1 - t12_0_3;
  e[21] = t12_1_0;
  e[23] = t12_1_1;
  e[24] = t12_1_2;
  e[22] = t12_1_3;
  const T c13_0 = fma(T(9), l[4], l[0]);
  const T c13_x = fma(T(27), l[10], mul_rn(T(3), l[1]));
  const T t13_0_0 = c13_0 + c13_x;
  const T t13_0_1 = c13_0 - c13_x;
  e[33] = t13_0_0;
  e[34] = t13_0_1;
}

// The same with the z-odd multipliers zero (lattice one cell thick in z, u_z = 0).
template <class T>
__device__ __forceinline__ void exponents2d(const T (&l)[13], T (&e)[39]) {
  const T c0_0 = l[0];
  e[0] = c0_0;
  const T c1_0 = l[0] + l[6];
  e[5] = c1_0;
  e[6] = c1_0;
  const T c2_0 = fma(T(4), l[6], l[0]);
  e[19] = c2_0;
  e[20] = c2_0;
  const T c3_0 = fma(T(9), l[6], l[0]);
  e[37] = c3_0;
  e[38] = c3_0;
  const T c4_0 = l[0] + l[5];
  const T c4_y = l[2] + l[11];
  const T t4_0_0 = c4_0 + c4_y;
  const T t4_0_1 = c4_0 - c4_y;
  e[3] = t4_0_0;
  e[4] = t4_0_1;
  const T c5_0 = fma(T(4), l[5], l[0]);
  const T c5_y = fma(T(8), l[11], mul_rn(T(2), l[2]));
  const T t5_0_0 = c5_0 + c5_y;
  const T t5_0_1 = c5_0 - c5_y;
  e[17] = t5_0_0;
  e[18] = t5_0_1;
  const T c6_0 = fma(T(4), l[6], fma(T(4), l[5], l[0]));
  const T c6_y = fma(T(16), l[11], mul_rn(T(2), l[2]));
  const T t6_0_0 = c6_0 + c6_y;
  const T t6_0_1 = c6_0 - c6_y;
  e[29] = t6_0_0;
  e[31] = t6_0_0;
  e[32] = t6_0_1;
  e[30] = t6_0_1;
  const T c7_0 = fma(T(9), l[5], l[0]);
  const T c7_y = fma(T(27), l[11], mul_rn(T(3), l[2]));
  const T t7_0_0 = c7_0 + c7_y;
  const T t7_0_1 = c7_0 - c7_y;
  e[35] = t7_0_0;
  e[36] = t7_0_1;
  const T c8_0 = l[0] + l[4];
  const T c8_x = l[1] + l[10];
  const T t8_0_0 = c8_0 + c8_x;
  const T t8_0_1 = c8_0 - c8_x;
  e[1] = t8_0_0;
  e[2] = t8_0_1;
  const T c9_0 = l[0] + l[4] + l[5] + l[6];
  const T c9_x = fma(T(3), l[10], l[1]);
  const T c9_y = fma(T(3), l[11], l[2]);
  const T c9_xy = l[7];
  const T t9_0_0 = c9_0 + c9_x;
  const T t9_0_1 = c9_0 - c9_x;
  const T t9_0_2 = c9_y + c9_xy;
  const T t9_0_3 = c9_y - c9_xy;
  const T t9_1_0 = t9_0_0 + t9_0_2;
  const T t9_1_1 = t9_0_0 - t9_0_2;
  const T t9_1_2 = t9_0_1 + t9_0_3;
  const T t9_1_3 = t9_0_1 - t9_0_3;
  e[7] = t9_1_0;
  e[9] = t9_1_0;
  e[11] = t9_1_1;
  e[14] = t9_1_1;
  e[13] = t9_1_2;
  e[12] = t9_1_2;
  e[10] = t9_1_3;
  e[8] = t9_1_3;
  const T c10_0 = fma(T(4), l[4], l[0]);
  const T c10_x = fma(T(8), l[10], mul_rn(T(2), l[1]));
  const T t10_0_0 = c10_0 + c10_x;
  const T t10_0_1 = c10_0 - c10_x;
  e[15] = t10_0_0;
  e[16] = t10_0_1;
  const T c11_0 = fma(T(4), l[6], fma(T(4), l[4], l[0]));
  const T c11_x = fma(T(16), l[10], mul_rn(T(2), l[1]));
  const T t11_0_0 = c11_0 + c11_x;
  const T t11_0_1 = c11_0 - c11_x;
  e[25] = t11_0_0;
  e[27] = t11_0_0;
  e[28] = t11_0_1;
  e[26] = t11_0_1;
  const T c12_0 = fma(T(4), l[5], fma(T(4), l[4], l[0]));
  const T c12_x = fma(T(16), l[10], mul_rn(T(2), l[1]));
  const T c12_y = fma(T(16), l[11], mul_rn(T(2), l[2]));
  const T c12_xy = mul_rn(T(4), l[7]);
  const T t12_0_0 = c12_0 + c12_x;
  const T t12_0_1 = c12_0 - c12_x;
  const T t12_0_2 = c12_y + c12_xy;
  const T t12_0_3 = c12_y - c12_xy;
  const T t12_1_0 = t12_0_0 + t12_0_2;
  const T t12_1_1 = t12_0_0 - t12_0_2;
  const T t12_1_2 = t12_0_1 + t12_0_3;
  const T t12_1_3 = t12_0_1 - t12_0_3;
  e[21] = t12_1_0;
  e[23] = t12_1_1;
  e[24] = t12_1_2;
  e[22] = t12_1_3;
  const T c13_0 = fma(T(9), l[4], l[0]);
  const T c13_x = fma(T(27), l[10], mul_rn(T(3), l[1]));
  const T t13_0_0 = c13_0 + c13_x;
  const T t13_0_1 = c13_0 - c13_x;
  e[33] = t13_0_0;
  e[34] = t13_0_1;
}

// s_k = sum_i F_i phi_k(xi_i) and J_kl = sum_i F_i phi_k(xi_i) phi_l(xi_i) (l <= k,
// packed) from the Walsh-Hadamard coefficients of the sign orbits.
template <class T, class A>
__device__ __forceinline__ void moments(const A& F, T (&s)[13], T (&J)[91]) {
  const T h000_0 = F[0];
  const T w1_0_0 = F[5] + F[6];
  const T w1_0_1 = F[5] - F[6];
  const T h001_0 = w1_0_0;
  const T h001_z = w1_0_1;
  const T w2_0_0 = F[19] + F[20];
  const T w2_0_1 = F[19] - F[20];
  const T h002_0 = w2_0_0;
  const T h002_z = w2_0_1;
  const T w3_0_0 = F[37] + F[38];
  const T w3_0_1 = F[37] - F[38];
  const T h003_0 = w3_0_0;
  const T h003_z = w3_0_1;
  const T w4_0_0 = F[3] + F[4];
  const T w4_0_1 = F[3] - F[4];
  const T h010_0 = w4_0_0;
  const T h010_y = w4_0_1;
  const T w5_0_0 = F[17] + F[18];
  const T w5_0_1 = F[17] - F[18];
  const T h020_0 = w5_0_0;
  const T h020_y = w5_0_1;
  const T w6_0_0 = F[29] + F[32];
  const T w6_0_1 = F[29] - F[32];
  const T w6_0_2 = F[31] + F[30];
  const T w6_0_3 = F[31] - F[30];
  const T w6_1_0 = w6_0_0 + w6_0_2;
  const T w6_1_1 = w6_0_0 - w6_0_2;
  const T w6_1_2 = w6_0_1 + w6_0_3;
  const T w6_1_3 = w6_0_1 - w6_0_3;
  const T h022_0 = w6_1_0;
  const T h022_z = w6_1_1;
  const T h022_y = w6_1_2;
  const T h022_yz = w6_1_3;
  const T w7_0_0 = F[35] + F[36];
  const T w7_0_1 = F[35] - F[36];
  const T h030_0 = w7_0_0;
  const T h030_y = w7_0_1;
  const T w8_0_0 = F[1] + F[2];
  const T w8_0_1 = F[1] - F[2];
  const T h100_0 = w8_0_0;
  const T h100_x = w8_0_1;
  const T w9_0_0 = F[7] + F[13];
  const T w9_0_1 = F[7] - F[13];
  const T w9_0_2 = F[9] + F[12];
  const T w9_0_3 = F[9] - F[12];
  const T w9_0_4 = F[11] + F[10];
  const T w9_0_5 = F[11] - F[10];
  const T w9_0_6 = F[14] + F[8];
  const T w9_0_7 = F[14] - F[8];
  const T w9_1_0 = w9_0_0 + w9_0_4;
  const T w9_1_1 = w9_0_0 - w9_0_4;
  const T w9_1_2 = w9_0_1 + w9_0_5;
  const T w9_1_3 = w9_0_1 - w9_0_5;
  const T w9_1_4 = w9_0_2 + w9_0_6;
  const T w9_1_5 = w9_0_2 - w9_0_6;
  const T w9_1_6 = w9_0_3 + w9_0_7;
  const T w9_1_7 = w9_0_3 - w9_0_7;
  const T w9_2_0 = w9_1_0 + w9_1_4;
  const T w9_2_1 = w9_1_0 - w9_1_4;
  const T w9_2_2 = w9_1_1 + w9_1_5;
  const T w9_2_3 = w9_1_1 - w9_1_5;
  const T w9_2_4 = w9_1_2 + w9_1_6;
  const T w9_2_5 = w9_1_2 - w9_1_6;
  const T w9_2_6 = w9_1_3 + w9_1_7;
  const T w9_2_7 = w9_1_3 - w9_1_7;
  const T h111_0 = w9_2_0;
  const T h111_z = w9_2_1;
  const T h111_y = w9_2_2;
  const T h111_yz = w9_2_3;
  const T h111_x = w9_2_4;
  const T h111_xz = w9_2_5;
  const T h111_xy = w9_2_6;
  const T h111_xyz = w9_2_7;
  const T w10_0_0 = F[15] + F[16];
  const T w10_0_1 = F[15] - F[16];
  const T h200_0 = w10_0_0;
  const T h200_x = w10_0_1;
  const T w11_0_0 = F[25] + F[28];
  const T w11_0_1 = F[25] - F[28];
  const T w11_0_2 = F[27] + F[26];
  const T w11_0_3 = F[27] - F[26];
  const T w11_1_0 = w11_0_0 + w11_0_2;
  const T w11_1_1 = w11_0_0 - w11_0_2;
  const T w11_1_2 = w11_0_1 + w11_0_3;
  const T w11_1_3 = w11_0_1 - w11_0_3;
  const T h202_0 = w11_1_0;
  const T h202_z = w11_1_1;
  const T h202_x = w11_1_2;
  const T h202_xz = w11_1_3;
  const T w12_0_0 = F[21] + F[24];
  const T w12_0_1 = F[21] - F[24];
  const T w12_0_2 = F[23] + F[22];
  const T w12_0_3 = F[23] - F[22];
  const T w12_1_0 = w12_0_0 + w12_0_2;
  const T w12_1_1 = w12_0_0 - w12_0_2;
  const T w12_1_2 = w12_0_1 + w12_0_3;
  const T w12_1_3 = w12_0_1 - w12_0_3;
  const T h220_0 = w12_1_0;
  const T h220_y = w12_1_1;
  const T h220_x = w12_1_2;
  const T h220_xy = w12_1_3;
  const T w13_0_0 = F[33] + F[34];
  const T w13_0_1 = F[33] - F[34];
  const T h300_0 = w13_0_0;
  const T h300_x = w13_0_1;
  const T M000_0 = (((h000_0 + h010_0 + h100_0 + h220_0) + (h001_0 + h020_0 + h111_0 + h300_0)) + ((h002_0 + h022_0 + h200_0) + (h003_0 + h030_0 + h202_0)));
  const T M001_0 = ((fma(T(2), h022_z, fma(T(2), h002_z, h001_z))) + (fma(T(2), h202_z, fma(T(3), h003_z, h111_z))));
  const T M010_0 = ((fma(T(3), h030_y, fma(T(2), h020_y, h010_y))) + (fma(T(2), h220_y, fma(T(2), h022_y, h111_y))));
  const T M100_0 = ((fma(T(2), h220_x, fma(T(2), h200_x, h100_x))) + (fma(T(3), h300_x, fma(T(2), h202_x, h111_x))));
  const T M002_0 = ((fma(T(4), h022_0, fma(T(4), h002_0, h001_0))) + (fma(T(4), h202_0, fma(T(9), h003_0, h111_0))));
  const T M011_0 = fma(T(4), h022_yz, h111_yz);
  const T M020_0 = ((fma(T(9), h030_0, fma(T(4), h020_0, h010_0))) + (fma(T(4), h220_0, fma(T(4), h022_0, h111_0))));
  const T M101_0 = fma(T(4), h202_xz, h111_xz);
  const T M110_0 = fma(T(4), h220_xy, h111_xy);
  const T M200_0 = ((fma(T(4), h220_0, fma(T(4), h200_0, h100_0))) + (fma(T(9), h300_0, fma(T(4), h202_0, h111_0))));
  const T M003_0 = ((fma(T(8), h022_z, fma(T(8), h002_z, h001_z))) + (fma(T(8), h202_z, fma(T(27), h003_z, h111_z))));
  const T M012_0 = fma(T(8), h022_y, h111_y);
  const T M021_0 = fma(T(8), h022_z, h111_z);
  const T M030_0 = ((fma(T(27), h030_y, fma(T(8), h020_y, h010_y))) + (fma(T(8), h220_y, fma(T(8), h022_y, h111_y))));
  const T M102_0 = fma(T(8), h202_x, h111_x);
  const T M111_0 = h111_xyz;
  const T M120_0 = fma(T(8), h220_x, h111_x);
  const T M201_0 = fma(T(8), h202_z, h111_z);
  const T M210_0 = fma(T(8), h220_y, h111_y);
  const T M300_0 = ((fma(T(8), h220_x, fma(T(8), h200_x, h100_x))) + (fma(T(27), h300_x, fma(T(8), h202_x, h111_x))));
  const T M004_0 = ((fma(T(16), h022_0, fma(T(16), h002_0, h001_0))) + (fma(T(16), h202_0, fma(T(81), h003_0, h111_0))));
  const T M013_0 = fma(T(16), h022_yz, h111_yz);
  const T M022_0 = fma(T(16), h022_0, h111_0);
  const T M031_0 = fma(T(16), h022_yz, h111_yz);
  const T M040_0 = ((fma(T(81), h030_0, fma(T(16), h020_0, h010_0))) + (fma(T(16), h220_0, fma(T(16), h022_0, h111_0))));
  const T M103_0 = fma(T(16), h202_xz, h111_xz);
  const T M112_0 = h111_xy;
  const T M121_0 = h111_xz;
  const T M130_0 = fma(T(16), h220_xy, h111_xy);
  const T M202_0 = fma(T(16), h202_0, h111_0);
  const T M211_0 = h111_yz;
  const T M220_0 = fma(T(16), h220_0, h111_0);
  const T M301_0 = fma(T(16), h202_xz, h111_xz);
  const T M310_0 = fma(T(16), h220_xy, h111_xy);
  const T M400_0 = ((fma(T(16), h220_0, fma(T(16), h200_0, h100_0))) + (fma(T(81), h300_0, fma(T(16), h202_0, h111_0))));
  const T M001_1 = ((fma(T(16), h202_z, fma(T(16), h022_z, fma(T(8), h002_z, h001_z)))) + (fma(T(3), h111_z, mul_rn(T(27), h003_z))));
  const T M010_1 = ((fma(T(16), h220_y, fma(T(27), h030_y, fma(T(8), h020_y, h010_y)))) + (fma(T(3), h111_y, mul_rn(T(16), h022_y))));
  const T M100_1 = ((fma(T(27), h300_x, fma(T(16), h202_x, fma(T(3), h111_x, h100_x)))) + (fma(T(16), h220_x, mul_rn(T(8), h200_x))));
  const T M002_1 = ((fma(T(32), h202_0, fma(T(32), h022_0, fma(T(16), h002_0, h001_0)))) + (fma(T(3), h111_0, mul_rn(T(81), h003_0))));
  const T M011_1 = fma(T(3), h111_yz, mul_rn(T(32), h022_yz));
  const T M020_1 = ((fma(T(32), h220_0, fma(T(81), h030_0, fma(T(16), h020_0, h010_0)))) + (fma(T(3), h111_0, mul_rn(T(32), h022_0))));
  const T M101_1 = fma(T(32), h202_xz, mul_rn(T(3), h111_xz));
  const T M110_1 = fma(T(32), h220_xy, mul_rn(T(3), h111_xy));
  const T M200_1 = ((fma(T(81), h300_0, fma(T(32), h202_0, fma(T(3), h111_0, h100_0)))) + (fma(T(32), h220_0, mul_rn(T(16), h200_0))));
  const T M003_1 = ((fma(T(64), h202_z, fma(T(64), h022_z, fma(T(32), h002_z, h001_z)))) + (fma(T(3), h111_z, mul_rn(T(243), h003_z))));
  const T M012_1 = fma(T(3), h111_y, mul_rn(T(64), h022_y));
  const T M021_1 = fma(T(3), h111_z, mul_rn(T(64), h022_z));
  const T M030_1 = ((fma(T(64), h220_y, fma(T(243), h030_y, fma(T(32), h020_y, h010_y)))) + (fma(T(3), h111_y, mul_rn(T(64), h022_y))));
  const T M102_1 = fma(T(64), h202_x, mul_rn(T(3), h111_x));
  const T M111_1 = mul_rn(T(3), h111_xyz);
  const T M120_1 = fma(T(64), h220_x, mul_rn(T(3), h111_x));
  const T M201_1 = fma(T(64), h202_z, mul_rn(T(3), h111_z));
  const T M210_1 = fma(T(64), h220_y, mul_rn(T(3), h111_y));
  const T M300_1 = ((fma(T(243), h300_x, fma(T(64), h202_x, fma(T(3), h111_x, h100_x)))) + (fma(T(64), h220_x, mul_rn(T(32), h200_x))));
  const T M002_2 = ((fma(T(256), h202_0, fma(T(256), h022_0, fma(T(64), h002_0, h001_0)))) + (fma(T(9), h111_0, mul_rn(T(729), h003_0))));
  const T M011_2 = fma(T(9), h111_yz, mul_rn(T(256), h022_yz));
  const T M020_2 = ((fma(T(256), h220_0, fma(T(729), h030_0, fma(T(64), h020_0, h010_0)))) + (fma(T(9), h111_0, mul_rn(T(256), h022_0))));
  const T M101_2 = fma(T(256), h202_xz, mul_rn(T(9), h111_xz));
  const T M110_2 = fma(T(256), h220_xy, mul_rn(T(9), h111_xy));
  const T M200_2 = ((fma(T(729), h300_0, fma(T(256), h202_0, fma(T(9), h111_0, h100_0)))) + (fma(T(256), h220_0, mul_rn(T(64), h200_0))));
  s[0] = M000_0;
  s[1] = M100_0;
  s[2] = M010_0;
  s[3] = M001_0;
  s[4] = M200_0;
  s[5] = M020_0;
  s[6] = M002_0;
  s[7] = M110_0;
  s[8] = M101_0;
  s[9] = M011_0;
  s[10] = M100_1;
  s[11] = M010_1;
  s[12] = M001_1;
  J[0] = M000_0;
  J[1] = M100_0;
  J[2] = M200_0;
  J[3] = M010_0;
  J[4] = M110_0;
  J[5] = M020_0;
  J[6] = M001_0;
  J[7] = M101_0;
  J[8] = M011_0;
  J[9] = M002_0;
  J[10] = M200_0;
  J[11] = M300_0;
  J[12] = M210_0;
  J[13] = M201_0;
  J[14] = M400_0;
  J[15] = M020_0;
  J[16] = M120_0;
  J[17] = M030_0;
  J[18] = M021_0;
  J[19] = M220_0;
  J[20] = M040_0;
  J[21] = M002_0;
  J[22] = M102_0;
  J[23] = M012_0;
  J[24] = M003_0;
  J[25] = M202_0;
  J[26] = M022_0;
  J[27] = M004_0;
  J[28] = M110_0;
  J[29] = M210_0;
  J[30] = M120_0;
  J[31] = M111_0;
  J[32] = M310_0;
  J[33] = M130_0;
  J[34] = M112_0;
  J[35] = M220_0;
  J[36] = M101_0;
  J[37] = M201_0;
  J[38] = M111_0;
  J[39] = M102_0;
  J[40] = M301_0;
  J[41] = M121_0;
  J[42] = M103_0;
  J[43] = M211_0;
  J[44] = M202_0;
  J[45] = M011_0;
  J[46] = M111_0;
  J[47] = M021_0;
  J[48] = M012_0;
  J[49] = M211_0;
  J[50] = M031_0;
  J[51] = M013_0;
  J[52] = M121_0;
  J[53] = M112_0;
  J[54] = M022_0;
  J[55] = M100_1;
  J[56] = M200_1;
  J[57] = M110_1;
  J[58] = M101_1;
  J[59] = M300_1;
  J[60] = M120_1;
  J[61] = M102_1;
  J[62] = M210_1;
  J[63] = M201_1;
  J[64] = M111_1;
  J[65] = M200_2;
  J[66] = M010_1;
  J[67] = M110_1;
  J[68] = M020_1;
  J[69] = M011_1;
  J[70] = M210_1;
  J[71] = M030_1;
  J[72] = M012_1;
  J[73] = M120_1;
  J[74] = M111_1;
  J[75] = M021_1;
  J[76] = M110_2;
  J[77] = M020_2;
  J[78] = M001_1;
  J[79] = M101_1;
  J[80] = M011_1;
  J[81] = M002_1;
  J[82] = M201_1;
  J[83] = M021_1;
  J[84] = M003_1;
  J[85] = M111_1;
  J[86] = M102_1;
  J[87] = M012_1;
  J[88] = M101_2;
  J[89] = M011_2;
  J[90] = M002_2;
}

// s_k = sum_i F_i phi_k(xi_i) only.
template <class T, class A>
__device__ __forceinline__ void moments_s(const A& F, T (&s)[13]) {
  const T h000_0 = F[0];
  const T w1_0_0 = F[5] + F[6];
  const T w1_0_1 = F[5] - F[6];
  const T h001_0 = w1_0_0;
  const T h001_z = w1_0_1;
  const T w2_0_0 = F[19] + F[20];
  const T w2_0_1 = F[19] - F[20];
  const T h002_0 = w2_0_0;
  const T h002_z = w2_0_1;
  const T w3_0_0 = F[37] + F[38];
  const T w3_0_1 = F[37] - F[38];
  const T h003_0 = w3_0_0;
  const T h003_z = w3_0_1;
  const T w4_0_0 = F[3] + F[4];
  const T w4_0_1 = F[3] - F[4];
  const T h010_0 = w4_0_0;
  const T h010_y = w4_0_1;
  const T w5_0_0 = F[17] + F[18];
  const T w5_0_1 = F[17] - F[18];
  const T h020_0 = w5_0_0;
  const T h020_y = w5_0_1;
  const T w6_0_0 = F[29] + F[32];
  const T w6_0_1 = F[29] - F[32];
  const T w6_0_2 = F[31] + F[30];
  const T w6_0_3 = F[31] - F[30];
  const T w6_1_0 = w6_0_0 + w6_0_2;
  const T w6_1_1 = w6_0_0 - w6_0_2;
  const T w6_1_2 = w6_0_1 + w6_0_3;
  const T w6_1_3 = w6_0_1 - w6_0_3;
  const T h022_0 = w6_1_0;
  const T h022_z = w6_1_1;
  const T h022_y = w6_1_2;
  const T h022_yz = w6_1_3;
  const T w7_0_0 = F[35] + F[36];
  const T w7_0_1 = F[35] - F[36];
  const T h030_0 = w7_0_0;
  const T h030_y = w7_0_1;
  const T w8_0_0 = F[1] + F[2];
  const T w8_0_1 = F[1] - F[2];
  const T h100_0 = w8_0_0;
  const T h100_x = w8_0_1;
  const T w9_0_0 = F[7] + F[13];
  const T w9_0_1 = F[7] - F[13];
  const T w9_0_2 = F[9] + F[12];
  const T w9_0_3 = F[9] - F[12];
  const T w9_0_4 = F[11] + F[10];
  const T w9_0_5 = F[11] - F[10];
  const T w9_0_6 = F[14] + F[8];
  const T w9_0_7 = F[14] - F[8];
  const T w9_1_0 = w9_0_0 + w9_0_4;
  const T w9_1_1 = w9_0_0 - w9_0_4;
  const T w9_1_2 = w9_0_1 + w9_0_5;
  const T w9_1_3 = w9_0_1 - w9_0_5;
  const T w9_1_4 = w9_0_2 + w9_0_6;
  const T w9_1_5 = w9_0_2 - w9_0_6;
  const T w9_1_6 = w9_0_3 + w9_0_7;
  const T w9_1_7 = w9_0_3 - w9_0_7;
  const T w9_2_0 = w9_1_0 + w9_1_4;
  const T w9_2_1 = w9_1_0 - w9_1_4;
  const T w9_2_2 = w9_1_1 + w9_1_5;
  const T w9_2_3 = w9_1_1 - w9_1_5;
  const T w9_2_4 = w9_1_2 + w9_1_6;
  const T w9_2_5 = w9_1_2 - w9_1_6;
  const T w9_2_6 = w9_1_3 + w9_1_7;
  const T w9_2_7 = w9_1_3 - w9_1_7;
  const T h111_0 = w9_2_0;
  const T h111_z = w9_2_1;
  const T h111_y = w9_2_2;
  const T h111_yz = w9_2_3;
  const T h111_x = w9_2_4;
  const T h111_xz = w9_2_5;
  const T h111_xy = w9_2_6;
  const T h111_xyz = w9_2_7;
  const T w10_0_0 = F[15] + F[16];
  const T w10_0_1 = F[15] - F[16];
  const T h200_0 = w10_0_0;
  const T h200_x = w10_0_1;
  const T w11_0_0 = F[25] + F[28];
  const T w11_0_1 = F[25] - F[28];
  const T w11_0_2 = F[27] + F[26];
  const T w11_0_3 = F[27] - F[26];
  const T w11_1_0 = w11_0_0 + w11_0_2;
  const T w11_1_1 = w11_0_0 - w11_0_2;
  const T w11_1_2 = w11_0_1 + w11_0_3;
  const T w11_1_3 = w11_0_1 - w11_0_3;
  const T h202_0 = w11_1_0;
  const T h202_z = w11_1_1;
  const T h202_x = w11_1_2;
  const T h202_xz = w11_1_3;
  const T w12_0_0 = F[21] + F[24];
  const T w12_0_1 = F[21] - F[24];
  const T w12_0_2 = F[23] + F[22];
  const T w12_0_3 = F[23] - F[22];
  const T w12_1_0 = w12_0_0 + w12_0_2;
  const T w12_1_1 = w12_0_0 - w12_0_2;
  const T w12_1_2 = w12_0_1 + w12_0_3;
  const T w12_1_3 = w12_0_1 - w12_0_3;
  const T h220_0 = w12_1_0;
  const T h220_y = w12_1_1;
  const T h220_x = w12_1_2;
  const T h220_xy = w12_1_3;
  const T w13_0_0 = F[33] + F[34];
  const T w13_0_1 = F[33] - F[34];
  const T h300_0 = w13_0_0;
  const T h300_x = w13_0_1;
  const T M000_0 = (((h000_0 + h010_0 + h100_0 + h220_0) + (h001_0 + h020_0 + h111_0 + h300_0)) + ((h002_0 + h022_0 + h200_0) + (h003_0 + h030_0 + h202_0)));
  const T M001_0 = ((fma(T(2), h022_z, fma(T(2), h002_z, h001_z))) + (fma(T(2), h202_z, fma(T(3), h003_z, h111_z))));
  const T M010_0 = ((fma(T(3), h030_y, fma(T(2), h020_y, h010_y))) + (fma(T(2), h220_y, fma(T(2), h022_y, h111_y))));
  const T M100_0 = ((fma(T(2), h220_x, fma(T(2), h200_x, h100_x))) + (fma(T(3), h300_x, fma(T(2), h202_x, h111_x))));
  const T M002_0 = ((fma(T(4), h022_0, fma(T(4), h002_0, h001_0))) + (fma(T(4), h202_0, fma(T(9), h003_0, h111_0))));
  const T M011_0 = fma(T(4), h022_yz, h111_yz);
  const T M020_0 = ((fma(T(9), h030_0, fma(T(4), h020_0, h010_0))) + (fma(T(4), h220_0, fma(T(4), h022_0, h111_0))));
  const T M101_0 = fma(T(4), h202_xz, h111_xz);
  const T M110_0 = fma(T(4), h220_xy, h111_xy);
  const T M200_0 = ((fma(T(4), h220_0, fma(T(4), h200_0, h100_0))) + (fma(T(9), h300_0, fma(T(4), h202_0, h111_0))));
  const T M001_1 = ((fma(T(16), h202_z, fma(T(16), h022_z, fma(T(8), h002_z, h001_z)))) + (fma(T(3), h111_z, mul_rn(T(27), h003_z))));
  const T M010_1 = ((fma(T(16), h220_y, fma(T(27), h030_y, fma(T(8), h020_y, h010_y)))) + (fma(T(3), h111_y, mul_rn(T(16), h022_y))));
  const T M100_1 = ((fma(T(27), h300_x, fma(T(16), h202_x, fma(T(3), h111_x, h100_x)))) + (fma(T(16), h220_x, mul_rn(T(8), h200_x))));
  s[0] = M000_0;
  s[1] = M100_0;
  s[2] = M010_0;
  s[3] = M001_0;
  s[4] = M200_0;
  s[5] = M020_0;
  s[6] = M002_0;
  s[7] = M110_0;
  s[8] = M101_0;
  s[9] = M011_0;
  s[10] = M100_1;
  s[11] = M010_1;
  s[12] = M001_1;
}

// z-mirror-symmetric F: s and J of the nine z-even basis functions (ZEVEN order).
template <class T, class A>
__device__ __forceinline__ void moments2d(const A& F, T (&s)[9], T (&J)[45]) {
  const T h000_0 = F[0];
  const T w1_0_0 = F[5] + F[6];
  const T w1_0_1 = F[5] - F[6];
  const T h001_0 = w1_0_0;
  const T h001_z = w1_0_1;
  const T w2_0_0 = F[19] + F[20];
  const T w2_0_1 = F[19] - F[20];
  const T h002_0 = w2_0_0;
  const T h002_z = w2_0_1;
  const T w3_0_0 = F[37] + F[38];
  const T w3_0_1 = F[37] - F[38];
  const T h003_0 = w3_0_0;
  const T h003_z = w3_0_1;
  const T w4_0_0 = F[3] + F[4];
  const T w4_0_1 = F[3] - F[4];
  const T h010_0 = w4_0_0;
  const T h010_y = w4_0_1;
  const T w5_0_0 = F[17] + F[18];
  const T w5_0_1 = F[17] - F[18];
  const T h020_0 = w5_0_0;
  const T h020_y = w5_0_1;
  const T w6_0_0 = F[29] + F[32];
  const T w6_0_1 = F[29] - F[32];
  const T w6_0_2 = F[31] + F[30];
  const T w6_0_3 = F[31] - F[30];
  const T w6_1_0 = w6_0_0 + w6_0_2;
  const T w6_1_1 = w6_0_0 - w6_0_2;
  const T w6_1_2 = w6_0_1 + w6_0_3;
  const T w6_1_3 = w6_0_1 - w6_0_3;
  const T h022_0 = w6_1_0;
  const T h022_z = w6_1_1;
  const T h022_y = w6_1_2;
  const T h022_yz = w6_1_3;
  const T w7_0_0 = F[35] + F[36];
  const T w7_0_1 = F[35] - F[36];
  const T h030_0 = w7_0_0;
  const T h030_y = w7_0_1;
  const T w8_0_0 = F[1] + F[2];
  const T w8_0_1 = F[1] - F[2];
  const T h100_0 = w8_0_0;
  const T h100_x = w8_0_1;
  const T w9_0_0 = F[7] + F[13];
  const T w9_0_1 = F[7] - F[13];
  const T w9_0_2 = F[9] + F[12];
  const T w9_0_3 = F[9] - F[12];
  const T w9_0_4 = F[11] + F[10];
  const T w9_0_5 = F[11] - F[10];
  const T w9_0_6 = F[14] + F[8];
  const T w9_0_7 = F[14] - F[8];
  const T w9_1_0 = w9_0_0 + w9_0_4;
  const T w9_1_1 = w9_0_0 - w9_0_4;
  const T w9_1_2 = w9_0_1 + w9_0_5;
  const T w9_1_3 = w9_0_1 - w9_0_5;
  const T w9_1_4 = w9_0_2 + w9_0_6;
  const T w9_1_5 = w9_0_2 - w9_0_6;
  const T w9_1_6 = w9_0_3 + w9_0_7;
  const T w9_1_7 = w9_0_3 - w9_0_7;
  const T w9_2_0 = w9_1_0 + w9_1_4;
  const T w9_2_1 = w9_1_0 - w9_1_4;
  const T w9_2_2 = w9_1_1 + w9_1_5;
  const T w9_2_3 = w9_1_1 - w9_1_5;
  const T w9_2_4 = w9_1_2 + w9_1_6;
  const T w9_2_5 = w9_1_2 - w9_1_6;
  const T w9_2_6 = w9_1_3 + w9_1_7;
  const T w9_2_7 = w9_1_3 - w9_1_7;
  const T h111_0 = w9_2_0;
  const T h111_z = w9_2_1;
  const T h111_y = w9_2_2;
  const T h111_yz = w9_2_3;
  const T h111_x = w9_2_4;
  const T h111_xz = w9_2_5;
  const T h111_xy = w9_2_6;
  const T h111_xyz = w9_2_7;
  const T w10_0_0 = F[15] + F[16];
  const T w10_0_1 = F[15] - F[16];
  const T h200_0 = w10_0_0;
  const T h200_x = w10_0_1;
  const T w11_0_0 = F[25] + F[28];
  const T w11_0_1 = F[25] - F[28];
  const T w11_0_2 = F[27] + F[26];
  const T w11_0_3 = F[27] - F[26];
  const T w11_1_0 = w11_0_0 + w11_0_2;
  const T w11_1_1 = w11_0_0 - w11_0_2;
  const T w11_1_2 = w11_0_1 + w11_0_3;
  const T w11_1_3 = w11_0_1 - w11_0_3;
  const T h202_0 = w11_1_0;
  const T h202_z = w11_1_1;
  const T h202_x = w11_1_2;
  const T h202_xz = w11_1_3;
  const T w12_0_0 = F[21] + F[24];
  const T w12_0_1 = F[21] - F[24];
  const T w12_0_2 = F[23] + F[22];
  const T w12_0_3 = F[23] - F[22];
  const T w12_1_0 = w12_0_0 + w12_0_2;
  const T w12_1_1 = w12_0_0 - w12_0_2;
  const T w12_1_2 = w12_0_1 + w12_0_3;
  const T w12_1_3 = w12_0_1 - w12_0_3;
  const T h220_0 = w12_1_0;
  const T h220_y = w12_1_1;
  const T h220_x = w12_1_2;
  const T h220_xy = w12_1_3;
  const T w13_0_0 = F[33] + F[34];
  const T w13_0_1 = F[33] - F[34];
  const T h300_0 = w13_0_0;
  const T h300_x = w13_0_1;
  const T M000_0 = (((h000_0 + h010_0 + h100_0 + h220_0) + (h001_0 + h020_0 + h111_0 + h300_0)) + ((h002_0 + h022_0 + h200_0) + (h003_0 + h030_0 + h202_0)));
  const T M010_0 = ((fma(T(3), h030_y, fma(T(2), h020_y, h010_y))) + (fma(T(2), h220_y, fma(T(2), h022_y, h111_y))));
  const T M100_0 = ((fma(T(2), h220_x, fma(T(2), h200_x, h100_x))) + (fma(T(3), h300_x, fma(T(2), h202_x, h111_x))));
  const T M002_0 = ((fma(T(4), h022_0, fma(T(4), h002_0, h001_0))) + (fma(T(4), h202_0, fma(T(9), h003_0, h111_0))));
  const T M020_0 = ((fma(T(9), h030_0, fma(T(4), h020_0, h010_0))) + (fma(T(4), h220_0, fma(T(4), h022_0, h111_0))));
  const T M110_0 = fma(T(4), h220_xy, h111_xy);
  const T M200_0 = ((fma(T(4), h220_0, fma(T(4), h200_0, h100_0))) + (fma(T(9), h300_0, fma(T(4), h202_0, h111_0))));
  const T M012_0 = fma(T(8), h022_y, h111_y);
  const T M030_0 = ((fma(T(27), h030_y, fma(T(8), h020_y, h010_y))) + (fma(T(8), h220_y, fma(T(8), h022_y, h111_y))));
  const T M102_0 = fma(T(8), h202_x, h111_x);
  const T M120_0 = fma(T(8), h220_x, h111_x);
  const T M210_0 = fma(T(8), h220_y, h111_y);
  const T M300_0 = ((fma(T(8), h220_x, fma(T(8), h200_x, h100_x))) + (fma(T(27), h300_x, fma(T(8), h202_x, h111_x))));
  const T M004_0 = ((fma(T(16), h022_0, fma(T(16), h002_0, h001_0))) + (fma(T(16), h202_0, fma(T(81), h003_0, h111_0))));
  const T M022_0 = fma(T(16), h022_0, h111_0);
  const T M040_0 = ((fma(T(81), h030_0, fma(T(16), h020_0, h010_0))) + (fma(T(16), h220_0, fma(T(16), h022_0, h111_0))));
  const T M112_0 = h111_xy;
  const T M130_0 = fma(T(16), h220_xy, h111_xy);
  const T M202_0 = fma(T(16), h202_0, h111_0);
  const T M220_0 = fma(T(16), h220_0, h111_0);
  const T M310_0 = fma(T(16), h220_xy, h111_xy);
  const T M400_0 = ((fma(T(16), h220_0, fma(T(16), h200_0, h100_0))) + (fma(T(81), h300_0, fma(T(16), h202_0, h111_0))));
  const T M010_1 = ((fma(T(16), h220_y, fma(T(27), h030_y, fma(T(8), h020_y, h010_y)))) + (fma(T(3), h111_y, mul_rn(T(16), h022_y))));
  const T M100_1 = ((fma(T(27), h300_x, fma(T(16), h202_x, fma(T(3), h111_x, h100_x)))) + (fma(T(16), h220_x, mul_rn(T(8), h200_x))));
  const T M020_1 = ((fma(T(32), h220_0, fma(T(81), h030_0, fma(T(16), h020_0, h010_0)))) + (fma(T(3), h111_0, mul_rn(T(32), h022_0))));
  const T M110_1 = fma(T(32), h220_xy, mul_rn(T(3), h111_xy));
  const T M200_1 = ((fma(T(81), h300_0, fma(T(32), h202_0, fma(T(3), h111_0, h100_0)))) + (fma(T(32), h220_0, mul_rn(T(16), h200_0))));
  const T M012_1 = fma(T(3), h111_y, mul_rn(T(64), h022_y));
  const T M030_1 = ((fma(T(64), h220_y, fma(T(243), h030_y, fma(T(32), h020_y, h010_y)))) + (fma(T(3), h111_y, mul_rn(T(64), h022_y))));
  const T M102_1 = fma(T(64), h202_x, mul_rn(T(3), h111_x));
  const T M120_1 = fma(T(64), h220_x, mul_rn(T(3), h111_x));
  const T M210_1 = fma(T(64), h220_y, mul_rn(T(3), h111_y));
  const T M300_1 = ((fma(T(243), h300_x, fma(T(64), h202_x, fma(T(3), h111_x, h100_x)))) + (fma(T(64), h220_x, mul_rn(T(32), h200_x))));
  const T M020_2 = ((fma(T(256), h220_0, fma(T(729), h030_0, fma(T(64), h020_0, h010_0)))) + (fma(T(9), h111_0, mul_rn(T(256), h022_0))));
  const T M110_2 = fma(T(256), h220_xy, mul_rn(T(9), h111_xy));
  const T M200_2 = ((fma(T(729), h300_0, fma(T(256), h202_0, fma(T(9), h111_0, h100_0)))) + (fma(T(256), h220_0, mul_rn(T(64), h200_0))));
  s[0] = M000_0;
  s[1] = M100_0;
  s[2] = M010_0;
  s[3] = M200_0;
  s[4] = M020_0;
  s[5] = M002_0;
  s[6] = M110_0;
  s[7] = M100_1;
  s[8] = M010_1;
  J[0] = M000_0;
  J[1] = M100_0;
  J[2] = M200_0;
  J[3] = M010_0;
  J[4] = M110_0;
  J[5] = M020_0;
  J[6] = M200_0;
  J[7] = M300_0;
  J[8] = M210_0;
  J[9] = M400_0;
  J[10] = M020_0;
  J[11] = M120_0;
  J[12] = M030_0;
  J[13] = M220_0;
  J[14] = M040_0;
  J[15] = M002_0;
  J[16] = M102_0;
  J[17] = M012_0;
  J[18] = M202_0;
  J[19] = M022_0;
  J[20] = M004_0;
  J[21] = M110_0;
  J[22] = M210_0;
  J[23] = M120_0;
  J[24] = M310_0;
  J[25] = M130_0;
  J[26] = M112_0;
  J[27] = M220_0;
  J[28] = M100_1;
  J[29] = M200_1;
  J[30] = M110_1;
  J[31] = M300_1;
  J[32] = M120_1;
  J[33] = M102_1;
  J[34] = M210_1;
  J[35] = M200_2;
  J[36] = M010_1;
  J[37] = M110_1;
  J[38] = M020_1;
  J[39] = M210_1;
  J[40] = M030_1;
  J[41] = M012_1;
  J[42] = M120_1;
  J[43] = M110_2;
  J[44] = M020_2;
}

template <class T, class A>
__device__ __forceinline__ void moments_s2d(const A& F, T (&s)[9]) {
  const T h000_0 = F[0];
  const T w1_0_0 = F[5] + F[6];
  const T w1_0_1 = F[5] - F[6];
  const T h001_0 = w1_0_0;
  const T h001_z = w1_0_1;
  const T w2_0_0 = F[19] + F[20];
  const T w2_0_1 = F[19] - F[20];
  const T h002_0 = w2_0_0;
  const T h002_z = w2_0_1;
  const T w3_0_0 = F[37] + F[38];
  const T w3_0_1 = F[37] - F[38];
  const T h003_0 = w3_0_0;
  const T h003_z = w3_0_1;
  const T w4_0_0 = F[3] + F[4];
  const T w4_0_1 = F[3] - F[4];
  const T h010_0 = w4_0_0;
  const T h010_y = w4_0_1;
  const T w5_0_0 = F[17] + F[18];
  const T w5_0_1 = F[17] - F[18];
  const T h020_0 = w5_0_0;
  const T h020_y = w5_0_1;
  const T w6_0_0 = F[29] + F[32];
  const T w6_0_1 = F[29] - F[32];
  const T w6_0_2 = F[31] + F[30];
  const T w6_0_3 = F[31] - F[30];
  const T w6_1_0 = w6_0_0 + w6_0_2;
  const T w6_1_1 = w6_0_0 - w6_0_2;
  const T w6_1_2 = w6_0_1 + w6_0_3;
  const T w6_1_3 = w6_0_1 - w6_0_3;
  const T h022_0 = w6_1_0;
  const T h022_z = w6_1_1;
  const T h022_y = w6_1_2;
  const T h022_yz = w6_1_3;
  const T w7_0_0 = F[35] + F[36];
  const T w7_0_1 = F[35] - F[36];
  const T h030_0 = w7_0_0;
  const T h030_y = w7_0_1;
  const T w8_0_0 = F[1] + F[2];
  const T w8_0_1 = F[1] - F[2];
  const T h100_0 = w8_0_0;
  const T h100_x = w8_0_1;
  const T w9_0_0 = F[7] + F[13];
  const T w9_0_1 = F[7] - F[13];
  const T w9_0_2 = F[9] + F[12];
  const T w9_0_3 = F[9] - F[12];
  const T w9_0_4 = F[11] + F[10];
  const T w9_0_5 = F[11] - F[10];
  const T w9_0_6 = F[14] + F[8];
  const T w9_0_7 = F[14] - F[8];
  const T w9_1_0 = w9_0_0 + w9_0_4;
  const T w9_1_1 = w9_0_0 - w9_0_4;
  const T w9_1_2 = w9_0_1 + w9_0_5;
  const T w9_1_3 = w9_0_1 - w9_0_5;
  const T w9_1_4 = w9_0_2 + w9_0_6;
  const T w9_1_5 = w9_0_2 - w9_0_6;
  const T w9_1_6 = w9_0_3 + w9_0_7;
  const T w9_1_7 = w9_0_3 - w9_0_7;
  const T w9_2_0 = w9_1_0 + w9_1_4;
  const T w9_2_1 = w9_1_0 - w9_1_4;
  const T w9_2_2 = w9_1_1 + w9_1_5;
  const T w9_2_3 = w9_1_1 - w9_1_5;
  const T w9_2_4 = w9_1_2 + w9_1_6;
  const T w9_2_5 = w9_1_2 - w9_1_6;
  const T w9_2_6 = w9_1_3 + w9_1_7;
  const T w9_2_7 = w9_1_3 - w9_1_7;
  const T h111_0 = w9_2_0;
  const T h111_z = w9_2_1;
  const T h111_y = w9_2_2;
  const T h111_yz = w9_2_3;
  const T h111_x = w9_2_4;
  const T h111_xz = w9_2_5;
  const T h111_xy = w9_2_6;
  const T h111_xyz = w9_2_7;
  const T w10_0_0 = F[15] + F[16];
  const T w10_0_1 = F[15] - F[16];
  const T h200_0 = w10_0_0;
  const T h200_x = w10_0_1;
  const T w11_0_0 = F[25] + F[28];
  const T w11_0_1 = F[25] - F[28];
  const T w11_0_2 = F[27] + F[26];
  const T w11_0_3 = F[27] - F[26];
  const T w11_1_0 = w11_0_0 + w11_0_2;
  const T w11_1_1 = w11_0_0 - w11_0_2;
  const T w11_1_2 = w11_0_1 + w11_0_3;
  const T w11_1_3 = w11_0_1 - w11_0_3;
  const T h202_0 = w11_1_0;
  const T h202_z = w11_1_1;
  const T h202_x = w11_1_2;
  const T h202_xz = w11_1_3;
  const T w12_0_0 = F[21] + F[24];
  const T w12_0_1 = F[21] - F[24];
  const T w12_0_2 = F[23] + F[22];
  const T w12_0_3 = F[23] - F[22];
  const T w12_1_0 = w12_0_0 + w12_0_2;
  const T w12_1_1 = w12_0_0 - w12_0_2;
  const T w12_1_2 = w12_0_1 + w12_0_3;
  const T w12_1_3 = w12_0_1 - w12_0_3;
  const T h220_0 = w12_1_0;
  const T h220_y = w12_1_1;
  const T h220_x = w12_1_2;
  const T h220_xy = w12_1_3;
  const T w13_0_0 = F[33] + F[34];
  const T w13_0_1 = F[33] - F[34];
  const T h300_0 = w13_0_0;
  const T h300_x = w13_0_1;
  const T M000_0 = (((h000_0 + h010_0 + h100_0 + h220_0) + (h001_0 + h020_0 + h111_0 + h300_0)) + ((h002_0 + h022_0 + h200_0) + (h003_0 + h030_0 + h202_0)));
  const T M010_0 = ((fma(T(3), h030_y, fma(T(2), h020_y, h010_y))) + (fma(T(2), h220_y, fma(T(2), h022_y, h111_y))));
  const T M100_0 = ((fma(T(2), h220_x, fma(T(2), h200_x, h100_x))) + (fma(T(3), h300_x, fma(T(2), h202_x, h111_x))));
  const T M002_0 = ((fma(T(4), h022_0, fma(T(4), h002_0, h001_0))) + (fma(T(4), h202_0, fma(T(9), h003_0, h111_0))));
  const T M020_0 = ((fma(T(9), h030_0, fma(T(4), h020_0, h010_0))) + (fma(T(4), h220_0, fma(T(4), h022_0, h111_0))));
  const T M110_0 = fma(T(4), h220_xy, h111_xy);
  const T M200_0 = ((fma(T(4), h220_0, fma(T(4), h200_0, h100_0))) + (fma(T(9), h300_0, fma(T(4), h202_0, h111_0))));
  const T M010_1 = ((fma(T(16), h220_y, fma(T(27), h030_y, fma(T(8), h020_y, h010_y)))) + (fma(T(3), h111_y, mul_rn(T(16), h022_y))));
  const T M100_1 = ((fma(T(27), h300_x, fma(T(16), h202_x, fma(T(3), h111_x, h100_x)))) + (fma(T(16), h220_x, mul_rn(T(8), h200_x))));
  s[0] = M000_0;
  s[1] = M100_0;
  s[2] = M010_0;
  s[3] = M200_0;
  s[4] = M020_0;
  s[5] = M002_0;
  s[6] = M110_0;
  s[7] = M100_1;
  s[8] = M010_1;
}

// rho = sum f, j = sum f xi, e2f = sum f |xi|^2 (Sec. 3, macroscopic step).
template <class T, class A>
__device__ __forceinline__ void f_moments(const A& f, T& rho, T& jx, T& jy, T& jz,
                                          T& e2f) {
  const T ps1 = f[1] + f[2], pd1 = f[1] - f[2];
  const T ps3 = f[3] + f[4], pd3 = f[3] - f[4];
  const T ps5 = f[5] + f[6], pd5 = f[5] - f[6];
  const T ps7 = f[7] + f[8], pd7 = f[7] - f[8];
  const T ps9 = f[9] + f[10], pd9 = f[9] - f[10];
  const T ps11 = f[11] + f[12], pd11 = f[11] - f[12];
  const T ps13 = f[13] + f[14], pd13 = f[13] - f[14];
  const T ps15 = f[15] + f[16], pd15 = f[15] - f[16];
  const T ps17 = f[17] + f[18], pd17 = f[17] - f[18];
  const T ps19 = f[19] + f[20], pd19 = f[19] - f[20];
  const T ps21 = f[21] + f[22], pd21 = f[21] - f[22];
  const T ps23 = f[23] + f[24], pd23 = f[23] - f[24];
  const T ps25 = f[25] + f[26], pd25 = f[25] - f[26];
  const T ps27 = f[27] + f[28], pd27 = f[27] - f[28];
  const T ps29 = f[29] + f[30], pd29 = f[29] - f[30];
  const T ps31 = f[31] + f[32], pd31 = f[31] - f[32];
  const T ps33 = f[33] + f[34], pd33 = f[33] - f[34];
  const T ps35 = f[35] + f[36], pd35 = f[35] - f[36];
  const T ps37 = f[37] + f[38], pd37 = f[37] - f[38];
  rho = f[0] + (((((ps1 + ps3) + ps5) + (ps7 + ps9)) + (((ps11 + ps13) + ps15) + (ps17 + ps19))) + ((((ps21 + ps23) + ps25) + (ps27 + ps29)) + ((ps31 + ps33) + (ps35 + ps37))));
  jx = (((fma(T(2), pd25, pd1 - pd13)) + (fma(T(2), pd27, fma(T(2), pd15, pd7)))) + ((fma(T(3), pd33, fma(T(2), pd21, pd9))) + (fma(T(2), pd23, pd11))));
  jy = (((fma(T(2), pd29, pd3 - pd11)) + (fma(T(2), pd31, fma(T(2), pd17, pd7)))) + ((fma(T(3), pd35, fma(T(2), pd21, pd9))) + (fma(T(-2), pd23, pd13))));
  jz = (((fma(T(2), pd29, pd5 - pd9)) + (fma(T(-2), pd31, fma(T(2), pd19, pd7)))) + ((fma(T(3), pd37, fma(T(2), pd25, pd11))) + (fma(T(-2), pd27, pd13))));
  const T sh1 = ((ps1 + ps3) + ps5);
  const T sh3 = ((ps7 + ps9) + (ps11 + ps13));
  const T sh4 = ((ps15 + ps17) + ps19);
  const T sh8 = (((ps21 + ps23) + ps25) + ((ps27 + ps29) + ps31));
  const T sh9 = ((ps33 + ps35) + ps37);
  e2f = ((fma(T(8), sh8, fma(T(3), sh3, sh1))) + (fma(T(9), sh9, mul_rn(T(4), sh4))));
}

// sum g (the second population's share of the total energy).
template <class T, class A>
__device__ __forceinline__ T g_sum(const A& g) {
  const T gs = ((((((g[0] + g[1]) + g[2]) + (g[3] + g[4])) + (((g[5] + g[6]) + g[7]) + (g[8] + g[9]))) + ((((g[10] + g[11]) + g[12]) + (g[13] + g[14])) + (((g[15] + g[16]) + g[17]) + (g[18] + g[19])))) + (((((g[20] + g[21]) + g[22]) + (g[23] + g[24])) + (((g[25] + g[26]) + g[27]) + (g[28] + g[29]))) + ((((g[30] + g[31]) + g[32]) + (g[33] + g[34])) + ((g[35] + g[36]) + (g[37] + g[38])))));
  return gs;
}

// exp(x) = 2^(k/256) exp(r), x = k ln2/256 + r (table-driven method of P. T. P. Tang,
// ACM TOMS 15(2), 1989, with a 256-entry table): 256/ln2, ln2/256 = head + tail.
constexpr double EXP_INV_L = 369.3299304675746;
constexpr double EXP_L_HI = 0.0027076061742263846;
constexpr double EXP_L_LO = -1.6409824502660487e-13;
// 2^(j/256), j = 0..255, each the double nearest the exact value.
__device__ const double kExp2Table[256] = {
    1.0, 1.0027112750502025, 1.0054299011128027, 1.0081558981184175,
    1.0108892860517005, 1.0136300849514894, 1.016378314910953, 1.019133996077738,
    1.0218971486541166, 1.0246677928971357, 1.0274459491187637, 1.030231637686041,
    1.0330248790212284, 1.0358256936019572, 1.0386341019613787, 1.041450124688316,
    1.0442737824274138, 1.0471050958792898, 1.0499440858006872, 1.0527907730046264,
    1.0556451783605572, 1.0585073227945128, 1.061377227289262, 1.0642549128844645,
    1.0671404006768237, 1.0700337118202419, 1.0729348675259756, 1.075843889062791,
    1.0787607977571199, 1.0816856149932152, 1.0846183622133092, 1.0875590609177697,
    1.0905077326652577, 1.0934643990728858, 1.0964290818163769, 1.099401802630222,
    1.102382583307841, 1.1053714457017412, 1.1083684117236787, 1.1113735033448175,
    1.1143867425958924, 1.1174081515673693, 1.1204377524096067, 1.12347556733302,
    1.1265216186082418, 1.129575928566288, 1.1326385195987192, 1.1357094141578055,
    1.1387886347566916, 1.1418762039695616, 1.1449721444318042, 1.148076478840179,
    1.1511892299529827, 1.154310420590216, 1.1574400736337511, 1.1605782120274988,
    1.1637248587775775, 1.1668800369524817, 1.1700437696832502, 1.1732160801636373,
    1.1763969916502812, 1.1795865274628758, 1.182784710984341, 1.1859915656609938,
    1.189207115002721, 1.1924313825831512, 1.1956643920398273, 1.1989061670743806,
    1.202156731452703, 1.2054161090051239, 1.2086843236265816, 1.2119613992768012,
    1.215247359980469, 1.2185422298274085, 1.2218460329727576, 1.2251587936371455,
    1.22848053610687, 1.2318112847340759, 1.2351510639369334, 1.2384998981998165,
    1.241857812073484, 1.245224830175258, 1.2486009771892048, 1.2519862778663162,
    1.255380757024691, 1.2587844395497165, 1.2621973503942507, 1.2656195145788063,
    1.2690509571917332, 1.2724917033894028, 1.275941778396392, 1.2794012075056693,
    1.2828700160787783, 1.2863482295460256, 1.2898358734066657, 1.2933329732290895,
    1.2968395546510096, 1.3003556433796506, 1.3038812651919358, 1.3074164459346773,
    1.3109612115247644, 1.3145155879493546, 1.318079601266064, 1.3216532776031575,
    1.3252366431597413, 1.3288297242059544, 1.3324325470831615, 1.3360451382041458,
    1.339667524053303, 1.3432997311868353, 1.3469417862329458, 1.3505937158920345,
    1.3542555469368927, 1.3579273062129011, 1.3616090206382248, 1.365300717204012,
    1.3690024229745905, 1.3727141650876684, 1.3764359707545302, 1.380167867260238,
    1.383909881963832, 1.387662042298529, 1.3914243757719262, 1.3951969099662003,
    1.3989796725383112, 1.4027726912202048, 1.4065759938190154, 1.4103896082172707,
    1.4142135623730951, 1.4180478843204152, 1.4218926021691656, 1.4257477441054942,
    1.42961333839197, 1.433489413367789, 1.4373759974489824, 1.4412731191286257,
    1.4451808069770467, 1.449099089642035, 1.4530279958490526, 1.4569675544014438,
    1.460917794180647, 1.4648787441464057, 1.4688504333369818, 1.4728328908693675,
    1.4768261459394993, 1.4808302278224719, 1.4848451658727524, 1.488870989524397,
    1.4929077282912648, 1.4969554117672355, 1.5010140696264256, 1.5050837316234065,
    1.5091644275934228, 1.5132561874526098, 1.5173590411982147, 1.5214730189088146,
    1.5255981507445384, 1.529734466947287, 1.533881997840956, 1.5380407738316568,
    1.5422108254079407, 1.5463921831410214, 1.550584877685, 1.5547889397770887,
    1.559004400237837, 1.5632312899713576, 1.567469639965553, 1.5717194812923414,
    1.5759808451078865, 1.5802537626528246, 1.5845382652524937, 1.588834384317164,
    1.593142151342267, 1.597461597908627, 1.6017927556826934, 1.606135656416771,
    1.6104903319492543, 1.6148568142048607, 1.6192351351948637, 1.6236253270173289,
    1.6280274218573478, 1.632441451987275, 1.6368674497669644, 1.6413054476440063,
    1.645755478153965, 1.6502175739206177, 1.6546917676561943, 1.6591780921616162,
    1.6636765803267364, 1.6681872651305825, 1.6727101796415966, 1.6772453570178785,
    1.681792830507429, 1.6863526334483934, 1.6909247992693053, 1.6955093614893326,
    1.7001063537185235, 1.7047158096580513, 1.709337763100463, 1.713972247929926,
    1.718619298122478, 1.723278947746274, 1.7279512309618377, 1.732636182022311,
    1.7373338352737062, 1.7420442251551564, 1.746767386199169, 1.7515033530318782,
    1.7562521603732995, 1.761013843037584, 1.7657884359332727, 1.7705759740635547,
    1.7753764925265212, 1.7801900265154245, 1.785016611318935, 1.789856282321401,
    1.7947090750031072, 1.7995750249405351, 1.804454167806624, 1.809346539371032,
    1.8142521755003989, 1.8191711121586085, 1.8241033854070534, 1.8290490314048973,
    1.8340080864093424, 1.8389805867758937, 1.843966568958626, 1.8489660695104508,
    1.8539791250833855, 1.8590057724288205, 1.864046048397789, 1.8690999899412386,
    1.8741676341103, 1.8792490180565602, 1.8843441790323345, 1.8894531543909392,
    1.8945759815869656, 1.8997126981765553, 1.9048633418176741, 1.9100279502703899,
    1.9152065613971474, 1.9203992131630474, 1.925605943636125, 1.930826790987627,
    1.9360617934922943, 1.9413109895286405, 1.9465744175792332, 1.9518521162309783,
    1.9571441241754002, 1.9624504802089273, 1.9677712232331759, 1.9731063922552343,
    1.978456026387951, 1.9838201648502194, 1.9891988469672663, 1.9945921121709402,
};

// A velocity index as a type.
template <int I>
struct Idx {
  static constexpr int value = I;
};

// s_k = sum_i v(i) phi_k(xi_i) in 64-bit integers.
template <class V>
__device__ __forceinline__ void sums_fx(const V& v, unsigned long long (&s)[13]) {
  const unsigned long long v0 = v(Idx<0>{});
  s[0] = v0;
  const unsigned long long v5 = v(Idx<5>{});
  const unsigned long long v6 = v(Idx<6>{});
  const unsigned long long w1_0_0 = v5 + v6;
  const unsigned long long w1_0_1 = v5 - v6;
  s[0] += w1_0_0;
  s[6] = w1_0_0;
  s[3] = w1_0_1;
  s[12] = w1_0_1;
  const unsigned long long v19 = v(Idx<19>{});
  const unsigned long long v20 = v(Idx<20>{});
  const unsigned long long w2_0_0 = v19 + v20;
  const unsigned long long w2_0_1 = v19 - v20;
  s[0] += w2_0_0;
  s[6] += 4ull * w2_0_0;
  s[3] += 2ull * w2_0_1;
  s[12] += 8ull * w2_0_1;
  const unsigned long long v37 = v(Idx<37>{});
  const unsigned long long v38 = v(Idx<38>{});
  const unsigned long long w3_0_0 = v37 + v38;
  const unsigned long long w3_0_1 = v37 - v38;
  s[0] += w3_0_0;
  s[6] += 9ull * w3_0_0;
  s[3] += 3ull * w3_0_1;
  s[12] += 27ull * w3_0_1;
  const unsigned long long v3 = v(Idx<3>{});
  const unsigned long long v4 = v(Idx<4>{});
  const unsigned long long w4_0_0 = v3 + v4;
  const unsigned long long w4_0_1 = v3 - v4;
  s[0] += w4_0_0;
  s[5] = w4_0_0;
  s[2] = w4_0_1;
  s[11] = w4_0_1;
  const unsigned long long v17 = v(Idx<17>{});
  const unsigned long long v18 = v(Idx<18>{});
  const unsigned long long w5_0_0 = v17 + v18;
  const unsigned long long w5_0_1 = v17 - v18;
  s[0] += w5_0_0;
  s[5] += 4ull * w5_0_0;
  s[2] += 2ull * w5_0_1;
  s[11] += 8ull * w5_0_1;
  const unsigned long long v29 = v(Idx<29>{});
  const unsigned long long v30 = v(Idx<30>{});
  const unsigned long long v31 = v(Idx<31>{});
  const unsigned long long v32 = v(Idx<32>{});
  const unsigned long long w6_0_0 = v31 + v30;
  const unsigned long long w6_0_1 = v31 - v30;
  const unsigned long long w6_0_2 = v29 + v32;
  const unsigned long long w6_0_3 = v29 - v32;
  const unsigned long long w6_1_0 = w6_0_2 + w6_0_0;
  const unsigned long long w6_1_1 = w6_0_2 - w6_0_0;
  const unsigned long long w6_1_2 = w6_0_3 + w6_0_1;
  const unsigned long long w6_1_3 = w6_0_3 - w6_0_1;
  s[0] += w6_1_0;
  s[5] += 4ull * w6_1_0;
  s[6] += 4ull * w6_1_0;
  s[3] += 2ull * w6_1_1;
  s[12] += 16ull * w6_1_1;
  s[2] += 2ull * w6_1_2;
  s[11] += 16ull * w6_1_2;
  s[9] = 4ull * w6_1_3;
  const unsigned long long v35 = v(Idx<35>{});
  const unsigned long long v36 = v(Idx<36>{});
  const unsigned long long w7_0_0 = v35 + v36;
  const unsigned long long w7_0_1 = v35 - v36;
  s[0] += w7_0_0;
  s[5] += 9ull * w7_0_0;
  s[2] += 3ull * w7_0_1;
  s[11] += 27ull * w7_0_1;
  const unsigned long long v1 = v(Idx<1>{});
  const unsigned long long v2 = v(Idx<2>{});
  const unsigned long long w8_0_0 = v1 + v2;
  const unsigned long long w8_0_1 = v1 - v2;
  s[0] += w8_0_0;
  s[4] = w8_0_0;
  s[1] = w8_0_1;
  s[10] = w8_0_1;
  const unsigned long long v7 = v(Idx<7>{});
  const unsigned long long v8 = v(Idx<8>{});
  const unsigned long long v9 = v(Idx<9>{});
  const unsigned long long v10 = v(Idx<10>{});
  const unsigned long long v11 = v(Idx<11>{});
  const unsigned long long v12 = v(Idx<12>{});
  const unsigned long long v13 = v(Idx<13>{});
  const unsigned long long v14 = v(Idx<14>{});
  const unsigned long long w9_0_0 = v14 + v8;
  const unsigned long long w9_0_1 = v14 - v8;
  const unsigned long long w9_0_2 = v11 + v10;
  const unsigned long long w9_0_3 = v11 - v10;
  const unsigned long long w9_0_4 = v9 + v12;
  const unsigned long long w9_0_5 = v9 - v12;
  const unsigned long long w9_0_6 = v7 + v13;
  const unsigned long long w9_0_7 = v7 - v13;
  const unsigned long long w9_1_0 = w9_0_4 + w9_0_0;
  const unsigned long long w9_1_1 = w9_0_4 - w9_0_0;
  const unsigned long long w9_1_2 = w9_0_6 + w9_0_2;
  const unsigned long long w9_1_3 = w9_0_6 - w9_0_2;
  const unsigned long long w9_1_4 = w9_0_5 + w9_0_1;
  const unsigned long long w9_1_5 = w9_0_5 - w9_0_1;
  const unsigned long long w9_1_6 = w9_0_7 + w9_0_3;
  const unsigned long long w9_1_7 = w9_0_7 - w9_0_3;
  const unsigned long long w9_2_0 = w9_1_2 + w9_1_0;
  const unsigned long long w9_2_1 = w9_1_2 - w9_1_0;
  const unsigned long long w9_2_2 = w9_1_3 + w9_1_1;
  const unsigned long long w9_2_3 = w9_1_3 - w9_1_1;
  const unsigned long long w9_2_4 = w9_1_6 + w9_1_4;
  const unsigned long long w9_2_5 = w9_1_6 - w9_1_4;
  const unsigned long long w9_2_6 = w9_1_7 + w9_1_5;
  const unsigned long long w9_2_7 = w9_1_7 - w9_1_5;
  s[0] += w9_2_0;
  s[4] += w9_2_0;
  s[5] += w9_2_0;
  s[6] += w9_2_0;
  s[3] += w9_2_1;
  s[12] += 3ull * w9_2_1;
  s[2] += w9_2_2;
  s[11] += 3ull * w9_2_2;
  s[9] += w9_2_3;
  s[1] += w9_2_4;
  s[10] += 3ull * w9_2_4;
  s[8] = w9_2_5;
  s[7] = w9_2_6;
  const unsigned long long v15 = v(Idx<15>{});
  const unsigned long long v16 = v(Idx<16>{});
  const unsigned long long w10_0_0 = v15 + v16;
  const unsigned long long w10_0_1 = v15 - v16;
  s[0] += w10_0_0;
  s[4] += 4ull * w10_0_0;
  s[1] += 2ull * w10_0_1;
  s[10] += 8ull * w10_0_1;
  const unsigned long long v25 = v(Idx<25>{});
  const unsigned long long v26 = v(Idx<26>{});
  const unsigned long long v27 = v(Idx<27>{});
  const unsigned long long v28 = v(Idx<28>{});
  const unsigned long long w11_0_0 = v27 + v26;
  const unsigned long long w11_0_1 = v27 - v26;
  const unsigned long long w11_0_2 = v25 + v28;
  const unsigned long long w11_0_3 = v25 - v28;
  const unsigned long long w11_1_0 = w11_0_2 + w11_0_0;
  const unsigned long long w11_1_1 = w11_0_2 - w11_0_0;
  const unsigned long long w11_1_2 = w11_0_3 + w11_0_1;
  const unsigned long long w11_1_3 = w11_0_3 - w11_0_1;
  s[0] += w11_1_0;
  s[4] += 4ull * w11_1_0;
  s[6] += 4ull * w11_1_0;
  s[3] += 2ull * w11_1_1;
  s[12] += 16ull * w11_1_1;
  s[1] += 2ull * w11_1_2;
  s[10] += 16ull * w11_1_2;
  s[8] += 4ull * w11_1_3;
  const unsigned long long v21 = v(Idx<21>{});
  const unsigned long long v22 = v(Idx<22>{});
  const unsigned long long v23 = v(Idx<23>{});
  const unsigned long long v24 = v(Idx<24>{});
  const unsigned long long w12_0_0 = v23 + v22;
  const unsigned long long w12_0_1 = v23 - v22;
  const unsigned long long w12_0_2 = v21 + v24;
  const unsigned long long w12_0_3 = v21 - v24;
  const unsigned long long w12_1_0 = w12_0_2 + w12_0_0;
  const unsigned long long w12_1_1 = w12_0_2 - w12_0_0;
  const unsigned long long w12_1_2 = w12_0_3 + w12_0_1;
  const unsigned long long w12_1_3 = w12_0_3 - w12_0_1;
  s[0] += w12_1_0;
  s[4] += 4ull * w12_1_0;
  s[5] += 4ull * w12_1_0;
  s[2] += 2ull * w12_1_1;
  s[11] += 16ull * w12_1_1;
  s[1] += 2ull * w12_1_2;
  s[10] += 16ull * w12_1_2;
  s[7] += 4ull * w12_1_3;
  const unsigned long long v33 = v(Idx<33>{});
  const unsigned long long v34 = v(Idx<34>{});
  const unsigned long long w13_0_0 = v33 + v34;
  const unsigned long long w13_0_1 = v33 - v34;
  s[0] += w13_0_0;
  s[4] += 9ull * w13_0_0;
  s[1] += 3ull * w13_0_1;
  s[10] += 27ull * w13_0_1;
}

// s_k = sum_i p(i, y_i) phi_k(xi_i) in 64-bit integers.
template <class V>
__device__ __forceinline__ void jvec_fx(const int (&d)[13], const V& p, unsigned long long (&s)[13]) {
  const int c0_0 = d[0];
  const unsigned long long p0 = p(Idx<0>{}, c0_0);
  s[0] = p0;
  const int c1_0 = d[0] + d[6];
  const int c1_z = d[3] + d[12];
  const int y1_0_0 = c1_0 + c1_z;
  const int y1_0_1 = c1_0 - c1_z;
  const unsigned long long p5 = p(Idx<5>{}, y1_0_0);
  const unsigned long long p6 = p(Idx<6>{}, y1_0_1);
  const unsigned long long w1_0_0 = p5 + p6;
  const unsigned long long w1_0_1 = p5 - p6;
  s[0] += w1_0_0;
  s[6] = w1_0_0;
  s[3] = w1_0_1;
  s[12] = w1_0_1;
  const int c2_0 = d[0] + 4 * d[6];
  const int c2_z = 2 * d[3] + 8 * d[12];
  const int y2_0_0 = c2_0 + c2_z;
  const int y2_0_1 = c2_0 - c2_z;
  const unsigned long long p19 = p(Idx<19>{}, y2_0_0);
  const unsigned long long p20 = p(Idx<20>{}, y2_0_1);
  const unsigned long long w2_0_0 = p19 + p20;
  const unsigned long long w2_0_1 = p19 - p20;
  s[0] += w2_0_0;
  s[6] += 4ull * w2_0_0;
  s[3] += 2ull * w2_0_1;
  s[12] += 8ull * w2_0_1;
  const int c3_0 = d[0] + 9 * d[6];
  const int c3_z = 3 * d[3] + 27 * d[12];
  const int y3_0_0 = c3_0 + c3_z;
  const int y3_0_1 = c3_0 - c3_z;
  const unsigned long long p37 = p(Idx<37>{}, y3_0_0);
  const unsigned long long p38 = p(Idx<38>{}, y3_0_1);
  const unsigned long long w3_0_0 = p37 + p38;
  const unsigned long long w3_0_1 = p37 - p38;
  s[0] += w3_0_0;
  s[6] += 9ull * w3_0_0;
  s[3] += 3ull * w3_0_1;
  s[12] += 27ull * w3_0_1;
  const int c4_0 = d[0] + d[5];
  const int c4_y = d[2] + d[11];
  const int y4_0_0 = c4_0 + c4_y;
  const int y4_0_1 = c4_0 - c4_y;
  const unsigned long long p3 = p(Idx<3>{}, y4_0_0);
  const unsigned long long p4 = p(Idx<4>{}, y4_0_1);
  const unsigned long long w4_0_0 = p3 + p4;
  const unsigned long long w4_0_1 = p3 - p4;
  s[0] += w4_0_0;
  s[5] = w4_0_0;
  s[2] = w4_0_1;
  s[11] = w4_0_1;
  const int c5_0 = d[0] + 4 * d[5];
  const int c5_y = 2 * d[2] + 8 * d[11];
  const int y5_0_0 = c5_0 + c5_y;
  const int y5_0_1 = c5_0 - c5_y;
  const unsigned long long p17 = p(Idx<17>{}, y5_0_0);
  const unsigned long long p18 = p(Idx<18>{}, y5_0_1);
  const unsigned long long w5_0_0 = p17 + p18;
  const unsigned long long w5_0_1 = p17 - p18;
  s[0] += w5_0_0;
  s[5] += 4ull * w5_0_0;
  s[2] += 2ull * w5_0_1;
  s[11] += 8ull * w5_0_1;
  const int c6_0 = d[0] + 4 * d[5] + 4 * d[6];
  const int c6_y = 2 * d[2] + 16 * d[11];
  const int c6_z = 2 * d[3] + 16 * d[12];
  const int c6_yz = 4 * d[9];
  const int y6_0_0 = c6_0 + c6_y;
  const int y6_0_1 = c6_0 - c6_y;
  const int y6_0_2 = c6_z + c6_yz;
  const int y6_0_3 = c6_z - c6_yz;
  const int y6_1_0 = y6_0_1 + y6_0_3;
  const int y6_1_1 = y6_0_1 - y6_0_3;
  const int y6_1_2 = y6_0_0 + y6_0_2;
  const int y6_1_3 = y6_0_0 - y6_0_2;
  const unsigned long long p29 = p(Idx<29>{}, y6_1_2);
  const unsigned long long p30 = p(Idx<30>{}, y6_1_1);
  const unsigned long long p31 = p(Idx<31>{}, y6_1_3);
  const unsigned long long p32 = p(Idx<32>{}, y6_1_0);
  const unsigned long long w6_0_0 = p31 + p30;
  const unsigned long long w6_0_1 = p31 - p30;
  const unsigned long long w6_0_2 = p29 + p32;
  const unsigned long long w6_0_3 = p29 - p32;
  const unsigned long long w6_1_0 = w6_0_2 + w6_0_0;
  const unsigned long long w6_1_1 = w6_0_2 - w6_0_0;
  const unsigned long long w6_1_2 = w6_0_3 + w6_0_1;
  const unsigned long long w6_1_3 = w6_0_3 - w6_0_1;
  s[0] += w6_1_0;
  s[5] += 4ull * w6_1_0;
  s[6] += 4ull * w6_1_0;
  s[3] += 2ull * w6_1_1;
  s[12] += 16ull * w6_1_1;
  s[2] += 2ull * w6_1_2;
  s[11] += 16ull * w6_1_2;
  s[9] = 4ull * w6_1_3;
  const int c7_0 = d[0] + 9 * d[5];
  const int c7_y = 3 * d[2] + 27 * d[11];
  const int y7_0_0 = c7_0 + c7_y;
  const int y7_0_1 = c7_0 - c7_y;
  const unsigned long long p35 = p(Idx<35>{}, y7_0_0);
  const unsigned long long p36 = p(Idx<36>{}, y7_0_1);
  const unsigned long long w7_0_0 = p35 + p36;
  const unsigned long long w7_0_1 = p35 - p36;
  s[0] += w7_0_0;
  s[5] += 9ull * w7_0_0;
  s[2] += 3ull * w7_0_1;
  s[11] += 27ull * w7_0_1;
  const int c8_0 = d[0] + d[4];
  const int c8_x = d[1] + d[10];
  const int y8_0_0 = c8_0 + c8_x;
  const int y8_0_1 = c8_0 - c8_x;
  const unsigned long long p1 = p(Idx<1>{}, y8_0_0);
  const unsigned long long p2 = p(Idx<2>{}, y8_0_1);
  const unsigned long long w8_0_0 = p1 + p2;
  const unsigned long long w8_0_1 = p1 - p2;
  s[0] += w8_0_0;
  s[4] = w8_0_0;
  s[1] = w8_0_1;
  s[10] = w8_0_1;
  const int c9_0 = d[0] + d[4] + d[5] + d[6];
  const int c9_x = d[1] + 3 * d[10];
  const int c9_y = d[2] + 3 * d[11];
  const int c9_z = d[3] + 3 * d[12];
  const int c9_xy = d[7];
  const int c9_xz = d[8];
  const int c9_yz = d[9];
  const int y9_0_0 = c9_0 + c9_x;
  const int y9_0_1 = c9_0 - c9_x;
  const int y9_0_2 = c9_y + c9_xy;
  const int y9_0_3 = c9_y - c9_xy;
  const int y9_0_6 = c9_z + c9_xz;
  const int y9_0_7 = c9_z - c9_xz;
  const int y9_1_0 = y9_0_1 + y9_0_3;
  const int y9_1_1 = y9_0_1 - y9_0_3;
  const int y9_1_2 = y9_0_7 + c9_yz;
  const int y9_1_3 = y9_0_7 - c9_yz;
  const int y9_1_4 = y9_0_0 + y9_0_2;
  const int y9_1_5 = y9_0_0 - y9_0_2;
  const int y9_1_6 = y9_0_6 + c9_yz;
  const int y9_1_7 = y9_0_6 - c9_yz;
  const int y9_2_0 = y9_1_1 + y9_1_3;
  const int y9_2_1 = y9_1_1 - y9_1_3;
  const int y9_2_2 = y9_1_0 + y9_1_2;
  const int y9_2_3 = y9_1_0 - y9_1_2;
  const int y9_2_4 = y9_1_5 + y9_1_7;
  const int y9_2_5 = y9_1_5 - y9_1_7;
  const int y9_2_6 = y9_1_4 + y9_1_6;
  const int y9_2_7 = y9_1_4 - y9_1_6;
  const unsigned long long p7 = p(Idx<7>{}, y9_2_6);
  const unsigned long long p8 = p(Idx<8>{}, y9_2_1);
  const unsigned long long p9 = p(Idx<9>{}, y9_2_7);
  const unsigned long long p10 = p(Idx<10>{}, y9_2_0);
  const unsigned long long p11 = p(Idx<11>{}, y9_2_4);
  const unsigned long long p12 = p(Idx<12>{}, y9_2_3);
  const unsigned long long p13 = p(Idx<13>{}, y9_2_2);
  const unsigned long long p14 = p(Idx<14>{}, y9_2_5);
  const unsigned long long w9_0_0 = p14 + p8;
  const unsigned long long w9_0_1 = p14 - p8;
  const unsigned long long w9_0_2 = p11 + p10;
  const unsigned long long w9_0_3 = p11 - p10;
  const unsigned long long w9_0_4 = p9 + p12;
  const unsigned long long w9_0_5 = p9 - p12;
  const unsigned long long w9_0_6 = p7 + p13;
  const unsigned long long w9_0_7 = p7 - p13;
  const unsigned long long w9_1_0 = w9_0_4 + w9_0_0;
  const unsigned long long w9_1_1 = w9_0_4 - w9_0_0;
  const unsigned long long w9_1_2 = w9_0_6 + w9_0_2;
  const unsigned long long w9_1_3 = w9_0_6 - w9_0_2;
  const unsigned long long w9_1_4 = w9_0_5 + w9_0_1;
  const unsigned long long w9_1_5 = w9_0_5 - w9_0_1;
  const unsigned long long w9_1_6 = w9_0_7 + w9_0_3;
  const unsigned long long w9_1_7 = w9_0_7 - w9_0_3;
  const unsigned long long w9_2_0 = w9_1_2 + w9_1_0;
  const unsigned long long w9_2_1 = w9_1_2 - w9_1_0;
  const unsigned long long w9_2_2 = w9_1_3 + w9_1_1;
  const unsigned long long w9_2_3 = w9_1_3 - w9_1_1;
  const unsigned long long w9_2_4 = w9_1_6 + w9_1_4;
  const unsigned long long w9_2_5 = w9_1_6 - w9_1_4;
  const unsigned long long w9_2_6 = w9_1_7 + w9_1_5;
  const unsigned long long w9_2_7 = w9_1_7 - w9_1_5;
  s[0] += w9_2_0;
  s[4] += w9_2_0;
  s[5] += w9_2_0;
  s[6] += w9_2_0;
  s[3] += w9_2_1;
  s[12] += 3ull * w9_2_1;
  s[2] += w9_2_2;
  s[11] += 3ull * w9_2_2;
  s[9] += w9_2_3;
  s[1] += w9_2_4;
  s[10] += 3ull * w9_2_4;
  s[8] = w9_2_5;
  s[7] = w9_2_6;
  const int c10_0 = d[0] + 4 * d[4];
  const int c10_x = 2 * d[1] + 8 * d[10];
  const int y10_0_0 = c10_0 + c10_x;
  const int y10_0_1 = c10_0 - c10_x;
  const unsigned long long p15 = p(Idx<15>{}, y10_0_0);
  const unsigned long long p16 = p(Idx<16>{}, y10_0_1);
  const unsigned long long w10_0_0 = p15 + p16;
  const unsigned long long w10_0_1 = p15 - p16;
  s[0] += w10_0_0;
  s[4] += 4ull * w10_0_0;
  s[1] += 2ull * w10_0_1;
  s[10] += 8ull * w10_0_1;
  const int c11_0 = d[0] + 4 * d[4] + 4 * d[6];
  const int c11_x = 2 * d[1] + 16 * d[10];
  const int c11_z = 2 * d[3] + 16 * d[12];
  const int c11_xz = 4 * d[8];
  const int y11_0_0 = c11_0 + c11_x;
  const int y11_0_1 = c11_0 - c11_x;
  const int y11_0_2 = c11_z + c11_xz;
  const int y11_0_3 = c11_z - c11_xz;
  const int y11_1_0 = y11_0_1 + y11_0_3;
  const int y11_1_1 = y11_0_1 - y11_0_3;
  const int y11_1_2 = y11_0_0 + y11_0_2;
  const int y11_1_3 = y11_0_0 - y11_0_2;
  const unsigned long long p25 = p(Idx<25>{}, y11_1_2);
  const unsigned long long p26 = p(Idx<26>{}, y11_1_1);
  const unsigned long long p27 = p(Idx<27>{}, y11_1_3);
  const unsigned long long p28 = p(Idx<28>{}, y11_1_0);
  const unsigned long long w11_0_0 = p27 + p26;
  const unsigned long long w11_0_1 = p27 - p26;
  const unsigned long long w11_0_2 = p25 + p28;
  const unsigned long long w11_0_3 = p25 - p28;
  const unsigned long long w11_1_0 = w11_0_2 + w11_0_0;
  const unsigned long long w11_1_1 = w11_0_2 - w11_0_0;
  const unsigned long long w11_1_2 = w11_0_3 + w11_0_1;
  const unsigned long long w11_1_3 = w11_0_3 - w11_0_1;
  s[0] += w11_1_0;
  s[4] += 4ull * w11_1_0;
  s[6] += 4ull * w11_1_0;
  s[3] += 2ull * w11_1_1;
  s[12] += 16ull * w11_1_1;
  s[1] += 2ull * w11_1_2;
  s[10] += 16ull * w11_1_2;
  s[8] += 4ull * w11_1_3;
  const int c12_0 = d[0] + 4 * d[4] + 4 * d[5];
  const int c12_x = 2 * d[1] + 16 * d[10];
  const int c12_y = 2 * d[2] + 16 * d[11];
  const int c12_xy = 4 * d[7];
  const int y12_0_0 = c12_0 + c12_x;
  const int y12_0_1 = c12_0 - c12_x;
  const int y12_0_2 = c12_y + c12_xy;
  const int y12_0_3 = c12_y - c12_xy;
  const int y12_1_0 = y12_0_1 + y12_0_3;
  const int y12_1_1 = y12_0_1 - y12_0_3;
  const int y12_1_2 = y12_0_0 + y12_0_2;
  const int y12_1_3 = y12_0_0 - y12_0_2;
  const unsigned long long p21 = p(Idx<21>{}, y12_1_2);
  const unsigned long long p22 = p(Idx<22>{}, y12_1_1);
  const unsigned long long p23 = p(Idx<23>{}, y12_1_3);
  const unsigned long long p24 = p(Idx<24>{}, y12_1_0);
  const unsigned long long w12_0_0 = p23 + p22;
  const unsigned long long w12_0_1 = p23 - p22;
  const unsigned long long w12_0_2 = p21 + p24;
  const unsigned long long w12_0_3 = p21 - p24;
  const unsigned long long w12_1_0 = w12_0_2 + w12_0_0;
  const unsigned long long w12_1_1 = w12_0_2 - w12_0_0;
  const unsigned long long w12_1_2 = w12_0_3 + w12_0_1;
  const unsigned long long w12_1_3 = w12_0_3 - w12_0_1;
  s[0] += w12_1_0;
  s[4] += 4ull * w12_1_0;
  s[5] += 4ull * w12_1_0;
  s[2] += 2ull * w12_1_1;
  s[11] += 16ull * w12_1_1;
  s[1] += 2ull * w12_1_2;
  s[10] += 16ull * w12_1_2;
  s[7] += 4ull * w12_1_3;
  const int c13_0 = d[0] + 9 * d[4];
  const int c13_x = 3 * d[1] + 27 * d[10];
  const int y13_0_0 = c13_0 + c13_x;
  const int y13_0_1 = c13_0 - c13_x;
  const unsigned long long p33 = p(Idx<33>{}, y13_0_0);
  const unsigned long long p34 = p(Idx<34>{}, y13_0_1);
  const unsigned long long w13_0_0 = p33 + p34;
  const unsigned long long w13_0_1 = p33 - p34;
  s[0] += w13_0_0;
  s[4] += 9ull * w13_0_0;
  s[1] += 3ull * w13_0_1;
  s[10] += 27ull * w13_0_1;
}

// sum_i v(i) [1, xi_i, |xi_i|^2] in 64-bit integers.
template <class V>
__device__ __forceinline__ void macro_fx(const V& v, unsigned long long (&s)[5]) {
  const unsigned long long v0 = v(Idx<0>{});
  s[0] = v0;
  const unsigned long long v5 = v(Idx<5>{});
  const unsigned long long v6 = v(Idx<6>{});
  const unsigned long long w1_0_0 = v5 + v6;
  const unsigned long long w1_0_1 = v5 - v6;
  s[0] += w1_0_0;
  s[4] = w1_0_0;
  s[3] = w1_0_1;
  const unsigned long long v19 = v(Idx<19>{});
  const unsigned long long v20 = v(Idx<20>{});
  const unsigned long long w2_0_0 = v19 + v20;
  const unsigned long long w2_0_1 = v19 - v20;
  s[0] += w2_0_0;
  s[4] += 4ull * w2_0_0;
  s[3] += 2ull * w2_0_1;
  const unsigned long long v37 = v(Idx<37>{});
  const unsigned long long v38 = v(Idx<38>{});
  const unsigned long long w3_0_0 = v37 + v38;
  const unsigned long long w3_0_1 = v37 - v38;
  s[0] += w3_0_0;
  s[4] += 9ull * w3_0_0;
  s[3] += 3ull * w3_0_1;
  const unsigned long long v3 = v(Idx<3>{});
  const unsigned long long v4 = v(Idx<4>{});
  const unsigned long long w4_0_0 = v3 + v4;
  const unsigned long long w4_0_1 = v3 - v4;
  s[0] += w4_0_0;
  s[4] += w4_0_0;
  s[2] = w4_0_1;
  const unsigned long long v17 = v(Idx<17>{});
  const unsigned long long v18 = v(Idx<18>{});
  const unsigned long long w5_0_0 = v17 + v18;
  const unsigned long long w5_0_1 = v17 - v18;
  s[0] += w5_0_0;
  s[4] += 4ull * w5_0_0;
  s[2] += 2ull * w5_0_1;
  const unsigned long long v29 = v(Idx<29>{});
  const unsigned long long v30 = v(Idx<30>{});
  const unsigned long long v31 = v(Idx<31>{});
  const unsigned long long v32 = v(Idx<32>{});
  const unsigned long long w6_0_0 = v31 + v30;
  const unsigned long long w6_0_1 = v31 - v30;
  const unsigned long long w6_0_2 = v29 + v32;
  const unsigned long long w6_0_3 = v29 - v32;
  const unsigned long long w6_1_0 = w6_0_2 + w6_0_0;
  const unsigned long long w6_1_1 = w6_0_2 - w6_0_0;
  const unsigned long long w6_1_2 = w6_0_3 + w6_0_1;
  const unsigned long long w6_1_3 = w6_0_3 - w6_0_1;
  s[0] += w6_1_0;
  s[4] += 8ull * w6_1_0;
  s[3] += 2ull * w6_1_1;
  s[2] += 2ull * w6_1_2;
  const unsigned long long v35 = v(Idx<35>{});
  const unsigned long long v36 = v(Idx<36>{});
  const unsigned long long w7_0_0 = v35 + v36;
  const unsigned long long w7_0_1 = v35 - v36;
  s[0] += w7_0_0;
  s[4] += 9ull * w7_0_0;
  s[2] += 3ull * w7_0_1;
  const unsigned long long v1 = v(Idx<1>{});
  const unsigned long long v2 = v(Idx<2>{});
  const unsigned long long w8_0_0 = v1 + v2;
  const unsigned long long w8_0_1 = v1 - v2;
  s[0] += w8_0_0;
  s[4] += w8_0_0;
  s[1] = w8_0_1;
  const unsigned long long v7 = v(Idx<7>{});
  const unsigned long long v8 = v(Idx<8>{});
  const unsigned long long v9 = v(Idx<9>{});
  const unsigned long long v10 = v(Idx<10>{});
  const unsigned long long v11 = v(Idx<11>{});
  const unsigned long long v12 = v(Idx<12>{});
  const unsigned long long v13 = v(Idx<13>{});
  const unsigned long long v14 = v(Idx<14>{});
  const unsigned long long w9_0_0 = v14 + v8;
  const unsigned long long w9_0_1 = v14 - v8;
  const unsigned long long w9_0_2 = v11 + v10;
  const unsigned long long w9_0_3 = v11 - v10;
  const unsigned long long w9_0_4 = v9 + v12;
  const unsigned long long w9_0_5 = v9 - v12;
  const unsigned long long w9_0_6 = v7 + v13;
  const unsigned long long w9_0_7 = v7 - v13;
  const unsigned long long w9_1_0 = w9_0_4 + w9_0_0;
  const unsigned long long w9_1_1 = w9_0_4 - w9_0_0;
  const unsigned long long w9_1_2 = w9_0_6 + w9_0_2;
  const unsigned long long w9_1_3 = w9_0_6 - w9_0_2;
  const unsigned long long w9_1_4 = w9_0_5 + w9_0_1;
  const unsigned long long w9_1_5 = w9_0_5 - w9_0_1;
  const unsigned long long w9_1_6 = w9_0_7 + w9_0_3;
  const unsigned long long w9_1_7 = w9_0_7 - w9_0_3;
  const unsigned long long w9_2_0 = w9_1_2 + w9_1_0;
  const unsigned long long w9_2_1 = w9_1_2 - w9_1_0;
  const unsigned long long w9_2_2 = w9_1_3 + w9_1_1;
  const unsigned long long w9_2_3 = w9_1_3 - w9_1_1;
  const unsigned long long w9_2_4 = w9_1_6 + w9_1_4;
  const unsigned long long w9_2_5 = w9_1_6 - w9_1_4;
  const unsigned long long w9_2_6 = w9_1_7 + w9_1_5;
  const unsigned long long w9_2_7 = w9_1_7 - w9_1_5;
  s[0] += w9_2_0;
  s[4] += 3ull * w9_2_0;
  s[3] += w9_2_1;
  s[2] += w9_2_2;
  s[1] += w9_2_4;
  const unsigned long long v15 = v(Idx<15>{});
  const unsigned long long v16 = v(Idx<16>{});
  const unsigned long long w10_0_0 = v15 + v16;
  const unsigned long long w10_0_1 = v15 - v16;
  s[0] += w10_0_0;
  s[4] += 4ull * w10_0_0;
  s[1] += 2ull * w10_0_1;
  const unsigned long long v25 = v(Idx<25>{});
  const unsigned long long v26 = v(Idx<26>{});
  const unsigned long long v27 = v(Idx<27>{});
  const unsigned long long v28 = v(Idx<28>{});
  const unsigned long long w11_0_0 = v27 + v26;
  const unsigned long long w11_0_1 = v27 - v26;
  const unsigned long long w11_0_2 = v25 + v28;
  const unsigned long long w11_0_3 = v25 - v28;
  const unsigned long long w11_1_0 = w11_0_2 + w11_0_0;
  const unsigned long long w11_1_1 = w11_0_2 - w11_0_0;
  const unsigned long long w11_1_2 = w11_0_3 + w11_0_1;
  const unsigned long long w11_1_3 = w11_0_3 - w11_0_1;
  s[0] += w11_1_0;
  s[4] += 8ull * w11_1_0;
  s[3] += 2ull * w11_1_1;
  s[1] += 2ull * w11_1_2;
  const unsigned long long v21 = v(Idx<21>{});
  const unsigned long long v22 = v(Idx<22>{});
  const unsigned long long v23 = v(Idx<23>{});
  const unsigned long long v24 = v(Idx<24>{});
  const unsigned long long w12_0_0 = v23 + v22;
  const unsigned long long w12_0_1 = v23 - v22;
  const unsigned long long w12_0_2 = v21 + v24;
  const unsigned long long w12_0_3 = v21 - v24;
  const unsigned long long w12_1_0 = w12_0_2 + w12_0_0;
  const unsigned long long w12_1_1 = w12_0_2 - w12_0_0;
  const unsigned long long w12_1_2 = w12_0_3 + w12_0_1;
  const unsigned long long w12_1_3 = w12_0_3 - w12_0_1;
  s[0] += w12_1_0;
  s[4] += 8ull * w12_1_0;
  s[2] += 2ull * w12_1_1;
  s[1] += 2ull * w12_1_2;
  const unsigned long long v33 = v(Idx<33>{});
  const unsigned long long v34 = v(Idx<34>{});
  const unsigned long long w13_0_0 = v33 + v34;
  const unsigned long long w13_0_1 = v33 - v34;
  s[0] += w13_0_0;
  s[4] += 9ull * w13_0_0;
  s[1] += 3ull * w13_0_1;
}

// s_k = sum_i v(i) phi_k(xi_i) in 64-bit integers (the nine z-even k, values mirror-symmetric in z).
template <class V>
__device__ __forceinline__ void sums_fx2d(const V& v, unsigned long long (&s)[9]) {
  const unsigned long long v0 = v(Idx<0>{});
  s[0] = v0;
  const unsigned long long v5 = v(Idx<5>{});
  s[0] += 2ull * v5;
  s[5] = 2ull * v5;
  const unsigned long long v19 = v(Idx<19>{});
  s[0] += 2ull * v19;
  s[5] += 8ull * v19;
  const unsigned long long v37 = v(Idx<37>{});
  s[0] += 2ull * v37;
  s[5] += 18ull * v37;
  const unsigned long long v3 = v(Idx<3>{});
  const unsigned long long v4 = v(Idx<4>{});
  const unsigned long long w4_0_0 = v3 + v4;
  const unsigned long long w4_0_1 = v3 - v4;
  s[0] += w4_0_0;
  s[4] = w4_0_0;
  s[2] = w4_0_1;
  s[8] = w4_0_1;
  const unsigned long long v17 = v(Idx<17>{});
  const unsigned long long v18 = v(Idx<18>{});
  const unsigned long long w5_0_0 = v17 + v18;
  const unsigned long long w5_0_1 = v17 - v18;
  s[0] += w5_0_0;
  s[4] += 4ull * w5_0_0;
  s[2] += 2ull * w5_0_1;
  s[8] += 8ull * w5_0_1;
  const unsigned long long v29 = v(Idx<29>{});
  const unsigned long long v30 = v(Idx<30>{});
  const unsigned long long w6_0_0 = v29 + v30;
  const unsigned long long w6_0_1 = v29 - v30;
  s[0] += 2ull * w6_0_0;
  s[4] += 8ull * w6_0_0;
  s[5] += 8ull * w6_0_0;
  s[2] += 4ull * w6_0_1;
  s[8] += 32ull * w6_0_1;
  const unsigned long long v35 = v(Idx<35>{});
  const unsigned long long v36 = v(Idx<36>{});
  const unsigned long long w7_0_0 = v35 + v36;
  const unsigned long long w7_0_1 = v35 - v36;
  s[0] += w7_0_0;
  s[4] += 9ull * w7_0_0;
  s[2] += 3ull * w7_0_1;
  s[8] += 27ull * w7_0_1;
  const unsigned long long v1 = v(Idx<1>{});
  const unsigned long long v2 = v(Idx<2>{});
  const unsigned long long w8_0_0 = v1 + v2;
  const unsigned long long w8_0_1 = v1 - v2;
  s[0] += w8_0_0;
  s[3] = w8_0_0;
  s[1] = w8_0_1;
  s[7] = w8_0_1;
  const unsigned long long v7 = v(Idx<7>{});
  const unsigned long long v8 = v(Idx<8>{});
  const unsigned long long v11 = v(Idx<11>{});
  const unsigned long long v12 = v(Idx<12>{});
  const unsigned long long w9_0_0 = v11 + v8;
  const unsigned long long w9_0_1 = v11 - v8;
  const unsigned long long w9_0_2 = v7 + v12;
  const unsigned long long w9_0_3 = v7 - v12;
  const unsigned long long w9_1_0 = w9_0_2 + w9_0_0;
  const unsigned long long w9_1_1 = w9_0_2 - w9_0_0;
  const unsigned long long w9_1_2 = w9_0_3 + w9_0_1;
  const unsigned long long w9_1_3 = w9_0_3 - w9_0_1;
  s[0] += 2ull * w9_1_0;
  s[3] += 2ull * w9_1_0;
  s[4] += 2ull * w9_1_0;
  s[5] += 2ull * w9_1_0;
  s[2] += 2ull * w9_1_1;
  s[8] += 6ull * w9_1_1;
  s[1] += 2ull * w9_1_2;
  s[7] += 6ull * w9_1_2;
  s[6] = 2ull * w9_1_3;
  const unsigned long long v15 = v(Idx<15>{});
  const unsigned long long v16 = v(Idx<16>{});
  const unsigned long long w10_0_0 = v15 + v16;
  const unsigned long long w10_0_1 = v15 - v16;
  s[0] += w10_0_0;
  s[3] += 4ull * w10_0_0;
  s[1] += 2ull * w10_0_1;
  s[7] += 8ull * w10_0_1;
  const unsigned long long v25 = v(Idx<25>{});
  const unsigned long long v26 = v(Idx<26>{});
  const unsigned long long w11_0_0 = v25 + v26;
  const unsigned long long w11_0_1 = v25 - v26;
  s[0] += 2ull * w11_0_0;
  s[3] += 8ull * w11_0_0;
  s[5] += 8ull * w11_0_0;
  s[1] += 4ull * w11_0_1;
  s[7] += 32ull * w11_0_1;
  const unsigned long long v21 = v(Idx<21>{});
  const unsigned long long v22 = v(Idx<22>{});
  const unsigned long long v23 = v(Idx<23>{});
  const unsigned long long v24 = v(Idx<24>{});
  const unsigned long long w12_0_0 = v23 + v22;
  const unsigned long long w12_0_1 = v23 - v22;
  const unsigned long long w12_0_2 = v21 + v24;
  const unsigned long long w12_0_3 = v21 - v24;
  const unsigned long long w12_1_0 = w12_0_2 + w12_0_0;
  const unsigned long long w12_1_1 = w12_0_2 - w12_0_0;
  const unsigned long long w12_1_2 = w12_0_3 + w12_0_1;
  const unsigned long long w12_1_3 = w12_0_3 - w12_0_1;
  s[0] += w12_1_0;
  s[3] += 4ull * w12_1_0;
  s[4] += 4ull * w12_1_0;
  s[2] += 2ull * w12_1_1;
  s[8] += 16ull * w12_1_1;
  s[1] += 2ull * w12_1_2;
  s[7] += 16ull * w12_1_2;
  s[6] += 4ull * w12_1_3;
  const unsigned long long v33 = v(Idx<33>{});
  const unsigned long long v34 = v(Idx<34>{});
  const unsigned long long w13_0_0 = v33 + v34;
  const unsigned long long w13_0_1 = v33 - v34;
  s[0] += w13_0_0;
  s[3] += 9ull * w13_0_0;
  s[1] += 3ull * w13_0_1;
  s[7] += 27ull * w13_0_1;
}

// s_k = sum_i p(i, y_i) phi_k(xi_i) in 64-bit integers (the nine z-even k, values mirror-symmetric in z).
template <class V>
__device__ __forceinline__ void jvec_fx2d(const int (&d)[9], const V& p, unsigned long long (&s)[9]) {
  const int c0_0 = d[0];
  const unsigned long long p0 = p(Idx<0>{}, c0_0);
  s[0] = p0;
  const int c1_0 = d[0] + d[5];
  const unsigned long long p5 = p(Idx<5>{}, c1_0);
  s[0] += 2ull * p5;
  s[5] = 2ull * p5;
  const int c2_0 = d[0] + 4 * d[5];
  const unsigned long long p19 = p(Idx<19>{}, c2_0);
  s[0] += 2ull * p19;
  s[5] += 8ull * p19;
  const int c3_0 = d[0] + 9 * d[5];
  const unsigned long long p37 = p(Idx<37>{}, c3_0);
  s[0] += 2ull * p37;
  s[5] += 18ull * p37;
  const int c4_0 = d[0] + d[4];
  const int c4_y = d[2] + d[8];
  const int y4_0_0 = c4_0 + c4_y;
  const int y4_0_1 = c4_0 - c4_y;
  const unsigned long long p3 = p(Idx<3>{}, y4_0_0);
  const unsigned long long p4 = p(Idx<4>{}, y4_0_1);
  const unsigned long long w4_0_0 = p3 + p4;
  const unsigned long long w4_0_1 = p3 - p4;
  s[0] += w4_0_0;
  s[4] = w4_0_0;
  s[2] = w4_0_1;
  s[8] = w4_0_1;
  const int c5_0 = d[0] + 4 * d[4];
  const int c5_y = 2 * d[2] + 8 * d[8];
  const int y5_0_0 = c5_0 + c5_y;
  const int y5_0_1 = c5_0 - c5_y;
  const unsigned long long p17 = p(Idx<17>{}, y5_0_0);
  const unsigned long long p18 = p(Idx<18>{}, y5_0_1);
  const unsigned long long w5_0_0 = p17 + p18;
  const unsigned long long w5_0_1 = p17 - p18;
  s[0] += w5_0_0;
  s[4] += 4ull * w5_0_0;
  s[2] += 2ull * w5_0_1;
  s[8] += 8ull * w5_0_1;
  const int c6_0 = d[0] + 4 * d[4] + 4 * d[5];
  const int c6_y = 2 * d[2] + 16 * d[8];
  const int y6_0_0 = c6_0 + c6_y;
  const int y6_0_1 = c6_0 - c6_y;
  const unsigned long long p29 = p(Idx<29>{}, y6_0_0);
  const unsigned long long p30 = p(Idx<30>{}, y6_0_1);
  const unsigned long long w6_0_0 = p29 + p30;
  const unsigned long long w6_0_1 = p29 - p30;
  s[0] += 2ull * w6_0_0;
  s[4] += 8ull * w6_0_0;
  s[5] += 8ull * w6_0_0;
  s[2] += 4ull * w6_0_1;
  s[8] += 32ull * w6_0_1;
  const int c7_0 = d[0] + 9 * d[4];
  const int c7_y = 3 * d[2] + 27 * d[8];
  const int y7_0_0 = c7_0 + c7_y;
  const int y7_0_1 = c7_0 - c7_y;
  const unsigned long long p35 = p(Idx<35>{}, y7_0_0);
  const unsigned long long p36 = p(Idx<36>{}, y7_0_1);
  const unsigned long long w7_0_0 = p35 + p36;
  const unsigned long long w7_0_1 = p35 - p36;
  s[0] += w7_0_0;
  s[4] += 9ull * w7_0_0;
  s[2] += 3ull * w7_0_1;
  s[8] += 27ull * w7_0_1;
  const int c8_0 = d[0] + d[3];
  const int c8_x = d[1] + d[7];
  const int y8_0_0 = c8_0 + c8_x;
  const int y8_0_1 = c8_0 - c8_x;
  const unsigned long long p1 = p(Idx<1>{}, y8_0_0);
  const unsigned long long p2 = p(Idx<2>{}, y8_0_1);
  const unsigned long long w8_0_0 = p1 + p2;
  const unsigned long long w8_0_1 = p1 - p2;
  s[0] += w8_0_0;
  s[3] = w8_0_0;
  s[1] = w8_0_1;
  s[7] = w8_0_1;
  const int c9_0 = d[0] + d[3] + d[4] + d[5];
  const int c9_x = d[1] + 3 * d[7];
  const int c9_y = d[2] + 3 * d[8];
  const int c9_xy = d[6];
  const int y9_0_0 = c9_0 + c9_x;
  const int y9_0_1 = c9_0 - c9_x;
  const int y9_0_2 = c9_y + c9_xy;
  const int y9_0_3 = c9_y - c9_xy;
  const int y9_1_0 = y9_0_1 + y9_0_3;
  const int y9_1_1 = y9_0_1 - y9_0_3;
  const int y9_1_2 = y9_0_0 + y9_0_2;
  const int y9_1_3 = y9_0_0 - y9_0_2;
  const unsigned long long p7 = p(Idx<7>{}, y9_1_2);
  const unsigned long long p8 = p(Idx<8>{}, y9_1_1);
  const unsigned long long p11 = p(Idx<11>{}, y9_1_3);
  const unsigned long long p12 = p(Idx<12>{}, y9_1_0);
  const unsigned long long w9_0_0 = p11 + p8;
  const unsigned long long w9_0_1 = p11 - p8;
  const unsigned long long w9_0_2 = p7 + p12;
  const unsigned long long w9_0_3 = p7 - p12;
  const unsigned long long w9_1_0 = w9_0_2 + w9_0_0;
  const unsigned long long w9_1_1 = w9_0_2 - w9_0_0;
  const unsigned long long w9_1_2 = w9_0_3 + w9_0_1;
  const unsigned long long w9_1_3 = w9_0_3 - w9_0_1;
  s[0] += 2ull * w9_1_0;
  s[3] += 2ull * w9_1_0;
  s[4] += 2ull * w9_1_0;
  s[5] += 2ull * w9_1_0;
  s[2] += 2ull * w9_1_1;
  s[8] += 6ull * w9_1_1;
  s[1] += 2ull * w9_1_2;
  s[7] += 6ull * w9_1_2;
  s[6] = 2ull * w9_1_3;
  const int c10_0 = d[0] + 4 * d[3];
  const int c10_x = 2 * d[1] + 8 * d[7];
  const int y10_0_0 = c10_0 + c10_x;
  const int y10_0_1 = c10_0 - c10_x;
  const unsigned long long p15 = p(Idx<15>{}, y10_0_0);
  const unsigned long long p16 = p(Idx<16>{}, y10_0_1);
  const unsigned long long w10_0_0 = p15 + p16;
  const unsigned long long w10_0_1 = p15 - p16;
  s[0] += w10_0_0;
  s[3] += 4ull * w10_0_0;
  s[1] += 2ull * w10_0_1;
  s[7] += 8ull * w10_0_1;
  const int c11_0 = d[0] + 4 * d[3] + 4 * d[5];
  const int c11_x = 2 * d[1] + 16 * d[7];
  const int y11_0_0 = c11_0 + c11_x;
  const int y11_0_1 = c11_0 - c11_x;
  const unsigned long long p25 = p(Idx<25>{}, y11_0_0);
  const unsigned long long p26 = p(Idx<26>{}, y11_0_1);
  const unsigned long long w11_0_0 = p25 + p26;
  const unsigned long long w11_0_1 = p25 - p26;
  s[0] += 2ull * w11_0_0;
  s[3] += 8ull * w11_0_0;
  s[5] += 8ull * w11_0_0;
  s[1] += 4ull * w11_0_1;
  s[7] += 32ull * w11_0_1;
  const int c12_0 = d[0] + 4 * d[3] + 4 * d[4];
  const int c12_x = 2 * d[1] + 16 * d[7];
  const int c12_y = 2 * d[2] + 16 * d[8];
  const int c12_xy = 4 * d[6];
  const int y12_0_0 = c12_0 + c12_x;
  const int y12_0_1 = c12_0 - c12_x;
  const int y12_0_2 = c12_y + c12_xy;
  const int y12_0_3 = c12_y - c12_xy;
  const int y12_1_0 = y12_0_1 + y12_0_3;
  const int y12_1_1 = y12_0_1 - y12_0_3;
  const int y12_1_2 = y12_0_0 + y12_0_2;
  const int y12_1_3 = y12_0_0 - y12_0_2;
  const unsigned long long p21 = p(Idx<21>{}, y12_1_2);
  const unsigned long long p22 = p(Idx<22>{}, y12_1_1);
  const unsigned long long p23 = p(Idx<23>{}, y12_1_3);
  const unsigned long long p24 = p(Idx<24>{}, y12_1_0);
  const unsigned long long w12_0_0 = p23 + p22;
  const unsigned long long w12_0_1 = p23 - p22;
  const unsigned long long w12_0_2 = p21 + p24;
  const unsigned long long w12_0_3 = p21 - p24;
  const unsigned long long w12_1_0 = w12_0_2 + w12_0_0;
  const unsigned long long w12_1_1 = w12_0_2 - w12_0_0;
  const unsigned long long w12_1_2 = w12_0_3 + w12_0_1;
  const unsigned long long w12_1_3 = w12_0_3 - w12_0_1;
  s[0] += w12_1_0;
  s[3] += 4ull * w12_1_0;
  s[4] += 4ull * w12_1_0;
  s[2] += 2ull * w12_1_1;
  s[8] += 16ull * w12_1_1;
  s[1] += 2ull * w12_1_2;
  s[7] += 16ull * w12_1_2;
  s[6] += 4ull * w12_1_3;
  const int c13_0 = d[0] + 9 * d[3];
  const int c13_x = 3 * d[1] + 27 * d[7];
  const int y13_0_0 = c13_0 + c13_x;
  const int y13_0_1 = c13_0 - c13_x;
  const unsigned long long p33 = p(Idx<33>{}, y13_0_0);
  const unsigned long long p34 = p(Idx<34>{}, y13_0_1);
  const unsigned long long w13_0_0 = p33 + p34;
  const unsigned long long w13_0_1 = p33 - p34;
  s[0] += w13_0_0;
  s[3] += 9ull * w13_0_0;
  s[1] += 3ull * w13_0_1;
  s[7] += 27ull * w13_0_1;
}

// sum_i v(i) [1, xi_i, |xi_i|^2] in 64-bit integers (values mirror-symmetric in z: no xi_z).
template <class V>
__device__ __forceinline__ void macro_fx2d(const V& v, unsigned long long (&s)[4]) {
  const unsigned long long v0 = v(Idx<0>{});
  s[0] = v0;
  const unsigned long long v5 = v(Idx<5>{});
  s[0] += 2ull * v5;
  s[3] = 2ull * v5;
  const unsigned long long v19 = v(Idx<19>{});
  s[0] += 2ull * v19;
  s[3] += 8ull * v19;
  const unsigned long long v37 = v(Idx<37>{});
  s[0] += 2ull * v37;
  s[3] += 18ull * v37;
  const unsigned long long v3 = v(Idx<3>{});
  const unsigned long long v4 = v(Idx<4>{});
  const unsigned long long w4_0_0 = v3 + v4;
  const unsigned long long w4_0_1 = v3 - v4;
  s[0] += w4_0_0;
  s[3] += w4_0_0;
  s[2] = w4_0_1;
  const unsigned long long v17 = v(Idx<17>{});
  const unsigned long long v18 = v(Idx<18>{});
  const unsigned long long w5_0_0 = v17 + v18;
  const unsigned long long w5_0_1 = v17 - v18;
  s[0] += w5_0_0;
  s[3] += 4ull * w5_0_0;
  s[2] += 2ull * w5_0_1;
  const unsigned long long v29 = v(Idx<29>{});
  const unsigned long long v30 = v(Idx<30>{});
  const unsigned long long w6_0_0 = v29 + v30;
  const unsigned long long w6_0_1 = v29 - v30;
  s[0] += 2ull * w6_0_0;
  s[3] += 16ull * w6_0_0;
  s[2] += 4ull * w6_0_1;
  const unsigned long long v35 = v(Idx<35>{});
  const unsigned long long v36 = v(Idx<36>{});
  const unsigned long long w7_0_0 = v35 + v36;
  const unsigned long long w7_0_1 = v35 - v36;
  s[0] += w7_0_0;
  s[3] += 9ull * w7_0_0;
  s[2] += 3ull * w7_0_1;
  const unsigned long long v1 = v(Idx<1>{});
  const unsigned long long v2 = v(Idx<2>{});
  const unsigned long long w8_0_0 = v1 + v2;
  const unsigned long long w8_0_1 = v1 - v2;
  s[0] += w8_0_0;
  s[3] += w8_0_0;
  s[1] = w8_0_1;
  const unsigned long long v7 = v(Idx<7>{});
  const unsigned long long v8 = v(Idx<8>{});
  const unsigned long long v11 = v(Idx<11>{});
  const unsigned long long v12 = v(Idx<12>{});
  const unsigned long long w9_0_0 = v11 + v8;
  const unsigned long long w9_0_1 = v11 - v8;
  const unsigned long long w9_0_2 = v7 + v12;
  const unsigned long long w9_0_3 = v7 - v12;
  const unsigned long long w9_1_0 = w9_0_2 + w9_0_0;
  const unsigned long long w9_1_1 = w9_0_2 - w9_0_0;
  const unsigned long long w9_1_2 = w9_0_3 + w9_0_1;
  const unsigned long long w9_1_3 = w9_0_3 - w9_0_1;
  s[0] += 2ull * w9_1_0;
  s[3] += 6ull * w9_1_0;
  s[2] += 2ull * w9_1_1;
  s[1] += 2ull * w9_1_2;
  const unsigned long long v15 = v(Idx<15>{});
  const unsigned long long v16 = v(Idx<16>{});
  const unsigned long long w10_0_0 = v15 + v16;
  const unsigned long long w10_0_1 = v15 - v16;
  s[0] += w10_0_0;
  s[3] += 4ull * w10_0_0;
  s[1] += 2ull * w10_0_1;
  const unsigned long long v25 = v(Idx<25>{});
  const unsigned long long v26 = v(Idx<26>{});
  const unsigned long long w11_0_0 = v25 + v26;
  const unsigned long long w11_0_1 = v25 - v26;
  s[0] += 2ull * w11_0_0;
  s[3] += 16ull * w11_0_0;
  s[1] += 4ull * w11_0_1;
  const unsigned long long v21 = v(Idx<21>{});
  const unsigned long long v22 = v(Idx<22>{});
  const unsigned long long v23 = v(Idx<23>{});
  const unsigned long long v24 = v(Idx<24>{});
  const unsigned long long w12_0_0 = v23 + v22;
  const unsigned long long w12_0_1 = v23 - v22;
  const unsigned long long w12_0_2 = v21 + v24;
  const unsigned long long w12_0_3 = v21 - v24;
  const unsigned long long w12_1_0 = w12_0_2 + w12_0_0;
  const unsigned long long w12_1_1 = w12_0_2 - w12_0_0;
  const unsigned long long w12_1_2 = w12_0_3 + w12_0_1;
  const unsigned long long w12_1_3 = w12_0_3 - w12_0_1;
  s[0] += w12_1_0;
  s[3] += 8ull * w12_1_0;
  s[2] += 2ull * w12_1_1;
  s[1] += 2ull * w12_1_2;
  const unsigned long long v33 = v(Idx<33>{});
  const unsigned long long v34 = v(Idx<34>{});
  const unsigned long long w13_0_0 = v33 + v34;
  const unsigned long long w13_0_1 = v33 - v34;
  s[0] += w13_0_0;
  s[3] += 9ull * w13_0_0;
  s[1] += 3ull * w13_0_1;
}

// 2^(j/1024) in units of 2^-55, j = 0..1023, each the integer nearest the exact value.
__device__ const unsigned long long kExp2Fixed[1024] = {
    36028797018963968ull, 36053193223259766ull, 36077605946974287ull, 36102035201293337ull,
    36126480997410295ull, 36150943346526120ull, 36175422259849356ull, 36199917748596135ull,
    36224429823990187ull, 36248958497262839ull, 36273503779653025ull, 36298065682407286ull,
    36322644216779783ull, 36347239394032294ull, 36371851225434223ull, 36396479722262608ull,
    36421124895802119ull, 36445786757345070ull, 36470465318191420ull, 36495160589648779ull,
    36519872583032416ull, 36544601309665260ull, 36569346780877907ull, 36594109008008627ull,
    36618888002403366ull, 36643683775415753ull, 36668496338407104ull, 36693325702746431ull,
    36718171879810441ull, 36743034880983547ull, 36767914717657869ull, 36792811401233241ull,
    36817724943117218ull, 36842655354725077ull, 36867602647479827ull, 36892566832812210ull,
    36917547922160709ull, 36942545926971552ull, 36967560858698718ull, 36992592728803942ull,
    37017641548756718ull, 37042707330034310ull, 37067790084121750ull, 37092889822511850ull,
    37118006556705201ull, 37143140298210185ull, 37168291058542973ull, 37193458849227536ull,
    37218643681795648ull, 37243845567786892ull, 37269064518748664ull, 37294300546236179ull,
    37319553661812477ull, 37344823877048427ull, 37370111203522734ull, 37395415652821942ull,
    37420737236540442ull, 37446075966280475ull, 37471431853652138ull, 37496804910273390ull,
    37522195147770057ull, 37547602577775838ull, 37573027211932307ull, 37598469061888924ull,
    37623928139303035ull, 37649404455839880ull, 37674898023172599ull, 37700408852982234ull,
    37725936956957739ull, 37751482346795981ull, 37777045034201749ull, 37802625030887757ull,
    37828222348574650ull, 37853836998991009ull, 37879468993873356ull, 37905118344966163ull,
    37930785064021853ull, 37956469162800805ull, 37982170653071364ull, 38007889546609843ull,
    38033625855200528ull, 38059379590635686ull, 38085150764715569ull, 38110939389248418ull,
    38136745476050469ull, 38162569036945963ull, 38188410083767143ull, 38214268628354266ull,
    38240144682555608ull, 38266038258227464ull, 38291949367234161ull, 38317878021448059ull,
    38343824232749554ull, 38369788013027090ull, 38395769374177160ull, 38421768328104313ull,
    38447784886721157ull, 38473819061948369ull, 38499870865714696ull, 38525940309956962ull,
    38552027406620076ull, 38578132167657034ull, 38604254605028925ull, 38630394730704939ull,
    38656552556662368ull, 38682728094886617ull, 38708921357371205ull, 38735132356117773ull,
    38761361103136088ull, 38787607610444049ull, 38813871890067695ull, 38840153954041206ull,
    38866453814406910ull, 38892771483215290ull, 38919106972524991ull, 38945460294402821ull,
    38971831460923758ull, 38998220484170959ull, 39024627376235760ull, 39051052149217687ull,
    39077494815224457ull, 39103955386371987ull, 39130433874784397ull, 39156930292594017ull,
    39183444651941392ull, 39209976964975288ull, 39236527243852698ull, 39263095500738845ull,
    39289681747807191ull, 39316285997239440ull, 39342908261225546ull, 39369548551963716ull,
    39396206881660417ull, 39422883262530381ull, 39449577706796612ull, 39476290226690390ull,
    39503020834451278ull, 39529769542327125ull, 39556536362574074ull, 39583321307456568ull,
    39610124389247355ull, 39636945620227490ull, 39663785012686348ull, 39690642578921624ull,
    39717518331239338ull, 39744412281953846ull, 39771324443387840ull, 39798254827872358ull,
    39825203447746787ull, 39852170315358868ull, 39879155443064706ull, 39906158843228769ull,
    39933180528223901ull, 39960220510431321ull, 39987278802240634ull, 40014355416049833ull,
    40041450364265306ull, 40068563659301843ull, 40095695313582640ull, 40122845339539303ull,
    40150013749611860ull, 40177200556248758ull, 40204405771906877ull, 40231629409051529ull,
    40258871480156469ull, 40286131997703897ull, 40313410974184465ull, 40340708422097283ull,
    40368024353949926ull, 40395358782258435ull, 40422711719547330ull, 40450083178349609ull,
    40477473171206757ull, 40504881710668751ull, 40532308809294067ull, 40559754479649683ull,
    40587218734311090ull, 40614701585862290ull, 40642203046895808ull, 40669723130012696ull,
    40697261847822538ull, 40724819212943457ull, 40752395238002120ull, 40779989935633742ull,
    40807603318482097ull, 40835235399199518ull, 40862886190446906ull, 40890555704893735ull,
    40918243955218058ull, 40945950954106513ull, 40973676714254328ull, 41001421248365328ull,
    41029184569151939ull, 41056966689335197ull, 41084767621644748ull, 41112587378818863ull,
    41140425973604434ull, 41168283418756986ull, 41196159727040681ull, 41224054911228324ull,
    41251968984101370ull, 41279901958449926ull, 41307853847072763ull, 41335824662777315ull,
    41363814418379690ull, 41391823126704676ull, 41419850800585742ull, 41447897452865047ull,
    41475963096393449ull, 41504047744030505ull, 41532151408644479ull, 41560274103112352ull,
    41588415840319820ull, 41616576633161307ull, 41644756494539969ull, 41672955437367697ull,
    41701173474565125ull, 41729410619061637ull, 41757666883795373ull, 41785942281713232ull,
    41814236825770879ull, 41842550528932754ull, 41870883404172074ull, 41899235464470842ull,
    41927606722819849ull, 41955997192218686ull, 41984406885675743ull, 42012835816208221ull,
    42041283996842133ull, 42069751440612314ull, 42098238160562425ull, 42126744169744959ull,
    42155269481221248ull, 42183814108061466ull, 42212378063344640ull, 42240961360158652ull,
    42269564011600245ull, 42298186030775033ull, 42326827430797501ull, 42355488224791017ull,
    42384168425887834ull, 42412868047229097ull, 42441587101964849ull, 42470325603254038ull,
    42499083564264524ull, 42527860998173079ull, 42556657918165402ull, 42585474337436117ull,
    42614310269188785ull, 42643165726635905ull, 42672040722998926ull, 42700935271508246ull,
    42729849385403224ull, 42758783077932183ull, 42787736362352417ull, 42816709251930197ull,
    42845701759940777ull, 42874713899668401ull, 42903745684406305ull, 42932797127456730ull,
    42961868242130922ull, 42990959041749141ull, 43020069539640668ull, 43049199749143808ull,
    43078349683605898ull, 43107519356383313ull, 43136708780841472ull, 43165917970354845ull,
    43195146938306956ull, 43224395698090395ull, 43253664263106818ull, 43282952646766955ull,
    43312260862490618ull, 43341588923706708ull, 43370936843853214ull, 43400304636377230ull,
    43429692314734951ull, 43459099892391686ull, 43488527382821861ull, 43517974799509026ull,
    43547442155945862ull, 43576929465634185ull, 43606436742084954ull, 43635963998818276ull,
    43665511249363414ull, 43695078507258792ull, 43724665786052001ull, 43754273099299806ull,
    43783900460568149ull, 43813547883432162ull, 43843215381476167ull, 43872902968293683ull,
    43902610657487437ull, 43932338462669364ull, 43962086397460617ull, 43991854475491572ull,
    44021642710401836ull, 44051451115840250ull, 44081279705464898ull, 44111128492943111ull,
    44140997491951477ull, 44170886716175842ull, 44200796179311322ull, 44230725895062304ull,
    44260675877142455ull, 44290646139274730ull, 44320636695191374ull, 44350647558633931ull,
    44380678743353251ull, 44410730263109493ull, 44440802131672135ull, 44470894362819979ull,
    44501006970341156ull, 44531139968033134ull, 44561293369702723ull, 44591467189166083ull,
    44621661440248729ull, 44651876136785537ull, 44682111292620752ull, 44712366921607992ull,
    44742643037610258ull, 44772939654499935ull, 44803256786158805ull, 44833594446478047ull,
    44863952649358246ull, 44894331408709402ull, 44924730738450933ull, 44955150652511679ull,
    44985591164829917ull, 45016052289353358ull, 45046534040039159ull, 45077036430853928ull,
    45107559475773730ull, 45138103188784092ull, 45168667583880014ull, 45199252675065971ull,
    45229858476355920ull, 45260485001773308ull, 45291132265351078ull, 45321800281131675ull,
    45352489063167053ull, 45383198625518680ull, 45413928982257545ull, 45444680147464168ull,
    45475452135228599ull, 45506244959650432ull, 45537058634838808ull, 45567893174912419ull,
    45598748593999522ull, 45629624906237935ull, 45660522125775054ull, 45691440266767852ull,
    45722379343382888ull, 45753339369796316ull, 45784320360193886ull, 45815322328770956ull,
    45846345289732496ull, 45877389257293092ull, 45908454245676958ull, 45939540269117938ull,
    45970647341859516ull, 46001775478154818ull, 46032924692266624ull, 46064094998467370ull,
    46095286411039156ull, 46126498944273756ull, 46157732612472616ull, 46188987429946871ull,
    46220263411017345ull, 46251560570014556ull, 46282878921278731ull, 46314218479159803ull,
    46345579258017423ull, 46376961272220966ull, 46408364536149536ull, 46439789064191976ull,
    46471234870746867ull, 46502701970222545ull, 46534190377037101ull, 46565700105618385ull,
    46597231170404023ull, 46628783585841412ull, 46660357366387734ull, 46691952526509960ull,
    46723569080684857ull, 46755207043398995ull, 46786866429148753ull, 46818547252440325ull,
    46850249527789730ull, 46881973269722814ull, 46913718492775260ull, 46945485211492593ull,
    46977273440430187ull, 47009083194153273ull, 47040914487236944ull, 47072767334266162ull,
    47104641749835765ull, 47136537748550474ull, 47168455345024899ull, 47200394553883545ull,
    47232355389760821ull, 47264337867301047ull, 47296342001158455ull, 47328367805997202ull,
    47360415296491377ull, 47392484487325001ull, 47424575393192039ull, 47456688028796409ull,
    47488822408851982ull, 47520978548082593ull, 47553156461222048ull, 47585356163014128ull,
    47617577668212599ull, 47649820991581217ull, 47682086147893734ull, 47714373151933907ull,
    47746682018495503ull, 47779012762382306ull, 47811365398408124ull, 47843739941396797ull,
    47876136406182201ull, 47908554807608259ull, 47940995160528942ull, 47973457479808282ull,
    48005941780320374ull, 48038448076949386ull, 48070976384589563ull, 48103526718145236ull,
    48136099092530830ull, 48168693522670866ull, 48201310023499973ull, 48233948609962892ull,
    48266609297014483ull, 48299292099619734ull, 48331997032753764ull, 48364724111401833ull,
    48397473350559350ull, 48430244765231875ull, 48463038370435129ull, 48495854181195004ull,
    48528692212547561ull, 48561552479539047ull, 48594434997225896ull, 48627339780674736ull,
    48660266844962397ull, 48693216205175920ull, 48726187876412561ull, 48759181873779798ull,
    48792198212395339ull, 48825236907387129ull, 48858297973893357ull, 48891381427062462ull,
    48924487282053141ull, 48957615554034353ull, 48990766258185333ull, 49023939409695590ull,
    49057135023764920ull, 49090353115603412ull, 49123593700431453ull, 49156856793479736ull,
    49190142409989268ull, 49223450565211377ull, 49256781274407716ull, 49290134552850274ull,
    49323510415821379ull, 49356908878613710ull, 49390329956530299ull, 49423773664884540ull,
    49457240019000198ull, 49490729034211413ull, 49524240725862708ull, 49557775109308996ull,
    49591332199915590ull, 49624912013058202ull, 49658514564122961ull, 49692139868506412ull,
    49725787941615524ull, 49759458798867701ull, 49793152455690785ull, 49826868927523065ull,
    49860608229813286ull, 49894370378020649ull, 49928155387614828ull, 49961963274075968ull,
    49995794052894699ull, 50029647739572138ull, 50063524349619901ull, 50097423898560103ull,
    50131346401925374ull, 50165291875258860ull, 50199260334114230ull, 50233251794055687ull,
    50267266270657973ull, 50301303779506374ull, 50335364336196733ull, 50369447956335449ull,
    50403554655539493ull, 50437684449436406ull, 50471837353664315ull, 50506013383871934ull,
    50540212555718574ull, 50574434884874149ull, 50608680387019183ull, 50642949077844819ull,
    50677240973052824ull, 50711556088355598ull, 50745894439476180ull, 50780256042148255ull,
    50814640912116162ull, 50849049065134901ull, 50883480516970141ull, 50917935283398225ull,
    50952413380206181ull, 50986914823191723ull, 51021439628163266ull, 51055987810939928ull,
    51090559387351537ull, 51125154373238642ull, 51159772784452518ull, 51194414636855171ull,
    51229079946319351ull, 51263768728728554ull, 51298480999977032ull, 51333216775969798ull,
    51367976072622636ull, 51402758905862107ull, 51437565291625556ull, 51472395245861120ull,
    51507248784527736ull, 51542125923595144ull, 51577026679043901ull, 51611951066865384ull,
    51646899103061798ull, 51681870803646182ull, 51716866184642421ull, 51751885262085248ull,
    51786928052020254ull, 51821994570503897ull, 51857084833603503ull, 51892198857397282ull,
    51927336657974328ull, 51962498251434632ull, 51997683653889086ull, 52032892881459489ull,
    52068125950278559ull, 52103382876489937ull, 52138663676248197ull, 52173968365718848ull,
    52209296961078350ull, 52244649478514112ull, 52280025934224507ull, 52315426344418876ull,
    52350850725317534ull, 52386299093151782ull, 52421771464163909ull, 52457267854607204ull,
    52492788280745962ull, 52528332758855489ull, 52563901305222113ull, 52599493936143190ull,
    52635110667927110ull, 52670751516893308ull, 52706416499372268ull, 52742105631705532ull,
    52777818930245707ull, 52813556411356475ull, 52849318091412596ull, 52885103986799919ull,
    52920914113915387ull, 52956748489167048ull, 52992607128974058ull, 53028490049766693ull,
    53064397267986354ull, 53100328800085574ull, 53136284662528028ull, 53172264871788537ull,
    53208269444353079ull, 53244298396718795ull, 53280351745393997ull, 53316429506898175ull,
    53352531697762005ull, 53388658334527355ull, 53424809433747296ull, 53460985011986108ull,
    53497185085819284ull, 53533409671833544ull, 53569658786626838ull, 53605932446808355ull,
    53642230668998530ull, 53678553469829055ull, 53714900865942879ull, 53751272873994226ull,
    53787669510648593ull, 53824090792582762ull, 53860536736484810ull, 53897007359054112ull,
    53933502677001351ull, 53970022707048525ull, 54006567465928956ull, 54043136970387295ull,
    54079731237179534ull, 54116350283073007ull, 54152994124846406ull, 54189662779289782ull,
    54226356263204555ull, 54263074593403521ull, 54299817786710864ull, 54336585859962157ull,
    54373378830004372ull, 54410196713695893ull, 54447039527906514ull, 54483907289517457ull,
    54520800015421371ull, 54557717722522346ull, 54594660427735916ull, 54631628147989071ull,
    54668620900220262ull, 54705638701379411ull, 54742681568427913ull, 54779749518338654ull,
    54816842568096008ull, 54853960734695852ull, 54891104035145571ull, 54928272486464067ull,
    54965466105681764ull, 55002684909840620ull, 55039928915994130ull, 55077198141207341ull,
    55114492602556849ull, 55151812317130819ull, 55189157302028984ull, 55226527574362655ull,
    55263923151254731ull, 55301344049839706ull, 55338790287263675ull, 55376261880684344ull,
    55413758847271036ull, 55451281204204700ull, 55488828968677921ull, 55526402157894922ull,
    55564000789071579ull, 55601624879435422ull, 55639274446225650ull, 55676949506693132ull,
    55714650078100420ull, 55752376177721754ull, 55790127822843070ull, 55827905030762013ull,
    55865707818787935ull, 55903536204241914ull, 55941390204456752ull, 55979269836776992ull,
    56017175118558917ull, 56055106067170566ull, 56093062699991738ull, 56131045034413998ull,
    56169053087840689ull, 56207086877686940ull, 56245146421379669ull, 56283231736357597ull,
    56321342840071251ull, 56359479749982976ull, 56397642483566941ull, 56435831058309148ull,
    56474045491707436ull, 56512285801271497ull, 56550552004522876ull, 56588844118994984ull,
    56627162162233103ull, 56665506151794397ull, 56703876105247917ull, 56742272040174612ull,
    56780693974167336ull, 56819141924830852ull, 56857615909781849ull, 56896115946648940ull,
    56934642053072678ull, 56973194246705560ull, 57011772545212036ull, 57050376966268517ull,
    57089007527563383ull, 57127664246796993ull, 57166347141681689ull, 57205056229941807ull,
    57243791529313688ull, 57282553057545678ull, 57321340832398144ull, 57360154871643479ull,
    57398995193066108ull, 57437861814462502ull, 57476754753641178ull, 57515674028422716ull,
    57554619656639761ull, 57593591656137032ull, 57632590044771333ull, 57671614840411558ull,
    57710666060938702ull, 57749743724245866ull, 57788847848238269ull, 57827978450833253ull,
    57867135549960292ull, 57906319163561002ull, 57945529309589145ull, 57984766006010644ull,
    58024029270803585ull, 58063319121958227ull, 58102635577477011ull, 58141978655374570ull,
    58181348373677733ull, 58220744750425537ull, 58260167803669232ull, 58299617551472293ull,
    58339094011910425ull, 58378597203071573ull, 58418127143055931ull, 58457683849975947ull,
    58497267341956335ull, 58536877637134082ull, 58576514753658455ull, 58616178709691011ull,
    58655869523405606ull, 58695587212988399ull, 58735331796637867ull, 58775103292564806ull,
    58814901718992348ull, 58854727094155958ull, 58894579436303456ull, 58934458763695011ull,
    58974365094603163ull, 59014298447312820ull, 59054258840121274ull, 59094246291338205ull,
    59134260819285693ull, 59174302442298222ull, 59214371178722694ull, 59254467046918431ull,
    59294590065257188ull, 59334740252123161ull, 59374917625912994ull, 59415122205035786ull,
    59455354007913104ull, 59495613052978988ull, 59535899358679960ull, 59576212943475031ull,
    59616553825835715ull, 59656922024246031ull, 59697317557202515ull, 59737740443214226ull,
    59778190700802757ull, 59818668348502245ull, 59859173404859373ull, 59899705888433384ull,
    59940265817796090ull, 59980853211531876ull, 60021468088237712ull, 60062110466523161ull,
    60102780365010386ull, 60143477802334160ull, 60184202797141876ull, 60224955368093550ull,
    60265735533861838ull, 60306543313132036ull, 60347378724602093ull, 60388241786982621ull,
    60429132518996899ull, 60470050939380886ull, 60510997066883227ull, 60551970920265262ull,
    60592972518301035ull, 60634001879777303ull, 60675059023493543ull, 60716143968261963ull,
    60757256732907509ull, 60798397336267874ull, 60839565797193504ull, 60880762134547614ull,
    60921986367206189ull, 60963238514057994ull, 61004518594004588ull, 61045826625960325ull,
    61087162628852371ull, 61128526621620703ull, 61169918623218126ull, 61211338652610278ull,
    61252786728775640ull, 61294262870705541ull, 61335767097404174ull, 61377299427888596ull,
    61418859881188743ull, 61460448476347438ull, 61502065232420396ull, 61543710168476237ull,
    61585383303596492ull, 61627084656875614ull, 61668814247420983ull, 61710572094352920ull,
    61752358216804690ull, 61794172633922517ull, 61836015364865587ull, 61877886428806061ull,
    61919785844929079ull, 61961713632432777ull, 62003669810528285ull, 62045654398439745ull,
    62087667415404317ull, 62129708880672183ull, 62171778813506563ull, 62213877233183721ull,
    62256004158992972ull, 62298159610236693ull, 62340343606230331ull, 62382556166302413ull,
    62424797309794552ull, 62467067056061460ull, 62509365424470953ull, 62551692434403964ull,
    62594048105254545ull, 62636432456429885ull, 62678845507350311ull, 62721287277449303ull,
    62763757786173496ull, 62806257052982697ull, 62848785097349886ull, 62891341938761234ull,
    62933927596716100ull, 62976542090727052ull, 63019185440319869ull, 63061857665033550ull,
    63104558784420326ull, 63147288818045667ull, 63190047785488292ull, 63232835706340176ull,
    63275652600206561ull, 63318498486705965ull, 63361373385470189ull, 63404277316144329ull,
    63447210298386781ull, 63490172351869255ull, 63533163496276778ull, 63576183751307710ull,
    63619233136673747ull, 63662311672099933ull, 63705419377324669ull, 63748556272099720ull,
    63791722376190226ull, 63834917709374712ull, 63878142291445095ull, 63921396142206693ull,
    63964679281478234ull, 64007991729091869ull, 64051333504893175ull, 64094704628741167ull,
    64138105120508310ull, 64181535000080523ull, 64224994287357190ull, 64268483002251171ull,
    64312001164688809ull, 64355548794609939ull, 64399125911967899ull, 64442732536729537ull,
    64486368688875223ull, 64530034388398853ull, 64573729655307866ull, 64617454509623244ull,
    64661208971379529ull, 64704993060624827ull, 64748806797420822ull, 64792650201842779ull,
    64836523293979559ull, 64880426093933624ull, 64924358621821050ull, 64968320897771533ull,
    65012312941928398ull, 65056334774448613ull, 65100386415502792ull, 65144467885275209ull,
    65188579203963805ull, 65232720391780196ull, 65276891468949686ull, 65321092455711273ull,
    65365323372317660ull, 65409584239035264ull, 65453875076144225ull, 65498195903938413ull,
    65542546742725443ull, 65586927612826678ull, 65631338534577245ull, 65675779528326036ull,
    65720250614435724ull, 65764751813282772ull, 65809283145257437ull, 65853844630763785ull,
    65898436290219698ull, 65943058144056884ull, 65987710212720884ull, 66032392516671086ull,
    66077105076380729ull, 66121847912336917ull, 66166621045040626ull, 66211424495006714ull,
    66256258282763928ull, 66301122428854920ull, 66346016953836248ull, 66390941878278391ull,
    66435897222765758ull, 66480883007896694ull, 66525899254283495ull, 66570945982552411ull,
    66616023213343659ull, 66661130967311435ull, 66706269265123918ull, 66751438127463282ull,
    66796637575025708ull, 66841867628521387ull, 66887128308674537ull, 66932419636223408ull,
    66977741631920293ull, 67023094316531534ull, 67068477710837539ull, 67113891835632784ull,
    67159336711725826ull, 67204812359939314ull, 67250318801109994ull, 67295856056088723ull,
    67341424145740476ull, 67387023090944357ull, 67432652912593607ull, 67478313631595614ull,
    67524005268871926ull, 67569727845358253ull, 67615481382004486ull, 67661265899774698ull,
    67707081419647159ull, 67752927962614345ull, 67798805549682945ull, 67844714201873873ull,
    67890653940222277ull, 67936624785777548ull, 67982626759603331ull, 68028659882777532ull,
    68074724176392333ull, 68120819661554194ull, 68166946359383871ull, 68213104291016418ull,
    68259293477601201ull, 68305513940301909ull, 68351765700296559ull, 68398048778777511ull,
    68444363196951471ull, 68490708976039508ull, 68537086137277060ull, 68583494701913943ull,
    68629934691214362ull, 68676406126456923ull, 68722909028934637ull, 68769443419954936ull,
    68816009320839678ull, 68862606752925159ull, 68909235737562123ull, 68955896296115771ull,
    69002588449965772ull, 69049312220506270ull, 69096067629145897ull, 69142854697307780ull,
    69189673446429555ull, 69236523897963370ull, 69283406073375904ull, 69330319994148366ull,
    69377265681776516ull, 69424243157770667ull, 69471252443655695ull, 69518293560971055ull,
    69565366531270786ull, 69612471376123521ull, 69659608117112497ull, 69706776775835568ull,
    69753977373905212ull, 69801209932948539ull, 69848474474607307ull, 69895771020537925ull,
    69943099592411470ull, 69990460211913688ull, 70037852900745015ull, 70085277680620576ull,
    70132734573270202ull, 70180223600438440ull, 70227744783884557ull, 70275298145382555ull,
    70322883706721183ull, 70370501489703940ull, 70418151516149090ull, 70465833807889672ull,
    70513548386773507ull, 70561295274663211ull, 70609074493436204ull, 70656886064984718ull,
    70704730011215812ull, 70752606354051376ull, 70800515115428146ull, 70848456317297711ull,
    70896429981626524ull, 70944436130395913ull, 70992474785602090ull, 71040545969256161ull,
    71088649703384136ull, 71136786010026940ull, 71184954911240422ull, 71233156429095368ull,
    71281390585677505ull, 71329657403087519ull, 71377956903441057ull, 71426289108868745ull,
    71474654041516191ull, 71523051723544001ull, 71571482177127785ull, 71619945424458170ull,
    71668441487740808ull, 71716970389196388ull, 71765532151060644ull, 71814126795584367ull,
    71862754345033417ull, 71911414821688726ull, 71960108247846319ull, 72008834645817313ull,
};

}  // namespace gen
}  // namespace lbm39
