// GENERATED by gen_expansion.py -- do not edit by hand.
// Straight-line Cartesian expansion pieces over scaled symmetric
// coefficients (multi-index alpha, divided by alpha!).  Multi-indices are
// ordered by degree, then a descending, then b descending.
#pragma once

#define SFMM_NM_0 1  /* potential coefficients, |beta| <= 0 */
#define SFMM_NF_0 3  /* acceleration coefficients, 1 <= |gamma| <= 1 */
#define SFMM_NM_1 4  /* potential coefficients, |beta| <= 1 */
#define SFMM_NF_1 9  /* acceleration coefficients, 1 <= |gamma| <= 2 */
#define SFMM_NM_2 10  /* potential coefficients, |beta| <= 2 */
#define SFMM_NF_2 19  /* acceleration coefficients, 1 <= |gamma| <= 3 */
#define SFMM_NM_3 20  /* potential coefficients, |beta| <= 3 */
#define SFMM_NF_3 34  /* acceleration coefficients, 1 <= |gamma| <= 4 */
#define SFMM_NM_4 35  /* potential coefficients, |beta| <= 4 */
#define SFMM_NF_4 55  /* acceleration coefficients, 1 <= |gamma| <= 5 */

template <typename T> __device__ __forceinline__ void sfmm_mono_0(T vx, T vy, T vz, T* o) {
  o[0] = T(1);
}

template <typename T> __device__ __forceinline__ void sfmm_mono_1(T vx, T vy, T vz, T* o) {
  o[0] = T(1);
  o[1] = o[0] * vx;
  o[2] = o[0] * vy;
  o[3] = o[0] * vz;
}

template <typename T> __device__ __forceinline__ void sfmm_mono_2(T vx, T vy, T vz, T* o) {
  o[0] = T(1);
  o[1] = o[0] * vx;
  o[2] = o[0] * vy;
  o[3] = o[0] * vz;
  o[4] = o[1] * (vx * T(0.5));
  o[5] = o[2] * vx;
  o[6] = o[3] * vx;
  o[7] = o[2] * (vy * T(0.5));
  o[8] = o[3] * vy;
  o[9] = o[3] * (vz * T(0.5));
}

template <typename T> __device__ __forceinline__ void sfmm_mono_3(T vx, T vy, T vz, T* o) {
  o[0] = T(1);
  o[1] = o[0] * vx;
  o[2] = o[0] * vy;
  o[3] = o[0] * vz;
  o[4] = o[1] * (vx * T(0.5));
  o[5] = o[2] * vx;
  o[6] = o[3] * vx;
  o[7] = o[2] * (vy * T(0.5));
  o[8] = o[3] * vy;
  o[9] = o[3] * (vz * T(0.5));
  o[10] = o[4] * (vx * T(0.3333333333333333));
  o[11] = o[5] * (vx * T(0.5));
  o[12] = o[6] * (vx * T(0.5));
  o[13] = o[7] * vx;
  o[14] = o[8] * vx;
  o[15] = o[9] * vx;
  o[16] = o[7] * (vy * T(0.3333333333333333));
  o[17] = o[8] * (vy * T(0.5));
  o[18] = o[9] * vy;
  o[19] = o[9] * (vz * T(0.3333333333333333));
}

template <typename T> __device__ __forceinline__ void sfmm_mono_4(T vx, T vy, T vz, T* o) {
  o[0] = T(1);
  o[1] = o[0] * vx;
  o[2] = o[0] * vy;
  o[3] = o[0] * vz;
  o[4] = o[1] * (vx * T(0.5));
  o[5] = o[2] * vx;
  o[6] = o[3] * vx;
  o[7] = o[2] * (vy * T(0.5));
  o[8] = o[3] * vy;
  o[9] = o[3] * (vz * T(0.5));
  o[10] = o[4] * (vx * T(0.3333333333333333));
  o[11] = o[5] * (vx * T(0.5));
  o[12] = o[6] * (vx * T(0.5));
  o[13] = o[7] * vx;
  o[14] = o[8] * vx;
  o[15] = o[9] * vx;
  o[16] = o[7] * (vy * T(0.3333333333333333));
  o[17] = o[8] * (vy * T(0.5));
  o[18] = o[9] * vy;
  o[19] = o[9] * (vz * T(0.3333333333333333));
  o[20] = o[10] * (vx * T(0.25));
  o[21] = o[11] * (vx * T(0.3333333333333333));
  o[22] = o[12] * (vx * T(0.3333333333333333));
  o[23] = o[13] * (vx * T(0.5));
  o[24] = o[14] * (vx * T(0.5));
  o[25] = o[15] * (vx * T(0.5));
  o[26] = o[16] * vx;
  o[27] = o[17] * vx;
  o[28] = o[18] * vx;
  o[29] = o[19] * vx;
  o[30] = o[16] * (vy * T(0.25));
  o[31] = o[17] * (vy * T(0.3333333333333333));
  o[32] = o[18] * (vy * T(0.5));
  o[33] = o[19] * vy;
  o[34] = o[19] * (vz * T(0.25));
}

template <typename T> __device__ __forceinline__ void sfmm_mono_5(T vx, T vy, T vz, T* o) {
  o[0] = T(1);
  o[1] = o[0] * vx;
  o[2] = o[0] * vy;
  o[3] = o[0] * vz;
  o[4] = o[1] * (vx * T(0.5));
  o[5] = o[2] * vx;
  o[6] = o[3] * vx;
  o[7] = o[2] * (vy * T(0.5));
  o[8] = o[3] * vy;
  o[9] = o[3] * (vz * T(0.5));
  o[10] = o[4] * (vx * T(0.3333333333333333));
  o[11] = o[5] * (vx * T(0.5));
  o[12] = o[6] * (vx * T(0.5));
  o[13] = o[7] * vx;
  o[14] = o[8] * vx;
  o[15] = o[9] * vx;
  o[16] = o[7] * (vy * T(0.3333333333333333));
  o[17] = o[8] * (vy * T(0.5));
  o[18] = o[9] * vy;
  o[19] = o[9] * (vz * T(0.3333333333333333));
  o[20] = o[10] * (vx * T(0.25));
  o[21] = o[11] * (vx * T(0.3333333333333333));
  o[22] = o[12] * (vx * T(0.3333333333333333));
  o[23] = o[13] * (vx * T(0.5));
  o[24] = o[14] * (vx * T(0.5));
  o[25] = o[15] * (vx * T(0.5));
  o[26] = o[16] * vx;
  o[27] = o[17] * vx;
  o[28] = o[18] * vx;
  o[29] = o[19] * vx;
  o[30] = o[16] * (vy * T(0.25));
  o[31] = o[17] * (vy * T(0.3333333333333333));
  o[32] = o[18] * (vy * T(0.5));
  o[33] = o[19] * vy;
  o[34] = o[19] * (vz * T(0.25));
  o[35] = o[20] * (vx * T(0.2));
  o[36] = o[21] * (vx * T(0.25));
  o[37] = o[22] * (vx * T(0.25));
  o[38] = o[23] * (vx * T(0.3333333333333333));
  o[39] = o[24] * (vx * T(0.3333333333333333));
  o[40] = o[25] * (vx * T(0.3333333333333333));
  o[41] = o[26] * (vx * T(0.5));
  o[42] = o[27] * (vx * T(0.5));
  o[43] = o[28] * (vx * T(0.5));
  o[44] = o[29] * (vx * T(0.5));
  o[45] = o[30] * vx;
  o[46] = o[31] * vx;
  o[47] = o[32] * vx;
  o[48] = o[33] * vx;
  o[49] = o[34] * vx;
  o[50] = o[30] * (vy * T(0.2));
  o[51] = o[31] * (vy * T(0.25));
  o[52] = o[32] * (vy * T(0.3333333333333333));
  o[53] = o[33] * (vy * T(0.5));
  o[54] = o[34] * vy;
  o[55] = o[34] * (vz * T(0.2));
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_1(T ux, T uy, T uz, T rinv, T* D) {
  const T R0_100 = ux * T(-1.0);
  const T R0_010 = uy * T(-1.0);
  const T R0_001 = uz * T(-1.0);
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_2(T ux, T uy, T uz, T rinv, T* D) {
  const T R0_100 = ux * T(-1.0);
  const T R0_010 = uy * T(-1.0);
  const T R0_001 = uz * T(-1.0);
  const T R1_100 = ux * T(3.0);
  const T R0_200 = fma(ux, R1_100, T(1.0) * T(-1.0));
  const T R1_010 = uy * T(3.0);
  const T R0_110 = ux * R1_010;
  const T R1_001 = uz * T(3.0);
  const T R0_101 = ux * R1_001;
  const T R0_020 = fma(uy, R1_010, T(1.0) * T(-1.0));
  const T R0_011 = uy * R1_001;
  const T R0_002 = fma(uz, R1_001, T(1.0) * T(-1.0));
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
  D[9] = R0_002 * s;
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_3(T ux, T uy, T uz, T rinv, T* D) {
  const T R0_100 = ux * T(-1.0);
  const T R0_010 = uy * T(-1.0);
  const T R0_001 = uz * T(-1.0);
  const T R1_100 = ux * T(3.0);
  const T R0_200 = fma(ux, R1_100, T(1.0) * T(-1.0));
  const T R1_010 = uy * T(3.0);
  const T R0_110 = ux * R1_010;
  const T R1_001 = uz * T(3.0);
  const T R0_101 = ux * R1_001;
  const T R0_020 = fma(uy, R1_010, T(1.0) * T(-1.0));
  const T R0_011 = uy * R1_001;
  const T R0_002 = fma(uz, R1_001, T(1.0) * T(-1.0));
  const T R2_100 = ux * T(-15.0);
  const T R1_200 = fma(ux, R2_100, T(1.0) * T(3.0));
  const T R0_300 = fma(ux, R1_200, T(2.0) * R1_100);
  const T R2_010 = uy * T(-15.0);
  const T R1_110 = ux * R2_010;
  const T R0_210 = fma(ux, R1_110, T(1.0) * R1_010);
  const T R2_001 = uz * T(-15.0);
  const T R1_101 = ux * R2_001;
  const T R0_201 = fma(ux, R1_101, T(1.0) * R1_001);
  const T R1_020 = fma(uy, R2_010, T(1.0) * T(3.0));
  const T R0_120 = ux * R1_020;
  const T R1_011 = uy * R2_001;
  const T R0_111 = ux * R1_011;
  const T R1_002 = fma(uz, R2_001, T(1.0) * T(3.0));
  const T R0_102 = ux * R1_002;
  const T R0_030 = fma(uy, R1_020, T(2.0) * R1_010);
  const T R0_021 = fma(uy, R1_011, T(1.0) * R1_001);
  const T R0_012 = uy * R1_002;
  const T R0_003 = fma(uz, R1_002, T(2.0) * R1_001);
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
  D[9] = R0_002 * s;
  s = s * rinv;
  D[10] = R0_300 * s;
  D[11] = R0_210 * s;
  D[12] = R0_201 * s;
  D[13] = R0_120 * s;
  D[14] = R0_111 * s;
  D[15] = R0_102 * s;
  D[16] = R0_030 * s;
  D[17] = R0_021 * s;
  D[18] = R0_012 * s;
  D[19] = R0_003 * s;
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_4(T ux, T uy, T uz, T rinv, T* D) {
  const T R0_100 = ux * T(-1.0);
  const T R0_010 = uy * T(-1.0);
  const T R0_001 = uz * T(-1.0);
  const T R1_100 = ux * T(3.0);
  const T R0_200 = fma(ux, R1_100, T(1.0) * T(-1.0));
  const T R1_010 = uy * T(3.0);
  const T R0_110 = ux * R1_010;
  const T R1_001 = uz * T(3.0);
  const T R0_101 = ux * R1_001;
  const T R0_020 = fma(uy, R1_010, T(1.0) * T(-1.0));
  const T R0_011 = uy * R1_001;
  const T R0_002 = fma(uz, R1_001, T(1.0) * T(-1.0));
  const T R2_100 = ux * T(-15.0);
  const T R1_200 = fma(ux, R2_100, T(1.0) * T(3.0));
  const T R0_300 = fma(ux, R1_200, T(2.0) * R1_100);
  const T R2_010 = uy * T(-15.0);
  const T R1_110 = ux * R2_010;
  const T R0_210 = fma(ux, R1_110, T(1.0) * R1_010);
  const T R2_001 = uz * T(-15.0);
  const T R1_101 = ux * R2_001;
  const T R0_201 = fma(ux, R1_101, T(1.0) * R1_001);
  const T R1_020 = fma(uy, R2_010, T(1.0) * T(3.0));
  const T R0_120 = ux * R1_020;
  const T R1_011 = uy * R2_001;
  const T R0_111 = ux * R1_011;
  const T R1_002 = fma(uz, R2_001, T(1.0) * T(3.0));
  const T R0_102 = ux * R1_002;
  const T R0_030 = fma(uy, R1_020, T(2.0) * R1_010);
  const T R0_021 = fma(uy, R1_011, T(1.0) * R1_001);
  const T R0_012 = uy * R1_002;
  const T R0_003 = fma(uz, R1_002, T(2.0) * R1_001);
  const T R3_100 = ux * T(105.0);
  const T R2_200 = fma(ux, R3_100, T(1.0) * T(-15.0));
  const T R1_300 = fma(ux, R2_200, T(2.0) * R2_100);
  const T R0_400 = fma(ux, R1_300, T(3.0) * R1_200);
  const T R3_010 = uy * T(105.0);
  const T R2_110 = ux * R3_010;
  const T R1_210 = fma(ux, R2_110, T(1.0) * R2_010);
  const T R0_310 = fma(ux, R1_210, T(2.0) * R1_110);
  const T R3_001 = uz * T(105.0);
  const T R2_101 = ux * R3_001;
  const T R1_201 = fma(ux, R2_101, T(1.0) * R2_001);
  const T R0_301 = fma(ux, R1_201, T(2.0) * R1_101);
  const T R2_020 = fma(uy, R3_010, T(1.0) * T(-15.0));
  const T R1_120 = ux * R2_020;
  const T R0_220 = fma(ux, R1_120, T(1.0) * R1_020);
  const T R2_011 = uy * R3_001;
  const T R1_111 = ux * R2_011;
  const T R0_211 = fma(ux, R1_111, T(1.0) * R1_011);
  const T R2_002 = fma(uz, R3_001, T(1.0) * T(-15.0));
  const T R1_102 = ux * R2_002;
  const T R0_202 = fma(ux, R1_102, T(1.0) * R1_002);
  const T R1_030 = fma(uy, R2_020, T(2.0) * R2_010);
  const T R0_130 = ux * R1_030;
  const T R1_021 = fma(uy, R2_011, T(1.0) * R2_001);
  const T R0_121 = ux * R1_021;
  const T R1_012 = uy * R2_002;
  const T R0_112 = ux * R1_012;
  const T R1_003 = fma(uz, R2_002, T(2.0) * R2_001);
  const T R0_103 = ux * R1_003;
  const T R0_040 = fma(uy, R1_030, T(3.0) * R1_020);
  const T R0_031 = fma(uy, R1_021, T(2.0) * R1_011);
  const T R0_022 = fma(uy, R1_012, T(1.0) * R1_002);
  const T R0_013 = uy * R1_003;
  const T R0_004 = fma(uz, R1_003, T(3.0) * R1_002);
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
  D[9] = R0_002 * s;
  s = s * rinv;
  D[10] = R0_300 * s;
  D[11] = R0_210 * s;
  D[12] = R0_201 * s;
  D[13] = R0_120 * s;
  D[14] = R0_111 * s;
  D[15] = R0_102 * s;
  D[16] = R0_030 * s;
  D[17] = R0_021 * s;
  D[18] = R0_012 * s;
  D[19] = R0_003 * s;
  s = s * rinv;
  D[20] = R0_400 * s;
  D[21] = R0_310 * s;
  D[22] = R0_301 * s;
  D[23] = R0_220 * s;
  D[24] = R0_211 * s;
  D[25] = R0_202 * s;
  D[26] = R0_130 * s;
  D[27] = R0_121 * s;
  D[28] = R0_112 * s;
  D[29] = R0_103 * s;
  D[30] = R0_040 * s;
  D[31] = R0_031 * s;
  D[32] = R0_022 * s;
  D[33] = R0_013 * s;
  D[34] = R0_004 * s;
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_5(T ux, T uy, T uz, T rinv, T* D) {
  const T R0_100 = ux * T(-1.0);
  const T R0_010 = uy * T(-1.0);
  const T R0_001 = uz * T(-1.0);
  const T R1_100 = ux * T(3.0);
  const T R0_200 = fma(ux, R1_100, T(1.0) * T(-1.0));
  const T R1_010 = uy * T(3.0);
  const T R0_110 = ux * R1_010;
  const T R1_001 = uz * T(3.0);
  const T R0_101 = ux * R1_001;
  const T R0_020 = fma(uy, R1_010, T(1.0) * T(-1.0));
  const T R0_011 = uy * R1_001;
  const T R0_002 = fma(uz, R1_001, T(1.0) * T(-1.0));
  const T R2_100 = ux * T(-15.0);
  const T R1_200 = fma(ux, R2_100, T(1.0) * T(3.0));
  const T R0_300 = fma(ux, R1_200, T(2.0) * R1_100);
  const T R2_010 = uy * T(-15.0);
  const T R1_110 = ux * R2_010;
  const T R0_210 = fma(ux, R1_110, T(1.0) * R1_010);
  const T R2_001 = uz * T(-15.0);
  const T R1_101 = ux * R2_001;
  const T R0_201 = fma(ux, R1_101, T(1.0) * R1_001);
  const T R1_020 = fma(uy, R2_010, T(1.0) * T(3.0));
  const T R0_120 = ux * R1_020;
  const T R1_011 = uy * R2_001;
  const T R0_111 = ux * R1_011;
  const T R1_002 = fma(uz, R2_001, T(1.0) * T(3.0));
  const T R0_102 = ux * R1_002;
  const T R0_030 = fma(uy, R1_020, T(2.0) * R1_010);
  const T R0_021 = fma(uy, R1_011, T(1.0) * R1_001);
  const T R0_012 = uy * R1_002;
  const T R0_003 = fma(uz, R1_002, T(2.0) * R1_001);
  const T R3_100 = ux * T(105.0);
  const T R2_200 = fma(ux, R3_100, T(1.0) * T(-15.0));
  const T R1_300 = fma(ux, R2_200, T(2.0) * R2_100);
  const T R0_400 = fma(ux, R1_300, T(3.0) * R1_200);
  const T R3_010 = uy * T(105.0);
  const T R2_110 = ux * R3_010;
  const T R1_210 = fma(ux, R2_110, T(1.0) * R2_010);
  const T R0_310 = fma(ux, R1_210, T(2.0) * R1_110);
  const T R3_001 = uz * T(105.0);
  const T R2_101 = ux * R3_001;
  const T R1_201 = fma(ux, R2_101, T(1.0) * R2_001);
  const T R0_301 = fma(ux, R1_201, T(2.0) * R1_101);
  const T R2_020 = fma(uy, R3_010, T(1.0) * T(-15.0));
  const T R1_120 = ux * R2_020;
  const T R0_220 = fma(ux, R1_120, T(1.0) * R1_020);
  const T R2_011 = uy * R3_001;
  const T R1_111 = ux * R2_011;
  const T R0_211 = fma(ux, R1_111, T(1.0) * R1_011);
  const T R2_002 = fma(uz, R3_001, T(1.0) * T(-15.0));
  const T R1_102 = ux * R2_002;
  const T R0_202 = fma(ux, R1_102, T(1.0) * R1_002);
  const T R1_030 = fma(uy, R2_020, T(2.0) * R2_010);
  const T R0_130 = ux * R1_030;
  const T R1_021 = fma(uy, R2_011, T(1.0) * R2_001);
  const T R0_121 = ux * R1_021;
  const T R1_012 = uy * R2_002;
  const T R0_112 = ux * R1_012;
  const T R1_003 = fma(uz, R2_002, T(2.0) * R2_001);
  const T R0_103 = ux * R1_003;
  const T R0_040 = fma(uy, R1_030, T(3.0) * R1_020);
  const T R0_031 = fma(uy, R1_021, T(2.0) * R1_011);
  const T R0_022 = fma(uy, R1_012, T(1.0) * R1_002);
  const T R0_013 = uy * R1_003;
  const T R0_004 = fma(uz, R1_003, T(3.0) * R1_002);
  const T R4_100 = ux * T(-945.0);
  const T R3_200 = fma(ux, R4_100, T(1.0) * T(105.0));
  const T R2_300 = fma(ux, R3_200, T(2.0) * R3_100);
  const T R1_400 = fma(ux, R2_300, T(3.0) * R2_200);
  const T R0_500 = fma(ux, R1_400, T(4.0) * R1_300);
  const T R4_010 = uy * T(-945.0);
  const T R3_110 = ux * R4_010;
  const T R2_210 = fma(ux, R3_110, T(1.0) * R3_010);
  const T R1_310 = fma(ux, R2_210, T(2.0) * R2_110);
  const T R0_410 = fma(ux, R1_310, T(3.0) * R1_210);
  const T R4_001 = uz * T(-945.0);
  const T R3_101 = ux * R4_001;
  const T R2_201 = fma(ux, R3_101, T(1.0) * R3_001);
  const T R1_301 = fma(ux, R2_201, T(2.0) * R2_101);
  const T R0_401 = fma(ux, R1_301, T(3.0) * R1_201);
  const T R3_020 = fma(uy, R4_010, T(1.0) * T(105.0));
  const T R2_120 = ux * R3_020;
  const T R1_220 = fma(ux, R2_120, T(1.0) * R2_020);
  const T R0_320 = fma(ux, R1_220, T(2.0) * R1_120);
  const T R3_011 = uy * R4_001;
  const T R2_111 = ux * R3_011;
  const T R1_211 = fma(ux, R2_111, T(1.0) * R2_011);
  const T R0_311 = fma(ux, R1_211, T(2.0) * R1_111);
  const T R3_002 = fma(uz, R4_001, T(1.0) * T(105.0));
  const T R2_102 = ux * R3_002;
  const T R1_202 = fma(ux, R2_102, T(1.0) * R2_002);
  const T R0_302 = fma(ux, R1_202, T(2.0) * R1_102);
  const T R2_030 = fma(uy, R3_020, T(2.0) * R3_010);
  const T R1_130 = ux * R2_030;
  const T R0_230 = fma(ux, R1_130, T(1.0) * R1_030);
  const T R2_021 = fma(uy, R3_011, T(1.0) * R3_001);
  const T R1_121 = ux * R2_021;
  const T R0_221 = fma(ux, R1_121, T(1.0) * R1_021);
  const T R2_012 = uy * R3_002;
  const T R1_112 = ux * R2_012;
  const T R0_212 = fma(ux, R1_112, T(1.0) * R1_012);
  const T R2_003 = fma(uz, R3_002, T(2.0) * R3_001);
  const T R1_103 = ux * R2_003;
  const T R0_203 = fma(ux, R1_103, T(1.0) * R1_003);
  const T R1_040 = fma(uy, R2_030, T(3.0) * R2_020);
  const T R0_140 = ux * R1_040;
  const T R1_031 = fma(uy, R2_021, T(2.0) * R2_011);
  const T R0_131 = ux * R1_031;
  const T R1_022 = fma(uy, R2_012, T(1.0) * R2_002);
  const T R0_122 = ux * R1_022;
  const T R1_013 = uy * R2_003;
  const T R0_113 = ux * R1_013;
  const T R1_004 = fma(uz, R2_003, T(3.0) * R2_002);
  const T R0_104 = ux * R1_004;
  const T R0_050 = fma(uy, R1_040, T(4.0) * R1_030);
  const T R0_041 = fma(uy, R1_031, T(3.0) * R1_021);
  const T R0_032 = fma(uy, R1_022, T(2.0) * R1_012);
  const T R0_023 = fma(uy, R1_013, T(1.0) * R1_003);
  const T R0_014 = uy * R1_004;
  const T R0_005 = fma(uz, R1_004, T(4.0) * R1_003);
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
  D[9] = R0_002 * s;
  s = s * rinv;
  D[10] = R0_300 * s;
  D[11] = R0_210 * s;
  D[12] = R0_201 * s;
  D[13] = R0_120 * s;
  D[14] = R0_111 * s;
  D[15] = R0_102 * s;
  D[16] = R0_030 * s;
  D[17] = R0_021 * s;
  D[18] = R0_012 * s;
  D[19] = R0_003 * s;
  s = s * rinv;
  D[20] = R0_400 * s;
  D[21] = R0_310 * s;
  D[22] = R0_301 * s;
  D[23] = R0_220 * s;
  D[24] = R0_211 * s;
  D[25] = R0_202 * s;
  D[26] = R0_130 * s;
  D[27] = R0_121 * s;
  D[28] = R0_112 * s;
  D[29] = R0_103 * s;
  D[30] = R0_040 * s;
  D[31] = R0_031 * s;
  D[32] = R0_022 * s;
  D[33] = R0_013 * s;
  D[34] = R0_004 * s;
  s = s * rinv;
  D[35] = R0_500 * s;
  D[36] = R0_410 * s;
  D[37] = R0_401 * s;
  D[38] = R0_320 * s;
  D[39] = R0_311 * s;
  D[40] = R0_302 * s;
  D[41] = R0_230 * s;
  D[42] = R0_221 * s;
  D[43] = R0_212 * s;
  D[44] = R0_203 * s;
  D[45] = R0_140 * s;
  D[46] = R0_131 * s;
  D[47] = R0_122 * s;
  D[48] = R0_113 * s;
  D[49] = R0_104 * s;
  D[50] = R0_050 * s;
  D[51] = R0_041 * s;
  D[52] = R0_032 * s;
  D[53] = R0_023 * s;
  D[54] = R0_014 * s;
  D[55] = R0_005 * s;
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_0(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    C[0] += s; }
  { T s = D[1] * Q[0];
    C[1] -= s; }
  { T s = D[2] * Q[0];
    C[2] -= s; }
  { T s = D[3] * Q[0];
    C[3] -= s; }
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_0_nodip(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    C[0] += s; }
  { T s = D[1] * Q[0];
    C[1] -= s; }
  { T s = D[2] * Q[0];
    C[2] -= s; }
  { T s = D[3] * Q[0];
    C[3] -= s; }
}

template <typename T, typename C_T> __device__ __forceinline__ void sfmm_l2p_0(const T* am, const C_T* C, T* out) {
  T phi = T(0), ax = T(0), ay = T(0), az = T(0);
  phi = fma(am[0], T(C[0]), phi);
  ax = fma(am[0], T(C[1]), ax);
  ay = fma(am[0], T(C[2]), ay);
  az = fma(am[0], T(C[3]), az);
  out[0] = phi; out[1] = ax; out[2] = ay; out[3] = az;
}

template <typename T> __device__ __forceinline__ void sfmm_m2m_0(const T* gm, const T* Qc, T* Qp) {
  { T s = Qp[0];
    s = fma(gm[0], Qc[0], s);
    Qp[0] = s; }
}

#define SFMM_NT_0 1  /* steps of the L2L translation */
static __device__ const unsigned short sfmm_l2l_steps_0[1][32] = {
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static const int sfmm_moment_mi_0[1][3] = {{0,0,0}};

#define SFMM_MT_0 1  /* steps of the M2M translation */
static __device__ const unsigned short sfmm_m2m_steps_0[1][32] = {
  {0, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static __device__ const unsigned short sfmm_moment_exp_0[1] = {0};

template <typename T> __device__ __forceinline__ void sfmm_fold_0(const T* Q, T* q) {
  q[0] = Q[0];
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_fold_0(const T* D, const T* q, T* C) {
  C[0] = fma(D[0], q[0], C[0]);
  C[1] = fma(D[1], q[0], C[1]);
  C[2] = fma(D[2], q[0], C[2]);
  C[3] = fma(D[3], q[0], C[3]);
}

#define SFMM_NR_0 1  /* entries of a source row */
#define SFMM_NS_0 4  /* sums of an interaction */
#define SFMM_NX_0 1
static __device__ const signed char sfmm_unfold_0[4][1][2] = {
  {{0, 1}},
  {{1, -1}},
  {{2, -1}},
  {{3, -1}}};

template <typename T> __device__ __forceinline__ void sfmm_m2l_1(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    s = fma(D[1], Q[1], s);
    s = fma(D[2], Q[2], s);
    s = fma(D[3], Q[3], s);
    C[0] += s; }
  { T s = D[1] * Q[0];
    C[1] -= s; }
  { T s = D[2] * Q[0];
    C[2] -= s; }
  { T s = D[3] * Q[0];
    C[3] -= s; }
  { T s = D[1] * Q[0];
    s = fma(D[4], Q[1], s);
    s = fma(D[5], Q[2], s);
    s = fma(D[6], Q[3], s);
    C[4] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[5], Q[1], s);
    s = fma(D[7], Q[2], s);
    s = fma(D[8], Q[3], s);
    C[5] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[6], Q[1], s);
    s = fma(D[8], Q[2], s);
    s = fma(D[9], Q[3], s);
    C[6] -= s; }
  { T s = D[4] * Q[0];
    C[7] += s; }
  { T s = D[5] * Q[0];
    C[8] += s; }
  { T s = D[6] * Q[0];
    C[9] += s; }
  { T s = D[7] * Q[0];
    C[10] += s; }
  { T s = D[8] * Q[0];
    C[11] += s; }
  { T s = D[9] * Q[0];
    C[12] += s; }
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_1_nodip(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    C[0] += s; }
  { T s = D[1] * Q[0];
    C[1] -= s; }
  { T s = D[2] * Q[0];
    C[2] -= s; }
  { T s = D[3] * Q[0];
    C[3] -= s; }
  { T s = D[1] * Q[0];
    C[4] -= s; }
  { T s = D[2] * Q[0];
    C[5] -= s; }
  { T s = D[3] * Q[0];
    C[6] -= s; }
  { T s = D[4] * Q[0];
    C[7] += s; }
  { T s = D[5] * Q[0];
    C[8] += s; }
  { T s = D[6] * Q[0];
    C[9] += s; }
  { T s = D[7] * Q[0];
    C[10] += s; }
  { T s = D[8] * Q[0];
    C[11] += s; }
  { T s = D[9] * Q[0];
    C[12] += s; }
}

template <typename T, typename C_T> __device__ __forceinline__ void sfmm_l2p_1(const T* am, const C_T* C, T* out) {
  T phi = T(0), ax = T(0), ay = T(0), az = T(0);
  phi = fma(am[0], T(C[0]), phi);
  ax = fma(am[0], T(C[4]), ax);
  ay = fma(am[0], T(C[5]), ay);
  az = fma(am[0], T(C[6]), az);
  phi = fma(am[1], T(C[1]), phi);
  ax = fma(am[1], T(C[7]), ax);
  ay = fma(am[1], T(C[8]), ay);
  az = fma(am[1], T(C[9]), az);
  phi = fma(am[2], T(C[2]), phi);
  ax = fma(am[2], T(C[8]), ax);
  ay = fma(am[2], T(C[10]), ay);
  az = fma(am[2], T(C[11]), az);
  phi = fma(am[3], T(C[3]), phi);
  ax = fma(am[3], T(C[9]), ax);
  ay = fma(am[3], T(C[11]), ay);
  az = fma(am[3], T(C[12]), az);
  out[0] = phi; out[1] = ax; out[2] = ay; out[3] = az;
}

template <typename T> __device__ __forceinline__ void sfmm_m2m_1(const T* gm, const T* Qc, T* Qp) {
  { T s = Qp[0];
    s = fma(gm[0], Qc[0], s);
    Qp[0] = s; }
  { T s = Qp[1];
    s = fma(gm[1], Qc[0], s);
    s = fma(gm[0], Qc[1], s);
    Qp[1] = s; }
  { T s = Qp[2];
    s = fma(gm[2], Qc[0], s);
    s = fma(gm[0], Qc[2], s);
    Qp[2] = s; }
  { T s = Qp[3];
    s = fma(gm[3], Qc[0], s);
    s = fma(gm[0], Qc[3], s);
    Qp[3] = s; }
}

#define SFMM_NT_1 3  /* steps of the L2L translation */
static __device__ const unsigned short sfmm_l2l_steps_1[3][32] = {
  {257, 65535, 65535, 65535, 263, 264, 265, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {514, 65535, 65535, 65535, 520, 522, 523, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {771, 65535, 65535, 65535, 777, 779, 780, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static const int sfmm_moment_mi_1[4][3] = {{0,0,0}, {1,0,0}, {0,1,0}, {0,0,1}};

#define SFMM_MT_1 2  /* steps of the M2M translation */
static __device__ const unsigned short sfmm_m2m_steps_1[2][32] = {
  {0, 1, 2, 3, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 256, 512, 768, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static __device__ const unsigned short sfmm_moment_exp_1[4] = {0, 1, 8, 64};

template <typename T> __device__ __forceinline__ void sfmm_fold_1(const T* Q, T* q) {
  q[0] = Q[0];
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_fold_1(const T* D, const T* q, T* C) {
  C[0] = fma(D[0], q[0], C[0]);
  C[1] = fma(D[1], q[0], C[1]);
  C[2] = fma(D[2], q[0], C[2]);
  C[3] = fma(D[3], q[0], C[3]);
  C[4] = fma(D[4], q[0], C[4]);
  C[5] = fma(D[5], q[0], C[5]);
  C[6] = fma(D[6], q[0], C[6]);
  C[7] = fma(D[7], q[0], C[7]);
  C[8] = fma(D[8], q[0], C[8]);
}

#define SFMM_NR_1 1  /* entries of a source row */
#define SFMM_NS_1 9  /* sums of an interaction */
#define SFMM_NX_1 2
static __device__ const signed char sfmm_unfold_1[13][2][2] = {
  {{0, 1}, {0, 0}},
  {{1, -1}, {0, 0}},
  {{2, -1}, {0, 0}},
  {{3, -1}, {0, 0}},
  {{1, -1}, {0, 0}},
  {{2, -1}, {0, 0}},
  {{3, -1}, {0, 0}},
  {{4, 1}, {0, 0}},
  {{5, 1}, {0, 0}},
  {{6, 1}, {0, 0}},
  {{7, 1}, {0, 0}},
  {{8, 1}, {0, 0}},
  {{4, -1}, {7, -1}}};

template <typename T> __device__ __forceinline__ void sfmm_m2l_2(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    s = fma(D[1], Q[1], s);
    s = fma(D[2], Q[2], s);
    s = fma(D[3], Q[3], s);
    s = fma(D[4], Q[4], s);
    s = fma(D[5], Q[5], s);
    s = fma(D[6], Q[6], s);
    s = fma(D[7], Q[7], s);
    s = fma(D[8], Q[8], s);
    s = fma(D[9], Q[9], s);
    C[0] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[4], Q[1], s);
    s = fma(D[5], Q[2], s);
    s = fma(D[6], Q[3], s);
    C[1] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[5], Q[1], s);
    s = fma(D[7], Q[2], s);
    s = fma(D[8], Q[3], s);
    C[2] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[6], Q[1], s);
    s = fma(D[8], Q[2], s);
    s = fma(D[9], Q[3], s);
    C[3] -= s; }
  { T s = D[4] * Q[0];
    C[4] += s; }
  { T s = D[5] * Q[0];
    C[5] += s; }
  { T s = D[6] * Q[0];
    C[6] += s; }
  { T s = D[7] * Q[0];
    C[7] += s; }
  { T s = D[8] * Q[0];
    C[8] += s; }
  { T s = D[9] * Q[0];
    C[9] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[4], Q[1], s);
    s = fma(D[5], Q[2], s);
    s = fma(D[6], Q[3], s);
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    C[10] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[5], Q[1], s);
    s = fma(D[7], Q[2], s);
    s = fma(D[8], Q[3], s);
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    C[11] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[6], Q[1], s);
    s = fma(D[8], Q[2], s);
    s = fma(D[9], Q[3], s);
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    C[12] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[10], Q[1], s);
    s = fma(D[11], Q[2], s);
    s = fma(D[12], Q[3], s);
    C[13] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[11], Q[1], s);
    s = fma(D[13], Q[2], s);
    s = fma(D[14], Q[3], s);
    C[14] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[12], Q[1], s);
    s = fma(D[14], Q[2], s);
    s = fma(D[15], Q[3], s);
    C[15] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[13], Q[1], s);
    s = fma(D[16], Q[2], s);
    s = fma(D[17], Q[3], s);
    C[16] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[14], Q[1], s);
    s = fma(D[17], Q[2], s);
    s = fma(D[18], Q[3], s);
    C[17] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[15], Q[1], s);
    s = fma(D[18], Q[2], s);
    s = fma(D[19], Q[3], s);
    C[18] += s; }
  { T s = D[10] * Q[0];
    C[19] -= s; }
  { T s = D[11] * Q[0];
    C[20] -= s; }
  { T s = D[12] * Q[0];
    C[21] -= s; }
  { T s = D[13] * Q[0];
    C[22] -= s; }
  { T s = D[14] * Q[0];
    C[23] -= s; }
  { T s = D[15] * Q[0];
    C[24] -= s; }
  { T s = D[16] * Q[0];
    C[25] -= s; }
  { T s = D[17] * Q[0];
    C[26] -= s; }
  { T s = D[18] * Q[0];
    C[27] -= s; }
  { T s = D[19] * Q[0];
    C[28] -= s; }
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_2_nodip(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    s = fma(D[4], Q[4], s);
    s = fma(D[5], Q[5], s);
    s = fma(D[6], Q[6], s);
    s = fma(D[7], Q[7], s);
    s = fma(D[8], Q[8], s);
    s = fma(D[9], Q[9], s);
    C[0] += s; }
  { T s = D[1] * Q[0];
    C[1] -= s; }
  { T s = D[2] * Q[0];
    C[2] -= s; }
  { T s = D[3] * Q[0];
    C[3] -= s; }
  { T s = D[4] * Q[0];
    C[4] += s; }
  { T s = D[5] * Q[0];
    C[5] += s; }
  { T s = D[6] * Q[0];
    C[6] += s; }
  { T s = D[7] * Q[0];
    C[7] += s; }
  { T s = D[8] * Q[0];
    C[8] += s; }
  { T s = D[9] * Q[0];
    C[9] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    C[10] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    C[11] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    C[12] -= s; }
  { T s = D[4] * Q[0];
    C[13] += s; }
  { T s = D[5] * Q[0];
    C[14] += s; }
  { T s = D[6] * Q[0];
    C[15] += s; }
  { T s = D[7] * Q[0];
    C[16] += s; }
  { T s = D[8] * Q[0];
    C[17] += s; }
  { T s = D[9] * Q[0];
    C[18] += s; }
  { T s = D[10] * Q[0];
    C[19] -= s; }
  { T s = D[11] * Q[0];
    C[20] -= s; }
  { T s = D[12] * Q[0];
    C[21] -= s; }
  { T s = D[13] * Q[0];
    C[22] -= s; }
  { T s = D[14] * Q[0];
    C[23] -= s; }
  { T s = D[15] * Q[0];
    C[24] -= s; }
  { T s = D[16] * Q[0];
    C[25] -= s; }
  { T s = D[17] * Q[0];
    C[26] -= s; }
  { T s = D[18] * Q[0];
    C[27] -= s; }
  { T s = D[19] * Q[0];
    C[28] -= s; }
}

template <typename T, typename C_T> __device__ __forceinline__ void sfmm_l2p_2(const T* am, const C_T* C, T* out) {
  T phi = T(0), ax = T(0), ay = T(0), az = T(0);
  phi = fma(am[0], T(C[0]), phi);
  ax = fma(am[0], T(C[10]), ax);
  ay = fma(am[0], T(C[11]), ay);
  az = fma(am[0], T(C[12]), az);
  phi = fma(am[1], T(C[1]), phi);
  ax = fma(am[1], T(C[13]), ax);
  ay = fma(am[1], T(C[14]), ay);
  az = fma(am[1], T(C[15]), az);
  phi = fma(am[2], T(C[2]), phi);
  ax = fma(am[2], T(C[14]), ax);
  ay = fma(am[2], T(C[16]), ay);
  az = fma(am[2], T(C[17]), az);
  phi = fma(am[3], T(C[3]), phi);
  ax = fma(am[3], T(C[15]), ax);
  ay = fma(am[3], T(C[17]), ay);
  az = fma(am[3], T(C[18]), az);
  phi = fma(am[4], T(C[4]), phi);
  ax = fma(am[4], T(C[19]), ax);
  ay = fma(am[4], T(C[20]), ay);
  az = fma(am[4], T(C[21]), az);
  phi = fma(am[5], T(C[5]), phi);
  ax = fma(am[5], T(C[20]), ax);
  ay = fma(am[5], T(C[22]), ay);
  az = fma(am[5], T(C[23]), az);
  phi = fma(am[6], T(C[6]), phi);
  ax = fma(am[6], T(C[21]), ax);
  ay = fma(am[6], T(C[23]), ay);
  az = fma(am[6], T(C[24]), az);
  phi = fma(am[7], T(C[7]), phi);
  ax = fma(am[7], T(C[22]), ax);
  ay = fma(am[7], T(C[25]), ay);
  az = fma(am[7], T(C[26]), az);
  phi = fma(am[8], T(C[8]), phi);
  ax = fma(am[8], T(C[23]), ax);
  ay = fma(am[8], T(C[26]), ay);
  az = fma(am[8], T(C[27]), az);
  phi = fma(am[9], T(C[9]), phi);
  ax = fma(am[9], T(C[24]), ax);
  ay = fma(am[9], T(C[27]), ay);
  az = fma(am[9], T(C[28]), az);
  out[0] = phi; out[1] = ax; out[2] = ay; out[3] = az;
}

template <typename T> __device__ __forceinline__ void sfmm_m2m_2(const T* gm, const T* Qc, T* Qp) {
  { T s = Qp[0];
    s = fma(gm[0], Qc[0], s);
    Qp[0] = s; }
  { T s = Qp[1];
    s = fma(gm[1], Qc[0], s);
    s = fma(gm[0], Qc[1], s);
    Qp[1] = s; }
  { T s = Qp[2];
    s = fma(gm[2], Qc[0], s);
    s = fma(gm[0], Qc[2], s);
    Qp[2] = s; }
  { T s = Qp[3];
    s = fma(gm[3], Qc[0], s);
    s = fma(gm[0], Qc[3], s);
    Qp[3] = s; }
  { T s = Qp[4];
    s = fma(gm[4], Qc[0], s);
    s = fma(gm[1], Qc[1], s);
    s = fma(gm[0], Qc[4], s);
    Qp[4] = s; }
  { T s = Qp[5];
    s = fma(gm[5], Qc[0], s);
    s = fma(gm[2], Qc[1], s);
    s = fma(gm[1], Qc[2], s);
    s = fma(gm[0], Qc[5], s);
    Qp[5] = s; }
  { T s = Qp[6];
    s = fma(gm[6], Qc[0], s);
    s = fma(gm[3], Qc[1], s);
    s = fma(gm[1], Qc[3], s);
    s = fma(gm[0], Qc[6], s);
    Qp[6] = s; }
  { T s = Qp[7];
    s = fma(gm[7], Qc[0], s);
    s = fma(gm[2], Qc[2], s);
    s = fma(gm[0], Qc[7], s);
    Qp[7] = s; }
  { T s = Qp[8];
    s = fma(gm[8], Qc[0], s);
    s = fma(gm[3], Qc[2], s);
    s = fma(gm[2], Qc[3], s);
    s = fma(gm[0], Qc[8], s);
    Qp[8] = s; }
  { T s = Qp[9];
    s = fma(gm[9], Qc[0], s);
    s = fma(gm[3], Qc[3], s);
    s = fma(gm[0], Qc[9], s);
    Qp[9] = s; }
}

#define SFMM_NT_2 9  /* steps of the L2L translation */
static __device__ const unsigned short sfmm_l2l_steps_2[9][32] = {
  {257, 260, 261, 262, 65535, 65535, 65535, 65535, 65535, 65535, 269, 270, 271, 275, 276, 277, 278, 279, 280, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {514, 517, 519, 520, 65535, 65535, 65535, 65535, 65535, 65535, 526, 528, 529, 532, 534, 535, 537, 538, 539, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {771, 774, 776, 777, 65535, 65535, 65535, 65535, 65535, 65535, 783, 785, 786, 789, 791, 792, 794, 795, 796, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1028, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1043, 1044, 1045, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1285, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1300, 1302, 1303, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1542, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1557, 1559, 1560, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1799, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1814, 1817, 1818, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2056, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2071, 2074, 2075, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2313, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2328, 2331, 2332, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static const int sfmm_moment_mi_2[10][3] = {{0,0,0}, {1,0,0}, {0,1,0}, {0,0,1}, {2,0,0}, {1,1,0}, {1,0,1}, {0,2,0}, {0,1,1}, {0,0,2}};

#define SFMM_MT_2 4  /* steps of the M2M translation */
static __device__ const unsigned short sfmm_m2m_steps_2[4][32] = {
  {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 256, 512, 768, 257, 258, 259, 514, 515, 771, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 1024, 513, 769, 1792, 770, 2304, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 1280, 1536, 65535, 2048, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static __device__ const unsigned short sfmm_moment_exp_2[10] = {0, 1, 8, 64, 2, 9, 65, 16, 72, 128};

template <typename T> __device__ __forceinline__ void sfmm_fold_2(const T* Q, T* q) {
  q[0] = Q[0];
  q[1] = Q[4] - Q[9];
  q[2] = Q[5];
  q[3] = Q[6];
  q[4] = Q[7] - Q[9];
  q[5] = Q[8];
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_fold_2(const T* D, const T* q, T* C) {
  { T s = D[4] * q[1];
    s = fma(D[5], q[2], s);
    s = fma(D[6], q[3], s);
    s = fma(D[7], q[4], s);
    s = fma(D[8], q[5], s);
    C[0] += fma(D[0], q[0], s); }
  C[1] = fma(D[1], q[0], C[1]);
  C[2] = fma(D[2], q[0], C[2]);
  C[3] = fma(D[3], q[0], C[3]);
  C[4] = fma(D[4], q[0], C[4]);
  C[5] = fma(D[5], q[0], C[5]);
  C[6] = fma(D[6], q[0], C[6]);
  C[7] = fma(D[7], q[0], C[7]);
  C[8] = fma(D[8], q[0], C[8]);
  C[9] = fma(D[10], q[1], C[9]);
  C[9] = fma(D[11], q[2], C[9]);
  C[9] = fma(D[12], q[3], C[9]);
  C[9] = fma(D[13], q[4], C[9]);
  C[9] = fma(D[14], q[5], C[9]);
  C[10] = fma(D[11], q[1], C[10]);
  C[10] = fma(D[13], q[2], C[10]);
  C[10] = fma(D[14], q[3], C[10]);
  C[10] = fma(D[16], q[4], C[10]);
  C[10] = fma(D[17], q[5], C[10]);
  C[11] = fma(D[12], q[1], C[11]);
  C[11] = fma(D[14], q[2], C[11]);
  C[11] = fma(D[15], q[3], C[11]);
  C[11] = fma(D[17], q[4], C[11]);
  C[11] = fma(D[18], q[5], C[11]);
  C[12] = fma(D[10], q[0], C[12]);
  C[13] = fma(D[11], q[0], C[13]);
  C[14] = fma(D[12], q[0], C[14]);
  C[15] = fma(D[13], q[0], C[15]);
  C[16] = fma(D[14], q[0], C[16]);
  C[17] = fma(D[16], q[0], C[17]);
  C[18] = fma(D[17], q[0], C[18]);
}

#define SFMM_NR_2 6  /* entries of a source row */
#define SFMM_NS_2 19  /* sums of an interaction */
#define SFMM_NX_2 2
static __device__ const signed char sfmm_unfold_2[29][2][2] = {
  {{0, 1}, {0, 0}},
  {{1, -1}, {0, 0}},
  {{2, -1}, {0, 0}},
  {{3, -1}, {0, 0}},
  {{4, 1}, {0, 0}},
  {{5, 1}, {0, 0}},
  {{6, 1}, {0, 0}},
  {{7, 1}, {0, 0}},
  {{8, 1}, {0, 0}},
  {{4, -1}, {7, -1}},
  {{1, -1}, {9, -1}},
  {{2, -1}, {10, -1}},
  {{3, -1}, {11, -1}},
  {{4, 1}, {0, 0}},
  {{5, 1}, {0, 0}},
  {{6, 1}, {0, 0}},
  {{7, 1}, {0, 0}},
  {{8, 1}, {0, 0}},
  {{4, -1}, {7, -1}},
  {{12, -1}, {0, 0}},
  {{13, -1}, {0, 0}},
  {{14, -1}, {0, 0}},
  {{15, -1}, {0, 0}},
  {{16, -1}, {0, 0}},
  {{12, 1}, {15, 1}},
  {{17, -1}, {0, 0}},
  {{18, -1}, {0, 0}},
  {{13, 1}, {17, 1}},
  {{14, 1}, {18, 1}}};

template <typename T> __device__ __forceinline__ void sfmm_m2l_3(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    s = fma(D[1], Q[1], s);
    s = fma(D[2], Q[2], s);
    s = fma(D[3], Q[3], s);
    s = fma(D[4], Q[4], s);
    s = fma(D[5], Q[5], s);
    s = fma(D[6], Q[6], s);
    s = fma(D[7], Q[7], s);
    s = fma(D[8], Q[8], s);
    s = fma(D[9], Q[9], s);
    s = fma(D[10], Q[10], s);
    s = fma(D[11], Q[11], s);
    s = fma(D[12], Q[12], s);
    s = fma(D[13], Q[13], s);
    s = fma(D[14], Q[14], s);
    s = fma(D[15], Q[15], s);
    s = fma(D[16], Q[16], s);
    s = fma(D[17], Q[17], s);
    s = fma(D[18], Q[18], s);
    s = fma(D[19], Q[19], s);
    C[0] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[4], Q[1], s);
    s = fma(D[5], Q[2], s);
    s = fma(D[6], Q[3], s);
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    C[1] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[5], Q[1], s);
    s = fma(D[7], Q[2], s);
    s = fma(D[8], Q[3], s);
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    C[2] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[6], Q[1], s);
    s = fma(D[8], Q[2], s);
    s = fma(D[9], Q[3], s);
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    C[3] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[10], Q[1], s);
    s = fma(D[11], Q[2], s);
    s = fma(D[12], Q[3], s);
    C[4] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[11], Q[1], s);
    s = fma(D[13], Q[2], s);
    s = fma(D[14], Q[3], s);
    C[5] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[12], Q[1], s);
    s = fma(D[14], Q[2], s);
    s = fma(D[15], Q[3], s);
    C[6] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[13], Q[1], s);
    s = fma(D[16], Q[2], s);
    s = fma(D[17], Q[3], s);
    C[7] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[14], Q[1], s);
    s = fma(D[17], Q[2], s);
    s = fma(D[18], Q[3], s);
    C[8] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[15], Q[1], s);
    s = fma(D[18], Q[2], s);
    s = fma(D[19], Q[3], s);
    C[9] += s; }
  { T s = D[10] * Q[0];
    C[10] -= s; }
  { T s = D[11] * Q[0];
    C[11] -= s; }
  { T s = D[12] * Q[0];
    C[12] -= s; }
  { T s = D[13] * Q[0];
    C[13] -= s; }
  { T s = D[14] * Q[0];
    C[14] -= s; }
  { T s = D[15] * Q[0];
    C[15] -= s; }
  { T s = D[16] * Q[0];
    C[16] -= s; }
  { T s = D[17] * Q[0];
    C[17] -= s; }
  { T s = D[18] * Q[0];
    C[18] -= s; }
  { T s = D[19] * Q[0];
    C[19] -= s; }
  { T s = D[1] * Q[0];
    s = fma(D[4], Q[1], s);
    s = fma(D[5], Q[2], s);
    s = fma(D[6], Q[3], s);
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    s = fma(D[20], Q[10], s);
    s = fma(D[21], Q[11], s);
    s = fma(D[22], Q[12], s);
    s = fma(D[23], Q[13], s);
    s = fma(D[24], Q[14], s);
    s = fma(D[25], Q[15], s);
    s = fma(D[26], Q[16], s);
    s = fma(D[27], Q[17], s);
    s = fma(D[28], Q[18], s);
    s = fma(D[29], Q[19], s);
    C[20] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[5], Q[1], s);
    s = fma(D[7], Q[2], s);
    s = fma(D[8], Q[3], s);
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    s = fma(D[21], Q[10], s);
    s = fma(D[23], Q[11], s);
    s = fma(D[24], Q[12], s);
    s = fma(D[26], Q[13], s);
    s = fma(D[27], Q[14], s);
    s = fma(D[28], Q[15], s);
    s = fma(D[30], Q[16], s);
    s = fma(D[31], Q[17], s);
    s = fma(D[32], Q[18], s);
    s = fma(D[33], Q[19], s);
    C[21] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[6], Q[1], s);
    s = fma(D[8], Q[2], s);
    s = fma(D[9], Q[3], s);
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    s = fma(D[22], Q[10], s);
    s = fma(D[24], Q[11], s);
    s = fma(D[25], Q[12], s);
    s = fma(D[27], Q[13], s);
    s = fma(D[28], Q[14], s);
    s = fma(D[29], Q[15], s);
    s = fma(D[31], Q[16], s);
    s = fma(D[32], Q[17], s);
    s = fma(D[33], Q[18], s);
    s = fma(D[34], Q[19], s);
    C[22] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[10], Q[1], s);
    s = fma(D[11], Q[2], s);
    s = fma(D[12], Q[3], s);
    s = fma(D[20], Q[4], s);
    s = fma(D[21], Q[5], s);
    s = fma(D[22], Q[6], s);
    s = fma(D[23], Q[7], s);
    s = fma(D[24], Q[8], s);
    s = fma(D[25], Q[9], s);
    C[23] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[11], Q[1], s);
    s = fma(D[13], Q[2], s);
    s = fma(D[14], Q[3], s);
    s = fma(D[21], Q[4], s);
    s = fma(D[23], Q[5], s);
    s = fma(D[24], Q[6], s);
    s = fma(D[26], Q[7], s);
    s = fma(D[27], Q[8], s);
    s = fma(D[28], Q[9], s);
    C[24] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[12], Q[1], s);
    s = fma(D[14], Q[2], s);
    s = fma(D[15], Q[3], s);
    s = fma(D[22], Q[4], s);
    s = fma(D[24], Q[5], s);
    s = fma(D[25], Q[6], s);
    s = fma(D[27], Q[7], s);
    s = fma(D[28], Q[8], s);
    s = fma(D[29], Q[9], s);
    C[25] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[13], Q[1], s);
    s = fma(D[16], Q[2], s);
    s = fma(D[17], Q[3], s);
    s = fma(D[23], Q[4], s);
    s = fma(D[26], Q[5], s);
    s = fma(D[27], Q[6], s);
    s = fma(D[30], Q[7], s);
    s = fma(D[31], Q[8], s);
    s = fma(D[32], Q[9], s);
    C[26] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[14], Q[1], s);
    s = fma(D[17], Q[2], s);
    s = fma(D[18], Q[3], s);
    s = fma(D[24], Q[4], s);
    s = fma(D[27], Q[5], s);
    s = fma(D[28], Q[6], s);
    s = fma(D[31], Q[7], s);
    s = fma(D[32], Q[8], s);
    s = fma(D[33], Q[9], s);
    C[27] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[15], Q[1], s);
    s = fma(D[18], Q[2], s);
    s = fma(D[19], Q[3], s);
    s = fma(D[25], Q[4], s);
    s = fma(D[28], Q[5], s);
    s = fma(D[29], Q[6], s);
    s = fma(D[32], Q[7], s);
    s = fma(D[33], Q[8], s);
    s = fma(D[34], Q[9], s);
    C[28] += s; }
  { T s = D[10] * Q[0];
    s = fma(D[20], Q[1], s);
    s = fma(D[21], Q[2], s);
    s = fma(D[22], Q[3], s);
    C[29] -= s; }
  { T s = D[11] * Q[0];
    s = fma(D[21], Q[1], s);
    s = fma(D[23], Q[2], s);
    s = fma(D[24], Q[3], s);
    C[30] -= s; }
  { T s = D[12] * Q[0];
    s = fma(D[22], Q[1], s);
    s = fma(D[24], Q[2], s);
    s = fma(D[25], Q[3], s);
    C[31] -= s; }
  { T s = D[13] * Q[0];
    s = fma(D[23], Q[1], s);
    s = fma(D[26], Q[2], s);
    s = fma(D[27], Q[3], s);
    C[32] -= s; }
  { T s = D[14] * Q[0];
    s = fma(D[24], Q[1], s);
    s = fma(D[27], Q[2], s);
    s = fma(D[28], Q[3], s);
    C[33] -= s; }
  { T s = D[15] * Q[0];
    s = fma(D[25], Q[1], s);
    s = fma(D[28], Q[2], s);
    s = fma(D[29], Q[3], s);
    C[34] -= s; }
  { T s = D[16] * Q[0];
    s = fma(D[26], Q[1], s);
    s = fma(D[30], Q[2], s);
    s = fma(D[31], Q[3], s);
    C[35] -= s; }
  { T s = D[17] * Q[0];
    s = fma(D[27], Q[1], s);
    s = fma(D[31], Q[2], s);
    s = fma(D[32], Q[3], s);
    C[36] -= s; }
  { T s = D[18] * Q[0];
    s = fma(D[28], Q[1], s);
    s = fma(D[32], Q[2], s);
    s = fma(D[33], Q[3], s);
    C[37] -= s; }
  { T s = D[19] * Q[0];
    s = fma(D[29], Q[1], s);
    s = fma(D[33], Q[2], s);
    s = fma(D[34], Q[3], s);
    C[38] -= s; }
  { T s = D[20] * Q[0];
    C[39] += s; }
  { T s = D[21] * Q[0];
    C[40] += s; }
  { T s = D[22] * Q[0];
    C[41] += s; }
  { T s = D[23] * Q[0];
    C[42] += s; }
  { T s = D[24] * Q[0];
    C[43] += s; }
  { T s = D[25] * Q[0];
    C[44] += s; }
  { T s = D[26] * Q[0];
    C[45] += s; }
  { T s = D[27] * Q[0];
    C[46] += s; }
  { T s = D[28] * Q[0];
    C[47] += s; }
  { T s = D[29] * Q[0];
    C[48] += s; }
  { T s = D[30] * Q[0];
    C[49] += s; }
  { T s = D[31] * Q[0];
    C[50] += s; }
  { T s = D[32] * Q[0];
    C[51] += s; }
  { T s = D[33] * Q[0];
    C[52] += s; }
  { T s = D[34] * Q[0];
    C[53] += s; }
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_3_nodip(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    s = fma(D[4], Q[4], s);
    s = fma(D[5], Q[5], s);
    s = fma(D[6], Q[6], s);
    s = fma(D[7], Q[7], s);
    s = fma(D[8], Q[8], s);
    s = fma(D[9], Q[9], s);
    s = fma(D[10], Q[10], s);
    s = fma(D[11], Q[11], s);
    s = fma(D[12], Q[12], s);
    s = fma(D[13], Q[13], s);
    s = fma(D[14], Q[14], s);
    s = fma(D[15], Q[15], s);
    s = fma(D[16], Q[16], s);
    s = fma(D[17], Q[17], s);
    s = fma(D[18], Q[18], s);
    s = fma(D[19], Q[19], s);
    C[0] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    C[1] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    C[2] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    C[3] -= s; }
  { T s = D[4] * Q[0];
    C[4] += s; }
  { T s = D[5] * Q[0];
    C[5] += s; }
  { T s = D[6] * Q[0];
    C[6] += s; }
  { T s = D[7] * Q[0];
    C[7] += s; }
  { T s = D[8] * Q[0];
    C[8] += s; }
  { T s = D[9] * Q[0];
    C[9] += s; }
  { T s = D[10] * Q[0];
    C[10] -= s; }
  { T s = D[11] * Q[0];
    C[11] -= s; }
  { T s = D[12] * Q[0];
    C[12] -= s; }
  { T s = D[13] * Q[0];
    C[13] -= s; }
  { T s = D[14] * Q[0];
    C[14] -= s; }
  { T s = D[15] * Q[0];
    C[15] -= s; }
  { T s = D[16] * Q[0];
    C[16] -= s; }
  { T s = D[17] * Q[0];
    C[17] -= s; }
  { T s = D[18] * Q[0];
    C[18] -= s; }
  { T s = D[19] * Q[0];
    C[19] -= s; }
  { T s = D[1] * Q[0];
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    s = fma(D[20], Q[10], s);
    s = fma(D[21], Q[11], s);
    s = fma(D[22], Q[12], s);
    s = fma(D[23], Q[13], s);
    s = fma(D[24], Q[14], s);
    s = fma(D[25], Q[15], s);
    s = fma(D[26], Q[16], s);
    s = fma(D[27], Q[17], s);
    s = fma(D[28], Q[18], s);
    s = fma(D[29], Q[19], s);
    C[20] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    s = fma(D[21], Q[10], s);
    s = fma(D[23], Q[11], s);
    s = fma(D[24], Q[12], s);
    s = fma(D[26], Q[13], s);
    s = fma(D[27], Q[14], s);
    s = fma(D[28], Q[15], s);
    s = fma(D[30], Q[16], s);
    s = fma(D[31], Q[17], s);
    s = fma(D[32], Q[18], s);
    s = fma(D[33], Q[19], s);
    C[21] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    s = fma(D[22], Q[10], s);
    s = fma(D[24], Q[11], s);
    s = fma(D[25], Q[12], s);
    s = fma(D[27], Q[13], s);
    s = fma(D[28], Q[14], s);
    s = fma(D[29], Q[15], s);
    s = fma(D[31], Q[16], s);
    s = fma(D[32], Q[17], s);
    s = fma(D[33], Q[18], s);
    s = fma(D[34], Q[19], s);
    C[22] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[20], Q[4], s);
    s = fma(D[21], Q[5], s);
    s = fma(D[22], Q[6], s);
    s = fma(D[23], Q[7], s);
    s = fma(D[24], Q[8], s);
    s = fma(D[25], Q[9], s);
    C[23] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[21], Q[4], s);
    s = fma(D[23], Q[5], s);
    s = fma(D[24], Q[6], s);
    s = fma(D[26], Q[7], s);
    s = fma(D[27], Q[8], s);
    s = fma(D[28], Q[9], s);
    C[24] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[22], Q[4], s);
    s = fma(D[24], Q[5], s);
    s = fma(D[25], Q[6], s);
    s = fma(D[27], Q[7], s);
    s = fma(D[28], Q[8], s);
    s = fma(D[29], Q[9], s);
    C[25] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[23], Q[4], s);
    s = fma(D[26], Q[5], s);
    s = fma(D[27], Q[6], s);
    s = fma(D[30], Q[7], s);
    s = fma(D[31], Q[8], s);
    s = fma(D[32], Q[9], s);
    C[26] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[24], Q[4], s);
    s = fma(D[27], Q[5], s);
    s = fma(D[28], Q[6], s);
    s = fma(D[31], Q[7], s);
    s = fma(D[32], Q[8], s);
    s = fma(D[33], Q[9], s);
    C[27] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[25], Q[4], s);
    s = fma(D[28], Q[5], s);
    s = fma(D[29], Q[6], s);
    s = fma(D[32], Q[7], s);
    s = fma(D[33], Q[8], s);
    s = fma(D[34], Q[9], s);
    C[28] += s; }
  { T s = D[10] * Q[0];
    C[29] -= s; }
  { T s = D[11] * Q[0];
    C[30] -= s; }
  { T s = D[12] * Q[0];
    C[31] -= s; }
  { T s = D[13] * Q[0];
    C[32] -= s; }
  { T s = D[14] * Q[0];
    C[33] -= s; }
  { T s = D[15] * Q[0];
    C[34] -= s; }
  { T s = D[16] * Q[0];
    C[35] -= s; }
  { T s = D[17] * Q[0];
    C[36] -= s; }
  { T s = D[18] * Q[0];
    C[37] -= s; }
  { T s = D[19] * Q[0];
    C[38] -= s; }
  { T s = D[20] * Q[0];
    C[39] += s; }
  { T s = D[21] * Q[0];
    C[40] += s; }
  { T s = D[22] * Q[0];
    C[41] += s; }
  { T s = D[23] * Q[0];
    C[42] += s; }
  { T s = D[24] * Q[0];
    C[43] += s; }
  { T s = D[25] * Q[0];
    C[44] += s; }
  { T s = D[26] * Q[0];
    C[45] += s; }
  { T s = D[27] * Q[0];
    C[46] += s; }
  { T s = D[28] * Q[0];
    C[47] += s; }
  { T s = D[29] * Q[0];
    C[48] += s; }
  { T s = D[30] * Q[0];
    C[49] += s; }
  { T s = D[31] * Q[0];
    C[50] += s; }
  { T s = D[32] * Q[0];
    C[51] += s; }
  { T s = D[33] * Q[0];
    C[52] += s; }
  { T s = D[34] * Q[0];
    C[53] += s; }
}

template <typename T, typename C_T> __device__ __forceinline__ void sfmm_l2p_3(const T* am, const C_T* C, T* out) {
  T phi = T(0), ax = T(0), ay = T(0), az = T(0);
  phi = fma(am[0], T(C[0]), phi);
  ax = fma(am[0], T(C[20]), ax);
  ay = fma(am[0], T(C[21]), ay);
  az = fma(am[0], T(C[22]), az);
  phi = fma(am[1], T(C[1]), phi);
  ax = fma(am[1], T(C[23]), ax);
  ay = fma(am[1], T(C[24]), ay);
  az = fma(am[1], T(C[25]), az);
  phi = fma(am[2], T(C[2]), phi);
  ax = fma(am[2], T(C[24]), ax);
  ay = fma(am[2], T(C[26]), ay);
  az = fma(am[2], T(C[27]), az);
  phi = fma(am[3], T(C[3]), phi);
  ax = fma(am[3], T(C[25]), ax);
  ay = fma(am[3], T(C[27]), ay);
  az = fma(am[3], T(C[28]), az);
  phi = fma(am[4], T(C[4]), phi);
  ax = fma(am[4], T(C[29]), ax);
  ay = fma(am[4], T(C[30]), ay);
  az = fma(am[4], T(C[31]), az);
  phi = fma(am[5], T(C[5]), phi);
  ax = fma(am[5], T(C[30]), ax);
  ay = fma(am[5], T(C[32]), ay);
  az = fma(am[5], T(C[33]), az);
  phi = fma(am[6], T(C[6]), phi);
  ax = fma(am[6], T(C[31]), ax);
  ay = fma(am[6], T(C[33]), ay);
  az = fma(am[6], T(C[34]), az);
  phi = fma(am[7], T(C[7]), phi);
  ax = fma(am[7], T(C[32]), ax);
  ay = fma(am[7], T(C[35]), ay);
  az = fma(am[7], T(C[36]), az);
  phi = fma(am[8], T(C[8]), phi);
  ax = fma(am[8], T(C[33]), ax);
  ay = fma(am[8], T(C[36]), ay);
  az = fma(am[8], T(C[37]), az);
  phi = fma(am[9], T(C[9]), phi);
  ax = fma(am[9], T(C[34]), ax);
  ay = fma(am[9], T(C[37]), ay);
  az = fma(am[9], T(C[38]), az);
  phi = fma(am[10], T(C[10]), phi);
  ax = fma(am[10], T(C[39]), ax);
  ay = fma(am[10], T(C[40]), ay);
  az = fma(am[10], T(C[41]), az);
  phi = fma(am[11], T(C[11]), phi);
  ax = fma(am[11], T(C[40]), ax);
  ay = fma(am[11], T(C[42]), ay);
  az = fma(am[11], T(C[43]), az);
  phi = fma(am[12], T(C[12]), phi);
  ax = fma(am[12], T(C[41]), ax);
  ay = fma(am[12], T(C[43]), ay);
  az = fma(am[12], T(C[44]), az);
  phi = fma(am[13], T(C[13]), phi);
  ax = fma(am[13], T(C[42]), ax);
  ay = fma(am[13], T(C[45]), ay);
  az = fma(am[13], T(C[46]), az);
  phi = fma(am[14], T(C[14]), phi);
  ax = fma(am[14], T(C[43]), ax);
  ay = fma(am[14], T(C[46]), ay);
  az = fma(am[14], T(C[47]), az);
  phi = fma(am[15], T(C[15]), phi);
  ax = fma(am[15], T(C[44]), ax);
  ay = fma(am[15], T(C[47]), ay);
  az = fma(am[15], T(C[48]), az);
  phi = fma(am[16], T(C[16]), phi);
  ax = fma(am[16], T(C[45]), ax);
  ay = fma(am[16], T(C[49]), ay);
  az = fma(am[16], T(C[50]), az);
  phi = fma(am[17], T(C[17]), phi);
  ax = fma(am[17], T(C[46]), ax);
  ay = fma(am[17], T(C[50]), ay);
  az = fma(am[17], T(C[51]), az);
  phi = fma(am[18], T(C[18]), phi);
  ax = fma(am[18], T(C[47]), ax);
  ay = fma(am[18], T(C[51]), ay);
  az = fma(am[18], T(C[52]), az);
  phi = fma(am[19], T(C[19]), phi);
  ax = fma(am[19], T(C[48]), ax);
  ay = fma(am[19], T(C[52]), ay);
  az = fma(am[19], T(C[53]), az);
  out[0] = phi; out[1] = ax; out[2] = ay; out[3] = az;
}

template <typename T> __device__ __forceinline__ void sfmm_m2m_3(const T* gm, const T* Qc, T* Qp) {
  { T s = Qp[0];
    s = fma(gm[0], Qc[0], s);
    Qp[0] = s; }
  { T s = Qp[1];
    s = fma(gm[1], Qc[0], s);
    s = fma(gm[0], Qc[1], s);
    Qp[1] = s; }
  { T s = Qp[2];
    s = fma(gm[2], Qc[0], s);
    s = fma(gm[0], Qc[2], s);
    Qp[2] = s; }
  { T s = Qp[3];
    s = fma(gm[3], Qc[0], s);
    s = fma(gm[0], Qc[3], s);
    Qp[3] = s; }
  { T s = Qp[4];
    s = fma(gm[4], Qc[0], s);
    s = fma(gm[1], Qc[1], s);
    s = fma(gm[0], Qc[4], s);
    Qp[4] = s; }
  { T s = Qp[5];
    s = fma(gm[5], Qc[0], s);
    s = fma(gm[2], Qc[1], s);
    s = fma(gm[1], Qc[2], s);
    s = fma(gm[0], Qc[5], s);
    Qp[5] = s; }
  { T s = Qp[6];
    s = fma(gm[6], Qc[0], s);
    s = fma(gm[3], Qc[1], s);
    s = fma(gm[1], Qc[3], s);
    s = fma(gm[0], Qc[6], s);
    Qp[6] = s; }
  { T s = Qp[7];
    s = fma(gm[7], Qc[0], s);
    s = fma(gm[2], Qc[2], s);
    s = fma(gm[0], Qc[7], s);
    Qp[7] = s; }
  { T s = Qp[8];
    s = fma(gm[8], Qc[0], s);
    s = fma(gm[3], Qc[2], s);
    s = fma(gm[2], Qc[3], s);
    s = fma(gm[0], Qc[8], s);
    Qp[8] = s; }
  { T s = Qp[9];
    s = fma(gm[9], Qc[0], s);
    s = fma(gm[3], Qc[3], s);
    s = fma(gm[0], Qc[9], s);
    Qp[9] = s; }
  { T s = Qp[10];
    s = fma(gm[10], Qc[0], s);
    s = fma(gm[4], Qc[1], s);
    s = fma(gm[1], Qc[4], s);
    s = fma(gm[0], Qc[10], s);
    Qp[10] = s; }
  { T s = Qp[11];
    s = fma(gm[11], Qc[0], s);
    s = fma(gm[5], Qc[1], s);
    s = fma(gm[4], Qc[2], s);
    s = fma(gm[2], Qc[4], s);
    s = fma(gm[1], Qc[5], s);
    s = fma(gm[0], Qc[11], s);
    Qp[11] = s; }
  { T s = Qp[12];
    s = fma(gm[12], Qc[0], s);
    s = fma(gm[6], Qc[1], s);
    s = fma(gm[4], Qc[3], s);
    s = fma(gm[3], Qc[4], s);
    s = fma(gm[1], Qc[6], s);
    s = fma(gm[0], Qc[12], s);
    Qp[12] = s; }
  { T s = Qp[13];
    s = fma(gm[13], Qc[0], s);
    s = fma(gm[7], Qc[1], s);
    s = fma(gm[5], Qc[2], s);
    s = fma(gm[2], Qc[5], s);
    s = fma(gm[1], Qc[7], s);
    s = fma(gm[0], Qc[13], s);
    Qp[13] = s; }
  { T s = Qp[14];
    s = fma(gm[14], Qc[0], s);
    s = fma(gm[8], Qc[1], s);
    s = fma(gm[6], Qc[2], s);
    s = fma(gm[5], Qc[3], s);
    s = fma(gm[3], Qc[5], s);
    s = fma(gm[2], Qc[6], s);
    s = fma(gm[1], Qc[8], s);
    s = fma(gm[0], Qc[14], s);
    Qp[14] = s; }
  { T s = Qp[15];
    s = fma(gm[15], Qc[0], s);
    s = fma(gm[9], Qc[1], s);
    s = fma(gm[6], Qc[3], s);
    s = fma(gm[3], Qc[6], s);
    s = fma(gm[1], Qc[9], s);
    s = fma(gm[0], Qc[15], s);
    Qp[15] = s; }
  { T s = Qp[16];
    s = fma(gm[16], Qc[0], s);
    s = fma(gm[7], Qc[2], s);
    s = fma(gm[2], Qc[7], s);
    s = fma(gm[0], Qc[16], s);
    Qp[16] = s; }
  { T s = Qp[17];
    s = fma(gm[17], Qc[0], s);
    s = fma(gm[8], Qc[2], s);
    s = fma(gm[7], Qc[3], s);
    s = fma(gm[3], Qc[7], s);
    s = fma(gm[2], Qc[8], s);
    s = fma(gm[0], Qc[17], s);
    Qp[17] = s; }
  { T s = Qp[18];
    s = fma(gm[18], Qc[0], s);
    s = fma(gm[9], Qc[2], s);
    s = fma(gm[8], Qc[3], s);
    s = fma(gm[3], Qc[8], s);
    s = fma(gm[2], Qc[9], s);
    s = fma(gm[0], Qc[18], s);
    Qp[18] = s; }
  { T s = Qp[19];
    s = fma(gm[19], Qc[0], s);
    s = fma(gm[9], Qc[3], s);
    s = fma(gm[3], Qc[9], s);
    s = fma(gm[0], Qc[19], s);
    Qp[19] = s; }
}

#define SFMM_NT_3 19  /* steps of the L2L translation */
static __device__ const unsigned short sfmm_l2l_steps_3[19][64] = {
  {257, 260, 261, 262, 266, 267, 268, 269, 270, 271, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 279, 280, 281, 285, 286, 287, 288, 289, 290, 295, 296, 297, 298, 299, 300, 301, 302, 303, 304, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {514, 517, 519, 520, 523, 525, 526, 528, 529, 530, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 536, 538, 539, 542, 544, 545, 547, 548, 549, 552, 554, 555, 557, 558, 559, 561, 562, 563, 564, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {771, 774, 776, 777, 780, 782, 783, 785, 786, 787, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 793, 795, 796, 799, 801, 802, 804, 805, 806, 809, 811, 812, 814, 815, 816, 818, 819, 820, 821, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1028, 1034, 1035, 1036, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1053, 1054, 1055, 1063, 1064, 1065, 1066, 1067, 1068, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1285, 1291, 1293, 1294, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1310, 1312, 1313, 1320, 1322, 1323, 1325, 1326, 1327, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1542, 1548, 1550, 1551, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1567, 1569, 1570, 1577, 1579, 1580, 1582, 1583, 1584, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1799, 1805, 1808, 1809, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1824, 1827, 1828, 1834, 1837, 1838, 1841, 1842, 1843, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2056, 2062, 2065, 2066, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2081, 2084, 2085, 2091, 2094, 2095, 2098, 2099, 2100, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2313, 2319, 2322, 2323, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2338, 2341, 2342, 2348, 2351, 2352, 2355, 2356, 2357, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2570, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2599, 2600, 2601, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2827, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2856, 2858, 2859, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3084, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3113, 3115, 3116, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3341, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3370, 3373, 3374, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3598, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3627, 3630, 3631, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3855, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3884, 3887, 3888, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4112, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4141, 4145, 4146, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4369, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4398, 4402, 4403, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4626, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4655, 4659, 4660, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4883, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4912, 4916, 4917, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static const int sfmm_moment_mi_3[20][3] = {{0,0,0}, {1,0,0}, {0,1,0}, {0,0,1}, {2,0,0}, {1,1,0}, {1,0,1}, {0,2,0}, {0,1,1}, {0,0,2}, {3,0,0}, {2,1,0}, {2,0,1}, {1,2,0}, {1,1,1}, {1,0,2}, {0,3,0}, {0,2,1}, {0,1,2}, {0,0,3}};

#define SFMM_MT_3 8  /* steps of the M2M translation */
static __device__ const unsigned short sfmm_m2m_steps_3[8][32] = {
  {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 256, 512, 768, 257, 258, 259, 514, 515, 771, 260, 261, 262, 263, 264, 265, 519, 520, 521, 777, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 1024, 513, 769, 1792, 770, 2304, 1025, 516, 772, 517, 518, 774, 1794, 775, 776, 2307, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 1280, 1536, 65535, 2048, 65535, 2560, 1026, 1027, 1282, 773, 1539, 4096, 1795, 2051, 4864, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1281, 1537, 1793, 1283, 2305, 65535, 2050, 2306, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2816, 3072, 3328, 1538, 3840, 65535, 4352, 4608, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2049, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3584, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static __device__ const unsigned short sfmm_moment_exp_3[20] = {0, 1, 8, 64, 2, 9, 65, 16, 72, 128, 3, 10, 66, 17, 73, 129, 24, 80, 136, 192};

template <typename T> __device__ __forceinline__ void sfmm_fold_3(const T* Q, T* q) {
  q[0] = Q[0];
  q[1] = Q[4] - Q[9];
  q[2] = Q[5];
  q[3] = Q[6];
  q[4] = Q[7] - Q[9];
  q[5] = Q[8];
  q[6] = Q[10] - Q[15];
  q[7] = Q[11] - Q[18];
  q[8] = Q[12] - Q[19];
  q[9] = Q[13] - Q[15];
  q[10] = Q[14];
  q[11] = Q[16] - Q[18];
  q[12] = Q[17] - Q[19];
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_fold_3(const T* D, const T* q, T* C) {
  { T s = D[4] * q[1];
    s = fma(D[5], q[2], s);
    s = fma(D[6], q[3], s);
    s = fma(D[7], q[4], s);
    s = fma(D[8], q[5], s);
    s = fma(D[10], q[6], s);
    s = fma(D[11], q[7], s);
    s = fma(D[12], q[8], s);
    s = fma(D[13], q[9], s);
    s = fma(D[14], q[10], s);
    s = fma(D[16], q[11], s);
    s = fma(D[17], q[12], s);
    C[0] += fma(D[0], q[0], s); }
  { T s = D[10] * q[1];
    s = fma(D[11], q[2], s);
    s = fma(D[12], q[3], s);
    s = fma(D[13], q[4], s);
    s = fma(D[14], q[5], s);
    C[1] += fma(D[1], q[0], s); }
  { T s = D[11] * q[1];
    s = fma(D[13], q[2], s);
    s = fma(D[14], q[3], s);
    s = fma(D[16], q[4], s);
    s = fma(D[17], q[5], s);
    C[2] += fma(D[2], q[0], s); }
  { T s = D[12] * q[1];
    s = fma(D[14], q[2], s);
    s = fma(D[15], q[3], s);
    s = fma(D[17], q[4], s);
    s = fma(D[18], q[5], s);
    C[3] += fma(D[3], q[0], s); }
  C[4] = fma(D[4], q[0], C[4]);
  C[5] = fma(D[5], q[0], C[5]);
  C[6] = fma(D[6], q[0], C[6]);
  C[7] = fma(D[7], q[0], C[7]);
  C[8] = fma(D[8], q[0], C[8]);
  C[9] = fma(D[10], q[0], C[9]);
  C[10] = fma(D[11], q[0], C[10]);
  C[11] = fma(D[12], q[0], C[11]);
  C[12] = fma(D[13], q[0], C[12]);
  C[13] = fma(D[14], q[0], C[13]);
  C[14] = fma(D[16], q[0], C[14]);
  C[15] = fma(D[17], q[0], C[15]);
  C[16] = fma(D[20], q[6], C[16]);
  C[16] = fma(D[21], q[7], C[16]);
  C[16] = fma(D[22], q[8], C[16]);
  C[16] = fma(D[23], q[9], C[16]);
  C[16] = fma(D[24], q[10], C[16]);
  C[16] = fma(D[26], q[11], C[16]);
  C[16] = fma(D[27], q[12], C[16]);
  C[17] = fma(D[21], q[6], C[17]);
  C[17] = fma(D[23], q[7], C[17]);
  C[17] = fma(D[24], q[8], C[17]);
  C[17] = fma(D[26], q[9], C[17]);
  C[17] = fma(D[27], q[10], C[17]);
  C[17] = fma(D[30], q[11], C[17]);
  C[17] = fma(D[31], q[12], C[17]);
  C[18] = fma(D[22], q[6], C[18]);
  C[18] = fma(D[24], q[7], C[18]);
  C[18] = fma(D[25], q[8], C[18]);
  C[18] = fma(D[27], q[9], C[18]);
  C[18] = fma(D[28], q[10], C[18]);
  C[18] = fma(D[31], q[11], C[18]);
  C[18] = fma(D[32], q[12], C[18]);
  C[19] = fma(D[20], q[1], C[19]);
  C[19] = fma(D[21], q[2], C[19]);
  C[19] = fma(D[22], q[3], C[19]);
  C[19] = fma(D[23], q[4], C[19]);
  C[19] = fma(D[24], q[5], C[19]);
  C[20] = fma(D[21], q[1], C[20]);
  C[20] = fma(D[23], q[2], C[20]);
  C[20] = fma(D[24], q[3], C[20]);
  C[20] = fma(D[26], q[4], C[20]);
  C[20] = fma(D[27], q[5], C[20]);
  C[21] = fma(D[22], q[1], C[21]);
  C[21] = fma(D[24], q[2], C[21]);
  C[21] = fma(D[25], q[3], C[21]);
  C[21] = fma(D[27], q[4], C[21]);
  C[21] = fma(D[28], q[5], C[21]);
  C[22] = fma(D[23], q[1], C[22]);
  C[22] = fma(D[26], q[2], C[22]);
  C[22] = fma(D[27], q[3], C[22]);
  C[22] = fma(D[30], q[4], C[22]);
  C[22] = fma(D[31], q[5], C[22]);
  C[23] = fma(D[24], q[1], C[23]);
  C[23] = fma(D[27], q[2], C[23]);
  C[23] = fma(D[28], q[3], C[23]);
  C[23] = fma(D[31], q[4], C[23]);
  C[23] = fma(D[32], q[5], C[23]);
  C[24] = fma(D[20], q[0], C[24]);
  C[25] = fma(D[21], q[0], C[25]);
  C[26] = fma(D[22], q[0], C[26]);
  C[27] = fma(D[23], q[0], C[27]);
  C[28] = fma(D[24], q[0], C[28]);
  C[29] = fma(D[26], q[0], C[29]);
  C[30] = fma(D[27], q[0], C[30]);
  C[31] = fma(D[30], q[0], C[31]);
  C[32] = fma(D[31], q[0], C[32]);
}

#define SFMM_NR_3 13  /* entries of a source row */
#define SFMM_NS_3 33  /* sums of an interaction */
#define SFMM_NX_3 4
static __device__ const signed char sfmm_unfold_3[54][4][2] = {
  {{0, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{1, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{2, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{3, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{4, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{5, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{6, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{7, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{8, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{4, -1}, {7, -1}, {0, 0}, {0, 0}},
  {{9, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{10, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{11, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{12, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{13, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{9, 1}, {12, 1}, {0, 0}, {0, 0}},
  {{14, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{15, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{10, 1}, {14, 1}, {0, 0}, {0, 0}},
  {{11, 1}, {15, 1}, {0, 0}, {0, 0}},
  {{1, -1}, {16, -1}, {0, 0}, {0, 0}},
  {{2, -1}, {17, -1}, {0, 0}, {0, 0}},
  {{3, -1}, {18, -1}, {0, 0}, {0, 0}},
  {{4, 1}, {19, 1}, {0, 0}, {0, 0}},
  {{5, 1}, {20, 1}, {0, 0}, {0, 0}},
  {{6, 1}, {21, 1}, {0, 0}, {0, 0}},
  {{7, 1}, {22, 1}, {0, 0}, {0, 0}},
  {{8, 1}, {23, 1}, {0, 0}, {0, 0}},
  {{4, -1}, {19, -1}, {7, -1}, {22, -1}},
  {{9, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{10, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{11, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{12, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{13, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{9, 1}, {12, 1}, {0, 0}, {0, 0}},
  {{14, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{15, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{10, 1}, {14, 1}, {0, 0}, {0, 0}},
  {{11, 1}, {15, 1}, {0, 0}, {0, 0}},
  {{24, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{25, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{26, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{27, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{28, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{24, -1}, {27, -1}, {0, 0}, {0, 0}},
  {{29, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{30, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{25, -1}, {29, -1}, {0, 0}, {0, 0}},
  {{26, -1}, {30, -1}, {0, 0}, {0, 0}},
  {{31, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{32, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{27, -1}, {31, -1}, {0, 0}, {0, 0}},
  {{28, -1}, {32, -1}, {0, 0}, {0, 0}},
  {{24, 1}, {27, 2}, {31, 1}, {0, 0}}};

template <typename T> __device__ __forceinline__ void sfmm_m2l_4(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    s = fma(D[1], Q[1], s);
    s = fma(D[2], Q[2], s);
    s = fma(D[3], Q[3], s);
    s = fma(D[4], Q[4], s);
    s = fma(D[5], Q[5], s);
    s = fma(D[6], Q[6], s);
    s = fma(D[7], Q[7], s);
    s = fma(D[8], Q[8], s);
    s = fma(D[9], Q[9], s);
    s = fma(D[10], Q[10], s);
    s = fma(D[11], Q[11], s);
    s = fma(D[12], Q[12], s);
    s = fma(D[13], Q[13], s);
    s = fma(D[14], Q[14], s);
    s = fma(D[15], Q[15], s);
    s = fma(D[16], Q[16], s);
    s = fma(D[17], Q[17], s);
    s = fma(D[18], Q[18], s);
    s = fma(D[19], Q[19], s);
    s = fma(D[20], Q[20], s);
    s = fma(D[21], Q[21], s);
    s = fma(D[22], Q[22], s);
    s = fma(D[23], Q[23], s);
    s = fma(D[24], Q[24], s);
    s = fma(D[25], Q[25], s);
    s = fma(D[26], Q[26], s);
    s = fma(D[27], Q[27], s);
    s = fma(D[28], Q[28], s);
    s = fma(D[29], Q[29], s);
    s = fma(D[30], Q[30], s);
    s = fma(D[31], Q[31], s);
    s = fma(D[32], Q[32], s);
    s = fma(D[33], Q[33], s);
    s = fma(D[34], Q[34], s);
    C[0] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[4], Q[1], s);
    s = fma(D[5], Q[2], s);
    s = fma(D[6], Q[3], s);
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    s = fma(D[20], Q[10], s);
    s = fma(D[21], Q[11], s);
    s = fma(D[22], Q[12], s);
    s = fma(D[23], Q[13], s);
    s = fma(D[24], Q[14], s);
    s = fma(D[25], Q[15], s);
    s = fma(D[26], Q[16], s);
    s = fma(D[27], Q[17], s);
    s = fma(D[28], Q[18], s);
    s = fma(D[29], Q[19], s);
    C[1] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[5], Q[1], s);
    s = fma(D[7], Q[2], s);
    s = fma(D[8], Q[3], s);
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    s = fma(D[21], Q[10], s);
    s = fma(D[23], Q[11], s);
    s = fma(D[24], Q[12], s);
    s = fma(D[26], Q[13], s);
    s = fma(D[27], Q[14], s);
    s = fma(D[28], Q[15], s);
    s = fma(D[30], Q[16], s);
    s = fma(D[31], Q[17], s);
    s = fma(D[32], Q[18], s);
    s = fma(D[33], Q[19], s);
    C[2] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[6], Q[1], s);
    s = fma(D[8], Q[2], s);
    s = fma(D[9], Q[3], s);
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    s = fma(D[22], Q[10], s);
    s = fma(D[24], Q[11], s);
    s = fma(D[25], Q[12], s);
    s = fma(D[27], Q[13], s);
    s = fma(D[28], Q[14], s);
    s = fma(D[29], Q[15], s);
    s = fma(D[31], Q[16], s);
    s = fma(D[32], Q[17], s);
    s = fma(D[33], Q[18], s);
    s = fma(D[34], Q[19], s);
    C[3] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[10], Q[1], s);
    s = fma(D[11], Q[2], s);
    s = fma(D[12], Q[3], s);
    s = fma(D[20], Q[4], s);
    s = fma(D[21], Q[5], s);
    s = fma(D[22], Q[6], s);
    s = fma(D[23], Q[7], s);
    s = fma(D[24], Q[8], s);
    s = fma(D[25], Q[9], s);
    C[4] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[11], Q[1], s);
    s = fma(D[13], Q[2], s);
    s = fma(D[14], Q[3], s);
    s = fma(D[21], Q[4], s);
    s = fma(D[23], Q[5], s);
    s = fma(D[24], Q[6], s);
    s = fma(D[26], Q[7], s);
    s = fma(D[27], Q[8], s);
    s = fma(D[28], Q[9], s);
    C[5] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[12], Q[1], s);
    s = fma(D[14], Q[2], s);
    s = fma(D[15], Q[3], s);
    s = fma(D[22], Q[4], s);
    s = fma(D[24], Q[5], s);
    s = fma(D[25], Q[6], s);
    s = fma(D[27], Q[7], s);
    s = fma(D[28], Q[8], s);
    s = fma(D[29], Q[9], s);
    C[6] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[13], Q[1], s);
    s = fma(D[16], Q[2], s);
    s = fma(D[17], Q[3], s);
    s = fma(D[23], Q[4], s);
    s = fma(D[26], Q[5], s);
    s = fma(D[27], Q[6], s);
    s = fma(D[30], Q[7], s);
    s = fma(D[31], Q[8], s);
    s = fma(D[32], Q[9], s);
    C[7] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[14], Q[1], s);
    s = fma(D[17], Q[2], s);
    s = fma(D[18], Q[3], s);
    s = fma(D[24], Q[4], s);
    s = fma(D[27], Q[5], s);
    s = fma(D[28], Q[6], s);
    s = fma(D[31], Q[7], s);
    s = fma(D[32], Q[8], s);
    s = fma(D[33], Q[9], s);
    C[8] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[15], Q[1], s);
    s = fma(D[18], Q[2], s);
    s = fma(D[19], Q[3], s);
    s = fma(D[25], Q[4], s);
    s = fma(D[28], Q[5], s);
    s = fma(D[29], Q[6], s);
    s = fma(D[32], Q[7], s);
    s = fma(D[33], Q[8], s);
    s = fma(D[34], Q[9], s);
    C[9] += s; }
  { T s = D[10] * Q[0];
    s = fma(D[20], Q[1], s);
    s = fma(D[21], Q[2], s);
    s = fma(D[22], Q[3], s);
    C[10] -= s; }
  { T s = D[11] * Q[0];
    s = fma(D[21], Q[1], s);
    s = fma(D[23], Q[2], s);
    s = fma(D[24], Q[3], s);
    C[11] -= s; }
  { T s = D[12] * Q[0];
    s = fma(D[22], Q[1], s);
    s = fma(D[24], Q[2], s);
    s = fma(D[25], Q[3], s);
    C[12] -= s; }
  { T s = D[13] * Q[0];
    s = fma(D[23], Q[1], s);
    s = fma(D[26], Q[2], s);
    s = fma(D[27], Q[3], s);
    C[13] -= s; }
  { T s = D[14] * Q[0];
    s = fma(D[24], Q[1], s);
    s = fma(D[27], Q[2], s);
    s = fma(D[28], Q[3], s);
    C[14] -= s; }
  { T s = D[15] * Q[0];
    s = fma(D[25], Q[1], s);
    s = fma(D[28], Q[2], s);
    s = fma(D[29], Q[3], s);
    C[15] -= s; }
  { T s = D[16] * Q[0];
    s = fma(D[26], Q[1], s);
    s = fma(D[30], Q[2], s);
    s = fma(D[31], Q[3], s);
    C[16] -= s; }
  { T s = D[17] * Q[0];
    s = fma(D[27], Q[1], s);
    s = fma(D[31], Q[2], s);
    s = fma(D[32], Q[3], s);
    C[17] -= s; }
  { T s = D[18] * Q[0];
    s = fma(D[28], Q[1], s);
    s = fma(D[32], Q[2], s);
    s = fma(D[33], Q[3], s);
    C[18] -= s; }
  { T s = D[19] * Q[0];
    s = fma(D[29], Q[1], s);
    s = fma(D[33], Q[2], s);
    s = fma(D[34], Q[3], s);
    C[19] -= s; }
  { T s = D[20] * Q[0];
    C[20] += s; }
  { T s = D[21] * Q[0];
    C[21] += s; }
  { T s = D[22] * Q[0];
    C[22] += s; }
  { T s = D[23] * Q[0];
    C[23] += s; }
  { T s = D[24] * Q[0];
    C[24] += s; }
  { T s = D[25] * Q[0];
    C[25] += s; }
  { T s = D[26] * Q[0];
    C[26] += s; }
  { T s = D[27] * Q[0];
    C[27] += s; }
  { T s = D[28] * Q[0];
    C[28] += s; }
  { T s = D[29] * Q[0];
    C[29] += s; }
  { T s = D[30] * Q[0];
    C[30] += s; }
  { T s = D[31] * Q[0];
    C[31] += s; }
  { T s = D[32] * Q[0];
    C[32] += s; }
  { T s = D[33] * Q[0];
    C[33] += s; }
  { T s = D[34] * Q[0];
    C[34] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[4], Q[1], s);
    s = fma(D[5], Q[2], s);
    s = fma(D[6], Q[3], s);
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    s = fma(D[20], Q[10], s);
    s = fma(D[21], Q[11], s);
    s = fma(D[22], Q[12], s);
    s = fma(D[23], Q[13], s);
    s = fma(D[24], Q[14], s);
    s = fma(D[25], Q[15], s);
    s = fma(D[26], Q[16], s);
    s = fma(D[27], Q[17], s);
    s = fma(D[28], Q[18], s);
    s = fma(D[29], Q[19], s);
    s = fma(D[35], Q[20], s);
    s = fma(D[36], Q[21], s);
    s = fma(D[37], Q[22], s);
    s = fma(D[38], Q[23], s);
    s = fma(D[39], Q[24], s);
    s = fma(D[40], Q[25], s);
    s = fma(D[41], Q[26], s);
    s = fma(D[42], Q[27], s);
    s = fma(D[43], Q[28], s);
    s = fma(D[44], Q[29], s);
    s = fma(D[45], Q[30], s);
    s = fma(D[46], Q[31], s);
    s = fma(D[47], Q[32], s);
    s = fma(D[48], Q[33], s);
    s = fma(D[49], Q[34], s);
    C[35] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[5], Q[1], s);
    s = fma(D[7], Q[2], s);
    s = fma(D[8], Q[3], s);
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    s = fma(D[21], Q[10], s);
    s = fma(D[23], Q[11], s);
    s = fma(D[24], Q[12], s);
    s = fma(D[26], Q[13], s);
    s = fma(D[27], Q[14], s);
    s = fma(D[28], Q[15], s);
    s = fma(D[30], Q[16], s);
    s = fma(D[31], Q[17], s);
    s = fma(D[32], Q[18], s);
    s = fma(D[33], Q[19], s);
    s = fma(D[36], Q[20], s);
    s = fma(D[38], Q[21], s);
    s = fma(D[39], Q[22], s);
    s = fma(D[41], Q[23], s);
    s = fma(D[42], Q[24], s);
    s = fma(D[43], Q[25], s);
    s = fma(D[45], Q[26], s);
    s = fma(D[46], Q[27], s);
    s = fma(D[47], Q[28], s);
    s = fma(D[48], Q[29], s);
    s = fma(D[50], Q[30], s);
    s = fma(D[51], Q[31], s);
    s = fma(D[52], Q[32], s);
    s = fma(D[53], Q[33], s);
    s = fma(D[54], Q[34], s);
    C[36] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[6], Q[1], s);
    s = fma(D[8], Q[2], s);
    s = fma(D[9], Q[3], s);
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    s = fma(D[22], Q[10], s);
    s = fma(D[24], Q[11], s);
    s = fma(D[25], Q[12], s);
    s = fma(D[27], Q[13], s);
    s = fma(D[28], Q[14], s);
    s = fma(D[29], Q[15], s);
    s = fma(D[31], Q[16], s);
    s = fma(D[32], Q[17], s);
    s = fma(D[33], Q[18], s);
    s = fma(D[34], Q[19], s);
    s = fma(D[37], Q[20], s);
    s = fma(D[39], Q[21], s);
    s = fma(D[40], Q[22], s);
    s = fma(D[42], Q[23], s);
    s = fma(D[43], Q[24], s);
    s = fma(D[44], Q[25], s);
    s = fma(D[46], Q[26], s);
    s = fma(D[47], Q[27], s);
    s = fma(D[48], Q[28], s);
    s = fma(D[49], Q[29], s);
    s = fma(D[51], Q[30], s);
    s = fma(D[52], Q[31], s);
    s = fma(D[53], Q[32], s);
    s = fma(D[54], Q[33], s);
    s = fma(D[55], Q[34], s);
    C[37] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[10], Q[1], s);
    s = fma(D[11], Q[2], s);
    s = fma(D[12], Q[3], s);
    s = fma(D[20], Q[4], s);
    s = fma(D[21], Q[5], s);
    s = fma(D[22], Q[6], s);
    s = fma(D[23], Q[7], s);
    s = fma(D[24], Q[8], s);
    s = fma(D[25], Q[9], s);
    s = fma(D[35], Q[10], s);
    s = fma(D[36], Q[11], s);
    s = fma(D[37], Q[12], s);
    s = fma(D[38], Q[13], s);
    s = fma(D[39], Q[14], s);
    s = fma(D[40], Q[15], s);
    s = fma(D[41], Q[16], s);
    s = fma(D[42], Q[17], s);
    s = fma(D[43], Q[18], s);
    s = fma(D[44], Q[19], s);
    C[38] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[11], Q[1], s);
    s = fma(D[13], Q[2], s);
    s = fma(D[14], Q[3], s);
    s = fma(D[21], Q[4], s);
    s = fma(D[23], Q[5], s);
    s = fma(D[24], Q[6], s);
    s = fma(D[26], Q[7], s);
    s = fma(D[27], Q[8], s);
    s = fma(D[28], Q[9], s);
    s = fma(D[36], Q[10], s);
    s = fma(D[38], Q[11], s);
    s = fma(D[39], Q[12], s);
    s = fma(D[41], Q[13], s);
    s = fma(D[42], Q[14], s);
    s = fma(D[43], Q[15], s);
    s = fma(D[45], Q[16], s);
    s = fma(D[46], Q[17], s);
    s = fma(D[47], Q[18], s);
    s = fma(D[48], Q[19], s);
    C[39] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[12], Q[1], s);
    s = fma(D[14], Q[2], s);
    s = fma(D[15], Q[3], s);
    s = fma(D[22], Q[4], s);
    s = fma(D[24], Q[5], s);
    s = fma(D[25], Q[6], s);
    s = fma(D[27], Q[7], s);
    s = fma(D[28], Q[8], s);
    s = fma(D[29], Q[9], s);
    s = fma(D[37], Q[10], s);
    s = fma(D[39], Q[11], s);
    s = fma(D[40], Q[12], s);
    s = fma(D[42], Q[13], s);
    s = fma(D[43], Q[14], s);
    s = fma(D[44], Q[15], s);
    s = fma(D[46], Q[16], s);
    s = fma(D[47], Q[17], s);
    s = fma(D[48], Q[18], s);
    s = fma(D[49], Q[19], s);
    C[40] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[13], Q[1], s);
    s = fma(D[16], Q[2], s);
    s = fma(D[17], Q[3], s);
    s = fma(D[23], Q[4], s);
    s = fma(D[26], Q[5], s);
    s = fma(D[27], Q[6], s);
    s = fma(D[30], Q[7], s);
    s = fma(D[31], Q[8], s);
    s = fma(D[32], Q[9], s);
    s = fma(D[38], Q[10], s);
    s = fma(D[41], Q[11], s);
    s = fma(D[42], Q[12], s);
    s = fma(D[45], Q[13], s);
    s = fma(D[46], Q[14], s);
    s = fma(D[47], Q[15], s);
    s = fma(D[50], Q[16], s);
    s = fma(D[51], Q[17], s);
    s = fma(D[52], Q[18], s);
    s = fma(D[53], Q[19], s);
    C[41] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[14], Q[1], s);
    s = fma(D[17], Q[2], s);
    s = fma(D[18], Q[3], s);
    s = fma(D[24], Q[4], s);
    s = fma(D[27], Q[5], s);
    s = fma(D[28], Q[6], s);
    s = fma(D[31], Q[7], s);
    s = fma(D[32], Q[8], s);
    s = fma(D[33], Q[9], s);
    s = fma(D[39], Q[10], s);
    s = fma(D[42], Q[11], s);
    s = fma(D[43], Q[12], s);
    s = fma(D[46], Q[13], s);
    s = fma(D[47], Q[14], s);
    s = fma(D[48], Q[15], s);
    s = fma(D[51], Q[16], s);
    s = fma(D[52], Q[17], s);
    s = fma(D[53], Q[18], s);
    s = fma(D[54], Q[19], s);
    C[42] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[15], Q[1], s);
    s = fma(D[18], Q[2], s);
    s = fma(D[19], Q[3], s);
    s = fma(D[25], Q[4], s);
    s = fma(D[28], Q[5], s);
    s = fma(D[29], Q[6], s);
    s = fma(D[32], Q[7], s);
    s = fma(D[33], Q[8], s);
    s = fma(D[34], Q[9], s);
    s = fma(D[40], Q[10], s);
    s = fma(D[43], Q[11], s);
    s = fma(D[44], Q[12], s);
    s = fma(D[47], Q[13], s);
    s = fma(D[48], Q[14], s);
    s = fma(D[49], Q[15], s);
    s = fma(D[52], Q[16], s);
    s = fma(D[53], Q[17], s);
    s = fma(D[54], Q[18], s);
    s = fma(D[55], Q[19], s);
    C[43] += s; }
  { T s = D[10] * Q[0];
    s = fma(D[20], Q[1], s);
    s = fma(D[21], Q[2], s);
    s = fma(D[22], Q[3], s);
    s = fma(D[35], Q[4], s);
    s = fma(D[36], Q[5], s);
    s = fma(D[37], Q[6], s);
    s = fma(D[38], Q[7], s);
    s = fma(D[39], Q[8], s);
    s = fma(D[40], Q[9], s);
    C[44] -= s; }
  { T s = D[11] * Q[0];
    s = fma(D[21], Q[1], s);
    s = fma(D[23], Q[2], s);
    s = fma(D[24], Q[3], s);
    s = fma(D[36], Q[4], s);
    s = fma(D[38], Q[5], s);
    s = fma(D[39], Q[6], s);
    s = fma(D[41], Q[7], s);
    s = fma(D[42], Q[8], s);
    s = fma(D[43], Q[9], s);
    C[45] -= s; }
  { T s = D[12] * Q[0];
    s = fma(D[22], Q[1], s);
    s = fma(D[24], Q[2], s);
    s = fma(D[25], Q[3], s);
    s = fma(D[37], Q[4], s);
    s = fma(D[39], Q[5], s);
    s = fma(D[40], Q[6], s);
    s = fma(D[42], Q[7], s);
    s = fma(D[43], Q[8], s);
    s = fma(D[44], Q[9], s);
    C[46] -= s; }
  { T s = D[13] * Q[0];
    s = fma(D[23], Q[1], s);
    s = fma(D[26], Q[2], s);
    s = fma(D[27], Q[3], s);
    s = fma(D[38], Q[4], s);
    s = fma(D[41], Q[5], s);
    s = fma(D[42], Q[6], s);
    s = fma(D[45], Q[7], s);
    s = fma(D[46], Q[8], s);
    s = fma(D[47], Q[9], s);
    C[47] -= s; }
  { T s = D[14] * Q[0];
    s = fma(D[24], Q[1], s);
    s = fma(D[27], Q[2], s);
    s = fma(D[28], Q[3], s);
    s = fma(D[39], Q[4], s);
    s = fma(D[42], Q[5], s);
    s = fma(D[43], Q[6], s);
    s = fma(D[46], Q[7], s);
    s = fma(D[47], Q[8], s);
    s = fma(D[48], Q[9], s);
    C[48] -= s; }
  { T s = D[15] * Q[0];
    s = fma(D[25], Q[1], s);
    s = fma(D[28], Q[2], s);
    s = fma(D[29], Q[3], s);
    s = fma(D[40], Q[4], s);
    s = fma(D[43], Q[5], s);
    s = fma(D[44], Q[6], s);
    s = fma(D[47], Q[7], s);
    s = fma(D[48], Q[8], s);
    s = fma(D[49], Q[9], s);
    C[49] -= s; }
  { T s = D[16] * Q[0];
    s = fma(D[26], Q[1], s);
    s = fma(D[30], Q[2], s);
    s = fma(D[31], Q[3], s);
    s = fma(D[41], Q[4], s);
    s = fma(D[45], Q[5], s);
    s = fma(D[46], Q[6], s);
    s = fma(D[50], Q[7], s);
    s = fma(D[51], Q[8], s);
    s = fma(D[52], Q[9], s);
    C[50] -= s; }
  { T s = D[17] * Q[0];
    s = fma(D[27], Q[1], s);
    s = fma(D[31], Q[2], s);
    s = fma(D[32], Q[3], s);
    s = fma(D[42], Q[4], s);
    s = fma(D[46], Q[5], s);
    s = fma(D[47], Q[6], s);
    s = fma(D[51], Q[7], s);
    s = fma(D[52], Q[8], s);
    s = fma(D[53], Q[9], s);
    C[51] -= s; }
  { T s = D[18] * Q[0];
    s = fma(D[28], Q[1], s);
    s = fma(D[32], Q[2], s);
    s = fma(D[33], Q[3], s);
    s = fma(D[43], Q[4], s);
    s = fma(D[47], Q[5], s);
    s = fma(D[48], Q[6], s);
    s = fma(D[52], Q[7], s);
    s = fma(D[53], Q[8], s);
    s = fma(D[54], Q[9], s);
    C[52] -= s; }
  { T s = D[19] * Q[0];
    s = fma(D[29], Q[1], s);
    s = fma(D[33], Q[2], s);
    s = fma(D[34], Q[3], s);
    s = fma(D[44], Q[4], s);
    s = fma(D[48], Q[5], s);
    s = fma(D[49], Q[6], s);
    s = fma(D[53], Q[7], s);
    s = fma(D[54], Q[8], s);
    s = fma(D[55], Q[9], s);
    C[53] -= s; }
  { T s = D[20] * Q[0];
    s = fma(D[35], Q[1], s);
    s = fma(D[36], Q[2], s);
    s = fma(D[37], Q[3], s);
    C[54] += s; }
  { T s = D[21] * Q[0];
    s = fma(D[36], Q[1], s);
    s = fma(D[38], Q[2], s);
    s = fma(D[39], Q[3], s);
    C[55] += s; }
  { T s = D[22] * Q[0];
    s = fma(D[37], Q[1], s);
    s = fma(D[39], Q[2], s);
    s = fma(D[40], Q[3], s);
    C[56] += s; }
  { T s = D[23] * Q[0];
    s = fma(D[38], Q[1], s);
    s = fma(D[41], Q[2], s);
    s = fma(D[42], Q[3], s);
    C[57] += s; }
  { T s = D[24] * Q[0];
    s = fma(D[39], Q[1], s);
    s = fma(D[42], Q[2], s);
    s = fma(D[43], Q[3], s);
    C[58] += s; }
  { T s = D[25] * Q[0];
    s = fma(D[40], Q[1], s);
    s = fma(D[43], Q[2], s);
    s = fma(D[44], Q[3], s);
    C[59] += s; }
  { T s = D[26] * Q[0];
    s = fma(D[41], Q[1], s);
    s = fma(D[45], Q[2], s);
    s = fma(D[46], Q[3], s);
    C[60] += s; }
  { T s = D[27] * Q[0];
    s = fma(D[42], Q[1], s);
    s = fma(D[46], Q[2], s);
    s = fma(D[47], Q[3], s);
    C[61] += s; }
  { T s = D[28] * Q[0];
    s = fma(D[43], Q[1], s);
    s = fma(D[47], Q[2], s);
    s = fma(D[48], Q[3], s);
    C[62] += s; }
  { T s = D[29] * Q[0];
    s = fma(D[44], Q[1], s);
    s = fma(D[48], Q[2], s);
    s = fma(D[49], Q[3], s);
    C[63] += s; }
  { T s = D[30] * Q[0];
    s = fma(D[45], Q[1], s);
    s = fma(D[50], Q[2], s);
    s = fma(D[51], Q[3], s);
    C[64] += s; }
  { T s = D[31] * Q[0];
    s = fma(D[46], Q[1], s);
    s = fma(D[51], Q[2], s);
    s = fma(D[52], Q[3], s);
    C[65] += s; }
  { T s = D[32] * Q[0];
    s = fma(D[47], Q[1], s);
    s = fma(D[52], Q[2], s);
    s = fma(D[53], Q[3], s);
    C[66] += s; }
  { T s = D[33] * Q[0];
    s = fma(D[48], Q[1], s);
    s = fma(D[53], Q[2], s);
    s = fma(D[54], Q[3], s);
    C[67] += s; }
  { T s = D[34] * Q[0];
    s = fma(D[49], Q[1], s);
    s = fma(D[54], Q[2], s);
    s = fma(D[55], Q[3], s);
    C[68] += s; }
  { T s = D[35] * Q[0];
    C[69] -= s; }
  { T s = D[36] * Q[0];
    C[70] -= s; }
  { T s = D[37] * Q[0];
    C[71] -= s; }
  { T s = D[38] * Q[0];
    C[72] -= s; }
  { T s = D[39] * Q[0];
    C[73] -= s; }
  { T s = D[40] * Q[0];
    C[74] -= s; }
  { T s = D[41] * Q[0];
    C[75] -= s; }
  { T s = D[42] * Q[0];
    C[76] -= s; }
  { T s = D[43] * Q[0];
    C[77] -= s; }
  { T s = D[44] * Q[0];
    C[78] -= s; }
  { T s = D[45] * Q[0];
    C[79] -= s; }
  { T s = D[46] * Q[0];
    C[80] -= s; }
  { T s = D[47] * Q[0];
    C[81] -= s; }
  { T s = D[48] * Q[0];
    C[82] -= s; }
  { T s = D[49] * Q[0];
    C[83] -= s; }
  { T s = D[50] * Q[0];
    C[84] -= s; }
  { T s = D[51] * Q[0];
    C[85] -= s; }
  { T s = D[52] * Q[0];
    C[86] -= s; }
  { T s = D[53] * Q[0];
    C[87] -= s; }
  { T s = D[54] * Q[0];
    C[88] -= s; }
  { T s = D[55] * Q[0];
    C[89] -= s; }
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_4_nodip(const T* D, const T* Q, T* C) {
  { T s = D[0] * Q[0];
    s = fma(D[4], Q[4], s);
    s = fma(D[5], Q[5], s);
    s = fma(D[6], Q[6], s);
    s = fma(D[7], Q[7], s);
    s = fma(D[8], Q[8], s);
    s = fma(D[9], Q[9], s);
    s = fma(D[10], Q[10], s);
    s = fma(D[11], Q[11], s);
    s = fma(D[12], Q[12], s);
    s = fma(D[13], Q[13], s);
    s = fma(D[14], Q[14], s);
    s = fma(D[15], Q[15], s);
    s = fma(D[16], Q[16], s);
    s = fma(D[17], Q[17], s);
    s = fma(D[18], Q[18], s);
    s = fma(D[19], Q[19], s);
    s = fma(D[20], Q[20], s);
    s = fma(D[21], Q[21], s);
    s = fma(D[22], Q[22], s);
    s = fma(D[23], Q[23], s);
    s = fma(D[24], Q[24], s);
    s = fma(D[25], Q[25], s);
    s = fma(D[26], Q[26], s);
    s = fma(D[27], Q[27], s);
    s = fma(D[28], Q[28], s);
    s = fma(D[29], Q[29], s);
    s = fma(D[30], Q[30], s);
    s = fma(D[31], Q[31], s);
    s = fma(D[32], Q[32], s);
    s = fma(D[33], Q[33], s);
    s = fma(D[34], Q[34], s);
    C[0] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    s = fma(D[20], Q[10], s);
    s = fma(D[21], Q[11], s);
    s = fma(D[22], Q[12], s);
    s = fma(D[23], Q[13], s);
    s = fma(D[24], Q[14], s);
    s = fma(D[25], Q[15], s);
    s = fma(D[26], Q[16], s);
    s = fma(D[27], Q[17], s);
    s = fma(D[28], Q[18], s);
    s = fma(D[29], Q[19], s);
    C[1] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    s = fma(D[21], Q[10], s);
    s = fma(D[23], Q[11], s);
    s = fma(D[24], Q[12], s);
    s = fma(D[26], Q[13], s);
    s = fma(D[27], Q[14], s);
    s = fma(D[28], Q[15], s);
    s = fma(D[30], Q[16], s);
    s = fma(D[31], Q[17], s);
    s = fma(D[32], Q[18], s);
    s = fma(D[33], Q[19], s);
    C[2] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    s = fma(D[22], Q[10], s);
    s = fma(D[24], Q[11], s);
    s = fma(D[25], Q[12], s);
    s = fma(D[27], Q[13], s);
    s = fma(D[28], Q[14], s);
    s = fma(D[29], Q[15], s);
    s = fma(D[31], Q[16], s);
    s = fma(D[32], Q[17], s);
    s = fma(D[33], Q[18], s);
    s = fma(D[34], Q[19], s);
    C[3] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[20], Q[4], s);
    s = fma(D[21], Q[5], s);
    s = fma(D[22], Q[6], s);
    s = fma(D[23], Q[7], s);
    s = fma(D[24], Q[8], s);
    s = fma(D[25], Q[9], s);
    C[4] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[21], Q[4], s);
    s = fma(D[23], Q[5], s);
    s = fma(D[24], Q[6], s);
    s = fma(D[26], Q[7], s);
    s = fma(D[27], Q[8], s);
    s = fma(D[28], Q[9], s);
    C[5] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[22], Q[4], s);
    s = fma(D[24], Q[5], s);
    s = fma(D[25], Q[6], s);
    s = fma(D[27], Q[7], s);
    s = fma(D[28], Q[8], s);
    s = fma(D[29], Q[9], s);
    C[6] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[23], Q[4], s);
    s = fma(D[26], Q[5], s);
    s = fma(D[27], Q[6], s);
    s = fma(D[30], Q[7], s);
    s = fma(D[31], Q[8], s);
    s = fma(D[32], Q[9], s);
    C[7] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[24], Q[4], s);
    s = fma(D[27], Q[5], s);
    s = fma(D[28], Q[6], s);
    s = fma(D[31], Q[7], s);
    s = fma(D[32], Q[8], s);
    s = fma(D[33], Q[9], s);
    C[8] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[25], Q[4], s);
    s = fma(D[28], Q[5], s);
    s = fma(D[29], Q[6], s);
    s = fma(D[32], Q[7], s);
    s = fma(D[33], Q[8], s);
    s = fma(D[34], Q[9], s);
    C[9] += s; }
  { T s = D[10] * Q[0];
    C[10] -= s; }
  { T s = D[11] * Q[0];
    C[11] -= s; }
  { T s = D[12] * Q[0];
    C[12] -= s; }
  { T s = D[13] * Q[0];
    C[13] -= s; }
  { T s = D[14] * Q[0];
    C[14] -= s; }
  { T s = D[15] * Q[0];
    C[15] -= s; }
  { T s = D[16] * Q[0];
    C[16] -= s; }
  { T s = D[17] * Q[0];
    C[17] -= s; }
  { T s = D[18] * Q[0];
    C[18] -= s; }
  { T s = D[19] * Q[0];
    C[19] -= s; }
  { T s = D[20] * Q[0];
    C[20] += s; }
  { T s = D[21] * Q[0];
    C[21] += s; }
  { T s = D[22] * Q[0];
    C[22] += s; }
  { T s = D[23] * Q[0];
    C[23] += s; }
  { T s = D[24] * Q[0];
    C[24] += s; }
  { T s = D[25] * Q[0];
    C[25] += s; }
  { T s = D[26] * Q[0];
    C[26] += s; }
  { T s = D[27] * Q[0];
    C[27] += s; }
  { T s = D[28] * Q[0];
    C[28] += s; }
  { T s = D[29] * Q[0];
    C[29] += s; }
  { T s = D[30] * Q[0];
    C[30] += s; }
  { T s = D[31] * Q[0];
    C[31] += s; }
  { T s = D[32] * Q[0];
    C[32] += s; }
  { T s = D[33] * Q[0];
    C[33] += s; }
  { T s = D[34] * Q[0];
    C[34] += s; }
  { T s = D[1] * Q[0];
    s = fma(D[10], Q[4], s);
    s = fma(D[11], Q[5], s);
    s = fma(D[12], Q[6], s);
    s = fma(D[13], Q[7], s);
    s = fma(D[14], Q[8], s);
    s = fma(D[15], Q[9], s);
    s = fma(D[20], Q[10], s);
    s = fma(D[21], Q[11], s);
    s = fma(D[22], Q[12], s);
    s = fma(D[23], Q[13], s);
    s = fma(D[24], Q[14], s);
    s = fma(D[25], Q[15], s);
    s = fma(D[26], Q[16], s);
    s = fma(D[27], Q[17], s);
    s = fma(D[28], Q[18], s);
    s = fma(D[29], Q[19], s);
    s = fma(D[35], Q[20], s);
    s = fma(D[36], Q[21], s);
    s = fma(D[37], Q[22], s);
    s = fma(D[38], Q[23], s);
    s = fma(D[39], Q[24], s);
    s = fma(D[40], Q[25], s);
    s = fma(D[41], Q[26], s);
    s = fma(D[42], Q[27], s);
    s = fma(D[43], Q[28], s);
    s = fma(D[44], Q[29], s);
    s = fma(D[45], Q[30], s);
    s = fma(D[46], Q[31], s);
    s = fma(D[47], Q[32], s);
    s = fma(D[48], Q[33], s);
    s = fma(D[49], Q[34], s);
    C[35] -= s; }
  { T s = D[2] * Q[0];
    s = fma(D[11], Q[4], s);
    s = fma(D[13], Q[5], s);
    s = fma(D[14], Q[6], s);
    s = fma(D[16], Q[7], s);
    s = fma(D[17], Q[8], s);
    s = fma(D[18], Q[9], s);
    s = fma(D[21], Q[10], s);
    s = fma(D[23], Q[11], s);
    s = fma(D[24], Q[12], s);
    s = fma(D[26], Q[13], s);
    s = fma(D[27], Q[14], s);
    s = fma(D[28], Q[15], s);
    s = fma(D[30], Q[16], s);
    s = fma(D[31], Q[17], s);
    s = fma(D[32], Q[18], s);
    s = fma(D[33], Q[19], s);
    s = fma(D[36], Q[20], s);
    s = fma(D[38], Q[21], s);
    s = fma(D[39], Q[22], s);
    s = fma(D[41], Q[23], s);
    s = fma(D[42], Q[24], s);
    s = fma(D[43], Q[25], s);
    s = fma(D[45], Q[26], s);
    s = fma(D[46], Q[27], s);
    s = fma(D[47], Q[28], s);
    s = fma(D[48], Q[29], s);
    s = fma(D[50], Q[30], s);
    s = fma(D[51], Q[31], s);
    s = fma(D[52], Q[32], s);
    s = fma(D[53], Q[33], s);
    s = fma(D[54], Q[34], s);
    C[36] -= s; }
  { T s = D[3] * Q[0];
    s = fma(D[12], Q[4], s);
    s = fma(D[14], Q[5], s);
    s = fma(D[15], Q[6], s);
    s = fma(D[17], Q[7], s);
    s = fma(D[18], Q[8], s);
    s = fma(D[19], Q[9], s);
    s = fma(D[22], Q[10], s);
    s = fma(D[24], Q[11], s);
    s = fma(D[25], Q[12], s);
    s = fma(D[27], Q[13], s);
    s = fma(D[28], Q[14], s);
    s = fma(D[29], Q[15], s);
    s = fma(D[31], Q[16], s);
    s = fma(D[32], Q[17], s);
    s = fma(D[33], Q[18], s);
    s = fma(D[34], Q[19], s);
    s = fma(D[37], Q[20], s);
    s = fma(D[39], Q[21], s);
    s = fma(D[40], Q[22], s);
    s = fma(D[42], Q[23], s);
    s = fma(D[43], Q[24], s);
    s = fma(D[44], Q[25], s);
    s = fma(D[46], Q[26], s);
    s = fma(D[47], Q[27], s);
    s = fma(D[48], Q[28], s);
    s = fma(D[49], Q[29], s);
    s = fma(D[51], Q[30], s);
    s = fma(D[52], Q[31], s);
    s = fma(D[53], Q[32], s);
    s = fma(D[54], Q[33], s);
    s = fma(D[55], Q[34], s);
    C[37] -= s; }
  { T s = D[4] * Q[0];
    s = fma(D[20], Q[4], s);
    s = fma(D[21], Q[5], s);
    s = fma(D[22], Q[6], s);
    s = fma(D[23], Q[7], s);
    s = fma(D[24], Q[8], s);
    s = fma(D[25], Q[9], s);
    s = fma(D[35], Q[10], s);
    s = fma(D[36], Q[11], s);
    s = fma(D[37], Q[12], s);
    s = fma(D[38], Q[13], s);
    s = fma(D[39], Q[14], s);
    s = fma(D[40], Q[15], s);
    s = fma(D[41], Q[16], s);
    s = fma(D[42], Q[17], s);
    s = fma(D[43], Q[18], s);
    s = fma(D[44], Q[19], s);
    C[38] += s; }
  { T s = D[5] * Q[0];
    s = fma(D[21], Q[4], s);
    s = fma(D[23], Q[5], s);
    s = fma(D[24], Q[6], s);
    s = fma(D[26], Q[7], s);
    s = fma(D[27], Q[8], s);
    s = fma(D[28], Q[9], s);
    s = fma(D[36], Q[10], s);
    s = fma(D[38], Q[11], s);
    s = fma(D[39], Q[12], s);
    s = fma(D[41], Q[13], s);
    s = fma(D[42], Q[14], s);
    s = fma(D[43], Q[15], s);
    s = fma(D[45], Q[16], s);
    s = fma(D[46], Q[17], s);
    s = fma(D[47], Q[18], s);
    s = fma(D[48], Q[19], s);
    C[39] += s; }
  { T s = D[6] * Q[0];
    s = fma(D[22], Q[4], s);
    s = fma(D[24], Q[5], s);
    s = fma(D[25], Q[6], s);
    s = fma(D[27], Q[7], s);
    s = fma(D[28], Q[8], s);
    s = fma(D[29], Q[9], s);
    s = fma(D[37], Q[10], s);
    s = fma(D[39], Q[11], s);
    s = fma(D[40], Q[12], s);
    s = fma(D[42], Q[13], s);
    s = fma(D[43], Q[14], s);
    s = fma(D[44], Q[15], s);
    s = fma(D[46], Q[16], s);
    s = fma(D[47], Q[17], s);
    s = fma(D[48], Q[18], s);
    s = fma(D[49], Q[19], s);
    C[40] += s; }
  { T s = D[7] * Q[0];
    s = fma(D[23], Q[4], s);
    s = fma(D[26], Q[5], s);
    s = fma(D[27], Q[6], s);
    s = fma(D[30], Q[7], s);
    s = fma(D[31], Q[8], s);
    s = fma(D[32], Q[9], s);
    s = fma(D[38], Q[10], s);
    s = fma(D[41], Q[11], s);
    s = fma(D[42], Q[12], s);
    s = fma(D[45], Q[13], s);
    s = fma(D[46], Q[14], s);
    s = fma(D[47], Q[15], s);
    s = fma(D[50], Q[16], s);
    s = fma(D[51], Q[17], s);
    s = fma(D[52], Q[18], s);
    s = fma(D[53], Q[19], s);
    C[41] += s; }
  { T s = D[8] * Q[0];
    s = fma(D[24], Q[4], s);
    s = fma(D[27], Q[5], s);
    s = fma(D[28], Q[6], s);
    s = fma(D[31], Q[7], s);
    s = fma(D[32], Q[8], s);
    s = fma(D[33], Q[9], s);
    s = fma(D[39], Q[10], s);
    s = fma(D[42], Q[11], s);
    s = fma(D[43], Q[12], s);
    s = fma(D[46], Q[13], s);
    s = fma(D[47], Q[14], s);
    s = fma(D[48], Q[15], s);
    s = fma(D[51], Q[16], s);
    s = fma(D[52], Q[17], s);
    s = fma(D[53], Q[18], s);
    s = fma(D[54], Q[19], s);
    C[42] += s; }
  { T s = D[9] * Q[0];
    s = fma(D[25], Q[4], s);
    s = fma(D[28], Q[5], s);
    s = fma(D[29], Q[6], s);
    s = fma(D[32], Q[7], s);
    s = fma(D[33], Q[8], s);
    s = fma(D[34], Q[9], s);
    s = fma(D[40], Q[10], s);
    s = fma(D[43], Q[11], s);
    s = fma(D[44], Q[12], s);
    s = fma(D[47], Q[13], s);
    s = fma(D[48], Q[14], s);
    s = fma(D[49], Q[15], s);
    s = fma(D[52], Q[16], s);
    s = fma(D[53], Q[17], s);
    s = fma(D[54], Q[18], s);
    s = fma(D[55], Q[19], s);
    C[43] += s; }
  { T s = D[10] * Q[0];
    s = fma(D[35], Q[4], s);
    s = fma(D[36], Q[5], s);
    s = fma(D[37], Q[6], s);
    s = fma(D[38], Q[7], s);
    s = fma(D[39], Q[8], s);
    s = fma(D[40], Q[9], s);
    C[44] -= s; }
  { T s = D[11] * Q[0];
    s = fma(D[36], Q[4], s);
    s = fma(D[38], Q[5], s);
    s = fma(D[39], Q[6], s);
    s = fma(D[41], Q[7], s);
    s = fma(D[42], Q[8], s);
    s = fma(D[43], Q[9], s);
    C[45] -= s; }
  { T s = D[12] * Q[0];
    s = fma(D[37], Q[4], s);
    s = fma(D[39], Q[5], s);
    s = fma(D[40], Q[6], s);
    s = fma(D[42], Q[7], s);
    s = fma(D[43], Q[8], s);
    s = fma(D[44], Q[9], s);
    C[46] -= s; }
  { T s = D[13] * Q[0];
    s = fma(D[38], Q[4], s);
    s = fma(D[41], Q[5], s);
    s = fma(D[42], Q[6], s);
    s = fma(D[45], Q[7], s);
    s = fma(D[46], Q[8], s);
    s = fma(D[47], Q[9], s);
    C[47] -= s; }
  { T s = D[14] * Q[0];
    s = fma(D[39], Q[4], s);
    s = fma(D[42], Q[5], s);
    s = fma(D[43], Q[6], s);
    s = fma(D[46], Q[7], s);
    s = fma(D[47], Q[8], s);
    s = fma(D[48], Q[9], s);
    C[48] -= s; }
  { T s = D[15] * Q[0];
    s = fma(D[40], Q[4], s);
    s = fma(D[43], Q[5], s);
    s = fma(D[44], Q[6], s);
    s = fma(D[47], Q[7], s);
    s = fma(D[48], Q[8], s);
    s = fma(D[49], Q[9], s);
    C[49] -= s; }
  { T s = D[16] * Q[0];
    s = fma(D[41], Q[4], s);
    s = fma(D[45], Q[5], s);
    s = fma(D[46], Q[6], s);
    s = fma(D[50], Q[7], s);
    s = fma(D[51], Q[8], s);
    s = fma(D[52], Q[9], s);
    C[50] -= s; }
  { T s = D[17] * Q[0];
    s = fma(D[42], Q[4], s);
    s = fma(D[46], Q[5], s);
    s = fma(D[47], Q[6], s);
    s = fma(D[51], Q[7], s);
    s = fma(D[52], Q[8], s);
    s = fma(D[53], Q[9], s);
    C[51] -= s; }
  { T s = D[18] * Q[0];
    s = fma(D[43], Q[4], s);
    s = fma(D[47], Q[5], s);
    s = fma(D[48], Q[6], s);
    s = fma(D[52], Q[7], s);
    s = fma(D[53], Q[8], s);
    s = fma(D[54], Q[9], s);
    C[52] -= s; }
  { T s = D[19] * Q[0];
    s = fma(D[44], Q[4], s);
    s = fma(D[48], Q[5], s);
    s = fma(D[49], Q[6], s);
    s = fma(D[53], Q[7], s);
    s = fma(D[54], Q[8], s);
    s = fma(D[55], Q[9], s);
    C[53] -= s; }
  { T s = D[20] * Q[0];
    C[54] += s; }
  { T s = D[21] * Q[0];
    C[55] += s; }
  { T s = D[22] * Q[0];
    C[56] += s; }
  { T s = D[23] * Q[0];
    C[57] += s; }
  { T s = D[24] * Q[0];
    C[58] += s; }
  { T s = D[25] * Q[0];
    C[59] += s; }
  { T s = D[26] * Q[0];
    C[60] += s; }
  { T s = D[27] * Q[0];
    C[61] += s; }
  { T s = D[28] * Q[0];
    C[62] += s; }
  { T s = D[29] * Q[0];
    C[63] += s; }
  { T s = D[30] * Q[0];
    C[64] += s; }
  { T s = D[31] * Q[0];
    C[65] += s; }
  { T s = D[32] * Q[0];
    C[66] += s; }
  { T s = D[33] * Q[0];
    C[67] += s; }
  { T s = D[34] * Q[0];
    C[68] += s; }
  { T s = D[35] * Q[0];
    C[69] -= s; }
  { T s = D[36] * Q[0];
    C[70] -= s; }
  { T s = D[37] * Q[0];
    C[71] -= s; }
  { T s = D[38] * Q[0];
    C[72] -= s; }
  { T s = D[39] * Q[0];
    C[73] -= s; }
  { T s = D[40] * Q[0];
    C[74] -= s; }
  { T s = D[41] * Q[0];
    C[75] -= s; }
  { T s = D[42] * Q[0];
    C[76] -= s; }
  { T s = D[43] * Q[0];
    C[77] -= s; }
  { T s = D[44] * Q[0];
    C[78] -= s; }
  { T s = D[45] * Q[0];
    C[79] -= s; }
  { T s = D[46] * Q[0];
    C[80] -= s; }
  { T s = D[47] * Q[0];
    C[81] -= s; }
  { T s = D[48] * Q[0];
    C[82] -= s; }
  { T s = D[49] * Q[0];
    C[83] -= s; }
  { T s = D[50] * Q[0];
    C[84] -= s; }
  { T s = D[51] * Q[0];
    C[85] -= s; }
  { T s = D[52] * Q[0];
    C[86] -= s; }
  { T s = D[53] * Q[0];
    C[87] -= s; }
  { T s = D[54] * Q[0];
    C[88] -= s; }
  { T s = D[55] * Q[0];
    C[89] -= s; }
}

template <typename T, typename C_T> __device__ __forceinline__ void sfmm_l2p_4(const T* am, const C_T* C, T* out) {
  T phi = T(0), ax = T(0), ay = T(0), az = T(0);
  phi = fma(am[0], T(C[0]), phi);
  ax = fma(am[0], T(C[35]), ax);
  ay = fma(am[0], T(C[36]), ay);
  az = fma(am[0], T(C[37]), az);
  phi = fma(am[1], T(C[1]), phi);
  ax = fma(am[1], T(C[38]), ax);
  ay = fma(am[1], T(C[39]), ay);
  az = fma(am[1], T(C[40]), az);
  phi = fma(am[2], T(C[2]), phi);
  ax = fma(am[2], T(C[39]), ax);
  ay = fma(am[2], T(C[41]), ay);
  az = fma(am[2], T(C[42]), az);
  phi = fma(am[3], T(C[3]), phi);
  ax = fma(am[3], T(C[40]), ax);
  ay = fma(am[3], T(C[42]), ay);
  az = fma(am[3], T(C[43]), az);
  phi = fma(am[4], T(C[4]), phi);
  ax = fma(am[4], T(C[44]), ax);
  ay = fma(am[4], T(C[45]), ay);
  az = fma(am[4], T(C[46]), az);
  phi = fma(am[5], T(C[5]), phi);
  ax = fma(am[5], T(C[45]), ax);
  ay = fma(am[5], T(C[47]), ay);
  az = fma(am[5], T(C[48]), az);
  phi = fma(am[6], T(C[6]), phi);
  ax = fma(am[6], T(C[46]), ax);
  ay = fma(am[6], T(C[48]), ay);
  az = fma(am[6], T(C[49]), az);
  phi = fma(am[7], T(C[7]), phi);
  ax = fma(am[7], T(C[47]), ax);
  ay = fma(am[7], T(C[50]), ay);
  az = fma(am[7], T(C[51]), az);
  phi = fma(am[8], T(C[8]), phi);
  ax = fma(am[8], T(C[48]), ax);
  ay = fma(am[8], T(C[51]), ay);
  az = fma(am[8], T(C[52]), az);
  phi = fma(am[9], T(C[9]), phi);
  ax = fma(am[9], T(C[49]), ax);
  ay = fma(am[9], T(C[52]), ay);
  az = fma(am[9], T(C[53]), az);
  phi = fma(am[10], T(C[10]), phi);
  ax = fma(am[10], T(C[54]), ax);
  ay = fma(am[10], T(C[55]), ay);
  az = fma(am[10], T(C[56]), az);
  phi = fma(am[11], T(C[11]), phi);
  ax = fma(am[11], T(C[55]), ax);
  ay = fma(am[11], T(C[57]), ay);
  az = fma(am[11], T(C[58]), az);
  phi = fma(am[12], T(C[12]), phi);
  ax = fma(am[12], T(C[56]), ax);
  ay = fma(am[12], T(C[58]), ay);
  az = fma(am[12], T(C[59]), az);
  phi = fma(am[13], T(C[13]), phi);
  ax = fma(am[13], T(C[57]), ax);
  ay = fma(am[13], T(C[60]), ay);
  az = fma(am[13], T(C[61]), az);
  phi = fma(am[14], T(C[14]), phi);
  ax = fma(am[14], T(C[58]), ax);
  ay = fma(am[14], T(C[61]), ay);
  az = fma(am[14], T(C[62]), az);
  phi = fma(am[15], T(C[15]), phi);
  ax = fma(am[15], T(C[59]), ax);
  ay = fma(am[15], T(C[62]), ay);
  az = fma(am[15], T(C[63]), az);
  phi = fma(am[16], T(C[16]), phi);
  ax = fma(am[16], T(C[60]), ax);
  ay = fma(am[16], T(C[64]), ay);
  az = fma(am[16], T(C[65]), az);
  phi = fma(am[17], T(C[17]), phi);
  ax = fma(am[17], T(C[61]), ax);
  ay = fma(am[17], T(C[65]), ay);
  az = fma(am[17], T(C[66]), az);
  phi = fma(am[18], T(C[18]), phi);
  ax = fma(am[18], T(C[62]), ax);
  ay = fma(am[18], T(C[66]), ay);
  az = fma(am[18], T(C[67]), az);
  phi = fma(am[19], T(C[19]), phi);
  ax = fma(am[19], T(C[63]), ax);
  ay = fma(am[19], T(C[67]), ay);
  az = fma(am[19], T(C[68]), az);
  phi = fma(am[20], T(C[20]), phi);
  ax = fma(am[20], T(C[69]), ax);
  ay = fma(am[20], T(C[70]), ay);
  az = fma(am[20], T(C[71]), az);
  phi = fma(am[21], T(C[21]), phi);
  ax = fma(am[21], T(C[70]), ax);
  ay = fma(am[21], T(C[72]), ay);
  az = fma(am[21], T(C[73]), az);
  phi = fma(am[22], T(C[22]), phi);
  ax = fma(am[22], T(C[71]), ax);
  ay = fma(am[22], T(C[73]), ay);
  az = fma(am[22], T(C[74]), az);
  phi = fma(am[23], T(C[23]), phi);
  ax = fma(am[23], T(C[72]), ax);
  ay = fma(am[23], T(C[75]), ay);
  az = fma(am[23], T(C[76]), az);
  phi = fma(am[24], T(C[24]), phi);
  ax = fma(am[24], T(C[73]), ax);
  ay = fma(am[24], T(C[76]), ay);
  az = fma(am[24], T(C[77]), az);
  phi = fma(am[25], T(C[25]), phi);
  ax = fma(am[25], T(C[74]), ax);
  ay = fma(am[25], T(C[77]), ay);
  az = fma(am[25], T(C[78]), az);
  phi = fma(am[26], T(C[26]), phi);
  ax = fma(am[26], T(C[75]), ax);
  ay = fma(am[26], T(C[79]), ay);
  az = fma(am[26], T(C[80]), az);
  phi = fma(am[27], T(C[27]), phi);
  ax = fma(am[27], T(C[76]), ax);
  ay = fma(am[27], T(C[80]), ay);
  az = fma(am[27], T(C[81]), az);
  phi = fma(am[28], T(C[28]), phi);
  ax = fma(am[28], T(C[77]), ax);
  ay = fma(am[28], T(C[81]), ay);
  az = fma(am[28], T(C[82]), az);
  phi = fma(am[29], T(C[29]), phi);
  ax = fma(am[29], T(C[78]), ax);
  ay = fma(am[29], T(C[82]), ay);
  az = fma(am[29], T(C[83]), az);
  phi = fma(am[30], T(C[30]), phi);
  ax = fma(am[30], T(C[79]), ax);
  ay = fma(am[30], T(C[84]), ay);
  az = fma(am[30], T(C[85]), az);
  phi = fma(am[31], T(C[31]), phi);
  ax = fma(am[31], T(C[80]), ax);
  ay = fma(am[31], T(C[85]), ay);
  az = fma(am[31], T(C[86]), az);
  phi = fma(am[32], T(C[32]), phi);
  ax = fma(am[32], T(C[81]), ax);
  ay = fma(am[32], T(C[86]), ay);
  az = fma(am[32], T(C[87]), az);
  phi = fma(am[33], T(C[33]), phi);
  ax = fma(am[33], T(C[82]), ax);
  ay = fma(am[33], T(C[87]), ay);
  az = fma(am[33], T(C[88]), az);
  phi = fma(am[34], T(C[34]), phi);
  ax = fma(am[34], T(C[83]), ax);
  ay = fma(am[34], T(C[88]), ay);
  az = fma(am[34], T(C[89]), az);
  out[0] = phi; out[1] = ax; out[2] = ay; out[3] = az;
}

template <typename T> __device__ __forceinline__ void sfmm_m2m_4(const T* gm, const T* Qc, T* Qp) {
  { T s = Qp[0];
    s = fma(gm[0], Qc[0], s);
    Qp[0] = s; }
  { T s = Qp[1];
    s = fma(gm[1], Qc[0], s);
    s = fma(gm[0], Qc[1], s);
    Qp[1] = s; }
  { T s = Qp[2];
    s = fma(gm[2], Qc[0], s);
    s = fma(gm[0], Qc[2], s);
    Qp[2] = s; }
  { T s = Qp[3];
    s = fma(gm[3], Qc[0], s);
    s = fma(gm[0], Qc[3], s);
    Qp[3] = s; }
  { T s = Qp[4];
    s = fma(gm[4], Qc[0], s);
    s = fma(gm[1], Qc[1], s);
    s = fma(gm[0], Qc[4], s);
    Qp[4] = s; }
  { T s = Qp[5];
    s = fma(gm[5], Qc[0], s);
    s = fma(gm[2], Qc[1], s);
    s = fma(gm[1], Qc[2], s);
    s = fma(gm[0], Qc[5], s);
    Qp[5] = s; }
  { T s = Qp[6];
    s = fma(gm[6], Qc[0], s);
    s = fma(gm[3], Qc[1], s);
    s = fma(gm[1], Qc[3], s);
    s = fma(gm[0], Qc[6], s);
    Qp[6] = s; }
  { T s = Qp[7];
    s = fma(gm[7], Qc[0], s);
    s = fma(gm[2], Qc[2], s);
    s = fma(gm[0], Qc[7], s);
    Qp[7] = s; }
  { T s = Qp[8];
    s = fma(gm[8], Qc[0], s);
    s = fma(gm[3], Qc[2], s);
    s = fma(gm[2], Qc[3], s);
    s = fma(gm[0], Qc[8], s);
    Qp[8] = s; }
  { T s = Qp[9];
    s = fma(gm[9], Qc[0], s);
    s = fma(gm[3], Qc[3], s);
    s = fma(gm[0], Qc[9], s);
    Qp[9] = s; }
  { T s = Qp[10];
    s = fma(gm[10], Qc[0], s);
    s = fma(gm[4], Qc[1], s);
    s = fma(gm[1], Qc[4], s);
    s = fma(gm[0], Qc[10], s);
    Qp[10] = s; }
  { T s = Qp[11];
    s = fma(gm[11], Qc[0], s);
    s = fma(gm[5], Qc[1], s);
    s = fma(gm[4], Qc[2], s);
    s = fma(gm[2], Qc[4], s);
    s = fma(gm[1], Qc[5], s);
    s = fma(gm[0], Qc[11], s);
    Qp[11] = s; }
  { T s = Qp[12];
    s = fma(gm[12], Qc[0], s);
    s = fma(gm[6], Qc[1], s);
    s = fma(gm[4], Qc[3], s);
    s = fma(gm[3], Qc[4], s);
    s = fma(gm[1], Qc[6], s);
    s = fma(gm[0], Qc[12], s);
    Qp[12] = s; }
  { T s = Qp[13];
    s = fma(gm[13], Qc[0], s);
    s = fma(gm[7], Qc[1], s);
    s = fma(gm[5], Qc[2], s);
    s = fma(gm[2], Qc[5], s);
    s = fma(gm[1], Qc[7], s);
    s = fma(gm[0], Qc[13], s);
    Qp[13] = s; }
  { T s = Qp[14];
    s = fma(gm[14], Qc[0], s);
    s = fma(gm[8], Qc[1], s);
    s = fma(gm[6], Qc[2], s);
    s = fma(gm[5], Qc[3], s);
    s = fma(gm[3], Qc[5], s);
    s = fma(gm[2], Qc[6], s);
    s = fma(gm[1], Qc[8], s);
    s = fma(gm[0], Qc[14], s);
    Qp[14] = s; }
  { T s = Qp[15];
    s = fma(gm[15], Qc[0], s);
    s = fma(gm[9], Qc[1], s);
    s = fma(gm[6], Qc[3], s);
    s = fma(gm[3], Qc[6], s);
    s = fma(gm[1], Qc[9], s);
    s = fma(gm[0], Qc[15], s);
    Qp[15] = s; }
  { T s = Qp[16];
    s = fma(gm[16], Qc[0], s);
    s = fma(gm[7], Qc[2], s);
    s = fma(gm[2], Qc[7], s);
    s = fma(gm[0], Qc[16], s);
    Qp[16] = s; }
  { T s = Qp[17];
    s = fma(gm[17], Qc[0], s);
    s = fma(gm[8], Qc[2], s);
    s = fma(gm[7], Qc[3], s);
    s = fma(gm[3], Qc[7], s);
    s = fma(gm[2], Qc[8], s);
    s = fma(gm[0], Qc[17], s);
    Qp[17] = s; }
  { T s = Qp[18];
    s = fma(gm[18], Qc[0], s);
    s = fma(gm[9], Qc[2], s);
    s = fma(gm[8], Qc[3], s);
    s = fma(gm[3], Qc[8], s);
    s = fma(gm[2], Qc[9], s);
    s = fma(gm[0], Qc[18], s);
    Qp[18] = s; }
  { T s = Qp[19];
    s = fma(gm[19], Qc[0], s);
    s = fma(gm[9], Qc[3], s);
    s = fma(gm[3], Qc[9], s);
    s = fma(gm[0], Qc[19], s);
    Qp[19] = s; }
  { T s = Qp[20];
    s = fma(gm[20], Qc[0], s);
    s = fma(gm[10], Qc[1], s);
    s = fma(gm[4], Qc[4], s);
    s = fma(gm[1], Qc[10], s);
    s = fma(gm[0], Qc[20], s);
    Qp[20] = s; }
  { T s = Qp[21];
    s = fma(gm[21], Qc[0], s);
    s = fma(gm[11], Qc[1], s);
    s = fma(gm[10], Qc[2], s);
    s = fma(gm[5], Qc[4], s);
    s = fma(gm[4], Qc[5], s);
    s = fma(gm[2], Qc[10], s);
    s = fma(gm[1], Qc[11], s);
    s = fma(gm[0], Qc[21], s);
    Qp[21] = s; }
  { T s = Qp[22];
    s = fma(gm[22], Qc[0], s);
    s = fma(gm[12], Qc[1], s);
    s = fma(gm[10], Qc[3], s);
    s = fma(gm[6], Qc[4], s);
    s = fma(gm[4], Qc[6], s);
    s = fma(gm[3], Qc[10], s);
    s = fma(gm[1], Qc[12], s);
    s = fma(gm[0], Qc[22], s);
    Qp[22] = s; }
  { T s = Qp[23];
    s = fma(gm[23], Qc[0], s);
    s = fma(gm[13], Qc[1], s);
    s = fma(gm[11], Qc[2], s);
    s = fma(gm[7], Qc[4], s);
    s = fma(gm[5], Qc[5], s);
    s = fma(gm[4], Qc[7], s);
    s = fma(gm[2], Qc[11], s);
    s = fma(gm[1], Qc[13], s);
    s = fma(gm[0], Qc[23], s);
    Qp[23] = s; }
  { T s = Qp[24];
    s = fma(gm[24], Qc[0], s);
    s = fma(gm[14], Qc[1], s);
    s = fma(gm[12], Qc[2], s);
    s = fma(gm[11], Qc[3], s);
    s = fma(gm[8], Qc[4], s);
    s = fma(gm[6], Qc[5], s);
    s = fma(gm[5], Qc[6], s);
    s = fma(gm[4], Qc[8], s);
    s = fma(gm[3], Qc[11], s);
    s = fma(gm[2], Qc[12], s);
    s = fma(gm[1], Qc[14], s);
    s = fma(gm[0], Qc[24], s);
    Qp[24] = s; }
  { T s = Qp[25];
    s = fma(gm[25], Qc[0], s);
    s = fma(gm[15], Qc[1], s);
    s = fma(gm[12], Qc[3], s);
    s = fma(gm[9], Qc[4], s);
    s = fma(gm[6], Qc[6], s);
    s = fma(gm[4], Qc[9], s);
    s = fma(gm[3], Qc[12], s);
    s = fma(gm[1], Qc[15], s);
    s = fma(gm[0], Qc[25], s);
    Qp[25] = s; }
  { T s = Qp[26];
    s = fma(gm[26], Qc[0], s);
    s = fma(gm[16], Qc[1], s);
    s = fma(gm[13], Qc[2], s);
    s = fma(gm[7], Qc[5], s);
    s = fma(gm[5], Qc[7], s);
    s = fma(gm[2], Qc[13], s);
    s = fma(gm[1], Qc[16], s);
    s = fma(gm[0], Qc[26], s);
    Qp[26] = s; }
  { T s = Qp[27];
    s = fma(gm[27], Qc[0], s);
    s = fma(gm[17], Qc[1], s);
    s = fma(gm[14], Qc[2], s);
    s = fma(gm[13], Qc[3], s);
    s = fma(gm[8], Qc[5], s);
    s = fma(gm[7], Qc[6], s);
    s = fma(gm[6], Qc[7], s);
    s = fma(gm[5], Qc[8], s);
    s = fma(gm[3], Qc[13], s);
    s = fma(gm[2], Qc[14], s);
    s = fma(gm[1], Qc[17], s);
    s = fma(gm[0], Qc[27], s);
    Qp[27] = s; }
  { T s = Qp[28];
    s = fma(gm[28], Qc[0], s);
    s = fma(gm[18], Qc[1], s);
    s = fma(gm[15], Qc[2], s);
    s = fma(gm[14], Qc[3], s);
    s = fma(gm[9], Qc[5], s);
    s = fma(gm[8], Qc[6], s);
    s = fma(gm[6], Qc[8], s);
    s = fma(gm[5], Qc[9], s);
    s = fma(gm[3], Qc[14], s);
    s = fma(gm[2], Qc[15], s);
    s = fma(gm[1], Qc[18], s);
    s = fma(gm[0], Qc[28], s);
    Qp[28] = s; }
  { T s = Qp[29];
    s = fma(gm[29], Qc[0], s);
    s = fma(gm[19], Qc[1], s);
    s = fma(gm[15], Qc[3], s);
    s = fma(gm[9], Qc[6], s);
    s = fma(gm[6], Qc[9], s);
    s = fma(gm[3], Qc[15], s);
    s = fma(gm[1], Qc[19], s);
    s = fma(gm[0], Qc[29], s);
    Qp[29] = s; }
  { T s = Qp[30];
    s = fma(gm[30], Qc[0], s);
    s = fma(gm[16], Qc[2], s);
    s = fma(gm[7], Qc[7], s);
    s = fma(gm[2], Qc[16], s);
    s = fma(gm[0], Qc[30], s);
    Qp[30] = s; }
  { T s = Qp[31];
    s = fma(gm[31], Qc[0], s);
    s = fma(gm[17], Qc[2], s);
    s = fma(gm[16], Qc[3], s);
    s = fma(gm[8], Qc[7], s);
    s = fma(gm[7], Qc[8], s);
    s = fma(gm[3], Qc[16], s);
    s = fma(gm[2], Qc[17], s);
    s = fma(gm[0], Qc[31], s);
    Qp[31] = s; }
  { T s = Qp[32];
    s = fma(gm[32], Qc[0], s);
    s = fma(gm[18], Qc[2], s);
    s = fma(gm[17], Qc[3], s);
    s = fma(gm[9], Qc[7], s);
    s = fma(gm[8], Qc[8], s);
    s = fma(gm[7], Qc[9], s);
    s = fma(gm[3], Qc[17], s);
    s = fma(gm[2], Qc[18], s);
    s = fma(gm[0], Qc[32], s);
    Qp[32] = s; }
  { T s = Qp[33];
    s = fma(gm[33], Qc[0], s);
    s = fma(gm[19], Qc[2], s);
    s = fma(gm[18], Qc[3], s);
    s = fma(gm[9], Qc[8], s);
    s = fma(gm[8], Qc[9], s);
    s = fma(gm[3], Qc[18], s);
    s = fma(gm[2], Qc[19], s);
    s = fma(gm[0], Qc[33], s);
    Qp[33] = s; }
  { T s = Qp[34];
    s = fma(gm[34], Qc[0], s);
    s = fma(gm[19], Qc[3], s);
    s = fma(gm[9], Qc[9], s);
    s = fma(gm[3], Qc[19], s);
    s = fma(gm[0], Qc[34], s);
    Qp[34] = s; }
}

#define SFMM_NT_4 34  /* steps of the L2L translation */
static __device__ const unsigned short sfmm_l2l_steps_4[34][96] = {
  {257, 260, 261, 262, 266, 267, 268, 269, 270, 271, 276, 277, 278, 279, 280, 281, 282, 283, 284, 285, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 294, 295, 296, 300, 301, 302, 303, 304, 305, 310, 311, 312, 313, 314, 315, 316, 317, 318, 319, 325, 326, 327, 328, 329, 330, 331, 332, 333, 334, 335, 336, 337, 338, 339, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {514, 517, 519, 520, 523, 525, 526, 528, 529, 530, 533, 535, 536, 538, 539, 540, 542, 543, 544, 545, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 551, 553, 554, 557, 559, 560, 562, 563, 564, 567, 569, 570, 572, 573, 574, 576, 577, 578, 579, 582, 584, 585, 587, 588, 589, 591, 592, 593, 594, 596, 597, 598, 599, 600, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {771, 774, 776, 777, 780, 782, 783, 785, 786, 787, 790, 792, 793, 795, 796, 797, 799, 800, 801, 802, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 808, 810, 811, 814, 816, 817, 819, 820, 821, 824, 826, 827, 829, 830, 831, 833, 834, 835, 836, 839, 841, 842, 844, 845, 846, 848, 849, 850, 851, 853, 854, 855, 856, 857, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1028, 1034, 1035, 1036, 1044, 1045, 1046, 1047, 1048, 1049, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1068, 1069, 1070, 1078, 1079, 1080, 1081, 1082, 1083, 1093, 1094, 1095, 1096, 1097, 1098, 1099, 1100, 1101, 1102, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1285, 1291, 1293, 1294, 1301, 1303, 1304, 1306, 1307, 1308, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1325, 1327, 1328, 1335, 1337, 1338, 1340, 1341, 1342, 1350, 1352, 1353, 1355, 1356, 1357, 1359, 1360, 1361, 1362, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1542, 1548, 1550, 1551, 1558, 1560, 1561, 1563, 1564, 1565, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1582, 1584, 1585, 1592, 1594, 1595, 1597, 1598, 1599, 1607, 1609, 1610, 1612, 1613, 1614, 1616, 1617, 1618, 1619, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {1799, 1805, 1808, 1809, 1815, 1818, 1819, 1822, 1823, 1824, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1839, 1842, 1843, 1849, 1852, 1853, 1856, 1857, 1858, 1864, 1867, 1868, 1871, 1872, 1873, 1876, 1877, 1878, 1879, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2056, 2062, 2065, 2066, 2072, 2075, 2076, 2079, 2080, 2081, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2096, 2099, 2100, 2106, 2109, 2110, 2113, 2114, 2115, 2121, 2124, 2125, 2128, 2129, 2130, 2133, 2134, 2135, 2136, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2313, 2319, 2322, 2323, 2329, 2332, 2333, 2336, 2337, 2338, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2353, 2356, 2357, 2363, 2366, 2367, 2370, 2371, 2372, 2378, 2381, 2382, 2385, 2386, 2387, 2390, 2391, 2392, 2393, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2570, 2580, 2581, 2582, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2614, 2615, 2616, 2629, 2630, 2631, 2632, 2633, 2634, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {2827, 2837, 2839, 2840, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2871, 2873, 2874, 2886, 2888, 2889, 2891, 2892, 2893, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3084, 3094, 3096, 3097, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3128, 3130, 3131, 3143, 3145, 3146, 3148, 3149, 3150, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3341, 3351, 3354, 3355, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3385, 3388, 3389, 3400, 3403, 3404, 3407, 3408, 3409, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3598, 3608, 3611, 3612, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3642, 3645, 3646, 3657, 3660, 3661, 3664, 3665, 3666, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {3855, 3865, 3868, 3869, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3899, 3902, 3903, 3914, 3917, 3918, 3921, 3922, 3923, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4112, 4122, 4126, 4127, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4156, 4160, 4161, 4171, 4175, 4176, 4180, 4181, 4182, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4369, 4379, 4383, 4384, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4413, 4417, 4418, 4428, 4432, 4433, 4437, 4438, 4439, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4626, 4636, 4640, 4641, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4670, 4674, 4675, 4685, 4689, 4690, 4694, 4695, 4696, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {4883, 4893, 4897, 4898, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 4927, 4931, 4932, 4942, 4946, 4947, 4951, 4952, 4953, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {5140, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 5189, 5190, 5191, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {5397, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 5446, 5448, 5449, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {5654, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 5703, 5705, 5706, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {5911, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 5960, 5963, 5964, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {6168, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 6217, 6220, 6221, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {6425, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 6474, 6477, 6478, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {6682, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 6731, 6735, 6736, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {6939, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 6988, 6992, 6993, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {7196, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 7245, 7249, 7250, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {7453, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 7502, 7506, 7507, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {7710, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 7759, 7764, 7765, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {7967, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 8016, 8021, 8022, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {8224, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 8273, 8278, 8279, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {8481, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 8530, 8535, 8536, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {8738, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 8787, 8792, 8793, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static const int sfmm_moment_mi_4[35][3] = {{0,0,0}, {1,0,0}, {0,1,0}, {0,0,1}, {2,0,0}, {1,1,0}, {1,0,1}, {0,2,0}, {0,1,1}, {0,0,2}, {3,0,0}, {2,1,0}, {2,0,1}, {1,2,0}, {1,1,1}, {1,0,2}, {0,3,0}, {0,2,1}, {0,1,2}, {0,0,3}, {4,0,0}, {3,1,0}, {3,0,1}, {2,2,0}, {2,1,1}, {2,0,2}, {1,3,0}, {1,2,1}, {1,1,2}, {1,0,3}, {0,4,0}, {0,3,1}, {0,2,2}, {0,1,3}, {0,0,4}};

#define SFMM_MT_4 12  /* steps of the M2M translation */
static __device__ const unsigned short sfmm_m2m_steps_4[12][64] = {
  {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 256, 512, 768, 257, 258, 259, 514, 515, 771, 260, 261, 262, 263, 264, 265, 519, 520, 521, 777, 266, 267, 268, 269, 270, 271, 272, 273, 274, 275, 528, 529, 530, 531, 787, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 1024, 513, 769, 1792, 770, 2304, 1025, 516, 772, 517, 518, 774, 1794, 775, 776, 2307, 1028, 522, 778, 523, 524, 780, 525, 526, 527, 783, 1799, 784, 785, 786, 2313, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 1280, 1536, 65535, 2048, 65535, 2560, 1026, 1027, 1282, 773, 1539, 4096, 1795, 2051, 4864, 2561, 1029, 1030, 1031, 779, 1033, 1287, 781, 782, 1545, 4098, 1800, 1801, 2057, 4867, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 1281, 1537, 1793, 1283, 2305, 65535, 2050, 2306, 65535, 5120, 1284, 1540, 1285, 1032, 1542, 1797, 1288, 1289, 2310, 7680, 2055, 2056, 2312, 8704, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2816, 3072, 3328, 1538, 3840, 65535, 4352, 4608, 65535, 65535, 2562, 2563, 1796, 1286, 2308, 3330, 1543, 1544, 3843, 65535, 4099, 2311, 4611, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 2049, 65535, 65535, 65535, 65535, 65535, 65535, 2817, 3073, 2818, 1541, 3075, 4097, 1798, 2054, 4865, 65535, 4354, 4355, 4866, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3584, 65535, 65535, 65535, 65535, 65535, 65535, 5376, 5632, 3329, 2052, 3841, 6656, 2053, 2309, 7424, 65535, 7936, 4610, 8448, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 5888, 2819, 6400, 65535, 3331, 3587, 65535, 65535, 65535, 8192, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3074, 65535, 65535, 3586, 3842, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 3585, 65535, 65535, 4353, 4609, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535},
  {65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 6144, 65535, 65535, 6912, 7168, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535, 65535}};
static __device__ const unsigned short sfmm_moment_exp_4[35] = {0, 1, 8, 64, 2, 9, 65, 16, 72, 128, 3, 10, 66, 17, 73, 129, 24, 80, 136, 192, 4, 11, 67, 18, 74, 130, 25, 81, 137, 193, 32, 88, 144, 200, 256};

template <typename T> __device__ __forceinline__ void sfmm_fold_4(const T* Q, T* q) {
  q[0] = Q[0];
  q[1] = Q[4] - Q[9];
  q[2] = Q[5];
  q[3] = Q[6];
  q[4] = Q[7] - Q[9];
  q[5] = Q[8];
  q[6] = Q[10] - Q[15];
  q[7] = Q[11] - Q[18];
  q[8] = Q[12] - Q[19];
  q[9] = Q[13] - Q[15];
  q[10] = Q[14];
  q[11] = Q[16] - Q[18];
  q[12] = Q[17] - Q[19];
  q[13] = Q[20] - Q[25] + Q[34];
  q[14] = Q[21] - Q[28];
  q[15] = Q[22] - Q[29];
  q[16] = Q[23] - Q[25] - Q[32] + T(2.0) * Q[34];
  q[17] = Q[24] - Q[33];
  q[18] = Q[26] - Q[28];
  q[19] = Q[27] - Q[29];
  q[20] = Q[30] - Q[32] + Q[34];
  q[21] = Q[31] - Q[33];
}

template <typename T> __device__ __forceinline__ void sfmm_m2l_fold_4(const T* D, const T* q, T* C) {
  { T s = D[4] * q[1];
    s = fma(D[5], q[2], s);
    s = fma(D[6], q[3], s);
    s = fma(D[7], q[4], s);
    s = fma(D[8], q[5], s);
    s = fma(D[10], q[6], s);
    s = fma(D[11], q[7], s);
    s = fma(D[12], q[8], s);
    s = fma(D[13], q[9], s);
    s = fma(D[14], q[10], s);
    s = fma(D[16], q[11], s);
    s = fma(D[17], q[12], s);
    s = fma(D[20], q[13], s);
    s = fma(D[21], q[14], s);
    s = fma(D[22], q[15], s);
    s = fma(D[23], q[16], s);
    s = fma(D[24], q[17], s);
    s = fma(D[26], q[18], s);
    s = fma(D[27], q[19], s);
    s = fma(D[30], q[20], s);
    s = fma(D[31], q[21], s);
    C[0] += fma(D[0], q[0], s); }
  { T s = D[10] * q[1];
    s = fma(D[11], q[2], s);
    s = fma(D[12], q[3], s);
    s = fma(D[13], q[4], s);
    s = fma(D[14], q[5], s);
    s = fma(D[20], q[6], s);
    s = fma(D[21], q[7], s);
    s = fma(D[22], q[8], s);
    s = fma(D[23], q[9], s);
    s = fma(D[24], q[10], s);
    s = fma(D[26], q[11], s);
    s = fma(D[27], q[12], s);
    C[1] += fma(D[1], q[0], s); }
  { T s = D[11] * q[1];
    s = fma(D[13], q[2], s);
    s = fma(D[14], q[3], s);
    s = fma(D[16], q[4], s);
    s = fma(D[17], q[5], s);
    s = fma(D[21], q[6], s);
    s = fma(D[23], q[7], s);
    s = fma(D[24], q[8], s);
    s = fma(D[26], q[9], s);
    s = fma(D[27], q[10], s);
    s = fma(D[30], q[11], s);
    s = fma(D[31], q[12], s);
    C[2] += fma(D[2], q[0], s); }
  { T s = D[12] * q[1];
    s = fma(D[14], q[2], s);
    s = fma(D[15], q[3], s);
    s = fma(D[17], q[4], s);
    s = fma(D[18], q[5], s);
    s = fma(D[22], q[6], s);
    s = fma(D[24], q[7], s);
    s = fma(D[25], q[8], s);
    s = fma(D[27], q[9], s);
    s = fma(D[28], q[10], s);
    s = fma(D[31], q[11], s);
    s = fma(D[32], q[12], s);
    C[3] += fma(D[3], q[0], s); }
  { T s = D[20] * q[1];
    s = fma(D[21], q[2], s);
    s = fma(D[22], q[3], s);
    s = fma(D[23], q[4], s);
    s = fma(D[24], q[5], s);
    C[4] += fma(D[4], q[0], s); }
  { T s = D[21] * q[1];
    s = fma(D[23], q[2], s);
    s = fma(D[24], q[3], s);
    s = fma(D[26], q[4], s);
    s = fma(D[27], q[5], s);
    C[5] += fma(D[5], q[0], s); }
  { T s = D[22] * q[1];
    s = fma(D[24], q[2], s);
    s = fma(D[25], q[3], s);
    s = fma(D[27], q[4], s);
    s = fma(D[28], q[5], s);
    C[6] += fma(D[6], q[0], s); }
  { T s = D[23] * q[1];
    s = fma(D[26], q[2], s);
    s = fma(D[27], q[3], s);
    s = fma(D[30], q[4], s);
    s = fma(D[31], q[5], s);
    C[7] += fma(D[7], q[0], s); }
  { T s = D[24] * q[1];
    s = fma(D[27], q[2], s);
    s = fma(D[28], q[3], s);
    s = fma(D[31], q[4], s);
    s = fma(D[32], q[5], s);
    C[8] += fma(D[8], q[0], s); }
  C[9] = fma(D[10], q[0], C[9]);
  C[10] = fma(D[11], q[0], C[10]);
  C[11] = fma(D[12], q[0], C[11]);
  C[12] = fma(D[13], q[0], C[12]);
  C[13] = fma(D[14], q[0], C[13]);
  C[14] = fma(D[16], q[0], C[14]);
  C[15] = fma(D[17], q[0], C[15]);
  C[16] = fma(D[20], q[0], C[16]);
  C[17] = fma(D[21], q[0], C[17]);
  C[18] = fma(D[22], q[0], C[18]);
  C[19] = fma(D[23], q[0], C[19]);
  C[20] = fma(D[24], q[0], C[20]);
  C[21] = fma(D[26], q[0], C[21]);
  C[22] = fma(D[27], q[0], C[22]);
  C[23] = fma(D[30], q[0], C[23]);
  C[24] = fma(D[31], q[0], C[24]);
  C[25] = fma(D[35], q[13], C[25]);
  C[25] = fma(D[36], q[14], C[25]);
  C[25] = fma(D[37], q[15], C[25]);
  C[25] = fma(D[38], q[16], C[25]);
  C[25] = fma(D[39], q[17], C[25]);
  C[25] = fma(D[41], q[18], C[25]);
  C[25] = fma(D[42], q[19], C[25]);
  C[25] = fma(D[45], q[20], C[25]);
  C[25] = fma(D[46], q[21], C[25]);
  C[26] = fma(D[36], q[13], C[26]);
  C[26] = fma(D[38], q[14], C[26]);
  C[26] = fma(D[39], q[15], C[26]);
  C[26] = fma(D[41], q[16], C[26]);
  C[26] = fma(D[42], q[17], C[26]);
  C[26] = fma(D[45], q[18], C[26]);
  C[26] = fma(D[46], q[19], C[26]);
  C[26] = fma(D[50], q[20], C[26]);
  C[26] = fma(D[51], q[21], C[26]);
  C[27] = fma(D[37], q[13], C[27]);
  C[27] = fma(D[39], q[14], C[27]);
  C[27] = fma(D[40], q[15], C[27]);
  C[27] = fma(D[42], q[16], C[27]);
  C[27] = fma(D[43], q[17], C[27]);
  C[27] = fma(D[46], q[18], C[27]);
  C[27] = fma(D[47], q[19], C[27]);
  C[27] = fma(D[51], q[20], C[27]);
  C[27] = fma(D[52], q[21], C[27]);
  C[28] = fma(D[35], q[6], C[28]);
  C[28] = fma(D[36], q[7], C[28]);
  C[28] = fma(D[37], q[8], C[28]);
  C[28] = fma(D[38], q[9], C[28]);
  C[28] = fma(D[39], q[10], C[28]);
  C[28] = fma(D[41], q[11], C[28]);
  C[28] = fma(D[42], q[12], C[28]);
  C[29] = fma(D[36], q[6], C[29]);
  C[29] = fma(D[38], q[7], C[29]);
  C[29] = fma(D[39], q[8], C[29]);
  C[29] = fma(D[41], q[9], C[29]);
  C[29] = fma(D[42], q[10], C[29]);
  C[29] = fma(D[45], q[11], C[29]);
  C[29] = fma(D[46], q[12], C[29]);
  C[30] = fma(D[37], q[6], C[30]);
  C[30] = fma(D[39], q[7], C[30]);
  C[30] = fma(D[40], q[8], C[30]);
  C[30] = fma(D[42], q[9], C[30]);
  C[30] = fma(D[43], q[10], C[30]);
  C[30] = fma(D[46], q[11], C[30]);
  C[30] = fma(D[47], q[12], C[30]);
  C[31] = fma(D[38], q[6], C[31]);
  C[31] = fma(D[41], q[7], C[31]);
  C[31] = fma(D[42], q[8], C[31]);
  C[31] = fma(D[45], q[9], C[31]);
  C[31] = fma(D[46], q[10], C[31]);
  C[31] = fma(D[50], q[11], C[31]);
  C[31] = fma(D[51], q[12], C[31]);
  C[32] = fma(D[39], q[6], C[32]);
  C[32] = fma(D[42], q[7], C[32]);
  C[32] = fma(D[43], q[8], C[32]);
  C[32] = fma(D[46], q[9], C[32]);
  C[32] = fma(D[47], q[10], C[32]);
  C[32] = fma(D[51], q[11], C[32]);
  C[32] = fma(D[52], q[12], C[32]);
  C[33] = fma(D[35], q[1], C[33]);
  C[33] = fma(D[36], q[2], C[33]);
  C[33] = fma(D[37], q[3], C[33]);
  C[33] = fma(D[38], q[4], C[33]);
  C[33] = fma(D[39], q[5], C[33]);
  C[34] = fma(D[36], q[1], C[34]);
  C[34] = fma(D[38], q[2], C[34]);
  C[34] = fma(D[39], q[3], C[34]);
  C[34] = fma(D[41], q[4], C[34]);
  C[34] = fma(D[42], q[5], C[34]);
  C[35] = fma(D[37], q[1], C[35]);
  C[35] = fma(D[39], q[2], C[35]);
  C[35] = fma(D[40], q[3], C[35]);
  C[35] = fma(D[42], q[4], C[35]);
  C[35] = fma(D[43], q[5], C[35]);
  C[36] = fma(D[38], q[1], C[36]);
  C[36] = fma(D[41], q[2], C[36]);
  C[36] = fma(D[42], q[3], C[36]);
  C[36] = fma(D[45], q[4], C[36]);
  C[36] = fma(D[46], q[5], C[36]);
  C[37] = fma(D[39], q[1], C[37]);
  C[37] = fma(D[42], q[2], C[37]);
  C[37] = fma(D[43], q[3], C[37]);
  C[37] = fma(D[46], q[4], C[37]);
  C[37] = fma(D[47], q[5], C[37]);
  C[38] = fma(D[41], q[1], C[38]);
  C[38] = fma(D[45], q[2], C[38]);
  C[38] = fma(D[46], q[3], C[38]);
  C[38] = fma(D[50], q[4], C[38]);
  C[38] = fma(D[51], q[5], C[38]);
  C[39] = fma(D[42], q[1], C[39]);
  C[39] = fma(D[46], q[2], C[39]);
  C[39] = fma(D[47], q[3], C[39]);
  C[39] = fma(D[51], q[4], C[39]);
  C[39] = fma(D[52], q[5], C[39]);
  C[40] = fma(D[35], q[0], C[40]);
  C[41] = fma(D[36], q[0], C[41]);
  C[42] = fma(D[37], q[0], C[42]);
  C[43] = fma(D[38], q[0], C[43]);
  C[44] = fma(D[39], q[0], C[44]);
  C[45] = fma(D[41], q[0], C[45]);
  C[46] = fma(D[42], q[0], C[46]);
  C[47] = fma(D[45], q[0], C[47]);
  C[48] = fma(D[46], q[0], C[48]);
  C[49] = fma(D[50], q[0], C[49]);
  C[50] = fma(D[51], q[0], C[50]);
}

#define SFMM_NR_4 22  /* entries of a source row */
#define SFMM_NS_4 51  /* sums of an interaction */
#define SFMM_NX_4 4
static __device__ const signed char sfmm_unfold_4[90][4][2] = {
  {{0, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{1, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{2, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{3, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{4, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{5, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{6, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{7, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{8, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{4, -1}, {7, -1}, {0, 0}, {0, 0}},
  {{9, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{10, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{11, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{12, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{13, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{9, 1}, {12, 1}, {0, 0}, {0, 0}},
  {{14, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{15, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{10, 1}, {14, 1}, {0, 0}, {0, 0}},
  {{11, 1}, {15, 1}, {0, 0}, {0, 0}},
  {{16, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{17, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{18, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{19, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{20, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{16, -1}, {19, -1}, {0, 0}, {0, 0}},
  {{21, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{22, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{17, -1}, {21, -1}, {0, 0}, {0, 0}},
  {{18, -1}, {22, -1}, {0, 0}, {0, 0}},
  {{23, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{24, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{19, -1}, {23, -1}, {0, 0}, {0, 0}},
  {{20, -1}, {24, -1}, {0, 0}, {0, 0}},
  {{16, 1}, {19, 2}, {23, 1}, {0, 0}},
  {{1, -1}, {25, -1}, {0, 0}, {0, 0}},
  {{2, -1}, {26, -1}, {0, 0}, {0, 0}},
  {{3, -1}, {27, -1}, {0, 0}, {0, 0}},
  {{4, 1}, {28, 1}, {0, 0}, {0, 0}},
  {{5, 1}, {29, 1}, {0, 0}, {0, 0}},
  {{6, 1}, {30, 1}, {0, 0}, {0, 0}},
  {{7, 1}, {31, 1}, {0, 0}, {0, 0}},
  {{8, 1}, {32, 1}, {0, 0}, {0, 0}},
  {{4, -1}, {28, -1}, {7, -1}, {31, -1}},
  {{9, -1}, {33, -1}, {0, 0}, {0, 0}},
  {{10, -1}, {34, -1}, {0, 0}, {0, 0}},
  {{11, -1}, {35, -1}, {0, 0}, {0, 0}},
  {{12, -1}, {36, -1}, {0, 0}, {0, 0}},
  {{13, -1}, {37, -1}, {0, 0}, {0, 0}},
  {{9, 1}, {33, 1}, {12, 1}, {36, 1}},
  {{14, -1}, {38, -1}, {0, 0}, {0, 0}},
  {{15, -1}, {39, -1}, {0, 0}, {0, 0}},
  {{10, 1}, {34, 1}, {14, 1}, {38, 1}},
  {{11, 1}, {35, 1}, {15, 1}, {39, 1}},
  {{16, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{17, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{18, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{19, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{20, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{16, -1}, {19, -1}, {0, 0}, {0, 0}},
  {{21, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{22, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{17, -1}, {21, -1}, {0, 0}, {0, 0}},
  {{18, -1}, {22, -1}, {0, 0}, {0, 0}},
  {{23, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{24, 1}, {0, 0}, {0, 0}, {0, 0}},
  {{19, -1}, {23, -1}, {0, 0}, {0, 0}},
  {{20, -1}, {24, -1}, {0, 0}, {0, 0}},
  {{16, 1}, {19, 2}, {23, 1}, {0, 0}},
  {{40, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{41, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{42, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{43, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{44, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{40, 1}, {43, 1}, {0, 0}, {0, 0}},
  {{45, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{46, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{41, 1}, {45, 1}, {0, 0}, {0, 0}},
  {{42, 1}, {46, 1}, {0, 0}, {0, 0}},
  {{47, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{48, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{43, 1}, {47, 1}, {0, 0}, {0, 0}},
  {{44, 1}, {48, 1}, {0, 0}, {0, 0}},
  {{40, -1}, {43, -2}, {47, -1}, {0, 0}},
  {{49, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{50, -1}, {0, 0}, {0, 0}, {0, 0}},
  {{45, 1}, {49, 1}, {0, 0}, {0, 0}},
  {{46, 1}, {50, 1}, {0, 0}, {0, 0}},
  {{41, -1}, {45, -2}, {49, -1}, {0, 0}},
  {{42, -1}, {46, -2}, {50, -1}, {0, 0}}};

template <typename T> __device__ __forceinline__ void sfmm_derivs_fold_1(T x, T y, T z, T rinv, T* D) {
  const T ri2 = rinv * rinv, b0 = rinv;
  const T b1 = b0 * (ri2 * T(-1.0));
  const T R0_100 = x * b1;
  const T R0_010 = y * b1;
  const T R0_001 = z * b1;
  D[0] = b0;
  D[1] = R0_100;
  D[2] = R0_010;
  D[3] = R0_001;
}

template <typename T> __device__ __forceinline__ void sfmm_uderivs_fold_1(T x, T y, T z, T rinv, T* D) {
  const T R0_100 = x * T(-1.0);
  const T R0_010 = y * T(-1.0);
  const T R0_001 = z * T(-1.0);
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_fold_2(T x, T y, T z, T rinv, T* D) {
  const T ri2 = rinv * rinv, b0 = rinv;
  const T b1 = b0 * (ri2 * T(-1.0));
  const T b2 = b1 * (ri2 * T(-3.0));
  const T R0_100 = x * b1;
  const T R0_010 = y * b1;
  const T R0_001 = z * b1;
  const T R1_100 = x * b2;
  const T R0_200 = fma(x, R1_100, b1);
  const T R1_010 = y * b2;
  const T R0_110 = x * R1_010;
  const T R1_001 = z * b2;
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, b1);
  const T R0_011 = y * R1_001;
  D[0] = b0;
  D[1] = R0_100;
  D[2] = R0_010;
  D[3] = R0_001;
  D[4] = R0_200;
  D[5] = R0_110;
  D[6] = R0_101;
  D[7] = R0_020;
  D[8] = R0_011;
}

template <typename T> __device__ __forceinline__ void sfmm_uderivs_fold_2(T x, T y, T z, T rinv, T* D) {
  const T R0_100 = x * T(-1.0);
  const T R0_010 = y * T(-1.0);
  const T R0_001 = z * T(-1.0);
  const T R1_100 = x * T(3.0);
  const T R0_200 = fma(x, R1_100, T(-1.0));
  const T R1_010 = y * T(3.0);
  const T R0_110 = x * R1_010;
  const T R1_001 = z * T(3.0);
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, T(-1.0));
  const T R0_011 = y * R1_001;
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_fold_3(T x, T y, T z, T rinv, T* D) {
  const T ri2 = rinv * rinv, b0 = rinv;
  const T b1 = b0 * (ri2 * T(-1.0));
  const T b2 = b1 * (ri2 * T(-3.0));
  const T b3 = b2 * (ri2 * T(-5.0));
  const T R0_100 = x * b1;
  const T R0_010 = y * b1;
  const T R0_001 = z * b1;
  const T R1_100 = x * b2;
  const T R0_200 = fma(x, R1_100, b1);
  const T R1_010 = y * b2;
  const T R0_110 = x * R1_010;
  const T R1_001 = z * b2;
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, b1);
  const T R0_011 = y * R1_001;
  const T R2_100 = x * b3;
  const T R1_200 = fma(x, R2_100, b2);
  const T R0_300 = fma(x, R1_200, T(2.0) * R1_100);
  const T R0_210 = y * R1_200;
  const T R0_201 = z * R1_200;
  const T R2_010 = y * b3;
  const T R1_020 = fma(y, R2_010, b2);
  const T R0_120 = x * R1_020;
  const T R2_001 = z * b3;
  const T R1_011 = y * R2_001;
  const T R0_111 = x * R1_011;
  const T R0_030 = fma(y, R1_020, T(2.0) * R1_010);
  const T R0_021 = z * R1_020;
  D[0] = b0;
  D[1] = R0_100;
  D[2] = R0_010;
  D[3] = R0_001;
  D[4] = R0_200;
  D[5] = R0_110;
  D[6] = R0_101;
  D[7] = R0_020;
  D[8] = R0_011;
  D[10] = R0_300;
  D[11] = R0_210;
  D[12] = R0_201;
  D[13] = R0_120;
  D[14] = R0_111;
  D[16] = R0_030;
  D[17] = R0_021;
  D[15] = -D[10] - D[13];
  D[18] = -D[11] - D[16];
}

template <typename T> __device__ __forceinline__ void sfmm_uderivs_fold_3(T x, T y, T z, T rinv, T* D) {
  const T R0_100 = x * T(-1.0);
  const T R0_010 = y * T(-1.0);
  const T R0_001 = z * T(-1.0);
  const T R1_100 = x * T(3.0);
  const T R0_200 = fma(x, R1_100, T(-1.0));
  const T R1_010 = y * T(3.0);
  const T R0_110 = x * R1_010;
  const T R1_001 = z * T(3.0);
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, T(-1.0));
  const T R0_011 = y * R1_001;
  const T R2_100 = x * T(-15.0);
  const T R1_200 = fma(x, R2_100, T(3.0));
  const T R0_300 = fma(x, R1_200, T(2.0) * R1_100);
  const T R0_210 = y * R1_200;
  const T R0_201 = z * R1_200;
  const T R2_010 = y * T(-15.0);
  const T R1_020 = fma(y, R2_010, T(3.0));
  const T R0_120 = x * R1_020;
  const T R2_001 = z * T(-15.0);
  const T R1_011 = y * R2_001;
  const T R0_111 = x * R1_011;
  const T R0_030 = fma(y, R1_020, T(2.0) * R1_010);
  const T R0_021 = z * R1_020;
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
  s = s * rinv;
  D[10] = R0_300 * s;
  D[11] = R0_210 * s;
  D[12] = R0_201 * s;
  D[13] = R0_120 * s;
  D[14] = R0_111 * s;
  D[16] = R0_030 * s;
  D[17] = R0_021 * s;
  D[15] = -D[10] - D[13];
  D[18] = -D[11] - D[16];
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_fold_4(T x, T y, T z, T rinv, T* D) {
  const T ri2 = rinv * rinv, b0 = rinv;
  const T b1 = b0 * (ri2 * T(-1.0));
  const T b2 = b1 * (ri2 * T(-3.0));
  const T b3 = b2 * (ri2 * T(-5.0));
  const T b4 = b3 * (ri2 * T(-7.0));
  const T R0_100 = x * b1;
  const T R0_010 = y * b1;
  const T R0_001 = z * b1;
  const T R1_100 = x * b2;
  const T R0_200 = fma(x, R1_100, b1);
  const T R1_010 = y * b2;
  const T R0_110 = x * R1_010;
  const T R1_001 = z * b2;
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, b1);
  const T R0_011 = y * R1_001;
  const T R2_100 = x * b3;
  const T R1_200 = fma(x, R2_100, b2);
  const T R0_300 = fma(x, R1_200, T(2.0) * R1_100);
  const T R0_210 = y * R1_200;
  const T R0_201 = z * R1_200;
  const T R2_010 = y * b3;
  const T R1_020 = fma(y, R2_010, b2);
  const T R0_120 = x * R1_020;
  const T R2_001 = z * b3;
  const T R1_011 = y * R2_001;
  const T R0_111 = x * R1_011;
  const T R0_030 = fma(y, R1_020, T(2.0) * R1_010);
  const T R0_021 = z * R1_020;
  const T R3_100 = x * b4;
  const T R2_200 = fma(x, R3_100, b3);
  const T R1_300 = fma(x, R2_200, T(2.0) * R2_100);
  const T R0_400 = fma(x, R1_300, T(3.0) * R1_200);
  const T R0_310 = y * R1_300;
  const T R0_301 = z * R1_300;
  const T R3_010 = y * b4;
  const T R2_020 = fma(y, R3_010, b3);
  const T R1_120 = x * R2_020;
  const T R0_220 = fma(x, R1_120, R1_020);
  const T R1_201 = z * R2_200;
  const T R0_211 = y * R1_201;
  const T R1_030 = fma(y, R2_020, T(2.0) * R2_010);
  const T R0_130 = x * R1_030;
  const T R1_021 = z * R2_020;
  const T R0_121 = x * R1_021;
  const T R0_040 = fma(y, R1_030, T(3.0) * R1_020);
  const T R0_031 = z * R1_030;
  D[0] = b0;
  D[1] = R0_100;
  D[2] = R0_010;
  D[3] = R0_001;
  D[4] = R0_200;
  D[5] = R0_110;
  D[6] = R0_101;
  D[7] = R0_020;
  D[8] = R0_011;
  D[10] = R0_300;
  D[11] = R0_210;
  D[12] = R0_201;
  D[13] = R0_120;
  D[14] = R0_111;
  D[16] = R0_030;
  D[17] = R0_021;
  D[15] = -D[10] - D[13];
  D[18] = -D[11] - D[16];
  D[20] = R0_400;
  D[21] = R0_310;
  D[22] = R0_301;
  D[23] = R0_220;
  D[24] = R0_211;
  D[26] = R0_130;
  D[27] = R0_121;
  D[30] = R0_040;
  D[31] = R0_031;
  D[25] = -D[20] - D[23];
  D[28] = -D[21] - D[26];
  D[32] = -D[23] - D[30];
}

template <typename T> __device__ __forceinline__ void sfmm_uderivs_fold_4(T x, T y, T z, T rinv, T* D) {
  const T R0_100 = x * T(-1.0);
  const T R0_010 = y * T(-1.0);
  const T R0_001 = z * T(-1.0);
  const T R1_100 = x * T(3.0);
  const T R0_200 = fma(x, R1_100, T(-1.0));
  const T R1_010 = y * T(3.0);
  const T R0_110 = x * R1_010;
  const T R1_001 = z * T(3.0);
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, T(-1.0));
  const T R0_011 = y * R1_001;
  const T R2_100 = x * T(-15.0);
  const T R1_200 = fma(x, R2_100, T(3.0));
  const T R0_300 = fma(x, R1_200, T(2.0) * R1_100);
  const T R0_210 = y * R1_200;
  const T R0_201 = z * R1_200;
  const T R2_010 = y * T(-15.0);
  const T R1_020 = fma(y, R2_010, T(3.0));
  const T R0_120 = x * R1_020;
  const T R2_001 = z * T(-15.0);
  const T R1_011 = y * R2_001;
  const T R0_111 = x * R1_011;
  const T R0_030 = fma(y, R1_020, T(2.0) * R1_010);
  const T R0_021 = z * R1_020;
  const T R3_100 = x * T(105.0);
  const T R2_200 = fma(x, R3_100, T(-15.0));
  const T R1_300 = fma(x, R2_200, T(2.0) * R2_100);
  const T R0_400 = fma(x, R1_300, T(3.0) * R1_200);
  const T R0_310 = y * R1_300;
  const T R0_301 = z * R1_300;
  const T R3_010 = y * T(105.0);
  const T R2_020 = fma(y, R3_010, T(-15.0));
  const T R1_120 = x * R2_020;
  const T R0_220 = fma(x, R1_120, R1_020);
  const T R1_201 = z * R2_200;
  const T R0_211 = y * R1_201;
  const T R1_030 = fma(y, R2_020, T(2.0) * R2_010);
  const T R0_130 = x * R1_030;
  const T R1_021 = z * R2_020;
  const T R0_121 = x * R1_021;
  const T R0_040 = fma(y, R1_030, T(3.0) * R1_020);
  const T R0_031 = z * R1_030;
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
  s = s * rinv;
  D[10] = R0_300 * s;
  D[11] = R0_210 * s;
  D[12] = R0_201 * s;
  D[13] = R0_120 * s;
  D[14] = R0_111 * s;
  D[16] = R0_030 * s;
  D[17] = R0_021 * s;
  D[15] = -D[10] - D[13];
  D[18] = -D[11] - D[16];
  s = s * rinv;
  D[20] = R0_400 * s;
  D[21] = R0_310 * s;
  D[22] = R0_301 * s;
  D[23] = R0_220 * s;
  D[24] = R0_211 * s;
  D[26] = R0_130 * s;
  D[27] = R0_121 * s;
  D[30] = R0_040 * s;
  D[31] = R0_031 * s;
  D[25] = -D[20] - D[23];
  D[28] = -D[21] - D[26];
  D[32] = -D[23] - D[30];
}

template <typename T> __device__ __forceinline__ void sfmm_derivs_fold_5(T x, T y, T z, T rinv, T* D) {
  const T ri2 = rinv * rinv, b0 = rinv;
  const T b1 = b0 * (ri2 * T(-1.0));
  const T b2 = b1 * (ri2 * T(-3.0));
  const T b3 = b2 * (ri2 * T(-5.0));
  const T b4 = b3 * (ri2 * T(-7.0));
  const T b5 = b4 * (ri2 * T(-9.0));
  const T R0_100 = x * b1;
  const T R0_010 = y * b1;
  const T R0_001 = z * b1;
  const T R1_100 = x * b2;
  const T R0_200 = fma(x, R1_100, b1);
  const T R1_010 = y * b2;
  const T R0_110 = x * R1_010;
  const T R1_001 = z * b2;
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, b1);
  const T R0_011 = y * R1_001;
  const T R2_100 = x * b3;
  const T R1_200 = fma(x, R2_100, b2);
  const T R0_300 = fma(x, R1_200, T(2.0) * R1_100);
  const T R0_210 = y * R1_200;
  const T R0_201 = z * R1_200;
  const T R2_010 = y * b3;
  const T R1_020 = fma(y, R2_010, b2);
  const T R0_120 = x * R1_020;
  const T R2_001 = z * b3;
  const T R1_011 = y * R2_001;
  const T R0_111 = x * R1_011;
  const T R0_030 = fma(y, R1_020, T(2.0) * R1_010);
  const T R0_021 = z * R1_020;
  const T R3_100 = x * b4;
  const T R2_200 = fma(x, R3_100, b3);
  const T R1_300 = fma(x, R2_200, T(2.0) * R2_100);
  const T R0_400 = fma(x, R1_300, T(3.0) * R1_200);
  const T R0_310 = y * R1_300;
  const T R0_301 = z * R1_300;
  const T R3_010 = y * b4;
  const T R2_020 = fma(y, R3_010, b3);
  const T R1_120 = x * R2_020;
  const T R0_220 = fma(x, R1_120, R1_020);
  const T R1_201 = z * R2_200;
  const T R0_211 = y * R1_201;
  const T R1_030 = fma(y, R2_020, T(2.0) * R2_010);
  const T R0_130 = x * R1_030;
  const T R1_021 = z * R2_020;
  const T R0_121 = x * R1_021;
  const T R0_040 = fma(y, R1_030, T(3.0) * R1_020);
  const T R0_031 = z * R1_030;
  const T R4_100 = x * b5;
  const T R3_200 = fma(x, R4_100, b4);
  const T R2_300 = fma(x, R3_200, T(2.0) * R3_100);
  const T R1_400 = fma(x, R2_300, T(3.0) * R2_200);
  const T R0_500 = fma(x, R1_400, T(4.0) * R1_300);
  const T R0_410 = y * R1_400;
  const T R0_401 = z * R1_400;
  const T R4_010 = y * b5;
  const T R3_020 = fma(y, R4_010, b4);
  const T R2_120 = x * R3_020;
  const T R1_220 = fma(x, R2_120, R2_020);
  const T R0_320 = fma(x, R1_220, T(2.0) * R1_120);
  const T R1_301 = z * R2_300;
  const T R0_311 = y * R1_301;
  const T R2_030 = fma(y, R3_020, T(2.0) * R3_010);
  const T R1_130 = x * R2_030;
  const T R0_230 = fma(x, R1_130, R1_030);
  const T R0_221 = z * R1_220;
  const T R1_040 = fma(y, R2_030, T(3.0) * R2_020);
  const T R0_140 = x * R1_040;
  const T R1_031 = z * R2_030;
  const T R0_131 = x * R1_031;
  const T R0_050 = fma(y, R1_040, T(4.0) * R1_030);
  const T R0_041 = z * R1_040;
  D[0] = b0;
  D[1] = R0_100;
  D[2] = R0_010;
  D[3] = R0_001;
  D[4] = R0_200;
  D[5] = R0_110;
  D[6] = R0_101;
  D[7] = R0_020;
  D[8] = R0_011;
  D[10] = R0_300;
  D[11] = R0_210;
  D[12] = R0_201;
  D[13] = R0_120;
  D[14] = R0_111;
  D[16] = R0_030;
  D[17] = R0_021;
  D[15] = -D[10] - D[13];
  D[18] = -D[11] - D[16];
  D[20] = R0_400;
  D[21] = R0_310;
  D[22] = R0_301;
  D[23] = R0_220;
  D[24] = R0_211;
  D[26] = R0_130;
  D[27] = R0_121;
  D[30] = R0_040;
  D[31] = R0_031;
  D[25] = -D[20] - D[23];
  D[28] = -D[21] - D[26];
  D[32] = -D[23] - D[30];
  D[35] = R0_500;
  D[36] = R0_410;
  D[37] = R0_401;
  D[38] = R0_320;
  D[39] = R0_311;
  D[41] = R0_230;
  D[42] = R0_221;
  D[45] = R0_140;
  D[46] = R0_131;
  D[50] = R0_050;
  D[51] = R0_041;
  D[40] = -D[35] - D[38];
  D[43] = -D[36] - D[41];
  D[47] = -D[38] - D[45];
  D[52] = -D[41] - D[50];
}

template <typename T> __device__ __forceinline__ void sfmm_uderivs_fold_5(T x, T y, T z, T rinv, T* D) {
  const T R0_100 = x * T(-1.0);
  const T R0_010 = y * T(-1.0);
  const T R0_001 = z * T(-1.0);
  const T R1_100 = x * T(3.0);
  const T R0_200 = fma(x, R1_100, T(-1.0));
  const T R1_010 = y * T(3.0);
  const T R0_110 = x * R1_010;
  const T R1_001 = z * T(3.0);
  const T R0_101 = x * R1_001;
  const T R0_020 = fma(y, R1_010, T(-1.0));
  const T R0_011 = y * R1_001;
  const T R2_100 = x * T(-15.0);
  const T R1_200 = fma(x, R2_100, T(3.0));
  const T R0_300 = fma(x, R1_200, T(2.0) * R1_100);
  const T R0_210 = y * R1_200;
  const T R0_201 = z * R1_200;
  const T R2_010 = y * T(-15.0);
  const T R1_020 = fma(y, R2_010, T(3.0));
  const T R0_120 = x * R1_020;
  const T R2_001 = z * T(-15.0);
  const T R1_011 = y * R2_001;
  const T R0_111 = x * R1_011;
  const T R0_030 = fma(y, R1_020, T(2.0) * R1_010);
  const T R0_021 = z * R1_020;
  const T R3_100 = x * T(105.0);
  const T R2_200 = fma(x, R3_100, T(-15.0));
  const T R1_300 = fma(x, R2_200, T(2.0) * R2_100);
  const T R0_400 = fma(x, R1_300, T(3.0) * R1_200);
  const T R0_310 = y * R1_300;
  const T R0_301 = z * R1_300;
  const T R3_010 = y * T(105.0);
  const T R2_020 = fma(y, R3_010, T(-15.0));
  const T R1_120 = x * R2_020;
  const T R0_220 = fma(x, R1_120, R1_020);
  const T R1_201 = z * R2_200;
  const T R0_211 = y * R1_201;
  const T R1_030 = fma(y, R2_020, T(2.0) * R2_010);
  const T R0_130 = x * R1_030;
  const T R1_021 = z * R2_020;
  const T R0_121 = x * R1_021;
  const T R0_040 = fma(y, R1_030, T(3.0) * R1_020);
  const T R0_031 = z * R1_030;
  const T R4_100 = x * T(-945.0);
  const T R3_200 = fma(x, R4_100, T(105.0));
  const T R2_300 = fma(x, R3_200, T(2.0) * R3_100);
  const T R1_400 = fma(x, R2_300, T(3.0) * R2_200);
  const T R0_500 = fma(x, R1_400, T(4.0) * R1_300);
  const T R0_410 = y * R1_400;
  const T R0_401 = z * R1_400;
  const T R4_010 = y * T(-945.0);
  const T R3_020 = fma(y, R4_010, T(105.0));
  const T R2_120 = x * R3_020;
  const T R1_220 = fma(x, R2_120, R2_020);
  const T R0_320 = fma(x, R1_220, T(2.0) * R1_120);
  const T R1_301 = z * R2_300;
  const T R0_311 = y * R1_301;
  const T R2_030 = fma(y, R3_020, T(2.0) * R3_010);
  const T R1_130 = x * R2_030;
  const T R0_230 = fma(x, R1_130, R1_030);
  const T R0_221 = z * R1_220;
  const T R1_040 = fma(y, R2_030, T(3.0) * R2_020);
  const T R0_140 = x * R1_040;
  const T R1_031 = z * R2_030;
  const T R0_131 = x * R1_031;
  const T R0_050 = fma(y, R1_040, T(4.0) * R1_030);
  const T R0_041 = z * R1_040;
  T s = rinv;
  D[0] = T(1.0) * s;
  s = s * rinv;
  D[1] = R0_100 * s;
  D[2] = R0_010 * s;
  D[3] = R0_001 * s;
  s = s * rinv;
  D[4] = R0_200 * s;
  D[5] = R0_110 * s;
  D[6] = R0_101 * s;
  D[7] = R0_020 * s;
  D[8] = R0_011 * s;
  s = s * rinv;
  D[10] = R0_300 * s;
  D[11] = R0_210 * s;
  D[12] = R0_201 * s;
  D[13] = R0_120 * s;
  D[14] = R0_111 * s;
  D[16] = R0_030 * s;
  D[17] = R0_021 * s;
  D[15] = -D[10] - D[13];
  D[18] = -D[11] - D[16];
  s = s * rinv;
  D[20] = R0_400 * s;
  D[21] = R0_310 * s;
  D[22] = R0_301 * s;
  D[23] = R0_220 * s;
  D[24] = R0_211 * s;
  D[26] = R0_130 * s;
  D[27] = R0_121 * s;
  D[30] = R0_040 * s;
  D[31] = R0_031 * s;
  D[25] = -D[20] - D[23];
  D[28] = -D[21] - D[26];
  D[32] = -D[23] - D[30];
  s = s * rinv;
  D[35] = R0_500 * s;
  D[36] = R0_410 * s;
  D[37] = R0_401 * s;
  D[38] = R0_320 * s;
  D[39] = R0_311 * s;
  D[41] = R0_230 * s;
  D[42] = R0_221 * s;
  D[45] = R0_140 * s;
  D[46] = R0_131 * s;
  D[50] = R0_050 * s;
  D[51] = R0_041 * s;
  D[40] = -D[35] - D[38];
  D[43] = -D[36] - D[41];
  D[47] = -D[38] - D[45];
  D[52] = -D[41] - D[50];
}

