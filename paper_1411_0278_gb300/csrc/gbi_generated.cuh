// Generated by paper_1411_0278_gb300/gen_tables.py -- do not edit.
// Pair-frame single-layer Galerkin couplings, packed-basis rotations and
// self scalars for the truncations l<=2, 3, 4, 5 (mode sets 1s 2a | 2s 3t | 3a 3s 4t | 4a 4s 5t |
// 5a 5s 6t) and the minimal truncation 40 (every mode of rank <= 4: l<=4 without 5t).
#pragma once

#include "df.cuh"   // gbi_fmac: a * b + c in the arithmetic of T

static constexpr int gbi_dm1_n = 5;
template <typename T> __host__ __device__ __forceinline__ void gbi_dmat1(T c, T s, T* __restrict__ dm) {
  const T c2 = c * c; const T c3 = c2 * c; const T c4 = c2 * c2;
  const T cp[5] = {T(1), c, c2, c3, c4}; (void)cp;
  const T sp[5] = {s, c * s, c2 * s, c3 * s, c4 * s}; (void)sp;
  dm[0] = T(1.0);   // (mu=-1, nu=-1)
  dm[1] = cp[1];   // (mu=0, nu=0)
  dm[2] = (-sp[0]);   // (mu=0, nu=1)
  dm[3] = sp[0];   // (mu=1, nu=0)
  dm[4] = cp[1];   // (mu=1, nu=1)
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapply1(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = in[0];
  out[1] = gbi_fmac(dm[2], in[2], gbi_mul(dm[1], in[1]));
  out[2] = gbi_fmac(dm[4], in[2], gbi_mul(dm[3], in[1]));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapplyT1(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = in[0];
  out[1] = gbi_fmac(dm[3], in[2], gbi_mul(dm[1], in[1]));
  out[2] = gbi_fmac(dm[4], in[2], gbi_mul(dm[2], in[1]));
}
static constexpr int gbi_dm2_n = 13;
template <typename T> __host__ __device__ __forceinline__ void gbi_dmat2(T c, T s, T* __restrict__ dm) {
  const T c2 = c * c; const T c3 = c2 * c; const T c4 = c2 * c2;
  const T cp[5] = {T(1), c, c2, c3, c4}; (void)cp;
  const T sp[5] = {s, c * s, c2 * s, c3 * s, c4 * s}; (void)sp;
  dm[0] = cp[1];   // (mu=-2, nu=-2)
  dm[1] = sp[0];   // (mu=-2, nu=-1)
  dm[2] = (-sp[0]);   // (mu=-1, nu=-2)
  dm[3] = cp[1];   // (mu=-1, nu=-1)
  dm[4] = gbi_fmac(1.5f, cp[2], T(-0.5));   // (mu=0, nu=0)
  dm[5] = T(-1.7320508075688774) * sp[1];   // (mu=0, nu=1)
  dm[6] = gbi_fmac(T(-0.8660254037844387), cp[2], T(0.8660254037844387));   // (mu=0, nu=2)
  dm[7] = T(1.7320508075688774) * sp[1];   // (mu=1, nu=0)
  dm[8] = gbi_fmac(2.0f, cp[2], T(-1.0));   // (mu=1, nu=1)
  dm[9] = (-sp[1]);   // (mu=1, nu=2)
  dm[10] = gbi_fmac(T(-0.8660254037844387), cp[2], T(0.8660254037844387));   // (mu=2, nu=0)
  dm[11] = sp[1];   // (mu=2, nu=1)
  dm[12] = gbi_fmac(0.5f, cp[2], T(0.5));   // (mu=2, nu=2)
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapply2(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[1], in[1], gbi_mul(dm[0], in[0]));
  out[1] = gbi_fmac(dm[3], in[1], gbi_mul(dm[2], in[0]));
  out[2] = gbi_fmac(dm[6], in[4], gbi_fmac(dm[5], in[3], gbi_mul(dm[4], in[2])));
  out[3] = gbi_fmac(dm[9], in[4], gbi_fmac(dm[8], in[3], gbi_mul(dm[7], in[2])));
  out[4] = gbi_fmac(dm[12], in[4], gbi_fmac(dm[11], in[3], gbi_mul(dm[10], in[2])));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapplyT2(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[2], in[1], gbi_mul(dm[0], in[0]));
  out[1] = gbi_fmac(dm[3], in[1], gbi_mul(dm[1], in[0]));
  out[2] = gbi_fmac(dm[10], in[4], gbi_fmac(dm[7], in[3], gbi_mul(dm[4], in[2])));
  out[3] = gbi_fmac(dm[11], in[4], gbi_fmac(dm[8], in[3], gbi_mul(dm[5], in[2])));
  out[4] = gbi_fmac(dm[12], in[4], gbi_fmac(dm[9], in[3], gbi_mul(dm[6], in[2])));
}
static constexpr int gbi_dm3_n = 25;
template <typename T> __host__ __device__ __forceinline__ void gbi_dmat3(T c, T s, T* __restrict__ dm) {
  const T c2 = c * c; const T c3 = c2 * c; const T c4 = c2 * c2;
  const T cp[5] = {T(1), c, c2, c3, c4}; (void)cp;
  const T sp[5] = {s, c * s, c2 * s, c3 * s, c4 * s}; (void)sp;
  dm[0] = gbi_fmac(0.75f, cp[2], T(0.25));   // (mu=-3, nu=-3)
  dm[1] = T(1.2247448713915892) * sp[1];   // (mu=-3, nu=-2)
  dm[2] = gbi_fmac(T(-0.9682458365518543), cp[2], T(0.9682458365518543));   // (mu=-3, nu=-1)
  dm[3] = T(-1.2247448713915892) * sp[1];   // (mu=-2, nu=-3)
  dm[4] = gbi_fmac(2.0f, cp[2], T(-1.0));   // (mu=-2, nu=-2)
  dm[5] = T(1.5811388300841898) * sp[1];   // (mu=-2, nu=-1)
  dm[6] = gbi_fmac(T(-0.9682458365518543), cp[2], T(0.9682458365518543));   // (mu=-1, nu=-3)
  dm[7] = T(-1.5811388300841898) * sp[1];   // (mu=-1, nu=-2)
  dm[8] = gbi_fmac(1.25f, cp[2], T(-0.25));   // (mu=-1, nu=-1)
  dm[9] = gbi_fmac(2.5f, cp[3], gbi_mul(-1.5f, cp[1]));   // (mu=0, nu=0)
  dm[10] = gbi_fmac(T(-3.061862178478973), sp[2], gbi_mul(T(0.6123724356957946), sp[0]));   // (mu=0, nu=1)
  dm[11] = gbi_fmac(T(-1.9364916731037085), cp[3], gbi_mul(T(1.9364916731037085), cp[1]));   // (mu=0, nu=2)
  dm[12] = gbi_fmac(T(0.7905694150420949), sp[2], gbi_mul(T(-0.7905694150420949), sp[0]));   // (mu=0, nu=3)
  dm[13] = gbi_fmac(T(3.061862178478973), sp[2], gbi_mul(T(-0.6123724356957946), sp[0]));   // (mu=1, nu=0)
  dm[14] = gbi_fmac(3.75f, cp[3], gbi_mul(-2.75f, cp[1]));   // (mu=1, nu=1)
  dm[15] = gbi_fmac(T(-2.3717082451262845), sp[2], gbi_mul(T(0.7905694150420949), sp[0]));   // (mu=1, nu=2)
  dm[16] = gbi_fmac(T(-0.9682458365518543), cp[3], gbi_mul(T(0.9682458365518543), cp[1]));   // (mu=1, nu=3)
  dm[17] = gbi_fmac(T(-1.9364916731037085), cp[3], gbi_mul(T(1.9364916731037085), cp[1]));   // (mu=2, nu=0)
  dm[18] = gbi_fmac(T(2.3717082451262845), sp[2], gbi_mul(T(-0.7905694150420949), sp[0]));   // (mu=2, nu=1)
  dm[19] = gbi_fmac(1.5f, cp[3], gbi_mul(-0.5f, cp[1]));   // (mu=2, nu=2)
  dm[20] = gbi_fmac(T(-0.6123724356957946), sp[2], gbi_mul(T(-0.6123724356957946), sp[0]));   // (mu=2, nu=3)
  dm[21] = gbi_fmac(T(-0.7905694150420949), sp[2], gbi_mul(T(0.7905694150420949), sp[0]));   // (mu=3, nu=0)
  dm[22] = gbi_fmac(T(-0.9682458365518543), cp[3], gbi_mul(T(0.9682458365518543), cp[1]));   // (mu=3, nu=1)
  dm[23] = gbi_fmac(T(0.6123724356957946), sp[2], gbi_mul(T(0.6123724356957946), sp[0]));   // (mu=3, nu=2)
  dm[24] = gbi_fmac(0.25f, cp[3], gbi_mul(0.75f, cp[1]));   // (mu=3, nu=3)
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapply3(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[2], in[2], gbi_fmac(dm[1], in[1], gbi_mul(dm[0], in[0])));
  out[1] = gbi_fmac(dm[5], in[2], gbi_fmac(dm[4], in[1], gbi_mul(dm[3], in[0])));
  out[2] = gbi_fmac(dm[8], in[2], gbi_fmac(dm[7], in[1], gbi_mul(dm[6], in[0])));
  out[3] = gbi_fmac(dm[12], in[6], gbi_fmac(dm[11], in[5], gbi_fmac(dm[10], in[4], gbi_mul(dm[9], in[3]))));
  out[4] = gbi_fmac(dm[16], in[6], gbi_fmac(dm[15], in[5], gbi_fmac(dm[14], in[4], gbi_mul(dm[13], in[3]))));
  out[5] = gbi_fmac(dm[20], in[6], gbi_fmac(dm[19], in[5], gbi_fmac(dm[18], in[4], gbi_mul(dm[17], in[3]))));
  out[6] = gbi_fmac(dm[24], in[6], gbi_fmac(dm[23], in[5], gbi_fmac(dm[22], in[4], gbi_mul(dm[21], in[3]))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapplyT3(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[6], in[2], gbi_fmac(dm[3], in[1], gbi_mul(dm[0], in[0])));
  out[1] = gbi_fmac(dm[7], in[2], gbi_fmac(dm[4], in[1], gbi_mul(dm[1], in[0])));
  out[2] = gbi_fmac(dm[8], in[2], gbi_fmac(dm[5], in[1], gbi_mul(dm[2], in[0])));
  out[3] = gbi_fmac(dm[21], in[6], gbi_fmac(dm[17], in[5], gbi_fmac(dm[13], in[4], gbi_mul(dm[9], in[3]))));
  out[4] = gbi_fmac(dm[22], in[6], gbi_fmac(dm[18], in[5], gbi_fmac(dm[14], in[4], gbi_mul(dm[10], in[3]))));
  out[5] = gbi_fmac(dm[23], in[6], gbi_fmac(dm[19], in[5], gbi_fmac(dm[15], in[4], gbi_mul(dm[11], in[3]))));
  out[6] = gbi_fmac(dm[24], in[6], gbi_fmac(dm[20], in[5], gbi_fmac(dm[16], in[4], gbi_mul(dm[12], in[3]))));
}
static constexpr int gbi_dm4_n = 41;
template <typename T> __host__ __device__ __forceinline__ void gbi_dmat4(T c, T s, T* __restrict__ dm) {
  const T c2 = c * c; const T c3 = c2 * c; const T c4 = c2 * c2;
  const T cp[5] = {T(1), c, c2, c3, c4}; (void)cp;
  const T sp[5] = {s, c * s, c2 * s, c3 * s, c4 * s}; (void)sp;
  dm[0] = gbi_fmac(0.5f, cp[3], gbi_mul(0.5f, cp[1]));   // (mu=-4, nu=-4)
  dm[1] = gbi_fmac(T(1.0606601717798212), sp[2], gbi_mul(T(0.35355339059327373), sp[0]));   // (mu=-4, nu=-3)
  dm[2] = gbi_fmac(T(-1.3228756555322954), cp[3], gbi_mul(T(1.3228756555322954), cp[1]));   // (mu=-4, nu=-2)
  dm[3] = gbi_fmac(T(-0.9354143466934854), sp[2], gbi_mul(T(0.9354143466934854), sp[0]));   // (mu=-4, nu=-1)
  dm[4] = gbi_fmac(T(-1.0606601717798212), sp[2], gbi_mul(T(-0.35355339059327373), sp[0]));   // (mu=-3, nu=-4)
  dm[5] = gbi_fmac(2.25f, cp[3], gbi_mul(-1.25f, cp[1]));   // (mu=-3, nu=-3)
  dm[6] = gbi_fmac(T(2.806243040080456), sp[2], gbi_mul(T(-0.9354143466934853), sp[0]));   // (mu=-3, nu=-2)
  dm[7] = gbi_fmac(T(-1.984313483298443), cp[3], gbi_mul(T(1.984313483298443), cp[1]));   // (mu=-3, nu=-1)
  dm[8] = gbi_fmac(T(-1.3228756555322954), cp[3], gbi_mul(T(1.3228756555322954), cp[1]));   // (mu=-2, nu=-4)
  dm[9] = gbi_fmac(T(-2.806243040080456), sp[2], gbi_mul(T(0.9354143466934853), sp[0]));   // (mu=-2, nu=-3)
  dm[10] = gbi_fmac(3.5f, cp[3], gbi_mul(-2.5f, cp[1]));   // (mu=-2, nu=-2)
  dm[11] = gbi_fmac(T(2.4748737341529163), sp[2], gbi_mul(T(-0.35355339059327373), sp[0]));   // (mu=-2, nu=-1)
  dm[12] = gbi_fmac(T(0.9354143466934854), sp[2], gbi_mul(T(-0.9354143466934854), sp[0]));   // (mu=-1, nu=-4)
  dm[13] = gbi_fmac(T(-1.984313483298443), cp[3], gbi_mul(T(1.984313483298443), cp[1]));   // (mu=-1, nu=-3)
  dm[14] = gbi_fmac(T(-2.4748737341529163), sp[2], gbi_mul(T(0.35355339059327373), sp[0]));   // (mu=-1, nu=-2)
  dm[15] = gbi_fmac(1.75f, cp[3], gbi_mul(-0.75f, cp[1]));   // (mu=-1, nu=-1)
  dm[16] = gbi_fmac(4.375f, cp[4], gbi_fmac(-3.75f, cp[2], T(0.375)));   // (mu=0, nu=0)
  dm[17] = gbi_fmac(T(-5.533985905294664), sp[3], gbi_mul(T(2.3717082451262845), sp[1]));   // (mu=0, nu=1)
  dm[18] = gbi_fmac(T(-3.9131189606246317), cp[4], gbi_fmac(T(4.472135954999579), cp[2], T(-0.5590169943749473)));   // (mu=0, nu=2)
  dm[19] = gbi_fmac(T(2.091650066335189), sp[3], gbi_mul(T(-2.091650066335189), sp[1]));   // (mu=0, nu=3)
  dm[20] = gbi_fmac(T(0.739509972887452), cp[4], gbi_fmac(T(-1.479019945774904), cp[2], T(0.739509972887452)));   // (mu=0, nu=4)
  dm[21] = gbi_fmac(T(5.533985905294664), sp[3], gbi_mul(T(-2.3717082451262845), sp[1]));   // (mu=1, nu=0)
  dm[22] = gbi_fmac(7.0f, cp[4], gbi_fmac(-6.75f, cp[2], T(0.75)));   // (mu=1, nu=1)
  dm[23] = gbi_fmac(T(-4.949747468305833), sp[3], gbi_mul(T(2.82842712474619), sp[1]));   // (mu=1, nu=2)
  dm[24] = gbi_fmac(T(-2.6457513110645907), cp[4], gbi_fmac(T(3.3071891388307386), cp[2], T(-0.6614378277661477)));   // (mu=1, nu=3)
  dm[25] = gbi_fmac(T(0.9354143466934854), sp[3], gbi_mul(T(-0.9354143466934854), sp[1]));   // (mu=1, nu=4)
  dm[26] = gbi_fmac(T(-3.9131189606246317), cp[4], gbi_fmac(T(4.472135954999579), cp[2], T(-0.5590169943749473)));   // (mu=2, nu=0)
  dm[27] = gbi_fmac(T(4.949747468305833), sp[3], gbi_mul(T(-2.82842712474619), sp[1]));   // (mu=2, nu=1)
  dm[28] = gbi_fmac(3.5f, cp[4], gbi_fmac(-3.0f, cp[2], T(0.5)));   // (mu=2, nu=2)
  dm[29] = T(-1.8708286933869707) * sp[3];   // (mu=2, nu=3)
  dm[30] = gbi_fmac(T(-0.6614378277661477), cp[4], T(0.6614378277661477));   // (mu=2, nu=4)
  dm[31] = gbi_fmac(T(-2.091650066335189), sp[3], gbi_mul(T(2.091650066335189), sp[1]));   // (mu=3, nu=0)
  dm[32] = gbi_fmac(T(-2.6457513110645907), cp[4], gbi_fmac(T(3.3071891388307386), cp[2], T(-0.6614378277661477)));   // (mu=3, nu=1)
  dm[33] = T(1.8708286933869707) * sp[3];   // (mu=3, nu=2)
  dm[34] = gbi_fmac(0.75f, cp[2], (T(-0.75) + cp[4]));   // (mu=3, nu=3)
  dm[35] = gbi_fmac(T(-0.35355339059327373), sp[3], gbi_mul(T(-1.0606601717798212), sp[1]));   // (mu=3, nu=4)
  dm[36] = gbi_fmac(T(0.739509972887452), cp[4], gbi_fmac(T(-1.479019945774904), cp[2], T(0.739509972887452)));   // (mu=4, nu=0)
  dm[37] = gbi_fmac(T(-0.9354143466934854), sp[3], gbi_mul(T(0.9354143466934854), sp[1]));   // (mu=4, nu=1)
  dm[38] = gbi_fmac(T(-0.6614378277661477), cp[4], T(0.6614378277661477));   // (mu=4, nu=2)
  dm[39] = gbi_fmac(T(0.35355339059327373), sp[3], gbi_mul(T(1.0606601717798212), sp[1]));   // (mu=4, nu=3)
  dm[40] = gbi_fmac(0.125f, cp[4], gbi_fmac(0.75f, cp[2], T(0.125)));   // (mu=4, nu=4)
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapply4(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[3], in[3], gbi_fmac(dm[2], in[2], gbi_fmac(dm[1], in[1], gbi_mul(dm[0], in[0]))));
  out[1] = gbi_fmac(dm[7], in[3], gbi_fmac(dm[6], in[2], gbi_fmac(dm[5], in[1], gbi_mul(dm[4], in[0]))));
  out[2] = gbi_fmac(dm[11], in[3], gbi_fmac(dm[10], in[2], gbi_fmac(dm[9], in[1], gbi_mul(dm[8], in[0]))));
  out[3] = gbi_fmac(dm[15], in[3], gbi_fmac(dm[14], in[2], gbi_fmac(dm[13], in[1], gbi_mul(dm[12], in[0]))));
  out[4] = gbi_fmac(dm[20], in[8], gbi_fmac(dm[19], in[7], gbi_fmac(dm[18], in[6], gbi_fmac(dm[17], in[5], gbi_mul(dm[16], in[4])))));
  out[5] = gbi_fmac(dm[25], in[8], gbi_fmac(dm[24], in[7], gbi_fmac(dm[23], in[6], gbi_fmac(dm[22], in[5], gbi_mul(dm[21], in[4])))));
  out[6] = gbi_fmac(dm[30], in[8], gbi_fmac(dm[29], in[7], gbi_fmac(dm[28], in[6], gbi_fmac(dm[27], in[5], gbi_mul(dm[26], in[4])))));
  out[7] = gbi_fmac(dm[35], in[8], gbi_fmac(dm[34], in[7], gbi_fmac(dm[33], in[6], gbi_fmac(dm[32], in[5], gbi_mul(dm[31], in[4])))));
  out[8] = gbi_fmac(dm[40], in[8], gbi_fmac(dm[39], in[7], gbi_fmac(dm[38], in[6], gbi_fmac(dm[37], in[5], gbi_mul(dm[36], in[4])))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapplyT4(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[12], in[3], gbi_fmac(dm[8], in[2], gbi_fmac(dm[4], in[1], gbi_mul(dm[0], in[0]))));
  out[1] = gbi_fmac(dm[13], in[3], gbi_fmac(dm[9], in[2], gbi_fmac(dm[5], in[1], gbi_mul(dm[1], in[0]))));
  out[2] = gbi_fmac(dm[14], in[3], gbi_fmac(dm[10], in[2], gbi_fmac(dm[6], in[1], gbi_mul(dm[2], in[0]))));
  out[3] = gbi_fmac(dm[15], in[3], gbi_fmac(dm[11], in[2], gbi_fmac(dm[7], in[1], gbi_mul(dm[3], in[0]))));
  out[4] = gbi_fmac(dm[36], in[8], gbi_fmac(dm[31], in[7], gbi_fmac(dm[26], in[6], gbi_fmac(dm[21], in[5], gbi_mul(dm[16], in[4])))));
  out[5] = gbi_fmac(dm[37], in[8], gbi_fmac(dm[32], in[7], gbi_fmac(dm[27], in[6], gbi_fmac(dm[22], in[5], gbi_mul(dm[17], in[4])))));
  out[6] = gbi_fmac(dm[38], in[8], gbi_fmac(dm[33], in[7], gbi_fmac(dm[28], in[6], gbi_fmac(dm[23], in[5], gbi_mul(dm[18], in[4])))));
  out[7] = gbi_fmac(dm[39], in[8], gbi_fmac(dm[34], in[7], gbi_fmac(dm[29], in[6], gbi_fmac(dm[24], in[5], gbi_mul(dm[19], in[4])))));
  out[8] = gbi_fmac(dm[40], in[8], gbi_fmac(dm[35], in[7], gbi_fmac(dm[30], in[6], gbi_fmac(dm[25], in[5], gbi_mul(dm[20], in[4])))));
}
static constexpr int gbi_dm5_n = 61;
template <typename T> __host__ __device__ __forceinline__ void gbi_dmat5(T c, T s, T* __restrict__ dm) {
  const T c2 = c * c; const T c3 = c2 * c; const T c4 = c2 * c2; const T c5 = c4 * c;
  const T cp[6] = {T(1), c, c2, c3, c4, c5}; (void)cp;
  const T sp[6] = {s, c * s, c2 * s, c3 * s, c4 * s, c5 * s}; (void)sp;
  dm[0] = gbi_fmac(0.3125f, cp[4], gbi_fmac(0.625f, cp[2], T(0.0625)));   // (mu=-5, nu=-5)
  dm[1] = gbi_fmac(T(0.7905694150420949), sp[3], gbi_mul(T(0.7905694150420949), sp[1]));   // (mu=-5, nu=-4)
  dm[2] = gbi_fmac(T(-1.2577882373436315), cp[4], gbi_fmac(T(0.8385254915624211), cp[2], T(0.41926274578121053)));   // (mu=-5, nu=-3)
  dm[3] = gbi_fmac(T(-1.3693063937629153), sp[3], gbi_mul(T(1.3693063937629153), sp[1]));   // (mu=-5, nu=-2)
  dm[4] = gbi_fmac(T(0.9057110466368398), cp[4], gbi_fmac(T(-1.8114220932736795), cp[2], T(0.9057110466368398)));   // (mu=-5, nu=-1)
  dm[5] = gbi_fmac(T(-0.7905694150420949), sp[3], gbi_mul(T(-0.7905694150420949), sp[1]));   // (mu=-4, nu=-5)
  dm[6] = gbi_fmac(2.0f, cp[4], gbi_fmac(-0.5f, cp[2], T(-0.5)));   // (mu=-4, nu=-4)
  dm[7] = gbi_fmac(T(3.181980515339464), sp[3], gbi_mul(T(-1.0606601717798212), sp[1]));   // (mu=-4, nu=-3)
  dm[8] = gbi_fmac(T(-3.464101615137755), cp[4], gbi_fmac(T(4.330127018922194), cp[2], T(-0.8660254037844387)));   // (mu=-4, nu=-2)
  dm[9] = gbi_fmac(T(-2.29128784747792), sp[3], gbi_mul(T(2.29128784747792), sp[1]));   // (mu=-4, nu=-1)
  dm[10] = gbi_fmac(T(-1.2577882373436315), cp[4], gbi_fmac(T(0.8385254915624211), cp[2], T(0.41926274578121053)));   // (mu=-3, nu=-5)
  dm[11] = gbi_fmac(T(-3.181980515339464), sp[3], gbi_mul(T(1.0606601717798212), sp[1]));   // (mu=-3, nu=-4)
  dm[12] = gbi_fmac(5.0625f, cp[4], gbi_fmac(-4.875f, cp[2], T(0.8125)));   // (mu=-3, nu=-3)
  dm[13] = gbi_fmac(T(5.5113519212621505), sp[3], gbi_mul(T(-3.061862178478972), sp[1]));   // (mu=-3, nu=-2)
  dm[14] = gbi_fmac(T(-3.6454166428544217), cp[4], gbi_fmac(T(4.050462936504913), cp[2], T(-0.4050462936504913)));   // (mu=-3, nu=-1)
  dm[15] = gbi_fmac(T(1.3693063937629153), sp[3], gbi_mul(T(-1.3693063937629153), sp[1]));   // (mu=-2, nu=-5)
  dm[16] = gbi_fmac(T(-3.464101615137755), cp[4], gbi_fmac(T(4.330127018922194), cp[2], T(-0.8660254037844387)));   // (mu=-2, nu=-4)
  dm[17] = gbi_fmac(T(-5.5113519212621505), sp[3], gbi_mul(T(3.061862178478972), sp[1]));   // (mu=-2, nu=-3)
  dm[18] = gbi_fmac(6.0f, cp[4], gbi_fmac(-5.5f, cp[2], T(0.5)));   // (mu=-2, nu=-2)
  dm[19] = gbi_fmac(T(3.968626966596886), sp[3], gbi_mul(T(-1.3228756555322954), sp[1]));   // (mu=-2, nu=-1)
  dm[20] = gbi_fmac(T(0.9057110466368398), cp[4], gbi_fmac(T(-1.8114220932736795), cp[2], T(0.9057110466368398)));   // (mu=-1, nu=-5)
  dm[21] = gbi_fmac(T(2.29128784747792), sp[3], gbi_mul(T(-2.29128784747792), sp[1]));   // (mu=-1, nu=-4)
  dm[22] = gbi_fmac(T(-3.6454166428544217), cp[4], gbi_fmac(T(4.050462936504913), cp[2], T(-0.4050462936504913)));   // (mu=-1, nu=-3)
  dm[23] = gbi_fmac(T(-3.968626966596886), sp[3], gbi_mul(T(1.3228756555322954), sp[1]));   // (mu=-1, nu=-2)
  dm[24] = gbi_fmac(2.625f, cp[4], gbi_fmac(T(-1.7500000000000002), cp[2], T(0.125)));   // (mu=-1, nu=-1)
  dm[25] = gbi_fmac(7.875f, cp[5], gbi_fmac(-8.75f, cp[3], gbi_mul(1.875f, cp[1])));   // (mu=0, nu=0)
  dm[26] = gbi_fmac(T(-10.16658128379447), sp[4], gbi_fmac(T(6.77772085586298), sp[2], gbi_mul(T(-0.4841229182759271), sp[0])));   // (mu=0, nu=1)
  dm[27] = gbi_fmac(T(-7.685213074469699), cp[5], gbi_fmac(T(10.2469507659596), cp[3], gbi_mul(T(-2.5617376914899), cp[1])));   // (mu=0, nu=2)
  dm[28] = gbi_fmac(T(4.706212649254175), sp[4], gbi_fmac(T(-5.229125165837972), sp[2], gbi_mul(T(0.5229125165837972), sp[0])));   // (mu=0, nu=3)
  dm[29] = gbi_fmac(T(2.218529918662356), cp[5], gbi_fmac(T(-4.437059837324712), cp[3], gbi_mul(T(2.218529918662356), cp[1])));   // (mu=0, nu=4)
  dm[30] = gbi_fmac(T(-0.7015607600201139), sp[4], gbi_fmac(T(1.4031215200402278), sp[2], gbi_mul(T(-0.7015607600201139), sp[0])));   // (mu=0, nu=5)
  dm[31] = gbi_fmac(T(10.16658128379447), sp[4], gbi_fmac(T(-6.77772085586298), sp[2], gbi_mul(T(0.4841229182759271), sp[0])));   // (mu=1, nu=0)
  dm[32] = gbi_fmac(13.125f, cp[5], gbi_fmac(T(-15.750000000000002), cp[3], gbi_mul(T(3.6250000000000004), cp[1])));   // (mu=1, nu=1)
  dm[33] = gbi_fmac(T(-9.921567416492215), sp[4], gbi_fmac(T(7.937253933193772), sp[2], gbi_mul(T(-0.6614378277661477), sp[0])));   // (mu=1, nu=2)
  dm[34] = gbi_fmac(T(-6.075694404757369), cp[5], gbi_fmac(T(8.911018460310808), cp[3], gbi_mul(T(-2.835324055553439), cp[1])));   // (mu=1, nu=3)
  dm[35] = gbi_fmac(T(2.8641098093474), sp[4], gbi_fmac(T(-3.43693177121688), sp[2], gbi_mul(T(0.57282196186948), sp[0])));   // (mu=1, nu=4)
  dm[36] = gbi_fmac(T(0.9057110466368398), cp[5], gbi_fmac(T(-1.8114220932736795), cp[3], gbi_mul(T(0.9057110466368398), cp[1])));   // (mu=1, nu=5)
  dm[37] = gbi_fmac(T(-7.685213074469699), cp[5], gbi_fmac(T(10.2469507659596), cp[3], gbi_mul(T(-2.5617376914899), cp[1])));   // (mu=2, nu=0)
  dm[38] = gbi_fmac(T(9.921567416492215), sp[4], gbi_fmac(T(-7.937253933193772), sp[2], gbi_mul(T(0.6614378277661477), sp[0])));   // (mu=2, nu=1)
  dm[39] = gbi_fmac(7.5f, cp[5], gbi_fmac(-9.0f, cp[3], gbi_mul(2.5f, cp[1])));   // (mu=2, nu=2)
  dm[40] = gbi_fmac(T(-4.592793267718458), sp[4], gbi_fmac(T(2.449489742783178), sp[2], gbi_mul(T(-0.30618621784789724), sp[0])));   // (mu=2, nu=3)
  dm[41] = gbi_fmac(T(-2.165063509461097), cp[5], gbi_fmac(T(1.7320508075688774), cp[3], gbi_mul(T(0.43301270189221935), cp[1])));   // (mu=2, nu=4)
  dm[42] = gbi_fmac(T(0.6846531968814576), sp[4], gbi_mul(T(-0.6846531968814576), sp[0]));   // (mu=2, nu=5)
  dm[43] = gbi_fmac(T(-4.706212649254175), sp[4], gbi_fmac(T(5.229125165837972), sp[2], gbi_mul(T(-0.5229125165837972), sp[0])));   // (mu=3, nu=0)
  dm[44] = gbi_fmac(T(-6.075694404757369), cp[5], gbi_fmac(T(8.911018460310808), cp[3], gbi_mul(T(-2.835324055553439), cp[1])));   // (mu=3, nu=1)
  dm[45] = gbi_fmac(T(4.592793267718458), sp[4], gbi_fmac(T(-2.449489742783178), sp[2], gbi_mul(T(0.30618621784789724), sp[0])));   // (mu=3, nu=2)
  dm[46] = gbi_fmac(2.8125f, cp[5], gbi_fmac(-0.875f, cp[3], gbi_mul(-0.9375f, cp[1])));   // (mu=3, nu=3)
  dm[47] = gbi_fmac(T(-1.3258252147247764), sp[4], gbi_fmac(T(-1.590990257669732), sp[2], gbi_mul(T(0.795495128834866), sp[0])));   // (mu=3, nu=4)
  dm[48] = gbi_fmac(T(-0.41926274578121053), cp[5], gbi_fmac(T(-0.8385254915624211), cp[3], gbi_mul(T(1.2577882373436315), cp[1])));   // (mu=3, nu=5)
  dm[49] = gbi_fmac(T(2.218529918662356), cp[5], gbi_fmac(T(-4.437059837324712), cp[3], gbi_mul(T(2.218529918662356), cp[1])));   // (mu=4, nu=0)
  dm[50] = gbi_fmac(T(-2.8641098093474), sp[4], gbi_fmac(T(3.43693177121688), sp[2], gbi_mul(T(-0.57282196186948), sp[0])));   // (mu=4, nu=1)
  dm[51] = gbi_fmac(T(-2.165063509461097), cp[5], gbi_fmac(T(1.7320508075688774), cp[3], gbi_mul(T(0.43301270189221935), cp[1])));   // (mu=4, nu=2)
  dm[52] = gbi_fmac(T(1.3258252147247764), sp[4], gbi_fmac(T(1.590990257669732), sp[2], gbi_mul(T(-0.795495128834866), sp[0])));   // (mu=4, nu=3)
  dm[53] = gbi_fmac(0.625f, cp[5], gbi_fmac(1.75f, cp[3], gbi_mul(-1.375f, cp[1])));   // (mu=4, nu=4)
  dm[54] = gbi_fmac(T(-0.19764235376052372), sp[4], gbi_fmac(T(-1.1858541225631423), sp[2], gbi_mul(T(-0.19764235376052372), sp[0])));   // (mu=4, nu=5)
  dm[55] = gbi_fmac(T(0.7015607600201139), sp[4], gbi_fmac(T(-1.4031215200402278), sp[2], gbi_mul(T(0.7015607600201139), sp[0])));   // (mu=5, nu=0)
  dm[56] = gbi_fmac(T(0.9057110466368398), cp[5], gbi_fmac(T(-1.8114220932736795), cp[3], gbi_mul(T(0.9057110466368398), cp[1])));   // (mu=5, nu=1)
  dm[57] = gbi_fmac(T(-0.6846531968814576), sp[4], gbi_mul(T(0.6846531968814576), sp[0]));   // (mu=5, nu=2)
  dm[58] = gbi_fmac(T(-0.41926274578121053), cp[5], gbi_fmac(T(-0.8385254915624211), cp[3], gbi_mul(T(1.2577882373436315), cp[1])));   // (mu=5, nu=3)
  dm[59] = gbi_fmac(T(0.19764235376052372), sp[4], gbi_fmac(T(1.1858541225631423), sp[2], gbi_mul(T(0.19764235376052372), sp[0])));   // (mu=5, nu=4)
  dm[60] = gbi_fmac(0.0625f, cp[5], gbi_fmac(0.625f, cp[3], gbi_mul(0.3125f, cp[1])));   // (mu=5, nu=5)
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapply5(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[4], in[4], gbi_fmac(dm[3], in[3], gbi_fmac(dm[2], in[2], gbi_fmac(dm[1], in[1], gbi_mul(dm[0], in[0])))));
  out[1] = gbi_fmac(dm[9], in[4], gbi_fmac(dm[8], in[3], gbi_fmac(dm[7], in[2], gbi_fmac(dm[6], in[1], gbi_mul(dm[5], in[0])))));
  out[2] = gbi_fmac(dm[14], in[4], gbi_fmac(dm[13], in[3], gbi_fmac(dm[12], in[2], gbi_fmac(dm[11], in[1], gbi_mul(dm[10], in[0])))));
  out[3] = gbi_fmac(dm[19], in[4], gbi_fmac(dm[18], in[3], gbi_fmac(dm[17], in[2], gbi_fmac(dm[16], in[1], gbi_mul(dm[15], in[0])))));
  out[4] = gbi_fmac(dm[24], in[4], gbi_fmac(dm[23], in[3], gbi_fmac(dm[22], in[2], gbi_fmac(dm[21], in[1], gbi_mul(dm[20], in[0])))));
  out[5] = gbi_fmac(dm[30], in[10], gbi_fmac(dm[29], in[9], gbi_fmac(dm[28], in[8], gbi_fmac(dm[27], in[7], gbi_fmac(dm[26], in[6], gbi_mul(dm[25], in[5]))))));
  out[6] = gbi_fmac(dm[36], in[10], gbi_fmac(dm[35], in[9], gbi_fmac(dm[34], in[8], gbi_fmac(dm[33], in[7], gbi_fmac(dm[32], in[6], gbi_mul(dm[31], in[5]))))));
  out[7] = gbi_fmac(dm[42], in[10], gbi_fmac(dm[41], in[9], gbi_fmac(dm[40], in[8], gbi_fmac(dm[39], in[7], gbi_fmac(dm[38], in[6], gbi_mul(dm[37], in[5]))))));
  out[8] = gbi_fmac(dm[48], in[10], gbi_fmac(dm[47], in[9], gbi_fmac(dm[46], in[8], gbi_fmac(dm[45], in[7], gbi_fmac(dm[44], in[6], gbi_mul(dm[43], in[5]))))));
  out[9] = gbi_fmac(dm[54], in[10], gbi_fmac(dm[53], in[9], gbi_fmac(dm[52], in[8], gbi_fmac(dm[51], in[7], gbi_fmac(dm[50], in[6], gbi_mul(dm[49], in[5]))))));
  out[10] = gbi_fmac(dm[60], in[10], gbi_fmac(dm[59], in[9], gbi_fmac(dm[58], in[8], gbi_fmac(dm[57], in[7], gbi_fmac(dm[56], in[6], gbi_mul(dm[55], in[5]))))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_dapplyT5(const T* __restrict__ dm, const T* __restrict__ in, T* __restrict__ out) {
  out[0] = gbi_fmac(dm[20], in[4], gbi_fmac(dm[15], in[3], gbi_fmac(dm[10], in[2], gbi_fmac(dm[5], in[1], gbi_mul(dm[0], in[0])))));
  out[1] = gbi_fmac(dm[21], in[4], gbi_fmac(dm[16], in[3], gbi_fmac(dm[11], in[2], gbi_fmac(dm[6], in[1], gbi_mul(dm[1], in[0])))));
  out[2] = gbi_fmac(dm[22], in[4], gbi_fmac(dm[17], in[3], gbi_fmac(dm[12], in[2], gbi_fmac(dm[7], in[1], gbi_mul(dm[2], in[0])))));
  out[3] = gbi_fmac(dm[23], in[4], gbi_fmac(dm[18], in[3], gbi_fmac(dm[13], in[2], gbi_fmac(dm[8], in[1], gbi_mul(dm[3], in[0])))));
  out[4] = gbi_fmac(dm[24], in[4], gbi_fmac(dm[19], in[3], gbi_fmac(dm[14], in[2], gbi_fmac(dm[9], in[1], gbi_mul(dm[4], in[0])))));
  out[5] = gbi_fmac(dm[55], in[10], gbi_fmac(dm[49], in[9], gbi_fmac(dm[43], in[8], gbi_fmac(dm[37], in[7], gbi_fmac(dm[31], in[6], gbi_mul(dm[25], in[5]))))));
  out[6] = gbi_fmac(dm[56], in[10], gbi_fmac(dm[50], in[9], gbi_fmac(dm[44], in[8], gbi_fmac(dm[38], in[7], gbi_fmac(dm[32], in[6], gbi_mul(dm[26], in[5]))))));
  out[7] = gbi_fmac(dm[57], in[10], gbi_fmac(dm[51], in[9], gbi_fmac(dm[45], in[8], gbi_fmac(dm[39], in[7], gbi_fmac(dm[33], in[6], gbi_mul(dm[27], in[5]))))));
  out[8] = gbi_fmac(dm[58], in[10], gbi_fmac(dm[52], in[9], gbi_fmac(dm[46], in[8], gbi_fmac(dm[40], in[7], gbi_fmac(dm[34], in[6], gbi_mul(dm[28], in[5]))))));
  out[9] = gbi_fmac(dm[59], in[10], gbi_fmac(dm[53], in[9], gbi_fmac(dm[47], in[8], gbi_fmac(dm[41], in[7], gbi_fmac(dm[35], in[6], gbi_mul(dm[29], in[5]))))));
  out[10] = gbi_fmac(dm[60], in[10], gbi_fmac(dm[54], in[9], gbi_fmac(dm[48], in[8], gbi_fmac(dm[42], in[7], gbi_fmac(dm[36], in[6], gbi_mul(dm[30], in[5]))))));
}

template <typename T> __host__ __device__ __forceinline__ void gbi_pack2(T x, T y, T z, T* __restrict__ out) {
  out[0] = T(1.414213562373095) * x * y;
  out[1] = T(1.414213562373095) * y * z;
  out[2] = T(0.816496580927726) * z * z + T(-0.408248290463863) * y * y + T(-0.408248290463863) * x * x;
  out[3] = T(1.414213562373095) * x * z;
  out[4] = T(-0.7071067811865475) * y * y + T(0.7071067811865475) * x * x;
}
template <typename T> __host__ __device__ __forceinline__ void gbi_unpack2(const T* __restrict__ yv, T* __restrict__ s6) {
  s6[0] = T(-0.408248290463863) * yv[2] + T(0.7071067811865475) * yv[4];
  s6[1] = T(0.7071067811865475) * yv[0];
  s6[2] = T(0.7071067811865475) * yv[3];
  s6[3] = T(-0.408248290463863) * yv[2] + T(-0.7071067811865475) * yv[4];
  s6[4] = T(0.7071067811865475) * yv[1];
  s6[5] = T(0.816496580927726) * yv[2];
}

// ---------------- truncation l <= 2: 14 components per sphere
struct GbiTrunc2 {
  static constexpr int D = 14;      // components per sphere (L + H)
  static constexpr int NL = 6;
  static constexpr int H = 8;
  static constexpr int NMODE = 4;
  static constexpr int MAXK = 2;
};
__host__ __device__ constexpr int gbi_t2_k(int m) { constexpr int v[4] = {1, 1, 2, 1}; return v[m]; }
__host__ __device__ constexpr int gbi_t2_L(int m) { constexpr int v[4] = {1, 2, 2, 3}; return v[m]; }
__host__ __device__ constexpr int gbi_t2_off(int m) { constexpr int v[4] = {0, 3, 6, 11}; return v[m]; }
// internal coordinate x = scale * packed coordinate of the paper's irreducible tensor
static const double gbi_t2_scale[14] = {1.0, 1.0, 1.0, 0.7071067811865476, 0.7071067811865476, 0.7071067811865476, 1.0, 1.0, 1.0, 1.0, 1.0, 0.7745966692414834, 0.7745966692414834, 0.7745966692414834};
// self scalar g per component (units 1/a): 8 pi eta V = -g Q for an isolated sphere
static const double gbi_t2_self[14] = {1.3333333333333333, 1.3333333333333333, 1.3333333333333333, 2.0, 2.0, 2.0, 1.2, 1.2, 1.2, 1.2, 1.2, 4.0, 4.0, 4.0};
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_all_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0]), gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0])));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1]), gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])));
  y[2] = gbi_fmac(e2, gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2]), gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2])));
  y[3] = gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]));
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]));
  y[6] = gbi_fmac(e2, T(2.4) * xs[6], T(0));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0]), gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5])));
  y[8] = gbi_fmac(e2, gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1]), gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2]), gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3])));
  y[10] = gbi_fmac(e2, T(2.4) * xs[10], T(0));
  y[11] = gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0]);
  y[12] = gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1]);
  y[13] = gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_all_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_all_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(2.262741699796952) * xs[7], T(-0.5163977794943223) * xs[11]);
  y[1] = gbi_fmac(e2, T(-3.919183588453085) * xs[8], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]));
  y[2] = gbi_fmac(e2, T(2.262741699796952) * xs[9], T(-0.5163977794943223) * xs[13]);
  y[3] = T(-3.0) * xs[9];
  y[4] = T(0);
  y[5] = T(3.0) * xs[7];
  y[6] = gbi_fmac(e2, T(2.4) * xs[6], T(0));
  y[7] = gbi_fmac(e2, T(-9.6) * xs[7], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7]));
  y[8] = gbi_fmac(e2, T(14.4) * xs[8], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]));
  y[9] = gbi_fmac(e2, T(-9.6) * xs[9], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9]));
  y[10] = gbi_fmac(e2, T(2.4) * xs[10], T(0));
  y[11] = T(-2.1908902300206647) * xs[7];
  y[12] = T(3.7947331922020555) * xs[8];
  y[13] = T(-2.1908902300206647) * xs[9];
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_L_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0]), gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0])));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1]), gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])));
  y[2] = gbi_fmac(e2, gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2]), gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2])));
  y[3] = gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]));
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_L_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_L_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(2.262741699796952) * xs[7], T(-0.5163977794943223) * xs[11]);
  y[1] = gbi_fmac(e2, T(-3.919183588453085) * xs[8], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]));
  y[2] = gbi_fmac(e2, T(2.262741699796952) * xs[9], T(-0.5163977794943223) * xs[13]);
  y[3] = T(-3.0) * xs[9];
  y[4] = T(0);
  y[5] = T(3.0) * xs[7];
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_H_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, T(2.4) * xs[6], T(0));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0]), gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5])));
  y[8] = gbi_fmac(e2, gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1]), gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2]), gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3])));
  y[10] = gbi_fmac(e2, T(2.4) * xs[10], T(0));
  y[11] = gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0]);
  y[12] = gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1]);
  y[13] = gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_H_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_H_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, T(2.4) * xs[6], T(0));
  y[7] = gbi_fmac(e2, T(-9.6) * xs[7], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7]));
  y[8] = gbi_fmac(e2, T(14.4) * xs[8], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]));
  y[9] = gbi_fmac(e2, T(-9.6) * xs[9], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9]));
  y[10] = gbi_fmac(e2, T(2.4) * xs[10], T(0));
  y[11] = T(-2.1908902300206647) * xs[7];
  y[12] = T(3.7947331922020555) * xs[8];
  y[13] = T(-2.1908902300206647) * xs[9];
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t2_couple_P_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // point target: 1s rows only, beta from the source's finite-size operator alone
  y[0] = gbi_fmac(e2, gbi_fmac(T(0.848528137423857), xs[7], T(0.3333333333333333) * xs[0]), gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0])));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-1.469693845669907), xs[8], T(-0.6666666666666666) * xs[1]), gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])));
  y[2] = gbi_fmac(e2, gbi_fmac(T(0.848528137423857), xs[9], T(0.3333333333333333) * xs[2]), gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2])));
}
static constexpr int gbi_t2_nnz = 37;   // pair-frame nonzeros (all rows, all columns)
static constexpr int gbi_t2_flops_point = 250;   // per (point, sphere): 1s rows from all columns
// algorithmic flops per ordered pair, [rows][cols] with 0 = all, 1 = L, 2 = H
static constexpr int gbi_t2_flops[3][3] = {{420, 316, 343}, {290, 166, 231}, {324, 238, 273}};

// ---------------- truncation l <= 3: 31 components per sphere
struct GbiTrunc3 {
  static constexpr int D = 31;      // components per sphere (L + H)
  static constexpr int NL = 6;
  static constexpr int H = 25;
  static constexpr int NMODE = 7;
  static constexpr int MAXK = 3;
};
__host__ __device__ constexpr int gbi_t3_k(int m) { constexpr int v[7] = {1, 1, 2, 1, 2, 3, 2}; return v[m]; }
__host__ __device__ constexpr int gbi_t3_L(int m) { constexpr int v[7] = {1, 2, 2, 3, 3, 3, 4}; return v[m]; }
__host__ __device__ constexpr int gbi_t3_off(int m) { constexpr int v[7] = {0, 3, 6, 11, 14, 19, 26}; return v[m]; }
// internal coordinate x = scale * packed coordinate of the paper's irreducible tensor
static const double gbi_t3_scale[31] = {1.0, 1.0, 1.0, 0.7071067811865476, 0.7071067811865476, 0.7071067811865476, 1.0, 1.0, 1.0, 1.0, 1.0, 0.7745966692414834, 0.7745966692414834, 0.7745966692414834, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422};
// self scalar g per component (units 1/a): 8 pi eta V = -g Q for an isolated sphere
static const double gbi_t3_self[31] = {1.3333333333333333, 1.3333333333333333, 1.3333333333333333, 2.0, 2.0, 2.0, 1.2, 1.2, 1.2, 1.2, 1.2, 4.0, 4.0, 4.0, 12.0, 12.0, 12.0, 12.0, 12.0, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 72.0, 72.0, 72.0, 72.0, 72.0};
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_all_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0])), gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1])), gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2])), gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))));
  y[3] = gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))));
  y[4] = gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4]);
  y[5] = gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))));
  y[6] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]), gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0])), gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5]))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1])), gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2])), gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3]))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]), gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])));
  y[11] = gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0]));
  y[12] = gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1]));
  y[13] = gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2]));
  y[14] = gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]));
  y[15] = gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))));
  y[16] = gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4]);
  y[17] = gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))));
  y[18] = gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]));
  y[19] = gbi_fmac(e2, T(25.71428571428571) * xs[19], T(-6.0) * xs[19]);
  y[20] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]), gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0])), gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0])))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1])), gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1])))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2])), gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2])))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]), gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))));
  y[25] = gbi_fmac(e2, T(25.71428571428571) * xs[25], T(-6.0) * xs[25]);
  y[26] = gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]);
  y[27] = gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0]));
  y[28] = gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1]));
  y[29] = gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2]));
  y[30] = gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_all_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_all_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7]), gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11]))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8]), gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9]), gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13]))));
  y[3] = gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]));
  y[4] = T(8.485281374238571) * xs[16];
  y[5] = gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]));
  y[6] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]), gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7]), gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7])))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8]), gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9]), gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9])))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]), gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])));
  y[11] = gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7]);
  y[12] = gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8]);
  y[13] = gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9]);
  y[14] = gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]));
  y[15] = gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]));
  y[16] = T(-48.0) * xs[16];
  y[17] = gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]));
  y[18] = gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]));
  y[19] = gbi_fmac(e2, T(25.71428571428571) * xs[19], T(-6.0) * xs[19]);
  y[20] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]), gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7]), gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7])))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8]), gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8]))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9]), gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9])))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]), gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))));
  y[25] = gbi_fmac(e2, T(25.71428571428571) * xs[25], T(-6.0) * xs[25]);
  y[26] = gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]);
  y[27] = gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7]);
  y[28] = gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8]);
  y[29] = gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9]);
  y[30] = gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_L_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0])), gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1])), gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2])), gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))));
  y[3] = gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))));
  y[4] = gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4]);
  y[5] = gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_L_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_L_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7]), gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11]))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8]), gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9]), gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13]))));
  y[3] = gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]));
  y[4] = T(8.485281374238571) * xs[16];
  y[5] = gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_H_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]), gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0])), gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5]))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1])), gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2])), gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3]))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]), gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])));
  y[11] = gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0]));
  y[12] = gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1]));
  y[13] = gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2]));
  y[14] = gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]));
  y[15] = gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))));
  y[16] = gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4]);
  y[17] = gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))));
  y[18] = gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]));
  y[19] = gbi_fmac(e2, T(25.71428571428571) * xs[19], T(-6.0) * xs[19]);
  y[20] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]), gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0])), gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0])))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1])), gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1])))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2])), gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2])))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]), gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))));
  y[25] = gbi_fmac(e2, T(25.71428571428571) * xs[25], T(-6.0) * xs[25]);
  y[26] = gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]);
  y[27] = gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0]));
  y[28] = gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1]));
  y[29] = gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2]));
  y[30] = gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_H_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_H_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]), gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7]), gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7])))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8]), gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9]), gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9])))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]), gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])));
  y[11] = gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7]);
  y[12] = gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8]);
  y[13] = gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9]);
  y[14] = gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]));
  y[15] = gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]));
  y[16] = T(-48.0) * xs[16];
  y[17] = gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]));
  y[18] = gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]));
  y[19] = gbi_fmac(e2, T(25.71428571428571) * xs[19], T(-6.0) * xs[19]);
  y[20] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]), gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7]), gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7])))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8]), gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8]))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9]), gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9])))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]), gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))));
  y[25] = gbi_fmac(e2, T(25.71428571428571) * xs[25], T(-6.0) * xs[25]);
  y[26] = gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]);
  y[27] = gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7]);
  y[28] = gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8]);
  y[29] = gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9]);
  y[30] = gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t3_couple_P_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // point target: 1s rows only, beta from the source's finite-size operator alone
  y[0] = gbi_fmac(e2, gbi_fmac(T(3.319700011034928), xs[21], gbi_fmac(T(0.848528137423857), xs[7], T(0.3333333333333333) * xs[0])), gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-5.421047417431508), xs[22], gbi_fmac(T(-1.469693845669907), xs[8], T(-0.6666666666666666) * xs[1])), gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(3.319700011034928), xs[23], gbi_fmac(T(0.848528137423857), xs[9], T(0.3333333333333333) * xs[2])), gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))));
}
static constexpr int gbi_t3_nnz = 127;   // pair-frame nonzeros (all rows, all columns)
static constexpr int gbi_t3_flops_point = 531;   // per (point, sphere): 1s rows from all columns
// algorithmic flops per ordered pair, [rows][cols] with 0 = all, 1 = L, 2 = H
static constexpr int gbi_t3_flops[3][3] = {{1105, 658, 996}, {581, 166, 522}, {977, 580, 894}};

// ---------------- truncation l <= 4: 54 components per sphere
struct GbiTrunc4 {
  static constexpr int D = 54;      // components per sphere (L + H)
  static constexpr int NL = 6;
  static constexpr int H = 48;
  static constexpr int NMODE = 10;
  static constexpr int MAXK = 4;
};
__host__ __device__ constexpr int gbi_t4_k(int m) { constexpr int v[10] = {1, 1, 2, 1, 2, 3, 2, 3, 4, 3}; return v[m]; }
__host__ __device__ constexpr int gbi_t4_L(int m) { constexpr int v[10] = {1, 2, 2, 3, 3, 3, 4, 4, 4, 5}; return v[m]; }
__host__ __device__ constexpr int gbi_t4_off(int m) { constexpr int v[10] = {0, 3, 6, 11, 14, 19, 26, 31, 38, 47}; return v[m]; }
// internal coordinate x = scale * packed coordinate of the paper's irreducible tensor
static const double gbi_t4_scale[54] = {1.0, 1.0, 1.0, 0.7071067811865476, 0.7071067811865476, 0.7071067811865476, 1.0, 1.0, 1.0, 1.0, 1.0, 0.7745966692414834, 0.7745966692414834, 0.7745966692414834, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424};
// self scalar g per component (units 1/a): 8 pi eta V = -g Q for an isolated sphere
static const double gbi_t4_self[54] = {1.3333333333333333, 1.3333333333333333, 1.3333333333333333, 2.0, 2.0, 2.0, 1.2, 1.2, 1.2, 1.2, 1.2, 4.0, 4.0, 4.0, 12.0, 12.0, 12.0, 12.0, 12.0, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 72.0, 72.0, 72.0, 72.0, 72.0, 180.0, 180.0, 180.0, 180.0, 180.0, 180.0, 180.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 2160.0, 2160.0, 2160.0, 2160.0, 2160.0, 2160.0, 2160.0};
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_all_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0]))), gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0])))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1]))), gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2]))), gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2])))))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4]));
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))))));
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18]))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0]))), gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5])))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1]))), gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2]))), gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3])))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14]))))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0])));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1])));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2])));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4]));
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19]))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6])))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0]))), gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]))))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1]))), gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1])))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2]))), gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]))))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10])))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25]))));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0])));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1])));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2])));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], gbi_fmac(T(-47.434164902525694), xs[9], gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]))))));
  y[34] = gbi_fmac(2700.0f, xs[34], gbi_fmac(T(328.63353450309967), xs[16], T(46.475800154489) * xs[4]));
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], gbi_fmac(T(47.434164902525694), xs[7], gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]))))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19]))));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6])))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], gbi_fmac(T(-419.06562731868144), xs[7], T(-70.55336829505575) * xs[0]))), gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], gbi_fmac(T(120.26755886059097), xs[7], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]))))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], gbi_fmac(T(573.8292428937376), xs[8], T(111.55467020454341) * xs[1]))), gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], gbi_fmac(T(-175.662013130736), xs[8], T(-35.85685828003181) * xs[1])))))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], gbi_fmac(T(-419.06562731868144), xs[9], T(-70.55336829505575) * xs[2]))), gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], gbi_fmac(T(120.26755886059097), xs[9], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]))))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10])))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25]))));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
  y[47] = gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]);
  y[48] = gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6]));
  y[49] = gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], gbi_fmac(T(-124.21180068162376), xs[7], T(-17.5662013130736) * xs[0])));
  y[50] = gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], gbi_fmac(T(175.66201313073597), xs[8], T(28.685486624025447) * xs[1])));
  y[51] = gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], gbi_fmac(T(-124.21180068162376), xs[9], T(-17.5662013130736) * xs[2])));
  y[52] = gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10]));
  y[53] = gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_all_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
  y[31] = T(0);
  y[32] = T(0);
  y[33] = gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]);
  y[34] = T(46.475800154489) * xs[4];
  y[35] = gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]);
  y[36] = T(0);
  y[37] = T(0);
  y[38] = T(0);
  y[39] = T(0);
  y[40] = T(0);
  y[41] = gbi_fmac(e2, T(-70.55336829505575) * xs[0], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]));
  y[42] = gbi_fmac(e2, T(111.55467020454341) * xs[1], T(-35.85685828003181) * xs[1]);
  y[43] = gbi_fmac(e2, T(-70.55336829505575) * xs[2], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]));
  y[44] = T(0);
  y[45] = T(0);
  y[46] = T(0);
  y[47] = T(0);
  y[48] = T(0);
  y[49] = T(-17.5662013130736) * xs[0];
  y[50] = T(28.685486624025447) * xs[1];
  y[51] = T(-17.5662013130736) * xs[2];
  y[52] = T(0);
  y[53] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_all_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7])), gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11])))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8])), gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9])), gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13])))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], T(8.485281374238571) * xs[16]);
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]))));
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18]))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7])), gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7]))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8])), gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9])), gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9]))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14]))))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7]));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8]));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9]));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], T(-48.0) * xs[16]);
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19]))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6])))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7])), gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7]))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8])), gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8]))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9])), gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9]))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10])))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25]))));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7]));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8]));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9]));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], T(-47.434164902525694) * xs[9]))));
  y[34] = gbi_fmac(2700.0f, xs[34], T(328.63353450309967) * xs[16]);
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], T(47.434164902525694) * xs[7]))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19]))));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6])))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], T(-419.06562731868144) * xs[7])), gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], T(120.26755886059097) * xs[7]))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], T(573.8292428937376) * xs[8])), gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], T(-175.662013130736) * xs[8]))))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], T(-419.06562731868144) * xs[9])), gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], T(120.26755886059097) * xs[9]))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10])))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25]))));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
  y[47] = gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]);
  y[48] = gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6]));
  y[49] = gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], T(-124.21180068162376) * xs[7]));
  y[50] = gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], T(175.66201313073597) * xs[8]));
  y[51] = gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], T(-124.21180068162376) * xs[9]));
  y[52] = gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10]));
  y[53] = gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_L_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0]))), gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0])))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1]))), gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2]))), gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2])))))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4]));
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_L_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_L_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7])), gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11])))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8])), gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9])), gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13])))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], T(8.485281374238571) * xs[16]);
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_H_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18]))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0]))), gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5])))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1]))), gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2]))), gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3])))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14]))))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0])));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1])));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2])));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4]));
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19]))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6])))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0]))), gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]))))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1]))), gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1])))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2]))), gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]))))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10])))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25]))));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0])));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1])));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2])));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], gbi_fmac(T(-47.434164902525694), xs[9], gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]))))));
  y[34] = gbi_fmac(2700.0f, xs[34], gbi_fmac(T(328.63353450309967), xs[16], T(46.475800154489) * xs[4]));
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], gbi_fmac(T(47.434164902525694), xs[7], gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]))))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19]))));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6])))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], gbi_fmac(T(-419.06562731868144), xs[7], T(-70.55336829505575) * xs[0]))), gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], gbi_fmac(T(120.26755886059097), xs[7], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]))))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], gbi_fmac(T(573.8292428937376), xs[8], T(111.55467020454341) * xs[1]))), gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], gbi_fmac(T(-175.662013130736), xs[8], T(-35.85685828003181) * xs[1])))))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], gbi_fmac(T(-419.06562731868144), xs[9], T(-70.55336829505575) * xs[2]))), gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], gbi_fmac(T(120.26755886059097), xs[9], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]))))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10])))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25]))));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
  y[47] = gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]);
  y[48] = gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6]));
  y[49] = gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], gbi_fmac(T(-124.21180068162376), xs[7], T(-17.5662013130736) * xs[0])));
  y[50] = gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], gbi_fmac(T(175.66201313073597), xs[8], T(28.685486624025447) * xs[1])));
  y[51] = gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], gbi_fmac(T(-124.21180068162376), xs[9], T(-17.5662013130736) * xs[2])));
  y[52] = gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10]));
  y[53] = gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_H_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
  y[31] = T(0);
  y[32] = T(0);
  y[33] = gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]);
  y[34] = T(46.475800154489) * xs[4];
  y[35] = gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]);
  y[36] = T(0);
  y[37] = T(0);
  y[38] = T(0);
  y[39] = T(0);
  y[40] = T(0);
  y[41] = gbi_fmac(e2, T(-70.55336829505575) * xs[0], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]));
  y[42] = gbi_fmac(e2, T(111.55467020454341) * xs[1], T(-35.85685828003181) * xs[1]);
  y[43] = gbi_fmac(e2, T(-70.55336829505575) * xs[2], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]));
  y[44] = T(0);
  y[45] = T(0);
  y[46] = T(0);
  y[47] = T(0);
  y[48] = T(0);
  y[49] = T(-17.5662013130736) * xs[0];
  y[50] = T(28.685486624025447) * xs[1];
  y[51] = T(-17.5662013130736) * xs[2];
  y[52] = T(0);
  y[53] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_H_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18]))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7])), gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7]))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8])), gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9])), gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9]))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14]))))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7]));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8]));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9]));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], T(-48.0) * xs[16]);
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19]))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6])))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7])), gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7]))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8])), gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8]))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9])), gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9]))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10])))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25]))));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7]));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8]));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9]));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], T(-47.434164902525694) * xs[9]))));
  y[34] = gbi_fmac(2700.0f, xs[34], T(328.63353450309967) * xs[16]);
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], T(47.434164902525694) * xs[7]))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19]))));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6])))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], T(-419.06562731868144) * xs[7])), gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], T(120.26755886059097) * xs[7]))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], T(573.8292428937376) * xs[8])), gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], T(-175.662013130736) * xs[8]))))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], T(-419.06562731868144) * xs[9])), gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], T(120.26755886059097) * xs[9]))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10])))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25]))));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
  y[47] = gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]);
  y[48] = gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6]));
  y[49] = gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], T(-124.21180068162376) * xs[7]));
  y[50] = gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], T(175.66201313073597) * xs[8]));
  y[51] = gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], T(-124.21180068162376) * xs[9]));
  y[52] = gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10]));
  y[53] = gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t4_couple_P_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // point target: 1s rows only, beta from the source's finite-size operator alone
  y[0] = gbi_fmac(e2, gbi_fmac(T(17.638342073763937), xs[41], gbi_fmac(T(3.319700011034928), xs[21], gbi_fmac(T(0.848528137423857), xs[7], T(0.3333333333333333) * xs[0]))), gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0])))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-27.888667551135853), xs[42], gbi_fmac(T(-5.421047417431508), xs[22], gbi_fmac(T(-1.469693845669907), xs[8], T(-0.6666666666666666) * xs[1]))), gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(17.638342073763937), xs[43], gbi_fmac(T(3.319700011034928), xs[23], gbi_fmac(T(0.848528137423857), xs[9], T(0.3333333333333333) * xs[2]))), gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2])))))))));
}
static constexpr int gbi_t4_nnz = 297;   // pair-frame nonzeros (all rows, all columns)
static constexpr int gbi_t4_flops_point = 1002;   // per (point, sphere): 1s rows from all columns
// algorithmic flops per ordered pair, [rows][cols] with 0 = all, 1 = L, 2 = H
static constexpr int gbi_t4_flops[3][3] = {{2288, 1208, 2147}, {1062, 166, 1003}, {2128, 1130, 2013}};

// ---------------- truncation l <= 5: 83 components per sphere
struct GbiTrunc5 {
  static constexpr int D = 83;      // components per sphere (L + H)
  static constexpr int NL = 6;
  static constexpr int H = 77;
  static constexpr int NMODE = 13;
  static constexpr int MAXK = 5;
};
__host__ __device__ constexpr int gbi_t5_k(int m) { constexpr int v[13] = {1, 1, 2, 1, 2, 3, 2, 3, 4, 3, 4, 5, 4}; return v[m]; }
__host__ __device__ constexpr int gbi_t5_L(int m) { constexpr int v[13] = {1, 2, 2, 3, 3, 3, 4, 4, 4, 5, 5, 5, 6}; return v[m]; }
__host__ __device__ constexpr int gbi_t5_off(int m) { constexpr int v[13] = {0, 3, 6, 11, 14, 19, 26, 31, 38, 47, 54, 63, 74}; return v[m]; }
// internal coordinate x = scale * packed coordinate of the paper's irreducible tensor
static const double gbi_t5_scale[83] = {1.0, 1.0, 1.0, 0.7071067811865476, 0.7071067811865476, 0.7071067811865476, 1.0, 1.0, 1.0, 1.0, 1.0, 0.7745966692414834, 0.7745966692414834, 0.7745966692414834, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424, 1.259881576697424, 0.8944271909999159, 0.8944271909999159, 0.8944271909999159, 0.8944271909999159, 0.8944271909999159, 0.8944271909999159, 0.8944271909999159, 0.8944271909999159, 0.8944271909999159, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.5075567228888183, 1.5075567228888183, 1.5075567228888183, 1.5075567228888183, 1.5075567228888183, 1.5075567228888183, 1.5075567228888183, 1.5075567228888183, 1.5075567228888183};
// self scalar g per component (units 1/a): 8 pi eta V = -g Q for an isolated sphere
static const double gbi_t5_self[83] = {1.3333333333333333, 1.3333333333333333, 1.3333333333333333, 2.0, 2.0, 2.0, 1.2, 1.2, 1.2, 1.2, 1.2, 4.0, 4.0, 4.0, 12.0, 12.0, 12.0, 12.0, 12.0, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 72.0, 72.0, 72.0, 72.0, 72.0, 180.0, 180.0, 180.0, 180.0, 180.0, 180.0, 180.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 2160.0, 2160.0, 2160.0, 2160.0, 2160.0, 2160.0, 2160.0, 5040.0, 5040.0, 5040.0, 5040.0, 5040.0, 5040.0, 5040.0, 5040.0, 5040.0, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 2749.090909090909, 100800.0, 100800.0, 100800.0, 100800.0, 100800.0, 100800.0, 100800.0, 100800.0, 100800.0};
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_all_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[67], gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0])))), gbi_fmac(T(-127.63584563479449), xs[77], gbi_fmac(T(-86.94826047713663), xs[67], gbi_fmac(T(-70.99295739719538), xs[59], gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-857.1796922427575), xs[68], gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1])))), gbi_fmac(T(201.8099916438052), xs[78], gbi_fmac(T(224.49944320643647), xs[68], gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[69], gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2])))), gbi_fmac(T(-127.63584563479449), xs[79], gbi_fmac(T(-86.94826047713663), xs[69], gbi_fmac(T(70.99295739719538), xs[57], gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))))))))));
  y[3] = gbi_fmac(T(-368.8902275745455), xs[69], gbi_fmac(T(-200.79840636817812), xs[57], gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))))))));
  y[4] = gbi_fmac(T(317.49015732775086), xs[58], gbi_fmac(T(46.475800154489), xs[34], gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4])));
  y[5] = gbi_fmac(T(368.8902275745455), xs[67], gbi_fmac(T(-200.79840636817812), xs[59], gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))))))));
  y[6] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[66], gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]))), gbi_fmac(T(-382.90753690438345), xs[76], gbi_fmac(T(-325.330601081423), xs[66], gbi_fmac(T(-212.9788721915862), xs[60], gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[67], gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0])))), gbi_fmac(T(1083.026063650111), xs[77], gbi_fmac(T(983.7072735321215), xs[67], gbi_fmac(T(301.1976095522672), xs[59], gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5]))))))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(5039.166873289622), xs[68], gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1])))), gbi_fmac(T(-1482.994513567979), xs[78], gbi_fmac(T(-1374.772708486752), xs[68], gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])))))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[69], gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2])))), gbi_fmac(T(1083.026063650111), xs[79], gbi_fmac(T(983.7072735321215), xs[69], gbi_fmac(T(-301.1976095522672), xs[57], gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3]))))))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[70], gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]))), gbi_fmac(T(-382.90753690438345), xs[80], gbi_fmac(T(-325.330601081423), xs[70], gbi_fmac(T(212.9788721915862), xs[56], gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))))))));
  y[11] = gbi_fmac(T(-673.4983296193094), xs[67], gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0]))));
  y[12] = gbi_fmac(T(1043.3791257256396), xs[68], gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1]))));
  y[13] = gbi_fmac(T(-673.4983296193094), xs[69], gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2]))));
  y[14] = gbi_fmac(T(-1593.7879407248633), xs[70], gbi_fmac(T(-695.586083817093), xs[56], gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))))));
  y[15] = gbi_fmac(T(2108.3832668658706), xs[69], gbi_fmac(T(1967.4145470642432), xs[57], gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))))))));
  y[16] = gbi_fmac(T(-2693.993318477238), xs[58], gbi_fmac(T(-328.63353450309967), xs[34], gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4])));
  y[17] = gbi_fmac(T(-2108.3832668658706), xs[67], gbi_fmac(T(1967.4145470642432), xs[59], gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))))))));
  y[18] = gbi_fmac(T(1593.7879407248633), xs[66], gbi_fmac(T(-695.586083817093), xs[60], gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))))));
  y[19] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[65], gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19])), gbi_fmac(T(-1013.0781177812858), xs[75], gbi_fmac(T(-1126.978260659894), xs[65], gbi_fmac(T(-563.4891303299471), xs[61], gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])))))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[66], gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]))), gbi_fmac(T(4642.50715963613), xs[76], gbi_fmac(T(4507.913042639577), xs[66], gbi_fmac(T(1721.4877286812125), xs[60], gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[67], gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0])))), gbi_fmac(T(-10380.961594975855), xs[77], gbi_fmac(T(-9428.976614670333), xs[67], gbi_fmac(T(-1924.681791881453), xs[59], gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0])))))))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-41821.305812166014), xs[68], gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1])))), gbi_fmac(T(13401.763791653422), xs[78], gbi_fmac(T(11926.816842728827), xs[68], gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1])))))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[69], gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2])))), gbi_fmac(T(-10380.961594975855), xs[79], gbi_fmac(T(-9428.976614670333), xs[69], gbi_fmac(T(1924.681791881453), xs[57], gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2])))))))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[70], gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]))), gbi_fmac(T(4642.50715963613), xs[80], gbi_fmac(T(4507.913042639577), xs[70], gbi_fmac(T(-1721.4877286812125), xs[56], gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))))))));
  y[25] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[71], gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25])), gbi_fmac(T(-1013.0781177812858), xs[81], gbi_fmac(T(-1126.978260659894), xs[71], gbi_fmac(T(563.4891303299471), xs[55], gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])))))));
  y[26] = gbi_fmac(T(-3299.4545003682047), xs[66], gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6])));
  y[27] = gbi_fmac(T(8729.536070147142), xs[67], gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0]))));
  y[28] = gbi_fmac(T(-11711.901638931227), xs[68], gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1]))));
  y[29] = gbi_fmac(T(8729.536070147142), xs[69], gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2]))));
  y[30] = gbi_fmac(T(-3299.4545003682047), xs[70], gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10])));
  y[31] = gbi_fmac(T(-5855.950819465615), xs[71], gbi_fmac(T(-1951.983606488538), xs[55], gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]))));
  y[32] = gbi_fmac(T(15615.868851908304), xs[70], gbi_fmac(T(8945.11263204662), xs[56], gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))))));
  y[33] = gbi_fmac(T(-16331.46655998781), xs[69], gbi_fmac(T(-20001.879911648302), xs[57], gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], gbi_fmac(T(-47.434164902525694), xs[9], gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]))))))));
  y[34] = gbi_fmac(T(25822.315930218192), xs[58], gbi_fmac(2700.0f, xs[34], gbi_fmac(T(328.63353450309967), xs[16], T(46.475800154489) * xs[4])));
  y[35] = gbi_fmac(T(16331.46655998781), xs[67], gbi_fmac(T(-20001.879911648302), xs[59], gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], gbi_fmac(T(47.434164902525694), xs[7], gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]))))))));
  y[36] = gbi_fmac(T(-15615.868851908304), xs[66], gbi_fmac(T(8945.11263204662), xs[60], gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))))));
  y[37] = gbi_fmac(T(5855.950819465615), xs[65], gbi_fmac(T(-1951.983606488538), xs[61], gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]))));
  y[38] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[64], T(560.0) * xs[38]), gbi_fmac(T(-2026.1562355625713), xs[74], gbi_fmac(T(-3380.934781979682), xs[64], gbi_fmac(T(-1126.978260659894), xs[62], T(-180.0) * xs[38]))));
  y[39] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[65], gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19])), gbi_fmac(T(16209.24988450057), xs[75], gbi_fmac(T(19158.630431218196), xs[65], gbi_fmac(T(6761.869563959364), xs[61], gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])))))));
  y[40] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[66], gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6]))), gbi_fmac(T(-56732.374595752), xs[76], gbi_fmac(T(-56071.31459133092), xs[66], gbi_fmac(T(-15777.695649238518), xs[60], gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))))))));
  y[41] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[67], gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], gbi_fmac(T(-419.06562731868144), xs[7], T(-70.55336829505575) * xs[0])))), gbi_fmac(T(113464.749191504), xs[77], gbi_fmac(T(102139.30252356337), xs[67], gbi_fmac(T(15777.695649238516), xs[59], gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], gbi_fmac(T(120.26755886059097), xs[7], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0])))))))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(T(430300.7904337778), xs[68], gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], gbi_fmac(T(573.8292428937376), xs[8], T(111.55467020454341) * xs[1])))), gbi_fmac(T(-141830.93648938002), xs[78], gbi_fmac(T(-123967.60867258835), xs[68], gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], gbi_fmac(T(-175.662013130736), xs[8], T(-35.85685828003181) * xs[1])))))))));
  y[43] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[69], gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], gbi_fmac(T(-419.06562731868144), xs[9], T(-70.55336829505575) * xs[2])))), gbi_fmac(T(113464.749191504), xs[79], gbi_fmac(T(102139.30252356337), xs[69], gbi_fmac(T(-15777.695649238516), xs[57], gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], gbi_fmac(T(120.26755886059097), xs[9], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2])))))))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[70], gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10]))), gbi_fmac(T(-56732.374595752), xs[80], gbi_fmac(T(-56071.31459133092), xs[70], gbi_fmac(T(15777.695649238518), xs[56], gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))))))));
  y[45] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[71], gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25])), gbi_fmac(T(16209.24988450057), xs[81], gbi_fmac(T(19158.630431218196), xs[71], gbi_fmac(T(-6761.869563959364), xs[55], gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])))))));
  y[46] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[72], T(560.0) * xs[46]), gbi_fmac(T(-2026.1562355625713), xs[82], gbi_fmac(T(-3380.934781979682), xs[72], gbi_fmac(T(1126.978260659894), xs[54], T(-180.0) * xs[46]))));
  y[47] = gbi_fmac(T(-12778.73233149517), xs[65], gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]));
  y[48] = gbi_fmac(T(51114.92932598069), xs[66], gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6])));
  y[49] = gbi_fmac(T(-106914.54531540598), xs[67], gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], gbi_fmac(T(-124.21180068162376), xs[7], T(-17.5662013130736) * xs[0]))));
  y[50] = gbi_fmac(T(135237.3912791873), xs[68], gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], gbi_fmac(T(175.66201313073597), xs[8], T(28.685486624025447) * xs[1]))));
  y[51] = gbi_fmac(T(-106914.54531540598), xs[69], gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], gbi_fmac(T(-124.21180068162376), xs[9], T(-17.5662013130736) * xs[2]))));
  y[52] = gbi_fmac(T(51114.92932598069), xs[70], gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10])));
  y[53] = gbi_fmac(T(-12778.73233149517), xs[71], gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]));
  y[54] = gbi_fmac(-18144.0f, xs[72], gbi_fmac(T(-4031.9999999999995), xs[54], T(-1126.978260659894) * xs[46]));
  y[55] = gbi_fmac(81648.0f, xs[71], gbi_fmac(T(32255.999999999996), xs[55], gbi_fmac(T(6761.869563959364), xs[45], gbi_fmac(T(1951.983606488538), xs[31], T(563.4891303299471) * xs[25]))));
  y[56] = gbi_fmac(T(-166292.5068185575), xs[70], gbi_fmac(-112896.0f, xs[56], gbi_fmac(T(-15777.695649238518), xs[44], gbi_fmac(T(-8945.11263204662), xs[32], gbi_fmac(T(-1721.4877286812125), xs[24], gbi_fmac(T(-695.586083817093), xs[14], T(-212.9788721915862) * xs[10]))))));
  y[57] = gbi_fmac(T(155552.39662570294), xs[69], gbi_fmac(225792.0f, xs[57], gbi_fmac(T(15777.695649238516), xs[43], gbi_fmac(T(20001.879911648302), xs[33], gbi_fmac(T(1924.681791881453), xs[23], gbi_fmac(T(1967.4145470642432), xs[15], gbi_fmac(T(301.1976095522672), xs[9], gbi_fmac(T(200.79840636817812), xs[3], T(70.99295739719538) * xs[2]))))))));
  y[58] = gbi_fmac(-282240.0f, xs[58], gbi_fmac(T(-25822.315930218192), xs[34], gbi_fmac(T(-2693.993318477238), xs[16], T(-317.49015732775086) * xs[4])));
  y[59] = gbi_fmac(T(-155552.39662570294), xs[67], gbi_fmac(225792.0f, xs[59], gbi_fmac(T(-15777.695649238516), xs[41], gbi_fmac(T(20001.879911648302), xs[35], gbi_fmac(T(-1924.681791881453), xs[21], gbi_fmac(T(1967.4145470642432), xs[17], gbi_fmac(T(-301.1976095522672), xs[7], gbi_fmac(T(200.79840636817812), xs[5], T(-70.99295739719538) * xs[0]))))))));
  y[60] = gbi_fmac(T(166292.5068185575), xs[66], gbi_fmac(-112896.0f, xs[60], gbi_fmac(T(15777.695649238518), xs[40], gbi_fmac(T(-8945.11263204662), xs[36], gbi_fmac(T(1721.4877286812125), xs[20], gbi_fmac(T(-695.586083817093), xs[18], T(212.9788721915862) * xs[6]))))));
  y[61] = gbi_fmac(-81648.0f, xs[65], gbi_fmac(T(32255.999999999996), xs[61], gbi_fmac(T(-6761.869563959364), xs[39], gbi_fmac(T(1951.983606488538), xs[37], T(-563.4891303299471) * xs[19]))));
  y[62] = gbi_fmac(18144.0f, xs[64], gbi_fmac(T(-4031.9999999999995), xs[62], T(1126.978260659894) * xs[38]));
  y[63] = gbi_fmac(e2, T(20618.18181818182) * xs[63], T(-7560.0) * xs[63]);
  y[64] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[64], T(-10245.256915089945) * xs[38]), gbi_fmac(T(40775.60768177688), xs[74], gbi_fmac(69552.0f, xs[64], gbi_fmac(18144.0f, xs[62], T(3380.934781979682) * xs[38]))));
  y[65] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[65], gbi_fmac(T(61471.54149053967), xs[39], T(3951.741952963265) * xs[19])), gbi_fmac(T(-244653.6460906613), xs[75], gbi_fmac(-291816.0f, xs[65], gbi_fmac(-81648.0f, xs[61], gbi_fmac(T(-12778.73233149517), xs[47], gbi_fmac(T(-19158.630431218196), xs[39], gbi_fmac(T(-5855.950819465615), xs[37], T(-1126.978260659894) * xs[19])))))));
  y[66] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[66], gbi_fmac(T(-187798.66131067774), xs[40], gbi_fmac(T(-15806.96781185306), xs[20], T(-1419.6244410825732) * xs[6]))), gbi_fmac(T(747429.2348382615), xs[76], gbi_fmac(737856.0f, xs[66], gbi_fmac(T(166292.5068185575), xs[60], gbi_fmac(T(51114.92932598069), xs[48], gbi_fmac(T(56071.31459133092), xs[40], gbi_fmac(T(15615.868851908304), xs[36], gbi_fmac(T(3299.4545003682047), xs[26], gbi_fmac(T(4507.913042639577), xs[20], gbi_fmac(T(1593.7879407248633), xs[18], T(325.330601081423) * xs[6]))))))))));
  y[67] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[67], gbi_fmac(T(351339.1241596774), xs[41], gbi_fmac(T(33062.645272220645), xs[21], gbi_fmac(T(3755.9732262135544), xs[7], T(553.3071121272332) * xs[0])))), gbi_fmac(T(-1398312.0588116883), xs[77], gbi_fmac(-1248912.0f, xs[67], gbi_fmac(T(-155552.39662570294), xs[59], gbi_fmac(T(-106914.54531540598), xs[49], gbi_fmac(T(-102139.30252356337), xs[41], gbi_fmac(T(-16331.46655998781), xs[35], gbi_fmac(T(-8729.536070147142), xs[27], gbi_fmac(T(-9428.976614670333), xs[21], gbi_fmac(T(-2108.3832668658706), xs[17], gbi_fmac(T(-673.4983296193094), xs[11], gbi_fmac(T(-983.7072735321215), xs[7], gbi_fmac(T(-368.8902275745455), xs[5], T(-86.94826047713663) * xs[0])))))))))))));
  y[68] = gbi_fmac(e2, gbi_fmac(T(-5195781.818181818), xs[68], gbi_fmac(T(-430300.7904337778), xs[42], gbi_fmac(T(-41821.305812166014), xs[22], gbi_fmac(T(-5039.166873289622), xs[8], T(-857.1796922427575) * xs[1])))), gbi_fmac(T(1712575.5226346292), xs[78], gbi_fmac(1481760.0f, xs[68], gbi_fmac(T(135237.3912791873), xs[50], gbi_fmac(T(123967.60867258835), xs[42], gbi_fmac(T(11711.901638931227), xs[28], gbi_fmac(T(11926.816842728827), xs[22], gbi_fmac(T(1043.3791257256396), xs[12], gbi_fmac(T(1374.772708486752), xs[8], T(224.49944320643647) * xs[1])))))))));
  y[69] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[69], gbi_fmac(T(351339.1241596774), xs[43], gbi_fmac(T(33062.645272220645), xs[23], gbi_fmac(T(3755.9732262135544), xs[9], T(553.3071121272332) * xs[2])))), gbi_fmac(T(-1398312.0588116883), xs[79], gbi_fmac(-1248912.0f, xs[69], gbi_fmac(T(155552.39662570294), xs[57], gbi_fmac(T(-106914.54531540598), xs[51], gbi_fmac(T(-102139.30252356337), xs[43], gbi_fmac(T(16331.46655998781), xs[33], gbi_fmac(T(-8729.536070147142), xs[29], gbi_fmac(T(-9428.976614670333), xs[23], gbi_fmac(T(2108.3832668658706), xs[15], gbi_fmac(T(-673.4983296193094), xs[13], gbi_fmac(T(-983.7072735321215), xs[9], gbi_fmac(T(368.8902275745455), xs[3], T(-86.94826047713663) * xs[2])))))))))))));
  y[70] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[70], gbi_fmac(T(-187798.66131067774), xs[44], gbi_fmac(T(-15806.96781185306), xs[24], T(-1419.6244410825732) * xs[10]))), gbi_fmac(T(747429.2348382615), xs[80], gbi_fmac(737856.0f, xs[70], gbi_fmac(T(-166292.5068185575), xs[56], gbi_fmac(T(51114.92932598069), xs[52], gbi_fmac(T(56071.31459133092), xs[44], gbi_fmac(T(-15615.868851908304), xs[32], gbi_fmac(T(3299.4545003682047), xs[30], gbi_fmac(T(4507.913042639577), xs[24], gbi_fmac(T(-1593.7879407248633), xs[14], T(325.330601081423) * xs[10]))))))))));
  y[71] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[71], gbi_fmac(T(61471.54149053967), xs[45], T(3951.741952963265) * xs[25])), gbi_fmac(T(-244653.6460906613), xs[81], gbi_fmac(-291816.0f, xs[71], gbi_fmac(81648.0f, xs[55], gbi_fmac(T(-12778.73233149517), xs[53], gbi_fmac(T(-19158.630431218196), xs[45], gbi_fmac(T(5855.950819465615), xs[31], T(-1126.978260659894) * xs[25])))))));
  y[72] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[72], T(-10245.256915089945) * xs[46]), gbi_fmac(T(40775.60768177688), xs[82], gbi_fmac(69552.0f, xs[72], gbi_fmac(-18144.0f, xs[54], T(3380.934781979682) * xs[46]))));
  y[73] = gbi_fmac(e2, T(20618.18181818182) * xs[73], T(-7560.0) * xs[73]);
  y[74] = gbi_fmac(T(-40775.60768177688), xs[64], T(-2026.1562355625713) * xs[38]);
  y[75] = gbi_fmac(T(244653.6460906613), xs[65], gbi_fmac(T(16209.24988450057), xs[39], T(1013.0781177812858) * xs[19]));
  y[76] = gbi_fmac(T(-747429.2348382615), xs[66], gbi_fmac(T(-56732.374595752), xs[40], gbi_fmac(T(-4642.50715963613), xs[20], T(-382.90753690438345) * xs[6])));
  y[77] = gbi_fmac(T(1398312.0588116883), xs[67], gbi_fmac(T(113464.749191504), xs[41], gbi_fmac(T(10380.961594975855), xs[21], gbi_fmac(T(1083.026063650111), xs[7], T(127.63584563479449) * xs[0]))));
  y[78] = gbi_fmac(T(-1712575.5226346292), xs[68], gbi_fmac(T(-141830.93648938002), xs[42], gbi_fmac(T(-13401.763791653422), xs[22], gbi_fmac(T(-1482.994513567979), xs[8], T(-201.8099916438052) * xs[1]))));
  y[79] = gbi_fmac(T(1398312.0588116883), xs[69], gbi_fmac(T(113464.749191504), xs[43], gbi_fmac(T(10380.961594975855), xs[23], gbi_fmac(T(1083.026063650111), xs[9], T(127.63584563479449) * xs[2]))));
  y[80] = gbi_fmac(T(-747429.2348382615), xs[70], gbi_fmac(T(-56732.374595752), xs[44], gbi_fmac(T(-4642.50715963613), xs[24], T(-382.90753690438345) * xs[10])));
  y[81] = gbi_fmac(T(244653.6460906613), xs[71], gbi_fmac(T(16209.24988450057), xs[45], T(1013.0781177812858) * xs[25]));
  y[82] = gbi_fmac(T(-40775.60768177688), xs[72], T(-2026.1562355625713) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_all_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
  y[31] = T(0);
  y[32] = T(0);
  y[33] = gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]);
  y[34] = T(46.475800154489) * xs[4];
  y[35] = gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]);
  y[36] = T(0);
  y[37] = T(0);
  y[38] = T(0);
  y[39] = T(0);
  y[40] = T(0);
  y[41] = gbi_fmac(e2, T(-70.55336829505575) * xs[0], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]));
  y[42] = gbi_fmac(e2, T(111.55467020454341) * xs[1], T(-35.85685828003181) * xs[1]);
  y[43] = gbi_fmac(e2, T(-70.55336829505575) * xs[2], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]));
  y[44] = T(0);
  y[45] = T(0);
  y[46] = T(0);
  y[47] = T(0);
  y[48] = T(0);
  y[49] = T(-17.5662013130736) * xs[0];
  y[50] = T(28.685486624025447) * xs[1];
  y[51] = T(-17.5662013130736) * xs[2];
  y[52] = T(0);
  y[53] = T(0);
  y[54] = T(0);
  y[55] = T(0);
  y[56] = T(0);
  y[57] = gbi_fmac(T(200.79840636817812), xs[3], T(70.99295739719538) * xs[2]);
  y[58] = T(-317.49015732775086) * xs[4];
  y[59] = gbi_fmac(T(200.79840636817812), xs[5], T(-70.99295739719538) * xs[0]);
  y[60] = T(0);
  y[61] = T(0);
  y[62] = T(0);
  y[63] = T(0);
  y[64] = T(0);
  y[65] = T(0);
  y[66] = T(0);
  y[67] = gbi_fmac(e2, T(553.3071121272332) * xs[0], gbi_fmac(T(-368.8902275745455), xs[5], T(-86.94826047713663) * xs[0]));
  y[68] = gbi_fmac(e2, T(-857.1796922427575) * xs[1], T(224.49944320643647) * xs[1]);
  y[69] = gbi_fmac(e2, T(553.3071121272332) * xs[2], gbi_fmac(T(368.8902275745455), xs[3], T(-86.94826047713663) * xs[2]));
  y[70] = T(0);
  y[71] = T(0);
  y[72] = T(0);
  y[73] = T(0);
  y[74] = T(0);
  y[75] = T(0);
  y[76] = T(0);
  y[77] = T(127.63584563479449) * xs[0];
  y[78] = T(-201.8099916438052) * xs[1];
  y[79] = T(127.63584563479449) * xs[2];
  y[80] = T(0);
  y[81] = T(0);
  y[82] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_all_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[67], gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7]))), gbi_fmac(T(-127.63584563479449), xs[77], gbi_fmac(T(-86.94826047713663), xs[67], gbi_fmac(T(-70.99295739719538), xs[59], gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11]))))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-857.1796922427575), xs[68], gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8]))), gbi_fmac(T(201.8099916438052), xs[78], gbi_fmac(T(224.49944320643647), xs[68], gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]))))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[69], gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9]))), gbi_fmac(T(-127.63584563479449), xs[79], gbi_fmac(T(-86.94826047713663), xs[69], gbi_fmac(T(70.99295739719538), xs[57], gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13]))))))))));
  y[3] = gbi_fmac(T(-368.8902275745455), xs[69], gbi_fmac(T(-200.79840636817812), xs[57], gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]))))));
  y[4] = gbi_fmac(T(317.49015732775086), xs[58], gbi_fmac(T(46.475800154489), xs[34], T(8.485281374238571) * xs[16]));
  y[5] = gbi_fmac(T(368.8902275745455), xs[67], gbi_fmac(T(-200.79840636817812), xs[59], gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]))))));
  y[6] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[66], gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]))), gbi_fmac(T(-382.90753690438345), xs[76], gbi_fmac(T(-325.330601081423), xs[66], gbi_fmac(T(-212.9788721915862), xs[60], gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[67], gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7]))), gbi_fmac(T(1083.026063650111), xs[77], gbi_fmac(T(983.7072735321215), xs[67], gbi_fmac(T(301.1976095522672), xs[59], gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7])))))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(5039.166873289622), xs[68], gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8]))), gbi_fmac(T(-1482.994513567979), xs[78], gbi_fmac(T(-1374.772708486752), xs[68], gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]))))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[69], gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9]))), gbi_fmac(T(1083.026063650111), xs[79], gbi_fmac(T(983.7072735321215), xs[69], gbi_fmac(T(-301.1976095522672), xs[57], gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9])))))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[70], gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]))), gbi_fmac(T(-382.90753690438345), xs[80], gbi_fmac(T(-325.330601081423), xs[70], gbi_fmac(T(212.9788721915862), xs[56], gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))))))));
  y[11] = gbi_fmac(T(-673.4983296193094), xs[67], gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7])));
  y[12] = gbi_fmac(T(1043.3791257256396), xs[68], gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8])));
  y[13] = gbi_fmac(T(-673.4983296193094), xs[69], gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9])));
  y[14] = gbi_fmac(T(-1593.7879407248633), xs[70], gbi_fmac(T(-695.586083817093), xs[56], gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))))));
  y[15] = gbi_fmac(T(2108.3832668658706), xs[69], gbi_fmac(T(1967.4145470642432), xs[57], gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]))))));
  y[16] = gbi_fmac(T(-2693.993318477238), xs[58], gbi_fmac(T(-328.63353450309967), xs[34], T(-48.0) * xs[16]));
  y[17] = gbi_fmac(T(-2108.3832668658706), xs[67], gbi_fmac(T(1967.4145470642432), xs[59], gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]))))));
  y[18] = gbi_fmac(T(1593.7879407248633), xs[66], gbi_fmac(T(-695.586083817093), xs[60], gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))))));
  y[19] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[65], gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19])), gbi_fmac(T(-1013.0781177812858), xs[75], gbi_fmac(T(-1126.978260659894), xs[65], gbi_fmac(T(-563.4891303299471), xs[61], gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])))))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[66], gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]))), gbi_fmac(T(4642.50715963613), xs[76], gbi_fmac(T(4507.913042639577), xs[66], gbi_fmac(T(1721.4877286812125), xs[60], gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[67], gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7]))), gbi_fmac(T(-10380.961594975855), xs[77], gbi_fmac(T(-9428.976614670333), xs[67], gbi_fmac(T(-1924.681791881453), xs[59], gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7])))))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-41821.305812166014), xs[68], gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8]))), gbi_fmac(T(13401.763791653422), xs[78], gbi_fmac(T(11926.816842728827), xs[68], gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8]))))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[69], gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9]))), gbi_fmac(T(-10380.961594975855), xs[79], gbi_fmac(T(-9428.976614670333), xs[69], gbi_fmac(T(1924.681791881453), xs[57], gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9])))))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[70], gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]))), gbi_fmac(T(4642.50715963613), xs[80], gbi_fmac(T(4507.913042639577), xs[70], gbi_fmac(T(-1721.4877286812125), xs[56], gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))))))));
  y[25] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[71], gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25])), gbi_fmac(T(-1013.0781177812858), xs[81], gbi_fmac(T(-1126.978260659894), xs[71], gbi_fmac(T(563.4891303299471), xs[55], gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])))))));
  y[26] = gbi_fmac(T(-3299.4545003682047), xs[66], gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6])));
  y[27] = gbi_fmac(T(8729.536070147142), xs[67], gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7])));
  y[28] = gbi_fmac(T(-11711.901638931227), xs[68], gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8])));
  y[29] = gbi_fmac(T(8729.536070147142), xs[69], gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9])));
  y[30] = gbi_fmac(T(-3299.4545003682047), xs[70], gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10])));
  y[31] = gbi_fmac(T(-5855.950819465615), xs[71], gbi_fmac(T(-1951.983606488538), xs[55], gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]))));
  y[32] = gbi_fmac(T(15615.868851908304), xs[70], gbi_fmac(T(8945.11263204662), xs[56], gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))))));
  y[33] = gbi_fmac(T(-16331.46655998781), xs[69], gbi_fmac(T(-20001.879911648302), xs[57], gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], T(-47.434164902525694) * xs[9]))))));
  y[34] = gbi_fmac(T(25822.315930218192), xs[58], gbi_fmac(2700.0f, xs[34], T(328.63353450309967) * xs[16]));
  y[35] = gbi_fmac(T(16331.46655998781), xs[67], gbi_fmac(T(-20001.879911648302), xs[59], gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], T(47.434164902525694) * xs[7]))))));
  y[36] = gbi_fmac(T(-15615.868851908304), xs[66], gbi_fmac(T(8945.11263204662), xs[60], gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))))));
  y[37] = gbi_fmac(T(5855.950819465615), xs[65], gbi_fmac(T(-1951.983606488538), xs[61], gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]))));
  y[38] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[64], T(560.0) * xs[38]), gbi_fmac(T(-2026.1562355625713), xs[74], gbi_fmac(T(-3380.934781979682), xs[64], gbi_fmac(T(-1126.978260659894), xs[62], T(-180.0) * xs[38]))));
  y[39] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[65], gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19])), gbi_fmac(T(16209.24988450057), xs[75], gbi_fmac(T(19158.630431218196), xs[65], gbi_fmac(T(6761.869563959364), xs[61], gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])))))));
  y[40] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[66], gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6]))), gbi_fmac(T(-56732.374595752), xs[76], gbi_fmac(T(-56071.31459133092), xs[66], gbi_fmac(T(-15777.695649238518), xs[60], gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))))))));
  y[41] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[67], gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], T(-419.06562731868144) * xs[7]))), gbi_fmac(T(113464.749191504), xs[77], gbi_fmac(T(102139.30252356337), xs[67], gbi_fmac(T(15777.695649238516), xs[59], gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], T(120.26755886059097) * xs[7])))))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(T(430300.7904337778), xs[68], gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], T(573.8292428937376) * xs[8]))), gbi_fmac(T(-141830.93648938002), xs[78], gbi_fmac(T(-123967.60867258835), xs[68], gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], T(-175.662013130736) * xs[8]))))))));
  y[43] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[69], gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], T(-419.06562731868144) * xs[9]))), gbi_fmac(T(113464.749191504), xs[79], gbi_fmac(T(102139.30252356337), xs[69], gbi_fmac(T(-15777.695649238516), xs[57], gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], T(120.26755886059097) * xs[9])))))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[70], gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10]))), gbi_fmac(T(-56732.374595752), xs[80], gbi_fmac(T(-56071.31459133092), xs[70], gbi_fmac(T(15777.695649238518), xs[56], gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))))))));
  y[45] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[71], gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25])), gbi_fmac(T(16209.24988450057), xs[81], gbi_fmac(T(19158.630431218196), xs[71], gbi_fmac(T(-6761.869563959364), xs[55], gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])))))));
  y[46] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[72], T(560.0) * xs[46]), gbi_fmac(T(-2026.1562355625713), xs[82], gbi_fmac(T(-3380.934781979682), xs[72], gbi_fmac(T(1126.978260659894), xs[54], T(-180.0) * xs[46]))));
  y[47] = gbi_fmac(T(-12778.73233149517), xs[65], gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]));
  y[48] = gbi_fmac(T(51114.92932598069), xs[66], gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6])));
  y[49] = gbi_fmac(T(-106914.54531540598), xs[67], gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], T(-124.21180068162376) * xs[7])));
  y[50] = gbi_fmac(T(135237.3912791873), xs[68], gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], T(175.66201313073597) * xs[8])));
  y[51] = gbi_fmac(T(-106914.54531540598), xs[69], gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], T(-124.21180068162376) * xs[9])));
  y[52] = gbi_fmac(T(51114.92932598069), xs[70], gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10])));
  y[53] = gbi_fmac(T(-12778.73233149517), xs[71], gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]));
  y[54] = gbi_fmac(-18144.0f, xs[72], gbi_fmac(T(-4031.9999999999995), xs[54], T(-1126.978260659894) * xs[46]));
  y[55] = gbi_fmac(81648.0f, xs[71], gbi_fmac(T(32255.999999999996), xs[55], gbi_fmac(T(6761.869563959364), xs[45], gbi_fmac(T(1951.983606488538), xs[31], T(563.4891303299471) * xs[25]))));
  y[56] = gbi_fmac(T(-166292.5068185575), xs[70], gbi_fmac(-112896.0f, xs[56], gbi_fmac(T(-15777.695649238518), xs[44], gbi_fmac(T(-8945.11263204662), xs[32], gbi_fmac(T(-1721.4877286812125), xs[24], gbi_fmac(T(-695.586083817093), xs[14], T(-212.9788721915862) * xs[10]))))));
  y[57] = gbi_fmac(T(155552.39662570294), xs[69], gbi_fmac(225792.0f, xs[57], gbi_fmac(T(15777.695649238516), xs[43], gbi_fmac(T(20001.879911648302), xs[33], gbi_fmac(T(1924.681791881453), xs[23], gbi_fmac(T(1967.4145470642432), xs[15], T(301.1976095522672) * xs[9]))))));
  y[58] = gbi_fmac(-282240.0f, xs[58], gbi_fmac(T(-25822.315930218192), xs[34], T(-2693.993318477238) * xs[16]));
  y[59] = gbi_fmac(T(-155552.39662570294), xs[67], gbi_fmac(225792.0f, xs[59], gbi_fmac(T(-15777.695649238516), xs[41], gbi_fmac(T(20001.879911648302), xs[35], gbi_fmac(T(-1924.681791881453), xs[21], gbi_fmac(T(1967.4145470642432), xs[17], T(-301.1976095522672) * xs[7]))))));
  y[60] = gbi_fmac(T(166292.5068185575), xs[66], gbi_fmac(-112896.0f, xs[60], gbi_fmac(T(15777.695649238518), xs[40], gbi_fmac(T(-8945.11263204662), xs[36], gbi_fmac(T(1721.4877286812125), xs[20], gbi_fmac(T(-695.586083817093), xs[18], T(212.9788721915862) * xs[6]))))));
  y[61] = gbi_fmac(-81648.0f, xs[65], gbi_fmac(T(32255.999999999996), xs[61], gbi_fmac(T(-6761.869563959364), xs[39], gbi_fmac(T(1951.983606488538), xs[37], T(-563.4891303299471) * xs[19]))));
  y[62] = gbi_fmac(18144.0f, xs[64], gbi_fmac(T(-4031.9999999999995), xs[62], T(1126.978260659894) * xs[38]));
  y[63] = gbi_fmac(e2, T(20618.18181818182) * xs[63], T(-7560.0) * xs[63]);
  y[64] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[64], T(-10245.256915089945) * xs[38]), gbi_fmac(T(40775.60768177688), xs[74], gbi_fmac(69552.0f, xs[64], gbi_fmac(18144.0f, xs[62], T(3380.934781979682) * xs[38]))));
  y[65] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[65], gbi_fmac(T(61471.54149053967), xs[39], T(3951.741952963265) * xs[19])), gbi_fmac(T(-244653.6460906613), xs[75], gbi_fmac(-291816.0f, xs[65], gbi_fmac(-81648.0f, xs[61], gbi_fmac(T(-12778.73233149517), xs[47], gbi_fmac(T(-19158.630431218196), xs[39], gbi_fmac(T(-5855.950819465615), xs[37], T(-1126.978260659894) * xs[19])))))));
  y[66] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[66], gbi_fmac(T(-187798.66131067774), xs[40], gbi_fmac(T(-15806.96781185306), xs[20], T(-1419.6244410825732) * xs[6]))), gbi_fmac(T(747429.2348382615), xs[76], gbi_fmac(737856.0f, xs[66], gbi_fmac(T(166292.5068185575), xs[60], gbi_fmac(T(51114.92932598069), xs[48], gbi_fmac(T(56071.31459133092), xs[40], gbi_fmac(T(15615.868851908304), xs[36], gbi_fmac(T(3299.4545003682047), xs[26], gbi_fmac(T(4507.913042639577), xs[20], gbi_fmac(T(1593.7879407248633), xs[18], T(325.330601081423) * xs[6]))))))))));
  y[67] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[67], gbi_fmac(T(351339.1241596774), xs[41], gbi_fmac(T(33062.645272220645), xs[21], T(3755.9732262135544) * xs[7]))), gbi_fmac(T(-1398312.0588116883), xs[77], gbi_fmac(-1248912.0f, xs[67], gbi_fmac(T(-155552.39662570294), xs[59], gbi_fmac(T(-106914.54531540598), xs[49], gbi_fmac(T(-102139.30252356337), xs[41], gbi_fmac(T(-16331.46655998781), xs[35], gbi_fmac(T(-8729.536070147142), xs[27], gbi_fmac(T(-9428.976614670333), xs[21], gbi_fmac(T(-2108.3832668658706), xs[17], gbi_fmac(T(-673.4983296193094), xs[11], T(-983.7072735321215) * xs[7])))))))))));
  y[68] = gbi_fmac(e2, gbi_fmac(T(-5195781.818181818), xs[68], gbi_fmac(T(-430300.7904337778), xs[42], gbi_fmac(T(-41821.305812166014), xs[22], T(-5039.166873289622) * xs[8]))), gbi_fmac(T(1712575.5226346292), xs[78], gbi_fmac(1481760.0f, xs[68], gbi_fmac(T(135237.3912791873), xs[50], gbi_fmac(T(123967.60867258835), xs[42], gbi_fmac(T(11711.901638931227), xs[28], gbi_fmac(T(11926.816842728827), xs[22], gbi_fmac(T(1043.3791257256396), xs[12], T(1374.772708486752) * xs[8]))))))));
  y[69] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[69], gbi_fmac(T(351339.1241596774), xs[43], gbi_fmac(T(33062.645272220645), xs[23], T(3755.9732262135544) * xs[9]))), gbi_fmac(T(-1398312.0588116883), xs[79], gbi_fmac(-1248912.0f, xs[69], gbi_fmac(T(155552.39662570294), xs[57], gbi_fmac(T(-106914.54531540598), xs[51], gbi_fmac(T(-102139.30252356337), xs[43], gbi_fmac(T(16331.46655998781), xs[33], gbi_fmac(T(-8729.536070147142), xs[29], gbi_fmac(T(-9428.976614670333), xs[23], gbi_fmac(T(2108.3832668658706), xs[15], gbi_fmac(T(-673.4983296193094), xs[13], T(-983.7072735321215) * xs[9])))))))))));
  y[70] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[70], gbi_fmac(T(-187798.66131067774), xs[44], gbi_fmac(T(-15806.96781185306), xs[24], T(-1419.6244410825732) * xs[10]))), gbi_fmac(T(747429.2348382615), xs[80], gbi_fmac(737856.0f, xs[70], gbi_fmac(T(-166292.5068185575), xs[56], gbi_fmac(T(51114.92932598069), xs[52], gbi_fmac(T(56071.31459133092), xs[44], gbi_fmac(T(-15615.868851908304), xs[32], gbi_fmac(T(3299.4545003682047), xs[30], gbi_fmac(T(4507.913042639577), xs[24], gbi_fmac(T(-1593.7879407248633), xs[14], T(325.330601081423) * xs[10]))))))))));
  y[71] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[71], gbi_fmac(T(61471.54149053967), xs[45], T(3951.741952963265) * xs[25])), gbi_fmac(T(-244653.6460906613), xs[81], gbi_fmac(-291816.0f, xs[71], gbi_fmac(81648.0f, xs[55], gbi_fmac(T(-12778.73233149517), xs[53], gbi_fmac(T(-19158.630431218196), xs[45], gbi_fmac(T(5855.950819465615), xs[31], T(-1126.978260659894) * xs[25])))))));
  y[72] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[72], T(-10245.256915089945) * xs[46]), gbi_fmac(T(40775.60768177688), xs[82], gbi_fmac(69552.0f, xs[72], gbi_fmac(-18144.0f, xs[54], T(3380.934781979682) * xs[46]))));
  y[73] = gbi_fmac(e2, T(20618.18181818182) * xs[73], T(-7560.0) * xs[73]);
  y[74] = gbi_fmac(T(-40775.60768177688), xs[64], T(-2026.1562355625713) * xs[38]);
  y[75] = gbi_fmac(T(244653.6460906613), xs[65], gbi_fmac(T(16209.24988450057), xs[39], T(1013.0781177812858) * xs[19]));
  y[76] = gbi_fmac(T(-747429.2348382615), xs[66], gbi_fmac(T(-56732.374595752), xs[40], gbi_fmac(T(-4642.50715963613), xs[20], T(-382.90753690438345) * xs[6])));
  y[77] = gbi_fmac(T(1398312.0588116883), xs[67], gbi_fmac(T(113464.749191504), xs[41], gbi_fmac(T(10380.961594975855), xs[21], T(1083.026063650111) * xs[7])));
  y[78] = gbi_fmac(T(-1712575.5226346292), xs[68], gbi_fmac(T(-141830.93648938002), xs[42], gbi_fmac(T(-13401.763791653422), xs[22], T(-1482.994513567979) * xs[8])));
  y[79] = gbi_fmac(T(1398312.0588116883), xs[69], gbi_fmac(T(113464.749191504), xs[43], gbi_fmac(T(10380.961594975855), xs[23], T(1083.026063650111) * xs[9])));
  y[80] = gbi_fmac(T(-747429.2348382615), xs[70], gbi_fmac(T(-56732.374595752), xs[44], gbi_fmac(T(-4642.50715963613), xs[24], T(-382.90753690438345) * xs[10])));
  y[81] = gbi_fmac(T(244653.6460906613), xs[71], gbi_fmac(T(16209.24988450057), xs[45], T(1013.0781177812858) * xs[25]));
  y[82] = gbi_fmac(T(-40775.60768177688), xs[72], T(-2026.1562355625713) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_L_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[67], gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0])))), gbi_fmac(T(-127.63584563479449), xs[77], gbi_fmac(T(-86.94826047713663), xs[67], gbi_fmac(T(-70.99295739719538), xs[59], gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-857.1796922427575), xs[68], gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1])))), gbi_fmac(T(201.8099916438052), xs[78], gbi_fmac(T(224.49944320643647), xs[68], gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[69], gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2])))), gbi_fmac(T(-127.63584563479449), xs[79], gbi_fmac(T(-86.94826047713663), xs[69], gbi_fmac(T(70.99295739719538), xs[57], gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))))))))));
  y[3] = gbi_fmac(T(-368.8902275745455), xs[69], gbi_fmac(T(-200.79840636817812), xs[57], gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))))))));
  y[4] = gbi_fmac(T(317.49015732775086), xs[58], gbi_fmac(T(46.475800154489), xs[34], gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4])));
  y[5] = gbi_fmac(T(368.8902275745455), xs[67], gbi_fmac(T(-200.79840636817812), xs[59], gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))))))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_L_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_L_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[67], gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7]))), gbi_fmac(T(-127.63584563479449), xs[77], gbi_fmac(T(-86.94826047713663), xs[67], gbi_fmac(T(-70.99295739719538), xs[59], gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11]))))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-857.1796922427575), xs[68], gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8]))), gbi_fmac(T(201.8099916438052), xs[78], gbi_fmac(T(224.49944320643647), xs[68], gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8]))))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(553.3071121272332), xs[69], gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9]))), gbi_fmac(T(-127.63584563479449), xs[79], gbi_fmac(T(-86.94826047713663), xs[69], gbi_fmac(T(70.99295739719538), xs[57], gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13]))))))))));
  y[3] = gbi_fmac(T(-368.8902275745455), xs[69], gbi_fmac(T(-200.79840636817812), xs[57], gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]))))));
  y[4] = gbi_fmac(T(317.49015732775086), xs[58], gbi_fmac(T(46.475800154489), xs[34], T(8.485281374238571) * xs[16]));
  y[5] = gbi_fmac(T(368.8902275745455), xs[67], gbi_fmac(T(-200.79840636817812), xs[59], gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]))))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_H_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[66], gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]))), gbi_fmac(T(-382.90753690438345), xs[76], gbi_fmac(T(-325.330601081423), xs[66], gbi_fmac(T(-212.9788721915862), xs[60], gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[67], gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0])))), gbi_fmac(T(1083.026063650111), xs[77], gbi_fmac(T(983.7072735321215), xs[67], gbi_fmac(T(301.1976095522672), xs[59], gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5]))))))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(5039.166873289622), xs[68], gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1])))), gbi_fmac(T(-1482.994513567979), xs[78], gbi_fmac(T(-1374.772708486752), xs[68], gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1])))))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[69], gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2])))), gbi_fmac(T(1083.026063650111), xs[79], gbi_fmac(T(983.7072735321215), xs[69], gbi_fmac(T(-301.1976095522672), xs[57], gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3]))))))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[70], gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]))), gbi_fmac(T(-382.90753690438345), xs[80], gbi_fmac(T(-325.330601081423), xs[70], gbi_fmac(T(212.9788721915862), xs[56], gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))))))));
  y[11] = gbi_fmac(T(-673.4983296193094), xs[67], gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0]))));
  y[12] = gbi_fmac(T(1043.3791257256396), xs[68], gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1]))));
  y[13] = gbi_fmac(T(-673.4983296193094), xs[69], gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2]))));
  y[14] = gbi_fmac(T(-1593.7879407248633), xs[70], gbi_fmac(T(-695.586083817093), xs[56], gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))))));
  y[15] = gbi_fmac(T(2108.3832668658706), xs[69], gbi_fmac(T(1967.4145470642432), xs[57], gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))))))));
  y[16] = gbi_fmac(T(-2693.993318477238), xs[58], gbi_fmac(T(-328.63353450309967), xs[34], gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4])));
  y[17] = gbi_fmac(T(-2108.3832668658706), xs[67], gbi_fmac(T(1967.4145470642432), xs[59], gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))))))));
  y[18] = gbi_fmac(T(1593.7879407248633), xs[66], gbi_fmac(T(-695.586083817093), xs[60], gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))))));
  y[19] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[65], gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19])), gbi_fmac(T(-1013.0781177812858), xs[75], gbi_fmac(T(-1126.978260659894), xs[65], gbi_fmac(T(-563.4891303299471), xs[61], gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])))))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[66], gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]))), gbi_fmac(T(4642.50715963613), xs[76], gbi_fmac(T(4507.913042639577), xs[66], gbi_fmac(T(1721.4877286812125), xs[60], gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[67], gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0])))), gbi_fmac(T(-10380.961594975855), xs[77], gbi_fmac(T(-9428.976614670333), xs[67], gbi_fmac(T(-1924.681791881453), xs[59], gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0])))))))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-41821.305812166014), xs[68], gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1])))), gbi_fmac(T(13401.763791653422), xs[78], gbi_fmac(T(11926.816842728827), xs[68], gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1])))))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[69], gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2])))), gbi_fmac(T(-10380.961594975855), xs[79], gbi_fmac(T(-9428.976614670333), xs[69], gbi_fmac(T(1924.681791881453), xs[57], gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2])))))))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[70], gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]))), gbi_fmac(T(4642.50715963613), xs[80], gbi_fmac(T(4507.913042639577), xs[70], gbi_fmac(T(-1721.4877286812125), xs[56], gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))))))));
  y[25] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[71], gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25])), gbi_fmac(T(-1013.0781177812858), xs[81], gbi_fmac(T(-1126.978260659894), xs[71], gbi_fmac(T(563.4891303299471), xs[55], gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])))))));
  y[26] = gbi_fmac(T(-3299.4545003682047), xs[66], gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6])));
  y[27] = gbi_fmac(T(8729.536070147142), xs[67], gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0]))));
  y[28] = gbi_fmac(T(-11711.901638931227), xs[68], gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1]))));
  y[29] = gbi_fmac(T(8729.536070147142), xs[69], gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2]))));
  y[30] = gbi_fmac(T(-3299.4545003682047), xs[70], gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10])));
  y[31] = gbi_fmac(T(-5855.950819465615), xs[71], gbi_fmac(T(-1951.983606488538), xs[55], gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]))));
  y[32] = gbi_fmac(T(15615.868851908304), xs[70], gbi_fmac(T(8945.11263204662), xs[56], gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))))));
  y[33] = gbi_fmac(T(-16331.46655998781), xs[69], gbi_fmac(T(-20001.879911648302), xs[57], gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], gbi_fmac(T(-47.434164902525694), xs[9], gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]))))))));
  y[34] = gbi_fmac(T(25822.315930218192), xs[58], gbi_fmac(2700.0f, xs[34], gbi_fmac(T(328.63353450309967), xs[16], T(46.475800154489) * xs[4])));
  y[35] = gbi_fmac(T(16331.46655998781), xs[67], gbi_fmac(T(-20001.879911648302), xs[59], gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], gbi_fmac(T(47.434164902525694), xs[7], gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]))))))));
  y[36] = gbi_fmac(T(-15615.868851908304), xs[66], gbi_fmac(T(8945.11263204662), xs[60], gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))))));
  y[37] = gbi_fmac(T(5855.950819465615), xs[65], gbi_fmac(T(-1951.983606488538), xs[61], gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]))));
  y[38] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[64], T(560.0) * xs[38]), gbi_fmac(T(-2026.1562355625713), xs[74], gbi_fmac(T(-3380.934781979682), xs[64], gbi_fmac(T(-1126.978260659894), xs[62], T(-180.0) * xs[38]))));
  y[39] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[65], gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19])), gbi_fmac(T(16209.24988450057), xs[75], gbi_fmac(T(19158.630431218196), xs[65], gbi_fmac(T(6761.869563959364), xs[61], gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])))))));
  y[40] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[66], gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6]))), gbi_fmac(T(-56732.374595752), xs[76], gbi_fmac(T(-56071.31459133092), xs[66], gbi_fmac(T(-15777.695649238518), xs[60], gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))))))));
  y[41] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[67], gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], gbi_fmac(T(-419.06562731868144), xs[7], T(-70.55336829505575) * xs[0])))), gbi_fmac(T(113464.749191504), xs[77], gbi_fmac(T(102139.30252356337), xs[67], gbi_fmac(T(15777.695649238516), xs[59], gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], gbi_fmac(T(120.26755886059097), xs[7], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0])))))))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(T(430300.7904337778), xs[68], gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], gbi_fmac(T(573.8292428937376), xs[8], T(111.55467020454341) * xs[1])))), gbi_fmac(T(-141830.93648938002), xs[78], gbi_fmac(T(-123967.60867258835), xs[68], gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], gbi_fmac(T(-175.662013130736), xs[8], T(-35.85685828003181) * xs[1])))))))));
  y[43] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[69], gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], gbi_fmac(T(-419.06562731868144), xs[9], T(-70.55336829505575) * xs[2])))), gbi_fmac(T(113464.749191504), xs[79], gbi_fmac(T(102139.30252356337), xs[69], gbi_fmac(T(-15777.695649238516), xs[57], gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], gbi_fmac(T(120.26755886059097), xs[9], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2])))))))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[70], gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10]))), gbi_fmac(T(-56732.374595752), xs[80], gbi_fmac(T(-56071.31459133092), xs[70], gbi_fmac(T(15777.695649238518), xs[56], gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))))))));
  y[45] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[71], gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25])), gbi_fmac(T(16209.24988450057), xs[81], gbi_fmac(T(19158.630431218196), xs[71], gbi_fmac(T(-6761.869563959364), xs[55], gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])))))));
  y[46] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[72], T(560.0) * xs[46]), gbi_fmac(T(-2026.1562355625713), xs[82], gbi_fmac(T(-3380.934781979682), xs[72], gbi_fmac(T(1126.978260659894), xs[54], T(-180.0) * xs[46]))));
  y[47] = gbi_fmac(T(-12778.73233149517), xs[65], gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]));
  y[48] = gbi_fmac(T(51114.92932598069), xs[66], gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6])));
  y[49] = gbi_fmac(T(-106914.54531540598), xs[67], gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], gbi_fmac(T(-124.21180068162376), xs[7], T(-17.5662013130736) * xs[0]))));
  y[50] = gbi_fmac(T(135237.3912791873), xs[68], gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], gbi_fmac(T(175.66201313073597), xs[8], T(28.685486624025447) * xs[1]))));
  y[51] = gbi_fmac(T(-106914.54531540598), xs[69], gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], gbi_fmac(T(-124.21180068162376), xs[9], T(-17.5662013130736) * xs[2]))));
  y[52] = gbi_fmac(T(51114.92932598069), xs[70], gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10])));
  y[53] = gbi_fmac(T(-12778.73233149517), xs[71], gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]));
  y[54] = gbi_fmac(-18144.0f, xs[72], gbi_fmac(T(-4031.9999999999995), xs[54], T(-1126.978260659894) * xs[46]));
  y[55] = gbi_fmac(81648.0f, xs[71], gbi_fmac(T(32255.999999999996), xs[55], gbi_fmac(T(6761.869563959364), xs[45], gbi_fmac(T(1951.983606488538), xs[31], T(563.4891303299471) * xs[25]))));
  y[56] = gbi_fmac(T(-166292.5068185575), xs[70], gbi_fmac(-112896.0f, xs[56], gbi_fmac(T(-15777.695649238518), xs[44], gbi_fmac(T(-8945.11263204662), xs[32], gbi_fmac(T(-1721.4877286812125), xs[24], gbi_fmac(T(-695.586083817093), xs[14], T(-212.9788721915862) * xs[10]))))));
  y[57] = gbi_fmac(T(155552.39662570294), xs[69], gbi_fmac(225792.0f, xs[57], gbi_fmac(T(15777.695649238516), xs[43], gbi_fmac(T(20001.879911648302), xs[33], gbi_fmac(T(1924.681791881453), xs[23], gbi_fmac(T(1967.4145470642432), xs[15], gbi_fmac(T(301.1976095522672), xs[9], gbi_fmac(T(200.79840636817812), xs[3], T(70.99295739719538) * xs[2]))))))));
  y[58] = gbi_fmac(-282240.0f, xs[58], gbi_fmac(T(-25822.315930218192), xs[34], gbi_fmac(T(-2693.993318477238), xs[16], T(-317.49015732775086) * xs[4])));
  y[59] = gbi_fmac(T(-155552.39662570294), xs[67], gbi_fmac(225792.0f, xs[59], gbi_fmac(T(-15777.695649238516), xs[41], gbi_fmac(T(20001.879911648302), xs[35], gbi_fmac(T(-1924.681791881453), xs[21], gbi_fmac(T(1967.4145470642432), xs[17], gbi_fmac(T(-301.1976095522672), xs[7], gbi_fmac(T(200.79840636817812), xs[5], T(-70.99295739719538) * xs[0]))))))));
  y[60] = gbi_fmac(T(166292.5068185575), xs[66], gbi_fmac(-112896.0f, xs[60], gbi_fmac(T(15777.695649238518), xs[40], gbi_fmac(T(-8945.11263204662), xs[36], gbi_fmac(T(1721.4877286812125), xs[20], gbi_fmac(T(-695.586083817093), xs[18], T(212.9788721915862) * xs[6]))))));
  y[61] = gbi_fmac(-81648.0f, xs[65], gbi_fmac(T(32255.999999999996), xs[61], gbi_fmac(T(-6761.869563959364), xs[39], gbi_fmac(T(1951.983606488538), xs[37], T(-563.4891303299471) * xs[19]))));
  y[62] = gbi_fmac(18144.0f, xs[64], gbi_fmac(T(-4031.9999999999995), xs[62], T(1126.978260659894) * xs[38]));
  y[63] = gbi_fmac(e2, T(20618.18181818182) * xs[63], T(-7560.0) * xs[63]);
  y[64] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[64], T(-10245.256915089945) * xs[38]), gbi_fmac(T(40775.60768177688), xs[74], gbi_fmac(69552.0f, xs[64], gbi_fmac(18144.0f, xs[62], T(3380.934781979682) * xs[38]))));
  y[65] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[65], gbi_fmac(T(61471.54149053967), xs[39], T(3951.741952963265) * xs[19])), gbi_fmac(T(-244653.6460906613), xs[75], gbi_fmac(-291816.0f, xs[65], gbi_fmac(-81648.0f, xs[61], gbi_fmac(T(-12778.73233149517), xs[47], gbi_fmac(T(-19158.630431218196), xs[39], gbi_fmac(T(-5855.950819465615), xs[37], T(-1126.978260659894) * xs[19])))))));
  y[66] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[66], gbi_fmac(T(-187798.66131067774), xs[40], gbi_fmac(T(-15806.96781185306), xs[20], T(-1419.6244410825732) * xs[6]))), gbi_fmac(T(747429.2348382615), xs[76], gbi_fmac(737856.0f, xs[66], gbi_fmac(T(166292.5068185575), xs[60], gbi_fmac(T(51114.92932598069), xs[48], gbi_fmac(T(56071.31459133092), xs[40], gbi_fmac(T(15615.868851908304), xs[36], gbi_fmac(T(3299.4545003682047), xs[26], gbi_fmac(T(4507.913042639577), xs[20], gbi_fmac(T(1593.7879407248633), xs[18], T(325.330601081423) * xs[6]))))))))));
  y[67] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[67], gbi_fmac(T(351339.1241596774), xs[41], gbi_fmac(T(33062.645272220645), xs[21], gbi_fmac(T(3755.9732262135544), xs[7], T(553.3071121272332) * xs[0])))), gbi_fmac(T(-1398312.0588116883), xs[77], gbi_fmac(-1248912.0f, xs[67], gbi_fmac(T(-155552.39662570294), xs[59], gbi_fmac(T(-106914.54531540598), xs[49], gbi_fmac(T(-102139.30252356337), xs[41], gbi_fmac(T(-16331.46655998781), xs[35], gbi_fmac(T(-8729.536070147142), xs[27], gbi_fmac(T(-9428.976614670333), xs[21], gbi_fmac(T(-2108.3832668658706), xs[17], gbi_fmac(T(-673.4983296193094), xs[11], gbi_fmac(T(-983.7072735321215), xs[7], gbi_fmac(T(-368.8902275745455), xs[5], T(-86.94826047713663) * xs[0])))))))))))));
  y[68] = gbi_fmac(e2, gbi_fmac(T(-5195781.818181818), xs[68], gbi_fmac(T(-430300.7904337778), xs[42], gbi_fmac(T(-41821.305812166014), xs[22], gbi_fmac(T(-5039.166873289622), xs[8], T(-857.1796922427575) * xs[1])))), gbi_fmac(T(1712575.5226346292), xs[78], gbi_fmac(1481760.0f, xs[68], gbi_fmac(T(135237.3912791873), xs[50], gbi_fmac(T(123967.60867258835), xs[42], gbi_fmac(T(11711.901638931227), xs[28], gbi_fmac(T(11926.816842728827), xs[22], gbi_fmac(T(1043.3791257256396), xs[12], gbi_fmac(T(1374.772708486752), xs[8], T(224.49944320643647) * xs[1])))))))));
  y[69] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[69], gbi_fmac(T(351339.1241596774), xs[43], gbi_fmac(T(33062.645272220645), xs[23], gbi_fmac(T(3755.9732262135544), xs[9], T(553.3071121272332) * xs[2])))), gbi_fmac(T(-1398312.0588116883), xs[79], gbi_fmac(-1248912.0f, xs[69], gbi_fmac(T(155552.39662570294), xs[57], gbi_fmac(T(-106914.54531540598), xs[51], gbi_fmac(T(-102139.30252356337), xs[43], gbi_fmac(T(16331.46655998781), xs[33], gbi_fmac(T(-8729.536070147142), xs[29], gbi_fmac(T(-9428.976614670333), xs[23], gbi_fmac(T(2108.3832668658706), xs[15], gbi_fmac(T(-673.4983296193094), xs[13], gbi_fmac(T(-983.7072735321215), xs[9], gbi_fmac(T(368.8902275745455), xs[3], T(-86.94826047713663) * xs[2])))))))))))));
  y[70] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[70], gbi_fmac(T(-187798.66131067774), xs[44], gbi_fmac(T(-15806.96781185306), xs[24], T(-1419.6244410825732) * xs[10]))), gbi_fmac(T(747429.2348382615), xs[80], gbi_fmac(737856.0f, xs[70], gbi_fmac(T(-166292.5068185575), xs[56], gbi_fmac(T(51114.92932598069), xs[52], gbi_fmac(T(56071.31459133092), xs[44], gbi_fmac(T(-15615.868851908304), xs[32], gbi_fmac(T(3299.4545003682047), xs[30], gbi_fmac(T(4507.913042639577), xs[24], gbi_fmac(T(-1593.7879407248633), xs[14], T(325.330601081423) * xs[10]))))))))));
  y[71] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[71], gbi_fmac(T(61471.54149053967), xs[45], T(3951.741952963265) * xs[25])), gbi_fmac(T(-244653.6460906613), xs[81], gbi_fmac(-291816.0f, xs[71], gbi_fmac(81648.0f, xs[55], gbi_fmac(T(-12778.73233149517), xs[53], gbi_fmac(T(-19158.630431218196), xs[45], gbi_fmac(T(5855.950819465615), xs[31], T(-1126.978260659894) * xs[25])))))));
  y[72] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[72], T(-10245.256915089945) * xs[46]), gbi_fmac(T(40775.60768177688), xs[82], gbi_fmac(69552.0f, xs[72], gbi_fmac(-18144.0f, xs[54], T(3380.934781979682) * xs[46]))));
  y[73] = gbi_fmac(e2, T(20618.18181818182) * xs[73], T(-7560.0) * xs[73]);
  y[74] = gbi_fmac(T(-40775.60768177688), xs[64], T(-2026.1562355625713) * xs[38]);
  y[75] = gbi_fmac(T(244653.6460906613), xs[65], gbi_fmac(T(16209.24988450057), xs[39], T(1013.0781177812858) * xs[19]));
  y[76] = gbi_fmac(T(-747429.2348382615), xs[66], gbi_fmac(T(-56732.374595752), xs[40], gbi_fmac(T(-4642.50715963613), xs[20], T(-382.90753690438345) * xs[6])));
  y[77] = gbi_fmac(T(1398312.0588116883), xs[67], gbi_fmac(T(113464.749191504), xs[41], gbi_fmac(T(10380.961594975855), xs[21], gbi_fmac(T(1083.026063650111), xs[7], T(127.63584563479449) * xs[0]))));
  y[78] = gbi_fmac(T(-1712575.5226346292), xs[68], gbi_fmac(T(-141830.93648938002), xs[42], gbi_fmac(T(-13401.763791653422), xs[22], gbi_fmac(T(-1482.994513567979), xs[8], T(-201.8099916438052) * xs[1]))));
  y[79] = gbi_fmac(T(1398312.0588116883), xs[69], gbi_fmac(T(113464.749191504), xs[43], gbi_fmac(T(10380.961594975855), xs[23], gbi_fmac(T(1083.026063650111), xs[9], T(127.63584563479449) * xs[2]))));
  y[80] = gbi_fmac(T(-747429.2348382615), xs[70], gbi_fmac(T(-56732.374595752), xs[44], gbi_fmac(T(-4642.50715963613), xs[24], T(-382.90753690438345) * xs[10])));
  y[81] = gbi_fmac(T(244653.6460906613), xs[71], gbi_fmac(T(16209.24988450057), xs[45], T(1013.0781177812858) * xs[25]));
  y[82] = gbi_fmac(T(-40775.60768177688), xs[72], T(-2026.1562355625713) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_H_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
  y[31] = T(0);
  y[32] = T(0);
  y[33] = gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]);
  y[34] = T(46.475800154489) * xs[4];
  y[35] = gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]);
  y[36] = T(0);
  y[37] = T(0);
  y[38] = T(0);
  y[39] = T(0);
  y[40] = T(0);
  y[41] = gbi_fmac(e2, T(-70.55336829505575) * xs[0], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]));
  y[42] = gbi_fmac(e2, T(111.55467020454341) * xs[1], T(-35.85685828003181) * xs[1]);
  y[43] = gbi_fmac(e2, T(-70.55336829505575) * xs[2], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]));
  y[44] = T(0);
  y[45] = T(0);
  y[46] = T(0);
  y[47] = T(0);
  y[48] = T(0);
  y[49] = T(-17.5662013130736) * xs[0];
  y[50] = T(28.685486624025447) * xs[1];
  y[51] = T(-17.5662013130736) * xs[2];
  y[52] = T(0);
  y[53] = T(0);
  y[54] = T(0);
  y[55] = T(0);
  y[56] = T(0);
  y[57] = gbi_fmac(T(200.79840636817812), xs[3], T(70.99295739719538) * xs[2]);
  y[58] = T(-317.49015732775086) * xs[4];
  y[59] = gbi_fmac(T(200.79840636817812), xs[5], T(-70.99295739719538) * xs[0]);
  y[60] = T(0);
  y[61] = T(0);
  y[62] = T(0);
  y[63] = T(0);
  y[64] = T(0);
  y[65] = T(0);
  y[66] = T(0);
  y[67] = gbi_fmac(e2, T(553.3071121272332) * xs[0], gbi_fmac(T(-368.8902275745455), xs[5], T(-86.94826047713663) * xs[0]));
  y[68] = gbi_fmac(e2, T(-857.1796922427575) * xs[1], T(224.49944320643647) * xs[1]);
  y[69] = gbi_fmac(e2, T(553.3071121272332) * xs[2], gbi_fmac(T(368.8902275745455), xs[3], T(-86.94826047713663) * xs[2]));
  y[70] = T(0);
  y[71] = T(0);
  y[72] = T(0);
  y[73] = T(0);
  y[74] = T(0);
  y[75] = T(0);
  y[76] = T(0);
  y[77] = T(127.63584563479449) * xs[0];
  y[78] = T(-201.8099916438052) * xs[1];
  y[79] = T(127.63584563479449) * xs[2];
  y[80] = T(0);
  y[81] = T(0);
  y[82] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_H_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[66], gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6]))), gbi_fmac(T(-382.90753690438345), xs[76], gbi_fmac(T(-325.330601081423), xs[66], gbi_fmac(T(-212.9788721915862), xs[60], gbi_fmac(T(-39.27922024247863), xs[48], gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))))))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[67], gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7]))), gbi_fmac(T(1083.026063650111), xs[77], gbi_fmac(T(983.7072735321215), xs[67], gbi_fmac(T(301.1976095522672), xs[59], gbi_fmac(T(124.21180068162376), xs[49], gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7])))))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(5039.166873289622), xs[68], gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8]))), gbi_fmac(T(-1482.994513567979), xs[78], gbi_fmac(T(-1374.772708486752), xs[68], gbi_fmac(T(-175.66201313073597), xs[50], gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8]))))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-3755.9732262135544), xs[69], gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9]))), gbi_fmac(T(1083.026063650111), xs[79], gbi_fmac(T(983.7072735321215), xs[69], gbi_fmac(T(-301.1976095522672), xs[57], gbi_fmac(T(124.21180068162376), xs[51], gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9])))))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(1419.6244410825732), xs[70], gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10]))), gbi_fmac(T(-382.90753690438345), xs[80], gbi_fmac(T(-325.330601081423), xs[70], gbi_fmac(T(212.9788721915862), xs[56], gbi_fmac(T(-39.27922024247863), xs[52], gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))))))));
  y[11] = gbi_fmac(T(-673.4983296193094), xs[67], gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7])));
  y[12] = gbi_fmac(T(1043.3791257256396), xs[68], gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8])));
  y[13] = gbi_fmac(T(-673.4983296193094), xs[69], gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9])));
  y[14] = gbi_fmac(T(-1593.7879407248633), xs[70], gbi_fmac(T(-695.586083817093), xs[56], gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))))));
  y[15] = gbi_fmac(T(2108.3832668658706), xs[69], gbi_fmac(T(1967.4145470642432), xs[57], gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]))))));
  y[16] = gbi_fmac(T(-2693.993318477238), xs[58], gbi_fmac(T(-328.63353450309967), xs[34], T(-48.0) * xs[16]));
  y[17] = gbi_fmac(T(-2108.3832668658706), xs[67], gbi_fmac(T(1967.4145470642432), xs[59], gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]))))));
  y[18] = gbi_fmac(T(1593.7879407248633), xs[66], gbi_fmac(T(-695.586083817093), xs[60], gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))))));
  y[19] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[65], gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19])), gbi_fmac(T(-1013.0781177812858), xs[75], gbi_fmac(T(-1126.978260659894), xs[65], gbi_fmac(T(-563.4891303299471), xs[61], gbi_fmac(T(-68.0336051416609), xs[47], gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])))))));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[66], gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6]))), gbi_fmac(T(4642.50715963613), xs[76], gbi_fmac(T(4507.913042639577), xs[66], gbi_fmac(T(1721.4877286812125), xs[60], gbi_fmac(T(408.20163084996545), xs[48], gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[67], gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7]))), gbi_fmac(T(-10380.961594975855), xs[77], gbi_fmac(T(-9428.976614670333), xs[67], gbi_fmac(T(-1924.681791881453), xs[59], gbi_fmac(T(-1020.5040771249135), xs[49], gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7])))))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-41821.305812166014), xs[68], gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8]))), gbi_fmac(T(13401.763791653422), xs[78], gbi_fmac(T(11926.816842728827), xs[68], gbi_fmac(T(1360.6721028332179), xs[50], gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8]))))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(33062.645272220645), xs[69], gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9]))), gbi_fmac(T(-10380.961594975855), xs[79], gbi_fmac(T(-9428.976614670333), xs[69], gbi_fmac(T(1924.681791881453), xs[57], gbi_fmac(T(-1020.5040771249135), xs[51], gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9])))))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-15806.96781185306), xs[70], gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10]))), gbi_fmac(T(4642.50715963613), xs[80], gbi_fmac(T(4507.913042639577), xs[70], gbi_fmac(T(-1721.4877286812125), xs[56], gbi_fmac(T(408.20163084996545), xs[52], gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))))))));
  y[25] = gbi_fmac(e2, gbi_fmac(T(3951.741952963265), xs[71], gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25])), gbi_fmac(T(-1013.0781177812858), xs[81], gbi_fmac(T(-1126.978260659894), xs[71], gbi_fmac(T(563.4891303299471), xs[55], gbi_fmac(T(-68.0336051416609), xs[53], gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])))))));
  y[26] = gbi_fmac(T(-3299.4545003682047), xs[66], gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6])));
  y[27] = gbi_fmac(T(8729.536070147142), xs[67], gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7])));
  y[28] = gbi_fmac(T(-11711.901638931227), xs[68], gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8])));
  y[29] = gbi_fmac(T(8729.536070147142), xs[69], gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9])));
  y[30] = gbi_fmac(T(-3299.4545003682047), xs[70], gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10])));
  y[31] = gbi_fmac(T(-5855.950819465615), xs[71], gbi_fmac(T(-1951.983606488538), xs[55], gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]))));
  y[32] = gbi_fmac(T(15615.868851908304), xs[70], gbi_fmac(T(8945.11263204662), xs[56], gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))))));
  y[33] = gbi_fmac(T(-16331.46655998781), xs[69], gbi_fmac(T(-20001.879911648302), xs[57], gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], T(-47.434164902525694) * xs[9]))))));
  y[34] = gbi_fmac(T(25822.315930218192), xs[58], gbi_fmac(2700.0f, xs[34], T(328.63353450309967) * xs[16]));
  y[35] = gbi_fmac(T(16331.46655998781), xs[67], gbi_fmac(T(-20001.879911648302), xs[59], gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], T(47.434164902525694) * xs[7]))))));
  y[36] = gbi_fmac(T(-15615.868851908304), xs[66], gbi_fmac(T(8945.11263204662), xs[60], gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))))));
  y[37] = gbi_fmac(T(5855.950819465615), xs[65], gbi_fmac(T(-1951.983606488538), xs[61], gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]))));
  y[38] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[64], T(560.0) * xs[38]), gbi_fmac(T(-2026.1562355625713), xs[74], gbi_fmac(T(-3380.934781979682), xs[64], gbi_fmac(T(-1126.978260659894), xs[62], T(-180.0) * xs[38]))));
  y[39] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[65], gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19])), gbi_fmac(T(16209.24988450057), xs[75], gbi_fmac(T(19158.630431218196), xs[65], gbi_fmac(T(6761.869563959364), xs[61], gbi_fmac(T(952.4704719832527), xs[47], gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])))))));
  y[40] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[66], gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6]))), gbi_fmac(T(-56732.374595752), xs[76], gbi_fmac(T(-56071.31459133092), xs[66], gbi_fmac(T(-15777.695649238518), xs[60], gbi_fmac(T(-4364.768035073571), xs[48], gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))))))));
  y[41] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[67], gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], T(-419.06562731868144) * xs[7]))), gbi_fmac(T(113464.749191504), xs[77], gbi_fmac(T(102139.30252356337), xs[67], gbi_fmac(T(15777.695649238516), xs[59], gbi_fmac(T(9759.91803244269), xs[49], gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], T(120.26755886059097) * xs[7])))))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(T(430300.7904337778), xs[68], gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], T(573.8292428937376) * xs[8]))), gbi_fmac(T(-141830.93648938002), xs[78], gbi_fmac(T(-123967.60867258835), xs[68], gbi_fmac(-12600.0f, xs[50], gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], T(-175.662013130736) * xs[8]))))))));
  y[43] = gbi_fmac(e2, gbi_fmac(T(-351339.1241596774), xs[69], gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], T(-419.06562731868144) * xs[9]))), gbi_fmac(T(113464.749191504), xs[79], gbi_fmac(T(102139.30252356337), xs[69], gbi_fmac(T(-15777.695649238516), xs[57], gbi_fmac(T(9759.91803244269), xs[51], gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], T(120.26755886059097) * xs[9])))))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(T(187798.66131067774), xs[70], gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10]))), gbi_fmac(T(-56732.374595752), xs[80], gbi_fmac(T(-56071.31459133092), xs[70], gbi_fmac(T(15777.695649238518), xs[56], gbi_fmac(T(-4364.768035073571), xs[52], gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))))))));
  y[45] = gbi_fmac(e2, gbi_fmac(T(-61471.54149053967), xs[71], gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25])), gbi_fmac(T(16209.24988450057), xs[81], gbi_fmac(T(19158.630431218196), xs[71], gbi_fmac(T(-6761.869563959364), xs[55], gbi_fmac(T(952.4704719832527), xs[53], gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])))))));
  y[46] = gbi_fmac(e2, gbi_fmac(T(10245.256915089945), xs[72], T(560.0) * xs[46]), gbi_fmac(T(-2026.1562355625713), xs[82], gbi_fmac(T(-3380.934781979682), xs[72], gbi_fmac(T(1126.978260659894), xs[54], T(-180.0) * xs[46]))));
  y[47] = gbi_fmac(T(-12778.73233149517), xs[65], gbi_fmac(T(-952.4704719832527), xs[39], T(-68.0336051416609) * xs[19]));
  y[48] = gbi_fmac(T(51114.92932598069), xs[66], gbi_fmac(T(4364.768035073571), xs[40], gbi_fmac(T(408.20163084996545), xs[20], T(39.27922024247863) * xs[6])));
  y[49] = gbi_fmac(T(-106914.54531540598), xs[67], gbi_fmac(T(-9759.91803244269), xs[41], gbi_fmac(T(-1020.5040771249135), xs[21], T(-124.21180068162376) * xs[7])));
  y[50] = gbi_fmac(T(135237.3912791873), xs[68], gbi_fmac(12600.0f, xs[42], gbi_fmac(T(1360.6721028332179), xs[22], T(175.66201313073597) * xs[8])));
  y[51] = gbi_fmac(T(-106914.54531540598), xs[69], gbi_fmac(T(-9759.91803244269), xs[43], gbi_fmac(T(-1020.5040771249135), xs[23], T(-124.21180068162376) * xs[9])));
  y[52] = gbi_fmac(T(51114.92932598069), xs[70], gbi_fmac(T(4364.768035073571), xs[44], gbi_fmac(T(408.20163084996545), xs[24], T(39.27922024247863) * xs[10])));
  y[53] = gbi_fmac(T(-12778.73233149517), xs[71], gbi_fmac(T(-952.4704719832527), xs[45], T(-68.0336051416609) * xs[25]));
  y[54] = gbi_fmac(-18144.0f, xs[72], gbi_fmac(T(-4031.9999999999995), xs[54], T(-1126.978260659894) * xs[46]));
  y[55] = gbi_fmac(81648.0f, xs[71], gbi_fmac(T(32255.999999999996), xs[55], gbi_fmac(T(6761.869563959364), xs[45], gbi_fmac(T(1951.983606488538), xs[31], T(563.4891303299471) * xs[25]))));
  y[56] = gbi_fmac(T(-166292.5068185575), xs[70], gbi_fmac(-112896.0f, xs[56], gbi_fmac(T(-15777.695649238518), xs[44], gbi_fmac(T(-8945.11263204662), xs[32], gbi_fmac(T(-1721.4877286812125), xs[24], gbi_fmac(T(-695.586083817093), xs[14], T(-212.9788721915862) * xs[10]))))));
  y[57] = gbi_fmac(T(155552.39662570294), xs[69], gbi_fmac(225792.0f, xs[57], gbi_fmac(T(15777.695649238516), xs[43], gbi_fmac(T(20001.879911648302), xs[33], gbi_fmac(T(1924.681791881453), xs[23], gbi_fmac(T(1967.4145470642432), xs[15], T(301.1976095522672) * xs[9]))))));
  y[58] = gbi_fmac(-282240.0f, xs[58], gbi_fmac(T(-25822.315930218192), xs[34], T(-2693.993318477238) * xs[16]));
  y[59] = gbi_fmac(T(-155552.39662570294), xs[67], gbi_fmac(225792.0f, xs[59], gbi_fmac(T(-15777.695649238516), xs[41], gbi_fmac(T(20001.879911648302), xs[35], gbi_fmac(T(-1924.681791881453), xs[21], gbi_fmac(T(1967.4145470642432), xs[17], T(-301.1976095522672) * xs[7]))))));
  y[60] = gbi_fmac(T(166292.5068185575), xs[66], gbi_fmac(-112896.0f, xs[60], gbi_fmac(T(15777.695649238518), xs[40], gbi_fmac(T(-8945.11263204662), xs[36], gbi_fmac(T(1721.4877286812125), xs[20], gbi_fmac(T(-695.586083817093), xs[18], T(212.9788721915862) * xs[6]))))));
  y[61] = gbi_fmac(-81648.0f, xs[65], gbi_fmac(T(32255.999999999996), xs[61], gbi_fmac(T(-6761.869563959364), xs[39], gbi_fmac(T(1951.983606488538), xs[37], T(-563.4891303299471) * xs[19]))));
  y[62] = gbi_fmac(18144.0f, xs[64], gbi_fmac(T(-4031.9999999999995), xs[62], T(1126.978260659894) * xs[38]));
  y[63] = gbi_fmac(e2, T(20618.18181818182) * xs[63], T(-7560.0) * xs[63]);
  y[64] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[64], T(-10245.256915089945) * xs[38]), gbi_fmac(T(40775.60768177688), xs[74], gbi_fmac(69552.0f, xs[64], gbi_fmac(18144.0f, xs[62], T(3380.934781979682) * xs[38]))));
  y[65] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[65], gbi_fmac(T(61471.54149053967), xs[39], T(3951.741952963265) * xs[19])), gbi_fmac(T(-244653.6460906613), xs[75], gbi_fmac(-291816.0f, xs[65], gbi_fmac(-81648.0f, xs[61], gbi_fmac(T(-12778.73233149517), xs[47], gbi_fmac(T(-19158.630431218196), xs[39], gbi_fmac(T(-5855.950819465615), xs[37], T(-1126.978260659894) * xs[19])))))));
  y[66] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[66], gbi_fmac(T(-187798.66131067774), xs[40], gbi_fmac(T(-15806.96781185306), xs[20], T(-1419.6244410825732) * xs[6]))), gbi_fmac(T(747429.2348382615), xs[76], gbi_fmac(737856.0f, xs[66], gbi_fmac(T(166292.5068185575), xs[60], gbi_fmac(T(51114.92932598069), xs[48], gbi_fmac(T(56071.31459133092), xs[40], gbi_fmac(T(15615.868851908304), xs[36], gbi_fmac(T(3299.4545003682047), xs[26], gbi_fmac(T(4507.913042639577), xs[20], gbi_fmac(T(1593.7879407248633), xs[18], T(325.330601081423) * xs[6]))))))))));
  y[67] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[67], gbi_fmac(T(351339.1241596774), xs[41], gbi_fmac(T(33062.645272220645), xs[21], T(3755.9732262135544) * xs[7]))), gbi_fmac(T(-1398312.0588116883), xs[77], gbi_fmac(-1248912.0f, xs[67], gbi_fmac(T(-155552.39662570294), xs[59], gbi_fmac(T(-106914.54531540598), xs[49], gbi_fmac(T(-102139.30252356337), xs[41], gbi_fmac(T(-16331.46655998781), xs[35], gbi_fmac(T(-8729.536070147142), xs[27], gbi_fmac(T(-9428.976614670333), xs[21], gbi_fmac(T(-2108.3832668658706), xs[17], gbi_fmac(T(-673.4983296193094), xs[11], T(-983.7072735321215) * xs[7])))))))))));
  y[68] = gbi_fmac(e2, gbi_fmac(T(-5195781.818181818), xs[68], gbi_fmac(T(-430300.7904337778), xs[42], gbi_fmac(T(-41821.305812166014), xs[22], T(-5039.166873289622) * xs[8]))), gbi_fmac(T(1712575.5226346292), xs[78], gbi_fmac(1481760.0f, xs[68], gbi_fmac(T(135237.3912791873), xs[50], gbi_fmac(T(123967.60867258835), xs[42], gbi_fmac(T(11711.901638931227), xs[28], gbi_fmac(T(11926.816842728827), xs[22], gbi_fmac(T(1043.3791257256396), xs[12], T(1374.772708486752) * xs[8]))))))));
  y[69] = gbi_fmac(e2, gbi_fmac(T(4329818.181818183), xs[69], gbi_fmac(T(351339.1241596774), xs[43], gbi_fmac(T(33062.645272220645), xs[23], T(3755.9732262135544) * xs[9]))), gbi_fmac(T(-1398312.0588116883), xs[79], gbi_fmac(-1248912.0f, xs[69], gbi_fmac(T(155552.39662570294), xs[57], gbi_fmac(T(-106914.54531540598), xs[51], gbi_fmac(T(-102139.30252356337), xs[43], gbi_fmac(T(16331.46655998781), xs[33], gbi_fmac(T(-8729.536070147142), xs[29], gbi_fmac(T(-9428.976614670333), xs[23], gbi_fmac(T(2108.3832668658706), xs[15], gbi_fmac(T(-673.4983296193094), xs[13], T(-983.7072735321215) * xs[9])))))))))));
  y[70] = gbi_fmac(e2, gbi_fmac(T(-2474181.8181818184), xs[70], gbi_fmac(T(-187798.66131067774), xs[44], gbi_fmac(T(-15806.96781185306), xs[24], T(-1419.6244410825732) * xs[10]))), gbi_fmac(T(747429.2348382615), xs[80], gbi_fmac(737856.0f, xs[70], gbi_fmac(T(-166292.5068185575), xs[56], gbi_fmac(T(51114.92932598069), xs[52], gbi_fmac(T(56071.31459133092), xs[44], gbi_fmac(T(-15615.868851908304), xs[32], gbi_fmac(T(3299.4545003682047), xs[30], gbi_fmac(T(4507.913042639577), xs[24], gbi_fmac(T(-1593.7879407248633), xs[14], T(325.330601081423) * xs[10]))))))))));
  y[71] = gbi_fmac(e2, gbi_fmac(T(927818.1818181819), xs[71], gbi_fmac(T(61471.54149053967), xs[45], T(3951.741952963265) * xs[25])), gbi_fmac(T(-244653.6460906613), xs[81], gbi_fmac(-291816.0f, xs[71], gbi_fmac(81648.0f, xs[55], gbi_fmac(T(-12778.73233149517), xs[53], gbi_fmac(T(-19158.630431218196), xs[45], gbi_fmac(T(5855.950819465615), xs[31], T(-1126.978260659894) * xs[25])))))));
  y[72] = gbi_fmac(e2, gbi_fmac(T(-206181.8181818182), xs[72], T(-10245.256915089945) * xs[46]), gbi_fmac(T(40775.60768177688), xs[82], gbi_fmac(69552.0f, xs[72], gbi_fmac(-18144.0f, xs[54], T(3380.934781979682) * xs[46]))));
  y[73] = gbi_fmac(e2, T(20618.18181818182) * xs[73], T(-7560.0) * xs[73]);
  y[74] = gbi_fmac(T(-40775.60768177688), xs[64], T(-2026.1562355625713) * xs[38]);
  y[75] = gbi_fmac(T(244653.6460906613), xs[65], gbi_fmac(T(16209.24988450057), xs[39], T(1013.0781177812858) * xs[19]));
  y[76] = gbi_fmac(T(-747429.2348382615), xs[66], gbi_fmac(T(-56732.374595752), xs[40], gbi_fmac(T(-4642.50715963613), xs[20], T(-382.90753690438345) * xs[6])));
  y[77] = gbi_fmac(T(1398312.0588116883), xs[67], gbi_fmac(T(113464.749191504), xs[41], gbi_fmac(T(10380.961594975855), xs[21], T(1083.026063650111) * xs[7])));
  y[78] = gbi_fmac(T(-1712575.5226346292), xs[68], gbi_fmac(T(-141830.93648938002), xs[42], gbi_fmac(T(-13401.763791653422), xs[22], T(-1482.994513567979) * xs[8])));
  y[79] = gbi_fmac(T(1398312.0588116883), xs[69], gbi_fmac(T(113464.749191504), xs[43], gbi_fmac(T(10380.961594975855), xs[23], T(1083.026063650111) * xs[9])));
  y[80] = gbi_fmac(T(-747429.2348382615), xs[70], gbi_fmac(T(-56732.374595752), xs[44], gbi_fmac(T(-4642.50715963613), xs[24], T(-382.90753690438345) * xs[10])));
  y[81] = gbi_fmac(T(244653.6460906613), xs[71], gbi_fmac(T(16209.24988450057), xs[45], T(1013.0781177812858) * xs[25]));
  y[82] = gbi_fmac(T(-40775.60768177688), xs[72], T(-2026.1562355625713) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t5_couple_P_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // point target: 1s rows only, beta from the source's finite-size operator alone
  y[0] = gbi_fmac(e2, gbi_fmac(T(118.56580974154997), xs[67], gbi_fmac(T(17.638342073763937), xs[41], gbi_fmac(T(3.319700011034928), xs[21], gbi_fmac(T(0.848528137423857), xs[7], T(0.3333333333333333) * xs[0])))), gbi_fmac(T(-127.63584563479449), xs[77], gbi_fmac(T(-86.94826047713663), xs[67], gbi_fmac(T(-70.99295739719538), xs[59], gbi_fmac(T(-17.5662013130736), xs[49], gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-183.68136262344808), xs[68], gbi_fmac(T(-27.888667551135853), xs[42], gbi_fmac(T(-5.421047417431508), xs[22], gbi_fmac(T(-1.469693845669907), xs[8], T(-0.6666666666666666) * xs[1])))), gbi_fmac(T(201.8099916438052), xs[78], gbi_fmac(T(224.49944320643647), xs[68], gbi_fmac(T(28.685486624025447), xs[50], gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1])))))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(118.56580974154997), xs[69], gbi_fmac(T(17.638342073763937), xs[43], gbi_fmac(T(3.319700011034928), xs[23], gbi_fmac(T(0.848528137423857), xs[9], T(0.3333333333333333) * xs[2])))), gbi_fmac(T(-127.63584563479449), xs[79], gbi_fmac(T(-86.94826047713663), xs[69], gbi_fmac(T(70.99295739719538), xs[57], gbi_fmac(T(-17.5662013130736), xs[51], gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))))))))));
}
static constexpr int gbi_t5_nnz = 571;   // pair-frame nonzeros (all rows, all columns)
static constexpr int gbi_t5_flops_point = 1753;   // per (point, sphere): 1s rows from all columns
// algorithmic flops per ordered pair, [rows][cols] with 0 = all, 1 = L, 2 = H
static constexpr int gbi_t5_flops[3][3] = {{4139, 2056, 3966}, {1823, 166, 1764}, {3947, 1978, 3800}};

// ---------------- minimal truncation (every mode of rank <= 4): 47 components per sphere
struct GbiTrunc40 {
  static constexpr int D = 47;      // components per sphere (L + H)
  static constexpr int NL = 6;
  static constexpr int H = 41;
  static constexpr int NMODE = 9;
  static constexpr int MAXK = 4;
};
__host__ __device__ constexpr int gbi_t40_k(int m) { constexpr int v[9] = {1, 1, 2, 1, 2, 3, 2, 3, 4}; return v[m]; }
__host__ __device__ constexpr int gbi_t40_L(int m) { constexpr int v[9] = {1, 2, 2, 3, 3, 3, 4, 4, 4}; return v[m]; }
__host__ __device__ constexpr int gbi_t40_off(int m) { constexpr int v[9] = {0, 3, 6, 11, 14, 19, 26, 31, 38}; return v[m]; }
// internal coordinate x = scale * packed coordinate of the paper's irreducible tensor
static const double gbi_t40_scale[47] = {1.0, 1.0, 1.0, 0.7071067811865476, 0.7071067811865476, 0.7071067811865476, 1.0, 1.0, 1.0, 1.0, 1.0, 0.7745966692414834, 0.7745966692414834, 0.7745966692414834, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 0.816496580927726, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422, 1.01418510567422, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 0.8660254037844386, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0};
// self scalar g per component (units 1/a): 8 pi eta V = -g Q for an isolated sphere
static const double gbi_t40_self[47] = {1.3333333333333333, 1.3333333333333333, 1.3333333333333333, 2.0, 2.0, 2.0, 1.2, 1.2, 1.2, 1.2, 1.2, 4.0, 4.0, 4.0, 12.0, 12.0, 12.0, 12.0, 12.0, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 6.857142857142857, 72.0, 72.0, 72.0, 72.0, 72.0, 180.0, 180.0, 180.0, 180.0, 180.0, 180.0, 180.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0, 100.0};
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_all_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0]))), gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1]))), gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1]))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2]))), gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4]));
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))))));
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0]))), gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5]))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1]))), gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1]))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2]))), gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3]))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0])));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1])));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2])));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4]));
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0]))), gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0])))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1]))), gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1]))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2]))), gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2])))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0])));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1])));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2])));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], gbi_fmac(T(-47.434164902525694), xs[9], gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]))))));
  y[34] = gbi_fmac(2700.0f, xs[34], gbi_fmac(T(328.63353450309967), xs[16], T(46.475800154489) * xs[4]));
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], gbi_fmac(T(47.434164902525694), xs[7], gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]))))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], gbi_fmac(T(-419.06562731868144), xs[7], T(-70.55336829505575) * xs[0]))), gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], gbi_fmac(T(120.26755886059097), xs[7], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0])))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], gbi_fmac(T(573.8292428937376), xs[8], T(111.55467020454341) * xs[1]))), gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], gbi_fmac(T(-175.662013130736), xs[8], T(-35.85685828003181) * xs[1]))))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], gbi_fmac(T(-419.06562731868144), xs[9], T(-70.55336829505575) * xs[2]))), gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], gbi_fmac(T(120.26755886059097), xs[9], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2])))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_all_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
  y[31] = T(0);
  y[32] = T(0);
  y[33] = gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]);
  y[34] = T(46.475800154489) * xs[4];
  y[35] = gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]);
  y[36] = T(0);
  y[37] = T(0);
  y[38] = T(0);
  y[39] = T(0);
  y[40] = T(0);
  y[41] = gbi_fmac(e2, T(-70.55336829505575) * xs[0], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]));
  y[42] = gbi_fmac(e2, T(111.55467020454341) * xs[1], T(-35.85685828003181) * xs[1]);
  y[43] = gbi_fmac(e2, T(-70.55336829505575) * xs[2], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]));
  y[44] = T(0);
  y[45] = T(0);
  y[46] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_all_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7])), gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11]))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8])), gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8])))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9])), gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13]))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], T(8.485281374238571) * xs[16]);
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]))));
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7])), gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7])))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8])), gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8])))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9])), gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9])))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7]));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8]));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9]));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], T(-48.0) * xs[16]);
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7])), gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7])))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8])), gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8])))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9])), gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9])))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7]));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8]));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9]));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], T(-47.434164902525694) * xs[9]))));
  y[34] = gbi_fmac(2700.0f, xs[34], T(328.63353450309967) * xs[16]);
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], T(47.434164902525694) * xs[7]))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], T(-419.06562731868144) * xs[7])), gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], T(120.26755886059097) * xs[7])))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], T(573.8292428937376) * xs[8])), gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], T(-175.662013130736) * xs[8])))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], T(-419.06562731868144) * xs[9])), gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], T(120.26755886059097) * xs[9])))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_L_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], gbi_fmac(T(2.262741699796952), xs[7], T(0.6666666666666666) * xs[0]))), gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], gbi_fmac(T(-3.919183588453085), xs[8], T(-1.3333333333333333) * xs[1]))), gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1]))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], gbi_fmac(T(2.262741699796952), xs[9], T(0.6666666666666666) * xs[2]))), gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], gbi_fmac(-3.0f, xs[9], gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]))))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], gbi_fmac(T(8.485281374238571), xs[16], T(2.0) * xs[4]));
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], gbi_fmac(3.0f, xs[7], gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]))))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_L_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, T(0.6666666666666666) * xs[0], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]));
  y[1] = gbi_fmac(e2, T(-1.3333333333333333) * xs[1], T(2.0) * xs[1]);
  y[2] = gbi_fmac(e2, T(0.6666666666666666) * xs[2], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]));
  y[3] = gbi_fmac(-1.0f, xs[3], T(-1.4142135623730951) * xs[2]);
  y[4] = T(2.0) * xs[4];
  y[5] = gbi_fmac(-1.0f, xs[5], T(1.4142135623730951) * xs[0]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_L_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[0] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[41], gbi_fmac(T(11.06566670344976), xs[21], T(2.262741699796952) * xs[7])), gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], T(-0.5163977794943223) * xs[11]))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-111.55467020454341), xs[42], gbi_fmac(T(-18.070158058105026), xs[22], T(-3.919183588453085) * xs[8])), gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], T(2.449489742783178) * xs[8])))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(70.55336829505575), xs[43], gbi_fmac(T(11.06566670344976), xs[23], T(2.262741699796952) * xs[9])), gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], T(-0.5163977794943223) * xs[13]))))));
  y[3] = gbi_fmac(T(-56.124860801609124), xs[43], gbi_fmac(T(-28.460498941515414), xs[33], gbi_fmac(T(-10.95445115010332), xs[23], gbi_fmac(T(-4.898979485566356), xs[15], T(-3.0) * xs[9]))));
  y[4] = gbi_fmac(T(46.475800154489), xs[34], T(8.485281374238571) * xs[16]);
  y[5] = gbi_fmac(T(56.124860801609124), xs[41], gbi_fmac(T(-28.460498941515414), xs[35], gbi_fmac(T(10.95445115010332), xs[21], gbi_fmac(T(-4.898979485566356), xs[17], T(3.0) * xs[7]))));
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_H_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], gbi_fmac(T(-9.6), xs[7], T(-2.262741699796952) * xs[0]))), gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], gbi_fmac(3.0f, xs[7], T(3.0) * xs[5]))))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], gbi_fmac(T(14.4), xs[8], T(3.919183588453085) * xs[1]))), gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], gbi_fmac(-6.0f, xs[8], T(-2.449489742783178) * xs[1]))))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], gbi_fmac(T(-9.6), xs[9], T(-2.262741699796952) * xs[2]))), gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], gbi_fmac(3.0f, xs[9], T(-3.0) * xs[3]))))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], gbi_fmac(T(-2.1908902300206647), xs[7], T(-0.5163977794943223) * xs[0])));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], gbi_fmac(T(3.7947331922020555), xs[8], T(1.0327955589886446) * xs[1])));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], gbi_fmac(T(-2.1908902300206647), xs[9], T(-0.5163977794943223) * xs[2])));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], gbi_fmac(T(9.797958971132712), xs[9], gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]))))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], gbi_fmac(-48.0f, xs[16], T(-8.485281374238571) * xs[4]));
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], gbi_fmac(T(-9.797958971132712), xs[7], gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]))))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], gbi_fmac(T(56.33717734338851), xs[7], T(11.06566670344976) * xs[0]))), gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], gbi_fmac(T(-17.527121840165314), xs[7], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0])))))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], gbi_fmac(T(-79.67280026483827), xs[8], T(-18.070158058105026) * xs[1]))), gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], gbi_fmac(T(27.8854800926934), xs[8], T(7.58946638440411) * xs[1]))))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], gbi_fmac(T(56.33717734338851), xs[9], T(11.06566670344976) * xs[2]))), gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], gbi_fmac(T(-17.527121840165314), xs[9], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2])))))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], gbi_fmac(T(16.22696169078752), xs[7], T(2.868548662402545) * xs[0])));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], gbi_fmac(T(-24.34044253618128), xs[8], T(-4.9684720272649505) * xs[1])));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], gbi_fmac(T(16.22696169078752), xs[9], T(2.868548662402545) * xs[2])));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], gbi_fmac(T(-47.434164902525694), xs[9], gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]))))));
  y[34] = gbi_fmac(2700.0f, xs[34], gbi_fmac(T(328.63353450309967), xs[16], T(46.475800154489) * xs[4]));
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], gbi_fmac(T(47.434164902525694), xs[7], gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]))))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], gbi_fmac(T(-419.06562731868144), xs[7], T(-70.55336829505575) * xs[0]))), gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], gbi_fmac(T(120.26755886059097), xs[7], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0])))))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], gbi_fmac(T(573.8292428937376), xs[8], T(111.55467020454341) * xs[1]))), gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], gbi_fmac(T(-175.662013130736), xs[8], T(-35.85685828003181) * xs[1]))))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], gbi_fmac(T(-419.06562731868144), xs[9], T(-70.55336829505575) * xs[2]))), gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], gbi_fmac(T(120.26755886059097), xs[9], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2])))))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_H_L(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = T(0);
  y[7] = gbi_fmac(e2, T(-2.262741699796952) * xs[0], T(3.0) * xs[5]);
  y[8] = gbi_fmac(e2, T(3.919183588453085) * xs[1], T(-2.449489742783178) * xs[1]);
  y[9] = gbi_fmac(e2, T(-2.262741699796952) * xs[2], T(-3.0) * xs[3]);
  y[10] = T(0);
  y[11] = T(-0.5163977794943223) * xs[0];
  y[12] = T(1.0327955589886446) * xs[1];
  y[13] = T(-0.5163977794943223) * xs[2];
  y[14] = T(0);
  y[15] = gbi_fmac(T(4.898979485566356), xs[3], T(3.4641016151377544) * xs[2]);
  y[16] = T(-8.485281374238571) * xs[4];
  y[17] = gbi_fmac(T(4.898979485566356), xs[5], T(-3.4641016151377544) * xs[0]);
  y[18] = T(0);
  y[19] = T(0);
  y[20] = T(0);
  y[21] = gbi_fmac(e2, T(11.06566670344976) * xs[0], gbi_fmac(T(-10.95445115010332), xs[5], T(-1.5491933384829666) * xs[0]));
  y[22] = gbi_fmac(e2, T(-18.070158058105026) * xs[1], T(7.58946638440411) * xs[1]);
  y[23] = gbi_fmac(e2, T(11.06566670344976) * xs[2], gbi_fmac(T(10.95445115010332), xs[3], T(-1.5491933384829666) * xs[2]));
  y[24] = T(0);
  y[25] = T(0);
  y[26] = T(0);
  y[27] = T(2.868548662402545) * xs[0];
  y[28] = T(-4.9684720272649505) * xs[1];
  y[29] = T(2.868548662402545) * xs[2];
  y[30] = T(0);
  y[31] = T(0);
  y[32] = T(0);
  y[33] = gbi_fmac(T(-28.460498941515414), xs[3], T(-13.416407864998739) * xs[2]);
  y[34] = T(46.475800154489) * xs[4];
  y[35] = gbi_fmac(T(-28.460498941515414), xs[5], T(13.416407864998739) * xs[0]);
  y[36] = T(0);
  y[37] = T(0);
  y[38] = T(0);
  y[39] = T(0);
  y[40] = T(0);
  y[41] = gbi_fmac(e2, T(-70.55336829505575) * xs[0], gbi_fmac(T(56.124860801609124), xs[5], T(11.338934190276817) * xs[0]));
  y[42] = gbi_fmac(e2, T(111.55467020454341) * xs[1], T(-35.85685828003181) * xs[1]);
  y[43] = gbi_fmac(e2, T(-70.55336829505575) * xs[2], gbi_fmac(T(-56.124860801609124), xs[3], T(11.338934190276817) * xs[2]));
  y[44] = T(0);
  y[45] = T(0);
  y[46] = T(0);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_H_H(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // xs[q] = (a/r)^l_q * x'_q in the pair frame; y[p] = sum_q (alpha_pq + beta_pq (a/r)^2) xs[q]
  y[6] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[40], gbi_fmac(T(17.815379734994163), xs[20], T(2.4) * xs[6])), gbi_fmac(T(-34.01680257083045), xs[40], gbi_fmac(-30.0f, xs[36], gbi_fmac(T(-4.05674042269688), xs[26], gbi_fmac(T(-3.4641016151377544), xs[20], T(-4.898979485566356) * xs[18])))));
  y[7] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[41], gbi_fmac(T(-56.33717734338851), xs[21], T(-9.6) * xs[7])), gbi_fmac(T(120.26755886059097), xs[41], gbi_fmac(T(47.434164902525694), xs[35], gbi_fmac(T(16.22696169078752), xs[27], gbi_fmac(T(17.527121840165314), xs[21], gbi_fmac(T(9.797958971132712), xs[17], gbi_fmac(T(2.1908902300206647), xs[11], T(3.0) * xs[7])))))));
  y[8] = gbi_fmac(e2, gbi_fmac(T(573.8292428937376), xs[42], gbi_fmac(T(79.67280026483827), xs[22], T(14.4) * xs[8])), gbi_fmac(T(-175.662013130736), xs[42], gbi_fmac(T(-24.34044253618128), xs[28], gbi_fmac(T(-27.8854800926934), xs[22], gbi_fmac(T(-3.7947331922020555), xs[12], T(-6.0) * xs[8])))));
  y[9] = gbi_fmac(e2, gbi_fmac(T(-419.06562731868144), xs[43], gbi_fmac(T(-56.33717734338851), xs[23], T(-9.6) * xs[9])), gbi_fmac(T(120.26755886059097), xs[43], gbi_fmac(T(-47.434164902525694), xs[33], gbi_fmac(T(16.22696169078752), xs[29], gbi_fmac(T(17.527121840165314), xs[23], gbi_fmac(T(-9.797958971132712), xs[15], gbi_fmac(T(2.1908902300206647), xs[13], T(3.0) * xs[9])))))));
  y[10] = gbi_fmac(e2, gbi_fmac(T(148.16207341961706), xs[44], gbi_fmac(T(17.815379734994163), xs[24], T(2.4) * xs[10])), gbi_fmac(T(-34.01680257083045), xs[44], gbi_fmac(30.0f, xs[32], gbi_fmac(T(-4.05674042269688), xs[30], gbi_fmac(T(-3.4641016151377544), xs[24], T(4.898979485566356) * xs[14])))));
  y[11] = gbi_fmac(T(-81.9756061276768), xs[41], gbi_fmac(-12.0f, xs[21], T(-2.1908902300206647) * xs[7]));
  y[12] = gbi_fmac(T(129.6148139681572), xs[42], gbi_fmac(T(19.595917942265423), xs[22], T(3.7947331922020555) * xs[8]));
  y[13] = gbi_fmac(T(-81.9756061276768), xs[43], gbi_fmac(-12.0f, xs[23], T(-2.1908902300206647) * xs[9]));
  y[14] = gbi_fmac(T(-194.42222095223582), xs[44], gbi_fmac(T(-73.48469228349535), xs[32], gbi_fmac(T(-28.284271247461902), xs[24], gbi_fmac(-8.0f, xs[14], T(-4.898979485566356) * xs[10]))));
  y[15] = gbi_fmac(T(274.9545416973504), xs[43], gbi_fmac(T(232.379000772445), xs[33], gbi_fmac(T(44.721359549995796), xs[23], gbi_fmac(32.0f, xs[15], T(9.797958971132712) * xs[9]))));
  y[16] = gbi_fmac(T(-328.63353450309967), xs[34], T(-48.0) * xs[16]);
  y[17] = gbi_fmac(T(-274.9545416973504), xs[41], gbi_fmac(T(232.379000772445), xs[35], gbi_fmac(T(-44.721359549995796), xs[21], gbi_fmac(32.0f, xs[17], T(-9.797958971132712) * xs[7]))));
  y[18] = gbi_fmac(T(194.42222095223582), xs[40], gbi_fmac(T(-73.48469228349535), xs[36], gbi_fmac(T(28.284271247461902), xs[20], gbi_fmac(-8.0f, xs[18], T(4.898979485566356) * xs[6]))));
  y[19] = gbi_fmac(e2, gbi_fmac(320.0f, xs[39], T(25.71428571428571) * xs[19]), gbi_fmac(-90.0f, xs[39], gbi_fmac(T(-51.96152422706632), xs[37], T(-6.0) * xs[19])));
  y[20] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[40], gbi_fmac(T(-154.28571428571428), xs[20], T(-17.815379734994163) * xs[6])), gbi_fmac(T(432.0714226672649), xs[40], gbi_fmac(T(207.84609690826528), xs[36], gbi_fmac(T(35.13240262614719), xs[26], gbi_fmac(44.0f, xs[20], gbi_fmac(T(28.284271247461902), xs[18], T(3.4641016151377544) * xs[6]))))));
  y[21] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[41], gbi_fmac(T(385.71428571428567), xs[21], T(56.33717734338851) * xs[7])), gbi_fmac(T(-992.4903741886583), xs[41], gbi_fmac(T(-259.8076211353316), xs[35], gbi_fmac(T(-111.09841197270617), xs[27], gbi_fmac(-122.0f, xs[21], gbi_fmac(T(-44.721359549995796), xs[17], gbi_fmac(-12.0f, xs[11], T(-17.527121840165314) * xs[7])))))));
  y[22] = gbi_fmac(e2, gbi_fmac(T(-4233.202097703344), xs[42], gbi_fmac(T(-514.2857142857143), xs[22], T(-79.67280026483827) * xs[8])), gbi_fmac(T(1292.638497691557), xs[42], gbi_fmac(T(157.11688096991452), xs[28], gbi_fmac(168.0f, xs[22], gbi_fmac(T(19.595917942265423), xs[12], T(27.8854800926934) * xs[8])))));
  y[23] = gbi_fmac(e2, gbi_fmac(T(3279.0242451070717), xs[43], gbi_fmac(T(385.71428571428567), xs[23], T(56.33717734338851) * xs[9])), gbi_fmac(T(-992.4903741886583), xs[43], gbi_fmac(T(259.8076211353316), xs[33], gbi_fmac(T(-111.09841197270617), xs[29], gbi_fmac(-122.0f, xs[23], gbi_fmac(T(44.721359549995796), xs[15], gbi_fmac(-12.0f, xs[13], T(-17.527121840165314) * xs[9])))))));
  y[24] = gbi_fmac(e2, gbi_fmac(T(-1466.424222385869), xs[44], gbi_fmac(T(-154.28571428571428), xs[24], T(-17.815379734994163) * xs[10])), gbi_fmac(T(432.0714226672649), xs[44], gbi_fmac(T(-207.84609690826528), xs[32], gbi_fmac(T(35.13240262614719), xs[30], gbi_fmac(44.0f, xs[24], gbi_fmac(T(-28.284271247461902), xs[14], T(3.4641016151377544) * xs[10]))))));
  y[25] = gbi_fmac(e2, gbi_fmac(320.0f, xs[45], T(25.71428571428571) * xs[25]), gbi_fmac(-90.0f, xs[45], gbi_fmac(T(51.96152422706632), xs[31], T(-6.0) * xs[25])));
  y[26] = gbi_fmac(T(-321.9937887599697), xs[40], gbi_fmac(T(-35.13240262614719), xs[20], T(-4.05674042269688) * xs[6]));
  y[27] = gbi_fmac(T(910.7359661284933), xs[41], gbi_fmac(T(111.09841197270617), xs[21], T(16.22696169078752) * xs[7]));
  y[28] = gbi_fmac(T(-1247.0765814495917), xs[42], gbi_fmac(T(-157.11688096991452), xs[22], T(-24.34044253618128) * xs[8]));
  y[29] = gbi_fmac(T(910.7359661284933), xs[43], gbi_fmac(T(111.09841197270617), xs[23], T(16.22696169078752) * xs[9]));
  y[30] = gbi_fmac(T(-321.9937887599697), xs[44], gbi_fmac(T(-35.13240262614719), xs[24], T(-4.05674042269688) * xs[10]));
  y[31] = gbi_fmac(T(-545.5960043841964), xs[45], gbi_fmac(-135.0f, xs[31], T(-51.96152422706632) * xs[25]));
  y[32] = gbi_fmac(T(1666.8233259706922), xs[44], gbi_fmac(810.0f, xs[32], gbi_fmac(T(207.84609690826528), xs[24], gbi_fmac(T(73.48469228349535), xs[14], T(30.0) * xs[10]))));
  y[33] = gbi_fmac(T(-1863.5651316763792), xs[43], gbi_fmac(-2025.0f, xs[33], gbi_fmac(T(-259.8076211353316), xs[23], gbi_fmac(T(-232.379000772445), xs[15], T(-47.434164902525694) * xs[9]))));
  y[34] = gbi_fmac(2700.0f, xs[34], T(328.63353450309967) * xs[16]);
  y[35] = gbi_fmac(T(1863.5651316763792), xs[41], gbi_fmac(-2025.0f, xs[35], gbi_fmac(T(259.8076211353316), xs[21], gbi_fmac(T(-232.379000772445), xs[17], T(47.434164902525694) * xs[7]))));
  y[36] = gbi_fmac(T(-1666.8233259706922), xs[40], gbi_fmac(810.0f, xs[36], gbi_fmac(T(-207.84609690826528), xs[20], gbi_fmac(T(73.48469228349535), xs[18], T(-30.0) * xs[6]))));
  y[37] = gbi_fmac(T(545.5960043841964), xs[39], gbi_fmac(-135.0f, xs[37], T(51.96152422706632) * xs[19]));
  y[38] = gbi_fmac(e2, T(560.0) * xs[38], T(-180.0) * xs[38]);
  y[39] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[39], T(-320.0) * xs[19]), gbi_fmac(1395.0f, xs[39], gbi_fmac(T(545.5960043841964), xs[37], T(90.0) * xs[19])));
  y[40] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[40], gbi_fmac(T(1466.424222385869), xs[20], T(148.16207341961706) * xs[6])), gbi_fmac(-4770.0f, xs[40], gbi_fmac(T(-1666.8233259706922), xs[36], gbi_fmac(T(-321.9937887599697), xs[26], gbi_fmac(T(-432.0714226672649), xs[20], gbi_fmac(T(-194.42222095223582), xs[18], T(-34.01680257083045) * xs[6]))))));
  y[41] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[41], gbi_fmac(T(-3279.0242451070717), xs[21], T(-419.06562731868144) * xs[7])), gbi_fmac(9405.0f, xs[41], gbi_fmac(T(1863.5651316763792), xs[35], gbi_fmac(T(910.7359661284933), xs[27], gbi_fmac(T(992.4903741886583), xs[21], gbi_fmac(T(274.9545416973504), xs[17], gbi_fmac(T(81.9756061276768), xs[11], T(120.26755886059097) * xs[7])))))));
  y[42] = gbi_fmac(e2, gbi_fmac(39200.0f, xs[42], gbi_fmac(T(4233.202097703344), xs[22], T(573.8292428937376) * xs[8])), gbi_fmac(-11700.0f, xs[42], gbi_fmac(T(-1247.0765814495917), xs[28], gbi_fmac(T(-1292.638497691557), xs[22], gbi_fmac(T(-129.6148139681572), xs[12], T(-175.662013130736) * xs[8])))));
  y[43] = gbi_fmac(e2, gbi_fmac(-31360.0f, xs[43], gbi_fmac(T(-3279.0242451070717), xs[23], T(-419.06562731868144) * xs[9])), gbi_fmac(9405.0f, xs[43], gbi_fmac(T(-1863.5651316763792), xs[33], gbi_fmac(T(910.7359661284933), xs[29], gbi_fmac(T(992.4903741886583), xs[23], gbi_fmac(T(-274.9545416973504), xs[15], gbi_fmac(T(81.9756061276768), xs[13], T(120.26755886059097) * xs[9])))))));
  y[44] = gbi_fmac(e2, gbi_fmac(15680.0f, xs[44], gbi_fmac(T(1466.424222385869), xs[24], T(148.16207341961706) * xs[10])), gbi_fmac(-4770.0f, xs[44], gbi_fmac(T(1666.8233259706922), xs[32], gbi_fmac(T(-321.9937887599697), xs[30], gbi_fmac(T(-432.0714226672649), xs[24], gbi_fmac(T(194.42222095223582), xs[14], T(-34.01680257083045) * xs[10]))))));
  y[45] = gbi_fmac(e2, gbi_fmac(-4480.0f, xs[45], T(-320.0) * xs[25]), gbi_fmac(1395.0f, xs[45], gbi_fmac(T(-545.5960043841964), xs[31], T(90.0) * xs[25])));
  y[46] = gbi_fmac(e2, T(560.0) * xs[46], T(-180.0) * xs[46]);
}
template <typename T> __host__ __device__ __forceinline__ void gbi_t40_couple_P_all(T e2, const T* __restrict__ xs, T* __restrict__ y) {
  // point target: 1s rows only, beta from the source's finite-size operator alone
  y[0] = gbi_fmac(e2, gbi_fmac(T(17.638342073763937), xs[41], gbi_fmac(T(3.319700011034928), xs[21], gbi_fmac(T(0.848528137423857), xs[7], T(0.3333333333333333) * xs[0]))), gbi_fmac(T(-11.338934190276817), xs[41], gbi_fmac(T(-13.416407864998739), xs[35], gbi_fmac(T(-2.868548662402545), xs[27], gbi_fmac(T(-1.5491933384829666), xs[21], gbi_fmac(T(-3.4641016151377544), xs[17], gbi_fmac(T(-0.5163977794943223), xs[11], gbi_fmac(T(-1.4142135623730951), xs[5], xs[0]))))))));
  y[1] = gbi_fmac(e2, gbi_fmac(T(-27.888667551135853), xs[42], gbi_fmac(T(-5.421047417431508), xs[22], gbi_fmac(T(-1.469693845669907), xs[8], T(-0.6666666666666666) * xs[1]))), gbi_fmac(T(35.85685828003181), xs[42], gbi_fmac(T(4.9684720272649505), xs[28], gbi_fmac(T(7.58946638440411), xs[22], gbi_fmac(T(1.0327955589886446), xs[12], gbi_fmac(T(2.449489742783178), xs[8], T(2.0) * xs[1]))))));
  y[2] = gbi_fmac(e2, gbi_fmac(T(17.638342073763937), xs[43], gbi_fmac(T(3.319700011034928), xs[23], gbi_fmac(T(0.848528137423857), xs[9], T(0.3333333333333333) * xs[2]))), gbi_fmac(T(-11.338934190276817), xs[43], gbi_fmac(T(13.416407864998739), xs[33], gbi_fmac(T(-2.868548662402545), xs[29], gbi_fmac(T(-1.5491933384829666), xs[23], gbi_fmac(T(3.4641016151377544), xs[15], gbi_fmac(T(-0.5163977794943223), xs[13], gbi_fmac(T(1.4142135623730951), xs[3], xs[2]))))))));
}
static constexpr int gbi_t40_nnz = 253;   // pair-frame nonzeros (all rows, all columns)
static constexpr int gbi_t40_flops_point = 921;   // per (point, sphere): 1s rows from all columns
// algorithmic flops per ordered pair, [rows][cols] with 0 = all, 1 = L, 2 = H
static constexpr int gbi_t40_flops[3][3] = {{2035, 1106, 1900}, {981, 166, 922}, {1881, 1028, 1772}};

