// Spheres above a plane no-slip wall (z = 0, fluid z > 0): the superposition
// approximation of Sec. IV with the wall's Green's function in place of the Oseen tensor
// (Sec. VI: another geometry enters through its Green's function).
//
// Blake's Green's function is the Oseen tensor plus an image system at
// y* = (y1, y2, -y3), h = y3, R = x - y*, m = (1, 1, -1):
//
//   W_ij(x, y) = -G_ij(R) + 2 h m_j [ h (d_ij/|R|^3 - 3 R_i R_j/|R|^5) + d_i3 R_j/|R|^3
//                                      - (d_ij R_3 + R_i d_j3)/|R|^3 + 3 R_i R_3 R_j/|R|^5 ].
//
// gbi_wall_superpose adds to the unbounded superposition (gbi_superpose, l <= 2) the image
// flows, at the point-singularity level, of every sphere's force F, torque T and
// stresslet S = (20/3) pi eta a^2 V^(2s) (what it exerts on the fluid), its own images
// included:
//
//   8 pi eta u(x) = sum_m W_ij(x, R_m) F_j + D_jk d/dy_k W_ij(x, y)|_{y = R_m},
//   D_jk = S_jk + (1/2) eps_kjl T_l,   V_n += u(R_n),   Omega_n += curl u (R_n) / 2.
//
// In closed form, with phi = 1/|R|, z = x_3 and m = (1, 1, -1): the bracket is
// z d_i d_j phi - d_i3 d_j phi + d_j3 d_i phi, d/dy_k = -m_k d/dR_k (+ d/dh for k = 3), so with
//   Dt_jk = -D_jk m_k,   E_j = m_j (h F_j + D_j3),   H_jk = h m_j Dt_jk (symmetrised),   c_k = h m_3 Dt_3k,
//   Phi = -E.R/|R|^3 + 3 (R.H R)/|R|^5 - tr H / |R|^3,   chi = E_3/|R| - (c.R)/|R|^3
// (both harmonic), and q = R.Dt R, v = Dt R, a_i = eps_ijk Dt_jk,
//   u = -F/|R| - (F.R) R/|R|^3 - (a x R + tr Dt R)/|R|^3 + 3 q R/|R|^5 + 2 (z grad Phi - e_3 Phi + grad chi),
//   curl u = -2 (F x R + a)/|R|^3 + 6 (v x R)/|R|^5 + 4 e_3 x grad Phi.
// Everything that depends on the source alone is formed once per source (k_wall_records), so a
// pair costs about 100 floating-point instructions (nested dual numbers, which this replaces:
// 1 089 in the compiled FP32 kernel).  Measured, with the unbounded superposition: FP64 N = 1500
// 5.73 -> 1.02 ms, FP32 N = 10^4 4.29 -> 0.85 ms; the error against 64 bits of the FP32 sums fell from
// 2.9e-7 to 1.9e-7 (N = 4000), that of V in FP64 (rms over N = 1500, of the largest; extended precision as the
// reference) from 3.1e-16 to 2.6e-16.
// Sources in shared-memory tiles, split over gridDim.y slices whose partial sums are added in
// slice order by a second kernel, so the result does not depend on timing.
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "ctx.cuh"
#include "df.cuh"
#include "gbi_generated.cuh"

namespace gbi {
namespace {

constexpr int kWallThreads = 128;
constexpr int kWallTile = 32;
constexpr int kWallRec = 32;   // words per source record (layout at k_wall_records)

// Flops of one (target, source) term as written below (FMA = 2, rsqrt = 1)
constexpr int kWallPairFlops = 170;

__device__ __forceinline__ float wall_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double wall_rsqrt(double x) { return rsqrt(x); }

// a x b + c
template <typename T>
__device__ __forceinline__ void cross_add(const T* a, const T* b, T c0, T c1, T c2, T* o) {
  o[0] = gbi_fmac(a[1], b[2], gbi_fmac(-a[2], b[1], c0));
  o[1] = gbi_fmac(a[2], b[0], gbi_fmac(-a[0], b[2], c1));
  o[2] = gbi_fmac(a[0], b[1], gbi_fmac(-a[1], b[0], c2));
}

// Image flow at target x (times 8 pi eta) of the source record r added to u, its curl to c.
template <typename T>
__device__ __forceinline__ void wall_image_pair(const T* x, const T* __restrict__ r, T* u, T* c) {
  const T R[3] = {x[0] - r[0], x[1] - r[1], x[2] + r[2]};
  const T* F = r + 3;     // F
  const T* Dt = r + 6;    // Dt, row-major
  const T* a = r + 15;    // a
  const T* H = r + 18;    // 2 H: xx xy xz yy yz zz
  const T* E = r + 24;    // 2 E
  const T* cc = r + 27;   // 2 c
  const T tr = r[30];     // tr Dt + 2 E_3
  const T th = r[31];     // 2 tr H
  const T r2 = gbi_fmac(R[2], R[2], gbi_fmac(R[1], R[1], R[0] * R[0]));
  const T i1 = wall_rsqrt(r2);
  const T i2 = i1 * i1, i3 = i1 * i2, i5 = i3 * i2;
  const T FR = gbi_fmac(F[2], R[2], gbi_fmac(F[1], R[1], gbi_fmac(F[0], R[0], tr)));
  const T v[3] = {gbi_fmac(Dt[2], R[2], gbi_fmac(Dt[1], R[1], Dt[0] * R[0])),
                  gbi_fmac(Dt[5], R[2], gbi_fmac(Dt[4], R[1], Dt[3] * R[0])),
                  gbi_fmac(Dt[8], R[2], gbi_fmac(Dt[7], R[1], Dt[6] * R[0]))};
  const T q = gbi_fmac(R[2], v[2] + cc[2], gbi_fmac(R[1], v[1] + cc[1], R[0] * (v[0] + cc[0])));
  const T g[3] = {gbi_fmac(H[2], R[2], gbi_fmac(H[1], R[1], H[0] * R[0])),
                  gbi_fmac(H[4], R[2], gbi_fmac(H[3], R[1], H[1] * R[0])),
                  gbi_fmac(H[5], R[2], gbi_fmac(H[4], R[1], H[2] * R[0]))};
  const T qh = gbi_fmac(R[2], g[2], gbi_fmac(R[1], g[1], R[0] * g[0]));
  const T ER = gbi_fmac(E[2], R[2], gbi_fmac(E[1], R[1], gbi_fmac(E[0], R[0], th)));
  // 2 Phi and 2 grad Phi = 6 g i5 - E i3 + kp R
  const T t5 = T(3) * i5;
  const T phi = gbi_fmac(t5, qh, -(ER * i3));
  const T kp = gbi_fmac(T(-15) * i2, qh, T(3) * ER) * i5;
  const T s5 = T(6) * i5;
  T dp[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) dp[k] = gbi_fmac(s5, g[k], gbi_fmac(-i3, E[k], kp * R[k]));
  // u: the R-parallel terms of the Oseen part and grad chi, the others, z 2 grad Phi - 2 e_3 Phi;
  // a pair's terms are added together before the sum takes them (one rounding against the sum:
  // accumulating term by term measured 20 % more FP32 error)
  const T k0 = gbi_fmac(t5, q, -(FR * i3));
  T w[3];
  cross_add<T>(a, R, cc[0], cc[1], cc[2], w);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const T pre = k == 2 ? -gbi_fmac(i1, F[k], phi) : -(i1 * F[k]);
    u[k] += gbi_fmac(x[2], dp[k], gbi_fmac(k0, R[k], gbi_fmac(-i3, w[k], pre)));
  }
  // curl: -2 (F x R + a) i3 + 6 (v x R) i5 + 2 e_3 x (2 grad Phi)
  T f[3], vr[3];
  cross_add<T>(F, R, a[0], a[1], a[2], f);
  cross_add<T>(v, R, T(0), T(0), T(0), vr);
  const T m3 = T(-2) * i3;
  c[0] += gbi_fmac(T(-2), dp[1], gbi_fmac(m3, f[0], s5 * vr[0]));
  c[1] += gbi_fmac(T(2), dp[0], gbi_fmac(m3, f[1], s5 * vr[1]));
  c[2] += gbi_fmac(m3, f[2], s5 * vr[2]);
}

// Source records: 0..2 position, 3..5 F, 6..14 Dt, 15..17 a, 18..23 2 H, 24..26 2 E, 27..29 2 c,
// 30 tr Dt + 2 E_3, 31 2 tr H -- formed in FP64 and rounded to T.
template <typename T>
__global__ void k_wall_records(int N, double a, double eta, const double* __restrict__ R,
                               const double* __restrict__ VH, int h, const double* __restrict__ Fe,
                               const double* __restrict__ Te, T* __restrict__ rec) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= N) return;
  T* o = rec + (size_t)m * kWallRec;
  const double cs = (20.0 / 3.0) * kPi * eta * a * a;
  double s6[6];   // xx xy xz yy yz zz of the packed V^(2s)
  gbi_unpack2<double>(VH + (size_t)h * m, s6);
  const double S[9] = {s6[0], s6[1], s6[2], s6[1], s6[3], s6[4], s6[2], s6[4], s6[5]};
  const double T0 = Te[3 * (size_t)m], T1 = Te[3 * (size_t)m + 1], T2 = Te[3 * (size_t)m + 2];
  // D = S + A, A_jk = (1/2) eps_kjl T_l
  const double A[9] = {0.0, -0.5 * T2, 0.5 * T1, 0.5 * T2, 0.0, -0.5 * T0, -0.5 * T1, 0.5 * T0, 0.0};
  const double sg[3] = {1.0, 1.0, -1.0};
  const double y3 = R[3 * (size_t)m + 2];
  double F[3], D[9], Dt[9], E[3], Hf[9];
  for (int k = 0; k < 3; ++k) F[k] = Fe[3 * (size_t)m + k];
  for (int q = 0; q < 9; ++q) D[q] = cs * S[q] + A[q];
  for (int j = 0; j < 3; ++j) {
    for (int k = 0; k < 3; ++k) {
      Dt[3 * j + k] = -sg[k] * D[3 * j + k];
      Hf[3 * j + k] = y3 * sg[j] * Dt[3 * j + k];
    }
    E[j] = sg[j] * (y3 * F[j] + D[3 * j + 2]);
  }
  for (int k = 0; k < 3; ++k) {
    o[k] = T(R[3 * (size_t)m + k]);
    o[3 + k] = T(F[k]);
    o[24 + k] = T(2.0 * E[k]);
    o[27 + k] = T(2.0 * Hf[6 + k]);
  }
  for (int q = 0; q < 9; ++q) o[6 + q] = T(Dt[q]);
  o[15] = T(Dt[5] - Dt[7]);
  o[16] = T(Dt[6] - Dt[2]);
  o[17] = T(Dt[1] - Dt[3]);
  o[18] = T(2.0 * Hf[0]);
  o[19] = T(Hf[1] + Hf[3]);
  o[20] = T(Hf[2] + Hf[6]);
  o[21] = T(2.0 * Hf[4]);
  o[22] = T(Hf[5] + Hf[7]);
  o[23] = T(2.0 * Hf[8]);
  o[30] = T(Dt[0] + Dt[4] + Dt[8] + 2.0 * E[2]);
  o[31] = T(2.0 * (Hf[0] + Hf[4] + Hf[8]));
}

// Partial image sums of the targets over the sources of slice blockIdx.y.
template <typename T>
__global__ void __launch_bounds__(kWallThreads) k_wall_pairs(int N, int per_slice, const T* __restrict__ rec,
                                                             T* __restrict__ part) {
  __shared__ __align__(32) T s_rec[kWallTile * kWallRec];
  const int n = blockIdx.x * kWallThreads + threadIdx.x;
  const int m0 = blockIdx.y * per_slice;
  const int m1 = min(N, m0 + per_slice);
  T x[3] = {T(0), T(0), T(0)};
  if (n < N)
    for (int k = 0; k < 3; ++k) x[k] = rec[(size_t)n * kWallRec + k];
  T u[3] = {T(0), T(0), T(0)}, c[3] = {T(0), T(0), T(0)};
  for (int base = m0; base < m1; base += kWallTile) {
    const int len = min(kWallTile, m1 - base);
    __syncthreads();
    for (int q = threadIdx.x; q < len * kWallRec; q += kWallThreads) s_rec[q] = rec[(size_t)base * kWallRec + q];
    __syncthreads();
    if (n < N)
      for (int j = 0; j < len; ++j) wall_image_pair<T>(x, s_rec + j * kWallRec, u, c);
  }
  if (n < N) {
    T* o = part + ((size_t)blockIdx.y * N + n) * 6;
    for (int k = 0; k < 3; ++k) {
      o[k] = u[k];
      o[3 + k] = c[k];
    }
  }
}

// V += u / (8 pi eta), Omega += c / (16 pi eta), the slices added in order.
// One thread per (sphere, component), component fastest, eight slices' loads in flight.
template <typename T>
__global__ void k_wall_reduce(int N, int slices, double eta, const T* __restrict__ part, double* V, double* Om) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long rows = 6LL * N;
  if (i >= rows) return;
  const long long n = i / 6;
  const int c = (int)(i - 6 * n);
  double acc = 0.0;
  for (int q = 0; q < slices; q += 8) {
    T p[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) p[k] = q + k < slices ? part[(long long)(q + k) * rows + i] : T(0);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (q + k < slices) acc += double(p[k]);
  }
  const double f = 1.0 / (8.0 * kPi * eta);
  if (c < 3) V[3 * n + c] += f * acc;
  else Om[3 * n + c - 3] += 0.5 * f * acc;
}

int wall_slices(int N) {
  // about four blocks per SM on 152 SMs, at least 8 sources per slice: at small N the slices
  // are the only parallelism, and a source costs a thread a chain of dependent operations
  const int tb = (N + kWallThreads - 1) / kWallThreads;
  int s = (608 + tb - 1) / tb;
  const int maxs = (N + 7) / 8;
  if (s > maxs) s = maxs;
  return s < 1 ? 1 : s;
}

template <typename T>
cudaError_t launch_wall_t(int N, double a, double eta, const double* R, const double* VH, int h, const double* Fe,
                          const double* Te, double* V, double* Om, void* scratch, cudaStream_t st) {
  T* rec = static_cast<T*>(scratch);
  const int slices = wall_slices(N);
  const int per = (N + slices - 1) / slices;
  T* part = rec + (size_t)N * kWallRec;
  k_wall_records<T><<<(N + 255) / 256, 256, 0, st>>>(N, a, eta, R, VH, h, Fe, Te, rec);
  k_wall_pairs<T><<<dim3((N + kWallThreads - 1) / kWallThreads, slices), kWallThreads, 0, st>>>(N, per, rec, part);
  k_wall_reduce<T><<<(unsigned)((6LL * N + 127) / 128), 128, 0, st>>>(N, slices, eta, part, V, Om);
  return cudaGetLastError();
}

size_t wall_scratch_bytes(int N, bool fp32) {
  const size_t w = fp32 ? sizeof(float) : sizeof(double);
  return w * ((size_t)N * kWallRec + (size_t)wall_slices(N) * N * 6) + 256;
}

}  // namespace
}  // namespace gbi

using namespace gbi;

extern "C" gbi_status gbi_wall_superpose(gbi_ctx* ctx, const gbi_params* prm, int N, const double* R,
                                         const double* Va, const double* Oa, const double* VH, const double* Fe,
                                         const double* Te, double* V, double* Omega) {
  if (!ctx || !valid_params(prm) || N < 0 || prm->trunc != 2) return GBI_ERR_ARG;
  if (N == 0) return GBI_OK;
  if (!R || !Va || !Oa || !VH || !Fe || !Te || !V || !Omega) return GBI_ERR_ARG;
  // the unbounded superposition first (direct pairs with their finite-size terms)
  GBI_TRY(gbi_superpose(ctx, prm, N, R, Va, Oa, VH, Fe, Te, V, Omega));
  cudaSetDevice(ctx->device);
  const bool fp32 = prm->precision != 0 && prm->precision != 2;
  GBI_TRY(ensure(ctx, ctx->wallbuf, wall_scratch_bytes(N, fp32)));
  const int h = gbi_h(prm->trunc);
  const double flops = double(kWallPairFlops) * double(N) * double(N);
  const cudaError_t e = timed(ctx, fp32 ? 32 : 31, flops, 3, [&] {
    return fp32 ? launch_wall_t<float>(N, prm->a, prm->eta, R, VH, h, Fe, Te, V, Omega, ctx->wallbuf.p, ctx->stream)
                : launch_wall_t<double>(N, prm->a, prm->eta, R, VH, h, Fe, Te, V, Omega, ctx->wallbuf.p,
                                        ctx->stream);
  });
  GBI_CHECK(e);
  return GBI_OK;
}
