// Forward-Euler superposition steps of one suspension in a trap (Sec. V, Eq. trap_eom) at l <= 2
// in FP32: what gbi_trap_step / gbi_squirmer_step run with superposition set.
//
// In these steps the forcing is F = -k R and no torque, and the active modes are V^(2s) = s0 (pp -
// I/3) and V^(3t) = d0 p, so the pair sum of trap_kernel.cu loses its torque terms (and, with d0 =
// 0, the potential dipole).  With rho = R_n - R_m, F and S divided by 8 pi eta, d = (a^3/10) V^(32):
//   V_n += (1/r + 2a^2/(3r^3)) F - (16/5) a^2 S.rho/r^5 - d/r^3
//        + [ (1/r^3 - 2a^2/r^5)(rho.F) + (8a^2/r^7 - 3/r^5)(rho.S.rho) + 3 (rho.d)/r^5 ] rho
//   Omega_n += (F x rho)/r^3 + 3 rho x (S.rho)/r^5
// -- 65 floating-point instructions per pair (72 with the dipole) against 86 in general.  The
// operations that stay keep trap_pairs_f2's order, so a pair's terms are the same bits: where
// squirmers overlap, one pair's terms are so large that their last bits show in the orbits.  (The
// form (F/r^3 - 3 S.rho/r^5) x rho would save six more; its orientations after four steps of 10^4
// squirmers, with closest pairs at 0.2 a, differed by 1.1e-9.)
//
// A step is two kernels: the pair sums, and one that adds the splits, moves the spheres and
// writes the next step's source records (the general call sequence: six).  Up to kStepsSmall
// spheres one block runs all the steps in one launch.  Microseconds a step, before -> now:
// N = 2: 26.7 -> 2.0, 64: 44 -> 7.8, 128: 45 -> 14.7, 1000: 53 -> 16.5, 10^4: 348 -> 256 (pairs 310 -> 242).
#include <cuda_runtime.h>

#include <type_traits>

#include "ctx.cuh"
#include "f2.cuh"

namespace gbi {
namespace {

struct StepPar {
  int N;
  double a, dt, k, vs;
  double i8;     // 1 / (8 pi eta): F / (8 pi eta) = (-k R) i8
  double ss;     // S / (8 pi eta) = ss (pp - |p|^2/3 I)   (-(5/6) a^2 s0)
  double ds;     // d = ds (d0 p)   (a^3 / 10)
  double d0;
  double mt;     // V += mt F (one body): 1/(6 pi eta a)
};

// Source record: hi (3), lo (3) of the centre, F (3), S xx xy xz yy yz zz (6), d (3) with the
// dipole; padded to whole 16-byte words
template <bool DIP> struct StepRec { static constexpr int W = DIP ? 20 : 16; };

template <bool DIP>
__device__ __forceinline__ void step_record(const StepPar& c, const double* R, const double* p, float* r) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float h = float(R[i]);
    r[i] = h;
    r[3 + i] = float(R[i] - double(h));
    r[6 + i] = float((-c.k * R[i]) * c.i8);
  }
  const double xx = p[0] * p[0], yy = p[1] * p[1], zz = p[2] * p[2];
  const double t = (xx + yy + zz) * (1.0 / 3.0);
  r[9] = float(c.ss * (xx - t));
  r[10] = float(c.ss * (p[0] * p[1]));
  r[11] = float(c.ss * (p[0] * p[2]));
  r[12] = float(c.ss * (yy - t));
  r[13] = float(c.ss * (p[1] * p[2]));
  r[14] = float(c.ss * (zz - t));
  r[15] = 0.f;
  if constexpr (DIP) {
    r[15] = float(c.ds * (c.d0 * p[0]));
    r[16] = float(c.ds * (c.d0 * p[1]));
    r[17] = float(c.ds * (c.d0 * p[2]));
    r[18] = r[19] = 0.f;
  }
}

// constants of the radius
template <typename T> struct StepC {
  T c23, c2a, c8a, c165;
  __device__ __forceinline__ explicit StepC(double a) {
    const float a2 = float(a * a);
    c23 = T((2.0f / 3.0f) * a2);
    c2a = T(-2.0f * a2);
    c8a = T(8.0f * a2);
    c165 = T((-16.0f / 5.0f) * a2);
  }
};

// The pair terms of source q (record words) on targets with centre parts ph, pl; dead(ri) zeroes
// 1/r of a target's own sphere, whose rho is exactly 0 (every term is then a product with 0).
template <bool DIP, typename T, typename K>
__device__ __forceinline__ void step_pair(const T* q, const T* ph, const T* pl, const StepC<T>& c, T* v, T* w, K&& dead) {
  const T x = (ph[0] - q[0]) + (pl[0] - q[3]);
  const T y = (ph[1] - q[1]) + (pl[1] - q[4]);
  const T z = (ph[2] - q[2]) + (pl[2] - q[5]);
  const T r2 = fma2(z, z, fma2(y, y, x * x));
  T ri = rsqrt2(r2);
  dead(ri);
  const T ri2 = ri * ri, ri3 = ri * ri2, ri5 = ri3 * ri2, ri7 = ri5 * ri2;
  const T *F = q + 6, *S = q + 9;
  const T rF = fma2(z, F[2], fma2(y, F[1], x * F[0]));
  const T sx = fma2(S[2], z, fma2(S[1], y, S[0] * x));
  const T sy = fma2(S[4], z, fma2(S[3], y, S[1] * x));
  const T sz = fma2(S[5], z, fma2(S[4], y, S[2] * x));
  const T rSr = fma2(z, sz, fma2(y, sy, x * sx));
  const T c1 = fma2(c.c23, ri3, ri);
  const T t3 = T(3.0f) * ri5;
  T cx = fma2(c.c8a, ri7, -t3);
  if constexpr (DIP) cx = fma2(cx, rSr, t3 * fma2(z, q[17], fma2(y, q[16], x * q[15])));
  else cx = cx * rSr;
  cx = fma2(fma2(c.c2a, ri5, ri3), rF, cx);
  const T cs = c.c165 * ri5;
  v[0] = fma2(cs, sx, fma2(cx, x, fma2(c1, F[0], v[0])));
  v[1] = fma2(cs, sy, fma2(cx, y, fma2(c1, F[1], v[1])));
  v[2] = fma2(cs, sz, fma2(cx, z, fma2(c1, F[2], v[2])));
  if constexpr (DIP) {
    v[0] = fma2(ri3, -q[15], v[0]);
    v[1] = fma2(ri3, -q[16], v[1]);
    v[2] = fma2(ri3, -q[17], v[2]);
  }
  const T e0 = fma2(F[1], z, -F[2] * y), e1 = fma2(F[2], x, -F[0] * z), e2 = fma2(F[0], y, -F[1] * x);
  const T tx = t3 * x, ty = t3 * y, tz = t3 * z;
  w[0] = fma2(ty, sz, fma2(-tz, sy, fma2(ri3, e0, w[0])));
  w[1] = fma2(tz, sx, fma2(-tx, sz, fma2(ri3, e1, w[1])));
  w[2] = fma2(tx, sy, fma2(-ty, sx, fma2(ri3, e2, w[2])));
}

// R, p of one sphere moved by dt with V = vs p + mt F + dv, Omega = dw (the FP64 pair sums)
__device__ __forceinline__ void step_move(const StepPar& c, const double* dv, const double* dw, double* R, double* p) {
#pragma unroll
  for (int i = 0; i < 3; ++i) R[i] += c.dt * (c.vs * p[i] + c.mt * (-c.k * R[i]) + dv[i]);
  const double qx = p[0] + c.dt * (dw[1] * p[2] - dw[2] * p[1]);
  const double qy = p[1] + c.dt * (dw[2] * p[0] - dw[0] * p[2]);
  const double qz = p[2] + c.dt * (dw[0] * p[1] - dw[1] * p[0]);
  const double inv = rsqrt(qx * qx + qy * qy + qz * qz);
  p[0] = qx * inv;
  p[1] = qy * inv;
  p[2] = qz * inv;
}

template <bool DIP>
__global__ void k_steps_records(const StepPar c, const double* __restrict__ R, const double* __restrict__ p,
                                float* __restrict__ rec) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= c.N) return;
  step_record<DIP>(c, R + 3 * (size_t)n, p + 3 * (size_t)n, rec + (size_t)n * StepRec<DIP>::W);
}

// Pair sums of the sources [blockIdx.y chunk, + chunk) for 2 kStepTG targets per thread, two at a
// time in paired instructions; the tile's records sit in shared memory with every word doubled,
// so that one 16-byte load gives two broadcast operands (as trap_pairs_f2).
// (The sources are split and added up as in trap_kernel.cu, so the sums are the same bits.)  Up to
// kStepsNarrow spheres, where that leaves a few blocks (N = 1000: 32), the block is one warp with two
// targets per thread; us a step: N = 1900 24.5, 2048 25.0, then 2049 with the wide block 39.6, 3000 41.2 (the general
// sequence 57, 56, 70, 74), so the narrow one still wins at this limit.
constexpr int kStepTile = 128;
constexpr int kStepsNarrow = 2048;

template <bool DIP, int kStepThreads, int kStepTG, int kMinBlocks>
__global__ void __launch_bounds__(kStepThreads, kMinBlocks)
    k_steps_pairs(const StepPar c, const float* __restrict__ rec, int chunk, float* __restrict__ partial) {
  constexpr int W = StepRec<DIP>::W, TI = 2 * kStepTG;
  pdl_wait();
  __shared__ __align__(16) float4 s_dup[kStepTile * W / 2];
  const int N = c.N;
  const int n0 = (blockIdx.x * kStepThreads + threadIdx.x) * TI;
  const int m_begin = blockIdx.y * chunk, m_end = min(N, m_begin + chunk);
  const int blk0 = blockIdx.x * kStepThreads * TI, blk1 = blk0 + kStepThreads * TI;
  const StepC<f2> k(c.a);
  f2 ph[kStepTG][3], pl[kStepTG][3], v[kStepTG][3], w[kStepTG][3];
#pragma unroll
  for (int g = 0; g < kStepTG; ++g) {
    const float* ra = rec + (size_t)min(n0 + 2 * g, N - 1) * W;
    const float* rb = rec + (size_t)min(n0 + 2 * g + 1, N - 1) * W;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      ph[g][i] = f2(ra[i], rb[i]);
      pl[g][i] = f2(ra[3 + i], rb[3 + i]);
      v[g][i] = w[g][i] = f2(0.f);
    }
  }
  for (int base = m_begin; base < m_end; base += kStepTile) {
    const int len = min(kStepTile, m_end - base);
    __syncthreads();
    const float2* src = reinterpret_cast<const float2*>(rec + (size_t)base * W);
    for (int i = threadIdx.x; i < len * (W / 2); i += kStepThreads) {
      const float2 t = src[i];
      s_dup[i] = make_float4(t.x, t.x, t.y, t.y);
    }
    __syncthreads();
    // only a tile that holds one of this block's targets can hold a thread's own sphere
    const bool self = base < blk1 && base + len > blk0;
    auto tile = [&](auto own) {
      for (int j = 0; j < len; ++j) {
        f2 q[W];
        const float4* r4 = s_dup + j * (W / 2);
#pragma unroll
        for (int i = 0; i < W / 2; ++i) {
          const float4 t = r4[i];
          q[2 * i] = f2(t.x, t.y);
          q[2 * i + 1] = f2(t.z, t.w);
        }
#pragma unroll
        for (int g = 0; g < kStepTG; ++g)
          step_pair<DIP>(q, ph[g], pl[g], k, v[g], w[g], [&](f2& ri) {
            if constexpr (decltype(own)::value) {
              if (base + j == n0 + 2 * g) ri.v.x = 0.f;
              if (base + j == n0 + 2 * g + 1) ri.v.y = 0.f;
            }
          });
      }
    };
    if (self) tile(std::true_type{});
    else tile(std::false_type{});
  }
#pragma unroll
  for (int t = 0; t < TI; ++t) {
    const int n = n0 + t;
    if (n < N) {
      float* o = partial + ((size_t)blockIdx.y * N + n) * 6;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        o[i] = (t & 1) ? v[t >> 1][i].v.y : v[t >> 1][i].v.x;
        o[3 + i] = (t & 1) ? w[t >> 1][i].v.y : w[t >> 1][i].v.x;
      }
    }
  }
}

// The splits' sums in order (FP64, one thread per sphere and component, eight loads in flight),
// then one thread per sphere moves it and writes its next record.
constexpr int kMoveSpheres = 32;

template <bool DIP>
__global__ void __launch_bounds__(6 * kMoveSpheres)
    k_steps_move(const StepPar c, const float* __restrict__ partial, int nsplit, double* __restrict__ R,
                 double* __restrict__ p, float* __restrict__ rec) {
  pdl_wait();
  __shared__ double s_sum[kMoveSpheres * 6];
  const long long rows = 6LL * c.N;
  const long long i = (long long)blockIdx.x * (6 * kMoveSpheres) + threadIdx.x;
  double acc = 0.0;
  if (i < rows) {
    for (int s = 0; s < nsplit; s += 8) {
      float q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = s + u < nsplit ? partial[(long long)(s + u) * rows + i] : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (s + u < nsplit) acc += double(q[u]);
    }
  }
  s_sum[threadIdx.x] = acc;
  __syncthreads();
  const int n = blockIdx.x * kMoveSpheres + threadIdx.x;
  if (threadIdx.x >= kMoveSpheres || n >= c.N) return;
  double Rn[3], pn[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    Rn[q] = R[3 * (size_t)n + q];
    pn[q] = p[3 * (size_t)n + q];
  }
  step_move(c, s_sum + 6 * threadIdx.x, s_sum + 6 * threadIdx.x + 3, Rn, pn);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    R[3 * (size_t)n + q] = Rn[q];
    p[3 * (size_t)n + q] = pn[q];
  }
  step_record<DIP>(c, Rn, pn, rec + (size_t)n * StepRec<DIP>::W);
}

// All the steps of a small suspension in one block.  Four lanes per sphere hold its centre and
// orientation, one component each (the fourth idles): an FP64 instruction takes the SM's pipe 16
// cycles and its result 64, whatever the lanes, so the update and the next record are written
// with the components side by side.  A target's sources are summed one after the other, as in
// trap_kernel.cu, so that orbits with close encounters, which amplify a last bit by ten thousand within
// fifty steps, stay the same; V and Omega are summed by different threads.  (Several lanes per target added
// in FP64 took 8.3 us at N = 64 and left R 8e-9 off.)  A step is bound by the latency of the pair sums and of the
// FP64 chain from them to the next record: 2.0 us at N = 2, 4.8 at 32, 7.8 at 64, 8.1 at 72; the two kernels take
// 11.0 at 73.  It still wins at this limit, up to which two splits hold every target's sources.
constexpr int kSmallThreads = 512;
constexpr int kStepsSmall = 72;

template <bool DIP>
__global__ void __launch_bounds__(kSmallThreads)
    k_steps_small(const StepPar c, int nsteps, int G, int chunk, int half, double* __restrict__ R,
                  double* __restrict__ p) {
  constexpr int W = StepRec<DIP>::W;
  constexpr unsigned int kAll = 0xffffffffu;
  __shared__ __align__(16) float s_rec[kStepsSmall * W];
  __shared__ float s_part[2][kStepsSmall][6];
  const int tid = threadIdx.x, N = c.N;
  // the sums' threads: split `sub` of target n, the velocity in the first part of the block, the
  // angular velocity in the second
  const bool angular = tid >= half;
  const int item = angular ? tid - half : tid, n = item / G, sub = item - n * G;
  const StepC<float> k(c.a);
  // the state's lanes: sphere tid / 4, component tid % 4
  const bool owner = (tid & ~31) < 4 * N;   // the whole warp takes part in the exchanges
  const int on = min(tid >> 2, N - 1), oc = min(tid & 3, 2);
  const bool live = tid < 4 * N && (tid & 3) < 3;
  const int l0 = (tid & 31) & ~3, l1 = l0 + (oc == 2 ? 0 : oc + 1), l2 = l0 + (oc == 0 ? 2 : oc - 1);
  const int c1 = oc == 2 ? 0 : oc + 1, c2 = oc == 0 ? 2 : oc - 1;
  double Rc = 0.0, pc = 0.0;
  float* my = s_rec + on * W;
  auto record = [&]() {
    const double p1 = __shfl_sync(kAll, pc, l1);
    const double sq = pc * pc;
    const double s0 = __shfl_sync(kAll, sq, l0), s1 = __shfl_sync(kAll, sq, l0 + 1), s2 = __shfl_sync(kAll, sq, l0 + 2);
    const double t = (s0 + s1 + s2) * (1.0 / 3.0);
    if (!live) return;
    const float hi = float(Rc);
    my[oc] = hi;
    my[3 + oc] = float(Rc - double(hi));
    my[6 + oc] = float((-c.k * Rc) * c.i8);
    my[oc == 0 ? 9 : (oc == 1 ? 12 : 14)] = float(c.ss * (sq - t));
    my[oc == 0 ? 10 : (oc == 1 ? 13 : 11)] = float(c.ss * (pc * p1));
    if constexpr (DIP) my[15 + oc] = float(c.ds * (c.d0 * pc));
  };
  if (owner) {
    Rc = R[3 * on + oc];
    pc = p[3 * on + oc];
    record();
  }
  for (int step = 0; step < nsteps; ++step) {
    __syncthreads();
    if (n < N) {
      float ph[3], pl[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        ph[q] = s_rec[n * W + q];
        pl[q] = s_rec[n * W + 3 + q];
      }
      const int m0 = sub * chunk, m1 = min(N, m0 + chunk);
      // both sums of every source; the one that a thread does not keep drops out
      auto sum = [&](float* v, float* w) {
#pragma unroll 2
        for (int m = m0; m < m1; ++m) {
          float q[W];
          const float4* r4 = reinterpret_cast<const float4*>(s_rec + m * W);
#pragma unroll
          for (int i = 0; i < W / 4; ++i) {
            const float4 t = r4[i];
            q[4 * i] = t.x;
            q[4 * i + 1] = t.y;
            q[4 * i + 2] = t.z;
            q[4 * i + 3] = t.w;
          }
          step_pair<DIP>(q, ph, pl, k, v, w, [&](float& ri) {
            if (m == n) ri = 0.f;
          });
        }
      };
      float v[3] = {0.f, 0.f, 0.f}, w[3] = {0.f, 0.f, 0.f};
      float* o = s_part[sub][n] + (angular ? 3 : 0);
      if (angular) {
        sum(v, w);
        o[0] = w[0], o[1] = w[1], o[2] = w[2];
      } else {
        sum(v, w);
        o[0] = v[0], o[1] = v[1], o[2] = v[2];
      }
    }
    __syncthreads();
    if (owner) {
      // step_move, a component per lane
      // (the splits' sums in order)
      auto total = [&](int q) {
        double t = double(s_part[0][on][q]);
        if (G > 1) t += double(s_part[1][on][q]);
        return t;
      };
      const double p1 = __shfl_sync(kAll, pc, l1), p2 = __shfl_sync(kAll, pc, l2);
      Rc += c.dt * (c.vs * pc + c.mt * (-c.k * Rc) + total(oc));
      const double q = pc + c.dt * (total(3 + c1) * p2 - total(3 + c2) * p1);
      const double sq = q * q;
      const double s0 = __shfl_sync(kAll, sq, l0), s1 = __shfl_sync(kAll, sq, l0 + 1), s2 = __shfl_sync(kAll, sq, l0 + 2);
      pc = q * rsqrt(s0 + s1 + s2);
      record();
    }
  }
  if (live) {
    R[3 * on + oc] = Rc;
    p[3 * on + oc] = pc;
  }
}

template <bool DIP>
gbi_status run_steps(gbi_ctx* ctx, const StepPar& c, int nsteps, double* R, double* p) {
  constexpr int W = StepRec<DIP>::W;
  // per pair: rho 9, r^2 5, rsqrt 1, powers 4, rho.F 5, S.rho 15, rho.S.rho 5, coefficients 11, V 18, Omega 30;
  // the dipole 13 more
  const double flops = (DIP ? 116.0 : 103.0) * double(c.N) * double(c.N - 1);
  const int ns = trap_splits(c.N, 1), chunk = (c.N + ns - 1) / ns;   // at most 2 splits up to kStepsSmall
  if (c.N <= kStepsSmall) {
    const int half = (c.N * ns + 31) / 32 * 32;   // threads of one kind of sum
    const int threads = half + half > 4 * c.N ? half + half : (4 * c.N + 31) / 32 * 32;
    // a launch stays below 40 ms (4096 steps of 72 spheres: 33)
    for (int done = 0; done < nsteps; done += 4096) {
      const int n = nsteps - done < 4096 ? nsteps - done : 4096;
      GBI_CHECK(timed(ctx, 28, n * flops, 1, [&] {
        k_steps_small<DIP><<<1, threads, 0, ctx->stream>>>(c, n, ns, chunk, half, R, p);
        return cudaGetLastError();
      }));
    }
    return GBI_OK;
  }
  GBI_TRY(ensure(ctx, ctx->trapbuf, sizeof(float) * ((size_t)c.N * W + (size_t)ns * c.N * 6)));
  float* rec = P<float>(ctx->trapbuf);
  float* partial = rec + (size_t)c.N * W;
  const unsigned move = (unsigned)((c.N + kMoveSpheres - 1) / kMoveSpheres);
  k_steps_records<DIP><<<grid1(c.N, 128), 128, 0, ctx->stream>>>(c, R, p, rec);
  ++ctx->launches;
  GBI_CHECK(cudaGetLastError());
  const float* crec = rec;
  const float* cpart = partial;
  for (int s = 0; s < nsteps; ++s) {
    GBI_CHECK(timed(ctx, 28, flops, 1, [&] {
      if (c.N <= kStepsNarrow)
        return launch_pdl(ctx->pdl && !ctx->prof, dim3((c.N + 63) / 64, ns), dim3(32), ctx->stream,
                          k_steps_pairs<DIP, 32, 1, 16>, c, crec, chunk, partial);
      return launch_pdl(ctx->pdl && !ctx->prof, dim3((c.N + 511) / 512, ns), dim3(128), ctx->stream,
                        k_steps_pairs<DIP, 128, 2, 4>, c, crec, chunk, partial);
    }));
    GBI_CHECK(launch_pdl(ctx->pdl && !ctx->prof, dim3(move), dim3(6 * kMoveSpheres), ctx->stream, k_steps_move<DIP>, c,
                         cpart, ns, R, p, rec));
    ++ctx->launches;
  }
  return GBI_OK;
}

}  // namespace

gbi_status superposition_steps(gbi_ctx* ctx, const gbi_params* prm, int N, double dt, double k_trap, double vs,
                               double s0, double d0, int nsteps, double* R, double* p) {
  const double a = prm->a, i8 = 1.0 / (8.0 * kPi * prm->eta);
  StepPar c;
  c.N = N;
  c.a = a;
  c.dt = dt;
  c.k = k_trap;
  c.vs = vs;
  c.i8 = i8;
  c.ss = -(5.0 / 6.0) * a * a * s0;
  c.ds = a * a * a / 10.0;
  c.d0 = d0;
  c.mt = 1.0 / (6.0 * kPi * prm->eta * a);
  return d0 != 0.0 ? run_steps<true>(ctx, c, nsteps, R, p) : run_steps<false>(ctx, c, nsteps, R, p);
}

}  // namespace gbi
