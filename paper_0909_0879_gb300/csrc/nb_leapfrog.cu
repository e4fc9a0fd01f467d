// Differentiable leapfrog: the paper's second-order symplectic integrator
// (Sec. 3.1, kick-drift-kick form) in FP32 on the GPU, with a hand-written
// adjoint of the force sum and a checkpointed reverse pass.
//
// Force (acceleration only):  a_i = G sum_{j != i} m_j d / s^3,
//   d = x_j - x_i, s^2 = |d|^2 + eps^2.
// Adjoint of the force map for a cotangent g_i = dL/da_i, with the softened
// tidal tensor T(d) = I / s^3 - 3 d d^T / s^5 (symmetric, even in d):
//   dL/dx_k = G sum_{j != k} T(x_j - x_k) (m_k g_j - m_j g_k)
//   dL/dm_k = G sum_{i != k} g_i . (x_k - x_i) / s_ik^3
// Both sums are i-parallel: several lanes split a particle's j-range and meet
// by a warp-shuffle butterfly, so the results do not depend on launch order.
// The i == j term is exactly zero for eps > 0 and masked for eps == 0.
//
// Reverse of one KDK step (x, v) -> (x', v'):
//   v_h = v + A(x) dt/2, x' = x + v_h dt, v' = v_h + A(x') dt/2
//   lv_h = lv'; (lx', lm) += vjp_A(x'; lv' dt/2); lv_h += lx' dt;
//   (lx, lm) += vjp_A(x; lv_h dt/2); lx = lx', lv = lv_h
// The first kick of a step and the second kick of the step before it meet at
// the same x and lv, so a reverse pass takes one vjp_A(x; lv dt) there: n + 1
// of them for n steps.  The forward pass stores (x, v) every `ckpt_every`
// steps; the reverse pass re-runs each segment from its checkpoint, keeping
// the segment's positions, then walks it backwards.
#include "../../include/nbody.h"
#include "nb_device.cuh"

#include <algorithm>
#include <cmath>

namespace nbi {
namespace {

constexpr int kLfT = 256;              // threads per CTA, wide shape
constexpr int kLfJT = 256;             // j-records per shared tile, wide shape

// Small and middle N.  A particle's sum runs over eight chains of every
// eighth record.  A group of four warps holds 32 particles, one per lane;
// each warp takes two chains, side by side in packed FP32x2 instructions, so
// that a pair of records is one shared-memory broadcast.  The elementwise
// work around a force (kicks, drift, checkpoint) is done by the CTA that holds
// the particles, so a step is one launch.  Records come in tiles by
// asynchronous copies, the next tile while the current one is summed, stored
// in pairs so that a packed instruction takes two of them without a move.
// Measured per evaluation, N = 1,000 / 4,096 / 16,000 / 60,000: 6.5 / 16.7 / 132
// / 1,612 us (eight threads per particle, synchronous tile loads: 8.3 / 21.3 /
// 162 / 1,784, and a second launch for the step).  At N = 4,096 the eight
// chains leave one warp per scheduler, whose latencies set the time.  Lanes
// that split a particle's records, with one, two or four particles per lane,
// give 18.7 / 16.7 / - us at N = 4,096 and 1,860 / 1,786 / 1,763 at 60,000;
// programmatic dependent launch stacks waiting CTAs on some SMs (22 us).
constexpr int kLfTile = 512;
constexpr int kLfVjpTile = 1024;
constexpr int kLfAccWarps = 4;  // warps of a group of 32 particles
constexpr int kLfVjpTpi = 64;   // threads of a particle pair: vector-Jacobian product
constexpr int kLfMaxThreads = 512, kLfVjpMaxThreads = 1024;

__device__ __forceinline__ float2 dup(float s) { return make_float2(s, s); }

template <int MASK>
__device__ __forceinline__ float2 lf_rsq2(float2 s2) {
  float2 r;
  r.x = MASK ? (s2.x > 0.f ? rsqrtf(s2.x) : 0.f) : rsqrtf(s2.x);
  r.y = MASK ? (s2.y > 0.f ? rsqrtf(s2.y) : 0.f) : rsqrtf(s2.y);
  return r;
}

// A rounded packed product that no following addition is fused with.
__device__ __forceinline__ float2 mul2_alone(float2 a, float2 b) {
  float2 c;
  asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "mul.rn.f32x2 c, a, b;\n\tmov.b64 {%0, %1}, c;\n\t}"
      : "=f"(c.x), "=f"(c.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return c;
}

// Asynchronous copy of one float, completed by copies_wait().
__device__ __forceinline__ void copy_float(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void copies_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int LEFT>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// Queue the copies of records (x, y, z, w) of a tile, w from m;
// past the end: no mass, far away.
__device__ __forceinline__ void stage_xm(float4 *t, int64_t j0, int64_t n, const float *x,
                                         const float *m) {
  for (int r = threadIdx.x; r < kLfVjpTile; r += blockDim.x) {
    const int64_t j = j0 + r;
    float *const d = reinterpret_cast<float *>(t + r);
    if (j < n) {
#pragma unroll
      for (int c = 0; c < 3; ++c) copy_float(d + c, x + 3 * j + c);
      copy_float(d + 3, m + j);
    } else {
      t[r] = make_float4(1.0e15f, 1.0e15f, 1.0e15f, 0.f);
    }
  }
}
// The same in pairs: planes of (x0 x1 y0 y1) and (z0 z1 m0 m1), kLfTile / 2
// each.
__device__ __forceinline__ void stage_pairs(float4 *t, int64_t j0, int64_t n, const float *x,
                                            const float *m) {
  for (int r = threadIdx.x; r < kLfTile; r += blockDim.x) {
    const int64_t j = j0 + r;
    float *const xy = reinterpret_cast<float *>(t) + 4 * (r >> 1) + (r & 1);
    float *const zm = xy + 2 * kLfTile;
    if (j < n) {
      copy_float(xy, x + 3 * j);
      copy_float(xy + 2, x + 3 * j + 1);
      copy_float(zm, x + 3 * j + 2);
      copy_float(zm + 2, m + j);
    } else {
      xy[0] = xy[2] = zm[0] = 1.0e15f;
      zm[2] = 0.f;
    }
  }
}
// The same for cotangents (zero past the end).
__device__ __forceinline__ void stage_g(float4 *t, int64_t j0, int64_t n, const float *g) {
  for (int r = threadIdx.x; r < kLfVjpTile; r += blockDim.x) {
    const int64_t j = j0 + r;
    float *const d = reinterpret_cast<float *>(t + r);
    if (j < n) {
#pragma unroll
      for (int c = 0; c < 3; ++c) copy_float(d + c, g + 3 * j + c);
    } else {
      t[r] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

// What follows a force evaluation, per element: with close, the kick v += a
// h that ends the previous step; then, when ck is set, the checkpoint (x, v)
// of the step boundary; then, when x_out is set, this step's opening kick v +=
// a h and the drift x_out = x + v dt.  acc (may be null) receives a.
struct LfTail {
  const float *v_in = nullptr;
  float *v_out = nullptr;
  float *x_out = nullptr;
  float *acc = nullptr;
  float *ck = nullptr;
  int close = 0;
  float h = 0.f, dt = 0.f;
};

template <int MASK>
__global__ void __launch_bounds__(kLfMaxThreads)
    lf_eval_kernel(int64_t n, int per_cta, const float *__restrict__ x,
                   const float *__restrict__ m, float eps2, float G, const LfTail T) {
  __shared__ float4 tiles[2][kLfTile];
  __shared__ float part[kLfMaxThreads][3];
  constexpr int kPairs = kLfTile / 2;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r = wid % kLfAccWarps;  // the warp's chains
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * per_cta;
  const int64_t i = i0 + wid / kLfAccWarps * 32 + lane;
  const int64_t ii = i < n ? i : 0;
  const float2 nx = dup(-x[3 * ii]), ny = dup(-x[3 * ii + 1]), nz = dup(-x[3 * ii + 2]);
  const float2 e2 = dup(eps2);
  float2 px = dup(0.f), py = px, pz = px;
  stage_pairs(tiles[0], 0, n, x, m);
  copies_commit();
  int b = 0;
  for (int64_t j0 = 0; j0 < n; j0 += kLfTile, b ^= 1) {
    if (j0 + kLfTile < n) stage_pairs(tiles[b ^ 1], j0 + kLfTile, n, x, m);
    copies_commit();
    copies_wait<1>();
    __syncthreads();
    const float4 *t = tiles[b];
    auto pair = [&](int k) {
      const float4 q = t[k], w = t[kPairs + k];
      const float2 dx = __fadd2_rn(make_float2(q.x, q.y), nx);
      const float2 dy = __fadd2_rn(make_float2(q.z, q.w), ny);
      const float2 dz = __fadd2_rn(make_float2(w.x, w.y), nz);
      const float2 s2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
      const float2 ri = lf_rsq2<MASK>(s2);
      const float2 f = __fmul2_rn(__fmul2_rn(make_float2(w.z, w.w), ri), __fmul2_rn(ri, ri));
      px = __ffma2_rn(f, dx, px);
      py = __ffma2_rn(f, dy, py);
      pz = __ffma2_rn(f, dz, pz);
    };
    // what lies past the end adds zero
#pragma unroll 8
    for (int k = r; k < kPairs; k += kLfAccWarps) pair(k);
    __syncthreads();  // the tile's readers are done
  }
  part[threadIdx.x][0] = px.x + px.y;
  part[threadIdx.x][1] = py.x + py.y;
  part[threadIdx.x][2] = pz.x + pz.y;
  __syncthreads();
  for (int q = threadIdx.x; q < 3 * per_cta; q += blockDim.x) {
    const int64_t e = 3 * i0 + q;
    if (e >= 3 * n) return;
    const int p = q / 3, c = q - 3 * p;
    const float(*s)[3] = part + (p / 32 * kLfAccWarps * 32 + p % 32);
    const float a = G * ((s[0][c] + s[32][c]) + (s[64][c] + s[96][c]));
    if (T.acc) T.acc[e] = a;
    if (!T.v_out) continue;
    const float xe = x[e];
    float v = T.v_in[e];
    if (T.close) v = fmaf(a, T.h, v);
    if (T.ck) {
      T.ck[e] = xe;
      T.ck[3 * n + e] = v;
    }
    if (T.x_out) {
      v = fmaf(a, T.h, v);
      T.x_out[e] = fmaf(v, T.dt, xe);
    }
    T.v_out[e] = v;
  }
}

// Wide shape for large N: each thread holds 4 i-particles, two per packed
// FP32x2 instruction (per-lane IEEE rounding), and TPI threads share an
// i-particle group, splitting every shared-memory tile's j-range (their sums
// meet by a warp-shuffle butterfly); 1,024 / TPI i-particles per CTA.  The
// next tile is read into registers while the current one is summed, and each
// tile's sum is added to the running total, so no FP32 sum runs over more
// than 256 / TPI terms plus one term per tile.
constexpr int kLfWideIpt = 4;

template <int MASK, int TPI>
__global__ void __launch_bounds__(kLfT) lf_acc_wide_kernel(int64_t n, const float *__restrict__ x,
                                                           const float *__restrict__ m,
                                                           float eps2, float G,
                                                           float *__restrict__ acc) {
  __shared__ float4 sj[kLfJT];
  constexpr int NQ = kLfWideIpt / 2;
  constexpr int NG = kLfT / TPI;            // i-particle groups per CTA
  constexpr int BI = NG * kLfWideIpt;       // i-particles per CTA
  const int tid = threadIdx.x, g = tid / TPI, r = tid % TPI;
  float2 nx[NQ], ny[NQ], nz[NQ];  // negated i-positions, two particles per pair
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * BI + g + (2 * q) * NG;
    const int64_t i1 = i0 + NG;
    const int64_t a0 = i0 < n ? i0 : 0, a1 = i1 < n ? i1 : 0;
    nx[q] = make_float2(-x[3 * a0], -x[3 * a1]);
    ny[q] = make_float2(-x[3 * a0 + 1], -x[3 * a1 + 1]);
    nz[q] = make_float2(-x[3 * a0 + 2], -x[3 * a1 + 2]);
  }
  const float2 e2 = make_float2(eps2, eps2);
  float2 tx[NQ], ty[NQ], tz[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) tx[q] = ty[q] = tz[q] = make_float2(0.f, 0.f);
  auto fetch = [&](int64_t j) {
    return j < n ? make_float4(x[3 * j], x[3 * j + 1], x[3 * j + 2], m[j])
                 : make_float4(1.0e15f, 1.0e15f, 1.0e15f, 0.f);
  };
  float4 next = fetch(tid);
  for (int64_t j0 = 0; j0 < n; j0 += kLfJT) {
    __syncthreads();  // the previous tile's readers are done
    sj[tid] = next;
    __syncthreads();
    next = fetch(j0 + kLfJT + tid);
    float2 px[NQ], py[NQ], pz[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) px[q] = py[q] = pz[q] = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int t = r; t < kLfJT; t += TPI) {
      const float4 qj = sj[t];
      const float2 xj = make_float2(qj.x, qj.x), yj = make_float2(qj.y, qj.y);
      const float2 zj = make_float2(qj.z, qj.z), mj = make_float2(qj.w, qj.w);
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const float2 dx = __fadd2_rn(xj, nx[q]), dy = __fadd2_rn(yj, ny[q]);
        const float2 dz = __fadd2_rn(zj, nz[q]);
        const float2 s2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
        const float2 ri = lf_rsq2<MASK>(s2);
        const float2 f = __fmul2_rn(__fmul2_rn(mj, ri), __fmul2_rn(ri, ri));
        px[q] = __ffma2_rn(f, dx, px[q]);
        py[q] = __ffma2_rn(f, dy, py[q]);
        pz[q] = __ffma2_rn(f, dz, pz[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      tx[q] = __fadd2_rn(tx[q], px[q]);
      ty[q] = __fadd2_rn(ty[q], py[q]);
      tz[q] = __fadd2_rn(tz[q], pz[q]);
    }
  }
  if (TPI > 1) {
#pragma unroll
    for (int off = 1; off < TPI; off <<= 1)
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        tx[q].x += __shfl_xor_sync(0xffffffffu, tx[q].x, off);
        tx[q].y += __shfl_xor_sync(0xffffffffu, tx[q].y, off);
        ty[q].x += __shfl_xor_sync(0xffffffffu, ty[q].x, off);
        ty[q].y += __shfl_xor_sync(0xffffffffu, ty[q].y, off);
        tz[q].x += __shfl_xor_sync(0xffffffffu, tz[q].x, off);
        tz[q].y += __shfl_xor_sync(0xffffffffu, tz[q].y, off);
      }
  }
  if (r != 0) return;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * BI + g + (2 * q) * NG;
    const int64_t i1 = i0 + NG;
    if (i0 < n) {
      acc[3 * i0] = G * tx[q].x;
      acc[3 * i0 + 1] = G * ty[q].x;
      acc[3 * i0 + 2] = G * tz[q].x;
    }
    if (i1 < n) {
      acc[3 * i1] = G * tx[q].y;
      acc[3 * i1 + 1] = G * ty[q].y;
      acc[3 * i1 + 2] = G * tz[q].y;
    }
  }
}

// lx_k += dL/dx_k and lm_k += dL/dm_k for the cotangent g = h * lv; with
// lv_out set, also lv_out_k = lv_k + dlv lx_k with the updated lx_k (the
// adjoint of the drift).  Bound by the FP32 pipe, 32 lane-operations per
// pair; two warps per IPT particles, so that N = 4096 has seven per scheduler.
// N = 1,000 / 4,096 / 16,000: 11.9 / 30.9 / 342 us, the two clears of the stand-alone
// call included (8 threads per particle: 17.9 / 43.2 / 399).
template <int MASK, int IPT>
__global__ void __launch_bounds__(kLfVjpMaxThreads)
    lf_vjp_kernel(int64_t n, int slots, const float *__restrict__ x,
                  const float *__restrict__ m, const float *__restrict__ lv, float h, float eps2,
                  float G, float *__restrict__ lx, float *__restrict__ lm,
                  float *__restrict__ lv_out, float dlv) {
  extern __shared__ __align__(16) float4 vtiles[];  // [2][2][kLfVjpTile]: x, m; cotangents
  __shared__ float half[kLfVjpMaxThreads / kLfVjpTpi][4 * IPT];
  constexpr int TPI = kLfVjpTpi;
  const int g = threadIdx.x / TPI, r = threadIdx.x % TPI;
  const int64_t k0 = (static_cast<int64_t>(blockIdx.x) * slots + g) * IPT;
  constexpr int NQ = IPT / 2;
  // two particles side by side; positions and cotangents negated
  float2 nx[NQ][3], ng[NQ][3], mk[NQ], o[NQ][4];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int64_t a = k0 + 2 * q < n ? k0 + 2 * q : 0, b = k0 + 2 * q + 1 < n ? k0 + 2 * q + 1 : 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      nx[q][c] = make_float2(-x[3 * a + c], -x[3 * b + c]);
      ng[q][c] = make_float2(-lv[3 * a + c], -lv[3 * b + c]);
    }
    mk[q] = make_float2(m[a], m[b]);
    o[q][0] = o[q][1] = o[q][2] = o[q][3] = dup(0.f);
  }
  const float2 e2 = dup(eps2);
  auto stage = [&](int b, int64_t j0) {
    stage_xm(vtiles + b * 2 * kLfVjpTile, j0, n, x, m);
    stage_g(vtiles + (b * 2 + 1) * kLfVjpTile, j0, n, lv);
  };
  stage(0, 0);
  copies_commit();
  int b = 0;
  for (int64_t j0 = 0; j0 < n; j0 += kLfVjpTile, b ^= 1) {
    if (j0 + kLfVjpTile < n) stage(b ^ 1, j0 + kLfVjpTile);
    copies_commit();
    copies_wait<1>();
    __syncthreads();
    const float4 *t = vtiles + b * 2 * kLfVjpTile, *tg = t + kLfVjpTile;
    const int cnt = n - j0 < kLfVjpTile ? static_cast<int>(n - j0) : kLfVjpTile;
#pragma unroll 1
    for (int p0 = r; p0 < cnt; p0 += 4 * TPI)
#pragma unroll 2
    for (int p = p0; p < p0 + 4 * TPI; p += TPI) {
      const float4 j = t[p], gq = tg[p];
      const float2 xj[3] = {dup(j.x), dup(j.y), dup(j.z)}, mj = dup(j.w);
      const float2 gj[3] = {dup(gq.x), dup(gq.y), dup(gq.z)};
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        float2 d[3], u[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          d[c] = __fadd2_rn(xj[c], nx[q][c]);
          // u = m_k g_j - m_j g_k with both products rounded alike, so that
          // the i == j term is exactly zero (a fused form would leave the
          // rounding error of one product, amplified by 1/eps^3)
          u[c] = __fadd2_rn(mul2_alone(mk[q], gj[c]), mul2_alone(mj, ng[q][c]));
        }
        const float2 s2 =
            __ffma2_rn(d[0], d[0], __ffma2_rn(d[1], d[1], __ffma2_rn(d[2], d[2], e2)));
        const float2 ri = lf_rsq2<MASK>(s2);
        const float2 ri2 = __fmul2_rn(ri, ri);
        const float2 s3 = __fmul2_rn(ri, ri2);
        const float2 du = __ffma2_rn(d[0], u[0], __ffma2_rn(d[1], u[1], __fmul2_rn(d[2], u[2])));
        const float2 c3 = __fmul2_rn(__fmul2_rn(du, ri2), dup(-3.f));
        // (I - 3 d d^T / s^2) u / s^3
#pragma unroll
        for (int c = 0; c < 3; ++c) o[q][c] = __ffma2_rn(s3, __ffma2_rn(c3, d[c], u[c]), o[q][c]);
        // (g_j . d) / s^3
        const float2 gd =
            __ffma2_rn(gj[0], d[0], __ffma2_rn(gj[1], d[1], __fmul2_rn(gj[2], d[2])));
        o[q][3] = __ffma2_rn(gd, s3, o[q][3]);
      }
    }
    __syncthreads();
  }
  // lane 4 q + c ends component c of particle q (c = 3: the mass)
  float mine = 0.f;
  const int lane = r % 32;
#pragma unroll
  for (int q = 0; q < IPT; ++q)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float s = q % 2 ? o[q / 2][c].y : o[q / 2][c].x;
      if (c == 3) s = -s;
#pragma unroll
      for (int f = 1; f < 32; f <<= 1) s += __shfl_xor_sync(0xffffffffu, s, f);
      if (lane == 4 * q + c) mine = s;
    }
  if (r >= 32 && lane < 4 * IPT) half[g][lane] = mine;
  __syncthreads();
  const int64_t k = k0 + r / 4;
  const int c = r % 4;
  if (r >= 4 * IPT || k >= n) return;
  mine += half[g][r];
  // the sums are linear in the cotangent: its factor h comes in here
  const float val = G * (h * mine);
  if (c == 3) {
    lm[k] += val;
  } else {
    const float lxn = lx[3 * k + c] + val;
    lx[3 * k + c] = lxn;
    if (lv_out) lv_out[3 * k + c] = fmaf(dlv, lxn, lv[3 * k + c]);
  }
}

// v += a h.
__global__ void lf_kick_kernel(int64_t n3, float *__restrict__ v, const float *__restrict__ a,
                               float h) {
  const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q < n3) v[q] = fmaf(a[q], h, v[q]);
}

// One drift of a run of KDK steps with the kicks around it merged: with
// close set, the previous step's closing kick v += a h first; then, when
// ck_x is set, the checkpoint (x, v) of the step boundary; then this step's
// opening kick v += a h and the drift x_out = x_in + v dt.  The same
// per-element operations in the same order as separate kick and drift
// launches.  x_in may equal x_out, v_in v_out.
__global__ void lf_step_kernel(int64_t n3, const float *x_in, float *x_out, const float *v_in,
                               float *v_out, const float *__restrict__ a, float h, float dt,
                               int close, float *__restrict__ ck_x, float *__restrict__ ck_v) {
  const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q >= n3) return;
  const float aq = a[q], xq = x_in[q];
  float vq = v_in[q];
  if (close) vq = fmaf(aq, h, vq);
  if (ck_x) {
    ck_x[q] = xq;
    ck_v[q] = vq;
  }
  vq = fmaf(aq, h, vq);
  v_out[q] = vq;
  x_out[q] = fmaf(vq, dt, xq);
}

// The same for a run with the pair-symmetric force, one CTA per 256-record
// tile and one thread per particle: the step (with move set), then the new
// position's records for the force kernel.
__global__ void __launch_bounds__(kJT)
    lf_sym_step_kernel(int64_t n, const float *x_in, float *x_out, const float *v_in, float *v_out,
                       const float *__restrict__ a, float h, float dt, int move, int close,
                       float *__restrict__ ck_x, float *__restrict__ ck_v,
                       const float *__restrict__ m, float4 *__restrict__ jhi,
                       unsigned char *__restrict__ recs, const SymScale *__restrict__ scale) {
  const int64_t j = static_cast<int64_t>(blockIdx.x) * kJT + threadIdx.x;
  float4 r = make_float4(dev::kNowhere, dev::kNowhere, dev::kNowhere, 0.f);
  if (j < n) {
    float xn[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int64_t q = 3 * j + c;
      xn[c] = x_in[q];
      if (move) {
        const float aq = a[q];
        float vq = v_in[q];
        if (close) vq = fmaf(aq, h, vq);
        if (ck_x) {
          ck_x[q] = xn[c];
          ck_v[q] = vq;
        }
        vq = fmaf(aq, h, vq);
        v_out[q] = vq;
        xn[c] = fmaf(vq, dt, xn[c]);
        x_out[q] = xn[c];
      }
    }
    r = make_float4(xn[0], xn[1], xn[2], m[j]);
  }
  const float sc = scale->sc, sm = scale->sm;
  if (j < n) r = make_float4(r.x * sc, r.y * sc, r.z * sc, r.w * sm);
  jhi[j] = r;
  dev::put_rec4(recs + static_cast<size_t>(blockIdx.x) * dev::rec_bytes(0), 0, threadIdx.x, r);
}

// The pair-symmetric kernel's scale, from the size of the largest mass (masses
// come in any units and, while they are fitted, with any sign).  One CTA, once per
// run: N = 131,101 / 1,000,000 12 / 68 us (a forward step: 4.62 / 260 ms).
constexpr int kLfScaleT = 1024;

__global__ void __launch_bounds__(kLfScaleT)
    lf_scale_kernel(int64_t n, const float *__restrict__ m, float eps2, double G,
                    SymScale *__restrict__ out) {
  __shared__ float sh[kLfScaleT / 32];
  float top = 0.f;
#pragma unroll 8
  for (int64_t i = threadIdx.x; i < n; i += kLfScaleT) top = fmaxf(top, fabsf(m[i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (threadIdx.x % 32 == 0) sh[threadIdx.x / 32] = top;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < kLfScaleT / 32; ++w) top = fmaxf(top, sh[w]);
  const int e = sym_exponent(top, eps2);
  out->sc = ldexpf(1.f, e);
  out->sm = ldexpf(1.f, 3 * e);
  out->eps2 = eps2 * ldexpf(1.f, e) * ldexpf(1.f, e);
  out->g_acc = ldexp(G, -e);
}

struct LfCtx {
  int64_t n;
  const float *m;
  float eps2, G;
  int mask;
  int sms;
  cudaStream_t s;
  int64_t launches;
  // the pair-symmetric force, when the caller lent the scratch for it
  bool sym = false;
  SymArgs S;
  float4 *jhi = nullptr;
};

// Smallest n of the pair-symmetric force (nb_symforce.cu) for the forward
// steps, and the most scratch it may ask for (1.9 kB per particle).  A step
// with it against the one-sided shapes, N = 16,384 / 16,385 (a block more) /
// 20,000 / 60,000 / 131,101 / 262,144: 0.105 / 0.126 / 0.148 / 1.03 / 4.62 /
// 17.7 ms against 0.133 / 0.137 / 0.225 / 1.61 / 6.57 / 25.8; its sums fold in
// split precision, error against 64 bits 3 .. 4e-8 against 1.2 .. 4.6e-7.
constexpr int64_t kLfSymMin = 16384;
constexpr int64_t kLfSymMaxBytes = int64_t(16) << 30;

struct LfSymLayout {
  SymSplit split;
  size_t recs, ipart, jpart, err, scale, bytes;  // offsets behind the records jhi
};

bool lf_sym_layout(int64_t n, int mask, int sms, LfSymLayout *L) {
  if (n < kLfSymMin) return false;
  const int64_t n_jt = (n + kJT - 1) / kJT;
  if (!sym_split(n_jt, sym_block_i(0, mask, false, n_jt), sms, &L->split)) return false;
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  L->recs = up(static_cast<size_t>(n_jt) * kJT * sizeof(float4));
  L->ipart = L->recs + up(sym_record_bytes(n_jt, 0));
  L->jpart = L->ipart + up(sym_ipart_bytes(L->split, false));
  L->err = L->jpart + up(sym_jpart_bytes(L->split, false));
  L->scale = L->err + 128;
  L->bytes = L->err + 256;
  return L->bytes <= static_cast<size_t>(kLfSymMaxBytes);
}

int lf_sms() {
  // A failed query leaves its error for the launch's error check to report.
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms < 1 ? 1 : sms;
}

// Takes the pair-symmetric force where the scratch suffices.
cudaError_t lf_lend(LfCtx &C, void *scratch, int64_t bytes) {
  LfSymLayout L;
  if (!scratch || reinterpret_cast<uintptr_t>(scratch) % 256 != 0 ||
      !lf_sym_layout(C.n, C.mask, C.sms, &L) || bytes < static_cast<int64_t>(L.bytes))
    return cudaSuccess;
  unsigned char *b = static_cast<unsigned char *>(scratch);
  C.jhi = reinterpret_cast<float4 *>(b);
  C.S = SymArgs();
  C.S.jhi = C.jhi;
  C.S.jlo = C.S.jvel = C.S.jrel = C.S.tinfo = nullptr;
  C.S.n_jt = (C.n + kJT - 1) / kJT;
  C.S.n = C.n;
  C.S.eps2 = C.eps2;
  C.S.G = C.G;
  SymScale *scale = reinterpret_cast<SymScale *>(b + L.scale);
  C.S.dscale = scale;
  C.S.acc = C.S.jerk = nullptr;
  C.S.recs = b + L.recs;
  C.S.ipart = reinterpret_cast<float2 *>(b + L.ipart);
  C.S.jpart = reinterpret_cast<float2 *>(b + L.jpart);
  C.S.err = reinterpret_cast<int *>(b + L.err);
  C.S.split = L.split;
  C.sym = true;
  cudaError_t e = sym_prepare(0, C.mask, false, false, C.S.n_jt);
  if (e == cudaSuccess) e = cudaMemsetAsync(C.S.err, 0, sizeof(int), C.s);
  if (e != cudaSuccess) return e;
  lf_scale_kernel<<<1, kLfScaleT, 0, C.s>>>(C.n, C.m, C.eps2, C.G, scale);
  ++C.launches;
  return cudaGetLastError();
}

// N >= kLfWideMin takes the wide shape (4 particles per thread, records
// broadcast) for the force.
constexpr int64_t kLfWideMin = 65536;

// Groups of 32 particles per CTA of the small force shape: the count that
// leaves an SM the fewest groups to run, the larger one where two are equal
// (a CTA's copies of the records serve all its groups).
int lf_groups(int64_t n, int sms) {
  int best = 1;
  int64_t cost = INT64_MAX;
  for (int g = 1; g <= kLfMaxThreads / (32 * kLfAccWarps); ++g) {
    const int64_t ctas = (n + 32 * g - 1) / (32 * g);
    const int64_t c = (ctas + sms - 1) / sms * g;
    if (c < cost || (c == cost && n > 32 * static_cast<int64_t>(sms))) {
      cost = c;
      best = g;
    }
  }
  return best;
}

// Slots (groups of ipt particles) per CTA of the vector-Jacobian product: the
// CTAs fill whole rounds of the SMs (N = 4096, 152 SMs: 147 CTAs of 14 pairs).
int lf_slots(int64_t n, int ipt, int most, int sms) {
  const int64_t total = (n + ipt - 1) / ipt;
  const int64_t rounds = (total + sms * most - 1) / (sms * most);
  return static_cast<int>((total + sms * rounds - 1) / (sms * rounds));
}

// Threads per i-particle group of the wide shape, 4 or 8.  CTAs take the
// same time, so an SM's share is ceil(grid / SMs) CTAs run one after
// another; 8 threads halve the i-particles per CTA, and are taken where the
// grid then divides more evenly over the SMs (N = 131072 on 152 SMs: 3.4
// against 6.7 CTAs per SM).
int lf_wide_tpi(int64_t n, int sms) {
  auto balance = [&](int tpi) {
    const int64_t bi = kLfT / tpi * kLfWideIpt;
    const int64_t grid = (n + bi - 1) / bi;
    const int64_t rounds = (grid + sms - 1) / sms;
    return static_cast<double>(grid) / static_cast<double>(rounds * sms);
  };
  return balance(8) > balance(4) + 0.01 ? 8 : 4;
}

template <int TPI>
void launch_lf_wide(const LfCtx &C, const float *x, float *acc) {
  constexpr int bi = kLfT / TPI * kLfWideIpt;
  const unsigned grid = static_cast<unsigned>((C.n + bi - 1) / bi);
  if (C.mask)
    lf_acc_wide_kernel<1, TPI><<<grid, kLfT, 0, C.s>>>(C.n, x, C.m, C.eps2, C.G, acc);
  else
    lf_acc_wide_kernel<0, TPI><<<grid, kLfT, 0, C.s>>>(C.n, x, C.m, C.eps2, C.G, acc);
}

// A(x) and what follows it (see LfTail), n < kLfWideMin.
cudaError_t lf_eval(LfCtx &C, const float *x, const LfTail &T) {
  const int g = lf_groups(C.n, C.sms);
  // one group per CTA at most: spread over all SMs
  const int per = g == 1 && C.n <= 32 * static_cast<int64_t>(C.sms)
                      ? static_cast<int>((C.n + C.sms - 1) / C.sms)
                      : 32 * g;
  const unsigned grid = static_cast<unsigned>((C.n + per - 1) / per);
  const int nt = 32 * kLfAccWarps * g;
  if (C.mask)
    lf_eval_kernel<1><<<grid, nt, 0, C.s>>>(C.n, per, x, C.m, C.eps2, C.G, T);
  else
    lf_eval_kernel<0><<<grid, nt, 0, C.s>>>(C.n, per, x, C.m, C.eps2, C.G, T);
  ++C.launches;
  return cudaGetLastError();
}

// acc = A(x_out) after the step that leads there (with v_in set), or A(x_in).
cudaError_t lf_sym_eval(LfCtx &C, const float *x_in, float *x_out, const float *v_in, float *v_out,
                        float *acc, float h, float dt, bool close, float *ck) {
  lf_sym_step_kernel<<<static_cast<unsigned>(C.S.n_jt), kJT, 0, C.s>>>(
      C.n, x_in, x_out, v_in, v_out, acc, h, dt, v_in ? 1 : 0, close ? 1 : 0, ck,
      ck ? ck + 3 * C.n : nullptr, C.m, C.jhi, C.S.recs, C.S.dscale);
  ++C.launches;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  C.S.acc_f = acc;
  int nl = 0;
  e = launch_sym_force(0, C.mask, C.S, C.s, &nl);
  C.launches += nl;
  return e;
}

cudaError_t lf_acc(LfCtx &C, const float *x, float *acc) {
  if (C.sym) return lf_sym_eval(C, x, nullptr, nullptr, nullptr, acc, 0.f, 0.f, false, nullptr);
  if (C.n < kLfWideMin) {
    LfTail T;
    T.acc = acc;
    return lf_eval(C, x, T);
  }
  if (lf_wide_tpi(C.n, C.sms) == 8)
    launch_lf_wide<8>(C, x, acc);
  else
    launch_lf_wide<4>(C, x, acc);
  ++C.launches;
  return cudaGetLastError();
}

template <int MASK, int IPT>
cudaError_t launch_lf_vjp(const LfCtx &C, const float *x, const float *lv, float h, float *lx,
                          float *lm, float *lv_out, float dlv) {
  constexpr int smem = 4 * kLfVjpTile * sizeof(float4);
  cudaError_t e = cudaFuncSetAttribute(lf_vjp_kernel<MASK, IPT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int slots = lf_slots(C.n, IPT, kLfVjpMaxThreads / kLfVjpTpi, C.sms);
  const unsigned grid = static_cast<unsigned>((C.n + slots * IPT - 1) / (slots * IPT));
  lf_vjp_kernel<MASK, IPT><<<grid, slots * kLfVjpTpi, smem, C.s>>>(
      C.n, slots, x, C.m, lv, h, C.eps2, C.G, lx, lm, lv_out, dlv);
  return cudaGetLastError();
}

cudaError_t lf_vjp(LfCtx &C, const float *x, const float *lv, float h, float *lx, float *lm,
                   float *lv_out = nullptr, float dlv = 0.f) {
  ++C.launches;
  return C.mask ? launch_lf_vjp<1, 2>(C, x, lv, h, lx, lm, lv_out, dlv)
                : launch_lf_vjp<0, 2>(C, x, lv, h, lx, lm, lv_out, dlv);
}

cudaError_t lf_kick(LfCtx &C, float *v, const float *a, float h) {
  const int64_t n3 = 3 * C.n;
  lf_kick_kernel<<<static_cast<unsigned>((n3 + 255) / 256), 256, 0, C.s>>>(n3, v, a, h);
  ++C.launches;
  return cudaGetLastError();
}

// Whether acc carries A(x) from one half step to the next (and x_in may be
// x_out), or every half step computes it.
bool lf_carries(const LfCtx &C) { return C.sym || C.n >= kLfWideMin; }

// The drift of one KDK step with the kicks around it: from A(x_in) (where
// lf_carries, acc holds it and receives A(x_out); otherwise it is computed
// here and x_out must differ from x_in).  The step's own closing kick is left
// to the next call (close) or to the end of the run.
cudaError_t lf_half_step(LfCtx &C, const float *x_in, float *x_out, const float *v_in,
                         float *v_out, float *acc, float dt, bool close, float *ck) {
  if (C.sym)
    return lf_sym_eval(C, x_in, x_out, v_in, v_out, acc, 0.5f * dt, dt, close, ck);
  if (C.n < kLfWideMin) {
    LfTail T;
    T.v_in = v_in;
    T.v_out = v_out;
    T.x_out = x_out;
    T.ck = ck;
    T.close = close ? 1 : 0;
    T.h = 0.5f * dt;
    T.dt = dt;
    return lf_eval(C, x_in, T);
  }
  const int64_t n3 = 3 * C.n;
  lf_step_kernel<<<static_cast<unsigned>((n3 + 255) / 256), 256, 0, C.s>>>(
      n3, x_in, x_out, v_in, v_out, acc, 0.5f * dt, dt, close ? 1 : 0, ck,
      ck ? ck + n3 : nullptr);
  ++C.launches;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = lf_acc(C, x_out, acc);
  return e;
}

nb_status lf_check(int64_t n, float eps, float G, const void *a, const void *b) {
  if (n < 1 || n > (int64_t(1) << 30))
    return static_cast<nb_status>(set_error(NB_ERR_INVALID_ARG, "n out of range [1, 2^30]"));
  if (!(eps >= 0.f) || !(G > 0.f))
    return static_cast<nb_status>(set_error(NB_ERR_INVALID_ARG, "need eps >= 0 and G > 0"));
  if (!a || !b) return static_cast<nb_status>(set_error(NB_ERR_INVALID_ARG, "null device pointer"));
  return NB_OK;
}

nb_status lf_err(cudaError_t e) {
  return static_cast<nb_status>(
      set_error(NB_ERR_CUDA, "leapfrog kernel launch failed: %s", cudaGetErrorString(e)));
}

LfCtx make_ctx(int64_t n, const float *m, float eps, float G, void *stream) {
  LfCtx C;
  C.n = n;
  C.m = m;
  // eps^2 not a normal float: the kernels zero the i == j term (and take
  // eps^2 = 0, which is what the device's flush of subnormals would make of it)
  C.mask = eps * eps < FLT_MIN ? 1 : 0;
  C.eps2 = C.mask ? 0.f : eps * eps;
  C.G = G;
  C.sms = lf_sms();
  C.s = static_cast<cudaStream_t>(stream);
  C.launches = 0;
  return C;
}

}  // namespace
}  // namespace nbi

using namespace nbi;

extern "C" {

nb_status nb_lf_acc(int64_t n, const float *d_x, const float *d_m, float eps, float G,
                    float *d_acc, void *stream) {
  nb_status s = lf_check(n, eps, G, d_x, d_m);
  if (s != NB_OK) return s;
  if (!d_acc) return static_cast<nb_status>(set_error(NB_ERR_INVALID_ARG, "null output"));
  LfCtx C = make_ctx(n, d_m, eps, G, stream);
  cudaError_t e = lf_acc(C, d_x, d_acc);
  return e == cudaSuccess ? NB_OK : lf_err(e);
}

nb_status nb_lf_acc_vjp(int64_t n, const float *d_x, const float *d_m, const float *d_g,
                        float eps, float G, float *d_gx, float *d_gm, void *stream) {
  nb_status s = lf_check(n, eps, G, d_x, d_m);
  if (s != NB_OK) return s;
  if (!d_g || !d_gx || !d_gm)
    return static_cast<nb_status>(set_error(NB_ERR_INVALID_ARG, "null device pointer"));
  LfCtx C = make_ctx(n, d_m, eps, G, stream);
  cudaError_t e = cudaMemsetAsync(d_gx, 0, 3 * n * sizeof(float), C.s);
  if (e == cudaSuccess) e = cudaMemsetAsync(d_gm, 0, n * sizeof(float), C.s);
  if (e == cudaSuccess) e = lf_vjp(C, d_x, d_g, 1.f, d_gx, d_gm);
  return e == cudaSuccess ? NB_OK : lf_err(e);
}

int64_t nb_lf_ckpt_floats(int64_t n, int64_t nsteps, int32_t ckpt_every) {
  if (n < 1 || nsteps < 0 || ckpt_every < 1) return -1;
  const int64_t K = (nsteps + ckpt_every - 1) / ckpt_every;
  return std::max<int64_t>(K, 1) * 6 * n;
}

int64_t nb_lf_work_floats(int64_t n, int32_t ckpt_every) {
  if (n < 1 || ckpt_every < 1) return -1;
  return (static_cast<int64_t>(ckpt_every) + 1) * 3 * n + 6 * n;
}

int64_t nb_lf_scratch_bytes(int64_t n) {
  int64_t most = 0;
  if (n < kLfSymMin || n > (int64_t(1) << 30)) return 0;
  const int sms = lf_sms();
  for (int mask = 0; mask < 2; ++mask) {
    LfSymLayout L;
    if (lf_sym_layout(n, mask, sms, &L)) most = std::max(most, static_cast<int64_t>(L.bytes));
  }
  return most;
}

nb_status nb_lf_forward(int64_t n, const float *d_m, float *d_x, float *d_v, float *d_acc,
                        int64_t nsteps, float dt, float eps, float G, int32_t ckpt_every,
                        float *d_ckpt, void *stream) {
  return nb_lf_forward_lent(n, d_m, d_x, d_v, d_acc, nsteps, dt, eps, G, ckpt_every, d_ckpt,
                            nullptr, 0, stream);
}

nb_status nb_lf_forward_lent(int64_t n, const float *d_m, float *d_x, float *d_v, float *d_acc,
                             int64_t nsteps, float dt, float eps, float G, int32_t ckpt_every,
                             float *d_ckpt, void *d_scratch, int64_t scratch_bytes,
                             void *stream) {
  nb_status s = lf_check(n, eps, G, d_m, d_x);
  if (s != NB_OK) return s;
  if (!d_v || !d_acc || nsteps < 0 || ckpt_every < 1 || !(std::isfinite(dt)))
    return static_cast<nb_status>(set_error(NB_ERR_INVALID_ARG, "bad leapfrog arguments"));
  LfCtx C = make_ctx(n, d_m, eps, G, stream);
  const size_t n3b = 3 * static_cast<size_t>(n) * sizeof(float);
  auto ck = [&](int64_t st) {
    return d_ckpt && st % ckpt_every == 0 ? d_ckpt + (st / ckpt_every) * 6 * n : nullptr;
  };
  cudaError_t e = lf_lend(C, d_scratch, scratch_bytes);
  if (!lf_carries(C)) {
    // every force evaluation ends with the drift to the next positions, which
    // go to the other of d_x and d_acc (free until the last evaluation)
    float *cur = d_x, *other = d_acc;
    for (int64_t st = 0; st < nsteps && e == cudaSuccess; ++st) {
      e = lf_half_step(C, cur, other, d_v, d_v, nullptr, dt, st > 0, ck(st));
      std::swap(cur, other);
    }
    if (e == cudaSuccess && cur != d_x)
      e = cudaMemcpyAsync(d_x, cur, n3b, cudaMemcpyDeviceToDevice, C.s);
    LfTail T;
    T.acc = d_acc;
    if (nsteps > 0) {
      T.v_in = d_v;
      T.v_out = d_v;
      T.close = 1;
      T.h = 0.5f * dt;
    }
    if (e == cudaSuccess) e = lf_eval(C, d_x, T);
    return e == cudaSuccess ? NB_OK : lf_err(e);
  }
  if (e == cudaSuccess) e = lf_acc(C, d_x, d_acc);
  for (int64_t st = 0; st < nsteps && e == cudaSuccess; ++st)
    e = lf_half_step(C, d_x, d_x, d_v, d_v, d_acc, dt, st > 0, ck(st));
  if (e == cudaSuccess && nsteps > 0) e = lf_kick(C, d_v, d_acc, 0.5f * dt);
  return e == cudaSuccess ? NB_OK : lf_err(e);
}

nb_status nb_lf_backward(int64_t n, const float *d_m, const float *d_ckpt, int64_t nsteps,
                         float dt, float eps, float G, int32_t ckpt_every, float *d_lx,
                         float *d_lv, float *d_lm, float *d_work, void *stream) {
  return nb_lf_backward_lent(n, d_m, d_ckpt, nsteps, dt, eps, G, ckpt_every, d_lx, d_lv, d_lm,
                             d_work, nullptr, 0, stream);
}

nb_status nb_lf_backward_lent(int64_t n, const float *d_m, const float *d_ckpt, int64_t nsteps,
                              float dt, float eps, float G, int32_t ckpt_every, float *d_lx,
                              float *d_lv, float *d_lm, float *d_work, void *d_scratch,
                              int64_t scratch_bytes, void *stream) {
  nb_status s = lf_check(n, eps, G, d_m, d_ckpt);
  if (s != NB_OK) return s;
  if (!d_lx || !d_lv || !d_lm || !d_work || nsteps < 0 || ckpt_every < 1)
    return static_cast<nb_status>(set_error(NB_ERR_INVALID_ARG, "bad leapfrog adjoint arguments"));
  LfCtx C = make_ctx(n, d_m, eps, G, stream);
  const size_t n3 = 3 * static_cast<size_t>(n);
  const size_t n3b = n3 * sizeof(float);
  float *xs = d_work;                               // (ckpt_every + 1) positions
  float *v = d_work + (ckpt_every + 1) * n3;        // velocity during recompute
  float *acc = v + n3;                              // acceleration during recompute
  cudaError_t e = lf_lend(C, d_scratch, scratch_bytes);
  if (e == cudaSuccess) e = cudaMemsetAsync(d_lm, 0, n * sizeof(float), C.s);
  const int64_t K = (nsteps + ckpt_every - 1) / ckpt_every;
  for (int64_t seg = K - 1; seg >= 0 && e == cudaSuccess; --seg) {
    const int64_t s0 = seg * ckpt_every;
    const int64_t L = std::min<int64_t>(ckpt_every, nsteps - s0);
    const float *slot = d_ckpt + seg * 6 * n;  // x, v at step s0
    // positions of the segment's steps: xs[q] for q > 0, the checkpoint
    // itself for q = 0; the end of the last segment is needed too, the ends
    // of the others are the next one's checkpoint
    const int64_t upto = seg == K - 1 ? L : L - 1;
    auto pos = [&](int64_t q) -> const float * { return q == 0 ? slot : xs + q * n3; };
    if (upto > 0 && lf_carries(C)) e = lf_acc(C, slot, acc);
    for (int64_t q = 0; q < upto && e == cudaSuccess; ++q)
      e = lf_half_step(C, pos(q), xs + (q + 1) * n3, q == 0 ? slot + n3 : v, v, acc, dt, q > 0,
                       nullptr);
    // the sweep: at every x the merged kicks, then the drift that led there
    // (fused, writing the new lv to the other of d_lv and the now free
    // velocity buffer); half a kick at the two ends of the run
    float *cur = d_lv, *other = v;
    if (seg == K - 1 && e == cudaSuccess) {
      e = lf_vjp(C, pos(L), cur, 0.5f * dt, d_lx, d_lm, other, dt);
      std::swap(cur, other);
    }
    for (int64_t q = L - 1; q >= 0 && e == cudaSuccess; --q) {
      if (s0 + q > 0) {
        e = lf_vjp(C, pos(q), cur, dt, d_lx, d_lm, other, dt);
        std::swap(cur, other);
      } else {
        e = lf_vjp(C, pos(q), cur, 0.5f * dt, d_lx, d_lm);
      }
    }
    if (e == cudaSuccess && cur != d_lv)
      e = cudaMemcpyAsync(d_lv, cur, n3b, cudaMemcpyDeviceToDevice, C.s);
  }
  return e == cudaSuccess ? NB_OK : lf_err(e);
}

}  // extern "C"
