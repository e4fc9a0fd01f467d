// Energy of a state: kinetic, softened pair potential and external field.
//
//   K = 1/2 sum m v^2,  W = -G sum_{i<j} m_i m_j / sqrt(r_ij^2 + eps^2)
//
// The pair sum is O(N^2).  In FP64 it is bound by the FP64 pipe of this
// part (one warp instruction per ~64 cycles per scheduler, ~18 of them per
// pair, and one CTA per 256 rows of a triangle: 84.1 ms at N = 65,536, 18.3 at
// 20,000, 0.90 at 1,024).  From kSplitMin particles on the pair terms are
// evaluated on the FP32 pipe in split precision, about 89 packed operations
// for two pairs, every term to about 2^-46 of itself with unbiased rounding,
// and summed in split precision and, every 64 records, FP64; the triangle is
// cut into equal ranges over 2 CTAs per SM: 6.06 / 0.64 / 0.094 ms, bound by
// the FP32 pipe (0.76 of its rate).  The total is as exact as the FP64 sum,
// whose own rounding it replaces, because the term errors are independent
// and average over the N^2 / 2 pairs: relative error against extended
// precision, rms over 36 systems of N = 1,024 to 40,000 (Salpeter masses,
// softening 0 to 1e-2, with and without hard binaries), 1.2e-16 against
// 1.6e-16.  Systems whose term errors are not independent, or too few, take the
// FP64 sum after all (see energy_final_kernel).
//
// Pair term:
//  * Positions, scaled by a power of two to |x| <= 1, are three words: h a
//    multiple of 2^-23, l a multiple of 2^-46 (|l| <= 2^-24) and the rest.  The
//    differences of h and of l are then exact in FP32, a fast two-sum makes
//    them a pair D + E, and the rest's difference joins E: |E| < 2^-46 beside the
//    rounding of D, good to 2^-70.  From a softened distance of 2^-24 on (kEnNear)
//    that is 2^-46 of the distance, and D alone is good enough to start from.
//  * y0 = rsqrt(|D|^2 + eps^2) from the MUFU (2^-22).  Each component u of y0
//    (d, eps) is g + its error term, g rounded to the grid 2^-21 (adding 6 and
//    subtracting it again); g^2 is split at 2^-23 (adding 1), so that 1 - sum
//    g^2 is exact, and the residual e = 1 - sum u^2 is good to 2^-46.  The grid
//    matters: squares of full 24-bit values have structured last bits, and
//    rounding those biases the total by 5e-16.  1/r = y0 (1 + e/2 + 3 e^2/8) is
//    a Newton step with its second-order term.
//  * m_j / r as a pair, added by an error-free two-sum.  m_j is three words: what
//    two leave out (2^-49) is the same for all particles of one mass and would
//    not average out (up to 1.8e-15 of the total).  The third is a product of its
//    own: taken into the one with e / 2 it leaves a bias of 1e-15.
// A closer pair, or one whose term is a visible part of the total (hard
// binaries), takes FP64.  (With every softened distance from 2^-46 on in split
// precision a close pair of light particles was off by up to 1e-1 of its term.)
#include "nb_device.cuh"

#include <algorithm>

namespace nbi {

namespace {

constexpr int kEnThreads = 256;

// Smallest n of the split-precision pair sum: below it the term errors have
// too few pairs to average over, and the FP64 sum takes tens of microseconds.
constexpr int64_t kSplitMin = 1024;

// Fixed-order block reduction of one double per thread.
__device__ __forceinline__ double block_sum(double v, double *sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

__global__ void kinetic_kernel(int64_t n, const double *__restrict__ m,
                               const double *__restrict__ v, double *__restrict__ part) {
  __shared__ double sh[kEnThreads];
  double s = 0.0;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) {
    const double vx = v[3 * i], vy = v[3 * i + 1], vz = v[3 * i + 2];
    s = 0.5 * m[i] * (vx * vx + vy * vy + vz * vz);
  }
  s = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// w_i = m_i sum_{j > i} m_j / sqrt(r^2 + eps^2), FP64, j staged in tiles
// from the CTA's own diagonal tile on (each pair once); the block's sum of
// w_i goes to part[blockIdx.x].
__global__ void potential_kernel(int64_t n, const double *__restrict__ m,
                                 const double *__restrict__ x, double eps2,
                                 double *__restrict__ part) {
  __shared__ double sx[kEnThreads], sy[kEnThreads], sz[kEnThreads], sm[kEnThreads];
  __shared__ double sh[kEnThreads];
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x;
  const int64_t i = i0 + threadIdx.x;
  const bool valid = i < n;
  const double xi = valid ? x[3 * i] : 0.0;
  const double yi = valid ? x[3 * i + 1] : 0.0;
  const double zi = valid ? x[3 * i + 2] : 0.0;
  double w = 0.0;
  for (int64_t j0 = i0; j0 < n; j0 += kEnThreads) {
    const int64_t jl = j0 + threadIdx.x;
    if (jl < n) {
      sx[threadIdx.x] = x[3 * jl];
      sy[threadIdx.x] = x[3 * jl + 1];
      sz[threadIdx.x] = x[3 * jl + 2];
      sm[threadIdx.x] = m[jl];
    }
    __syncthreads();
    const int cnt = (n - j0) < kEnThreads ? static_cast<int>(n - j0) : kEnThreads;
    // on the diagonal tile only j > i counts
    const int t0 = (j0 == i0) ? static_cast<int>(threadIdx.x) + 1 : 0;
    for (int t = t0; t < cnt; ++t) {
      const double dx = sx[t] - xi, dy = sy[t] - yi, dz = sz[t] - zi;
      const double s2 = dx * dx + dy * dy + dz * dz + eps2;
      w += sm[t] * rsqrt(s2);
    }
    __syncthreads();
  }
  const double wi = valid ? m[i] * w : 0.0;
  const double s = block_sum(wi, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// e_i = m_i Phi_ext(x_i); the block's sum goes to part[blockIdx.x].
__global__ void ext_potential_kernel(int64_t n, const ExtField E, const double *__restrict__ m,
                                     const double *__restrict__ x, double *__restrict__ part) {
  __shared__ double sh[kEnThreads];
  double s = 0.0;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) {
    const double xv[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
    double av[3] = {0.0, 0.0, 0.0}, phi = 0.0;
    dev::ext_field(E, xv, nullptr, av, nullptr, &phi);
    s = m[i] * phi;
  }
  s = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// ---- split-precision pair sum

// Kinetic energy and mass of the block's particles into part[blockIdx.x]
// and mpart[blockIdx.x], and the bit patterns of the largest |coordinate| and mass (non-negative doubles
// order like integers) into top[0], top[1].
__global__ void energy_scan_kernel(int64_t n, const double *__restrict__ m,
                                   const double *__restrict__ x, const double *__restrict__ v,
                                   double *__restrict__ part, double *__restrict__ mpart,
                                   unsigned long long *top) {
  __shared__ double sh[kEnThreads];
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  double s = 0.0, mi = 0.0;
  unsigned long long mx = 0, mm = 0;
  if (i < n) {
    const double vx = v[3 * i], vy = v[3 * i + 1], vz = v[3 * i + 2];
    mi = m[i];
    s = 0.5 * mi * (vx * vx + vy * vy + vz * vz);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const unsigned long long b =
          static_cast<unsigned long long>(__double_as_longlong(x[3 * i + c])) & ~(1ull << 63);
      mx = b > mx ? b : mx;
    }
    mm = static_cast<unsigned long long>(__double_as_longlong(mi)) & ~(1ull << 63);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long a = __shfl_xor_sync(0xffffffffu, mx, o);
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, mm, o);
    mx = a > mx ? a : mx;
    mm = b > mm ? b : mm;
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(top, mx);
    atomicMax(top + 1, mm);
  }
  s = block_sum(s, sh);
  mi = block_sum(mi, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = s;
    mpart[blockIdx.x] = mi;
  }
}

// Power of two that brings a positive double below 1 (its bit pattern in b);
// 1 for zero; the exponent is held to +-1000 so that it and its inverse are
// normal numbers.
__device__ __forceinline__ int down_exp(unsigned long long b) {
  if (b == 0) return 0;
  const int e = static_cast<int>(b >> 52) - 1022;
  return e < -1000 ? -1000 : (e > 1000 ? 1000 : e);
}
__device__ __forceinline__ double pow2d(int k) {
  return __longlong_as_double(static_cast<long long>(1023 + k) << 52);
}
__device__ __forceinline__ int length_exp(const unsigned long long *top, double eps) {
  const unsigned long long be = static_cast<unsigned long long>(__double_as_longlong(eps));
  return down_exp(top[0] > be ? top[0] : be);
}

// Records of a tile of kJT particles in pairs: planes of 128 float4
// (h x, y), (h z, m), (l x, y), (l z, m's low word), (rest x, y), (rest z, m's
// rest), each value of both particles side by side.
constexpr int kEnPairs = kJT / 2;
constexpr int kEnPlane = kEnPairs;  // float4 per plane
// distance of what does not count: its reciprocal root, and so every product, is 0
constexpr float kEnInf = __builtin_huge_valf();
constexpr float kEnNear = 0x1p-48f;  // square of the least softened distance
constexpr int kEnPlanes = 6;
constexpr size_t kEnTileBytes = kEnPlanes * kEnPlane * sizeof(float4);
// j-records of a unit of work: 32 pairs, a quarter of a tile
constexpr int kEnSub = 32;
constexpr int kEnSubs = kEnPairs / kEnSub;

struct EnWord {
  float h[3], l[3], r[3], mh, ml, mr;
};

__device__ __forceinline__ EnWord energy_words(const double *__restrict__ m,
                                               const double *__restrict__ x, int64_t i,
                                               double sx, double sm) {
  EnWord w;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double xs = x[3 * i + c] * sx;
    const double h = rint(xs * 0x1p23) * 0x1p-23;
    const double t = xs - h;
    const double l = rint(t * 0x1p46) * 0x1p-46;
    w.h[c] = static_cast<float>(h);
    w.l[c] = static_cast<float>(l);
    w.r[c] = static_cast<float>(t - l);
  }
  const double ms = m[i] * sm;
  w.mh = static_cast<float>(ms);
  const double mt = ms - static_cast<double>(w.mh);
  w.ml = static_cast<float>(mt);
  w.mr = static_cast<float>(mt - static_cast<double>(w.ml));
  return w;
}

// The records of a tile, and the sum of its squared (scaled) masses into
// m2part[blockIdx.x].
__global__ void __launch_bounds__(kEnPairs)
    energy_records_kernel(int64_t n, const double *__restrict__ m, const double *__restrict__ x,
                          double eps, const unsigned long long *top, unsigned char *recs,
                          double *__restrict__ m2part) {
  __shared__ double sh[kEnPairs];
  double m2 = 0.0;
  const double sx = pow2d(-length_exp(top, eps)), sm = pow2d(-down_exp(top[1]));
  const int k = threadIdx.x;
  float4 *p = reinterpret_cast<float4 *>(recs + static_cast<size_t>(blockIdx.x) * kEnTileBytes);
  EnWord w[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * kJT + 2 * k + q;
    if (j < n) {
      w[q] = energy_words(m, x, j, sx, sm);
      m2 += (m[j] * sm) * (m[j] * sm);
    } else {  // no mass, outside the box
      w[q] = EnWord{{2.f, 2.f, 2.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, 0.f, 0.f, 0.f};
    }
  }
  const EnWord &a = w[0], &b = w[1];
  p[k] = make_float4(a.h[0], b.h[0], a.h[1], b.h[1]);
  p[kEnPlane + k] = make_float4(a.h[2], b.h[2], a.mh, b.mh);
  p[2 * kEnPlane + k] = make_float4(a.l[0], b.l[0], a.l[1], b.l[1]);
  p[3 * kEnPlane + k] = make_float4(a.l[2], b.l[2], a.ml, b.ml);
  p[4 * kEnPlane + k] = make_float4(a.r[0], b.r[0], a.r[1], b.r[1]);
  p[5 * kEnPlane + k] = make_float4(a.r[2], b.r[2], a.mr, b.mr);
  m2 = block_sum(m2, sh);
  if (k == 0) m2part[blockIdx.x] = m2;
}

// Sum of the blocks' mass sums, by the whole CTA in a fixed order.
__device__ __forceinline__ double mass_sum(int64_t nb, const double *__restrict__ mpart,
                                           double *sh) {
  double s = 0.0;
  for (int64_t b = threadIdx.x; b < nb; b += blockDim.x) s += mpart[b];
  return block_sum(s, sh);
}

// First unit of row ib (i-block of kEnThreads = kJT particles) of the
// triangle of quarter tiles at and after the row's own tile.
__host__ __device__ __forceinline__ int64_t tri_start(int64_t n_t, int64_t ib) {
  return kEnSubs * (ib * n_t - ib * (ib - 1) / 2);
}

// One thread per i-particle, two j-records per packed instruction; every
// CTA takes an equal contiguous range of units and leaves the sum of its
// m_i w_i, w_i = sum_{j > i} m_j / s_ij, in part[blockIdx.x].
template <int SOFT>
__global__ void __launch_bounds__(kEnThreads, 2)
    energy_pairs_kernel(int64_t n, int64_t n_t, const double *__restrict__ m,
                        const double *__restrict__ x, double eps, const unsigned long long *top,
                        const unsigned char *__restrict__ recs,
                        const double *__restrict__ mpart, double *__restrict__ part) {
  using V = float2;
  using O = dev::VOps<V>;
  __shared__ float4 sj[kEnPlanes][kEnSub];
  __shared__ double sh[kEnThreads];
  const int tid = threadIdx.x;
  const int ex = length_exp(top, eps), em = down_exp(top[1]);
  const double sx = pow2d(-ex), sm = pow2d(-em);
  const double eps_s = eps * sx;
  const float eh = static_cast<float>(eps_s);
  const float el = static_cast<float>(eps_s - static_cast<double>(eh));
  const double msum = mass_sum(n_t, mpart, sh) * sm;
  const int64_t units = tri_start(n_t, n_t);
  const int64_t u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
  double total = 0.0;
  if (u0 < u1) {
    int64_t lo = 0, hi = n_t - 1;  // row of u0
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) / 2;
      if (tri_start(n_t, mid) <= u0)
        lo = mid;
      else
        hi = mid - 1;
    }
    int64_t ib = lo;
    int64_t sub = kEnSubs * ib + (u0 - tri_start(n_t, ib));  // quarter tile
    for (int64_t u = u0; u < u1; ++ib, sub = kEnSubs * ib) {
      const int64_t i = ib * kJT + tid;
      const bool real = i < n;
      EnWord w = EnWord{{3.f, 3.f, 3.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, 0.f, 0.f, 0.f};
      if (real) w = energy_words(m, x, i, sx, sm);
      // m_j / r of a pair that is 1.4e-3 of the least |W| can be, M^2 / (10 L) where
      // no particle dominates (see energy_final_kernel)
      const float p_max = real ? static_cast<float>(1.4e-4 * msum * msum / (m[i] * sm)) : 3e38f;
      V nh[3], nl[3], nr[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        nh[c] = O::bc(-w.h[c]);
        nl[c] = O::bc(-w.l[c]);
        nr[c] = O::bc(-w.r[c]);
      }
      const V one = O::bc(1.f), mone = O::bc(-1.f), two = O::bc(2.f);
      const V grid = O::bc(6.f), ngrid = O::bc(-6.f);  // ulp 2^-21 in [4, 8)
      const V veh = O::bc(eh), vel = O::bc(el), ve2 = O::bc(eh * eh);
      auto sub2 = [&](V a, V b) { return O::fma(b, mone, a); };  // a - b
      double wi = 0.0;
      V ah = O::bc(0.f), nal = O::bc(0.f);  // sum of m_j / r: ah - nal
      auto flush = [&]() {
        wi += (dev::f2d(ah.x) - dev::f2d(nal.x)) + (dev::f2d(ah.y) - dev::f2d(nal.y));
        ah = nal = O::bc(0.f);
      };
      for (; u < u1 && sub < kEnSubs * n_t; ++u, ++sub) {
        const int64_t jt = sub / kEnSubs;
        const int k0 = static_cast<int>(sub - jt * kEnSubs) * kEnSub;
        const float4 *src =
            reinterpret_cast<const float4 *>(recs + static_cast<size_t>(jt) * kEnTileBytes);
        __syncthreads();
        if (tid < kEnPlanes * kEnSub)
          sj[tid / kEnSub][tid % kEnSub] = src[(tid / kEnSub) * kEnPlane + k0 + tid % kEnSub];
        __syncthreads();
        const bool own = jt == ib;
#pragma unroll 2
        for (int k = 0; k < kEnSub; ++k) {
          const float4 a = sj[0][k], b = sj[1][k], c4 = sj[2][k], d4 = sj[3][k], e4 = sj[4][k];
          const float2 f2 = reinterpret_cast<const float2 *>(&sj[5][k])[0];
          const V hj[3] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y)};
          const V lj[3] = {make_float2(c4.x, c4.y), make_float2(c4.z, c4.w),
                           make_float2(d4.x, d4.y)};
          const V rj[3] = {make_float2(e4.x, e4.y), make_float2(e4.z, e4.w),
                           f2};
          V mh = make_float2(b.z, b.w), ml = make_float2(d4.z, d4.w);
          V D[3], E[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const V dh = O::add(hj[c], nh[c]), dl = O::add(lj[c], nl[c]);
            D[c] = O::add(dh, dl);
            E[c] = O::add(sub2(dl, sub2(D[c], dh)), O::add(rj[c], nr[c]));
          }
          V R = O::mul(D[2], D[2]);
          if (SOFT) R = O::fma(D[2], D[2], ve2);
          R = O::fma(D[0], D[0], O::fma(D[1], D[1], R));
          if (own) {  // only j > i counts
            const int j = 2 * (k0 + k);
            if (j <= tid) R.x = kEnInf;
            if (j + 1 <= tid) R.y = kEnInf;
          }
          // pairs in FP64: distances too short for the words, and terms so large
          // that their own rounding would show in the total
          V y = O::rsq<0>(R), p = O::mul(mh, y);
          const bool bx = R.x < kEnNear || p.x > p_max, by = R.y < kEnNear || p.y > p_max;
          if (__any_sync(0xffffffffu, bx || by)) {
            for (int q = 0; q < 2; ++q) {
              if (!(q ? by : bx)) continue;
              const int64_t j = jt * kJT + 2 * (k0 + k) + q;
              if (real && j < n) {
                const double dx = (x[3 * j] - x[3 * i]) * sx;
                const double dy = (x[3 * j + 1] - x[3 * i + 1]) * sx;
                const double dz = (x[3 * j + 2] - x[3 * i + 2]) * sx;
                wi += m[j] * sm * rsqrt(dx * dx + dy * dy + dz * dz + eps_s * eps_s);
              }
            }
            if (bx) p.x = y.x = 0.f;
            if (by) p.y = y.y = 0.f;
          }
          const V ny = O::mul(y, mone);
          V s = one, qe = O::bc(0.f), zz = O::bc(0.f);
          V gs[4], ngs[4];
          // a component y (d + e) of the unit vector as g - ng, g on the grid
          // 2^-21; 1 - sum g^2 is s - qe exactly
          auto comp = [&](int q, V d, V e) {
            const V g = O::add(O::fma(y, d, grid), ngrid);
            const V ng = O::fma(ny, e, O::fma(ny, d, g));
            const V nq = O::fma(O::fma(g, g, one), mone, one);
            s = O::add(s, nq);
            qe = O::add(qe, O::fma(g, g, nq));
            zz = O::fma(ng, ng, zz);
            gs[q] = g;
            ngs[q] = ng;
          };
          comp(0, D[0], E[0]);
          comp(1, D[1], E[1]);
          comp(2, D[2], E[2]);
          if (SOFT) comp(3, veh, vel);
          // the small square first: each later rounding then falls anywhere
          // between two floats, so none of them is biased
          V cr = O::mul(zz, O::bc(-0.5f));
#pragma unroll
          for (int q = 0; q < (SOFT ? 4 : 3); ++q) cr = O::fma(ngs[q], gs[q], cr);
          const V e = O::fma(two, cr, sub2(s, qe));
          // m / r = m y (1 + e / 2 + 3 e^2 / 8) = p - np
          const V w2 = O::mul(e, O::mul(e, O::bc(-0.375f)));
          // read here, where it is needed: 3 % of the time
          const V mr = reinterpret_cast<const float2 *>(&sj[5][k])[1];
          V np = O::fma(p, w2, O::fma(mr, ny, O::fma(mh, ny, p)));
          np = O::fma(mh, O::mul(ny, O::mul(e, O::bc(0.5f))), O::fma(ml, ny, np));
          const V t = O::add(ah, p);
          const V bb = sub2(t, ah);
          const V err = O::add(sub2(ah, sub2(t, bb)), sub2(p, bb));
          ah = t;
          nal = sub2(O::add(nal, np), err);
        }
        // 64 records at a time: the low words' own rounding grows with the
        // number of terms
        flush();
      }
      if (real) total += m[i] * wi;
    }
  }
  const double t = block_sum(total, sh);
  // w_i is in units of (scaled mass) / (scaled length)
  if (tid == 0) part[blockIdx.x] = t * pow2d(-ex) * pow2d(em);
}

// Sums in a fixed order: out = {sum kin, -G sum pot, sum ext}; out[3] says whether
// the split-precision pair sum is to be thrown away for the FP64 one, because its
// terms' roundings would not average out:
//  * One particle dominates: the squares of the masses add up to more than a
//    fourth of the square of their sum.  The pair energy is then the terms of that
//    particle, too few of them (1,100 particles around a heavy one: 1.5e-15 against
//    6e-16 in FP64), and with light particles below 2^-64 of the heavy one the
//    correction of a term leaves the FP32 range (5e-31: 2e-8, below 1e-38 the
//    whole term).
//  * The softening is more than a fourth of the harmonic mean softened distance:
//    the distances hardly differ, and neither do the roundings (Plummer spheres of
//    1,024 and 1,500, softening over that distance 0.1 / 0.26 / 0.49 / 0.99: mean
//    error 6e-17 / 1.1e-16 / 2.5e-16 / 3e-16, FP64 1e-16 throughout).
__global__ void energy_final_kernel(int64_t nb, const double *__restrict__ kin, int64_t n_pot,
                                    const double *__restrict__ pot, int64_t n_ext,
                                    const double *__restrict__ ext, double G, double eps,
                                    const unsigned long long *top,
                                    const double *__restrict__ mpart,
                                    const double *__restrict__ m2part,
                                    double *__restrict__ out) {
  // the five sums side by side
  __shared__ double sh[5][kEnThreads];
  const double *const src[5] = {kin, pot, ext, mpart, m2part};
  const int64_t cnt[5] = {nb, n_pot, n_ext, mpart ? nb : 0, mpart ? nb : 0};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    double s = 0.0;
    for (int64_t b = threadIdx.x; b < cnt[k]; b += blockDim.x) s += src[k][b];
    sh[k][threadIdx.x] = s;
  }
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o)
#pragma unroll
      for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  const double w = sh[1][0];
  bool redo = false;
  if (mpart) {
    const double sm = pow2d(-down_exp(top[1]));
    const double mass = sh[3][0] * sm, m2 = sh[4][0], most = 0.25 * mass * mass;
    redo = !(m2 <= most) || !(2.0 * eps * (w * sm * sm) <= most);
  }
  out[0] = sh[0][0];
  out[1] = -G * w;
  out[2] = sh[2][0];
  out[3] = redo ? 1.0 : 0.0;
}

}  // namespace

int64_t energy_scratch_doubles(int64_t n) {
  const int64_t nb = (n + kEnThreads - 1) / kEnThreads;
  return 4 * nb + std::max<int64_t>(nb, kEnMaxCtas) + 6;
}

size_t energy_record_bytes(int64_t n) {
  return n < kSplitMin ? 0 : static_cast<size_t>((n + kJT - 1) / kJT) * kEnTileBytes;
}

cudaError_t launch_energy(int64_t n, const double *m, const double *x, const double *v,
                          double G, double eps, const ExtField &E, double *red,
                          unsigned char *recs, int num_sms, double *d_out, cudaStream_t s,
                          int *launches) {
  const int64_t nb = (n + kEnThreads - 1) / kEnThreads;
  const unsigned g = static_cast<unsigned>(nb);
  double *pk = red;
  double *pe = pk + nb;
  double *pw = pe + nb;
  unsigned long long *top =
      reinterpret_cast<unsigned long long *>(red + energy_scratch_doubles(n) - 6);
  double *pm = pw + std::max<int64_t>(nb, kEnMaxCtas);
  double *pm2 = pm + nb;
  int64_t np = nb;
  if (recs) {
    cudaError_t e = cudaMemsetAsync(top, 0, 2 * sizeof(*top), s);
    if (e != cudaSuccess) return e;
    energy_scan_kernel<<<g, kEnThreads, 0, s>>>(n, m, x, v, pk, pm, top);
    energy_records_kernel<<<g, kEnPairs, 0, s>>>(n, m, x, eps, top, recs, pm2);
    np = std::min<int64_t>(std::min<int64_t>(2 * num_sms, kEnMaxCtas), tri_start(nb, nb));
    const unsigned gp = static_cast<unsigned>(np);
    if (eps > 0.0)
      energy_pairs_kernel<1><<<gp, kEnThreads, 0, s>>>(n, nb, m, x, eps, top, recs, pm, pw);
    else
      energy_pairs_kernel<0><<<gp, kEnThreads, 0, s>>>(n, nb, m, x, eps, top, recs, pm, pw);
    if (launches) *launches += 3;
  } else {
    kinetic_kernel<<<g, kEnThreads, 0, s>>>(n, m, v, pk);
    potential_kernel<<<g, kEnThreads, 0, s>>>(n, m, x, eps * eps, pw);
    if (launches) *launches += 2;
  }
  if (E.on) ext_potential_kernel<<<g, kEnThreads, 0, s>>>(n, E, m, x, pe);
  energy_final_kernel<<<1, kEnThreads, 0, s>>>(nb, pk, np, pw, E.on ? nb : 0, pe, G, eps, top,
                                               recs ? pm : nullptr, pm2, d_out);
  if (launches) *launches += E.on ? 2 : 1;
  return cudaGetLastError();
}

}  // namespace nbi
