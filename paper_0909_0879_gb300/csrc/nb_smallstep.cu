// One shared Hermite step of a small system in one launch: prediction of
// every particle, force + jerk of all of them, correction (paper Sec. 2.2); and
// its symplectic runs (below).
//
// Bound: latency.  At N = 1,024 the pairs take 1 us of the FP32 pipes, while
// three launches (predictor, force, fix-up + corrector) cost a launch, a drain
// and cold loads each: 24.4 us per step.  Here a CTA owns 8 or 16 particles
// from the prediction to the correction; the only exchange is that of the
// records, through global memory and one grid barrier (cooperative launch: all
// CTAs are resident).  Split precision, per step: N = 256 12.4 us, N = 1,024
// 14.4 us (18.4 with 16 particles per CTA), N = 2,048 22.6 us; FP32 12.3 / 14.4 /
// 20.5 us.  Up to 2,288 particles the SMs hold them at 16 each, from there to
// 4,096 (the records' shared memory) at 32, two per warp: N = 2,500 / 3,000 /
// 4,096 38.9 / 45.1 / 61.3 us with three launches -> 34.8 / 38.9 / 45.1.
//
// The sums are those of the short-list force shape (a warp per i-particle,
// 8 records per lane and tile), segment by segment of its split over CTAs, and
// of the fix-up: the same bits as the separate launches.
#include "nb_device.cuh"

namespace nbi {
namespace {

constexpr int kWarps = 16;   // per CTA
constexpr int kBlock = 16;   // i-particles per block of the short-list shape's split
constexpr int kSmallMostTiles = 16;

// All CTAs arrive and leave together.  *bar counts arrivals for good: every
// launch adds a whole multiple of the grid.  False (for all threads) after
// kWaitLimit unsuccessful polls.
__device__ __forceinline__ bool grid_barrier(unsigned long long *bar) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned long long G = gridDim.x;
    const unsigned long long goal = (atomicAdd(bar, 1ull) / G + 1) * G;
    int ok = 0;
    for (uint32_t it = 0; it < kWaitLimit && !ok; ++it) {
      unsigned long long now;
      asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(now) : "l"(bar) : "memory");
      ok = now >= goal;
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// NI i-particles per CTA: 16 / NI warps each, the segments of the split going to
// the warps in turn, or NI / 16 per warp.
template <int PREC, int NI>
__global__ void __launch_bounds__(32 * kWarps, 1) small_step_kernel(const SmallStepArgs A) {
  constexpr int WPI = NI < kWarps ? kWarps / NI : 1, IPW = NI > kWarps ? NI / kWarps : 1;
  static_assert(NI <= 32, "the prediction is one warp's");
  using O = dev::VOps<float>;
  extern __shared__ __align__(16) float4 rec[];
  __shared__ double s_f[NI][6];
  __shared__ float2 s_seg[NI][kSmallMostTiles][6];  // the split's partial sums
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int n = static_cast<int>(A.n), n_jt = static_cast<int>(A.n_jt), n_pad = n_jt * kJT;
  const int ctas = (n + NI - 1) / NI;  // the CTAs after them write tile frames
  const int b = blockIdx.x, k0 = b * NI;

  // the corrector's particle: three lanes each, ten per warp
  dev::PState st;
  const int eq = lane < 30 ? wid * 10 + lane / 3 : NI, cq = lane % 3;
  const int ci = eq < NI && b < ctas && k0 + eq < n ? k0 + eq : -1;
  if (ci >= 0) dev::load_state(ci, A.x, A.v, A.a, A.jk, A.t_tick, A.lev, st);
  if (b < ctas && wid == 2 && lane < NI && k0 + lane < n) {
    const int k = k0 + lane;
    const float dt = static_cast<float>(A.t_next - A.t_tick[k]) * static_cast<float>(dev::kTick);
    float xh[3], xl[3], vp[3];
    float4 l;
    dev::predict_ds(A.x, A.v, A.a, A.jk, k, dt, xh, xl, vp);
    dev::store_records_ds(k, xh, xl, vp, A.m[k], PREC, A.jhi, A.jlo, A.jvel, &l);
  }
  if (!grid_barrier(A.bar)) {
    if (tid == 0) atomicOr(A.err, kErrWaitTimeout);
    return;
  }
  if (b >= ctas) {
    // a tile's frame, for whoever takes the far field at this prediction
    const int64_t jt = b - ctas, j = jt * kJT + tid;
    if (tid >= kJT) return;
    dev::tile_frame(jt, j, j < n, __ldcg(A.jhi + j), __ldcg(A.jlo + j), A.jrel, A.tinfo);
    return;
  }
  float4 *s_hi = rec, *s_lo = rec + n_pad, *s_v = rec + (PREC ? 2 : 1) * n_pad;
  for (int j = tid; j < n_pad; j += 32 * kWarps) {
    s_hi[j] = __ldcg(A.jhi + j);
    if (PREC) s_lo[j] = __ldcg(A.jlo + j);
    s_v[j] = __ldcg(A.jvel + j);
  }
  __syncthreads();

  // the segments of the i-block's tiles: owners plo .. phi of the split (a
  // warp's particles lie in one i-block of 16)
  const int blocks = (n + kBlock - 1) / kBlock;
  const uint64_t U = static_cast<uint64_t>(blocks) * n_jt;
  const int blk = NI <= kBlock ? k0 / kBlock  // (the last: warps past n)
                               : min((k0 + wid / WPI * IPW) / kBlock, blocks - 1);
  const uint64_t u0 = static_cast<uint64_t>(blk) * n_jt;
  const int plo = dev::owner_of(u0, U, A.P), phi = dev::owner_of(u0 + n_jt - 1, U, A.P);
  {
    const int e0 = wid / WPI * IPW;
    float nx[IPW][3], nl[IPW][3], nv[IPW][3];
#pragma unroll
    for (int w = 0; w < IPW; ++w) {
      const int i = k0 + e0 + w < n ? k0 + e0 + w : 0;
      const float4 hi = s_hi[i], wi = s_v[i];
      const float4 li = PREC ? s_lo[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      nx[w][0] = -hi.x, nx[w][1] = -hi.y, nx[w][2] = -hi.z;
      nl[w][0] = -li.x, nl[w][1] = -li.y, nl[w][2] = -li.z;
      nv[w][0] = -wi.x, nv[w][1] = -wi.y, nv[w][2] = -wi.z;
    }
    int t0 = 0;
    for (int p = plo; p <= phi; ++p) {
      const uint64_t ue = dev::udiv(U * static_cast<uint64_t>(p + 1), static_cast<uint64_t>(A.P));
      const int t1 = p == phi ? n_jt : static_cast<int>(ue - u0);
      if ((p - plo) % WPI == wid % WPI) {
        float sh[IPW][6], sl[IPW][6];
#pragma unroll
        for (int w = 0; w < IPW; ++w)
#pragma unroll
          for (int c = 0; c < 6; ++c) sh[w][c] = sl[w][c] = 0.f;
        for (int jt = t0; jt < t1; ++jt) {
          float pa[IPW][3], p1[IPW][3], p2[IPW][3];
#pragma unroll
          for (int w = 0; w < IPW; ++w)
#pragma unroll
            for (int c = 0; c < 3; ++c) pa[w][c] = p1[w][c] = p2[w][c] = 0.f;
#pragma unroll
          for (int q = 0; q < kJT / 32; ++q) {
            const int j = jt * kJT + q * 32 + lane;
            const float4 hj = s_hi[j], wj = s_v[j];
            const float4 lj = PREC ? s_lo[j] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < IPW; ++w) {
              float dx, dy, dz;
              if (PREC) {
                dx = O::add(O::add(hj.x, nx[w][0]), O::add(lj.x, nl[w][0]));
                dy = O::add(O::add(hj.y, nx[w][1]), O::add(lj.y, nl[w][1]));
                dz = O::add(O::add(hj.z, nx[w][2]), O::add(lj.z, nl[w][2]));
              } else {
                dx = O::add(hj.x, nx[w][0]);
                dy = O::add(hj.y, nx[w][1]);
                dz = O::add(hj.z, nx[w][2]);
              }
              const float ux = O::add(wj.x, nv[w][0]), uy = O::add(wj.y, nv[w][1]),
                          uz = O::add(wj.z, nv[w][2]);
              const float r2 = O::fma(dx, dx, O::fma(dy, dy, O::fma(dz, dz, A.eps2)));
              const float rinv = O::rsq<0>(r2);
              const float rinv2 = O::mul(rinv, rinv);
              const float mr3 = O::mul(O::mul(hj.w, rinv), rinv2);
              const float rv = O::fma(dx, ux, O::fma(dy, uy, O::mul(dz, uz)));
              const float cc = O::mul(O::mul(rv, rinv2), mr3);
              pa[w][0] = O::fma(mr3, dx, pa[w][0]);
              pa[w][1] = O::fma(mr3, dy, pa[w][1]);
              pa[w][2] = O::fma(mr3, dz, pa[w][2]);
              p1[w][0] = O::fma(mr3, ux, p1[w][0]);
              p1[w][1] = O::fma(mr3, uy, p1[w][1]);
              p1[w][2] = O::fma(mr3, uz, p1[w][2]);
              p2[w][0] = O::fma(cc, dx, p2[w][0]);
              p2[w][1] = O::fma(cc, dy, p2[w][1]);
              p2[w][2] = O::fma(cc, dz, p2[w][2]);
            }
          }
#pragma unroll
          for (int w = 0; w < IPW; ++w)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              const float jt3 = fmaf(-3.f, p2[w][c], p1[w][c]);
              if (PREC) {
                dev::ds_add(sh[w][c], sl[w][c], pa[w][c]);
                dev::ds_add(sh[w][3 + c], sl[w][3 + c], jt3);
              } else {
                sh[w][c] += pa[w][c];
                sh[w][3 + c] += jt3;
              }
            }
        }
#pragma unroll
        for (int w = 0; w < IPW; ++w) {
#pragma unroll
          for (int off = 1; off < 32; off <<= 1)
#pragma unroll
            for (int c = 0; c < 6; ++c) {
              const float oh = __shfl_xor_sync(0xffffffffu, sh[w][c], off);
              const float ol = __shfl_xor_sync(0xffffffffu, sl[w][c], off);
              dev::ds_add_pair(sh[w][c], sl[w][c], oh, ol, sh[w][c], sl[w][c]);
            }
          if (lane == 0)
#pragma unroll
            for (int c = 0; c < 6; ++c) s_seg[e0 + w][p - plo][c] = make_float2(sh[w][c], sl[w][c]);
        }
      }
      t0 = t1;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < IPW; ++q) {
    const int e = wid * IPW + q;
    if (e >= NI) break;
    // the fix-up's sum: lane q has segment q
    float h[6], l[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      h[c] = l[c] = 0.f;
      if (plo == phi) {
        h[c] = s_seg[e][0][c].x;
        l[c] = s_seg[e][0][c].y;
      } else if (lane <= phi - plo) {
        const float2 w = s_seg[e][lane][c];
        dev::ds_add_pair(h[c], l[c], w.x, w.y, h[c], l[c]);
      }
    }
    if (plo != phi) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          const float oh = __shfl_xor_sync(0xffffffffu, h[c], off);
          const float ol = __shfl_xor_sync(0xffffffffu, l[c], off);
          dev::ds_add_pair(h[c], l[c], oh, ol, h[c], l[c]);
        }
    }
    if (lane < 6) {
      float hh = h[0], ll = l[0];
#pragma unroll
      for (int c = 1; c < 6; ++c)
        if (lane == c) {
          hh = h[c];
          ll = l[c];
        }
      s_f[e][lane] = dev::ds_to_double(hh, ll, A.G);
    }
  }
  __syncthreads();
  if (ci >= 0) {
    const double an[3] = {s_f[eq][0], s_f[eq][1], s_f[eq][2]};
    const double jn[3] = {s_f[eq][3], s_f[eq][4], s_f[eq][5]};
    int nv = min(n - k0, NI) - wid * 10;  // this warp's particles
    nv = nv < 10 ? nv : 10;
    const unsigned mask = (1u << (3 * nv)) - 1u;
    dev::correct_vals3(cq, mask, lane - cq, ci, st, an, jn, A.t_next, A.x, A.v, A.a, A.jk,
                       A.t_tick, A.lev, A.eta, A.lev_min, A.lev_max, 0, A.n_clamped, nullptr,
                       &A.ext, nullptr, nullptr);
  }
}

// Acceleration of the CTA's NI particles (k0 ..) from the records in shared
// memory, into s_f: the sums of the acceleration-only short-list shape and its
// fix-up.  Called by the whole CTA.
template <int PREC, int NI>
__device__ __forceinline__ void small_acc(int n, int n_jt, int k0, int P, float eps2, double G,
                                          const float4 *s_hi, const float4 *s_lo,
                                          float2 (*s_seg)[kSmallMostTiles][3], double (*s_f)[3]) {
  using O = dev::VOps<float>;
  constexpr int WPI = NI < kWarps ? kWarps / NI : 1, IPW = NI > kWarps ? NI / kWarps : 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int blocks = (n + kBlock - 1) / kBlock;
  const uint64_t U = static_cast<uint64_t>(blocks) * n_jt;
  const int blk = NI <= kBlock ? k0 / kBlock
                               : min((k0 + wid / WPI * IPW) / kBlock, blocks - 1);
  const uint64_t u0 = static_cast<uint64_t>(blk) * n_jt;
  const int plo = dev::owner_of(u0, U, P), phi = dev::owner_of(u0 + n_jt - 1, U, P);
  const int e0 = wid / WPI * IPW;
  float nx[IPW][3], nl[IPW][3];
#pragma unroll
  for (int w = 0; w < IPW; ++w) {
    const int i = k0 + e0 + w < n ? k0 + e0 + w : 0;
    const float4 hi = s_hi[i];
    const float4 li = PREC ? s_lo[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    nx[w][0] = -hi.x, nx[w][1] = -hi.y, nx[w][2] = -hi.z;
    nl[w][0] = -li.x, nl[w][1] = -li.y, nl[w][2] = -li.z;
  }
  int t0 = 0;
  for (int p = plo; p <= phi; ++p) {
    const uint64_t ue = dev::udiv(U * static_cast<uint64_t>(p + 1), static_cast<uint64_t>(P));
    const int t1 = p == phi ? n_jt : static_cast<int>(ue - u0);
    if ((p - plo) % WPI == wid % WPI) {
      float sh[IPW][3], sl[IPW][3];
#pragma unroll
      for (int w = 0; w < IPW; ++w)
#pragma unroll
        for (int c = 0; c < 3; ++c) sh[w][c] = sl[w][c] = 0.f;
      for (int jt = t0; jt < t1; ++jt) {
        float pa[IPW][3];
#pragma unroll
        for (int w = 0; w < IPW; ++w)
#pragma unroll
          for (int c = 0; c < 3; ++c) pa[w][c] = 0.f;
#pragma unroll
        for (int q = 0; q < kJT / 32; ++q) {
          const int j = jt * kJT + q * 32 + lane;
          const float4 hj = s_hi[j];
          const float4 lj = PREC ? s_lo[j] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int w = 0; w < IPW; ++w) {
            float dx, dy, dz;
            if (PREC) {
              dx = O::add(O::add(hj.x, nx[w][0]), O::add(lj.x, nl[w][0]));
              dy = O::add(O::add(hj.y, nx[w][1]), O::add(lj.y, nl[w][1]));
              dz = O::add(O::add(hj.z, nx[w][2]), O::add(lj.z, nl[w][2]));
            } else {
              dx = O::add(hj.x, nx[w][0]);
              dy = O::add(hj.y, nx[w][1]);
              dz = O::add(hj.z, nx[w][2]);
            }
            const float r2 = O::fma(dx, dx, O::fma(dy, dy, O::fma(dz, dz, eps2)));
            const float rinv = O::rsq<0>(r2);
            const float mr3 = O::mul(O::mul(hj.w, rinv), O::mul(rinv, rinv));
            pa[w][0] = O::fma(mr3, dx, pa[w][0]);
            pa[w][1] = O::fma(mr3, dy, pa[w][1]);
            pa[w][2] = O::fma(mr3, dz, pa[w][2]);
          }
        }
#pragma unroll
        for (int w = 0; w < IPW; ++w)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            if (PREC)
              dev::ds_add(sh[w][c], sl[w][c], pa[w][c]);
            else
              sh[w][c] += pa[w][c];
          }
      }
#pragma unroll
      for (int w = 0; w < IPW; ++w) {
#pragma unroll
        for (int off = 1; off < 32; off <<= 1)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float oh = __shfl_xor_sync(0xffffffffu, sh[w][c], off);
            const float ol = __shfl_xor_sync(0xffffffffu, sl[w][c], off);
            dev::ds_add_pair(sh[w][c], sl[w][c], oh, ol, sh[w][c], sl[w][c]);
          }
        if (lane == 0)
#pragma unroll
          for (int c = 0; c < 3; ++c) s_seg[e0 + w][p - plo][c] = make_float2(sh[w][c], sl[w][c]);
      }
    }
    t0 = t1;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < IPW; ++q) {
    const int e = wid * IPW + q;
    if (e >= NI) break;
    float h[3], l[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      h[c] = l[c] = 0.f;
      if (plo == phi) {
        h[c] = s_seg[e][0][c].x;
        l[c] = s_seg[e][0][c].y;
      } else if (lane <= phi - plo) {
        const float2 w = s_seg[e][lane][c];
        dev::ds_add_pair(h[c], l[c], w.x, w.y, h[c], l[c]);
      }
    }
    if (plo != phi) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float oh = __shfl_xor_sync(0xffffffffu, h[c], off);
          const float ol = __shfl_xor_sync(0xffffffffu, l[c], off);
          dev::ds_add_pair(h[c], l[c], oh, ol, h[c], l[c]);
        }
    }
    if (lane < 3)
      s_f[e][lane] = dev::ds_to_double(dev::sel3(h, lane), dev::sel3(l, lane), G);
  }
  __syncthreads();
}

// A run of symplectic steps of a small system in one launch: a CTA keeps its
// particles' x and v in registers (one thread each) from the first step to the
// last; per stage the records cross one grid barrier, through two buffers in
// turn (a CTA writes a buffer again only after the barrier that all CTAs enter
// with their reads of it done).  With init the acceleration at the start is
// evaluated first, otherwise A.a holds it.  The arithmetic of kick_drift_kernel,
// the acceleration-only force and its fix-up: the same bits.  Bound: latency (a
// stage of separate launches is three of them).  Whole calls of one step with
// read-back, before -> now: leapfrog in the Galactic field N = 1,191 114 -> 66 us,
// sixth order FP32 N = 1,000 124 -> 82, split precision N = 2,300 200 -> 132, with
// the field N = 3,500 424 -> 270 (no graph to capture: a first call 192 -> 109 at
// N = 1,191).
template <int PREC, int NI>
__global__ void __launch_bounds__(32 * kWarps, 1) small_symplectic_kernel(const SmallSympArgs A) {
  extern __shared__ __align__(16) float4 rec[];
  __shared__ double s_f[NI][3];
  __shared__ float2 s_seg[NI][kSmallMostTiles][3];
  const int tid = threadIdx.x;
  const int n = static_cast<int>(A.n), n_jt = static_cast<int>(A.n_jt), n_pad = n_jt * kJT;
  const int k0 = blockIdx.x * NI, k = k0 + tid;
  const bool own = tid < NI && k < n;
  float4 *s_hi = rec, *s_lo = rec + n_pad;
  if (blockIdx.x == 0)  // padding of the second buffer: zero mass far away
    for (int j = n + tid; j < n_pad; j += 32 * kWarps) {
      A.hi[1][j] = make_float4(1.0e15f, 1.0e15f, 1.0e15f, 0.f);
      if (PREC) A.lo[1][j] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  double x[3], v[3], a[3], m = 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    x[c] = own ? A.x[3 * k + c] : 0.0;
    v[c] = own ? A.v[3 * k + c] : 0.0;
    a[c] = own ? A.a[3 * k + c] : 0.0;
  }
  if (own) m = A.m[k];
  int buf = 0;
  // stage -1: the acceleration at the start
  for (int64_t q = A.init ? -1 : 0; q < A.stages; ++q) {
    const int st = q < 0 ? 0 : static_cast<int>(q % A.S);
    if (own) {
      if (q >= 0) {
        if (A.h[st] != 0.0)
#pragma unroll
          for (int c = 0; c < 3; ++c) v[c] = fma(A.h[st], a[c], v[c]);
        if (A.d[st] != 0.0)
#pragma unroll
          for (int c = 0; c < 3; ++c) x[c] = fma(A.d[st], v[c], x[c]);
      }
      float hx[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) hx[c] = dev::d2f_rn(x[c]);
      A.hi[buf][k] = make_float4(hx[0], hx[1], hx[2], dev::d2f_rn(m));
      if (PREC)
        A.lo[buf][k] = make_float4(dev::d2f_rn(x[0] - dev::f2d(hx[0])),
                                   dev::d2f_rn(x[1] - dev::f2d(hx[1])),
                                   dev::d2f_rn(x[2] - dev::f2d(hx[2])), 0.f);
    }
    if (!grid_barrier(A.bar)) {
      if (tid == 0) atomicOr(A.err, kErrWaitTimeout);
      return;
    }
    for (int j = tid; j < n_pad; j += 32 * kWarps) {
      s_hi[j] = __ldcg(A.hi[buf] + j);
      if (PREC) s_lo[j] = __ldcg(A.lo[buf] + j);
    }
    __syncthreads();
    small_acc<PREC, NI>(n, n_jt, k0, A.P, A.eps2, A.G, s_hi, s_lo, s_seg, s_f);
    if (own) {
#pragma unroll
      for (int c = 0; c < 3; ++c) a[c] = s_f[tid][c];
      if (A.ext.on) dev::ext_acc(A.ext, x, a);
      if (q >= 0 && st == A.S - 1 && A.close != 0.0)
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = fma(A.close, a[c], v[c]);
    }
    buf ^= 1;
  }
  if (own)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      A.x[3 * k + c] = x[c];
      A.v[3 * k + c] = v[c];
      A.a[3 * k + c] = a[c];
    }
}

}  // namespace

// 8 particles per CTA where that leaves an SM for each CTA, otherwise 16 or 32; 0:
// too many.
static int small_ni(int64_t n, int64_t n_jt, int num_sms) {
  for (int ni = 8; ni <= 32; ni *= 2)
    if ((n + ni - 1) / ni + n_jt <= num_sms) return ni;
  return 0;
}

bool small_step_fits(int64_t n, int64_t n_jt, int prec, int mask, int num_sms) {
  if (mask || n_jt > kSmallMostTiles || small_ni(n, n_jt, num_sms) == 0) return false;
  const Variant &V = variant_at(choose_variant(prec, mask, n, n_jt, num_sms));
  return V.ipt == 1 && V.tpi == 32 && V.threads == 32 * kBlock && !V.rel;
}

size_t small_step_smem(int64_t n_jt, int prec) {
  return static_cast<size_t>(n_jt) * kJT * (prec ? 3 : 2) * sizeof(float4);
}

using SmallKernel = void (*)(const SmallStepArgs);
static SmallKernel small_kernel(int prec, int ni) {
  if (ni == 8) return prec ? small_step_kernel<1, 8> : small_step_kernel<0, 8>;
  if (ni == 16) return prec ? small_step_kernel<1, 16> : small_step_kernel<0, 16>;
  return prec ? small_step_kernel<1, 32> : small_step_kernel<0, 32>;
}

// The limit belongs to the kernel, which systems of many sizes share: always the
// most that any of them takes.
cudaError_t small_step_prepare(int64_t n, int64_t n_jt, int prec, int num_sms) {
  return cudaFuncSetAttribute(small_kernel(prec, small_ni(n, n_jt, num_sms)),
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(small_step_smem(kSmallMostTiles, prec)));
}

cudaError_t launch_small_step(const SmallStepArgs &A, int prec, int num_sms, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  const int ni = small_ni(A.n, A.n_jt, num_sms);
  const int64_t ctas = (A.n + ni - 1) / ni + (prec ? A.n_jt : 0);
  cfg.gridDim = dim3(static_cast<unsigned>(ctas));
  cfg.blockDim = dim3(32 * kWarps);
  cfg.dynamicSmemBytes = small_step_smem(A.n_jt, prec);
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, small_kernel(prec, ni), A);
}

// ---- symplectic runs

static int small_symp_ni(int64_t n, int num_sms) {
  for (int ni = 8; ni <= 32; ni *= 2)
    if ((n + ni - 1) / ni <= num_sms) return ni;
  return 0;
}

using SmallSympKernel = void (*)(const SmallSympArgs);
static SmallSympKernel small_symp_kernel(int prec, int ni) {
  if (ni == 8) return prec ? small_symplectic_kernel<1, 8> : small_symplectic_kernel<0, 8>;
  if (ni == 16) return prec ? small_symplectic_kernel<1, 16> : small_symplectic_kernel<0, 16>;
  return prec ? small_symplectic_kernel<1, 32> : small_symplectic_kernel<0, 32>;
}

static size_t small_symp_smem(int64_t n_jt, int prec) {
  return static_cast<size_t>(n_jt) * kJT * (prec ? 2 : 1) * sizeof(float4);
}

bool small_symp_fits(int64_t n, int64_t n_jt, int prec, int mask, int num_sms) {
  if (mask || n_jt > kSmallMostTiles || small_symp_ni(n, num_sms) == 0) return false;
  const Variant &V = variant_at(acc_shape(choose_variant(prec, mask, n, n_jt, num_sms)));
  return V.ipt == 1 && V.tpi == 32 && V.threads == 32 * kBlock && !V.rel;
}

cudaError_t small_symp_prepare(int64_t n, int prec, int num_sms) {
  return cudaFuncSetAttribute(small_symp_kernel(prec, small_symp_ni(n, num_sms)),
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(small_symp_smem(kSmallMostTiles, prec)));
}

cudaError_t launch_small_symplectic(const SmallSympArgs &A, int prec, int num_sms,
                                    cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  const int ni = small_symp_ni(A.n, num_sms);
  cfg.gridDim = dim3(static_cast<unsigned>((A.n + ni - 1) / ni));
  cfg.blockDim = dim3(32 * kWarps);
  cfg.dynamicSmemBytes = small_symp_smem(A.n_jt, prec);
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, small_symp_kernel(prec, ni), A);
}

}  // namespace nbi
