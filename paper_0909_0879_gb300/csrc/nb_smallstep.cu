// One shared Hermite step of a small system in one launch: prediction of
// every particle, force + jerk of all of them, correction (paper Sec. 2.2).
//
// Bound: latency.  At N = 1,024 the pairs take 2.6 us of an SM's FP32 pipe,
// while three launches (predictor, force, fix-up + corrector) cost a launch,
// a drain and cold loads each: 24.4 us per step.  Here a CTA owns an i-block
// of 16 particles from the prediction to the correction; the only exchange is
// that of the records, through global memory and one grid barrier (cooperative
// launch: all CTAs are resident).  SMALLSTEP_FIGS
//
// The sums are those of the short-list force shape (a warp per i-particle,
// 8 records per lane and tile), segment by segment of its split over CTAs, and
// of the fix-up: the same bits as the separate launches.
#include "nb_device.cuh"

namespace nbi {
namespace {

constexpr int kSmallI = 16;  // i-particles (warps) per CTA

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

template <int PREC>
__global__ void __launch_bounds__(32 * kSmallI, 1) small_step_kernel(const SmallStepArgs A) {
  using O = dev::VOps<float>;
  extern __shared__ __align__(16) float4 rec[];
  __shared__ double s_f[kSmallI][6];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int n = static_cast<int>(A.n), n_jt = static_cast<int>(A.n_jt), n_pad = n_jt * kJT;
  const int n_ib = (n + kSmallI - 1) / kSmallI;
  const int b = blockIdx.x;

  // the corrector's particle: three lanes each, ten per warp
  dev::PState st;
  const int eq = lane < 30 ? wid * 10 + lane / 3 : kSmallI, cq = lane % 3;
  const int ci = eq < kSmallI && b < n_ib && b * kSmallI + eq < n ? b * kSmallI + eq : -1;
  if (ci >= 0) dev::load_state(ci, A.x, A.v, A.a, A.jk, A.t_tick, A.lev, st);
  if (b < n_ib && wid == 2 && lane < kSmallI && b * kSmallI + lane < n) {
    const int k = b * kSmallI + lane;
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
  if (b >= n_ib) {
    // a tile's frame, for whoever takes the far field at this prediction
    const int64_t jt = b - n_ib, j = jt * kJT + tid;
    if (tid >= kJT) return;
    dev::tile_frame(jt, j, j < n, __ldcg(A.jhi + j), __ldcg(A.jlo + j), A.jrel, A.tinfo);
    return;
  }
  float4 *s_hi = rec, *s_lo = rec + n_pad, *s_v = rec + (PREC ? 2 : 1) * n_pad;
  for (int j = tid; j < n_pad; j += 32 * kSmallI) {
    s_hi[j] = __ldcg(A.jhi + j);
    if (PREC) s_lo[j] = __ldcg(A.jlo + j);
    s_v[j] = __ldcg(A.jvel + j);
  }
  __syncthreads();

  {
    const int k = b * kSmallI + wid;
    const int i = k < n ? k : 0;
    const float4 hi = s_hi[i], wi = s_v[i];
    const float4 li = PREC ? s_lo[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float nx[3] = {-hi.x, -hi.y, -hi.z}, nl[3] = {-li.x, -li.y, -li.z};
    const float nv[3] = {-wi.x, -wi.y, -wi.z};
    const uint64_t U = static_cast<uint64_t>(n_ib) * n_jt;
    const uint64_t u0 = static_cast<uint64_t>(b) * n_jt;
    const int plo = dev::owner_of(u0, U, A.P), phi = dev::owner_of(u0 + n_jt - 1, U, A.P);
    float h[6], l[6];  // the partial sums of the split, lane by lane
#pragma unroll
    for (int c = 0; c < 6; ++c) h[c] = l[c] = 0.f;
    int p = plo;
    uint64_t end = dev::udiv(U * static_cast<uint64_t>(p + 1), static_cast<uint64_t>(A.P));
    float sh[6], sl[6];  // this segment's sums
#pragma unroll
    for (int c = 0; c < 6; ++c) sh[c] = sl[c] = 0.f;
    for (int jt = 0; jt < n_jt; ++jt) {
      float pa[3] = {0.f, 0.f, 0.f}, p1[3] = {0.f, 0.f, 0.f}, p2[3] = {0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < kJT / 32; ++q) {
        const int j = jt * kJT + q * 32 + lane;
        const float4 hj = s_hi[j], wj = s_v[j];
        float dx, dy, dz;
        if (PREC) {
          const float4 lj = s_lo[j];
          dx = O::add(O::add(hj.x, nx[0]), O::add(lj.x, nl[0]));
          dy = O::add(O::add(hj.y, nx[1]), O::add(lj.y, nl[1]));
          dz = O::add(O::add(hj.z, nx[2]), O::add(lj.z, nl[2]));
        } else {
          dx = O::add(hj.x, nx[0]);
          dy = O::add(hj.y, nx[1]);
          dz = O::add(hj.z, nx[2]);
        }
        const float ux = O::add(wj.x, nv[0]), uy = O::add(wj.y, nv[1]), uz = O::add(wj.z, nv[2]);
        const float r2 = O::fma(dx, dx, O::fma(dy, dy, O::fma(dz, dz, A.eps2)));
        const float rinv = O::rsq<0>(r2);
        const float rinv2 = O::mul(rinv, rinv);
        const float mr3 = O::mul(O::mul(hj.w, rinv), rinv2);
        const float rv = O::fma(dx, ux, O::fma(dy, uy, O::mul(dz, uz)));
        const float cc = O::mul(O::mul(rv, rinv2), mr3);
        pa[0] = O::fma(mr3, dx, pa[0]);
        pa[1] = O::fma(mr3, dy, pa[1]);
        pa[2] = O::fma(mr3, dz, pa[2]);
        p1[0] = O::fma(mr3, ux, p1[0]);
        p1[1] = O::fma(mr3, uy, p1[1]);
        p1[2] = O::fma(mr3, uz, p1[2]);
        p2[0] = O::fma(cc, dx, p2[0]);
        p2[1] = O::fma(cc, dy, p2[1]);
        p2[2] = O::fma(cc, dz, p2[2]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float jt3 = fmaf(-3.f, p2[c], p1[c]);
        if (PREC) {
          dev::ds_add(sh[c], sl[c], pa[c]);
          dev::ds_add(sh[3 + c], sl[3 + c], jt3);
        } else {
          sh[c] += pa[c];
          sh[3 + c] += jt3;
        }
      }
      if (jt + 1 == n_jt || u0 + jt + 1 == end) {
        // a segment of the split ends
#pragma unroll
        for (int off = 1; off < 32; off <<= 1)
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            const float oh = __shfl_xor_sync(0xffffffffu, sh[c], off);
            const float ol = __shfl_xor_sync(0xffffffffu, sl[c], off);
            dev::ds_add_pair(sh[c], sl[c], oh, ol, sh[c], sl[c]);
          }
        if (plo == phi) {
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            h[c] = sh[c];
            l[c] = sl[c];
          }
        } else if (lane == ((p - plo) & 31)) {
#pragma unroll
          for (int c = 0; c < 6; ++c) dev::ds_add_pair(h[c], l[c], sh[c], sl[c], h[c], l[c]);
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) sh[c] = sl[c] = 0.f;
        ++p;
        end = dev::udiv(U * static_cast<uint64_t>(p + 1), static_cast<uint64_t>(A.P));
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
      s_f[wid][lane] = dev::ds_to_double(hh, ll, A.G);
    }
  }
  __syncthreads();
  if (ci >= 0) {
    const double an[3] = {s_f[eq][0], s_f[eq][1], s_f[eq][2]};
    const double jn[3] = {s_f[eq][3], s_f[eq][4], s_f[eq][5]};
    int nv = min(n - b * kSmallI, kSmallI) - wid * 10;  // this warp's particles
    nv = nv < 10 ? nv : 10;
    const unsigned mask = (1u << (3 * nv)) - 1u;
    dev::correct_vals3(cq, mask, lane - cq, ci, st, an, jn, A.t_next, A.x, A.v, A.a, A.jk,
                       A.t_tick, A.lev, A.eta, A.lev_min, A.lev_max, 0, A.n_clamped, nullptr,
                       &A.ext, nullptr, nullptr);
  }
}

}  // namespace

bool small_step_fits(int64_t n, int64_t n_jt, int prec, int mask, int num_sms) {
  if (mask) return false;
  const int64_t ctas = (n + kSmallI - 1) / kSmallI + n_jt;
  if (ctas > num_sms) return false;
  const Variant &V = variant_at(choose_variant(prec, mask, n, n_jt, num_sms));
  return V.ipt == 1 && V.tpi == 32 && V.threads == 32 * kSmallI && !V.rel;
}

size_t small_step_smem(int64_t n_jt, int prec) {
  return static_cast<size_t>(n_jt) * kJT * (prec ? 3 : 2) * sizeof(float4);
}

cudaError_t small_step_prepare(int64_t n_jt, int prec) {
  return cudaFuncSetAttribute(prec ? small_step_kernel<1> : small_step_kernel<0>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(small_step_smem(n_jt, prec)));
}

cudaError_t launch_small_step(const SmallStepArgs &A, int prec, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  const int64_t ctas = (A.n + kSmallI - 1) / kSmallI + (prec ? A.n_jt : 0);
  cfg.gridDim = dim3(static_cast<unsigned>(ctas));
  cfg.blockDim = dim3(32 * kSmallI);
  cfg.dynamicSmemBytes = small_step_smem(A.n_jt, prec);
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, prec ? small_step_kernel<1> : small_step_kernel<0>, A);
}

}  // namespace nbi
