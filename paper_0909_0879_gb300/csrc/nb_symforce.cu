// Pair-symmetric force + jerk kernels for sm_103a: every particle against
// every particle, each pair evaluated once.
//
// What is computed: the sums of nb_force.cu (paper eq. 1, Sec. 2, softened,
// and their time derivative) for all n particles.  The pair's difference,
// reciprocal square root and jerk vector c = w - 3 (d.w) d / s^2 serve both
// particles: i takes m_j / s^3 (d, c), j takes -m_i / s^3 (d, c).
//
// Bound: FP32 pipe and, with packed instructions holding the issue port for
// two cycles, the issue slots of everything else.  Per pair 19
// lane-operations are shared and 7 belong to each side: 33 for two
// interactions against 2 x 26 in the one-sided kernel (acceleration only 16
// against 2 x 12; split-precision near tiles 6 more, shared).
//
// Design:
//  * An i-block lives in registers (IPT particles per thread, each value
//    twice, as both halves of a packed operand); 256-record j-tiles come
//    through shared memory by bulk copies, records stored in pairs so that a
//    packed FP32x2 instruction takes two records without a move.  (Packing
//    two i-particles instead needs a move per record value and adds the
//    halves of the record's sums in every step: FP32 5.78 against 6.09 ms per
//    evaluation, N = 100,003.)
//  * Within a warp the 32 record pairs of a chunk go round: at step s lane l
//    holds pair l ^ s, and the pair's own sums travel with it by warp
//    shuffles, so after 32 steps every record has met the warp's 32 x IPT
//    particles and no sum crosses a warp through shared memory in the loop.
//  * Each warp leaves its records' sums in its own shared-memory rows; a
//    tile later the CTA adds the rows in warp order (split precision), so
//    the reduction of one tile overlaps the pair work of the next and one
//    barrier per tile remains.
//  * Work: i-blocks lie on a ring and row ib takes its own block and the
//    blocks at distances 1 .. (nb - 1) / 2 (for even nb the rows of the first
//    half also take distance nb / 2), so every pair of blocks belongs to one
//    row and the rows are equally long.  The rows' tiles form one list that
//    is cut into equal contiguous ranges, one per persistent CTA.
//  * No atomics: a CTA keeps its j-side sums in its own part of the scratch
//    (tiles it meets again in its next row are added by the same thread), and
//    the fix-up adds a particle's i-side and j-side partial sums in an order
//    fixed by the split: results are deterministic.  The scratch holds
//    about n / 2 records per CTA (split-precision pairs: 3.9 GB at N = 1M).
//  * m / r^3 is m (1 / r^3) on scaled positions and masses (sym_exponent), one
//    product less than (m y) y^2, whose FP32 range it has.  One mass for all
//    particles (EQ) comes in after the sums and leaves one 1 / r^3 for both
//    sides, 31 lane-operations (acceleration 14).  N = 1,048,576 King with EQ
//    622 -> 568 ms per step (577 without the scaling), N = 65,536 acceleration
//    (masses of a power law, near tiles) 1.68 -> 1.64 ms.
//  * Own-block tiles take the same loop and drop the j-side sums.
//  * Sums: near tiles fold the acceleration every 32 terms on both sides, far
//    tiles every 64 (i) and 32 IPT (j), the jerk every 128; no FP32 sum is
//    longer than in the one-sided kernel, and everything after the first
//    fold is split precision.  Against FP64 over 12 clusters of N = 33,000
//    (Salpeter masses): acceleration rms error 4.75e-8 against 4.79e-8
//    one-sided, jerk 3.5e-7 against 4.9e-7.
//  * One CTA of 8 warps per SM, IPT = 4 (8 for the FP32 acceleration of many
//    particles, see sym_pick).  The jerk kernel in split precision
//    keeps its i-side split-precision accumulators in shared memory (two
//    copy stages make room): 41.0 against 42.0 ms (N = 262,144 King, spatial
//    order) with them in registers.  Measured and not taken: IPT 3 / 2 with
//    as many or more warps (42.2 / 43.7), 12 warps for the acceleration (4.07
//    against 3.91 ms, N = 100,003), unrolls of 4 / 16 (41.8 / 42.9), units of
//    128 records (41.9), two CTAs of 4 warps (7.28 against 6.80 ms, N =
//    100,003).
//
// Measured (GB300, per evaluation, one-sided kernel -> this one):
//   N = 1,048,576 King, split precision, jerk, EQ 848 -> 568 ms
//   N = 100,003 sphere, FP32, jerk                7.86 -> 5.60 ms
//   N = 65,536 sphere, acceleration, DS           2.39 -> 1.64 ms
//   N = 131,101, acceleration, FP32               6.57 -> 4.62 ms
//   N = 16,384, acceleration, FP32                0.133 -> 0.105 ms
#include "nb_device.cuh"
#include "nb_pipe.cuh"

#include <algorithm>
#include <cmath>

namespace nbi {
namespace {

using dev::DsAcc;
using dev::ds_add;
using dev::VOps;
using dev::kNowhere;
using dev::kPairs;
using dev::kPlane2;
using dev::kPlane4;
using dev::rec_bytes;
using dev::rec_lo;
using dev::rec_rel;
using dev::rec_vel;

// Row of unit u and the unit's offset in it: tile offset `off` of row ib is
// tile off % TB of the block at ring distance off / TB.
__host__ __device__ __forceinline__ uint32_t sym_row(const SymSplit &S, uint32_t u,
                                                     uint32_t *off) {
  if (u < S.u1) {
    const uint32_t r = u / S.l1;
    *off = u - r * S.l1;
    return r;
  }
  const uint32_t w = u - S.u1, r = w / S.l2;
  *off = w - r * S.l2;
  return S.rows1 + r;
}

__host__ __device__ __forceinline__ uint32_t sym_row_start(const SymSplit &S, uint32_t row) {
  return row <= S.rows1 ? row * S.l1 : S.u1 + (row - S.rows1) * S.l2;
}

__host__ __device__ __forceinline__ uint32_t sym_row_len(const SymSplit &S, uint32_t row) {
  return row < S.rows1 ? S.l1 : S.l2;
}

// First unit of CTA p.
__host__ __device__ __forceinline__ uint32_t sym_begin(const SymSplit &S, uint32_t p) {
  return static_cast<uint32_t>(static_cast<uint64_t>(S.units) * p / S.ctas);
}

__host__ __device__ __forceinline__ uint32_t sym_owner(const SymSplit &S, uint32_t u) {
  return static_cast<uint32_t>(((static_cast<uint64_t>(u) + 1) * S.ctas - 1) / S.units);
}

// Tile of offset off in row ib (may lie past the last record tile in the
// last block).
__host__ __device__ __forceinline__ uint32_t sym_tile(const SymSplit &S, uint32_t row,
                                                      uint32_t off) {
  const uint32_t d = off / S.tb;
  uint32_t b = row + d;
  if (b >= S.nb) b -= S.nb;
  return b * S.tb + (off - d * S.tb);
}

// The jerk kernel's records from the predictor's; one CTA per tile, one thread
// per pair.
template <int PREC>
__global__ void __launch_bounds__(kPairs) sym_records_kernel(const SymArgs A) {
  if (A.ctl && A.ctl[kCtlNact] != A.n) return;
  const int k = threadIdx.x;
  const size_t j = static_cast<size_t>(blockIdx.x) * kJT + 2 * k;
  unsigned char *t = A.recs + static_cast<size_t>(blockIdx.x) * rec_bytes(PREC);
  const float4 none = make_float4(kNowhere, kNowhere, kNowhere, 0.f);
  auto scaled = [](float4 p, float s, float w) {
    return make_float4(p.x * s, p.y * s, p.z * s, p.w * w);
  };
  auto put = [&](const float4 *src, uint32_t at, bool four, float s) {
    const int64_t i = static_cast<int64_t>(j);
    const float4 p = four && i >= A.n ? none : scaled(src[j], s, A.sm);
    const float4 q = four && i + 1 >= A.n ? none : scaled(src[j + 1], s, A.sm);
    reinterpret_cast<float4 *>(t + at)[k] = make_float4(p.x, q.x, p.y, q.y);
    if (four)
      reinterpret_cast<float4 *>(t + at + kPlane4)[k] = make_float4(p.z, q.z, p.w, q.w);
    else
      reinterpret_cast<float2 *>(t + at + kPlane4)[k] = make_float2(p.z, q.z);
  };
  put(A.jhi, 0, true, A.sc);
  if (PREC) {
    put(A.jlo, rec_lo(), false, A.sc);
    put(A.jrel, rec_rel(), true, A.sc);
  }
  put(A.jvel, rec_vel(PREC), false, 1.f);
}

template <int PREC, int MASK, int JRK, int EQ, int IPT, int NT, int ST, int SACC>
struct SymShape {
  static constexpr int NW = NT / 32;
  static constexpr int NROW = (PREC ? 6 : 3) + (JRK ? 3 : 0);  // acc hi (lo), jerk
  static constexpr uint32_t kStageBytes = JRK ? rec_bytes(PREC) : rec_vel(PREC);
  static constexpr size_t kRowFloats = static_cast<size_t>(NW) * NROW * kJT;
  static constexpr size_t kAccOff = ST * kStageBytes + 2 * kRowFloats * sizeof(float);
  static constexpr size_t kSmem = kAccOff + (SACC ? 12 * IPT * NT * sizeof(float) : 0);
};

template <int PREC, int MASK, int JRK, int EQ, int IPT, int NT, int ST, int SACC>
__global__ void __launch_bounds__(NT, 256 / NT)
    sym_force_kernel(const SymArgs A) {
  using SH = SymShape<PREC, MASK, JRK, EQ, IPT, NT, ST, SACC>;
  using V = float2;  // two records j
  using O = VOps<V>;
  constexpr int BI = NT * IPT;
  constexpr int NC = JRK ? 6 : 3;
  constexpr int NROW = SH::NROW, NW = SH::NW;
  constexpr int kChunks = kPairs / 32;  // chunks of 32 pairs

  extern __shared__ __align__(128) unsigned char smem_raw[];
  float *rows = reinterpret_cast<float *>(smem_raw + ST * SH::kStageBytes);
  __shared__ __align__(8) uint64_t bars[ST];
  __shared__ uint32_t s_tile[ST];

  if (A.ctl && A.ctl[kCtlNact] != A.n) return;  // this step is not for all particles
  const SymSplit S = A.split;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint32_t p = blockIdx.x;
  const uint32_t u0 = sym_begin(S, p), u1 = sym_begin(S, p + 1);
  if (u0 >= u1) return;
  const uint32_t n_jt = static_cast<uint32_t>(A.n_jt);

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) pipe::mbar_init(&bars[s], 1);
    pipe::mbar_fence_init();
  }
  __syncthreads();

  uint32_t off, row = sym_row(S, u0, &off);
  const uint32_t slot_base = sym_tile(S, row, 0);  // the range's first row's first tile
  const uint32_t first_row = row;
  // thread 0's issue cursor runs ST units ahead
  uint32_t i_row = row, i_off = off;
  auto issue = [&](uint32_t s_idx) {
    const int st = static_cast<int>(s_idx % ST);
    uint32_t jt = sym_tile(S, i_row, i_off);
    s_tile[st] = jt;
    if (jt >= n_jt) jt = n_jt - 1;  // past the records: loaded, not used
    pipe::mbar_expect_tx(&bars[st], SH::kStageBytes);
    pipe::bulk_g2s(smem_raw + st * SH::kStageBytes,
                   A.recs + static_cast<size_t>(jt) * rec_bytes(PREC), SH::kStageBytes,
                   &bars[st]);
    if (++i_off == sym_row_len(S, i_row)) {
      i_off = 0;
      ++i_row;
    }
  };
  const uint32_t nunits = u1 - u0;
  if (tid == 0)
    for (uint32_t s = 0; s < nunits && s < ST; ++s) issue(s);

  // the tile whose j-side rows wait to be added: its partial-sum slot
  // (relative to the CTA's scratch), whether it is the slot's first, and
  // whether its rows have low words
  bool pend = false, pend_first = false, pend_lo = false;
  uint32_t pend_slot = 0;
  float2 *const my_j = A.jpart + static_cast<size_t>(p) * S.jslots * NC * kJT;

  auto reduce_rows = [&](int buf) {
    const float *rb = rows + static_cast<size_t>(buf) * SH::kRowFloats;
#pragma unroll
    for (int j = tid; j < kJT; j += NT) {
      float2 *dst = my_j + static_cast<size_t>(pend_slot) * NC * kJT + j;
      float2 old[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c)
        old[c] = pend_first ? make_float2(0.f, 0.f) : dst[c * kJT];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int r = c < 3 ? c : (PREC ? c + 3 : c);
        const bool lo = PREC && c < 3 && pend_lo;
        float h = rb[r * kJT + j], l = lo ? rb[(3 + c) * kJT + j] : 0.f;
#pragma unroll
        for (int w = 1; w < NW; ++w) {
          const float *rw = rb + static_cast<size_t>(w) * NROW * kJT;
          ds_add(h, l, rw[r * kJT + j]);
          if (lo) l += rw[(3 + c) * kJT + j];
        }
        dev::ds_add_pair(h, l, old[c].x, old[c].y, h, l);
        dst[c * kJT] = make_float2(h, l);
      }
    }
  };

  uint32_t s_idx = 0, u = u0;
  while (u < u1) {
    const uint32_t seg = min(sym_row_len(S, row) - off, u1 - u);
    // i-particle data, negated so that every difference is an addition;
    // lanes past n stand opposite the records past n
    float nxh[IPT][3], nxl[IPT][3], nvi[IPT][3], mi[IPT];
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      const int64_t k = static_cast<int64_t>(row) * BI + tid + q * NT;
      const int64_t i = k < A.n ? k : 0;
      const float4 h = A.jhi[i];
      const float4 w = JRK ? A.jvel[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 l = PREC ? A.jlo[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < A.n) {
        nxh[q][0] = -h.x * A.sc; nxh[q][1] = -h.y * A.sc; nxh[q][2] = -h.z * A.sc;
      } else {
        nxh[q][0] = nxh[q][1] = nxh[q][2] = kNowhere;
      }
      nxl[q][0] = -l.x * A.sc; nxl[q][1] = -l.y * A.sc; nxl[q][2] = -l.z * A.sc;
      nvi[q][0] = -w.x; nvi[q][1] = -w.y; nvi[q][2] = -w.z;
      mi[q] = k < A.n ? h.w * A.sm : 0.f;
    }
    const V veps2 = O::bc(!PREC && !JRK && !EQ && A.dscale ? A.dscale->eps2
                                                           : A.eps2 * A.sc * A.sc);
    float bc_i[3] = {0.f, 0.f, 0.f}, bh_i[3] = {0.f, 0.f, 0.f};
    if (PREC) {
      // bounding box of the i-block (far test), as in the one-sided kernel
      __shared__ float s_mn[3][NW], s_mx[3][NW];
      float mn[3] = {3.0e38f, 3.0e38f, 3.0e38f}, mx[3] = {-3.0e38f, -3.0e38f, -3.0e38f};
#pragma unroll
      for (int q = 0; q < IPT; ++q)
        if (static_cast<int64_t>(row) * BI + tid + q * NT < A.n) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            mn[c] = fminf(mn[c], -nxh[q][c]);
            mx[c] = fmaxf(mx[c], -nxh[q][c]);
          }
        }
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          mn[c] = fminf(mn[c], __shfl_xor_sync(0xffffffffu, mn[c], o));
          mx[c] = fmaxf(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], o));
        }
      __syncthreads();
      if (lane == 0)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          s_mn[c][wid] = mn[c];
          s_mx[c][wid] = mx[c];
        }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float a = s_mn[c][0], b = s_mx[c][0];
        for (int w = 1; w < NW; ++w) {
          a = fminf(a, s_mn[c][w]);
          b = fmaxf(b, s_mx[c][w]);
        }
        bc_i[c] = 0.5f * a + 0.5f * b;
        const float big = fmaxf(fabsf(a), fabsf(b));
        bh_i[c] = fmaxf(bc_i[c] - a, b - bc_i[c]) * (1.0f + 1.0e-6f) + big * 1.2e-7f;
      }
    }
    DsAcc<IPT, NT, SACC != 0> D;
    D.init(reinterpret_cast<float *>(smem_raw + SH::kAccOff), tid);

    for (uint32_t t = 0; t < seg; ++t, ++s_idx, ++off) {
      const int st = static_cast<int>(s_idx % ST);
      const bool ok = pipe::mbar_wait(&bars[st], (s_idx / ST) & 1);
      const uint32_t jt = s_tile[st];
      const int buf = static_cast<int>(s_idx & 1);
      float *my_rows = rows + static_cast<size_t>(buf) * SH::kRowFloats +
                       static_cast<size_t>(wid) * NROW * kJT;
      const unsigned char *rec = smem_raw + st * SH::kStageBytes;
      const bool live = jt < n_jt;
      const bool own = off < S.tb;
      bool far = false;
      float ox[3] = {0.f, 0.f, 0.f};
      if (PREC && live) {
        const float4 to = __ldg(&A.tinfo[2 * jt]);
        const float4 th = __ldg(&A.tinfo[2 * jt + 1]);
        ox[0] = to.x * A.sc; ox[1] = to.y * A.sc; ox[2] = to.z * A.sc;
        const float hw[3] = {th.x * A.sc, th.y * A.sc, th.z * A.sc};
        float d2 = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float d = fmaxf(0.f, fabsf(bc_i[c] - ox[c]) - (bh_i[c] + hw[c]));
          d2 = fmaf(d, d, d2);
        }
        const float lim = kRelKappa * (to.w * A.sc) * (1.0f + 1.0e-5f);
        far = d2 >= lim * lim;
      }

      // turn() passes a pair of records' sums to the lane that holds the
      // pair next.
      auto turn = [&](V &a, int mask) {
        a.x = __shfl_xor_sync(0xffffffffu, a.x, mask);
        a.y = __shfl_xor_sync(0xffffffffu, a.y, mask);
      };
      auto walk = [&](auto far_tag) {
        constexpr bool FAR = decltype(far_tag)::value;
        constexpr bool NEAR2 = PREC && !FAR;  // split-precision differences
        V xi[IPT][3], xl[IPT][3], vi[IPT][3], wi[IPT];
#pragma unroll
        for (int q = 0; q < IPT; ++q) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            // far: the i-particle relative to the tile's origin
            xi[q][c] = O::bc(FAR ? (nxh[q][c] + ox[c]) + nxl[q][c] : nxh[q][c]);
            if (NEAR2) xl[q][c] = O::bc(nxl[q][c]);
            if (JRK) vi[q][c] = O::bc(nvi[q][c]);
          }
          wi[q] = O::bc(mi[q]);
        }
        V pa[IPT][3], pj[IPT][3];
#pragma unroll
        for (int q = 0; q < IPT; ++q)
#pragma unroll
          for (int c = 0; c < 3; ++c) pa[q][c] = pj[q][c] = O::bc(0.f);
#pragma unroll 1
        for (int ch = 0; ch < kChunks; ++ch) {
          if (ch == kChunks / 2 && pend) reduce_rows(buf ^ 1);
          V ta[3], tj[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) ta[c] = tj[c] = O::bc(0.f);
          float2 *rw = reinterpret_cast<float2 *>(my_rows) + ch * 32;
          if (NEAR2) {
#pragma unroll
            for (int c = 0; c < 6; ++c) rw[c * kPairs + lane] = make_float2(0.f, 0.f);
            __syncwarp();
          }
#pragma unroll 1
          for (int s0 = 0; s0 < 32; s0 += 8) {
            const int base = lane ^ s0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int jj = ch * 32 + (base ^ k);
              const unsigned char *rp = rec + (FAR ? rec_rel() : 0);
              const float4 qa = reinterpret_cast<const float4 *>(rp)[jj];
              const float4 qb = reinterpret_cast<const float4 *>(rp + kPlane4)[jj];
              const V xj = make_float2(qa.x, qa.y), yj = make_float2(qa.z, qa.w);
              const V zj = make_float2(qb.x, qb.y), mj = make_float2(qb.z, qb.w);
              V xlj, ylj, zlj, vxj, vyj, vzj;
              if (NEAR2) {
                const float4 la = reinterpret_cast<const float4 *>(rec + rec_lo())[jj];
                xlj = make_float2(la.x, la.y);
                ylj = make_float2(la.z, la.w);
                zlj = reinterpret_cast<const float2 *>(rec + rec_lo() + kPlane4)[jj];
              }
              if (JRK) {
                const float4 va = reinterpret_cast<const float4 *>(rec + rec_vel(PREC))[jj];
                vxj = make_float2(va.x, va.y);
                vyj = make_float2(va.z, va.w);
                vzj = reinterpret_cast<const float2 *>(rec + rec_vel(PREC) + kPlane4)[jj];
              }
#pragma unroll
              for (int q = 0; q < IPT; ++q) {
                V dx = O::add(xj, xi[q][0]);
                V dy = O::add(yj, xi[q][1]);
                V dz = O::add(zj, xi[q][2]);
                if (NEAR2) {
                  dx = O::add(dx, O::add(xlj, xl[q][0]));
                  dy = O::add(dy, O::add(ylj, xl[q][1]));
                  dz = O::add(dz, O::add(zlj, xl[q][2]));
                }
                const V r2 = O::fma(dx, dx, O::fma(dy, dy, O::fma(dz, dz, veps2)));
                const V y = O::template rsq<MASK>(r2);
                // k = y^2, f = y^3; the jerk kernel for equal masses has -3 y^2
                // and 9 y^3 instead (the sums' factor makes up for it)
                const V ym = EQ && JRK ? O::mul(y, O::bc(-3.f)) : y;
                const V k2 = O::mul(ym, y), y3 = O::mul(ym, k2);
                const V fi = EQ ? y3 : O::mul(mj, y3);    // on i from j
                const V fj = EQ ? y3 : O::mul(wi[q], y3);  // on j from i
                pa[q][0] = O::fma(fi, dx, pa[q][0]);
                pa[q][1] = O::fma(fi, dy, pa[q][1]);
                pa[q][2] = O::fma(fi, dz, pa[q][2]);
                ta[0] = O::fma(fj, dx, ta[0]);
                ta[1] = O::fma(fj, dy, ta[1]);
                ta[2] = O::fma(fj, dz, ta[2]);
                if (JRK) {
                  V ux = O::add(vxj, vi[q][0]);
                  V uy = O::add(vyj, vi[q][1]);
                  V uz = O::add(vzj, vi[q][2]);
                  const V rv = O::fma(dx, ux, O::fma(dy, uy, O::mul(dz, uz)));
                  const V a3 = EQ ? O::mul(rv, k2) : O::mul(O::mul(rv, k2), O::bc(-3.f));
                  ux = O::fma(a3, dx, ux);
                  uy = O::fma(a3, dy, uy);
                  uz = O::fma(a3, dz, uz);
                  pj[q][0] = O::fma(fi, ux, pj[q][0]);
                  pj[q][1] = O::fma(fi, uy, pj[q][1]);
                  pj[q][2] = O::fma(fi, uz, pj[q][2]);
                  tj[0] = O::fma(fj, ux, tj[0]);
                  tj[1] = O::fma(fj, uy, tj[1]);
                  tj[2] = O::fma(fj, uz, tj[2]);
                }
              }
              if (k < 7) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                  turn(ta[c], k ^ (k + 1));
                  if (JRK) turn(tj[c], k ^ (k + 1));
                }
              }
            }
            // records after eight steps: 8 IPT terms
            if (NEAR2) {
              float2 *ra = rw + (base ^ 7);
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                float2 h = ra[c * kPairs], l = ra[(3 + c) * kPairs];
                ds_add(h.x, l.x, ta[c].x);
                ds_add(h.y, l.y, ta[c].y);
                ra[c * kPairs] = h;
                ra[(3 + c) * kPairs] = l;
                ta[c] = O::bc(0.f);
              }
              __syncwarp();
            }
            if (s0 < 24) {
              const int mask = (s0 + 7) ^ (s0 + 8);
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                if (!NEAR2) turn(ta[c], mask);
                if (JRK) turn(tj[c], mask);
              }
            }
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            if (!NEAR2) rw[c * kPairs + (lane ^ 31)] = ta[c];
            if (JRK) rw[((PREC ? 6 : 3) + c) * kPairs + (lane ^ 31)] = tj[c];
          }
          if (!FAR || ch % 2 == 1) {
#pragma unroll
            for (int q = 0; q < IPT; ++q)
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                float h = D.AH(q, c), l = D.AL(q, c);
                ds_add(h, l, pa[q][c].x);
                ds_add(h, l, pa[q][c].y);
                D.AH(q, c) = h;
                D.AL(q, c) = l;
                pa[q][c] = O::bc(0.f);
              }
          }
        }
        if (JRK) {
#pragma unroll
          for (int q = 0; q < IPT; ++q)
#pragma unroll
            for (int c = 0; c < 3; ++c) ds_add(D.JH(q, c), D.JL(q, c), pj[q][c].x + pj[q][c].y);
        }
      };
      if (live) {
        if (PREC && far)
          walk(std::true_type{});
        else
          walk(std::false_type{});
      } else if (pend) {
        reduce_rows(buf ^ 1);
      }
      // this tile's rows are added during the next tile
      pend = live && !own;
      if (pend) {
        pend_lo = PREC && !far;
        pend_slot = jt + (jt < slot_base ? S.nb * S.tb : 0) - slot_base;
        // met before by this CTA: the row before holds the tile one block
        // further along, inside the CTA's range
        const uint32_t po = off + S.tb;
        pend_first = row == first_row || po >= sym_row_len(S, row - 1) ||
                     sym_row_start(S, row - 1) + po < u0;
      }
      if (__syncthreads_or(!ok)) {
        // A copy never arrived: record it, wait (bounded) for the copies
        // still in flight so none lands after exit, and leave.
        if (tid == 0) {
          atomicOr(A.err, kErrWaitTimeout);
          const uint32_t last = min(s_idx + ST, nunits);
          for (uint32_t s2 = s_idx; s2 < last; ++s2)
            (void)pipe::mbar_wait(&bars[s2 % ST], (s2 / ST) & 1);
        }
        return;
      }
      if (tid == 0 && s_idx + ST < nunits) issue(s_idx + ST);
    }

    // the row's i-side sums
    float2 *dst = A.ipart + (static_cast<size_t>(p) * S.irows + (row - first_row)) * NC * BI + tid;
#pragma unroll
    for (int q = 0; q < IPT; ++q)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dst[c * BI + q * NT] = make_float2(D.AH(q, c), D.AL(q, c));
        if (JRK) dst[(3 + c) * BI + q * NT] = make_float2(D.JH(q, c), D.JL(q, c));
      }
    u += seg;
    if (off == sym_row_len(S, row)) {
      off = 0;
      ++row;
    }
  }
  if (pend) reduce_rows(static_cast<int>((s_idx - 1) & 1));
}

// Sums of every particle: its i-side partial sums (ascending CTAs), then
// the j-side ones by ring distance, in split precision; then, for a symplectic
// step, the external field at x and the closing kick v += kick a.
//
// Bound: latency of the chain of loads and additions (about nb / 2 links)
// and, with the field, the FP64 pipe.  One thread per (particle, component)
// and 32 particles per CTA: six or three short chains instead of one long
// one, and the field's particles spread over all SMs.  The partial sums'
// places (divisions) are worked out once per CTA, into a list of those that
// exist.  N = 20,011, acceleration, with the field: 20 us + 18 us per kick
// for the field with a thread per particle and 256 particles per CTA -> 17.8 us
// with everything in it; N = 100,003, jerk, FP32: 52 us.
constexpr int kFixP = 32, kFixList = 192;

template <int NC>
__global__ void __launch_bounds__(kFixP *NC) sym_fixup_kernel(const SymArgs A) {
  if (A.ctl && A.ctl[kCtlNact] != A.n) return;
  __shared__ uint32_t s_raw[kFixList], s_src[kFixList], s_n;
  __shared__ double s_a[3][kFixP];
  constexpr uint32_t kNone = 0xffffffffu;
  const SymSplit S = A.split;
  const uint32_t tid = threadIdx.x, c = tid / kFixP, pl = tid - c * kFixP, lane = tid & 31;
  const uint32_t jt = blockIdx.x / (kJT / kFixP);
  const uint32_t t = (blockIdx.x - jt * (kJT / kFixP)) * kFixP + pl;
  const uint32_t BI = S.tb * kJT;
  const uint32_t row = jt / S.tb, jo = jt - row * S.tb;

  // adds base[place(k) * stride] for k = 0 .. count - 1, without the kNone ones
  auto sum = [&](uint32_t count, auto place, const float2 *base, size_t stride, float &h,
                 float &l) {
    for (uint32_t b = 0; b < count; b += kFixList) {
      const uint32_t m = min(count - b, static_cast<uint32_t>(kFixList));
      __syncthreads();
      for (uint32_t k = tid; k < m; k += kFixP * NC) s_raw[k] = place(b + k);
      __syncthreads();
      if (tid < 32) {
        uint32_t cnt = 0;
        for (uint32_t k0 = 0; k0 < m; k0 += 32) {
          const uint32_t v = k0 + lane < m ? s_raw[k0 + lane] : kNone;
          const uint32_t mk = __ballot_sync(0xffffffffu, v != kNone);
          if (v != kNone) s_src[cnt + __popc(mk & ((1u << lane) - 1))] = v;
          cnt += __popc(mk);
        }
        if (lane == 0) s_n = cnt;
      }
      __syncthreads();
      const uint32_t cnt = s_n;
#pragma unroll 8
      for (uint32_t k = 0; k < cnt; ++k) {
        const float2 w = base[s_src[k] * stride];
        dev::ds_add_pair(h, l, w.x, w.y, h, l);
      }
    }
  };

  float h = 0.f, l = 0.f, gh = 0.f, gl = 0.f;
  const uint32_t us = sym_row_start(S, row), ue = us + sym_row_len(S, row) - 1;
  const uint32_t p0 = sym_owner(S, us);
  sum(sym_owner(S, ue) - p0 + 1,
      [&](uint32_t k) {
        uint32_t o;
        return (p0 + k) * S.irows + (row - sym_row(S, sym_begin(S, p0 + k), &o));
      },
      A.ipart + static_cast<size_t>(c) * BI + jo * kJT + t, static_cast<size_t>(NC) * BI, h, l);
  // owner of this tile as seen from the row at ring distance d (kNone: not
  // that row's)
  auto owner = [&](uint32_t d) {
    const uint32_t r = row >= d ? row - d : row + S.nb - d;
    const uint32_t o = d * S.tb + jo;
    return o >= sym_row_len(S, r) ? kNone : sym_owner(S, sym_row_start(S, r) + o);
  };
  sum(S.nb / 2,
      [&](uint32_t k) {
        const uint32_t p = owner(k + 1);
        // one slot for all rows of a CTA
        if (p == kNone || (k > 0 && p == owner(k))) return kNone;
        uint32_t fo;
        const uint32_t sb = sym_row(S, sym_begin(S, p), &fo) * S.tb;
        return p * S.jslots + (jt + (jt < sb ? S.nb * S.tb : 0) - sb);
      },
      A.jpart + static_cast<size_t>(c) * kJT + t, static_cast<size_t>(NC) * kJT, gh, gl);

  const int64_t i = static_cast<int64_t>(jt) * kJT + t;
  const bool real = i < A.n;
  dev::ds_add_pair(h, l, -gh, -gl, h, l);
  const double g_acc = NC == 3 && A.dscale ? A.dscale->g_acc : A.g_acc;
  double val = dev::ds_to_double(h, l, c < 3 ? g_acc : A.g_jerk);
  if (A.ext.on) {
    if (c < 3) s_a[c][pl] = val;
    __syncthreads();
    if (c == 0 && real) {
      const double xv[3] = {A.x[3 * i], A.x[3 * i + 1], A.x[3 * i + 2]};
      double at[3] = {s_a[0][pl], s_a[1][pl], s_a[2][pl]};
      dev::ext_acc(A.ext, xv, at);
#pragma unroll
      for (int q = 0; q < 3; ++q) s_a[q][pl] = at[q];
    }
    __syncthreads();
    if (c < 3) val = s_a[c][pl];
  }
  if (!real) return;
  if (NC == 3 && A.acc_f) {
    A.acc_f[3 * i + c] = *A.err ? __int_as_float(0x7fffffff) : static_cast<float>(val);
  } else if (c < 3) {
    A.acc[3 * i + c] = val;
    if (A.kick != 0.0) A.v[3 * i + c] = fma(A.kick, val, A.v[3 * i + c]);
  } else {
    A.jerk[3 * i + c - 3] = val;
  }
}

struct SymEntry {
  void (*fn)(const SymArgs);
  int ipt, nt;
  size_t smem;
};

template <int PREC, int MASK, int JRK, int EQ, int IPT, int NT, int ST, int SACC>
SymEntry sym_entry() {
  return {&sym_force_kernel<PREC, MASK, JRK, EQ, IPT, NT, ST, SACC>, IPT, NT,
          SymShape<PREC, MASK, JRK, EQ, IPT, NT, ST, SACC>::kSmem};
}

template <int MASK, int EQ>
const SymEntry &sym_shape(int prec, int jrk) {
  static const SymEntry kE[2][2] = {
      {sym_entry<0, MASK, 0, EQ, 4, 256, 3, 0>(), sym_entry<0, MASK, 1, EQ, 4, 256, 3, 0>()},
      {sym_entry<1, MASK, 0, EQ, 4, 256, 3, 0>(), sym_entry<1, MASK, 1, EQ, 4, 256, 2, 1>()}};
  return kE[prec ? 1 : 0][jrk ? 1 : 0];
}

// The FP32 acceleration takes eight i-particles per thread from N = 65,536
// (generic masses: N = 65,536 1.209 -> 1.163, N = 131,101 4.81 -> 4.62, N = 262,144
// 18.9 -> 17.7 ms): the loads, turns and address arithmetic of a record pair
// serve twice the pairs.  Below it the ring of 2,048-particle blocks divides
// worse (N = 16,385 0.126 against 0.144 ms, 24,000 0.193 against 0.227,
// 60,000 1.033 against 1.037), with eps = 0 there is nothing in it (N = 65,536
// 1.27 both), and in split precision the records' sums of 64 terms between
// folds cost accuracy (rms 4.55e-8 against 4.27e-8, N = 66,000).
constexpr int64_t kWideTiles = 65536 / kJT;

template <int EQ>
const SymEntry &sym_wide() {
  static const SymEntry kE = sym_entry<0, 0, 0, EQ, 8, 256, 4, 0>();
  return kE;
}

const SymEntry &sym_pick(int prec, int mask, int jrk, bool eq, int64_t n_jt) {
  if (!prec && !mask && !jrk && n_jt >= kWideTiles) return eq ? sym_wide<1>() : sym_wide<0>();
  if (mask) return eq ? sym_shape<1, 1>(prec, jrk) : sym_shape<1, 0>(prec, jrk);
  return eq ? sym_shape<0, 1>(prec, jrk) : sym_shape<0, 0>(prec, jrk);
}

}  // namespace

bool sym_split(int64_t n_jt, int bi, int ctas, SymSplit *out) {
  const int64_t tb = bi / kJT;
  const int64_t nb = (n_jt + tb - 1) / tb;
  if (nb < 4 || nb > (int64_t(1) << 15)) return false;
  SymSplit S;
  const int64_t h = (nb - 1) / 2;
  S.tb = static_cast<uint32_t>(tb);
  S.nb = static_cast<uint32_t>(nb);
  S.l2 = static_cast<uint32_t>(tb * (1 + h));
  S.l1 = nb % 2 ? S.l2 : S.l2 + S.tb;
  S.rows1 = static_cast<uint32_t>(nb % 2 ? nb : nb / 2);
  S.u1 = S.rows1 * S.l1;
  const int64_t units = static_cast<int64_t>(S.u1) + (nb - S.rows1) * S.l2;
  if (units >= (int64_t(1) << 31) || ctas < 4) return false;
  S.units = static_cast<uint32_t>(units);
  S.ctas = static_cast<uint32_t>(std::min<int64_t>(ctas, units));
  // rows a CTA's range can touch, and tiles of the ring from its first
  // row's first tile to its last row's last
  const int64_t per = (units + S.ctas - 1) / S.ctas;
  const int64_t r = (per + S.l2 - 2) / S.l2 + 1;
  if (r >= nb / 2) return false;
  S.irows = static_cast<uint32_t>(r);
  S.jslots = static_cast<uint32_t>(std::min<int64_t>(nb * tb, S.l1 + (r - 1) * tb));
  *out = S;
  return true;
}

size_t sym_ipart_bytes(const SymSplit &S, bool jrk) {
  return static_cast<size_t>(S.ctas) * S.irows * (jrk ? 6 : 3) * S.tb * kJT * sizeof(float2);
}

size_t sym_jpart_bytes(const SymSplit &S, bool jrk) {
  return static_cast<size_t>(S.ctas) * S.jslots * (jrk ? 6 : 3) * kJT * sizeof(float2);
}

size_t sym_record_bytes(int64_t n_jt, int prec) {
  return static_cast<size_t>(n_jt) * rec_bytes(prec);
}

int sym_block_i(int prec, int mask, bool jrk, int64_t n_jt) {
  const SymEntry &E = sym_pick(prec, mask, jrk, false, n_jt);
  return E.ipt * E.nt;
}

cudaError_t sym_prepare(int prec, int mask, bool jrk, bool eq, int64_t n_jt) {
  const SymEntry &E = sym_pick(prec, mask, jrk, eq, n_jt);
  return cudaFuncSetAttribute(E.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(E.smem));
}

cudaError_t launch_sym_force(int prec, int mask, const SymArgs &A0, cudaStream_t s,
                             int *launches) {
  SymArgs A = A0;
  const bool jrk = A.jerk != nullptr;
  A.sc = static_cast<float>(std::ldexp(1.0, A.sexp));
  A.sm = static_cast<float>(std::ldexp(1.0, 3 * A.sexp));
  A.g_jerk = A.eq ? A.G * std::ldexp(A.m_eq, 3 * A.sexp) / (jrk ? 9.0 : 1.0) : A.G;
  A.g_acc = std::ldexp(A.g_jerk, -A.sexp);
  const SymEntry &E = sym_pick(prec, mask, jrk, A.eq != 0, A.n_jt);
  const unsigned tiles = static_cast<unsigned>(A.n_jt);
  if (jrk) {  // a drift has written the acceleration's records
    if (prec)
      sym_records_kernel<1><<<tiles, kPairs, 0, s>>>(A);
    else
      sym_records_kernel<0><<<tiles, kPairs, 0, s>>>(A);
    if (launches) *launches += 1;
  }
  E.fn<<<A.split.ctas, E.nt, E.smem, s>>>(A);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const unsigned ctas = tiles * (kJT / kFixP);
  if (jrk)
    sym_fixup_kernel<6><<<ctas, 6 * kFixP, 0, s>>>(A);
  else
    sym_fixup_kernel<3><<<ctas, 3 * kFixP, 0, s>>>(A);
  if (launches) *launches += 2;
  return cudaGetLastError();
}

}  // namespace nbi
