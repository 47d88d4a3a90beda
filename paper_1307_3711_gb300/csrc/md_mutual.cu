// md_mutual.cu -- the step with every pair of records evaluated once.
//
// The step kernel of md_device.cuh evaluates each unordered pair twice, once
// for either record: 11 FP32 lane operations per interaction on tiles of one
// charge.  What bounds both kernels is the register file: a packed f32x2
// operation reads one 64-bit operand per cycle and scheduler, and ptxas leaves
// few of them to the operand reuse cache (probes: 2.0 cycles for an operation
// with two different operands, 2.6 with three).  The one-sided pair reads 25
// operands per two pairs and runs at 25.0 cycles (0.905 of the FP32 roofline,
// 13.2 ms per step at 200k records), so only fewer operands make a large step
// faster.  Here one evaluation of the displacement and of 1/r^3 feeds the sums
// of both records: 34 operands for four interactions, 36 cycles with the
// shuffles: 9.5 ms at 200k records, 2.46 against 3.41 at 100k, 0.67 against
// 0.91 at 50k, 0.123 against 0.20 at 19k.  (Unrolling by 1, 2 or 8 steps,
// prefetching the next source, one scalar instead of two packed partial sums
// of a source, tiles of 256 sources and 6, 10, 14 or 16 targets per thread
// were slower or no faster.)
//
//   * The records of a cluster are cut into i-blocks of 128 R (R = 8 or 12).  Block I
//     meets the source tiles of its own block one-sided (every target of the
//     block sums the tile) and the tiles of all later blocks mutually.
//   * A mutual tile is summed in chunks of 32 sources.  Lane l of a warp holds
//     R targets in registers, starts with source l of the chunk and moves on
//     to source l + 1 after each of 32 steps; the source's own partial sum
//     moves with it by a shuffle, from lane l + 1 to lane l, and after 32
//     steps is back at the lane that it belongs to, having met the warp's
//     32 R targets.  No atomics: the order of every sum is fixed.
//   * The four warps' sums of a source are added and written to `jpart`, one
//     FP32 value per component, block I and later record; the targets' sums
//     (Kahan, folded once per tile) go to `ipart` per work unit.  k_mut_push
//     adds a record's partials in a fixed order and pushes it.  The traffic is
//     12 bytes per i-block and later record each way: 0.24 GB written and read
//     per step at 200k records, 1 % of its time.
//   * Work units are runs of tiles of one i-block.  The whole context's tiles (a
//     mutual tile weighs 4, a one-sided tile 3) are cut into shares that a ticket
//     hands out, in rounds of three eighths of the work that is left (auto_configure).
#include <algorithm>

#include "md_device.cuh"
#include "md_internal.h"

namespace md {

namespace {

constexpr int kMutThreads = 128;
constexpr int kMutWarps = kMutThreads / 32;
constexpr int kTile = kMutTile;

// Far away from every record, where a source adds exactly 0 to a field: r^2 =
// 3e36 is finite and 1/r^3 underflows to 0 (to a potential, before its charge of 0
// or the tile's is applied, 6e-19).
constexpr float kFar = 1.0e18f;

// A source tile expanded for packed use, (x,x | y,y) and (z,z | q,q) apart, so
// that 32 lanes reading 32 consecutive sources meet no bank conflict.
template <int TILE>
struct MutTile {
  alignas(16) ulonglong2 xy[TILE];
  alignas(16) ulonglong2 zq[TILE];
};

// Accumulators of one lane: its targets' partial sums of the current tile.
template <int P, bool POT>
struct MutAcc {
  u64 ax[P], ay[P], az[P], ap[POT ? P : 1];
};

template <int P, bool POT>
struct MutSmem {
  // Kahan sums and compensations (as KahanSmem); before a unit's sums start,
  // its packed targets, read back as register pairs
  u64 v[POT ? 8 : 6][P][kMutThreads];
  u64 q[P][kMutThreads];  // the targets' charges (tiles of mixed charge)
  u64 e2[kMutThreads];
};

__device__ __forceinline__ u64 shfl_u64(u64 v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}

// Fold of the potential's partial (every 8 sources) of this thread's targets.
template <int P>
__device__ __forceinline__ void fold_phi(MutSmem<P, true>& ks, MutAcc<P, true>& a, u64 qq,
                                         bool scale) {
#pragma unroll
  for (int p = 0; p < P; ++p) {
    u64 sp = ks.v[6][p][threadIdx.x], cp = ks.v[7][p][threadIdx.x];
    kahan_add2(sp, cp, scale ? f2_mul(a.ap[p], qq) : a.ap[p]);
    ks.v[6][p][threadIdx.x] = sp;
    ks.v[7][p][threadIdx.x] = cp;
    a.ap[p] = 0ull;
  }
}

// One warp: the sources of a mutual tile (cnt32, a multiple of 32, the last
// ones possibly kFar with no charge) against this warp's targets.  UNI: the
// tile's sources have one charge and the block's targets have one charge;
// neither is applied here.  Otherwise each pair takes its charges.  jout
// (component c at jout[c * TILE + source]) receives the sources' sums, jphi
// their potentials.
template <int P, int TILE, bool UNI, bool POT, bool IMG>
__device__ __forceinline__ void mutual_tile(const MutTile<TILE>& dup, int cnt32,
                                            const u64 (&xi)[P], const u64 (&yi)[P],
                                            const u64 (&zi)[P], u64 e2, MutAcc<P, POT>& a,
                                            MutSmem<P, POT>& ks, float* jout, double* jphi, u64 qq,
                                            const u64 (&mi)[3]) {
  const int lane = threadIdx.x & 31, next = (lane + 1) & 31;
  const uint32_t bxy = smem_u32(&dup.xy[0]), bzq = smem_u32(&dup.zq[0]);
#pragma unroll 1
  for (int c = 0; c < cnt32; c += 32) {
    u64 jx = 0ull, jy = 0ull, jz = 0ull, jp = 0ull, jc = 0ull;
    uint32_t o = 16u * lane;
#pragma unroll 1
    for (int k0 = 0; k0 < 32; k0 += 4) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const ulonglong2 xy = lds_u64x2(bxy + 16u * c + o);
        u64 zz, qj = 0ull;
        if constexpr (UNI) {
          zz = lds_u64(bzq + 16u * c + o);
        } else {
          const ulonglong2 zq = lds_u64x2(bzq + 16u * c + o);
          zz = zq.x;
          qj = zq.y;
        }
        o = (o + 16u) & 511u;
        u64 ps = 0ull;
#pragma unroll
        for (int p = 0; p < P; ++p) {
          u64 dx = f2_sub(xy.x, xi[p]);
          u64 dy = f2_sub(xy.y, yi[p]);
          u64 dz = f2_sub(zz, zi[p]);
          if constexpr (IMG) {
            dx = f2_min_image(dx, mi);
            dy = f2_min_image(dy, mi);
            dz = f2_min_image(dz, mi);
          }
          u64 r2 = f2_fma(dx, dx, e2);
          r2 = f2_fma(dy, dy, r2);
          r2 = f2_fma(dz, dz, r2);
          float lo, hi;
          f2_unpack(r2, lo, hi);
          const u64 ri = f2_pack(rsqrt_mufu(lo), rsqrt_mufu(hi));
          const u64 ri2 = f2_mul(ri, ri);
          if constexpr (UNI) {
            const u64 s = f2_mul(ri2, ri);
            a.ax[p] = f2_fma(dx, s, a.ax[p]);
            a.ay[p] = f2_fma(dy, s, a.ay[p]);
            a.az[p] = f2_fma(dz, s, a.az[p]);
            jx = f2_fma(dx, s, jx);
            jy = f2_fma(dy, s, jy);
            jz = f2_fma(dz, s, jz);
            if constexpr (POT) {
              a.ap[p] = f2_add(a.ap[p], ri);
              ps = f2_add(ps, ri);
            }
          } else {
            const u64 qi = lds_u64(smem_u32(&ks.q[p][threadIdx.x]));
            const u64 pi = f2_mul(qj, ri), pj = f2_mul(qi, ri);
            const u64 si = f2_mul(pi, ri2), sj = f2_mul(pj, ri2);
            a.ax[p] = f2_fma(dx, si, a.ax[p]);
            a.ay[p] = f2_fma(dy, si, a.ay[p]);
            a.az[p] = f2_fma(dz, si, a.az[p]);
            jx = f2_fma(dx, sj, jx);
            jy = f2_fma(dy, sj, jy);
            jz = f2_fma(dz, sj, jz);
            if constexpr (POT) {
              a.ap[p] = f2_add(a.ap[p], pi);
              ps = f2_add(ps, pj);
            }
          }
        }
        if constexpr (POT) kahan_add2(jp, jc, ps);
        jx = shfl_u64(jx, next);
        jy = shfl_u64(jy, next);
        jz = shfl_u64(jz, next);
        if constexpr (POT) {
          jp = shfl_u64(jp, next);
          jc = shfl_u64(jc, next);
        }
      }
      if constexpr (POT) {
        if (k0 & 4) fold_phi(ks, a, qq, UNI);
      }
    }
    float lo, hi;
    f2_unpack(jx, lo, hi);
    jout[c + lane] = lo + hi;
    f2_unpack(jy, lo, hi);
    jout[TILE + c + lane] = lo + hi;
    f2_unpack(jz, lo, hi);
    jout[2 * TILE + c + lane] = lo + hi;
    if constexpr (POT) {
      float clo, chi;
      f2_unpack(jp, lo, hi);
      f2_unpack(jc, clo, chi);
      jphi[c + lane] = (static_cast<double>(lo) - clo) + (static_cast<double>(hi) - chi);
    }
  }
}

// One warp: every source of a tile against this warp's targets, one-sided
// (the tiles of the block's own records).
template <int P, int TILE, bool UNI, bool POT, bool IMG>
__device__ __forceinline__ void own_tile(const MutTile<TILE>& dup, int cnt,
                                         const u64 (&xi)[P], const u64 (&yi)[P],
                                         const u64 (&zi)[P], u64 e2, MutAcc<P, POT>& a,
                                         MutSmem<P, POT>& ks, u64 qq, const u64 (&mi)[3]) {
  const uint32_t bxy = smem_u32(&dup.xy[0]), bzq = smem_u32(&dup.zq[0]);
  AccP<P, POT> b;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    b.ax[p] = a.ax[p];
    b.ay[p] = a.ay[p];
    b.az[p] = a.az[p];
    b.ap[p] = 0ull;
  }
  // cnt is a multiple of kPad
#pragma unroll 1
  for (int j = 0; j < cnt; j += 4) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const ulonglong2 xy = lds_u64x2(bxy + 16u * (j + k)), zq = lds_u64x2(bzq + 16u * (j + k));
      if constexpr (UNI)
        pair2_u<P, POT, IMG>(xy, zq, xi, yi, zi, e2, b, mi);
      else
        pair2<P, POT, IMG>(xy, zq, xi, yi, zi, e2, b, mi);
    }
    if constexpr (POT) {
      if (j & 4) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
          a.ap[p] = b.ap[p];
          b.ap[p] = 0ull;
        }
        fold_phi(ks, a, qq, UNI);
      }
    }
  }
#pragma unroll
  for (int p = 0; p < P; ++p) {
    a.ax[p] = b.ax[p];
    a.ay[p] = b.ay[p];
    a.az[p] = b.az[p];
  }
}

template <int R, int TILE, bool POT, bool MI>
__global__ void __launch_bounds__(kMutThreads) k_mut_pairs(const MutArgs a) {
  static_assert(R % 2 == 0, "two targets per packed register");
  constexpr int P = R / 2, kBlock = kMutThreads * R;
  static_assert(kBlock % TILE == 0 && TILE % 32 == 0, "tiles of one block, chunks of 32");
  __shared__ Stage<TILE, 1> sm;
  __shared__ MutTile<TILE> dup;
  __shared__ MutSmem<P, POT> ks;
  __shared__ float s_j[kMutWarps][3 * TILE];
  __shared__ double s_jp[POT ? kMutWarps : 1][POT ? TILE : 1];
  __shared__ u64 s_mi[3][MI ? kMutThreads : 1];
  __shared__ float s_tb[6];
  __shared__ int s_unit, s_abort;
  __shared__ MutUnit s_un;
  __shared__ ClusterDev s_c;

  const int tid = threadIdx.x, warp = tid >> 5;
  const long long step = __ldcg(a.s.step);
  if (tid == 0) {
    mbar_init(&sm.full[0], 1);
    fence_mbar_init();
    s_abort = 0;
  }
  // the clusters' laser fields for the push, one CTA each
  if (tid == 32) {
    for (int c = blockIdx.x; c < a.n_clusters; c += gridDim.x) {
      const ClusterDev& cl = a.s.cl[c];
      laser_field(cl, cl.t0 + static_cast<double>(step) * cl.dt, a.las + 6 * c);
    }
  }
  __syncthreads();
  const float4* __restrict__ cur = (step & 1) ? a.s.posq1 : a.s.posq0;
  unsigned it = 0;  // tiles consumed (the barrier's phase)
  for (;;) {
    if (tid == 0) s_unit = static_cast<int>(atomicAdd(a.s.ticket, 1u));
    __syncthreads();
    const int share = s_unit;
    __syncthreads();
    if (share >= a.n_shares) break;
    const int u_end = a.share_first[share + 1];
#pragma unroll 1
    for (int u = a.share_first[share]; u < u_end; ++u) {
      if (tid == 0) {
        s_un = a.units[u];
        s_c = a.s.cl[s_un.cluster];
      }
      __syncthreads();
      // (checked build; the whole CTA decides alike) the unit, and its tiles in the cluster
      if (!MD_IN_RANGE(a.s.err, u, 0, a.n_units) ||
          !MD_IN_RANGE(a.s.err, s_un.cluster, 0, a.n_clusters) ||
          !MD_IN_RANGE(a.s.err, static_cast<long long>(s_un.block) * kBlock, 0, s_c.n_pad) ||
          !MD_IN_RANGE(a.s.err, s_un.t0, 0, s_un.t0 + s_un.nt) ||
          !MD_IN_RANGE(a.s.err,
                       static_cast<long long>(s_un.block) * kBlock +
                           static_cast<long long>(s_un.t0 + s_un.nt - 1) * TILE,
                       0, s_c.n_pad) ||
          !MD_IN_RANGE(a.s.err, s_c.off + s_c.n_pad, 1, a.s.n_total + 1) ||
          !MD_IN_RANGE(a.s.err, s_un.jrow, 0, a.n_jrecs + 1) ||
          !MD_IN_RANGE(a.s.err,
                       s_un.jrow + s_c.n_pad - static_cast<long long>(s_un.block + 1) * kBlock,
                       -kBlock, a.n_jrecs + 1)) {
        __syncthreads();
        continue;
      }
      const long long i0 = static_cast<long long>(s_un.block) * kBlock;
      const float4* __restrict__ blk = cur + s_c.off + i0;
      const int left = s_c.n_pad - static_cast<int>(i0);  // records from this block on
      const int t_end = s_un.t0 + s_un.nt;
      // tile s_un.t0 is on its way while the targets are loaded
      if (tid == 0) issue_tile<TILE, 1>(sm, it, blk, left, s_un.t0);
      u64 xi2[P], yi2[P], zi2[P];
      MutAcc<P, POT> acc;
      bool uni_i = true;
      const float q_i = blk[0].w;
      {
        float xi[R], yi[R], zi[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int k = tid + r * kMutThreads;
          const float4 p = k < left ? blk[k] : make_float4(0.f, 0.f, 0.f, q_i);
          xi[r] = p.x;
          yi[r] = p.y;
          zi[r] = p.z;
          uni_i = uni_i && p.w == q_i;
          float* qs = reinterpret_cast<float*>(&ks.q[r >> 1][tid]);
          qs[r & 1] = p.w;
        }
#pragma unroll
        for (int p = 0; p < P; ++p) {
          // through shared memory, so that ptxas keeps register pairs (KahanSmem)
          ks.v[0][p][tid] = f2_pack(xi[2 * p], xi[2 * p + 1]);
          ks.v[1][p][tid] = f2_pack(yi[2 * p], yi[2 * p + 1]);
          ks.v[2][p][tid] = f2_pack(zi[2 * p], zi[2 * p + 1]);
          xi2[p] = lds_u64(smem_u32(&ks.v[0][p][tid]));
          yi2[p] = lds_u64(smem_u32(&ks.v[1][p][tid]));
          zi2[p] = lds_u64(smem_u32(&ks.v[2][p][tid]));
          acc.ax[p] = acc.ay[p] = acc.az[p] = 0ull;
          if constexpr (POT) acc.ap[p] = 0ull;
#pragma unroll
          for (int k = 0; k < (POT ? 8 : 6); ++k) ks.v[k][p][tid] = 0ull;
        }
        if constexpr (MI) target_bounds<kMutThreads, R>(xi, yi, zi, s_tb);
      }
      uni_i = __syncthreads_and(uni_i);
      const bool dark_i = uni_i && q_i == 0.0f;
      ks.e2[tid] = f2_pack(s_c.eps2, s_c.eps2);
      const u64 e2 = lds_u64(smem_u32(&ks.e2[tid]));
      u64 mi[3] = {0ull, 0ull, 0ull};
      bool mi_on = false;
      float L = 0.0f;
      if constexpr (MI) {
        const double t_n = s_c.t0 + static_cast<double>(step) * s_c.dt;
        mi_on = a.s.min_image && a.s.min_image[s_un.cluster] &&
                (s_c.boundary == 1 || (s_c.boundary == 2 && t_n < s_c.t_switch));
        L = static_cast<float>(s_c.box);
        const float invL = 1.0f / L;
        s_mi[0][tid] = f2_pack(-L, -L);
        s_mi[1][tid] = f2_pack(invL, invL);
        s_mi[2][tid] = f2_pack(12582912.0f, 12582912.0f);
#pragma unroll
        for (int k = 0; k < 3; ++k) mi[k] = lds_u64(smem_u32(&s_mi[k][tid]));
      }
      // records after this block: the columns of its jpart rows
      const long long later = left - kBlock;
      float* jrow = a.jpart + 3 * (s_un.jrow);
      double* prow = POT ? a.jphi + s_un.jrow : nullptr;

#pragma unroll 1
      for (int t = s_un.t0; t < t_end; ++t, ++it) {
        if (!mbar_wait(&sm.full[0], it & 1u)) {
          atomicOr(a.s.err, kErrTimeout);
          s_abort = 1;
        }
        const int rem = left - t * TILE;
        const int cnt = rem < TILE ? rem : TILE;
        const int cnt32 = (cnt + 31) & ~31;
        float qt = 0.0f;
        bool uni = false, img = false;
        if (!*reinterpret_cast<volatile int*>(&s_abort)) {
          uni = tile_uniform_q(smem_u32(&sm.tile[0][0]), cnt, qt);
          if constexpr (MI)
            img = mi_on && tile_needs_image(smem_u32(&sm.tile[0][0]), cnt, s_tb, L);
          for (int k = tid; k < cnt32; k += kMutThreads) {
            const float4 p = k < cnt ? sm.tile[0][k] : make_float4(kFar, kFar, kFar, 0.0f);
            dup.xy[k] = make_ulonglong2(f2_pack(p.x, p.x), f2_pack(p.y, p.y));
            dup.zq[k] = make_ulonglong2(f2_pack(p.z, p.z), f2_pack(p.w, p.w));
          }
        }
        __syncthreads();
        // an expired wait: the one copy in flight is awaited once more (bounded)
        if (*reinterpret_cast<volatile int*>(&s_abort)) {
          if (tid == 0) mbar_wait(&sm.full[0], it & 1u);
          return;
        }
        if (tid == 0 && t + 1 < t_end) issue_tile<TILE, 1>(sm, it + 1, blk, left, t + 1);
        const u64 qq = f2_pack(qt, qt);
        const bool mutual = t * TILE >= kBlock;
        const long long col = static_cast<long long>(t) * TILE - kBlock;
        // what carries no charge adds to no field: nothing of an uncharged tile
        // at its own block or at uncharged targets, only the targets' side of a
        // tile of an uncharged block (an uncharged tile's own fields are summed:
        // its records may be test particles of no weight).  100k records, the
        // last half of them unused slots: 1.99 ms per step, 2.51 with every tile
        // summed, 2.20 with the step kernel
        const bool dark = uni && qt == 0.0f;
        if (dark && (!mutual || dark_i)) {
          if (mutual) {
            for (int k = tid; k < cnt; k += kMutThreads) {
              if (!MD_IN_RANGE(a.s.err, col + k, 0, later)) continue;
#pragma unroll
              for (int c = 0; c < 3; ++c) __stcg(jrow + c * later + col + k, 0.0f);
              if constexpr (POT) __stcg(prow + col + k, 0.0);
            }
          }
          continue;
        }
        const bool one_sided = !mutual || dark_i;
        // (a minimum image would bring a far padding source near, so a padded
        // tile that needs images applies the charges, 0 for the padding)
        const bool charged_alike = uni && (one_sided || (uni_i && !(img && cnt32 != cnt)));
        auto sum = [&](auto img_tag) {
          constexpr bool IMG = decltype(img_tag)::value;
          float* jo = s_j[warp];
          double* jph = s_jp[POT ? warp : 0];
          if (!one_sided) {
            if (charged_alike)
              mutual_tile<P, TILE, true, POT, IMG>(dup, cnt32, xi2, yi2, zi2, e2, acc, ks, jo, jph, qq,
                                                mi);
            else
              mutual_tile<P, TILE, false, POT, IMG>(dup, cnt32, xi2, yi2, zi2, e2, acc, ks, jo, jph,
                                                 qq, mi);
          } else {
            if (charged_alike)
              own_tile<P, TILE, true, POT, IMG>(dup, cnt, xi2, yi2, zi2, e2, acc, ks, qq, mi);
            else
              own_tile<P, TILE, false, POT, IMG>(dup, cnt, xi2, yi2, zi2, e2, acc, ks, qq, mi);
          }
        };
        if (MI && img)
          sum(std::integral_constant<bool, MI>{});
        else
          sum(std::false_type{});
        const u64 qf = charged_alike ? qq : f2_pack(1.0f, 1.0f);
#pragma unroll
        for (int p = 0; p < P; ++p) {
          if (!dark) {
            u64 sv, cv;
            sv = ks.v[0][p][tid]; cv = ks.v[3][p][tid];
            kahan_add2(sv, cv, f2_mul(acc.ax[p], qf));
            ks.v[0][p][tid] = sv; ks.v[3][p][tid] = cv;
            sv = ks.v[1][p][tid]; cv = ks.v[4][p][tid];
            kahan_add2(sv, cv, f2_mul(acc.ay[p], qf));
            ks.v[1][p][tid] = sv; ks.v[4][p][tid] = cv;
            sv = ks.v[2][p][tid]; cv = ks.v[5][p][tid];
            kahan_add2(sv, cv, f2_mul(acc.az[p], qf));
            ks.v[2][p][tid] = sv; ks.v[5][p][tid] = cv;
          }
          acc.ax[p] = acc.ay[p] = acc.az[p] = 0ull;
        }
        __syncthreads();  // dup is rewritten by the next tile; the warps' s_j are complete
        if (mutual) {
          // (s_j is written again only after the next tile's barrier)
          const float qi = charged_alike ? q_i : 1.0f;
          for (int k = tid; k < cnt; k += kMutThreads) {
            if (!MD_IN_RANGE(a.s.err, col + k, 0, later)) continue;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              const float s = (s_j[0][c * TILE + k] + s_j[1][c * TILE + k]) +
                              (s_j[2][c * TILE + k] + s_j[3][c * TILE + k]);
              __stcg(jrow + c * later + col + k, one_sided ? 0.0f : s * qi);
            }
            if constexpr (POT)
              __stcg(prow + col + k,
                     one_sided ? 0.0
                               : ((s_jp[0][k] + s_jp[1][k]) + (s_jp[2][k] + s_jp[3][k])) * qi);
          }
        }
      }
      // this unit's Kahan sums and compensations at its targets (of
      // sum Q (x_j - x_i)/r^3, and of the potential)
      float2* ip = a.ipart + (POT ? 4 : 3) * static_cast<long long>(kBlock) * u;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int k = tid + r * kMutThreads;
#pragma unroll
        for (int c = 0; c < (POT ? 4 : 3); ++c) {
          const int kc = c < 3 ? c : 6, cc = c < 3 ? c + 3 : 7;
          float s0, s1, c0, c1;
          f2_unpack(ks.v[kc][r >> 1][tid], s0, s1);
          f2_unpack(ks.v[cc][r >> 1][tid], c0, c1);
          __stcg(ip + c * kBlock + k, (r & 1) ? make_float2(s1, c1) : make_float2(s0, c0));
        }
      }
      __syncthreads();  // s_un, s_c and ks are rewritten by the next unit
    }
  }
}

// The push of every record: its partials in a fixed order, laser, kick, drift.
// Runs after k_mut_pairs, whose ticket it resets; its last CTA advances the
// step.  A CTA takes 32 records: warp w of W adds the work units and the earlier
// blocks' rows w, w + W, ... in Kahan-compensated FP32, and the first warp joins
// the W sums and pushes with the laser field that the pair kernel left.  86 us at
// 200k records (0.3 GB of partials) with W = 4, 10.9 at 19k with 8; one thread per
// record with FP64 adds, which the narrow FP64 pipe bounds, took 240 and 32, the
// laser's sine in every CTA 136 and 14, the W sums in FP64 99 and 12.2.
constexpr int kPushRec = 32;

template <int kPushWarps, bool DET, bool POT>
__global__ void __launch_bounds__(32 * kPushWarps) k_mut_push(const MutArgs a) {
  constexpr int C = POT ? 4 : 3;
  __shared__ float2 s_e[3][kPushWarps][kPushRec];  // the warps' sums (value x - y)
  __shared__ double s_ph[POT ? kPushWarps : 1][kPushRec];
  __shared__ ClusterDev s_c;
  __shared__ float s_las[6];
  const long long step = __ldcg(a.s.step);
  // a wait of k_mut_pairs ran out: its partials are incomplete, push nothing
  if (__ldcg(a.s.err) & kErrTimeout) return;
  const int per = a.block / kPushRec;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const MutBlk b = a.blks[blockIdx.x / per];
  const ClusterDev* cl = a.s.cl + b.cluster;
  const int n_pad = cl->n_pad;
  const int k = static_cast<int>(blockIdx.x % per) * kPushRec + lane;  // in the block
  const long long j = static_cast<long long>(b.block) * a.block + k;   // in the cluster
  const bool live = j < n_pad && MD_IN_RANGE(a.s.err, cl->off + j, 0, a.s.n_total) &&
                    MD_IN_RANGE(a.s.err, b.unit0, 0, a.n_units) &&
                    MD_IN_RANGE(a.s.err, b.unit0 + b.units, 1, a.n_units + 1);
  RecState st;
  static_assert(sizeof(ClusterDev) % 4 == 0, "copied by words");
  for (int q = threadIdx.x; q < static_cast<int>(sizeof(ClusterDev) / 4); q += 32 * kPushWarps)
    reinterpret_cast<int*>(&s_c)[q] = reinterpret_cast<const int*>(cl)[q];
  if (threadIdx.x < 6) s_las[threadIdx.x] = a.las[6 * b.cluster + threadIdx.x];
  if (live) {
    if (warp == 0) st = load_state(a.s, cl->off + j);
    float s[3] = {0.f, 0.f, 0.f}, c[3] = {0.f, 0.f, 0.f};
    double ph = 0.0;
    const float2* ip = a.ipart + C * static_cast<long long>(a.block) * b.unit0 + k;
#pragma unroll 2
    for (int p = warp; p < b.units; p += kPushWarps) {
      const float2* q = ip + static_cast<long long>(p) * C * a.block;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        // the units sum x_j - x_i: their field has the other sign
        const float2 v = __ldcg(q + m * a.block);
        kahan_add(s[m], c[m], -v.x);
        kahan_add(s[m], c[m], v.y);
      }
      if constexpr (POT) {
        const float2 v = __ldcg(q + 3 * a.block);
        ph += static_cast<double>(v.x) - v.y;
      }
    }
    // row I: the records after block I, `later` of them, three components apart
#pragma unroll 4
    for (int I = warp; I < b.block; I += kPushWarps) {
      const long long skipped = static_cast<long long>(I) * n_pad -
                                static_cast<long long>(a.block) * I * (I + 1) / 2;
      const long long later = n_pad - static_cast<long long>(I + 1) * a.block;
      const long long col = j - static_cast<long long>(I + 1) * a.block;
      if (!MD_IN_RANGE(a.s.err, col, 0, later) ||
          !MD_IN_RANGE(a.s.err, b.jbase + skipped + later, 1, a.n_jrecs + 1))
        continue;
      const float* row = a.jpart + 3 * (b.jbase + skipped) + col;
#pragma unroll
      for (int m = 0; m < 3; ++m) kahan_add(s[m], c[m], __ldcg(row + m * later));
      if constexpr (POT) ph += __ldcg(a.jphi + b.jbase + skipped + col);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) s_e[m][warp][lane] = make_float2(s[m], c[m]);
    if constexpr (POT) s_ph[warp][lane] = ph;
  }
  __syncthreads();
  if (warp == 0) {
    if (live) {
      double e[C];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        float2 v = s_e[m][0][lane];
#pragma unroll
        for (int w = 1; w < kPushWarps; ++w)
          join_sums(v.x, v.y, s_e[m][w][lane].x, s_e[m][w][lane].y);
        e[m] = static_cast<double>(v.x) - v.y;
      }
      if constexpr (POT) {
        e[3] = 0.0;
#pragma unroll
        for (int w = 0; w < kPushWarps; ++w) e[3] += s_ph[w][lane];
      }
      const float4* __restrict__ cur = (step & 1) ? a.s.posq1 : a.s.posq0;
      float4* __restrict__ nxt = (step & 1) ? a.s.posq0 : a.s.posq1;
      const double t_next = s_c.t0 + static_cast<double>(step + 1) * s_c.dt;
      const long long i = s_c.off + j;
      if constexpr (POT) {
        // the potential without the record's own term
        const double phi = e[3] - static_cast<double>(cur[i].w * rsqrt_mufu(s_c.eps2));
        push_loaded<DET, true>(a.s, s_c, i, st, e[0], e[1], e[2], s_las, t_next, cur, nxt, phi);
      } else {
        push_loaded<DET>(a.s, s_c, i, st, e[0], e[1], e[2], s_las, t_next, cur, nxt);
      }
    }
  } else if (threadIdx.x == 32) {
    const unsigned prev = atomicAdd(a.s.done, 1u);  // every warp here has read the step
    if (prev == gridDim.x - 1) {
      atomicExch(a.s.ticket, 0u);
      atomicExch(a.s.done, 0u);
      *reinterpret_cast<volatile long long*>(a.s.step) = step + 1;
    }
  }
}

template <int R>
cudaError_t blocks_per_sm_r(bool pot, bool mi, int* out) {
  if (mi)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_mut_pairs<R, kTile, false, true>,
                                                         kMutThreads, 0);
  if (pot)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_mut_pairs<R, kTile, true, false>,
                                                         kMutThreads, 0);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_mut_pairs<R, kTile, false, false>,
                                                       kMutThreads, 0);
}

template <int R>
void launch_pairs_r(const MutArgs& a, int grid, bool pot, bool mi, cudaStream_t s) {
  if (mi)
    k_mut_pairs<R, kTile, false, true><<<grid, kMutThreads, 0, s>>>(a);
  else if (pot)
    k_mut_pairs<R, kTile, true, false><<<grid, kMutThreads, 0, s>>>(a);
  else
    k_mut_pairs<R, kTile, false, false><<<grid, kMutThreads, 0, s>>>(a);
}

template <int W>
void launch_push_w(const MutArgs& a, unsigned g, bool det, bool pot, cudaStream_t s) {
  if (det)
    k_mut_push<W, true, false><<<g, 32 * W, 0, s>>>(a);
  else if (pot)
    k_mut_push<W, false, true><<<g, 32 * W, 0, s>>>(a);
  else
    k_mut_push<W, false, false><<<g, 32 * W, 0, s>>>(a);
}

}  // namespace

cudaError_t mut_blocks_per_sm(int block, bool pot, bool mi, int* out) {
  return block == kMutThreads * 12 ? blocks_per_sm_r<12>(pot, mi, out)
                                   : blocks_per_sm_r<8>(pot, mi, out);
}

cudaError_t launch_mut_step(const MutArgs& a, int grid, bool det, bool pot, bool mi,
                            cudaStream_t s) {
  if (a.block == kMutThreads * 12)
    launch_pairs_r<12>(a, grid, pot, mi, s);
  else if (a.block == kMutThreads * 8)
    launch_pairs_r<8>(a, grid, pot, mi, s);
  else
    return cudaErrorInvalidValue;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const unsigned g = static_cast<unsigned>(a.n_blks) * static_cast<unsigned>(a.block / kPushRec);
  // eight warps while the CTAs are few (19k records: 12.5 us against 18 with
  // four), four once they fill the SMs (a scan of 290k records: 81 against 125;
  // both sides with the warps' sums in FP64, now 10.9 and 59)
  if (g >= 8u * static_cast<unsigned>(a.sms))
    launch_push_w<4>(a, g, det, pot, s);
  else
    launch_push_w<8>(a, g, det, pot, s);
  return cudaGetLastError();
}

}  // namespace md
