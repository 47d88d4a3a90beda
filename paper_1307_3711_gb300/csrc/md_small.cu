// md_small.cu -- the step of a few thousand records.
//
// Such a step is bound by latency, not by the pair sums (2000 records: 1.2 us
// of the FP32 pipe), and the large kernels' blocks leave most of the chip idle.
// Here a CTA takes kTargets targets, few enough that the CTAs cover the SMs,
// and all its warps share them: every (target lane, slice) thread sums the
// sources j = slice, slice + kSlices, ... of each staged tile, the slices' sums
// are added in a fixed order as compensated FP32 pairs (an FP64 instruction takes
// its pipe 16 cycles) through shared memory, and the targets are
// pushed by the CTA that summed them: one launch, no partial sums
// in memory, no ticket.  The laser's FP64 envelope and sine run in two warps of
// their own beside the sums, the targets' state is loaded before them, and the
// step counter is advanced beside the push.
//
// A wait that runs out: the CTA pushes nothing, waits (bounded) for its copies
// still in flight and leaves; the step does not advance, and the launches that
// follow (of the same graph) find the error bit and push nothing.
//
// Measured (graph replay, us per step): 7.0 at 2000 records (53 with the step
// kernel's default configuration; 8.1 with the slices' sums in FP64 and the last
// few sources of a tile one by one), 5.1 at 1000, 11.9 at 3000, 14.6 at 4000, 41.6
// at 8000; about 5 us of each are the launch, the loads and the push.  More
// threads per CTA (512, 768), two or four targets per thread, 8 targets per
// CTA, two stages, a register cap for a fourth CTA per SM and programmatic
// launches were slower or no faster.
#include "md_device.cuh"
#include "md_internal.h"

namespace md {

namespace {

constexpr int kTile = 1024;   // sources per stage
constexpr int kStages = 4;

template <int THREADS, int TL, int R, bool POT>
struct SmallSmem {
  Stage<kTile, kStages> st;
  float2 e[POT ? 4 : 3][THREADS / 32][TL * R];  // the warps' sums (value x - y)
  float2 sum[POT ? 4 : 3][TL * R];
  ClusterDev c;
  double amp, sn, cs;  // the laser at t_n
};

// One target group: TL lanes x R targets, THREADS / TL slices of the sources.
template <int THREADS, int TL, int R, bool DET, bool POT>
__global__ void __launch_bounds__(THREADS + 64) k_step_small(const StepArgs a,
                                                             const SmallBlk* blks) {
  constexpr int kTargets = TL * R;
  constexpr int kSlices = THREADS / TL;
  constexpr int C = POT ? 4 : 3;
  __shared__ SmallSmem<THREADS, TL, R, POT> S;

  const int tid = threadIdx.x;
  const SmallBlk b = blks ? blks[blockIdx.x] : SmallBlk{0, static_cast<int>(blockIdx.x) * kTargets};
  const ClusterDev* cl = a.cl + b.cluster;
  const long long off = cl->off;
  const int n_pad = cl->n_pad;
  const float eps2 = cl->eps2;
  if (tid == THREADS) {
    for (int s = 0; s < kStages; ++s) mbar_init(&S.st.full[s], 1);
    fence_mbar_init();
  }
  const long long step = __ldcg(a.step);
  const float4* __restrict__ cur = ((step & 1) ? a.posq1 : a.posq0);
  float4* __restrict__ nxt = (step & 1) ? a.posq0 : a.posq1;
  const float4* __restrict__ src = cur + off;
  const int ntiles = (n_pad + kTile - 1) / kTile;
  const int lead = ntiles < kStages ? ntiles : kStages;
  const int tl = tid % TL, slice = tid / TL;
  float xi[R], yi[R], zi[R];
  RecState st;
  const bool pushes = tid < kTargets && b.t0 + tid < n_pad &&
                      MD_IN_RANGE(a.err, off + b.t0 + tid, 0, a.n_total);
  if (tid >= THREADS) {
    if (tid == THREADS)
      for (int t = 0; t < lead; ++t)
        issue_tile<kTile, kStages>(S.st, static_cast<unsigned>(t), src, n_pad, t);
    static_assert(sizeof(ClusterDev) % 4 == 0, "copied by words");
    const int* from = reinterpret_cast<const int*>(cl);
    int* to = reinterpret_cast<int*>(&S.c);
    for (int k = tid - THREADS; k < static_cast<int>(sizeof(ClusterDev) / 4); k += 64) to[k] = from[k];
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = b.t0 + tl + r * TL;
      const float4 p = i < n_pad ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      xi[r] = p.x;
      yi[r] = p.y;
      zi[r] = p.z;
    }
    if (pushes) st = load_state(a, off + b.t0 + tid);
  }
  __syncthreads();  // the first copies are issued, the descriptor is in place
  // the tiles of the group from t0 on, before their CTA leaves
  auto drain = [&](int t0) {
    if (tid == THREADS)
      for (int t = t0; t < ntiles && t < t0 + kStages; ++t)
        mbar_wait(&S.st.full[t % kStages], (t / kStages) & 1u);
  };
  // a wait of this thread ran out, or (the thread that asks) one of an earlier launch
  bool late = false;
  if (tid >= THREADS) {
    const double t_n = S.c.t0 + static_cast<double>(step) * S.c.dt;
    if (tid == THREADS) {
      S.amp = S.c.a0 * envelope(t_n, S.c.env, S.c.tau);
      late = __ldcg(a.err) & kErrTimeout;
    } else if (tid == THREADS + 32) {
      sincos(t_n, &S.sn, &S.cs);
    }
  }
  Acc<R, POT> acc;
  acc.zero();
  for (int t0 = 0; t0 < ntiles; t0 += kStages) {
    if (tid < THREADS) {
      for (int t = t0; t < ntiles && t < t0 + kStages; ++t) {
        const int s = t % kStages;
        if (!mbar_wait(&S.st.full[s], (t / kStages) & 1u)) {
          atomicOr(a.err, kErrTimeout);
          late = true;
          break;
        }
        const int rem = n_pad - t * kTile, cnt = rem < kTile ? rem : kTile;
        const uint32_t tile = smem_u32(&S.st.tile[s][0]);
        auto fold_phi = [&] {
          if constexpr (POT) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
              kahan_add(acc.sp[r], acc.cp[r], acc.ap[r]);
              acc.ap[r] = 0.0f;
            }
          }
        };
        int k = slice;
        for (; k + 7 * kSlices < cnt; k += 8 * kSlices) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            pair<R, POT>(lds_f4(tile + 16u * (k + q * kSlices)), xi, yi, zi, eps2, acc);
          fold_phi();
        }
        if (k < cnt) {
          // the last few at once too: past the end the tile's last source, uncharged
#pragma unroll
          for (int q = 0; q < 7; ++q) {
            const int j = k + q * kSlices;
            float4 p = lds_f4(tile + 16u * (j < cnt ? j : cnt - 1));
            p.w = j < cnt ? p.w : 0.0f;
            pair<R, POT>(p, xi, yi, zi, eps2, acc);
          }
          fold_phi();
        }
        fold<R, POT>(acc);
      }
    }
    if (t0 + kStages < ntiles) {
      // every stage is read: refill (a cluster of more than kStages tiles)
      if (__syncthreads_or(late)) {
        drain(t0);
        return;
      }
      if (tid == THREADS)
        for (int t = t0 + kStages; t < ntiles && t < t0 + 2 * kStages; ++t)
          issue_tile<kTile, kStages>(S.st, static_cast<unsigned>(t), src, n_pad, t);
    }
  }
  if (tid < THREADS) {
    auto put = [&](int c, int r, float v, float w) {
#pragma unroll
      for (int d = TL; d < 32; d <<= 1)
        join_sums(v, w, __shfl_xor_sync(0xffffffffu, v, d), __shfl_xor_sync(0xffffffffu, w, d));
      if ((tid & 31) < TL) S.e[c][tid >> 5][tl + r * TL] = make_float2(v, w);
    };
#pragma unroll
    for (int r = 0; r < R; ++r) {
      put(0, r, acc.sx[r], acc.cx[r]);
      put(1, r, acc.sy[r], acc.cy[r]);
      put(2, r, acc.sz[r], acc.cz[r]);
      if constexpr (POT) put(3, r, acc.sp[r], acc.cp[r]);
    }
  }
  if (__syncthreads_or(late)) {
    drain((ntiles - 1) / kStages * kStages);
    return;
  }
  if (tid >= THREADS) {
    // every thread of this CTA has read the step, and its sums are complete: the
    // last CTA to get here advances it (beside the join and the push of the others)
    if (tid == THREADS) {
      const unsigned prev = atomicAdd(a.done, 1u);
      if (prev == gridDim.x - 1) {
        atomicExch(a.done, 0u);
        *reinterpret_cast<volatile long long*>(a.step) = step + 1;
      }
    }
    return;
  }
  // each value's warps: kJoin neighbouring lanes add some each, then each other's
  constexpr int kWarps = THREADS / 32, kJoin = THREADS / (4 * kTargets);
  static_assert(kJoin >= 1 && kJoin <= kWarps, "lanes per value");
  {
    const int k = tid / kJoin, c = k / kTargets, t = k % kTargets;
    float2 v = make_float2(0.0f, 0.0f);
    if (k < C * kTargets) {
      v = S.e[c][tid % kJoin][t];
#pragma unroll
      for (int w = tid % kJoin + kJoin; w < kWarps; w += kJoin)
        join_sums(v.x, v.y, S.e[c][w][t].x, S.e[c][w][t].y);
    }
#pragma unroll
    for (int d = kJoin / 2; d > 0; d >>= 1)
      join_sums(v.x, v.y, __shfl_xor_sync(0xffffffffu, v.x, d),
                __shfl_xor_sync(0xffffffffu, v.y, d));
    if (k < C * kTargets && tid % kJoin == 0) S.sum[c][t] = v;
  }
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");  // the summing threads
  if (pushes) {
    const long long i = off + b.t0 + tid;
    float las[6];
    laser_of(S.amp, S.sn, S.cs, S.c.pol, las);
    const double t_next = S.c.t0 + static_cast<double>(step + 1) * S.c.dt;
    auto value = [&](int c) {
      const float2 v = S.sum[c][tid];
      return static_cast<double>(v.x) - static_cast<double>(v.y);
    };
    if constexpr (POT) {
      const double ph = value(3) - static_cast<double>(cur[i].w * rsqrt_mufu(S.c.eps2));
      push_loaded<DET, true>(a, S.c, i, st, -value(0), -value(1), -value(2), las, t_next, cur,
                             nxt, ph);
    } else {
      push_loaded<DET>(a, S.c, i, st, -value(0), -value(1), -value(2), las, t_next, cur, nxt);
    }
  }
}

template <int THREADS, int TL, int R, bool DET, bool POT>
cudaError_t launch_k(const StepArgs& a, const SmallBlk* blks, int n_blks, cudaStream_t s) {
  k_step_small<THREADS, TL, R, DET, POT><<<n_blks, THREADS + 64, 0, s>>>(a, blks);
  return cudaGetLastError();
}

template <int THREADS, int TL, int R>
cudaError_t launch_t(const StepArgs& a, const SmallBlk* blks, int n_blks, bool det, bool pot,
                     cudaStream_t s) {
  if (det) return launch_k<THREADS, TL, R, true, false>(a, blks, n_blks, s);
  if (pot) return launch_k<THREADS, TL, R, false, true>(a, blks, n_blks, s);
  return launch_k<THREADS, TL, R, false, false>(a, blks, n_blks, s);
}

}  // namespace

cudaError_t launch_small_step(const StepArgs& a, const SmallBlk* blks, int n_blks, int targets,
                              bool det, bool pot, cudaStream_t s) {
  if (targets == 16) return launch_t<256, 16, 1>(a, blks, n_blks, det, pot, s);
  if (targets == 32) return launch_t<256, 32, 1>(a, blks, n_blks, det, pot, s);
  return cudaErrorInvalidValue;
}

}  // namespace md
