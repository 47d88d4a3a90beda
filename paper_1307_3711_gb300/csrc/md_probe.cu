// md_probe.cu -- field and potential at caller-given targets in one launch and
// without scratch memory.
//
// The field kernel of md_device.cuh gives a CTA 1024 targets and adds partial
// fields through memory: at a few hundred targets most of its lanes hold none.
// Here a cluster of CTAs takes kTargets targets; its CTAs share the sources,
// the warps of a CTA share its part (every TL lanes another source of the
// staged tile), the slices' sums are added in FP64 in shared memory and the
// CTAs' through distributed shared memory by the cluster's first CTA.
//
// Measured (us, field without the potential; in brackets the field kernel with
// its partials in memory, and the allocation-free kernel of 256-target blocks
// that this one replaced): 300 targets x 150k sources 49 (185, 657), 1000 x
// 4001 10.3 (237, 146), 1 x 150k 19 (171, 655), 1000 x 1M 586 (948, 4320), 3000
// x 1M 1650 (1756, 4325), 10000 x 150k 757 (675, 1012).  One target per thread
// reads a source from shared memory per pair, so where the field kernel's
// blocks fill the SMs it stays faster (field_uses_probe).
#include <algorithm>
#include <cmath>
#include <utility>

#include <cooperative_groups.h>

#include "md_device.cuh"
#include "md_internal.h"

namespace md {

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 512;
constexpr int kTile = 1024;  // sources per stage
constexpr int kStages = 3;
constexpr int kMaxCluster = 8;

template <int TL, int R, bool POT>
struct ProbeSmem {
  Stage<kTile, kStages> st;
  double e[POT ? 4 : 3][kThreads / TL][TL * R];       // the slices' sums
  double part[kMaxCluster][POT ? 4 : 3][TL * R];      // first CTA: the CTAs' sums
  int abort;
};

// CTA (x, rank) of cluster x: targets [x kTargets, ...), sources [rank seg, ...).
template <int TL, int R, bool POT>
__global__ void __launch_bounds__(kThreads) k_probe(const FieldArgs a, long long seg) {
  constexpr int kTargets = TL * R;
  constexpr int kSlices = kThreads / TL;
  constexpr int C = POT ? 4 : 3;
  __shared__ ProbeSmem<TL, R, POT> S;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank());
  const int ranks = static_cast<int>(cluster.num_blocks());
  // (the cluster's CTAs have all started before one writes to another's memory)
  auto started = cluster.barrier_arrive();
  const int tid = threadIdx.x;
  const long long group = blockIdx.x / ranks;
  const long long j0 = rank * seg;
  const long long ns = j0 >= a.ns ? 0 : (a.ns - j0 < seg ? a.ns - j0 : seg);
  const float4* __restrict__ src = a.src + j0;
  const int ntiles = static_cast<int>((ns + kTile - 1) / kTile);
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(&S.st.full[s], 1);
    fence_mbar_init();
    S.abort = 0;
    for (int t = 0; t < kStages && t < ntiles; ++t)
      issue_tile<kTile, kStages>(S.st, static_cast<unsigned>(t), src, ns, t);
  }
  const int tl = tid % TL, slice = tid / TL;
  const long long i0 = group * kTargets;
  float xi[R], yi[R], zi[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const long long i = i0 + tl + r * TL;
    const float4 p = i < a.nt ? a.tgt[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    xi[r] = p.x;
    yi[r] = p.y;
    zi[r] = p.z;
  }
  __syncthreads();
  Acc<R, POT> acc;
  acc.zero();
  for (int t = 0; t < ntiles; ++t) {
    const int s = t % kStages;
    if (!mbar_wait(&S.st.full[s], (t / kStages) & 1u)) {
      atomicOr(a.err, kErrTimeout);
      S.abort = 1;
    }
    const long long rem = ns - static_cast<long long>(t) * kTile;
    const int cnt = static_cast<int>(rem < kTile ? rem : kTile);
    const uint32_t tile = smem_u32(&S.st.tile[s][0]);
    int k = slice;
    for (; k + 7 * kSlices < cnt; k += 8 * kSlices) {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        pair<R, POT>(lds_f4(tile + 16u * (k + q * kSlices)), xi, yi, zi, a.eps2, acc);
      if constexpr (POT) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          kahan_add(acc.sp[r], acc.cp[r], acc.ap[r]);
          acc.ap[r] = 0.0f;
        }
      }
    }
    for (; k < cnt; k += kSlices)
      pair<R, POT>(lds_f4(tile + 16u * k), xi, yi, zi, a.eps2, acc);
    fold<R, POT>(acc);
    if (t + kStages < ntiles) {
      __syncthreads();  // the stage has been read by every warp
      if (tid == 0 && !S.abort)
        issue_tile<kTile, kStages>(S.st, static_cast<unsigned>(t + kStages), src, ns, t + kStages);
      if (S.abort) {  // an expired wait: no further copies, those in flight are awaited
        if (tid == 0)
          for (int q = t + 1; q < t + kStages && q < ntiles; ++q)
            mbar_wait(&S.st.full[q % kStages], (q / kStages) & 1u);
        break;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    S.e[0][slice][tl + r * TL] = -(static_cast<double>(acc.sx[r]) - acc.cx[r]);
    S.e[1][slice][tl + r * TL] = -(static_cast<double>(acc.sy[r]) - acc.cy[r]);
    S.e[2][slice][tl + r * TL] = -(static_cast<double>(acc.sz[r]) - acc.cz[r]);
    if constexpr (POT) S.e[3][slice][tl + r * TL] = static_cast<double>(acc.sp[r]) - acc.cp[r];
  }
  __syncthreads();
  cluster.barrier_wait(std::move(started));
  // each value's slices: eight neighbouring lanes add every eighth, then each other's
  constexpr int kVals = C * kTargets;
  double* to = &cluster.map_shared_rank(&S.part[0][0][0], 0)[rank * kVals];
  for (int v0 = 0; v0 < kVals; v0 += kThreads / 8) {
    const int v = v0 + tid / 8, c = v / kTargets, t = v % kTargets;
    double s = 0.0;
    if (v < kVals)
      for (int q = tid % 8; q < kSlices; q += 8) s += S.e[c][q][t];
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (v < kVals && tid % 8 == 0) to[v] = s;
  }
  cluster.sync();
  if (rank != 0 || tid >= kTargets) return;
  const long long i = i0 + tid;
  if (i >= a.nt) return;
  double e[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    e[c] = 0.0;
    for (int r = 0; r < ranks; ++r) e[c] += S.part[r][c][tid];
  }
  a.e[3 * i + 0] = e[0];
  a.e[3 * i + 1] = e[1];
  a.e[3 * i + 2] = e[2];
  if constexpr (POT) {
    if (a.self_offset >= 0) {
      const long long js = i + a.self_offset;
      if (js < a.ns) e[3] -= static_cast<double>(a.src[js].w * rsqrt_mufu(a.eps2));
    }
    a.phi[i] = e[3];
  }
}

template <int TL, int R, bool POT>
cudaError_t launch_t(const FieldArgs& a, int cluster, cudaStream_t s) {
  const long long groups = (a.nt + TL * R - 1) / (TL * R);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(groups * cluster));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = static_cast<unsigned>(cluster);
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  // whole cache lines of sources per CTA
  const long long seg = ((a.ns + cluster - 1) / cluster + 7) / 8 * 8;
  return cudaLaunchKernelEx(&cfg, k_probe<TL, R, POT>, a, seg);
}

template <int TL, int R>
cudaError_t launch_p(const FieldArgs& a, bool potential, int cluster, cudaStream_t s) {
  return potential ? launch_t<TL, R, true>(a, cluster, s) : launch_t<TL, R, false>(a, cluster, s);
}

// Field of few sources at many targets, two per thread.
template <bool POT>
__global__ void __launch_bounds__(128) k_few(const FieldArgs a) {
  constexpr int R = 2, kTileFew = 512;
  __shared__ Stage<kTileFew, 1> sm;
  __shared__ int s_abort;
  if (threadIdx.x == 0) {
    mbar_init(&sm.full[0], 1);
    fence_mbar_init();
    s_abort = 0;
  }
  __syncthreads();
  const long long i0 = static_cast<long long>(blockIdx.x) * (128 * R);
  float xi[R], yi[R], zi[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const long long i = i0 + threadIdx.x + r * 128;
    const float4 p = (i < a.nt) ? a.tgt[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    xi[r] = p.x;
    yi[r] = p.y;
    zi[r] = p.z;
  }
  Acc<R, POT> acc;
  acc.zero();
  unsigned it = 0;
  if (!sum_sources<128, R, kTileFew, 1, POT>(sm, it, a.src, a.ns, xi, yi, zi, a.eps2, acc, a.err,
                                             &s_abort))
    return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const long long i = i0 + threadIdx.x + r * 128;
    if (i >= a.nt) continue;
    a.e[3 * i + 0] = -(static_cast<double>(acc.sx[r]) - acc.cx[r]);
    a.e[3 * i + 1] = -(static_cast<double>(acc.sy[r]) - acc.cy[r]);
    a.e[3 * i + 2] = -(static_cast<double>(acc.sz[r]) - acc.cz[r]);
    if constexpr (POT) {
      double ph = static_cast<double>(acc.sp[r]) - acc.cp[r];
      if (a.self_offset >= 0 && i + a.self_offset < a.ns)
        ph -= static_cast<double>(a.src[i + a.self_offset].w * rsqrt_mufu(a.eps2));
      a.phi[i] = ph;
    }
  }
}

// With few sources for many targets a cluster per few targets costs more than
// it sums: 30000 targets x 100 sources 13 us with k_few, 27 with clusters; 10000
// x 100 12.7 and 14.5, 3000 x 100 11.7 and 13.3 (k_few takes 35 ns per source).
bool few_sources(long long nt, long long ns) {
  return ns < 512 && nt > (ns < 160 ? 1024 : 8192);
}

}  // namespace

cudaError_t launch_field_direct(const FieldArgs& a, bool potential, int sms, cudaStream_t s) {
  if (a.nt <= 0) return cudaSuccess;
  if (few_sources(a.nt, a.ns)) {
    const unsigned g = static_cast<unsigned>((a.nt + 255) / 256);
    if (potential)
      k_few<true><<<g, 128, 0, s>>>(a);
    else
      k_few<false><<<g, 128, 0, s>>>(a);
    return cudaGetLastError();
  }
  // as many CTAs per cluster as leave each a stage of sources; then the most
  // targets per CTA that still give five CTAs to three SMs (fewer targets: the
  // sources are staged more often; fewer CTAs: idle SMs)
  int cluster = 1;
  while (cluster < kMaxCluster && a.ns / (2 * cluster) >= 1000) cluster *= 2;
  const long long want = 5LL * sms / 3;
  auto ctas = [&](long long tl) { return (a.nt + tl - 1) / tl * cluster; };
  // two targets per thread halve the loads per pair once there is work for it
  // (30000 x 30000: 489 us with one, 440 with two; 3000 x 150k: 262 and 277),
  // and enough targets need fewer CTAs per cluster (four: 440, eight: 469)
  if (a.nt >= 8192 && a.ns >= 8192)
    return launch_p<32, 2>(a, potential, a.nt >= 16384 ? std::min(cluster, 4) : cluster, s);
  // (many targets and few sources: no more CTAs than that; 30000 x 4001: 105 us
  // with clusters of four, 74 without)
  while (cluster > 1 && ctas(32) >= 4 * want) cluster /= 2;
  if (ctas(32) >= want) return launch_p<32, 1>(a, potential, cluster, s);
  if (ctas(16) >= want) return launch_p<16, 1>(a, potential, cluster, s);
  if (ctas(8) >= want) return launch_p<8, 1>(a, potential, cluster, s);
  return launch_p<4, 1>(a, potential, cluster, s);
}

// Whether launch_field_direct is the faster of the two for nt targets and ns
// sources in nseg segments of the field kernel.  Estimates in us from the
// timings above: this kernel 7 + 0.53 per million pairs; the field kernel 12 +
// (8 + 49 k) ns per source of a segment, k = 1024-target CTAs per SM (three
// run at once).
bool field_uses_probe(long long nt, long long ns, long long nseg, int sms) {
  const double pairs = static_cast<double>(nt) * static_cast<double>(ns);
  const double k = static_cast<double>((nt + 1023) / 1024 * nseg) / sms;
  const double at_once = k < 3.0 ? std::ceil(k) : 3.0, rounds = k < 3.0 ? 1.0 : k / 3.0;
  const double split = 12.0 + static_cast<double>(ns) / static_cast<double>(nseg) *
                                  (0.008 + 0.049 * at_once) * rounds;
  return few_sources(nt, ns) || 7.0 + 5.3e-7 * pairs < split;
}

}  // namespace md
