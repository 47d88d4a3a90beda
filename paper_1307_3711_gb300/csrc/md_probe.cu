// md_probe.cu -- field and potential at caller-given targets in one launch and
// without scratch memory.
//
// The field kernel of md_device.cuh gives a CTA 1024 targets and adds partial
// fields through memory: at a few hundred targets most of its lanes hold none.
// Here a cluster of CTAs takes kTargets targets; its CTAs share the sources,
// the warps of a CTA share its part (every TL lanes another source of the
// staged tile), the warps' sums are joined as compensated FP32 pairs through
// shared memory, and the CTAs' are added in FP64 by the cluster's first CTA, which
// receives them through distributed shared memory.
//
// A tile is released warp by warp instead of by a CTA-wide barrier and a full
// tile's loop has a fixed length (3 to 4 % of a large field); FP32 pairs, for an
// FP64 instruction takes its pipe 16 cycles (every slice in FP64: 2 us more per call).  Up to four targets per SM the sources' tiles
// are what a CTA waits for: tiles of 4096, two stages, one CTA per SM and small
// clusters, which the SMs hold evenly (300 x 150k: 49 us with tiles of 1024 and
// clusters of eight, 29 so).
//
// Measured (us, field without the potential; in brackets the field kernel with
// its partials in memory, and the allocation-free kernel of 256-target blocks
// that this one replaced): 300 targets x 150k sources 29 (185, 657), 1000 x
// 4001 10.5 (237, 146), 1 x 150k 10.4 (171, 655), 1000 x 1M 559 (948, 4320), 3000
// x 1M 1610 (1756, 4325), 10000 x 150k 711 (675, 1012).  One target per thread
// reads a source from shared memory per pair, so where the field kernel's
// blocks fill the SMs it stays faster (field_uses_probe).
#include <algorithm>
#include <utility>

#include <cooperative_groups.h>

#include "md_device.cuh"
#include "md_internal.h"

namespace md {

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCluster = 8;
constexpr int kLargeTile = 4096;  // (two stages of it leave room for one CTA per SM)

template <int TL, int R, bool POT, int kTile, int kStages>
struct ProbeSmem {
  Stage<kTile, kStages> st;
  float2 e[POT ? 4 : 3][kWarps][TL * R];              // the warps' sums (value x - y)
  double part[kMaxCluster][POT ? 4 : 3][TL * R];      // first CTA: the CTAs' sums
  uint64_t empty[kStages];
  int abort;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// CTA (x, rank) of cluster x: targets [x kTargets, ...), sources [rank seg, ...).
template <int TL, int R, bool POT, int kTile, int kStages>
__global__ void __launch_bounds__(kThreads) k_probe(const FieldArgs a, long long seg) {
  constexpr int kTargets = TL * R;
  constexpr int kSlices = kThreads / TL;
  constexpr int C = POT ? 4 : 3;
  __shared__ ProbeSmem<TL, R, POT, kTile, kStages> S;
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
  // (checked build: sources outside the array are left out)
  const int ntiles = ns > 0 && MD_IN_RANGE(a.err, j0 + ns, 1, a.ns + 1)
                         ? static_cast<int>((ns + kTile - 1) / kTile)
                         : 0;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&S.st.full[s], 1);
      mbar_init(&S.empty[s], kWarps);
    }
    fence_mbar_init();
    S.abort = 0;
    for (int t = 0; t < kStages && t < ntiles; ++t)
      issue_tile<kTile, kStages>(S.st, static_cast<unsigned>(t), src, ns, t);
  }
  const int tl = tid % TL, slice = tid / TL, lane = tid & 31;
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
  // (a thread meets kTile / kSlices sources of a tile: several tiles to a fold)
  constexpr int kFold = 64 * kSlices > kTile ? 64 * kSlices / kTile : 1;
  auto stop = [&] {
    atomicOr(a.err, kErrTimeout);
    *reinterpret_cast<volatile int*>(&S.abort) = 1;
  };
  int issued = kStages < ntiles ? kStages : ntiles;  // (thread 0)
  for (int t = 0; t < ntiles; ++t) {
    const int s = t % kStages;
    // the first thread refills the stage of the tile before this one once every
    // warp has read it: the warps run up to a tile apart
    if (tid == 0 && t > 0 && issued < ntiles) {
      if (mbar_wait(&S.empty[(t - 1) % kStages], ((t - 1) / kStages) & 1u)) {
        issue_tile<kTile, kStages>(S.st, static_cast<unsigned>(issued), src, ns, issued);
        ++issued;
      } else {
        stop();
      }
    }
    // (the lanes of a warp decide alike)
    if (!__all_sync(0xffffffffu, mbar_try_wait(&S.st.full[s], (t / kStages) & 1u))) {
      const bool go = *reinterpret_cast<volatile int*>(&S.abort) == 0 &&
                      mbar_wait(&S.st.full[s], (t / kStages) & 1u);
      if (!__all_sync(0xffffffffu, go)) {
        stop();
        break;
      }
    }
    const long long rem = ns - static_cast<long long>(t) * kTile;
    const uint32_t tile = smem_u32(&S.st.tile[s][0]) + 16u * slice;
    auto eight = [&](uint32_t from) {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        pair<R, POT>(lds_f4(from + 16u * (q * kSlices)), xi, yi, zi, a.eps2, acc);
      if constexpr (POT) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          kahan_add(acc.sp[r], acc.cp[r], acc.ap[r]);
          acc.ap[r] = 0.0f;
        }
      }
    };
    if (rem >= kTile) {
      constexpr int kEach = kTile / kSlices;  // a full tile's sources per thread
      static_assert(kEach % 8 == 0, "eights");
#pragma unroll(kEach <= 32 ? kEach / 8 : 2)
      for (int k = 0; k < kEach; k += 8) eight(tile + 16u * (k * kSlices));
    } else {
      const int cnt = static_cast<int>(rem);
      int k = slice;
      for (; k + 7 * kSlices < cnt; k += 8 * kSlices) eight(tile + 16u * (k - slice));
      for (; k < cnt; k += kSlices)
        pair<R, POT>(lds_f4(tile + 16u * (k - slice)), xi, yi, zi, a.eps2, acc);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.empty[s]);
    if ((t + 1) % kFold == 0) fold<R, POT>(acc);
  }
  fold<R, POT>(acc);
  // (an expired wait: no further copies, those in flight are awaited)
  if (tid == 0 && S.abort)
    for (int q = issued > kStages ? issued - kStages : 0; q < issued; ++q)
      mbar_wait(&S.st.full[q % kStages], (q / kStages) & 1u);
  auto put = [&](int c, int r, float v, float w) {
#pragma unroll
    for (int d = TL; d < 32; d <<= 1)
      join_sums(v, w, __shfl_xor_sync(0xffffffffu, v, d), __shfl_xor_sync(0xffffffffu, w, d));
    if (lane < TL) S.e[c][tid >> 5][tl + r * TL] = make_float2(v, w);
  };
#pragma unroll
  for (int r = 0; r < R; ++r) {
    put(0, r, acc.sx[r], acc.cx[r]);
    put(1, r, acc.sy[r], acc.cy[r]);
    put(2, r, acc.sz[r], acc.cz[r]);
    if constexpr (POT) put(3, r, acc.sp[r], acc.cp[r]);
  }
  __syncthreads();
  cluster.barrier_wait(std::move(started));
  // each value's warps: eight neighbouring lanes add two each, then each other's
  constexpr int kVals = C * kTargets;
  double* to = &cluster.map_shared_rank(&S.part[0][0][0], 0)[rank * kVals];
  for (int v0 = 0; v0 < kVals; v0 += kThreads / 8) {
    const int v = v0 + tid / 8, c = v / kTargets, t = v % kTargets;
    float2 s = make_float2(0.0f, 0.0f);
    if (v < kVals) {
      s = S.e[c][tid % 8][t];
      const float2 o = S.e[c][tid % 8 + 8][t];
      join_sums(s.x, s.y, o.x, o.y);
    }
#pragma unroll
    for (int d = 4; d > 0; d >>= 1)
      join_sums(s.x, s.y, __shfl_xor_sync(0xffffffffu, s.x, d), __shfl_xor_sync(0xffffffffu, s.y, d));
    if (v < kVals && tid % 8 == 0) {
      const double val = static_cast<double>(s.x) - s.y;
      to[v] = c < 3 ? -val : val;
    }
  }
  cluster.sync();
  if (rank != 0 || tid >= kTargets) return;
  const long long i = i0 + tid;
  if (i >= a.nt || !MD_IN_RANGE(a.err, i, 0, a.nt)) return;
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

template <int TL, int R, bool POT, int TILE, int STAGES>
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
  return cudaLaunchKernelEx(&cfg, k_probe<TL, R, POT, TILE, STAGES>, a, seg);
}

template <int TL, int R, int TILE = 1024, int STAGES = 3>
cudaError_t launch_p(const FieldArgs& a, bool potential, int cluster, cudaStream_t s) {
  return potential ? launch_t<TL, R, true, TILE, STAGES>(a, cluster, s)
                   : launch_t<TL, R, false, TILE, STAGES>(a, cluster, s);
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

// With few sources for many targets a cluster per few targets costs more than it
// sums: k_few takes 4.5 us + 35 ns per source (the mean of with and without the
// potential), k_probe 6.2 us + a third of a ns per target.  30000 targets x 100
// sources 8.4 and 17 us, 10000 x 100 8.4 and 10.4, 3000 x 100 8.4 and 6.6.
bool few_sources(long long nt, long long ns) { return ns < 512 && 105 * ns < 5100 + nt; }

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
  // up to four targets per SM and many sources: one CTA per SM with large tiles,
  // the fewest targets per CTA that its cluster size lets run at once (clusters of
  // two fill every SM, of four all but four SMs, of eight nine in ten)
  if (a.ns >= 12000) {
    const long long c8 = sms / 9, c4 = sms / 4 - 1, c2 = sms / 2;
    if (a.nt <= 2 * c8) return launch_p<2, 1, kLargeTile, 2>(a, potential, 8, s);
    if (a.nt <= 2 * c4) return launch_p<2, 1, kLargeTile, 2>(a, potential, 4, s);
    if (a.nt <= 4 * c4) return launch_p<4, 1, kLargeTile, 2>(a, potential, 4, s);
    if (a.nt <= 4 * c2) return launch_p<4, 1, kLargeTile, 2>(a, potential, 2, s);
    // (400 x 150k: 53 us, 47 with the smaller tiles below; 400 x 30k: 14.7 and 16.7)
    if (a.nt > (a.ns < 60000 ? 4 : 6) * c2 && a.nt <= 8 * c2)
      return launch_p<8, 1, kLargeTile, 2>(a, potential, 2, s);
  }
  // as many CTAs per cluster as leave each a stage of sources; then the most
  // targets per CTA that still give five CTAs to three SMs (fewer targets: the
  // sources are staged more often; fewer CTAs: idle SMs)
  int cluster = 1;
  while (cluster < kMaxCluster && a.ns / (2 * cluster) >= 1000) cluster *= 2;
  const long long want = 5LL * sms / 3;
  auto ctas = [&](long long tl) { return (a.nt + tl - 1) / tl * cluster; };
  // two targets per thread halve the loads per pair once there is work for it
  // (30000 x 30000: 440 us with one, 421 with two; 10000 x 150k: 750 and 711), with
  // the cluster size that loads the busiest SM least: it holds L of the CTAs, each
  // 1.6 us and 4.3 ns per source of its part, the fewer the less they hide of each
  // other's waits (us with clusters of one, two, four and eight: 8192 x 30000 133,
  // 134, 138, 140; 10000 x 30000 257, 196, 166, 158; 14000 x 17000 150, 116, 119, 140;
  // 20000 x 80000 998, 835, 758, 771; 30000 x 89000 1289 with two, 1207 with four;
  // 28000 x 16000 209, 210, 219, 247; with the potential 8192 x 200k 1012, 955, 964, 936)
  if (a.nt >= 8192 && a.ns >= 8192) {
    const long long groups = (a.nt + 63) / 64;
    int best = 1;
    double least = 0.0;
    for (int c = 1; c <= cluster; c *= 2) {
      // (clusters of four leave four SMs empty, of eight a dozen, whose CTAs are
      // many and even out)
      const long long on = c == 4 ? sms - 4 : sms;
      const double L = c == 8 ? 8.0 * groups / (sms - 12) + 0.4
                              : static_cast<double>((groups * c + on - 1) / on);
      const double t = (L + 0.08) * (1.6 + 0.0043 * static_cast<double>(a.ns) / c);
      if (c == 1 || t < least) {
        least = t;
        best = c;
      }
    }
    return launch_p<32, 2>(a, potential, best, s);
  }
  // (many targets and few sources: no more CTAs than that; 30000 x 4001: 105 us
  // with clusters of four, 74 without)
  while (cluster > 1 && ctas(32) >= 4 * want) cluster /= 2;
  if (ctas(32) >= want) return launch_p<32, 1>(a, potential, cluster, s);
  if (ctas(16) >= want) return launch_p<16, 1>(a, potential, cluster, s);
  if (ctas(8) >= want) return launch_p<8, 1>(a, potential, cluster, s);
  return launch_p<4, 1>(a, potential, cluster, s);
}

// Whether launch_field_direct is the faster of the two for nt targets and ns
// sources in nseg segments of the field kernel; the same with and without the
// potential, so that the field has the same bits.  Estimates in us from the
// timings above: this kernel 7 + 0.53 per million pairs, with few sources per
// target 7 + 0.25 ns per target + 0.4 per million pairs (the clusters' start and
// join); k_few 4.5 + 35 ns per source or 8 + 16.3 for each of the busiest SM's CTAs;
// the field kernel 10.5 + (3.5 + 56.2 k) ns per source of a segment, k = 1024-target
// CTAs per SM (three run at once).  Either side of the lines, us, field kernel and this
// one: 100000 x 520 41 and 49, x 1300 88 and 84, 200000 x 800 103 and 117, 50000 x 600
// 45 and 34; field kernel and k_few 300000 x 510 68 and 74, 527000 x 307 81 and 77.
bool field_uses_probe(long long nt, long long ns, long long nseg, int sms) {
  const double t = static_cast<double>(nt), n = static_cast<double>(ns), pairs = t * n;
  const long long k = ((nt + 1023) / 1024 * nseg + sms - 1) / sms;
  const double each = 0.172 * (k / 3) + (k % 3 ? 0.0035 + 0.0562 * (k % 3) : 0.0);
  const double split = 10.5 + each * n / static_cast<double>(nseg);
  if (few_sources(nt, ns)) {
    const double L = static_cast<double>(((nt + 255) / 256 + sms - 1) / sms);
    return 4.5 + std::max(0.035, 0.008 + 0.0163 * L) * n < split;
  }
  return 7.0 + std::max(5.3e-7 * pairs, 2.5e-4 * t + 4.0e-7 * pairs) < split;
}

}  // namespace md
