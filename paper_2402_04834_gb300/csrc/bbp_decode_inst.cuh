// Instantiation of the decoder kernel for one scalar type.
#pragma once

#include "bbp_fused.cuh"
#include "bbp_kernels.cuh"
#include "bbp_launch.h"

namespace bbp {

template <typename T, int DM = kMaxD>
int smem_bytes_for(const Geo& g, int M, int warps = kWarps) {
  return cta_layout(g, M, kMaxK, warps, (int)sizeof(WarpWS<T, kMaxK, DM>)).total;
}

template <typename T, int DM, int NW, bool CL>
cudaError_t launch_decode_nw(const LaunchArgs& a, int cluster, cudaStream_t st) {
  KArgs<T> k;
  k.geo = a.geo; k.M = a.M; k.D = a.D; k.max_iter = a.max_iter; k.arena_elems = a.arena_elems;
  k.p = a.p; k.eta = a.eta; k.delta0 = a.delta0; k.delta1 = a.delta1; k.cutoff = a.cutoff;
  k.synd = a.synd; k.arena = static_cast<T*>(a.arena);
  k.logp = a.logp; k.delta = a.delta; k.iters = a.iters; k.flags = a.flags;
  k.init_msgs = nullptr; k.final_msgs = nullptr;
  k.n_items = 0; k.slot_elems = 0;
  set_working(k);
  const int smem = smem_bytes_for<T, DM>(a.geo, a.M, NW);
  auto kern = decode_kernel<T, kMaxK, DM, NW, CL>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.B * 4 * cluster));
  cfg.blockDim = dim3(NW * 32);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, k);
}

// Warps per CTA (one message update each) and CTAs per network.  The linear
// algebra is a chain of short dependent steps, and one SM holds 8 warps in FP64
// and 16 in FP32 (the warps' shared memory; 16 in FP64 with DM = 4 by the
// registers), so what a batch leaves idle goes to clusters that share a
// network's half-round (60 updates at d = 11, 12 at d = 5 with k = 3), up to a
// warp per update:
// - FP64: four-warp CTAs, as many per network as are resident together, from
//   three on; eight-warp CTAs where even those leave half the chip idle; else
//   pairs of eight-warp CTAs at any batch size (shorter rounds, a fuller last
//   wave).  Half-rounds of fewer than 16 updates: four-warp CTAs, a warp per
//   update (d = 5, k = 3, 200 syndromes: 3 x 4 warps 54.5 ms, 1 x 8 56.0, 2 x 8
//   67.6).
// - FP32: eight-warp CTAs, as many per network as are resident, at least two.
//   Half-rounds of fewer than 16 updates, whose warps the edge blocks leave
//   idle, and k = 1, where an update is shorter than what a cluster adds to it,
//   are shared only as far as CTAs are resident (d = 5, 150 syndromes: 1 x 4 9.4
//   ms, 3 x 4 11.9; k = 1, d = 9, 76 syndromes: 1 x 8 7.7 ms, 2 x 8 8.8).  A
//   long half-round at k = 1 in a batch that fills the chip with four-warp CTAs
//   takes those (d = 5, 144 updates, 300 syndromes: 1 x 4 7.4 ms, 1 x 8 8.5; d =
//   3, 40 updates: 2.3 and 2.0).
// ms, one CTA per network -> clusters: FP64 d = 11, 1 syndrome 223 -> 40 (8 x 8
// warps; 8 x 4: 49), 5: 223 -> 59 (8 x 4; 8 x 8: 63), 12: 224 -> 84, 24: 225 ->
// 150 (3 x 4; 2 x 8: 180), 48: 348 -> 285, 100: 558 -> 495, 200: 973 -> 927;
// d = 5, k = 3, 1 syndrome 10.1 -> 4.9, 200: 57.9 -> 54.5.  FP32 d = 11:
// 1 syndrome 39 -> 10, 24: 52 -> 36, 100: 147 -> 126, 300: 379 -> 343.
template <typename T, int DM>
cudaError_t launch_decode_dm(const LaunchArgs& a, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int half = (a.M + 1) / 2;   // updates of a half-round
  auto fits = [&](int warps) { return smem_bytes_for<T, DM>(a.geo, a.M, warps) <= kMaxSmemBytes; };
  auto warps_per_sm = [&](int warps) {   // at most 16
    const long long per_sm = kSmemPerSm / (smem_bytes_for<T, DM>(a.geo, a.M, warps) + kSmemReservedPerCta);
    return per_sm * warps < 16 ? per_sm * warps : 16;
  };
  // CTAs per network in one wave.
  auto resident = [&](int warps) { return warps_per_sm(warps) / warps * sms / (4 * a.B); };
  auto cluster = [&](int warps, long long n) {
    const long long cap = (half + warps - 1) / warps;
    n = n < cap ? n : cap;
    return (int)(n < 1 ? 1 : n > kMaxCluster ? kMaxCluster : n);
  };
  const bool small = half < 16;
  bool four = !fits(8) || small;
  int least = 2, most = kMaxCluster;   // CTAs per network, before the cap of a warp per update
  if (sizeof(T) == 8) {
    if (!four) four = resident(4) >= 3 && !(64 * a.B <= sms && half > 4 * kMaxCluster);
    if (small) least = kMaxCluster;
  } else if (small) {
    least = 1;
  } else if (a.geo.k == 1 && resident(8) < 2) {
    least = most = 1;
    if (!four) four = half >= 64 && resident(4) < 2 && warps_per_sm(4) >= warps_per_sm(8);
  }
  const int warps = four ? 4 : 8;
  const long long n = resident(warps);
  int cs = cluster(warps, n < least ? least : n > most ? most : n);
  if (4 * a.B * cs > 0x7fffffff) cs = 1;   // grid limit
  if constexpr (sizeof(T) == 4) {
    if (cs == 1) return four ? launch_decode_nw<T, DM, 4, false>(a, 1, st) : launch_decode_nw<T, DM, 8, false>(a, 1, st);
  }
  return four ? launch_decode_nw<T, DM, 4, true>(a, cs, st) : launch_decode_nw<T, DM, 8, true>(a, cs, st);
}

// D <= 4 in FP64 takes an instance of that capacity: 7 KB a warp instead of
// 27, 8 columns over 4 lanes each instead of 16 over 2, so half the FP64
// operations of a step and 16 warps an SM.  d = 5, k = 3, D = 4: 200 syndromes
// 54.4 -> 34.4 ms, 1 syndrome 4.9 -> 3.6; d = 9, 60: 92.9 -> 60.2.  FP32, whose
// rounding a change of summation order would move, keeps the one instance.
template <typename T>
cudaError_t launch_decode_t(const LaunchArgs& a, cudaStream_t st) {
  if constexpr (sizeof(T) == 8) {
    if (a.D <= 4) return launch_decode_dm<T, 4>(a, st);
  }
  return launch_decode_dm<T, kMaxD>(a, st);
}

template <typename T, int K>
int fused_smem_for(const Geo& g, int M, int warps, int cosets, bool gm = (K > 4), int lean = 0) {
  return fused_layout<T, K>(g, M, warps, cosets, gm, lean).total;
}

// Dynamic shared memory of a launch with its messages in workspace slots.  They
// are read through L1, which gets what shared memory leaves, and the runtime
// sets shared memory aside for every CTA that could be resident: with one CTA
// per SM to run, room for a second takes that much from L1, so the request is
// raised until a second would not fit (where two would leave less).  FP32, up to
// 152 CTAs, without -> with: k = 2, 60 syndromes at d = 25 19.6 -> 14.0 ms and at
// d = 13 5.66 -> 4.05 ms; k = 3 at d = 18 7.66 -> 6.11 ms.  With more CTAs than
// SMs a second one pays (d = 25, 150 syndromes 26.0 ms, alone on its SM 27.9).
inline int slot_smem(int smem, long long items, int sms) {
  const int one = kSmemPerSm / 2;
  return items <= sms && smem < one && 2 * (smem + kSmemReservedPerCta) > one ? one : smem;
}

template <typename T>
KArgs<T> fused_args(const LaunchArgs& a) {
  KArgs<T> k;
  k.geo = a.geo; k.M = a.M; k.D = a.D; k.max_iter = a.max_iter; k.arena_elems = 0;
  k.p = a.p; k.eta = a.eta; k.delta0 = a.delta0; k.delta1 = a.delta1; k.cutoff = a.cutoff;
  k.synd = a.synd; k.arena = nullptr;
  k.logp = a.logp; k.delta = a.delta; k.iters = a.iters; k.flags = a.flags;
  k.init_msgs = a.init_msgs; k.final_msgs = a.final_msgs;
  k.n_items = 0; k.slot_elems = 0;
  set_working(k);
  return k;
}

inline cudaError_t sm_count(int* sms) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

// Persistent grid of a launch with its messages in workspace slots:
// resident CTAs, at most one per item and per message slot.
template <typename Kern>
cudaError_t persistent_grid(Kern kern, int threads, int smem, int ctas_per_sm, int sms, long long items,
                            long long slots, long long* grid) {
  cudaError_t e;
  int per_sm = ctas_per_sm;
  if (per_sm <= 0) {
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem)) != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
  }
  long long g = (long long)sms * per_sm;
  if (g > items) g = items;
  if (g > slots) g = slots;
  *grid = g;
  return g > 0 ? cudaSuccess : cudaErrorInvalidValue;
}

// GM: messages in the workspace (a.arena, a.slots slots of G * M * vec
// scalars), a persistent grid; always for k = 5, 6.
template <typename T, int NW, int G, int K, bool GM = (K > 4), int LB = 0>
cudaError_t launch_fused_nw(const LaunchArgs& a, cudaStream_t st) {
  const KArgs<T> k = fused_args<T>(a);
  int smem = fused_smem_for<T, K>(a.geo, a.M, NW, G, GM, LB == 0 ? 0 : (K == 4 && LB >= kEvenLB ? 2 : 1));
  auto kern = fused_kernel<T, NW, G, K, GM, LB>;
  const long long items = a.B * (4 / G);
  int sms = 0;
  cudaError_t e;
  if (GM) {
    if ((e = sm_count(&sms)) != cudaSuccess) return e;
    smem = slot_smem(smem, items, sms);
  }
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
  if (GM) {
    KArgs<T> kp = k;
    kp.arena = static_cast<T*>(a.arena);
    kp.n_items = items;
    kp.slot_elems = (long long)G * a.M * FusedDim<K>::vec;
    long long grid = 0;
    if ((e = persistent_grid(kern, NW * 32, smem, 0, sms, items, a.slots, &grid)) != cudaSuccess) return e;
    kern<<<(unsigned)grid, NW * 32, smem, st>>>(kp);
    return cudaGetLastError();
  }
  kern<<<(unsigned)items, NW * 32, smem, st>>>(k);
  return cudaGetLastError();
}

template <typename T, int NW, int G, int K, bool GM = (K > 4), int LB = 0>
cudaError_t launch_fused_mixed_nw(const LaunchArgs& a, const MixedLaunch& m, cudaStream_t st) {
  const KArgs<T> k = fused_args<T>(a);
  const Geo gmax = make_geo(m.d_max, a.geo.k);
  int Mmax = 0, ae = 0;
  count_messages(gmax, 1, &Mmax, &ae);
  int smem = fused_smem_for<T, K>(gmax, Mmax, NW, G, GM, LB == 0 ? 0 : (K == 4 && LB >= kEvenLB ? 2 : 1));
  auto kern = fused_mixed_kernel<T, NW, G, K, GM, LB>;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  if (GM) smem = slot_smem(smem, a.B * (4 / G), sms);
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
  int per_sm = m.ctas_per_sm;
  if (per_sm <= 0) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NW * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
  }
  MixedArgs mx;
  mx.d_of = m.d_of; mx.offsets = m.offsets; mx.order = m.order; mx.counter = m.counter;
  mx.n_items = a.B * (4 / G); mx.k = a.geo.k;
  mx.B = a.B; mx.d_max = m.d_max;
  long long grid = (long long)sms * per_sm;
  if (grid > mx.n_items) grid = mx.n_items;
  KArgs<T> kp = k;
  if (GM) {      // messages in the workspace, one slot per CTA
    kp.arena = static_cast<T*>(m.slot_base);
    kp.slot_elems = (long long)G * Mmax * FusedDim<K>::vec;
    if (grid > m.slots) grid = m.slots;
    if (grid < 1) return cudaErrorInvalidValue;
  }
  if ((e = cudaMemsetAsync(m.counter, 0, sizeof(unsigned long long), st)) != cudaSuccess) return e;
  kern<<<(unsigned)grid, NW * 32, smem, st>>>(kp, mx);
  return cudaGetLastError();
}

}  // namespace bbp
