// Persistent batched launch: many scenarios of one (tier, scheme and order) group
// advanced by one kernel that takes its work from a device ticket queue.
//
// A ticket, taken by one warp, is one tile of elements (kBatchStageTile; the stage kernel: R,
// Adams-Bashforth commit and positivity limiter, Algorithms 1 and 3;
// kBatchTvbTile: the TVB limiter, Section 5.3) of one phase of one scenario, a phase being one
// of those two kernels at one finest substep of the scenario's multirate schedule.
// Tickets are ordered phase by phase, round-robin over the scenarios (the host builds
// the segment table), and a ticket runs only after every tile of its scenario's
// earlier phases has completed, since a neighbour of any element may sit in any tile.
// Every wait is bounded in time: a scenario whose wait gives up is marked
// SWE_ETIMEOUT in its status word and the rest of its tickets are skipped, while the
// other scenarios carry on. The first phase of a scenario also waits for its release
// flag, which the host sets for every scenario it does not hold back.
//
// Memory ordering: a warp that finishes a tile orders its lanes' stores before its
// counter update with a warp barrier followed by a device-scope fence in the lane
// that updates the counter (cumulative over what the barrier ordered, the pattern of
// a grid-wide barrier); a warp that
// waits reads the counter with acquire semantics, then the arrays other CTAs wrote
// with ordinary (coherent) loads, never through the read-only data path.
#pragma once

#include <cstddef>

#include "kernels.cuh"
#include "kernels_tc.cuh"
#include "kernels_team.cuh"

namespace swe {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Lane 0 of the warp: wait until ticket segment S may run. Returns 1 to run the tile, 0 to
// skip it (its scenario failed, or this wait gave up and failed it). A warp may hold a
// ticket several phases ahead, and a thousand warps polling one counter delay the very
// updates they wait for: it sleeps 2 us while more than the phase before its own is
// outstanding, half a microsecond while many tiles of that are, and only then polls fast.
template <typename T>
__device__ __forceinline__ int batch_wait(const BatchLaunch<T>& bl, const BatchSeg& S) {
  BatchCnt* cnt = bl.cnt + S.scn;
  if (ld_acquire(&cnt->status) != 0) return 0;
  const unsigned long long limit = (unsigned long long)__ldcg(&bl.ctl->wait_ns);
  const unsigned long long t0 = global_ns();
  if (S.first) {
    while (ld_acquire(bl.release + S.scn) == 0) {
      if (global_ns() - t0 > limit) {
        atomicCAS(&cnt->status, 0, -5 /* SWE_ETIMEOUT */);
        return 0;
      }
      __nanosleep(256);
    }
  }
  for (long long rem; (rem = S.need - (long long)ld_acquire(&cnt->done)) > 0;) {
    if (ld_acquire(&cnt->status) != 0) return 0;
    if (global_ns() - t0 > limit) {
      atomicCAS(&cnt->status, 0, -5 /* SWE_ETIMEOUT */);
      return 0;
    }
    __nanosleep(rem > S.prev ? 2000 : (rem > 16 ? 500 : 64));
  }
  return 1;
}

// L2 prefetch of the node planes of the state and the bed of elements [e0, e0 + n)
// of a scenario at substep k (the buffer each element reads: the parity of its
// level's activation count), one 128-byte line per lane and plane. Hints only:
// every address lies inside its array.
template <typename T, int N>
__device__ __forceinline__ void batch_prefetch_stage(const StageParams<T>& B, long long k, int e0, int n, int lane) {
  constexpr int NP = Dims<N>::NP;
  const size_t ks = (size_t)B.sc.KS, fstride = (size_t)NP * ks;
  const long long a = k >> (level_of(B.sc, e0) - 1);
  const T* q = B.s.q + (size_t)(a & 1) * 3 * fstride + e0;
  constexpr int per_line = 128 / sizeof(T);
  const int lines = (n + per_line - 1) / per_line;
  for (int w = lane; w < 4 * NP * lines; w += 32) {
    const int pl = w / lines, ln = w - pl * lines;
    const T* base = pl < 3 * NP ? q + (size_t)pl * ks : B.s.B + e0 + (size_t)(pl - 3 * NP) * ks;
    prefetch_l2(base + ln * per_line);
  }
}

__device__ __forceinline__ BatchSeg load_seg(const BatchSeg* p) {
  BatchSeg S;
  const int4* src = reinterpret_cast<const int4*>(p);
  int4* dst = reinterpret_cast<int4*>(&S);
  dst[0] = __ldg(src);
  dst[1] = __ldg(src + 1);
  dst[2] = __ldg(src + 2);
  return S;
}

// kTC: the tensor-core stage body (FP32 tier); otherwise the SIMT body (T = float
// or double). Every warp of the CTA takes tickets on its own (no barrier in the
// loop). It holds its next ticket with that ticket's segment record, fetched before the
// current one runs, and lane 0 waits only when a ticket opens a segment the warp has not
// yet waited for (the tiles a segment needs are the same for all its tickets). The warp
// prefetches the next stage ticket's node planes to L2, as the separate launch does a tile
// ahead.
template <typename T, int N, bool kTC>
__global__ void __launch_bounds__(kTC ? 32 * TcSmem<N>::LIMIT : kBatchTile, 1) k_batch(const __grid_constant__ BatchLaunch<T> bl) {
  static_assert(kBatchStageTile % TcSmem<N>::E == 0 && kBatchStageTile % Team<T, N>::E == 0 && kBatchTvbTile % 32 == 0,
                "whole warp-tiles per ticket");
  static_assert(sizeof(BatchLaunch<T>) <= 32000, "batch launch parameters exceed the kernel-parameter space");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ long long s_k0[kBatchMaxScn];   // finest substep count at the start of the call
  T* sops = reinterpret_cast<T*>(smem_raw);
  // the macro counters move only after the launch (the finish kernel): read once
  for (int i = threadIdx.x; i < bl.nscn; i += blockDim.x)
    s_k0[i] = __ldcg(bl.scn[i].s.macro) * (long long)bl.period[i];
  // every scenario of the group has the same operators: stage the first one's
  // (the staging ends with a CTA barrier, which also publishes s_k0)
  if constexpr (kTC) {
    tc_ops_begin<N>(sops, bl.scn[0].s.ops, bl.scn[0].s.tcops);
    stage_tc_init<N>(sops + TcSmem<N>::CTA + (threadIdx.x >> 5) * TcSmem<N>::WARP);
    team_ops_ready();
  } else {
    team_ops_begin<T, N>(sops, bl.scn[0].s.ops);
    team_ops_ready();
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long total = (long long)__ldcg(&bl.ctl->total);
  const unsigned nseg = (unsigned)__ldcg(&bl.ctl->nseg);
  auto take = [&]() {   // the warp's next ticket
    unsigned long long t = 0;
    if (lane == 0) t = atomicAdd(&bl.ctl->head, 1ull);
    return (long long)__shfl_sync(0xffffffffu, t, 0);
  };
  // the warp's next ticket and its segment, in every lane
  long long ticket = take();
  int sg = 0, ok_sg = -1;
  BatchSeg S = {};
  auto find = [&]() {
    if (ticket < S.t0 + S.ntiles) return;   // still in the segment at hand
    sg = batch_find((unsigned)sg, nseg, [&](unsigned base, unsigned stride) {
      const unsigned i = base + lane * stride;
      return (unsigned)__popc(__ballot_sync(0xffffffffu, i < nseg && __ldg(&bl.segs[i].t0) <= ticket));
    });
    S = load_seg(bl.segs + sg);
  };
  if (ticket < total) find();
  while (ticket < total) {
    // take the held ticket, wait if it opens a segment, and fetch the next
    const int tile = (int)(ticket - S.t0), scn = S.scn, kind = S.kind, nactive = S.nactive, kofs = S.kofs;
    int go = 1;
    if (sg != ok_sg) {
      if (lane == 0) go = batch_wait(bl, S);
      go = __shfl_sync(0xffffffffu, go, 0);
      if (go) ok_sg = sg;
    }
    ticket = take();
    if (ticket < total) find();
    if (go) {
      // the scenario's parameters, in the kernel-parameter space
      const StageParams<T>& wp = bl.scn[scn];
      // the substep count: the scenario's count at the start of the call plus the
      // phase's offset in this call
      const long long k = s_k0[scn] + kofs;
      // the warp's next stage ticket: its planes start moving to L2 now
      if (ticket < total && S.kind == 0) {
        const int e0 = (int)(ticket - S.t0) * kBatchStageTile;
        batch_prefetch_stage<T, N>(bl.scn[S.scn], s_k0[S.scn] + S.kofs, e0, min(kBatchStageTile, S.nactive - e0), lane);
      }
      double injected = 0.0;
      if (kind == 0) {
        if constexpr (kTC) {
          using SM = TcSmem<N>;
          float* sw = sops + SM::CTA + warp * SM::WARP;
          const int t0 = tile * (kBatchStageTile / SM::E);
          const int t1 = min(t0 + kBatchStageTile / SM::E, (nactive + SM::E - 1) / SM::E);
          injected = stage_tc_range<N>(wp, k, nactive, sops, sw, t0, 1, t1, false);
        } else {
          using C = Team<T, N>;
          T* sw = sops + C::OPS + warp * C::WARP;
          const int t0 = tile * (kBatchStageTile / C::E);
          const int t1 = min(t0 + kBatchStageTile / C::E, (nactive + C::E - 1) / C::E);
          injected = team_range<T, N>(wp, sops, sops + C::PRE, sw, t0, 1, t1, nactive, k);
        }
      } else {
        const int e0 = tile * kBatchTvbTile;
        tvb_range<T, N>(wp, 1, sops, e0 + lane, 32, min(e0 + kBatchTvbTile, nactive), k);
      }
      if (injected != 0.0) atomicAdd(wp.s.acc, injected);
    }
    __syncwarp();   // the lanes' stores of the tile are issued and ordered before lane 0's
    if (lane == 0) {
      __threadfence();   // ... which a device-scope fence makes visible before the counter moves
      if (!go) atomicAdd(&bl.cnt[scn].skipped, 1ull);
      atomicAdd(&bl.cnt[scn].done, 1ull);
    }
  }
}

}  // namespace swe
