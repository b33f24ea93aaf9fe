// Ticket segments of the persistent batch kernel: the records that the device reads, their
// construction from the scenarios' schedules, and the search for a ticket's segment. Plain
// C++ (no CUDA types), shared by the library, the kernels and a test program.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

#if defined(__CUDACC__)
#define SWE_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SWE_HOST_DEVICE inline
#endif

namespace swe {

// Elements per ticket: one tensor-core tile of the stage phase, one element per lane of
// the TVB phase. A ticket's elements run one tile after the other on one warp and the next
// phase waits for the last of them, so the smallest ticket gives the shortest phase: an
// ensemble of eight scenarios of 5 k to 100 k elements takes 1.34 ms per macro step with
// tickets of 16, 1.35 with 16 to 64 by phase size, 2.21 with 64.
constexpr int kBatchStageTile = 16;
constexpr int kBatchTvbTile = 32;

// One phase of one scenario: tickets [t0, t0 + ntiles). Tickets are counted in 64 bits:
// sixteen scenarios of 200,000 elements and 5,000 macro steps have 6e9 of them.
struct alignas(16) BatchSeg {
  long long t0;
  long long need;   // tiles of this scenario that must be complete first
  int ntiles;
  int scn;          // scenario (index in the group)
  int nactive;      // active elements
  int kind;         // 0: stage kernel, 1: TVB limiter
  int kofs;         // k of this phase minus k at the start of the call
  int first;        // the scenario's first phase in this call: waits for its release
  int prev;         // tiles of the scenario's phase before this one
  int pad;
};
static_assert(sizeof(BatchSeg) == 48, "a segment is three 16-byte words");

// Counters of one scenario, a 128-byte line each (the scenarios' waits poll different lines).
struct alignas(128) BatchCnt {
  unsigned long long done;      // tiles completed (run or skipped)
  unsigned long long skipped;   // tiles skipped
  int status;                   // 0, or SWE_ETIMEOUT when a wait gave up
};
static_assert(sizeof(BatchCnt) == 128, "a line per scenario");

struct BatchCtl {   // per group, in the batch workspace
  unsigned long long head;   // next ticket
  unsigned long long total;  // tickets of this call
  long long wait_ns;         // bound of every wait
  int nseg;                  // segments of this call
  int pad;
};

// A scenario's schedule as the tables need it.
struct BatchSchedule {
  int kinds = 1;              // phases per finest substep: the stage, then (2) the TVB limiter
  std::vector<int> nactive;   // active elements of each finest substep of a macro step
};

inline int batch_tiles(int nactive, int kind) {   // tickets of one phase
  const int t = kind == 0 ? kBatchStageTile : kBatchTvbTile;
  return nactive / t + (nactive % t != 0);
}

// Segments of `macro` macro steps of a scenario.
inline int64_t batch_segment_count(const BatchSchedule& s, int64_t macro) {
  return macro * (int64_t)s.nactive.size() * s.kinds;
}

// Segments of one call: the phases of every scenario (per macro step and finest substep:
// the stage kernel, then the TVB limiter), ordered phase by phase, round-robin over the
// scenarios, each after the tickets of its scenario's earlier phases.
inline void batch_segments(const std::vector<BatchSchedule>& scn, const std::vector<int32_t>& nmacro,
                           std::vector<BatchSeg>& out) {
  out.clear();
  const size_t n = scn.size();
  std::vector<int64_t> nph(n), need(n, 0);
  std::vector<int> prev(n, 0);
  int64_t maxp = 0, total = 0, t0 = 0;
  for (size_t a = 0; a < n; ++a) {
    nph[a] = batch_segment_count(scn[a], nmacro[a]);
    maxp = std::max(maxp, nph[a]);
    total += nph[a];
  }
  out.reserve((size_t)total);
  for (int64_t ph = 0; ph < maxp; ++ph)
    for (size_t a = 0; a < n; ++a) {
      if (ph >= nph[a]) continue;
      const BatchSchedule& s = scn[a];
      const int64_t step = ph / s.kinds;   // substeps since the start of the call
      BatchSeg sg = {};
      sg.t0 = t0;
      sg.need = need[a];
      sg.nactive = s.nactive[(size_t)(step % (int64_t)s.nactive.size())];
      sg.kind = (int)(ph % s.kinds);
      sg.ntiles = batch_tiles(sg.nactive, sg.kind);
      sg.prev = prev[a];
      sg.scn = (int)a;
      sg.kofs = (int)step;
      sg.first = ph == 0 ? 1 : 0;
      prev[a] = sg.ntiles;
      need[a] += sg.ntiles;
      t0 += sg.ntiles;
      out.push_back(sg);
    }
}

// The segment of a ticket: the last one whose t0 is at most the ticket (segments without
// tickets share their successor's t0). lo: a segment known to start at or before it (a
// warp's tickets only grow, so its previous segment); the ticket is below the total.
// probe(base, stride) counts, over i < 32, the segments base + i stride below nseg that
// start at or before the ticket. The 32 segments after lo are looked at first, then the
// rest is narrowed 32-fold per probe. A table with one int per ticket costs 4 bytes per
// ticket on the device, on the host and in the upload (24 GB for the schedule at BatchSeg)
// and two loads per ticket where most tickets stay in the segment at hand: the ensemble of
// eight at kBatchStageTile, 8 macro steps with transfers, 13.49 ms with it, 12.24 without.
template <typename Probe>
SWE_HOST_DEVICE int batch_find(unsigned lo, unsigned nseg, Probe&& probe) {
  unsigned c = probe(lo + 1u, 1u);
  lo += c;
  if (c < 32u) return (int)lo;
  for (unsigned hi = nseg; hi - lo > 1u;) {
    const unsigned stride = (hi - lo + 31u) / 32u;
    c = probe(lo + stride, stride);
    lo += c * stride;
    hi = hi - lo > stride ? lo + stride : hi;
  }
  return (int)lo;
}

}  // namespace swe
