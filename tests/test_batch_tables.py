"""Ticket segments of the persistent batch kernel (csrc/batch_tables.hpp), compiled into a
small host program: tickets counted in 64 bits over long schedules, and the segment of a
ticket found by the kernel's search as by a plain scan.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1403_1661_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "batch_tables.hpp"
using namespace swe;
#define CHECK(x) do { if (!(x)) { std::printf("failed at line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)

// the kernel's search on the host: a probe counts over the 32 lanes
int find(const std::vector<BatchSeg>& s, int64_t ticket, int lo) {
  return batch_find((unsigned)lo, (unsigned)s.size(), [&](unsigned base, unsigned stride) {
    unsigned c = 0;
    for (unsigned lane = 0; lane < 32; ++lane) {
      const unsigned i = base + lane * stride;
      c += i < s.size() && s[i].t0 <= ticket;
    }
    return c;
  });
}

int main(int argc, char** argv) {
  if (argc > 4) {   // scenarios, elements, macro steps, expected tickets per macro step: 4 levels, both limiters
    const int n = std::atoi(argv[1]), K = std::atoi(argv[2]), macro = std::atoi(argv[3]);
    const int64_t per_macro = std::atoll(argv[4]);
    BatchSchedule s;
    s.kinds = 2;
    s.nactive = {K, K / 8, K / 4, K / 8, K / 2, K / 8, K / 4, K / 8};
    std::vector<BatchSeg> seg;
    batch_segments(std::vector<BatchSchedule>(n, s), std::vector<int32_t>(n, macro), seg);
    CHECK((int64_t)seg.size() == n * batch_segment_count(s, macro));
    int64_t t = 0;
    std::vector<int64_t> done(n, 0);
    for (const BatchSeg& g : seg) {
      CHECK(g.t0 == t && g.need == done[g.scn] && g.first == (done[g.scn] == 0));
      t += g.ntiles;
      done[g.scn] += g.ntiles;
    }
    CHECK(t == per_macro * n * macro);
    for (int64_t x : {(int64_t)0, t / 3, t - 1}) {
      const BatchSeg& g = seg[find(seg, x, 0)];
      CHECK(g.t0 <= x && x < g.t0 + g.ntiles);
    }
    std::printf("ok\n");
    return 0;
  }
  std::mt19937 rng(7);
  auto u = [&](int a, int b) { return std::uniform_int_distribution<int>(a, b)(rng); };
  for (int rep = 0; rep < 300; ++rep) {
    std::vector<BatchSchedule> scn(u(1, 48));
    std::vector<int32_t> nm;
    for (BatchSchedule& s : scn) {
      s.kinds = u(1, 2);
      const int per = 1 << u(0, 3);
      int K = rep % 3 ? u(1, 40) : u(1, 3000);
      for (int j = 0; j < per; ++j) s.nactive.push_back(j == 0 ? K : u(0, K));   // a level may hold no element
      nm.push_back(u(0, 12));
    }
    nm[0] = 1;
    std::vector<BatchSeg> seg;
    batch_segments(scn, nm, seg);
    int64_t last = 0;
    int at = 0;
    for (int q = 0; q < (int)seg.size(); ++q)
      for (int t = 0; t < seg[q].ntiles; ++t) {
        const int64_t ticket = seg[q].t0 + t;
        CHECK(find(seg, ticket, u(0, q)) == q);
        if (ticket - last > u(0, 400)) {   // a warp's tickets, from one to a later one
          at = find(seg, ticket, at);
          CHECK(at == q);
          last = ticket;
        }
      }
  }
  std::printf("ok\n");
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("tables")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ftrapv", "-Wall", "-Werror", f"-I{CSRC}", str(d / "t.cpp"), "-o",
                    str(d / "t")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("n,K,macro", [(16, 200_000, 5000), (8, 1_000_000, 1000), (48, 500_000, 300), (1, 17, 3)])
def test_long_schedules_are_counted_in_64_bits(program, n, K, macro):
    active = [K, K // 8, K // 4, K // 8, K // 2, K // 8, K // 4, K // 8]
    per_macro = sum(-(-a // 16) + -(-a // 32) for a in active)
    r = subprocess.run([program, str(n), str(K), str(macro), str(per_macro)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_search_finds_the_segment_of_every_ticket(program):
    r = subprocess.run([program], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
