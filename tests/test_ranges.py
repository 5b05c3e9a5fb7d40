"""csrc/ranges.h on the host: the path ranges of the adjoint for every path count, limit and failing
allocation."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "ranges.h"

static void must(bool ok, const char *what) { if (!ok) { std::printf("FAILED %s\n", what); std::exit(1); } }

int main()
{
    const uint64_t counts[] = {1, 2, 255, 256, 257, 511, 512, 513, 70001, 131072, 1000003, 0x7fffffffull};
    const size_t limits[] = {0, 1, 1000, 100000, 10u << 20, 1400ull << 20, 1ull << 50};
    for (uint64_t M : counts)
        for (size_t limit : limits)
            for (int fine = 0; fine < 2; ++fine) {
                // fine: a small range is split into more blocks and takes more than its share
                auto bytes = [&](uint64_t m) { return (size_t)m * 40000 + (fine && m < 4096 ? 3000000u : 30000u); };
                auto covers = [&](const cva::RangePlan &p) {
                    must(p.ranges >= 1 && p.per % cva::kRangeBlock == 0, "whole blocks");
                    must((p.ranges - 1) * p.per < M && p.ranges * p.per >= M, "ranges cover the paths");
                    const uint64_t last = M - (p.ranges - 1) * p.per;
                    must(p.bytes >= bytes(last) && (p.ranges == 1 || p.bytes >= bytes(p.per)), "the arrays of every range fit");
                };
                const cva::RangePlan p = cva::plan_ranges(M, limit, bytes);
                covers(p);
                const uint64_t last = M - (p.ranges - 1) * p.per;
                must(bytes(p.per < M ? p.per : M) <= limit || p.per == cva::kRangeBlock, "the limit");
                must(p.bytes == (bytes(last) > bytes(p.per < M ? p.per : M) ? bytes(last) : bytes(p.per < M ? p.per : M)), "size");
                // an allocator with `room` bytes: the first plan it takes fits, and it is asked
                // for narrower ranges until then
                for (size_t room : {(size_t)0, (size_t)5000000, (size_t)13000000, (size_t)(300u << 20), (size_t)1 << 60}) {
                    cva::RangePlan got;
                    uint64_t tried = ~0ull;
                    auto allocate = [&](const cva::RangePlan &q) {
                        covers(q);
                        must(q.per <= tried, "narrower after a failure");
                        tried = q.per;
                        return q.bytes + 8 * q.ranges <= room;
                    };
                    const bool ok = cva::fit_ranges(M, limit, bytes, allocate, &got);
                    if (ok) must(got.bytes + 8 * got.ranges <= room, "taken plan fits");
                    else must(got.per == cva::kRangeBlock, "gives up at one block only");
                }
            }
    std::printf("ok\n");
}
"""


def test_ranges_cover_the_paths_and_fit_what_can_be_allocated(tmp_path):
    src = tmp_path / "ranges.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "ranges"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2211_17005_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
