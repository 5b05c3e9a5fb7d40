"""csrc/inflight.h on the host: the copy waits of the training kernels under every pattern of waits
that give up. The fake barriers complete their copies late and in order; what is checked is
what the hardware asks for: at most one copy in flight per barrier, none issued after a wait of the issuing
thread gave up, and none in flight at the end."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "inflight.h"

static void must(bool ok, const char *what) { if (!ok) { std::printf("FAILED %s\n", what); std::exit(1); } }

template <unsigned B>
struct Bars {
    std::vector<int> left;        // polls until copy u completes (in issue order)
    unsigned done = 0;            // copies complete
    int limit = 1 + std::rand() % 40;   // polls of the waits until one gives up; enough after that
    bool gave_up = false;
    unsigned phase(unsigned b) const { return done / B + (done % B > b); }   // phases complete
    void issue(unsigned b)
    {
        must(!gave_up, "issued after a wait gave up");
        must(b == left.size() % B, "barriers in turn");
        must(left.size() - done < B, "one copy in flight per barrier");
        left.push_back(std::rand() % 12);
    }
    void poll() { if (done < left.size() && left[done]-- <= 0) ++done; }
    bool wait(unsigned b, unsigned parity)
    {
        for (int i = 0; i < (gave_up ? 1000 : limit); ++i) {
            if ((phase(b) & 1u) != parity) return true;   // the phase of that parity is complete
            poll();
        }
        must(!gave_up, "waited for a phase that does not come");
        gave_up = true;
        return false;
    }
    auto bounded() { return [this](unsigned b, unsigned parity) { return wait(b, parity); }; }
};

int main()
{
    for (int trial = 0; trial < 200000; ++trial) {
        std::srand(trial);
        {   // a tile's copy requested while the last one is worked on
            Bars<1> bars;
            unsigned issued = 1;
            bool good = true;
            bars.issue(0);
            for (unsigned tile = 0; tile < 6 && good; ++tile) {
                good = bars.wait(0, tile & 1u);
                if (good && tile + 1 < 6) { bars.issue(0); ++issued; }
            }
            if (!good) cva::settle_copies<1>(issued, bars.bounded());
            must(good == !bars.gave_up, "status");
            must(bars.done == bars.left.size(), "a copy in flight at the end");
        }
        const unsigned K = 1 + std::rand() % 9;
        {   // input copies two tiles ahead in two buffers
            Bars<2> bars;
            bool good = true;
            auto stage = [&](unsigned i) {
                if (good && !bars.wait(i & 1u, (i >> 1) & 1u)) {
                    good = false;
                    cva::settle_copies<2>(K < i + 2 ? K : i + 2, bars.bounded());
                }
            };
            for (unsigned i = 0; i < K && i < 2; ++i) bars.issue(i & 1u);
            stage(0);
            for (unsigned i = 0; i < K; ++i) {
                if (i + 2 < K && good) bars.issue(i & 1u);
                if (i + 1 < K) stage(i + 1);
            }
            must(bars.done == bars.left.size(), "copies in flight at the end");
        }
    }
    std::printf("ok\n");
}
"""


def test_no_copy_outlives_a_wait_that_gave_up(tmp_path):
    src = tmp_path / "inflight.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "inflight"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2211_17005_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
