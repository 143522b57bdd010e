"""Give-up path of the kernels on pairs of CTAs, on the CPU: after any history of two producers that stop at different loads,
every copy in flight has landed once the leader has waited for what `open_loads` names (csrc/drain.cuh)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# A barrier as the hardware keeps it: one arrival (the leader's, which also announces bytes) and a byte balance per phase.  The
# producers run ahead of one another as far as the consumer's frees let them, copies land in any order.
MODEL = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "drain.cuh"
struct Bar {
    int phase = 0, pending = 1, bytes = 0;
    void settle() { if (pending == 0 && bytes == 0) { ++phase; pending = 1; } }
    void arrive_expect(int n) { bytes += n; --pending; settle(); }
    void complete(int n) { bytes -= n; settle(); }
};
int main() {
    std::mt19937 rng(1);
    auto upto = [&](int n) { return (int)(rng() % (unsigned)n); };
    const int half = 16;
    long opened = 0, uneven = 0;
    for (int trial = 0; trial < 200000; ++trial) {
        const int streams = 1 + upto(3), stages = 1 + upto(4), slots = streams * stages, total = upto(6 * slots);
        std::vector<Bar> bar(slots);
        std::vector<int> flight;                        // barrier of each copy under way
        int issued[2] = {0, 0}, freed = 0;              // loads begun by each CTA, loads whose slot is free again
        auto index = [&](uint32_t m) { return libra::stream_barrier(m, streams, stages); };
        const int steps = upto(6 * slots + 8);
        for (int s = 0; s < steps; ++s) {
            const int what = upto(4);
            if (what < 2) {
                const int m = issued[what];
                if (m >= total || m >= freed + slots) continue;
                if (what == 0) bar[index(m)].arrive_expect(2 * half);
                flight.push_back(index(m));
                ++issued[what];
            } else if (what == 2 && !flight.empty()) {
                const int x = upto((int)flight.size()), b = flight[x];
                flight.erase(flight.begin() + x);
                bar[b].complete(half);
            } else if (freed < issued[0] && bar[index(freed)].phase > freed / slots) {
                ++freed;                                // the consumer waits for a load's phase, then frees its slot
            }
        }
        uneven += issued[0] != issued[1];
        bool failed = false;
        libra::open_loads(issued[0], issued[1], slots, index, [&](uint32_t b, uint32_t parity, bool leader, bool peer) {
            ++opened;
            if (!leader) bar[b].arrive_expect(half);
            if (!peer) bar[b].complete(half);
            while ((bar[b].phase & 1) == (int)parity) {   // the phase of that parity is still open
                size_t x = 0;
                while (x < flight.size() && flight[x] != (int)b) ++x;
                if (x == flight.size()) { failed = true; return; }   // it would never end
                flight.erase(flight.begin() + x);
                bar[b].complete(half);
            }
        });
        if (failed || !flight.empty()) {
            std::printf("trial %d: %d / %d loads, %zu copies left, stuck %d\n", trial, issued[0], issued[1], flight.size(), failed);
            return 1;
        }
    }
    std::printf("%ld %ld\n", opened, uneven);
    return opened > 100000 && uneven > 10000 ? 0 : 2;
}
"""


def test_every_copy_in_flight_is_waited_for(tmp_path):
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(MODEL)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-x", "c++", "-I",
                           os.path.join(ROOT, "paper_2607_23250_b200", "csrc"), str(src), "-o", str(exe)])
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
