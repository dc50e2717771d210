"""Loads in flight when a CTA pair gives up (csrc/rid_pair_loads.cuh), on CPU.  A
model of the pair's weight stream is stopped at a random point: loads land in any
order, either producer may be ahead of the other, either may have stopped alone.
The even CTA then settles each stage as the kernel does.  No stage's wait may end
before every load issued into it has landed, and each must end once they have."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "rid_pair_loads.cuh"
struct Bar {                                    // an mbarrier of one arrival and a byte count
    int pending = 1, phase = 0;
    long tx = 0;
    void check() { if (pending == 0 && tx == 0) { pending = 1; ++phase; } }
    void arrive_tx(long b) { tx += b; --pending; check(); }
    void complete(long b) { tx -= b; check(); }
    bool past(int parity) const { return (phase & 1) != parity; }
};
struct Load { int it, cta; long bytes; };
int main() {
    std::mt19937 rng(5);
    auto rnd = [&](int n) { return (int)(rng() % n); };
    long early = 0, never = 0, ahead[2] = {0, 0}, stops = 0;
    for (int trial = 0; trial < 20000; ++trial) {
        const int ns = 2 + rnd(5), total = 1 + rnd(30);
        std::vector<long> part[2];
        for (int i = 0; i < total; ++i) { part[0].push_back(128 * (1 + rnd(4))); part[1].push_back(128 * (1 + rnd(4))); }
        std::vector<Bar> full(ns);
        std::vector<Load> fly;
        int issued[2] = {0, 0}, used = 0;
        bool stopped[2] = {false, false};
        auto land = [&](int k) {
            const Load l = fly[k];
            fly.erase(fly.begin() + k);
            full[l.it % ns].complete(l.bytes);
        };
        const int events = rnd(6 * total + 1);
        for (int e = 0; e < events; ++e) {
            const int what = rnd(4);
            if (what < 2) {
                if (rnd(40) == 0) stopped[what] = true;               // this CTA's producer gives up
                int& it = issued[what];
                if (stopped[what] || it >= total || it >= used + ns) continue;
                if (what == 0) full[it % ns].arrive_tx(part[0][it] + part[1][it]);
                fly.push_back({it, what, part[what][it]});
                ++it;
            } else if (what == 2) {
                if (!fly.empty()) land(rnd((int)fly.size()));
            } else if (used < total && full[used % ns].phase > used / ns) {
                ++used;                                               // the MMAs have read it
            }
        }
        ++stops;
        ahead[0] += issued[0] > issued[1];
        ahead[1] += issued[1] > issued[0];
        std::vector<PairStageLoads> q(ns);
        for (int s = 0; s < ns; ++s) {
            q[s] = pair_stage_loads(issued[0], issued[1], ns, s);
            if (q[s].it < 0 || q[s].even == q[s].odd) continue;
            if (q[s].even) full[s].complete(part[1][q[s].it]);
            else full[s].arrive_tx(part[1][q[s].it]);
        }
        for (;;) {
            for (int s = 0; s < ns; ++s) {
                bool waiting = false;
                for (const Load& l : fly) waiting |= l.it % ns == s;
                const bool done = q[s].it < 0 || full[s].past((q[s].it / ns) & 1);
                early += done && waiting;
                never += !done && !waiting;
            }
            if (fly.empty()) break;
            land(rnd((int)fly.size()));
        }
    }
    std::printf("%ld %ld %ld %ld %ld\n", early, never, ahead[0], ahead[1], stops);
    return 0;
}
"""


def test_every_load_lands_before_a_pair_leaves(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "loads.cpp", tmp_path / "loads"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2408_14070_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    early, never, even_ahead, odd_ahead, stops = map(int, out.split())
    assert even_ahead > stops // 10 and odd_ahead > stops // 10      # the model reaches both
    assert early == 0 and never == 0
