"""The staged kernels' ring of shared-memory stages on the CPU (csrc/lks_ring.cuh): a host program takes the consumer
warps' walk from the header and plays the ring with mbarriers modelled by their phase parity, copies that land in
any order and warps that run at any pace.  No wait may return before the phase it stands for is complete, no
arrival may count for another task, every item is taken once, and nothing may be left waiting."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "lks_ring.cuh"

struct Bar {  // an mbarrier: the phase being filled, and what it still waits for
    int count, pending, phase = 0;
    explicit Bar(int n) : count(n), pending(n) {}
    bool done(unsigned parity) const { return (phase & 1u) != parity; }
    void arrive() { if (--pending == 0) ++phase, pending = count; }
};
struct Op { int kind, task, item; };  // 0: wait for the task's copies, 1: arrive on its stage's `empty`, 2: item

// every operation of a consumer warp, from the walk that the kernels use
template <int WARPS>
std::vector<Op> ops_of(int warp, int ntask, int items) {
    std::vector<Op> ops;
    auto skip = [&](uint32_t it) { ops.push_back({0, (int)it, 0}); ops.push_back({1, (int)it, 0}); return true; };
    lks::ItemWalk<WARPS> i(warp);
    for (; i.next(ntask, items, skip); i.c += WARPS) {
        ops.push_back({0, (int)i.it, 0});
        ops.push_back({2, (int)i.it, i.c});
        ops.push_back({1, (int)i.it, 0});
    }
    return ops;
}

template <int WARPS, int STAGES>
const char* play(int items, int ntask, unsigned seed) {
    std::vector<std::vector<Op>> ops;
    for (int w = 0; w < WARPS; ++w) ops.push_back(ops_of<WARPS>(w, ntask, items));
    std::vector<Bar> full(STAGES, Bar(1)), empty(STAGES, Bar(lks::ring_arrivals(items, WARPS)));
    std::vector<size_t> at(WARPS, 0);
    std::vector<int> taken(ntask * items, 0), landing;  // tasks whose copies are in flight
    int issued = 0;
    srand(seed);
    const int lag = seed % 3 == 0 ? -1 : rand() % ntask, slow = rand() % WARPS;  // one late copy, one slow warp
    for (long idle = 0, n = 0; idle < 200000; ++n, ++idle) {
        const int who = rand() % (WARPS + 2);
        if (who == WARPS) {  // the producer
            if (issued == ntask) continue;
            const int s = issued % STAGES, u = issued / STAGES;
            if (u > 0 && !empty[s].done((u - 1) & 1u)) continue;
            if (u > 0 && empty[s].phase != u) return "the producer's wait returned early";
            landing.push_back(issued++);
        } else if (who > WARPS) {  // one of the copies lands
            if (landing.empty()) continue;
            const size_t k = rand() % landing.size();
            if (landing[k] == lag && rand() % 200) { idle = 0; continue; }
            if (full[landing[k] % STAGES].phase != landing[k] / STAGES) return "a stage was filled twice";
            full[landing[k] % STAGES].arrive();
            landing.erase(landing.begin() + k);
        } else {
            if (at[who] == ops[who].size() || (who == slow && rand() % 50)) continue;
            const Op o = ops[who][at[who]];
            const int s = o.task % STAGES, u = o.task / STAGES;
            if (o.kind == 0) {
                if (!full[s].done(u & 1u)) continue;
                if (full[s].phase != u + 1) return "a consumer's wait returned early";
            } else if (o.kind == 1) {
                if (empty[s].phase != u) return "an arrival counted for another task";
                empty[s].arrive();
            } else {
                ++taken[o.task * items + o.item];
            }
            ++at[who];
        }
        idle = 0;
    }
    for (int w = 0; w < WARPS; ++w)
        if (at[w] != ops[w].size()) return "a warp is left waiting";
    for (int n : taken)
        if (n != 1) return "an item was not taken once";
    return issued == ntask && landing.empty() ? nullptr : "a task was not staged";
}

int main(int argc, char** argv) {
    const int warps = atoi(argv[1]), first = atoi(argv[2]), last = atoi(argv[3]);
    for (int items = first; items <= last; ++items)
        for (int ntask : {1, 2, 7, 40})
            for (unsigned seed = 0; seed < 16; ++seed) {
                const char* m = warps == 15 ? play<15, 3>(items, ntask, seed) : play<11, 4>(items, ntask, seed);
                if (m) {
                    printf("%s: %d items, %d tasks, seed %u\n", m, items, ntask, seed);
                    return 1;
                }
            }
    return 0;
}
"""


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    (d / "ring.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2112_13930_gb300", "csrc"),
                    str(d / "ring.cpp"), "-o", str(d / "ring")], check=True)
    return str(d / "ring")


# 2D: 15 consumer warps, three stages, rows of 1024 nodes and more have 9 to 16 items a task; 3D: 11 consumer warps,
# four stages, 8 items a task
@pytest.mark.parametrize("warps,first,last", [(15, 1, 17), (11, 8, 8)])
def test_every_wait_of_the_ring_is_exact(ring, warps, first, last):
    r = subprocess.run([ring, str(warps), str(first), str(last)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
