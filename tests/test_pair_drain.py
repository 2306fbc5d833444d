"""What the leader of a CTA pair owes its load barriers after an abort (PairDrain), run on the host against a model of an mbarrier: wherever
the two producers stopped, each phase ends, and none before the loads under way have landed."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_05699_b200", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "kvq_umma.cuh"
struct Bar {   // an mbarrier of one arrival: a phase ends when the arrival is in and no bytes are owed
    int phase = 0, pending = 1, tx = 0;
    void look() { if (pending == 0 && tx == 0) ++phase, pending = 1; }
    void arrive_expect(int b) { tx += b, --pending; look(); }
    void complete(int b) { tx -= b; look(); }
};
int main()
{
    srand(1);
    for (int it = 0; it < 200000; ++it) {
        const int ring = 2 + rand() % 11, base = rand() % 40;
        int n[2] = {base, base};
        n[rand() & 1] += rand() % (ring + 1);
        std::vector<Bar> bar(ring);
        std::vector<int> flying;   // block of each load that has not landed
        const int top = n[0] > n[1] ? n[0] : n[1];
        // blocks up to top - ring have been used, so both loads of them have landed; of the others some have
        for (int u = 0; u < top; ++u) {
            if (u < n[0]) bar[u % ring].arrive_expect(2);
            for (int c = 0; c < 2; ++c)
                if (u < n[c]) {
                    if (u < top - ring || (rand() & 1)) bar[u % ring].complete(1);
                    else flying.push_back(u);
                }
        }
        const kvq::PairDrain d{n[0], n[1], ring};
        for (int u = d.begin(); u < d.end(); ++u) {
            Bar &b = bar[d.slot(u)];
            if (d.owes_arrival(u)) b.arrive_expect(1);
            if (d.owes_bytes(u)) b.complete(1);
            bool out = false;
            for (int f : flying) out |= f == u;
            if (out && b.phase != u / ring) return printf("ring %d, %d and %d blocks: the phase of block %d ended early\n", ring, n[0], n[1], u), 1;
            for (int f : flying)
                if (f == u) b.complete(1);
            if (b.phase != u / ring + 1 || d.parity(u) != (unsigned)(u / ring) % 2)
                return printf("ring %d, %d and %d blocks: the phase of block %d never ends\n", ring, n[0], n[1], u), 1;
        }
        for (int f : flying)
            if (f < d.begin()) return printf("ring %d, %d and %d blocks: block %d is not waited for\n", ring, n[0], n[1], f), 1;
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_every_load_under_way_is_waited_for(tmp_path):
    src, exe = tmp_path / "drain.cu", tmp_path / "drain"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True, text=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
