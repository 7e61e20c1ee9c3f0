"""The rules of the TTI passes' plane rings (csrc/plane_ring.cuh) on the host, against a model of
an mbarrier (arrivals, pending bytes, phases; a wait by parity returns at once when the phase of
that parity is over): a march without incident, readers that never leave a slot, and a copy that
lands only after the wait for it has given up.  Whatever happens, no arrival may reach a phase
whose arrivals are complete, no copy may start into a slot that was not seen empty, a wait that
gives up must raise the error flag, and no copy may be in flight once the block has drained."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2201_06914_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "plane_ring.cuh"

struct Bar {
    int pending = 1, phase = 0, late = -1;   // late: phase whose bytes land one wait too late
    int tx = 0;
    bool bad = false;
    void arrive_expect() { if (pending == 0) bad = true; pending--; tx++; step(); }
    void land() { tx--; step(); }
    void step() { if (pending == 0 && tx == 0) { phase++; pending = 1; } }
    bool over(unsigned parity) const { return (unsigned)(phase & 1) != parity; }
};

// NS slots, LA ahead, n planes.  stuck: plane the readers never leave (-1: none); late: plane whose
// copy lands only at the second wait for it (-1: none).
template <int NS, int LA, bool EMPTY>
static int march(int n, int stuck, int late)
{
    Bar full[NS];
    wp::PlaneRing<NS, LA> r;
    int raised = 0, gave_up = 0, seen_late = 0, torn = 0, count[NS] = {0};
    auto issue = [&](int i) {
        const int s = i % NS;
        if (stuck >= 0 && i > stuck && s == stuck % NS) torn = 1;
        full[s].arrive_expect();
        count[s]++;
        if (i == late) full[s].late = i / NS;
        else full[s].land();
    };
    auto wait = [&](int s, unsigned parity) {
        if (full[s].over(parity)) return true;
        if (full[s].late == full[s].phase && seen_late++ > 0) { full[s].late = -1; full[s].land(); return true; }
        gave_up = 1;
        return false;
    };
    auto raise = [&] { raised = 1; };
    for (int g = 0; g < LA && g < n; g++) issue(g);
    for (int i = 0; i < n; i++) {
        r.refill(i, n, [&] {
            if (!EMPTY || stuck < 0 || (i + LA) % NS != stuck % NS || i + LA <= stuck) return true;
            gave_up = 1;
            return false;
        }, raise, [&] { issue(i + LA); });
        r.await(i, n, [&] { return wait(i % NS, (unsigned)(i / NS) & 1); }, raise);
    }
    int in_flight = 0, total = 0;
    if (raised) r.drain(n, [&](int s, unsigned p) { return wait(s, p); });
    for (int s = 0; s < NS; s++) { in_flight += full[s].tx != 0; total += count[s]; if (full[s].bad) return 1; }
    if (torn) return 2;
    if (raised != gave_up) return 3;
    if (in_flight) return 4;
    if (stuck < 0 && late < 0 && (raised || total != n)) return 5;
    if ((late >= 0 && !raised)) return 6;
    return 0;
}

int main()
{
    int fails = 0;
    auto check = [&](const char *w, int n, int k, int rc) {
        if (rc) { fails++; if (fails < 20) printf("%s n=%d plane=%d: rule %d broken\n", w, n, k, rc); }
    };
    for (int n = 1; n <= 23; n++) {
        check("pass 1", n, -1, march<4, 2, true>(n, -1, -1));
        check("pass 2", n, -1, march<3, 2, false>(n, -1, -1));
        for (int k = 0; k < n; k++) {
            check("pass 1 stuck", n, k, march<4, 2, true>(n, k, -1));
            check("pass 1 late", n, k, march<4, 2, true>(n, -1, k));
            check("pass 2 late", n, k, march<3, 2, false>(n, -1, k));
        }
    }
    return fails ? 1 : 0;
}
"""


def test_plane_ring_rules(tmp_path):
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout
