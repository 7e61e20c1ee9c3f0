"""The rule for the cluster size of the range finder's QR (csrc/qr_plan.cuh), run on the host with
the numbers of clusters a GB300 holds: the size it takes must be within a tenth of the fastest one,
by the time of the call measured at every size (us, one power, 200 columns)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2201_06914_gb300", "csrc")

# clusters of 1 .. 8 resident at once: with one CTA an SM, with the small shared memory
FIT_SMEM = (152, 76, 46, 36, 28, 23, 15, 15)
FIT_GLOBAL = (456, 228, 148, 110, 87, 74, 59, 51)
# (nt, r, shots): us at clusters of 1 .. 8
TIMES = {
    (300, 16, 1): (218, 177, 166, 156, 155, 152, 152, 150),
    (500, 8, 1): (159, 127, 117, 114, 109, 104, 106, 108),
    (1000, 4, 16): (153, 124, 113, 112, 108, 104, 109, 108),
    (300, 256, 16): (22100, 9860, 5057, 4121, 3405, 3241, 4903, 4750),
    (2000, 64, 16): (9421, 4848, 4045, 2605, 1427, 1257, 2061, 1942),
    (2000, 96, 16): (19170, 9824, 8111, 5194, 4552, 4277, 4865, 3610),
    (2000, 128, 1): (32772, 16667, 13607, 8539, 7501, 7042, 6561, 4828),
    (1000, 96, 64): (9395, 4950, 4930, 3673, 4717, 4215, 6184, 5590),
    (500, 192, 64): (17175, 9406, 8980, 6757, 9249, 7955, 12497, 10859),
    (4000, 256, 64): (464392, 224852, 182087, 131494, 133233, 125216, 170097, 125725),
}

DRIVER = """
#include <cstdio>
#include <cstdlib>
#include "qr_plan.cuh"
int main(int, char **v)
{
    const int fs[8] = {%s}, fg[8] = {%s};
    printf("%%d", wp::qr_cluster(atoi(v[1]), atoi(v[2]), atoi(v[3]), [&](int c, bool smem) { return smem ? fs[c - 1] : fg[c - 1]; }));
    // no cluster size is refused for want of residency: one CTA is the last resort
    return wp::qr_cluster(100, 8, 1, [](int, bool) { return 0; }) == 1 ? 0 : 1;
}
"""


def test_cluster_size_is_near_the_fastest(tmp_path):
    src, exe = tmp_path / "qr.cpp", tmp_path / "qr"
    src.write_text(DRIVER % (", ".join(map(str, FIT_SMEM)), ", ".join(map(str, FIT_GLOBAL))))
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    for k, us in TIMES.items():
        p = subprocess.run([str(exe), *map(str, k)], capture_output=True, text=True, check=True)
        c = int(p.stdout)
        assert 1 <= c <= 8 and us[c - 1] <= 1.1 * min(us), (k, c, us)
