"""Index arithmetic of the device code, compiled for the host: the cell indices that
the field passes take from a cell number, below and above 2^31 (a run without
particles may have more cells than a particle's cell index can name)."""
import os
import subprocess

import pytest

from paper_1101_0809_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include "pic_device.cuh"
using namespace pic;
int main()
{
    const int sizes[][3] = {{1290, 1290, 1291}, {65537, 65536, 1}, {5, 5, 1 << 28}, {7, 5, 9}, {1073741827, 7, 1}, {8, 1 << 30, 1}};
    long long bad = 0, done = 0;
    for (auto &n : sizes) {
        RunDev rn{};
        for (int a = 0; a < 3; ++a) rn.n[a] = n[a];
        rn.inv_nx = make_inv(n[0]);
        rn.inv_ny = make_inv(n[1]);
        const long long cells = (long long)n[0] * n[1] * n[2], edge = 1LL << 31;
        for (long long at : {0LL, cells / 2, edge - 70000, edge - 3, edge, 2 * edge - 3, cells - 70000, cells - 3})
            for (long long l = at < 0 ? 0 : at; l < cells && l < at + 70000; ++l) {
                int i = -1, j = -1, k = -1;
                yee_ijk(rn, l, i, j, k);
                const long long r = l / n[0];
                bad += i != (int)(l % n[0]) || j != (int)(r % n[1]) || k != (int)(r / n[1]);
                ++done;
            }
    }
    printf("%lld %lld\n", done, bad);
    return 0;
}
"""


def host_run(tmp_path, source):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("the CUDA toolkit is not installed")
    src, exe = str(tmp_path / "host.cu"), str(tmp_path / "host")
    with open(src, "w") as f:
        f.write(source)
    subprocess.run([nvcc, *B.ARCH, "-std=c++17", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), src, "-o", exe],
                   check=True, capture_output=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()


def test_cell_indices_below_and_above_two_to_the_31(tmp_path):
    done, bad = map(int, host_run(tmp_path, SOURCE))
    assert done > 1_000_000 and bad == 0


DRIFT = r"""
#include <cstdio>
#include "pic_device.cuh"
int main()
{
    const int most = 0x7fffffff;
    int sum = 0, bad = 0;
    for (long long step = 1; step <= 300000; ++step) {   // 8192 particles a step pass 2^31 after 262144
        sum = pic::add_drifted(sum, 8192);
        const long long want = 8192 * step;
        bad += sum != (want < most ? (int)want : most);
    }
    bad += pic::add_drifted(most, 0) != most || pic::add_drifted(0, most) != most || pic::add_drifted(3, 4) != 7;
    printf("%d\n", bad);
    return 0;
}
"""


def test_drift_sums_stay_at_the_largest_int(tmp_path):
    assert host_run(tmp_path, DRIFT) == ["0"]
