"""Host check of the rules that choose a kernel's form by size (kernels.h, compiled for the host with
nvcc): the L2 prefetch of the FP32 two-site sweep, over the sizes lbm_create accepts (a group of rows of
2^30 sites times 4 does not fit 32 bits), stays off in the forms it was measured to slow down, and where
it is on a group is a few kB and the distance within the sites it was measured at."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1105_2904_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include "kernels.h"
using namespace lbmp;
static int ahead(long long nx, long long ny, long long nz, double share, int bx)
{
    Geom g{};
    g.nx = (int)nx; g.ny = (int)ny; g.nz = (int)nz; g.N = (unsigned)(nx * ny * nz);
    return prefetch_groups(g, (long long)(share * (double)g.N), bx, bx > 64 ? 1 : 64 / bx);
}
int main()
{
    for (int bx : {16, 32, 64, 128})
        for (double share : {0.0, 0.05, 0.1, 0.3})
            for (long long nx = 2; nx < (1ll << 31); nx += nx < 5000 ? 2 : nx / 3 / 2 * 2)
                for (long long ny : {1ll, 2ll, 5ll, 64ll, 65535ll})
                    for (long long nz : {1ll, 3ll, 512ll}) {
                        if (nx * ny * nz >= (1ll << 31)) continue;
                        const long long group = nx * (bx > 64 ? 1 : 64 / bx);
                        const int a = ahead(nx, ny, nz, share, bx);
                        if (a < 0 || (a && (group > 16384 || (a - 1) * group > 131072 || share == 0.0 || bx != 16))) {
                            std::printf("%lld x %lld x %lld, share %g, bx %d: %d\n", nx, ny, nz, share, bx, a);
                            return 1;
                        }
                    }
    if (ahead(1 << 30, 1, 1, 0.3, 16) || ahead(512, 512, 512, 0.08, 16) || ahead(64, 512, 256, 0.256, 16)) return 2;
    if (!ahead(512, 512, 512, 0.256, 16) || !ahead(1024, 2048, 1, 0.075, 16)) return 3;
    std::printf("ok\n");
    return 0;
}
'''


def test_prefetch_rule(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "rules.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "rules"
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", (out.returncode, out.stdout)
