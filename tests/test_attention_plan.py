"""How the attention kernels' work is cut into items (csrc/nfd_attn_plan.h), on the CPU: the plan of a configuration."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "nfd_attn_plan.h"
extern "C" void own_plan(int T, int tiles, int n_blocks, const int *clusters, int *out) {
    AttnPlan pl;
    attn_blocks(pl, T);
    attn_own_plan(pl, tiles, n_blocks, [&](int k) { return clusters[k]; });
    out[0] = pl.MAXSPLIT, out[1] = pl.CH;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SOURCE)
    subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2506_01380_b200", "csrc"), "-o", str(d / "plan.so"), str(d / "plan.cpp")], check=True)
    return C.CDLL(str(d / "plan.so"))


# clusters of k CTAs that a 148-SM B200 holds at once, k = 0 .. 8
B200 = [0, 148, 74, 45, 33, 26, 22, 15, 15]


@pytest.mark.parametrize("T", [40, 77, 220, 336])
def test_clusters_of_the_caller_s_pages_fit_the_machine(lib, T):
    """Every tile's cluster is resident at once, on a whole B200, and on a machine that holds few or no clusters."""
    out = (C.c_int * 2)()
    for machine in (B200, [0, 148, 74, 45, 33, 0, 0, 0, 0], [0, 20, 10, 4, 2, 1, 1, 1, 1], [0, 20] + [0] * 7):
        for tiles in range(1, 160):
            for n_blocks in (1, 2, 9, 33, 51, 400):
                lib.own_plan(T, tiles, n_blocks, (C.c_int * 9)(*machine), out)
                k, ch = out
                assert k == 1 or tiles <= machine[k], (machine, tiles, n_blocks, k)
                assert 1 <= k <= n_blocks and (k - 1) * ch < n_blocks <= k * ch
    lib.own_plan(40, 16, 33, (C.c_int * 9)(*B200), out)
    assert out[0] not in (7, 8)          # 16 clusters of either do not fit
