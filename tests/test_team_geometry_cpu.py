"""CPU tests of the whole-row kernels' geometry (host code of the library), through a small program linked to it."""
import os
import subprocess

import pytest

from paper_2609_01864_gb300 import build as B

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "credit_host.h"
using namespace credit;
int main(int, char **v) {  // SMs, rows, cols, element size, gamma / beta arrays, cluster size
    DeviceInfo di{};
    di.sm_count = atoi(v[1]);
    di.smem_optin = di.smem_per_sm = 232448;
    TeamCfg c{};
    const bool ok = team_config(di, atoll(v[2]), atoll(v[3]), atoi(v[4]), atoi(v[5]), atoi(v[6]), 0, &c);
    if (!ok) return puts("no"), 0;
    printf("%d %d %d %d %lld %d\n", c.P, c.threads, c.teams, c.stages, c.smem, c.grid);
}
"""


@pytest.fixture(scope="module")
def geometry(tmp_path_factory):
    lib = B.build()
    d = tmp_path_factory.mktemp("geometry")
    src, exe = d / "g.cpp", d / "g"
    src.write_text(SRC)
    cuda = os.path.dirname(os.path.dirname(B._nvcc()))
    subprocess.run(["g++", "-O1", "-std=c++17", f"-I{B.CSRC}", f"-I{os.path.join(B.ROOT, 'include')}",
                    f"-I{os.path.join(cuda, 'include')}", str(src), lib, f"-Wl,-rpath,{os.path.dirname(lib)}", "-o",
                    str(exe)], check=True)

    def run(*a):
        r = subprocess.run([str(exe), *map(str, a)], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.returncode
        return None if r.stdout == "no\n" else [int(x) for x in r.stdout.split()]
    return run


@pytest.mark.parametrize("sms", [1, 2, 7, 8, 15])
@pytest.mark.parametrize("P", [1, 2, 4, 8, 16])
def test_a_cluster_wider_than_the_device_is_refused(geometry, sms, P):
    got = geometry(sms, 500, 40000, 4, 1, P)
    if P > sms:
        assert got is None
    elif got is not None:
        assert got[0] == P and 1 <= got[5] <= sms // P


@pytest.mark.parametrize("P", [0, 3, 6, 32, -1])
def test_other_cluster_sizes_are_refused(geometry, P):
    assert geometry(152, 500, 40000, 4, 1, P) is None
