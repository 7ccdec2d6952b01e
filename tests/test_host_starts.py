"""Cell starts of a checkpoint image become particle keys on the host; starts
that do not rise from 0 to the particle count are refused before a key is
written."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1704_01202_gb300", "csrc", "pic_host.cuh")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "%s"

int main(int argc, char **v)
{
    const int n = atoi(v[1]), ncell = argc - 3;
    std::vector<int> starts, key(n + 64, -7);
    for (int k = 2; k < argc; ++k) starts.push_back(atoi(v[k]));
    printf("%%d", (int)pic::keys_of_starts(starts.data(), ncell, n, key.data()));
    for (int x : key) printf(" %%d", x);
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("starts")
    src = d / "starts.cpp"
    src.write_text(MAIN % SRC)
    exe = d / "starts"
    subprocess.run(["g++", "-std=c++17", "-pthread", "-o", str(exe), str(src)], check=True)
    return lambda n, s: [int(x) for x in subprocess.run([str(exe), str(n)] + [str(x) for x in s], capture_output=True,
                                                        text=True, check=True).stdout.split()]


@pytest.mark.parametrize("n,starts", [(0, [0, 0]), (5, [0, 5]), (5, [0, 0, 2, 2, 5, 5]), (3, [0, 1, 2, 3])])
def test_keys(prog, n, starts):
    r = prog(n, starts)
    assert r[0] == 1
    assert r[1:n + 1] == np.repeat(np.arange(len(starts) - 1), np.diff(starts)).tolist()
    assert set(r[n + 1:]) == {-7}


@pytest.mark.parametrize("n,starts", [(5, [0, 40, 2, 5]), (5, [0, 2, 40, 5]), (5, [0, -3, 2, 5]), (5, [1, 2, 5]), (5, [0, 2, 4]),
                                      (5, [0, 4, 3, 5])])
def test_damaged_starts_write_nothing(prog, n, starts):
    r = prog(n, starts)
    assert r[0] == 0 and set(r[1:]) == {-7}
