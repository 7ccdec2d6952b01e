"""Loading splits its records over host threads; with fewer to be had than
wanted, or none, the same shares are done and nothing ends the process."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1704_01202_gb300", "csrc", "pic_host.cuh")

MAIN = r"""
#include <atomic>
#include <cerrno>
#include <cstdio>
#include <cstdlib>
#include <dlfcn.h>
#include <pthread.h>
#include "%s"

static std::atomic<int> left{0};
extern "C" int pthread_create(pthread_t *t, const pthread_attr_t *a, void *(*f)(void *), void *x) noexcept
{
    if (left.fetch_sub(1) <= 0) return EAGAIN;
    typedef int (*fn)(pthread_t *, const pthread_attr_t *, void *(*)(void *), void *);
    return ((fn)dlsym(RTLD_NEXT, "pthread_create"))(t, a, f, x);
}

int main(int, char **v)
{
    const int shares = atoi(v[1]);
    left = atoi(v[2]);
    std::vector<int> done(shares + 1, 0);
    pic::host_shares(shares, [&](int t) { done[t] += t + 1; });
    for (int t = 0; t < shares; ++t)
        if (done[t] != t + 1) return 1;
    printf("created %%d\n", atoi(v[2]) - std::max(left.load(), 0));
    return done[shares] != 0;
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("threads")
    src = d / "shares.cpp"
    src.write_text("#include <algorithm>\n" + MAIN % SRC)
    exe = d / "shares"
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-o", str(exe), str(src), "-ldl"], check=True)
    return str(exe)


@pytest.mark.parametrize("shares", [0, 1, 2, 16])
@pytest.mark.parametrize("threads", [0, 1, 3, 100])
def test_shares_without_enough_threads(prog, shares, threads):
    r = subprocess.run([prog, str(shares), str(threads)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr)
    assert r.stdout == f"created {min(threads, max(shares - 1, 0))}\n"


def test_load_uses_them():
    api = open(os.path.join(os.path.dirname(SRC), "pic_api.cu")).read()
    assert "std::thread" not in api.replace("std::thread::hardware_concurrency", "")
    assert "host_shares(" in api
