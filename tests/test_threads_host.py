"""parallel_for, the host loops of mesh and simulation creation, when a thread cannot start or
a loop body throws: every item is still done once, or the exception reaches the caller (who
turns it into a status), and no thread is left behind."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SOURCE = r"""
#include <atomic>
#include <cerrno>
#include <cstdio>
#include <cstdlib>
#include <dlfcn.h>
#include <pthread.h>
#include "pic_internal.h"

static std::atomic<int> starts{0};
static int allowed = 0;

// the system's, for the first `allowed` threads
extern "C" int pthread_create(pthread_t *t, const pthread_attr_t *a, void *(*f)(void *), void *x) {
    using Fn = int (*)(pthread_t *, const pthread_attr_t *, void *(*)(void *), void *);
    static const Fn real = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "pthread_create"));
    return starts++ < allowed ? real(t, a, f, x) : EAGAIN;
}

int main(int argc, char **argv) {
    allowed = atoi(argv[1]);
    const long fail_at = atol(argv[2]);
    const int64_t n = 100003;
    std::vector<std::atomic<int>> seen(n);
    try {
        pic::parallel_for(n, [&](int64_t a, int64_t b) {
            for (int64_t i = a; i < b; i++) {
                if (i == fail_at) throw std::bad_alloc();
                seen[i]++;
            }
        });
    } catch (const std::bad_alloc &) {
        puts("bad_alloc");
        return fail_at >= 0 ? 0 : 1;
    }
    if (fail_at >= 0) return 2;
    for (int64_t i = 0; i < n; i++)
        if (seen[i] != 1) return 3;
    puts("all once");
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("threads")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-D_GNU_SOURCE", "-I", os.path.join(CUDA, "include"),
                    "-I", os.path.join(ROOT, "paper_1701_03784_gb300", "csrc"), str(src), "-o", str(exe),
                    "-lpthread", "-ldl"], check=True, capture_output=True, text=True)
    return str(exe)


@pytest.mark.parametrize("threads", [0, 1, 3, 1000])
@pytest.mark.parametrize("fail_at", [-1, 0, 50000, 100002])
def test_every_item_or_an_exception(program, threads, fail_at):
    if (os.cpu_count() or 1) < 2:
        pytest.skip("one core: no threads are started")
    r = subprocess.run([program, str(threads), str(fail_at)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    assert r.stdout.strip() == ("all once" if fail_at < 0 else "bad_alloc")
