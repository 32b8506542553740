"""Host-side state of the library that outlives one call, against a fake CUDA runtime: a small
program with its own definitions of the calls that the header makes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2203_06513_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

pytestmark = pytest.mark.skipif(shutil.which("g++") is None or
                                not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")),
                                reason="needs g++ and the CUDA headers")


def _run(tmp_path, source):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-I", os.path.join(CUDA, "include"), str(src),
                    "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True, timeout=60)


def test_shared_memory_limits_are_kept_by_device(tmp_path):
    """A limit raised on one device says nothing about another; it is never lowered, and a
    refusal is not remembered as allowed."""
    _run(tmp_path, r"""
#include <cassert>
#include <map>
#include <utility>
#include "pic_optin.h"
int device = 0, calls = 0;
bool refuse = false;
std::map<std::pair<int, const void *>, int> limit;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v)
{
    ++calls;
    if (refuse) return cudaErrorInvalidValue;
    limit[{device, f}] = v;
    return cudaSuccess;
}
int main()
{
    char a, b;
    pic::SmemOptin one, two;
    assert(one.raise(&a, 40000) && calls == 0);               // the default suffices
    assert(two.raise(&b, 48 * 1024) && calls == 1);           // not with what the kernel has statically
    calls = 0;
    assert(one.raise(&a, 100000) && limit[std::make_pair(0, (const void *)&a)] == 100000);
    assert(one.raise(&a, 90000) && calls == 1 && one.allowed(90000));
    device = 1;
    assert(!one.allowed(90000));
    assert(one.raise(&a, 90000) && calls == 2 && limit[std::make_pair(1, (const void *)&a)] == 90000);
    device = 0;
    assert(one.raise(&a, 100000) && calls == 2);
    const void *const both[] = {&a, &b};
    assert(two.raise(both, 70000) && calls == 4);
    refuse = true;
    assert(!two.raise(both, 80000) && !two.allowed(80000));
    device = 1000;                                            // beyond the table: asked for every time
    refuse = false;
    assert(one.raise(&a, 60000) && one.raise(&a, 60000) && calls == 7);
}
""")
