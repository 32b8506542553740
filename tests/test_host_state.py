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


def test_handles_of_a_device_share_the_copy_buffers(tmp_path):
    """One set of page-locked pieces and streams per device however many handles copy; the
    last handle gives it back; a second copy at the same time is left to the caller; the
    caller's current device stays."""
    _run(tmp_path, r"""
#include <cassert>
#include <memory>
#include <cstdlib>
#include "pic_hostcopy.h"
std::atomic<int> pinned{0}, pins{0}, streams{0};
std::atomic<bool> hold{false}, inside{false};
thread_local int device = 3;
bool full = false;
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n)
{
    if (full) return cudaErrorMemoryAllocation;
    ++pinned; ++pins;
    *p = std::malloc(n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { --pinned; std::free(p); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { ++streams; *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { --streams; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    assert(device == 5);
    inside = true;
    while (hold) {}
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}
int main()
{
    const size_t n = (9u << 20) + 77;
    std::vector<char> a(n), b(n);
    for (size_t i = 0; i < n; ++i) a[i] = (char)(i * 31 >> 3);
    {
        std::vector<std::unique_ptr<pic::HostCopy>> h;
        for (int i = 0; i < 100; ++i) {
            h.emplace_back(new pic::HostCopy);
            std::fill(b.begin(), b.end(), 0);
            assert(h.back()->run(b.data(), a.data(), n, 5) && a == b);
            assert(!h.back()->run(b.data(), a.data(), 100, 5));
        }
        assert(pinned == 1 && pins == 1 && streams == 8 && device == 3);
        hold = true;
        inside = false;
        std::vector<char> c(n);
        std::thread t([&] { assert(h[0]->run(c.data(), a.data(), n, 5)); });
        while (!inside) {}
        assert(!h[1]->run(b.data(), a.data(), n, 5));
        hold = false;
        t.join();
        assert(a == c);
        h.resize(1);
        assert(pinned == 1 && h[0]->run(b.data(), a.data(), n, 5));
    }
    assert(pinned == 0 && streams == 0);
    pic::HostCopy again, none;
    assert(again.run(b.data(), a.data(), n, 5) && pinned == 1);
    full = true;
    assert(!none.run(b.data(), a.data(), n, 6) && device == 3);
}
""")
