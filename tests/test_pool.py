"""The pool of context memory (pool.cu) on a made-up device of a few megabytes,
without a GPU: pool.cu itself, compiled for the host against the CUDA calls that
it makes."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_02012_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

DEVICE = r"""
#include <stdio.h>
#include <stdlib.h>
#include <map>
#include <new>
#include "pool.cu"

static size_t g_room = 8 << 20, g_pins = 8;      // what is left of the device's memory, and pinned blocks
static cudaError_t g_last = cudaSuccess;
static std::map<void*, size_t> g_dev, g_pin;
static bool g_no_new = false;
static unsigned long long g_context = 7;         // 0: none is current

void* operator new(size_t n)
{
    if (g_no_new) throw std::bad_alloc();
    return malloc(n);
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
static unsigned long long g_next = 8;
cudaError_t cudaSetDevice(int)
{
    if (!g_context) g_context = g_next++;
    return cudaSuccess;
}
static CUresult context(CUcontext, unsigned long long* id)
{
    *id = g_context;
    return g_context ? CUDA_SUCCESS : CUDA_ERROR_INVALID_CONTEXT;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q)
{
    *p = (void*)context;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t cudaMalloc(void** p, size_t n)
{
    if (n > g_room) return g_last = cudaErrorMemoryAllocation;
    g_room -= n;
    g_dev[*p = malloc(1)] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    if (!p) return cudaSuccess;
    if (!g_dev.count(p)) return g_last = cudaErrorInvalidValue;
    g_room += g_dev[p];
    g_dev.erase(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t)
{
    if (!g_pins) return g_last = cudaErrorMemoryAllocation;
    --g_pins;
    g_pin[*p = malloc(64)] = 1;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p)
{
    if (!p) return cudaSuccess;
    if (!g_pin.count(p)) return g_last = cudaErrorInvalidValue;
    ++g_pins;
    g_pin.erase(p);
    return cudaSuccess;
}
}

#define CHECK(x) do { if (!(x)) { fprintf(stderr, "line %d: %s\n", __LINE__, #x); exit(1); } } while (0)

using namespace rr;
"""


@pytest.fixture
def run(tmp_path):
    def go(body):
        src, exe = tmp_path / "pool_test.cpp", tmp_path / "pool_test"
        src.write_text(DEVICE + "int main()\n{\n" + body + "\n}\n")
        cmd = ["g++", "-std=c++17", "-O1", "-w", "-pthread", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
               "-I" + os.path.join(CUDA, "include"), str(src), "-o", str(exe)]
        p = subprocess.run(cmd, capture_output=True, text=True)
        assert p.returncode == 0, p.stderr[:3000]
        p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
        assert p.returncode == 0, p.stderr
    return go


def test_short_memory_takes_the_kept_blocks(run):
    run(r"""
    Block a, b;
    void* p = nullptr;
    CHECK(pool_take(6 << 20, &a) == cudaSuccess);
    pool_give(a, true);
    CHECK(device_alloc(&p, 4 << 20) == cudaSuccess);             // does not fit beside the kept block
    CHECK(g_dev.size() == 1 && cudaGetLastError() == cudaSuccess);
    CHECK(device_alloc(&p, 5 << 20) == cudaErrorMemoryAllocation);
    CHECK(cudaGetLastError() == cudaSuccess);                    // (no launch after it fails)
    cudaFree(p);
    // pinned memory, the pool's own words among it
    g_pins = 1;
    CHECK(pool_take(1 << 20, &a) == cudaSuccess && g_pins == 0);
    pool_give(a, true);
    CHECK(pinned_alloc(&p, 64) == cudaSuccess && g_dev.empty());
    cudaFreeHost(p);
    CHECK(pool_take(1 << 20, &a) == cudaSuccess);
    pool_give(a, true);
    CHECK(pool_take(4 << 20, &b) == cudaSuccess);
    pool_give(b, true);
    CHECK(g_dev.size() == 1 && g_pins == 0);
    rr_release_cached();
    CHECK(g_dev.empty() && g_pin.empty());
    """)


def test_giving_back_takes_no_memory(run):
    """A block is kept, an old one dropped and all released while the host has
    no memory left (a C++ exception through the C interface otherwise)."""
    run(r"""
    g_pins = g_room = (size_t)1 << 40;
    Block a[70];
    for (Block& b : a) CHECK(pool_take(64, &b) == cudaSuccess);
    g_no_new = true;
    for (Block& b : a) pool_give(b, true);
    CHECK(g_dev.size() == 64);                                   // the most that are kept
    pool_clear();
    CHECK(g_dev.empty());
    g_no_new = false;
    // the oldest go first, and the smallest that fits is taken
    Block x, y, z;
    CHECK(pool_take((size_t)600 << 20, &x) == cudaSuccess && pool_take((size_t)500 << 20, &y) == cudaSuccess);
    pool_give(x, true);
    pool_give(y, true);                                          // over 1 GiB together
    CHECK(g_dev.size() == 1 && g_dev.count(y.dev));
    CHECK(pool_take((size_t)450 << 20, &z) == cudaSuccess && z.dev == y.dev);
    pool_give(z, false);                                         // not idle: freed
    CHECK(g_dev.empty());
    CHECK(pool_take((size_t)2 << 30, &z) == cudaSuccess);
    pool_give(z, true);                                          // larger than what is kept
    CHECK(g_dev.empty() && g_pin.empty());
    """)


def test_blocks_go_with_their_context(run):
    """After a device reset the kept blocks are neither handed out nor freed (the
    memory at their addresses is someone else's); a thread that has no context
    current yet gets the device's own."""
    run(r"""
    Block a, b, c;
    CHECK(pool_take(1 << 20, &a) == cudaSuccess && pool_take(1 << 20, &b) == cudaSuccess);
    pool_give(a, true);
    g_context = 0;
    g_next = 7;                                                  // no context current in this thread
    CHECK(pool_take(1 << 20, &c) == cudaSuccess && c.dev == a.dev);
    pool_give(c, true);
    g_context = 0;
    g_next = 9;                                                  // the device was reset
    CHECK(pool_take(1 << 20, &c) == cudaSuccess && c.dev != a.dev && c.dev != b.dev);
    pool_give(b, true);                                          // of a context made before it
    pool_give(c, true);
    rr_release_cached();
    CHECK(g_dev.size() == 2 && g_dev.count(a.dev) && g_dev.count(b.dev) && cudaGetLastError() == cudaSuccess);
    """)


def test_every_allocation_can_take_them():
    """No file but pool.cu asks the driver for memory itself."""
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        if name != "pool.cu":
            assert not re.search(r"\bcuda(Malloc\w*|HostAlloc)\s*\(", text), name
