"""The library's device allocations (csrc/scratch_cache.h) over an allocator
that holds a stated number of bytes: requests that fail are tried again without
the idle blocks, whether they are for the cache or not, and what lies idle stays
within its bounds.  No device."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_02818_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "scratch_cache.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
static size_t g_room, g_used;
static uintptr_t g_next = 4096;
static std::map<void *, std::pair<size_t, int>> g_held;
static int g_dev;
struct Ops {
    static constexpr int kNoMemory = 2;
    static int allocate(void **p, size_t n)
    {
        if (g_used + n > g_room) return kNoMemory;
        *p = reinterpret_cast<void *>(g_next);
        g_next += n;
        g_used += n;
        g_held[*p] = {n, g_dev};
        return 0;
    }
    static void release(void *p, int dev)
    {
        const auto it = g_held.find(p);
        if (it == g_held.end() || it->second.second != dev) std::abort();
        g_used -= it->second.first;
        g_held.erase(it);
    }
};
using Cache = gbmc::ScratchCache<Ops>;
int main()
{
    const size_t MB = size_t(1) << 20, GB = size_t(1) << 30;
    void *a, *b, *c;
    {   // reuse; the smallest block that fits, at most twice the size
        Cache k;
        g_room = GB;
        CHECK(k.take(0, 3 * MB, &a) == 0 && k.take(0, 2 * MB, &b) == 0);
        k.give(a);
        k.give(b);
        CHECK(k.take(0, 3 * MB / 2, &c) == 0 && c == b);
        CHECK(k.take(0, MB, &b) == 0 && b != a);
        CHECK(k.take(0, 100, &a) == 0 && g_used == 6 * MB + 256);
        k.give(a), k.give(b), k.give(c);
        k.release(-1);
        CHECK(g_used == 0);
    }
    {   // short of memory: idle blocks go, for a cached request and for one past the cache; live ones stay
        Cache k;
        g_room = 100 * MB;
        CHECK(k.take(0, 60 * MB, &a) == 0 && k.take(0, 30 * MB, &b) == 0);
        k.give(a);
        CHECK(k.take_uncached(0, 65 * MB, &c) == 0 && g_used == 95 * MB);
        Ops::release(c, 0);
        k.give(b);
        CHECK(k.take(0, 90 * MB, &a) == 0 && g_used == 90 * MB);
        CHECK(k.take(0, 20 * MB, &b) == Ops::kNoMemory && k.take_uncached(0, 20 * MB, &b) == Ops::kNoMemory);
        k.give(a);
        k.release(0);
        CHECK(g_used == 0);
    }
    {   // another device's idle blocks do not help, and are not given up
        Cache k;
        g_room = 100 * MB;
        g_dev = 1;
        CHECK(k.take(1, 60 * MB, &a) == 0);
        k.give(a);
        g_dev = 0;
        CHECK(k.take(0, 60 * MB, &b) == Ops::kNoMemory && g_used == 60 * MB);
        k.release(1);
        CHECK(g_used == 0);
    }
    {   // bounds on what lies idle: the oldest go first
        Cache k;
        g_room = 64 * GB;
        void *p[40];
        for (int i = 0; i < 40; ++i) CHECK(k.take(0, GB / 2 + i * MB, &p[i]) == 0);
        for (int i = 0; i < 40; ++i) k.give(p[i]);
        CHECK(g_used <= Cache::kIdleBytes && g_used > Cache::kIdleBytes - GB);
        CHECK(g_held.count(p[39]) == 1 && g_held.count(p[0]) == 0);
        const size_t before = g_used;
        CHECK(k.take(0, 10 * GB, &a) == 0);
        k.give(a);
        CHECK(g_used == before);
        k.release(0);
        static void *q[3000];
        for (auto &x : q) CHECK(k.take(0, 256, &x) == 0);
        for (auto &x : q) k.give(x);
        CHECK(g_held.size() == Cache::kIdleBlocks && g_held.count(q[2999]) == 1);
        k.release(-1);
        CHECK(g_used == 0 && g_held.empty());
    }
    std::puts("ok");
    return 0;
}
"""


def test_cache_over_an_allocator_that_fails(tmp_path):
    src, exe = tmp_path / "cache.cpp", tmp_path / "cache"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-include", "cstdint", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout


def test_every_device_allocation_has_the_retry():
    """One call of cudaMalloc, the cache's."""
    hits = [(os.path.basename(f), m.start()) for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
            for m in re.finditer(r"\bcudaMalloc(?:Async)?\(", open(f).read())]
    assert [h[0] for h in hits] == ["mc_api.cu"], hits
