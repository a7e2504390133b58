"""The bookkeeping of a context's block cache (csrc/blocks.cuh), host code compiled
with g++: classes, reuse, the limit on held bytes, a block freed twice, no host memory, and blocks freed while a graph is captured."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r"""
#include <stdio.h>
#include <stdlib.h>
#include <vector>
#include "blocks.cuh"
using tid::BlockCache;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
static void *addr(size_t i) { return (void *)(4096 + 256 * i); }
"""


def _run(tmp_path, body, head=""):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(HEAD + head + "int main() {\n" + body + "\nreturn 0;\n}\n")
    csrc = os.path.join(ROOT, "paper_1807_01409_gb300", "csrc")
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", csrc, "-x", "c++", "-o", str(exe), str(src),
                           "-pthread"])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_blocks_are_reused_by_class_and_bounded(tmp_path):
    _run(tmp_path, r"""
    static BlockCache b;
    CHECK(BlockCache::class_bytes(BlockCache::class_of(1)) == 256);
    CHECK(BlockCache::class_bytes(BlockCache::class_of(257)) == 320);
    CHECK(BlockCache::class_of(BlockCache::MAX_BLOCK) == BlockCache::CLASSES - 1);
    for (size_t n = 1; n <= BlockCache::MAX_BLOCK; n = n * 3 / 2 + 1)
        CHECK(BlockCache::class_bytes(BlockCache::class_of(n)) >= n && BlockCache::class_bytes(BlockCache::class_of(n)) <= (n < 256 ? 256 : n + n / 4 + 1));
    CHECK(b.take(3) == nullptr && b.put(addr(9)) == BlockCache::POOL);
    for (int i = 0; i < 40; ++i) b.add(addr(i), i % 4);
    for (int i = 0; i < 40; ++i) CHECK(b.put(addr(i)) == BlockCache::KEPT);
    std::vector<int> seen(40, 0);
    for (int i = 0; i < 40; ++i) {
        void *p = b.take(i % 4);
        CHECK(p != nullptr);
        ++seen[((size_t)p - 4096) / 256];
    }
    for (int i = 0; i < 40; ++i) CHECK(seen[i] == 1);
    CHECK(b.held() == 0 && b.take(0) == nullptr);
    const int big = BlockCache::CLASSES - 1;
    for (int i = 0; i < 6; ++i) b.add(addr(100 + i), big);
    for (int i = 0; i < 6; ++i) CHECK(b.put(addr(100 + i)) == (i < 4 ? BlockCache::KEPT : BlockCache::POOL));
    CHECK(b.held() <= BlockCache::MAX_HELD);
    int given = 0;
    CHECK(b.drop([&](void *) { ++given; }) && given == 4 && b.held() == 0);
    CHECK(!b.drop([&](void *) { ++given; }) && b.take(big) == nullptr);
    CHECK(b.put(addr(0)) == BlockCache::KEPT);   // those in use stay known
    """)


def test_a_block_freed_twice_is_reported(tmp_path):
    """Not kept a second time, where two owners would get it, and not passed over in silence."""
    _run(tmp_path, r"""
    static BlockCache b;
    b.add(addr(1), 2);
    b.add(addr(2), 2);
    CHECK(b.put(addr(1)) == BlockCache::KEPT);
    CHECK(b.put(addr(1)) == BlockCache::TWICE);
    CHECK(b.put(addr(2)) == BlockCache::KEPT);
    void *p = b.take(2), *q = b.take(2);
    CHECK(p && q && p != q && b.take(2) == nullptr);
    """)


def test_no_host_memory_is_no_exception(tmp_path):
    """Bookkeeping that finds no host memory does without: nothing is thrown through the C entries (a freed
    block among them, also while an exception or an error path unwinds)."""
    _run(tmp_path, r"""
    static BlockCache b;
    b.add(addr(0), 1);
    refuse = true;
    for (int i = 1; i < 1000; ++i) b.add(addr(i), 1);
    for (int i = 1; i < 1000; ++i) CHECK(b.put(addr(i)) == BlockCache::POOL);   // unknown: the pool's
    CHECK(b.put(addr(0)) == BlockCache::KEPT);
    CHECK(b.take(1) == addr(0));
    refuse = false;
    """, head="""
static bool refuse = false;
void *operator new(size_t n) { if (refuse) throw std::bad_alloc(); return malloc(n); }
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
""")


def test_blocks_freed_under_capture_are_set_aside(tmp_path):
    _run(tmp_path, r"""
    static BlockCache b;
    b.add(addr(1), 2);
    b.add(addr(2), 2);
    b.add(addr(3), BlockCache::LARGE);
    b.add(addr(4), BlockCache::LARGE);
    CHECK(b.put(addr(1), true) == BlockCache::KEPT && b.take(2) == nullptr);
    CHECK(b.put(addr(3), true) == BlockCache::KEPT && b.put(addr(3)) == BlockCache::TWICE);
    CHECK(b.put(addr(9), true) == BlockCache::POOL);    // the graph's own
    CHECK(b.put(addr(4)) == BlockCache::POOL && b.put(addr(4)) == BlockCache::POOL);
    CHECK(b.put(addr(2)) == BlockCache::KEPT);
    int given = 0;
    CHECK(b.drop([&](void *) { ++given; }) && given == 1);
    CHECK(b.drop([&](void *) { ++given; }, true) && given == 3);
    """)
