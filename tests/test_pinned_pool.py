"""The pool of pinned blocks (csrc/lbm_pinned_pool.h) over a driver of the
test's own: no GPU.  Its memory comes from one arena, so that an allocation
made after a context was lost lies where the lost one did."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1412_7228_gb300", "csrc")

FAKE = r"""
#include <cassert>
#include <cstdint>
#include <cstring>
#include <map>
#include <set>
#include <thread>
#include "lbm_pinned_pool.h"
using lbm::Pinned;
struct Fake {
    alignas(256) static char arena[1 << 20];
    std::map<char*, std::pair<size_t, std::pair<unsigned long long, int>>> live;   // address: size, (id, context)
    unsigned long long next = 1;
    int now = 1, fail = 0, allocations = 0;
    void* allocate(size_t bytes) {
        if (fail) return nullptr;
        char* p = arena;
        for (auto& a : live) if (p + bytes > a.first && p < a.first + a.second.first) p = a.first + a.second.first;
        assert(p + bytes <= arena + sizeof arena);
        live[p] = {bytes, {next++, now}};
        ++allocations;
        return p;
    }
    void release(void* p) { assert(live.erase(static_cast<char*>(p)) == 1); }
    unsigned long long context() { return now; }
    unsigned long long id(void* p) {
        auto it = live.find(static_cast<char*>(p));
        return it == live.end() ? 0 : it->second.second.first;
    }
    void lose(int c) {   // the context and its allocations are gone
        for (auto it = live.begin(); it != live.end();) it = it->second.second.second == c ? live.erase(it) : std::next(it);
    }
};
alignas(256) char Fake::arena[1 << 20];
int main() {
%s
    return 0;
}
"""


def check(tmp_path, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(FAKE.replace("%s", body))
    r = subprocess.run([cxx, "-std=c++17", "-Wall", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def test_blocks_are_distinct_and_used_again(tmp_path):
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 4);
    Pinned b[6];
    std::set<void*> seen;
    for (auto& x : b) { x = pool.get(200); assert(x.p && seen.insert(x.p).second); memset(x.p, 1, 200); }
    Pinned big = pool.get(5000);
    assert(big.p && big.slab == 0);
    pool.put(big);
    for (auto& x : b) pool.put(x);
    Pinned again = pool.get(256);
    assert(again.slab == b[0].slab && again.p == b[0].p);
    pool.put(again);
    pool.put({});
    """)


def test_a_lost_context_takes_its_slab_with_it(tmp_path):
    """Its blocks are never handed out again, nor given back into the slab
    that now lies where it did."""
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 4);
    Pinned old = pool.get(256);
    pool.driver().lose(1);
    Pinned young = pool.get(256);
    assert(young.p == old.p && young.slab != old.slab);       // the same address
    assert(pool.driver().id(young.p) == young.slab);          // and live
    pool.put(old);
    Pinned other = pool.get(256);
    assert(other.p != young.p);
    pool.put(young);
    pool.put(other);
    """)


def test_each_context_has_its_own_slab(tmp_path):
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 4);
    Pinned a = pool.get(256);
    pool.driver().now = 2;
    Pinned b = pool.get(256);
    assert(a.slab != b.slab);
    pool.driver().lose(1);
    memset(b.p, 1, 256);
    assert(pool.driver().id(static_cast<char*>(b.p)) == b.slab);   // the second context's is still there
    Pinned c = pool.get(256);
    assert(c.slab == b.slab && c.p != b.p);
    pool.put(a); pool.put(b); pool.put(c);
    """)


def test_no_memory_and_no_ids(tmp_path):
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 4);
    pool.driver().fail = 1;
    assert(!pool.get(256).p && !pool.get(5000).p);
    pool.driver().fail = 0;
    Pinned a = pool.get(256);
    assert(a.p);
    pool.put(a);
    struct NoId : Fake { unsigned long long id(void*) { return 0; } };
    lbm::PinnedPool<NoId> blind(256, 4);
    Pinned b = blind.get(256);
    assert(b.p && b.slab == 0 && blind.driver().live.size() == 1);
    blind.put(b);
    assert(blind.driver().live.empty());
    """)


def test_threads(tmp_path):
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 16);
    Pinned first = pool.get(256);                              // the slab is there: threads only share its blocks
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] {
            for (int i = 0; i < 2000; ++i) {
                Pinned b = pool.get(256);
                memset(b.p, k + 1, 256);
                std::this_thread::yield();
                for (int j = 0; j < 256; ++j) assert(static_cast<char*>(b.p)[j] == k + 1);
                pool.put(b);
            }
        });
    for (auto& x : t) x.join();
    pool.put(first);
    """)
