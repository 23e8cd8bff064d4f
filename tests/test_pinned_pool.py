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
    const void* context() { return reinterpret_cast<void*>(static_cast<intptr_t>(now)); }
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
    for (auto& x : b) { x = pool.get(); assert(x.p && x.slab && seen.insert(x.p).second); memset(x.p, 1, 256); }
    for (auto& x : b) assert(pool.put(x));
    Pinned again = pool.get();
    assert(seen.count(again.p));
    assert(pool.put(again));
    assert(!pool.put({}));
    """)


def test_a_lost_context_takes_its_slab_with_it(tmp_path):
    """Its blocks are never handed out again, nor given back into the slab
    that now lies where it did."""
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 4);
    Pinned old = pool.get();
    pool.driver().lose(1);
    Pinned young = pool.get();
    assert(young.p == old.p && young.slab != old.slab);       // the same address
    assert(pool.driver().id(young.p) == young.slab);          // and live
    pool.put(old);
    Pinned other = pool.get();
    assert(other.p != young.p);
    pool.put(young);
    pool.put(other);
    """)


def test_each_context_has_its_own_slab(tmp_path):
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 4);
    Pinned a = pool.get();
    pool.driver().now = 2;
    Pinned b = pool.get();
    assert(a.slab != b.slab);
    pool.driver().lose(1);
    memset(b.p, 1, 256);
    assert(pool.driver().id(static_cast<char*>(b.p)) == b.slab);   // the second context's is still there
    Pinned c = pool.get();
    assert(c.slab == b.slab && c.p != b.p);
    pool.put(a); pool.put(b); pool.put(c);
    """)


def test_no_memory_and_no_ids(tmp_path):
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 4);
    pool.driver().fail = 1;
    assert(!pool.get().p);
    pool.driver().fail = 0;
    Pinned a = pool.get();
    assert(a.p);
    pool.put(a);
    struct NoId : Fake { unsigned long long id(void*) { return 0; } };
    lbm::PinnedPool<NoId> blind(256, 4);
    Pinned b = blind.get();
    assert(b.p && b.slab == 0 && blind.driver().live.size() == 1);
    assert(!blind.put(b));                                    // the owner's to release
    """)


def test_many_owners_share_slabs_which_are_given_back(tmp_path):
    """No owner beyond a slab's blocks pays for memory of its own, and no
    more than one empty slab stays."""
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 8);
    std::vector<Pinned> b(100);
    for (int round = 0; round < 3; ++round) {
        const int before = pool.driver().allocations;
        for (auto& x : b) { x = pool.get(); assert(x.p && x.slab); }
        assert(pool.driver().live.size() == 13 && pool.driver().allocations - before == (round ? 12 : 13));
        for (size_t k = 0; k < b.size(); ++k) assert(pool.put(b[(k * 37) % 100]));
        assert(pool.driver().live.size() == 1);
    }
    for (int k = 0; k < 50; ++k) {                            // one owner after another, at a full slab's edge too
        for (int i = 0; i < 8; ++i) b[i] = pool.get();
        const int before = pool.driver().allocations;
        for (int i = 0; i < 5; ++i) assert(pool.put(pool.get()));
        assert(pool.driver().allocations - before == 1 && pool.driver().live.size() == 2);
        for (int i = 0; i < 8; ++i) assert(pool.put(b[i]));
        assert(pool.driver().live.size() <= 2);
        b[8] = pool.get(); b[9] = pool.get();
        assert(pool.put(b[8]) && pool.put(b[9]));
    }
    """)


def test_threads(tmp_path):
    check(tmp_path, """
    lbm::PinnedPool<Fake> pool(256, 16);
    Pinned first = pool.get();                              // the slab is there: threads only share its blocks
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] {
            for (int i = 0; i < 2000; ++i) {
                Pinned b = pool.get();
                memset(b.p, k + 1, 256);
                std::this_thread::yield();
                for (int j = 0; j < 256; ++j) assert(static_cast<char*>(b.p)[j] == k + 1);
                pool.put(b);
            }
        });
    for (auto& x : t) x.join();
    pool.put(first);
    """)
