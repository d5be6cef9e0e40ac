"""The mesh's device memory (csrc/arena.h) on the host, over a stand-in for the device: blocks never
overlap, free neighbours join, what calls return is bounded, a refused chunk gives the unused ones back,
and a rebuild after a change of device takes new memory."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include "arena.h"
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>
using ue::Arena;
static std::map<char*, size_t> dev;      // chunks out
static size_t total, most, limit = SIZE_MAX;
static int cur, gets, idles;
static char* next_p = (char*)(uintptr_t)0x10000000000;   // never followed
static void* get(size_t n) {
    if (total + n > limit) return nullptr;
    char* p = next_p;
    next_p += n + 4096;
    dev[p] = n;
    total += n;
    most = total > most ? total : most;
    ++gets;
    return p;
}
static void put(void* p) {
    auto it = dev.find((char*)p);
    if (it == dev.end()) { puts("put of an unknown chunk"); exit(1); }
    total -= it->second;
    dev.erase(it);
}
static void idle() { ++idles; }
static int device() { return cur; }
static const Arena::Ops ops{get, put, idle, device};
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

static std::map<char*, size_t> live;
static bool sound(char* p, size_t n) {   // inside one chunk, apart from every live block, aligned
    if (((uintptr_t)p & 255) != 0) return false;
    bool in = false;
    for (auto& c : dev) in = in || (p >= c.first && p + n <= c.first + c.second);
    auto a = live.lower_bound(p);
    if (a != live.end() && p + n > a->first) return false;
    if (a != live.begin() && std::prev(a)->first + std::prev(a)->second > p) return false;
    return in;
}

int blocks() {
    Arena a(ops);
    std::mt19937 r(1);
    a.reserve(9 << 20);
    for (int i = 0; i < 4000; ++i) {
        if (live.size() < 40 && r() % 2) {
            const size_t n = r() % 8 ? 1 + r() % 90000 : r() % 3000000;
            const bool temp = r() % 3 == 0;
            char* p = (char*)a.alloc(n, temp);
            CHECK(p && sound(p, n ? n : 1));
            live[p] = n ? n : 1;
        } else if (!live.empty()) {
            auto it = live.begin();
            std::advance(it, r() % live.size());
            CHECK(a.release(it->first));
            CHECK(!a.release(it->first) || live.size() > 1);
            live.erase(it);
        }
        CHECK(a.held() == total);
    }
    CHECK(!a.release((void*)16));
    live.clear();
    return 0;
}

int joining() {   // any order of release leaves one block of the whole chunk
    for (unsigned seed = 0; seed < 20; ++seed) {
        Arena a(ops);
        a.reserve(4 << 20);
        std::vector<void*> p;
        for (int i = 0; i < 16; ++i) p.push_back(a.alloc(1 << 18, false));
        const int g = gets;
        CHECK(a.held() == (size_t)4 << 20);
        std::mt19937 r(seed);
        std::shuffle(p.begin(), p.end(), r);
        for (void* x : p) CHECK(a.release(x));
        CHECK(idles > 0 && a.alloc(4 << 20, false) && gets == g);
    }
    CHECK(total == 0);
    return 0;
}

int calls() {   // eigenmode calls of varying width between a build's arrays: 60k triangles, 1 to 24 modes
    Arena a(ops);
    a.reserve(12 << 20);
    for (int i = 0; i < 25; ++i) a.alloc(480000, false);
    const size_t built = total, n = 60000;
    std::mt19937 r(3);
    most = 0;
    for (int i = 0; i < 1000; ++i) {
        const size_t k = 1 + r() % 24, m = 2 * k < 32 ? 2 * k : 32, work = 8 * (3 * n * m + 6 * n);
        void* w = a.alloc(work, true);
        void* b = a.alloc(8 * k * n, true);
        CHECK(w && b && a.release(w) && a.release(b));
        CHECK(total <= built + Arena::kKeep);
    }
    CHECK(most <= built + Arena::kKeep + 62000000 + 2 * Arena::kChunk);
    const int g = gets;
    for (int i = 0; i < 9; ++i) {   // the same call again takes nothing new
        void* w = a.alloc(20000000, true);
        void* b = a.alloc(4000000, true);
        CHECK(a.release(b) && a.release(w));
    }
    CHECK(gets <= g + 2);
    return 0;
}

int large() {   // large blocks apart, chunks of several bounded
    Arena a(ops);
    a.reserve(300 << 20);
    std::vector<char*> p;
    for (int i = 0; i < 60; ++i) p.push_back((char*)a.alloc(i % 6 == 0 ? 20 << 20 : 3 << 20, false));
    size_t own = 0;
    for (auto& c : dev) {
        CHECK(c.second <= Arena::kGrow);
        own += c.second == (size_t)20 << 20;
    }
    CHECK(own == 10);
    const int g = gets;
    a.reset(true);
    for (int i = 0; i < 60; ++i) CHECK(a.alloc(i % 6 == 0 ? 20 << 20 : 3 << 20, false));
    CHECK(gets == g);
    return 0;
}

int refused() {
    Arena a(ops);
    limit = 40 << 20;
    a.reserve(10 << 20);
    void* x = a.alloc(9 << 20, false);
    void* t = a.alloc(24 << 20, true);
    CHECK(x && t && a.release(t));
    CHECK(a.alloc(20 << 20, false));   // the returned chunk makes room
    CHECK(!a.alloc(20 << 20, false) && !a.alloc(20 << 20, true));
    CHECK(a.release(x) && a.alloc(19 << 20, true));   // a build's chunk, wholly free, as well
    a.reset(false);
    CHECK(total == 0);
    limit = (3 << 20) + (1 << 19);     // less than a chunk more: no more than asked for
    CHECK(a.alloc(2 << 20, false) && a.alloc(1 << 20, false) && a.alloc(1 << 18, false));
    limit = SIZE_MAX;
    return 0;
}

int rebuilds() {
    Arena a(ops);
    auto build = [&](int n, size_t r) {
        a.reserve(r);
        for (int i = 0; i < n; ++i)
            if (!a.alloc(1 << 20, false)) return false;
        return true;
    };
    CHECK(build(8, 8 << 20));
    int g = gets;
    a.reset(true);
    CHECK(build(8, 8 << 20) && gets == g);       // the same chunk
    CHECK(build(20, 0) && dev.size() > 1);       // grown past it
    g = gets;
    a.reset(true);
    CHECK(build(28, 28 << 20) && gets == g);     // the same chunks
    void* t = a.alloc(20 << 20, true);
    CHECK(t && a.release(t));
    g = gets;
    a.reset(true);
    CHECK((t = a.alloc(20 << 20, true)) && gets == g && a.release(t));   // and what a call returned
    CHECK(build(3, 3 << 20) && gets == g);
    a.reset(true);                               // far larger than the last build: not kept
    CHECK(total == 0 && build(3, 3 << 20) && total == (size_t)4 << 20);
    g = gets;
    cur = 1;                                     // another device
    a.reset(true);
    CHECK(total == 0 && build(3, 3 << 20) && gets == g + 1);
    a.reset(true);
    CHECK(build(3, 3 << 20) && gets == g + 1);
    return 0;
}

int main(int, char** v) {
    const std::string s = v[1];
    const int rc = s == "blocks" ? blocks() : s == "joining" ? joining() : s == "calls" ? calls() : s == "refused" ? refused() : s == "large" ? large() : rebuilds();
    if (rc == 0 && total != 0) { puts("chunks left"); return 1; }
    return rc;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("arena")
    (d / "driver.cpp").write_text("#include <string>\n" + DRIVER)
    exe = d / "driver"
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_1812_01448_gb300", "csrc"),
                    str(d / "driver.cpp"), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("case", ["blocks", "joining", "calls", "large", "refused", "rebuilds"])
def test_arena(driver, case):
    r = subprocess.run([driver, case], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
