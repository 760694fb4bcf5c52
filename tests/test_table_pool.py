"""Bookkeeping of the device memory kept for the next handle (csrc/table_pool.h), on the CPU: the pool is
compiled against a made-up device whose contexts, failures and blocks the checks below control."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "table_pool.h"
#include <cassert>
#include <cstdio>
#include <cstdlib>
#include <map>

static unsigned long long g_ctx = 1;                 // the calling thread's context
static std::map<void *, unsigned long long> g_live;  // block -> context it was allocated in
static int g_fail = 0;                               // allocations to refuse for want of memory

struct Dev {
    static unsigned long long context(bool) { return g_ctx; }
    static int alloc(void **p, size_t bytes) {
        if (g_fail) { g_fail--; return 2; }
        *p = malloc(bytes);
        g_live[*p] = g_ctx;
        return 0;
    }
    static bool out_of_memory(int e) { return e == 2; }
    static void release(void *p) { assert(g_live.erase(p) == 1); free(p); }
};
#define CHECK(c) do { if (!(c)) { printf("failed, line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main() {
    using namespace guide;
    TableBlock a, b, c, d;
    {   // a block comes back under its own context only, and is still there afterwards
        TablePool<Dev> pool;
        g_ctx = 1;
        CHECK(pool.take(1000, 1, &a) == 0 && a.context == 1 && a.bytes >= 1000);
        pool.give(a);
        g_ctx = 2;
        CHECK(pool.take(1000, 1, &b) == 0 && b.p != a.p && b.context == 2);
        CHECK(g_live.size() == 2);
        pool.give(b);
        g_ctx = 1;
        CHECK(pool.take(1000, 1, &c) == 0 && c.p == a.p && c.context == 1);
        // handed back while another context is current: not kept as that one's
        g_ctx = 2;
        pool.give(c);
        CHECK(g_live.count(c.p) == 0);
        CHECK(pool.take(1000, 1, &d) == 0 && d.p == b.p);
        Dev::release(d.p);
        CHECK(g_live.empty());
    }
    {   // no context to be had: nothing is taken from the pool, nothing of it is forgotten, nothing is put in
        TablePool<Dev> pool;
        g_ctx = 1;
        CHECK(pool.take(1000, 1, &a) == 0);
        pool.give(a);
        g_ctx = 0;
        CHECK(pool.take(1000, 1, &b) == 0 && b.p != a.p && b.context == 0);
        g_ctx = 1;
        pool.give(b);
        CHECK(g_live.size() == 1);
        CHECK(pool.take(1000, 1, &c) == 0 && c.p == a.p);
        Dev::release(c.p);
        CHECK(g_live.empty());
    }
    {   // a refused allocation gives this context's blocks back first, no other's
        TablePool<Dev> pool;
        g_ctx = 1; CHECK(pool.take(1000, 1, &a) == 0); pool.give(a);
        g_ctx = 2; CHECK(pool.take(1000, 1, &b) == 0); pool.give(b);
        g_fail = 1;
        CHECK(pool.take(500000, 1, &c) == 0);
        CHECK(g_live.count(b.p) == 0 && g_live.count(a.p) == 1);
        Dev::release(c.p);
        g_fail = 2;
        CHECK(pool.take(500000, 1, &c) == 2);
        g_ctx = 1;
        CHECK(pool.take(1000, 1, &c) == 0 && c.p == a.p);
        Dev::release(c.p);
        CHECK(g_live.empty());
    }
    {   // bounded: so many blocks per context and in all, none larger than the limit; the rest is freed
        TablePool<Dev> pool;
        TableBlock many[8];
        for (unsigned long long ctx = 1; ctx <= 40; ctx++) {
            g_ctx = ctx;
            for (TableBlock &m : many) CHECK(pool.take(1000, 1, &m) == 0);
            for (TableBlock &m : many) pool.give(m);
        }
        CHECK(g_live.size() == TablePool<Dev>::TOTAL);
        g_ctx = 1;
        CHECK(pool.take(TablePool<Dev>::BYTES + 1, 1, &a) == 0);
        pool.give(a);
        CHECK(g_live.count(a.p) == 0);
        size_t mine = 0;
        for (auto &l : g_live) mine += l.second == 1;
        CHECK(mine == TablePool<Dev>::PER_CONTEXT);
        for (unsigned long long ctx = 1; ctx <= 40; ctx++) { g_ctx = ctx; pool.drop(ctx); }
        CHECK(g_live.empty());
    }
    {   // the smallest block that is large enough
        TablePool<Dev> pool;
        g_ctx = 1;
        CHECK(pool.take(600000, 1, &a) == 0 && pool.take(100000, 1, &b) == 0 && pool.take(300000, 1, &c) == 0);
        pool.give(a); pool.give(b); pool.give(c);
        CHECK(pool.take(200000, 1, &d) == 0 && d.p == c.p);
        Dev::release(d.p);
        CHECK(!g_live.empty());
    }
    {   // for uploads on the stream its handle was used on only, wherever that was destroyed; any stream if none has used it
        TablePool<Dev> pool;
        g_ctx = 1;
        CHECK(pool.take(1000, 7, &a) == 0);
        a.used_on(7); a.used_on(7);
        pool.give(a);
        CHECK(pool.take(1000, 8, &b) == 0 && b.p != a.p);
        CHECK(pool.take(1000, 7, &c) == 0 && c.p == a.p && c.stream == 0 && c.one_stream);
        pool.give(c);                                // not used since its upload
        CHECK(pool.take(1000, 9, &d) == 0 && d.p == a.p);
        d.used_on(9); d.used_on(7);                  // two streams: freed
        pool.give(d);
        CHECK(g_live.count(a.p) == 0);
        b.used_on(8); b.used_on(0); b.used_on(8);    // once in a capture: freed
        pool.give(b);
        CHECK(g_live.empty());
    }
    {   // the blocks given back last are kept: those of streams that are gone make room
        TablePool<Dev> pool;
        TableBlock many[6];
        g_ctx = 1;
        for (unsigned long long i = 0; i < 6; i++) { CHECK(pool.take(1000, i + 1, &many[i]) == 0); many[i].used_on(i + 1); }
        for (TableBlock &m : many) pool.give(m);
        CHECK(g_live.size() == TablePool<Dev>::PER_CONTEXT && !g_live.count(many[0].p) && !g_live.count(many[1].p));
        for (unsigned long long i = 2; i < 6; i++) {
            CHECK(pool.take(1000, i + 1, &a) == 0 && a.p == many[i].p);
            a.used_on(i + 1);
            pool.give(a);
        }
    }
    CHECK(g_live.empty());                           // freed with the pool
    printf("ok\n");
    return 0;
}
"""


def test_bookkeeping(tmp_path):
    src = tmp_path / "pool.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "pool")
    subprocess.run(["g++", "-std=c++17", "-g", "-fsanitize=address,undefined", "-Wall", "-I",
                    os.path.join(ROOT, "paper_2412_04788_b200", "csrc"), str(src), "-o", exe], check=True, timeout=120)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0 and res.stdout == "ok\n", res.stdout + res.stderr[-2000:]
