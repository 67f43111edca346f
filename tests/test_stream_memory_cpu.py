"""When a stream's device buffers may move (csrc/stream_memory.h), against a
counted allocator on the host: a buffer whose address a captured graph holds is
never freed, and optional memory is never had at the expense of what is there."""
import subprocess

from paper_2001_02620_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <set>
#include "stream_memory.h"
using namespace qrt;

struct Fake {
    std::set<void*> live;
    size_t largest = 1u << 20;
    int allocs = 0, drains = 0;
    int alloc(void** p, size_t n) {
        ++allocs;
        if (n > largest) return kNoMemory;
        live.insert(*p = std::malloc(n));
        return 0;
    }
    void release(void* p) {
        if (!live.erase(p)) std::exit(2);  // freed twice, or never had
        std::free(p);
    }
    int drain() { ++drains; return 0; }
    size_t spare_bytes = 1u << 20;
    size_t spare() { return spare_bytes; }
};
#define CHECK(c) if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; }

int main() {
    std::vector<void*> retired;
    {   // an adjoint after a captured render leaves the workspace where it is
        Fake m;
        StreamBuffer ws, hits;
        CHECK(need(ws, 1000, false, retired, m) == 0);
        void* const p = ws.ptr;
        CHECK(need(ws, 1000, true, retired, m) == 0 && ws.captured);
        CHECK(need(ws, 1000, false, retired, m) == 0 && want(hits, 100, 5000 / 100, false, retired, m) == 0);
        CHECK(ws.ptr == p && hits.bytes == 5000 && m.live.size() == 2 && retired.empty());
        // a larger render takes another one, and the captured one stays
        CHECK(need(ws, 2000, false, retired, m) == 0);
        CHECK(ws.ptr != p && ws.bytes == 2000 && !ws.captured);
        CHECK(m.live.count(p) && retired.size() == 1 && retired[0] == p);
        // one that no capture saw is freed, after the stream has drained
        void* const q = ws.ptr;
        const int drains = m.drains;
        CHECK(need(ws, 3000, false, retired, m) == 0);
        CHECK(!m.live.count(q) && m.drains == drains + 1 && retired.size() == 1);
    }
    retired.clear();
    {   // nothing is allocated during a capture
        Fake m;
        StreamBuffer ws, hits;
        CHECK(need(ws, 10, true, retired, m) == kCapturing && !ws.ptr && !ws.captured);
        CHECK(want(hits, 10, 1, true, retired, m) == 0 && !hits.ptr && !hits.captured && m.allocs == 0);
        CHECK(need(ws, 10, false, retired, m) == 0);
        CHECK(need(ws, 11, true, retired, m) == kCapturing && ws.bytes == 10 && !ws.captured);
    }
    {   // kept hits of a captured adjoint, and a deeper one after it
        Fake m;
        StreamBuffer hits;
        CHECK(want(hits, 100, 100 / 100, false, retired, m) == 0);
        void* const p = hits.ptr;
        CHECK(want(hits, 100, 300 / 100, true, retired, m) == 0 && hits.ptr == p && hits.captured);
        CHECK(want(hits, 100, 300 / 100, false, retired, m) == 0 && hits.bytes == 300);
        CHECK(m.live.count(p) && retired.size() == 1 && retired[0] == p);
        // memory that is not there: what is there stays, and is not asked for again
        m.largest = 400;
        void* const q = hits.ptr;
        CHECK(want(hits, 100, 500 / 100, false, retired, m) == 0 && hits.ptr == q && hits.bytes == 300);
        const int allocs = m.allocs;
        CHECK(want(hits, 100, 500 / 100, false, retired, m) == 0 && want(hits, 100, 600 / 100, false, retired, m) == 0);
        CHECK(m.allocs == allocs && hits.ptr == q);
        CHECK(want(hits, 100, 400 / 100, false, retired, m) == 0 && hits.bytes == 400 && !m.live.count(q));
        // little memory to spare: as many units as fit it, and no second try
        StreamBuffer few;
        m.spare_bytes = 350;
        CHECK(want(few, 100, 8, false, retired, m) == 0 && few.bytes == 300);
        m.spare_bytes = 1000;
        CHECK(want(few, 100, 8, false, retired, m) == 0 && few.bytes == 300);
        m.spare_bytes = 0;
        StreamBuffer none;
        CHECK(want(none, 100, 2, false, retired, m) == 0 && !none.ptr);
        // a workspace that cannot be had is an error, and holds nothing
        StreamBuffer ws;
        CHECK(need(ws, 401, false, retired, m) == kNoMemory && !ws.ptr && ws.bytes == 0);
    }
    return 0;
}
"""


def test_buffers_of_captured_calls_stay(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", B.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True)
    assert r.returncode == 0, r.stdout
