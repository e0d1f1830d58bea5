"""The scratch of hs_sign_mixed's kept graph under memory pressure, with a
fake device in place of cudaMalloc: a call whose full request is refused signs
in the lean layout, identical calls after it leave the buffer alone (so the
graph in it is relaunched), and the full request is made again once more
memory is free."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <map>
#include "graph_scratch.h"
using namespace hs;
struct Fake {                       // a device of 'room' bytes, 2 MB granules
    size_t room, used = 0;
    int allocs = 0, frees = 0;
    std::map<void*, size_t> held;
    static size_t up(size_t n) { return (n + 2097151) / 2097152 * 2097152; }
    bool alloc(void** p, size_t n) {
        allocs++;
        if (used + up(n) > room) return false;
        *p = reinterpret_cast<void*>((size_t)allocs << 30);
        held[*p] = up(n);
        used += up(n);
        return true;
    }
    void release(void* p) { frees++; used -= held[p]; held.erase(p); }
    size_t avail() { return room - used; }
};
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); bad++; } } while (0)
int main() {
    int bad = 0;
    const size_t M = 1 << 20;
    Fake d{100 * M};
    GraphScratch g;
    CHECK(reserve_graph_scratch(g, 60 * M, 30 * M, d) == Layout::full && g.cap == 60 * M);
    CHECK(reserve_graph_scratch(g, 50 * M, 30 * M, d) == Layout::full && d.allocs == 1);
    CHECK(reserve_graph_scratch(g, 120 * M, 70 * M, d) == Layout::lean && g.cap == 70 * M && d.held.size() == 1);
    const int a = d.allocs, f = d.frees;
    void* const p = g.p;
    for (int i = 0; i < 5; i++) CHECK(reserve_graph_scratch(g, 120 * M, 70 * M, d) == Layout::lean);
    CHECK(d.allocs == a && d.frees == f && g.p == p);                      // nothing given back, nothing asked
    CHECK(reserve_graph_scratch(g, 65 * M, 40 * M, d) == Layout::full && g.p == p);
    CHECK(reserve_graph_scratch(g, 130 * M, 60 * M, d) == Layout::lean && g.p == p);
    CHECK(reserve_graph_scratch(g, 130 * M, 80 * M, d) == Layout::lean && g.cap == 80 * M);   // lean itself grows
    CHECK(reserve_graph_scratch(g, 99 * M, 80 * M, d) == Layout::full && g.cap == 99 * M);    // less than was refused
    CHECK(reserve_graph_scratch(g, 120 * M, 100 * M, d) == Layout::lean && g.cap == 100 * M);
    d.room = 200 * M;                                                       // others freed memory
    CHECK(reserve_graph_scratch(g, 120 * M, 100 * M, d) == Layout::full && g.cap == 120 * M && g.refused == 0);
    CHECK(reserve_graph_scratch(g, 300 * M, 250 * M, d) == Layout::none && g.p == nullptr && g.cap == 0);
    CHECK(reserve_graph_scratch(g, 300 * M, 300 * M, d) == Layout::none);
    CHECK(reserve_graph_scratch(g, 10 * M, 10 * M, d) == Layout::full && d.held.size() == 1);
    return bad;
}
"""


def test_refused_request_is_not_repeated(tmp_path):
    src, exe = str(tmp_path / "g.cpp"), str(tmp_path / "g")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", src, "-o", exe, "-I",
                    os.path.join(ROOT, "paper_2512_23969_gb300", "csrc")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
