// graph_scratch.h -- the fixed scratch of hs_sign_mixed's kept graph.
//
// A call asks for 'full' bytes (shared trees and chain ends are extra) and can
// do with 'lean'.  Where the device refused full, the call signs in the lean
// layout, and an identical next call must neither give the buffer back nor
// ask again while the memory it could get has not grown: the graph in the
// buffer is then relaunched as it is.
#pragma once
#include <cstddef>

namespace hs {

struct GraphScratch {
    void* p = nullptr;
    size_t cap = 0;
    size_t refused = 0;        // the request refused last (0: none since the last that held)
    size_t refused_avail = 0;  // free bytes at that time, the buffer given back
};

enum class Layout { full, lean, none };

// Mem: alloc(void**, size_t) -- true if it holds; release(void*) -- after the
// last graph; avail() -- free bytes.
template <class Mem>
Layout reserve_graph_scratch(GraphScratch& g, size_t full, size_t lean, Mem& mem) {
    auto grow = [&](size_t n) {
        if (g.p) mem.release(g.p);
        g.p = nullptr;
        g.cap = 0;
        if (mem.alloc(&g.p, n)) g.cap = n;
        return g.cap != 0;
    };
    if (full <= g.cap) return Layout::full;
    if (g.refused == 0 || full < g.refused || lean >= full || mem.avail() + g.cap > g.refused_avail) {
        if (grow(full)) {
            g.refused = 0;
            return Layout::full;
        }
        if (lean >= full) return Layout::none;
        g.refused = full;
        g.refused_avail = mem.avail();
    }
    return lean <= g.cap || grow(lean) ? Layout::lean : Layout::none;
}

}  // namespace hs
