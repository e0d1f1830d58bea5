"""The scratch regions of a batch, checked on the host: carve_scratch lays out
exactly the bytes that scratch_bytes sizes, every region lies inside them and
none overlaps another, for batches with their own keys and with a keyset's
resident ones (whose key blocks are not scratch), signing and verifying, in
every form.  A small C++ program linked with the library's objects does it;
no kernel is launched and no region is touched."""
import glob
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = r"""
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <utility>
#include <vector>
#include "hs_launch.h"
using namespace hs;
static int bad = 0;
"""

LAYOUT = COMMON + r"""
struct R { const void* p; size_t n; };
static void check(Batch b, const char* what) {
    SetShape s;
    set_shape(b.pset, &s);
    const size_t w = s.n, cnt = b.count, own = b.dedup_layer ? b.dedup_layer : s.d;
    const size_t mu = b.cached ? 0 : b.max_uniq, per = b.ck ? 16 / b.ck : 0;
    const size_t len = 2 * s.n + 3;
    KeyBlock* const resident = reinterpret_cast<KeyBlock*>(8);
    if (b.resident) b.keys = resident;
    char* base = reinterpret_cast<char*>(1 << 20);
    const size_t want = scratch_bytes(b), got = carve_scratch(b, base);
    bool ok = want == got && (!b.resident || b.keys == resident);
    std::vector<R> r = {{b.offsets, (cnt + 1) * 8}, {b.infos, cnt * sizeof(MsgInfo)}, {b.pk_fors, cnt * w},
                        {b.roots, cnt * s.d * w}, {b.chk, cnt * s.d * len * per * w}};
    if (!b.resident) r.push_back({b.keys, b.num_keys * sizeof(KeyBlock)});
    if (b.ends) r.push_back({b.ends, (b.verify ? cnt : (cnt * own + mu) * s.leaves) * len * w});
    if (b.mj_id) r.push_back({b.mj_id, cnt * (s.d - own) * 4});
    if (mu) r.push_back({b.nodes_u, mu * 2 * s.leaves * w});
    if (mu && b.chk_u) r.push_back({b.chk_u, mu * s.leaves * len * per * w});
    if (b.leafv) r.push_back({b.leafv, cnt * s.d * s.leaves * w});
    if (b.vends) r.push_back({b.vends, cnt * s.d * len * 16 * w});
    if (b.vorder) r.push_back({b.vorder, cnt * len * 4});
    std::sort(r.begin(), r.end(), [](const R& x, const R& y) { return x.p < y.p; });
    const char* at = base;
    for (const R& x : r) {
        if (!x.n) continue;
        ok = ok && static_cast<const char*>(x.p) >= at;
        at = static_cast<const char*>(x.p) + x.n;
    }
    ok = ok && at <= base + want;
    if (!ok) { printf("%s: set %d keys %u count %u ck %u split %d: sized %zu, carved %zu\n", what, b.pset, b.num_keys, b.count, b.ck, b.split, want, got); bad++; }
}
int main() {
    for (int p = 0; p < kNumSets; p++) {
        SetShape s;
        set_shape(p, &s);
        for (unsigned keys : {1u, 1000u})
            for (unsigned count : {1u, 7u, 2100u})
                for (unsigned ck : {0u, 1u, 2u, 8u})
                    for (int split = 0; split < 2; split++) {
                        Batch b;
                        memset(&b, 0, sizeof b);
                        b.pset = p; b.num_keys = keys; b.count = count; b.ck = ck; b.split = split;
                        check(b, "sign");
                        plan_dedup(b);
                        check(b, "sign, shared trees");
                        b.resident = true;
                        check(b, "keyset, shared trees");
                        const size_t one = (b.num_keys = 1, scratch_bytes(b));
                        b.num_keys = 1000;
                        if (scratch_bytes(b) != one) { printf("set %d: key blocks of a keyset in the scratch\n", p); bad++; }
                        b.num_keys = keys;
                        drop_dedup(b);
                        check(b, "keyset");
                        b.cached = true; b.dedup_layer = s.d - 1; b.cache_tpk = 1;
                        check(b, "keyset, cached layer");
                    }
        for (int walk = 0; walk < 2; walk++)
            for (unsigned count : {1u, 33u, 100u}) {
                Batch b;
                memset(&b, 0, sizeof b);
                b.pset = p; b.num_keys = 3; b.count = count; b.verify = true; b.walk = walk;
                check(b, "verify");
            }
    }
    return bad != 0;
}
"""


KEYSET = COMMON + r"""
int main() {
    uint32_t own_nodes = 0, own_chk = 0;
    for (int p = 0; p < kNumSets; p++)
        for (unsigned layers : {0u, 1u})
            for (unsigned count : {3u, 4u, 5000u}) {
                SetShape s;
                set_shape(p, &s);
                hs_keyset ks;
                ks.pset = p; ks.num_keys = 2; ks.layers = layers; ks.first_layer = s.d - layers; ks.tpk = layers; ks.ck = 2;
                ks.kb = reinterpret_cast<KeyBlock*>(64);
                if (layers) { ks.nodes = &own_nodes; ks.chk = &own_chk; }      // null without layers
                Batch b;
                memset(&b, 0, sizeof b);
                b.pset = p; b.count = count;
                use_keyset(b, ks);
                if (!b.cached) plan_dedup(b);
                carve_scratch(b, reinterpret_cast<char*>(1 << 20));
                const bool built = b.max_uniq != 0;
                bool ok = b.keys == ks.kb && b.num_keys == 2 && b.ck == 2 && (b.cached != 0) == (layers != 0);
                ok = ok && built == (layers == 0 && count >= 4);
                if (built) ok = ok && b.desc && b.nodes_u > reinterpret_cast<uint32_t*>(1 << 20);
                if (layers) ok = ok && b.nodes_u == &own_nodes && b.chk_u == &own_chk && b.dedup_layer == (unsigned)s.d - 1;
                if (!ok) { printf("set %d layers %u count %u: nodes_u %p\n", p, layers, count, (void*)b.nodes_u); bad++; }
            }
    return bad != 0;
}
"""


WIDE = COMMON + r"""
int main() {
    for (int p = 0; p < kNumSets; p++) {
        SetShape s;
        set_shape(p, &s);
        if (s.leaves <= 32) continue;
        for (unsigned keys : {1u, 16u}) {
            Batch b;
            memset(&b, 0, sizeof b);
            b.pset = p; b.num_keys = keys; b.count = 16384; b.ck = 2;
            const size_t own = scratch_bytes(b);
            plan_dedup(b);
            const size_t shared = scratch_bytes(b);
            if (!b.max_uniq || shared > own + (own >> 2)) { printf("set %d, %u keys: %zu bytes alone, %zu shared\n", p, keys, own, shared); bad++; }
        }
    }
    return bad != 0;
}
"""


ENDS = COMMON + r"""
int main() {
    for (int p = 0; p < kNumSets; p++) {
        const int below = tune_get(p, 2);                    // no tuned cache: the default line
        if (below <= 1) continue;
        SetShape s;
        set_shape(p, &s);
        const double ends = (below - 1.0) * s.d * s.leaves * (2 * s.n + 3) * s.n;
        if (ends > 2.5e9) { printf("set %d: %.2f GB of chain ends at %d messages\n", p, ends / 1e9, below - 1); bad++; }
    }
    return bad != 0;
}
"""


@pytest.fixture(scope="module")
def run_cpp(tmp_path_factory):
    """Compile a program against the library's objects and run it."""
    from paper_2512_23969_gb300 import build
    build.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    csrc = os.path.join(ROOT, "paper_2512_23969_gb300", "csrc")
    libs = [d for d in (os.path.join(cuda, "lib64"), *glob.glob(os.path.join(cuda, "targets", "*", "lib")))
            if os.path.exists(os.path.join(d, "libcudart_static.a"))]
    incs = [d for d in (os.path.join(cuda, "include"), *glob.glob(os.path.join(cuda, "targets", "*", "include")))
            if os.path.exists(os.path.join(d, "cuda_runtime.h"))]
    objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    assert objs and libs and incs

    def run(name, source):
        d = tmp_path_factory.mktemp(name)
        src, exe = str(d / (name + ".cpp")), str(d / name)
        with open(src, "w") as f:
            f.write(source)
        subprocess.run(["g++", "-std=c++17", "-O1", src, "-o", exe, "-I", csrc] + ["-I" + i for i in incs] + objs +
                       ["-L" + libs[0], "-lcudart_static", "-ldl", "-lrt", "-lpthread"], check=True)
        return subprocess.run([exe], capture_output=True, text=True)
    return run


def test_layout_matches_size(run_cpp):
    r = run_cpp("layout", LAYOUT)
    assert r.returncode == 0, r.stdout[-2000:]


def test_keyset_trees_have_memory(run_cpp):
    """The trees a keyset call builds itself live in its scratch; only a
    keyset with prebuilt layers brings its own."""
    r = run_cpp("keyset", KEYSET)
    assert r.returncode == 0, r.stdout[-2000:]


def test_sharing_wide_trees_adds_little_memory(run_cpp):
    """16384 messages of an s set with shared top layers: at most a quarter
    more scratch than with every message's own trees (a checkpoint of every
    chain of every leaf of those trees would be 18 GB and more)."""
    r = run_cpp("wide", WIDE)
    assert r.returncode == 0, r.stdout[-2000:]


def test_default_forms_bound_the_chain_ends(run_cpp):
    r = run_cpp("ends", ENDS)
    assert r.returncode == 0, r.stdout[-2000:]
