// dispatch.cu -- routes each launch to the parameter set's table with the
// tuned launch shape (see hs_tune_set in include/hs.h).
#include <algorithm>
#include <atomic>
#include "hs_launch.h"

namespace hs {

const SetOps* set_ops(int pset) {
    switch (pset) {
    case 0: return &kOps_128F;
    case 1: return &kOps_192F;
    case 2: return &kOps_256F;
    case 3: return &kOps_Toy;
    case 4: return &kOps_128S;
    case 5: return &kOps_192S;
    case 6: return &kOps_256S;
    case 7: return &kOps_K128F;
    case 8: return &kOps_K192F;
    case 9: return &kOps_K256F;
    case 10: return &kOps_K128S;
    case 11: return &kOps_K192S;
    case 12: return &kOps_K256S;
    case 13: return &kOps_R128F;
    case 14: return &kOps_R192F;
    case 15: return &kOps_R256F;
    }
    return nullptr;
}

namespace {
// -1 = not set: use the table's default (knob 5: the process-wide stride).
struct TuneSlots {
    std::atomic<int> v[kNumSets][kNumKnobs];
    TuneSlots() {
        for (auto& row : v)
            for (auto& x : row) x.store(-1);
    }
};
TuneSlots g_slots;
auto& g_tune = g_slots.v;
std::atomic<int> g_ck_default{2};
// TREE_Sign's form without a tuned cache, per set, as measured on GB300: the
// batch size below which it runs chain-parallel (chain-parallel / per leaf,
// ms: 128f 1024 messages 5.84 / 5.87, 2048 11.63 / 11.12; 192f 256 2.54 /
// 2.71, 1024 9.99 / 8.88; 256f 32 0.76 / 1.27, 64 1.46 / 1.26), and above that
// the cost model's coefficients (split_faster below).  At the SHAKE and robust
// f sets the chain-parallel form is ahead at every size measured (TREE_Sign,
// ms: shake-256f 4096 226 / 232, 8192 437 / 442; robust-256f 4096 193 / 215),
// but for 0.3 - 2.5 % at robust-192f between 512 and 2048 messages, so there the line bounds its scratch: the chain ends (98, 215 and 583 KB a
// message) stay at 2.4 GB or less.
constexpr int kSplitDefault[kNumSets] = {1024, 256, 64, 0, 16, 16, 0, 16384, 8192, 4096, 256, 256, 256,
                                         16384, 8192, 4096};
constexpr int kStepUsDefault[kNumSets] = {637, 958, 1262, 0, 655, 1015, 1300, 2379, 3510, 4615, 2414, 3534, 4635,
                                          2379, 3606, 6405};
constexpr int kSplitNsDefault[kNumSets] = {5741, 9833, 22514, 0, 116992, 197938, 167196, 20966, 30673, 62918,
                                           425882, 626482, 473714, 11576, 17815, 54806};
constexpr int kStrides[] = {0, 1, 2, 4, 8};
// Default batch size below which the message stage runs a warp per message
// (SHA-2 sets; the SHAKE sets always run a thread per message): up to two warps
// per SM sub-partition, 1216 messages.  The warp form is then ahead at every
// length; with a third, long messages wait for issue slots (every lane runs
// the rounds), while the thread form leaves most of them free.  Measured on GB300, whole calls of
// messages of one length, thread / warp form (ms): 128f 32 bytes 1200 messages
// 6.53 / 6.43, 2047 10.69 / 10.66; 64 KB 1200 10.86 / 10.24, 1500 12.46 /
// 13.36, 2047 15.29 / 18.06 (verification 4.15 / 5.51); 192f 64 KB 1200 17.4 /
// 16.7, 1500 20.3 / 21.6, 2047 25.7 / 29.3; 256f 64 KB 1200 31.0 / 30.3, 2047
// 47.9 / 51.6.
constexpr int kMsgWarpDefault[kNumSets] = {1217, 1217, 1217, 1217, 1217, 1217, 1217, 0, 0, 0, 0, 0, 0,
                                           1217, 1217, 1217};
bool is_shake(int pset) { return pset >= 7 && pset <= 12; }
}

int tune_get(int pset, int knob) {
    const SetOps* o = set_ops(pset);
    if (!o || knob < 0 || knob >= kNumKnobs) return -1;
    const int v = g_tune[pset][knob].load();
    if (v >= 0) return v;
    switch (knob) {
    case 0: return o->fors_lpt_default;
    case 1: return o->tree_minb_default;
    case 2: return kSplitDefault[pset];
    case 3: return o->tree_pol_default;
    case 4: return 1;
    case 5: return g_ck_default.load();
    case 8: return kMsgWarpDefault[pset];
    case 6: return kStepUsDefault[pset];
    case 7: return kSplitNsDefault[pset];
    default: return 0;
    }
}

uint32_t chain_checkpoint_stride(int pset) {
    const int v = tune_get(pset, 5);
    return v < 0 ? (uint32_t)g_ck_default.load() : (uint32_t)v;
}

void set_default_checkpoint(uint32_t stride) {
    g_ck_default.store((int)stride);
    for (auto& row : g_tune) row[5].store(-1);       // one stride for every set again
}

int tune_options(int pset, int knob, int32_t* values, int max) {
    const SetOps* o = set_ops(pset);
    if (!o || knob < 0 || knob >= kNumKnobs) return -1;
    int32_t buf[16];
    int n = 0;
    switch (knob) {
    case 0: for (int i = 0; i < o->n_fors_lpt; i++) buf[n++] = o->fors_lpt[i]; break;
    case 1: for (int i = 0; i < o->n_tree_minb; i++) buf[n++] = o->tree_minb[i]; break;
    case 2: for (int v : {0, 16, 64, 256, 512, 1024, 2048, 4096, 8192, 16384}) buf[n++] = v; break;   // suggestions: any value works
    case 3: for (int v : {7, 15}) if (o->tree_has(0, v, 1)) buf[n++] = v; break;
    case 4: for (int v : {1, 2}) if (o->tree_has(0, o->tree_pol_default, v)) buf[n++] = v; break;
    case 5: for (int v : kStrides) buf[n++] = v; break;
    case 8:                             // suggestions: any value works (SHAKE sets: 0 only)
        if (is_shake(pset)) buf[n++] = 0;
        else for (int v : {0, 64, 256, 512, 1024, 1217, 2048, 4096}) buf[n++] = v;
        break;
    default:                            // 6, 7: measured coefficients, any value >= 0
        buf[n++] = 0;
        if (const int d = knob == 6 ? kStepUsDefault[pset] : kSplitNsDefault[pset]) buf[n++] = d;
        break;
    }
    for (int i = 0; i < n && i < max; i++)
        if (values) values[i] = buf[i];
    return n;
}

// The two forms of building XMSS trees.  A thread per leaf: the time is a
// staircase -- one warp per SM sub-partition already keeps the ALU pipe
// busy, so it takes about step_us x ceil(warps / sub-partitions).
// Chain-parallel: it grows with the trees (split_ns per message's d trees).
// True if the second is predicted faster.
static bool split_faster(int pset, const SetShape& sh, uint64_t trees, uint64_t max_steps) {
    const int step_us = tune_get(pset, 6), split_ns = tune_get(pset, 7);
    if (step_us <= 0 || split_ns <= 0) return false;
    const uint64_t warps = (trees * sh.leaves + 31) / 32, smsp = 4ull * (uint64_t)sm_count();
    const uint64_t steps = (warps + smsp - 1) / smsp;
    if (steps > max_steps) return false;
    return (uint64_t)split_ns * trees / sh.d < (uint64_t)step_us * 1000ull * steps;
}

bool tree_split(int pset, uint32_t count) {
    const int below = tune_get(pset, 2);
    if (below > 0 && count < (uint32_t)below) return true;
    // Above the threshold: within the first few steps, where a batch just
    // past a step wastes most of its last one, take the form predicted faster.
    SetShape sh{};
    return set_shape(pset, &sh) && split_faster(pset, sh, (uint64_t)count * sh.d, 4);
}

// Key generation builds one tree per key.
bool keygen_split(int pset, uint32_t count) {
    SetShape sh{};
    return set_shape(pset, &sh) && split_faster(pset, sh, count, 4);
}

bool msg_warp(int pset, uint32_t count) {
    return !is_shake(pset) && count < (uint32_t)std::max(0, tune_get(pset, 8));
}

// Verification: the walk over every digit's chain ends runs 16 times the
// chain steps in parallel in place of d serial chain launches, so it pays up
// to a number of chains per layer that hardly depends on the set.  Measured
// on GB300, walk against layer by layer (us): 128f 1 signature 536 / 1129,
// 96 1064 / 1153, 128 1227 / 1151; 256f 1 1413 / 1971, 64 2101 / 2118, 96
// 2367 / 2116; 128s 96 474 / 491, 128 527 / 491; shake-128f 64 2475 / 2957,
// 96 3089 / 2956.
bool verify_walk(int pset, uint32_t count) {
    SetShape sh{};
    if (!set_shape(pset, &sh)) return false;
    return (uint64_t)count * (2 * sh.n + 3) <= (is_shake(pset) ? 3000u : 3500u);
}

// SM count of the current device (looked up once per device).
int sm_count() {
    static std::atomic<int> cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 152;
    }
    int v = cache[dev].load();
    if (v > 0) return v;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
        cudaGetLastError();
        return 152;
    }
    cache[dev].store(v);
    return v;
}

int fors_lanes(int pset, uint32_t count) {
    const SetOps* o = set_ops(pset);
    SetShape sh{};
    if (!o || !set_shape(pset, &sh)) return -1;
    int lpt = tune_get(pset, 0);
    const uint64_t want = (uint64_t)sm_count() * 1024;
    while ((uint64_t)count * sh.k * lpt < want) {
        int wider = 0;                    // smallest compiled value above lpt
        for (int i = 0; i < o->n_fors_lpt; i++)
            if (o->fors_lpt[i] > lpt && (wider == 0 || o->fors_lpt[i] < wider)) wider = o->fors_lpt[i];
        if (wider == 0) break;
        lpt = wider;
    }
    return lpt;
}

bool tune_set(int pset, int knob, int value) {
    const SetOps* o = set_ops(pset);
    if (!o || knob < 0 || knob >= kNumKnobs) return false;
    if (knob == 2 || knob == 6 || knob == 7 || knob == 8) {   // batch-size thresholds, cost coefficients
        if (value < 0 || (knob == 8 && value > 0 && is_shake(pset))) return false;
        g_tune[pset][knob].store(value);
        return true;
    }
    if (knob == 1 || knob == 3 || knob == 4) {   // a compiled TREE_Sign combination
        int t[3] = {tune_get(pset, 1), tune_get(pset, 3), tune_get(pset, 4)};
        t[knob == 1 ? 0 : (knob == 3 ? 1 : 2)] = value;
        if (!o->tree_has(t[0], t[1], t[2])) return false;
        g_tune[pset][knob].store(value);
        return true;
    }
    int32_t opts[16];
    const int n = tune_options(pset, knob, opts, 16);
    for (int i = 0; i < n; i++)
        if (opts[i] == value) {
            g_tune[pset][knob].store(value);
            return true;
        }
    return false;
}

cudaError_t launch_keyprep(const Batch& b, bool from_pk, cudaStream_t s) {
    const SetOps* o = set_ops(b.pset);
    return o ? o->keyprep(b, from_pk, s) : cudaErrorInvalidValue;
}
cudaError_t launch_message(const Batch& b, bool verify, cudaStream_t s) {
    const SetOps* o = set_ops(b.pset);
    return o ? o->message(b, verify, s) : cudaErrorInvalidValue;
}
cudaError_t launch_fors(const Batch& b, cudaStream_t s) {
    const SetOps* o = set_ops(b.pset);
    return o ? o->fors(b, fors_lanes(b.pset, b.count), s) : cudaErrorInvalidValue;
}
cudaError_t launch_fors_pk(const Batch& b, cudaStream_t s) {
    const SetOps* o = set_ops(b.pset);
    return o ? o->fors_pk(b, s) : cudaErrorInvalidValue;
}
static cudaError_t tree_beside(const Batch& b, BesideFn beside, cudaStream_t s) {
    const SetOps* o = set_ops(b.pset);
    if (!o) return cudaErrorInvalidValue;
    // The shared layers' auth paths and roots: from a keyset's prebuilt trees
    // first, where the small launch runs while other batches fill the GPU;
    // behind the trees it lengthened the batch's serial end (serving mix, 2
    // cached layers, 87.5k requests/s: p50 4.8 ms behind, 3.95 first).
    cudaError_t e = b.cached ? o->tree_shared(b, s) : cudaSuccess;
    if (e == cudaSuccess)
        e = b.split ? o->tree_split(b, beside, s)
                    : o->tree(b, tune_get(b.pset, 1), tune_get(b.pset, 3), tune_get(b.pset, 4), beside, s);
    if (e == cudaSuccess && b.dedup_layer && !b.cached) e = o->tree_shared(b, s);
    return e;
}
cudaError_t launch_tree(const Batch& b, cudaStream_t s) { return tree_beside(b, nullptr, s); }
static bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) == cudaSuccess) return cap != cudaStreamCaptureStatusNone;
    cudaGetLastError();
    return true;
}
bool can_overlap(cudaStream_t s) { return !capturing(s); }
cudaError_t launch_prep(const Batch& b, bool verify, cudaStream_t s) {
    cudaError_t e = launch_keyprep(b, verify, s);
    if (needs_offsets(b) || !can_overlap(s)) {
        if (e == cudaSuccess) e = launch_offsets(b, s);
        return e == cudaSuccess ? launch_message(b, verify, s) : e;
    }
    Batch c = b;                          // the warp form reads the keys themselves
    c.beside = true;
    return e == cudaSuccess ? launch_message(c, verify, s) : e;
}
cudaError_t launch_sign_trees(const Batch& b, cudaStream_t s) {
    if (b.crowded || !can_overlap(s)) {
        cudaError_t e = launch_fors(b, s);
        if (e == cudaSuccess) e = launch_fors_pk(b, s);
        return e == cudaSuccess ? launch_tree(b, s) : e;
    }
    Batch c = b;
    c.beside = true;
    return tree_beside(c, [](const Batch& x, int stage, cudaStream_t st) {
        return stage == 0 ? launch_fors(x, st) : launch_fors_pk(x, st);
    }, s);
}
cudaError_t launch_wots(const Batch& b, cudaStream_t s) {
    const SetOps* o = set_ops(b.pset);
    return o ? o->wots(b, s) : cudaErrorInvalidValue;
}
cudaError_t launch_verify(const Batch& b, cudaStream_t s) {
    const SetOps* o = set_ops(b.pset);
    return o ? o->verify(b, s) : cudaErrorInvalidValue;
}
cudaError_t launch_keygen(int pset, const uint8_t* seeds, uint32_t count, uint8_t* pk, uint8_t* sk,
                          cudaStream_t s) {
    const SetOps* o = set_ops(pset);
    // The chain-parallel form allocates.  In a captured graph that would be
    // an allocation node, and such a graph cannot be instantiated twice, cloned
    // or used as a child: there a thread per leaf (at the f sets one kernel and
    // no allocation).
    return o ? o->keygen(seeds, count, pk, sk, keygen_split(pset, count) && !capturing(s), s) : cudaErrorInvalidValue;
}

}  // namespace hs
