// set_impl.cuh -- host launchers of every kernel for one parameter set P.
// Each set_<name>.cu instantiates SetImpl<P> and the launch-shape variants
// the tuner may choose from, and exports them as one SetOps table.
#pragma once
#include <cuda_runtime.h>
#include "hs_launch.h"
#include "kern_msg.cuh"
#include "kern_fors.cuh"
#include "kern_tree.cuh"
#include "kern_wots.cuh"
#include "kern_verify.cuh"
#include "kern_dedup.cuh"
#include "kern_stree.cuh"

namespace hs {

// Launch on s; beside = true: the launch may start beside the previous one
// of the stream (hs_common.cuh), with the guard block that makes it end after
// it.  The kernel's last parameter is the guard's block index.
template <class... K, class... A>
inline cudaError_t launch_beside(bool beside, void (*kernel)(K...), uint32_t grid, uint32_t threads, cudaStream_t s,
                                 A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid + (beside ? 1u : 0u));
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = beside ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args..., beside ? grid : kNoGuard);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <class P>
struct SetImpl {
    // XMSS trees wider than a warp (s sets) take the two-launch form of
    // kern_stree.cuh, also for the shared and cached trees.
    static constexpr bool kWide = P::LEAVES > 32;

    // Whether a T_l launch over this many groups of 32 items runs by groups:
    // while the SMs hold them all at once.
    static bool tl_groups_pay(uint64_t groups) { return groups <= (uint64_t)kTlGroupsPerSm * sm_count(); }

    // layers each message builds itself: all of them unless the upper
    // layers are shared within the batch (dedup_layer = first shared layer)
    static uint32_t own_layers(const Batch& b) { return b.dedup_layer ? b.dedup_layer : (uint32_t)P::D; }

    static cudaError_t keyprep(const Batch& b, bool from_pk, cudaStream_t s) {
        const uint64_t threads = (uint64_t)b.num_keys * (P::BIG ? 2 : 1);
        const uint32_t T = 128, G = (uint32_t)((threads + T - 1) / T);
        keyprep_kernel<P><<<G, T, 0, s>>>(b.keys_in, b.num_keys, from_pk ? 1 : 0, b.keys);
        return cudaGetLastError();
    }
    static cudaError_t message(const Batch& b, bool verify, cudaStream_t s) {
        if constexpr (!P::SHAKE) {
            if (b.msg_warp) {                               // a warp per message
                const uint32_t T = 32 * kMsgWarpsPerBlock, G = (b.count + kMsgWarpsPerBlock - 1) / kMsgWarpsPerBlock;
                return launch_beside(b.beside, message_warp_kernel<P>, G, T, s, b.keys_in, b.num_keys, b.key_idx, b.msgs,
                                     b.lens, (const uint64_t*)(needs_offsets(b) ? b.offsets : nullptr), b.count,
                                     b.sigs, b.infos, b.status, verify ? 1 : 0, b.prefix, b.prefix_len,
                                     b.fips ? 1 : 0);
            }
        }
        const uint32_t T = 64, G = (b.count + T - 1) / T;
        message_kernel<P><<<G, T, 0, s>>>(b.keys, b.num_keys, b.key_idx, b.msgs, b.offsets, b.count, b.sigs,
                                          b.infos, b.status, verify ? 1 : 0, b.prefix, b.prefix_len,
                                          b.fips ? 1 : 0);
        return cudaGetLastError();
    }
    template <int LPT>
    static cudaError_t fors(const Batch& b, cudaStream_t s) {
        const uint64_t threads = (uint64_t)b.count * P::K * LPT;
        const uint32_t T = 256;
        const uint32_t G = (uint32_t)((threads + T - 1) / T);
        return launch_beside(b.beside, fors_kernel<P, fors_pol<P>(), LPT>, G, T, s, (const KeyBlock*)b.keys,
                             (const MsgInfo*)b.infos, b.count, b.sigs, b.fors_roots, 1u);
    }
    // The widest form (the knob's value 32 at the f sets): a thread per leaf
    // while that is the faster one, else lane groups of 32.  A block of the
    // former holds its 2^a threads' registers while a few lanes climb the
    // upper levels, so at a = 8 / 9 it pays for a few trees per SM only:
    // measured on GB300, 256f 1 message 215 -> 61 us, 96 messages 632 -> 987;
    // 192f 123 -> 47 and 360 -> 397; at a = 6 (128f) the blocks are small,
    // 30 -> 20 us and 76 -> 65.  Beside other batches (crowded) the line lies
    // at 2 trees per SM at every set: serving mix, p50 at 20k / 40k / 60k / 76k
    // requests/s 0.55 / 0.85 / 1.48 / 2.96 ms; without a line 0.55 / 0.85 /
    // 1.51 / 3.04, never a thread per leaf 0.64 / 0.94 / 1.42 / 2.94.
    static cudaError_t fors_widest(const Batch& b, cudaStream_t s) {
        constexpr int T = P::A < 7 ? 1 << (7 - P::A) : 1;          // trees per block: at least 128 threads
        const uint64_t trees = (uint64_t)b.count * P::K;
        if (b.crowded && trees > (uint64_t)sm_count() * 2) return fors<32>(b, s);
        if constexpr (P::A >= 8) {
            if (trees > (uint64_t)sm_count() * (P::A == 8 ? 6 : 4)) return fors<32>(b, s);
        }
        return launch_beside(b.beside, fors_wide_kernel<P, fors_pol<P>(), T>, (uint32_t)((trees + T - 1) / T), T << P::A,
                             s, (const KeyBlock*)b.keys, (const MsgInfo*)b.infos, b.count, b.sigs, b.fors_roots, 1u);
    }
    // T_k has no climbs behind it, so its groups pay a little beyond what the
    // SMs hold at once (robust sets: no further, the mask is hashed by the
    // group's warps in turn).  Measured on GB300, groups / a thread per message
    // (us): 128f 24352 messages 37 / 43, 32768 45 / 47, 65536 74 / 68, 131072
    // 131 / 109; 192f 24352 59 / 78, 49152 109 / 102; 256f 24352 82 / 100,
    // 49152 150 / 137; robust-256f 24352 263 / 242.
    static cudaError_t fors_pk(const Batch& b, cudaStream_t s) {
        const uint32_t G = (b.count + 31) / 32;
        if (!b.crowded && G <= (P::ROBUST ? kTlGroupsPerSm : 7u) * (uint32_t)sm_count())
            return launch_beside(b.beside, fors_pk_kernel<P, true>, G, TlShape<P>::THREADS, s, (const KeyBlock*)b.keys,
                                 (const MsgInfo*)b.infos, b.count, b.fors_roots, b.pk_fors);
        return launch_beside(b.beside, fors_pk_kernel<P, false>, (b.count + 127) / 128, 128u, s, (const KeyBlock*)b.keys,
                             (const MsgInfo*)b.infos, b.count, b.fors_roots, b.pk_fors);
    }
    template <int MINB, int POL = tree_pol<P>(), int ILP = 1>
    static cudaError_t tree(const Batch& b, BesideFn beside, cudaStream_t s) {
        const uint32_t L = own_layers(b);
        const uint64_t threads = (uint64_t)b.count * L * P::LEAVES;
        const uint32_t T = 128;
        const uint32_t G = (uint32_t)((threads + T - 1) / T);
        if (threads == 0) return cudaSuccess;
        // the shared trees first; the messages' own start beside them, as their
        // last wave is far from full
        cudaError_t e = describe_shared(b, s);
        if (e == cudaSuccess && b.max_uniq) e = build_leaves(b.keys, b.desc, b.max_uniq, b.nodes_u, b.chk_u, b.ck, s);
        if (e != cudaSuccess) return e;
        const bool own_beside = beside != nullptr && b.max_uniq != 0;
        if constexpr (kWide) {
            e = launch_beside(own_beside, bleaf_kernel<P, POL, MINB, ILP>, G, T, s, (const KeyBlock*)b.keys,
                              (const MsgInfo*)b.infos, b.count, b.leafv, b.chk, b.ck, L, 1u);
            if (e == cudaSuccess && beside) e = beside(b, 0, s);
            if (e == cudaSuccess) e = build_merge(b.keys, b.desc, b.max_uniq, b.nodes_u, s);
            if (e == cudaSuccess) e = merge(b, s);
            if (e == cudaSuccess && beside) e = beside(b, 1, s);
        } else {
            e = launch_beside(own_beside, tree_kernel<P, POL, MINB, ILP>, G, T, s, (const KeyBlock*)b.keys,
                              (const MsgInfo*)b.infos, b.count, b.sigs, b.roots, b.chk, b.ck, L, 1u);
            if (e == cudaSuccess && beside) e = beside(b, 0, s);
            if (e == cudaSuccess && beside) {           // T_k reads what the launch before it writes
                Batch after = b;
                after.beside = false;
                e = beside(after, 1, s);
            }
        }
        return e;
    }
    // The descriptions of the trees this call builds for several messages.
    static cudaError_t describe_shared(const Batch& b, cudaStream_t s) {
        if (b.max_uniq == 0) return cudaSuccess;
        cache_desc_kernel<P><<<(b.max_uniq + 127) / 128, 128, 0, s>>>(b.num_keys, own_layers(b), b.cache_tpk, b.desc);
        return cudaGetLastError();
    }
    // Wide trees: one block per (message, layer) merges the stored leaves.
    static cudaError_t merge(const Batch& b, cudaStream_t s) {
        const uint32_t L = own_layers(b);
        const uint64_t blocks = (uint64_t)b.count * L;
        if (blocks == 0) return cudaSuccess;
        bmerkle_kernel<P><<<(uint32_t)blocks, kMergeThreads, 0, s>>>(b.keys, b.infos, b.count, b.leafv, b.sigs,
                                                                     b.roots, L);
        return cudaGetLastError();
    }
    // The ndesc trees of desc, all nodes and the checkpoints of every leaf: a
    // thread per leaf; wide trees leave the levels above to build_merge.
    static cudaError_t build_leaves(const KeyBlock* keys, const DedupDesc* desc, uint32_t ndesc, uint32_t* nodes,
                                    uint32_t* chk, uint32_t ck, cudaStream_t s) {
        const uint32_t T = 128;
        const uint64_t th = (uint64_t)ndesc * P::LEAVES;
        if (th == 0) return cudaSuccess;
        const uint32_t G = (uint32_t)((th + T - 1) / T);
        if constexpr (kWide)
            wtree_leaf_kernel<P, tree_pol<P>()><<<G, T, 0, s>>>(keys, desc, ndesc, nodes, chk, ck, 1u);
        else
            utree_kernel<P, tree_pol<P>()><<<G, T, 0, s>>>(keys, desc, ndesc, nodes, chk, ck, 1u);
        return cudaGetLastError();
    }
    static cudaError_t build_merge(const KeyBlock* keys, const DedupDesc* desc, uint32_t ndesc, uint32_t* nodes,
                                   cudaStream_t s) {
        if constexpr (kWide) {
            if (ndesc) wtree_merge_kernel<P><<<ndesc, kMergeThreads, 0, s>>>(keys, desc, ndesc, nodes);
        }
        return cudaGetLastError();
    }
    // Shared or cached top layers: auth paths, roots and tree ids from their nodes.
    static cudaError_t tree_shared(const Batch& b, cudaStream_t s) {
        const uint32_t T = 128, L = own_layers(b);
        const uint64_t mj = (uint64_t)b.count * (P::D - L);
        if (mj == 0) return cudaSuccess;
        cache_scatter_kernel<P><<<(uint32_t)((mj + T - 1) / T), T, 0, s>>>(b.infos, b.count, L, b.cache_tpk,
                                                                           b.nodes_u, b.sigs, b.roots, b.mj_id);
        return cudaGetLastError();
    }
    // Build every tree of layers L..D-1 of num_keys resident keys.
    static cudaError_t cache_build(const KeyBlock* keys, uint32_t num_keys, uint32_t L, uint32_t tpk,
                                   DedupDesc* desc, uint32_t* nodes, uint32_t* chk, uint32_t ck, cudaStream_t s) {
        const uint32_t T = 128;
        const uint64_t trees = (uint64_t)num_keys * tpk;
        if (trees == 0) return cudaSuccess;
        cache_desc_kernel<P><<<(uint32_t)((trees + T - 1) / T), T, 0, s>>>(num_keys, L, tpk, desc);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        e = build_leaves(keys, desc, (uint32_t)trees, nodes, chk, ck, s);
        return e == cudaSuccess ? build_merge(keys, desc, (uint32_t)trees, nodes, s) : e;
    }
    // Chain-parallel form: the messages' own trees and the ndesc trees of
    // desc in the same launches (either may be none).  T_len's launch starts
    // after FORS_Sign's (it waits for the whole stream), so T_k beside it
    // finds the FORS roots complete.
    static cudaError_t split_trees(const KeyBlock* keys, const MsgInfo* infos, uint32_t count, uint32_t L,
                                   uint32_t* ends, uint32_t* chk, uint32_t ck, const DedupDesc* desc, uint32_t ndesc,
                                   uint32_t* nodes_u, uint32_t* chk_u, uint32_t* leafv, uint8_t* sigs,
                                   uint32_t* roots, const Batch* b, BesideFn beside, cudaStream_t s) {
        const uint32_t T = 128;
        const uint64_t own = (uint64_t)count * L * P::LEAVES, shared = (uint64_t)ndesc * P::LEAVES;
        const uint64_t chains = (own + shared) * P::LEN;
        if (chains == 0) return cudaSuccess;
        chains_kernel<P, tree_pol<P>()><<<(uint32_t)((chains + T - 1) / T), T, 0, s>>>(
            keys, infos, count, ends, chk, ck, L, desc, ndesc, chk_u, 1u);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess && beside) e = beside(*b, 0, s);
        if (e != cudaSuccess) return e;
        const bool group = !(b && b->crowded) && tl_groups_pay((own + 31) / 32 + (shared + 31) / 32);
        const uint32_t per = group ? 32 : 128, TL = group ? TlShape<P>::THREADS : 128;
        const uint32_t G = (uint32_t)((own + per - 1) / per + (shared + per - 1) / per);
        if constexpr (kWide) {
            if (group)
                bleaf_from_ends_kernel<P, true><<<G, TL, 0, s>>>(keys, infos, count, ends, leafv, L, desc, ndesc, nodes_u);
            else
                bleaf_from_ends_kernel<P, false><<<G, TL, 0, s>>>(keys, infos, count, ends, leafv, L, desc, ndesc, nodes_u);
            e = cudaGetLastError();
            if (e == cudaSuccess && beside) e = beside(*b, 1, s);
            if (e != cudaSuccess || ndesc == 0) return e;
            wtree_merge_kernel<P><<<ndesc, kMergeThreads, 0, s>>>(keys, desc, ndesc, nodes_u);
            return cudaGetLastError();
        } else {
            if (group)
                leaves_kernel<P, true><<<G, TL, 0, s>>>(keys, infos, count, ends, sigs, roots, L, desc, ndesc, nodes_u);
            else
                leaves_kernel<P, false><<<G, TL, 0, s>>>(keys, infos, count, ends, sigs, roots, L, desc, ndesc, nodes_u);
            e = cudaGetLastError();
            return e == cudaSuccess && beside ? beside(*b, 1, s) : e;
        }
    }
    static cudaError_t tree_split(const Batch& b, BesideFn beside, cudaStream_t s) {
        cudaError_t e = describe_shared(b, s);
        if (e == cudaSuccess)
            e = split_trees(b.keys, b.infos, b.count, own_layers(b), b.ends, b.chk, b.ck, b.desc, b.max_uniq,
                            b.nodes_u, b.chk_u, b.leafv, b.sigs, b.roots, &b, beside, s);
        if constexpr (kWide) {
            if (e == cudaSuccess) e = merge(b, s);
        }
        return e;
    }
    static cudaError_t wots(const Batch& b, cudaStream_t s) {
        const uint64_t threads = (uint64_t)b.count * P::D * P::LEN;
        const uint32_t T = 256;
        const uint32_t G = (uint32_t)((threads + T - 1) / T);
        wots_kernel<P, kChainPol><<<G, T, 0, s>>>(b.keys, b.infos, b.count, b.pk_fors, b.roots, b.sigs, b.chk,
                                                   b.ck, own_layers(b), b.mj_id, b.chk_u, 1u);
        return cudaGetLastError();
    }
    // Few signatures: the chain ends for every digit, the FORS roots beside
    // them, then one walk over the layers (scratch: fors_roots, vends, ends).
    static cudaError_t verify_few(const Batch& b, cudaStream_t s) {
        const uint32_t T = 128;
        const uint64_t ct = (uint64_t)b.count * P::D * P::LEN * 16, ft = (uint64_t)b.count * P::K;
        vspec_kernel<P, kChainPol><<<(uint32_t)((ct + T - 1) / T), T, 0, s>>>(b.keys, b.infos, b.count, b.sigs, b.vends,
                                                                              1u);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess)
            e = launch_beside(can_overlap(s), vfors_kernel<P>, (uint32_t)((ft + T - 1) / T), T, s, (const KeyBlock*)b.keys,
                              (const MsgInfo*)b.infos, b.count, (const uint8_t*)b.sigs, b.fors_roots);
        if (e != cudaSuccess) return e;
        vwalk_kernel<P><<<(b.count + 31) / 32, kWalkThreads, 0, s>>>(b.keys, b.infos, b.count, b.sigs, b.vends, b.ends,
                                                                     b.fors_roots, b.ok);
        return cudaGetLastError();
    }
    // Verification: FORS roots, PK_FORS, then per layer chains and T_len +
    // climbs (layers are serial), then the comparison with PK.root.  The
    // layer messages live in pk_fors (layer 0) and roots (layers >= 1).
    // Scratch: fors_roots, pk_fors, roots (root_j of the current layer),
    // ends (chain ends of one layer), vcnt (16 step buckets per layer),
    // vsitem / vorder (one word per chain of a layer).
    static cudaError_t verify(const Batch& b, cudaStream_t s) {
        if (b.walk) return verify_few(b, s);
        const uint32_t T = 128;
        cudaError_t e = cudaMemsetAsync(b.vcnt, 0, sizeof(uint32_t) * 16 * P::D, s);
        const uint64_t ft = (uint64_t)b.count * P::K;
        if (e == cudaSuccess) {
            vfors_kernel<P><<<(uint32_t)((ft + T - 1) / T), T, 0, s>>>(b.keys, b.infos, b.count, b.sigs,
                                                                       b.fors_roots, kNoGuard);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = fors_pk(b, s);
        const uint64_t ct = (uint64_t)b.count * P::LEN;
        const uint32_t G1 = (b.count + T - 1) / T, G32 = (b.count + 31) / 32;
        if (e == cudaSuccess) {
            vcount0_kernel<P><<<G32, T, 0, s>>>(b.infos, b.count, b.pk_fors, b.vcnt, b.vsitem);
            e = cudaGetLastError();
        }
        for (uint32_t j = 0; j < (uint32_t)P::D && e == cudaSuccess; j++) {
            vscatter_kernel<P><<<(uint32_t)((ct + 255) / 256), 256, 0, s>>>(b.count, b.vcnt + 16 * j, b.vsitem,
                                                                            b.vorder);
            if ((e = cudaGetLastError()) != cudaSuccess) break;
            vchain_kernel<P, kChainPol><<<(uint32_t)((ct + T - 1) / T), T, 0, s>>>(
                b.keys, b.infos, b.count, b.sigs, b.vorder, b.vsitem, b.ends, j, 1u);
            if ((e = cudaGetLastError()) != cudaSuccess) break;
            uint32_t* next = j + 1 < (uint32_t)P::D ? b.vcnt + 16 * (j + 1) : nullptr;
            if (tl_groups_pay(G32))
                vleaf_kernel<P, true><<<G32, TlShape<P>::THREADS, 0, s>>>(b.keys, b.infos, b.count, b.sigs, b.ends,
                                                                          b.roots, j, next, b.vsitem);
            else
                vleaf_kernel<P, false><<<G32, 32, 0, s>>>(b.keys, b.infos, b.count, b.sigs, b.ends, b.roots, j, next,
                                                          b.vsitem);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return e;
        vfinal_kernel<P><<<G1, T, 0, s>>>(b.keys, b.infos, b.count, b.roots, b.ok);
        return cudaGetLastError();
    }
    // split: chain-parallel, one XMSS tree per key as the trees of desc.
    static cudaError_t keygen(const uint8_t* seeds, uint32_t count, uint8_t* pk, uint8_t* sk, bool split,
                              cudaStream_t s) {
        const uint64_t threads = (uint64_t)count * P::LEAVES;
        const uint32_t T = 128;
        const uint32_t G = (uint32_t)((threads + T - 1) / T);
        if (!kWide && !split) {
            if constexpr (!kWide) keygen_kernel<P><<<G, T, 0, s>>>(seeds, count, pk, sk, 1u);
            return cudaGetLastError();
        }
        auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
        const size_t kb_bytes = al((size_t)count * sizeof(KeyBlock));
        const size_t node_bytes = al((split ? 2 : 1) * threads * P::NW * 4);      // heap, or the leaves alone
        const size_t desc_bytes = split ? al((size_t)count * sizeof(DedupDesc)) : 0;
        const size_t end_bytes = split ? threads * P::LEN * P::NW * 4 : 0;
        void* scratch = nullptr;
        cudaError_t e = pool_alloc(&scratch, kb_bytes + node_bytes + desc_bytes + end_bytes, s);
        if (e == cudaErrorMemoryAllocation && split) {       // the chain ends are extra scratch
            cudaGetLastError();
            return keygen(seeds, count, pk, sk, false, s);
        }
        if (e != cudaSuccess) return e;
        KeyBlock* kbs = static_cast<KeyBlock*>(scratch);
        char* at = static_cast<char*>(scratch) + kb_bytes;
        uint32_t* nodes = reinterpret_cast<uint32_t*>(at);
        seed_keys_kernel<P><<<(count + T - 1) / T, T, 0, s>>>(seeds, count, kbs);
        e = cudaGetLastError();
        if (split) {
            DedupDesc* desc = reinterpret_cast<DedupDesc*>(at + node_bytes);
            uint32_t* ends = reinterpret_cast<uint32_t*>(at + node_bytes + desc_bytes);
            if (e == cudaSuccess) {
                cache_desc_kernel<P><<<(count + T - 1) / T, T, 0, s>>>(count, (uint32_t)P::D - 1, 1u, desc);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess)
                e = split_trees(kbs, nullptr, 0, 0, ends, nullptr, 0, desc, count, nodes, nullptr, nullptr, nullptr,
                                nullptr, nullptr, nullptr, s);
            if (e == cudaSuccess) {
                const uint64_t bytes = (uint64_t)count * 4 * P::N;
                keygen_out_kernel<P><<<(uint32_t)((bytes + T - 1) / T), T, 0, s>>>(seeds, count, nodes, pk, sk);
                e = cudaGetLastError();
            }
        } else if constexpr (kWide) {       // top-tree leaves, then one block per key for the root
            if (e == cudaSuccess) {
                bkeygen_leaf_kernel<P, kChainPol><<<G, T, 0, s>>>(kbs, count, nodes, 1u);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess) {
                bkeygen_root_kernel<P><<<count, kMergeThreads, 0, s>>>(kbs, seeds, count, nodes, pk, sk);
                e = cudaGetLastError();
            }
        }
        const cudaError_t f = cudaFreeAsync(scratch, s);
        return e == cudaSuccess ? f : e;
    }
};

// The compiled variants of TREE_Sign's per-leaf kernel for one set, as
// (min blocks per SM, addition policy, chains per thread): the default
// (0, tree_pol<P>(), 1); the other addition policy and two interleaved
// chains per thread (simple SHA-2 sets other than toy); and MB_ALT min blocks
// (0 = none) -- each alternative with the other two at their defaults.
template <class P, int MB_ALT>
struct TreeVariants {
    static constexpr int PD = tree_pol<P>();
    static constexpr bool kAlts = !P::SHAKE && !P::ROBUST && P::LEAVES >= 8;   // simple SHA-2, not toy
    static constexpr int PA = PD == 7 ? 15 : 7;
    static bool has(int minb, int pol, int ilp) {
        if (minb == 0 && pol == PD && ilp == 1) return true;
        if (MB_ALT != 0 && minb == MB_ALT && pol == PD && ilp == 1) return true;
        return kAlts && minb == 0 && ((pol == PA && ilp == 1) || (pol == PD && ilp == 2));
    }
    static cudaError_t run(const Batch& b, int minb, int pol, int ilp, BesideFn beside, cudaStream_t s) {
        if (minb == 0 && pol == PD && ilp == 1) return SetImpl<P>::template tree<1, PD, 1>(b, beside, s);
        if constexpr (MB_ALT != 0)
            if (minb == MB_ALT && pol == PD && ilp == 1) return SetImpl<P>::template tree<MB_ALT, PD, 1>(b, beside, s);
        if constexpr (kAlts) {
            if (minb == 0 && pol == PA && ilp == 1) return SetImpl<P>::template tree<1, PA, 1>(b, beside, s);
            if (minb == 0 && pol == PD && ilp == 2) return SetImpl<P>::template tree<1, PD, 2>(b, beside, s);
        }
        return cudaErrorInvalidValue;
    }
};

}  // namespace hs
