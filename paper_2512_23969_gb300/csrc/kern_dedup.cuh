// kern_dedup.cuh -- XMSS trees built once for all the messages that sign with
// them: the shared upper layers of a batch, and the layers a keyset keeps.
//
// The tree of layer j that message m signs with is fixed by (key, j,
// t_j = idx_tree >> (j h')) alone (paper Fig. 2: every layer's tree and leaf
// come from the digest), and layer j holds only 2^((d-1-j) h') trees per key
// -- the top layer is tree 0 for every message.  So the trees of the top
// layers L..D-1 are built once per key, with all their Merkle nodes and, when
// chain checkpoints are on, the checkpoints of every leaf; each message then
// copies its own auth path and root from its tree.  Every signature byte is
// the same as when each message builds its own.  Within a batch the host
// picks the layers whose trees are at most half as many as the messages
// (plan_dedup): measured on GB300, 16384 128f messages over 16 keys build
// 9360 trees in place of 65536.  All of a layer's trees are built, not only
// those the batch uses: there the unused ones are 0.4 % of the work, and the
// direct index needs no hash table.
#pragma once
#include <cuda_runtime.h>
#include "hs_common.cuh"
#include "hs_launch.h"
#include "sha256_chain.cuh"
#include "kern_tree.cuh"

namespace hs {

constexpr uint32_t kNoSlot = 0xFFFFFFFFu;

// One lane group per tree: every leaf (with all its checkpoints) and every
// Merkle node, stored heap-ordered.
template <class P, int POL>
__global__ void __launch_bounds__(128) utree_kernel(const KeyBlock* __restrict__ keys,
                                                    const DedupDesc* __restrict__ desc, uint32_t ndesc,
                                                    uint32_t* __restrict__ nodes, uint32_t* __restrict__ chk_u,
                                                    uint32_t ck, uint32_t one) {
    allow_next();
    constexpr int NW = P::NW, LV = P::LEAVES;
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t id = gid / LV;
    const uint32_t l = (uint32_t)(gid % LV);
    if (id >= ndesc) return;                         // whole trees exit together
    const unsigned gmask = ((LV == 32) ? 0xFFFFFFFFu : ((1u << LV) - 1u)) << (lane & ~(uint32_t)(LV - 1));
    const DedupDesc d = desc[id];
    const KeyBlock& kb = keys[d.key];
    uint32_t ms256[8], msT[P::BIG ? 16 : 8], skseed[NW];
#pragma unroll
    for (int w = 0; w < 8; w++) ms256[w] = kb.ms256[w];
#pragma unroll
    for (int w = 0; w < (P::BIG ? 16 : 8); w++) msT[w] = P::BIG ? kb.ms512[w] : kb.ms256[w];
#pragma unroll
    for (int w = 0; w < NW; w++) skseed[w] = kb.sk_seed[w];
    const Pipes<POL> pp(one);
    uint32_t* mychk = ck ? chk_u + ((size_t)id * LV + l) * (size_t)P::LEN * (16u / ck) * NW : nullptr;
    uint32_t node[NW];
    wots_leaf<P, POL>(ms256, msT, skseed, d.layer, d.tree, l, node, mychk, ck, pp, kb.pk_seed);
    heap_finish<P>(ms256, msT, gmask, d.layer, d.tree, l, node, nodes + (size_t)id * 2 * LV * NW, kb.pk_seed);
}

// Layer j holds 2^((D-1-j) h') trees (the possible values of
// idx_tree >> (j h')).  Trees of one key are stored top layer first, so the
// tree t of layer j has id  key * tpk + cache_off(j) + t.

// Trees of the layers above j: sum over u < D-1-j of 2^(u h').
template <class P>
__host__ __device__ __forceinline__ uint64_t cache_off(uint32_t j) {
    uint64_t off = 0;
    for (uint32_t u = 0; u + 1 + j < (uint32_t)P::D; u++) off += 1ull << (u * P::HP);
    return off;
}

// One thread per tree: its (key, layer, tree) description.
template <class P>
__global__ void cache_desc_kernel(uint32_t num_keys, uint32_t L, uint32_t tpk, DedupDesc* __restrict__ desc) {
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (uint64_t)num_keys * tpk) return;
    const uint32_t key = (uint32_t)(gid / tpk);
    uint64_t r = gid % tpk;
    uint32_t j = (uint32_t)P::D - 1;
    while (j > L && r >= (1ull << ((P::D - 1 - j) * P::HP))) {
        r -= 1ull << ((P::D - 1 - j) * P::HP);
        j--;
    }
    DedupDesc d;
    d.tree = r;
    d.layer = j;
    d.key = key;
    desc[gid] = d;
}

// One thread per (message, layer from L up): auth path and root from its tree.
template <class P>
__global__ void cache_scatter_kernel(const MsgInfo* __restrict__ infos, uint32_t count, uint32_t L, uint32_t tpk,
                                     const uint32_t* __restrict__ nodes, uint8_t* __restrict__ sigs,
                                     uint32_t* __restrict__ roots, uint32_t* __restrict__ mj_id) {
    constexpr int NW = P::NW, HP = P::HP, LV = P::LEAVES;
    const uint32_t per_msg = (uint32_t)P::D - L;
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (uint64_t)count * per_msg) return;
    const uint32_t m = (uint32_t)(gid / per_msg);
    const uint32_t j = L + (uint32_t)(gid % per_msg);
    const MsgInfo& info = infos[m];
    if (info.key == KEY_INVALID) { mj_id[gid] = kNoSlot; return; }
    const uint64_t id = (uint64_t)info.key * tpk + cache_off<P>(j) + layer_tree<P>(info.idx_tree, (int)j);
    mj_id[gid] = (uint32_t)id;
    const uint32_t sl = layer_leaf<P>(info.idx_tree, info.idx_leaf, (int)j);
    const uint32_t* tn = nodes + id * 2 * LV * NW;
    uint8_t* auth = sigs + (size_t)m * P::SIG_BYTES + P::N + P::FORS_BYTES + (size_t)j * P::LAYER_BYTES +
                    (size_t)P::LEN * P::N;
#pragma unroll
    for (int z = 0; z < HP; z++) store_be<NW>(auth + (size_t)z * P::N, tn + ((LV >> z) + ((sl >> z) ^ 1u)) * NW);
    uint32_t* rt = roots + ((size_t)m * P::D + j) * NW;
#pragma unroll
    for (int w = 0; w < NW; w++) rt[w] = tn[1 * NW + w];
}

// Key generation in its chain-parallel form: PK.root from the top trees'
// nodes (tree id = key), then pk = PK.seed || PK.root and sk = SK.seed ||
// SK.prf || PK.seed || PK.root.
template <class P>
__global__ void keygen_out_kernel(const uint8_t* __restrict__ seeds, uint32_t count,
                                  const uint32_t* __restrict__ nodes, uint8_t* __restrict__ pk,
                                  uint8_t* __restrict__ sk) {
    constexpr int NW = P::NW, N = P::N;
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;      // one byte of sk
    const uint64_t key = gid / (4 * N);
    const uint32_t b = (uint32_t)(gid % (4 * N));
    if (key >= count) return;
    const uint32_t* root = nodes + (key * 2 * P::LEAVES + 1) * NW;
    const uint32_t r = b - 3 * N;
    const uint8_t v = b < 3 * N ? seeds[key * 3 * N + b] : (uint8_t)(root[r >> 2] >> (24 - 8 * (r & 3)));
    sk[gid] = v;
    if (b >= 2 * N) pk[key * 2 * N + (b - 2 * N)] = v;
}

}  // namespace hs
