// kern_verify.cuh -- batched signature verification on the GPU.
//
// The scheme's verification (the paper signs only; this is the definition's
// inverse of Fig. 2): PK_FORS from the FORS signature (leaf from the
// revealed secret, a climbs with the auth path, T_k over the roots), then
// for each layer j the WOTS+ public key from the signature of msg_j (chain i
// advanced from digit_i to w-1), T_len, and h' climbs with the auth path to
// root_j = msg_{j+1}.  Valid iff root_{d-1} equals PK.root.
//
// GB300 mapping: verification is serial across layers (layer j's digits
// come from root_{j-1}), but a batch has count x len independent chains in
// every layer.  So: one thread per (message, FORS tree) for the FORS roots
// (then the signer's T_k kernel for PK_FORS); then for each layer one
// thread per (message, chain) advancing its chain to the end, and a block
// per 32 messages for T_len and the h' climbs, which leaves root_j in
// scratch for the next layer; finally a comparison with PK.root.
// A chain needs w - 1 - digit steps (0 .. 15), so a warp of chains in
// message order waits for its longest.  The chains of a layer are
// therefore bucketed by their step count (the block that produced msg_j
// counts its messages' digits), scattered longest first, and the chain
// kernel runs them in that order: the chains of a warp then have the same
// length.  Few signatures take another form (vwalk_kernel).
#pragma once
#include <cuda_runtime.h>
#include "hs_common.cuh"
#include "hs_launch.h"
#include "sha256_chain.cuh"
#include "kern_tl.cuh"

namespace hs {

// FORS root i of message m from the signature: leaf from the revealed
// secret, a climbs with the auth path.
template <class P>
__global__ void __launch_bounds__(128) vfors_kernel(const KeyBlock* __restrict__ keys,
                                                    const MsgInfo* __restrict__ infos, uint32_t count,
                                                    const uint8_t* __restrict__ sigs,
                                                    uint32_t* __restrict__ fors_roots, uint32_t guard) {
    if (blockIdx.x == guard) { wait_previous(); return; }
    constexpr int NW = P::NW, A = P::A, K = P::K;
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t m = gid / K;
    const uint32_t i = (uint32_t)(gid % K);
    if (m >= count) return;
    const MsgInfo& info = infos[m];
    if (info.key == KEY_INVALID) return;
    const KeyBlock& kb = keys[info.key];
    uint32_t ms256[8], msT[P::BIG ? 16 : 8];
#pragma unroll
    for (int w = 0; w < 8; w++) ms256[w] = kb.ms256[w];
#pragma unroll
    for (int w = 0; w < (P::BIG ? 16 : 8); w++) msT[w] = P::BIG ? kb.ms512[w] : kb.ms256[w];
    const uint8_t* s = sigs + (size_t)m * P::SIG_BYTES + P::N + (size_t)i * (A + 1) * P::N;
    const uint32_t g = (i << A) + info.fors_idx[i];
    uint32_t sk[NW], node[NW];
    load_be<NW>(s, sk);
    hashF<P, false>(ms256, make_adrs(0, info.idx_tree, T_FORS_TREE, info.idx_leaf, 0, g), sk, node, kb.pk_seed);
#pragma unroll 1
    for (int z = 0; z < A; z++) {
        const uint32_t gz = g >> z;
        uint32_t au[NW], lr[2 * NW];
        load_be<NW>(s + (size_t)(1 + z) * P::N, au);
#pragma unroll
        for (int w = 0; w < NW; w++) {
            lr[w] = (gz & 1) ? au[w] : node[w];
            lr[NW + w] = (gz & 1) ? node[w] : au[w];
        }
        hashH_ms<P>(ms256, msT, make_adrs(0, info.idx_tree, T_FORS_TREE, info.idx_leaf, z + 1, gz >> 1), lr, node,
                    kb.pk_seed);
    }
    uint32_t* r = fors_roots + ((size_t)m * K + i) * NW;
#pragma unroll
    for (int w = 0; w < NW; w++) r[w] = node[w];
}

constexpr uint32_t kRankBits = 28;        // sitem = steps << 28 | rank within the steps bucket

// The step counts of the chains of a block's messages (32 of them from m0 on:
// digit sources and checksums in msg / csum, valid = false: 0 steps), counted
// into the layer's 16 buckets, with each chain's rank inside its bucket
// recorded in sitem.  The whole block works on the 32 * LEN chains: ranks in
// the block from shared-memory counters, one global atomic per bucket and
// block.  (A thread per message counting in registers, 16 selects per digit
// and 80 shuffles, took about as long as T_len itself.)
template <class P>
struct CountSmem {
    uint32_t msg[32 * P::NW];
    uint32_t csum[32];
    uint32_t valid[32];
    uint32_t hist[16], base[16];
};
template <class P>
__device__ __forceinline__ void set_count_msg(CountSmem<P>& c, uint32_t lane, const uint32_t* msg, bool valid) {
    uint32_t cs = 0;
#pragma unroll
    for (int w = 0; w < P::NW; w++) {
        c.msg[lane * P::NW + w] = msg[w];
#pragma unroll
        for (int b = 0; b < 8; b++) cs += 15u - ((msg[w] >> (28 - 4 * b)) & 15u);
    }
    c.csum[lane] = cs << 4;
    c.valid[lane] = valid ? 1u : 0u;
    if (lane < 16) c.hist[lane] = 0;
}
// buf: 32 * LEN words of shared memory.  Every thread of the block calls it,
// after a barrier behind set_count_msg.
template <class P>
__device__ __forceinline__ void count_block(CountSmem<P>& c, uint32_t* buf, uint32_t m0, uint32_t nmsg,
                                            uint32_t* __restrict__ cnt, uint32_t* __restrict__ sitem) {
    constexpr int LEN = P::LEN;
    const uint32_t items = nmsg * LEN;
    for (uint32_t it = threadIdx.x; it < items; it += blockDim.x) {
        const uint32_t mm = it / LEN, i = it % LEN;
        const uint32_t d = i < (uint32_t)P::LEN1 ? (c.msg[mm * P::NW + (i >> 3)] >> (28 - 4 * (i & 7))) & 15u
                                                 : (c.csum[mm] >> (12 - 4 * (i - P::LEN1))) & 15u;
        const uint32_t st = c.valid[mm] ? 15u - d : 0u;
        buf[it] = (st << kRankBits) | atomicAdd(&c.hist[st], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 16) c.base[threadIdx.x] = c.hist[threadIdx.x] ? atomicAdd(&cnt[threadIdx.x], c.hist[threadIdx.x]) : 0u;
    __syncthreads();
    for (uint32_t it = threadIdx.x; it < items; it += blockDim.x) {
        const uint32_t v = buf[it];
        sitem[(size_t)m0 * LEN + it] = v + c.base[v >> kRankBits];
    }
}

// Layer 0: count from PK_FORS, 32 messages per block.
template <class P>
__global__ void __launch_bounds__(128) vcount0_kernel(const MsgInfo* __restrict__ infos, uint32_t count,
                                                      const uint32_t* __restrict__ pk_fors, uint32_t* __restrict__ cnt,
                                                      uint32_t* __restrict__ sitem) {
    __shared__ CountSmem<P> c;
    __shared__ uint32_t buf[32 * P::LEN];
    const uint32_t m0 = blockIdx.x * 32, m = m0 + threadIdx.x;
    if (threadIdx.x < 32) {
        const bool valid = m < count && infos[m].key != KEY_INVALID;
        uint32_t msg[P::NW];
#pragma unroll
        for (int w = 0; w < P::NW; w++) msg[w] = valid ? pk_fors[(size_t)m * P::NW + w] : 0u;
        set_count_msg<P>(c, threadIdx.x, msg, valid);
    }
    __syncthreads();
    count_block<P>(c, buf, m0, min(32u, count - m0), cnt, sitem);
}

// Place every chain of the layer at its sorted position (longest first).
template <class P>
__global__ void __launch_bounds__(256) vscatter_kernel(uint32_t count, const uint32_t* __restrict__ cnt,
                                                       const uint32_t* __restrict__ sitem, uint32_t* __restrict__ order) {
    const uint64_t it = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= (uint64_t)count * P::LEN) return;
    const uint32_t v = sitem[it];
    const uint32_t st = v >> kRankBits, r = v & ((1u << kRankBits) - 1u);
    uint32_t base = 0;
#pragma unroll
    for (int b = 15; b >= 0; b--) base += ((uint32_t)b > st) ? cnt[b] : 0u;
    order[base + r] = (uint32_t)it;
}

// Layer j, chain i of message m: its digit from msg_j (PK_FORS for j = 0,
// else root_{j-1} in vroot), then F from the signed position to w - 1.
template <class P, int POL>
__global__ void __launch_bounds__(128) vchain_kernel(const KeyBlock* __restrict__ keys,
                                                     const MsgInfo* __restrict__ infos, uint32_t count,
                                                     const uint8_t* __restrict__ sigs,
                                                     const uint32_t* __restrict__ order,
                                                     const uint32_t* __restrict__ sitem,
                                                     uint32_t* __restrict__ ends, uint32_t j, uint32_t one) {
    constexpr int NW = P::NW, LEN = P::LEN;
    const uint64_t pos = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= (uint64_t)count * LEN) return;
    const uint64_t gid = order[pos];             // chains in order of decreasing length
    const uint64_t m = gid / LEN;
    const uint32_t i = (uint32_t)(gid % LEN);
    const MsgInfo& info = infos[m];
    if (info.key == KEY_INVALID) return;
    const KeyBlock& kb = keys[info.key];
    const uint32_t digit = 15u - (sitem[gid] >> kRankBits);
    const uint64_t tree = layer_tree<P>(info.idx_tree, (int)j);
    const uint32_t kp = layer_leaf<P>(info.idx_tree, info.idx_leaf, (int)j);
    uint32_t ms256[8], x[NW];
#pragma unroll
    for (int w = 0; w < 8; w++) ms256[w] = kb.ms256[w];
    load_be<NW>(sigs + (size_t)m * P::SIG_BYTES + P::N + P::FORS_BYTES + (size_t)j * P::LAYER_BYTES +
                    (size_t)i * P::N, x);
    const Pipes<POL> pp(one);
    if (digit < 15u) {
        if constexpr (P::SHAKE) {
#pragma unroll 1
            for (uint32_t q = digit; q < 15u; q++)
                hashF_p<P, POL>(ms256, make_adrs(j, tree, T_WOTS_HASH, kp, i, q), x, x, pp);
        } else if constexpr (P::ROBUST) {
            ChainCtx cx;
            MaskCtx<NW> mk;
            const Adrs ah = make_adrs(j, tree, T_WOTS_HASH, kp, i, 0);
            chain_ctx<POL>(ms256, ah, cx, pp);
            mask_ctx<POL, NW>(kb.pk_seed, ah, mk, pp);
#pragma unroll 1
            for (uint32_t q = digit; q < 15u; q++) chain_step_p<P, POL>(cx, mk, ms256, q, x, x, pp);
        } else {
            ChainCtx cx;
            chain_ctx<POL>(ms256, make_adrs(j, tree, T_WOTS_HASH, kp, i, 0), cx, pp);
#pragma unroll 1
            for (uint32_t q = digit; q < 15u; q++) chain_step<POL, NW>(cx, ms256, q, x, x, pp);
        }
    }
    uint32_t* e = ends + gid * NW;
#pragma unroll
    for (int w = 0; w < NW; w++) e[w] = x[w];
}

// Layer j of 32 messages per block: T_len over the chain ends (kern_tl.cuh),
// then h' climbs with the auth path; root_j replaces msg_j in vroot and its
// digits are counted for the next layer.
// GROUP = false: one warp per block, a thread per message alone.
template <class P, bool GROUP>
__global__ void __launch_bounds__(GROUP ? TlShape<P>::THREADS : 32) vleaf_kernel(const KeyBlock* __restrict__ keys,
                                                                    const MsgInfo* __restrict__ infos, uint32_t count,
                                                                    const uint8_t* __restrict__ sigs,
                                                                    uint32_t* __restrict__ ends,
                                                                    uint32_t* __restrict__ vroot, uint32_t j,
                                                                    uint32_t* __restrict__ cnt_next,
                                                                    uint32_t* __restrict__ sitem) {
    constexpr int NW = P::NW, LEN = P::LEN, HP = P::HP;
    constexpr int TLW = GROUP ? TlShape<P>::SMEM_WORDS : 1, BUF = TLW > 32 * LEN ? TLW : 32 * LEN;
    __shared__ __align__(16) uint32_t smem[BUF];
    __shared__ CountSmem<P> c;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t m0 = blockIdx.x * 32, m = m0 + lane;
    const uint32_t key = m < count ? infos[m].key : KEY_INVALID;
    const bool active = key != KEY_INVALID;
    const MsgInfo& info = infos[active ? m : 0];
    const KeyBlock& kb = keys[active ? key : 0];
    const uint64_t tree = layer_tree<P>(info.idx_tree, (int)j);
    const uint32_t kp = layer_leaf<P>(info.idx_tree, info.idx_leaf, (int)j);
    uint32_t node[NW];
    tl_group<P, LEN, GROUP>(P::BIG ? kb.ms512 : kb.ms256, make_adrs(j, tree, T_WOTS_PK, kp, 0, 0),
                     ends + (size_t)m * LEN * NW, active, kb.pk_seed, smem, node);
    if (threadIdx.x < 32) {
        if (active) {
            uint32_t ms256[8], msT[P::BIG ? 16 : 8];
#pragma unroll
            for (int w = 0; w < 8; w++) ms256[w] = kb.ms256[w];
#pragma unroll
            for (int w = 0; w < (P::BIG ? 16 : 8); w++) msT[w] = P::BIG ? kb.ms512[w] : kb.ms256[w];
            const uint8_t* auth = sigs + (size_t)m * P::SIG_BYTES + P::N + P::FORS_BYTES + (size_t)j * P::LAYER_BYTES +
                                  (size_t)LEN * P::N;
#pragma unroll 1
            for (int z = 0; z < HP; z++) {
                const uint32_t iz = kp >> z;
                uint32_t au[NW], lr[2 * NW];
                load_be<NW>(auth + (size_t)z * P::N, au);
#pragma unroll
                for (int w = 0; w < NW; w++) {
                    lr[w] = (iz & 1) ? au[w] : node[w];
                    lr[NW + w] = (iz & 1) ? node[w] : au[w];
                }
                hashH_ms<P>(ms256, msT, make_adrs(j, tree, T_TREE, 0, z + 1, iz >> 1), lr, node, kb.pk_seed);
            }
#pragma unroll
            for (int w = 0; w < NW; w++) vroot[(size_t)m * NW + w] = node[w];
        }
        if (cnt_next) set_count_msg<P>(c, lane, node, active);
    }
    if (cnt_next) {                                // the next layer's chains
        __syncthreads();
        count_block<P>(c, smem, m0, min(32u, count - m0), cnt_next, sitem);
    }
}

// ---------------------------------------------------------------- few signatures
// With few signatures a layer's chains and T_len are each one warp's latency,
// and the layers are serial.  The chains need not be: only the number of
// steps of a chain depends on the layer below, so the ends of every chain for
// each of the 16 digits it might have are computed for all layers at once
// (120 steps a chain in place of 7.5, in parallel), and what remains serial is
// picking the ends by digit, T_len and the climbs -- one launch that walks the
// layers of 32 signatures per block.  Pays while the extra steps are cheaper
// than d chain launches (verify_walk in dispatch.cu).

// End of chain i of layer j of message m for digit d, at
// [m][j][i][d][NW words]; the longest (d = 0) first.
template <class P, int POL>
__global__ void __launch_bounds__(128) vspec_kernel(const KeyBlock* __restrict__ keys,
                                                    const MsgInfo* __restrict__ infos, uint32_t count,
                                                    const uint8_t* __restrict__ sigs, uint32_t* __restrict__ vends,
                                                    uint32_t one) {
    allow_next();
    constexpr int NW = P::NW, LEN = P::LEN, D = P::D;
    const uint64_t gid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t per = (uint64_t)count * D * LEN;
    const uint32_t d = (uint32_t)(gid / per);
    if (d > 15) return;
    const uint64_t r = gid % per;
    const uint32_t m = (uint32_t)(r / (D * LEN)), j = (uint32_t)(r / LEN) % D, i = (uint32_t)(r % LEN);
    const MsgInfo& info = infos[m];
    if (info.key == KEY_INVALID) return;
    const KeyBlock& kb = keys[info.key];
    const uint64_t tree = layer_tree<P>(info.idx_tree, (int)j);
    const uint32_t kp = layer_leaf<P>(info.idx_tree, info.idx_leaf, (int)j);
    uint32_t ms256[8], x[NW];
#pragma unroll
    for (int w = 0; w < 8; w++) ms256[w] = kb.ms256[w];
    load_be<NW>(sigs + (size_t)m * P::SIG_BYTES + P::N + P::FORS_BYTES + (size_t)j * P::LAYER_BYTES +
                    (size_t)i * P::N, x);
    const Pipes<POL> pp(one);
    if constexpr (P::SHAKE) {
#pragma unroll 1
        for (uint32_t q = d; q < 15u; q++) hashF_p<P, POL>(ms256, make_adrs(j, tree, T_WOTS_HASH, kp, i, q), x, x, pp);
    } else {
        const Adrs ah = make_adrs(j, tree, T_WOTS_HASH, kp, i, 0);
        ChainCtx cx;
        MaskCtx<NW> mk;
        chain_ctx<POL>(ms256, ah, cx, pp);
        if constexpr (P::ROBUST) mask_ctx<POL, NW>(kb.pk_seed, ah, mk, pp);
#pragma unroll 1
        for (uint32_t q = d; q < 15u; q++) chain_step_p<P, POL>(cx, mk, ms256, q, x, x, pp);
    }
    uint32_t* e = vends + (r * 16 + d) * NW;
#pragma unroll
    for (int w = 0; w < NW; w++) e[w] = x[w];
}

// PK_FORS, then every layer of 32 signatures, then the comparison.  ends:
// count * LEN * NW words (the picked ends of the current layer).
constexpr int kWalkThreads = 256;
template <class P>
__global__ void __launch_bounds__(kWalkThreads) vwalk_kernel(const KeyBlock* __restrict__ keys,
                                                             const MsgInfo* __restrict__ infos, uint32_t count,
                                                             const uint8_t* __restrict__ sigs,
                                                             const uint32_t* __restrict__ vends, uint32_t* ends,
                                                             uint32_t* fors_roots, uint8_t* __restrict__ ok) {
    constexpr int NW = P::NW, LEN = P::LEN, HP = P::HP, D = P::D;
    __shared__ __align__(16) uint32_t smem[TlShape<P>::SMEM_WORDS];
    __shared__ uint32_t nodes[32 * NW], msg[32 * NW], csum[32], valid[32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t m0 = blockIdx.x * 32, m = m0 + lane, nmsg = min(32u, count - m0);
    const uint32_t key = m < count ? infos[m].key : KEY_INVALID;
    const bool active = key != KEY_INVALID;
    const MsgInfo& info = infos[active ? m : 0];
    const KeyBlock& kb = keys[active ? key : 0];
    const uint64_t idx_tree = info.idx_tree;
    const uint32_t idx_leaf = info.idx_leaf;
    const uint32_t* msT = P::BIG ? kb.ms512 : kb.ms256;
    uint32_t node[NW];
    if (warp == 0) valid[lane] = active ? 1u : 0u;
    tl_group<P, P::K>(msT, make_adrs(0, idx_tree, T_FORS_ROOTS, idx_leaf, 0, 0), fors_roots + (size_t)m * P::K * NW,
                      active, kb.pk_seed, smem, node);
#pragma unroll 1
    for (uint32_t j = 0; j < (uint32_t)D; j++) {
        if (warp == 0) {
            uint32_t cs = 0;
#pragma unroll
            for (int w = 0; w < NW; w++) {
                msg[lane * NW + w] = node[w];
#pragma unroll
                for (int b = 0; b < 8; b++) cs += 15u - ((node[w] >> (28 - 4 * b)) & 15u);
            }
            csum[lane] = cs << 4;
        }
        __syncthreads();
        for (uint32_t it = threadIdx.x; it < nmsg * LEN; it += kWalkThreads) {
            const uint32_t mm = it / LEN, i = it % LEN;
            if (!valid[mm]) continue;
            const uint32_t d = i < (uint32_t)P::LEN1 ? (msg[mm * NW + (i >> 3)] >> (28 - 4 * (i & 7))) & 15u
                                                     : (csum[mm] >> (12 - 4 * (i - P::LEN1))) & 15u;
            const uint32_t* e = vends + ((((size_t)(m0 + mm) * D + j) * LEN + i) * 16 + d) * NW;
            uint32_t* o = ends + ((size_t)(m0 + mm) * LEN + i) * NW;
#pragma unroll
            for (int w = 0; w < NW; w += 2) *reinterpret_cast<uint2*>(o + w) = *reinterpret_cast<const uint2*>(e + w);
        }
        __syncthreads();
        const uint64_t tree = layer_tree<P>(idx_tree, (int)j);
        const uint32_t kp = layer_leaf<P>(idx_tree, idx_leaf, (int)j);
        const uint8_t* auth = sigs + (size_t)(active ? m : 0) * P::SIG_BYTES + P::N + P::FORS_BYTES +
                              (size_t)j * P::LAYER_BYTES + (size_t)LEN * P::N;
        tl_group<P, LEN>(msT, make_adrs(j, tree, T_WOTS_PK, kp, 0, 0), ends + (size_t)m * LEN * NW, active, kb.pk_seed,
                         smem, node);
        uint32_t au[NW], nx[NW];
        const bool loads = active && warp == (P::SHAKE ? 0u : 1u);
#pragma unroll
        for (int w = 0; w < NW; w++) au[w] = nx[w] = 0;
        if (loads) load_be<NW>(auth, au);
#pragma unroll 1
        for (int z = 0; z < HP; z++) {
            const uint32_t iz = kp >> z;
            const Adrs a = make_adrs(j, tree, T_TREE, 0, z + 1, iz >> 1);
            if (loads && z + 1 < HP) load_be<NW>(auth + (size_t)(z + 1) * P::N, nx);
            if constexpr (P::SHAKE) {
                if (loads) {
                    uint32_t lr[2 * NW];
#pragma unroll
                    for (int w = 0; w < NW; w++) {
                        lr[w] = (iz & 1) ? au[w] : node[w];
                        lr[NW + w] = (iz & 1) ? node[w] : au[w];
                    }
                    hashH_ms<P>(kb.ms256, nullptr, a, lr, node, nullptr);
                }
            } else {
                h_group<P>(kb, a, iz & 1, au, smem, nodes, node);
            }
#pragma unroll
            for (int w = 0; w < NW; w++) au[w] = nx[w];
        }
    }
    if (warp == 0 && m < count) {
        uint32_t diff = active ? 0u : 1u;
#pragma unroll
        for (int w = 0; w < NW; w++) diff |= active ? node[w] ^ kb.pk_root[w] : 0u;
        ok[m] = diff == 0 ? 1 : 0;
    }
}

// ok[m] = 1 iff the top root equals PK.root.
template <class P>
__global__ void vfinal_kernel(const KeyBlock* __restrict__ keys, const MsgInfo* __restrict__ infos, uint32_t count,
                              const uint32_t* __restrict__ vroot, uint8_t* __restrict__ ok) {
    const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= count) return;
    const MsgInfo& info = infos[m];
    if (info.key == KEY_INVALID) { ok[m] = 0; return; }
    const KeyBlock& kb = keys[info.key];
    uint32_t diff = 0;
#pragma unroll
    for (int w = 0; w < P::NW; w++) diff |= vroot[(size_t)m * P::NW + w] ^ kb.pk_root[w];
    ok[m] = diff == 0 ? 1 : 0;
}

}  // namespace hs
