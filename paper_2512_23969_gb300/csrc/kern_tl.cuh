// kern_tl.cuh -- T_l of many items at once: one lane per item, the message
// schedules of the blocks computed by other warps.
//
// T_len (WOTS+ public keys) and T_k (FORS public key) hash 9 to 18 blocks in
// series: each block starts from the previous block's state.  A thread that
// hashes alone runs at one warp's latency with the schedule's instructions
// on the serial path (measured on GB300: 3500 cycles per SHA-256 block and
// 8400 or more per SHA-512 block), and the launches that do it hold few
// warps: 32 leaves or messages to a warp.  The payload is complete before the
// launch, and a block's schedule W_t + K_t depends on the payload alone, so
// here a group of 32 items takes 1 + CH warps: warps 1 .. CH compute the
// schedules of the next CH blocks (lane = item) into shared memory while
// warp 0 runs the rounds of the current ones.  The work is the same, split
// over warps on different SM sub-partitions; the serial path keeps the
// rounds only (about 2000 cycles per SHA-256 block, 5000 per SHA-512 block).
// Rows are [round][lane], so every shared-memory access of a warp is one
// conflict-free row.  CH: the producers' time per block is below the rounds'
// at both widths; two at SHA-256 halve the barriers (32 KB of shared memory),
// one at SHA-512 keeps the two buffers at 40 KB, five groups to an SM.
#pragma once
#include <cuda_runtime.h>
#include "hs_common.cuh"

namespace hs {

// Groups of 32 items per SM up to which a launch runs by groups: as many as an
// SM holds at SHA-512 (40 KB of shared memory each); the same line at SHA-256
// (32 KB, one more would fit).
constexpr uint32_t kTlGroupsPerSm = 5;

template <class P>
struct TlShape {
    static constexpr int CH = P::SHAKE ? 0 : (P::BIG ? 1 : 2);       // producer warps = blocks per buffer
    static constexpr int ROUNDS = P::BIG ? 80 : 64;
    static constexpr int SLOT = ROUNDS * 32 * (P::BIG ? 2 : 1);      // words of one block's rows
    static constexpr int THREADS = 32 * (1 + CH);                    // per 32 items
    static constexpr int SMEM_WORDS = P::SHAKE ? 1 : 2 * CH * SLOT;
};

// Block b of T_l's input after the midstate (as tl_block), its payload words
// loaded in one batch (p is 8-byte aligned: whole nodes from an aligned
// base): the words around the payload are what the 2-byte
// offset reads there -- the address's last half word before it, the pad byte
// and zeros behind it.
template <bool BIG, int PW>
__device__ __forceinline__ void tl_block_batch(const Adrs& a, const uint32_t* p, int b, uint32_t* W) {
    constexpr int BW = BIG ? 32 : 16;
    constexpr int NB = tl_blocks<BIG, PW>();
    static_assert(PW % 2 == 0, "pairs of payload words");
    uint32_t raw[BW + 2];
    if (BIG && b > 0 && b < NB - 1) {          // inside the payload: 8-byte loads (b BW - 6 is even)
#pragma unroll
        for (int k = 0; k <= BW; k += 2) {
            const int q = b * BW + k - 6;
            const uint2 t = q < PW ? *reinterpret_cast<const uint2*>(p + q) : make_uint2(q == PW ? 0x80000000u : 0u, 0u);
            raw[k] = t.x;
            raw[k + 1] = t.y;
        }
#pragma unroll
        for (int k = 0; k < BW; k++) W[k] = mid16(raw[k], raw[k + 1]);
        return;
    }
#pragma unroll
    for (int k = 0; k <= BW; k++) {
        const int q = b * BW + k - 6;
        raw[k] = (uint32_t)q < (uint32_t)PW ? p[q] : (q == -1 ? a.half : (q == PW ? 0x80000000u : 0u));
    }
#pragma unroll
    for (int k = 0; k < BW; k++) W[k] = mid16(raw[k], raw[k + 1]);
    if (b == 0) { W[0] = a.w0; W[1] = a.w1; W[2] = a.w2; W[3] = a.w3; W[4] = a.w4; }
    if (b == NB - 1) W[BW - 1] = ((BIG ? 128u : 64u) + 22u + 4u * PW) * 8u;
}

// One block's schedule into rows[t * 32 + lane]: W_t + K_t (SHA-256), W_t
// alone (SHA-512, where the producer is the slower side and the rounds add
// K_t).
__device__ __forceinline__ void tl_rows256(uint32_t W[16], uint32_t* rows, uint32_t lane) {
#pragma unroll 1
    for (int t0 = 0; t0 < 64; t0 += 16) {
#pragma unroll
        for (int i = 0; i < 16; i++) {
            if (t0 > 0) W[i] += s1_256(W[(i + 14) & 15]) + W[(i + 9) & 15] + s0_256(W[(i + 1) & 15]);
            rows[(t0 + i) * 32 + lane] = W[i] + c_K256[t0 + i];
        }
    }
}
__device__ __forceinline__ void tl_rows512(const uint32_t blk[32], uint64_t* rows, uint32_t lane) {
    uint64_t W[16];
#pragma unroll
    for (int i = 0; i < 16; i++) W[i] = ((uint64_t)blk[2 * i] << 32) | blk[2 * i + 1];
#pragma unroll 1
    for (int t0 = 0; t0 < 80; t0 += 16) {
#pragma unroll
        for (int i = 0; i < 16; i++) {
            if (t0 > 0) W[i] += s1_512(W[(i + 14) & 15]) + W[(i + 9) & 15] + s0_512(W[(i + 1) & 15]);
            rows[(t0 + i) * 32 + lane] = W[i];
        }
    }
}

// The rounds and the feed-forward from those rows; the next rows are loaded
// while the current ones are used.  SHA-256: the new e is formed as
// (d + h + W_t + K_t) + Sigma1 + Ch, its first sum ready before Sigma1 (the
// empty asm keeps it), as in the message stage's warp form.
__device__ __forceinline__ void tl_rounds256(uint32_t st[8], const uint32_t* rows, uint32_t lane) {
    uint32_t v[8], xa[8], xb[8];
#pragma unroll
    for (int i = 0; i < 8; i++) { v[i] = st[i]; xa[i] = rows[i * 32 + lane]; }
    auto eight = [&](const uint32_t* x) {
#pragma unroll
        for (int j = 0; j < 8; j++) {
            uint32_t &a = v[(8 - j) & 7], &b = v[(9 - j) & 7], &c = v[(10 - j) & 7], &d = v[(11 - j) & 7];
            uint32_t &e = v[(12 - j) & 7], &f = v[(13 - j) & 7], &g = v[(14 - j) & 7], &h = v[(15 - j) & 7];
            const uint32_t hx = h + x[j];
            uint32_t dhx = d + hx;
            asm("" : "+r"(dhx));
            const uint32_t s1 = S1_256(e), ch = ch32(e, f, g);
            d = dhx + s1 + ch;
            h = (hx + s1 + ch) + S0_256(a) + maj32(a, b, c);
        }
    };
#pragma unroll 1
    for (int t = 0; t < 64; t += 16) {
        const uint32_t* r = rows + t * 32 + lane;
#pragma unroll
        for (int i = 0; i < 8; i++) xb[i] = r[(8 + i) * 32];
        eight(xa);
        if (t < 48) {
#pragma unroll
            for (int i = 0; i < 8; i++) xa[i] = r[(16 + i) * 32];
        }
        eight(xb);
    }
#pragma unroll
    for (int i = 0; i < 8; i++) st[i] += v[i];
}
__device__ __forceinline__ void tl_rounds512(uint64_t st[8], const uint64_t* rows, uint32_t lane) {
    uint64_t v[8], xa[4], xb[4];
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = st[i];
#pragma unroll
    for (int i = 0; i < 4; i++) xa[i] = rows[i * 32 + lane];
    auto round = [&](int j, uint64_t x, uint64_t k) {
        uint64_t &a = v[(8 - j) & 7], &b = v[(9 - j) & 7], &c = v[(10 - j) & 7], &d = v[(11 - j) & 7];
        uint64_t &e = v[(12 - j) & 7], &f = v[(13 - j) & 7], &g = v[(14 - j) & 7], &h = v[(15 - j) & 7];
        const uint64_t t1 = h + S1_512(e) + ((e & f) ^ (~e & g)) + (x + k);
        const uint64_t t2 = S0_512(a) + ((a & b) | (c & (a | b)));
        d += t1;
        h = t1 + t2;
    };
#pragma unroll 1
    for (int t = 0; t < 80; t += 8) {
        const uint64_t* r = rows + t * 32 + lane;
#pragma unroll
        for (int i = 0; i < 4; i++) xb[i] = r[(4 + i) * 32];
#pragma unroll
        for (int i = 0; i < 4; i++) round(i, xa[i], c_K512[t + i]);
        if (t < 72) {
#pragma unroll
            for (int i = 0; i < 4; i++) xa[i] = r[(8 + i) * 32];
        }
#pragma unroll
        for (int i = 0; i < 4; i++) round(4 + i, xb[i], c_K512[t + 4 + i]);
    }
#pragma unroll
    for (int i = 0; i < 8; i++) st[i] += v[i];
}

// T_l of l = L n-byte values for the 32 items of a block (lane = item, the
// same item in every warp); TlShape<P>::THREADS threads or more, all of them
// call it.  p: the item's payload, complete before the launch; active: the lane
// has an item (others read nothing).  The result is in warp 0.  ms: the
// midstate (SHAKE: PK.seed); pks: PK.seed (robust sets: the payload is
// masked in place first, the mask's blocks shared by the warps).
// GROUP = false: every thread hashes its own item alone (tl_groups_pay).
template <class P, int L, bool GROUP = true>
__device__ __forceinline__ void tl_group(const uint32_t* ms, const Adrs& a, uint32_t* p, bool active,
                                         const uint32_t* pks, uint32_t* smem, uint32_t* out) {
    constexpr int NW = P::NW, PW = L * NW;
    if constexpr (!P::SHAKE && !GROUP) {
        if (active) {
            if constexpr (P::ROBUST) mask_mem<P::BIG, NW, PW>(pks, a, p);
            tl_from_mem<P::BIG, PW, NW>(ms, a, p, out);
        }
    } else if constexpr (P::SHAKE) {
        if (active && (!GROUP || threadIdx.x < 32)) {
            TStreamP<P> ts;
            ts.init(ms, a);
#pragma unroll 1
            for (int i = 0; i < L; i++) ts.template push_n<NW>(p + i * NW);
            ts.template finish<NW>(L * P::N, out);
        }
    } else {
        using S = TlShape<P>;
        constexpr int NB = tl_blocks<P::BIG, PW>(), NC = (NB + S::CH - 1) / S::CH;
        const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if constexpr (P::ROBUST) {
            if (active) mask_mem<P::BIG, NW, PW>(pks, a, p, (int)warp, (int)(blockDim.x >> 5));
            __syncthreads();
        }
        uint32_t st[P::BIG ? 1 : 8];
        uint64_t st64[P::BIG ? 8 : 1];
        if constexpr (P::BIG) {
#pragma unroll
            for (int i = 0; i < 8; i++) st64[i] = ((uint64_t)ms[2 * i] << 32) | ms[2 * i + 1];
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) st[i] = ms[i];
        }
#pragma unroll 1
        for (int c = -1; c < NC; c++) {           // c = -1: the first buffer is filled
            if (warp == 0) {
#pragma unroll 1
                for (int k = 0; k < S::CH; k++) {
                    if (c < 0 || c * S::CH + k >= NB) break;
                    const uint32_t* rows = smem + ((c & 1) * S::CH + k) * S::SLOT;
                    if constexpr (P::BIG) tl_rounds512(st64, reinterpret_cast<const uint64_t*>(rows), lane);
                    else tl_rounds256(st, rows, lane);
                }
            } else if (warp <= (uint32_t)S::CH) {
                const int b = (c + 1) * S::CH + (int)warp - 1;
                if (b < NB && active) {
                    uint32_t W[P::BIG ? 32 : 16];
                    uint32_t* rows = smem + (((c + 1) & 1) * S::CH + warp - 1) * S::SLOT;
                    tl_block_batch<P::BIG, PW>(a, p, b, W);
                    if constexpr (P::BIG) tl_rows512(W, reinterpret_cast<uint64_t*>(rows), lane);
                    else tl_rows256(W, rows, lane);
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < NW; i++) {
            if constexpr (P::BIG) out[i] = (i & 1) ? (uint32_t)st64[i / 2] : (uint32_t)(st64[i / 2] >> 32);
            else out[i] = st[i];
        }
    }
}

// H of two children for the same 32 items (SHA-2): one block each, warp 1
// computing the next 16 rounds' schedule while warp 0 runs the current 16.
// node (warp 0) is one child and receives the parent; right: it is the right
// child.  sib: the other child (warp 1); nodes: 32 * NW words of shared
// memory.
template <class P>
__device__ __forceinline__ void h_group(const KeyBlock& kb, const Adrs& a, bool right, const uint32_t* sib,
                                        uint32_t* smem, uint32_t* nodes, uint32_t* node) {
    constexpr int NW = P::NW, NCH = P::BIG ? 5 : 4, BW = P::BIG ? 32 : 16;
    constexpr int ROW = 16 * 32 * (P::BIG ? 2 : 1);      // words of 16 rows
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {
#pragma unroll
        for (int w = 0; w < NW; w++) nodes[w * 32 + lane] = node[w];
    }
    __syncthreads();
    uint32_t W[16], v[8];
    uint64_t W64[P::BIG ? 16 : 1], v64[P::BIG ? 8 : 1];
    if (warp == 1) {
        uint32_t lr[2 * NW], blk[BW];
#pragma unroll
        for (int w = 0; w < NW; w++) {
            const uint32_t n = nodes[w * 32 + lane];
            lr[w] = right ? sib[w] : n;
            lr[NW + w] = right ? n : sib[w];
        }
        if constexpr (P::ROBUST) mask_regs<P::BIG, NW, 2 * NW>(kb.pk_seed, a, lr);
        fill_block<BW, 2 * NW>(blk, a, lr);
        blk[BW - 1] = ((P::BIG ? 128 : 64) + 22 + 8 * NW) * 8;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            if constexpr (P::BIG) W64[i] = ((uint64_t)blk[2 * i] << 32) | blk[2 * i + 1];
            else W[i] = blk[i];
        }
    } else if (warp == 0) {
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if constexpr (P::BIG) v64[i] = ((uint64_t)kb.ms512[2 * i] << 32) | kb.ms512[2 * i + 1];
            else v[i] = kb.ms256[i];
        }
    }
#pragma unroll 1
    for (int c = -1; c < NCH; c++) {
        if (warp == 0 && c >= 0) {
            const uint32_t* rows = smem + (c & 1) * ROW;
            if constexpr (P::BIG) {
                const uint64_t* r = reinterpret_cast<const uint64_t*>(rows) + lane;
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    uint64_t &a_ = v64[(16 - j) & 7], &b_ = v64[(17 - j) & 7], &c_ = v64[(18 - j) & 7],
                             &d_ = v64[(19 - j) & 7], &e_ = v64[(20 - j) & 7], &f_ = v64[(21 - j) & 7],
                             &g_ = v64[(22 - j) & 7], &h_ = v64[(23 - j) & 7];
                    const uint64_t t1 = h_ + S1_512(e_) + ((e_ & f_) ^ (~e_ & g_)) + (r[j * 32] + c_K512[16 * c + j]);
                    const uint64_t t2 = S0_512(a_) + ((a_ & b_) | (c_ & (a_ | b_)));
                    d_ += t1;
                    h_ = t1 + t2;
                }
            } else {
                const uint32_t* r = rows + lane;
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    uint32_t &a_ = v[(16 - j) & 7], &b_ = v[(17 - j) & 7], &c_ = v[(18 - j) & 7],
                             &d_ = v[(19 - j) & 7], &e_ = v[(20 - j) & 7], &f_ = v[(21 - j) & 7],
                             &g_ = v[(22 - j) & 7], &h_ = v[(23 - j) & 7];
                    const uint32_t hx = h_ + r[j * 32];
                    uint32_t dhx = d_ + hx;
                    asm("" : "+r"(dhx));
                    const uint32_t s1 = S1_256(e_), ch = ch32(e_, f_, g_);
                    d_ = dhx + s1 + ch;
                    h_ = (hx + s1 + ch) + S0_256(a_) + maj32(a_, b_, c_);
                }
            }
        } else if (warp == 1 && c + 1 < NCH) {
            const int t0 = 16 * (c + 1);
            uint32_t* rows = smem + ((c + 1) & 1) * ROW;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                if constexpr (P::BIG) {
                    if (t0 > 0) W64[i] += s1_512(W64[(i + 14) & 15]) + W64[(i + 9) & 15] + s0_512(W64[(i + 1) & 15]);
                    reinterpret_cast<uint64_t*>(rows)[i * 32 + lane] = W64[i];
                } else {
                    if (t0 > 0) W[i] += s1_256(W[(i + 14) & 15]) + W[(i + 9) & 15] + s0_256(W[(i + 1) & 15]);
                    rows[i * 32 + lane] = W[i] + c_K256[t0 + i];
                }
            }
        }
        __syncthreads();
    }
    if (warp == 0) {
#pragma unroll
        for (int i = 0; i < NW; i++) {
            if constexpr (P::BIG) {
                const uint64_t s = v64[i / 2] + (((uint64_t)kb.ms512[i & ~1] << 32) | kb.ms512[i | 1]);
                node[i] = (i & 1) ? (uint32_t)s : (uint32_t)(s >> 32);
            } else {
                node[i] = v[i] + kb.ms256[i];
            }
        }
    }
}

}  // namespace hs
