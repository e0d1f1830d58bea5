// kern_msg.cuh -- per-key preparation and the message stage (kernel templates).
//
// Message stage (the paper's hash_message + message_to_indices, Fig. 2):
//   R      = Trunc_n(HMAC-SHA-x(SK.prf, PK.seed || M))          (PRF_msg)
//   digest = MGF1-SHA-x(R || PK.seed || SHA-x(R || PK.seed || PK.root || M), m)
//   digest = md || tree bytes || leaf bytes -> k FORS indices, idx_tree, idx_leaf
// FIPS 205 mode: M is preceded by a per-call prefix (0x00 || len(ctx) || ctx
// for pure SLH-DSA) in both hashes, and the FORS indices are read from md
// most significant bit first (FIPS 205 base_2b).
// The work is serial in the message length (two passes over M), the only
// length-dependent part of signing.  Large batches run a thread per message;
// small ones (SHA-2 sets) a warp per message, which takes the message
// schedules off the serial path (message_warp).
#pragma once
#include <cuda_runtime.h>
#include "hs_common.cuh"
#include "hs_launch.h"
#include "../../include/hs.h"

namespace hs {

// ------------------------------------------------------------- a warp per message
// A message's hash is one serial chain of compressions (FIPS 180-4 Sec.
// 6.2.2 / 6.4.2: each block starts from the previous block's state), so a
// thread hashing alone runs at one warp's latency with the message
// schedule's instructions on the same serial path.  The schedule of a block
// depends on the block alone, so a warp computes the schedules of up to 32
// blocks at once, one block per lane, and keeps W_t + K_t in shared memory
// (a row per block, padded by 4 words so that the lanes' rows start in
// different banks); every lane then runs the same rounds over them, which
// leaves only the rounds on the serial path.
template <bool BIG> struct CoopShape;
template <> struct CoopShape<false> { static constexpr int CH = 32, WKW = 64 + 4; };
template <> struct CoopShape<true> { static constexpr int CH = 32, WKW = 2 * 80 + 4; };

// W_t + K_t (t = 0..63) of one SHA-256 block (16 big-endian words) into o.
__device__ __forceinline__ void wk256_store(uint32_t W[16], uint32_t* o) {
#pragma unroll 1
    for (int t = 0; t < 64; t += 16) {
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
            uint32_t v[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int i = j + q;
                if (t > 0) W[i] += s1_256(W[(i + 14) & 15]) + W[(i + 9) & 15] + s0_256(W[(i + 1) & 15]);
                v[q] = W[i] + c_K256[t + i];
            }
            *reinterpret_cast<uint4*>(o + t + j) = make_uint4(v[0], v[1], v[2], v[3]);
        }
    }
}
// The same for SHA-512 (32 big-endian 32-bit words), (hi, lo) word pairs.
__device__ __forceinline__ void wk512_store(const uint32_t w[32], uint32_t* o) {
    uint64_t W[16];
#pragma unroll
    for (int i = 0; i < 16; i++) W[i] = ((uint64_t)w[2 * i] << 32) | w[2 * i + 1];
#pragma unroll 1
    for (int t = 0; t < 80; t += 16) {
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            uint64_t v[2];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int i = j + q;
                if (t > 0) W[i] += s1_512(W[(i + 14) & 15]) + W[(i + 9) & 15] + s0_512(W[(i + 1) & 15]);
                v[q] = W[i] + c_K512[t + i];
            }
            *reinterpret_cast<uint4*>(o + 2 * (t + j)) =
                make_uint4((uint32_t)(v[0] >> 32), (uint32_t)v[0], (uint32_t)(v[1] >> 32), (uint32_t)v[1]);
        }
    }
}

// The 64 SHA-256 rounds and the feed-forward, W_t + K_t read from wk.
// Latency form: the new e is d + T1 = (d + h + W_t + K_t) + Sigma1(e) +
// Ch(e, f, g), with the first sum formed before Sigma1 is ready (h and d
// are known rounds ahead), so only one three-input addition follows
// Sigma1 on the serial path; the empty asm keeps the compiler from folding
// that sum back into d + T1.  Measured 13 % faster than d + T1 in the warp
// form; the same restructuring made the SHA-512 rounds 8 % slower.  All 64
// rounds unrolled: in a loop of 8 a 64 KB message took 2.44 ms in place of
// 2.02.  Splitting a round over two lanes, one with (e, f, g, h) and one with
// (a, b, c, d) two rounds behind, trading T1 and a by shuffles, was slower
// too (3.07 ms, and 20 % at SHA-512): the shuffles outweigh the halved work.
__device__ __forceinline__ void rounds256_wk(uint32_t st[8], const uint32_t* wk) {
    uint32_t a = st[0], b = st[1], c = st[2], d = st[3], e = st[4], f = st[5], g = st[6], h = st[7];
#define HS_RW256(a, b, c, d, e, f, g, h, x)                         \
    do {                                                            \
        const uint32_t hx_ = h + (x);                               \
        uint32_t dhx_ = d + hx_;                                    \
        asm("" : "+r"(dhx_));                                       \
        const uint32_t s1_ = S1_256(e), ch_ = ch32(e, f, g);        \
        d = dhx_ + s1_ + ch_;                                       \
        h = (hx_ + s1_ + ch_) + S0_256(a) + maj32(a, b, c);         \
    } while (0)
#pragma unroll
    for (int t = 0; t < 64; t += 8) {
        const uint4 u = *reinterpret_cast<const uint4*>(wk + t);
        const uint4 v = *reinterpret_cast<const uint4*>(wk + t + 4);
        HS_RW256(a, b, c, d, e, f, g, h, u.x);
        HS_RW256(h, a, b, c, d, e, f, g, u.y);
        HS_RW256(g, h, a, b, c, d, e, f, u.z);
        HS_RW256(f, g, h, a, b, c, d, e, u.w);
        HS_RW256(e, f, g, h, a, b, c, d, v.x);
        HS_RW256(d, e, f, g, h, a, b, c, v.y);
        HS_RW256(c, d, e, f, g, h, a, b, v.z);
        HS_RW256(b, c, d, e, f, g, h, a, v.w);
    }
#undef HS_RW256
    st[0] += a; st[1] += b; st[2] += c; st[3] += d; st[4] += e; st[5] += f; st[6] += g; st[7] += h;
}

// The 80 SHA-512 rounds and the feed-forward on a state of 16 big-endian
// words (hi, lo pairs); W_t + K_t are loaded four rounds ahead (a 64 KB
// message at 192f 2.52 -> 2.46 ms).
__device__ __forceinline__ void rounds512_wk(uint32_t st[16], const uint32_t* wk) {
    uint64_t s[8], v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = s[i] = ((uint64_t)st[2 * i] << 32) | st[2 * i + 1];
    auto round = [&](int j, uint32_t khi, uint32_t klo) {
        uint64_t &a = v[(8 - j) & 7], &b = v[(9 - j) & 7], &c = v[(10 - j) & 7], &d = v[(11 - j) & 7];
        uint64_t &e = v[(12 - j) & 7], &f = v[(13 - j) & 7], &g = v[(14 - j) & 7], &h = v[(15 - j) & 7];
        const uint64_t t1 = h + S1_512(e) + ((e & f) ^ (~e & g)) + (((uint64_t)khi << 32) | klo);
        const uint64_t t2 = S0_512(a) + ((a & b) | (c & (a | b)));
        d += t1;
        h = t1 + t2;
    };
    const uint4* w4 = reinterpret_cast<const uint4*>(wk);
    uint4 k0 = w4[0], k1 = w4[1];
#pragma unroll 1
    for (int t = 0; t < 80; t += 8) {
        const uint4 n0 = w4[t / 2 + 2], n1 = w4[t / 2 + 3];
        round(0, k0.x, k0.y);
        round(1, k0.z, k0.w);
        round(2, k1.x, k1.y);
        round(3, k1.z, k1.w);
        if (t < 72) { k0 = w4[t / 2 + 4]; k1 = w4[t / 2 + 5]; }
        round(4, n0.x, n0.y);
        round(5, n0.z, n0.w);
        round(6, n1.x, n1.y);
        round(7, n1.z, n1.w);
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        s[i] += v[i];
        st[2 * i] = (uint32_t)(s[i] >> 32);
        st[2 * i + 1] = (uint32_t)s[i];
    }
}

// ------------------------------------------------------------- byte SHA-x
// Streaming SHA-256 / SHA-512 over bytes and big-endian words.  Only the
// message stage uses it: key words, pads and digests are appended a word at
// a time from registers; message bytes arrive through aligned word loads,
// whole blocks with the next block's loads in flight (blocks()), the partial
// blocks at either end through one batch of loads each (append()).
template <bool BIG>
struct ByteSha {
    static constexpr int B = BIG ? 128 : 64;   // block bytes
    static constexpr int BW = B / 4;
    uint32_t st[BIG ? 16 : 8];
    uint32_t blk[BW];
    uint32_t fill;      // bytes in blk
    uint64_t total;     // message bytes so far

    __device__ void init() {
        if constexpr (BIG) {
            uint64_t s[8];
            sha512_iv(s);
            for (int i = 0; i < 8; i++) { st[2 * i] = (uint32_t)(s[i] >> 32); st[2 * i + 1] = (uint32_t)s[i]; }
        } else {
            sha256_iv(st);
        }
        for (int i = 0; i < BW; i++) blk[i] = 0;
        fill = 0;
        total = 0;
    }
    __device__ void compress() {
        if constexpr (BIG) {
            uint64_t s[8];
            for (int i = 0; i < 8; i++) s[i] = ((uint64_t)st[2 * i] << 32) | st[2 * i + 1];
            sha512_compress_w32(s, blk);
            for (int i = 0; i < 8; i++) { st[2 * i] = (uint32_t)(s[i] >> 32); st[2 * i + 1] = (uint32_t)s[i]; }
        } else {
            uint32_t W[16];
            for (int i = 0; i < 16; i++) W[i] = blk[i];
            sha256_compress_rolled(st, W);
        }
        for (int i = 0; i < BW; i++) blk[i] = 0;
        fill = 0;
    }
    __device__ void byte(uint32_t b) {
        blk[fill >> 2] |= (b & 0xFFu) << (24 - 8 * (fill & 3));
        fill++;
        total++;
        if (fill == B) compress();
    }
    // Append the top nb (1..4) bytes of the big-endian word w at any byte
    // offset; the caller keeps fill + nb <= B and compresses a full block.
    __device__ __forceinline__ void put(uint32_t w, uint32_t nb) {
        if (nb < 4) w &= 0xFFFFFFFFu << (32 - 8 * nb);
        const uint32_t s = 8 * (fill & 3), j = fill >> 2;
        if (s == 0) {
            blk[j] = w;
        } else {
            blk[j] |= w >> s;
            if (s + 8 * nb > 32) blk[j + 1] |= w << (32 - s);
        }
        fill += nb;
        total += nb;
    }
    // nbytes of a big-endian word array (register data: keys, pads, digests)
    __device__ void words(const uint32_t* w, int nbytes) {
#pragma unroll 1
        for (int i = 0; i < nbytes; i += 4) {
            const uint32_t avail = nbytes - i < 4 ? (uint32_t)(nbytes - i) : 4u;
            const uint32_t room = (uint32_t)B - fill;
            if (avail <= room) {
                put(w[i >> 2], avail);
            } else {                                  // the word straddles the block end
                put(w[i >> 2], room);
                compress();
                put(w[i >> 2] << (8 * room), avail - room);
            }
            if (fill == (uint32_t)B) compress();
        }
    }
    // The message word selector: big-endian word k of bytes q[4k .. 4k+3]
    // from the aligned little-endian words around it (q & 3 = sh).
    static __device__ __forceinline__ uint32_t be_sel(uint32_t sh) {
        return (sh << 12) | ((sh + 1) << 8) | ((sh + 2) << 4) | (sh + 3);
    }
    __device__ __forceinline__ void compress_words(const uint32_t w[BW]) {
        if constexpr (BIG) {
            uint64_t s[8], W[16];
#pragma unroll
            for (int i = 0; i < 8; i++) s[i] = ((uint64_t)st[2 * i] << 32) | st[2 * i + 1];
#pragma unroll
            for (int i = 0; i < 16; i++) W[i] = ((uint64_t)w[2 * i] << 32) | w[2 * i + 1];
            sha512_compress(s, W);
#pragma unroll
            for (int i = 0; i < 8; i++) { st[2 * i] = (uint32_t)(s[i] >> 32); st[2 * i + 1] = (uint32_t)s[i]; }
        } else {
            uint32_t W[16];
#pragma unroll
            for (int i = 0; i < 16; i++) W[i] = w[i];
            sha256_compress_full(st, W);
        }
    }
    // Append r < B message bytes at q (any alignment) without crossing the
    // end of the open block.  The bytes arrive through aligned 32-bit loads
    // issued together, each holding at least one byte of q[0, r), so nothing
    // outside the message is read.
    __device__ void append(const uint8_t* q, uint32_t r) {
        if (r == 0) return;
        const uintptr_t addr = reinterpret_cast<uintptr_t>(q);
        const uint32_t* a = reinterpret_cast<const uint32_t*>(addr & ~(uintptr_t)3);
        const uint32_t sh = (uint32_t)(addr & 3), sel = be_sel(sh);
        const uint32_t nl = (sh + r + 3) >> 2;
        uint32_t raw[BW + 1];
#pragma unroll
        for (int k = 0; k < BW + 1; k++) raw[k] = ((uint32_t)k < nl) ? __ldg(a + k) : 0u;
#pragma unroll
        for (int k = 0; k < BW; k++)
            if ((uint32_t)(4 * k) < r) put(__byte_perm(raw[k], raw[k + 1], sel), min(4u, r - 4u * k));
        if (fill == (uint32_t)B) compress();
    }
    // nb whole blocks from q at any alignment: aligned 32-bit loads (every
    // word holds at least one byte of the blocks), one prmt per big-endian
    // word, and the next block's loads in flight during this compression.
    __device__ void blocks(const uint8_t* q, uint64_t nb) {
        const uintptr_t addr = reinterpret_cast<uintptr_t>(q);
        const uint32_t* a = reinterpret_cast<const uint32_t*>(addr & ~(uintptr_t)3);
        const uint32_t sh = (uint32_t)(addr & 3), sel = be_sel(sh);
        uint32_t raw[BW + 1];
#pragma unroll
        for (int k = 0; k < BW; k++) raw[k] = __ldg(a + k);
        raw[BW] = sh ? __ldg(a + BW) : 0u;
        for (uint64_t b = 0; b < nb; b++) {
            uint32_t w[BW];
#pragma unroll
            for (int k = 0; k < BW; k++) w[k] = __byte_perm(raw[k], raw[k + 1], sel);
            if (b + 1 < nb) {
                const uint32_t* an = a + (b + 1) * BW;
#pragma unroll
                for (int k = 0; k < BW; k++) raw[k] = __ldg(an + k);
                raw[BW] = sh ? __ldg(an + BW) : 0u;
            }
            compress_words(w);
        }
        total += nb * B;
    }
    // raw bytes from global memory at any alignment: the rest of the open
    // block, whole blocks, then the tail
    __device__ void mem(const uint8_t* p, uint64_t len) {
        uint64_t i = 0;
        if (fill != 0 && len != 0) {
            i = ((uint64_t)B - fill < len) ? (uint64_t)B - fill : len;
            append(p, (uint32_t)i);
        }
        const uint64_t nb = (len - i) / B;
        if (nb) {
            blocks(p + i, nb);
            i += nb * B;
        }
        if (i < len) append(p + i, (uint32_t)(len - i));
    }
    // Pad (0x80, zeros, bit length) and return the digest words (8 or 16).
    __device__ void finish(uint32_t* out) {
        const uint64_t bits = total * 8;
        blk[fill >> 2] |= 0x80u << (24 - 8 * (fill & 3));
        fill++;
        if (fill > (uint32_t)(B - (BIG ? 16 : 8))) compress();
        blk[BW - 1] = (uint32_t)bits;
        blk[BW - 2] = (uint32_t)(bits >> 32);
        compress();
        for (int i = 0; i < (BIG ? 16 : 8); i++) out[i] = st[i];
    }
};

// ------------------------------------------------------------- keyprep
// KeyBlock from a key buffer: sign keys are SK.seed||SK.prf||PK.seed||PK.root
// (4n); verify keys are PK.seed||PK.root (2n).  The midstates are the SHA-2
// state after the first block BlockPad(PK.seed).  At n = 24 / 32 two threads
// share a key, one per midstate: with few keys the launch is one thread's
// latency.
template <class P>
__global__ void keyprep_kernel(const uint8_t* __restrict__ in, uint32_t num_keys, int from_pk,
                               KeyBlock* __restrict__ out) {
    allow_next();
    constexpr int NW = P::NW, TPK = P::BIG ? 2 : 1;
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, k = t / TPK;
    if (k >= num_keys) return;
    KeyBlock& kb = out[k];
    const uint8_t* pk = in + (from_pk ? (size_t)k * 2 * P::N : (size_t)k * 4 * P::N + 2 * P::N);
    uint32_t seed[8];
#pragma unroll
    for (int i = 0; i < 8; i++) seed[i] = 0;
    load_be_unaligned<NW>(pk, seed);
    if (t % TPK == 0) {
        uint32_t v[8];
#pragma unroll
        for (int i = 0; i < 8; i++) { kb.pk_seed[i] = seed[i]; kb.pad[i] = 0; v[i] = 0; }
        load_be_unaligned<NW>(pk + P::N, v);
#pragma unroll
        for (int i = 0; i < 8; i++) { kb.pk_root[i] = v[i]; v[i] = 0; }
        if (!from_pk) load_be_unaligned<NW>(pk - 2 * P::N, v);
#pragma unroll
        for (int i = 0; i < 8; i++) { kb.sk_seed[i] = v[i]; v[i] = 0; }
        if (!from_pk) load_be_unaligned<NW>(pk - P::N, v);
#pragma unroll
        for (int i = 0; i < 8; i++) { kb.sk_prf[i] = v[i]; v[i] = seed[i]; }
        if constexpr (!P::SHAKE) {    // the SHAKE hashes take PK.seed itself
            uint32_t W[16];
#pragma unroll
            for (int i = 0; i < 16; i++) W[i] = (i < NW) ? seed[i] : 0u;
            sha256_iv(v);
            sha256_compress_rolled(v, W);
        }
#pragma unroll
        for (int i = 0; i < 8; i++) kb.ms256[i] = v[i];
        if constexpr (!P::BIG) {
#pragma unroll
            for (int i = 0; i < 16; i++) kb.ms512[i] = 0;
        }
    } else {
        uint32_t blk[32];
#pragma unroll
        for (int i = 0; i < 32; i++) blk[i] = (i < NW) ? seed[i] : 0u;
        uint64_t s[8];
        sha512_iv(s);
        sha512_compress_w32(s, blk);
#pragma unroll
        for (int i = 0; i < 8; i++) { kb.ms512[2 * i] = (uint32_t)(s[i] >> 32); kb.ms512[2 * i + 1] = (uint32_t)s[i]; }
    }
}

// ------------------------------------------------------------- message stage
template <class P>
__device__ __forceinline__ uint32_t digest_byte(const uint32_t* dw, int i) {
    return (dw[i >> 2] >> (24 - 8 * (i & 3))) & 0xFFu;
}

// One message's stage.  verify = 0: compute R (PRF_msg) and write it to
// sig[0:n]; verify = 1: R is read from the signature.
template <class P>
__device__ __forceinline__ void message_one(uint32_t m, const KeyBlock* __restrict__ keys,
                                            uint32_t num_keys, const uint32_t* __restrict__ key_idx,
                                            const uint8_t* __restrict__ msgs, const uint64_t* __restrict__ off,
                                            uint8_t* __restrict__ sigs, MsgInfo* __restrict__ infos,
                                            uint32_t* __restrict__ status, int verify,
                                            const uint8_t* __restrict__ prefix, uint32_t plen, int msb_first) {
    constexpr int NW = P::NW;
    constexpr int DW = P::BIG ? 16 : 8;            // digest words of SHA-x
    uint8_t* sig = sigs + (size_t)m * P::SIG_BYTES;
    MsgInfo info;
    info.pad[0] = info.pad[1] = 0;
    const uint32_t key = key_idx ? key_idx[m] : 0u;
    if (key >= num_keys) {
        atomicOr(status, 1u << HS_EKEY);
        info.key = KEY_INVALID;
        info.idx_tree = 0;
        info.idx_leaf = 0;
        for (int i = 0; i < 36; i++) info.fors_idx[i] = 0;
        infos[m] = info;
        if (!verify) {
            uint4* s4 = reinterpret_cast<uint4*>(sig);
            for (uint32_t i = 0; i < (uint32_t)(P::SIG_BYTES / 16); i++) s4[i] = make_uint4(0, 0, 0, 0);
        }
        return;
    }
    const KeyBlock& kb = keys[key];
    const uint8_t* M = msgs + off[m];
    const uint64_t mlen = off[m + 1] - off[m];

    uint32_t R[8];
    uint32_t dg[16];                     // digest words, >= m bytes (m <= 49)
    if constexpr (P::SHAKE) {
        // PRF_msg = SHAKE256(SK.prf || opt_rand || M, 8n), H_msg =
        // SHAKE256(R || PK.seed || PK.root || M, 8m); M may carry a prefix
        ByteShake k;
        if (!verify) {
            k.init();
            k.words(kb.sk_prf, P::N);
            k.words(kb.pk_seed, P::N);
            if (plen) k.mem(prefix, plen);
            k.mem(M, mlen);
            k.finish(R, P::N);
            store_be<NW>(sig, R);
        } else {
            load_be<NW>(sig, R);
        }
        k.init();
        k.words(R, P::N);
        k.words(kb.pk_seed, P::N);
        k.words(kb.pk_root, P::N);
        if (plen) k.mem(prefix, plen);
        k.mem(M, mlen);
        k.finish(dg, P::M);
    } else {
    using Sha = ByteSha<P::BIG>;
    Sha h;
    if (!verify) {
        // PRF_msg = HMAC-SHA-x(SK.prf, opt_rand || M), opt_rand = PK.seed
        uint32_t kw[Sha::BW];
        for (int i = 0; i < Sha::BW; i++) kw[i] = (i < NW) ? kb.sk_prf[i] : 0u;
        uint32_t inner[DW];
        h.init();
        for (int i = 0; i < Sha::BW; i++) {
            uint32_t x = kw[i] ^ 0x36363636u;
            h.words(&x, 4);
        }
        h.words(kb.pk_seed, P::N);
        if (plen) h.mem(prefix, plen);
        h.mem(M, mlen);
        h.finish(inner);
        h.init();
        for (int i = 0; i < Sha::BW; i++) {
            uint32_t x = kw[i] ^ 0x5c5c5c5cu;
            h.words(&x, 4);
        }
        h.words(inner, 4 * DW);
        uint32_t mac[DW];
        h.finish(mac);
        for (int i = 0; i < NW; i++) R[i] = mac[i];
        store_be<NW>(sig, R);
    } else {
        load_be<NW>(sig, R);
    }
    // H_msg
    uint32_t inner[DW];
    h.init();
    h.words(R, P::N);
    h.words(kb.pk_seed, P::N);
    h.words(kb.pk_root, P::N);
    if (plen) h.mem(prefix, plen);
    h.mem(M, mlen);
    h.finish(inner);
    int got = 0;
    for (uint32_t c = 0; got < P::M; c++) {
        h.init();
        h.words(R, P::N);
        h.words(kb.pk_seed, P::N);
        h.words(inner, 4 * DW);
        h.words(&c, 4);
        uint32_t blockd[DW];
        h.finish(blockd);
        for (int i = 0; i < DW && got < P::M; i++, got += 4) dg[got >> 2] = blockd[i];
    }
    }
    // md -> FORS indices: md read as a little-endian bit stream, index i from
    // stream bits i*a .. i*a+a-1, first bit least significant; in FIPS 205
    // mode bit q is bit 7 - q mod 8 of byte q/8 and the first bit read is the
    // most significant.
    for (int i = 0; i < P::K; i++) {
        uint32_t v = 0;
        for (int j = 0; j < P::A; j++) {
            const int q = i * P::A + j;
            if (msb_first) v |= ((digest_byte<P>(dg, q >> 3) >> (7 - (q & 7))) & 1u) << (P::A - 1 - j);
            else v |= ((digest_byte<P>(dg, q >> 3) >> (q & 7)) & 1u) << j;
        }
        info.fors_idx[i] = (uint16_t)v;
    }
    for (int i = P::K; i < 36; i++) info.fors_idx[i] = 0;
    uint64_t t = 0;
    for (int b = 0; b < P::TREE_BYTES; b++) t = (t << 8) | digest_byte<P>(dg, P::MD_BYTES + b);
    if (P::TREE_BITS < 64) t &= (1ull << (P::TREE_BITS & 63)) - 1ull;
    uint32_t l = 0;
    for (int b = 0; b < P::LEAF_BYTES; b++) l = (l << 8) | digest_byte<P>(dg, P::MD_BYTES + P::TREE_BYTES + b);
    l &= (uint32_t)(P::LEAVES - 1);
    info.idx_tree = t;
    info.idx_leaf = l;
    info.key = key;
    infos[m] = info;
}

// One thread per message: the throughput form for large batches.
template <class P>
__global__ void message_kernel(const KeyBlock* __restrict__ keys, uint32_t num_keys,
                               const uint32_t* __restrict__ key_idx, const uint8_t* __restrict__ msgs,
                               const uint64_t* __restrict__ off, uint32_t count, uint8_t* __restrict__ sigs,
                               MsgInfo* __restrict__ infos, uint32_t* __restrict__ status, int verify,
                               const uint8_t* __restrict__ prefix, uint32_t plen, int msb_first) {
    const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= count) return;
    message_one<P>(m, keys, num_keys, key_idx, msgs, off, sigs, infos, status, verify, prefix, plen, msb_first);
}

// One warp per message (SHA-2 sets): the latency form for small batches,
// where the message's serial hashes are on the batch's critical path.
// Each hash's input is a header of whole words (keys, R, digests; in shared
// memory), then -- where it hashes M -- the prefix and the message: whole
// blocks of M are loaded by the lane that schedules them, the others ("edge"
// blocks) are put together a word per lane.  HMAC's two pad blocks, and
// MGF1's two counters at n = 16, are independent: the warp's halves hash
// them side by side (dual).  One loop over the hashes keeps one copy of the
// schedule and round code, which a single message otherwise waits to fetch.
// Measured on GB300 against one lane feeding a byte-wise hash: a 32-byte
// message 53 -> 28 us at 128f, 74 -> 41 at 192f, 82 -> 43 at 256f; 4 KB at
// 192f 242 -> 193 us; at 64 KB the rounds are everything (31 cycles per
// SHA-256 round, 61 per SHA-512 round).
template <class P>
struct MsgWarp {
    static constexpr bool BIG = P::BIG;
    static constexpr int B = BIG ? 128 : 64, BW = B / 4, DW = BIG ? 16 : 8, WKW = CoopShape<BIG>::WKW;
    uint32_t rows[32 * WKW];
    uint32_t hdr[2][40];         // the header, per half
    uint32_t R[8];
    uint32_t dg[16];             // digest words, >= m bytes (m <= 49)
};

template <class P>
__device__ __forceinline__ void message_warp(MsgWarp<P>& sm, uint32_t m, const uint8_t* __restrict__ raw_keys,
                                             uint32_t num_keys, const uint32_t* __restrict__ key_idx,
                                             const uint8_t* __restrict__ msgs, const uint64_t* __restrict__ lens,
                                             const uint64_t* __restrict__ off, uint8_t* __restrict__ sigs,
                                             MsgInfo* __restrict__ infos, uint32_t* __restrict__ status, int verify,
                                             const uint8_t* __restrict__ prefix, uint32_t plen, int msb_first) {
    using S = MsgWarp<P>;
    constexpr int NW = P::NW, N = P::N, DW = S::DW, BW = S::BW, B = S::B, WKW = S::WKW;
    constexpr int NC = (P::M + 4 * DW - 1) / (4 * DW);            // MGF1 counters
    static_assert(NC <= 2 && 2 * N + 4 * DW + 4 <= 160, "two counters; the header fits");
    const uint32_t lane = threadIdx.x & 31, half = lane >> 4;
    uint8_t* sig = sigs + (size_t)m * P::SIG_BYTES;
    const uint32_t key = key_idx ? key_idx[m] : 0u;
    MsgInfo* info = infos + m;
    if (key >= num_keys) {                          // the whole warp
        if (lane == 0) {
            atomicOr(status, 1u << HS_EKEY);
            info->idx_tree = 0;
            info->idx_leaf = 0;
            info->key = KEY_INVALID;
            info->pad[0] = info->pad[1] = 0;
        }
        for (uint32_t i = lane; i < 36; i += 32) info->fors_idx[i] = 0;
        if (!verify) {
            uint4* s4 = reinterpret_cast<uint4*>(sig);
            for (uint32_t i = lane; i < (uint32_t)(P::SIG_BYTES / 16); i += 32) s4[i] = make_uint4(0, 0, 0, 0);
        }
        return;
    }
    // SK.prf, PK.seed and PK.root from the caller's key bytes, so that the
    // launch need not wait for keyprep
    const uint8_t* kb = raw_keys + (verify ? (size_t)key * 2 * N : (size_t)key * 4 * N + 2 * N);     // PK.seed
    auto key_word = [&](int at) { uint32_t w; load_be_unaligned<1>(kb + at, &w); return w; };
    const uint32_t pk_seed = lane < NW ? key_word(4 * lane) : 0u, pk_root = lane < NW ? key_word(N + 4 * lane) : 0u;
    // the message's offset: up to kSumLens messages, the warp sums the lengths
    // before it and no launch is needed for a prefix sum (off is null)
    uint64_t before = 0;
    if (off) {
        before = off[m];
    } else {
#pragma unroll 4
        for (uint32_t i = lane; i < m; i += 32) before += lens[i];
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, w);
    }
    const uint8_t* M = msgs + before;
    const uint64_t mlen = lens[m];

    uint32_t st[DW], outer[DW];
#pragma unroll
    for (int i = 0; i < DW; i++) outer[i] = 0;
    // 0: HMAC's pad blocks; 1: its inner hash; 2: its outer hash = R;
    // 3: H_msg's hash over M; 4: MGF1.
#pragma unroll 1
    for (int ph = verify ? 3 : 0; ph < 5; ph++) {
        uint32_t hl = 0;                            // header bytes
        uint64_t done = 0;                          // bytes hashed into st before
        if (ph == 1) {
#pragma unroll
            for (int i = 0; i < DW; i++) {
                outer[i] = __shfl_sync(0xFFFFFFFFu, st[i], 16);
                st[i] = __shfl_sync(0xFFFFFFFFu, st[i], 0);
            }
            if (lane < NW) sm.hdr[0][lane] = pk_seed;
            hl = N;
            done = B;
        } else if (ph == 2) {
            if (lane == 0) {
#pragma unroll
                for (int i = 0; i < DW; i++) sm.hdr[0][i] = st[i];
            }
#pragma unroll
            for (int i = 0; i < DW; i++) st[i] = outer[i];
            hl = 4 * DW;
            done = B;
        } else {
            if (ph == 0) {
                if (lane < BW) {
                    const uint32_t kw = lane < NW ? key_word(4 * (int)lane - N) : 0u;
                    sm.hdr[0][lane] = kw ^ 0x36363636u;
                    sm.hdr[1][lane] = kw ^ 0x5c5c5c5cu;
                }
                hl = B;
            } else if (ph == 3) {
                if (lane == 0) {
                    uint32_t R[NW];
                    if (verify) {
                        load_be<NW>(sig, R);
                    } else {
#pragma unroll
                        for (int i = 0; i < NW; i++) R[i] = st[i];
                        store_be<NW>(sig, R);
                    }
#pragma unroll
                    for (int i = 0; i < NW; i++) sm.R[i] = sm.hdr[0][i] = R[i];
                }
                if (lane < NW) {
                    sm.hdr[0][NW + lane] = pk_seed;
                    sm.hdr[0][2 * NW + lane] = pk_root;
                }
                hl = 3 * N;
            } else {
#pragma unroll 1
                for (int h = 0; h < 2; h++) {
                    if (lane < NW) {
                        sm.hdr[h][lane] = sm.R[lane];
                        sm.hdr[h][NW + lane] = pk_seed;
                    }
                    if (lane == 0) {
#pragma unroll
                        for (int i = 0; i < DW; i++) sm.hdr[h][2 * NW + i] = st[i];
                        sm.hdr[h][2 * NW + DW] = h;
                    }
                }
                hl = 2 * N + 4 * DW + 4;
            }
            if constexpr (P::BIG) {
                uint64_t iv[8];
                sha512_iv(iv);
#pragma unroll
                for (int i = 0; i < 8; i++) { st[2 * i] = (uint32_t)(iv[i] >> 32); st[2 * i + 1] = (uint32_t)iv[i]; }
            } else {
                sha256_iv(st);
            }
        }
        __syncwarp();
        const bool raw = ph == 0, body = ph == 1 || ph == 3, dual = ph == 0 || (ph == 4 && NC == 2);
        const uint64_t pl = body ? plen : 0u, ml = body ? mlen : 0u, total = hl + pl + ml;
        const uint64_t nb = raw ? 1u : (total + 1 + (P::BIG ? 16 : 8) + B - 1) / B;
        const uint64_t in0 = (hl + pl + B - 1) / B, in1 = (hl + pl + ml) / B;    // blocks in0 .. in1 - 1 lie in M
        const uint64_t bits = (done + total) * 8;
#pragma unroll 1
        for (uint64_t b0 = 0; b0 < nb; b0 += 32) {
            const uint32_t c = nb - b0 < 32 ? (uint32_t)(nb - b0) : 32u;
#pragma unroll 1
            for (uint32_t j = 0; j < c; j++) {      // the edge blocks' words, one per lane
                const uint64_t b = b0 + j;
                if (b >= in0 && b < in1) continue;
                if (lane < (uint32_t)BW) {
                    const uint64_t o = b * B + 4 * lane;
                    uint32_t w[2] = {0u, 0u};
                    if (o < hl) {                   // the header is whole words
                        w[0] = sm.hdr[0][o >> 2];
                        w[1] = sm.hdr[1][o >> 2];
                    } else if (!raw) {
                        const uint64_t q = o - hl;
#pragma unroll
                        for (int i = 0; i < 4; i++) {
                            const uint64_t x = q + i;
                            const uint32_t v = x < pl ? prefix[x] : (x < pl + ml ? M[x - pl] : (x == pl + ml ? 0x80u : 0u));
                            w[0] = (w[0] << 8) | v;
                        }
                        if (b == nb - 1 && lane == (uint32_t)BW - 1) w[0] = (uint32_t)bits;
                        if (b == nb - 1 && lane == (uint32_t)BW - 2) w[0] = (uint32_t)(bits >> 32);
                        w[1] = w[0];
                    }
                    sm.rows[j * WKW + lane] = w[0];
                    if (dual) sm.rows[(16 + j) * WKW + lane] = w[1];
                }
            }
            __syncwarp();
            const uint32_t j = dual ? lane & 15 : lane;
            if (j < c) {
                uint32_t* row = sm.rows + lane * WKW;
                const uint64_t b = b0 + j;
                uint32_t w[BW];
                if (b >= in0 && b < in1) {          // aligned words around the block, each holding a byte of it
                    const uintptr_t addr = reinterpret_cast<uintptr_t>(M + (b * B - hl - pl));
                    const uint32_t* a = reinterpret_cast<const uint32_t*>(addr & ~(uintptr_t)3);
                    const uint32_t sh = (uint32_t)(addr & 3), sel = ByteSha<P::BIG>::be_sel(sh);
                    uint32_t raww[BW + 1];
#pragma unroll
                    for (int k = 0; k < BW; k++) raww[k] = __ldg(a + k);
                    raww[BW] = sh ? __ldg(a + BW) : 0u;
#pragma unroll
                    for (int k = 0; k < BW; k++) w[k] = __byte_perm(raww[k], raww[k + 1], sel);
                } else {
#pragma unroll
                    for (int k = 0; k < BW; k++) w[k] = row[k];
                }
                if constexpr (P::BIG) wk512_store(w, row);
                else wk256_store(w, row);
            }
            __syncwarp();
            const uint32_t* wk = sm.rows + (dual ? half * 16 * WKW : 0u);
#pragma unroll 1
            for (uint32_t k = 0; k < c; k++) {
                if constexpr (P::BIG) rounds512_wk(st, wk + k * WKW);
                else rounds256_wk(st, wk + k * WKW);
            }
            __syncwarp();
        }
    }
    if (lane == 0 || (NC == 2 && lane == 16)) {
#pragma unroll
        for (int i = 0; i < DW; i++)
            if (i + (lane ? DW : 0) < 16) sm.dg[i + (lane ? DW : 0)] = st[i];
    }
    __syncwarp();
    // md -> FORS indices (a <= 14 bits of the stream, as in message_one), a lane per index
    auto byte = [&](uint32_t i) { return (sm.dg[i >> 2] >> (24 - 8 * (i & 3))) & 0xFFu; };
    for (uint32_t i = lane; i < 36; i += 32) {
        uint32_t v = 0;
        if (i < (uint32_t)P::K) {
            const uint32_t q = i * P::A, o = q >> 3, s = q & 7;
            v = msb_first ? ((byte(o) << 16) | (byte(o + 1) << 8) | byte(o + 2)) >> (24 - s - P::A)
                          : (byte(o) | (byte(o + 1) << 8) | (byte(o + 2) << 16)) >> s;
            v &= (1u << P::A) - 1u;
        }
        info->fors_idx[i] = (uint16_t)v;
    }
    if (lane == 0) {
        uint64_t t = 0;
        for (int b = 0; b < P::TREE_BYTES; b++) t = (t << 8) | byte(P::MD_BYTES + b);
        if (P::TREE_BITS < 64) t &= (1ull << (P::TREE_BITS & 63)) - 1ull;
        uint32_t l = 0;
        for (int b = 0; b < P::LEAF_BYTES; b++) l = (l << 8) | byte(P::MD_BYTES + P::TREE_BYTES + b);
        info->idx_tree = t;
        info->idx_leaf = l & (uint32_t)(P::LEAVES - 1);
        info->key = key;
        info->pad[0] = info->pad[1] = 0;
    }
}

// Two warps per block, each with its own message.
constexpr int kMsgWarpsPerBlock = 2;
template <class P>
__global__ void __launch_bounds__(32 * kMsgWarpsPerBlock)
    message_warp_kernel(const uint8_t* __restrict__ raw_keys, uint32_t num_keys,
                        const uint32_t* __restrict__ key_idx, const uint8_t* __restrict__ msgs,
                        const uint64_t* __restrict__ lens, const uint64_t* __restrict__ off, uint32_t count,
                        uint8_t* __restrict__ sigs, MsgInfo* __restrict__ infos, uint32_t* __restrict__ status,
                        int verify, const uint8_t* __restrict__ prefix, uint32_t plen, int msb_first, uint32_t guard) {
    if (blockIdx.x == guard) { wait_previous(); return; }
    __shared__ __align__(16) MsgWarp<P> sm[kMsgWarpsPerBlock];
    const uint32_t warp = threadIdx.x >> 5;
    const uint32_t m = blockIdx.x * kMsgWarpsPerBlock + warp;
    if (m >= count) return;                        // the whole warp
    message_warp<P>(sm[warp], m, raw_keys, num_keys, key_idx, msgs, lens, off, sigs, infos, status, verify, prefix,
                    plen, msb_first);
}

}  // namespace hs
