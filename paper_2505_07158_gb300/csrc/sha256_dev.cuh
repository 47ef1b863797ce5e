// Device code of the sub-frame SHA-256 (FIPS 180-4) shared by the digest kernels and the persistent batch
// kernel: the producer/consumer message pipeline and the tree digest.  See sha256.cu for the design.
#pragma once
#include "bounds.cuh"
#include "common.cuh"
#include "sha256_core.cuh"

namespace fhd {
namespace {

__device__ __forceinline__ uint32_t rotr(uint32_t x, int n) { return __funnelshift_r(x, x, n); }
__device__ __forceinline__ uint32_t bswap(uint32_t x) { return __byte_perm(x, 0, 0x0123); }

struct ShaState {
    uint32_t h[8];
    __device__ __forceinline__ void init() { sha256_init(h); }
};

__device__ __forceinline__ void store_digest(uint8_t *dst, const uint32_t h[8]) {
    uint32_t *d = reinterpret_cast<uint32_t *>(dst);   // 32-byte slots, 4-byte aligned
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = bswap(h[k]);
}

constexpr int kMsgPerCta = 32;
constexpr uint64_t kPrefetchBlocks = 8;
constexpr uint64_t kRing = 4;

// Blocks of a padded message of len bytes (FIPS 180-4 Sec. 5.1.1).
__device__ __forceinline__ uint64_t padded_blocks(uint64_t len) { return (len >> 6) + ((len & 63) + 9 <= 64 ? 1 : 2); }

// Block b of the padded message (p, len) as 16 big-endian words, by byte loads.
__device__ __forceinline__ void message_block(const uint8_t *p, uint64_t len, uint64_t b, uint32_t w[16]) {
    const uint64_t full = len >> 6;
    if (b < full) {
        if (!FHD_IN(64 * b + 63, len, kSiteShaBlock)) {
#pragma unroll
            for (int k = 0; k < 16; ++k) w[k] = 0;
            return;
        }
        const uint8_t *q = p + 64 * b;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            w[k] = ((uint32_t)q[4 * k] << 24) | ((uint32_t)q[4 * k + 1] << 16) | ((uint32_t)q[4 * k + 2] << 8) |
                   (uint32_t)q[4 * k + 3];
        return;
    }
    const uint32_t rem = (uint32_t)(len & 63);
    const uint32_t blk = (uint32_t)(b - full);           // 0 or 1 within the tail
    const uint8_t *tail = p + 64 * full;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        uint32_t word = 0;
#pragma unroll
        for (int byte = 0; byte < 4; ++byte) {
            const uint32_t pos = blk * 64 + 4 * k + byte;
            uint32_t v = 0;
            if (pos < rem) v = tail[pos];
            else if (pos == rem) v = 0x80u;
            word = (word << 8) | v;
        }
        w[k] = word;
    }
    if (b == padded_blocks(len) - 1) {
        const uint64_t bits = len * 8;
        w[14] = (uint32_t)(bits >> 32);
        w[15] = (uint32_t)bits;
    }
}

// 16-byte asynchronous global -> shared copy (Ampere-class cp.async, L2 only), its commit and wait.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Threads of a pipeline: two consumer warps and the producer warp.
constexpr uint32_t kShaThreads = 96;

// The warps of one pipeline meet at hardware barrier `id`.
template <uint32_t kThreads = kShaThreads>
__device__ __forceinline__ void pipeline_barrier(uint32_t id) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kThreads) : "memory");
}

// a * one + b, with one a 1 that the compiler does not know: an addition on the multiplier's pipe, for the rounds'
// off-chain sums.  The shifts and LOP3s fill the other one (two cycles an instruction); a value in constant memory
// (blockDim.y below) costs no register port.
__device__ __forceinline__ uint32_t mul_add(uint32_t a, uint32_t one, uint32_t b) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(one), "r"(b));
    return d;
}

// Shared memory of one pipeline: the W + K ring the consumers read (four rounds to a 16-byte word; column m is
// message m's, column 32 zero) and the block ring the producer fills.
struct ShaSmem {
    uint4 wk[2][16][33];
    uint4 ring[kRing][4][32];
};

// What a pipeline that may share its SM keeps in shared memory (sha_pipeline).
struct ShaShare {
    uint32_t hand[8][32];   // the states handed from two lanes to one
    uint32_t start;         // sm_pair_roomy when the pipeline came,
    uint32_t roomy[2];      // and while each block was made, by its parity
};

// The pipelines on a pair of SMs: a word with a bit each, sixteen to an SM (which has room for eight).
__device__ __forceinline__ uint32_t sm_id() {
    uint32_t id;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(id));
    return id;
}
// No SM of the pair has a second pipeline.
__device__ __forceinline__ bool sm_pair_roomy(uint32_t w) { return __popc(w & 0xffffu) <= 1 && __popc(w >> 16) <= 1; }
// Takes a bit of SM `id` (0: none is left) and says whether the pair is roomy.
__device__ __forceinline__ uint32_t take_sm_bit(uint32_t *taken, uint32_t id, uint32_t &roomy) {
    uint32_t bit = id & 1 ? 0x10000u : 1u, old = 0;
    for (int k = 0; k < 16; ++k, bit <<= 1) {
        old = atomicOr(taken, bit);
        if (!(old & bit)) {
            roomy = sm_pair_roomy(old | bit);
            return bit;
        }
    }
    roomy = 0;
    return 0;
}

// Producer warp of a pipeline: lane = message (p, len; nothing if !active), NB blocks in all.
//
// Message bytes reach shared memory by cp.async, kRing - 1 blocks ahead of the block being expanded (one commit
// group per block, empty when the lane has nothing to copy), so no register waits on a load in flight; an L2
// prefetch runs kPrefetchBlocks ahead of that.  The copies are the 16-byte aligned pieces that lie inside the
// message, so a message that starts s bytes into a piece takes its block b from pieces 4b .. 4b + 4, shifted by s
// (a select by the words of s, a byte permute that also turns the word round); blocks that reach into a piece at
// the message's edge, and the padded tail, come by byte loads.  Byte loads throughout took such a message
// 2300 cycles a block, longer than the rounds (241 x 317 grey, 6 sub-frames: 0.24 -> 0.18 ms).
template <bool kShared>
__device__ __forceinline__ void sha_producer(const uint8_t *p, uint64_t len, bool active, uint64_t nb, uint64_t NB,
                                             uint32_t lane, uint32_t bar, ShaSmem &sm, ShaShare *share,
                                             const uint32_t *sm_pipelines) {
    const uint32_t s = (uint32_t)reinterpret_cast<uintptr_t>(p) & 15u;
    const bool shifted = __any_sync(0xffffffffu, active && s != 0);
    const uint64_t first = s ? 1 : 0, pieces = active ? (s + len) >> 4 : 0;   // whole pieces: first .. pieces - 1
    const uint64_t full = len >> 6;
    const uint32_t turn = 0x0123u + 0x1111u * (s & 3);
    auto issue = [&](uint64_t blk) {
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) {
            const uint64_t j = 4 * blk + q;
            if (j >= first && j < pieces && FHD_IN(16 * j + 15 - s, len, kSiteShaBlock))
                cp_async16(&sm.ring[blk % kRing][q][lane], p - s + 16 * j);
        }
        cp_async_commit();
    };
    for (uint64_t k = 0; k + 1 < kRing; ++k) issue(k);
    for (uint64_t b = 0; b < NB; ++b) {
        // Refills the slot of block b - 1, whose bytes were consumed in the previous iteration.
        issue(b + kRing - 1);
        uint32_t taken = 0;
        if (kShared) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(taken) : "l"(sm_pipelines));
        if (b < nb) {
            if (b + kPrefetchBlocks < full) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 64 * (b + kPrefetchBlocks)));
            cp_async_wait<kRing - 2>();     // blocks b and b + 1 have landed
            uint32_t w[16];
            if (4 * b >= first && 4 * b + (s ? 5 : 4) <= pieces) {
                uint32_t x[20];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 v = sm.ring[b % kRing][q][lane];
                    x[4 * q] = v.x;
                    x[4 * q + 1] = v.y;
                    x[4 * q + 2] = v.z;
                    x[4 * q + 3] = v.w;
                }
                if (shifted) {
                    const uint4 v = sm.ring[(b + 1) % kRing][0][lane];   // s == 0: not used
                    x[16] = v.x;
                    x[17] = v.y;
                    x[18] = v.z;
                    x[19] = v.w;
#pragma unroll
                    for (int q = 0; q < 18; ++q) x[q] = s & 8 ? x[q + 2] : x[q];
#pragma unroll
                    for (int q = 0; q < 17; ++q) x[q] = s & 4 ? x[q + 1] : x[q];
#pragma unroll
                    for (int q = 0; q < 16; ++q) w[q] = __byte_perm(x[q], x[q + 1], turn);
                } else {
#pragma unroll
                    for (int q = 0; q < 16; ++q) w[q] = bswap(x[q]);
                }
            } else {
                message_block(p, len, b, w);
            }
            uint4(*dst)[33] = sm.wk[b & 1];
            uint32_t o[4];
#pragma unroll
            for (int t = 0; t < 64; ++t) {
                uint32_t wt;
                if (t < 16) {
                    wt = w[t];
                } else {
                    const uint32_t w15 = w[(t - 15) & 15], w2 = w[(t - 2) & 15];
                    const uint32_t s0 = rotr(w15, 7) ^ rotr(w15, 18) ^ (w15 >> 3);
                    const uint32_t s1 = rotr(w2, 17) ^ rotr(w2, 19) ^ (w2 >> 10);
                    wt = w[t & 15] + s0 + w[(t - 7) & 15] + s1;
                    w[t & 15] = wt;
                }
                o[t & 3] = wt + kSha256K[t];
                if ((t & 3) == 3) dst[t >> 2][lane] = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        if (kShared && lane == 0) share->roomy[b & 1] = sm_pair_roomy(taken);
        pipeline_barrier(bar);     // block b is ready; block b-1 has been consumed
    }
    pipeline_barrier(bar);         // pairs with the consumers' last wait
    cp_async_wait<0>();
}

// 32 messages per pipeline: of its threads (rtid = 0 ..), the first two warps compress and the last one
// produces W + K.  Pipeline `unit` takes messages 32 unit .. 32 unit + 31 of the nmsg messages; message m is
// located by locate(m, p, len, out) and its digest goes to out (32 bytes); locate returns false for a message that
// failed a range check (checked builds), which is then skipped.  `bar` is the hardware barrier id the
// pipeline's warps use; the consumers of a pipeline with a `share` meet at bar + 1.
//
// What bounds a pipeline is the consumers' chain of rounds.  One lane per message needs ~28 cycles
// a round: 14 shifts, LOP3s and additions at two cycles an instruction on one pipe, the other additions on the
// multiplier's.  Split, two lanes of a consumer warp share a message: lane E holds e, f, g, h and lane A holds
// a, b, c, d, two rounds behind E, which needs a only four rounds later.  Both run the same instructions -- three
// rotations by their own amounts, one choice function, two sums -- and trade their new word by one shuffle, ~23
// cycles a round:
//   E, round t:  e' = (S1(e) + Ch(e, f, g)) + (h + K + W + a[t-4])      a[t-4] = d, from A
//   A, round t:  a' = (S0(a) + Maj(a, b, c)) + (e' - d)                 e' from E; e' - d is the round's T1
// with Ch and Maj as z ^ (e & x) and z ^ (a & x) of two words made from older ones (E: x = f ^ g, z = g; A: x =
// b ^ c, z = b & c).
//
// Split messages take twice the issue slots, so they pay only where a pipeline has its SM to itself: two split
// pipelines on one SM took 1.5 times as long as two unsplit ones.  With kShared the producer looks at the word of its SMs'
// pipelines (sm_pipelines) once a block, and the consumers, from the first block that found another one there, go on with one
// lane per message in the first warp; whether the others come from the same launch, from another stream's or from a launch
// confined to a few SMs makes no difference.  The two SMs of a pair do so together: with one of them split and the
// other not, the loops of both kinds miss the instruction cache that the two appear to share, and 153 pipelines took
// 3.59 ms where 154 took 2.90.  Digests of 30 720p frames on k streams, k = 1, 6, 8, 12: 1.17, 1.51, 1.64, 2.41 ms;
// always split 1.17, 1.96, 2.06, 2.95; always unsplit 1.30, 1.50, 1.61, 2.52.  Without kShared (the persistent kernel,
// one pipeline per SM) a pipeline stays split.
template <bool kShared, class Locate>
__device__ void sha_pipeline(Locate locate, uint32_t nmsg, uint32_t unit, uint32_t rtid, uint32_t bar, ShaSmem &sm,
                             ShaShare *share = nullptr, uint32_t *sm_pipelines = nullptr) {
    const uint32_t lane = rtid & 31;
    const uint32_t one = blockDim.y;       // every launch is one-dimensional
    const uint8_t *p = nullptr;
    uint64_t len = 0;
    uint8_t *out = nullptr;
    const uint32_t m = unit * kMsgPerCta + lane;
    bool active = m < nmsg;
    if (active) active = locate(m, p, len, out);
    const uint64_t nb = active ? padded_blocks(len) : 0;
    const uint64_t NB = __reduce_max_sync(0xffffffffu, (unsigned)nb);   // < 2^32 blocks per message
    if (rtid >= kShaThreads - 32) {
        sha_producer<kShared>(p, len, active, nb, NB, lane, bar, sm, share, sm_pipelines);
        return;
    }
    uint64_t b = 0;
    uint32_t own = 0;
    if (kShared && rtid == 0) own = take_sm_bit(sm_pipelines, sm_id(), share->start);   // while block 0 is made
    if (rtid < 32) sm.wk[rtid >> 4][rtid & 15][32] = make_uint4(0, 0, 0, 0);
    pipeline_barrier(bar);                 // block 0 ready
    bool split = !kShared || share->start != 0;
    ShaState st;
    st.init();
    if (split) {
        const bool A = rtid & 1;
        const uint32_t m2 = unit * kMsgPerCta + (rtid >> 1);
        const uint8_t *p2 = nullptr;
        uint64_t len2 = 0;
        uint8_t *out2 = nullptr;
        bool active2 = m2 < nmsg;
        if (active2) active2 = locate(m2, p2, len2, out2);
        const uint64_t nb2 = active2 ? padded_blocks(len2) : 0;
        const uint32_t mask = A ? 0xffffffffu : 0u, sign = A ? 0xffffffffu : 1u;
        const uint32_t r0 = A ? 2 : 6, r1 = A ? 13 : 11, r2 = A ? 22 : 25;
        uint32_t H[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) H[q] = A ? st.h[q] : st.h[4 + q];
        const uint32_t column = A ? 32u : rtid >> 1;   // A adds no W + K
        while (b < NB && split) {
            if (kShared) split = share->roomy[b & 1] != 0;   // after this block
            uint32_t wk[64], first[4], traded[66];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const uint4 x = sm.wk[b & 1][q][column];
                wk[4 * q] = x.x;
                wk[4 * q + 1] = x.y;
                wk[4 * q + 2] = x.z;
                wk[4 * q + 3] = x.w;
            }
            uint32_t s0 = H[0], s1 = H[1], s2 = H[2], s3 = H[3];
#pragma unroll
            for (int q = 0; q < 4; ++q) first[q] = __shfl_xor_sync(0xffffffffu, H[3 - q], 1);
            uint32_t x = s1 ^ s2, z = s2 & (s1 | ~mask);
#pragma unroll
            for (int i = 0; i < 66; ++i) {     // E: round i; A: round i - 2
                const uint32_t other = i < 2 ? first[i] : i < 4 ? (A ? traded[i - 2] : first[i]) : traded[i - 2];
                const uint32_t own = mul_add(s3, sign, i < 64 ? wk[i] : 0u);
                const uint32_t S = __funnelshift_r(s0, s0, r0) ^ __funnelshift_r(s0, s0, r1) ^ __funnelshift_r(s0, s0, r2);
                const uint32_t F = z ^ (s0 & x);
                const uint32_t v = S + F + mul_add(own, one, other);
                traded[i] = __shfl_xor_sync(0xffffffffu, v, 1);
                const bool step = i < 2 ? !A : i >= 64 ? A : true;
                s3 = step ? s2 : s3;
                s2 = step ? s1 : s2;
                s1 = step ? s0 : s1;
                s0 = step ? v : s0;
                x = s1 ^ s2;
                z = s2 & (s1 | ~mask);
            }
            if (b < nb2) {
                H[0] += s0;
                H[1] += s1;
                H[2] += s2;
                H[3] += s3;
            }
            pipeline_barrier(bar);         // done with block b; block b+1 ready
            ++b;
        }
        if (split) {
            if (kShared && rtid == 0) atomicAnd(sm_pipelines, ~own);
            if (active2) {
                uint32_t *d = reinterpret_cast<uint32_t *>(out2) + (A ? 0 : 4);   // 32-byte slots, 4-byte aligned
#pragma unroll
                for (int q = 0; q < 4; ++q) d[q] = bswap(H[q]);
            }
            return;
        }
        if constexpr (kShared) {           // on with one lane per message
#pragma unroll
            for (int q = 0; q < 4; ++q) share->hand[A ? q : 4 + q][rtid >> 1] = H[q];
            pipeline_barrier<64>(bar + 1);
#pragma unroll
            for (int q = 0; q < 8; ++q) st.h[q] = share->hand[q][lane];
        }
    }
    if constexpr (kShared) {
        if (rtid >= 32) {
            for (; b < NB; ++b) pipeline_barrier(bar);
            return;
        }
        for (; b < NB; ++b) {
            if (b < nb) {
                // all 64 W+K words into registers first: the rounds never wait on shared memory
                uint32_t wk[64];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const uint4 x = sm.wk[b & 1][q][lane];
                    wk[4 * q] = x.x;
                    wk[4 * q + 1] = x.y;
                    wk[4 * q + 2] = x.z;
                    wk[4 * q + 3] = x.w;
                }
                uint32_t a = st.h[0], bb = st.h[1], c = st.h[2], d = st.h[3];
                uint32_t e = st.h[4], f = st.h[5], g = st.h[6], hh = st.h[7];
#pragma unroll
                for (int t = 0; t < 64; ++t) {
                    const uint32_t S1 = rotr(e, 6) ^ rotr(e, 11) ^ rotr(e, 25);
                    const uint32_t ch = (e & f) ^ (~e & g);
                    const uint32_t S0 = rotr(a, 2) ^ rotr(a, 13) ^ rotr(a, 22);
                    const uint32_t mj = (a & bb) ^ (a & c) ^ (bb & c);
                    const uint32_t t1 = mul_add(hh, one, wk[t]) + S1 + ch;
                    hh = g; g = f; f = e; e = mul_add(t1, one, d);
                    d = c; c = bb; bb = a; a = t1 + S0 + mj;
                }
                st.h[0] += a; st.h[1] += bb; st.h[2] += c; st.h[3] += d;
                st.h[4] += e; st.h[5] += f; st.h[6] += g; st.h[7] += hh;
            }
            pipeline_barrier(bar);         // done with block b; block b+1 ready
        }
        if (rtid == 0) atomicAnd(sm_pipelines, ~own);
        if (active) store_digest(out, st.h);
    }
}

// Tree digest (an option of this library, not of the paper): SHA-256 of the n sub-frame digests at `part`
// concatenated in order, 32 n bytes; one thread.  The stored digests are big-endian bytes, so each message
// word is the byte swap of a stored 32-bit word.  32 n bytes end on a half or a whole 64-byte block: the
// padding (0x80, zeros, the 64-bit bit length 256 n) always fits in the last block.
__device__ void tree_digest(const uint8_t *part, uint32_t n, uint32_t h[8]) {
    ShaState st;
    st.init();
    const uint32_t *p = reinterpret_cast<const uint32_t *>(part);
    const uint32_t words = 8 * n;
    uint32_t w[16];
    uint32_t i = 0;
    for (; i + 16 <= words; i += 16) {
#pragma unroll
        for (int k = 0; k < 16; ++k) w[k] = bswap(__ldcg(p + i + k));
        sha256_compress(st.h, w);
    }
    const uint32_t rem = words - i;   // 0 or 8
#pragma unroll
    for (int k = 0; k < 16; ++k) w[k] = (uint32_t)k < rem ? bswap(__ldcg(p + i + k)) : 0u;
    w[rem] = 0x80000000u;
    const uint64_t bits = 256ull * n;
    w[14] = (uint32_t)(bits >> 32);
    w[15] = (uint32_t)bits;
    sha256_compress(st.h, w);
#pragma unroll
    for (int k = 0; k < 8; ++k) h[k] = st.h[k];
}

}  // namespace
}  // namespace fhd
