// SHAKE256 hashes of a whole batch, sixteen to a warp: two threads hold one
// state (the sixteen-state form of dil_keccak16.cuh) in registers, and each
// pair of threads works through hashes of its own, so the single-sponge hashes
// of independent tasks (H(pk), mu, rho', c~) share the permutation's
// instructions instead of running one per warp.
//
// A lone chain takes 250 SM clocks per round for a warp on its own and about a
// thousand a block for absorbing, 224 and 150 in the 25-lane form (a 136-byte block
// 3.8 to 4.0 us against 2.7), so long messages of small batches go there
// (hash_split).  A loaded SM spends 3.2 clocks per state and round on this one, 18.7
// on that: the bound is the ALU pipe, which the logic and funnel shifts of a round
// occupy for 2.8.
#pragma once
#include "dil_keccak16.cuh"
#include "dil_sample.cuh"

namespace dil {

// Input of one hash: plen bytes at pre (a multiple of 8, at most 128), then the
// rest of the `total` bytes at msg; any alignment.
struct HashInput {
    const uint8_t *pre;
    const uint8_t *msg;
    size_t total;
    int plen;
};

// Shared words a warp's sixteen inputs are staged in: 8-byte unit u of a pair's
// current block at k16_word(pair, 2 u), u <= 17 (conflict-free for the 32
// threads reading the same unit or its neighbour).  The stage is 8-byte aligned.
constexpr int HASH16_STAGE_WORDS = 18 * K16_ROW;

__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Starts copying the 136-byte block at byte `off` of a pair's input into its
// stage: the prefix's units, then the aligned 8-byte units that hold the
// message's bytes (each holds one, so it lies in that byte's page and no copy
// can fault).  The copies run while the previous block is permuted; loading a
// block when it was needed, 17 words one after the other, took longer than
// permuting it.
__device__ __forceinline__ void hash16_fetch(const HashInput &in, size_t off, uint32_t stage, int pair, int p) {
    const int nblk = in.total - off < 136 ? (int)(in.total - off) : 136;   // input bytes in the block
    const int npre = off == 0 ? in.plen / 8 : 0;                           // prefix units in the block
    const uint32_t dst = stage + 4 * k16_word(pair, 2 * p);
    if (npre) {
        const bool aligned = (reinterpret_cast<uintptr_t>(in.pre) & 7) == 0;
        for (int u = p; u < npre; u += 2) {
            const uint32_t to = stage + 4 * k16_word(pair, 2 * u);
            if (aligned)
                cp_async8(to, in.pre + 8 * u);
            else
                asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(to), "r"(ld_bytes4(in.pre + 8 * u, 4)),
                             "r"(ld_bytes4(in.pre + 8 * u + 4, 4))
                             : "memory");
        }
    }
    const uint8_t *m = in.msg + (off == 0 ? 0 : off - in.plen);
    const int mis = (int)(reinterpret_cast<uintptr_t>(m) & 7);
    const int end = nblk > 8 * npre ? npre + (mis + nblk - 8 * npre + 7) / 8 : npre;
    const uint8_t *q = m - mis - 8 * npre + 8 * p;
#pragma unroll
    for (int i = 0; i < 9; ++i)   // units p + 2 i
        if (2 * i + p >= npre && 2 * i + p < end) cp_async8(dst + 8 * K16_ROW * i, q + 16 * i);
}

// XORs the staged, padded block at byte `off` of the input into the state
// halves of thread p of the pair (p = 0: low words).  True when it is the last.
__device__ __forceinline__ bool hash16_absorb(uint32_t (&a)[25], const HashInput &in, size_t off, uint32_t stage,
                                              int pair, int p) {
    const int left = in.total - off < 136 ? (int)(in.total - off) : 136;
    const int npre = off == 0 ? in.plen / 8 : 0;
    // the message's words start (msg & 7) bytes into its first unit; prefix and
    // blocks are whole units
    const int mis = (int)(reinterpret_cast<uintptr_t>(in.msg) & 7), shift = 8 * (mis & 3), d = mis >> 2;
    const uint32_t pre = stage + 4 * k16_word(pair, p);
    const uint32_t lo_at = stage + 4 * k16_word(pair, p + d), hi_at = stage + 4 * k16_word(pair, p + d + 1);
    const bool last = left < 136;
#pragma unroll
    for (int i = 0; i < 17; ++i) {
        uint32_t lo, hi;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(lo) : "r"((i >= npre ? lo_at : pre) + 4 * K16_ROW * i));
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(hi) : "r"(hi_at + 4 * K16_ROW * i));
        uint32_t v = __funnelshift_r(lo, hi, i >= npre ? shift : 0);
        if (last) {
            const int have = left - 8 * i - 4 * p;
            v = have <= 0 ? 0u : have < 4 ? v & ((1u << (8 * have)) - 1u) : v;
            if (have >= 0 && have < 4) v ^= 0x1Fu << (8 * have);
            if (i == 16 && p) v ^= 0x80000000u;
        }
        a[i] ^= v;
    }
    return last;
}

// 24 rounds on sixteen states held in registers (all 32 lanes).
__device__ __forceinline__ void hash16_permute(uint32_t (&a)[25], bool high) {
#pragma unroll 1
    for (int round = 0; round < 24; ++round) k16_round(a, high, c_keccak_rc[round]);
}

// Runs hashes until no pair has one left (all 32 lanes; stage: the warp's
// HASH16_STAGE_WORDS shared words).  Job: `bool next(HashInput &)` gives this
// thread's pair its next input (both threads of a pair get the same answer),
// `void done(const uint32_t (&a)[25])` takes the state after the last block
// (thread p holds words 2 i + p of the output).  Job::CHAINED: what done() writes to
// global memory may be the next input of the same pair.
template <class Job>
__device__ __forceinline__ void hash16_run(Job &job, uint32_t *stage_words, int lane) {
    const uint32_t stage = smem_addr(stage_words);
    const int pair = lane >> 1, p = lane & 1;
    uint32_t a[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) a[i] = 0;
    HashInput in;
    size_t off = 0;
    bool live = job.next(in);
    if (live) hash16_fetch(in, 0, stage, pair, p);
    while (__any_sync(FULL, live)) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        bool last = false;
        if (live) last = hash16_absorb(a, in, off, stage, pair, p);
        __syncwarp();
        if (live && !last) {
            off += 136;
            hash16_fetch(in, off, stage, pair, p);
        }
        hash16_permute(a, p);
        if (last) {
            job.done(a);
#pragma unroll
            for (int i = 0; i < 25; ++i) a[i] = 0;
            off = 0;
            if (Job::CHAINED) {   // a thread fetches 8-byte units, of which its partner wrote half
                __threadfence_block();
                __syncwarp(3u << (lane & 30));
            }
            live = job.next(in);
            if (live) hash16_fetch(in, 0, stage, pair, p);
        }
    }
}

// Both threads of a pair: the even one's value.
__device__ __forceinline__ int pair_bcast(int v, int lane) {
    return __shfl_sync(3u << (lane & 30), v, lane & 30);
}

// Shared words of a warp that draws sixteen challenges: the stage, then 256
// bytes each.
constexpr int CHALLENGE_STRIDE = 65;   // words from one pair's challenge to the next
constexpr int CHALLENGE_WORDS = HASH16_STAGE_WORDS + K16_STATES * CHALLENGE_STRIDE;

// c = SampleInBall(c~) of every pair with `more` (all 32 lanes; ct: this
// thread's words 2 i + p of c~): 256 bytes at the pair's challenge behind the
// stage.  The squeezed blocks go through the stage and the even thread of each
// pair draws and swaps in the order Alg 2 gives, sixteen challenges at a time:
// about 50 short steps for all of them, where a warp that works on one
// challenge needs 1.1 k instructions for its permutation alone.
template <int TAU>
__device__ __forceinline__ void challenge16(const uint32_t (&ct)[4], bool more, uint32_t *stage, int lane) {
    const int pair = lane >> 1, p = lane & 1;
    uint8_t *c = reinterpret_cast<uint8_t *>(stage + HASH16_STAGE_WORDS + pair * CHALLENGE_STRIDE);
    uint32_t a[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) a[i] = i < 4 ? ct[i] : 0u;
    if (!p) a[4] = 0x1Fu;
    if (p) a[16] = 0x80000000u;
    for (int i = p; i < 64; i += 2) reinterpret_cast<uint32_t *>(c)[i] = 0;
    int i = N - TAU, pos = 8;
    uint64_t signs = 0;
    for (int blk = 0; blk < MAX_SQUEEZE_BLOCKS && __any_sync(FULL, more); ++blk) {
        hash16_permute(a, p);
        __syncwarp();
#pragma unroll
        for (int w = 0; w < 17; ++w) stage[k16_word(pair, 2 * w + p)] = a[w];
        __syncwarp();
        if (more && !p) {
            if (blk == 0) signs = ((uint64_t)stage[k16_word(pair, 1)] << 32) | stage[k16_word(pair, 0)];
            while (i < N && pos < 136) {
                const int at = (stage[k16_word(pair, pos >> 2)] >> (8 * (pos & 3))) & 0xFF;
                ++pos;
                if (at > i) continue;
                c[i] = c[at];
                c[at] = (signs & 1) ? 0xFF : 1;
                signs >>= 1;
                ++i;
            }
            pos = 0;
        }
        more = more && pair_bcast(i, lane) < N;
    }
    __syncwarp();
}

// Challenge u of the warp to global memory (4-byte aligned; all 32 lanes).
__device__ __forceinline__ void put_challenge(uint8_t *dst, const uint32_t *stage, int u, int lane) {
    const uint32_t *src = stage + HASH16_STAGE_WORDS + u * CHALLENGE_STRIDE;
    uint32_t *d = reinterpret_cast<uint32_t *>(dst);
    d[lane] = src[lane];
    d[lane + 32] = src[lane + 32];
}

}  // namespace dil
