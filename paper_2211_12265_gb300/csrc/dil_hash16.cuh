// SHAKE256 hashes of a whole batch, sixteen to a warp: two threads hold one
// state (the sixteen-state form of dil_keccak16.cuh) in registers, and each
// pair of threads works through hashes of its own, so the single-sponge hashes
// of independent tasks (H(pk), mu, rho', c~) share the permutation's
// instructions instead of running one per warp.
//
// A lone chain is no slower this way (250 SM clocks per round for a warp on
// its own, 224 for the 25-lane form) and a loaded SM spends 3.2 clocks per
// state and round on it where the 25-lane form spends 18.7: the bound is the
// ALU pipe, which the logic and funnel shifts of a round occupy for 2.8.
#pragma once
#include "dil_keccak16.cuh"

namespace dil {

// 4 bytes of global memory at p (any alignment), bytes from p + have on read
// as 0.  Only aligned words that hold a byte below p + have are loaded, and
// such a word lies in that byte's page, so no load can fault.
__device__ __forceinline__ uint32_t ld_bytes4(const uint8_t *p, long long have) {
    if (have <= 0) return 0;
    const uint32_t mis = (uint32_t)reinterpret_cast<uintptr_t>(p) & 3u;
    const uint32_t *q = reinterpret_cast<const uint32_t *>(p - mis);
    uint32_t v = q[0];
    if (mis) v = __funnelshift_r(v, have > (long long)(4 - mis) ? q[1] : 0u, 8 * mis);
    return have < 4 ? v & ((1u << (8 * (int)have)) - 1u) : v;
}

// Input of one hash: plen bytes at pre (a multiple of 8, at most 128), then the
// rest of the `total` bytes at msg; any alignment.
struct HashInput {
    const uint8_t *pre;
    const uint8_t *msg;
    size_t total;
    int plen;
};

// Shared words a warp's sixteen inputs are staged in: stream word w of the
// pair's current block, w <= 34, at k16_word(pair, w) (conflict-free for the
// 32 threads reading the same w or its neighbour).
constexpr int HASH16_STAGE_WORDS = 18 * K16_ROW;

__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// Starts copying the 136-byte block at byte `off` of a pair's input into its
// stage: the prefix's words, then the aligned words that hold the message's
// bytes (each holds one, so no copy can fault).  The copies run while the
// previous block is permuted; loading a block when it was needed, 17 words one
// after the other, took longer than permuting it (a 16 KB message: 2.2x).
__device__ __forceinline__ void hash16_fetch(const HashInput &in, size_t off, uint32_t stage, int pair, int p) {
    const int nblk = in.total - off < 136 ? (int)(in.total - off) : 136;   // input bytes in the block
    const int npre = off == 0 ? in.plen / 4 : 0;                           // prefix words in the block
    if (npre) {
        const bool aligned = (reinterpret_cast<uintptr_t>(in.pre) & 3) == 0;
        for (int w = p; w < npre; w += 2) {
            const uint32_t dst = stage + 4 * k16_word(pair, w);
            if (aligned)
                cp_async4(dst, in.pre + 4 * w);
            else
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst), "r"(ld_bytes4(in.pre + 4 * w, 4)) : "memory");
        }
    }
    const uint8_t *m = in.msg + (off == 0 ? 0 : off - in.plen);
    const int mis = (int)(reinterpret_cast<uintptr_t>(m) & 3);
    const int end = nblk > 4 * npre ? npre + (mis + nblk - 4 * npre + 3) / 4 : npre;
    const uint8_t *q = m - mis - 4 * npre;
    for (int w = p; w < end; w += 2)
        if (w >= npre) cp_async4(stage + 4 * k16_word(pair, w), q + 4 * w);
}

// XORs the staged, padded block at byte `off` of the input into the state
// halves of thread p of the pair (p = 0: low words).  True when it is the last.
__device__ __forceinline__ bool hash16_absorb(uint32_t (&a)[25], const HashInput &in, size_t off, uint32_t stage,
                                              int pair, int p) {
    const int left = in.total - off < 136 ? (int)(in.total - off) : 136;
    const int npre = off == 0 ? in.plen / 4 : 0;
    const int shift = 8 * (int)(reinterpret_cast<uintptr_t>(in.msg) & 3);   // prefix and blocks are whole words
    const uint32_t base = stage + 4 * k16_word(pair, p), next = stage + 4 * k16_word(pair, p + 1);
    const bool last = left < 136;
#pragma unroll
    for (int i = 0; i < 17; ++i) {
        uint32_t lo, hi;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(lo) : "r"(base + 4 * K16_ROW * i));
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(hi) : "r"(next + 4 * K16_ROW * i));
        uint32_t v = __funnelshift_r(lo, hi, 2 * i + p >= npre ? shift : 0);
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
// (thread p holds words 2 i + p of the output).  What done() writes to global
// memory may be the next input of the same pair.
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
            __threadfence_block();
            live = job.next(in);
            if (live) hash16_fetch(in, 0, stage, pair, p);
        }
    }
}

// Both threads of a pair: the even one's value.
__device__ __forceinline__ int pair_bcast(int v, int lane) {
    return __shfl_sync(3u << (lane & 30), v, lane & 30);
}

}  // namespace dil
