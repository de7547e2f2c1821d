// ExpandA and ExpandS over the polynomials of a batch, sixteen to a warp
// whatever tasks they belong to, with the states in registers (dil_hash16.cuh).
#pragma once
#include "dil_hash16.cuh"
#include "dil_sample.cuh"

namespace dil {

// Shared words of a warp that samples sixteen polynomials at a time from whole
// squeezed streams: five 168-byte blocks (210 words) per state, which spaces
// the states' copies of one word over sixteen different pairs of banks, and
// the words that the last candidate slots beyond the blocks address.
constexpr int EXPAND16_STRIDE = 210;
constexpr int EXPAND16_WORDS = K16_STATES * EXPAND16_STRIDE + 8;

// ExpandA over a batch: polynomials [first, first + 16) of the `total` = tasks
// k l polynomials, numbered task by task, one warp.  seed_of(t): the 32 bytes
// of task t's rho (global memory, any alignment); out_of(t): task t's A^, in
// index order with INDEX, else in lane order.  BLOCKS: squeezed blocks taken at
// once (a test takes four, which never fill a polynomial).
// The states stay in registers over the five permutations; the blocks of all
// go to shared memory, and a lane then takes candidates lane + 32 m of one
// stream: 24 bits times 32 are whole words, so its shift is fixed and its
// word advances by 24.  (Voting on each block as it came, two states at a
// time, took a quarter of ExpandA's time.)  A stream of 280 candidates leaves
// fewer than 256 with probability below 1e-30; such a polynomial is sampled
// again by the form that squeezes until it has enough.
template <int LEVEL, bool INDEX, int BLOCKS = 5, class Seed, class Out>
__device__ __forceinline__ void expand_a_batch(long long first, long long total, Seed seed_of, Out out_of,
                                               uint32_t *st, int lane) {
    using V = Lv<LEVEL>;
    constexpr int KL = V::K * V::L;
    if (first >= total) return;
    const int s = lane >> 1, p = lane & 1;
    const long long at = first + s < total ? first + s : total - 1;
    const int task = (int)(at / KL), ij = (int)(at - (long long)task * KL);
    const uint8_t *rho = seed_of(task);
    uint32_t a[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) a[i] = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = ld_bytes4(rho + 8 * i + 4 * p, 4);
    if (!p) a[4] = (uint32_t)(ij % V::L) | ((uint32_t)(ij / V::L) << 8) | (0x1Fu << 16);
    if (p) a[20] = 0x80000000u;
#pragma unroll 1
    for (int blk = 0; blk < BLOCKS; ++blk) {
        hash16_permute(a, p);
#pragma unroll
        for (int i = 0; i < 21; ++i) st[s * EXPAND16_STRIDE + 42 * blk + 2 * i + p] = a[i];
    }
    __syncwarp();
    const int w0 = (24 * lane) >> 5, sh = (24 * lane) & 31;
    uint32_t few = 0;   // polynomials that the five blocks do not fill
#pragma unroll 1
    for (int u = 0; u < K16_STATES && first + u < total; ++u) {
        const int t = (int)((first + u) / KL);
        int32_t *dst = out_of(t) + (int)(first + u - (long long)t * KL) * N;
        const uint32_t *src = st + u * EXPAND16_STRIDE + w0;
        // the first 256 candidates all below q (0.78 of the polynomials): in place
        uint32_t v[9];
        bool all = 56 * BLOCKS >= N;
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            v[m] = __funnelshift_r(src[24 * m], src[24 * m + 1], sh) & 0x7FFFFFu;
            all = all && v[m] < (uint32_t)Q;
        }
        if (__all_sync(FULL, all)) {
            const int to = INDEX ? lane : lane_order(lane);   // candidate + 32: 32 or 16 words on
#pragma unroll
            for (int m = 0; m < 8; ++m) dst[to + (INDEX ? 32 : 16) * m] = (int32_t)v[m];
            continue;
        }
        v[8] = __funnelshift_r(src[192], src[193], sh) & 0x7FFFFFu;
        int c = 0;
#pragma unroll
        for (int m = 0; m < 9; ++m) {
            const bool acc = v[m] < (uint32_t)Q && (32 * m + 32 <= 56 * BLOCKS || 32 * m + lane < 56 * BLOCKS);
            const uint32_t mask = __ballot_sync(FULL, acc);
            const int to = c + __popc(mask & lanemask_lt(lane));
            if (acc && to < N) dst[INDEX ? to : lane_order(to)] = (int32_t)v[m];
            c += __popc(mask);
        }
        few |= (uint32_t)(c < N) << u;
    }
    if (!few) return;
    __syncwarp();
    uint8_t *seed = reinterpret_cast<uint8_t *>(st), *sq = seed + 32;
    int32_t *buf = reinterpret_cast<int32_t *>(st) + 64;
#pragma unroll 1
    for (int u = 0; u < K16_STATES; ++u) {
        if (!((few >> u) & 1u)) continue;
        const int t = (int)((first + u) / KL), q = (int)(first + u - (long long)t * KL);
        seed[lane] = seed_of(t)[lane];
        __syncwarp();
        expand_a_poly(seed, q / V::L, q % V::L, buf, sq, lane);
        for (int m = 0; m < 8; ++m)
            out_of(t)[q * N + (INDEX ? 8 * lane + m : lane_order(8 * lane + m))] = buf[9 * lane + m];
        __syncwarp();
    }
}

// As expand_a_batch for ExpandS: polynomials [first, first + 16) of the `total` =
// tasks (l + k), s1 then s2 of each task, coefficients in order.  seed_of(t):
// the 64 bytes of rho' (4-byte aligned); out_of(t): l + k polynomials.  Two
// blocks hold 544 candidates: always enough for eta = 2 (15 in 16 accepted),
// and for eta = 4 (9 in 16) in all but one polynomial of 10^5.
template <int LEVEL, class Seed, class Out>
__device__ __forceinline__ void expand_s_batch(long long first, long long total, Seed seed_of, Out out_of,
                                               uint32_t *st, int lane) {
    using V = Lv<LEVEL>;
    constexpr int KL = V::K + V::L;
    if (first >= total) return;
    const int s = lane >> 1, p = lane & 1;
    const long long at = first + s < total ? first + s : total - 1;
    const int task = (int)(at / KL), nonce = (int)(at - (long long)task * KL);
    const uint32_t *rhop = reinterpret_cast<const uint32_t *>(seed_of(task));
    uint32_t a[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) a[i] = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = rhop[2 * i + p];
    if (!p) a[8] = (uint32_t)nonce | (0x1Fu << 16);
    if (p) a[16] = 0x80000000u;
#pragma unroll 1
    for (int blk = 0; blk < 2; ++blk) {
        hash16_permute(a, p);
#pragma unroll
        for (int i = 0; i < 17; ++i) st[s * EXPAND16_STRIDE + 34 * blk + 2 * i + p] = a[i];
    }
    __syncwarp();
    uint32_t few = 0;
#pragma unroll 1
    for (int u = 0; u < K16_STATES && first + u < total; ++u) {
        const int t = (int)((first + u) / KL);
        int32_t *dst = out_of(t) + (int)(first + u - (long long)t * KL) * N;
        // candidate lane + 32 m: nibble lane mod 8 of word lane / 8 + 4 m
        const uint32_t *src = st + u * EXPAND16_STRIDE + (lane >> 3);
        int c = 0;
#pragma unroll 1
        for (int m = 0; m < 17 && c < N; ++m) {
            const uint32_t v = (src[4 * m] >> (4 * (lane & 7))) & 15u;
            const bool acc = V::ETA == 2 ? v < 15u : v < 9u;
            const uint32_t mask = __ballot_sync(FULL, acc);
            const int to = c + __popc(mask & lanemask_lt(lane));
            if (acc && to < N) dst[to] = V::ETA == 2 ? 2 - (int32_t)(v % 5u) : 4 - (int32_t)v;
            c += __popc(mask);
        }
        few |= (uint32_t)(c < N) << u;
    }
    if (!few) return;
    __syncwarp();
    uint8_t *seed = reinterpret_cast<uint8_t *>(st), *sq = seed + 64;
    int32_t *buf = reinterpret_cast<int32_t *>(st) + 64;
#pragma unroll 1
    for (int u = 0; u < K16_STATES; ++u) {
        if (!((few >> u) & 1u)) continue;
        const int t = (int)((first + u) / KL), q = (int)(first + u - (long long)t * KL);
        seed[lane] = seed_of(t)[lane];
        seed[lane + 32] = seed_of(t)[lane + 32];
        __syncwarp();
        expand_s_poly<V::ETA>(seed, q, buf, sq, lane);
        for (int m = 0; m < 8; ++m) out_of(t)[q * N + lane + 32 * m] = buf[lane + 36 * m];
        __syncwarp();
    }
}

}  // namespace dil
