// Verify of a batch (Alg 3).
//
// Batch form.  One kernel hashes tr = H(pk) and mu = H(tr || M), sixteen tasks
// to a warp (in small batches, and for their long messages, a warp each).  Beside
// it, on a stream of their own where the caller has one to spare, run SampleInBall(c~), sixteen tasks to a warp, with ExpandA, sixteen
// polynomials to a warp whatever tasks they belong to (dil_sample16.cuh; not
// with a resident key's or the caller's A^), and then the arithmetic up to the
// packed w1', one task per warp.  The last kernel recomputes c~ = H(mu || w1'),
// sixteen tasks to a warp, and compares.  Hashing inside the task's own warp
// (k_verify, kept for the launch shapes a caller asks for) runs the 18 blocks of
// a Dilithium2 task at 18.7 SM clocks per round, 8.1 k of the task's 20.7 k
// clocks; sixteen to a warp they take 1.4 k.  Fused -> batch: 10,000 Dilithium2
// tasks 655 -> 399 us, 10,000 Dilithium5 with messages up to 4 KB 1810 -> 1202,
// thirteen Dilithium3 162 -> 87.  Sampling A^ takes 228 of the 399 us (ALU pipe),
// the arithmetic about 100 (latency of its loads and exchanges), the comparison 45.
#include "dil_kern.cuh"
#include "dil_sample16.cuh"

namespace dil {

template <int LEVEL, int P>
__global__ void __launch_bounds__(256, 4) k_verify(int n, const uint8_t *__restrict__ pk,
                                                   const uint8_t *__restrict__ msg,
                                                   const uint64_t *__restrict__ off,
                                                   const uint8_t *__restrict__ sig, uint8_t *ok, int32_t *scratch) {
    extern __shared__ __align__(16) uint8_t smem[];
    const CtaView v = cta_setup<P>(smem);
    const int task = blockIdx.x * v.groups + v.group;
    if (task >= n) return;
    using V = Lv<LEVEL>;
    uint64_t m0;
    size_t mlen;
    if (!message_of(off, task, m0, mlen)) {   // decreasing offsets: reject
        if (v.g == 0 && v.lane == 0) ok[task] = 0;
        return;
    }
    int r = verify_task<LEVEL, P>(pk + (size_t)task * V::PK, msg + m0, mlen,
                                  sig + (size_t)task * V::SIG,
                                  scratch + (size_t)task * Scratch<LEVEL>::VERIFY_POLYS * N, *v.gs, *v.ws, v.zt,
                                  v.izt, v.g, v.bar, v.lane);
    if (v.g == 0 && v.lane == 0) ok[task] = (uint8_t)r;
}

cudaError_t launch_verify(int level, int n, const uint8_t *pk, const uint8_t *msg, const uint64_t *off,
                          const uint8_t *sig, uint8_t *ok, int32_t *scratch, int warps, int p, cudaStream_t s) {
    DIL_DISPATCH_GROUPS(k_verify, pk, msg, off, sig, ok, scratch)
}

// ---------------------------------------------------------------- batch form

// Scratch polynomials of one task of the batch form: the packed w1', then A^.
template <int LEVEL, int SRC>
__host__ __device__ constexpr int verify_polys() {
    return SRC == VERIFY_PLAIN ? 1 + Lv<LEVEL>::K * Lv<LEVEL>::L : 1;
}

// Task t's message (and resident key); false when the task is to be rejected.
template <int SRC>
__device__ __forceinline__ bool verify_input(const VerifyBatch &b, int t, int &key, uint64_t &m0, size_t &mlen) {
    key = t;
    if (SRC == VERIFY_KEYED) {
        key = b.key_idx[t];
        if (key < 0 || key >= b.n_keys) return false;
    }
    return message_of(b.off, t, m0, mlen);
}

// tr = H(pk) (not for resident keys) and mu = H(tr || M) of a pair's tasks:
// the first by the pair's index, the next ones from the batch's counter.
template <int LEVEL, int SRC>
struct VerifyMuJob {
    static constexpr bool CHAINED = true;
    const VerifyBatch &b;
    int task, lane;
    bool first, have_tr;

    __device__ VerifyMuJob(const VerifyBatch &b_, int first_task, int lane_)
        : b(b_), task(first_task), lane(lane_), first(true), have_tr(false) {}

    __device__ __forceinline__ bool next(HashInput &in) {
        using V = Lv<LEVEL>;
        uint64_t m0 = 0;
        size_t mlen = 0;
        int key;
        if (!have_tr) {
            for (;;) {
                if (!first) {
                    const int claimed = b.hash_warps * K16_STATES;   // one for every pair to start with
                    if (b.n <= claimed) return false;                // (the counter is not set up either)
                    int c = 0;
                    if (!(lane & 1)) c = atomicAdd(b.next, 1);
                    task = claimed + pair_bcast(c, lane);
                }
                first = false;
                if (task >= b.n) return false;
                if (verify_input<SRC>(b, task, key, m0, mlen)) break;
            }
            if (SRC != VERIFY_KEYED) {
                in = {nullptr, b.pk + (size_t)task * V::PK, (size_t)V::PK, 0};
                return true;
            }
        }
        verify_input<SRC>(b, task, key, m0, mlen);
        const uint8_t *tr = SRC == VERIFY_KEYED ? b.key_tr + (size_t)key * 32
                                                : reinterpret_cast<const uint8_t *>(b.tr + (size_t)task * 8);
        in = {tr, b.msg + m0, 32 + mlen, 32};
        return true;
    }

    __device__ __forceinline__ void done(const uint32_t (&a)[25]) {
        const int p = lane & 1;
        if (SRC != VERIFY_KEYED && !have_tr) {   // the pair reads them back as the prefix of mu's input
#pragma unroll
            for (int i = 0; i < 4; ++i) b.tr[(size_t)task * 8 + 2 * i + p] = a[i];
            have_tr = true;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) b.mu[(size_t)task * 16 + 2 * i + p] = a[i];
            have_tr = false;
        }
    }
};

// tr and mu of one task, a warp of a CTA of W on the 25-lane form.
template <int LEVEL, int SRC, int W>
__device__ __forceinline__ void verify_hash_wide(const VerifyBatch &b, int task, int lane) {
    __shared__ __align__(16) uint8_t trs[W][32];
    uint8_t *tr = trs[W > 1 ? threadIdx.x >> 5 : 0];
    using V = Lv<LEVEL>;
    int key;
    uint64_t m0;
    size_t mlen;
    if (!verify_input<SRC>(b, task, key, m0, mlen)) return;
    uint32_t lo = 0, hi = 0;
    if (SRC == VERIFY_KEYED) {
        tr[lane] = b.key_tr[(size_t)key * 32 + lane];
    } else {
        absorb_concat(lo, hi, tr, 0, b.pk + (size_t)task * V::PK, V::PK, 136, lane);
        squeeze_words(lo, hi, tr, 4, lane);
    }
    __syncwarp();
    lo = 0;
    hi = 0;
    absorb_concat(lo, hi, tr, 32, b.msg + m0, mlen, 136, lane);
    squeeze_words(lo, hi, reinterpret_cast<uint8_t *>(b.mu + (size_t)task * 16), 8, lane);
}

// The hashing warps, each a CTA of its own: they are chains (a 16 KB message is
// 121 blocks, 3.8 us each on a warp of its own), so they get the registers to
// keep a state and its input (at 64, a block took 4.5 us) and start first.
template <int LEVEL, int SRC>
__global__ void __launch_bounds__(32, 16) k_verify_hash(const VerifyBatch b) {
    __shared__ __align__(16) uint32_t stage[HASH16_STAGE_WORDS];
    VerifyMuJob<LEVEL, SRC> job(b, blockIdx.x * K16_STATES + (threadIdx.x >> 1), threadIdx.x);
    hash16_run(job, stage, threadIdx.x);
}

// With wide warps for long messages (hash_split) behind them, four to a CTA, since
// the batch's other kernels wait until all these CTAs have started.  The pairs'
// warps have a CTA each, or (pair_ctas fewer than hash_warps) are four to a CTA,
// which keeps them off most SMs once ExpandA fills all: 2,400 Dilithium2 tasks of
// 1,000 bytes 191 -> 165 us, 3,000 of 16 KB 843 -> 658; but 800 of 1,000 bytes 119 ->
// 128 and, with resident keys, 2,000 of 16 KB 506 -> 531.
template <int LEVEL, int SRC>
__global__ void __launch_bounds__(128, 4) k_verify_hash_both(const VerifyBatch b) {
    __shared__ __align__(16) uint32_t stage[4][HASH16_STAGE_WORDS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (blockIdx.x < b.pair_ctas) {
        const int w = b.pair_ctas < b.hash_warps ? blockIdx.x * 4 + warp : warp ? b.hash_warps : blockIdx.x;
        if (w >= b.hash_warps) return;
        const int t = w * K16_STATES + (lane >> 1);   // the pair's only task
        VerifyMuJob<LEVEL, SRC> job(b, has_wide_warp(b.off, b.n, t, b.long_bytes, b.per_group) ? b.n : t, lane);
        hash16_run(job, stage[warp], lane);
    } else {
        const int w = (blockIdx.x - b.pair_ctas) * 4 + warp;
        const int task = task_of_wide_warp(b.off, b.n, w, b.long_bytes, b.per_group, lane);
        if (task >= 0) verify_hash_wide<LEVEL, SRC, 4>(b, task, lane);
    }
}

// For a small batch, a block per task only.  A kernel of its own: with the code
// above beside it thirteen Dilithium3 tasks take 92 us instead of 87.
template <int LEVEL, int SRC>
__global__ void __launch_bounds__(32) k_verify_hash_wide(const VerifyBatch b) {
    verify_hash_wide<LEVEL, SRC, 1>(b, blockIdx.x, threadIdx.x);
}

// c = SampleInBall(c~) of the signatures of tasks [first, first + 16), one warp.
template <int LEVEL>
__device__ __forceinline__ void verify_challenges(const VerifyBatch &b, int first, uint32_t *stage, int lane) {
    using V = Lv<LEVEL>;
    if (first >= b.n) return;
    const int t = first + (lane >> 1);
    const uint8_t *ct = b.sig + (size_t)(t < b.n ? t : first) * V::SIG + 4 * (lane & 1);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = ld_bytes4(ct + 8 * i, 4);
    challenge16<V::TAU>(w, t < b.n, stage, lane);
    for (int u = 0; u < K16_STATES && first + u < b.n; ++u)
        put_challenge(b.challenge + (size_t)(first + u) * 256, stage, u, lane);
}

// Blocks [0, challenge_blocks) draw challenges, the others (VERIFY_PLAIN only)
// sample A^.  One warp per CTA, as in Sign's prepare kernel.
template <int LEVEL>
__global__ void __launch_bounds__(32, 16) k_verify_sample(const VerifyBatch b) {
    __shared__ __align__(16) uint32_t sm[EXPAND16_WORDS];
    static_assert(CHALLENGE_WORDS <= EXPAND16_WORDS, "the challenge blocks' shared memory");
    using V = Lv<LEVEL>;
    const int lane = threadIdx.x, blk = blockIdx.x;
    if (blk < b.challenge_blocks) {
        verify_challenges<LEVEL>(b, blk * K16_STATES, sm, lane);
        return;
    }
    expand_a_batch<LEVEL, false>(
        (long long)(blk - b.challenge_blocks) * K16_STATES, (long long)b.n * V::K * V::L,
        [&](int t) { return b.pk + (size_t)t * V::PK; },
        [&](int t) { return b.scratch + ((size_t)t * verify_polys<LEVEL, VERIFY_PLAIN>() + 1) * N; }, sm, lane);
}

// Starts the lines of a byte range on their way into L2.
__device__ __forceinline__ void prefetch_l2(const void *p, int nbytes, int lane) {
    for (int at = 128 * lane; at < nbytes; at += 128 * 32)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const uint8_t *>(p) + at));
}

// The arithmetic of one task, a CTA of P warps (g: this one, with an exchange
// buffer of its own): hint decoding, z^, and per row
// w1' = UseHint(h, INTT(A^ z^ - c^ NTT(t1 2^d))), packed to the start of its
// scratch.  False when the signature is malformed or z too large.
template <int LEVEL, int SRC, int P>
__device__ __forceinline__ bool verify_rows(const VerifyBatch &b, int task, int key, int32_t *buf, int32_t *zh,
                                            uint32_t *hmask, int g, int lane) {
    using V = Lv<LEVEL>;
    const uint8_t *sig = b.sig + (size_t)task * V::SIG, *pk = b.pk + (size_t)key * V::PK;
    uint8_t *sq = reinterpret_cast<uint8_t *>(buf);
    int32_t v[8], ch[8];
    // unpacked polynomial by polynomial between transforms: without this each waits
    // for DRAM in turn (10,000 Dilithium2 tasks 418 -> 406 us, 50,000 1837 -> 1786;
    // A^ as well: no better, Dilithium5 0.4% worse)
    if (g == 0) prefetch_l2(sig, V::SIG, lane);
    if (SRC != VERIFY_KEYED && g == P - 1) prefetch_l2(pk, V::PK, lane);
    // strict hint decoding into bit masks
    bool bad = false;
    if (g == 0) {
        stage_bytes(sq, sig + V::SIG_H, V::OMEGA + V::K, lane);
        hmask[lane] = 0;
        hmask[32 + lane] = 0;
        __syncwarp();
        int prev = 0;
#pragma unroll 1
        for (int i = 0; i < V::K; ++i) {
            const int end = sq[V::OMEGA + i];
            if (end < prev || end > V::OMEGA) {
                bad = true;
                break;
            }
            for (int j = prev + lane; j < end; j += 32) {
                const int idx = sq[j];
                if (j > prev && idx <= sq[j - 1]) bad = true;
                atomicOr(&hmask[i * 8 + (idx >> 5)], 1u << (idx & 31));
            }
            prev = end;
        }
        if (!bad)
            for (int j = prev + lane; j < V::OMEGA; j += 32)
                if (sq[j]) bad = true;
        bad = __any_sync(FULL, bad);
        if (P == 1 && bad) return false;
    }
    // z^ = NTT(z), ||z|| < gamma1 - beta
#pragma unroll 1
    for (int j = g; j < V::L; j += P) {
        unpack_buf_l0<V::ZBITS>(v, sig + V::SIG_Z + j * V::POLYZ, V::GAMMA1, buf, lane);
#pragma unroll
        for (int m = 0; m < 8; ++m) bad |= iabs(v[m]) >= V::GAMMA1 - V::BETA;
        if (P == 1 && __any_sync(FULL, bad)) return false;
        ntt_fwd_global(v, buf);
        store_l2(zh + j * N, v, lane);   // read back by the same lane
    }
    if (P > 1 && __syncthreads_or(bad)) return false;   // and every warp's z^ and the hints are there
    const int8_t *c = reinterpret_cast<const int8_t *>(b.challenge) + (size_t)task * 256;
#pragma unroll
    for (int m = 0; m < 8; ++m) ch[m] = c[lane + 32 * m];
    ntt_fwd_global(ch, buf);
    int32_t *scr = b.scratch + (size_t)task * verify_polys<LEVEL, SRC>() * N;
    const int32_t *keyp = SRC == VERIFY_KEYED ? b.keys + (size_t)key * Scratch<LEVEL>::KEY_POLYS * N : nullptr;
    const int32_t *ah = SRC == VERIFY_KEYED  ? keyp + Scratch<LEVEL>::AH * N
                        : SRC == VERIFY_AHAT ? b.ahat + (size_t)task * V::K * V::L * N
                                             : scr + N;
#pragma unroll 1
    for (int i = g; i < V::K; i += P) {
        int32_t a[V::L][8];   // every load of the row in flight during t1's transform
#pragma unroll
        for (int j = 0; j < V::L; ++j) {
            if (SRC == VERIFY_AHAT) load_seq(a[j], ah + (i * V::L + j) * N, lane);
            else load_l2(a[j], ah + (i * V::L + j) * N, lane);
        }
        if (SRC == VERIFY_KEYED) {
            load_l2(v, keyp + (Scratch<LEVEL>::T1H + i) * N, lane);
        } else {
            unpack_buf_l0<10>(v, pk + 32 + i * V::POLYT1, 0, buf, lane);
#pragma unroll
            for (int m = 0; m < 8; ++m) v[m] = (-v[m]) << D;   // t1 2^d, t1 unpacked as 0 - field
            ntt_fwd_global(v, buf);
        }
        // summed in 64 bits, |sum| < 7 q 9.1q + 9.1q 9.1q < 2^31 q
        long long acc[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) acc[m] = -(long long)ch[m] * v[m];
#pragma unroll
        for (int j = 0; j < V::L; ++j) {
            load_l2(v, zh + j * N, lane);
#pragma unroll
            for (int m = 0; m < 8; ++m) acc[m] += (long long)a[j][m] * v[m];
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = mont_reduce(acc[m]);
        ntt_inv_global(v, buf);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const int hbit = (hmask[i * 8 + m] >> lane) & 1u;
            v[m] = use_hint<LEVEL>(hbit, to_canonical(v[m]));
        }
        l0_to_seq(v, buf, lane);
        pack_w1<LEVEL>(reinterpret_cast<uint8_t *>(scr) + i * V::POLYW1, v, lane);
    }
    return true;
}

// Resident warps: it waits for loads more than it issues.  10,000 and 50,000
// Dilithium2 tasks with 20, 24, 28, 32 of them: 407, 406, 401, 400 and 1808, 1786,
// 1760, 1748 us, 5,000 (28, 32) 230, 233; 10,000 Dilithium5 with 16, 20, 24: 1201,
// 1202, 1212.
template <int LEVEL, int SRC, int P>
__global__ void __launch_bounds__(32 * P, LEVEL != 2 ? 20 / P : P > 1 ? 32 / P : 28) k_verify_rows(const VerifyBatch b) {
    __shared__ __align__(16) int32_t bufs[P][288], zh[Lv<LEVEL>::L * N];
    __shared__ uint32_t hmask[64];
    const int task = blockIdx.x, g = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int key;
    uint64_t m0;
    size_t mlen;
    const bool r = verify_input<SRC>(b, task, key, m0, mlen) &&
                   verify_rows<LEVEL, SRC, P>(b, task, key, bufs[g], zh, hmask, g, lane);
    if (threadIdx.x == 0) b.ok[task] = r;   // 1: c~ decides (k_verify_compare)
}

// c~ = H(mu || w1') of task `pair` against the signature's.
template <int LEVEL, int SRC>
struct VerifyCompareJob {
    static constexpr bool CHAINED = false;
    const VerifyBatch &b;
    int task, lane;
    bool todo;

    __device__ VerifyCompareJob(const VerifyBatch &b_, int pair, int lane_)
        : b(b_), task(pair), lane(lane_), todo(pair < b_.n && b_.ok[pair]) {}

    __device__ __forceinline__ bool next(HashInput &in) {
        using V = Lv<LEVEL>;
        if (!todo) return false;
        todo = false;
        in = {reinterpret_cast<const uint8_t *>(b.mu + (size_t)task * 16),
              reinterpret_cast<const uint8_t *>(b.scratch + (size_t)task * verify_polys<LEVEL, SRC>() * N),
              64 + V::K * V::POLYW1, 64};
        return true;
    }

    __device__ __forceinline__ void done(const uint32_t (&a)[25]) {
        const uint8_t *ct = b.sig + (size_t)task * Lv<LEVEL>::SIG + 4 * (lane & 1);
        bool eq = true;
#pragma unroll
        for (int i = 0; i < 4; ++i) eq &= ld_bytes4(ct + 8 * i, 4) == a[i];
        const bool other = __shfl_xor_sync(3u << (lane & 30), eq, 1);
        if (!(eq && other) && !(lane & 1)) b.ok[task] = 0;
    }
};

template <int LEVEL, int SRC>
__global__ void __launch_bounds__(128) k_verify_compare(const VerifyBatch b) {
    __shared__ __align__(16) uint32_t stage[4][HASH16_STAGE_WORDS];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w * K16_STATES >= b.n) return;
    VerifyCompareJob<LEVEL, SRC> job(b, w * K16_STATES + (lane >> 1), lane);
    hash16_run(job, stage[threadIdx.x >> 5], lane);
}

// The same for a small batch, a warp per task on the 25-lane form.
template <int LEVEL, int SRC>
__global__ void __launch_bounds__(32) k_verify_compare_wide(const VerifyBatch b) {
    using V = Lv<LEVEL>;
    constexpr int W1 = V::K * V::POLYW1;
    __shared__ __align__(16) uint32_t in[(64 + W1) / 4 + 2];
    const int task = blockIdx.x, lane = threadIdx.x;
    if (!b.ok[task]) return;
    const uint32_t *w1 = reinterpret_cast<const uint32_t *>(b.scratch + (size_t)task * verify_polys<LEVEL, SRC>() * N);
    if (lane < 16) in[lane] = b.mu[(size_t)task * 16 + lane];
#pragma unroll
    for (int i = 0; i < W1 / 128; ++i) in[16 + lane + 32 * i] = w1[lane + 32 * i];
    __syncwarp();
    uint32_t lo = 0, hi = 0;
    absorb_smem(lo, hi, reinterpret_cast<const uint8_t *>(in), 64 + W1, 136, lane);
    bool eq = true;
    if (lane < 4) {
        const uint8_t *ct = b.sig + (size_t)task * V::SIG + 8 * lane;
        eq = ld_bytes4(ct, 4) == lo && ld_bytes4(ct + 4, 4) == hi;
    }
    if (!__all_sync(FULL, eq) && lane == 0) b.ok[task] = 0;
}

namespace {

// The lines of hash_split.  Up to `all` tasks the rows, too, have four warps a task
// and the comparison one: the rows of so few leave most of the GPU idle (13 tasks
// of 32 bytes on Dilithium5 keys 70 us with one warp, 55 with four, 608 77 and 65,
// 13 Dilithium2 verifies 71 and 60; 609 and more beside ExpandA gain nothing).
// Without sampling (a resident key's or the caller's A^) that line is two hashing
// warps to a sub-partition: 800 tasks of 4 KB on Dilithium2 keys 155 -> 138 us and
// 1,216 of 32 bytes 64 -> 56 with it at 1,216 instead of 608; at 1,824 1,700
// Dilithium3 of 32 bytes 73 -> 80.
// Beside sampling warps two threads to a state are slowed more, so shorter
// messages and larger batches have wide warps: Dilithium3 up to 4 KB 609, 1,000 and
// 1,824 tasks 244, 262, 364 -> 210, 248, 316 us with the line at 2 KB instead of 8;
// Dilithium2 of 4 KB 609 203 -> 187, 1,250 215 -> 219, 1,500 217 -> 233.  Once the
// sampling warps alone fill the GPU the hashing ones start late: 2,400 Dilithium2
// of 16 KB 824 -> 660 us with a warp each, 2,000 599 -> 643.
constexpr int FULL_GPU = 152 * 16;   // sampling warps
template <int LEVEL> bool sampling_fills_gpu(int n) {
    return (long long)n * Lv<LEVEL>::K * Lv<LEVEL>::L > (FULL_GPU - 152LL) * K16_STATES;
}
template <int LEVEL, int SRC>
HashLines verify_lines(int n) {
    if (SRC != VERIFY_PLAIN) return {1216, HASH_LONG_MOST, HASH_FEW_MOST, HASH_LONG_BYTES};
    return {HASH_WIDE_MOST, sampling_fills_gpu<LEVEL>(n) ? FULL_GPU : 1824, HASH_FEW_MOST_SAMPLING,
            LEVEL == 2 && n > 1250 ? HASH_LONG_BYTES : HASH_LONG_BYTES / 4};
}

template <int LEVEL, int SRC>
cudaError_t launch_batch(VerifyBatch b, const VerifyFork &f, cudaStream_t s) {
    const int most = verify_lines<LEVEL, SRC>(b.n).all;
    const HashSplit split = hash_split(b.n, b.n, verify_lines<LEVEL, SRC>(b.n));
    b.hash_warps = split.warps;
    b.long_bytes = split.long_bytes;
    b.per_group = split.per_group;
    b.pair_ctas = SRC == VERIFY_PLAIN && sampling_fills_gpu<LEVEL>(b.n) ? (split.warps + 3) / 4 : split.warps;
    b.challenge_blocks = (b.n + K16_STATES - 1) / K16_STATES;
    const cudaStream_t hs = f.stream ? f.stream : s;
    cudaError_t e = cudaSuccess;
    if (f.stream && ((e = cudaEventRecord(f.fork, s)) != cudaSuccess ||
                     (e = cudaStreamWaitEvent(hs, f.fork, 0)) != cudaSuccess))
        return e;
    if (split.warps && b.n > split.warps * K16_STATES &&
        (e = cudaMemsetAsync(b.next, 0, sizeof(int), hs)) != cudaSuccess)
        return e;
    if (!split.warps)
        k_verify_hash_wide<LEVEL, SRC><<<split.wide, 32, 0, hs>>>(b);
    else if (split.wide)
        k_verify_hash_both<LEVEL, SRC><<<b.pair_ctas + (split.wide + 3) / 4, 128, 0, hs>>>(b);
    else
        k_verify_hash<LEVEL, SRC><<<split.warps, 32, 0, hs>>>(b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const long long polys = SRC == VERIFY_PLAIN ? (long long)b.n * Lv<LEVEL>::K * Lv<LEVEL>::L : 0;
    k_verify_sample<LEVEL><<<b.challenge_blocks + (int)((polys + K16_STATES - 1) / K16_STATES), 32, 0, s>>>(b);
    e = cudaGetLastError();
    if (e == cudaSuccess) {
        if (b.n <= most)
            k_verify_rows<LEVEL, SRC, 4><<<b.n, 128, 0, s>>>(b);
        else
            k_verify_rows<LEVEL, SRC, 1><<<b.n, 32, 0, s>>>(b);
        e = cudaGetLastError();
    }
    // the caller's stream waits for the hashes whatever went wrong on it
    if (f.stream) {
        const cudaError_t r = cudaEventRecord(f.join, hs), w = cudaStreamWaitEvent(s, f.join, 0);
        if (e == cudaSuccess) e = r != cudaSuccess ? r : w;
    }
    if (e != cudaSuccess) return e;
    const HashGrid h = hash_grid(b.n);
    if (b.n <= most)
        k_verify_compare_wide<LEVEL, SRC><<<b.n, 32, 0, s>>>(b);
    else
        k_verify_compare<LEVEL, SRC><<<h.blocks, h.threads, 0, s>>>(b);
    return cudaGetLastError();
}

template <int LEVEL>
cudaError_t launch_batch_src(int src, const VerifyBatch &b, const VerifyFork &f, cudaStream_t s) {
    switch (src) {
        case VERIFY_PLAIN: return launch_batch<LEVEL, VERIFY_PLAIN>(b, f, s);
        case VERIFY_AHAT: return launch_batch<LEVEL, VERIFY_AHAT>(b, f, s);
        case VERIFY_KEYED: return launch_batch<LEVEL, VERIFY_KEYED>(b, f, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_verify_batch(int level, int src, const VerifyBatch &b, const VerifyFork &f, cudaStream_t s) {
    if (b.n <= 0) return cudaSuccess;
    switch (level) {
        case 2: return launch_batch_src<2>(src, b, f, s);
        case 3: return launch_batch_src<3>(src, b, f, s);
        case 5: return launch_batch_src<5>(src, b, f, s);
    }
    return cudaErrorInvalidValue;
}

size_t verify_batch_polys(int level, int src) {
    const int all = level == 2 ? verify_polys<2, VERIFY_PLAIN>() : level == 3 ? verify_polys<3, VERIFY_PLAIN>()
                                                                           : verify_polys<5, VERIFY_PLAIN>();
    return src == VERIFY_PLAIN ? all : 1;
}

size_t cta_smem_bytes(int warps, int p) { return cta_bytes(warps, p); }

template <int LEVEL>
static size_t polys_for(int op) {
    using S = Scratch<LEVEL>;
    return op == OP_KEYGEN ? S::GEN_POLYS : op == OP_SIGN ? S::SIGN_POLYS : S::VERIFY_POLYS;
}

size_t scratch_polys(int op, int level) {
    switch (level) {
        case 2: return polys_for<2>(op);
        case 3: return polys_for<3>(op);
        case 5: return polys_for<5>(op);
    }
    return 0;
}

}  // namespace dil
