// Sign of a batch in rounds (Alg 2).
//
// A prepare kernel hashes mu and rho' of every task, sixteen tasks to a warp (in
// small batches, and for their long messages, a warp each), while its other
// blocks sample A^ and transform s1, s2 and t0.  Then every round evaluates the
// next m repetitions of each unfinished task (an "attempt" each, in a slot of its
// own), phase by phase over the whole batch:
//   mask   y = ExpandMask: sixteen polynomials to a warp
//   front  y^, w = INTT(A^ y^), w1: a warp per attempt
//   hash   c~ = H(mu || w1) and SampleInBall: sixteen attempts to a warp
//   back   z, r0 and hint checks: a warp per attempt; the warp that finishes a
//          task's last attempt of the round writes the signature of the
//          smallest accepting repetition, or keeps the task for the next round
// m grows as tasks finish (round_reps), so the long tail of the rejection loop
// is evaluated in parallel and a round keeps filling the GPU.
// The host launches as many rounds as leave at most 0.02 tasks over in
// expectation (a launch of valid keys in fifty keeps one, and each of a batch's
// parts counts), and then a kernel that runs the plain loop on whatever is left.
//
// Against one fused kernel with a task per warp (dil_sign.cu): every hash runs
// at 3.2 SM clocks per round and state instead of 18.7 (c~) or with a third of
// its output unused (masks sampled sixteen nonces ahead), each kernel's code
// fits the instruction cache (the fused kernel's first stall is instruction
// fetch), and no SM idles while a few tasks run 20 to 30 repetitions one after
// the other.  Fused -> rounds: 10,000 Dilithium2 tasks 3396 -> 1525 us, 10,000
// Dilithium3 (32 B - 4 KB) 5350 -> 2340 us, 150 Dilithium5 1580 -> 340 to 375, one
// Dilithium2 task 176 -> 101 us (of 256 KB 5568 -> 5431; 7862 with two threads to
// its hash's state).
//
// What bounds the phases at 10,000 Dilithium2 tasks and 20,000 attempts: mask and
// prepare the ALU pipe (82 and 71%), hash its few warps' chains (57% of that pipe),
// front DRAM (59% of its peak), back its loads and issue slots (47%; 18 of 32 warps).
#include <algorithm>
#include <climits>

#include "dil_kern.cuh"
#include "dil_sample16.cuh"

namespace dil {

// ---------------------------------------------------------------- slots
// A slot holds one attempt: y (l polynomials, z replaces them), w (k), and one
// polynomial's room for the packed w1, later c (256 bytes), the hint masks and
// c~.
template <int LEVEL> struct Slot {
    using V = Lv<LEVEL>;
    static constexpr int Y = 0, W = V::L, X = V::L + V::K, POLYS = X + 1;
    static constexpr int XC = 0, XHINT = 256, XCT = 512;   // bytes within X, once w1 is hashed
};

constexpr int ROUND_MAX_REPS = 32;     // repetitions of one task in one round
constexpr int MAX_ROUNDS = 24;
// Attempts of a round that are worth having in flight, speculative ones included:
// a round of fewer takes almost as long (its hashes alone are a chain of eight
// permutations), more are only wasted repetitions.  10,000 Dilithium2 tasks with
// 10, 15, 20, 30 k slots: 1770, 1662, 1579, 1812 us; 150 Dilithium5 tasks with
// 1.2, 2.4, 3.6, 4.8 k: 422, 460, 409, 430 us; 1,000 of them: 954, 687, 725, 776.
template <int LEVEL> constexpr int round_fill() { return 152 * (LEVEL == 2 ? 32 : LEVEL == 3 ? 28 : 24); }
// The same for all of several batches that share the GPU: the rounds of one fill
// the gaps of the others', and their last rounds, of a few tasks each, come at
// the same time.  10,000 Dilithium2 tasks in four batches with 4.8, 9.7, 14.6 k:
// 1517, 1524, 1566 us; Dilithium3: 2270, 2233, 2233; 3,000 Dilithium2: 784, 672
// (9.7 k slots; 723 with 6 k), 666.
constexpr int ROUND_SHARED = 152 * 64;
constexpr int ROUND_MOST = 152 * 192;
// Repetitions of a task in one round that are worth their time on a full GPU:
// all of a task's are run though the first accepted one ends it.  100,000
// Dilithium2 tasks with 1, 2, 3, 4, 6, 32: 12.5, 12.5, 12.1, 12.0, 12.3, 12.8 ms;
// 10,000 with 3, 5, 32: 1535, 1524, 1591 us; 10,000 Dilithium3: 2271, 2233, 2326.
constexpr int ROUND_CAP = 5;

// Repetitions of each of `pending` tasks in a round: as many as there are slots
// for, but more than ROUND_CAP only up to `fill` attempts in all.
__host__ __device__ __forceinline__ int round_reps(int pending, int slots, int fill) {
    if (pending <= 0) return 0;
    const int worth = fill / pending > ROUND_CAP ? fill / pending : ROUND_CAP;
    int m = slots / pending;
    if (m > worth) m = worth;
    return m < 1 ? 1 : m > ROUND_MAX_REPS ? ROUND_MAX_REPS : m;
}

// Round r: unfinished tasks, repetitions of each, first of them.
struct Round {
    int p, m, base;
};
__device__ __forceinline__ Round round_of(const SignBatch &b, int r) {
    Round q{b.count[r], 0, 0};
    for (int i = 0; i < r; ++i) q.base += round_reps(b.count[i], b.slots, b.fill);
    q.m = round_reps(q.p, b.slots, b.fill);
    return q;
}

__device__ __forceinline__ const int *pending_list(const SignBatch &b, int r) {
    return b.pending + (size_t)(r & 1) * b.n;
}

template <int LEVEL>
__device__ __forceinline__ int32_t *slot_of(const SignBatch &b, int s) {
    return b.slot_polys + (size_t)s * Slot<LEVEL>::POLYS * N;
}

// The precomputation (A^, s^1, s^2, t^0) of task t.
template <int LEVEL, int SRC>
__device__ __forceinline__ const int32_t *pre_of(const SignBatch &b, int t) {
    if (SRC == SIGN_KEYED) return b.keys + (size_t)b.key_idx[t] * Scratch<LEVEL>::KEY_POLYS * N;
    return b.pre + (size_t)t * Scratch<LEVEL>::PRE_POLYS * N;
}

// A host cancel of the batch (seen through L2; any lane).
__device__ __forceinline__ bool canceled(const SignBatch &b) { return b.cancel && __ldcg(b.cancel) != 0; }

// Status and repetitions of a task without a signature.
__device__ __forceinline__ void report(const SignBatch &b, int task, int status, int iters) {
    if (b.status) b.status[task] = status;
    if (b.iters) b.iters[task] = iters;
}

// ---------------------------------------------------------------- prepare
// Task t's message (and resident key); false when the task is to be rejected.
template <int SRC>
__device__ __forceinline__ bool sign_input(const SignBatch &b, int t, int &key, uint64_t &m0, size_t &mlen) {
    key = t;
    if (SRC == SIGN_KEYED) {
        key = b.key_idx[t];
        if (key < 0 || key >= b.n_keys) return false;
    }
    return message_of(b.off, t, m0, mlen);
}

// A hashed task enters round 0 (one thread).
__device__ __forceinline__ void enter(const SignBatch &b, int task) {
    b.best[task] = INT_MAX;
    b.done[task] = 0;
    b.pending[atomicAdd(b.count, 1)] = task;
}

// mu = H(tr || M) and rho' = H(K || mu) of a pair's tasks: the first by the
// pair's index, the next ones from the batch's counter.  A task with an
// unknown key or decreasing offsets is rejected here (and one met after a cancel
// ends), every other one enters round 0.
template <int LEVEL, int SRC>
struct SignMuJob {
    static constexpr bool CHAINED = true;
    const SignBatch &b;
    int task, lane;
    bool first, have_mu;

    __device__ SignMuJob(const SignBatch &b_, int first_task, int lane_)
        : b(b_), task(first_task), lane(lane_), first(true), have_mu(false) {}

    __device__ __forceinline__ bool next(HashInput &in) {
        using V = Lv<LEVEL>;
        uint64_t m0 = 0;
        size_t mlen = 0;
        int key;
        if (have_mu) {   // rho' = H(K || mu)
            sign_input<SRC>(b, task, key, m0, mlen);
            in = {b.sk + (size_t)key * V::SK + 32, reinterpret_cast<const uint8_t *>(b.mu + (size_t)task * 16), 96, 32};
            return true;
        }
        for (;;) {
            if (!first) {
                const int claimed = b.hash_warps * K16_STATES;   // one for every pair to start with
                if (b.n <= claimed) return false;
                int c = 0;
                if (!(lane & 1)) c = atomicAdd(b.next, 1);
                task = claimed + pair_bcast(c, lane);
            }
            first = false;
            if (task >= b.n) return false;
            const bool valid = sign_input<SRC>(b, task, key, m0, mlen), stop = pair_bcast(canceled(b), lane);
            if (valid && !stop) break;
            uint8_t *sig = b.sig + (size_t)task * V::SIG;
            for (int i = lane & 1; i < V::SIG; i += 2) sig[i] = 0;
            if (!(lane & 1)) report(b, task, valid ? DIL_ECANCELED : DIL_EINVAL, 0);
        }
        in = {b.sk + (size_t)key * V::SK + 64, b.msg + m0, 32 + mlen, 32};
        return true;
    }

    __device__ __forceinline__ void done(const uint32_t (&a)[25]) {
        uint32_t *dst = (have_mu ? b.rhop : b.mu) + (size_t)task * 16 + (lane & 1);
#pragma unroll
        for (int i = 0; i < 8; ++i) dst[2 * i] = a[i];
        if (have_mu && !(lane & 1)) enter(b, task);
        have_mu = !have_mu;
    }
};

// The same for the task of a wide block, a warp on the 25-lane form (hash_split).
template <int LEVEL, int SRC>
__device__ __forceinline__ void sign_mu_wide(const SignBatch &b, int blk, uint32_t *sm, int lane) {
    using V = Lv<LEVEL>;
    const int task = b.hash_warps ? task_of_wide_warp(b.off, b.n, blk, b.long_bytes, b.per_group, lane) : blk;
    if (task < 0) return;
    uint8_t *in = reinterpret_cast<uint8_t *>(sm);   // tr, then K || mu
    uint64_t m0 = 0;
    size_t mlen = 0;
    int key;
    const bool valid = sign_input<SRC>(b, task, key, m0, mlen);
    if (!valid || __shfl_sync(FULL, canceled(b), 0)) {
        sign_zero<LEVEL, 1>(b.sig + (size_t)task * V::SIG, 0, lane);
        if (lane == 0) report(b, task, valid ? DIL_ECANCELED : DIL_EINVAL, 0);
        return;
    }
    const uint8_t *sk = b.sk + (size_t)key * V::SK;
    uint32_t lo = 0, hi = 0;
    stage_bytes(in, sk + 64, 32, lane);
    __syncwarp();
    absorb_concat(lo, hi, in, 32, b.msg + m0, mlen, 136, lane);
    squeeze_words(lo, hi, reinterpret_cast<uint8_t *>(b.mu + (size_t)task * 16), 8, lane);
    __syncwarp();
    stage_bytes(in, sk + 32, 32, lane);
    squeeze_words(lo, hi, in + 32, 8, lane);
    __syncwarp();
    lo = 0;
    hi = 0;
    absorb_smem(lo, hi, in, 96, 136, lane);
    squeeze_words(lo, hi, reinterpret_cast<uint8_t *>(b.rhop + (size_t)task * 16), 8, lane);
    if (lane == 0) enter(b, task);
}

// s^1, s^2, t^0 of one task (one warp).
template <int LEVEL>
__device__ __forceinline__ void sign_secrets(const uint8_t *sk, int32_t *pre, int32_t *buf, int lane) {
    using V = Lv<LEVEL>;
    using S = Scratch<LEVEL>;
    int32_t r[8];
#pragma unroll 1
    for (int u = 0; u < V::L + 2 * V::K; ++u) {
        if (u < V::L + V::K)
            unpack_buf_l0<V::ETABITS>(r, sk + V::SK_S1 + u * V::POLYETA, V::ETA, buf, lane);   // s1, then s2
        else
            unpack_buf_l0<D>(r, sk + V::SK_T0 + (u - V::L - V::K) * V::POLYT0, 1 << (D - 1), buf, lane);
        ntt_fwd_global(r, buf);
        store_l2(pre + (S::S1H + u) * N, r, lane);
    }
}

constexpr int ROUND_WARPS = 4;   // warps per CTA of the hashing and checking kernels

// One warp per CTA: a sampling warp's 11 to 13 KB of shared memory let sixteen
// be resident on an SM, and single warps spread over the SMs to within one (in
// fours, 2,500 mask warps made 625 CTAs for 608 places, a second wave of 17).
// Blocks [0, hash_warps) hash, [.., + wide_blocks) hash a long message each
// (WIDE, hash_split), [.., + expand_blocks) sample A^ (SIGN_AHAT:
// none), the rest transform the secrets (SIGN_KEYED: none), one task each; with
// SIGN_AHAT they also copy the caller's A^.
template <int LEVEL, int SRC, bool WIDE>
__global__ void __launch_bounds__(32, 16) k_sign_prepare(const SignBatch b) {
    extern __shared__ __align__(16) uint32_t sm[];
    using V = Lv<LEVEL>;
    constexpr int KL = V::K * V::L;
    const int lane = threadIdx.x;
    int blk = blockIdx.x;
    if (blk < b.hash_warps) {
        int t = blk * K16_STATES + (lane >> 1);   // with WIDE the pair's only task
        if (WIDE && has_wide_warp(b.off, b.n, t, b.long_bytes, b.per_group)) t = b.n;
        SignMuJob<LEVEL, SRC> job(b, t, lane);
        hash16_run(job, sm, lane);
        return;
    }
    blk -= b.hash_warps;
    if (WIDE) {
        if (blk < b.wide_blocks) {
            sign_mu_wide<LEVEL, SRC>(b, blk, sm, lane);
            return;
        }
        blk -= b.wide_blocks;
    }
    // canceled before this batch began: the hashing blocks reject every task
    if (b.stop && *b.stop) return;
    if constexpr (SRC != SIGN_KEYED) {
        if (blk < b.expand_blocks) {
            expand_a_batch<LEVEL, false>(
                (long long)blk * K16_STATES, (long long)b.n * KL, [&](int t) { return b.sk + (size_t)t * V::SK; },
                [&](int t) { return b.pre + (size_t)t * Scratch<LEVEL>::PRE_POLYS * N; }, sm, lane);
            return;
        }
        const int t = blk - b.expand_blocks;
        int32_t *pre = b.pre + (size_t)t * Scratch<LEVEL>::PRE_POLYS * N;
        if (SRC == SIGN_AHAT) copy_polys(b.ahat + (size_t)t * KL * N, 0, KL, pre, lane);
        sign_secrets<LEVEL>(b.sk + (size_t)t * V::SK, pre, reinterpret_cast<int32_t *>(sm), lane);
    }
}

// ---------------------------------------------------------------- mask
// Words of one state's five squeezed blocks (170), spaced so that the sixteen
// states' copies of the same word fall into sixteen different pairs of banks.
constexpr int MASK_STRIDE = 178;
constexpr int MASK_WORDS = K16_STATES * MASK_STRIDE;

template <int LEVEL>
__global__ void __launch_bounds__(32, 16) k_sign_mask(const SignBatch b, int r) {
    __shared__ __align__(16) uint32_t st[MASK_WORDS];
    using V = Lv<LEVEL>;
    const int lane = threadIdx.x;
    const Round q = round_of(b, r);
    // a state per polynomial: polynomial j of the attempt in slot i is the round's i l + j-th
    const int polys = q.p * q.m * V::L, first = blockIdx.x * K16_STATES;
    if (first >= polys) return;
    const int s = lane >> 1, p = lane & 1;
    const int mine = min(first + s, polys - 1), slot = mine / V::L, i = slot / q.m;
    const int rep = q.base + slot - i * q.m;
    const uint32_t *seed = b.rhop + (size_t)pending_list(b, r)[i] * 16;
    uint32_t a[25];
#pragma unroll
    for (int w = 0; w < 25; ++w) a[w] = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) a[w] = seed[2 * w + p];
    if (!p) a[8] = ((uint32_t)(V::L * rep + mine - slot * V::L) & 0xFFFFu) | (0x1Fu << 16);
    if (p) a[16] = 0x80000000u;
#pragma unroll 1
    for (int blk = 0; blk < 5; ++blk) {
        hash16_permute(a, p);
#pragma unroll
        for (int w = 0; w < 17; ++w) st[s * MASK_STRIDE + 34 * blk + 2 * w + p] = a[w];
    }
    __syncwarp();
    // fields: coefficient lane + 32 m starts at bit ZBITS lane + 32 ZBITS m, so
    // the shift is the lane's own and the word advances by ZBITS
    const int w0 = (V::ZBITS * lane) >> 5, sh = (V::ZBITS * lane) & 31;
#pragma unroll 1
    for (int u = 0; u < K16_STATES; ++u) {
        const int at = (first + u) / V::L;
        if (first + u >= polys) break;
        int32_t *dst = slot_of<LEVEL>(b, at) + (Slot<LEVEL>::Y + first + u - at * V::L) * N;
        const uint32_t *src = st + u * MASK_STRIDE + w0;
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const uint32_t f = __funnelshift_r(src[V::ZBITS * m], src[V::ZBITS * m + 1], sh);
            dst[lane + 32 * m] = V::GAMMA1 - (int32_t)(f & ((1u << V::ZBITS) - 1u));
        }
    }
}

// ---------------------------------------------------------------- front
// Two polynomials at a time share their twiddles and y^ (10,000 Dilithium3 tasks
// 2586 -> 2556 us, Dilithium5 3353 -> 3309, Dilithium2 unchanged: the kernel waits
// for DRAM more than for its transforms, 69% of the copy rate).
template <int LEVEL, int SRC>
__global__ void __launch_bounds__(32, 20) k_sign_front(const SignBatch b, int r) {
    __shared__ __align__(16) int32_t buf[2 * 288], yh[Lv<LEVEL>::L * N];
    using V = Lv<LEVEL>;
    using S = Scratch<LEVEL>;
    const Round q = round_of(b, r);
    const int attempts = q.p * q.m, s = blockIdx.x, lane = threadIdx.x;
    if (s >= attempts) return;
    const int32_t *pre = pre_of<LEVEL, SRC>(b, pending_list(b, r)[s / q.m]);
    int32_t *slot = slot_of<LEVEL>(b, s);
    int32_t v[2][8];
#pragma unroll 1
    for (int j = 0; j + 1 < V::L; j += 2) {
        load_l0(v[0], slot + (Slot<LEVEL>::Y + j) * N, lane);
        load_l0(v[1], slot + (Slot<LEVEL>::Y + j + 1) * N, lane);
        ntt_fwd_global(v, buf);
        store_l2(yh + j * N, v[0], lane);   // read back by the same lane
        store_l2(yh + (j + 1) * N, v[1], lane);
    }
    if (V::L % 2) {
        load_l0(v[0], slot + (Slot<LEVEL>::Y + V::L - 1) * N, lane);
        ntt_fwd_global(v[0], buf);
        store_l2(yh + (V::L - 1) * N, v[0], lane);
    }
    static_assert(V::K % 2 == 0, "rows in pairs");
#pragma unroll 1
    for (int i = 0; i < V::K; i += 2) {
        // the l products of a row are summed in 64 bits (|sum| < 7 q 9.1q < 2^31 q) and reduced once
        long long acc[2][8];
#pragma unroll
        for (int m = 0; m < 8; ++m) acc[0][m] = acc[1][m] = 0;
        const int32_t *row = pre + (S::AH + i * V::L) * N;
#pragma unroll
        for (int j = 0; j < V::L; ++j) {
            int32_t a0[8], a1[8], y[8];
            load_l2(a0, row + j * N, lane);
            load_l2(a1, row + (V::L + j) * N, lane);
            load_l2(y, yh + j * N, lane);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                acc[0][m] += (long long)a0[m] * y[m];
                acc[1][m] += (long long)a1[m] * y[m];
            }
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            v[0][m] = mont_reduce(acc[0][m]);
            v[1][m] = mont_reduce(acc[1][m]);
        }
        ntt_inv_global(v, buf);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            int32_t h[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                v[c][m] = to_canonical(v[c][m]);
                h[m] = highbits<LEVEL>(v[c][m]);
            }
            store_l0(slot + (Slot<LEVEL>::W + i + c) * N, v[c], lane);
            l0_to_seq(h, buf, lane);
            pack_w1<LEVEL>(reinterpret_cast<uint8_t *>(slot + Slot<LEVEL>::X * N) + (i + c) * V::POLYW1, h, lane);
        }
    }
}

// ---------------------------------------------------------------- hash
// c~ = H(mu || w1) of the attempt in slot `pair`.
template <int LEVEL>
struct SignCtJob {
    static constexpr bool CHAINED = false;
    const SignBatch &b;
    const uint8_t *mu, *w1;
    bool todo;
    uint32_t ct[4];

    __device__ __forceinline__ bool next(HashInput &in) {
        if (!todo) return false;
        todo = false;
        in = {mu, w1, 64 + Lv<LEVEL>::K * Lv<LEVEL>::POLYW1, 64};
        return true;
    }
    __device__ __forceinline__ void done(const uint32_t (&a)[25]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) ct[i] = a[i];
    }
};

template <int LEVEL>
__global__ void __launch_bounds__(32 * ROUND_WARPS, 4) k_sign_hash(const SignBatch b, int r) {
    __shared__ __align__(16) uint32_t sm[ROUND_WARPS][CHALLENGE_WORDS];
    using V = Lv<LEVEL>;
    using SL = Slot<LEVEL>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, pair = lane >> 1, p = lane & 1;
    const Round q = round_of(b, r);
    const int attempts = q.p * q.m, first = (blockIdx.x * (blockDim.x >> 5) + warp) * K16_STATES;
    if (first >= attempts) return;
    uint32_t *stage = sm[warp];
    const int s = first + pair;
    const bool mine = s < attempts;
    const int task = mine ? pending_list(b, r)[s / q.m] : 0;
    uint8_t *x = reinterpret_cast<uint8_t *>(slot_of<LEVEL>(b, mine ? s : first) + SL::X * N);
    SignCtJob<LEVEL> job{b, reinterpret_cast<const uint8_t *>(b.mu + (size_t)task * 16), x, mine, {0, 0, 0, 0}};
    hash16_run(job, stage, lane);
    if (mine) {
#pragma unroll
        for (int i = 0; i < 4; ++i) reinterpret_cast<uint32_t *>(x + SL::XCT)[2 * i + p] = job.ct[i];
    }
    challenge16<V::TAU>(job.ct, mine, stage, lane);
    // over the slot's w1, which every pair of the warp has absorbed
    for (int u = 0; u < K16_STATES && first + u < attempts; ++u)
        put_challenge(reinterpret_cast<uint8_t *>(slot_of<LEVEL>(b, first + u) + SL::X * N), stage, u, lane);
}

// The same for a small round, a warp per attempt on the 25-lane form.
template <int LEVEL>
__global__ void __launch_bounds__(32) k_sign_hash_wide(const SignBatch b, int r) {
    using V = Lv<LEVEL>;
    using SL = Slot<LEVEL>;
    constexpr int W1 = V::K * V::POLYW1;
    __shared__ __align__(16) uint32_t in[(64 + W1) / 4 + 2];
    __shared__ __align__(16) int32_t buf[288];
    __shared__ __align__(16) uint8_t sq[688], ct[32];
    const Round q = round_of(b, r);
    const int s = blockIdx.x, lane = threadIdx.x;
    if (s >= q.p * q.m) return;
    const int task = pending_list(b, r)[s / q.m];
    uint32_t *x = reinterpret_cast<uint32_t *>(slot_of<LEVEL>(b, s) + SL::X * N);
    if (lane < 16) in[lane] = b.mu[(size_t)task * 16 + lane];
#pragma unroll
    for (int i = 0; i < W1 / 128; ++i) in[16 + lane + 32 * i] = x[lane + 32 * i];
    __syncwarp();
    uint32_t lo = 0, hi = 0;
    absorb_smem(lo, hi, reinterpret_cast<const uint8_t *>(in), 64 + W1, 136, lane);
    squeeze_words(lo, hi, ct, 4, lane);
    __syncwarp();
    sample_in_ball<V::TAU>(ct, buf, sq, lane);
    int32_t c[8];
    read_buf_l0(c, buf, lane);
    int8_t *out = reinterpret_cast<int8_t *>(x);
#pragma unroll
    for (int m = 0; m < 8; ++m) out[SL::XC + lane + 32 * m] = (int8_t)c[m];
    if (lane < 8) x[SL::XCT / 4 + lane] = reinterpret_cast<const uint32_t *>(ct)[lane];
}

// ---------------------------------------------------------------- back
// v_s = INTT(c^ o s^2) in v, w in d: d = w - v_s (kept for the hint); true when
// r0 = LowBits(w - v_s) is too large.
template <int LEVEL>
__device__ __forceinline__ bool check_r0(const int32_t (&v)[8], int32_t (&d)[8]) {
    using V = Lv<LEVEL>;
    bool bad = false;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        int32_t e = d[m] - v[m];                 // (-q, 2q)
        e += (e < 0) ? Q : 0;
        e -= (e >= Q) ? Q : 0;
        int32_t h1, l0;
        decompose<LEVEL>(e, h1, l0);
        bad |= iabs(l0) >= V::GAMMA2 - V::BETA;
        d[m] = e;
    }
    return __any_sync(FULL, bad);
}

// INTT(c^ o s^1) in v, y in d: v = z; true when ||z|| >= gamma1 - beta.
template <int LEVEL>
__device__ __forceinline__ bool check_z(int32_t (&v)[8], const int32_t (&d)[8]) {
    using V = Lv<LEVEL>;
    bool bad = false;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        v[m] = centre_small(to_canonical(v[m]) + d[m]);
        bad |= iabs(v[m]) >= V::GAMMA1 - V::BETA;
    }
    return __any_sync(FULL, bad);
}

// v_t = INTT(c^ o t^0) in v, w - v_s in d: h = MakeHint(-v_t, w - v_s + v_t) into
// eight masks, its ones added to count; true when ||v_t|| >= gamma2.
template <int LEVEL>
__device__ __forceinline__ bool check_hint(const int32_t (&v)[8], const int32_t (&d)[8], uint32_t *hint, int &count,
                                           int lane) {
    using V = Lv<LEVEL>;
    bool bad = false;
    uint32_t hbits = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        int32_t vt = to_canonical(v[m]);
        bad |= iabs(to_centred(vt)) >= V::GAMMA2;
        int32_t rr = d[m] + vt;
        rr -= (rr >= Q) ? Q : 0;
        int32_t z = vt ? Q - vt : 0;
        hbits |= (uint32_t)make_hint<LEVEL>(z, rr) << m;
    }
    if (__any_sync(FULL, bad)) return true;
    uint32_t mine = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const uint32_t x = __ballot_sync(FULL, (hbits >> m) & 1u);
        if (lane == m) mine = x;
        count += __popc(x);
    }
    if (lane < 8) hint[lane] = mine;
    return false;
}

// The hint masks of a slot, eight words per polynomial.
template <int LEVEL>
__device__ __forceinline__ uint32_t *hint_of(int32_t *slot) {
    return reinterpret_cast<uint32_t *>(slot + Slot<LEVEL>::X * N) + Slot<LEVEL>::XHINT / 4;
}

// The checks of the attempt in `slot` with challenge ch (L2 layout); z
// replaces y, the hint masks go behind the challenge.  True when accepted.
// One loop over the r0 polynomials (LowBits(w - c s2)), then z = y + c s1, then
// the hints (c t0), so that the transform exists once: r0 first, since its
// polynomials reject more often (Dilithium3: 0.17 against 0.09 each; 5.3
// transforms an attempt instead of 6.6).
template <int LEVEL>
__device__ __forceinline__ bool sign_checks(const int32_t *pre, int32_t *slot, const int32_t (&ch)[8], int32_t *buf,
                                            const int32_t *izt, int lane) {
    using V = Lv<LEVEL>;
    using S = Scratch<LEVEL>;
    using SL = Slot<LEVEL>;
    constexpr int R0 = V::K, ZS = V::K + V::L, ALL = 2 * V::K + V::L;   // ends of the three parts
    static_assert(SL::W == SL::Y + V::L, "w behind y");
    uint32_t *hint = hint_of<LEVEL>(slot);
    int32_t v[8], a[8], d[8];
    int count = 0;
#pragma unroll 1
    for (int u = 0; u < ALL; ++u) {
        int32_t *data = slot + (u < R0 ? SL::W + u : SL::Y + u - R0) * N;   // w, y, w again
        load_l2(a, pre + (u < R0 ? S::S2H + u : u < ZS ? S::S1H + u - R0 : S::T0H + u - ZS) * N, lane);
        load_l0(d, data, lane);
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = mont_mul(ch[m], a[m]);
        ntt_inv(v, buf, izt, lane);
        if (u < R0) {
            if (check_r0<LEVEL>(v, d)) return false;
            store_l0(data, d, lane);
        } else if (u < ZS) {
            if (check_z<LEVEL>(v, d)) return false;
            store_l0(data, v, lane);
        } else if (check_hint<LEVEL>(v, d, hint + (u - ZS) * 8, count, lane)) {
            return false;
        }
    }
    return count <= V::OMEGA;
}

// sig = c~ || z || h of the accepted attempt in `slot` (read through L2:
// another warp may have written it).
template <int LEVEL>
__device__ __forceinline__ void sign_emit(uint8_t *sig, const int32_t *slot, int32_t *buf, int lane) {
    using V = Lv<LEVEL>;
    using SL = Slot<LEVEL>;
#pragma unroll 1
    for (int j = 0; j < V::L; ++j) {
        int32_t v[8];
        load_seq_cg(v, slot + (SL::Y + j) * N, lane);   // 8 consecutive coefficients
        pack_poly<V::ZBITS>(sig + V::SIG_Z + j * V::POLYZ, v, V::GAMMA1, -1, buf, lane);
    }
    const uint8_t *x = reinterpret_cast<const uint8_t *>(slot + SL::X * N);
    sig[lane] = __ldcg(x + SL::XCT + lane);
    const uint32_t *hint = reinterpret_cast<const uint32_t *>(x + SL::XHINT);
    uint8_t *h = sig + V::SIG_H;
    int base = 0;
#pragma unroll 1
    for (int i = 0; i < V::K; ++i) {
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const uint32_t w = __ldcg(hint + i * 8 + m);
            if ((w >> lane) & 1u) h[base + __popc(w & lanemask_lt(lane))] = (uint8_t)(lane + 32 * m);
            base += __popc(w);
        }
        if (lane == 0) h[V::OMEGA + i] = (uint8_t)base;
    }
    for (int p = base + lane; p < V::OMEGA; p += 32) h[p] = 0;
}

// Task `task` (i-th of round r) after the last of its attempts: its signature,
// the cap, a cancel, or the next round.
template <int LEVEL>
__device__ __forceinline__ void settle(const SignBatch &b, const Round &q, int r, int i, int task, int best, int32_t *buf,
                                       int lane) {
    using V = Lv<LEVEL>;
    uint8_t *sig = b.sig + (size_t)task * V::SIG;
    if (best != INT_MAX) {
        sign_emit<LEVEL>(sig, slot_of<LEVEL>(b, i * q.m + best - q.base), buf, lane);
        if (lane == 0) report(b, task, DIL_OK, best + 1);
        return;
    }
    const bool capped = q.base + q.m >= b.max_iter;
    if (__shfl_sync(FULL, capped || canceled(b), 0)) {
        sign_zero<LEVEL, 1>(sig, 0, lane);
        if (lane == 0) report(b, task, capped ? DIL_EITER : DIL_ECANCELED, capped ? b.max_iter : 0);
    } else if (lane == 0) {
        b.done[task] = 0;
        int *list = b.pending + (size_t)((r + 1) & 1) * b.n;
        list[atomicAdd(b.count + r + 1, 1)] = task;
    }
}

// One warp per attempt, after its checks (what they wrote has been fenced: it is
// read through L2): the last of the task's attempts settles the round.  What an
// accepted one wrote is visible before its repetition, and that before its
// arrival.
template <int LEVEL>
__device__ __forceinline__ void arrive(const SignBatch &b, const Round &q, int r, int i, int task, int rep,
                                       bool accepted, int32_t *buf, int lane) {
    int best = accepted ? rep : INT_MAX;
    if (q.m > 1) {
        int arrived = 0;
        if (lane == 0) {
            if (accepted) {
                atomicMin(&b.best[task], rep);
                __threadfence();
            }
            arrived = atomicAdd(&b.done[task], 1);
        }
        if (__shfl_sync(FULL, arrived, 0) != q.m - 1) return;
        __threadfence();
        if (lane == 0) best = atomicOr(&b.best[task], 0);
        best = __shfl_sync(FULL, best, 0);
    }
    settle<LEVEL>(b, q, r, i, task, best, buf, lane);
}

template <int LEVEL, int SRC>
__global__ void __launch_bounds__(32 * ROUND_WARPS, 8) k_sign_back(const SignBatch b, int r) {
    __shared__ __align__(16) int32_t tables[2 * NTT_TABLE_WORDS], bufs[ROUND_WARPS][288];
    const Round q = round_of(b, r);
    const int attempts = q.p * q.m;
    if ((int)blockIdx.x * ROUND_WARPS >= attempts) return;
    load_zetas(tables);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, s = blockIdx.x * ROUND_WARPS + warp;
    if (s >= attempts) return;
    int32_t *buf = bufs[warp], *zt = tables, *izt = tables + NTT_TABLE_WORDS;
    const int i = s / q.m, task = pending_list(b, r)[i], rep = q.base + s - i * q.m;
    int32_t *slot = slot_of<LEVEL>(b, s);
    // a repetition past the cap, or past one that has been accepted, is not looked at
    int skip = 0;
    if (lane == 0) skip = rep >= b.max_iter || (q.m > 1 && atomicOr(&b.best[task], 0) < rep);
    bool accepted = false;
    if (!__shfl_sync(FULL, skip, 0)) {
        int32_t ch[8];
        const int8_t *c = reinterpret_cast<const int8_t *>(slot + Slot<LEVEL>::X * N);
#pragma unroll
        for (int m = 0; m < 8; ++m) ch[m] = c[lane + 32 * m];
        ntt_fwd(ch, buf, zt, lane);
        accepted = sign_checks<LEVEL>(pre_of<LEVEL, SRC>(b, task), slot, ch, buf, izt, lane);
    }
    if (accepted) __threadfence();
    __syncwarp();
    arrive<LEVEL>(b, q, r, i, task, rep, accepted, buf, lane);
}

// The same for a small round, four warps per attempt: its checks are 2 k + l
// transforms in a row on a warp of its own (20 us for Dilithium2), a quarter of
// that here, and the SMs have the room.
template <int LEVEL, int SRC>
__global__ void __launch_bounds__(128) k_sign_back_wide(const SignBatch b, int r) {
    __shared__ __align__(16) int32_t tables[2 * NTT_TABLE_WORDS], bufs[4][288];
    __shared__ int hints;
    using V = Lv<LEVEL>;
    using S = Scratch<LEVEL>;
    using SL = Slot<LEVEL>;
    const Round q = round_of(b, r);
    const int s = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (s >= q.p * q.m) return;
    load_zetas(tables);
    if (threadIdx.x == 0) hints = 0;
    __syncthreads();
    int32_t *buf = bufs[warp], *zt = tables, *izt = tables + NTT_TABLE_WORDS;
    const int i = s / q.m, task = pending_list(b, r)[i], rep = q.base + s - i * q.m;
    int32_t *slot = slot_of<LEVEL>(b, s);
    const int32_t *pre = pre_of<LEVEL, SRC>(b, task);
    bool bad = threadIdx.x == 0 && (rep >= b.max_iter || (q.m > 1 && atomicOr(&b.best[task], 0) < rep));
    bool accepted = !__syncthreads_or(bad);
    if (accepted) {
        int32_t ch[8];
        const int8_t *c = reinterpret_cast<const int8_t *>(slot + SL::X * N);
#pragma unroll
        for (int m = 0; m < 8; ++m) ch[m] = c[lane + 32 * m];
        ntt_fwd(ch, buf, zt, lane);
        // r0, z and hint polynomials in turn, a quarter of each to a warp
#pragma unroll 1
        for (int part = 0; part < 3 && accepted; ++part) {
            const int polys = part == 1 ? V::L : V::K;
            bad = false;
#pragma unroll 1
            for (int u = warp; u < polys && !bad; u += 4) {
                int32_t v[8], a[8], d[8];
                load_l2(a, pre + ((part == 0 ? S::S2H : part == 1 ? S::S1H : S::T0H) + u) * N, lane);
                int32_t *data = slot + ((part == 1 ? SL::Y : SL::W) + u) * N;
                load_l0(d, data, lane);
#pragma unroll
                for (int m = 0; m < 8; ++m) v[m] = mont_mul(ch[m], a[m]);
                ntt_inv(v, buf, izt, lane);
                if (part == 0) {
                    bad = check_r0<LEVEL>(v, d);
                    if (!bad) store_l0(data, d, lane);
                } else if (part == 1) {
                    bad = check_z<LEVEL>(v, d);
                    if (!bad) store_l0(data, v, lane);
                } else {
                    int count = 0;
                    bad = check_hint<LEVEL>(v, d, hint_of<LEVEL>(slot) + 8 * u, count, lane);
                    if (!bad && lane == 0) atomicAdd(&hints, count);
                }
            }
            accepted = !__syncthreads_or(bad);
        }
        accepted = accepted && *(volatile int *)&hints <= V::OMEGA;
    }
    // every warp of the CTA has written its part by the last barrier; warp 0 settles
    if (accepted) __threadfence();
    __syncthreads();
    if (warp == 0) arrive<LEVEL>(b, q, r, i, task, rep, accepted, buf, lane);
}

// ---------------------------------------------------------------- what is left
// The plain loop over the tasks still unfinished after round r - 1, from
// round r's first repetition on, one task per warp; the slots are its scratch.
// Of valid keys it is a task now and then; a damaged key may hold its task here
// for thousands of repetitions, and such tasks may be a whole batch, so there are
// as many warps as tasks, slots and the GPU allow (704 Dilithium2 tasks that hardly
// ever accept, up to 400 repetitions: 204 ms on 64 warps, 26 with two warps to each,
// 22 with one; 10,000: 823, 259, 130).
template <int LEVEL, int SRC>
__global__ void __launch_bounds__(256, 4) k_sign_rest(const SignBatch b, int r, int workers) {
    extern __shared__ __align__(16) uint8_t smem[];
    using V = Lv<LEVEL>;
    if (b.stop && blockIdx.x == 0 && threadIdx.x == 0 && canceled(b)) *b.stop = 1;   // for the next batch in line
    if (b.count[r] <= 0) return;
    const Round q = round_of(b, r);
    const CtaView v = cta_setup<1>(smem);
    const int w = blockIdx.x * v.groups + v.group;
    if (w >= workers) return;
    int32_t *itr = b.slot_polys + (size_t)w * Scratch<LEVEL>::ITR_POLYS * N;
    for (int i = w; i < q.p; i += workers) {
        const int task = pending_list(b, r)[i];
        const int32_t *pre = pre_of<LEVEL, SRC>(b, task);
        if (v.lane < 16) {
            reinterpret_cast<uint32_t *>(v.gs->hb + HB_MU)[v.lane] = b.mu[(size_t)task * 16 + v.lane];
            reinterpret_cast<uint32_t *>(v.gs->rhop)[v.lane] = b.rhop[(size_t)task * 16 + v.lane];
        }
        __syncwarp();
        int it = q.base;
        bool ok = false, stop = false;
        MaskStream ms{0, 0};
        while (it < b.max_iter && !(stop = __shfl_sync(FULL, canceled(b), 0))) {
            ok = sign_attempt<LEVEL, 1>(it * V::L, pre, itr, ms, *v.gs, *v.ws, v.zt, v.izt, 0, v.bar, v.lane);
            ++it;
            if (ok) break;
        }
        uint8_t *sig = b.sig + (size_t)task * V::SIG;
        if (ok)
            sign_pack<LEVEL, 1>(sig, itr, *v.gs, 0, v.lane);
        else
            sign_zero<LEVEL, 1>(sig, 0, v.lane);
        if (v.lane == 0) report(b, task, ok ? DIL_OK : stop ? DIL_ECANCELED : DIL_EITER, !ok && stop ? 0 : it);
        __syncwarp();
    }
}

// ---------------------------------------------------------------- host side
namespace {

// Mean acceptance of one repetition (Alg 2; 1 / 4.25, 1 / 5.1, 1 / 3.85).
double accept_of(int level) { return level == 2 ? 1 / 4.25 : level == 3 ? 1 / 5.1 : 1 / 3.85; }

constexpr int CTL_WORDS = 64;   // the hashing warps' counter, then the rounds' task counts
static_assert(MAX_ROUNDS + 3 <= CTL_WORDS, "a count per round, the counter and the round after the last");

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

template <int LEVEL>
int min_slots() { return (Scratch<LEVEL>::ITR_POLYS + Slot<LEVEL>::POLYS - 1) / Slot<LEVEL>::POLYS; }

struct Layout {
    size_t pre, slots, mu, rhop, pending, best, done, ctl, total;
};

template <int LEVEL>
Layout layout_of(int src, size_t n, size_t slots) {
    Layout L;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t here = at;
        at += al256(bytes);
        return here;
    };
    L.pre = take(src == SIGN_KEYED ? 0 : n * Scratch<LEVEL>::PRE_POLYS * N * 4);
    L.slots = take(slots * Slot<LEVEL>::POLYS * N * 4);
    L.mu = take(64 * n);
    L.rhop = take(64 * n);
    L.pending = take(8 * n);
    L.best = take(4 * n);
    L.done = take(4 * n);
    L.ctl = take(4 * CTL_WORDS);
    L.total = at;
    return L;
}

// Attempts worth having in flight in a batch that has 1 / parts of the GPU.
template <int LEVEL> int fill_of(int parts) { return parts > 1 ? ROUND_SHARED / parts : round_fill<LEVEL>(); }

// Rounds after which fewer than 0.02 tasks are expected to be left.
int rounds_of(int level, int n, const SignBatch &b) {
    double left = n;
    int r = 0;
    while (left > 0.02 && r < MAX_ROUNDS) {
        const int m = round_reps(left < 1 ? 1 : (int)left, b.slots, b.fill);
        for (int i = 0; i < m; ++i) left *= 1 - accept_of(level);
        ++r;
    }
    return r;
}

template <class Kern>
cudaError_t dynamic_smem(Kern kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

int blocks_for(long long items, int per) { return (int)((items + per - 1) / per); }

template <int LEVEL, int SRC>
cudaError_t launch_rounds(SignBatch b, void *ws, cudaStream_t s) {
    using V = Lv<LEVEL>;
    const Layout L = layout_of<LEVEL>(SRC, b.n, b.slots);
    uint8_t *base = static_cast<uint8_t *>(ws);
    b.pre = reinterpret_cast<int32_t *>(base + L.pre);
    b.slot_polys = reinterpret_cast<int32_t *>(base + L.slots);
    b.mu = reinterpret_cast<uint32_t *>(base + L.mu);
    b.rhop = reinterpret_cast<uint32_t *>(base + L.rhop);
    b.pending = reinterpret_cast<int *>(base + L.pending);
    b.best = reinterpret_cast<int *>(base + L.best);
    b.done = reinterpret_cast<int *>(base + L.done);
    b.next = reinterpret_cast<int *>(base + L.ctl);
    b.count = b.next + 1;
    b.fill = fill_of<LEVEL>(b.parts);
    cudaError_t e = cudaMemsetAsync(b.next, 0, 4 * CTL_WORDS, s);
    if (e != cudaSuccess) return e;

    // prepare
    const HashSplit split = hash_split(b.n, b.on_gpu, {HASH_WIDE_MOST, HASH_LONG_MOST, HASH_LONG_MOST, HASH_LONG_BYTES});
    b.hash_warps = split.warps;
    b.wide_blocks = split.wide;
    b.long_bytes = split.long_bytes;
    b.per_group = split.per_group;
    b.expand_blocks = SRC == SIGN_PLAIN ? blocks_for((long long)b.n * V::K * V::L, K16_STATES) : 0;
    const int secret_blocks = SRC == SIGN_KEYED ? 0 : b.n;
    const size_t prep_smem = 4 * (SRC == SIGN_PLAIN ? EXPAND16_WORDS : HASH16_STAGE_WORDS);
    static_assert(288 <= HASH16_STAGE_WORDS && HASH16_STAGE_WORDS <= EXPAND16_WORDS, "every block's shared memory");
    const auto prepare = split.wide ? k_sign_prepare<LEVEL, SRC, true> : k_sign_prepare<LEVEL, SRC, false>;
    if ((e = dynamic_smem(prepare, prep_smem)) != cudaSuccess) return e;
    prepare<<<b.hash_warps + b.wide_blocks + b.expand_blocks + secret_blocks, 32, prep_smem, s>>>(b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;

    const int rounds = rounds_of(LEVEL, b.n, b);
    const int most = b.slots;   // attempts of a round; blocks beyond the actual count return at once
    const HashGrid h = hash_grid(most);
    for (int r = 0; r < rounds; ++r) {
        k_sign_mask<LEVEL><<<blocks_for((long long)most * V::L, K16_STATES), 32, 0, s>>>(b, r);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_sign_front<LEVEL, SRC><<<most, 32, 0, s>>>(b, r);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (most <= HASH_WIDE_MOST)
            k_sign_hash_wide<LEVEL><<<most, 32, 0, s>>>(b, r);
        else
            k_sign_hash<LEVEL><<<h.blocks, h.threads, 0, s>>>(b, r);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (most <= HASH_WIDE_MOST)
            k_sign_back_wide<LEVEL, SRC><<<most, 128, 0, s>>>(b, r);
        else
            k_sign_back<LEVEL, SRC><<<blocks_for(most, ROUND_WARPS), 32 * ROUND_WARPS, 0, s>>>(b, r);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const long long room = (long long)b.slots * Slot<LEVEL>::POLYS / Scratch<LEVEL>::ITR_POLYS, gpu = 152 * 16;
    const int workers = (int)std::min({room, gpu, (long long)b.n}), ctas = blocks_for(workers, 4);
    const size_t rest_smem = cta_bytes(4, 1);
    if ((e = dynamic_smem(k_sign_rest<LEVEL, SRC>, rest_smem)) != cudaSuccess) return e;
    k_sign_rest<LEVEL, SRC><<<ctas, 128, rest_smem, s>>>(b, rounds, workers);
    return cudaGetLastError();
}

template <int LEVEL>
cudaError_t launch_src(int src, const SignBatch &b, void *ws, cudaStream_t s) {
    switch (src) {
        case SIGN_PLAIN: return launch_rounds<LEVEL, SIGN_PLAIN>(b, ws, s);
        case SIGN_AHAT: return launch_rounds<LEVEL, SIGN_AHAT>(b, ws, s);
        case SIGN_KEYED: return launch_rounds<LEVEL, SIGN_KEYED>(b, ws, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// Slots of a batch that has 1 / parts of the GPU: one per task at least, and for
// further repetitions up to ROUND_MAX_REPS per task within the fill, two per
// task within ROUND_MOST.
template <int LEVEL>
static int slots_of(int n, int parts) {
    const long long fill = fill_of<LEVEL>(parts), most = ROUND_MOST / parts;
    long long s = (long long)n * ROUND_MAX_REPS;
    if (s > fill) s = 2LL * n > fill ? 2LL * n : fill;
    if (s > most) s = n > most ? n : most;
    return (int)(s < min_slots<LEVEL>() ? min_slots<LEVEL>() : s);
}

int sign_batch_slots(int level, int n, int parts) {
    return level == 2 ? slots_of<2>(n, parts) : level == 3 ? slots_of<3>(n, parts) : slots_of<5>(n, parts);
}

size_t sign_batch_bytes(int level, int src, size_t n, size_t slots) {
    return level == 2   ? layout_of<2>(src, n, slots).total
           : level == 3 ? layout_of<3>(src, n, slots).total
                        : layout_of<5>(src, n, slots).total;
}

int sign_batch_min_slots(int level, int n) {
    const int least = level == 2 ? min_slots<2>() : level == 3 ? min_slots<3>() : min_slots<5>();
    return n > least ? n : least;
}

cudaError_t launch_sign_batch(int level, int src, const SignBatch &b, void *ws, cudaStream_t s) {
    if (b.n <= 0) return cudaSuccess;
    if (b.slots < sign_batch_min_slots(level, b.n)) return cudaErrorInvalidValue;
    switch (level) {
        case 2: return launch_src<2>(src, b, ws, s);
        case 3: return launch_src<3>(src, b, ws, s);
        case 5: return launch_src<5>(src, b, ws, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace dil
