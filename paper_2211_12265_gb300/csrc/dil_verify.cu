// Verify of a batch (Alg 3).
//
// Batch form.  The first kernel gives its leading blocks to the hashes
// tr = H(pk) and mu = H(tr || M) and to SampleInBall(c~), sixteen tasks to a
// warp, and the others to sampling A^, sixteen polynomials to a warp whatever tasks they belong to
// (dil_sample16.cuh).  The second does the arithmetic up to the packed w1', one
// task per warp; with a resident key's or the caller's A^ it is the other blocks
// of the first, one task per group of P warps.  The last recomputes c~ = H(mu || w1'),
// sixteen tasks to a warp, and compares.  Hashing inside
// the task's own warp (k_verify, kept for the launch shapes a caller asks for)
// runs the 18 blocks of a Dilithium2 task at 18.7 SM clocks per round, 8.1 k
// of the task's 20.7 k clocks; sixteen to a warp they take 1.4 k.  10,000 tasks,
// fused -> batch: Dilithium2 655 -> 462 us, Dilithium5 (32 B - 4 KB)
// 1813 -> 1351 us; 13 Dilithium3 tasks 162 -> 138 us.
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

// Scratch polynomials of one task of the batch form.
template <int LEVEL, int SRC>
__host__ __device__ constexpr int verify_polys() {
    return SRC == VERIFY_PLAIN ? Scratch<LEVEL>::VERIFY_POLYS : Scratch<LEVEL>::KEYED_VERIFY_POLYS;
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

static_assert(HASH16_STAGE_WORDS * sizeof(uint32_t) <= sizeof(WarpSmem), "the hashing warps' shared memory");

// tr = H(pk) (not for resident keys) and mu = H(tr || M) of a pair's tasks:
// the first by the pair's index, the next ones from the batch's counter.
template <int LEVEL, int SRC>
struct VerifyMuJob {
    const VerifyBatch &b;
    int task, lane;
    bool first, have_tr;

    __device__ VerifyMuJob(const VerifyBatch &b_, int pair, int lane_)
        : b(b_), task(pair), lane(lane_), first(true), have_tr(false) {}

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
        if (SRC != VERIFY_KEYED && !have_tr) {   // the words this thread reads back as the prefix of mu's input
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

// One hashing warp of the batch (w < hash_warps).
template <int LEVEL, int SRC>
__device__ __forceinline__ void verify_hashes(const VerifyBatch &b, int w, uint32_t *stage, int lane) {
    VerifyMuJob<LEVEL, SRC> job(b, w * K16_STATES + (lane >> 1), lane);
    hash16_run(job, stage, lane);
}

// The arithmetic of the tasks of CTA `blk`.
template <int LEVEL, int P, int SRC>
__device__ __forceinline__ void verify_tasks(const VerifyBatch &b, int blk, uint8_t *smem) {
    using V = Lv<LEVEL>;
    const CtaView v = cta_setup<P>(smem);
    const int task = blk * v.groups + v.group;
    if (task >= b.n) return;
    int key;
    uint64_t m0;
    size_t mlen;
    int r = 0;
    if (verify_input<SRC>(b, task, key, m0, mlen)) {
        int32_t *scr = b.scratch + (size_t)task * verify_polys<LEVEL, SRC>() * N;
        const int32_t *a = SRC == VERIFY_AHAT ? b.ahat + (size_t)task * V::K * V::L * N
                                              : b.keys + (size_t)key * Scratch<LEVEL>::KEY_POLYS * N;
        r = verify_task<LEVEL, P, SRC == VERIFY_KEYED, SRC == VERIFY_AHAT, true>(
            b.pk + (size_t)key * V::PK, nullptr, 0, b.sig + (size_t)task * V::SIG, scr, *v.gs, *v.ws, v.zt, v.izt,
            v.g, v.bar, v.lane, a);
    }
    if (v.g == 0 && v.lane == 0) b.ok[task] = (uint8_t)r;   // 1: c~ decides (k_verify_compare)
}

// VERIFY_AHAT, VERIFY_KEYED: hashes and arithmetic.
template <int LEVEL, int P, int SRC>
__global__ void __launch_bounds__(256, 4) k_verify_batch(const VerifyBatch b) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if ((int)blockIdx.x < b.hash_blocks) {
        const int w = blockIdx.x * warps + warp;
        if (w < b.hash_warps)
            verify_hashes<LEVEL, SRC>(b, w, reinterpret_cast<uint32_t *>(smem) + warp * HASH16_STAGE_WORDS, lane);
        return;
    }
    verify_tasks<LEVEL, P, SRC>(b, blockIdx.x - b.hash_blocks, smem);
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

// VERIFY_PLAIN: blocks [0, hash_warps) hash tr and mu, [.., + challenge_blocks)
// draw challenges, the others sample A^; the arithmetic follows.  One warp per
// CTA, as in Sign's prepare kernel.
template <int LEVEL>
__global__ void __launch_bounds__(32, 16) k_verify_prepare(const VerifyBatch b) {
    extern __shared__ __align__(16) uint32_t sm[];
    using V = Lv<LEVEL>;
    const int lane = threadIdx.x;
    int blk = blockIdx.x;
    if (blk < b.hash_warps) {
        verify_hashes<LEVEL, VERIFY_PLAIN>(b, blk, sm, lane);
        return;
    }
    blk -= b.hash_warps;
    if (blk < b.challenge_blocks) {
        verify_challenges<LEVEL>(b, blk * K16_STATES, sm, lane);
        return;
    }
    blk -= b.challenge_blocks;
    expand_a_batch<LEVEL>(
        (long long)blk * K16_STATES, (long long)b.n * V::K * V::L, [&](int t) { return b.pk + (size_t)t * V::PK; },
        [&](int t) { return b.scratch + ((size_t)t * verify_polys<LEVEL, VERIFY_PLAIN>() + V::L) * N; }, sm, lane);
}

// The arithmetic of one task, one warp: hint decoding, z^, and per row
// w1' = UseHint(h, INTT(A^ z^ - c^ NTT(t1 2^d))), packed to the start of its
// scratch.  False when the signature is malformed or z too large.
template <int LEVEL>
__device__ __forceinline__ bool verify_rows(const VerifyBatch &b, int task, int32_t *buf, int32_t *zh, uint32_t *hmask,
                                            int lane) {
    using V = Lv<LEVEL>;
    const uint8_t *sig = b.sig + (size_t)task * V::SIG, *pk = b.pk + (size_t)task * V::PK;
    uint8_t *sq = reinterpret_cast<uint8_t *>(buf);
    int32_t v[8], ch[8];
    // strict hint decoding into bit masks
    stage_bytes(sq, sig + V::SIG_H, V::OMEGA + V::K, lane);
    hmask[lane] = 0;
    hmask[32 + lane] = 0;
    __syncwarp();
    bool bad = false;
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
    if (__any_sync(FULL, bad)) return false;
    // z^ = NTT(z), ||z|| < gamma1 - beta
#pragma unroll 1
    for (int j = 0; j < V::L; ++j) {
        unpack_buf_l0<V::ZBITS>(v, sig + V::SIG_Z + j * V::POLYZ, V::GAMMA1, buf, lane);
#pragma unroll
        for (int m = 0; m < 8; ++m) bad |= iabs(v[m]) >= V::GAMMA1 - V::BETA;
        if (__any_sync(FULL, bad)) return false;
        ntt_fwd_global(v, buf);
        store_l2(zh + j * N, v, lane);   // read back by the same lane
    }
    const int8_t *c = reinterpret_cast<const int8_t *>(b.challenge) + (size_t)task * 256;
#pragma unroll
    for (int m = 0; m < 8; ++m) ch[m] = c[lane + 32 * m];
    ntt_fwd_global(ch, buf);
    int32_t *scr = b.scratch + (size_t)task * verify_polys<LEVEL, VERIFY_PLAIN>() * N;
#pragma unroll 1
    for (int i = 0; i < V::K; ++i) {
        int32_t a[V::L][8];   // every load of the row in flight during t1's transform
#pragma unroll
        for (int j = 0; j < V::L; ++j) load_l2(a[j], scr + (V::L + i * V::L + j) * N, lane);
        unpack_buf_l0<10>(v, pk + 32 + i * V::POLYT1, 0, buf, lane);
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = (-v[m]) << D;   // t1 2^d, t1 unpacked as 0 - field
        ntt_fwd_global(v, buf);
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

template <int LEVEL>
__global__ void __launch_bounds__(32, LEVEL == 2 ? 24 : 20) k_verify_rows(const VerifyBatch b) {
    __shared__ __align__(16) int32_t buf[288], zh[Lv<LEVEL>::L * N];
    __shared__ uint32_t hmask[64];
    const int task = blockIdx.x, lane = threadIdx.x;
    int key;
    uint64_t m0;
    size_t mlen;
    const bool r = verify_input<VERIFY_PLAIN>(b, task, key, m0, mlen) &&
                   verify_rows<LEVEL>(b, task, buf, zh, hmask, lane);
    if (lane == 0) b.ok[task] = r;   // 1: c~ decides (k_verify_compare)
}

// c~ = H(mu || w1') of task `pair` against the signature's.
template <int LEVEL, int SRC>
struct VerifyCompareJob {
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

namespace {

template <int LEVEL, int P, int SRC>
cudaError_t launch_batch(VerifyBatch b, int warps, cudaStream_t s) {
    b.hash_warps = batch_hash_warps(b.n);
    cudaError_t e = cudaSuccess;
    if (b.n > b.hash_warps * K16_STATES) e = cudaMemsetAsync(b.next, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    if constexpr (SRC == VERIFY_PLAIN) {
        b.challenge_blocks = (b.n + K16_STATES - 1) / K16_STATES;
        const long long polys = (long long)b.n * Lv<LEVEL>::K * Lv<LEVEL>::L;
        const int expand_blocks = (int)((polys + K16_STATES - 1) / K16_STATES);
        const int bytes = EXPAND16_WORDS * (int)sizeof(uint32_t);
        static_assert(CHALLENGE_WORDS <= EXPAND16_WORDS, "the hashing blocks' shared memory");
        e = cudaFuncSetAttribute(k_verify_prepare<LEVEL>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        k_verify_prepare<LEVEL><<<b.hash_warps + b.challenge_blocks + expand_blocks, 32, bytes, s>>>(b);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_verify_rows<LEVEL><<<b.n, 32, 0, s>>>(b);
    } else {
        const int blocks = (b.n + warps / P - 1) / (warps / P);
        const size_t smem = cta_bytes(warps, P);
        b.hash_blocks = (b.hash_warps + warps - 1) / warps;
        e = cudaFuncSetAttribute(k_verify_batch<LEVEL, P, SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_verify_batch<LEVEL, P, SRC><<<b.hash_blocks + blocks, warps * 32, smem, s>>>(b);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const HashGrid h = hash_grid(b.n);
    k_verify_compare<LEVEL, SRC><<<h.blocks, h.threads, 0, s>>>(b);
    return cudaGetLastError();
}

template <int LEVEL, int SRC>
cudaError_t launch_batch_p(const VerifyBatch &b, int warps, int p, cudaStream_t s) {
    if constexpr (SRC == VERIFY_PLAIN) return launch_batch<LEVEL, 1, SRC>(b, warps, s);
    switch (p) {
        case 1: return launch_batch<LEVEL, 1, SRC>(b, warps, s);
        case 4: return launch_batch<LEVEL, 4, SRC>(b, warps, s);
    }
    return cudaErrorInvalidValue;
}

template <int LEVEL>
cudaError_t launch_batch_src(int src, const VerifyBatch &b, int warps, int p, cudaStream_t s) {
    switch (src) {
        case VERIFY_PLAIN: return launch_batch_p<LEVEL, VERIFY_PLAIN>(b, warps, p, s);
        case VERIFY_AHAT: return launch_batch_p<LEVEL, VERIFY_AHAT>(b, warps, p, s);
        case VERIFY_KEYED: return launch_batch_p<LEVEL, VERIFY_KEYED>(b, warps, p, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_verify_batch(int level, int src, const VerifyBatch &b, int warps, int p, cudaStream_t s) {
    if (b.n <= 0) return cudaSuccess;
    switch (level) {
        case 2: return launch_batch_src<2>(src, b, warps, p, s);
        case 3: return launch_batch_src<3>(src, b, warps, p, s);
        case 5: return launch_batch_src<5>(src, b, warps, p, s);
    }
    return cudaErrorInvalidValue;
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
