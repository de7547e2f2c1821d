// KeyGen of a batch (Alg 1).
//
// Batch form, four kernels: H(zeta), sixteen tasks to a warp; ExpandA and
// ExpandS, sixteen polynomials to a warp whatever tasks they belong to
// (dil_sample16.cuh); t = A s1 + s2 and the packed keys, one task per warp;
// tr = H(pk), sixteen tasks to a warp.  In the task's own warp
// (k_keygen, kept for the launch shapes a caller asks for) the eleven blocks of
// a Dilithium2 key's hashes cost 4.9 k of the task's 19.4 k SM clocks (10,000
// keys, fused -> batch: 616 -> 433 us, 290 of them the sampling at 3.2 SM clocks
// per state and round).
#include "dil_kern.cuh"
#include "dil_sample16.cuh"

namespace dil {

template <int LEVEL, int P>
__global__ void __launch_bounds__(256, 4) k_keygen(int n, const uint8_t *__restrict__ seeds, uint8_t *pk,
                                                   uint8_t *sk, int32_t *scratch) {
    extern __shared__ __align__(16) uint8_t smem[];
    const CtaView v = cta_setup<P>(smem);
    const int task = blockIdx.x * v.groups + v.group;
    if (task >= n) return;
    using V = Lv<LEVEL>;
    gen_task<LEVEL, P>(seeds + (size_t)task * 32, pk + (size_t)task * V::PK, sk + (size_t)task * V::SK,
                       scratch + (size_t)task * Scratch<LEVEL>::GEN_POLYS * N, *v.gs, *v.ws, v.zt, v.izt, v.g, v.bar,
                       v.lane);
}

cudaError_t launch_keygen(int level, int n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk, int32_t *scratch,
                          int warps, int p, cudaStream_t s) {
    DIL_DISPATCH_GROUPS(k_keygen, seeds, pk, sk, scratch)
}

// ---------------------------------------------------------------- batch form

// Bytes this thread of a pair writes of 4-byte words a[lo .. lo + cnt) (every
// other word of a byte string of any alignment).
__device__ __forceinline__ void put_words(uint8_t *dst, const uint32_t (&a)[25], int lo, int cnt) {
#pragma unroll
    for (int i = 0; i < 25; ++i) {
        if (i < lo || i >= lo + cnt) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[8 * (i - lo) + q] = (uint8_t)(a[i] >> (8 * q));
    }
}

// (rho, rho', K) = H(zeta) of task `pair`: rho to pk, sk and the start of its
// scratch, rho' behind it, K to sk.
template <int LEVEL>
struct KeygenSeedJob {
    static constexpr bool CHAINED = false;
    const uint8_t *seed;
    uint8_t *pk, *sk;
    uint32_t *out;
    bool todo;
    int lane;

    __device__ __forceinline__ bool next(HashInput &in) {
        if (!todo) return false;
        todo = false;
        in = {nullptr, seed, 32, 0};
        return true;
    }

    __device__ __forceinline__ void done(const uint32_t (&a)[25]) {
        const int p = lane & 1;
#pragma unroll
        for (int i = 0; i < 12; ++i) out[2 * i + p] = a[i];   // rho (32 bytes), rho' (64)
        put_words(pk + 4 * p, a, 0, 4);
        put_words(sk + 4 * p, a, 0, 4);
        put_words(sk + 32 + 4 * p, a, 12, 4);
    }
};

template <int LEVEL>
__device__ __forceinline__ int32_t *gen_scratch(int32_t *scratch, int t) {
    return scratch + (size_t)t * Scratch<LEVEL>::GEN_POLYS * N;
}

template <int LEVEL>
__global__ void __launch_bounds__(128) k_keygen_seeds(int n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk,
                                                      int32_t *scratch) {
    __shared__ __align__(16) uint32_t stage[4][HASH16_STAGE_WORDS];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w * K16_STATES >= n) return;
    const int t = w * K16_STATES + (lane >> 1);
    const bool mine = t < n;
    const size_t at = mine ? t : 0;
    KeygenSeedJob<LEVEL> job{seeds + at * 32, pk + at * Lv<LEVEL>::PK, sk + at * Lv<LEVEL>::SK,
                             reinterpret_cast<uint32_t *>(gen_scratch<LEVEL>(scratch, (int)at)), mine, lane};
    hash16_run(job, stage[threadIdx.x >> 5], lane);
}

// Blocks [0, s_blocks) sample s1 || s2, the others A^.  One warp per CTA, as in
// Sign's prepare kernel.
template <int LEVEL>
__global__ void __launch_bounds__(32, 16) k_keygen_expand(int n, int32_t *scratch, int s_blocks) {
    __shared__ __align__(16) uint32_t st[EXPAND16_WORDS];
    using V = Lv<LEVEL>;
    using S = Scratch<LEVEL>;
    const int lane = threadIdx.x;
    const int blk = blockIdx.x;
    if (blk < s_blocks) {
        expand_s_batch<LEVEL>(
            (long long)blk * K16_STATES, (long long)n * (V::K + V::L),
            [&](int t) { return reinterpret_cast<const uint8_t *>(gen_scratch<LEVEL>(scratch, t)) + 32; },
            [&](int t) { return gen_scratch<LEVEL>(scratch, t) + S::GEN_S * N; }, st, lane);
    } else {
        expand_a_batch<LEVEL, false>(
            (long long)(blk - s_blocks) * K16_STATES, (long long)n * V::K * V::L,
            [&](int t) { return reinterpret_cast<const uint8_t *>(gen_scratch<LEVEL>(scratch, t)); },
            [&](int t) { return gen_scratch<LEVEL>(scratch, t) + V::L * N; }, st, lane);
    }
}

// s1, s2, t1 and t0 of one task, one warp: gen_rows with s^1 in shared memory and
// every load of a row of A^ in flight at once.
template <int LEVEL>
__global__ void __launch_bounds__(32, LEVEL == 2 ? 28 : 20) k_keygen_rows(uint8_t *pk, uint8_t *sk,
                                                                       const int32_t *scratch) {
    __shared__ __align__(16) int32_t buf[288], sh[Lv<LEVEL>::L * N];
    using V = Lv<LEVEL>;
    const int task = blockIdx.x, lane = threadIdx.x;
    pk += (size_t)task * V::PK;
    sk += (size_t)task * V::SK;
    const int32_t *ah = scratch + ((size_t)task * Scratch<LEVEL>::GEN_POLYS + V::L) * N;
    const int32_t *sraw = scratch + ((size_t)task * Scratch<LEVEL>::GEN_POLYS + Scratch<LEVEL>::GEN_S) * N;
    int32_t v[8], s[8];
#pragma unroll 1
    for (int j = 0; j < V::L; ++j) {
        load_seq(s, sraw + j * N, lane);
        load_l0(v, sraw + j * N, lane);
        pack_poly<V::ETABITS>(sk + V::SK_S1 + j * V::POLYETA, s, V::ETA, -1, buf, lane);
        ntt_fwd_global(v, buf);
        store_l2(sh + j * N, v, lane);   // read back by the same lane
    }
#pragma unroll 1
    for (int i = 0; i < V::K; ++i) {
        int32_t a[V::L][8];
#pragma unroll
        for (int j = 0; j < V::L; ++j) load_l2(a[j], ah + (i * V::L + j) * N, lane);
        load_seq(s, sraw + (V::L + i) * N, lane);
        pack_poly<V::ETABITS>(sk + V::SK_S2 + i * V::POLYETA, s, V::ETA, -1, buf, lane);
        long long acc[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) acc[m] = 0;
#pragma unroll
        for (int j = 0; j < V::L; ++j) {
            load_l2(v, sh + j * N, lane);
#pragma unroll
            for (int m = 0; m < 8; ++m) acc[m] += (long long)a[j][m] * v[m];
        }
        load_l0(s, sraw + (V::L + i) * N, lane);
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = mont_reduce(acc[m]);
        ntt_inv_global(v, buf);
        gen_split<LEVEL>(pk + 32 + i * V::POLYT1, sk + V::SK_T0 + i * V::POLYT0, v, s, buf, lane);
    }
}

// tr = H(pk) of task `pair` into its secret key.
template <int LEVEL>
struct KeygenTrJob {
    static constexpr bool CHAINED = false;
    const uint8_t *pk;
    uint8_t *sk;
    bool todo;
    int lane;

    __device__ __forceinline__ bool next(HashInput &in) {
        if (!todo) return false;
        todo = false;
        in = {nullptr, pk, (size_t)Lv<LEVEL>::PK, 0};
        return true;
    }

    __device__ __forceinline__ void done(const uint32_t (&a)[25]) { put_words(sk + 64 + 4 * (lane & 1), a, 0, 4); }
};

template <int LEVEL>
__global__ void __launch_bounds__(128) k_keygen_tr(int n, const uint8_t *pk, uint8_t *sk) {
    __shared__ __align__(16) uint32_t stage[4][HASH16_STAGE_WORDS];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w * K16_STATES >= n) return;
    const int t = w * K16_STATES + (lane >> 1);
    KeygenTrJob<LEVEL> job{pk + (size_t)t * Lv<LEVEL>::PK, sk + (size_t)t * Lv<LEVEL>::SK, t < n, lane};
    hash16_run(job, stage[threadIdx.x >> 5], lane);
}

// The same for a small batch, a warp per key on the 25-lane form.
template <int LEVEL>
__global__ void __launch_bounds__(32) k_keygen_tr_wide(const uint8_t *pk, uint8_t *sk) {
    __shared__ __align__(16) uint8_t none[8];
    const int t = blockIdx.x, lane = threadIdx.x;
    uint32_t lo = 0, hi = 0;
    absorb_concat(lo, hi, none, 0, pk + (size_t)t * Lv<LEVEL>::PK, Lv<LEVEL>::PK, 136, lane);
    if (lane >= 4) return;
    uint8_t *tr = sk + (size_t)t * Lv<LEVEL>::SK + 64 + 8 * lane;
#pragma unroll
    for (int q = 0; q < 8; ++q) tr[q] = (uint8_t)((q < 4 ? lo : hi) >> (8 * (q & 3)));
}

namespace {

template <int LEVEL>
cudaError_t launch_batch(int n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk, int32_t *scratch, cudaStream_t s) {
    using V = Lv<LEVEL>;
    const HashGrid h = hash_grid(n);
    k_keygen_seeds<LEVEL><<<h.blocks, h.threads, 0, s>>>(n, seeds, pk, sk, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const auto blocks = [&](long long polys) { return (int)((polys * n + K16_STATES - 1) / K16_STATES); };
    const int s_blocks = blocks(V::K + V::L);
    k_keygen_expand<LEVEL><<<s_blocks + blocks(V::K * V::L), 32, 0, s>>>(n, scratch, s_blocks);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_keygen_rows<LEVEL><<<n, 32, 0, s>>>(pk, sk, scratch);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (n <= HASH_WIDE_MOST)
        k_keygen_tr_wide<LEVEL><<<n, 32, 0, s>>>(pk, sk);
    else
        k_keygen_tr<LEVEL><<<h.blocks, h.threads, 0, s>>>(n, pk, sk);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_keygen_batch(int level, int n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk, int32_t *scratch,
                                cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    switch (level) {
        case 2: return launch_batch<2>(n, seeds, pk, sk, scratch, s);
        case 3: return launch_batch<3>(n, seeds, pk, sk, scratch, s);
        case 5: return launch_batch<5>(n, seeds, pk, sk, scratch, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace dil
