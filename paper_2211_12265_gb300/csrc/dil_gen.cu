// KeyGen of a batch (Alg 1).
//
// Batch form: one task per group of P warps up to the packed keys, then a
// kernel that hashes tr = H(pk) sixteen tasks to a warp.  In the task's own
// warp (k_keygen, kept for the launch shapes a caller asks for) the ten blocks
// of a Dilithium2 key cost 4.5 k of the task's 19.4 k SM clocks (10,000 keys:
// 616 -> 550 us).
#include "dil_hash16.cuh"
#include "dil_kern.cuh"

namespace dil {

template <int LEVEL, int P, bool SPLIT>
__device__ __forceinline__ void keygen_body(int n, const uint8_t *__restrict__ seeds, uint8_t *pk, uint8_t *sk,
                                            int32_t *scratch) {
    extern __shared__ __align__(16) uint8_t smem[];
    const CtaView v = cta_setup<P>(smem);
    const int task = blockIdx.x * v.groups + v.group;
    if (task >= n) return;
    using V = Lv<LEVEL>;
    gen_task<LEVEL, P, SPLIT>(seeds + (size_t)task * 32, pk + (size_t)task * V::PK, sk + (size_t)task * V::SK,
                              scratch + (size_t)task * Scratch<LEVEL>::GEN_POLYS * N, *v.gs, *v.ws, v.zt, v.izt, v.g,
                              v.bar, v.lane);
}

template <int LEVEL, int P>
__global__ void __launch_bounds__(256, 4) k_keygen(int n, const uint8_t *__restrict__ seeds, uint8_t *pk,
                                                   uint8_t *sk, int32_t *scratch) {
    keygen_body<LEVEL, P, false>(n, seeds, pk, sk, scratch);
}

cudaError_t launch_keygen(int level, int n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk, int32_t *scratch,
                          int warps, int p, cudaStream_t s) {
    DIL_DISPATCH_GROUPS(k_keygen, seeds, pk, sk, scratch)
}

// ---------------------------------------------------------------- batch form

template <int LEVEL, int P>
__global__ void __launch_bounds__(256, 4) k_keygen_batch(int n, const uint8_t *__restrict__ seeds, uint8_t *pk,
                                                         uint8_t *sk, int32_t *scratch) {
    keygen_body<LEVEL, P, true>(n, seeds, pk, sk, scratch);
}

// tr = H(pk) of task `pair` into its secret key.
template <int LEVEL>
struct KeygenTrJob {
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

    __device__ __forceinline__ void done(const uint32_t (&a)[25]) {
        uint8_t *tr = sk + 64 + 4 * (lane & 1);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) tr[8 * i + q] = (uint8_t)(a[i] >> (8 * q));
    }
};

template <int LEVEL>
__global__ void __launch_bounds__(128) k_keygen_tr(int n, const uint8_t *pk, uint8_t *sk) {
    __shared__ uint32_t stage[4][HASH16_STAGE_WORDS];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w * K16_STATES >= n) return;
    const int t = w * K16_STATES + (lane >> 1);
    KeygenTrJob<LEVEL> job{pk + (size_t)t * Lv<LEVEL>::PK, sk + (size_t)t * Lv<LEVEL>::SK, t < n, lane};
    hash16_run(job, stage[threadIdx.x >> 5], lane);
}

namespace {

template <int LEVEL>
cudaError_t launch_batch(int n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk, int32_t *scratch, int warps, int p,
                         cudaStream_t s) {
    const cudaError_t e = p == 1 ? launch_plain(k_keygen_batch<LEVEL, 1>, n, warps, p, s, seeds, pk, sk, scratch)
                                 : launch_plain(k_keygen_batch<LEVEL, 4>, n, warps, p, s, seeds, pk, sk, scratch);
    if (e != cudaSuccess) return e;
    const HashGrid h = hash_grid(n);
    k_keygen_tr<LEVEL><<<h.blocks, h.threads, 0, s>>>(n, pk, sk);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_keygen_batch(int level, int n, const uint8_t *seeds, uint8_t *pk, uint8_t *sk, int32_t *scratch,
                                int warps, int p, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (p != 1 && p != 4) return cudaErrorInvalidValue;
    switch (level) {
        case 2: return launch_batch<2>(n, seeds, pk, sk, scratch, warps, p, s);
        case 3: return launch_batch<3>(n, seeds, pk, sk, scratch, warps, p, s);
        case 5: return launch_batch<5>(n, seeds, pk, sk, scratch, warps, p, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace dil
