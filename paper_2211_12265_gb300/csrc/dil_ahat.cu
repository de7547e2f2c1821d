// Resident-A^ forms of the plain kernels: A^ = ExpandA(rho) written to a
// caller's buffer (Alg 4; the matrix Alg 1 samples and Alg 2 / Alg 3 use in the
// NTT domain), and Sign reading that A^ instead of sampling it (Verify's is a
// source of its batch form, dil_verify.cu; Sign's usual form, too, is one of
// the batch's, dil_rounds.cu).  The Sign here runs a task on one warp with the
// plain body (dil_procs.cuh) and the A^ source switched.
#include "dil_kern.cuh"
#include "dil_sample16.cuh"

namespace dil {

// A^ of task t at ahat + t k l N, polynomial (i, j) at index i l + j,
// coefficients in index order, each in [0, q).
template <int LEVEL, bool INDEX = true, int BLOCKS = 5>
__global__ void __launch_bounds__(32, 16) k_expand_a(int n, const uint8_t *rho, size_t rho_stride, int32_t *ahat) {
    __shared__ __align__(16) uint32_t st[EXPAND16_WORDS];
    constexpr int KL = Lv<LEVEL>::K * Lv<LEVEL>::L;
    expand_a_batch<LEVEL, INDEX, BLOCKS>((long long)blockIdx.x * K16_STATES, (long long)n * KL,
                                [&](int t) { return rho + (size_t)t * rho_stride; },
                                [&](int t) { return ahat + (size_t)t * KL * N; }, st, threadIdx.x);
}

template <int LEVEL>
__global__ void __launch_bounds__(256, 4) k_sign_a(int n, const uint8_t *__restrict__ sk,
                                                   const uint8_t *__restrict__ msg, const uint64_t *__restrict__ off,
                                                   const int32_t *__restrict__ ahat, uint8_t *sig, int32_t *status,
                                                   int32_t *iters, int32_t *scratch, int max_iter) {
    extern __shared__ __align__(16) uint8_t smem[];
    const CtaView v = cta_setup<1>(smem);
    const int task = blockIdx.x * v.groups + v.group;
    if (task >= n) return;
    using V = Lv<LEVEL>;
    int32_t *scr = scratch + (size_t)task * Scratch<LEVEL>::SIGN_POLYS * N;
    uint64_t m0;
    size_t mlen;
    uint8_t *tsig = sig + (size_t)task * V::SIG;
    if (!message_of(off, task, m0, mlen)) {   // decreasing offsets: reject the task
        sign_zero<LEVEL, 1>(tsig, 0, v.lane);
        if (v.lane == 0) {
            if (status) status[task] = DIL_EINVAL;
            if (iters) iters[task] = 0;
        }
        return;
    }
    sign_prepare<LEVEL, 1, true>(sk + (size_t)task * V::SK, msg + m0, mlen, scr, *v.gs, *v.ws, v.zt, 0, v.bar,
                                 v.lane, ahat + (size_t)task * V::K * V::L * N);
    int it = 0;
    bool ok = false;
    MaskStream ms{0, 0};
    while (it < max_iter) {
        ok = sign_attempt<LEVEL, 1>(it * V::L, scr, scr + Scratch<LEVEL>::PRE_POLYS * N, ms, *v.gs, *v.ws, v.zt,
                                    v.izt, 0, v.bar, v.lane);
        ++it;
        if (ok) break;
    }
    if (ok)
        sign_pack<LEVEL, 1>(tsig, scr + Scratch<LEVEL>::PRE_POLYS * N, *v.gs, 0, v.lane);
    else
        sign_zero<LEVEL, 1>(tsig, 0, v.lane);
    if (v.lane == 0) {
        if (status) status[task] = ok ? DIL_OK : DIL_EITER;
        if (iters) iters[task] = it;
    }
}

template <int LEVEL, bool INDEX = true, int BLOCKS = 5>
static cudaError_t launch_expand(int n, const uint8_t *rho, size_t rho_stride, int32_t *ahat, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const long long polys = (long long)n * Lv<LEVEL>::K * Lv<LEVEL>::L;
    k_expand_a<LEVEL, INDEX, BLOCKS><<<(int)((polys + K16_STATES - 1) / K16_STATES), 32, 0, s>>>(n, rho, rho_stride, ahat);
    return cudaGetLastError();
}

cudaError_t launch_expand_a(int level, int n, const uint8_t *rho, size_t rho_stride, int32_t *ahat, cudaStream_t s) {
    switch (level) {
        case 2: return launch_expand<2>(n, rho, rho_stride, ahat, s);
        case 3: return launch_expand<3>(n, rho, rho_stride, ahat, s);
        case 5: return launch_expand<5>(n, rho, rho_stride, ahat, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_test_expand_a_refill(int level, int n, const uint8_t *rho, bool index, int32_t *ahat,
                                        cudaStream_t s) {
    switch (2 * level + index) {
        case 4: return launch_expand<2, false, 4>(n, rho, 32, ahat, s);
        case 5: return launch_expand<2, true, 4>(n, rho, 32, ahat, s);
        case 6: return launch_expand<3, false, 4>(n, rho, 32, ahat, s);
        case 7: return launch_expand<3, true, 4>(n, rho, 32, ahat, s);
        case 10: return launch_expand<5, false, 4>(n, rho, 32, ahat, s);
        case 11: return launch_expand<5, true, 4>(n, rho, 32, ahat, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_sign_a(int level, int n, const uint8_t *sk, const uint8_t *msg, const uint64_t *off,
                          const int32_t *ahat, uint8_t *sig, int32_t *status, int32_t *iters, int32_t *scratch,
                          int max_iter, int warps, cudaStream_t s) {
    switch (level) {
        case 2: return launch_plain(k_sign_a<2>, n, warps, 1, s, sk, msg, off, ahat, sig, status, iters, scratch, max_iter);
        case 3: return launch_plain(k_sign_a<3>, n, warps, 1, s, sk, msg, off, ahat, sig, status, iters, scratch, max_iter);
        case 5: return launch_plain(k_sign_a<5>, n, warps, 1, s, sk, msg, off, ahat, sig, status, iters, scratch, max_iter);
    }
    return cudaErrorInvalidValue;
}

}  // namespace dil
