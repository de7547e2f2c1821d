// Shared prologue and launch helper of the plain one-launch-per-batch kernels
// (section 4.2 fusion: one kernel runs whole Gen, Sign or Verify tasks).  A CTA
// holds W warps = W / P task groups of P warps; the CTA shares the NTT twiddle
// tables in shared memory, each group its GroupSmem, each warp its WarpSmem.
#pragma once
#include "../../include/dil.h"
#include "dil_launch.h"
#include "dil_procs.cuh"

namespace dil {

__host__ __device__ constexpr size_t cta_bytes(int warps, int p) {
    return CTA_TABLE_BYTES + (size_t)(warps / p) * sizeof(GroupSmem) + (size_t)warps * sizeof(WarpSmem);
}

struct CtaView {
    int32_t *zt, *izt;
    GroupSmem *gs;
    WarpSmem *ws;
    int g, bar, lane, group, groups;
};

// Carves the dynamic shared memory, loads the twiddles (whole CTA) and locates
// this warp's group.
template <int P>
__device__ __forceinline__ CtaView cta_setup(uint8_t *smem) {
    CtaView v;
    const int warps = blockDim.x >> 5;
    v.groups = warps / P;
    v.zt = reinterpret_cast<int32_t *>(smem);
    v.izt = v.zt + NTT_TABLE_WORDS;
    GroupSmem *gsa = reinterpret_cast<GroupSmem *>(smem + CTA_TABLE_BYTES);
    WarpSmem *wsa = reinterpret_cast<WarpSmem *>(smem + CTA_TABLE_BYTES + v.groups * sizeof(GroupSmem));
    load_zetas(v.zt);
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    v.lane = threadIdx.x & 31;
    v.group = warp / P;
    v.g = warp % P;
    v.bar = 1 + v.group;   // named barrier 0 is __syncthreads
    v.gs = gsa + v.group;
    v.ws = wsa + warp;
    return v;
}

template <class Kern, class... Args>
static cudaError_t launch_plain(Kern kern, int n, int warps, int p, cudaStream_t s, Args... args) {
    if (n <= 0) return cudaSuccess;
    const size_t smem = cta_bytes(warps, p);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int groups = warps / p;
    kern<<<(n + groups - 1) / groups, warps * 32, smem, s>>>(n, args...);
    return cudaGetLastError();
}

// Warps that hash a batch of n tasks sixteen at a time.  One task to a pair of
// threads while that takes at most one warp per sub-partition (608 warps);
// beyond it two to a pair, taken as pairs come free: fewer warps then share
// the SMs with the arithmetic, and a pair with a short message goes on to the
// next task.
inline int batch_hash_warps(int n) {
    const int all = (n + 15) / 16;
    return all <= 608 ? all : (n + 31) / 32 > 608 ? (n + 31) / 32 : 608;
}

// Up to this many hashes a warp each, on the 25-lane form: while every warp has a
// sub-partition to itself a block takes 2.7 us that way and 3.8 two threads to a
// state (224 and 250 clocks a round; absorbing costs 150 and 1,000), and the
// chain of a hash's blocks is what a small batch waits for.
constexpr int HASH_WIDE_MOST = 608;

// How a batch's messages are hashed: `warps` warps of two threads to a state,
// and `wide` warps, one per task, that take the messages of at least
// `long_bytes` on the 25-lane form.  Beyond HASH_WIDE_MOST tasks on the GPU that
// form still ends a long message's chain sooner, while its chains are bound by
// latency (up to ten or twelve on an SM; more, and two threads to a state finish
// the same work in a sixth of the issue slots).  1,000 Dilithium2 tasks of 16 KB,
// Sign 914 us without and 818 with it, Verify 549 and 477; of 256 KB 8200 and
// 6719, 7460 and 6401.  Messages of 4 KB as well: Verify of 609 Dilithium2 tasks
// 203 -> 187 us, but Sign of 1,824 Dilithium3 1001 -> 1043; Sign of 1,500 Dilithium2
// of 16 KB 973 -> 936, of 1,800 of 64 KB 2536 -> 2597, Verify with resident keys of
// 1,800 505 -> 537.
constexpr size_t HASH_LONG_BYTES = 8192;
constexpr int HASH_LONG_MOST = 1520;
// Beyond that line only where at most HASH_FEW of sixteen tasks in a row have a
// long message.  Messages of 32 B - 16 KB (a ninth of them long), Verify: 3,000
// Dilithium3 tasks 863 -> 645 us (708 with four of sixteen, which a group now and
// then exceeds), 6,000 1034 -> 880, but 10,000 1259 -> 2377; with resident keys
// 3,000 519 -> 474, 4,000 522 -> 493, 8,191 552 -> 556 and all of 16 KB 574 -> 610.
constexpr int HASH_FEW = 8, HASH_FEW_MOST = 3072, HASH_FEW_MOST_SAMPLING = 6144;
static_assert(HASH_FEW_MOST_SAMPLING <= 608 * K16_STATES, "one task to a pair (batch_hash_warps) beside wide warps");
struct HashSplit {
    int warps, wide;
    size_t long_bytes;
    int per_group;   // wide warps of sixteen tasks in a row
};
// The tasks on the GPU up to which every message has a warp, every one of
// long_bytes or more, few such.
struct HashLines {
    int all, every_long, few_long;
    size_t long_bytes;
};
inline HashSplit hash_split(int n, int on_gpu, const HashLines &l) {   // n of the on_gpu tasks that run at a time
    if (on_gpu <= l.all) return {0, n, 0, 0};
    const int warps = batch_hash_warps(n);
    if (on_gpu > l.few_long) return {warps, 0, (size_t)-1, 0};
    const int groups = (n + K16_STATES - 1) / K16_STATES;
    if (on_gpu <= l.every_long) return {warps, groups * K16_STATES, l.long_bytes, K16_STATES};
    return {warps, groups * HASH_FEW, HASH_LONG_BYTES, HASH_FEW};
}

__device__ __forceinline__ bool is_long(const uint64_t *off, int n, int t, size_t least) {
    uint64_t m0;
    size_t mlen;
    return t < n && message_of(off, t, m0, mlen) && mlen >= least;
}

// Whether task t (n: none) is a wide warp's.
__device__ __forceinline__ bool has_wide_warp(const uint64_t *off, int n, int t, size_t least, int per_group) {
    if (!is_long(off, n, t, least)) return false;
    if (per_group >= K16_STATES) return true;
    const int first = t / K16_STATES * K16_STATES;
    int c = 0;
    for (int i = 0; i < K16_STATES; ++i) c += is_long(off, n, first + i, least);
    return c <= per_group;
}

// The task of wide warp w (all 32 lanes), or -1.
__device__ __forceinline__ int task_of_wide_warp(const uint64_t *off, int n, int w, size_t least, int per_group,
                                                 int lane) {
    const int first = w / per_group * K16_STATES, nth = w % per_group;
    const unsigned mask = __ballot_sync(FULL, lane < K16_STATES && is_long(off, n, first + lane, least));
    if (__popc(mask) > per_group || nth >= __popc(mask)) return -1;
    return first + (int)__fns(mask, 0, nth + 1);
}

// Launch shape of a kernel that only hashes, one task per pair of threads:
// single-warp CTAs spread a small batch over the SMs, four-warp ones put one
// warp on each of an SM's sub-partitions.
struct HashGrid {
    int blocks, threads;
};
inline HashGrid hash_grid(int n) {
    const int warps = (n + 15) / 16;
    return warps <= 152 ? HashGrid{warps, 32} : HashGrid{(warps + 3) / 4, 128};
}

// Dispatch on (level, warps per task) to kernel template K<LEVEL, P>.
#define DIL_DISPATCH(KERN, ...)                                                                  \
    switch (level * 10 + p) {                                                                    \
        case 21: return launch_plain(KERN<2, 1>, n, warps, p, s, __VA_ARGS__);                   \
        case 22: return launch_plain(KERN<2, 2>, n, warps, p, s, __VA_ARGS__);                   \
        case 24: return launch_plain(KERN<2, 4>, n, warps, p, s, __VA_ARGS__);                   \
        case 31: return launch_plain(KERN<3, 1>, n, warps, p, s, __VA_ARGS__);                   \
        case 32: return launch_plain(KERN<3, 2>, n, warps, p, s, __VA_ARGS__);                   \
        case 34: return launch_plain(KERN<3, 4>, n, warps, p, s, __VA_ARGS__);                   \
        case 51: return launch_plain(KERN<5, 1>, n, warps, p, s, __VA_ARGS__);                   \
        case 52: return launch_plain(KERN<5, 2>, n, warps, p, s, __VA_ARGS__);                   \
        case 54: return launch_plain(KERN<5, 4>, n, warps, p, s, __VA_ARGS__);                   \
    }                                                                                            \
    return cudaErrorInvalidValue;

// As DIL_DISPATCH for kernels that exist for groups of two and four warps only.
#define DIL_DISPATCH_GROUPS(KERN, ...)                                                           \
    switch (level * 10 + p) {                                                                    \
        case 22: return launch_plain(KERN<2, 2>, n, warps, p, s, __VA_ARGS__);                   \
        case 24: return launch_plain(KERN<2, 4>, n, warps, p, s, __VA_ARGS__);                   \
        case 32: return launch_plain(KERN<3, 2>, n, warps, p, s, __VA_ARGS__);                   \
        case 34: return launch_plain(KERN<3, 4>, n, warps, p, s, __VA_ARGS__);                   \
        case 52: return launch_plain(KERN<5, 2>, n, warps, p, s, __VA_ARGS__);                   \
        case 54: return launch_plain(KERN<5, 4>, n, warps, p, s, __VA_ARGS__);                   \
    }                                                                                            \
    return cudaErrorInvalidValue;

}  // namespace dil
