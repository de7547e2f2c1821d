// Warp-level 256-point negacyclic NTT / INTT mod q (section 2.2; section 3.2 of
// arXiv 2211.12265, single-warp form: each thread holds 8 coefficients in
// registers, three levels run in registers between two shared-memory exchanges,
// and the exchanges are padded so that no two lanes of a warp hit one bank).
//
// Output order (round-3 reading): index j holds f(zeta^(2 brv8(j) + 1)),
// zeta = 1753.  Twiddles are z = zeta^brv8(k) (forward) and zeta^-brv8(k)
// (inverse), centred, each with its quotient zs = round(2^32 z / q): a product
// by a known factor is then z b - floor(zs b / 2^32) q (Shoup), one high and
// two low multiplies with the additions of the butterfly folded in, instead of
// a Montgomery product's two high and two low ones and three additions.
//
// Register layouts of the 8 values r[0..7] held by lane t:
//   L0: coefficient t + 32 m           (natural order, coalesced loads)
//   L1: coefficient 32 (t>>2) + (t&3) + 4 m
//   L2: coefficient 8 t + m            (two 16-byte vector loads)
// Exchange L0<->L1 uses the padded index i + 4 (i >> 5) (4 words per 32),
// exchange L1<->L2 uses i + (i >> 3) (1 word per 8); both are conflict-free for
// the write and the read side.
#pragma once
#include "dil_arith.cuh"

namespace dil {

struct __align__(16) Zetas {
    int32_t z[256], zs[256];     // zeta^brv8(k) mod q, centred, and its quotient
    int32_t iz[256], izs[256];   // zeta^-brv8(k)
};
// Shared words of one direction's twiddles: z, then zs.
constexpr int NTT_TABLE_WORDS = 512;

namespace detail {
constexpr int64_t cpow(int64_t b, int64_t e) {
    int64_t r = 1;
    b %= Q;
    if (b < 0) b += Q;
    while (e) {
        if (e & 1) r = r * b % Q;
        b = b * b % Q;
        e >>= 1;
    }
    return r;
}
constexpr unsigned cbrv8(unsigned j) {
    unsigned r = 0;
    for (int b = 0; b < 8; ++b)
        if (j & (1u << b)) r |= 1u << (7 - b);
    return r;
}
constexpr int64_t MONT = (int64_t(1) << 32) % Q;  // 2^32 mod q
constexpr int32_t centre(int64_t v) {
    v %= Q;
    if (v < 0) v += Q;
    return (int32_t)(v > (Q - 1) / 2 ? v - Q : v);
}
// round(2^32 z / q) for |z| <= (q - 1) / 2; |result| < 2^31
constexpr int32_t quotient(int32_t z) {
    const int64_t a = z < 0 ? -(int64_t)z : z;
    const int64_t v = ((a << 32) + Q / 2) / Q;
    return (int32_t)(z < 0 ? -v : v);
}
constexpr Zetas make_zetas() {
    Zetas t{};
    for (unsigned k = 0; k < 256; ++k) {
        int64_t e = cbrv8(k);
        t.z[k] = centre(cpow(1753, e));
        t.zs[k] = quotient(t.z[k]);
        t.iz[k] = centre(cpow(1753, 512 - e));   // zeta^512 = 1
        t.izs[k] = quotient(t.iz[k]);
    }
    return t;
}
}  // namespace detail

static __constant__ Zetas c_zetas = detail::make_zetas();       // factors the code names one by one
static __device__ const Zetas g_zetas = detail::make_zetas();   // the source of the shared tables

// Final INTT level scale: mont(F, x) = x * 2^32 / 256 and
// mont(G, x) = x * zeta^-brv8(1) * 2^32 / 256 (mod q).
constexpr int32_t NTT_F = detail::centre(detail::MONT * detail::MONT % Q * detail::cpow(256, Q - 2));
constexpr int32_t NTT_G = detail::centre((int64_t)NTT_F * detail::cpow(1753, 512 - detail::cbrv8(1)) % Q);

// c + z b mod q, in c + [-|b| 2^-33 q, (1 + |b| 2^-33) q): the quotient's
// rounding moves floor(zs b / 2^32) by at most |b| 2^-33 from floor(z b / q).
// The sums are taken mod 2^32 and fit 32 bits.
__device__ __forceinline__ int32_t mul_add_z(int32_t c, int32_t b, int32_t z, int32_t zs) {
    return (int32_t)((uint32_t)c + (uint32_t)z * (uint32_t)b - (uint32_t)__mulhi(b, zs) * (uint32_t)Q);
}

// (a, b) <- (a + z b, a - z b)
__device__ __forceinline__ void ct_bfly(int32_t &a, int32_t &b, int32_t z, int32_t zs) {
    const int32_t s = mul_add_z(a, b, z, zs);
    b = (int32_t)(2u * (uint32_t)a - (uint32_t)s);
    a = s;
}

// (a, b) <- (a + b, z (a - b))
__device__ __forceinline__ void gs_bfly(int32_t &a, int32_t &b, int32_t z, int32_t zs) {
    const int32_t d = a - b;
    a = a + b;
    b = mul_add_z(0, d, z, zs);
}

// The same on coefficients a and b of C polynomials.
template <int C>
__device__ __forceinline__ void ct_bflies(int32_t (&r)[C][8], int a, int b, int32_t z, int32_t zs) {
#pragma unroll
    for (int c = 0; c < C; ++c) ct_bfly(r[c][a], r[c][b], z, zs);
}
template <int C>
__device__ __forceinline__ void gs_bflies(int32_t (&r)[C][8], int a, int b, int32_t z, int32_t zs) {
#pragma unroll
    for (int c = 0; c < C; ++c) gs_bfly(r[c][a], r[c][b], z, zs);
}

// Shared-memory accesses by 32-bit shared-window address (the out-of-line
// transforms receive addresses, not generic pointers).  Exchange-buffer
// accesses are ordered (volatile, memory clobber); twiddle loads read
// constant data and may be scheduled freely.
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void sts32(uint32_t a, int32_t v) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ int32_t lds32(uint32_t a) {
    int32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int32_t ldz32(uint32_t a) {
    int32_t v;
    asm("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ int2 ldz64(uint32_t a) {
    int2 v;
    asm("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ int4 ldz128(uint32_t a) {
    int4 v;
    asm("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}

// Twiddles z and zs [i, i + 1 / 2 / 4) of one direction, from a CTA's shared
// table or (kernels whose CTAs are too short-lived to fill one) from the global
// one through L1.
struct SharedTwiddles {
    uint32_t at;   // shared-memory address
    __device__ __forceinline__ int32_t z32(int i) const { return ldz32(at + 4 * i); }
    __device__ __forceinline__ int32_t zs32(int i) const { return ldz32(at + 1024 + 4 * i); }
    __device__ __forceinline__ int2 z64(int i) const { return ldz64(at + 4 * i); }
    __device__ __forceinline__ int2 zs64(int i) const { return ldz64(at + 1024 + 4 * i); }
    __device__ __forceinline__ int4 z128(int i) const { return ldz128(at + 4 * i); }
    __device__ __forceinline__ int4 zs128(int i) const { return ldz128(at + 1024 + 4 * i); }
};
template <bool INV>
struct GlobalTwiddles {
    __device__ __forceinline__ const int32_t *z(int i) const { return (INV ? g_zetas.iz : g_zetas.z) + i; }
    __device__ __forceinline__ const int32_t *zs(int i) const { return (INV ? g_zetas.izs : g_zetas.zs) + i; }
    __device__ __forceinline__ int32_t z32(int i) const { return __ldg(z(i)); }
    __device__ __forceinline__ int32_t zs32(int i) const { return __ldg(zs(i)); }
    __device__ __forceinline__ int2 z64(int i) const { return __ldg(reinterpret_cast<const int2 *>(z(i))); }
    __device__ __forceinline__ int2 zs64(int i) const { return __ldg(reinterpret_cast<const int2 *>(zs(i))); }
    __device__ __forceinline__ int4 z128(int i) const { return __ldg(reinterpret_cast<const int4 *>(z(i))); }
    __device__ __forceinline__ int4 zs128(int i) const { return __ldg(reinterpret_cast<const int4 *>(zs(i))); }
};

// Eight coefficients of one lane, passed by value to the out-of-line transforms.
struct Poly8 {
    int32_t v[8];
};
// The same for C polynomials that are transformed together.
template <int C>
struct Polys8 {
    int32_t v[C][8];
};

// Forward NTT.  In: L0, |r| < q.  Out: L2, |r| < 9.1q, unscaled (a level adds
// at most 1.01q).  buf: the warp's exchange buffer (288 words), zt: the
// forward twiddles (shared).
template <int C, class Table>
__device__ __forceinline__ void ntt_fwd_body(int32_t (&r)[C][8], uint32_t buf, Table zt) {
    const int lane = threadIdx.x & 31;
    // level 1 (len 128): pairs (m, m+4)
    {
        const int32_t z = c_zetas.z[1], zs = c_zetas.zs[1];
#pragma unroll
        for (int m = 0; m < 4; ++m) ct_bflies(r, m, m + 4, z, zs);
    }
    // level 2 (len 64): pairs (m, m+2), twiddle 2 + m/4
    ct_bflies(r, 0, 2, c_zetas.z[2], c_zetas.zs[2]);
    ct_bflies(r, 1, 3, c_zetas.z[2], c_zetas.zs[2]);
    ct_bflies(r, 4, 6, c_zetas.z[3], c_zetas.zs[3]);
    ct_bflies(r, 5, 7, c_zetas.z[3], c_zetas.zs[3]);
    // level 3 (len 32): pairs (m, m+1), twiddle 4 + m/2
    ct_bflies(r, 0, 1, c_zetas.z[4], c_zetas.zs[4]);
    ct_bflies(r, 2, 3, c_zetas.z[5], c_zetas.zs[5]);
    ct_bflies(r, 4, 5, c_zetas.z[6], c_zetas.zs[6]);
    ct_bflies(r, 6, 7, c_zetas.z[7], c_zetas.zs[7]);
    // exchange L0 -> L1
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) sts32(4 * 288 * c + buf + 4 * (lane + 36 * m), r[c][m]);
    __syncwarp();
    const int b = lane >> 2;
    const uint32_t base1 = buf + 4 * (36 * b + (lane & 3));
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) r[c][m] = lds32(4 * 288 * c + base1 + 16 * m);
    __syncwarp();
    // level 4 (len 16): pairs (m, m+4), twiddle 8 + b
    {
        const int32_t z = zt.z32(8 + b), zs = zt.zs32(8 + b);
#pragma unroll
        for (int m = 0; m < 4; ++m) ct_bflies(r, m, m + 4, z, zs);
    }
    // level 5 (len 8): pairs (m, m+2), twiddles 16 + 2b + {0, 1}
    {
        const int2 z = zt.z64(16 + 2 * b), zs = zt.zs64(16 + 2 * b);
        ct_bflies(r, 0, 2, z.x, zs.x);
        ct_bflies(r, 1, 3, z.x, zs.x);
        ct_bflies(r, 4, 6, z.y, zs.y);
        ct_bflies(r, 5, 7, z.y, zs.y);
    }
    // level 6 (len 4): pairs (m, m+1), twiddles 32 + 4b + {0..3}
    {
        const int4 z = zt.z128(32 + 4 * b), zs = zt.zs128(32 + 4 * b);
        ct_bflies(r, 0, 1, z.x, zs.x);
        ct_bflies(r, 2, 3, z.y, zs.y);
        ct_bflies(r, 4, 5, z.z, zs.z);
        ct_bflies(r, 6, 7, z.w, zs.w);
    }
    // exchange L1 -> L2
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) sts32(4 * 288 * c + base1 + 4 * (4 * m + (m >> 1)), r[c][m]);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) r[c][m] = lds32(4 * 288 * c + buf + 4 * (9 * lane + m));
    __syncwarp();
    // level 7 (len 2): pairs (m, m+2), twiddles 64 + 2t + {0, 1} (one 8-byte
    // load per lane: a half-warp reads 128 contiguous bytes, conflict-free)
    {
        const int2 z = zt.z64(64 + 2 * lane), zs = zt.zs64(64 + 2 * lane);
        ct_bflies(r, 0, 2, z.x, zs.x);
        ct_bflies(r, 1, 3, z.x, zs.x);
        ct_bflies(r, 4, 6, z.y, zs.y);
        ct_bflies(r, 5, 7, z.y, zs.y);
    }
    // level 8 (len 1): pairs (m, m+1), twiddles 128 + 4t + {0..3} (16-byte load)
    {
        const int4 z = zt.z128(128 + 4 * lane), zs = zt.zs128(128 + 4 * lane);
        ct_bflies(r, 0, 1, z.x, zs.x);
        ct_bflies(r, 2, 3, z.y, zs.y);
        ct_bflies(r, 4, 5, z.z, zs.z);
        ct_bflies(r, 6, 7, z.w, zs.w);
    }
}

// Inverse NTT.  In: L2, |r| < q.  Out: L0, |r| < q, equal to INTT(in) * 2^32,
// so it turns pointwise Montgomery products into plain coefficients.  A sum
// doubles per level and stays within 256 (q - 1) < 2^31 at the last; a product
// lies in [-q/4, 5q/4), so it never exceeds the sums of its level.  The last
// level keeps the Montgomery product, whose result is below q.
// izt: the inverse twiddles in shared memory.
template <int C, class Table>
__device__ __forceinline__ void ntt_inv_body(int32_t (&r)[C][8], uint32_t buf, Table izt) {
    const int lane = threadIdx.x & 31;
    // len 1: pairs (m, m+1), twiddles 128 + 4t + {0..3}
    {
        const int4 z = izt.z128(128 + 4 * lane), zs = izt.zs128(128 + 4 * lane);
        gs_bflies(r, 0, 1, z.x, zs.x);
        gs_bflies(r, 2, 3, z.y, zs.y);
        gs_bflies(r, 4, 5, z.z, zs.z);
        gs_bflies(r, 6, 7, z.w, zs.w);
    }
    // len 2: pairs (m, m+2), twiddles 64 + 2t + {0, 1}
    {
        const int2 z = izt.z64(64 + 2 * lane), zs = izt.zs64(64 + 2 * lane);
        gs_bflies(r, 0, 2, z.x, zs.x);
        gs_bflies(r, 1, 3, z.x, zs.x);
        gs_bflies(r, 4, 6, z.y, zs.y);
        gs_bflies(r, 5, 7, z.y, zs.y);
    }
    // exchange L2 -> L1
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) sts32(4 * 288 * c + buf + 4 * (9 * lane + m), r[c][m]);
    __syncwarp();
    const int b = lane >> 2;
    const uint32_t base1 = buf + 4 * (36 * b + (lane & 3));
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) r[c][m] = lds32(4 * 288 * c + base1 + 4 * (4 * m + (m >> 1)));
    __syncwarp();
    // len 4: pairs (m, m+1), twiddles 32 + 4b + {0..3}
    {
        const int4 z = izt.z128(32 + 4 * b), zs = izt.zs128(32 + 4 * b);
        gs_bflies(r, 0, 1, z.x, zs.x);
        gs_bflies(r, 2, 3, z.y, zs.y);
        gs_bflies(r, 4, 5, z.z, zs.z);
        gs_bflies(r, 6, 7, z.w, zs.w);
    }
    // len 8: pairs (m, m+2), twiddles 16 + 2b + {0, 1}
    {
        const int2 z = izt.z64(16 + 2 * b), zs = izt.zs64(16 + 2 * b);
        gs_bflies(r, 0, 2, z.x, zs.x);
        gs_bflies(r, 1, 3, z.x, zs.x);
        gs_bflies(r, 4, 6, z.y, zs.y);
        gs_bflies(r, 5, 7, z.y, zs.y);
    }
    // len 16: pairs (m, m+4), twiddle 8 + b
    {
        const int32_t z = izt.z32(8 + b), zs = izt.zs32(8 + b);
#pragma unroll
        for (int m = 0; m < 4; ++m) gs_bflies(r, m, m + 4, z, zs);
    }
    // exchange L1 -> L0
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) sts32(4 * 288 * c + base1 + 16 * m, r[c][m]);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 8; ++m) r[c][m] = lds32(4 * 288 * c + buf + 4 * (lane + 36 * m));
    __syncwarp();
    // len 32: pairs (m, m+1), twiddle 4 + m/2
    gs_bflies(r, 0, 1, c_zetas.iz[4], c_zetas.izs[4]);
    gs_bflies(r, 2, 3, c_zetas.iz[5], c_zetas.izs[5]);
    gs_bflies(r, 4, 5, c_zetas.iz[6], c_zetas.izs[6]);
    gs_bflies(r, 6, 7, c_zetas.iz[7], c_zetas.izs[7]);
    // len 64: pairs (m, m+2), twiddle 2 + m/4
    gs_bflies(r, 0, 2, c_zetas.iz[2], c_zetas.izs[2]);
    gs_bflies(r, 1, 3, c_zetas.iz[2], c_zetas.izs[2]);
    gs_bflies(r, 4, 6, c_zetas.iz[3], c_zetas.izs[3]);
    gs_bflies(r, 5, 7, c_zetas.iz[3], c_zetas.izs[3]);
    // len 128 with the factor 2^32/n folded in (twiddle 1)
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int32_t a = r[c][m], b2 = r[c][m + 4];
            r[c][m] = mont_mul(NTT_F, a + b2);
            r[c][m + 4] = mont_mul(NTT_G, a - b2);
        }
}

// Out of line: one copy of the code serves every call site, which keeps the
// fused kernels' instruction footprint small.
static __device__ __noinline__ Polys8<1> ntt_fwd_impl(Polys8<1> p, uint32_t buf, uint32_t zt) {
    ntt_fwd_body(p.v, buf, SharedTwiddles{zt});
    return p;
}
static __device__ __noinline__ Polys8<1> ntt_inv_impl(Polys8<1> p, uint32_t buf, uint32_t izt) {
    ntt_inv_body(p.v, buf, SharedTwiddles{izt});
    return p;
}
// With the twiddles of the global table, on one polynomial or on two whose
// chains fill each other's latencies and share the twiddles (exchange buffer:
// 288 words each).
template <int C>
__device__ __noinline__ Polys8<C> ntt_fwd_global_impl(Polys8<C> p, uint32_t buf) {
    ntt_fwd_body(p.v, buf, GlobalTwiddles<false>{});
    return p;
}
template <int C>
__device__ __noinline__ Polys8<C> ntt_inv_global_impl(Polys8<C> p, uint32_t buf) {
    ntt_inv_body(p.v, buf, GlobalTwiddles<true>{});
    return p;
}

__device__ __forceinline__ void ntt_fwd(int32_t r[8], int32_t *buf, const int32_t *zt, int lane) {
    (void)lane;
    Polys8<1> p;
#pragma unroll
    for (int m = 0; m < 8; ++m) p.v[0][m] = r[m];
    p = ntt_fwd_impl(p, smem_addr(buf), smem_addr(zt));
#pragma unroll
    for (int m = 0; m < 8; ++m) r[m] = p.v[0][m];
}

__device__ __forceinline__ void ntt_inv(int32_t r[8], int32_t *buf, const int32_t *izt, int lane) {
    (void)lane;
    Polys8<1> p;
#pragma unroll
    for (int m = 0; m < 8; ++m) p.v[0][m] = r[m];
    p = ntt_inv_impl(p, smem_addr(buf), smem_addr(izt));
#pragma unroll
    for (int m = 0; m < 8; ++m) r[m] = p.v[0][m];
}

// The same with the twiddles of the global table, on C polynomials.
template <int C>
__device__ __forceinline__ void ntt_fwd_global(int32_t (&r)[C][8], int32_t *buf) {
    Polys8<C> p;
#pragma unroll
    for (int i = 0; i < 8 * C; ++i) p.v[i / 8][i % 8] = r[i / 8][i % 8];
    p = ntt_fwd_global_impl<C>(p, smem_addr(buf));
#pragma unroll
    for (int i = 0; i < 8 * C; ++i) r[i / 8][i % 8] = p.v[i / 8][i % 8];
}
template <int C>
__device__ __forceinline__ void ntt_inv_global(int32_t (&r)[C][8], int32_t *buf) {
    Polys8<C> p;
#pragma unroll
    for (int i = 0; i < 8 * C; ++i) p.v[i / 8][i % 8] = r[i / 8][i % 8];
    p = ntt_inv_global_impl<C>(p, smem_addr(buf));
#pragma unroll
    for (int i = 0; i < 8 * C; ++i) r[i / 8][i % 8] = p.v[i / 8][i % 8];
}
__device__ __forceinline__ void ntt_fwd_global(int32_t (&r)[8], int32_t *buf) {
    ntt_fwd_global(reinterpret_cast<int32_t (&)[1][8]>(r), buf);
}
__device__ __forceinline__ void ntt_inv_global(int32_t (&r)[8], int32_t *buf) {
    ntt_inv_global(reinterpret_cast<int32_t (&)[1][8]>(r), buf);
}

// Copies the forward twiddles (NTT_TABLE_WORDS), or those and behind them the
// inverse ones, to 16-byte aligned shared memory (whole block participates).
// From global memory: constant memory serves lanes that ask for different words
// one after the other, 32 reads per warp and word.
template <int TABLES = 2>
__device__ __forceinline__ void load_zetas(int32_t *zt) {
    static_assert(sizeof(Zetas) == 2 * NTT_TABLE_WORDS * sizeof(int32_t), "forward, then inverse");
    for (int i = threadIdx.x; i < TABLES * NTT_TABLE_WORDS / 4; i += blockDim.x)
        reinterpret_cast<int4 *>(zt)[i] = __ldg(reinterpret_cast<const int4 *>(&g_zetas) + i);
}

// Transposes 8 values from L0 to 8 consecutive coefficients (8 lane + m).
__device__ __forceinline__ void l0_to_seq(int32_t v[8], int32_t *buf, int lane) {
#pragma unroll
    for (int m = 0; m < 8; ++m) buf[lane + 36 * m + (lane >> 3)] = v[m];
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 8; ++m) v[m] = buf[9 * lane + m];
    __syncwarp();
}

}  // namespace dil
