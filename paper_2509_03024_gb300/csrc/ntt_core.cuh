// ntt_core.cuh — butterfly arithmetic and the register-blocked stages shared by
// the plain NTT launches (ntt.cu) and the fused key-switch passes (ks.cu). See
// ntt.cu for the decomposition.
#pragma once

#include "core.cuh"

namespace fhe {
namespace nttc {

// Arithmetic of the transforms and of products with constants, a property of the prime (Prime::cls,
// uniform in a CTA). What bounds the transforms is the 32-bit multiply pipe: a mad.wide.u32 holds it
// for four cycles per warp, a 32-bit mad.lo for two, so the products are formed from as few wide
// multiplies as possible.
//
// Near primes, q = 2^b - delta with delta <= 2^26, b = 50 or 60 (the library's primes are the largest
// of their size that are 1 mod 2N, so this is the usual case). For a constant w the tables hold W0 = w
// and W1 = 2^32 w mod q, so y w = y0 W0 + y1 W1 (mod q) for any y = y0 + 2^32 y1. Both are split at bit
// `at`: A = y0 W0l + y1 W1l and B = y0 W0h + y1 W1h need no carries, the product is A + 2^at B, and
// 2^(32 + at) = 2^(32 + at - b) delta (mod q) folds the high word of B back in with one multiply. Six
// wide multiplies in all, where a Shoup product takes four wide ones for its quotient and two wide and
// four narrow ones for its low products.
//   AR_NEAR50  at = 20, y and the product signed: |y w| < T = 1.54 2^58. With 64 bits for a 50-bit prime
//              nothing is reduced between the stages of a forward transform (each adds at most T:
//              below 2^60.4 + 16 T < 2^63 at the end), and signed differences need no multiple of q;
//              the inverse folds every value once per register block
//   AR_NEAR60  at = 29, unsigned: y w < 2^62 + 2^61 + 2^59 < 7 q; values stay below 16 q < 2^64 with the
//              first operand folded in every other forward stage, the sum in every inverse one
//   AR_SHOUP   any prime up to 61 bits: Shoup products with a quotient from the three upper partial
//              products (at most two below the true one), y w < 4 q; values below 8 q, the first
//              operand of each butterfly brought below 4 q
//   AR_LAZY    the same for primes below 2^57, whose forward transforms (of many or short rows, with_arith) leave
//              the first operand as it is: 8 q and 4 q more per stage are below 72 q < 2^64 after 16 stages (1024
//              polynomials of four 40-bit limbs at N = 2^12 217 -> 197 us, 84 of six 45-bit limbs at 2^16 477 -> 420)
// Register-only rate of the forward butterfly (GB300, 10^9 per second, unrolled radix-8 blocks): Shoup
// with the exact quotient 998, NEAR50 1420 (13 instructions); the same with B's low word shifted by
// shift and add 1290, with unsigned values and a multiple of q in the difference 1120.
// Prime::cls holds one of the four (AR_LAZY where it applies).
enum Arith { AR_SHOUP = 0, AR_NEAR50 = 1, AR_NEAR60 = 2, AR_LAZY = 3 };
__host__ __device__ constexpr bool is_near(u32 cls) { return cls == AR_NEAR50 || cls == AR_NEAR60; }
__host__ __device__ constexpr int split_at(int ar) { return ar == AR_NEAR50 ? 20 : 29; }

__device__ __forceinline__ u64 mul_wide(u32 a, u32 b) {
    u64 r;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ u64 mad_wide(u32 a, u32 b, u64 c) {
    u64 r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
// the same with both factors signed (b is below 2^31 here, so only a's sign matters)
__device__ __forceinline__ u64 mad_wide_s(u32 a, u32 b, u64 c) {
    u64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// Constants of one prime's arithmetic.
template <int AR>
struct Mod {
    u64 q;
    u64 K;      // multiple of q: 2^13 q (NEAR50: makes any signed value non-negative), 7 q (NEAR60), 4 q (SHOUP)
    u32 delta;  // near primes
    static constexpr bool shoup = !is_near(AR);
    __device__ __forceinline__ explicit Mod(const Prime& p) : q(p.q) {
        K = AR == AR_NEAR50 ? p.q << 13 : AR == AR_NEAR60 ? p.q * 7 : p.q << 2;
        delta = p.delta;
    }
    // y w mod q for any y (NEAR50: signed), w a constant's two words; ranges above
    __device__ __forceinline__ u64 mul(u64 y, const ulonglong2& w) const {
        const u32 y0 = (u32)y, y1 = (u32)(y >> 32);
        const u32 a0 = (u32)w.x, a1 = (u32)(w.x >> 32), b0 = (u32)w.y, b1 = (u32)(w.y >> 32);
        if constexpr (shoup) {
            const u64 c0 = mul_wide(y0, b1), c1 = mul_wide(y1, b0);
            const u64 qh = mad_wide(y1, b1, (c0 >> 32) + (c1 >> 32));
            return y * w.x - qh * q;
        } else if constexpr (AR == AR_NEAR50) {
            const u64 A = mad_wide_s(y1, b0, mul_wide(y0, a0));
            const u64 B = mad_wide_s(y1, b1, mul_wide(y0, a1));
            return mad_wide_s((u32)(B >> 32), delta << 2, mad_wide((u32)B, 1u << 20, A));
        } else {
            const u64 A = mad_wide(y1, b0, mul_wide(y0, a0));
            const u64 B = mad_wide(y1, b1, mul_wide(y0, a1));
            return mad_wide((u32)(B >> 32), delta << 1, mad_wide((u32)B, 1u << 29, A));
        }
    }
    // a congruent value: NEAR50 any signed v to (-2^39, 2^50 + 2^39), NEAR60 any v below 2^60 + 2^30,
    // SHOUP v < 8 q below 4 q
    __device__ __forceinline__ u64 fold(u64 v) const {
        if constexpr (shoup) return v >= K ? v - K : v;
        else if constexpr (AR == AR_NEAR50) return mad_wide_s((u32)((i64)v >> 50), delta, v & (((u64)1 << 50) - 1));
        else return mad_wide((u32)(v >> 60), delta, v & (((u64)1 << 60) - 1));
    }
    // any v in the ranges above reduced to [0, q) (SHOUP: any v at all)
    __device__ __forceinline__ u64 canon(u64 v, u64 one_s) const {
        if constexpr (shoup) {
            v -= __umul64hi(v, one_s) * q;
        } else if constexpr (AR == AR_NEAR50) {
            v += K;  // in [0, 2^64)
            v = mad_wide((u32)(v >> 50), delta, v & (((u64)1 << 50) - 1));
        } else {
            v = fold(v);
        }
        const u64 d = v - q;  // v < 2 q < 2^62
        return (i64)d < 0 ? v : d;
    }
    // Forward Cooley-Tukey butterfly X <- X + W Y, Y <- X - W Y, in the i-th stage of a register block.
    __device__ __forceinline__ void ct(u64& x, u64& y, const ulonglong2& w, int i) const {
        const u64 t = mul(y, w);
        if constexpr (AR == AR_NEAR50) {
            y = x - t;
            x += t;
        } else {
            const u64 a = AR == AR_SHOUP || (AR == AR_NEAR60 && (i & 1) == 0) ? fold(x) : x;
            x = a + t;
            y = a + K - t;
        }
    }
    // Inverse Gentleman-Sande butterfly X <- X + Y, Y <- (X - Y) W. NEAR50: the block's inputs were folded,
    // so magnitudes are below 2^51, T, 2 T, 4 T before its four stages and 8 T < 2^63 after them. NEAR60
    // and SHOUP: values below 7 q, 4 q.
    __device__ __forceinline__ void gs(u64& x, u64& y, const ulonglong2& w) const {
        if constexpr (AR == AR_NEAR50) {
            const u64 d = x - y;
            x += y;
            y = mul(d, w);
        } else {
            const u64 d = x + K - y;
            x = fold(x + y);
            y = mul(d, w);
        }
    }
};

// Sum of products of two residues each, both variable. NEAR50: operands split at bit 25, four wide multiplies
// into three column sums (at most kTerms products), one folded product to reduce them all; otherwise
// Barrett per product. The tensor of 64 ciphertexts at N = 2^15, 8 limbs: 0.221 -> 0.186 ms (5.0 TB/s).
template <int AR>
struct Products {
    static constexpr int kTerms = 512;
    u64 c0 = 0, c1 = 0, c2 = 0;
    // the first product (the sum's start, which the Barrett form need not add to)
    __device__ __forceinline__ void start(u64 a, u64 b, const Prime& P) {
        if constexpr (AR == AR_NEAR50) add(a, b, P);
        else c0 = mul_mod(a, b, P);
    }
    __device__ __forceinline__ void add(u64 a, u64 b, const Prime& P) {
        if constexpr (AR == AR_NEAR50) {
            constexpr u32 m25 = (1u << 25) - 1;
            const u32 a0 = (u32)a & m25, a1 = (u32)(a >> 25), b0 = (u32)b & m25, b1 = (u32)(b >> 25);
            c0 = mad_wide(a0, b0, c0);
            c1 = mad_wide(a1, b0, mad_wide(a0, b1, c1));
            c2 = mad_wide(a1, b1, c2);
        } else {
            c0 = add_mod(c0, mul_mod(a, b, P), P.q);
        }
    }
    __device__ __forceinline__ void add_residue(u64 r, const Prime& P) {
        if constexpr (AR == AR_NEAR50) c0 += r;
        else c0 = add_mod(c0, r, P.q);
    }
    __device__ __forceinline__ u64 reduce(const Mod<AR>& m, const Prime& P) const {
        if constexpr (AR == AR_NEAR50) {
            const u64 d = c0 + ((c1 & ((1u << 25) - 1)) << 25), h = c2 + (c1 >> 25);  // below 2^60
            return m.canon(d + m.mul(h, make_ulonglong2(P.w50[0], P.w50[1])), 0);
        } else {
            return c0;
        }
    }
};
template <int AR>
__device__ __forceinline__ u64 product(u64 a, u64 b, const Mod<AR>& m, const Prime& P) {
    Products<AR> s;
    s.start(a, b, P);
    return s.reduce(m, P);
}

// Any 64-bit value reduced to [0, q): a lazy Shoup product by 1, then one correction.
__device__ __forceinline__ u64 reduce_any(u64 x, u64 q, u64 one_s) {
    u64 t = x - __umul64hi(x, one_s) * q;
    return t >= q ? t - q : t;
}

// m mod q for a signed m.
__device__ __forceinline__ u64 signed_residue(i64 m, const Prime& P) {
    const u64 r = reduce_any(m < 0 ? (u64)0 - (u64)m : (u64)m, P.q, P.one_s);
    return m < 0 && r ? P.q - r : r;
}

// Element x (within its sub-transform) that register u of the 2^RB-element group g holds in
// radix-2^RB block blk (block blk covers stages [RB blk, min(RB blk + RB, LOGM))).
template <int LOGM, int RB = 3>
__device__ __forceinline__ int block_elem(int blk, int g, int u) {
    constexpr int M = 1 << LOGM;
    const int s0 = RB * blk;
    const int b = (LOGM - s0) < RB ? (LOGM - s0) : RB;
    const int d = M >> (s0 + b);
    return (g / d) * ((1 << RB) * d) + (g % d) + u * d;
}

// Butterfly stages of one register block of a transform of M = 2^LOGM points: the 2^RB values of
// thread group g, elements block_elem(BLK, g, u), through stages [RB BLK, min(RB BLK + RB, LOGM))
// (forward ascending, inverse descending). tw(s, k) returns the twiddle of this thread's k-th
// sub-group at stage s (a block of b stages over 2^RB values holds 2^(RB-b+j) sub-groups at its stage j).
// FOLD: the inverse NEAR50 values may be large (every block but the first after reduced inputs).
template <int LOGM, int RB, int BLK, bool INV, bool FOLD, int AR, class TW>
__device__ __forceinline__ void block_stages(u64 (&v)[1 << RB], const Mod<AR>& m, TW&& tw) {
    constexpr int V = 1 << RB, S0 = RB * BLK;
    constexpr int b = (LOGM - S0) < RB ? (LOGM - S0) : RB;
    if (INV && FOLD && AR == AR_NEAR50) {
#pragma unroll
        for (int u = 0; u < V; u++) v[u] = m.fold(v[u]);
    }
#pragma unroll
    for (int i = 0; i < b; i++) {
        const int j = INV ? b - 1 - i : i;
        const int dist = 1 << (b - 1 - j);
#pragma unroll
        for (int u = 0; u < V; u++) {
            if (u & dist) continue;
            const ulonglong2 w = tw(S0 + j, u >> (b - j));
            if (INV) m.gs(v[u], v[u + dist], w);
            else m.ct(v[u], v[u + dist], w, i);
        }
    }
}

template <int V>
struct Tag {
    static constexpr int value = V;
};
// f is called with the arithmetic of prime p as a compile-time constant. LAZY: AR_LAZY is one of them, else its primes
// take AR_SHOUP: for forward transforms of many or short rows. In the passes of few rows a fourth copy of the code costs
// more than the reductions (two polynomials of three 32- and 40-bit limbs at N = 2^13, forward and inverse, 28.7 us
// without it and 29.5 with it).
template <bool LAZY, class F>
__device__ __forceinline__ void with_arith(const Prime& p, F&& f) {
    const u32 cls = p.cls;
    if (cls == AR_NEAR50) f(Tag<AR_NEAR50>{});
    else if (LAZY && cls == AR_LAZY) f(Tag<LAZY ? AR_LAZY : AR_SHOUP>{});
    else if (cls == AR_NEAR60) f(Tag<AR_NEAR60>{});
    else f(Tag<AR_SHOUP>{});
}

// The whole transform of one row of M = 2^LOGM points held in sm (element x at sm[x]) by M / 8
// threads, radix-8 register blocks between shared-memory exchanges (single-pass rings). The caller
// fills sm and synchronises before; the result is in sm after a final __syncthreads().
template <int LOGM, int BI, bool INV, int AR>
__device__ __forceinline__ void single_blocks(u64* sm, const ulonglong2* __restrict__ W, const Mod<AR>& m) {
    constexpr int RB = 3, V = 8, NB = (LOGM + RB - 1) / RB;
    if constexpr (BI < NB) {
        constexpr int BLK = INV ? NB - 1 - BI : BI, S0 = RB * BLK;
        const int g = threadIdx.x;
        u64 v[V];
#pragma unroll
        for (int u = 0; u < V; u++) v[u] = sm[block_elem<LOGM, RB>(BLK, g, u)];
        const int tb = block_elem<LOGM, RB>(BLK, g, 0) >> (LOGM - S0);  // the thread's first group at stage S0
        block_stages<LOGM, RB, BLK, INV, (BI > 0)>(v, m, [&](int s, int k) { return W[(1 << s) + (tb << (s - S0)) + k]; });
#pragma unroll
        for (int u = 0; u < V; u++) sm[block_elem<LOGM, RB>(BLK, g, u)] = v[u];
        __syncthreads();
        single_blocks<LOGM, BI + 1, INV>(sm, W, m);
    }
}

}  // namespace nttc
}  // namespace fhe
