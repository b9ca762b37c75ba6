// ks_inner.cu — key inner product of hybrid key switching (Han-Ki 2020), K3 of ks.cu:
//
//   acc[t][h][x][k] = sum_j M_j[x][k] * evk_j[h][px][k]        (plain / fan-out)
//   acc[t][h][x][k] = sum_r sum_j M_j[x][pi_r(k)] * evk_{r,j}[h][px][k]   (hoisted rotate-and-sum)
//
// M_j[x] is the raised digit j at extended limb x (K1 stores the limbs of digit j itself beside the
// converted ones, so every digit row is read alike), pi_r the slot map of rotation r. Products are
// summed exactly in 128 bits and reduced once, so the result is independent of the formulation; the
// variants differ in
//   * the multiply-accumulate: "C" (the product's low and high halves in C and a carry compare),
//     "P32" (a schoolbook chain of 32-bit mad.lo / mad.hi with carries) or, for data primes below
//     2^50, "S25" (operands split at bit 25: four mad.wide.u32 partial products into three 64-bit
//     column sums that cannot wrap, no additions at all),
//   * items per thread: items that share a key read each key pair once for all of them,
//   * the launch shape: blockIdx.y is the extended limb, so every block of one limb runs before the
//     next limb's, keeping that limb's key rows in L2 while every item reads them.
// An automorphism maps every aligned pair of evaluation slots onto an aligned pair, so a pair is
// one 128-bit load whatever the rotation; a key's two halves are interleaved, so the four key words of
// a slot pair are 32 contiguous bytes and one running pointer serves them.
//
// What bounds them: instruction issue (a wide multiply-add is two instructions, so the sums alone take 7 to 9
// per multiply-accumulate in registers, 13 to 15 in the kernels) and load latency at two blocks of 128
// registers per SM. 64 items, 15 rotations, N = 2^15, level 6 (S2, ms): 2.15 with digit rows selected
// between the raised digits and the input and keys in two rows, 1.93 as here, 1.83 with Karatsuba
// (S2L); one relinearisation 0.362 -> 0.229, most of it the shorter reduction (reduce128).
#include <algorithm>

#include "ks_inner.cuh"
#include "ntt_core.cuh"

namespace fhe {

const char* const kInnerVariantNames[INNER_N_VARIANTS] = {"v0", "c1", "p1", "s1", "s2", "s2l"};

namespace {

// (hi * 2^64 + lo) mod q for hi < 2^63. Near primes: hi times 2^64 mod q (one product of ntt_core.cuh) plus
// lo folded at 2^b, one correction: about 25 instructions. Otherwise hi and lo reduced with floor(2^64 / q),
// then hi * (2^64 mod q) + lo by Barrett, about 130. A relinearisation reduces after every dnum products,
// so this was most of its inner product (64 items at N = 2^15, level 6: 0.362 -> 0.274 ms with it).
template <int AR>
__device__ __forceinline__ u64 reduce128_near(u64 lo, u64 hi, const Prime& P) {
    const nttc::Mod<AR> m(P);
    constexpr int b = AR == nttc::AR_NEAR50 ? 50 : 60;
    const u64 l = nttc::mad_wide((u32)(lo >> b), P.delta, lo & (((u64)1 << b) - 1));
    return m.canon(l + m.mul(hi, make_ulonglong2(P.w64[0], P.w64[1])), 0);
}
__device__ __forceinline__ u64 reduce128(u64 lo, u64 hi, const Prime& P) {
    if (P.cls == nttc::AR_NEAR50) return reduce128_near<nttc::AR_NEAR50>(lo, hi, P);
    if (P.cls == nttc::AR_NEAR60) return reduce128_near<nttc::AR_NEAR60>(lo, hi, P);
    const u64 q = P.q;
    const u64 h = nttc::reduce_any(hi, q, P.one_s);
    const u64 l = nttc::reduce_any(lo, q, P.one_s);
    const u64 r64 = (u64)0 - q * P.one_s;  // 2^64 mod q
    return add_mod(mul_mod(h, r64, P), l, q);
}

// ---------------------------------------------------------------- multiply-accumulate forms

struct MacC {
    u64 lo = 0, hi = 0;
    __device__ __forceinline__ void mac(u64 a, u64 b) {
        const u64 pl = a * b, ph = __umul64hi(a, b);
        lo += pl;
        hi += ph + (lo < pl ? 1 : 0);
    }
    __device__ __forceinline__ u64 reduce(const Prime& P) const { return reduce128(lo, hi, P); }
    // packed: both operands are split at bit 25 (key_pack)
    __device__ __forceinline__ void macx(u64 a, u64 k, bool packed) {
        mac(packed ? key_unpack(a) : a, packed ? key_unpack(k) : k);
    }
};

struct MacP {  // PTX 64-bit multiply-add with carry (the one-item legacy form of the plain kernel)
    u64 lo = 0, hi = 0;
    __device__ __forceinline__ void mac(u64 a, u64 b) {
        asm("mad.lo.cc.u64 %0, %2, %3, %0;\n\tmadc.hi.u64 %1, %2, %3, %1;" : "+l"(lo), "+l"(hi) : "l"(a), "l"(b));
    }
    __device__ __forceinline__ u64 reduce(const Prime& P) const { return reduce128(lo, hi, P); }
    // packed: both operands are split at bit 25 (key_pack)
    __device__ __forceinline__ void macx(u64 a, u64 k, bool packed) {
        mac(packed ? key_unpack(a) : a, packed ? key_unpack(k) : k);
    }
};

// Schoolbook on 32-bit words in one carry chain per row: a0 b0 and a1 b1 first, then each cross
// product (eight mad.lo / mad.hi with carries and two carry propagations).
struct MacP32 {
    u32 r0 = 0, r1 = 0, r2 = 0, r3 = 0;
    __device__ __forceinline__ void mac(u64 a, u64 b) {
        const u32 a0 = (u32)a, a1 = (u32)(a >> 32), b0 = (u32)b, b1 = (u32)(b >> 32);
        asm("mad.lo.cc.u32 %0, %4, %6, %0;\n\t"
            "madc.hi.cc.u32 %1, %4, %6, %1;\n\t"
            "madc.lo.cc.u32 %2, %5, %7, %2;\n\t"
            "madc.hi.u32 %3, %5, %7, %3;\n\t"
            "mad.lo.cc.u32 %1, %4, %7, %1;\n\t"
            "madc.hi.cc.u32 %2, %4, %7, %2;\n\t"
            "addc.u32 %3, %3, 0;\n\t"
            "mad.lo.cc.u32 %1, %5, %6, %1;\n\t"
            "madc.hi.cc.u32 %2, %5, %6, %2;\n\t"
            "addc.u32 %3, %3, 0;"
            : "+r"(r0), "+r"(r1), "+r"(r2), "+r"(r3)
            : "r"(a0), "r"(a1), "r"(b0), "r"(b1));
    }
    __device__ __forceinline__ u64 reduce(const Prime& P) const {
        return reduce128(((u64)r1 << 32) | r0, ((u64)r3 << 32) | r2, P);
    }
    // packed: both operands are split at bit 25 (key_pack)
    __device__ __forceinline__ void macx(u64 a, u64 k, bool packed) {
        mac(packed ? key_unpack(a) : a, packed ? key_unpack(k) : k);
    }
};

// Operands below 2^50 split at bit 25: a b = a0 b0 + 2^25 (a0 b1 + a1 b0) + 2^50 a1 b1 with every
// partial product below 2^50, so three 64-bit column sums take up to 2^13 terms without a carry:
// four mad.wide.u32 per multiply-accumulate and no additions.
struct MacS25 {
    u64 C0 = 0, C1 = 0, C2 = 0;
    // packed operands (key_pack) hold their two halves in their two words
    __device__ __forceinline__ void macx(u64 a, u64 k, bool) {
        asm("mad.wide.u32 %0, %3, %5, %0;\n\t"
            "mad.wide.u32 %1, %3, %6, %1;\n\t"
            "mad.wide.u32 %1, %4, %5, %1;\n\t"
            "mad.wide.u32 %2, %4, %6, %2;"
            : "+l"(C0), "+l"(C1), "+l"(C2)
            : "r"((u32)a), "r"((u32)(a >> 32)), "r"((u32)k), "r"((u32)(k >> 32)));
    }
    // C0 + 2^25 cross + 2^50 C2: near primes d + 2^50 h with d, h below 2^60 (at most 512 terms), h times 2^50
    // mod q; otherwise as 128 bits
    static __device__ __forceinline__ u64 reduce_columns(u64 C0, u64 cross, u64 C2, const Prime& P) {
        const u64 d = C0 + ((cross & ((1u << 25) - 1)) << 25), h = C2 + (cross >> 25);
        if (P.cls == nttc::AR_NEAR50) {
            const nttc::Mod<nttc::AR_NEAR50> m(P);
            return m.canon(d + m.mul(h, make_ulonglong2(P.w50[0], P.w50[1])), 0);
        }
        const u64 lo = d + (h << 50);
        return reduce128(lo, (h >> 14) + (lo < d ? 1 : 0), P);
    }
    __device__ __forceinline__ u64 reduce(const Prime& P) const { return reduce_columns(C0, C1, C2, P); }
};

// S25 with both cross products from one multiply, (a0 + a1)(b0 + b1) - a0 b0 - a1 b1 (Karatsuba): three
// wide multiplies and an addition per operand, shared by the products an operand enters.
struct MacK25 {
    u64 C0 = 0, C1 = 0, C2 = 0;
    __device__ __forceinline__ void macx(u64 a, u64 k, bool) {
        const u32 a0 = (u32)a, a1 = (u32)(a >> 32), b0 = (u32)k, b1 = (u32)(k >> 32);
        C0 = nttc::mad_wide(a0, b0, C0);
        C1 = nttc::mad_wide(a0 + a1, b0 + b1, C1);
        C2 = nttc::mad_wide(a1, b1, C2);
    }
    __device__ __forceinline__ u64 reduce(const Prime& P) const { return MacS25::reduce_columns(C0, C1 - C0 - C2, C2, P); }
};

// Slots (2 k2, 2 k2 + 1) of phi_g(row): the automorphism maps the aligned pair onto an aligned pair.
__device__ __forceinline__ void load_pair_auto(const u64* __restrict__ row, int k2, int g, int log_n, u64& vx, u64& vy) {
    const int src = auto_src(2 * k2, g, log_n);
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(row)[src >> 1];
    vx = (src & 1) ? v.y : v.x;
    vy = (src & 1) ? v.x : v.y;
}

// (b, a) of slots 2 k2 and 2 k2 + 1 of a key row: key points at the row's first pair
struct KeyPair {
    ulonglong2 x, y;
};
__device__ __forceinline__ KeyPair load_key(const ulonglong2* __restrict__ p) { return {p[0], p[1]}; }

// c0sum at slot pair k2 of item t, limb x: c0 and its rotations (hoisted, data limbs)
__device__ __forceinline__ void store_c0sum(const InnerArgs& a, int t, int x, int k2, u64 q) {
    const u64* c0 = a.tab[t].addP0 + ((size_t)x << a.log_n);
    const ulonglong2 self = reinterpret_cast<const ulonglong2*>(c0)[k2];
    u64 sx = self.x, sy = self.y;
    for (int r = 0; r < a.n_steps; r++) {
        u64 vx, vy;
        load_pair_auto(c0, k2, (int)a.steps[r].galois, a.log_n, vx, vy);
        sx = add_mod(sx, vx, q);
        sy = add_mod(sy, vy, q);
    }
    reinterpret_cast<ulonglong2*>(a.c0sum + ((size_t)(t * (a.level + 1) + x) << a.log_n))[k2] = make_ulonglong2(sx, sy);
}

// The four sums (half 0 and 1 at slots 2 k2, 2 k2 + 1) of one item.
template <class MAC>
struct Sums {
    MAC b0, b1, a0, a1;
    __device__ __forceinline__ void add(u64 v0, u64 v1, const KeyPair& k, bool packed) {
        b0.macx(v0, k.x.x, packed);
        b1.macx(v1, k.y.x, packed);
        a0.macx(v0, k.x.y, packed);
        a1.macx(v1, k.y.y, packed);
    }
    __device__ __forceinline__ void store(const InnerArgs& a, int t, int x, int k2, const Prime& P) const {
        ulonglong2* acc = reinterpret_cast<ulonglong2*>(a.acc + ((size_t)(t * 2 * a.next + x) << a.log_n)) + k2;
        acc[0] = make_ulonglong2(b0.reduce(P), b1.reduce(P));
        acc[(size_t)a.next << (a.log_n - 1)] = make_ulonglong2(a0.reduce(P), a1.reduce(P));
    }
};

// ---------------------------------------------------------------- v0: the grid-stride forms

template <bool FANOUT>
__global__ void __launch_bounds__(256, 4) inner_v0_kernel(InnerArgs a) {
    const int hl = a.log_n - 1, l1 = a.level + 1;
    const size_t total = (size_t)a.items * a.next << hl;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int k2 = (int)(e & (((size_t)1 << hl) - 1));
        const size_t row = e >> hl;
        const int t = (int)(row % a.items), x = (int)(row / a.items);
        const int px = x < l1 ? x : x + (a.L - a.level);
        const KsItem it = a.tab[t];
        const bool packed = a.keys_packed && x < l1;
        const int st = FANOUT ? a.src_of[t] : t;
        const ulonglong2* kr = reinterpret_cast<const ulonglong2*>(it.key) + ((size_t)px << a.log_n) + 2 * k2;
        Sums<MacP> s;
        for (int j = 0; j < a.dn; j++) {
            u64 vx, vy;
            load_pair_auto(a.ext + ((size_t)((st * a.dn + j) * a.next + x) << a.log_n), k2, FANOUT ? (int)it.galois : 1,
                           a.log_n, vx, vy);
            s.add(vx, vy, load_key(kr + ((size_t)(j * a.n_ext) << a.log_n)), packed);
        }
        s.store(a, t, x, k2, a.pr[px]);
    }
}

__global__ void __launch_bounds__(256, 3) hoist_v0_kernel(InnerArgs a) {
    const int hl = a.log_n - 1, l1 = a.level + 1;
    const size_t total = (size_t)a.items * a.next << hl;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int k2 = (int)(e & (((size_t)1 << hl) - 1));
        const size_t row = e >> hl;
        const int t = (int)(row % a.items), x = (int)(row / a.items);
        const int px = x < l1 ? x : x + (a.L - a.level);
        const bool packed = a.keys_packed && x < l1;
        Sums<MacC> s;
        for (int r = 0; r < a.n_steps; r++) {
            const HoistStep st = a.steps[r];
            const ulonglong2* kr = reinterpret_cast<const ulonglong2*>(st.key) + ((size_t)px << a.log_n) + 2 * k2;
            for (int j = 0; j < a.dn; j++) {
                u64 vx, vy;
                load_pair_auto(a.ext + ((size_t)((t * a.dn + j) * a.next + x) << a.log_n), k2, (int)st.galois, a.log_n, vx, vy);
                s.add(vx, vy, load_key(kr + ((size_t)(j * a.n_ext) << a.log_n)), packed);
            }
        }
        s.store(a, t, x, k2, a.pr[px]);
        if (x < l1) store_c0sum(a, t, x, k2, a.pr[px].q);
    }
}

// ---------------------------------------------------------------- 2-D forms, IPT items per thread

// Thread (blockIdx.x * 256 + threadIdx.x) = (item group, pair k2) with k2 fastest; blockIdx.y = limb x.
// Items t0 .. t0 + IPT - 1 of a group; a ragged last group repeats its last item and skips its stores.
// The data limbs (x <= level) use the multiply-accumulate MACD when every data prime has at most 50
// bits (a.split25: digits and keys are packed), the special limbs and every other case MACS; the branch is
// uniform per block. Pointers run along the digits.

// Operands of one digit: the key words and each item's digit pair.
template <int IPT>
struct Operands {
    KeyPair k;
    ulonglong2 v[IPT];
};
template <class MAC, int IPT, bool PK>
__device__ __forceinline__ void mac_all(Sums<MAC> (&s)[IPT], const Operands<IPT>& o, bool swap) {
#pragma unroll
    for (int i = 0; i < IPT; i++) s[i].add(swap ? o.v[i].y : o.v[i].x, swap ? o.v[i].x : o.v[i].y, o.k, PK);
}

// Plain / fan-out: every item of a thread uses the same key (IPT > 1 only when the items share it); FANOUT
// reads item t's digits from source src_of[t] through its automorphism (plain digits were permuted by K1).
template <class MAC, int IPT, bool FANOUT, bool PK>
__device__ __forceinline__ void inner2_body(const InnerArgs& a, int x, int k2, int t0) {
    const int hl = a.log_n - 1, l1 = a.level + 1;
    const int px = x < l1 ? x : x + (a.L - a.level);
    const u64* key = IPT > 1 ? a.shared_key : a.tab[t0].key;
    const int src = FANOUT ? auto_src(2 * k2, (int)a.tab[t0].galois, a.log_n) : 2 * k2;
    const bool swap = FANOUT && (src & 1);
    const ulonglong2* kp = reinterpret_cast<const ulonglong2*>(key) + ((size_t)px << a.log_n) + 2 * k2;
    const ulonglong2* vp[IPT];
#pragma unroll
    for (int i = 0; i < IPT; i++) {
        const int t = min(t0 + i, a.items - 1), st = FANOUT ? a.src_of[t] : t;
        vp[i] = reinterpret_cast<const ulonglong2*>(a.ext) + (((size_t)st * a.dn * a.next + x) << hl) + (src >> 1);
    }
    const size_t vstride = (size_t)a.next << hl, kstride = (size_t)a.n_ext << a.log_n;
    auto load = [&](Operands<IPT>& o) {
        o.k = load_key(kp);
        kp += kstride;
#pragma unroll
        for (int i = 0; i < IPT; i++) {
            o.v[i] = *vp[i];
            vp[i] += vstride;
        }
    };
    Sums<MAC> s[IPT];
#pragma unroll 4
    for (int j = 0; j < a.dn; j++) {
        Operands<IPT> o;
        load(o);
        mac_all<MAC, IPT, PK>(s, o, swap);
    }
    const Prime P = a.pr[px];
#pragma unroll
    for (int i = 0; i < IPT; i++)
        if (t0 + i < a.items) s[i].store(a, t0 + i, x, k2, P);
}

template <class MACD, class MACS, int IPT, bool FANOUT>
__global__ void __launch_bounds__(256, IPT == 1 ? 3 : 2) inner2_kernel(InnerArgs a) {
    const int hl = a.log_n - 1;
    const int x = blockIdx.y;
    const unsigned e = blockIdx.x * 256u + threadIdx.x;
    const int k2 = (int)(e & ((1u << hl) - 1u));
    const int t0 = (int)(e >> hl) * IPT;
    if (t0 >= a.items) return;
    if (x <= a.level && a.split25) inner2_body<MACD, IPT, FANOUT, true>(a, x, k2, t0);
    else if (x <= a.level && a.keys_packed) inner2_body<MACS, IPT, FANOUT, true>(a, x, k2, t0);
    else inner2_body<MACS, IPT, FANOUT, false>(a, x, k2, t0);
}

template <class MAC, int IPT, bool PK>
__device__ __forceinline__ void hoist2_body(const InnerArgs& a, int x, int k2, int t0) {
    const int hl = a.log_n - 1, l1 = a.level + 1;
    const int px = x < l1 ? x : x + (a.L - a.level);
    const ulonglong2* row[IPT];
#pragma unroll
    for (int i = 0; i < IPT; i++)
        row[i] = reinterpret_cast<const ulonglong2*>(a.ext) + (((size_t)min(t0 + i, a.items - 1) * a.dn * a.next + x) << hl);
    const size_t vstride = (size_t)a.next << hl, kstride = (size_t)a.n_ext << a.log_n;
    const size_t koff = ((size_t)px << a.log_n) + 2 * k2;
    // packed residues are below 2^50, so c0 and its at most 31 rotations are summed unreduced beside the products
    const ulonglong2* c0[IPT];
    ulonglong2 c0s[IPT];
    if (PK && x < l1) {
#pragma unroll
        for (int i = 0; i < IPT; i++) {
            c0[i] = reinterpret_cast<const ulonglong2*>(a.tab[min(t0 + i, a.items - 1)].addP0) + ((size_t)x << hl);
            c0s[i] = c0[i][k2];
        }
    }
    Sums<MAC> s[IPT];
    for (int r = 0; r < a.n_steps; r++) {
        const HoistStep st = a.steps[r];
        const int src = auto_src(2 * k2, (int)st.galois, a.log_n);
        const bool swap = src & 1;
        const ulonglong2* kp = reinterpret_cast<const ulonglong2*>(st.key) + koff;
        const ulonglong2* vp[IPT];
#pragma unroll
        for (int i = 0; i < IPT; i++) vp[i] = row[i] + (src >> 1);
        auto load = [&](Operands<IPT>& o) {
            o.k = load_key(kp);
            kp += kstride;
#pragma unroll
            for (int i = 0; i < IPT; i++) {
                o.v[i] = *vp[i];
                vp[i] += vstride;
            }
        };
        // two digits at a time: 1.83 ms against 1.91 (one) and 1.90 (four) for the shape above
#pragma unroll 2
        for (int j = 0; j < a.dn; j++) {
            Operands<IPT> o;
            load(o);
            mac_all<MAC, IPT, PK>(s, o, swap);
        }
        if (PK && x < l1) {
#pragma unroll
            for (int i = 0; i < IPT; i++) {
                const ulonglong2 c = c0[i][src >> 1];
                c0s[i].x += swap ? c.y : c.x;
                c0s[i].y += swap ? c.x : c.y;
            }
        }
    }
    const Prime P = a.pr[px];
#pragma unroll
    for (int i = 0; i < IPT; i++)
        if (t0 + i < a.items) {
            s[i].store(a, t0 + i, x, k2, P);
            if (PK && x < l1)
                reinterpret_cast<ulonglong2*>(a.c0sum + ((size_t)((t0 + i) * l1 + x) << a.log_n))[k2] =
                    make_ulonglong2(nttc::reduce_any(c0s[i].x, P.q, P.one_s), nttc::reduce_any(c0s[i].y, P.q, P.one_s));
            else if (x < l1)
                store_c0sum(a, t0 + i, x, k2, P.q);
        }
}

template <class MACD, class MACS, int IPT>
__global__ void __launch_bounds__(256, IPT == 1 ? 3 : 2) hoist2_kernel(InnerArgs a) {
    const int hl = a.log_n - 1;
    const int x = blockIdx.y;
    const unsigned e = blockIdx.x * 256u + threadIdx.x;
    const int k2 = (int)(e & ((1u << hl) - 1u));
    const int t0 = (int)(e >> hl) * IPT;
    if (t0 >= a.items) return;
    if (x <= a.level && a.split25) hoist2_body<MACD, IPT, true>(a, x, k2, t0);
    else if (x <= a.level && a.keys_packed) hoist2_body<MACS, IPT, true>(a, x, k2, t0);
    else hoist2_body<MACS, IPT, false>(a, x, k2, t0);
}

inline unsigned grid1(size_t work) {
    size_t b = (work + 255) / 256;
    return (unsigned)std::min<size_t>(std::max<size_t>(b, 1), (size_t)1 << 30);
}

inline dim3 grid2(const InnerArgs& a, int ipt) {
    const size_t groups = (size_t)(a.items + ipt - 1) / ipt;
    const size_t threads = groups << (a.log_n - 1);
    return dim3((unsigned)((threads + 255) / 256), (unsigned)a.next);
}

}  // namespace

void launch_ks_inner(const InnerArgs& a0, bool fanout, int variant, int max_data_prime_bits, cudaStream_t s) {
    if (a0.items == 0) return;
    InnerArgs a = a0;
    if (variant <= INNER_V0 || variant >= INNER_N_VARIANTS) {
        if (fanout)
            inner_v0_kernel<true><<<grid1((size_t)a.items * a.next << (a.log_n - 1)), 256, 0, s>>>(a);
        else
            inner_v0_kernel<false><<<grid1((size_t)a.items * a.next << (a.log_n - 1)), 256, 0, s>>>(a);
        CK(cudaGetLastError());
        return;
    }
    // split at bit 25 needs data primes below 2^50 and at most 512 terms per sum (MacS25::reduce)
    a.split25 = a.keys_packed && max_data_prime_bits <= 50 && a.dn <= 512;
    const bool two = (variant == INNER_S2 || variant == INNER_S2L) && !fanout && a.shared_key && a.items > 1;
#define L2(MD, MS, I, F) inner2_kernel<MD, MS, I, F><<<grid2(a, I), 256, 0, s>>>(a)
    switch (variant) {
        case INNER_C1:
            if (fanout) L2(MacC, MacC, 1, true);
            else L2(MacC, MacC, 1, false);
            break;
        case INNER_P1:
            if (fanout) L2(MacP32, MacP32, 1, true);
            else L2(MacP32, MacP32, 1, false);
            break;
        case INNER_S2L:
            if (fanout) L2(MacK25, MacP32, 1, true);
            else if (two) L2(MacK25, MacP32, 2, false);
            else L2(MacK25, MacP32, 1, false);
            break;
        default:  // S1, S2
            if (fanout) L2(MacS25, MacP32, 1, true);
            else if (two) L2(MacS25, MacP32, 2, false);
            else L2(MacS25, MacP32, 1, false);
            break;
    }
#undef L2
    CK(cudaGetLastError());
}

void launch_ks_hoist_inner(const InnerArgs& a0, int variant, int max_data_prime_bits, cudaStream_t s) {
    if (a0.items == 0) return;
    InnerArgs a = a0;
    if (variant <= INNER_V0 || variant >= INNER_N_VARIANTS) {
        hoist_v0_kernel<<<grid1((size_t)a.items * a.next << (a.log_n - 1)), 256, 0, s>>>(a);
        CK(cudaGetLastError());
        return;
    }
    a.split25 = a.keys_packed && max_data_prime_bits <= 50 && (long long)a.dn * a.n_steps <= 512;
#define H2(MD, MS, I) hoist2_kernel<MD, MS, I><<<grid2(a, I), 256, 0, s>>>(a)
    switch (variant) {
        case INNER_C1: H2(MacC, MacC, 1); break;
        case INNER_P1: H2(MacP32, MacP32, 1); break;
        case INNER_S2:
            if (a.items > 1) H2(MacS25, MacP32, 2);
            else H2(MacS25, MacP32, 1);
            break;
        case INNER_S2L:
            if (a.items > 1) H2(MacK25, MacP32, 2);
            else H2(MacK25, MacP32, 1);
            break;
        default: H2(MacS25, MacP32, 1); break;
    }
#undef H2
    CK(cudaGetLastError());
}

}  // namespace fhe
