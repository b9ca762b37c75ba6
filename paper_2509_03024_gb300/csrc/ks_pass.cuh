// ks_pass.cuh — the fused NTT passes of key switching and rescaling (ks.cu): row descriptors,
// the load and store modes that fuse the base conversions and the combinations into the first and
// last pass of a transform, the pass kernel and its launchers. See ks.cu for the algorithm.
#pragma once

#include <type_traits>

#include "ks_inner.cuh"
#include "launch_rules.h"
#include "ntt_core.cuh"

namespace fhe {

namespace ksp {

enum LoadMode { LD_PLAIN = 0, LD_GATHER = 1, LD_CONV = 2, LD_AXPY = 3, LD_CENTRED = 4, LD_MUL = 5 };
enum StoreMode { ST_LAZY = 0, ST_LAST = 1, ST_SCALE = 2, ST_COMBINE = 3, ST_COMBINE_RS = 4, ST_RESCALE = 5 };

struct KsRow {
    u64* dst;        // the row's buffer (N residues)
    const u64* src;  // LD_GATHER: source row; LD_CONV: first source limb (limb stride N)
    const u64* cst;  // LD_CONV: constant words of the first source limb for this row's prime; ST_SCALE: words of the factor
    int prime;       // prime index of the row
    int galois;      // LD_GATHER: automorphism applied on load (1 = none)
    int src_cnt;     // LD_CONV: number of source limbs
    int cst_stride;  // LD_CONV: words between consecutive source limbs' constant pairs
    int item, half, limb;  // ST_COMBINE(_RS): output item, component and limb
    int pack;              // ST_LAST (forward), out2 of LD_GATHER: store the residue split at bit 25 (key_pack)
    const u64* src2;       // LD_AXPY / LD_MUL: second source row (LD_AXPY: null = none); ST_RESCALE: the input limb
    const u64* cst2;       // LD_AXPY: words of its factor; ST_RESCALE: words of q_l^-1 mod the row's prime
    u64* out2;             // ST_RESCALE: output row; LD_GATHER: second copy of the loaded row (null = none)
    const u64* src3;       // ST_RESCALE: when set, the input limb is src2 (.) src3 (a plaintext product)
};

constexpr int kMaxHoist = 31;

// Rotation keys of a hoisted rotate-and-sum (host side).
struct HoistKeys {
    const u64* key[kMaxHoist];
    int galois[kMaxHoist];
    int count;
};

struct CombineArgs {
    const KsItem* items;
    const u64* acc;    // [items][2][next][N]
    const u64* pinv;   // [L+1][2] words of P^-1 mod q_i (ST_COMBINE) or (P q_l)^-1 mod q_i (ST_COMBINE_RS)
    int next;
    const u64* qlinv;  // ST_COMBINE_RS: [L+1][2] words of q_l^-1 mod q_i
};

__device__ __forceinline__ ulonglong2 words(const u64* p) { return make_ulonglong2(p[0], p[1]); }

// Base conversion sum_i y_i c_i mod a 50-bit near prime: every c_i as two words split at bit 21, A and B
// the sums of the low and high partial products (y_i below 2^61: A below 2^55.2, B below 2^63.2 for
// four sources), folded once at 2^53 = 8 delta. The result, below 2^60.4, enters the forward transform
// as it is.
struct ConvSum {
    u64 A = 0, B = 0;
    __device__ __forceinline__ void add(u64 y, const ulonglong2& w) {
        const u32 y0 = (u32)y, y1 = (u32)(y >> 32);
        A = nttc::mad_wide(y1, (u32)w.y, nttc::mad_wide(y0, (u32)w.x, A));
        B = nttc::mad_wide(y1, (u32)(w.y >> 32), nttc::mad_wide(y0, (u32)(w.x >> 32), B));
    }
    __device__ __forceinline__ u64 value(u32 delta) const {
        return nttc::mad_wide((u32)(B >> 32), delta << 3, A + ((u64)(u32)B << kConvSplit));
    }
};

// Per-row constants of the first pass's loads, read once per row: the words of the (at most kConvMax)
// source limbs' constants of a base conversion, and the last limb's prime of a centred load.
constexpr int kConvMax = 4;
struct RowConst {
    u64 ql;
    ulonglong2 w[kConvMax];
};

template <int LOAD>
__device__ __forceinline__ RowConst row_const(const KsRow& r, const Prime* __restrict__ pr) {
    RowConst c;
    c.ql = LOAD == LD_CENTRED ? pr[r.limb].q : 0;
#pragma unroll
    for (int i = 0; i < kConvMax; i++)
        c.w[i] = LOAD == LD_CONV && i < r.src_cnt ? words(r.cst + (size_t)i * r.cst_stride) : make_ulonglong2(0, 0);
    return c;
}

// LD_CONV: the base conversion of residue k, sum_i src_i[k] c_i: over CNT sources already loaded to x ...
template <int AR, int CNT>
__device__ __forceinline__ u64 conv_sum(const u64 (&x)[CNT], const nttc::Mod<AR>& m, const RowConst& rc) {
    if constexpr (AR == nttc::AR_NEAR50) {
        ConvSum s;
#pragma unroll
        for (int i = 0; i < CNT; i++) s.add(x[i], rc.w[i]);
        return s.value(m.delta);
    } else {
        u64 acc = m.mul(x[0], rc.w[0]);
#pragma unroll
        for (int i = 1; i < CNT; i++) acc = m.fold(acc) + m.mul(x[i], rc.w[i]);
        return acc;
    }
}
// ... or over any number of them.
template <int AR>
__device__ __forceinline__ u64 conv_any(const KsRow& r, size_t k, int log_n, const nttc::Mod<AR>& m) {
    u64 acc = 0;
    for (int i0 = 0; i0 < r.src_cnt; i0 += kConvMax) {
        ConvSum s;
        for (int i = i0; i < min(i0 + kConvMax, r.src_cnt); i++) {
            const u64 x = r.src[((size_t)i << log_n) + k];
            const ulonglong2 w = words(r.cst + (size_t)i * r.cst_stride);
            if constexpr (AR == nttc::AR_NEAR50) s.add(x, w);
            else acc = m.fold(acc) + m.mul(x, w);
        }
        if constexpr (AR == nttc::AR_NEAR50) acc += m.fold(s.value(m.delta));
    }
    return acc;
}
// Conversions of V residues, at(u) = conversion of residue addr(u). The loads of several residues are issued
// together before anything is stored: a store to shared memory in between would order them (the compiler
// cannot tell the source rows from it), one round trip to L2 per residue.
template <int AR, int CNT, int V, class ADDR, class AT>
__device__ __forceinline__ void conv_rows(const KsRow& r, int log_n, const nttc::Mod<AR>& m, const RowConst& rc, ADDR&& addr,
                                          AT&& at) {
    if constexpr (CNT == 0) {
        for (int u = 0; u < V; u++) at(u) = conv_any(r, addr(u), log_n, m);
    } else {
        constexpr int G = CNT <= 2 ? 8 : 4;
        for (int u0 = 0; u0 < V; u0 += G) {
            u64 x[G][CNT];
#pragma unroll
            for (int u = 0; u < G; u++)
#pragma unroll
                for (int i = 0; i < CNT; i++) x[u][i] = r.src[((size_t)i << log_n) + addr(u0 + u)];
#pragma unroll
            for (int u = 0; u < G; u++) at(u0 + u) = conv_sum<AR, CNT>(x[u], m, rc);
        }
    }
}
// f is called with the number of sources as a compile-time constant (0: more than kConvMax).
template <class F>
__device__ __forceinline__ void with_count(int cnt, F&& f) {
    if (cnt == 1) f(nttc::Tag<1>{});
    else if (cnt == 2) f(nttc::Tag<2>{});
    else if (cnt == 3) f(nttc::Tag<3>{});
    else if (cnt == 4) f(nttc::Tag<4>{});
    else f(nttc::Tag<0>{});
}

// Residue k of the row as it stands in memory (LD_CONV: conv_rows). The single-pass kernel loads it before anything
// of the row's prime is known: behind the branch on the prime's arithmetic the loads wait for the prime, one more
// trip to L2 in a launch that may be a handful of them (two launches of three rows at N = 2^9 10.5 -> 9.1 us).
template <int LOAD>
__device__ __forceinline__ u64 load_raw(const KsRow& r, size_t k, int log_n) {
    if constexpr (LOAD == LD_PLAIN) return r.dst[k];
    else if constexpr (LOAD == LD_GATHER) return r.src[r.galois == 1 ? (int)k : auto_src((int)k, r.galois, log_n)];
    else return r.src[k];
}
// The same as the transform takes it: a congruent value, for a forward transform within 2^60.4 (NEAR50, signed),
// below 16 q (NEAR60) or 8 q (SHOUP); reduced for an inverse one.
template <int LOAD, int AR>
__device__ __forceinline__ u64 load_elem(const KsRow& r, u64 v, size_t k, const Prime& P, const nttc::Mod<AR>& m,
                                         const RowConst& rc) {
    if constexpr (LOAD == LD_PLAIN || LOAD == LD_GATHER) {
        return v;
    } else if constexpr (LOAD == LD_CENTRED) {  // the centred representative of src[k] (mod q_limb)
        const u64 ql = rc.ql;
        const bool neg = v > (ql >> 1);
        if constexpr (AR == nttc::AR_NEAR50) {
            return neg ? v - ql : v;  // signed, magnitude at most 2^60
        } else {
            const u64 mag = neg ? ql - v : v;
            const u64 t = nttc::reduce_any(mag, P.q, P.one_s);
            return neg ? (t ? P.q - t : 0) : t;
        }
    } else if constexpr (LOAD == LD_MUL) {
        return nttc::product(v, r.src2[k], m, P);
    } else {  // LD_AXPY: src + cst2 * src2
        static_assert(LOAD == LD_AXPY, "load mode");
        return r.src2 ? m.canon(v + m.mul(r.src2[k], words(r.cst2)), P.one_s) : v;
    }
}

// Residue k of the row from the transform's (unreduced) value v, in two steps so that the loads of several
// residues go out before the first store (which the compiler cannot tell from them): store_operands, then
// store_elem.
struct StoreIn {
    u64 a, b, c;
};
template <int STORE>
__device__ __forceinline__ StoreIn store_operands(const KsRow& r, size_t k, const CombineArgs& ca, int log_n) {
    StoreIn in{0, 0, 0};
    if constexpr (STORE == ST_RESCALE) {
        in.a = r.src2[k];
        if (r.src3) in.b = r.src3[k];
    } else if constexpr (STORE == ST_COMBINE || STORE == ST_COMBINE_RS) {
        const KsItem& it = ca.items[r.item];
        const size_t row_off = (size_t)r.limb << log_n;
        in.a = ca.acc[((((size_t)r.item * 2 + r.half) * ca.next + r.limb) << log_n) + k];
        const u64* add = r.half == 0 ? it.addI0 : it.addI1;
        if (add) in.b = add[row_off + k];
        if (STORE == ST_COMBINE && r.half == 0 && it.addP0)
            in.c = it.addP0[row_off + (it.galois == 1 ? (int)k : auto_src((int)k, (int)it.galois, log_n))];
    }
    return in;
}
template <bool INV, int STORE, int AR>
__device__ __forceinline__ void store_elem(const KsRow& r, size_t k, u64 v, const StoreIn& in, const Prime& P,
                                           const nttc::Mod<AR>& m, const u64* __restrict__ ninv, const CombineArgs& ca,
                                           int log_n) {
    const u64 q = m.q, one_s = P.one_s;
    if constexpr (STORE == ST_LAZY) {
        r.dst[k] = v;
    } else if constexpr (STORE == ST_LAST || STORE == ST_SCALE) {  // inverse: times N^-1, or the row's constant in its place
        const u64 t = m.canon(INV ? m.mul(v, words(STORE == ST_SCALE ? r.cst : ninv + 2 * r.prime)) : v, one_s);
        r.dst[k] = !INV && r.pack ? key_pack(t) : t;
    } else if constexpr (STORE == ST_RESCALE) {  // forward: out = (x - [x_l]) q_l^-1 with the transformed [x_l] in v
        const u64 x = r.src3 ? nttc::product(in.a, in.b, m, P) : in.a;
        r.out2[k] = m.canon(m.mul(x + q - m.canon(v, one_s), words(r.cst2)), one_s);
    } else {
        // out_h = (acc_h - v) P^-1 + add terms (Mod::mul's range and two reduced terms fit 64 bits); with the fused
        // rescale (acc_h - v) (P q_l)^-1 + c_h q_l^-1
        u64 s = m.mul(in.a + q - m.canon(v, one_s), words(ca.pinv + 2 * r.limb));
        s += STORE == ST_COMBINE_RS ? m.mul(in.b, words(ca.qlinv + 2 * r.limb)) : in.b + in.c;
        const KsItem& it = ca.items[r.item];
        (r.half == 0 ? it.out0 : it.out1)[((size_t)r.limb << log_n) + k] = m.canon(s, one_s);
    }
}

// ---------------------------------------------------------------- pass kernels

// Rows of a launch: a descriptor table in device memory, or the regular rows of a PolyBatch (plain NTT).
struct RowTable {
    const KsRow* rows;
    __device__ __forceinline__ KsRow get(int i, int) const { return rows[i]; }
};
struct RowBatch {
    PolyBatch pb;
    __device__ __forceinline__ KsRow get(int i, int log_n) const {
        const int li = i % pb.n_limbs, rest = i / pb.n_limbs, limb = pb.limb_lo + li;
        KsRow r{};
        r.dst = pb.base + (size_t)(rest / pb.n_parts) * pb.item_stride + (size_t)(rest % pb.n_parts) * pb.part_stride +
                ((size_t)(limb - pb.addr_lo) << log_n);
        r.prime = pb.prime_of(limb);
        return r;
    }
};

// Whole transform of one row per CTA (rings up to 2^12, see rules::single_pass).
template <class ROWS, int LOGN, bool INV, int LOAD, int STORE>
__global__ void __launch_bounds__((1 << LOGN) / 8, 1024 / ((1 << LOGN) / 8))
single_pass_kernel(ROWS rows, const Prime* __restrict__ primes, const ulonglong2* __restrict__ tw,
                   const u64* __restrict__ ninv, CombineArgs ca) {
    constexpr int N = 1 << LOGN, T = N / 8;
    extern __shared__ u64 sm[];
    const KsRow r = rows.get(blockIdx.x, LOGN);
    const Prime& P = primes[r.prime];
    const int tid = threadIdx.x;
    auto at = [&](int u) -> u64& { return sm[tid + u * T]; };
    auto addr = [&](int u) -> size_t { return tid + u * T; };
    u64 raw[LOAD == LD_CONV ? 1 : 8];
    if constexpr (LOAD != LD_CONV) {
#pragma unroll
        for (int u = 0; u < 8; u++) raw[u] = load_raw<LOAD>(r, addr(u), LOGN);
    }
    nttc::with_arith<!INV>(P, [&](auto ar) {
        constexpr int AR = decltype(ar)::value;
        const nttc::Mod<AR> m(P);
        const RowConst rc = row_const<LOAD>(r, primes);
        if constexpr (LOAD == LD_CONV) {
            with_count(r.src_cnt, [&](auto cnt) { conv_rows<AR, decltype(cnt)::value, 8>(r, LOGN, m, rc, addr, at); });
        } else {
            u64 v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) v[u] = load_elem<LOAD>(r, raw[u], addr(u), P, m, rc);
#pragma unroll
            for (int u = 0; u < 8; u++) {
                at(u) = v[u];
                if (LOAD == LD_GATHER && r.out2) r.out2[addr(u)] = r.pack ? key_pack(v[u]) : v[u];
            }
        }
        __syncthreads();
        nttc::single_blocks<LOGN, 0, INV>(sm, tw + ((size_t)r.prime << LOGN), m);
        StoreIn in[8];
#pragma unroll
        for (int u = 0; u < 8; u++) in[u] = store_operands<STORE>(r, addr(u), ca, LOGN);
#pragma unroll
        for (int u = 0; u < 8; u++) store_elem<INV, STORE>(r, addr(u), at(u), in[u], P, m, ninv, ca, LOGN);
    });
}

// One pass of the two-pass transform of a ring of 2^LOGN = N1 x N2 (N1 rows of N2): PASS 0 transforms
// columns of N1 = M points (R consecutive columns per CTA), PASS 1 rows of N2 = M points (R rows per CTA).
// A thread holds 2^RB residues. With RB = 4 and M = 128 or 256 that is two register blocks, so a residue
// makes one trip through shared memory between its global load and its store (two in a row pass, whose
// other side is a transposition that keeps the global access coalesced), where radix-8 tiles filled from
// and drained to shared memory made four; the T = M / 2^RB threads of one row of PASS 1 lie inside a warp,
// so its exchanges need no CTA barrier.
//   shared memory: PASS 0 element x of column c at x R + c (plus R per 2^RB elements when R < 16, which
//   puts the two element runs a half-warp reads on different banks); PASS 1 element x of a row at
//   x + x / 16, the rows M + M / 16 apart (stride-16 reads hit 16 different bank pairs).
//   twiddles: PASS 0 the column table (equal for all columns: broadcast loads); PASS 1 with RB = 4 the
//   table laid out so that the threads of a row read consecutive entries (see Ctx::d_tw2), RB = 3 the
//   natural table. A row pass's twiddles are as many words as its data, so a CTA takes `per_cta`
//   consecutive rows of the launch at the same tile and finds them in L1 when the rows share a prime.
// What bounds it: the 32-bit multiply pipe (ntt_core.cuh) and, in passes whose loads convert, the latency
// of their loads. Plain forward + inverse transform of 256 rows, N = 2^15 / 2^16 (ms): radix-8 tiles filled
// from shared memory with Shoup products 0.205 / 0.424, the same with split products 0.176 / 0.372,
// these passes 0.141 / 0.305; ModUp conversion pass set of 64 top-level inputs 1.032 / 4.66 -> 0.717 / 3.00, and
// 0.590 / 2.60 with the loads of several residues issued before the first store.
template <class ROWS, int LOGN, int LOGM, int R, bool INV, int PASS, int LOAD, int STORE, int RB, int MINB>
__global__ void __launch_bounds__(R * (1 << LOGM) / (1 << RB), MINB)
pass_kernel(ROWS rows, int n_rows, int per_cta, const Prime* __restrict__ primes, const ulonglong2* __restrict__ tw,
            const u64* __restrict__ ninv, CombineArgs ca) {
    constexpr int M = 1 << LOGM, V = 1 << RB, T = M >> RB, NB = (LOGM + RB - 1) / RB;
    constexpr int LOGN2 = PASS == 0 ? LOGN - LOGM : LOGM;
    constexpr int S1 = LOGN - LOGN2;
    extern __shared__ u64 sm_all[];
    const int lane_q = PASS == 0 ? threadIdx.x % R : threadIdx.x / T;  // column or row of the tile
    const int g = PASS == 0 ? threadIdx.x / R : threadIdx.x % T;       // thread within the sub-transform
    const int t0 = blockIdx.y * R + lane_q;                            // column or row of the ring
    u64* const sm = PASS == 0 ? sm_all + lane_q : sm_all + lane_q * (M + M / 16);
    auto at = [&](int x) -> u64& { return PASS == 0 ? sm[x * R + (R < 16 ? (x >> RB) * R : 0)] : sm[x + (x >> 4)]; };
    auto sync = [&] {
        if (PASS == 0) __syncthreads();
        else __syncwarp();
    };
    auto addr = [&](int x) -> size_t { return PASS == 0 ? (size_t)t0 + ((size_t)x << LOGN2) : ((size_t)t0 << LOGM) + x; };
    const int i1 = min(n_rows, (int)(blockIdx.x + 1) * per_cta);
    for (int i = blockIdx.x * per_cta; i < i1; i++) {
        const KsRow r = rows.get(i, LOGN);
        const Prime& P = primes[r.prime];
        const ulonglong2* const W = tw + ((size_t)r.prime << LOGN) + (PASS == 1 && RB == 4 ? (size_t)t0 << LOGM : 0);
        // register u holds element g + T u before block 0 and outside the blocks of a row pass (arrangement
        // -1), block_elem(k, g, u) in block k
        auto elem = [&](int blk, int u) { return blk < 0 ? g + T * u : nttc::block_elem<LOGM, RB>(blk, g, u); };
        auto load_addr = [&](int u) { return addr(INV && PASS == 0 ? elem(NB - 1, u) : g + T * u); };
        u64 v[V];
        nttc::with_arith<!INV && RB == 4>(P, [&](auto ar) {
            constexpr int AR = decltype(ar)::value;
            const nttc::Mod<AR> m(P);
            auto put = [&](int blk) {
#pragma unroll
                for (int u = 0; u < V; u++) at(elem(blk, u)) = v[u];
            };
            auto take = [&](int blk) {
#pragma unroll
                for (int u = 0; u < V; u++) v[u] = at(elem(blk, u));
            };
            auto exchange = [&](int from, int to) {
                put(from);
                sync();
                take(to);
                sync();
            };
            auto block = [&](auto tag) {
                constexpr int BLK = decltype(tag)::value, S0 = RB * BLK;
                const int tb = nttc::block_elem<LOGM, RB>(BLK, g, 0) >> (LOGM - S0);
                nttc::block_stages<LOGM, RB, BLK, INV, PASS == 0 || BLK != NB - 1>(v, m, [&](int s, int k) {
                    const int grp = (tb << (s - S0)) + k;
                    if (PASS == 0) return W[(1 << s) + grp];
                    if (RB == 4) return W[(1 << s) + (BLK == 0 ? grp : k * T + g)];
                    return W[(1 << (S1 + s)) + (t0 << s) + grp];
                });
            };
            // loads and stores with arithmetic of their own run in short loops over the thread's own
            // shared-memory elements: unrolled over the registers they overflow the instruction cache
            const RowConst rc = row_const<LOAD>(r, primes);
            if constexpr (LOAD == LD_CONV) {
                with_count(r.src_cnt, [&](auto cnt) {
                    conv_rows<AR, decltype(cnt)::value, V>(
                        r, LOGN, m, rc, [&](int u) { return addr(g + T * u); }, [&](int u) -> u64& { return at(g + T * u); });
                });
                take(-1);
            } else {
#pragma unroll
                for (int u = 0; u < V; u++)
                    v[u] = load_elem<LOAD>(r, load_raw<LOAD>(r, load_addr(u), LOGN), load_addr(u), P, m, rc);
                if (LOAD == LD_GATHER && r.out2) {
#pragma unroll
                    for (int u = 0; u < V; u++) r.out2[addr(g + T * u)] = r.pack ? key_pack(v[u]) : v[u];
                }
            }
            if constexpr (!INV) {
                block(nttc::Tag<0>{});
                if constexpr (NB > 1) {
                    exchange(0, 1);
                    block(nttc::Tag<1>{});
                }
                if constexpr (NB > 2) {
                    exchange(1, 2);
                    block(nttc::Tag<2>{});
                }
            } else {
                if (PASS == 1) exchange(-1, NB - 1);
                if constexpr (NB > 2) {
                    block(nttc::Tag<2>{});
                    exchange(2, 1);
                }
                if constexpr (NB > 1) {
                    block(nttc::Tag<1>{});
                    exchange(1, 0);
                }
                block(nttc::Tag<0>{});
            }
            if (!INV && PASS == 1) {
                put(NB - 1);
                sync();
                constexpr int G = STORE == ST_COMBINE || STORE == ST_RESCALE ? 4 : 8;
                for (int u0 = 0; u0 < V; u0 += G) {
                    StoreIn in[G];
#pragma unroll
                    for (int u = 0; u < G; u++) in[u] = store_operands<STORE>(r, addr(g + T * (u0 + u)), ca, LOGN);
#pragma unroll
                    for (int u = 0; u < G; u++)
                        store_elem<INV, STORE>(r, addr(g + T * (u0 + u)), at(g + T * (u0 + u)), in[u], P, m, ninv, ca, LOGN);
                }
                sync();
            } else {
#pragma unroll
                for (int u = 0; u < V; u++)
                    store_elem<INV, STORE>(r, addr(!INV ? elem(NB - 1, u) : g + T * u), v[u], StoreIn{}, P, m, ninv, ca, LOGN);
            }
        });
    }
}

template <class ROWS, int LOGN, int LOGM, int R, bool INV, int PASS, int LOAD, int STORE, int RB, int TPS>
void launch_pass(const Ctx& c, const ROWS& rows, int n_rows, const CombineArgs& ca, int cls, double bytes, cudaStream_t s) {
    constexpr int M = 1 << LOGM, threads = R * M / (1 << RB), tiles = (1 << LOGN) / M / R;
    constexpr int MINB = TPS / threads > 0 ? TPS / threads : 1;
    constexpr size_t smem = sizeof(u64) * (PASS == 0 ? R * (M + (R < 16 ? M >> RB : 0)) : R * (M + M / 16));
    const ulonglong2* tw = PASS == 1 && RB == 4 ? (INV ? c.d_itw2 : c.d_tw2) : (INV ? c.d_itw : c.d_tw);
    auto kernel = pass_kernel<ROWS, LOGN, LOGM, R, INV, PASS, LOAD, STORE, RB, MINB>;
    if (smem > 48 * 1024) CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int per_cta = PASS == 1 ? rules::rows_per_cta(c.n_sm, MINB, n_rows, tiles) : 1;
    LaunchScope _ls(c.prof, cls, bytes, s, (double)n_rows * ((size_t)1 << (c.log_n - 1)) * LOGM);
    kernel<<<dim3((n_rows + per_cta - 1) / per_cta, tiles), threads, smem, s>>>(rows, n_rows, per_cta, c.d_primes, tw,
                                                                             c.d_ninv, ca);
    CK(cudaGetLastError());
}

template <class ROWS, int LOGN, bool INV, int LOAD, int STORE>
void launch_single(const Ctx& c, const ROWS& rows, int n_rows, const CombineArgs& ca, int cls, double bytes, cudaStream_t s) {
    constexpr size_t smem = sizeof(u64) << LOGN;
    auto kernel = single_pass_kernel<ROWS, LOGN, INV, LOAD, STORE>;
    if (smem > 48 * 1024) CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    LaunchScope _ls(c.prof, cls, bytes, s, (double)n_rows * ((size_t)1 << (LOGN - 1)) * LOGN);
    kernel<<<n_rows, (1 << LOGN) / 8, smem, s>>>(rows, c.d_primes, INV ? c.d_itw : c.d_tw, c.d_ninv, ca);
    CK(cudaGetLastError());
}

// A full forward (INV = false) or inverse transform over the rows: the first pass applies LOAD, the
// last pass applies STORE (single-pass rings do both in one kernel). The column passes of a ring of 2^15
// have 2^7 points, its row passes 2^8. Rings of 2^13 in two passes: a row spreads over several SMs and the
// kernels are the register-direct ones. The shapes R = 16 with RB = 4 hold the single-pass kernels; rings of 2^12
// and 2^13 are otherwise transformed by the small tiles only. TPS: threads per SM the register cap of the
// kernels leaves room for.
template <class ROWS, bool INV, int LOAD, int STORE, int R, int RB, int TPS>
void transform_t(const Ctx& c, const ROWS& rows, int n_rows, const CombineArgs& ca, int cls, double bytes, cudaStream_t s) {
    if (n_rows == 0) return;
    // rows or columns per tile: with 8 residues per thread, 256-point sub-transforms take half as many, so that no CTA
    // has more than 256 threads. The ten rows of a rescale at N = 2^16 were 160 CTAs of 512 threads on 152 SMs: one
    // ciphertext, five 45-bit limbs left, 50.2 us, by rescale_noalloc 55.6; with 320 CTAs of half the size 40.6 and 45.4
    constexpr auto tile = [](int log_m) { return RB == 3 && log_m == 8 ? R / 2 : R; };
    constexpr bool single = R == 16 && RB == 4, small = R == 8 || RB == 3, plain = std::is_same<ROWS, RowBatch>::value;
#define ONE(LG)                                                                                    \
    case LG:                                                                                       \
        if constexpr (single) {                                                                    \
            launch_single<ROWS, LG, INV, LOAD, STORE>(c, rows, n_rows, ca, cls, bytes, s);         \
            return;                                                                                \
        }                                                                                          \
        break;
#define TWO(LG, LC, BUILT)                                                                                       \
    case LG:                                                                                                     \
        if constexpr (BUILT) {                                                                                   \
            constexpr int first = INV ? LG - LC : LC, last = LG - first;                                         \
            launch_pass<ROWS, LG, first, tile(first), INV, INV ? 1 : 0, LOAD, ST_LAZY, RB, TPS>(c, rows, n_rows, ca, cls, bytes, s); \
            launch_pass<ROWS, LG, last, tile(last), INV, INV ? 0 : 1, LD_PLAIN, STORE, RB, TPS>(c, rows, n_rows, ca, cls, bytes, s); \
            return;                                                                                              \
        }                                                                                                        \
        break;
    if (rules::single_pass(c.n_sm, c.log_n, !plain, INV, n_rows)) {
        switch (c.log_n) {
            ONE(9)
            ONE(10)
            ONE(11)
            ONE(12)
        }
    } else {
        switch (c.log_n) {
            TWO(12, 6, small && plain)
            TWO(13, 6, small)
            TWO(14, 7, true)
            TWO(15, 7, true)
            TWO(16, 8, true)
        }
    }
#undef ONE
#undef TWO
    fail(FHE_ERR_INVALID_ARG, "no transform of this ring in this shape");
}

// The tile shapes of the fused passes the autotuner chooses between (family "ks_pass"): rows or
// columns per tile of the two-pass rings, 16 residues per thread under a cap of 64 registers (r8x: 8 rows
// with 80 registers: fewer spills, a quarter fewer threads per SM); every shape computes the same bits.
// The exact rescale of 64 ciphertexts at N = 2^15 / 2^16 (ms): r16 0.306 / 0.969, r8 0.294 / 0.951, r8x
// 0.322 / 1.016 (the loads' latency needs the warps). Each shape's instantiations live in a translation
// unit of their own (ks_pass16.cu, ks_pass8.cu, ks_pass8x.cu).
enum KsTile { KS_R16 = 0, KS_R8, KS_R8X, KS_N_TILES };
extern const char* const kKsTileNames[KS_N_TILES];

#define KS_COMBOS(X)                      \
    X(true, LD_GATHER, ST_SCALE)          \
    X(false, LD_CONV, ST_LAST)            \
    X(false, LD_GATHER, ST_LAST)          \
    X(true, LD_AXPY, ST_SCALE)            \
    X(false, LD_CONV, ST_COMBINE_RS)      \
    X(false, LD_CONV, ST_COMBINE)         \
    X(true, LD_MUL, ST_SCALE)             \
    X(false, LD_CENTRED, ST_RESCALE)

template <bool INV, int LOAD, int STORE>
void ks_transform_r16(const Ctx& c, const KsRow* rows, int n_rows, const CombineArgs& ca, int cls, double bytes,
                      cudaStream_t s);
template <bool INV, int LOAD, int STORE>
void ks_transform_r8(const Ctx& c, const KsRow* rows, int n_rows, const CombineArgs& ca, int cls, double bytes,
                     cudaStream_t s);
template <bool INV, int LOAD, int STORE>
void ks_transform_few(const Ctx& c, const KsRow* rows, int n_rows, const CombineArgs& ca, int cls, double bytes,
                      cudaStream_t s);
template <bool INV, int LOAD, int STORE>
void ks_transform_r8x(const Ctx& c, const KsRow* rows, int n_rows, const CombineArgs& ca, int cls, double bytes,
                      cudaStream_t s);

// A full forward (INV = false) or inverse transform over a row table with the context's tile shape:
// the first pass applies LOAD, the last pass applies STORE (single-pass rings do both in one kernel).
template <bool INV, int LOAD, int STORE>
void ks_transform(const Ctx& c, const KsRow* rows, int n_rows, const CombineArgs& ca, int cls, double bytes,
                  cudaStream_t s) {
    // (rings below 2^14 are not tuned: 2^13 takes the small tiles, for the CTAs)
    if (rules::single_pass(c.n_sm, c.log_n, true, INV, n_rows)) ks_transform_r16<INV, LOAD, STORE>(c, rows, n_rows, ca, cls, bytes, s);
    else if (rules::few_rows(c.n_sm, c.log_n, n_rows)) ks_transform_few<INV, LOAD, STORE>(c, rows, n_rows, ca, cls, bytes, s);
    else if (c.log_n < 14 || c.tune.ks == KS_R8) ks_transform_r8<INV, LOAD, STORE>(c, rows, n_rows, ca, cls, bytes, s);
    else if (c.tune.ks == KS_R8X) ks_transform_r8x<INV, LOAD, STORE>(c, rows, n_rows, ca, cls, bytes, s);
    else ks_transform_r16<INV, LOAD, STORE>(c, rows, n_rows, ca, cls, bytes, s);
}

}  // namespace ksp
}  // namespace fhe
