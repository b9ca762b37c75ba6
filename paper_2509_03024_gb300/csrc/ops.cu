// ops.cu — batched RNS kernels over descriptor tables: element-wise add / sub /
// plaintext product / tensor product, segmented accumulation, integer-to-RNS
// conversion and the evaluation-domain automorphism. (Key switching and the
// rescale run as fused NTT passes in ks.cu.)
//
// Launch shape of the element-wise kernels: blockIdx.y selects the item (a
// table entry), the x dimension walks (component, limb, coefficient pair) with
// one 128-bit access per residue pair. Item tables are uploaded through the
// context's pinned descriptor arena.
#include <algorithm>

#include "ks_inner.cuh"
#include "ntt_core.cuh"

namespace fhe {

// ============================================================================ launch accounting

const char* const kKClassNames[K_COUNT] = {"ntt_forward", "ntt_inverse", "ks_inner", "tensor",
                                           "elementwise", "encode",      "other"};

cudaEvent_t Profiler::get_event() {
    if (pool_used == pool.size()) {
        cudaEvent_t e;
        CK(cudaEventCreate(&e));
        pool.push_back(e);
    }
    return pool[pool_used++];
}

void Profiler::reset() {
    for (int k = 0; k < K_COUNT; k++) {
        launches[k] = 0;
        bytes[k] = 0;
        work[k] = 0;
    }
    recs.clear();
    pool_used = 0;
}

Profiler::~Profiler() {
    for (cudaEvent_t e : pool) cudaEventDestroy(e);
}

thread_local bool tl_no_launch_events = false;

LaunchScope::LaunchScope(Profiler& prof, int k, double nbytes, cudaStream_t st, double work)
    : p(prof), cls(k), s(st) {
    p.launches[k]++;
    p.bytes[k] += nbytes;
    p.work[k] += work;
    if (p.timing && !tl_no_launch_events) {
        b = p.get_event();
        CK(cudaEventRecord(b, s));
    }
}

LaunchScope::~LaunchScope() {
    if (b) {
        cudaEvent_t e = p.get_event();
        cudaEventRecord(e, s);
        p.recs.push_back({cls, b, e});
    }
}

namespace {

constexpr int kThreads = 256;

template <typename T>
T* upload(Ctx& c, const std::vector<T>& v, cudaStream_t s) {
    return c.arena.push_vec(v, s);
}

inline dim3 grid2(size_t per_item, int items) {
    size_t bx = (per_item + kThreads - 1) / kThreads;
    if (bx > 65535u * 16) bx = 65535u * 16;
    return dim3((unsigned)std::max<size_t>(bx, 1), (unsigned)std::min(items, 65535));
}
inline unsigned grid1(size_t work) {
    size_t b = (work + kThreads - 1) / kThreads;
    return (unsigned)std::min<size_t>(std::max<size_t>(b, 1), (size_t)1 << 30);
}

// ---------------------------------------------------------------- element-wise

// For element e of an item: component p, limb i, coefficient pair k2.
struct PIdx {
    int part, limb, k2;
};
__device__ __forceinline__ PIdx pidx(size_t e, int log_half, int limbs) {
    PIdx r;
    r.k2 = (int)(e & ((1u << log_half) - 1));
    size_t row = e >> log_half;
    r.limb = (int)(row % limbs);
    r.part = (int)(row / limbs);
    return r;
}

__device__ __forceinline__ size_t off2(int part, int limb, int log_n, size_t part_words) {
    return (size_t)part * part_words + ((size_t)limb << log_n);
}

#define ITEM_LOOP(items_count)                                                                       \
    for (int it = blockIdx.y; it < (items_count); it += gridDim.y)                                   \
        for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < per;                      \
             e += (size_t)gridDim.x * blockDim.x)

__global__ void add_items_kernel(const BinItem* __restrict__ tab, int items, int parts, int limbs, int log_n,
                                 size_t part_words, const Prime* __restrict__ pr, bool sub) {
    const size_t per = (size_t)parts * limbs << (log_n - 1);
    ITEM_LOOP(items) {
        const BinItem t = tab[it];
        PIdx x = pidx(e, log_n - 1, limbs);
        size_t o = off2(x.part, x.limb, log_n, part_words);
        const u64 q = pr[x.limb].q;
        ulonglong2 va = reinterpret_cast<const ulonglong2*>(t.a + o)[x.k2];
        ulonglong2 vb = reinterpret_cast<const ulonglong2*>(t.b + o)[x.k2];
        ulonglong2 r;
        r.x = sub ? sub_mod(va.x, vb.x, q) : add_mod(va.x, vb.x, q);
        r.y = sub ? sub_mod(va.y, vb.y, q) : add_mod(va.y, vb.y, q);
        reinterpret_cast<ulonglong2*>(t.out + o)[x.k2] = r;
    }
}

__global__ void copy_items_kernel(const UnItem* __restrict__ tab, int items, int parts, int limbs, int log_n,
                                  size_t part_words) {
    const size_t per = (size_t)parts * limbs << (log_n - 1);
    ITEM_LOOP(items) {
        const UnItem t = tab[it];
        PIdx x = pidx(e, log_n - 1, limbs);
        size_t o = off2(x.part, x.limb, log_n, part_words);
        reinterpret_cast<ulonglong2*>(t.out + o)[x.k2] = reinterpret_cast<const ulonglong2*>(t.in + o)[x.k2];
    }
}

// Products of two residues modulo near 50-bit primes go to column sums (Products in ntt_core.cuh); N50 = false is
// the kernel of launches whose primes are all others. With the column sums' code beside it the Barrett form needs 80
// to 128 registers instead of 60 to 78: the tensor of 64 ciphertexts at N = 2^14, four 45-bit limbs, 65 us alone, 69 so;
// 64 plaintext products 66 and 69.
template <bool N50, class F>
__device__ __forceinline__ void with_products(const Prime& P, F&& f) {
    if (N50 && P.cls == nttc::AR_NEAR50) f(nttc::Tag<nttc::AR_NEAR50>{});
    else f(nttc::Tag<nttc::AR_SHOUP>{});
}
inline bool any_near50(const Ctx& c, int limbs) {
    for (int i = 0; i < limbs; i++)
        if (c.hprimes[i].cls == nttc::AR_NEAR50) return true;
    return false;
}

template <bool N50>
__global__ void mul_plain_items_kernel(const BinItem* __restrict__ tab, int items, int parts, int limbs,
                                       int log_n, size_t part_words, const Prime* __restrict__ pr) {
    const size_t per = (size_t)parts * limbs << (log_n - 1);
    ITEM_LOOP(items) {
        const BinItem t = tab[it];
        PIdx x = pidx(e, log_n - 1, limbs);
        size_t o = off2(x.part, x.limb, log_n, part_words);
        const Prime P = pr[x.limb];
        ulonglong2 va = reinterpret_cast<const ulonglong2*>(t.a + o)[x.k2];
        ulonglong2 vb = reinterpret_cast<const ulonglong2*>(t.b + ((size_t)x.limb << log_n))[x.k2];
        with_products<N50>(P, [&](auto ar) {
            const nttc::Mod<decltype(ar)::value> m(P);
            reinterpret_cast<ulonglong2*>(t.out + o)[x.k2] =
                make_ulonglong2(nttc::product(va.x, vb.x, m, P), nttc::product(va.y, vb.y, m, P));
        });
    }
}

__device__ __forceinline__ u64 signed_mod_q(long long v, u64 q) {
    if (v >= 0) return (u64)v % q;
    u64 m = (u64)(-(v + 1)) % q;
    return q - 1 - m;
}

__global__ void mul_const_items_kernel(const ConstItem* __restrict__ tab, int items, int parts, int limbs,
                                       int log_n, size_t part_words, const Prime* __restrict__ pr) {
    const size_t per = (size_t)parts * limbs << (log_n - 1);
    ITEM_LOOP(items) {
        const ConstItem t = tab[it];
        PIdx x = pidx(e, log_n - 1, limbs);
        size_t o = off2(x.part, x.limb, log_n, part_words);
        const Prime P = pr[x.limb];
        const u64 cv = signed_mod_q(t.value, P.q);
        ulonglong2 va = reinterpret_cast<const ulonglong2*>(t.in + o)[x.k2];
        ulonglong2 r;
        r.x = mul_mod(va.x, cv, P);
        r.y = mul_mod(va.y, cv, P);
        reinterpret_cast<ulonglong2*>(t.out + o)[x.k2] = r;
    }
}

// The three components of a (x) b at one slot pair, summed over several a, b before one reduction.
template <int AR>
struct TensorSum {
    nttc::Products<AR> x[3], y[3];
    template <bool START>
    __device__ __forceinline__ static void enter(nttc::Products<AR>& s, u64 a, u64 b, const Prime& P) {
        if (START) s.start(a, b, P);
        else s.add(a, b, P);
    }
    template <bool START>
    __device__ __forceinline__ void add(const u64* a, const u64* b, size_t o, size_t pw, int k2, const Prime& P) {
        const ulonglong2 a0 = reinterpret_cast<const ulonglong2*>(a + o)[k2];
        const ulonglong2 a1 = reinterpret_cast<const ulonglong2*>(a + pw + o)[k2];
        const ulonglong2 b0 = reinterpret_cast<const ulonglong2*>(b + o)[k2];
        const ulonglong2 b1 = reinterpret_cast<const ulonglong2*>(b + pw + o)[k2];
        enter<START>(x[0], a0.x, b0.x, P);
        enter<START>(y[0], a0.y, b0.y, P);
        enter<START>(x[1], a0.x, b1.x, P);
        x[1].add(a1.x, b0.x, P);
        enter<START>(y[1], a0.y, b1.y, P);
        y[1].add(a1.y, b0.y, P);
        enter<START>(x[2], a1.x, b1.x, P);
        enter<START>(y[2], a1.y, b1.y, P);
    }
    __device__ __forceinline__ void add_stored(const u64* out, size_t o, size_t pw, int k2, const Prime& P) {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const ulonglong2 v = reinterpret_cast<const ulonglong2*>(out + i * pw + o)[k2];
            x[i].add_residue(v.x, P);
            y[i].add_residue(v.y, P);
        }
    }
    __device__ __forceinline__ void store(u64* out, size_t o, size_t pw, int k2, const nttc::Mod<AR>& m, const Prime& P) const {
#pragma unroll
        for (int i = 0; i < 3; i++)
            reinterpret_cast<ulonglong2*>(out + i * pw + o)[k2] = make_ulonglong2(x[i].reduce(m, P), y[i].reduce(m, P));
    }
};

template <bool N50>
__global__ void tensor_items_kernel(const BinItem* __restrict__ tab, int items, int limbs, int log_n,
                                    size_t pw, const Prime* __restrict__ pr) {
    const size_t per = (size_t)limbs << (log_n - 1);
    ITEM_LOOP(items) {
        const BinItem t = tab[it];
        PIdx x = pidx(e, log_n - 1, limbs);
        size_t o = (size_t)x.limb << log_n;
        const Prime P = pr[x.limb];
        with_products<N50>(P, [&](auto ar) {
            constexpr int AR = decltype(ar)::value;
            TensorSum<AR> s;
            s.template add<true>(t.a, t.b, o, pw, x.k2, P);
            s.store(t.out, o, pw, x.k2, nttc::Mod<AR>(P), P);
        });
    }
}

template <bool N50>
__global__ void __launch_bounds__(kThreads, N50 ? 2 : 3) tensor_acc_kernel(const AccTarget* __restrict__ tg, const BinItem* __restrict__ cb, int targets,
                                  int limbs, int log_n, size_t pw, const Prime* __restrict__ pr) {
    const size_t per = (size_t)limbs << (log_n - 1);
    ITEM_LOOP(targets) {
        const AccTarget t = tg[it];
        PIdx x = pidx(e, log_n - 1, limbs);
        size_t o = (size_t)x.limb << log_n;
        const Prime& P = pr[x.limb];
        with_products<N50>(P, [&](auto ar) {
            constexpr int AR = decltype(ar)::value;
            const nttc::Mod<AR> m(P);
            // two products per contributor enter the middle component, and the stored value counts as one
            constexpr int kBatch = nttc::Products<AR>::kTerms / 2 - 1;
            for (int j0 = 0; j0 < t.cnt; j0 += kBatch) {
                TensorSum<AR> s;
                s.add_stored(t.out, o, pw, x.k2, P);
                for (int j = j0; j < min(j0 + kBatch, t.cnt); j++) s.template add<false>(cb[t.off + j].a, cb[t.off + j].b, o, pw, x.k2, P);
                s.store(t.out, o, pw, x.k2, m, P);
            }
        });
    }
}

__global__ void sum_acc_kernel(const AccTarget* __restrict__ tg, const BinItem* __restrict__ cb, int targets,
                               int parts, int limbs, int log_n, size_t pw, const Prime* __restrict__ pr) {
    const size_t per = (size_t)parts * limbs << (log_n - 1);
    ITEM_LOOP(targets) {
        const AccTarget t = tg[it];
        PIdx x = pidx(e, log_n - 1, limbs);
        size_t o = off2(x.part, x.limb, log_n, pw);
        const u64 q = pr[x.limb].q;
        ulonglong2 s = reinterpret_cast<const ulonglong2*>(t.out + o)[x.k2];
        for (int j = 0; j < t.cnt; j++) {
            ulonglong2 v = reinterpret_cast<const ulonglong2*>(cb[t.off + j].a + o)[x.k2];
            s.x = add_mod(s.x, v.x, q);
            s.y = add_mod(s.y, v.y, q);
        }
        reinterpret_cast<ulonglong2*>(t.out + o)[x.k2] = s;
    }
}

__global__ void int_to_rns_kernel(u64* out, size_t out_stride, const i64* __restrict__ in, size_t in_stride,
                                  int items, int limbs, int log_n, const Prime* __restrict__ pr) {
    const size_t total = (size_t)items * limbs << log_n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        int k = (int)(e & ((1u << log_n) - 1));
        size_t row = e >> log_n;
        int limb = (int)(row % limbs);
        int item = (int)(row / limbs);
        out[(size_t)item * out_stride + ((size_t)limb << log_n) + k] =
            nttc::signed_residue(in[(size_t)item * in_stride + k], pr[limb]);
    }
}

__global__ void int8_to_rns_kernel(u64* out, size_t out_stride, const int8_t* __restrict__ in, size_t in_stride,
                                   int items, int limbs, int log_n, int split, int jump,
                                   const Prime* __restrict__ pr) {
    const size_t total = (size_t)items * limbs << log_n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        int k = (int)(e & ((1u << log_n) - 1));
        size_t row = e >> log_n;
        int limb = (int)(row % limbs);
        int item = (int)(row / limbs);
        int prime = limb + (limb >= split ? jump : 0);
        int v = in[(size_t)item * in_stride + k];
        u64 q = pr[prime].q;
        out[(size_t)item * out_stride + ((size_t)limb << log_n) + k] = v >= 0 ? (u64)v : q - (u64)(-v);
    }
}

__global__ void automorphism_kernel(u64* out, const u64* __restrict__ in, int limbs, int log_n, int g) {
    const size_t total = (size_t)limbs << log_n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        int k = (int)(e & ((1u << log_n) - 1));
        size_t row = e >> log_n;
        out[e] = in[(row << log_n) + auto_src(k, g, log_n)];
    }
}

}  // namespace

// ============================================================================ launchers

void items_add(Ctx& c, const std::vector<BinItem>& it, int parts, int limbs, bool sub, cudaStream_t s) {
    if (it.empty()) return;
    const BinItem* d = upload(c, it, s);
    size_t per = (size_t)parts * limbs * c.n / 2;
    {
        LaunchScope _ls(c.prof, K_ELEMENTWISE, 3.0 * 8 * per * 2 * it.size(), s);
        add_items_kernel<<<grid2(per, (int)it.size()), kThreads, 0, s>>>(d, (int)it.size(), parts, limbs, c.log_n,
                                                                     (size_t)(c.L + 1) * c.n, c.d_primes, sub);
    CK(cudaGetLastError());
    }
}

void items_copy(Ctx& c, const std::vector<UnItem>& it, int parts, int limbs, cudaStream_t s) {
    if (it.empty()) return;
    const UnItem* d = upload(c, it, s);
    size_t per = (size_t)parts * limbs * c.n / 2;
    {
        LaunchScope _ls(c.prof, K_ELEMENTWISE, 2.0 * 8 * per * 2 * it.size(), s);
        copy_items_kernel<<<grid2(per, (int)it.size()), kThreads, 0, s>>>(d, (int)it.size(), parts, limbs, c.log_n,
                                                                      (size_t)(c.L + 1) * c.n);
    CK(cudaGetLastError());
    }
}

void items_mul_plain(Ctx& c, const std::vector<BinItem>& it, int parts, int limbs, cudaStream_t s) {
    if (it.empty()) return;
    const BinItem* d = upload(c, it, s);
    size_t per = (size_t)parts * limbs * c.n / 2;
    {
        LaunchScope _ls(c.prof, K_ELEMENTWISE, 2.5 * 8 * per * 2 * it.size(), s);
        auto kernel = any_near50(c, limbs) ? mul_plain_items_kernel<true> : mul_plain_items_kernel<false>;
        kernel<<<grid2(per, (int)it.size()), kThreads, 0, s>>>(d, (int)it.size(), parts, limbs,
                                                                           c.log_n, (size_t)(c.L + 1) * c.n,
                                                                           c.d_primes);
    CK(cudaGetLastError());
    }
}

void items_mul_const(Ctx& c, const std::vector<ConstItem>& it, int parts, int limbs, cudaStream_t s) {
    if (it.empty()) return;
    const ConstItem* d = upload(c, it, s);
    size_t per = (size_t)parts * limbs * c.n / 2;
    {
        LaunchScope _ls(c.prof, K_ELEMENTWISE, 2.0 * 8 * per * 2 * it.size(), s);
        mul_const_items_kernel<<<grid2(per, (int)it.size()), kThreads, 0, s>>>(d, (int)it.size(), parts, limbs, c.log_n,
                                                                              (size_t)(c.L + 1) * c.n, c.d_primes);
        CK(cudaGetLastError());
    }
}

void items_tensor(Ctx& c, const std::vector<BinItem>& it, int limbs, cudaStream_t s) {
    if (it.empty()) return;
    const BinItem* d = upload(c, it, s);
    size_t per = (size_t)limbs * c.n / 2;
    {
        LaunchScope _ls(c.prof, K_TENSOR, 7.0 * 8 * per * 2 * it.size(), s);
        auto kernel = any_near50(c, limbs) ? tensor_items_kernel<true> : tensor_items_kernel<false>;
        kernel<<<grid2(per, (int)it.size()), kThreads, 0, s>>>(d, (int)it.size(), limbs, c.log_n,
                                                                        (size_t)(c.L + 1) * c.n, c.d_primes);
    CK(cudaGetLastError());
    }
}

void items_tensor_acc(Ctx& c, const std::vector<AccTarget>& tg, const std::vector<BinItem>& contrib, int limbs,
                      cudaStream_t s) {
    if (tg.empty()) return;
    ArenaGather tables(c.arena);
    const AccTarget* dt = upload(c, tg, s);
    const BinItem* dc = upload(c, contrib, s);
    tables.upload(s);
    size_t per = (size_t)limbs * c.n / 2;
    {
        LaunchScope _ls(c.prof, K_TENSOR, 8.0 * per * 2 * (4.0 * contrib.size() + 6.0 * tg.size()), s);
        auto kernel = any_near50(c, limbs) ? tensor_acc_kernel<true> : tensor_acc_kernel<false>;
        kernel<<<grid2(per, (int)tg.size()), kThreads, 0, s>>>(dt, dc, (int)tg.size(), limbs, c.log_n,
                                                                      (size_t)(c.L + 1) * c.n, c.d_primes);
    CK(cudaGetLastError());
    }
}

void items_sum_acc(Ctx& c, const std::vector<AccTarget>& tg, const std::vector<BinItem>& contrib, int parts,
                   int limbs, cudaStream_t s) {
    if (tg.empty()) return;
    ArenaGather tables(c.arena);
    const AccTarget* dt = upload(c, tg, s);
    const BinItem* dc = upload(c, contrib, s);
    tables.upload(s);
    size_t per = (size_t)parts * limbs * c.n / 2;
    {
        LaunchScope _ls(c.prof, K_ELEMENTWISE, 8.0 * per * 2 * (contrib.size() + 2.0 * tg.size()), s);
        sum_acc_kernel<<<grid2(per, (int)tg.size()), kThreads, 0, s>>>(dt, dc, (int)tg.size(), parts, limbs, c.log_n,
                                                                   (size_t)(c.L + 1) * c.n, c.d_primes);
    CK(cudaGetLastError());
    }
}

void k_int_to_rns(const Ctx& c, u64* out, size_t out_item_stride, const i64* in, size_t in_stride, int items,
                  int limbs, cudaStream_t s) {
    size_t work = (size_t)items * limbs * c.n;
    if (!work) return;
    {
        LaunchScope _ls(c.prof, K_ELEMENTWISE, 8.0 * items * c.n + 8.0 * work, s);
        int_to_rns_kernel<<<grid1(work), kThreads, 0, s>>>(out, out_item_stride, in, in_stride, items, limbs, c.log_n,
                                                       c.d_primes);
    CK(cudaGetLastError());
    }
}

void k_int8_to_rns(const Ctx& c, u64* out, size_t out_item_stride, const int8_t* in, size_t in_stride, int items,
                   int limbs, int prime_split, int prime_jump, cudaStream_t s) {
    size_t work = (size_t)items * limbs * c.n;
    if (!work) return;
    {
        LaunchScope _ls(c.prof, K_ELEMENTWISE, 1.0 * items * c.n + 8.0 * work, s);
        int8_to_rns_kernel<<<grid1(work), kThreads, 0, s>>>(out, out_item_stride, in, in_stride, items, limbs, c.log_n,
                                                        prime_split, prime_jump, c.d_primes);
    CK(cudaGetLastError());
    }
}

void k_automorphism_poly(const Ctx& c, u64* out, const u64* in, int limbs, int galois, cudaStream_t s) {
    {
        LaunchScope _ls(c.prof, K_OTHER, 16.0 * limbs * c.n, s);
        automorphism_kernel<<<grid1((size_t)limbs * c.n), kThreads, 0, s>>>(out, in, limbs, c.log_n, galois);
    CK(cudaGetLastError());
    }
}

}  // namespace fhe
