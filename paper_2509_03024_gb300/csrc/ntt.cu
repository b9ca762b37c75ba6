// ntt.cu — batched negacyclic NTT over RNS limbs.
//
// Forward: Cooley-Tukey with merged psi powers (natural order in, bit-reversed
// order out): slot k holds a(psi^(2 brev(k) + 1)). Inverse: Gentleman-Sande
// (bit-reversed in, natural out) followed by the N^-1 scaling.
//
// Decomposition. A ring of N = N1 * N2 coefficients is viewed as N1 rows of
// N2: the first log2(N1) stages couple elements N2 apart (independent
// N1-point transforms on columns), the remaining stages couple elements inside
// one row (N2-point transforms with row-dependent twiddles). Rings up to 2^11
// run in one pass (one CTA per limb), rings from 2^13 on in two passes, one kernel each
// (pass_kernel in ks_pass.cuh), 2^12 in either (rules::single_pass). Values stay unreduced between stages
// wherever 64 bits allow it (ntt_core.cuh); the last pass reduces to [0, q).
#include "ntt_tile.cuh"

namespace fhe {

namespace ntt_tile {
const char* const kNttTileNames[NTT_N_TILES] = {"r16b4", "r8b4", "r32b4", "r16b3"};
}

namespace {

using namespace ntt_tile;

template <bool INV>
void run_ntt(const Ctx& c, const PolyBatch& pb, cudaStream_t s) {
    const double bytes = 16.0 * pb.rows() * ((size_t)1 << c.log_n);
    const int shape = rules::single_pass(c.n_sm, c.log_n, false, INV, pb.rows()) ? NTT_R16B4
                      : rules::few_rows(c.n_sm, c.log_n, pb.rows())              ? NTT_R16B3
                      : c.log_n < 14                                            ? NTT_R8B4
                                                                                : c.tune.ntt;
    switch (shape) {
        case NTT_R8B4: transform_r8b4(c, pb, INV, s, bytes); return;
        case NTT_R32B4: transform_r32b4(c, pb, INV, s, bytes); return;
        case NTT_R16B3: transform_r16b3(c, pb, INV, s, bytes); return;
        default: transform<INV, 16, 4>(c, pb, s, bytes); return;
    }
}

}  // namespace

void ntt_forward(const Ctx& c, const PolyBatch& pb, cudaStream_t s) { run_ntt<false>(c, pb, s); }
void ntt_inverse(const Ctx& c, const PolyBatch& pb, cudaStream_t s) { run_ntt<true>(c, pb, s); }

}  // namespace fhe
