// ntt_tiles.cu — the alternative tile shapes of the plain two-pass NTT (see ntt_tile.cuh), compiled in
// a translation unit of their own so that the library builds in parallel.
#include "ntt_tile.cuh"

namespace fhe {
namespace ntt_tile {

void transform_r8b4(const Ctx& c, const PolyBatch& pb, bool inv, cudaStream_t s, double bytes) {
    if (inv) transform<true, 8, 4>(c, pb, s, bytes);
    else transform<false, 8, 4>(c, pb, s, bytes);
}
void transform_r32b4(const Ctx& c, const PolyBatch& pb, bool inv, cudaStream_t s, double bytes) {
    if (inv) transform<true, 32, 4>(c, pb, s, bytes);
    else transform<false, 32, 4>(c, pb, s, bytes);
}
void transform_r16b3(const Ctx& c, const PolyBatch& pb, bool inv, cudaStream_t s, double bytes) {
    if (inv) transform<true, 16, 3>(c, pb, s, bytes);
    else transform<false, 16, 3>(c, pb, s, bytes);
}

}  // namespace ntt_tile
}  // namespace fhe
