// ntt_tile.cuh — the tile shapes of the plain NTT: the pass kernels of ks_pass.cuh over the regular
// rows of a PolyBatch. See ntt.cu for the decomposition.
#pragma once

#include "ks_pass.cuh"

namespace fhe {
namespace ntt_tile {

template <bool INV, int R, int RB>
void transform(const Ctx& c, const PolyBatch& pb, cudaStream_t s, double bytes) {
    const ksp::CombineArgs none{nullptr, nullptr, nullptr, 0, nullptr};
    ksp::transform_t<ksp::RowBatch, INV, ksp::LD_PLAIN, ksp::ST_LAST, R, RB, 768>(
        c, ksp::RowBatch{pb}, pb.rows(), none, INV ? K_NTT_INV : K_NTT_FWD, bytes, s);
}

// The tile shapes the autotuner chooses between (family "ntt"): rows or columns per tile R and
// residues per thread 2^RB of the two-pass rings; every shape computes the same bits.
enum NttTile { NTT_R16B4 = 0, NTT_R8B4, NTT_R32B4, NTT_R16B3, NTT_N_TILES };
extern const char* const kNttTileNames[NTT_N_TILES];
void transform_r8b4(const Ctx& c, const PolyBatch& pb, bool inv, cudaStream_t s, double bytes);
void transform_r32b4(const Ctx& c, const PolyBatch& pb, bool inv, cudaStream_t s, double bytes);
void transform_r16b3(const Ctx& c, const PolyBatch& pb, bool inv, cudaStream_t s, double bytes);

}  // namespace ntt_tile
}  // namespace fhe
