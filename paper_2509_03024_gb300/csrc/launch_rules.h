// launch_rules.h — the lines between launch shapes of the transforms, as functions of the ring, the rows of the
// launch and the GPU's SM count (Ctx::n_sm). Host code only.
#pragma once

#include <stddef.h>

#include <algorithm>

namespace fhe {
namespace rules {

// Launches of few rows leave an SM with a handful of warps, each a serial chain of 16-residue register
// blocks; with 8 residues per thread (ks_pass_few.cu, 16 rows or columns per tile) the chain is half as long and
// the warps twice as many. The line: less than 16 warps per SM at 16 residues per thread. One rotation at N = 2^16 with
// it and with one table upload per key switch 214 -> 170 us, one product at N = 2^13 111 -> 72 us.
inline bool few_rows(int n_sm, int log_n, size_t n_rows) { return (n_rows << (log_n - 4)) < (size_t)n_sm * 512; }

// A row pass takes several rows per CTA (they share its twiddles in L1) while at least eight waves of CTAs remain.
inline int rows_per_cta(int n_sm, int ctas_per_sm, size_t n_rows, size_t tiles) {
    return (int)std::min<size_t>(4, std::max<size_t>(1, n_rows * tiles / ((size_t)n_sm * ctas_per_sm * 8)));
}

}  // namespace rules
}  // namespace fhe
