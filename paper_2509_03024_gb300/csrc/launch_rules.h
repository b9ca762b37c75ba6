// launch_rules.h — the lines between launch shapes of the transforms, as functions of the ring, the rows of the
// launch and the GPU's SM count (Ctx::n_sm). Host code only.
#pragma once

#include <stddef.h>

#include <algorithm>

namespace fhe {
namespace rules {

// One pass (a CTA holds the whole row in shared memory) or two. Rings up to 2^11 take one, from 2^13 on two (at
// 2^13, 2048 rows: 323 us in one, 215 in two; two are ahead from the first row on). In between, at 2^12:
//   fused passes (key switches, rescales) one: a second pass costs every stored row another trip and every
//     conversion its own launch. 256 rotations of four 40-bit limbs 516 us in two, 496 in one; 64 rescales 58, 48;
//     one product 60 against 70 (50-bit limbs); 512 products of 60-bit limbs are the one place where two win, by 3 %
//   plain transforms (us, forward / inverse of 40-bit rows, reduced in every stage, in two : in one): 32 rows 8 : 10 / 8 : 10, 64 rows
//     11 : 10 / 12 : 10, 512 rows 31 : 28 / 34 : 31, 768 rows 37 : 39 / 43 : 43, 8192 rows 319 : 328 / 353 : 351.
//     Two up to a third of a row per SM, where one pass leaves most SMs idle, and in forward transforms of more
//     than four rows per SM, where the two passes' smaller tiles keep more warps in flight.
inline bool single_pass(int n_sm, int log_n, bool fused, bool inverse, size_t n_rows) {
    if (log_n != 12 || fused) return log_n <= 12;
    return 3 * n_rows > (size_t)n_sm && (inverse || n_rows <= 4 * (size_t)n_sm);
}

// Launches of few rows leave an SM with a handful of warps, each a serial chain of 16-residue register
// blocks; with 8 residues per thread (ks_pass_few.cu, 16 rows or columns per tile, 8 of 256 points) the chain is half as long and
// the warps twice as many. The line: less than 16 warps per SM at 16 residues per thread. One rotation at N = 2^16 with
// it and with one table upload per key switch 214 -> 170 us, one product at N = 2^13 111 -> 72 us.
inline bool few_rows(int n_sm, int log_n, size_t n_rows) { return (n_rows << (log_n - 4)) < (size_t)n_sm * 512; }

// A row pass takes several rows per CTA (they share its twiddles in L1) while at least eight waves of CTAs remain.
inline int rows_per_cta(int n_sm, int ctas_per_sm, size_t n_rows, size_t tiles) {
    return (int)std::min<size_t>(4, std::max<size_t>(1, n_rows * tiles / ((size_t)n_sm * ctas_per_sm * 8)));
}

}  // namespace rules
}  // namespace fhe
