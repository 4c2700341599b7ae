// Finite-lattice series kernel (Sec. 4.1-4.3): parameters and launcher.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cp {

constexpr int kMaxSeries = 128;  // longest series (terms) handled
constexpr int kMaxSeriesRects = 128;  // most rectangles of a band (4 per width)

struct SeriesParams {
    int lattice;  // CP_SQUARE / CP_TRIANGULAR
    int k;        // finite-lattice order: rectangles with k-3 <= r+s <= k, r <= s
    int n;        // terms per series
    int D1;       // coefficients per P~ row (D+1 >= n)
    int P;        // primes
    int Pg;       // primes per group
    int Pp;       // prime lanes per group (>= Pg): ptilde is laid out [P/Pg][n_rects][D1][Pp]
    int n_rects;
    int mmax;     // widest strip, (k-1)/2 when the extra square-lattice term applies
    int add_mu;   // 1: add the mu_{2m} z^{4m-1} terms (square lattice, odd k)
};

// ptilde [P/Pg][n_rects][D1][Pp] (signed representatives; each is replaced by its residue in [0, p)), rects (r, s),
// primes: a prime block per group -> out [3][P][n].  err |= 1 if a P~ lacks constant term 1.
// scratch: series_scratch_words(sp) words, the last P of them zero (left zero).
int launch_flm_series(uint32_t *ptilde, const int2 *rects, const uint32_t *primes, const SeriesParams &sp,
                      uint32_t *scratch, uint32_t *out, int *err, cudaStream_t st);
size_t series_scratch_words(const SeriesParams &sp);

}  // namespace cp
