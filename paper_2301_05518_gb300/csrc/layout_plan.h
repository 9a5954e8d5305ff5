// layout_plan.h -- how the kernels of k_layout.cu split their work.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace tls {

// Work of a CTA of 256 threads that moves vector pairs (k_move_pairs): `rows` canonical rows, each in
// `chunks` chunks of `pairs` vector pairs; consecutive threads take the pairs of a chunk at one site,
// then the next site.
// At most four pairs a chunk: a warp then reads runs of eight sites of eight vectors.  With all
// pairs of a site side by side it touched as many sectors as it has threads, and they had left
// L1 before the next site used the rest of them (pack and unpack of 72 FP32 vectors, 12 x 36 x 36 x
// 24: 1989 us with 36 pairs side by side, 735 with 12, 512 with 8, 494 with 4; 48^3 x 16: 10.6, 3.6,
// 2.5 and 2.2 ms; 24 vectors there 981, 988, 767 and 731 us).  Several rows where one leaves
// threads idle (4 x 48 x 48 x 24, 24 vectors in groups of eight: 211 us with one row, 125 with 16).
struct PairSplit {
    int rows, chunks, pairs;
};

// T pairs of rows of Lx sites, nrow rows a slice.
inline PairSplit pair_split(int T, int Lx, int nrow)
{
    PairSplit p;
    p.chunks = (T + 3) / 4;
    p.pairs = (T + p.chunks - 1) / p.chunks;
    p.rows = std::max(1, std::min(256 / (p.chunks * p.pairs * Lx), nrow));
    return p;
}

// Rows of a CTA that takes short rows of links together (an even number), 0: a row by itself, the
// better form from eight sites up (load and release, us, by itself / together: 2 x 96 x 96 x 96 1676 /
// 998, 4 x 64 x 64 x 64 709 / 576, 6 x 64 x 64 x 48 763 / 699, 8 x 32 x 32 x 32 262 / 266, 16 x 48 x 48 x
// 32 661 / 697) and where few CTAs are left (2 x 8 x 8 x 8 26.6 / 30.5).
inline int ingest_rows(int Lx, int sites, int64_t nrow)
{
    const int rows = sites / Lx & ~1;
    return Lx <= 6 && nrow >= (int64_t)304 * rows ? rows : 0;
}

// Strided subsets of a part of a slice's norm, `split` or one: by the slice alone, since it sets the
// order of the additions.  From 28^3 sites on a thread of `split` CTAs has eight reals or more.
inline int norm_subsets(int64_t slice_sites, int split) { return slice_sites * 6 >= 131072 ? split : 1; }

// Whether the subsets of a part are spread over a cluster: where one CTA per part (16 per slice
// and vector) leaves SMs idle.  The sums are the same either way.
inline bool norm_cluster(int nsl, int nvec) { return (int64_t)nsl * nvec * 16 < 8 * 152; }

}  // namespace tls
