// Pairs per staged chunk of the per-centre derivative kernels, and the shared memory that takes: host arithmetic on the
// layout of soap_device.cuh.
#pragma once
#include "soap_device.cuh"

namespace soap {

// The largest chunk that still leaves room for all the CTAs per SM that the registers allow (three of 256 threads), else
// two thirds of them, else whatever fits `max_smem` bytes (`extra` bytes follow the usual layout); false if nothing fits.
// Where the slab has room of its own a chunk may hold 96 pairs, so that most centres are staged once for both passes (3000
// atoms of 68 neighbours at (4, 3): 218 -> 193 us).
// CTAs of 128 threads stop at 32 pairs where a pair takes 96 words and more: six larger chunks leave the L1 too little
// for the radial table (64 or more against 32 pairs: 36,000 centres of 18 pairs at (4, 3) 682 -> 658 us, 3000 of 68 at
// (4, 4) 241 -> 224 us, at (2, 8) 327 -> 313 us; (2, 2), 48 words a pair, goes the other way, 83 against 93 us).
inline bool plan_chunk(int S, int n_max, int l_max, bool weighted, int warps, size_t extra, size_t max_smem, int& P_out, size_t& bytes_out) {
    const int ctas = 24 / warps;
    auto bytes_of = [&](int P) { return (size_t)make_layout(S, n_max, l_max, P, warps, weighted).total * 4 + extra; };
    const bool keep = make_layout(S, n_max, l_max, 32, warps, false).keep;
    const int L1 = l_max + 1, pair_words = 4 * ((L1 * L1) | 1) + 2 * n_max * L1;
    const int most = warps == 4 && pair_words >= 96 ? 32 : 32 * warps;
    int P = 4;
    for (int pass = 0; pass < 3; ++pass) {
        const size_t budget = pass == 2 ? max_smem : (size_t)228 * 1024 / (pass == 0 ? ctas : (2 * ctas + 2) / 3) - 1024;
        for (const int candidate : {96, 80, 64, 56, 48, 40, 32, 24, 16, 8, 4}) {
            P = candidate;
            if ((keep ? P <= most && (P != 24 || l_max < 8) : P <= 32 && P != 24) && bytes_of(P) <= budget) break;
        }
        if (P >= (pass == 2 ? 4 : 8) && bytes_of(P) <= budget) break;
    }
    P_out = P; bytes_out = bytes_of(P);
    return bytes_out <= max_smem;
}

}  // namespace soap
