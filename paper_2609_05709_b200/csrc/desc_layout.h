// Layout of the descriptor-only kernel (desc_kernel.cuh) and how a call is spread over it: host and device arithmetic.
#pragma once
#include <algorithm>

#include "soap_device.cuh"

namespace soap {

constexpr int kDescGroup = 64;                    // pairs whose geometry a warp holds in registers (two per lane)
constexpr int kDescMaxWarps = 16;                 // warps per CTA (one CTA per SM)
constexpr int kDescTeamWarps = 4;                 // most warps of a CTA that works on one centre
// atoms of a warp's share of such a search, and the bytes behind the layout: a slot per atom, and what each warp found
__host__ __device__ inline int desc_search_share(long long n_atoms, int warps) { return (int)((n_atoms + 32 * warps - 1) / (32 * warps)) * 32; }
__host__ __device__ inline size_t desc_search_bytes(long long n_atoms, int warps) { return n_atoms > 0 ? (size_t)desc_search_share(n_atoms, warps) * warps * 8 + kDescTeamWarps * 4 : 0; }

// tiles of four consecutive m of one l: tile index of the first tile of row l, and their number up to l_max
__host__ __device__ constexpr int desc_tile_base(int l) {
    int t = 0;
    for (int k = 0; k < l; ++k) t += (2 * k + 1 + 3) / 4;
    return t;
}
__host__ __device__ constexpr int desc_tiles(int l_max) { return desc_tile_base(l_max + 1); }
// n_max is padded to a multiple of four (NP = 4, 8, 12 or 16 is the template parameter; the padding channels have
// all-zero table rows, so they cost arithmetic but need no special cases)
__host__ __device__ constexpr int desc_np(int n_max) { return (n_max + 3) & ~3; }
// words per pair of the harmonics staging: the tiles, four words each, padded to an odd number of 16-byte chunks so
// that the 16-byte stores of eight lanes (eight pairs) fall into eight different bank groups
__host__ __device__ constexpr int desc_s_row(int l_max) { return 4 * (desc_tiles(l_max) | 1); }
// words per l of the radial staging.  Lanes that own tiles of different l read 16-byte chunks of different rows at
// once, and these must fall into different bank groups: with an odd number of chunks per l they do; with two
// (n_max up to 8) the two chunks of rows l >= 4 are swapped instead; with four the row is padded by one chunk.
__host__ __device__ constexpr int desc_g_l(int np) { return np == 16 ? 20 : np; }
__host__ __device__ constexpr int desc_g_swap(int np, int l) { return np == 8 ? (l >> 2) & 1 : 0; }

// The centre's coefficient tile c[lm][species, n]: S NP / 4 16-byte chunks per row, and with `pad` one more chunk of room
// after every four rows: the lanes of a warp, which own rows four apart, then do not all hit one group of banks when they
// store their sums.  Not in the plain kernel at l_max 8 with n_max 13 to 16, where two species keep eight warps without the
// room and seven with it (9000 atoms at (14, 8) 430 -> 389 us, 30,000 at (16, 8) 1659 -> 1565 us; one, three, four and five
// species, whose warps stay, 0 to 1.4 % faster).  Coefficients, read from the tile row by row, need it (899 centres 46
// against 52 us).  As an option of the launch, wherever the room costs a warp, it took registers from the largest bases ((7,
// 10) on 28,821 atoms 903 -> 988 us).
__host__ __device__ constexpr bool desc_tile_pad(int np, int l_max, bool plain) { return !(plain && np == 16 && l_max == 8); }
__host__ __device__ constexpr int desc_c_at(int row, int row_chunks, bool pad) { return row * row_chunks + (pad ? row >> 2 : 0); }
__host__ __device__ constexpr int desc_c_words(int S, int np, int lm, bool pad) { return 4 * (desc_c_at(lm - 1, S * np / 4, pad) + S * np / 4); }

// How the radial factors of a staged pair are taken from the table.  As quads: four adjacent n of one l per lane, the table as
// [interval][6][l][n], so that lanes side by side read side by side: 24 instructions for four values instead of 40 and no
// conflicts while eight lanes stay within one pair.  They do where 7 or 8 of every 8 lanes have a quad (`desc_quad_span`:
// a lane then keeps its quad), and conflicts weigh little with more than 16 quads; else two adjacent n per lane, the table as
// [interval][l][n / 2][6][2], which fills more lanes.  24,000 atoms of water, whole calls, pairs against quads: (8, 6) 202 ->
// 193 us, (8, 3) 148 -> 144, (14, 6) 714 -> 661, (2, 7) 175 -> 170, (10, 8) 623 -> 608; the other way, left as pairs,
// (8, 4) 164 -> 172, (2, 4) 131 -> 138, (10, 2) 169 -> 179, (8, 5) and (10, 3) equal or slower.  The bases that take quads do so
// with the table in global memory too (weighted, 3000 atoms, (3, 6) 53.6 -> 51.5 us, (8, 6) 65.9 -> 61.7, (14, 6) 122 -> 118) and
// in teams (300 atoms, (8, 6) 13.6 -> 12.4, (9, 4) 12.9 -> 12.1, (14, 6) 27.9 -> 27.3).
__host__ __device__ constexpr int desc_quad_span(int np, int l_max) {
    const int quads = (l_max + 1) * np / 4, span = (quads + 7) / 8 * 8;
    return span <= 32 && 32 % span == 0 && 8 * quads >= 7 * span ? span : 0;
}
__host__ __device__ constexpr bool desc_quads(int np, int l_max) { return desc_quad_span(np, l_max) > 0 || (l_max + 1) * np / 4 > 16; }

// Pairs staged at once by a warp: 32 where a staged pair is small, so that every lane has a pair's harmonics to form
// (80 words: sixteen warps still fit beside the table for two species), else 16; a team deals its chunks out to its warps
// and takes 16.
__host__ __device__ constexpr int desc_chunk(int l_max, int np, bool team) { return !team && desc_s_row(l_max) + (l_max + 1) * desc_g_l(np) <= 80 ? 32 : 16; }

// Blocks of 4 x 4 (species, n) pairs that Eq. 4 is computed in, and whether their places in the feature row are decoded
// once per CTA into a table (few blocks: up to S n_max = 32) or by every lane for every centre
__host__ __device__ constexpr int desc_blocks(int S, int np, bool crossover) {
    const int ta = S * np / 4, tb = np / 4;
    return crossover ? ta * (ta + 1) / 2 : S * (tb * (tb + 1) / 2);
}
constexpr int kDescTableBlocks = 36;
struct DescBlock {
    int rowoff[4];             // row i of the block starts at this feature (+ j (l_max+1) + l)
    int ta, tb;                // its column tiles
    unsigned valid;            // bit 4 i + j: whether (i, j) is a feature (n below n_max, n' >= n inside a diagonal species block)
    int pad;
};

// Shared memory in 4-byte words: [table (optional)] [block table (few blocks)] then one region per warp:
//   c [LM] rows | S staging [chunk][s_row] | G staging [chunk][L1 g_l] | pair staging [chunk][8 or 5]
// The feature row is assembled on top of the staging area when it fits there.  With the table in shared memory (many
// centres, no radial weighting) a staged pair is five words (dx, dy, dz, t; interval | species << 16) instead of eight (dx,
// dy, dz, r; interval, t, species, weight), for the room of it.
struct DescLayout {
    int table, blocks, warp0, per_warp, c, sS, sG, ring, slab_words, total;
};
__host__ __device__ inline DescLayout make_desc_layout(int S, int np, int l_max, int warps, int table_words, bool team, bool plain) {
    const int L1 = l_max + 1, LM = L1 * L1, n_blocks = desc_blocks(S, np, true), kDescChunk = desc_chunk(l_max, np, team);
    DescLayout o;
    o.table = 0;
    o.blocks = (table_words + 3) & ~3;
    o.warp0 = o.blocks + (n_blocks <= kDescTableBlocks ? n_blocks * (int)(sizeof(DescBlock) / 4) : 0);
    int off = 0;
    o.c = off; off += desc_c_words(S, np, LM, desc_tile_pad(np, l_max, plain));
    o.sS = off; off += kDescChunk * desc_s_row(l_max);
    o.sG = off; off += kDescChunk * L1 * desc_g_l(np);
    o.ring = off; off += kDescChunk * (table_words ? 5 : 8);
    off = (off + 3) & ~3;
    o.slab_words = off - o.sS;
    o.per_warp = off;
    o.total = o.warp0 + warps * off;
    return o;
}

// How a call on n_work centres runs.
struct DescPlan {
    int team;                  // warps that work on one centre, a CTA of them per centre; 0: a warp per centre, persistent CTAs
    bool table;                // whether the radial table is staged in shared memory
    int warps;                 // per CTA
    unsigned grid;
    size_t bytes;              // of shared memory
};

// Few centres: a team of warps per centre, four if the CTAs then run side by side in one wave (four of them fit an
// SM's registers), else two (eight; up to five centres per SM: beyond that a warp per centre is the faster one on half
// of the sizes).  Whole calls, (n_max, l_max) = (8, 6): 120 atoms 27 -> 17 us, 431 atoms of four species 66 -> 38 us,
// 600 atoms 31.2 -> 29.2 us; (12, 8), 600 atoms 60 -> 43 us.
// search_atoms: the team looks for its neighbours among that many atoms (0: it reads them).  Otherwise the radial table
// (table_words) goes to shared memory, unless pairs are weighted, when it leaves room for at least six warps and there is
// enough work to pay for staging it; small jobs use fewer warps per CTA so that they spread over the SMs.
inline DescPlan desc_plan(int S, int np, int l_max, bool plain, bool weighted, size_t table_words, int64_t n_work, int64_t search_atoms, int64_t sms,
                          size_t max_smem) {
    for (const int team : {kDescTeamWarps, 2}) {
        const size_t bytes = (size_t)make_desc_layout(S, np, l_max, team, 0, true, plain).total * 4 + desc_search_bytes(search_atoms, team);
        const int64_t per_sm = std::min<int64_t>(team == 2 ? 5 : 16 / kDescTeamWarps, (int64_t)(228 * 1024 / (bytes + 1024)));
        if (n_work <= per_sm * sms && bytes <= max_smem) return {team, false, team, (unsigned)n_work, bytes};
    }
    auto warps_beside = [&](size_t words) {
        const DescLayout one = make_desc_layout(S, np, l_max, 1, (int)words, false, plain);
        const size_t fixed = (size_t)one.warp0 * 4, each = (size_t)one.per_warp * 4;
        return fixed + each <= max_smem ? (int)std::min<size_t>(kDescMaxWarps, (max_smem - fixed) / each) : 0;
    };
    // (with the table in shared memory a warp's region is a little smaller: its staged pairs are five words, not eight)
    const int warps_fit = warps_beside(0), warps_table = table_words > 0 ? warps_beside(table_words) : 0;
    // The table pays from four centres per SM on, except where the warps it costs make a second round of centres that keeps
    // less than a quarter of them busy (coefficients, table against none: 1500 atoms at (8, 8) 46.1 against 39.6 us, 1000
    // atoms of three species at (6, 9) 48.2 against 36.8 us; with a fuller second round 48.1 against 48.5 us and less).
    const bool straggling = n_work <= warps_fit * sms && n_work > warps_table * sms && 4 * n_work <= 5 * warps_table * sms;
    DescPlan plan;
    plan.team = 0;
    plan.table = !weighted && warps_table >= 6 && n_work >= 4 * sms && !straggling;
    plan.warps = (int)std::max<int64_t>(1, std::min<int64_t>(plan.table ? warps_table : warps_fit, (n_work + sms - 1) / sms));
    plan.grid = (unsigned)std::min<int64_t>(sms, (n_work + plan.warps - 1) / plan.warps);
    plan.bytes = (size_t)make_desc_layout(S, np, l_max, plan.warps, plan.table ? (int)table_words : 0, false, plain).total * 4;
    return plan;
}

}  // namespace soap
