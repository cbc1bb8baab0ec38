// The descriptor-only kernel: expansion coefficients (Eq. 13 / Eqs. 18-19) and the power spectrum
// (Eq. 4) of every centre, one WARP per centre, persistent CTAs whose warps take the centres in turn.
//
// This build is bound by FP32 issue slots and by shared-memory bandwidth, not by HBM, so the layout is
// chosen for few instructions and few shared-memory wavefronts per pair:
//   * the radial table (value polynomials) sits in shared memory once per CTA when it fits; a lane evaluates four adjacent n
//     at once from six 16-byte loads and ten packed multiply-adds (fma.rn.f32x2: one issue slot for two multiply-adds), or two
//     from half as many, whichever fills more lanes (desc_quads);
//   * the pairs of a centre (up to 64 at a time) have their geometry formed in registers, are ranked by species with
//     ballots, and staged 16 or 32 at a time in species order: solid harmonics with a lane per pair from the fully
//     unrolled Q_l^m recursion, radial factors with the lanes side by side on the chunk's pairs and channels (a round per
//     pair left half of the lanes idle at l_max 3: 324,000 atoms at (4, 3) 2.03 -> 1.47 ms, 215,000 at (6, 4) 2.90 -> 2.33 ms,
//     with the chunks of 32);
//   * accumulation c[l,m][n] += S_lm G_nl is register-tiled: a lane owns four consecutive m of one l
//     times all n (an outer product of 4 x n_max per pair from one 16-byte load of S and n_max/4 of
//     G); with at most 16 such tiles the two half-warps work on two pairs at once.  Sums stay in
//     registers over all pairs of a species and are added to the centre's tile c[lm][species, n]
//     once per species; the staging rows are laid out so that all these loads are conflict-free;
//   * Eq. 4 is the Gram matrix of that tile per l: lanes take 4 x 4 blocks of (species, n) pairs,
//     two 16-byte loads per 16 multiply-adds, and the feature row is put together in shared memory
//     and handed to the copy engine.
// At (8, 6) on 30,000 atoms the kernel takes 212 us; the L1 data pipe is 82 % busy, the issue slots 50 %.
// Nothing but the pair list is read from HBM and nothing but the descriptor row is written.
#pragma once
#include "desc_layout.h"
#include "harmonic_tables.h"
#include "pair_test.cuh"
#include "soap_device.cuh"

namespace soap {

// harmonic normalisation up to l = 12: a_lm (sqrt2 folded in for m > 0), index l(l+1)/2 + m
struct HarmonicNorm { float a[kHarmonicTerms]; };
constexpr HarmonicNorm harmonic_norm() {
    constexpr HarmonicTables t = harmonic_tables();
    HarmonicNorm n{};
    for (int i = 0; i < kHarmonicTerms; ++i) n.a[i] = t.norm[i];
    return n;
}
__device__ __constant__ HarmonicNorm kd_norm = harmonic_norm();

// Real solid harmonics S_lm(d) = r^l Y_lm of one displacement, every (l, m), written as 16-byte tiles: tile
// desc_tile_base(l) + j holds m = 4j - l .. 4j + 3 - l of row l (zeros beyond m = l):
//   S_{l,+m} = a_lm Q_l^m Re (x+iy)^m,  S_{l,-m} = a_lm Q_l^m Im (x+iy)^m,
//   Q_m^m = (2m-1)!!,  (l+1-m) Q_{l+1}^m = (2l+1) z Q_l^m - (l+m) r^2 Q_{l-1}^m.
// Fully unrolled: every index is an immediate and the Q's live in registers.
template <int L>
__device__ __forceinline__ void harmonics_tiles(float x, float y, float z, float r2, float4* __restrict__ out) {
    float cm[L + 1], sm[L + 1];                   // (x+iy)^m
    cm[0] = 1.f; sm[0] = 0.f;
#pragma unroll
    for (int m = 1; m <= L; ++m) {
        cm[m] = x * cm[m - 1] - y * sm[m - 1];
        sm[m] = x * sm[m - 1] + y * cm[m - 1];
    }
    float q1[L + 1], q2[L + 1];                   // Q_l^m and Q_{l-1}^m while the loop is at l
#pragma unroll
    for (int m = 0; m <= L; ++m) { q1[m] = 0.f; q2[m] = 0.f; }
    float dfact = 1.f;                            // (2l-1)!!
#pragma unroll
    for (int l = 0; l <= L; ++l) {
        if (l > 0) dfact *= (float)(2 * l - 1);
        const float zl = (float)(2 * l - 1) * z;
        float row[2 * L + 4];                     // S_{l,m} at index m + l
#pragma unroll
        for (int i = 0; i < 2 * L + 4; ++i) row[i] = 0.f;
#pragma unroll
        for (int m = 0; m <= l; ++m) {
            float q;
            if (m == l) q = dfact;
            else q = (zl * q1[m] - (float)(l - 1 + m) * r2 * q2[m]) * (1.f / (float)(l - m));
            q2[m] = q1[m];
            q1[m] = q;
            const float aq = kd_norm.a[l * (l + 1) / 2 + m] * q;
            row[l + m] = aq * cm[m];
            if (m) row[l - m] = aq * sm[m];
        }
#pragma unroll
        for (int j = 0; j < (2 * l + 4) / 4; ++j)
            out[desc_tile_base(l) + j] = make_float4(row[4 * j], row[4 * j + 1], row[4 * j + 2], row[4 * j + 3]);
    }
}

// NP: n_max rounded up to a multiple of four.  PLAIN: the default configuration (atom centres, no weighting, every
// species pair, power spectrum out).  TS: the radial table is in shared memory (not with a weighting: a staged pair then
// has no word for the weight).
// TEAM: few centres, a CTA per centre: its warps take the chunks of pairs in turn, each into a tile of its own, and the
// tiles are added up; the blocks of Eq. 4 are spread over all of them.
// SEARCH: a team that looks for its centre's neighbours itself (CenterParams::numbers).  A kernel of its own: carried along by the
// teams that read their pairs it cost those registers and start-up (coefficients of 570 atoms at (4, 4) 20.6 -> 22.6 us, 200
// centres of 570 atoms 20.6 -> 22.6).
template <int L, int NP, bool PLAIN, bool TS, bool TEAM, bool SEARCH>
__global__ void __launch_bounds__(TEAM ? kDescTeamWarps * 32 : kDescMaxWarps * 32, TEAM ? 16 / kDescTeamWarps : 1) desc_kernel(const CenterParams p) {
    constexpr int L1 = L + 1, LM = L1 * L1;
    constexpr int NCHP = L1 * NP;                                        // channels (l, n), n padded
    constexpr int SROW = desc_s_row(L), GL = desc_g_l(NP), GROW = L1 * GL;
    constexpr int T = desc_tiles(L);
    constexpr int HALVES = T <= 16 ? 2 : 1, LANES_T = 32 / HALVES;
    constexpr int TPL = (T + LANES_T - 1) / LANES_T;                     // tiles per lane (1, or 2 from l_max = 10 on)
    constexpr int NB = (TPL * NP * 4 <= 64) ? NP : 64 / (4 * TPL);      // n handled per pass (at most 64 accumulators)
    constexpr int NPASS = (NP + NB - 1) / NB;
    constexpr bool QUADS = desc_quads(NP, L);
    constexpr int UNIT = QUADS ? 4 : 2, UNITS = NCHP / UNIT;             // units of the radial factors: adjacent n of one l
    constexpr int kDescChunk = desc_chunk(L, NP, TEAM);
    extern __shared__ __align__(16) float smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const bool o_cross = PLAIN || p.crossover, o_emit = !PLAIN && p.emit_coeff;
    const float* const o_cbar = PLAIN ? nullptr : p.c_bar;
    const float* const o_sites = PLAIN ? nullptr : p.sites;
    const float2* const o_pw = PLAIN ? nullptr : p.pair_w;
    const float o_w0 = PLAIN ? 1.f : p.w0;
    const int S = p.S, NMAX = p.n_max, F = p.F;
    const DescLayout lay = make_desc_layout(S, NP, L, warps, TS ? p.n_intervals * NCHP * 6 : 0, TEAM, PLAIN);

    if (TS) {
        const float4* src = reinterpret_cast<const float4*>(p.table_ln);
        float4* dst = reinterpret_cast<float4*>(smem);
        const int n4 = p.n_intervals * NCHP * 6 / 4;
        for (int e = threadIdx.x; e < n4; e += blockDim.x) dst[e] = __ldg(src + e);
        if (desc_blocks(S, NP, true) > kDescTableBlocks) __syncthreads();
    }
    // ---- the blocks of Eq. 4: where they lie in the tile and in the feature row (the same for every l and centre) ----
    constexpr int TB = NP / 4;                                           // 4-wide column tiles per species
    const int TA = S * TB, NTP = desc_blocks(S, NP, o_cross);
    const bool tabled = desc_blocks(S, NP, true) <= kDescTableBlocks;
    DescBlock* const blocks = reinterpret_cast<DescBlock*>(smem + lay.blocks);
    auto decode_block = [&](int rem) {
        DescBlock o;
        int ta = 0, tb;
        if (o_cross) {
            while (rem >= TA - ta) { rem -= TA - ta; ++ta; }
            tb = ta + rem;
        } else {
            const int sb = rem / (TB * (TB + 1) / 2);
            rem -= sb * (TB * (TB + 1) / 2);
            while (rem >= TB - ta) { rem -= TB - ta; ++ta; }
            tb = sb * TB + ta + rem;
            ta += sb * TB;
        }
        const int TRI = (NMAX * (NMAX + 1) / 2) * L1, SQ = NMAX * NMAX * L1;
        const int mu = (4 * ta) / NP, nu = (4 * tb) / NP, na = 4 * ta - mu * NP, nb = 4 * tb - nu * NP;
        const int before = o_cross ? mu * S - mu * (mu - 1) / 2 + (nu - mu) : mu, diag = o_cross ? mu + (nu > mu ? 1 : 0) : mu;
        const int base = diag * TRI + (before - diag) * SQ;
        o.ta = ta; o.tb = tb; o.valid = 0; o.pad = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int n1 = na + i;
            o.rowoff[i] = base + (mu < nu ? n1 * NMAX + nb : n1 * NMAX - n1 * (n1 - 1) / 2 - n1 + nb) * L1;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (n1 < NMAX && nb + j < NMAX && (mu < nu || n1 <= nb + j)) o.valid |= 1u << (4 * i + j);
        }
        return o;
    };
    if (tabled) {
        if ((int)threadIdx.x < NTP) blocks[threadIdx.x] = decode_block(threadIdx.x);
        if ((int)blockDim.x < NTP)
            for (int e = threadIdx.x + blockDim.x; e < NTP; e += blockDim.x) blocks[e] = decode_block(e);
        __syncthreads();
    }
    // the tables are this handle's own; everything below reads what the kernels before this one wrote
    grid_dependency_wait();
    // a failed neighbour build: write nothing
    if (!SEARCH && p.counters->n_pairs > p.pair_capacity) return;

    float* const wbase = smem + lay.warp0 + wid * lay.per_warp;
    float* const c_t = wbase + lay.c;                                               // [LM] rows of RC chunks, skewed
    const int RC = S * NP / 4;
    constexpr bool pad = desc_tile_pad(NP, L, PLAIN);
    auto c_chunk = [&](int r, int k) { return desc_c_at(r, RC, pad) + k; };              // 16-byte chunk k of row r
    auto c_word = [&](int r, int col) { return 4 * c_chunk(r, col >> 2) + (col & 3); };
    float4* const sS4 = reinterpret_cast<float4*>(wbase + lay.sS);                  // [chunk][SROW / 4] tiles of four m
    float* const sG = wbase + lay.sG;                                               // [chunk][L1][GL]
    float4* const ring_d = reinterpret_cast<float4*>(wbase + lay.ring);             // [chunk] dx, dy, dz, r
    int4* const ring_i = reinterpret_cast<int4*>(wbase + lay.ring + 4 * kDescChunk);// [chunk] interval, t, species, weight
    int* const ring_q = reinterpret_cast<int*>(wbase + lay.ring + 4 * kDescChunk);  // TS: [chunk] interval | species << 16, and t in ring_d.w
    const float4* const tab = TS ? reinterpret_cast<const float4*>(smem) : reinterpret_cast<const float4*>(p.table_ln);

    // the tiles of this lane: l, tile index, first row (l^2 + 4 j) and number of valid rows
    const int half = HALVES == 2 ? lane >> 4 : 0;
    int t_l[TPL], t_idx[TPL], t_lm0[TPL], t_kv[TPL];
#pragma unroll
    for (int tp = 0; tp < TPL; ++tp) {
        int t = tp * LANES_T + (lane & (LANES_T - 1)), l = 0;
        t_idx[tp] = t < T ? t : 0;
        if (t >= T) { t_l[tp] = 0; t_lm0[tp] = 0; t_kv[tp] = 0; continue; }
        while (t >= (2 * l + 4) / 4) { t -= (2 * l + 4) / 4; ++l; }
        t_l[tp] = l; t_lm0[tp] = l * l + 4 * t; t_kv[tp] = min(4, 2 * l + 1 - 4 * t);
    }
    // where the radial factors of unit u go in a pair's staging row, in words
    auto g_word = [](int u) {
        const int l = u / (NP / UNIT);
        return (UNIT * u + l * (GL - NP)) ^ (4 * desc_g_swap(NP, l));
    };
    const bool periodic = p.geom.pbc[0] | p.geom.pbc[1] | p.geom.pbc[2];
    const long long n_work = o_cbar ? 1 : p.n_centers;

    // Centres are dealt out to the warps of the grid in turn (neighbouring warps take neighbouring centres).
    constexpr int PPL = kDescGroup / 32;                                 // pairs per lane and group
    struct Head { float xi, yi, zi; int zsp; long long pair_base; int k_pairs; };
    struct Raw { unsigned long long key[PPL]; float wgt[PPL]; int spj[PPL]; float px[PPL], py[PPL], pz[PPL]; };
    // SEARCH: the team looks for its centre's neighbours itself, among all atoms of a small structure whose periodic axes are at least two
    // cutoffs high: an atom then has one image inside at most, the one nearest in each fractional coordinate.  The test is the
    // pair kernel's.  A warp takes a contiguous share of the atoms and leaves its finds in its own slots, in order.
    unsigned long long* const list = reinterpret_cast<unsigned long long*>(smem + lay.total);
    const int share = SEARCH ? desc_search_share(p.n_atoms, warps) : 0;
    int* const s_found = reinterpret_cast<int*>(list + share * warps);
    auto species_of = [&](int number) { return number >= 0 && number < 128 ? __ldg(p.z_lut + number) : -1; };
    auto search = [&](int i) {
        Head h;
        h.xi = p.pos[3 * i]; h.yi = p.pos[3 * i + 1]; h.zi = p.pos[3 * i + 2];
        h.zsp = species_of(p.numbers[i]);
        h.pair_base = 0;
        double fi[3] = {0.0, 0.0, 0.0};
        int status = 0, k = 0;
        if (h.zsp < 0) { status |= kStatusUnknownSpecies; h.zsp = 0; }
        if (periodic) {
            frac_coords(p.geom, h.xi, h.yi, h.zi, fi);
            for (int a = 0; a < 3; ++a)
                if (p.geom.pbc[a] && fabs(floor(fi[a])) > 100.0) status |= kStatusShiftRange;    // absurdly far outside the cell
        }
#pragma unroll 2
        for (int t = 0; t < share; t += 32) {
            const int j = wid * share + t + lane;
            bool valid = false;
            unsigned long long key = 0;
            if (j < p.n_atoms) {
                const float4 pj = make_float4(p.pos[3 * j], p.pos[3 * j + 1], p.pos[3 * j + 2], __int_as_float(j));
                const int zj = p.numbers[j];
                int n[3] = {0, 0, 0};
                if (periodic) {
                    double fj[3];
                    frac_coords(p.geom, pj.x, pj.y, pj.z, fj);
                    for (int a = 0; a < 3; ++a)
                        if (p.geom.pbc[a]) n[a] = -(int)rint(fj[a] - fi[a]);
                }
                valid = inside_cutoff(p.geom, pair_distance2(p.geom, periodic, pj, n[0], n[1], n[2], h.xi, h.yi, h.zi));
                if (valid && beyond_key(n[0], n[1], n[2])) { status |= kStatusShiftRange; valid = false; }
                if (valid) {
                    const int sj = species_of(zj);                            // (its own team reports an unknown one)
                    key = pair_key_of(pj, n[0], n[1], n[2]) | (unsigned long long)max(sj, 0) << 56;
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, valid);
            if (valid) list[wid * share + k + __popc(m & ((1u << lane) - 1))] = key;
            k += __popc(m);
        }
        status = (int)__reduce_or_sync(0xffffffffu, (unsigned)status);
        if (lane == 0) {
            s_found[wid] = k;
            if (status) atomicOr(&p.counters->status, status);
        }
        __syncthreads();
        h.k_pairs = 0;
        for (int w = 0; w < warps; ++w) h.k_pairs += s_found[w];
        return h;
    };
    auto found_key = [&](int e) {
        int w = 0;
        while (w + 1 < warps && e >= s_found[w]) e -= s_found[w++];
        return list[w * share + e];
    };
    auto load_head = [&](long long c_idx) {
        if constexpr (SEARCH) return search((int)c_idx);
        Head h;
        const int ci = o_sites ? -1 : (p.centers ? p.centers[c_idx] : (int)c_idx);
        const float* pc = o_sites ? o_sites + 3 * c_idx : p.pos + 3 * (long long)ci;
        h.xi = pc[0]; h.yi = pc[1]; h.zi = pc[2];
        h.zsp = o_sites ? 0 : p.species_idx[ci];
        h.pair_base = p.pair_start[c_idx];
        h.k_pairs = o_cbar ? 0 : p.pair_count[c_idx];
        return h;
    };
    auto load_keys = [&](const Head& h, int g0, Raw& r) {
#pragma unroll
        for (int b = 0; b < PPL; ++b) {
            const int e = g0 + 32 * b + lane;
            r.key[b] = e < h.k_pairs ? (SEARCH ? found_key(e) : p.pair_key[h.pair_base + e]) : 0ull;
            r.wgt[b] = (o_pw && e < h.k_pairs) ? o_pw[h.pair_base + e].x : 1.f;
        }
    };
    auto load_atoms = [&](const Head& h, int g0, Raw& r) {
#pragma unroll
        for (int b = 0; b < PPL; ++b) {
            const int e = g0 + 32 * b + lane;
            r.spj[b] = -1; r.px[b] = r.py[b] = r.pz[b] = 0.f;
            if (e < h.k_pairs) {
                const int j = key_atom(r.key[b]);
                r.spj[b] = S == 1 ? 0 : SEARCH ? (int)(r.key[b] >> 56) : p.species_idx[j];
                r.px[b] = p.pos[3 * (long long)j]; r.py[b] = p.pos[3 * (long long)j + 1]; r.pz[b] = p.pos[3 * (long long)j + 2];
            }
        }
    };
    // Full rounds give every warp of the grid one centre, CTA by CTA; the centres of the last, partial round are
    // dealt out across the CTAs first, so that every SM gets its share of them instead of a few SMs a full round.
    // (A team: the CTA's own centre.)
    auto wait_row = []() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); };   // this thread's row copies have read the slab
    const long long w_stride = TEAM ? gridDim.x : (long long)gridDim.x * warps, full_rounds = n_work / w_stride;
    for (long long round = 0; round <= full_rounds; ++round) {
        const long long c_idx = TEAM ? round * w_stride + blockIdx.x
                                     : round * w_stride + (round < full_rounds ? (long long)blockIdx.x * warps + wid
                                                                               : (long long)wid * gridDim.x + blockIdx.x);
        if (c_idx >= n_work) break;
        const Head hd = load_head(c_idx);
        Raw raw;
        const float xi = hd.xi, yi = hd.yi, zi = hd.zi;
        const int zi_species = hd.zsp, k_pairs = hd.k_pairs;

        for (int e = lane; e < desc_c_at(LM - 1, RC, pad) + RC; e += 32) reinterpret_cast<float4*>(c_t)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();

        for (int g0 = 0; g0 < k_pairs; g0 += kDescGroup) {
            // ---- geometry of up to 64 pairs, two per lane ----
            const int kg = min(kDescGroup, k_pairs - g0);
            load_keys(hd, g0, raw);
            load_atoms(hd, g0, raw);
            int sp[PPL], pos_sorted[PPL];
            float4 dd[PPL];
            int2 qt[PPL];                                                    // interval, offset bits
            float ww[PPL];
#pragma unroll
            for (int b = 0; b < PPL; ++b) {
                sp[b] = raw.spj[b];
                ww[b] = raw.wgt[b];
                dd[b] = make_float4(0.f, 0.f, 0.f, 0.f);
                qt[b] = make_int2(0, 0);
                pos_sorted[b] = -1;
                if (sp[b] >= 0) {
                    double dx = (double)raw.px[b] - (double)xi;
                    double dy = (double)raw.py[b] - (double)yi;
                    double dz = (double)raw.pz[b] - (double)zi;
                    if (periodic) {
                        int sh[3];
                        key_shift(raw.key[b], sh);
                        dx += sh[0] * p.geom.cell[0] + sh[1] * p.geom.cell[3] + sh[2] * p.geom.cell[6];
                        dy += sh[0] * p.geom.cell[1] + sh[1] * p.geom.cell[4] + sh[2] * p.geom.cell[7];
                        dz += sh[0] * p.geom.cell[2] + sh[1] * p.geom.cell[5] + sh[2] * p.geom.cell[8];
                    }
                    // interval and offset in the radial table, in fp64 so that the offset keeps its digits: r is the fp32
                    // root r0 (relative error 2^-23) and one Newton step on it, whose residual is formed in fp64 and
                    // whose own error is 2^-47
                    const double d2 = fma(dx, dx, fma(dy, dy, dz * dz));
                    const float r0 = sqrtf(fmaxf((float)d2, 1e-30f));
                    const double r = (double)r0 + (double)((float)fma(-(double)r0, (double)r0, d2) * __fdividef(0.5f, r0));
                    const double u = r * p.inv_h;
                    const int qi = min((int)u, p.n_intervals - 1);
                    dd[b] = make_float4((float)dx, (float)dy, (float)dz, (float)r);
                    qt[b] = make_int2(qi, __float_as_int((float)(u - qi)));
                }
            }
            // position of every pair in species order (stable): ballots, no memory traffic
            {
                int base = 0;
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int b = 0; b < PPL; ++b) {
                        const unsigned m = __ballot_sync(0xffffffffu, sp[b] == s);
                        if (sp[b] == s) pos_sorted[b] = base + __popc(m & ((1u << lane) - 1));
                        base += __popc(m);
                    }
            }

            if (!TEAM) {
                if (lane == 0) wait_row();                                   // the row of the centre before has left the staging area
                __syncwarp();
            }
#pragma unroll 1
            for (int ip = 0; ip < NPASS; ++ip) {
                const int n0 = ip * NB;
                // Packed multiply-adds take two products at once: (h_k g_n, h_k+1 g_n+1) into acc[..][k][n/2] and, with the two
                // h swapped, (h_k+1 g_n, h_k g_n+1) into acc[..][k+1][n/2] (k even): two swaps per tile instead of four copies
                // of an h into both halves of a register pair
                float2 acc[TPL][4][NB / 2];
#pragma unroll
                for (int tp = 0; tp < TPL; ++tp)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int n = 0; n < NB / 2; ++n) acc[tp][k][n] = make_float2(0.f, 0.f);
                auto sum_of = [&](int tp, int k, int n) {
                    const float2 even = acc[tp][k & ~1][n / 2], odd = acc[tp][k | 1][n / 2];
                    return (k & 1) == (n & 1) ? ((n & 1) ? even.y : even.x) : ((n & 1) ? odd.y : odd.x);
                };
                int cur = -1;
                const bool single = k_pairs <= kDescGroup;            // one group: every (row, species) is written once

                // sums of species s (columns n0 .. n0 + NB - 1) are added to the centre's tile; the two half-warps add up first
                auto flush = [&](int s) {
#pragma unroll
                    for (int tp = 0; tp < TPL; ++tp) {
#pragma unroll
                        for (int k2 = 0; k2 < (HALVES == 2 ? 2 : 4); ++k2) {
                            // (with two half-warps a lane keeps rows 0, 1 or rows 2, 3 of the tile and sends the others)
                            float v[NB];
#pragma unroll
                            for (int n = 0; n < NB; ++n) {
                                if (HALVES == 2) {
                                    const float low = sum_of(tp, k2, n), high = sum_of(tp, k2 + 2, n);
                                    v[n] = (half ? high : low) + __shfl_xor_sync(0xffffffffu, half ? low : high, 16);
                                } else {
                                    v[n] = sum_of(tp, k2, n);
                                }
                            }
                            const int k = HALVES == 2 ? k2 + 2 * half : k2;
                            if (k < t_kv[tp]) {
                                float4* const c4w = reinterpret_cast<float4*>(c_t);
                                const int r = t_lm0[tp] + k, k0 = (s * NP + n0) / 4;
#pragma unroll
                                for (int n4 = 0; n4 < NB / 4; ++n4)
                                    if (NPASS == 1 || n0 + 4 * n4 < NP) {
                                        float4 o = make_float4(v[4 * n4], v[4 * n4 + 1], v[4 * n4 + 2], v[4 * n4 + 3]);
                                        float4* dst = c4w + c_chunk(r, k0 + n4);
                                        if (!single) {
                                            const float4 old = *dst;
                                            o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w;
                                        }
                                        *dst = o;
                                    }
                            }
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k)
#pragma unroll
                            for (int n = 0; n < NB / 2; ++n) acc[tp][k][n] = make_float2(0.f, 0.f);
                    }
                };

                for (int c0 = TEAM ? wid * kDescChunk : 0; c0 < kg; c0 += TEAM ? warps * kDescChunk : kDescChunk) {
                    const int n_stage = min(kDescChunk, kg - c0);
                    // the pairs at sorted positions c0 .. c0 + 15 go to the staging slots
#pragma unroll
                    for (int b = 0; b < PPL; ++b)
                        if ((unsigned)(pos_sorted[b] - c0) < (unsigned)kDescChunk) {
                            if (TS) {
                                ring_d[pos_sorted[b] - c0] = make_float4(dd[b].x, dd[b].y, dd[b].z, __int_as_float(qt[b].y));
                                ring_q[pos_sorted[b] - c0] = qt[b].x | (sp[b] << 16);
                            } else {
                                ring_d[pos_sorted[b] - c0] = dd[b];
                                ring_i[pos_sorted[b] - c0] = make_int4(qt[b].x, qt[b].y, sp[b], __float_as_int(ww[b]));
                            }
                        }
                    __syncwarp();
                    // solid harmonics: a lane per pair
                    if (lane < n_stage) {
                        const float4 d = ring_d[lane];
                        harmonics_tiles<L>(d.x, d.y, d.z, TS ? fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z)) : d.w * d.w, sS4 + lane * (SROW / 4));
                    }
                    // radial factors of one unit of one pair
                    auto radial = [&](int pr, int u) {
                        int4 gi;
                        if (TS) { gi = make_int4(ring_q[pr] & 0xffff, __float_as_int(ring_d[pr].w), 0, 0); }
                        else gi = ring_i[pr];
                        const float t = __int_as_float(gi.y), wgt = !PLAIN && !TS ? __int_as_float(gi.w) : 1.f;
                        const float2 tt = make_float2(t, t);
                        float* const to = sG + pr * GROW + g_word(u);
                        if constexpr (QUADS) {
                            const float4* row = tab + (unsigned)(gi.x * 6 * UNITS + u);   // the coefficients of t^0 .. t^5, UNITS apart
                            float2 lo, hi;
#pragma unroll
                            for (int k = 5; k >= 0; --k) {
                                const float4 c = TS ? row[k * UNITS] : __ldg(row + k * UNITS);
                                const float2 c_lo = make_float2(c.x, c.y), c_hi = make_float2(c.z, c.w);
                                lo = k == 5 ? c_lo : __ffma2_rn(lo, tt, c_lo);
                                hi = k == 5 ? c_hi : __ffma2_rn(hi, tt, c_hi);
                            }
                            if (!PLAIN && !TS) { lo.x *= wgt; lo.y *= wgt; hi.x *= wgt; hi.y *= wgt; }
                            *reinterpret_cast<float4*>(to) = make_float4(lo.x, lo.y, hi.x, hi.y);
                        } else {
                            // coefficients of t^0 .. t^5 of two adjacent n, interleaved: (c0, c0', c1, c1'), (c2, ..), (c4, ..)
                            const float4* row = tab + (unsigned)(gi.x * UNITS + u) * 3u;
                            const float4 A = TS ? row[0] : __ldg(row), B = TS ? row[1] : __ldg(row + 1), C = TS ? row[2] : __ldg(row + 2);
                            float2 v = __ffma2_rn(make_float2(C.z, C.w), tt, make_float2(C.x, C.y));
                            v = __ffma2_rn(v, tt, make_float2(B.z, B.w));
                            v = __ffma2_rn(v, tt, make_float2(B.x, B.y));
                            v = __ffma2_rn(v, tt, make_float2(A.z, A.w));
                            v = __ffma2_rn(v, tt, make_float2(A.x, A.y));
                            if (!PLAIN && !TS) { v.x *= wgt; v.y *= wgt; }
                            *reinterpret_cast<float2*>(to) = v;
                        }
                    };
                    // (a team's warp has few rounds, and two of them at once make it spill: coefficients of 60 atoms at (14, 3) 18.5 ->
                    // 16.5 us, descriptors of 720 30.3 -> 27.8 us)
                    constexpr int SPAN = QUADS ? desc_quad_span(NP, L) : 0;
                    if constexpr (SPAN > 0) {
                        const int u = lane % SPAN;
                        if (u < UNITS) {
#pragma unroll (TEAM ? 1 : 2)
                            for (int pr = lane / SPAN; pr < n_stage; pr += 32 / SPAN) radial(pr, u);
                        }
                    } else {
                        // the lanes walk down the (pair, unit) list side by side, a warp's width at a time
                        int pr = lane / UNITS, u = lane - pr * UNITS;
#pragma unroll (!QUADS ? 4 : TEAM ? 1 : 2)
                        for (int e = lane; e < n_stage * UNITS; e += 32) {
                            radial(pr, u);
                            // 32 further down the list
                            pr += 32 / UNITS; u += 32 % UNITS;
                            if (u >= UNITS) { u -= UNITS; ++pr; }
                        }
                    }
                    __syncwarp();
                    const int tag = lane < n_stage ? (TS ? ring_q[lane] >> 16 : ring_i[lane].z) : -1;
                    for (int s = 0; s < S; ++s) {
                        const unsigned mask = __ballot_sync(0xffffffffu, tag == s);
                        if (!mask) continue;
                        const int a = __ffs(mask) - 1, b = a + __popc(mask);       // contiguous: staged in species order
                        if (s != cur) {
                            if (cur >= 0) flush(cur);
                            cur = s;
                        }
#pragma unroll 2
                        for (int q = a + half; q < b; q += HALVES) {
                            const float4* sp4 = sS4 + q * (SROW / 4);
                            const float4* gp = reinterpret_cast<const float4*>(sG + q * GROW + n0);
#pragma unroll
                            for (int tp = 0; tp < TPL; ++tp) {
                                const float4 h4 = sp4[t_idx[tp]];
                                const float2 h[4] = {make_float2(h4.x, h4.y), make_float2(h4.y, h4.x), make_float2(h4.z, h4.w),
                                                     make_float2(h4.w, h4.z)};
#pragma unroll
                                for (int n4 = 0; n4 < NB / 4; ++n4) {
                                    if (NPASS > 1 && n0 + 4 * n4 >= NP) break;
                                    const float4 g = gp[t_l[tp] * (GL / 4) + (n4 ^ desc_g_swap(NP, t_l[tp]))];
#pragma unroll
                                    for (int k = 0; k < 4; ++k) {
                                        acc[tp][k][2 * n4] = __ffma2_rn(h[k], make_float2(g.x, g.y), acc[tp][k][2 * n4]);
                                        acc[tp][k][2 * n4 + 1] = __ffma2_rn(h[k], make_float2(g.z, g.w), acc[tp][k][2 * n4 + 1]);
                                    }
                                }
                            }
                        }
                    }
                    __syncwarp();
                }
                if (cur >= 0) flush(cur);
                __syncwarp();
            }
        }

        if (!TEAM && k_pairs == 0) {
            if (lane == 0) wait_row();
            __syncwarp();
        }
        float4* const sum4 = reinterpret_cast<float4*>(TEAM ? smem + lay.warp0 + lay.c : c_t);       // the tile of the centre
        if (TEAM) {
            // the tiles of the team add up in the first warp's, in a fixed order
            __syncthreads();
            for (int e = threadIdx.x; e < desc_c_at(LM - 1, RC, pad) + RC; e += blockDim.x) {
                float4 v = sum4[e];
                for (int w = 1; w < warps; ++w) {
                    const float4 o = sum4[e + w * (lay.per_warp / 4)];
                    v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
                }
                sum4[e] = v;
            }
            __syncthreads();
        }
        // on-site term: the centre's own Gaussian, l = 0 only (second term of Eq. 13)
        if ((!TEAM || wid == 0) && !o_cbar && !o_sites && lane < NMAX) c_t[c_word(0, zi_species * NP + lane)] += o_w0 * __ldg(p.self_term + lane);
        if (o_cbar) {
            // given mean coefficients (inner average) take the place of the centre's own: index (mu n_max + n) LM + lm
            for (int e = lane; e < S * NMAX * LM; e += 32) {
                const int row = e / LM, lm = e - row * LM, mu = row / NMAX, n = row - mu * NMAX;
                c_t[c_word(lm, mu * NP + n)] = __ldg(o_cbar + e);
            }
        }
        if (TEAM) __syncthreads(); else __syncwarp();
        if (o_emit) {
            // coefficient mode: the tile itself is the result, index (mu n_max + n) (l_max+1)^2 + l^2 + l + m
            float* crow = p.out_desc + (size_t)c_idx * (S * NMAX * LM);
            const float* const tile = reinterpret_cast<const float*>(sum4);
            for (int e = TEAM ? (int)threadIdx.x : lane; e < S * NMAX * LM; e += TEAM ? (int)blockDim.x : 32) {
                const int row = e / LM, lm = e - row * LM, mu = row / NMAX, n = row - mu * NMAX;
                crow[e] = tile[c_word(lm, mu * NP + n)];
            }
            if (TEAM) __syncthreads(); else __syncwarp();
            continue;
        }

        // ---- power spectrum (Eq. 4): per l the Gram matrix of the tile's rows over (species, n) ----
        float* const desc_row = p.out_desc + (o_cbar ? (size_t)0 : (size_t)c_idx * F);
        const bool staged = F <= lay.slab_words;
        float* const slab = TEAM ? smem + lay.warp0 + lay.sS : wbase + lay.sS;
        float* const dst = staged ? slab : desc_row;
        // Lanes take blocks of 4 x 4 (species, n) pairs (ta <= tb in units of four columns); a block's place in the
        // feature row does not depend on l, and the lanes walk down the l (with few blocks, several l side by side:
        // group g of the lanes takes l = l_max - g, l_max - g - G, ...).
        const int lanes = TEAM ? (int)blockDim.x : 32, me = TEAM ? (int)threadIdx.x : lane;
        const int G = 2 * NTP <= lanes ? min(lanes / NTP, L1) : 1;   // l's side by side
        for (int tp0 = 0; tp0 < NTP; tp0 += lanes) {
            const int grp = G > 1 ? me / NTP : 0, rem = G > 1 ? me - grp * NTP : tp0 + me;
            const bool active = grp < G && rem < NTP;
            const DescBlock blk = tabled ? blocks[active ? rem : 0] : decode_block(active ? rem : 0);
            const unsigned valid = active ? blk.valid : 0u;
            for (int l0 = L; l0 >= 0; l0 -= G) {
                const int l = l0 - grp;                                // this lane's l (may fall below zero in the last trip)
                const int steps = (active && l >= 0) ? 2 * l + 1 : 0;
                // sums of (a_i b_j, a_i+1 b_j+1) in g[i][j / 2] and, with the two b swapped, (a_i b_j+1, a_i+1 b_j) in
                // g[i + 1][j / 2] (i, j even)
                float2 g[4][2];
#pragma unroll
                for (int i = 0; i < 4; ++i) g[i][0] = g[i][1] = make_float2(0.f, 0.f);
                int r = l >= 0 ? l * l : 0;
                const float4 *pa = sum4 + blk.ta, *pb = sum4 + blk.tb;
                for (int m = 0; m < steps; ++m, ++r) {
                    const int at = desc_c_at(r, RC, pad);
                    const float4 A = pa[at], B = pb[at];
                    const float2 a01 = make_float2(A.x, A.y), a23 = make_float2(A.z, A.w);
                    const float2 b[2] = {make_float2(B.x, B.y), make_float2(B.z, B.w)}, bs[2] = {make_float2(B.y, B.x), make_float2(B.w, B.z)};
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        g[0][j] = __ffma2_rn(a01, b[j], g[0][j]);
                        g[1][j] = __ffma2_rn(a01, bs[j], g[1][j]);
                        g[2][j] = __ffma2_rn(a23, b[j], g[2][j]);
                        g[3][j] = __ffma2_rn(a23, bs[j], g[3][j]);
                    }
                }
                if (steps) {
                    const float kl = __ldg(p.kl + l);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float* o = dst + blk.rowoff[i] + l;
                        // (i, j): the even rows of a pair sit in the first halves
                        const float2 u = g[i & 2][0], us = g[(i & 2) + 1][0], w = g[i & 2][1], ws = g[(i & 2) + 1][1];
                        const float v[4] = {(i & 1) ? us.y : u.x, (i & 1) ? u.y : us.x, (i & 1) ? ws.y : w.x, (i & 1) ? w.y : ws.x};
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (valid & (1u << (4 * i + j))) o[j * L1] = kl * v[j];
                    }
                }
            }
        }
        if (TEAM) __syncthreads(); else __syncwarp();
        if (staged) {
            // the copy engine takes the row where its place allows that (16-byte boundaries); the slab is not written
            // again before the copy has read it
            if ((F & 3) == 0 && (reinterpret_cast<size_t>(p.out_desc) & 15) == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (TEAM) __syncthreads(); else __syncwarp();
                if (me == 0) {
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                                 :: "l"(desc_row), "r"((unsigned)__cvta_generic_to_shared(slab)), "r"(4u * (unsigned)F) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    if (TEAM) wait_row();
                }
            } else {
                for (int e = me; e < F; e += lanes) desc_row[e] = slab[e];
            }
            if (TEAM) __syncthreads(); else __syncwarp();
        }
    }
    if (!TEAM && lane == 0) wait_row();                                      // the slab must outlive the copies that read it
    if (SEARCH && threadIdx.x == 0) {
        // the last team leaves the totals of the call
        int k = 0;
        for (int w = 0; w < warps; ++w) k += s_found[w];
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.counters->found), (unsigned long long)k);
        __threadfence();
        if (atomicAdd(&p.counters->finished, 1) == (int)gridDim.x - 1) {
            __threadfence();
            const long long total = (long long)atomicExch(reinterpret_cast<unsigned long long*>(&p.counters->found), 0ull);
            p.counters->finished = 0;
            p.counters->n_pairs = total;
            p.counters->n_rows = 0;
            if (total > p.pair_capacity) atomicOr(&p.counters->status, kStatusPairCapacity);
        }
    }
}

}  // namespace soap
