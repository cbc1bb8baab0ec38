// Device-side data structures shared by the neighbour kernels and the fused
// per-centre kernel.  sm_100a only.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace soap {

constexpr int kMaxSpecies = 8;
constexpr int kThreads = 256;            // largest CTA of the per-centre derivative kernels
constexpr int kMaxElements = 2048;       // soap_create refuses n_max (l_max+1)^2 above this (shared-memory budget of the tiles)

// status bits (device, sticky until soap_status)
constexpr int kStatusUnknownSpecies = 1;
constexpr int kStatusPairCapacity = 2;
constexpr int kStatusRowCapacity = 4;
constexpr int kStatusShiftRange = 8;

// pair_row flags
constexpr int kRowContinuation = 1 << 30;   // same atom (another image) as the previous pair
constexpr int kRowSelfImage = 1 << 29;      // a periodic image of the centre itself
constexpr int kRowMask = (1 << 29) - 1;

struct Geometry {                 // host-known, passed by value
    double cell[9];               // rows a, b, c (identity when no cell)
    double inv[9];                // inverse: frac = pos * inv
    double height[3];             // distance between opposite cell faces
    double r_cut, rc2;
    int pbc[3];
};

struct GridParams {               // device-resident, written by prep_kernel (above kPrepAtoms atoms by grid_setup_kernel)
    int nb[3];                    // bins per axis
    int R[3];                     // stencil half-width in bins
    int periodic[3];
    double smin[3];               // bin = (s - smin) * sscale
    double sscale[3];
    int n_cells;
    int thin;                     // no periodic axis, axes at right angles: bins a quarter as wide along axis 0 (for_each_candidate_runs)
};

struct Counters {                 // device-resident
    int status;
    int finished;                 // CTAs of a descriptor kernel that searches for itself that are done ...
    long long n_pairs;
    long long n_rows;
    long long found;              // ... and the pairs they found (both zero between calls)
};

// Shared memory of a per-centre derivative kernel (make_layout), offsets in 4-byte words.
struct SmemLayout {
    int c, geo, tri, xdec, zero, D, wUV, sSD, sG, slab, slab_words, total;
    bool keep;                    // the slab is apart from the staging area: what pass 1 staged is still there in pass 2
};

struct CenterParams {
    // structure
    const float* pos;             // [N,3]
    const int* centers;           // [C] or null
    const float* sites;           // [C,3] or null: centres at these points instead of at atoms (no on-site term, no own row)
    const int* order;             // [C] CTA -> centre slot (largest first) or null
    const int* species_idx;       // [N]
    const int* numbers;           // [N] or null: the descriptor kernel looks for its centres' neighbours among all atoms itself ...
    const int* z_lut;             // ... with the species of every atomic number below 128
    int n_atoms;
    long long n_centers;
    Geometry geom;
    // neighbour data
    const long long* pair_start;  // [C] first pair of the centre's segment
    const int* pair_count;        // [C]
    const unsigned long long* pair_key;
    const int* pair_row;
    const long long* row_ptr;     // [C+1]
    const int* self_row;          // [C]
    long long pair_capacity, row_capacity;
    Counters* counters;
    // basis
    const float* table;           // [nint][l][n / 2][6][2], n padded to even: coefficients of two adjacent n interleaved (derivative kernels)
    const float* table_ln;        // value polynomials on wider intervals as [nint][l][n / 2][6][2] or [nint][6][l][n] (desc_quads), n padded to a multiple of 4 (descriptor-only kernel)
    const float* self_term;       // [n_max]
    const int* l_of_lm;           // [lm] -> l
    const float* kl;
    const unsigned* row_ops;      // [S][F] or null: operands of feature f in the row of a neighbour of species s: g | g' << 8 | u << 16 | u' << 24
    const int* feat_pack;         // [F] n | n'<<5 | mu<<10 | nu<<14 | l<<18
    double inv_h;                 // intervals per Angstrom of the radial table in use
    int n_intervals;
    int S, n_max, l_max, F;
    int P;                        // pairs per staged chunk
    SmemLayout lay;               // shared memory of the derivative kernels, for this P
    unsigned nch_magic;           // floor(2^32 / (n_max (l_max+1))) + 1: x / n_ch == umulhi(x, magic) for x < 65536
    // output mode
    int crossover;                // 0: only the species pairs mu == nu are features
    int emit_coeff;               // descriptor build: write the coefficients c^mu_nlm instead of the power spectrum
    const float* c_bar;           // [S n_max (l_max+1)^2] or null: coefficients that replace the centre's own after pass 1
    // inner average over ALL atoms as centres: the kernel writes, for its atom a, d pbar / d r_a = own_scale times the
    // contraction of cbar with sum_i grad_a c(i) (pass 1 collects that sum) to out_jac[a], and no per-pair rows
    int inner_rows;
    float own_scale;
    // outer average over ALL atoms as centres: coefficients of every centre, [C][S n_max (l_max+1)^2] (index
    // (mu n_max + n) (l_max+1)^2 + l^2 + l + m, on-site terms included); the kernel of atom a adds to its own row
    // the rows that the centres it sees hold for it, all times own_scale, in out_jac[a]
    const float* c_all;
    // species-compact Jacobian rows: a neighbour's row holds only the blocks that involve its species (pitch Fc, a
    // multiple of 8 floats); the centre's own full row goes to out_center [C,3,F]
    int compact, Fc;
    float* out_center;
    // radial weighting of the neighbour density: per pair (w(d), w'(d)/d), null when off; w0 scales the on-site term
    const float2* pair_w;
    float w0;
    // outputs
    float* out_desc;              // [C,F]  (coefficient mode: [C, S n_max (l_max+1)^2]; with c_bar: [F])
    float* out_jac;               // [rows,3,F]  (coefficient mode: [rows, 3, S n_max (l_max+1)^2])
    int* row_atom;                // [rows]
};

// Programmatic dependent launch: a kernel launched with the attribute cudaLaunchAttributeProgrammaticStreamSerialization
// may start while the kernel before it in the stream still runs; it must call grid_dependency_wait() before it
// touches anything that kernel (or one before it) wrote - the wait returns once that kernel has finished and its
// writes are visible (at once when the launch carried no attribute).  grid_dependency_launch() lets the NEXT kernel
// of the stream start; without it that happens when this kernel's blocks exit.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// launch of a kernel that begins with grid_dependency_wait(), allowed to overlap the tail of its predecessor
template <class... KArgs, class... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
#endif

__host__ __device__ inline int key_atom(unsigned long long k) { return (int)(k >> 24); }
__host__ __device__ inline void key_shift(unsigned long long k, int s[3]) {
    s[0] = (int)((k >> 16) & 255) - 128;
    s[1] = (int)((k >> 8) & 255) - 128;
    s[2] = (int)(k & 255) - 128;
}

// Shared-memory carve-up of the per-centre kernel, in 4-byte words.  Every region
// starts on a 16-byte boundary.  Rows of the coefficient tiles and of the harmonics
// staging have the odd stride (l_max+1)^2 | 1, which keeps strided accesses off a
// single bank.
constexpr int kGeoPairs = 128;           // pairs whose geometry is staged at once

constexpr int kMaxZeroWords = 1024;      // largest block of zeros that bulk copies write into the structural-zero blocks of the rows

// whether the cross-species blocks of the rows are written in table-driven sweeps (a decode table in shared
// memory): several species, n_max from 9 to 12 and n_max (l_max+1) not a multiple of four (the other cases have
// faster paths with an operand in registers)
__host__ __device__ inline bool cross_table_wanted(int S, int n_max, int l_max) {
    return S > 1 && n_max > 8 && n_max <= 12 && ((n_max * (l_max + 1)) & 3) != 0;
}
__host__ __device__ inline int align4(int x) { return (x + 3) & ~3; }
constexpr int kGeoWords = kGeoPairs * 9 + 44;   // geometry (9 words per pair), species segments (9 + 32 words, padded)
// words of zeros: the largest block (two species, all n, n', l), when there is more than one species
__host__ __device__ inline int zero_words(int S, int n_max, int l_max) {
    const int block = align4(n_max * n_max * (l_max + 1));
    return S == 1 ? 0 : block < kMaxZeroWords ? block : kMaxZeroWords;
}
// Pass 1 of the per-centre kernel: threads that cover the lm index, and groups of them that split the n index.
__host__ __device__ constexpr int pass1_span(int l_max) {
    const int lm = (l_max + 1) * (l_max + 1);
    return lm <= 8 ? 8 : lm <= 16 ? 16 : (lm + 31) / 32 * 32;
}
__host__ __device__ constexpr int pass1_slots(int l_max, int n_max) {
    const int span = pass1_span(l_max), most = span <= 32 ? 64 / span : span <= 64 ? 2 : 256 / span;
    const int want = l_max >= 8 && n_max < 4 ? 1 : l_max <= 3 ? n_max : (n_max + 1) / 2;
    return want < most ? want : most;
}
// Bases whose Jacobian rows are written with the operands of every feature from a table (up to kKeepFeatures features).
__host__ __device__ constexpr bool row_table_wanted(int n_max, int l_max) { return n_max <= 4 && n_max * (l_max + 1) <= 20; }
// Features and l_max up to which the slab of the power spectrum has room of its own beside the staging area (16 bytes
// each), so that a centre's pairs can stay staged for pass 2.  With 100 harmonics and more a chunk holds 8 to 16 pairs, no
// centre's pairs fit, and the room halves the chunk (kernel, 3000 centres of 68 pairs, with and without the room: (3, 9)
// 445 -> 425 us, (4, 12) 851 -> 820 us, (3, 9) crossover off 373 -> 340 us; at l_max 8 and below 0.89 to 1.1 by the pairs).
constexpr int kKeepFeatures = 512, kKeepLmax = 8;
// by_table: the handle has a table of the rows' operands, whose zero behind the channels of every staged pair outlives the
// power spectrum: the slab must not reach it.  With crossover that holds anyway (the table stops at kKeepFeatures features,
// and what has no room of its own up to there has l_max above kKeepLmax and few features), so the plain kernels do not ask.
// (Writing that zero behind the power spectrum would do as well, but costs the kernel 14 of 660 us on 36,000 centres of 18
// pairs at (4, 3), where the slab has room of its own; asking there costs 4 us.)
__host__ __device__ inline SmemLayout make_layout(int S, int n_max, int l_max, int P, int warps, bool weighted, bool by_table = false) {
    const int L1 = l_max + 1, LMP = (L1 * L1) | 1, NCH = n_max * L1, CT = S * n_max * LMP, F = S * n_max * (S * n_max + 1) / 2 * L1;
    SmemLayout o;
    int off = 0;
    o.c = off; off = align4(off + CT);
    o.geo = off; off = align4(off + kGeoWords + (weighted ? 2 * kGeoPairs : 0));   // + per-pair weights
    o.tri = off; off = align4(off + ((n_max * (n_max + 1) / 2) * L1 + 1) / 2);   // 16-bit entries
    o.xdec = off; if (cross_table_wanted(S, n_max, l_max)) off = align4(off + (n_max * NCH + 1) / 2);   // 16-bit entries
    o.zero = off; off += zero_words(S, n_max, l_max);
    // the D tiles (pass 1, centre's row) and the per-warp U/V staging (pass 2) never live
    // at the same time and share space
    o.D = off; o.wUV = off;
    {
        const int a = 3 * CT, b = warps * S * NCH * 4;
        off = align4(off + (a > b ? a : b));
    }
    o.keep = F <= kKeepFeatures && l_max <= kKeepLmax;
    o.slab = off;
    if (o.keep) { o.slab_words = 4 * F; off += 4 * F; }
    o.sSD = off; off = align4(off + P * LMP * 4);
    o.sG = off; off = align4(off + P * (NCH + (row_table_wanted(n_max, l_max) ? 1 : 0)) * 2);
    if (!o.keep) o.slab_words = (by_table ? o.sG : off) - o.slab;
    o.total = off;
    return o;
}

}  // namespace soap
