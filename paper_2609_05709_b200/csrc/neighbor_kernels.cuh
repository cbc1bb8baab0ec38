// Cell list and neighbour compaction (the search step under Eq. 1).
//
// Atoms are binned in fractional coordinates of the cell (of the identity when
// there is none); periodic axes are wrapped for binning only.  A centre visits
// the stencil of bins around its own, and every candidate (atom j, lattice
// translation n) passes the exact test
//     0 < |(r_j - r_i) + ((n_a a + n_b b) + n_c c)|^2 < r_cut^2
// in fp64 on the raw fp32 inputs, each operation rounded separately, so the set
// does not depend on the binning and can be compared bit for bit with a
// reference.  Pairs of a centre come out sorted by (atom, n_a, n_b, n_c).
#pragma once
#include <cooperative_groups.h>

#include "pair_test.cuh"
#include "soap_device.cuh"

namespace soap {

#ifdef __CUDACC__
// launch of a grid that is one thread-block cluster; `dependent`: it begins with grid_dependency_wait() and may overlap
// the tail of its predecessor
template <class... KArgs, class... Args>
inline cudaError_t launch_cluster(void (*kernel)(KArgs...), int ctas, int threads, cudaStream_t st, bool dependent, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = ctas; cfg.blockDim = threads; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = dependent ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
#endif

// ---- order-preserving encoding of doubles for atomicMax ---------------------
__device__ inline unsigned long long enc_double(double x) {
    unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ inline double dec_double(unsigned long long e) {
    unsigned long long b = (e >> 63) ? (e & 0x7fffffffffffffffull) : ~e;
    return __longlong_as_double((long long)b);
}

// species index per atom, and the bounding box of the fractional coordinates
// bbox[0..2] = enc(max s), bbox[3..5] = enc(max -s); zero-initialised by the host
__global__ void species_bbox_kernel(const float* __restrict__ pos, const int* __restrict__ numbers, long long N,
                                    Geometry geom, const int* __restrict__ z_lut, int* __restrict__ species_idx,
                                    unsigned long long* bbox, Counters* counters) {
    double hi[3] = {-1e300, -1e300, -1e300}, lo[3] = {-1e300, -1e300, -1e300};
    bool bad = false;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        int z = numbers[i];
        int s = (z >= 0 && z < 128) ? z_lut[z] : -1;
        if (s < 0) { bad = true; s = 0; }
        species_idx[i] = s;
        double f[3];
        frac_coords(geom, pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], f);
        for (int a = 0; a < 3; ++a) { hi[a] = fmax(hi[a], f[a]); lo[a] = fmax(lo[a], -f[a]); }
    }
    for (int a = 0; a < 3; ++a)
        for (int o = 16; o > 0; o >>= 1) {
            hi[a] = fmax(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
            lo[a] = fmax(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
        }
    if ((threadIdx.x & 31) == 0)
        for (int a = 0; a < 3; ++a) {
            atomicMax(&bbox[a], enc_double(hi[a]));
            atomicMax(&bbox[3 + a], enc_double(lo[a]));
        }
    if (bad) atomicOr(&counters->status, kStatusUnknownSpecies);
}

constexpr int kThinBins = 4;
constexpr long long kThinAtoms = 65536;
constexpr double kThinAround = 160.0;
// Choose the bin grid; called by a whole warp, one lane per axis, the result in `g` (shared or global memory).  Bin
// width (measured perpendicular to the cell faces) is at least r_cut (1 + 1e-6) wherever more than one bin fits, so a
// stencil of +-1 bin covers the sphere; short periodic axes get one bin and a wider stencil of images.  Without a periodic
// axis, the axes at right angles, bins are a quarter as wide along axis 0 (stencil of +-4), where a row of bins is one run
// of the sorted atoms that can be cut to the width of the sphere there: 14.5 r_cut^3 of candidates for a sphere of 4.2
// instead of 27.  (Bins of r_cut / 2 along the other axes as well: 9.2, but 25 rows to look up instead of nine.)  That
// pays above kThinAtoms atoms, where the bins are counted and scanned by kernels of their own, and with many atoms around a
// centre; else the longer scan costs more than the candidates: descriptors of 1,000,002 atoms 8914 -> 8799 us, 3000 atoms of 274
// neighbours 1177 -> 1166, 30,000 of 46 neighbours (198 in a stencil) 280 -> 276, but 24,000 atoms of 37 (132) 1 to 2 us longer.
// may_thin: the caller walks by such runs.
__device__ inline void choose_grid(double hi, double lo, const Geometry& geom, long long N, int cell_cap, bool may_thin, GridParams* g) {
    const int a = threadIdx.x & 31;                       // lanes 3 .. 31 repeat axis 2
    const int ax = min(a, 2);
    const double rc = geom.r_cut * (1.0 + 1e-6);
    const bool periodic = geom.pbc[ax] != 0;
    if (N <= 0) { hi = 0.0; lo = 0.0; }
    const double span = hi - lo;
    const double* const c = geom.cell;
    const bool square = c[1] == 0.0 && c[2] == 0.0 && c[3] == 0.0 && c[5] == 0.0 && c[6] == 0.0 && c[7] == 0.0;
    double want = periodic ? floor(geom.height[ax] / rc) : floor(span * geom.height[ax] / rc);
    if (!(want >= 1.0)) want = 1.0;
    auto of = [&](int axis) { return __shfl_sync(0xffffffffu, want, axis); };
    const double around = 27.0 * (double)N / (of(0) * of(1) * of(2));          // atoms in a stencil of bins as wide as the cutoff
    const bool thin = may_thin && square && !(geom.pbc[0] | geom.pbc[1] | geom.pbc[2]) && (N > kThinAtoms || around >= kThinAround);
    const int split = thin && ax == 0 ? kThinBins : 1;
    if (split > 1) want = fmax(1.0, floor(span * geom.height[ax] * split / rc));
    if (want > 1024.0) want = 1024.0;
    // respect the scratch capacity: shrink the grid uniformly
    for (int it = 0; it < 64; ++it) {
        const double w0 = of(0), w1 = of(1), w2 = of(2);
        if (!(w0 * w1 * w2 > (double)cell_cap)) break;
        want = fmax(1.0, floor(want * 0.8));
    }
    const int nb = (int)want;
    const int n0 = __shfl_sync(0xffffffffu, nb, 0), n1 = __shfl_sync(0xffffffffu, nb, 1), n2 = __shfl_sync(0xffffffffu, nb, 2);
    if (a < 3) {
        g->nb[a] = nb;
        g->periodic[a] = periodic;
        g->smin[a] = periodic ? 0.0 : lo;
        g->sscale[a] = periodic ? (double)nb : (span > 0 ? nb / span : 0.0);
        g->R[a] = periodic ? (int)ceil(rc / (geom.height[a] / nb)) : min(nb - 1, split);
    }
    if (a == 0) { g->n_cells = n0 * n1 * n2; g->thin = thin; }
    __syncwarp();
}

__global__ void __launch_bounds__(32) grid_setup_kernel(const unsigned long long* bbox, Geometry geom, long long N, int cell_cap, GridParams* out,
                                  Counters* counters) {
    if (counters && threadIdx.x == 0) { counters->n_pairs = 0; counters->n_rows = 0; }      // the pair cursor of this call
    const int a = min((int)threadIdx.x, 2);
    choose_grid(dec_double(bbox[a]), -dec_double(bbox[3 + a]), geom, N, cell_cap, counters != nullptr, out);
}

__device__ inline void bin_of(const Geometry& geom, const GridParams& g, float x, float y, float z, int b[3], int w[3]) {
    double s[3];
    frac_coords(geom, x, y, z, s);
    for (int a = 0; a < 3; ++a) {
        double t = s[a];
        w[a] = 0;
        if (g.periodic[a]) {
            double fl = floor(t);
            w[a] = (int)fl;
            t -= fl;
        }
        int bi = (int)floor((t - g.smin[a]) * g.sscale[a]);
        b[a] = min(max(bi, 0), g.nb[a] - 1);
    }
}

__device__ inline int pack3(const int v[3]) { return ((v[0] + 512) << 20) | ((v[1] + 512) << 10) | (v[2] + 512); }
__device__ inline void unpack3(int p, int v[3]) { v[0] = ((p >> 20) & 1023) - 512; v[1] = ((p >> 10) & 1023) - 512; v[2] = (p & 1023) - 512; }

__global__ void bin_count_kernel(const float* __restrict__ pos, long long N, Geometry geom, const GridParams* __restrict__ gp,
                                 int* __restrict__ atom_cell, int* __restrict__ atom_wrap, int* cell_count, Counters* counters) {
    const GridParams g = *gp;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        int b[3], w[3];
        bin_of(geom, g, pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], b, w);
        if (abs(w[0]) > 100 || abs(w[1]) > 100 || abs(w[2]) > 100) {      // positions absurdly far outside the cell
            atomicOr(&counters->status, kStatusShiftRange);
            w[0] = w[1] = w[2] = 0;
        }
        int cell = (b[2] * g.nb[1] + b[1]) * g.nb[0] + b[0];
        atom_cell[i] = cell;
        atom_wrap[i] = pack3(w);
        atomicAdd(&cell_count[cell], 1);
    }
}

// Exclusive scan by ONE block (n is at most a few million here); out[n] = total.
template <typename OutT>
__global__ void scan_kernel(const int* __restrict__ in, OutT* __restrict__ out, long long n, long long* total_out,
                            const int* n_dev = nullptr) {
    if (n_dev) n = min(n, (long long)*n_dev);          // only the bins the grid really uses
    __shared__ long long warp_sums[32];
    __shared__ long long carry_s;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (long long base = 0; base < n; base += blockDim.x) {
        long long i = base + threadIdx.x;
        long long v = i < n ? (long long)in[i] : 0, x = v;
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sums[wid] = x;
        __syncthreads();
        if (wid == 0) {
            long long s = lane < nw ? warp_sums[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                long long y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            warp_sums[lane] = s;
        }
        __syncthreads();
        long long carry = carry_s;
        long long excl = carry + (wid > 0 ? warp_sums[wid - 1] : 0) + x - v;
        if (i < n) out[i] = (OutT)excl;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry_s = carry + warp_sums[nw - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[n] = (OutT)carry_s;
        if (total_out) *total_out = carry_s;
    }
}

// Exclusive scan of long arrays in three launches: sums of tiles of kScanTile items, a one-block
// scan of those sums, then every tile scans itself on top of its offset.
constexpr int kScanTile = 4096;          // 1024 threads x 4 items
__global__ void __launch_bounds__(1024) tile_sum_kernel(const int* __restrict__ in, long long n, int* __restrict__ tile_sums) {
    __shared__ int ws[32];
    const long long base = (long long)blockIdx.x * kScanTile;
    int v = 0;
    for (int k = 0; k < 4; ++k) {
        const long long i = base + k * 1024 + threadIdx.x;
        if (i < n) v += in[i];
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        int t = ws[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) tile_sums[blockIdx.x] = t;
    }
}
template <typename OutT>
__global__ void __launch_bounds__(1024) tile_scan_kernel(const int* __restrict__ in, OutT* __restrict__ out, long long n,
                                                         const long long* __restrict__ tile_offsets, long long n_tiles,
                                                         const Counters* counters = nullptr, Counters* host = nullptr) {
    __shared__ long long ws[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long base = (long long)blockIdx.x * kScanTile + threadIdx.x * 4;      // 4 consecutive items per thread
    int v[4];
    long long mine = 0;
    for (int k = 0; k < 4; ++k) { v[k] = base + k < n ? in[base + k] : 0; mine += v[k]; }
    long long x = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        long long t = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    long long run = tile_offsets[blockIdx.x] + (wid > 0 ? ws[wid - 1] : 0) + x - mine;
    for (int k = 0; k < 4; ++k) {
        if (base + k < n) out[base + k] = (OutT)run;
        run += v[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[n] = (OutT)tile_offsets[n_tiles];
        if (host) *host = *counters;                     // pinned host memory: the caller waits for the stream and reads it
    }
}

__global__ void bin_fill_kernel(const float* __restrict__ pos, long long N, const int* __restrict__ atom_cell,
                                const int* __restrict__ atom_wrap, const int* __restrict__ cell_start, int* cell_count,
                                float4* __restrict__ s_pos, int* __restrict__ s_wrap) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        int cell = atom_cell[i];
        int slot = cell_start[cell] + atomicSub(&cell_count[cell], 1) - 1;
        s_pos[slot] = make_float4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], __int_as_float((int)i));
        s_wrap[slot] = atom_wrap[i];
    }
}

// Species lookup, bounding box, grid choice, binning, bin scan and the sort of the atoms by bin in ONE launch (seven
// dependent launches otherwise; up to some ten thousand atoms the launches, not the work, set the time): of a single CTA
// up to kSmallPrepAtoms, bin counters on chip as long as they fit; of a thread-block cluster up to kPrepAtoms, whose CTAs
// exchange the bounding box and the totals of the bin scan through each other's shared memory, bin counters in global
// memory, zero before and after the call (the scan clears what it reads).  A thread keeps its atoms' positions, bins and
// places in registers through the phases; without a free axis there is no bounding box to form (whole search of 431
// atoms in a periodic box 22.2 -> 17.9 us with the pair kernel's loads ahead, 3000 atoms of water 25.5 -> 23.9 us).  At
// 4096 atoms and below the cluster is no faster (1111 atoms 11.0 against 12.0 us, 3000 atoms 14.5 us both); at 30,000
// atoms it takes 20 us, the seven launches 31 us and their gaps.
constexpr int kPrepThreads = 1024, kPrepCtas = 8, kPrepPerThread = 8, kSmallPrepPerThread = 4;
constexpr long long kPrepAtoms = (long long)kPrepThreads * kPrepCtas * kPrepPerThread, kSmallPrepAtoms = (long long)kPrepThreads * kSmallPrepPerThread;
constexpr int kPrepSmemCells = 4096;
template <bool CLUSTER, int PER_THREAD>
__global__ void __launch_bounds__(kPrepThreads)
prep_kernel(const float* __restrict__ pos, const int* __restrict__ numbers, long long N, Geometry geom,
            const int* __restrict__ z_lut, int* __restrict__ species_idx, int cell_cap, GridParams* grid_out,
            int* __restrict__ atom_cell, int* __restrict__ atom_wrap, int* cell_count, int* cell_start,
            float4* __restrict__ s_pos, int* __restrict__ s_wrap, Counters* counters) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double red[6][32], box[6];
    __shared__ GridParams sg;
    __shared__ int warp_sums[32], cta_total;
    __shared__ int s_count[CLUSTER ? 1 : kPrepSmemCells];
    grid_dependency_launch();                                                // the pair kernel may move in and wait
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rank = CLUSTER ? (int)cluster.block_rank() : 0, ctas = CLUSTER ? (int)cluster.num_blocks() : 1;
    const int stride = ctas * kPrepThreads, first = rank * kPrepThreads + tid, n = (int)N;
    if (!CLUSTER)
        for (int c = tid; c < kPrepSmemCells; c += kPrepThreads) s_count[c] = 0;
    // ---- species and bounding box of the fractional coordinates ----
    // (with more than four atoms per thread the positions do not fit the registers and are read again)
    constexpr int KEPT = PER_THREAD <= 4 ? PER_THREAD : 1;
    float x[KEPT], y[KEPT], z[KEPT];
    auto position = [&](int k, int i, float& px, float& py, float& pz) {
        if (PER_THREAD <= 4) { px = x[k % KEPT]; py = y[k % KEPT]; pz = z[k % KEPT]; }
        else { px = pos[3 * i]; py = pos[3 * i + 1]; pz = pos[3 * i + 2]; }
    };
    bool bad = false;
#pragma unroll
    for (int k = 0; k < PER_THREAD; ++k) {
        const int i = first + k * stride;
        x[k % KEPT] = y[k % KEPT] = z[k % KEPT] = 0.f;
        if (i < n) {
            if (PER_THREAD <= 4) { x[k % KEPT] = pos[3 * i]; y[k % KEPT] = pos[3 * i + 1]; z[k % KEPT] = pos[3 * i + 2]; }
            const int number = numbers[i];
            int s = (number >= 0 && number < 128) ? z_lut[number] : -1;
            if (s < 0) { bad = true; s = 0; }
            species_idx[i] = s;
        }
    }
    if (bad) atomicOr(&counters->status, kStatusUnknownSpecies);
    const bool free_axis = !(geom.pbc[0] && geom.pbc[1] && geom.pbc[2]);
    if (free_axis) {
        double m[6] = {-1e300, -1e300, -1e300, -1e300, -1e300, -1e300};       // max s, max -s
#pragma unroll
        for (int k = 0; k < PER_THREAD; ++k)
            if (first + k * stride < n) {
                float px, py, pz;
                position(k, first + k * stride, px, py, pz);
                double f[3];
                frac_coords(geom, px, py, pz, f);
                for (int a = 0; a < 3; ++a) { m[a] = fmax(m[a], f[a]); m[3 + a] = fmax(m[3 + a], -f[a]); }
            }
        for (int a = 0; a < 6; ++a) {
            for (int o = 16; o > 0; o >>= 1) m[a] = fmax(m[a], __shfl_xor_sync(0xffffffffu, m[a], o));
            if (lane == 0) red[a][wid] = m[a];
        }
        __syncthreads();
        if (wid < 6) {
            double v = red[wid][lane];
            for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (lane == 0) box[wid] = v;
        }
        if (CLUSTER) cluster.sync(); else __syncthreads();
    }
    if (wid == 0) {
        // every CTA makes the same choice from the boxes of all of them
        const int a = min(lane, 2);
        double hi = -1e300, lo = -1e300;
        if (free_axis)
            for (int r = 0; r < ctas; ++r) {
                const double* other = CLUSTER ? cluster.map_shared_rank(box, r) : box;
                hi = fmax(hi, other[a]); lo = fmax(lo, other[3 + a]);
            }
        choose_grid(hi, -lo, geom, N, cell_cap, true, &sg);
        if (rank == 0 && lane == 0) {
            *grid_out = sg;
            counters->n_pairs = 0;                                            // the pair cursor of this call
            counters->n_rows = 0;
        }
    }
    __syncthreads();
    const GridParams g = sg;
    int* const count = !CLUSTER && g.n_cells <= kPrepSmemCells ? s_count : cell_count;
    // ---- bin counts; the count an atom finds is its place within the bin ----
    int cell[KEPT], place[PER_THREAD];
#pragma unroll
    for (int k = 0; k < PER_THREAD; ++k) {
        const int i = first + k * stride;
        cell[k % KEPT] = place[k] = 0;
        if (i < n) {
            float px, py, pz;
            position(k, i, px, py, pz);
            int b[3], w[3];
            bin_of(geom, g, px, py, pz, b, w);
            if (abs(w[0]) > 100 || abs(w[1]) > 100 || abs(w[2]) > 100) {      // positions absurdly far outside the cell
                atomicOr(&counters->status, kStatusShiftRange);
                w[0] = w[1] = w[2] = 0;
            }
            const int own = (b[2] * g.nb[1] + b[1]) * g.nb[0] + b[0];
            if (PER_THREAD <= 4) cell[k % KEPT] = own;
            atom_cell[i] = own;
            atom_wrap[i] = pack3(w);
            place[k] = atomicAdd(&count[own], 1);
        }
    }
    if (CLUSTER) cluster.sync(); else __syncthreads();
    // ---- exclusive scan of the bin counts: a contiguous range of bins per CTA and per thread ----
    const int per_cta = (g.n_cells + ctas - 1) / ctas, c_end = min(g.n_cells, (rank + 1) * per_cta);
    const int per_thread = (per_cta + kPrepThreads - 1) / kPrepThreads;
    const int c0 = min(c_end, rank * per_cta + tid * per_thread), c1 = min(c_end, c0 + per_thread);
    int mine = 0;
    for (int c = c0; c < c1; ++c) mine += count[c];
    int incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
    }
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int w = warp_sums[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += up;
        }
        warp_sums[lane] = w;
        if (lane == 31) cta_total = w;
    }
    if (CLUSTER) cluster.sync(); else __syncthreads();
    int at = (wid > 0 ? warp_sums[wid - 1] : 0) + incl - mine;
    if (CLUSTER)
        for (int r = 0; r < rank; ++r) at += *cluster.map_shared_rank(&cta_total, r);
    for (int c = c0; c < c1; ++c) {
        const int v = count[c];
        cell_start[c] = at;
        count[c] = count == s_count ? at : 0;                                // (on chip: the bin's start, for the sort)
        at += v;
    }
    if (rank == 0 && tid == 0) cell_start[g.n_cells] = n;
    if (CLUSTER) cluster.sync(); else __syncthreads();
    // ---- atoms sorted by bin ----
    const int* const start = count == s_count ? s_count : cell_start;
#pragma unroll
    for (int k = 0; k < PER_THREAD; ++k) {
        const int i = first + k * stride;
        if (i < n) {
            float px, py, pz;
            position(k, i, px, py, pz);
            const int slot = start[PER_THREAD <= 4 ? cell[k % KEPT] : atom_cell[i]] + place[k];
            s_pos[slot] = make_float4(px, py, pz, __int_as_float(i));
            s_wrap[slot] = atom_wrap[i];
        }
    }
}

// floor division / modulo for the periodic wrap of a bin coordinate
__device__ inline void wrap_bin(int b, int nb, int& cell, int& image) {
    image = (b >= 0) ? b / nb : -((-b + nb - 1) / nb);
    cell = b - image * nb;
}

// Whether the atom pj (bin wrap `wrap`, in a bin at image `img`) is a neighbour of the centre, and its key.
__device__ __forceinline__ bool look_at(const Geometry& geom, bool any_periodic, float4 pj, int wrap, int img, float xi, float yi, float zi,
                                        const int wi[3], Counters* counters, unsigned long long& key) {
    int wj[3], im[3];
    unpack3(wrap, wj);
    unpack3(img, im);
    // translation on the raw (unwrapped) inputs
    const int na = im[0] - wj[0] + wi[0], nb = im[1] - wj[1] + wi[1], nc = im[2] - wj[2] + wi[2];
    bool valid = inside_cutoff(geom, pair_distance2(geom, any_periodic, pj, na, nb, nc, xi, yi, zi));
    if (valid && beyond_key(na, nb, nc)) {
        atomicOr(&counters->status, kStatusShiftRange);
        valid = false;
    }
    key = pair_key_of(pj, na, nb, nc);
    return valid;
}

// Calls f(valid, key) for every lane in lock step, over all candidates of one centre.
// key encodes (atom, lattice translation on the raw inputs); valid says whether this
// lane holds a pair inside the cutoff.
// The stencil is walked 32 bins at a time: each lane fetches the atom range of one bin (a single
// memory round trip for all of them), a warp scan turns the counts into offsets, and the lanes
// then run over the concatenated candidates, so they stay busy whatever the bin occupancy, AHEAD of them per lane at once.
// PERIODIC: an axis is periodic, as the caller knows; else that is looked up.
template <int AHEAD = 1, bool PERIODIC = false, class F>
__device__ inline void for_each_candidate(const Geometry& geom, const GridParams& g, const int* __restrict__ cell_start,
                                          const float4* __restrict__ s_pos, const int* __restrict__ s_wrap,
                                          float xi, float yi, float zi, const int bi[3], const int wi[3],
                                          int lane, Counters* counters, F f) {
    const int w0 = 2 * g.R[0] + 1, w1 = 2 * g.R[1] + 1, w2 = 2 * g.R[2] + 1;
    const int n_stencil = w0 * w1 * w2;
    const bool any_periodic = PERIODIC || (g.periodic[0] | g.periodic[1] | g.periodic[2]);
    for (int q0 = 0; q0 < n_stencil; q0 += 32) {
        // ---- this lane's bin of the stencil ----
        const int q = q0 + lane;
        int start = 0, cnt = 0, img = 0;                  // img: packed image of the bin (periodic axes)
        if (q < n_stencil) {
            int o[3] = {q % w0 - g.R[0], (q / w0) % w1 - g.R[1], q / (w0 * w1) - g.R[2]};
            int c[3], im[3];
            bool inside = true;
            for (int a = 0; a < 3; ++a) {
                if (g.periodic[a]) wrap_bin(bi[a] + o[a], g.nb[a], c[a], im[a]);
                else { c[a] = bi[a] + o[a]; im[a] = 0; inside &= (c[a] >= 0 && c[a] < g.nb[a]); }
            }
            if (inside) {
                const int cell = (c[2] * g.nb[1] + c[1]) * g.nb[0] + c[0];
                start = cell_start[cell];
                cnt = cell_start[cell + 1] - start;
                img = pack3(im);
            }
        }
        // ---- offsets of the bins in the concatenated candidate list ----
        int incl = cnt;
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        for (int t0 = 0; t0 < total; t0 += 32 * AHEAD) {
            // where the lane's next AHEAD candidates are, and their loads, before any of them is looked at
            float4 pj[AHEAD];
            int wrap[AHEAD], b_img[AHEAD];
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                const int t = t0 + 32 * u + lane;
                // bin of candidate t: the first lane whose inclusive offset exceeds t (binary search by shuffles)
                int lo = 0;
                for (int step = 16; step > 0; step >>= 1) {
                    const int probe = __shfl_sync(0xffffffffu, incl, lo + step - 1);
                    if (probe <= t) lo += step;
                }
                lo = min(lo, 31);
                const int b_incl = __shfl_sync(0xffffffffu, incl, lo), b_cnt = __shfl_sync(0xffffffffu, cnt, lo);
                const int b_start = __shfl_sync(0xffffffffu, start, lo);
                b_img[u] = __shfl_sync(0xffffffffu, img, lo);
                if (AHEAD == 1 || t < total) {
                    const int at = t < total ? b_start + (t - (b_incl - b_cnt)) : 0;
                    pj[u] = s_pos[at];
                    wrap[u] = s_wrap[at];
                }
            }
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                unsigned long long key = 0;
                const bool valid = t0 + 32 * u + lane < total && look_at(geom, any_periodic, pj[u], wrap[u], b_img[u], xi, yi, zi, wi, counters, key);
                f(valid, key);
            }
        }
    }
}

// The same walk for the common case (no periodic axis, stencil of +-1 bin across the rows): the bins of a stencil row along
// x are neighbours in the sorted atom array, so the stencil is 9 contiguous runs, each cut to the bins that the sphere
// reaches in its row (GridParams::thin).  Every lane keeps the nine run boundaries in registers, and a candidate finds its
// run with compares instead of shuffles.
template <class F>
__device__ inline void for_each_candidate_runs(const Geometry& geom, const GridParams& g, const int* __restrict__ cell_start,
                                               const float4* __restrict__ s_pos, float xi, float yi, float zi,
                                               const int bi[3], int lane, F f) {
    // lane r < 9 fetches run r = (dy + 1) + 3 (dz + 1)
    int start = 0, cnt = 0;
    if (lane < 9) {
        const int cy = bi[1] + lane % 3 - g.R[1], cz = bi[2] + lane / 3 - g.R[2];
        const bool inside = cy >= 0 && cy < g.nb[1] && cz >= 0 && cz < g.nb[2] && (lane % 3 <= 2 * g.R[1]) && (lane / 3 <= 2 * g.R[2]);
        if (inside) {
            int x0 = max(bi[0] - g.R[0], 0), x1 = min(bi[0] + g.R[0], g.nb[0] - 1);
            if (g.thin) {
                // how far the sphere reaches along x at the nearest point of this row of bins, a little rounded up (an
                // atom's bin and its edges carry rounding errors of the coordinates' last places)
                const double rc = geom.r_cut * (1.0 + 1e-6);
                double s[3], rest = rc * rc;
                frac_coords(geom, xi, yi, zi, s);
                const int row[3] = {0, cy, cz};
#pragma unroll
                for (int a = 1; a < 3; ++a) {
                    const double t = (s[a] - g.smin[a]) * g.sscale[a] - row[a];            // the bin is 0 .. 1
                    const double away = fmax(fmax(-t, t - 1.0) - 1e-6, 0.0);
                    if (away > 0.0) { const double d = away / g.sscale[a] * geom.height[a]; rest -= d * d; }
                }
                const double reach = rest > 0.0 ? sqrt(rest) / geom.height[0] : 0.0, at = s[0] - g.smin[0];
                x0 = max(x0, (int)floor((at - reach) * g.sscale[0] - 1e-6));
                x1 = min(x1, (int)floor((at + reach) * g.sscale[0] + 1e-6));
                if (rest <= 0.0) x1 = x0 - 1;
            }
            if (x0 <= x1) {
                const int first = (cz * g.nb[1] + cy) * g.nb[0];
                start = cell_start[first + x0];
                cnt = cell_start[first + x1 + 1] - start;
            }
        }
    }
    int r_start[9], r_end[9], total = 0;                 // run r covers candidates r_end[r] - count .. r_end[r] - 1
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const int c = __shfl_sync(0xffffffffu, cnt, r);
        r_start[r] = __shfl_sync(0xffffffffu, start, r) - total;      // atom index = r_start[r] + t for t inside run r
        total += c;
        r_end[r] = total;
    }
    for (int t0 = 0; t0 < total; t0 += 32) {
        const int t = t0 + lane;
        bool valid = false;
        unsigned long long key = 0;
        if (t < total) {
            int at = r_start[8];
#pragma unroll
            for (int r = 7; r >= 0; --r) at = t < r_end[r] ? r_start[r] : at;
            const float4 pj = s_pos[at + t];
            const double dx = __dsub_rn((double)pj.x, (double)xi);
            const double dy = __dsub_rn((double)pj.y, (double)yi);
            const double dz = __dsub_rn((double)pj.z, (double)zi);
            const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
            valid = (d2 < geom.rc2) && (d2 > 0.0);
            key = ((unsigned long long)(unsigned)__float_as_int(pj.w) << 24) | 0x808080ull;
        }
        f(valid, key);
    }
}

// One warp per centre: number of pairs.
__global__ void count_kernel(const float* __restrict__ pos, const int* __restrict__ centers, long long C, Geometry geom,
                             const GridParams* __restrict__ gp, const int* __restrict__ atom_cell, const int* __restrict__ atom_wrap,
                             const int* __restrict__ cell_start, const float4* __restrict__ s_pos, const int* __restrict__ s_wrap,
                             int* __restrict__ pair_count, Counters* counters) {
    const GridParams g = *gp;
    const int lane = threadIdx.x & 31;
    const long long c = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= C) return;
    const int i = centers ? centers[c] : (int)c;
    const float xi = pos[3 * (long long)i], yi = pos[3 * (long long)i + 1], zi = pos[3 * (long long)i + 2];
    int bi[3], wi[3];
    {
        int cell = atom_cell[i];
        bi[0] = cell % g.nb[0]; bi[1] = (cell / g.nb[0]) % g.nb[1]; bi[2] = cell / (g.nb[0] * g.nb[1]);
        unpack3(atom_wrap[i], wi);
    }
    int cnt = 0;
    for_each_candidate(geom, g, cell_start, s_pos, s_wrap, xi, yi, zi, bi, wi, lane, counters,
                       [&](bool valid, unsigned long long) { cnt += __popc(__ballot_sync(0xffffffffu, valid)); });
    if (lane == 0) pair_count[c] = cnt;
}

constexpr int kFillSmemKeys = 512;       // per warp; longer rows are sorted through global memory
constexpr int kFillSmemKeysSmall = 128;  // variant for structures with few pairs per centre: 4x less shared memory, more warps resident
constexpr int kFillWarps = 4;

// One warp per centre, one walk over the candidates: collect the pairs, reserve a segment of the
// pair arrays with one atomic add (segments follow the order in which warps arrive, so the pair
// arrays are addressed through pair_start / pair_count, not through a prefix sum), sort the keys,
// derive the Jacobian row bookkeeping (distinct atoms, the centre's own position among them).
// When the segment does not fit the planned capacity only the counts are produced and the status
// word says so; the caller plans again with the totals.
// ROWS = false (descriptor-only calls, which sum over the pairs in any order and have no Jacobian rows): the keys
// go out as they were found, unsorted, and the row bookkeeping is left out.
// AHEAD: candidates per lane whose loads are in flight at once where images have to be looked up: one on many centres (the
// warps hide each other's loads, and more cost registers), four on few, where a call waits for the longest warp (search
// of 60 atoms in a periodic box 31.6 -> 26.0 us, 431 atoms 21.1 -> 19.6 us, 2000 atoms 27.8 -> 26.0 us, 5000 atoms
// 35.7 -> 37.7 us).
// PERIODIC: an axis is periodic, and images have to be looked up; without one the centre walks runs of the sorted atoms.  A
// kernel holds one of the two walks only: with both (and the runs a second time, in the rare second walk below) the compiler
// spoilt the one that images take, at whatever bound on its registers (search and descriptors of a periodic box, r_cut 6, both
// walks against one: 60 atoms 34.2 -> 31.0 us, 150 atoms 55.7 -> 49.0 us, 1200 atoms 41.1 -> 37.8 us).
template <int KEYS, bool ROWS, bool PERIODIC, int AHEAD>
__global__ void __launch_bounds__(kFillWarps * 32)
pairs_kernel(const float* __restrict__ pos, const int* __restrict__ centers, const float* __restrict__ sites, long long C, Geometry geom,
             const GridParams* __restrict__ gp, const int* __restrict__ atom_cell, const int* __restrict__ atom_wrap,
             const int* __restrict__ cell_start, const float4* __restrict__ s_pos, const int* __restrict__ s_wrap,
             long long pair_capacity, unsigned long long* pair_tmp, unsigned long long* pair_key, int* __restrict__ pair_row,
             long long* __restrict__ pair_start, int* __restrict__ pair_count, int* __restrict__ row_count,
             int* __restrict__ self_row, Counters* counters) {
    constexpr int BUCKETS = KEYS < 256 ? KEYS : 256;
    __shared__ unsigned long long s_raw[kFillWarps][KEYS];
    __shared__ unsigned long long s_sorted[kFillWarps][ROWS ? KEYS : 1];
    __shared__ __align__(16) int s_bucket[kFillWarps][ROWS ? BUCKETS : 4];
    grid_dependency_launch();
    grid_dependency_wait();                                                  // the cell list of the kernel before
    const GridParams g = *gp;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long c = blockIdx.x * (long long)kFillWarps + wid;
    if (c >= C) return;
    // a centre is an atom, or (with `sites`) a point of its own: no atom index, no row of its own
    const bool site = sites != nullptr;
    const int i = site ? -1 : (centers ? centers[c] : (int)c);
    const float* pc = site ? sites + 3 * c : pos + 3 * (long long)i;
    const float xi = pc[0], yi = pc[1], zi = pc[2];
    int bi[3], wi[3];
    if (site) {
        bin_of(geom, g, xi, yi, zi, bi, wi);
        if (abs(wi[0]) > 100 || abs(wi[1]) > 100 || abs(wi[2]) > 100) {
            if (lane == 0) atomicOr(&counters->status, kStatusShiftRange);
            wi[0] = wi[1] = wi[2] = 0;
        }
    } else {
        int cell = atom_cell[i];
        bi[0] = cell % g.nb[0]; bi[1] = (cell / g.nb[0]) % g.nb[1]; bi[2] = cell / (g.nb[0] * g.nb[1]);
        unpack3(atom_wrap[i], wi);
    }
    // ---- walk the candidates; keep the keys on chip while they fit ----
    int k = 0;
    auto collect = [&](bool valid, unsigned long long key) {
        const unsigned m = __ballot_sync(0xffffffffu, valid);
        const int at = k + __popc(m & ((1u << lane) - 1));
        if (valid && at < KEYS) s_raw[wid][at] = key;
        k += __popc(m);
    };
    // (that an axis is periodic is told where several candidates are in flight: 150 atoms 50.6 -> 49.1 us; with one it costs registers,
    // 64 against 53, and 10,000 atoms 66.0 -> 68.0)
    if constexpr (PERIODIC) for_each_candidate<AHEAD, (AHEAD > 1)>(geom, g, cell_start, s_pos, s_wrap, xi, yi, zi, bi, wi, lane, counters, collect);
    else for_each_candidate_runs(geom, g, cell_start, s_pos, xi, yi, zi, bi, lane, collect);
    long long base = 0;
    if (lane == 0) base = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&counters->n_pairs), (unsigned long long)k);
    base = __shfl_sync(0xffffffffu, base, 0);
    const bool fits = base + k <= pair_capacity;
    const bool in_smem = k <= KEYS;
    if (lane == 0) { pair_start[c] = base; pair_count[c] = fits ? k : 0; }
    if (!fits) {
        if (lane == 0) {
            atomicOr(&counters->status, kStatusPairCapacity);
            row_count[c] = k + 1;                         // upper bound; exact once the plan fits
            self_row[c] = 0;
        }
        return;
    }
    if (!in_smem) {
        // rare: more pairs than the on-chip buffer holds; walk again, now with a place to put them
        int at0 = 0;
        for_each_candidate(geom, g, cell_start, s_pos, s_wrap, xi, yi, zi, bi, wi, lane, counters,
                           [&](bool valid, unsigned long long key) {
                               const unsigned m = __ballot_sync(0xffffffffu, valid);
                               const int at = at0 + __popc(m & ((1u << lane) - 1));
                               if (valid && at < k) pair_tmp[base + at] = key;
                               at0 += __popc(m);
                           });
    }
    __syncwarp();
    if (!ROWS) {
        const unsigned long long* raw = in_smem ? s_raw[wid] : pair_tmp + base;
        for (int q = lane; q < k; q += 32) pair_key[base + q] = raw[q];
        return;
    }
    // ---- sort by (atom, translation): the keys are distinct ----
    volatile unsigned long long* sorted = in_smem ? s_raw[wid] : pair_key + base;
    bool self_in = false;
    if (in_smem) {
        // Buckets of equal width between the smallest and the largest atom: one or two keys each as a rule, which are
        // ranked within their bucket (a rank sort over all k keys takes k^2 / 32 steps of a warp: 110 against 39 us for
        // the kernel on 3000 centres of 274 pairs, 16.8 against 14.6 us with 68 pairs each)
        unsigned long long* const raw = s_raw[wid];
        unsigned long long* const grouped = s_sorted[wid];
        int* const bucket_at = s_bucket[wid];
        unsigned lo = 0xffffffffu, hi = 0;
        for (int q = lane; q < k; q += 32) {
            const unsigned a = (unsigned)(raw[q] >> 24);
            lo = min(lo, a); hi = max(hi, a);
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        const float scale = (float)BUCKETS / (float)(hi - lo + 1u);                   // conversion and product keep the order
        auto bucket_of = [&](unsigned long long key) { return min(BUCKETS - 1, (int)((float)((unsigned)(key >> 24) - lo) * scale)); };
        constexpr int PER_LANE = BUCKETS / 32;
        int4* const mine = reinterpret_cast<int4*>(bucket_at) + lane * (PER_LANE / 4);
#pragma unroll
        for (int v = 0; v < PER_LANE / 4; ++v) mine[v] = make_int4(0, 0, 0, 0);
        __syncwarp();
        for (int q = lane; q < k; q += 32) atomicAdd(&bucket_at[bucket_of(raw[q])], 1);
        __syncwarp();
        int4 cnt[PER_LANE / 4];
        int sum = 0;
#pragma unroll
        for (int v = 0; v < PER_LANE / 4; ++v) { cnt[v] = mine[v]; sum += cnt[v].x + cnt[v].y + cnt[v].z + cnt[v].w; }
        int at = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += y;
        }
        at -= sum;
#pragma unroll
        for (int v = 0; v < PER_LANE / 4; ++v) {
            mine[v] = make_int4(at, at + cnt[v].x, at + cnt[v].x + cnt[v].y, at + cnt[v].x + cnt[v].y + cnt[v].z);
            at += cnt[v].x + cnt[v].y + cnt[v].z + cnt[v].w;
        }
        __syncwarp();
        for (int q = lane; q < k; q += 32) {
            const unsigned long long key = raw[q];
            grouped[atomicAdd(&bucket_at[bucket_of(key)], 1)] = key;
        }
        __syncwarp();                                                                  // bucket b now ends at bucket_at[b]
        for (int q = lane; q < k; q += 32) {
            const unsigned long long key = grouped[q];
            const int b = bucket_of(key), end = bucket_at[b];
            int rank = b > 0 ? bucket_at[b - 1] : 0;
            for (int r = rank; r < end; ++r) rank += grouped[r] < key;
            raw[rank] = key;
            self_in |= key_atom(key) == i;
        }
    } else {
        const volatile unsigned long long* raw = pair_tmp + base;
        for (int q = lane; q < k; q += 32) {
            const unsigned long long key = raw[q];
            int rank = 0;
            for (int r = 0; r < k; ++r) rank += raw[r] < key;
            sorted[rank] = key;
            self_in |= key_atom(key) == i;
        }
    }
    self_in = __any_sync(0xffffffffu, self_in);
    __syncwarp();
    // distinct atoms -> local Jacobian rows; the centre's own row sits in atom order
    int uniq = 0, below = 0;
    for (int q0 = 0; q0 < k; q0 += 32) {
        const int q = q0 + lane;
        int atom = -1, prev = -2;
        if (q < k) {
            const unsigned long long key = sorted[q];
            if (in_smem) pair_key[base + q] = key;
            atom = key_atom(key);
            prev = q > 0 ? key_atom(sorted[q - 1]) : -1;
        }
        const bool isnew = q < k && atom != prev;
        const unsigned m = __ballot_sync(0xffffffffu, isnew);
        const int u = uniq + __popc(m & ((1u << lane) - 1)) + (isnew ? 1 : 0) - 1;   // index among distinct atoms
        if (q < k) {
            int row = u + ((!site && !self_in && atom > i) ? 1 : 0);
            if (!isnew) row |= kRowContinuation;
            if (atom == i) row |= kRowSelfImage;
            pair_row[base + q] = row;
        }
        below += __popc(__ballot_sync(0xffffffffu, isnew && atom < i));
        uniq += __popc(m);
    }
    if (lane == 0) {
        row_count[c] = uniq + ((site || self_in) ? 0 : 1);
        self_row[c] = site ? -1 : below;
    }
}

// Many independent non-periodic structures in one launch: atoms of all structures in one list,
// struct_ptr[b] .. struct_ptr[b+1]-1 the atoms of structure b, every atom a centre that sees only its own
// structure.  One warp per centre runs over the atoms of its structure (brute force: the structures
// this is for are small molecules, where the cutoff sphere holds most of the structure anyway), with the same
// exact fp64 test as the cell-list path; neighbours come out in ascending atom order, so nothing is sorted.
// Writes what pairs_kernel writes (keys with zero lattice translation) plus the species index of the centre.
__global__ void __launch_bounds__(kFillWarps * 32)
batch_pairs_kernel(const float* __restrict__ pos, const int* __restrict__ numbers, const int* __restrict__ z_lut,
                   int* __restrict__ species_idx, const long long* __restrict__ struct_ptr, long long n_structs,
                   long long N, double rc2, long long pair_capacity, unsigned long long* pair_key,
                   int* __restrict__ pair_row, long long* __restrict__ pair_start, int* __restrict__ pair_count,
                   int* __restrict__ row_count, int* __restrict__ self_row, Counters* counters) {
    grid_dependency_launch();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long i = blockIdx.x * (long long)kFillWarps + wid;
    if (i >= N) return;
    if (lane == 0) {
        const int z = numbers[i];
        int s = (z >= 0 && z < 128) ? z_lut[z] : -1;
        if (s < 0) { atomicOr(&counters->status, kStatusUnknownSpecies); s = 0; }
        species_idx[i] = s;
    }
    // the structure that holds atom i: last b with struct_ptr[b] <= i (no offsets: one structure, all atoms)
    long long a = 0, b = N;
    if (struct_ptr) {
        long long lo = 0, hi = n_structs;
        while (hi - lo > 1) {
            const long long mid = (lo + hi) >> 1;
            if (struct_ptr[mid] <= i) lo = mid; else hi = mid;
        }
        a = struct_ptr[lo];
        b = min(struct_ptr[lo + 1], N);
    }
    const double xi = pos[3 * i], yi = pos[3 * i + 1], zi = pos[3 * i + 2];
    auto inside = [&](long long j) {
        if (j >= b) return false;
        const double dx = __dsub_rn((double)pos[3 * j], xi), dy = __dsub_rn((double)pos[3 * j + 1], yi),
                     dz = __dsub_rn((double)pos[3 * j + 2], zi);
        const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        return d2 < rc2 && d2 > 0.0;
    };
    int k = 0, below = 0;
    for (long long j0 = a; j0 < b; j0 += 32) {
        const bool v = inside(j0 + lane);
        k += __popc(__ballot_sync(0xffffffffu, v));
        below += __popc(__ballot_sync(0xffffffffu, v && j0 + lane < i));
    }
    long long base = 0;
    if (lane == 0) base = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&counters->n_pairs), (unsigned long long)k);
    base = __shfl_sync(0xffffffffu, base, 0);
    const bool fits = base + k <= pair_capacity;
    if (lane == 0) {
        pair_start[i] = base;
        pair_count[i] = fits ? k : 0;
        row_count[i] = k + 1;                     // the neighbours and the centre itself
        self_row[i] = below;
        if (!fits) atomicOr(&counters->status, kStatusPairCapacity);
    }
    if (!fits) return;
    int at = 0;
    for (long long j0 = a; j0 < b; j0 += 32) {
        const long long j = j0 + lane;
        const bool v = inside(j);
        const unsigned m = __ballot_sync(0xffffffffu, v);
        if (v) {
            const int q = at + __popc(m & ((1u << lane) - 1));
            pair_key[base + q] = ((unsigned long long)j << 24) | (128ull << 16) | (128ull << 8) | 128ull;
            pair_row[base + q] = q + (j > i ? 1 : 0);        // rows in atom order, the centre's own among them
        }
        at += __popc(m);
    }
}

// The test 0 < |d|^2 < r_cut^2 on the raw fp32 inputs, every operation rounded to fp64 on its own: what a pair is.
__device__ inline bool inside_exact(const Geometry& geom, float4 pj, float xi, float yi, float zi) {
    const double dx = __dsub_rn((double)pj.x, (double)xi), dy = __dsub_rn((double)pj.y, (double)yi), dz = __dsub_rn((double)pj.z, (double)zi);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return d2 < geom.rc2 && d2 > 0.0;
}
// The same answer, decided in fp32 wherever that is safe: the fp32 value of |d|^2 is off by at most 5 roundings (each
// difference one, counted twice by the square; the square; two sums), 5 x 2^-24 of itself, and the differences are zero
// when the coordinates are equal and only then; a band of +-2^-20 around r_cut^2 goes to the exact test.
__device__ __forceinline__ bool inside(const Geometry& geom, float rc2_lo, float rc2_hi, float4 pj, float xi, float yi, float zi) {
    const float dx = pj.x - xi, dy = pj.y - yi, dz = pj.z - zi;
    const float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    if (d2 < rc2_lo) return dx != 0.f || dy != 0.f || dz != 0.f;
    return d2 < rc2_hi && inside_exact(geom, pj, xi, yi, zi);
}

// The whole search of one non-periodic structure of up to kBruteForceAtoms atoms with every atom a centre, in ONE launch
// of a thread-block cluster: every CTA holds all positions in shared memory, its warps take the centres of a contiguous
// range and run over all atoms (neighbours come out in atom order, nothing is sorted); the pair totals of the CTAs
// before it come from their shared memory, so segments and row pointers are written directly.  At these sizes a call
// is a handful of launches and nothing else (24 atoms: memset, pair kernel and row scan took 10.7 us, this takes
// 7.7 us).  Writes what pairs_kernel and rows_order_kernel write, except a launch order.
constexpr int kBruteThreads = 1024, kBruteWarps = kBruteThreads / 32, kBruteCtas = 8, kBrutePerWarp = 2;
constexpr int kBruteForceAtoms = kBruteWarps * kBruteCtas * kBrutePerWarp, kBrutePerCta = kBruteWarps * kBrutePerWarp;
__global__ void __launch_bounds__(kBruteThreads)
brute_kernel(const float* __restrict__ pos, const int* __restrict__ numbers, const int* __restrict__ z_lut, int* __restrict__ species_idx,
             int n, Geometry geom, long long pair_capacity, unsigned long long* __restrict__ pair_key, int* __restrict__ pair_row,
             long long* __restrict__ pair_start, int* __restrict__ pair_count, int* __restrict__ self_row,
             long long* __restrict__ row_ptr, Counters* counters, Counters* host) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ float4 s_atom[kBruteForceAtoms];
    __shared__ int s_count[kBrutePerCta], cta_total;
    grid_dependency_launch();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rank = (int)cluster.block_rank(), ctas = (int)cluster.num_blocks();
    const int per_cta = (n + ctas - 1) / ctas, c_lo = min(n, rank * per_cta), c_hi = min(n, c_lo + per_cta);
    for (int i = tid; i < n; i += kBruteThreads) s_atom[i] = make_float4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], 0.f);
    if (c_lo + tid < c_hi) {
        const int z = numbers[c_lo + tid];
        int s = (z >= 0 && z < 128) ? z_lut[z] : -1;
        if (s < 0) { atomicOr(&counters->status, kStatusUnknownSpecies); s = 0; }
        species_idx[c_lo + tid] = s;
    }
    if (tid < kBrutePerCta) s_count[tid] = 0;
    __syncthreads();
    // ---- who sees whom: lane t of a warp keeps the mask of the atoms 32 t .. 32 t + 31 ----
    const float rc2_lo = (float)geom.rc2 * (1.f - 0x1p-20f), rc2_hi = (float)geom.rc2 * (1.f + 0x1p-20f);
    unsigned mask[kBrutePerWarp];
#pragma unroll
    for (int k = 0; k < kBrutePerWarp; ++k) {
        const int i = c_lo + wid + k * kBruteWarps;
        mask[k] = 0;
        if (i < c_hi) {
            const float4 pi = s_atom[i];
            int count = 0;
            for (int t = 0; 32 * t < n; ++t) {
                const int j = 32 * t + lane;
                const unsigned m = __ballot_sync(0xffffffffu, j < n && inside(geom, rc2_lo, rc2_hi, s_atom[j], pi.x, pi.y, pi.z));
                if (lane == t) mask[k] = m;
                count += __popc(m);
            }
            if (lane == 0) s_count[i - c_lo] = count;
        }
    }
    __syncthreads();
    // ---- first pair of every centre: exclusive scan over this CTA's centres, on top of the CTAs before it ----
    if (wid == 0) {
        constexpr int PER_LANE = kBrutePerCta / 32;
        int v[PER_LANE], sum = 0;
#pragma unroll
        for (int k = 0; k < PER_LANE; ++k) { v[k] = s_count[lane * PER_LANE + k]; sum += v[k]; }
        int at = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += y;
        }
        if (lane == 31) cta_total = at;
        at -= sum;
#pragma unroll
        for (int k = 0; k < PER_LANE; ++k) { s_count[lane * PER_LANE + k] = at; at += v[k]; }
    }
    cluster.sync();
    int before = 0, total = 0;
    for (int r = 0; r < ctas; ++r) {
        const int v = *cluster.map_shared_rank(&cta_total, r);
        if (r < rank) before += v;
        total += v;
    }
    cluster.sync();                                                          // nobody reads this CTA's shared memory any more
    const bool fits = total <= pair_capacity;
    if (rank == 0 && tid == 0) {
        if (!fits) atomicOr(&counters->status, kStatusPairCapacity);
        counters->n_pairs = total;
        counters->n_rows = total + n;                                        // the neighbours and the centres themselves
        row_ptr[n] = total + n;
        if (host) { __threadfence(); *host = *counters; }                    // pinned host memory: the caller waits for the stream and reads it
    }
#pragma unroll
    for (int k = 0; k < kBrutePerWarp; ++k) {
        const int i = c_lo + wid + k * kBruteWarps;
        if (i >= c_hi) continue;
        const int base = before + s_count[i - c_lo];
        int at = base, below = 0;
        for (int t = 0; 32 * t < n; ++t) {
            const unsigned m = __shfl_sync(0xffffffffu, mask[k], t);
            const int j = 32 * t + lane;
            if (fits && (m >> lane & 1)) {
                const int q = at + __popc(m & ((1u << lane) - 1));
                pair_key[q] = ((unsigned long long)j << 24) | 0x808080ull;
                pair_row[q] = q - base + (j > i ? 1 : 0);                    // rows in atom order, the centre's own among them
            }
            at += __popc(m);
            below += __popc(__ballot_sync(0xffffffffu, (m >> lane & 1) && j < i));
        }
        if (lane == 0) {
            pair_start[i] = base;
            pair_count[i] = fits ? at - base : 0;
            row_ptr[i] = base + i;
            self_row[i] = below;
        }
    }
}

// One cluster: exclusive scan of the row counts (rows of centre c start at row_ptr[c]), the totals to the host if it
// asks for them, and the launch order of the per-centre kernel, largest pair count first (bins of 4 pairs, counting
// sort), so that the long CTAs do not end up alone at the tail of the launch.  Every CTA takes a contiguous range of
// centres; sums and bin counts of the others come from their shared memory.  Up to kRowsPerCta centres one CTA does it,
// above that eight (36,000 centres: 46 us with one, 13 us with eight).
constexpr int kSizeBins = 256, kSizeBinShift = 2;
constexpr int kRowsCtas = 8, kRowsPerThread = 8, kRowsPerCta = 4096;
// Sum: what holds the rows of a CTA's centres (launch_neighbors: 64 bits where centres times atoms say that 32 do not do).
template <typename Sum>
__global__ void __launch_bounds__(1024)
rows_order_kernel(const int* __restrict__ row_count, const int* __restrict__ pair_count, int C,
                  long long* __restrict__ row_ptr, int* __restrict__ order, Counters* counters, Counters* host) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ Sum warp_sums[32], cta_sum;
    __shared__ int hist[kSizeBins], total[kSizeBins], first_slot[kSizeBins];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rank = (int)cluster.block_rank(), ctas = (int)cluster.num_blocks();
    grid_dependency_launch();
    if (tid < kSizeBins) hist[tid] = 0;
    // a contiguous range per CTA, consecutive centres per thread
    const int per_cta = (C + ctas - 1) / ctas, per_thread = (per_cta + 1023) / 1024;       // at most kRowsPerThread
    const int c_hi = min(C, (rank + 1) * per_cta), i0 = rank * per_cta + tid * per_thread;
    grid_dependency_wait();                                                  // the counts of the pair kernel
    __syncthreads();
    int v[kRowsPerThread], bin[kRowsPerThread];
    Sum mine = 0;
#pragma unroll
    for (int k = 0; k < kRowsPerThread; ++k) {
        v[k] = bin[k] = 0;
        if (k < per_thread && i0 + k < c_hi) {
            v[k] = row_count[i0 + k];
            bin[k] = min(pair_count[i0 + k] >> kSizeBinShift, kSizeBins - 1);
            atomicAdd(&hist[bin[k]], 1);
        }
        mine += v[k];
    }
    Sum incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const Sum y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        Sum w = warp_sums[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const Sum y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;
        if (lane == 31) cta_sum = w;
    }
    int before = 0;                                                          // centres of this thread's bin in the CTAs before this one
    long long base = 0, rows = 0;                                            // rows of the CTAs before this one, of all
    if (ctas > 1) {
        cluster.sync();
        if (tid < kSizeBins) {
            int all = 0;
            for (int r = 0; r < ctas; ++r) {
                const int h = cluster.map_shared_rank(hist, r)[tid];
                if (r < rank) before += h;
                all += h;
            }
            total[tid] = all;
        }
        for (int r = 0; r < ctas; ++r) {
            const Sum t = *cluster.map_shared_rank(&cta_sum, r);
            if (r < rank) base += t;
            rows += t;
        }
        cluster.sync();                                                      // (also: nobody reads this CTA's shared memory any more)
    } else {
        __syncthreads();
        rows = cta_sum;
    }
    if (rank == 0 && tid == 1023) {
        row_ptr[C] = rows;
        counters->n_rows = rows;
        if (host) *host = *counters;                                         // pinned host memory: the caller waits for the stream and reads it
    }
    if (wid == 0) {
        // first slot of every size bin, largest bin first: lane k scans the bins 255 - 8k down to 248 - 8k, a warp
        // scan adds what the lanes before it hold
        constexpr int per_lane = kSizeBins / 32;
        const int* const count = ctas > 1 ? total : hist;
        const int top = kSizeBins - 1 - lane * per_lane;
        int sum = 0;
        for (int k = 0; k < per_lane; ++k) sum += count[top - k];
        int at = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += y;
        }
        int run = at - sum;
        for (int k = 0; k < per_lane; ++k) { first_slot[top - k] = run; run += count[top - k]; }
    }
    __syncthreads();
    if (ctas > 1) {
        if (tid < kSizeBins) first_slot[tid] += before;
        __syncthreads();
    }
    long long at = base + (wid > 0 ? warp_sums[wid - 1] : 0) + incl - mine;
#pragma unroll
    for (int k = 0; k < kRowsPerThread; ++k) {
        if (k < per_thread && i0 + k < c_hi) {
            row_ptr[i0 + k] = at;
            order[atomicAdd(&first_slot[bin[k]], 1)] = i0 + k;
        }
        at += v[k];
    }
}

// Compact copy of the pair list (the pair arrays are addressed by segment): one warp per centre.
__global__ void export_pairs_kernel(const long long* __restrict__ pair_start, const long long* __restrict__ out_ptr,
                                    const unsigned long long* __restrict__ pair_key, long long C, long long capacity,
                                    int* out_atom, int* out_shift, Counters* counters) {
    if (out_ptr[C] > capacity) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&counters->status, kStatusPairCapacity);
        return;
    }
    const int lane = threadIdx.x & 31;
    for (long long c = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; c < C; c += ((long long)gridDim.x * blockDim.x) >> 5) {
        const long long src = pair_start[c], dst = out_ptr[c];
        const int k = (int)(out_ptr[c + 1] - dst);
        for (int q = lane; q < k; q += 32) {
            const unsigned long long key = pair_key[src + q];
            out_atom[dst + q] = key_atom(key);
            if (out_shift) {
                int sft[3];
                key_shift(key, sft);
                out_shift[3 * (dst + q)] = sft[0]; out_shift[3 * (dst + q) + 1] = sft[1]; out_shift[3 * (dst + q) + 2] = sft[2];
            }
        }
    }
}

}  // namespace soap
