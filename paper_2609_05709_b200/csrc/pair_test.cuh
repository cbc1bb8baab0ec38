// What a pair is: the test that every neighbour search with periodic images applies to a candidate.
#pragma once
#include "soap_device.cuh"

namespace soap {

__device__ inline void frac_coords(const Geometry& g, float x, float y, float z, double s[3]) {
    for (int a = 0; a < 3; ++a)
        s[a] = (double)x * g.inv[0 + a] + (double)y * g.inv[3 + a] + (double)z * g.inv[6 + a];
}

// Squared distance of the atom pj, translated by (na, nb, nc) cells, from the centre.  Every operation is rounded to fp64 on its
// own, on the raw fp32 inputs.
__device__ __forceinline__ double pair_distance2(const Geometry& geom, bool any_periodic, float4 pj, int na, int nb, int nc, float xi, float yi, float zi) {
    double dx = __dsub_rn((double)pj.x, (double)xi);
    double dy = __dsub_rn((double)pj.y, (double)yi);
    double dz = __dsub_rn((double)pj.z, (double)zi);
    if (any_periodic) {
        // T = (n_a a + n_b b) + n_c c, each product and sum rounded on its own
        const double fa = (double)na, fb = (double)nb, fc = (double)nc;
        double tx = __dadd_rn(__dadd_rn(__dmul_rn(fa, geom.cell[0]), __dmul_rn(fb, geom.cell[3])), __dmul_rn(fc, geom.cell[6]));
        double ty = __dadd_rn(__dadd_rn(__dmul_rn(fa, geom.cell[1]), __dmul_rn(fb, geom.cell[4])), __dmul_rn(fc, geom.cell[7]));
        double tz = __dadd_rn(__dadd_rn(__dmul_rn(fa, geom.cell[2]), __dmul_rn(fb, geom.cell[5])), __dmul_rn(fc, geom.cell[8]));
        dx = __dadd_rn(dx, tx); dy = __dadd_rn(dy, ty); dz = __dadd_rn(dz, tz);
    }
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Inside the cutoff: 0 < d2 < r_cut^2 (an atom is no neighbour of itself, its images are).
__device__ __forceinline__ bool inside_cutoff(const Geometry& geom, double d2) { return (d2 < geom.rc2) && (d2 > 0.0); }

// Whether a neighbour is too many cells away for its key.
__device__ __forceinline__ bool beyond_key(int na, int nb, int nc) { return abs(na) > 127 || abs(nb) > 127 || abs(nc) > 127; }

// The pair's key: the atom's number (in pj.w) and its translation.
__device__ __forceinline__ unsigned long long pair_key_of(float4 pj, int na, int nb, int nc) {
    return ((unsigned long long)(unsigned)__float_as_int(pj.w) << 24) |
           ((unsigned long long)(na + 128) << 16) | ((unsigned long long)(nb + 128) << 8) |
           (unsigned long long)(nc + 128);
}

}  // namespace soap
