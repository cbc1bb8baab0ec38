// Constants of the real solid harmonics up to l = 12, built by the compiler: a kernel's constant memory holds them when it is
// loaded, so that setting up a handle loads no kernels to fill it.
#pragma once

namespace soap {

constexpr int kHarmonicL = 12, kHarmonicTerms = (kHarmonicL + 1) * (kHarmonicL + 2) / 2;      // (l, m), 0 <= m <= l: index l(l+1)/2 + m

// square root by Heron's iteration, to the last bits of a double (x > 0; the iterates fall from the second one on)
constexpr double heron_sqrt(double x) {
    double r = x > 1.0 ? x : 1.0, next = 0.5 * (r + x / r);
    while (next < r) { r = next; next = 0.5 * (r + x / r); }
    return r;
}

struct HarmonicTables {
    float norm[kHarmonicTerms];          // a_lm = sqrt((2l+1)/4pi (l-m)!/(l+m)!), times sqrt2 for m > 0
    float norm_lm[kHarmonicTerms];       // (l+m) a_lm
    float step[kHarmonicTerms][4];       // coefficients that advance columns m and m+1 of the recursion from l to l+1
    float dfact[16];                     // (2m-1)!!
};

constexpr HarmonicTables harmonic_tables() {
    HarmonicTables t{};
    for (int l = 0; l <= kHarmonicL; ++l)
        for (int m = 0; m <= l; ++m) {
            const int i = l * (l + 1) / 2 + m;
            double ratio = m > 0 ? 2.0 : 1.0;
            for (int j = l - m + 1; j <= l + m; ++j) ratio /= j;
            t.norm[i] = (float)heron_sqrt((2 * l + 1) / (4.0 * 3.14159265358979323846) * ratio);
            t.norm_lm[i] = (float)(l + m) * t.norm[i];
            // ((2l+1)/(l+1-m), (l+m)/(l+1-m)) for column m and ((2l+1)/(l-m), (l+m+1)/(l-m)) for column m+1 (unused at l = m)
            t.step[i][0] = (float)(2 * l + 1) / (float)(l + 1 - m);
            t.step[i][1] = (float)(l + m) / (float)(l + 1 - m);
            t.step[i][2] = l > m ? (float)(2 * l + 1) / (float)(l - m) : 0.f;
            t.step[i][3] = l > m ? (float)(l + m + 1) / (float)(l - m) : 0.f;
        }
    double df = 1.0;
    for (int m = 0; m <= kHarmonicL; ++m) {
        if (m > 0) df *= 2 * m - 1;
        t.dfact[m] = (float)df;
    }
    return t;
}

}  // namespace soap
