// Every instantiation of the fused per-centre derivative kernels for one l_max and one family (center_launch.h): compiled
// once per value of SOAP_L (0..12) and SOAP_FAMILY (0..3), which the build passes on the command line.
#if !defined(SOAP_L) || !defined(SOAP_FAMILY)
#error "compile with -DSOAP_L=<l_max> -DSOAP_FAMILY=<0..3>"
#endif
#include "center_kernel.cuh"
#include "center_launch.h"

namespace soap {

#define SOAP_CAT2(a, b, c, d) a##b##c##d
#define SOAP_CAT(a, b, c, d) SOAP_CAT2(a, b, c, d)

// The kernels have an instantiation of their own for the usual n_max: loops over n unroll, the accumulators of pass 1
// fit the registers exactly.  The variant that reads n_max at run time spills 0.6 kB and serves what is left (n_max 1
// and 13 to 16, and the largest l_max, whose kernels take longest to compile).  Measured, run time against compile time:
// (n_max, l_max) = (5, 5) on 1021 centres 254 -> 159 us, (6, 6) with a weighting and compact rows on 1111 centres
// 368 -> 270 us, whole calls of the other sizes 1.2 to 1.7 times faster.
#if SOAP_L <= 10
#define SOAP_FOR_FIXED_NMAX(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12)
#elif SOAP_L == 12
#define SOAP_FOR_FIXED_NMAX(X) X(2) X(4) X(6) X(7) X(8) X(10) X(12)
#else
#define SOAP_FOR_FIXED_NMAX(X) X(4) X(8)
#endif
#if SOAP_L <= 8
#define SOAP_FOR_GENERAL_NMAX(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(10) X(12)
#elif SOAP_L <= 10
#define SOAP_FOR_GENERAL_NMAX(X) X(4) X(6) X(8) X(10) X(12)
#else
#define SOAP_FOR_GENERAL_NMAX(X) X(8)
#endif
#if SOAP_L % 2 == 0 || SOAP_L == 3
#define SOAP_FOR_COEFF_NMAX(X) X(4) X(8)
#else
#define SOAP_FOR_COEFF_NMAX(X) X(8)
#endif

#if SOAP_L <= 8
#define SOAP_FOR_AVERAGE_NMAX(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9)
#else
#define SOAP_FOR_AVERAGE_NMAX(X) X(8)
#endif

CenterKernel SOAP_CAT(center_kernel_l, SOAP_L, _f, SOAP_FAMILY)(int kind, int n_max) {
    (void)kind;
#if SOAP_FAMILY == 0
    switch (n_max) {
#define X(N) case N: return center_kernel<1, SOAP_L, N, true>;
        SOAP_FOR_FIXED_NMAX(X)
#undef X
    }
    return center_kernel<1, SOAP_L, 0, true>;
#elif SOAP_FAMILY == 1
    switch (n_max) {
#define X(N) case N: return center_kernel<1, SOAP_L, N, false>;
        SOAP_FOR_GENERAL_NMAX(X)
#undef X
    }
    return center_kernel<1, SOAP_L, 0, false>;
#elif SOAP_FAMILY == 2
    switch (n_max) {
#define X(N) case N: return center_kernel<2, SOAP_L, N, false>;
        SOAP_FOR_COEFF_NMAX(X)
#undef X
    }
    return center_kernel<2, SOAP_L, 0, false>;
#else
    if (kind == kCenterInner) {
        switch (n_max) {
#define X(N) case N: return center_kernel<3, SOAP_L, N, false>;
            SOAP_FOR_AVERAGE_NMAX(X)
#undef X
        }
        return center_kernel<3, SOAP_L, 0, false>;
    }
    switch (n_max) {
#define X(N) case N: return center_kernel<4, SOAP_L, N, false>;
        SOAP_FOR_AVERAGE_NMAX(X)
#undef X
    }
    return center_kernel<4, SOAP_L, 0, false>;
#endif
}

}  // namespace soap
