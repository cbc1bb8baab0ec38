// Every instantiation of the fused per-centre derivative kernels for one l_max: compiled once per value of
// SOAP_L (0..12), which the build passes on the command line.
#ifndef SOAP_L
#error "compile with -DSOAP_L=<l_max>"
#endif
#include "center_kernel.cuh"
#include "center_launch.h"

namespace soap {

#define SOAP_CAT2(a, b) a##b
#define SOAP_CAT(a, b) SOAP_CAT2(a, b)

// Fills this translation unit's constant tables (once per process and device is enough;
// it is cheap, so it runs whenever a handle sets up its kernels).
cudaError_t SOAP_CAT(center_constants_l, SOAP_L)(const float* anorm91, const float* dfact16) {
    // norm: (a_lm, (l+m) a_lm);  step: ((2l+1)/(l+1-m), (l+m)/(l+1-m)) for column m and
    // ((2l+1)/(l-m), (l+m+1)/(l-m)) for column m+1 (unused at l = m)
    float2 norm[91];
    float4 step[91];
    for (int l = 0; l <= 12; ++l)
        for (int m = 0; m <= l; ++m) {
            const int t = l * (l + 1) / 2 + m;
            norm[t] = make_float2(anorm91[t], (float)(l + m) * anorm91[t]);
            step[t].x = (float)(2 * l + 1) / (float)(l + 1 - m);
            step[t].y = (float)(l + m) / (float)(l + 1 - m);
            step[t].z = l > m ? (float)(2 * l + 1) / (float)(l - m) : 0.f;
            step[t].w = l > m ? (float)(l + m + 1) / (float)(l - m) : 0.f;
        }
    cudaError_t e = cudaMemcpyToSymbol(kc_norm, norm, sizeof(norm));
    if (e != cudaSuccess) return e;
    e = cudaMemcpyToSymbol(kc_step, step, sizeof(step));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(kc_dfact, dfact16, 16 * sizeof(float));
}

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

using Kernel = void (*)(CenterParams);

static Kernel kernel_of(int kind, int n_max, bool plain) {
    if (kind == kCenterInner) {
        switch (n_max) {
#define X(N) case N: return center_kernel<3, SOAP_L, N, false>;
            SOAP_FOR_AVERAGE_NMAX(X)
#undef X
        }
        return center_kernel<3, SOAP_L, 0, false>;
    }
    if (kind == kCenterOuter) {
        switch (n_max) {
#define X(N) case N: return center_kernel<4, SOAP_L, N, false>;
            SOAP_FOR_AVERAGE_NMAX(X)
#undef X
        }
        return center_kernel<4, SOAP_L, 0, false>;
    }
    if (kind == kCenterCoeff) {
        switch (n_max) {
#define X(N) case N: return center_kernel<2, SOAP_L, N, false>;
            SOAP_FOR_COEFF_NMAX(X)
#undef X
        }
        return center_kernel<2, SOAP_L, 0, false>;
    }
    if (!plain) {
        switch (n_max) {
#define X(N) case N: return center_kernel<1, SOAP_L, N, false>;
            SOAP_FOR_GENERAL_NMAX(X)
#undef X
        }
        return center_kernel<1, SOAP_L, 0, false>;
    }
    switch (n_max) {
#define X(N) case N: return center_kernel<1, SOAP_L, N, true>;
        SOAP_FOR_FIXED_NMAX(X)
#undef X
    }
    return center_kernel<1, SOAP_L, 0, true>;
}

// The dynamic shared memory that every kernel of this kind and n_max may be launched with.
cudaError_t SOAP_CAT(center_set_smem_l, SOAP_L)(int kind, int n_max, int bytes) {
    for (const bool plain : {false, true}) {
        const cudaError_t e = cudaFuncSetAttribute(kernel_of(kind, n_max, plain), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The kernel waits on the device for the kernel before it (the row scan, as a rule): its launch and its set-up overlap
// that kernel's tail.
cudaError_t SOAP_CAT(center_launch_l, SOAP_L)(int kind, int n_max, bool plain, int threads, const CenterParams& p, unsigned grid, size_t smem,
                                              cudaStream_t st) {
    return launch_dependent(kernel_of(kind, n_max, plain), grid, threads, smem, st, p);
}

}  // namespace soap
