// Dispatch of the per-centre kernel over its compile-time l_max (0..12) and n_max.
#pragma once
#include "soap_device.cuh"

namespace soap {
// kernel kinds: descriptor and Jacobian; coefficients c^mu_nlm and their Jacobian; Jacobian of the inner average;
// Jacobian of the outer average (the last two: every atom a centre, one row per atom)
constexpr int kCenterDeriv = 1, kCenterCoeff = 2, kCenterInner = 3, kCenterOuter = 4;
// Families of kernels that are compiled, and loaded when one of them is first launched, together (loading all of l_max 6 at
// once takes 22 ms, whatever the call needs of them): kind 1 as PLAIN and with options, kind 2, kinds 3 and 4.
constexpr int kFamilyPlain = 0, kFamilyOptions = 1, kFamilyCoeff = 2, kFamilyAverage = 3;
// whether the parameters ask for nothing beyond the default configuration (the kernels instantiated with
// PLAIN = true assume exactly this)
inline bool center_params_plain(const CenterParams& p) {
    return p.crossover && !p.compact && !p.emit_coeff && !p.c_bar && !p.sites && !p.pair_w && p.w0 == 1.f && !p.inner_rows && !p.c_all;
}
using CenterKernel = void (*)(CenterParams);
// The kernel of a kind (plain: kind 1 only), null where there is none.  It waits on the device for the kernel before it (the
// row scan, as a rule): launch it with launch_dependent, its launch and its set-up overlap that kernel's tail.
CenterKernel center_kernel_of(int kind, bool plain, int l_max, int n_max);

#define SOAP_DECLARE_L(LV)                                                                                                        \
    CenterKernel center_kernel_l##LV##_f0(int kind, int n_max); CenterKernel center_kernel_l##LV##_f1(int kind, int n_max);       \
    CenterKernel center_kernel_l##LV##_f2(int kind, int n_max); CenterKernel center_kernel_l##LV##_f3(int kind, int n_max);
SOAP_DECLARE_L(0) SOAP_DECLARE_L(1) SOAP_DECLARE_L(2) SOAP_DECLARE_L(3) SOAP_DECLARE_L(4) SOAP_DECLARE_L(5) SOAP_DECLARE_L(6)
SOAP_DECLARE_L(7) SOAP_DECLARE_L(8) SOAP_DECLARE_L(9) SOAP_DECLARE_L(10) SOAP_DECLARE_L(11) SOAP_DECLARE_L(12)
#undef SOAP_DECLARE_L
}  // namespace soap
