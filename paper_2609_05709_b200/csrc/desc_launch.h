// Dispatch of the descriptor-only kernel over its compile-time l_max (0..12) and padded n_max (4, 8, 12, 16).
#pragma once
#include "soap_device.cuh"

namespace soap {
using DescKernel = void (*)(CenterParams);
// plain: every option at its default (see desc_kernel); table_in_smem: the radial table is staged per CTA; team: a CTA per
// centre; search: a team that looks for its neighbours itself.  Null where there is none.  (It waits on the device for the kernel
// before it: launch it with launch_dependent, launch and table staging overlap that kernel's tail.)
DescKernel desc_kernel_of(int l_max, int np, bool plain, bool table_in_smem, bool team, bool search);

// compiled, and loaded, apart for the two values of `plain`
#define SOAP_DECLARE_L(LV)                                                                      \
    DescKernel desc_kernel_l##LV##_f0(int np, bool table_in_smem, bool team, bool search);         \
    DescKernel desc_kernel_l##LV##_f1(int np, bool table_in_smem, bool team, bool search);
SOAP_DECLARE_L(0) SOAP_DECLARE_L(1) SOAP_DECLARE_L(2) SOAP_DECLARE_L(3) SOAP_DECLARE_L(4) SOAP_DECLARE_L(5) SOAP_DECLARE_L(6)
SOAP_DECLARE_L(7) SOAP_DECLARE_L(8) SOAP_DECLARE_L(9) SOAP_DECLARE_L(10) SOAP_DECLARE_L(11) SOAP_DECLARE_L(12)
#undef SOAP_DECLARE_L
}  // namespace soap
