// Every instantiation of the descriptor-only kernel for one l_max, PLAIN (SOAP_FAMILY 0) or with options (1): compiled once
// per value of SOAP_L (0..12) and SOAP_FAMILY, which the build passes on the command line.
#if !defined(SOAP_L) || !defined(SOAP_FAMILY)
#error "compile with -DSOAP_L=<l_max> -DSOAP_FAMILY=<0..1>"
#endif
#include "desc_kernel.cuh"
#include "desc_launch.h"

namespace soap {

#define SOAP_CAT2(a, b, c, d) a##b##c##d
#define SOAP_CAT(a, b, c, d) SOAP_CAT2(a, b, c, d)

// a warp per centre with the table in shared memory or in global memory, or a team of warps per centre, which may search itself
template <int NP>
static DescKernel of_np(bool ts, bool team, bool search) {
    constexpr bool PLAIN = SOAP_FAMILY == 0;
    if (search) return desc_kernel<SOAP_L, NP, PLAIN, false, true, true>;
    if (team) return desc_kernel<SOAP_L, NP, PLAIN, false, true, false>;
    if (ts) return desc_kernel<SOAP_L, NP, PLAIN, true, false, false>;
    return desc_kernel<SOAP_L, NP, PLAIN, false, false, false>;
}

DescKernel SOAP_CAT(desc_kernel_l, SOAP_L, _f, SOAP_FAMILY)(int np, bool ts, bool team, bool search) {
    switch (np) {
        case 4: return of_np<4>(ts, team, search);
        case 8: return of_np<8>(ts, team, search);
        case 12: return of_np<12>(ts, team, search);
        case 16: return of_np<16>(ts, team, search);
    }
    return nullptr;
}

}  // namespace soap
