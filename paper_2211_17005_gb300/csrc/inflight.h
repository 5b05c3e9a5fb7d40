// Bounded waits for the copies that one thread issues on B mbarriers in turn: copy u completes
// phase u / B of barrier u % B. A barrier's parity tells two neighbouring phases apart and no
// more, so at most one copy may be in flight per barrier. After a wait that gave up, the issuer
// therefore requests nothing more, and before it leaves it waits once more, in full, for all it
// has in flight: no copy outlives its CTA.
//
// Plain C++, so that the protocol can be run on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define CVA_HD __host__ __device__ __forceinline__
#else
#define CVA_HD inline
#endif

namespace cva {

// The second wait, by wait(barrier, parity): of the copies issued so far the last B may be in
// flight.
template <uint32_t B, class Wait>
CVA_HD void settle_copies(uint32_t issued, Wait wait)
{
    for (uint32_t v = issued > B ? issued - B : 0u; v < issued; ++v) (void)wait(v % B, (v / B) & 1u);
}

}  // namespace cva
