// Launches of whole steps of mixed runs, n_states 1..8.
#include "resident.cuh"

namespace heom {

const void *mixed_run_kernel_a(int n) {
  switch (n) {
    case 1: return (const void *)el_run_kernel<kRunMixed, false, 1>;
    case 2: return (const void *)el_run_kernel<kRunMixed, false, 2>;
    case 3: return (const void *)el_run_kernel<kRunMixed, false, 3>;
    case 4: return (const void *)el_run_kernel<kRunMixed, false, 4>;
    case 5: return (const void *)el_run_kernel<kRunMixed, false, 5>;
    case 6: return (const void *)el_run_kernel<kRunMixed, false, 6>;
    case 7: return (const void *)el_run_kernel<kRunMixed, false, 7>;
    case 8: return (const void *)el_run_kernel<kRunMixed, false, 8>;
    default: return nullptr;
  }
}

}  // namespace heom
