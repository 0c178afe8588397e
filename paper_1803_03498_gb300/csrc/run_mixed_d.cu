// Launches of whole steps of mixed runs, n_states 20..24.
#include "resident.cuh"

namespace heom {

const void *mixed_run_kernel_d(int n) {
  switch (n) {
    case 20: return (const void *)el_run_kernel<kRunMixed, true, 20>;
    case 21: return (const void *)el_run_kernel<kRunMixed, true, 21>;
    case 22: return (const void *)el_run_kernel<kRunMixed, true, 22>;
    case 23: return (const void *)el_run_kernel<kRunOther, true, 23>;
    case 24: return (const void *)el_run_kernel<kRunOther, true, 24>;
    default: return nullptr;
  }
}

}  // namespace heom
