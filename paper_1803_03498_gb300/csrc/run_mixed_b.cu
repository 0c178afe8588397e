// Launches of whole steps of mixed runs, n_states 9..14.
#include "resident.cuh"

namespace heom {

const void *mixed_run_kernel_b(int n) {
  switch (n) {
    case 9: return (const void *)el_run_kernel<kRunMixed, true, 9>;
    case 10: return (const void *)el_run_kernel<kRunMixed, true, 10>;
    case 11: return (const void *)el_run_kernel<kRunMixed, true, 11>;
    case 12: return (const void *)el_run_kernel<kRunMixed, true, 12>;
    case 13: return (const void *)el_run_kernel<kRunMixed, true, 13>;
    case 14: return (const void *)el_run_kernel<kRunMixed, true, 14>;
    default: return nullptr;
  }
}

}  // namespace heom
