// Launches of whole steps of mixed runs, n_states 15..18.
#include "resident.cuh"

namespace heom {

const void *mixed_run_kernel_c(int n) {
  switch (n) {
    case 15: return (const void *)el_run_kernel<kRunMixed, true, 15>;
    case 16: return (const void *)el_run_kernel<kRunMixed, true, 16>;
    case 17: return (const void *)el_run_kernel<kRunMixed, true, 17>;
    case 18: return (const void *)el_run_kernel<kRunMixed, true, 18>;
    default: return nullptr;
  }
}

}  // namespace heom
