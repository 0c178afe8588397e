// Instantiations of the work-list stage kernel (FP32 bodies of mixed runs), n_states 17..24.
#include "stage_list.cuh"

namespace heom {

int launch_stage_list_c(int n, const ListLaunch &L, cudaStream_t st, int sm_count) {
  switch (n) {
    case 17: return launch_list_n<17>(L, st, sm_count);
    case 18: return launch_list_n<18>(L, st, sm_count);
    case 19: return launch_list_n<19>(L, st, sm_count);
    case 20: return launch_list_n<20>(L, st, sm_count);
    case 21: return launch_list_n<21>(L, st, sm_count);
    case 22: return launch_list_n<22>(L, st, sm_count);
    case 23: return launch_list_n<23>(L, st, sm_count);
    case 24: return launch_list_n<24>(L, st, sm_count);
    default:
      return 1;  // not in this translation unit
  }
}

}  // namespace heom
