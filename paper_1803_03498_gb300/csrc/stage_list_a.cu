// Instantiations of the work-list stage kernel (FP32 bodies of mixed runs), n_states 1..8.
#include "stage_list.cuh"

namespace heom {

int launch_stage_list_a(int n, const ListLaunch &L, cudaStream_t st, int sm_count) {
  switch (n) {
    case 1: return launch_list_n<1>(L, st, sm_count);
    case 2: return launch_list_n<2>(L, st, sm_count);
    case 3: return launch_list_n<3>(L, st, sm_count);
    case 4: return launch_list_n<4>(L, st, sm_count);
    case 5: return launch_list_n<5>(L, st, sm_count);
    case 6: return launch_list_n<6>(L, st, sm_count);
    case 7: return launch_list_n<7>(L, st, sm_count);
    case 8: return launch_list_n<8>(L, st, sm_count);
    default:
      return 1;  // not in this translation unit
  }
}

}  // namespace heom
