// Instantiations of the work-list stage kernel (FP32 bodies of mixed runs), n_states 9..16.
#include "stage_list.cuh"

namespace heom {

int launch_stage_list_b(int n, const ListLaunch &L, cudaStream_t st, int sm_count) {
  switch (n) {
    case 9: return launch_list_n<9>(L, st, sm_count);
    case 10: return launch_list_n<10>(L, st, sm_count);
    case 11: return launch_list_n<11>(L, st, sm_count);
    case 12: return launch_list_n<12>(L, st, sm_count);
    case 13: return launch_list_n<13>(L, st, sm_count);
    case 14: return launch_list_n<14>(L, st, sm_count);
    case 15: return launch_list_n<15>(L, st, sm_count);
    case 16: return launch_list_n<16>(L, st, sm_count);
    default:
      return 1;  // not in this translation unit
  }
}

}  // namespace heom
