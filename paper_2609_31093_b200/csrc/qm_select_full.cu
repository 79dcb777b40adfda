// Selection over every level from the dense scoring's tables (see qm_select.cuh).
#include "qm_select.cuh"

namespace pisa {

int launch_qm_select_full(const Geometry& g, const qm::Args& a, long long rows, int32_t* idx, float* margin, float* lse,
                          float* sel_lse, cudaStream_t s) {
  SelArgs sa = {};
  sa.idx = idx; sa.margin = margin; sa.lse = lse; sa.sel_lse = sel_lse;
  return launch_sel_mode<kSelFull>(g, a, sa, rows, s);
}

}  // namespace pisa
