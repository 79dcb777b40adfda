// Selection among the children of the kept level-2 nodes (see qm_select.cuh).
#include "qm_select.cuh"

namespace pisa {

int launch_qm_select_final(const Geometry& g, const qm::Args& a, long long rows, const int32_t* par, const float* blk,
                           int32_t* idx, float* margin, float* lse, float* sel_lse, cudaStream_t s) {
  SelArgs sa = {};
  sa.par = const_cast<int32_t*>(par); sa.blk = blk; sa.idx = idx; sa.margin = margin; sa.lse = lse; sa.sel_lse = sel_lse;
  return launch_sel_mode<kSelFinal>(g, a, sa, rows, s);
}

}  // namespace pisa
