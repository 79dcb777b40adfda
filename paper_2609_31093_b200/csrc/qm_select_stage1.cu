// Selection down to level 2: the kept level-2 nodes (see qm_select.cuh).
#include "qm_select.cuh"

namespace pisa {

int launch_qm_select_stage1(const Geometry& g, const qm::Args& a, long long rows, int32_t* par, float* margin, cudaStream_t s) {
  SelArgs sa = {};
  sa.par = par; sa.margin = margin;
  return launch_sel_mode<kSelStage1>(g, a, sa, rows, s);
}

}  // namespace pisa
