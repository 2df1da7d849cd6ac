// Instantiations of the fixed-point FP64 clover-inverse stencil (k_fx_clinv).
#include "fx.cuh"

namespace lq {

template <bool DAG, bool CLOV>
static int pick(int epi, dim3 gr, const FxArgs& m, cudaStream_t st) {
  if (epi == EPI_X) k_fx_clinv<DAG, CLOV, EPI_X><<<gr, 128, 0, st>>>(m);
  else if (epi == EPI_Y) k_fx_clinv<DAG, CLOV, EPI_Y><<<gr, 128, 0, st>>>(m);
  else if (epi == (EPI_X | EPI_Y)) k_fx_clinv<DAG, CLOV, EPI_X | EPI_Y><<<gr, 128, 0, st>>>(m);
  else return -1;
  return 0;
}

int fx_clinv_launch(bool dag, bool clov, int epi, dim3 gr, const FxArgs& m, cudaStream_t st) {
  if (dag) return clov ? pick<true, true>(epi, gr, m, st) : pick<true, false>(epi, gr, m, st);
  return clov ? pick<false, true>(epi, gr, m, st) : pick<false, false>(epi, gr, m, st);
}

}  // namespace lq
