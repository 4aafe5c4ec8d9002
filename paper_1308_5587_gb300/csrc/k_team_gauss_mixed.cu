// k_team_gauss_mixed.cu -- the gauss instances of the team kernel (k_team.cuh), mixed precision.
#include "k_team.cuh"

namespace gbmd {

void* k_team_gauss_mixed(int tpp, int mt, bool two_in_one) {
  return k_team_tpp<EVAL_GAUSS, GBMD_MIXED>(tpp, mt, two_in_one);
}

}  // namespace gbmd
