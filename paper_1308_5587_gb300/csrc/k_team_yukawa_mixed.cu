// k_team_yukawa_mixed.cu -- the yukawa instances of the team kernel (k_team.cuh), mixed precision.
#include "k_team.cuh"

namespace gbmd {

void* k_team_yukawa_mixed(int tpp, int mt, bool two_in_one) {
  return k_team_tpp<EVAL_YUKAWA, GBMD_MIXED>(tpp, mt, two_in_one);
}

}  // namespace gbmd
