// k_team_yukawa_fp64.cu -- the yukawa instances of the team kernel (k_team.cuh), FP64.
#include "k_team.cuh"

namespace gbmd {

void* k_team_yukawa_fp64(int tpp, int mt, bool two_in_one) {
  return k_team_tpp<EVAL_YUKAWA, GBMD_FP64>(tpp, mt, two_in_one);
}

}  // namespace gbmd
