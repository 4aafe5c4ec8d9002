// k_team_mie_mixed.cu -- the mie instances of the team kernel (k_team.cuh), mixed precision.
#include "k_team.cuh"

namespace gbmd {

void* k_team_mie_mixed(int tpp, int mt, bool two_in_one) {
  return k_team_tpp<EVAL_MIE, GBMD_MIXED>(tpp, mt, two_in_one);
}

}  // namespace gbmd
