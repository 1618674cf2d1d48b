// bp_pair_kernel on decomposed data (float32).
#include "bp_pair.cuh"

namespace fdkod {

cudaError_t launch_pair_od(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                           cudaStream_t st) {
    return launch_pair<float, false>(s, map, prm, nsq, st);
}

}  // namespace fdkod
