// bp_pair_kernel on Q stored as float32.
#include "bp_pair.cuh"

namespace fdkod {

cudaError_t launch_pair_f32(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                            cudaStream_t st) {
    return launch_pair<float, true>(s, map, prm, nsq, st);
}

}  // namespace fdkod
