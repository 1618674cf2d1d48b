// bp_pair_kernel on float32 windows: decomposed data, and Q stored as float32.
#include "bp_pair.cuh"

namespace fdkod {

cudaError_t launch_pair_f32(bool direct, const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                            cudaStream_t st) {
    return direct ? launch_pair<float, true>(s, map, prm, nsq, st) : launch_pair<float, false>(s, map, prm, nsq, st);
}

}  // namespace fdkod
