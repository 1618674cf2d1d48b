// bp_pair_kernel on Q stored as bfloat16.
#include "bp_pair.cuh"

namespace fdkod {

cudaError_t launch_pair_bf16(const PairShape &s, const CUtensorMap &map, const BpPairParams &prm, int nsq,
                             cudaStream_t st) {
    return launch_pair<__nv_bfloat16, true>(s, map, prm, nsq, st);
}

}  // namespace fdkod
