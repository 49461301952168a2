// The on-chip decoder's kernels: learned min-sum, FP16 messages.
#include "flow_chip.cuh"

namespace ldpc {
namespace chip {

ldpc_status run_noms16(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken) {
    return dispatch<2, flow::kFlowNOMS>(c, a, P, s, taken);
}

}  // namespace chip
}  // namespace ldpc
