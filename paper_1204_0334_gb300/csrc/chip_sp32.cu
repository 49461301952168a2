// The on-chip decoder's kernels: sum-product, FP32 messages.
#include "flow_chip.cuh"

namespace ldpc {
namespace chip {

ldpc_status run_sp32(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken) {
    return dispatch<1, flow::kFlowSP>(c, a, P, s, taken);
}

}  // namespace chip
}  // namespace ldpc
