// The on-chip decoder's kernels: sum-product, FP16 messages.
#include "flow_chip.cuh"

namespace ldpc {
namespace chip {

ldpc_status run_sp16(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken) {
    return dispatch<2, flow::kFlowSP>(c, a, P, s, taken);
}

}  // namespace chip
}  // namespace ldpc
