// The on-chip decoder's kernels: integer min-sum.
#include "flow_chip.cuh"

namespace ldpc {
namespace chip {

ldpc_status run_ms(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken) {
    return dispatch<4, flow::kFlowMS>(c, a, P, s, taken);
}

}  // namespace chip
}  // namespace ldpc
