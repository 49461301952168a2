// The flow decoder's kernels: learned min-sum, FP16 messages.
#include "flow.cuh"

namespace ldpc {
namespace flow {

ldpc_status run_noms16(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s) {
    return dispatch<2, kFlowNOMS>(a, st, g, tiles, s);
}

}  // namespace flow
}  // namespace ldpc
