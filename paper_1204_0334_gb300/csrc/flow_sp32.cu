// The flow decoder's kernels: sum-product, FP32 messages.
#include "flow.cuh"

namespace ldpc {
namespace flow {

ldpc_status run_sp32(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s) {
    return dispatch<1, kFlowSP>(a, st, g, tiles, s);
}

}  // namespace flow
}  // namespace ldpc
