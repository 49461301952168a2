// The flow decoder's kernels: integer min-sum.
#include "flow.cuh"

namespace ldpc {
namespace flow {

ldpc_status run_ms(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s) {
    return dispatch<4, kFlowMS>(a, st, g, tiles, s);
}

}  // namespace flow
}  // namespace ldpc
