// The FP64 build kernels for every ABF element dW0/dr d^alpha|r| (LABFM_ABF_DW0_ONLY).
#include "build_node.cuh"

namespace labfm {

cudaError_t launch_order_dw0(int k, int G, const BuildArgs &a, int num_sms, cudaStream_t s)
{
    return launch_order<false>(k, G, a, num_sms, s);
}

cudaError_t launch_items_dw0(const BuildArgs &a, const OrderItems &I, int num_sms, cudaStream_t s)
{
    return launch_persistent_build(k_build_fp64_items<false>, I.total, num_sms, s, a, I);
}

cudaError_t launch_any_dw0(const BuildArgs &a, const int8_t *order, int uniform_order, int num_sms, cudaStream_t s)
{
    return launch_persistent_build(k_build_fp64_any<false>, a.n_list, num_sms, s, a, order, uniform_order);
}

}  // namespace labfm
