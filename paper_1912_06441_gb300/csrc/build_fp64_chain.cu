// The FP64 build kernels for the full chain rule in the ABFs of degrees 2 and 3 (Appendix A as printed).
#include "build_node.cuh"

namespace labfm {

cudaError_t launch_order_chain(int k, int G, const BuildArgs &a, int num_sms, cudaStream_t s)
{
    return launch_order<true>(k, G, a, num_sms, s);
}

cudaError_t launch_items_chain(const BuildArgs &a, const OrderItems &I, int num_sms, cudaStream_t s)
{
    return launch_persistent_build(k_build_fp64_items<true>, I.total, num_sms, s, a, I);
}

cudaError_t launch_any_chain(const BuildArgs &a, const int8_t *order, int uniform_order, int num_sms, cudaStream_t s)
{
    return launch_persistent_build(k_build_fp64_any<true>, a.n_list, num_sms, s, a, order, uniform_order);
}

}  // namespace labfm
