// One-launch steps of small meshes: the synthetic 19-state model's kernels.
#include <mutex>

#include "esdc_small.cuh"

namespace {
std::mutex g_const_mu;
bool g_const_done[64] = {false};
}

cudaError_t esdc_small_constants_syn(int device)
{
    std::lock_guard<std::mutex> lk(g_const_mu);
    return upload_constants_local(g_const_done, device);
}

cudaError_t esdc_small_launch_syn(const StepArgs& a, const void* args, int M, int blocks, int threads, size_t smem,
                                  cudaStream_t s)
{
    return small_launch_M<esdc::SYN19>(a, *static_cast<const SmallArgs*>(args), M, blocks, threads, smem, s);
}
