// Step kernels instantiated for storage 1 (reduced single set, FP32).
#include "step_launch.cuh"

namespace lbcg {

template cudaError_t launch_phi_acc_t<1>(const Geo&, const StateBuf&, unsigned long long*, cudaStream_t);
template cudaError_t launch_step_s<1>(int, bool, bool, int, const Geo&, const Phys&, const StateBuf&, const InitBuf&,
                                      PhiSrc, AccBufs, StateBuf, void*, int, const FieldOut&, unsigned*, cudaStream_t);
template cudaError_t launch_phi_s<1>(const Geo&, const Phys&, const InitBuf&, PhiSrc, void*, int, cudaStream_t);
template cudaError_t launch_density_t<1>(int, const Geo&, const Phys&, const StateBuf&, const InitBuf&,
                                         const unsigned long long*, unsigned*, cudaStream_t);
template cudaError_t launch_export_t<1>(int, const Geo&, const Phys&, const StateBuf&, const InitBuf&, int, int, int,
                                        int, int, int, double*, double*, cudaStream_t);

template cudaError_t launch_batched_t<1>(const RunDesc*, const int*, long long, long long, int, int, long long, int, int, int,
                                         unsigned*, cudaStream_t);

}  // namespace lbcg
