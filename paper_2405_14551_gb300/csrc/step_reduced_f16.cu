// Step kernels instantiated for storage 2 (reduced single set, FP16 deviations).
#include "step_launch.cuh"

namespace lbcg {

template cudaError_t launch_phi_acc_t<2>(const Geo&, const StateBuf&, unsigned long long*, cudaStream_t);
template cudaError_t launch_step_s<2>(int, bool, bool, int, const Geo&, const Phys&, const StateBuf&, const InitBuf&,
                                      PhiSrc, AccBufs, StateBuf, void*, int, const FieldOut&, unsigned*, cudaStream_t);
template cudaError_t launch_phi_s<2>(const Geo&, const Phys&, const InitBuf&, PhiSrc, void*, int, cudaStream_t);
template cudaError_t launch_density_t<2>(int, const Geo&, const Phys&, const StateBuf&, const InitBuf&,
                                         const unsigned long long*, unsigned*, cudaStream_t);
template cudaError_t launch_export_t<2>(int, const Geo&, const Phys&, const StateBuf&, const InitBuf&, int, int, int,
                                        int, int, int, double*, double*, cudaStream_t);

template cudaError_t launch_batched_t<2>(const RunDesc*, const int*, long long, long long, int, int, long long, int, int, int,
                                         unsigned*, cudaStream_t);

}  // namespace lbcg
