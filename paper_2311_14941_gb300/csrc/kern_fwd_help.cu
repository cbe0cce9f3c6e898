// kern_fwd_help.cu -- integration kernels with one warp per cell and helper warps.
#include "kern_forward.cuh"

namespace chemgb {

template const void* plain_kernel<Grp1, HelpedView<1>>();
template cudaError_t launch_plain_g<Grp1, HelpedView<1>>(dim3, dim3, size_t, cudaStream_t, const MechView&, const CellLayout&, int, double*,
                                  const double*, double*, const double*, double*, int*, int*, int*, const IntOpts&,
                                  const unsigned long long*, unsigned long long);
template const void* persistent_kernel<Grp1, HelpedView<1>>();
template cudaError_t launch_persistent_g<Grp1, HelpedView<1>>(dim3, dim3, size_t, cudaStream_t, const MechView&, const CellLayout&, int,
                                       double*, const double*, double*, const double*, double*, int*, int*, int*,
                                       const int*, unsigned long long*, int, const IntOpts&,
                                       const unsigned long long*, unsigned long long);

template const void* plain_kernel<Grp1, HelpedView<3>>();
template cudaError_t launch_plain_g<Grp1, HelpedView<3>>(dim3, dim3, size_t, cudaStream_t, const MechView&, const CellLayout&, int, double*,
                                  const double*, double*, const double*, double*, int*, int*, int*, const IntOpts&,
                                  const unsigned long long*, unsigned long long);
template const void* persistent_kernel<Grp1, HelpedView<3>>();
template cudaError_t launch_persistent_g<Grp1, HelpedView<3>>(dim3, dim3, size_t, cudaStream_t, const MechView&, const CellLayout&, int,
                                       double*, const double*, double*, const double*, double*, int*, int*, int*,
                                       const int*, unsigned long long*, int, const IntOpts&,
                                       const unsigned long long*, unsigned long long);

}  // namespace chemgb
