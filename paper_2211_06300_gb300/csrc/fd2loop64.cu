// FP64 instantiations of the on-chip 2D time loops (fd2loop.h).
#include "fd2loop.h"

namespace esi {
template <>
cudaError_t launch_loop2<double>(unsigned flags, const StepArgs<double> &a, const LoopArgs<double> &g,
                                int nblk, int threads, size_t smem, cudaStream_t st) {
    return loop2::dispatch<double>(flags, a, g, nblk, threads, smem, st);
}
}  // namespace esi
