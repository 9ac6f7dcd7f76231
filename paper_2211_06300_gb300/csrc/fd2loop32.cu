// FP32 instantiations of the on-chip 2D time loops (fd2loop.h).
#include "fd2loop.h"

namespace esi {
template <>
cudaError_t launch_loop2<float>(unsigned flags, const StepArgs<float> &a, const LoopArgs<float> &g,
                                int nblk, int threads, size_t smem, cudaStream_t st) {
    return loop2::dispatch<float>(flags, a, g, nblk, threads, smem, st);
}
}  // namespace esi
