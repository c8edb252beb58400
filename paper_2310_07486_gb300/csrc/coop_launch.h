// coop_launch.h -- cooperative launches on as many blocks as can run at once (host code).
#pragma once
#include <cuda_runtime.h>

namespace qsg {

// launch(blocks) with `blocks` or, where they do not all fit on the GPU at once (a
// process may have fewer SMs than the device reports: a green context, a share of
// one), with half as many and so on; the kernel must take any number of blocks.
template <class Launch>
cudaError_t launch_resident_grid(int blocks, Launch launch) {
    cudaError_t e = launch(blocks);
    while (e == cudaErrorCooperativeLaunchTooLarge && blocks > 1) {
        cudaGetLastError();  // this attempt's
        blocks = (blocks + 1) / 2;
        e = launch(blocks);
    }
    return e;
}

}  // namespace qsg
