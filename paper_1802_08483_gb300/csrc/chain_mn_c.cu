// Recursions for frames with MN = 28, 29, 31, 33 received lengths per symbol.
#include "chain_kern.cuh"

namespace mdk {

cudaError_t launch_chain_c(int mn, const FrameDev *frames, const Work *work, int nwork, size_t smem,
                           int cluster, int threads, cudaStream_t st) {
    switch (mn) {
        case 28: return launch_chain_mn<28>(frames, work, nwork, smem, cluster, threads, st);
        case 29: return launch_chain_mn<29>(frames, work, nwork, smem, cluster, threads, st);
        case 31: return launch_chain_mn<31>(frames, work, nwork, smem, cluster, threads, st);
        case 33: return launch_chain_mn<33>(frames, work, nwork, smem, cluster, threads, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace mdk
