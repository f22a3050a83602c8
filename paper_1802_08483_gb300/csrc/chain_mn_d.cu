// Recursions for frames with MN = 34, 37, 41 received lengths per symbol.
#include "chain_kern.cuh"

namespace mdk {

cudaError_t launch_chain_d(int mn, const FrameDev *frames, const Work *work, int nwork, size_t smem,
                           int cluster, int threads, cudaStream_t st) {
    switch (mn) {
        case 34: return launch_chain_mn<34>(frames, work, nwork, smem, cluster, threads, st);
        case 37: return launch_chain_mn<37>(frames, work, nwork, smem, cluster, threads, st);
        case 41: return launch_chain_mn<41>(frames, work, nwork, smem, cluster, threads, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace mdk
