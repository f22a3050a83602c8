// Recursions for frames with MN = 45, 49 received lengths per symbol.
#include "chain_kern.cuh"

namespace mdk {

cudaError_t launch_chain_e(int mn, const FrameDev *frames, const Work *work, int nwork, size_t smem,
                           int cluster, int threads, cudaStream_t st) {
    switch (mn) {
        case 45: return launch_chain_mn<45>(frames, work, nwork, smem, cluster, threads, st);
        case 49: return launch_chain_mn<49>(frames, work, nwork, smem, cluster, threads, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace mdk
