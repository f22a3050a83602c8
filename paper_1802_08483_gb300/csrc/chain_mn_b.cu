// Recursions for frames with MN = 19, 21, 22, 23, 25 received lengths per symbol.
#include "chain_kern.cuh"

namespace mdk {

cudaError_t launch_chain_b(int mn, const FrameDev *frames, const Work *work, int nwork, size_t smem,
                           int cluster, int threads, cudaStream_t st) {
    switch (mn) {
        case 19: return launch_chain_mn<19>(frames, work, nwork, smem, cluster, threads, st);
        case 21: return launch_chain_mn<21>(frames, work, nwork, smem, cluster, threads, st);
        case 22: return launch_chain_mn<22>(frames, work, nwork, smem, cluster, threads, st);
        case 23: return launch_chain_mn<23>(frames, work, nwork, smem, cluster, threads, st);
        case 25: return launch_chain_mn<25>(frames, work, nwork, smem, cluster, threads, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace mdk
