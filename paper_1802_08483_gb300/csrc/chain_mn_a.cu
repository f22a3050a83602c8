// Recursions for frames with MN = 9, 11, 13, 15, 16, 17 received lengths per symbol.
#include "chain_kern.cuh"

namespace mdk {

cudaError_t launch_chain_a(int mn, const FrameDev *frames, const Work *work, int nwork, size_t smem,
                           int cluster, int threads, cudaStream_t st) {
    switch (mn) {
        case 9: return launch_chain_mn<9>(frames, work, nwork, smem, cluster, threads, st);
        case 11: return launch_chain_mn<11>(frames, work, nwork, smem, cluster, threads, st);
        case 13: return launch_chain_mn<13>(frames, work, nwork, smem, cluster, threads, st);
        case 15: return launch_chain_mn<15>(frames, work, nwork, smem, cluster, threads, st);
        case 16: return launch_chain_mn<16>(frames, work, nwork, smem, cluster, threads, st);
        case 17: return launch_chain_mn<17>(frames, work, nwork, smem, cluster, threads, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace mdk
