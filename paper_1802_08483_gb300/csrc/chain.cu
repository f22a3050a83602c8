// Sequential parts of the decoder and small helper kernels.
//
//   k_pack     : received bits (one per byte) -> 32-bit words.
//   k_chain    : the recursions (chain_kern.cuh, chain_crowd.cuh), dispatched here.
//   k_finalize : APPs (eq. L, normalised over D), extrinsic outputs (eq. L
//                without the symbol's own prior), d logP / d prior and the
//                FP64 reduction of the channel-parameter gradient
//                (k_grad_reduce adds the chunks of a frame in order).
#include <cstdlib>

#include "chain_kern.cuh"

namespace mdk {

// ---------------------------------------------------------------------------
__global__ void k_pack(const FrameDev *__restrict__ frames, const uint8_t *const *rx_bytes,
                       uint32_t *const *rx_words, int nframes) {
    const int fi = blockIdx.y;
    if (fi >= nframes) return;
    const long long rho = frames[fi].rho;
    const uint8_t *src = rx_bytes[fi];
    uint32_t *dst = rx_words[fi];
    const long long nwords = (rho + 31) / 32 + 3;
    for (long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x; w < nwords;
         w += (long long)gridDim.x * blockDim.x) {
        uint32_t v = 0;
        const long long b0 = w * 32;
        for (int b = 0; b < 32; ++b) {
            const long long k = b0 + b;
            if (k < rho && src[k]) v |= (1u << b);
        }
        dst[w] = v;
    }
}

// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kCrowdMaxThreads, 1) k_chain_crowd(const FrameDev *__restrict__ frames,
                                                         const Work *__restrict__ work) {
    const Work wk = work[blockIdx.x];
    crowd_recursion(frames[wk.frame], wk.tile);
}

// ---------------------------------------------------------------------------
// Finalize: one CTA per (frame, chunk of kFinChunk symbols), kFinSym symbols per
// warp at once, lanes over D.  Gradient sums of a chunk go to Gc[chunk]; a second
// kernel adds the chunks of a frame in order (deterministic).
//
// Bound by FP64: this GPU runs two FP64 lanes a clock and SM, so a warp's FP64
// instruction takes 16 clocks, and the normaliser's butterfly (5 additions) and
// division (about 20 instructions) per symbol outweighed everything else.  The
// kFinSym symbols of a warp share them: the butterflies run as one reduction that
// halves what a lane carries at each of the first exchanges (the additions and
// their order per symbol stay the same), leaving symbol k's sums in lanes
// 4 k .. 4 k + 3, where one division and one gradient formula serve all of them.
// One frame's finalize (N = 50, q = 16, n = 10) took 30 us, one symbol after another
// in each warp; its whole decode went from 267.5 to 255.3 us, and 256 frames of
// N = 64, q = 8 from 499 to 470 us.
constexpr int kFinSym = 8;
constexpr int kFinThreads = 64;
constexpr int kFinChunk = kFinSym * (kFinThreads / 32);
constexpr int kFinRegs = 2;  // 32-wide slices of q kept in registers (q <= 64)

// x[k]: this lane's part of sum k; returns, in lanes 4 k .. 4 k + 3, sum k over
// the warp (butterfly order 16, 8, 4, 2, 1).
__device__ __forceinline__ double fin_reduce(const double (&x)[kFinSym], int lane) {
    double y[4], z[2];
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        y[k] = (h4 ? x[k + 4] : x[k]) + __shfl_xor_sync(0xffffffffu, h4 ? x[k] : x[k + 4], 16);
#pragma unroll
    for (int k = 0; k < 2; ++k)
        z[k] = (h3 ? y[k + 2] : y[k]) + __shfl_xor_sync(0xffffffffu, h3 ? y[k] : y[k + 2], 8);
    double r = (h2 ? z[1] : z[0]) + __shfl_xor_sync(0xffffffffu, h2 ? z[0] : z[1], 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}

__global__ void __launch_bounds__(kFinThreads) k_finalize(const FrameDev *__restrict__ frames,
                                                          const Work *__restrict__ work,
                                                          int grad) {
    const Work wk = work[blockIdx.x];
    const FrameDev &f = frames[wk.frame];
    __shared__ double red[3][kFinThreads / 32];
    if (*f.status != ST_OK) return;
    const int q = f.q, n = f.n, xmax = f.xmax, S2 = f.S2, psT = f.psT, seg0 = f.seg_i0;
    const bool ps = f.ps != 0;
    // positions per row tile; row tiles whose sums are added first (gradients)
    const long long P2 = (long long)f.P * (f.group ? 1 : f.nsub);
    const unsigned group = max(1, f.group);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float *__restrict__ Lp = f.Lp;
    const float *__restrict__ priors = f.priors;
    float *const app = f.app, *const dpri = f.dpriors, *const ext = f.ext;
    const int c0 = seg0 + (wk.tile - f.fin_base) * kFinChunk;
    const int i1 = min(f.seg_i1, c0 + kFinChunk);
    const int i0 = c0 + warp * kFinSym;
    const int ns = max(0, min(kFinSym, i1 - i0));  // symbols of this warp
    // Rows of the APP partials of symbol i0 + k: tiles tlo .. tlo + cnt - 1, one row
    // each, looked up by lanes 4 k .. 4 k + 3.  Row of tile t: t S2 + i - (the
    // tile's first symbol), or t itself (per-symbol producers: rows are work items).
    const int mine = lane >> 2;
    long long tlo = 0;
    int cnt = 0;
    if (mine < ns) {
        const int i = i0 + mine;
        if (ps) {
            tlo = (long long)i * psT;
            cnt = psT;
        } else {
            tlo = max(0LL, (long long)n * i - xmax) / P2;
            cnt = (int)(min(f.rho, (long long)n * i + xmax) / P2 - tlo) + 1;
        }
    }
    const int most = __reduce_max_sync(0xffffffffu, cnt);
    auto row_of = [&](int i, long long t) -> long long {
        if (ps) return t;
        // i - ceil((t P2 - xmax) / n), the tile's first symbol not before the segment's
        const unsigned past = (unsigned)((long long)n * i - t * P2 + xmax) / (unsigned)n;
        return t * S2 + min(i - seg0, (int)past);
    };
    // Unnormalised sums L^u(D) (eq. L without the prior) of the warp's symbols at
    // D = D0 + lane, the rows of a symbol in order.  Four rows of every symbol are
    // loaded at a time: one symbol after another a warp waited for memory 2 to 40
    // times each (N = 50, q = 16: 22000 clocks of 36000).
    auto lsums = [&](int D0, float (&v)[kFinSym]) {
        const int D = D0 + lane;
        float part[kFinSym];
#pragma unroll
        for (int k = 0; k < kFinSym; ++k) v[k] = part[k] = 0.f;
        for (int t0 = 0; t0 < most; t0 += 4) {
            const int t = t0 + (lane & 3);
            const long long row = t < cnt ? row_of(i0 + mine, tlo + t) : -1;
            // rows that end a group (or the symbol's range)
            const unsigned last =
                __ballot_sync(0xffffffffu, (unsigned)(tlo + t) % group == group - 1 || t + 1 == cnt);
            float x[kFinSym][4];
#pragma unroll
            for (int k = 0; k < kFinSym; ++k)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const long long r = __shfl_sync(0xffffffffu, row, 4 * k + e);
                    x[k][e] = r >= 0 && D < q ? Lp[r * q + D] : 0.f;
                }
#pragma unroll
            for (int k = 0; k < kFinSym; ++k)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    part[k] += x[k][e];
                    if (last >> (4 * k + e) & 1u) {
                        v[k] += part[k];
                        part[k] = 0.f;
                    }
                }
        }
    };
    // pass 1: z = sum_D prior(D) L^u(D) and, for the extrinsic output, zu = sum_D L^u(D)
    float lu[kFinRegs][kFinSym], pr[kFinRegs][kFinSym];
    double z[kFinSym], zu[kFinSym];
#pragma unroll
    for (int k = 0; k < kFinSym; ++k) z[k] = zu[k] = 0.0;
    auto add = [&](int D0, const float (&v)[kFinSym], float (&p)[kFinSym]) {
#pragma unroll
        for (int k = 0; k < kFinSym; ++k)
            p[k] = k < ns && D0 + lane < q ? priors[(size_t)(i0 + k) * q + D0 + lane] : 0.f;
#pragma unroll
        for (int k = 0; k < kFinSym; ++k) {
            z[k] += (double)p[k] * (double)v[k];
            if (ext) zu[k] += (double)v[k];
        }
    };
#pragma unroll
    for (int r = 0; r < kFinRegs; ++r) {
#pragma unroll
        for (int k = 0; k < kFinSym; ++k) lu[r][k] = pr[r][k] = 0.f;
        if (32 * r >= q) continue;
        lsums(32 * r, lu[r]);
        add(32 * r, lu[r], pr[r]);
    }
    for (int D0 = 32 * kFinRegs; D0 < q; D0 += 32) {  // beyond the registers: through app
        float v[kFinSym], p[kFinSym];
        lsums(D0, v);
        add(D0, v, p);
#pragma unroll
        for (int k = 0; k < kFinSym; ++k)
            if (k < ns && D0 + lane < q) app[(size_t)(i0 + k) * q + D0 + lane] = v[k];
    }
    const double zs = fin_reduce(z, lane);
    const bool ok = mine < ns && zs > 0.0;
    const double iz = ok ? 1.0 / zs : 0.0;
    double izu = 0.0;
    if (ext) {
        const double zus = fin_reduce(zu, lane);
        izu = ok ? 1.0 / zus : 0.0;  // zu >= z / max prior > 0
    }
    const unsigned good = __ballot_sync(0xffffffffu, ok);
    // pass 2: each lane scales the entries it summed
#pragma unroll
    for (int k = 0; k < kFinSym; ++k) {
        const double izk = __shfl_sync(0xffffffffu, iz, 4 * k), izuk = __shfl_sync(0xffffffffu, izu, 4 * k);
        if (!(good >> (4 * k) & 1u)) continue;
        const size_t e0 = (size_t)(i0 + k) * q;
        auto put = [&](int D, float p, float v) {
            const double l = (double)v;
            app[e0 + D] = (float)((double)p * l * izk);
            if (dpri) dpri[e0 + D] = (float)(l * izk);
            if (ext) ext[e0 + D] = (float)(l * izuk);
        };
#pragma unroll
        for (int r = 0; r < kFinRegs; ++r)
            if (32 * r + lane < q) put(32 * r + lane, pr[r][k], lu[r][k]);
        for (int D = 32 * kFinRegs + lane; D < q; D += 32) put(D, priors[e0 + D], app[e0 + D]);
    }
    if (lane == 0 && good != (ns == kFinSym ? 0xffffffffu : (1u << (4 * ns)) - 1u))
        atomicMax(f.status, ST_ZERO);
    if (grad && f.Gc) {
        double g0 = 0.0, g1 = 0.0, g2 = 0.0;
        if (ok) {
            // the lattice ran with w' = k Pi/2, Q'm = k Pt (1-Ps), Q's = k Pt Ps
            const double Pt = f.dPt, Ps = f.dPs, Pd = f.dPd, k = f.kappa;
            const double Qm = k * Pt * (1.0 - Ps), Qs = k * Pt * Ps;
            double Sw = 0.0, Sd = 0.0, Ss = 0.0;
            const float *__restrict__ Gp = f.Gp;
            float sw = 0.f, sd = 0.f, ss = 0.f;
            int left = (int)(group - (unsigned)tlo % group);
            for (int t0 = 0; t0 < cnt; t0 += 4) {
                float x[4][3];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float *g = Gp + row_of(i0 + mine, tlo + min(t0 + e, cnt - 1)) * 3;
                    x[e][0] = g[0];
                    x[e][1] = g[1];
                    x[e][2] = g[2];
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (t0 + e >= cnt) break;
                    sw += x[e][0];
                    sd += x[e][1];
                    ss += x[e][2];
                    if (--left == 0 || t0 + e + 1 == cnt) {
                        Sw += sw;
                        Sd += sd;
                        Ss += ss;
                        sw = sd = ss = 0.f;
                        left = (int)group;
                    }
                }
            }
            // Sw, Sd, Ss: sums with dR~/dw', dR~/dPd, dR~/dQ's.  R~ is homogeneous
            // of degree n in (Pd, Q'm, Q's) (every bit is deleted or transmitted),
            // so Pd dR~/dPd + Q'm dR~/dQ'm + Q's dR~/dQ's = n R~ gives the Q'm sum.
            // Chain rule with w' = k Pi/2, Q'm = k Pt (1-Ps), Q's = k Pt Ps, Pt = 1-Pi-Pd.
            const double Sm = ((double)n * zs - Pd * Sd - Qs * Ss) / Qm;
            g0 = (0.5 * k * Sw - k * (1.0 - Ps) * Sm - k * Ps * Ss) * iz;
            g1 = (Sd - k * (1.0 - Ps) * Sm - k * Ps * Ss) * iz;
            g2 = (-k * Pt * Sm + k * Pt * Ss) * iz;
        }
        // over the warp's symbols (one lane in four), then the warps in order
#pragma unroll
        for (int o = 16; o > 2; o >>= 1) {
            g0 += __shfl_xor_sync(0xffffffffu, g0, o);
            g1 += __shfl_xor_sync(0xffffffffu, g1, o);
            g2 += __shfl_xor_sync(0xffffffffu, g2, o);
        }
        if (lane == 0) { red[0][warp] = g0; red[1][warp] = g1; red[2][warp] = g2; }
        __syncthreads();
        if (threadIdx.x < 3) {
            double s = 0.0;
            for (int w = 0; w < kFinThreads / 32; ++w) s += red[threadIdx.x][w];
            f.Gc[(size_t)wk.tile * 3 + threadIdx.x] = s;
        }
    }
}

// Sums the chunk gradients of every frame, a warp per frame: lane l adds chunks
// l, l + 32, .. in order, then a butterfly (deterministic).
__global__ void k_grad_reduce(const FrameDev *__restrict__ frames, int nframes) {
    const int fi = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (fi >= nframes) return;
    const FrameDev &f = frames[fi];
    if (!f.dchan || !f.Gc || *f.status != ST_OK) return;
    const int nch = f.fin_total;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int c = lane; c < nch; c += 32) {
        s0 += f.Gc[3 * c];
        s1 += f.Gc[3 * c + 1];
        s2 += f.Gc[3 * c + 2];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (lane == 0) {
        f.dchan[0] = s0;
        f.dchan[1] = s1;
        f.dchan[2] = s2;
    }
}

// ---------------------------------------------------------------------------
// Copies between pinned host memory and device memory by the SMs: 16 bytes per
// thread and step over a grid-stride loop, reading or writing the host side
// through its device mapping (NVLink-C2C).  Both pointers 16-byte aligned; n16
// 16-byte words.
__global__ void k_copy16(uint4 *__restrict__ dst, const uint4 *__restrict__ src, size_t n16) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n16; k += stride)
        dst[k] = src[k];
}

// ---------------------------------------------------------------------------
// Launch wrappers (host).
cudaError_t launch_copy16(void *dst, const void *src, size_t n16, int sms, cudaStream_t st) {
    if (n16 == 0) return cudaSuccess;
    const size_t per = 256;
    size_t blocks = (n16 + per - 1) / per;
    const size_t cap = (size_t)(sms > 0 ? sms : 152) * 4;
    if (blocks > cap) blocks = cap;
    k_copy16<<<(unsigned)blocks, (unsigned)per, 0, st>>>(static_cast<uint4 *>(dst),
                                                          static_cast<const uint4 *>(src), n16);
    return cudaGetLastError();
}

cudaError_t launch_pack(const FrameDev *frames, const uint8_t *const *rx_bytes,
                        uint32_t *const *rx_words, int nframes, long long max_words,
                        cudaStream_t st) {
    if (nframes <= 0) return cudaSuccess;
    int gx = (int)((max_words + 255) / 256);
    if (gx > 64) gx = 64;
    if (gx < 1) gx = 1;
    dim3 grid(gx, nframes);
    k_pack<<<grid, 256, 0, st>>>(frames, rx_bytes, rx_words, nframes);
    return cudaGetLastError();
}

size_t chain_smem_bytes(const FrameDev &f) {
    const size_t nck = (f.chainVC + f.chainCK - 1) / f.chainCK;
    // rows, lane groups and their lanes' places, chunk table (8 bytes each, to 16), stages
    return (size_t)f.chainRing * (f.Mp + 2 * kChainRowPad) * 4 + (size_t)f.chainWarps * f.chainList * sizeof(LaneGroup) +
           (size_t)f.chainWarps * (f.chainList - 1) * 32 * sizeof(int4) +
           ((nck * sizeof(ChunkGeom) + 15) & ~(size_t)15) +
           (size_t)f.chainStages * f.chainStageFloats * 4;
}

size_t crowd_smem_bytes(const FrameDev &f) {
    const size_t stageFloats = ((size_t)(f.crowdCD + f.MN + 1) * f.MNS + 8 + 3) & ~(size_t)3;
    return 4 * (2 * (size_t)f.Mp + (size_t)f.crowdStages * stageFloats);
}

cudaError_t launch_chain_crowd(const FrameDev *frames, const Work *work, int nwork, size_t smem,
                               int threads, cudaStream_t st) {
    if (nwork <= 0) return cudaSuccess;
    static std::atomic<uint64_t> attr{0};
    cudaError_t e = smem_optin_once(k_chain_crowd, attr);
    if (e != cudaSuccess) return e;
    if (threads != 128 && threads != 256 && threads != 512) threads = kCrowdThreads;
    k_chain_crowd<<<nwork, threads, smem, st>>>(frames, work);
    return cudaGetLastError();
}

cudaError_t launch_chain(int mn, const FrameDev *frames, const Work *work, int nwork, size_t smem,
                         int cluster, int threads, cudaStream_t st) {
    if (nwork <= 0) return cudaSuccess;
    if (threads < 96 || threads > kChainMaxThreads || threads % 32) return cudaErrorInvalidValue;
    // MN with a compiled kernel (launches whose frames share it): n = 4 .. 12, I = 1, 2, 3
    switch (mn) {
        case 9: case 11: case 13: case 15: case 16: case 17:
            return launch_chain_a(mn, frames, work, nwork, smem, cluster, threads, st);
        case 19: case 21: case 22: case 23: case 25:
            return launch_chain_b(mn, frames, work, nwork, smem, cluster, threads, st);
        case 28: case 29: case 31: case 33:
            return launch_chain_c(mn, frames, work, nwork, smem, cluster, threads, st);
        case 34: case 37: case 41:
            return launch_chain_d(mn, frames, work, nwork, smem, cluster, threads, st);
        case 45: case 49:
            return launch_chain_e(mn, frames, work, nwork, smem, cluster, threads, st);
        default: return launch_chain_mn<0>(frames, work, nwork, smem, cluster, threads, st);
    }
}

int finalize_chunks(int N) { return (N + kFinChunk - 1) / kFinChunk; }
size_t chain_state_bytes() { return sizeof(ChainState); }

cudaError_t launch_finalize(const FrameDev *frames, const Work *work, int nwork, int nframes,
                            int grad, cudaStream_t st, bool reduce) {
    if (nwork > 0) k_finalize<<<nwork, kFinThreads, 0, st>>>(frames, work, grad);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !grad || !reduce || nframes <= 0) return e;
    k_grad_reduce<<<(nframes + 3) / 4, 128, 0, st>>>(frames, nframes);
    return cudaGetLastError();
}

}  // namespace mdk
