// The recursion kernel (k_chain) and its launch template; one unit per group of
// received-length counts MN (chain_mn*.cu), dispatched in chain.cu.
#pragma once

#include <type_traits>

#include "chain_crowd.cuh"

namespace mdk {

// ---------------------------------------------------------------------------
constexpr int kChainMaxThreads = 512;
constexpr int kChainMostThreads = 320;  // one CTA: 8 virtual warps, mover and storer
// The work of one recursion: a CTA with a warp per virtual warp (its lanes then hold
// the partial sums), a CTA with a warp per lane group (rows of several chunks; the
// partial sums are read back from the rows), a cluster of such CTAs.
constexpr int kChainNarrow = 0, kChainWide = 1, kChainCluster = 2;

// Rows are divided by their power of two when their sums are formed (at tilt
// updates), or at once when their largest entry fell below this.
constexpr float kRowLow = 1.f / 65536.f;
// A sum of rows that were not scaled one by one is not used below this (2^-64): a step
// may have cost entries that a row scaled at once would have kept.  The launch is then
// run again with every row scaled (crowd_again), as where a sum left FP32's range:
// priors are used as given, whatever their rows' sums, and four steps may multiply a
// row by what a step may (2^+-126).
constexpr float kSumLow = 1.f / 18446744073709551616.f;
constexpr int kRunMost = 4;      // rows between two sums, at most
constexpr int kAliveSlots = 16;  // steps until a vote's place is used again (a power of two)

__device__ __forceinline__ bool tilt_due(int steps) {
    return steps < kTiltSettle || (steps & (kTiltEvery - 1)) == 0;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Store to `p`'s place in the shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ void st_cluster(const void *p, uint32_t rank, uint32_t v) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
// Barrier over the recursion's CTAs (one, or the cluster).
// relaxed (the helper warps of a cluster): the arrival orders nothing by itself, so
// it need not wait for the warp's earlier stores.  The storer's all go to global
// memory and are read by no CTA of the launch (waiting for a row's took about 1000
// clocks).  The mover hands the landed W on to its own CTA, by a fence of that scope
// (cta_release).  The compute warps' arrivals release rows and votes to the cluster.
// What a helper reads (rows, votes) is ordered before later writes of other warps by
// the CTA's barriers (__syncthreads) at the sums, one in four steps at least, and the
// compute warps' releases after them: the ring of rows and the votes' places are long
// enough for that.
template <bool CL>
__device__ __forceinline__ void chain_sync(bool relaxed = false) {
    if constexpr (CL) {
        __syncwarp();
        if (relaxed) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        else asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
}

// Orders what this warp saw or wrote before its relaxed arrival, for its own CTA.
__device__ __forceinline__ void cta_release() { asm volatile("fence.acq_rel.cta;" ::: "memory"); }

// The failure word: one past the step whose barrier the mover of a copy that did not
// land joins next (kNoFailure: none).  Every warp reads it between two runs of steps
// and stops if that step lies behind it: a mover that is already in the next run
// writes a later step, so that all warps of all CTAs stop at the same place,
// whichever of its writes they saw.
constexpr int kNoFailure = 0x7fffffff;
template <bool CL>
__device__ __forceinline__ int read_failure(const int *word) {
    int v;
    if constexpr (CL) asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(word)) : "memory");
    else asm volatile("ld.relaxed.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(word)) : "memory");
    return v;
}
// By the whole warp; the fence orders it before the warp's arrival for every CTA.
template <bool CL>
__device__ __forceinline__ void write_failure(int *word, int v, int lane, int ncta) {
    if constexpr (CL) {
        if (lane < ncta) {
            uint32_t a;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(word)), "r"(lane));
            asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
        }
        asm volatile("fence.acq_rel.cluster;" ::: "memory");
    } else if (lane == 0) {
        asm volatile("st.relaxed.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(word)), "r"(v) : "memory");
    }
}

// A lane group: 32 consecutive lanes of one chunk of states, JS = 2^lg adjacent
// lanes per state (state = s0 + (lane >> lg), below d1).
struct LaneGroup {
    int s0, d1, lg, v;  // first state, end of the chunk, lanes per state, number
};
__device__ __forceinline__ LaneGroup lane_group(const FrameDev &f, int v) {
    const int CD = f.chainCD, VW = f.chainVW;
    const int nck = (f.M + CD - 1) / CD;
    const int k = min(v / VW, nck - 1), idx = v - k * VW;
    LaneGroup g;
    g.d1 = min(f.M, (k + 1) * CD);
    g.lg = chain_lanes_lg(g.d1 - k * CD);
    g.s0 = k * CD + ((idx * 32) >> g.lg);
    g.v = v;
    return g;
}
// The W rows that lane groups [v0, v1) need, as a copy: aligned start (floats)
// and size within a symbol's block (blocks are 16-byte aligned).
struct ChunkGeom {
    int off;
    uint32_t bytes;
};
__device__ __forceinline__ ChunkGeom chunk_geom(const FrameDev &f, int dir, int v0, int v1) {
    const LaneGroup a = lane_group(f, v0), b = lane_group(f, v1 - 1);
    int r0 = a.s0, r1 = min(b.d1, b.s0 + (32 >> b.lg));
    if (dir == 0) {  // destination s gets sources s - nI .. s + n
        r0 = max(0, r0 - f.n * f.I);
        r1 = min(f.M, r1 + f.n);
    }
    ChunkGeom t;
    t.off = (r0 * f.MNS) & ~3;
    t.bytes = (uint32_t)(((r1 * f.MNS + 3) & ~3) - t.off) * 4u;
    return t;
}

// 2^-e for e in [-126, 127].
__device__ __forceinline__ float inv_pow2(int e) {
    return __int_as_float(e == 127 ? 0x00400000 : (127 - e) << 23);
}

// A lane's part in a step: its first term's place in a row, in the staged W and
// in the weights (floats), and its number of terms T.
struct Place {
    int s, T, coff, woff, voff;
    int sel;     // 8 direction + 4 edge + lg
    bool owner;  // the lane that writes the state
};

// One state's sum over the received lengths j = j0, j0 + J, ... (T terms; J = 2^LG
// lanes share the state), sum c[-+j] (w v[j]): four sums over t mod 4 of the full
// groups of four, the rest onto the first.  c, w, v point at the first term.
// A step waits for its slowest warp, so everything is straight-line code: MN at
// compile time makes every address an immediate offset, and a block's loads are
// issued before its arithmetic.  A row of 121 states (n = 8, I = 2) on 8 warps:
// 560 cycles a step so, 890-940 behind a jump on a run-time length, 760 with
// half the warps.
constexpr int kDotBlock = 4;  // groups whose loads are in flight together
template <int MN, int DIR, int LG>
__device__ __forceinline__ float chain_dot(const float *c, const float *w, const float *v, int js) {
    // every lane has all its lengths, j0 = js: v is the lane's row of weights
    constexpr int J = 1 << LG, MNS = MN | 1;
    constexpr int C = DIR == 0 ? -J : J, W = DIR == 0 ? J * (1 - MNS) : J;
    constexpr int Tmin = MN / J, Tmax = (MN + J - 1) / J, GF = Tmin / 4;
    float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int g0 = 0; g0 < GF; g0 += kDotBlock) {
        float4 q[kDotBlock];
        float cr[4 * kDotBlock], wr[4 * kDotBlock];
#pragma unroll
        for (int g = 0; g < kDotBlock; ++g) {
            if (g0 + g >= GF) break;
            q[g] = *reinterpret_cast<const float4 *>(v + 4 * (g0 + g));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                wr[4 * g + i] = w[(4 * (g0 + g) + i) * W];
                cr[4 * g + i] = c[(4 * (g0 + g) + i) * C];
            }
        }
#pragma unroll
        for (int g = 0; g < kDotBlock; ++g) {
            if (g0 + g >= GF) break;
            a[0] = fmaf(cr[4 * g], wr[4 * g] * q[g].x, a[0]);
            a[1] = fmaf(cr[4 * g + 1], wr[4 * g + 1] * q[g].y, a[1]);
            a[2] = fmaf(cr[4 * g + 2], wr[4 * g + 2] * q[g].z, a[2]);
            a[3] = fmaf(cr[4 * g + 3], wr[4 * g + 3] * q[g].w, a[3]);
        }
    }
    if constexpr (4 * GF < Tmax) {
        float cr[4], xr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 4 * GF + i;
            cr[i] = xr[i] = 0.f;
            if (t < Tmin || (t < Tmax && js + t * J < MN)) {
                cr[i] = c[t * C];
                xr[i] = w[t * W] * v[t];
            }
        }
        a[0] = fmaf(cr[0], xr[0], a[0]);
        if (Tmax >= 4 * GF + 4 && js + (4 * GF + 3) * J < MN) {  // four terms: a full group
            a[1] = fmaf(cr[1], xr[1], a[1]);
            a[2] = fmaf(cr[2], xr[2], a[2]);
            a[3] = fmaf(cr[3], xr[3], a[3]);
        } else {
            a[0] = fmaf(cr[1], xr[1], a[0]);
            a[0] = fmaf(cr[2], xr[2], a[0]);
        }
    }
    float r = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
    for (int o = 1; o < J; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}
// Any first length and number of terms per lane (a term past T loads nothing); v:
// the plain weights from j0 on.
template <int MN, int DIR, int LG>
__device__ __forceinline__ float chain_dot_edge(const float *c, const float *w, const float *v, int T) {
    constexpr int J = 1 << LG, MNS = MN | 1;
    constexpr int C = DIR == 0 ? -J : J, W = DIR == 0 ? J * (1 - MNS) : J;
    constexpr int NG = ((MN + J - 1) / J + 3) / 4;
    float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int g0 = 0; g0 < NG; g0 += 4) {
        float cr[16], wr[16], vr[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int t = 4 * g0 + i;
            cr[i] = wr[i] = vr[i] = 0.f;
            if (t < 4 * NG && t < T) {
                wr[i] = w[t * W];
                cr[i] = c[t * C];
                vr[i] = v[t * J];
            }
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            if (g0 + g >= NG) break;
            const bool full = 4 * (g0 + g) + 3 < T;
            a[0] = fmaf(cr[4 * g], wr[4 * g] * vr[4 * g], a[0]);
            const float x1 = wr[4 * g + 1] * vr[4 * g + 1], x2 = wr[4 * g + 2] * vr[4 * g + 2];
            const float b1 = fmaf(cr[4 * g + 1], x1, full ? a[1] : a[0]);
            a[1] = full ? b1 : a[1];
            a[0] = full ? a[0] : b1;
            const float b2 = fmaf(cr[4 * g + 2], x2, full ? a[2] : a[0]);
            a[2] = full ? b2 : a[2];
            a[0] = full ? a[0] : b2;
            a[3] = fmaf(cr[4 * g + 3], wr[4 * g + 3] * vr[4 * g + 3], a[3]);  // zero unless full
        }
    }
    float r = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
    for (int o = 1; o < J; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}
// Run-time MN (launches over several codes, uncommon lengths): the same sums in
// loops, plain weights.
template <int DIR>
__device__ __forceinline__ float chain_dot_any(int lg, int MNS, const float *c, const float *w,
                                               const float *v, int T) {
    const int J = 1 << lg, C = DIR == 0 ? -J : J, W = DIR == 0 ? J * (1 - MNS) : J;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    int t = 0;
#pragma unroll 2
    for (; t + 3 < T; t += 4) {
        const float w0 = w[0], w1 = w[W], w2 = w[2 * W], w3 = w[3 * W];
        const float c0 = c[0], c1 = c[C], c2 = c[2 * C], c3 = c[3 * C];
        const float v0 = v[0], v1 = v[J], v2 = v[2 * J], v3 = v[3 * J];
        a0 = fmaf(c0, w0 * v0, a0);
        a1 = fmaf(c1, w1 * v1, a1);
        a2 = fmaf(c2, w2 * v2, a2);
        a3 = fmaf(c3, w3 * v3, a3);
        c += 4 * C;
        w += 4 * W;
        v += 4 * J;
    }
    if (t < T) a0 = fmaf(c[0], w[0] * v[0], a0);
    if (t + 1 < T) a0 = fmaf(c[C], w[W] * v[J], a0);
    if (t + 2 < T) a0 = fmaf(c[2 * C], w[2 * W] * v[2 * J], a0);
    float r = (a0 + a1) + (a2 + a3);
    for (int o = 1; o < J; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}
// dot(c, w, v) of a lane group's kind `sel`, handed to fn at compile time.
template <int MN, typename Fn>
__device__ __forceinline__ void chain_with_dot(int sel, int MNS, int T, int js, Fn &&fn) {
    using F = const float *;
    if constexpr (MN == 0) {
        if (sel & 8) fn([&](F c, F w, F v) { return chain_dot_any<1>(sel & 3, MNS, c, w, v, T); });
        else fn([&](F c, F w, F v) { return chain_dot_any<0>(sel & 3, MNS, c, w, v, T); });
    } else {
#define MAPDEC_CHAIN_D(D, LG)                                                                     \
    case 8 * D + LG: fn([&](F c, F w, F v) { return chain_dot<MN, D, LG>(c, w, v, js); }); break; \
    case 8 * D + 4 + LG: fn([&](F c, F w, F v) { return chain_dot_edge<MN, D, LG>(c, w, v, T); }); break;
        switch (sel) {
            MAPDEC_CHAIN_D(0, 0) MAPDEC_CHAIN_D(0, 1) MAPDEC_CHAIN_D(0, 2) MAPDEC_CHAIN_D(0, 3)
            MAPDEC_CHAIN_D(1, 0) MAPDEC_CHAIN_D(1, 1) MAPDEC_CHAIN_D(1, 2) MAPDEC_CHAIN_D(1, 3)
        }
#undef MAPDEC_CHAIN_D
    }
}

// The weights 2^{(theta - 1) j} in shared memory, zero from j = MN on: the plain
// table, then for a chunk's lanes per state (2^lg) lane js's weights of its
// lengths js, js + 2^lg, ... in a row of their own, read four at a time.
constexpr int kWtPlain = 2 * kMaxMN, kWtLane = kMaxMN + 32;  // floats
__host__ __device__ constexpr int wt_stride(int lg) { return (kMaxMN >> lg) + 4; }
struct WeightTab {
    float plain[kWtPlain];
    float lane[2][kWtLane];  // full chunks, last chunk
};

// Exponential tilt.  The forward metric alpha_i(m) is the joint probability of
// a received prefix of L = n i + m bits, so a row falls off roughly like
// 2^{-h L} (h: entropy rate of the received bits) on top of the drift
// posterior; the backward metric rises the same way.  Far apart in FP32, the
// entries that carry the posterior would underflow.  The chains therefore store
//   alpha^_i(m) = alpha_i(m) 2^{theta_i L} / Z_i,   beta^_i(m) = beta_i(m) 2^{-theta'_i L} / Y_i
// with tilts theta driven toward h by the row sums: with a tilt theta a step
// grows the row sum by about 2^{(theta - h) n}, so theta_{i+1} = theta_i -
// g log2(growth) / n (g = 1/(steps+1), floored at kTiltGainMin); after the
// first kTiltSettle steps it is updated every kTiltEvery steps from the mean
// growth of the steps since.  The producers already weight every received bit
// by 2 (theta = 1), so a step multiplies the transition sums by
// 2^{(theta - 1) j} (j = received length) and pre-scales the source row by
// 2^{(theta_{i+1} - theta_i)(m - mean)}.  Rows are divided by powers of two
// (exact), so Z_i is a power of two times the tilt factors, kept exactly in an
// integer and FP64, and log P(Y) = log alpha^_N(rho - tau) + log Z_N - theta_N
// rho log 2.  The APP producer applies the matching exact factor; the per-row
// constants cancel in the APPs and in the gradient.
//
// One recursion is a serial chain of N steps, each a banded product of the row
// with W_i, so what counts is a step's latency: a single frame has no other
// work, and a batch waits for its longest frame.  What bounds a step is the
// number of dependent instructions of its slowest warp (a row of 121 states:
// about 1000 clocks, 500 of them the sums, 110 the barrier; W_i, 12 KB, streams
// in a fifth of that), so:
//   - A plain step has one barrier and no reduction.  Rows go round a ring of
//     shared buffers; the sums (power-of-two scaling, tilt controller) of the
//     rows since the last tilt update are formed together at the next one, eight
//     sums in one reduction of nine shuffles, and each thread runs the
//     controller on the same numbers, so nothing is broadcast.  A row whose
//     entries all fell below kRowLow (a vote in the step's barrier) is summed
//     and scaled at once.
//   - Plain steps run in a loop of their own, its sums compiled for the frame's
//     MN and the warp's kind (chain_dot).
//   - Two more warps do what is not arithmetic.  The mover issues the bulk copies
//     of W_i (cp.async.bulk on mbarriers, every wait bounded, several steps
//     ahead), waits for the next step's before it joins the step's barrier, and
//     writes the tilts and the FP64 record; the storer writes the summed rows,
//     scaled, to global memory, one a step (and in a cluster the tilts and means,
//     see chain_sync).
//   - A row of many states takes a warp per lane group, and, with SMs idle, the
//     CTAs of a cluster: each stages its part of W_i (one SM streams 64 bytes a
//     clock) and stores its states into every CTA's row buffers through
//     distributed shared memory.
// The order of the additions is the same for every split: states are summed in
// chunks of chainCD over 256 virtual lanes, whatever CTAs, warps and staged
// chunks do the work; k_chain_crowd adds in that order too with 256 threads and its
// default chunks (another block size or budget changes its lanes per state).
// Whole decodes with k_chain_crowd's kernel in its place and with this one: one
// frame N = 1000, M = 401, MN = 31: 3.24 -> 1.69 ms; N = 300, M = 81, MN = 25: 638 ->
// 420 us; gradients of N = 1000, M = 121, MN = 25: 2.36 -> 1.48 ms; 64 stream frames
// N = 1000, M = 171: 4.66 -> 3.68 ms; 8 frames N = 8000, M = 1661, MN = 49,
// checkpointed: 287 -> 208 ms.
// Bookkeeping that every warp repeats is kept to one step counter, and what only
// the storer needs to shared memory (with more live values the 512-thread modes
// spill, and a cluster barrier waits for the spills' stores: 1.45 -> 1.61 ms).
// Recursions alone, with a counter per quantity and so: N = 50, M = 41 99.9 -> 91.7
// us; N = 300, M = 81 298 -> 282; N = 1000, M = 121 861 -> 803; N = 1000, M = 401
// 1481 -> 1447; 64 stream frames M = 171 1141 -> 1070.
template <int MNT, int MODE>
__global__ void __launch_bounds__(MODE == kChainNarrow ? kChainMostThreads : kChainMaxThreads) k_chain(
    const FrameDev *__restrict__ frames, const Work *__restrict__ work) {
    constexpr bool CL = MODE == kChainCluster, WIDE = MODE != kChainNarrow;
    const int rank = CL ? (int)cluster_rank() : 0;
    const int ncta = CL ? (int)cluster_size() : 1;
    const Work wk = work[CL ? blockIdx.x / ncta : blockIdx.x];
    const FrameDev &f = frames[wk.frame];
    const int dir = wk.tile & 1;  // 0 = forward (alpha), 1 = backward (beta); bit 1: replay
    const int M = f.M, Mp = f.Mp, MNS = f.MNS, MN = MNT ? MNT : f.MN, n = f.n, N = f.N, xmax = f.xmax;
    const long long rho = f.rho, wblk = f.wblk;
    const int NST = f.chainStages, RB = f.chainRing;
    const uint32_t wait_limit = f.wait_limit;
    const int i0 = f.seg_i0, i1 = f.seg_i1;  // symbols of this launch (segment)
    const int nsteps = i1 - i0;
    const int send = (int)(rho - (long long)n * N) + xmax;  // state of the end drift
    const bool segm = (f.chain_flags & CH_SEGMENTED) != 0;
    const bool replay = dir == 0 && (wk.tile & 2) != 0;
    // first launch of this direction: the frame boundary; otherwise the row carried over
    const bool fresh = dir == 0 ? (i0 == 0) : (i1 == N);
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), NCW = (nthr >> 5) - 2;
    // the last two warps: copies and records; rows to global memory
    const bool mover = warp == NCW, storer = warp == NCW + 1, helper = warp >= NCW;
    // lane groups of this CTA and its staged chunks of CK of them
    const int NV = f.chainNV, VC = f.chainVC, CK = f.chainCK;
    const int vA = min(NV, rank * VC), vB = min(NV, vA + VC);
    const int nck = max(1, (vB - vA + CK - 1) / CK);  // a CTA without states steps along

    __shared__ uint64_t bar[kMaxStages];
    __shared__ int s_alive[kAliveSlots];  // clusters, by step: some entry >= kRowLow
    __shared__ int s_fail;      // see kNoFailure
    __shared__ __align__(16) float s_red[8][8];   // [2 row + (sum, moment)][virtual warp]
    __shared__ __align__(16) WeightTab wtab[2];
    extern __shared__ float4 sm4[];
    // RB rows of RS floats, state s at kChainRowPad + s, zero outside [0, M)
    const int RS = Mp + 2 * kChainRowPad;
    float *rows = reinterpret_cast<float *>(sm4) + kChainRowPad;
    // each compute warp's lane groups in order, then one past every chunk
    LaneGroup *grp = reinterpret_cast<LaneGroup *>(reinterpret_cast<float *>(sm4) + RB * RS);
    const int LL = f.chainList;  // entries per warp
    int4 *const ptab0 = reinterpret_cast<int4 *>(grp + NCW * LL);
    ChunkGeom *tab = reinterpret_cast<ChunkGeom *>(ptab0 + (size_t)NCW * (LL - 1) * 32);
    const int nckMax = (VC + CK - 1) / CK;
    float *stage0 = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(tab) +
                                              ((nckMax * sizeof(ChunkGeom) + 15) & ~(size_t)15));
    const size_t stageFloats = f.chainStageFloats;

    // Narrow: warp w takes the groups of virtual warp w (lanes 32 w .. of every
    // chunk, in rounds of 256), so its lanes hold the summation order's partial
    // sums in registers.  Else: contiguous groups in turn.
    for (int e = tid; e < NCW * LL; e += nthr) {
        const int w = e / LL, t = e - w * LL;
        int v;
        if (WIDE) {
            v = vA + w + t * NCW;
            if (v >= vB) v = -1;
        } else {
            const int VW = f.chainVW, ncan = (M + f.chainCD - 1) / f.chainCD;
            const int VL = NV - (ncan - 1) * VW;                    // groups of the last chunk
            const int cF = w < VW ? ((VW - 1 - w) >> 3) + 1 : 0;    // this warp's of a full one
            const int cL = w < VL ? ((VL - 1 - w) >> 3) + 1 : 0;    // and of the last
            const int tL = t - (ncan - 1) * cF;
            if (tL < 0) v = t / cF * VW + 8 * (t % cF) + w;
            else v = tL < cL ? (ncan - 1) * VW + 8 * tL + w : -1;
        }
        LaneGroup g = {0, 0, 0, 1 << 30};
        if (v >= 0) g = lane_group(f, v);
        grp[e] = g;
    }
    // Chunk table, and a self-check of every copy it implies: source inside
    // this launch's symbols of W (plus the 16-float tail slack), destination
    // inside its stage, 16-byte alignment and size.  The check covers the
    // chunks of every CTA of the cluster, so that they all take the same way:
    // a violation records ST_ARG and the recursion does not start.
    bool bad_geom = ((uintptr_t)f.W & 15) != 0 || (wblk & 3) != 0 || ((uintptr_t)stage0 & 15) != 0 ||
                    (stageFloats & 3) != 0 || (long long)VC * ncta < NV || NCW < 1 ||
                    NST > kMaxStages || RB < 2;
    for (int e = tid; e < ncta * nckMax && !bad_geom; e += nthr) {
        const int r = e / nckMax, k = e - r * nckMax;
        const int g0 = min(NV, r * VC), g1 = min(NV, g0 + VC), v0 = g0 + k * CK;
        if (v0 < g1) {
            const ChunkGeom g = chunk_geom(f, dir, v0, min(g1, v0 + CK));
            if (g.off + (long long)g.bytes / 4 > wblk + 16 || g.bytes / 4 > stageFloats) bad_geom = true;
            if (r == rank) tab[k] = g;
        }
    }
    if (tid == 0) {
        for (int st = 0; st < NST; ++st) mbar_init(&bar[st], 1);
        fence_mbar_init();
    }
    for (int e = tid; e < RB * RS; e += nthr) reinterpret_cast<float *>(sm4)[e] = 0.f;
    for (int e = tid; e < 2 * (int)(sizeof(WeightTab) / 4); e += nthr) wtab[0].plain[e] = 0.f;
    for (int e = tid; e < 64; e += nthr) s_red[0][e] = 0.f;
    if (tid < kAliveSlots) s_alive[tid] = 0;
    if (tid == 0) s_fail = kNoFailure;
    if (__syncthreads_or(bad_geom ? 1 : 0)) {  // nothing issued yet
        if (tid == 0) atomicMax(f.status, ST_ARG);
        return;
    }

    // The mover's copies: chunk g = (step, k) in order into stage g % NST.
    int total = vB > vA ? nsteps * nck : 0;
    int issued = 0, is_k = 0, is_slot = 0;
    const float *is_src = f.W + (size_t)(dir == 0 ? i0 : i1 - 1) * wblk;  // symbol block of the next copy
    const long long is_step = dir == 0 ? wblk : -wblk;
    // testing: a copy that is never issued, every CTA's first or a later one of the last CTA
    const int tcopy = f.test_flags >> kTestCopyShift;
    const int skip = (f.test_flags & TEST_SKIP_COPY) && (tcopy == 0 || rank == ncta - 1) ? tcopy : -1;
    auto issue_next = [&]() {
        if (lane == 0 && issued != skip) {
            const ChunkGeom g = tab[is_k];
            mbar_expect_tx(&bar[is_slot], g.bytes);
            bulk_g2s(stage0 + (size_t)is_slot * stageFloats, is_src + g.off, g.bytes, &bar[is_slot]);
        }
        ++issued;
        if (++is_k == nck) { is_k = 0; is_src += is_step; }
        if (++is_slot == NST) is_slot = 0;
    };
    // chunk `waited` has landed before the CTA passes the barrier of `step` that follows;
    // a wait that gives up tells every CTA, and issues no further copy (its stage's
    // barrier has not completed the phase that the next copy would count on)
    int waited = 0, wt_slot = 0;
    uint32_t wt_ph = 0;
    auto wait_next = [&](int step) {
        if (waited >= total) return;
        if (!__all_sync(0xffffffffu, mbar_wait(&bar[wt_slot], wt_ph, wait_limit))) {
            write_failure<CL>(&s_fail, step + 1, lane, ncta);
            total = issued;
        }
        ++waited;
        if (++wt_slot == NST) { wt_slot = 0; wt_ph ^= 1u; }
    };

    // Start row.  Stream decoding: a boundary drift prior replaces the point
    // mass (alpha_0 = phi0, beta_N = phiN; Sec. II-C).  In the tilted rows the
    // start row is alpha^_0(m) = phi0(m) 2^m / Z_0 (tilt 1, received length m)
    // and the end row beta^_N(m) is proportional to phiN(m) 2^-m; both are first
    // scaled by 2^-emax (emax the largest exponent over the prior's support,
    // exact), then divided by the power of two below their sum like every row,
    // and log2 Z_0 = emax + that exponent starts the forward record.
    const float *prior = !fresh ? nullptr : (dir == 0 ? f.phi0 : f.phiN);
    int zexp = 0;  // log2 Z of the last summed row: integer part
    float mean0 = (dir == 0) ? 0.f : (float)(send - xmax);
    if (prior) {
        __shared__ int s_emax;
        if (tid == 0) s_emax = -(1 << 30);
        __syncthreads();
        for (int s = tid; s < M; s += nthr)
            if (prior[s] > 0.f) atomicMax(&s_emax, dir == 0 ? s - xmax : xmax - s);
        __syncthreads();
        const int emax = s_emax;
        for (int s = tid; s < M; s += nthr) {
            const float w = prior[s];
            const int e = (dir == 0 ? s - xmax : xmax - s) - emax;  // <= 0
            rows[s] = (w > 0.f && e > -150) ? ldexpf(w, e) : 0.f;
        }
        __syncthreads();
        for (int wi = tid >> 5; wi < 8; wi += nthr >> 5) {
            float a = 0.f, b = 0.f;
            for (int s = wi * 32 + lane; s < M; s += 256) {
                a += rows[s];
                b = fmaf(rows[s], (float)(s - xmax), b);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                b += __shfl_xor_sync(0xffffffffu, b, o);
            }
            if (lane == 0) { s_red[0][wi] = a; s_red[1][wi] = b; }
        }
        __syncthreads();
        float c0 = 0.f, cm0 = 0.f;
        for (int w = 0; w < 8; ++w) { c0 += s_red[0][w]; cm0 += s_red[1][w]; }
        if (!(c0 > 0.f)) {  // no mass inside the drift limits (same in every thread and CTA)
            if (tid == 0) atomicMax(f.status, ST_ZERO);
            return;         // nothing issued yet
        }
        int ex;
        frexpf(c0, &ex);
        const float inv = ldexpf(1.f, 1 - ex);
        for (int s = tid; s < M; s += nthr) rows[s] *= inv;
        zexp = emax + ex - 1;
        mean0 = cm0 / c0;
    } else {
        for (int s = tid; s < M; s += nthr) {
            if (fresh) rows[s] = (s == (dir == 0 ? xmax : send)) ? 1.f : 0.f;
            else rows[s] = (dir == 0) ? f.ckpt[s] : f.bedge[s];
        }
    }
    float *const grow = (dir == 0) ? f.alpha + (size_t)i0 * Mp : f.beta + (size_t)i1 * Mp;
    const long long gstep = dir == 0 ? Mp : -Mp;  // row t of this launch: grow + t gstep
    if (rank == 0)
        for (int s = tid; s < M; s += nthr) grow[s] = rows[s];  // this thread's own entries

    // Controller state, the same in every thread; ztilt (the tilt terms of log2
    // Z, FP64) in the mover.
    float theta = 1.f, mean = mean0;
    float lrow = 0.f;     // log2 of the current row's sum
    float lc_prev = 0.f;  // sum of log2 growth since the last tilt update
    int lc_cnt = 0;       // number of steps in lc_prev
    int steps0 = 0;       // steps of this direction before this launch
    double ztilt = 0.0;
    if (!fresh && segm && !replay) {
        const ChainState &cs = f.cst[dir];
        theta = cs.theta;
        mean = cs.mean;
        lc_prev = cs.lc_sum;
        lrow = cs.lrow;
        lc_cnt = cs.lc_cnt;
        steps0 = cs.steps;
        zexp = (int)cs.zexp;
        ztilt = cs.ztilt;
    }
    double *const thr_ = dir == 0 ? f.thf : f.thb;
    double *const mcr = f.mcf;
    // replay: the recorded tilts, read a step ahead
    float th_next = 0.f, mc_next = 0.f;
    if (replay) {
        theta = (float)thr_[i0];
        th_next = (float)thr_[i0 + 1];
        mc_next = (float)mcr[i0];
    }
    const bool record = rank == 0 && !replay;
    // the warp that writes tilts and means: of a cluster the one whose stores nothing waits for
    const bool recorder = CL ? storer : mover;
    if (record && fresh && tid == 0) {
        thr_[dir == 0 ? 0 : N] = 1.0;
        if (dir == 0) mcr[0] = (double)mean0;
    }
    const int lgA = chain_lanes_lg(min(f.chainCD, M));
    const int lgB = chain_lanes_lg(M - (M - 1) / f.chainCD * f.chainCD);
    const int wtA = (tid & ((1 << lgA) - 1)) * wt_stride(lgA) + (tid >> lgA);
    const int wtB = (tid & ((1 << lgB) - 1)) * wt_stride(lgB) + (tid >> lgB);
    auto fill_weights = [&](WeightTab &t, float th) {
        for (int j = tid; j < MN; j += nthr) {  // one length a thread (64 threads or more)
            const float x = exp2f((th - 1.f) * (float)j);
            t.plain[j] = x;
            t.lane[0][wtA] = x;
            t.lane[1][wtB] = x;
        }
    };
    float th_tab = theta;  // the tilt wtab[vp] holds
    int vp = 0;
    fill_weights(wtab[0], theta);
    if (mover) {
        while (issued < NST && issued < total) issue_next();
    }

    // Sums of the rows built since the last time (pend of them), in the order of
    // 256 virtual lanes: partial sums and first moments x[2 k], x[2 k + 1] of this
    // lane (k = 3 the last row), butterflies into s_red[.][virtual warp].
    int pend = 0, cur = 0;  // cur: the last row's buffer in the ring (floats)
    const int rowE = RB * RS;
    const int CD = f.chainCD, nwi = f.chainVWarps;
    float x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = 0.f;
    auto reduce_rows = [&](int wi) {
        if (pend == 1) {
            float p = x[6], q = x[7];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                p += __shfl_xor_sync(0xffffffffu, p, o);
                q += __shfl_xor_sync(0xffffffffu, q, o);
            }
            if (lane == 0) {
                s_red[6][wi] = p;
                s_red[7][wi] = q;
            }
        } else {
            // eight butterfly sums at once: each exchange halves the sums a lane
            // carries; lanes 4 k .. 4 k + 3 end with sum k
            float y[4], z[2];
            const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                y[k] = (h4 ? x[k + 4] : x[k]) + __shfl_xor_sync(0xffffffffu, h4 ? x[k] : x[k + 4], 16);
#pragma unroll
            for (int k = 0; k < 2; ++k)
                z[k] = (h3 ? y[k + 2] : y[k]) + __shfl_xor_sync(0xffffffffu, h3 ? y[k] : y[k + 2], 8);
            float r = (h2 ? z[1] : z[0]) + __shfl_xor_sync(0xffffffffu, h2 ? z[0] : z[1], 4);
            r += __shfl_xor_sync(0xffffffffu, r, 2);
            r += __shfl_xor_sync(0xffffffffu, r, 1);
            if ((lane & 3) == 0) s_red[lane >> 2][wi] = r;
        }
    };
    // wide: the same partial sums from the rows in shared memory
    auto gather_rows = [&]() {
        for (int wi = warp; wi < nwi; wi += NCW + 2) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = 0.f;
            for (int s00 = 0; s00 < M; s00 += CD) {
                const int nst = min(CD, M - s00), lg = chain_lanes_lg(nst), js = (1 << lg) - 1;
                for (int l = wi * 32 + lane; l < (nst << lg); l += 256) {
                    const int s = s00 + (l >> lg);
                    const float m = (float)(s - xmax);
                    int q = cur;
#pragma unroll
                    for (int k = 3; k >= 0; --k) {
                        const float v = (l & js) || k < 4 - pend ? 0.f : rows[q + s];
                        x[2 * k] += v;
                        x[2 * k + 1] = fmaf(v, m, x[2 * k + 1]);
                        q = q == 0 ? rowE - RS : q - RS;
                    }
                }
            }
            reduce_rows(wi);
        }
    };
    // The sums' record for the tilt controller, and each row's power of two.
    // False: a row had no usable sum.
    float sc_last = 1.f;            // scales the last summed row
    int rec_row = -1;               // recorder: a row whose mean is to be recorded
    float rec_mean = 0.f;
    __shared__ float s_qs[4];       // storer: scales of the rows to store, the last in entry 3
    int qn = 0, qb = 0;             // how many, buffer of the first
    int qr = 0;                     // and its row number
    // st: the row number of the last one in this launch
    auto sum_rows = [&](int st) -> bool {
        bool good;
        float mn;
        if (pend == 1) {
            float c, cm;
            const float4 a0 = *reinterpret_cast<const float4 *>(&s_red[6][0]);
            const float4 a1 = *reinterpret_cast<const float4 *>(&s_red[6][4]);
            const float4 b0 = *reinterpret_cast<const float4 *>(&s_red[7][0]);
            const float4 b1 = *reinterpret_cast<const float4 *>(&s_red[7][4]);
            c = ((((((a0.x + a0.y) + a0.z) + a0.w) + a1.x) + a1.y) + a1.z) + a1.w;
            cm = ((((((b0.x + b0.y) + b0.z) + b0.w) + b1.x) + b1.y) + b1.z) + b1.w;
            good = c >= 1.2e-38f && c <= 3.0e38f;
            const int e = (__float_as_int(c) >> 23) - 127;  // c = m 2^e, m in [1, 2)
            const float l = log2f(c);
            mn = cm / c;
            lc_prev += l - lrow;
            lrow = l - (float)e;
            zexp += e;
            sc_last = inv_pow2(e);
            if (storer && lane == 0) s_qs[3] = sc_last;
            if (record && dir == 0 && recorder && lane == 0) { rec_row = i0 + st; rec_mean = mn; }
        } else {
            // lane 2 k: sum c of row k; lane 2 k + 1: its first moment
            const float4 ra = *reinterpret_cast<const float4 *>(&s_red[lane & 7][0]);
            const float4 rb = *reinterpret_cast<const float4 *>(&s_red[lane & 7][4]);
            const float c = ((((((ra.x + ra.y) + ra.z) + ra.w) + rb.x) + rb.y) + rb.z) + rb.w;
            const float cm = __shfl_xor_sync(0xffffffffu, c, 1);
            const int e = (__float_as_int(c) >> 23) - 127;
            const int k0 = 4 - pend;
            // the row before it still carried the power of two of its own sum
            int dp = __shfl_up_sync(0xffffffffu, e, 2);
            if ((lane & 7) < 2 * (k0 + 1)) dp = 0;
            const float co = c * inv_pow2(dp);
            const float lc = log2f(co);
            mn = cm / c;
            const unsigned ok = __ballot_sync(0xffffffffu, c >= kSumLow && c <= 3.0e38f && co >= 1.2e-38f && co <= 3.0e38f);
            good = (ok & ((0x55u << (2 * k0)) & 0x55u)) == ((0x55u << (2 * k0)) & 0x55u);
            const int row = (lane >> 1) - k0;  // rows since the last time
            if (record && dir == 0 && recorder && lane < 8 && !(lane & 1) && row >= 0) {
                rec_row = i0 + st - (pend - 1 - row);
                rec_mean = mn;
            }
            const int eo = e - dp;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (k >= k0) {
                    const float l = __shfl_sync(0xffffffffu, lc, 2 * k);
                    const int ek = __shfl_sync(0xffffffffu, eo, 2 * k);
                    lc_prev += l - lrow;
                    lrow = l - (float)ek;
                    zexp += ek;
                }
            }
            mn = __shfl_sync(0xffffffffu, mn, 6);
            const float sc = inv_pow2(e);
            sc_last = __shfl_sync(0xffffffffu, sc, 6);
            if (storer && lane < 8 && !(lane & 1)) s_qs[lane >> 1] = sc;
        }
        lc_cnt += pend;
        mean = mn;
        if (storer) {
            qn = pend;
            qb = cur - (pend - 1) * RS;
            if (qb < 0) qb += rowE;
            qr = st - (pend - 1);
            __syncwarp();
        }
        pend = 0;
        return good;
    };
    // The storer writes a summed row, scaled, to global memory: one a step.
    auto store_row = [&]() {
        if (qn == 0) return;
        const float *r = rows + qb;
        const float sc = s_qs[4 - qn];
        float *const g = grow + qr * gstep;
        for (int s = rank * 32 + lane; s < M; s += 32 * ncta) g[s] = r[s] * sc;
        ++qr;
        qb = qb + RS == rowE ? 0 : qb + RS;
        --qn;
    };

    auto place = [&](LaneGroup g, int vlo, int vhi) {
        g.lg &= 255;
        Place p;
        p.s = g.s0 + (lane >> g.lg);
        const int js = lane & ((1 << g.lg) - 1);
        p.owner = p.s < g.d1 && js == 0;
        const int s = min(p.s, g.d1 - 1);  // lanes past the chunk repeat its last state
        int jlo, jhi;
        if (dir == 0) {  // alpha'(s) = sum_j alpha(s - j + n) W[s - j + n][j] vtab[j]
            jlo = max(0, s + n - vhi);
            jhi = min(MN - 1, s + n - vlo);
        } else {         // beta'(s) = sum_j W[s][j] vtab[j] beta(s + j - n)
            jlo = max(0, n - s);
            jhi = s >= vlo && s <= vhi ? min(MN - 1, M - 1 - s + n) : -1;
        }
        int j0 = jlo + js;
        p.T = jhi >= j0 ? ((jhi - j0) >> g.lg) + 1 : 0;
        if (p.T == 0) j0 = js;  // no term: any place inside the tables
        const bool edge = MNT == 0 || __any_sync(0xffffffffu, jlo != 0 || jhi != MN - 1);
        p.sel = 8 * dir + (edge ? 4 : 0) + g.lg;
        p.coff = dir == 0 ? s + n - j0 : s - n + j0;
        p.woff = dir == 0 ? (s + n) * MNS + j0 * (1 - MNS) : s * MNS + j0;
        p.voff = edge ? j0 : kWtPlain + (g.d1 == M ? kWtLane : 0) + js * wt_stride(g.lg);
        return p;
    };
    // steps whose every W row is valid: window starts n i + s - xmax inside [0, rho]
    const int iin0 = (xmax + n - 1) / n;
    const int iin1 = rho >= xmax ? (int)min((rho - xmax) / n, (long long)N) : -1;
    // A warp with one lane group keeps its place of such a step.
    const LaneGroup *list = grp + (helper ? 0 : warp) * LL;
    // With several, the places of such a step are kept in shared memory (and the
    // kind of a group's sums in its lg field, from bit 8 on).
    int4 *const ptab = ptab0 + (helper ? 0 : warp) * (LL - 1) * 32;
    if (!helper && (nck > 1 || LL > 2 || CL))
        for (int t = 0; list[t].v < NV; ++t) {
            const Place p = place(list[t], 0, M - 1);
            ptab[t * 32 + lane] = make_int4(p.coff, p.woff, p.voff | p.T << 16, p.s | (p.owner ? 1 << 30 : 0));
            __syncwarp();
            if (lane == 0) grp[warp * LL + t].lg |= p.sel << 8;
            __syncwarp();
        }
    const LaneGroup g0 = list[0];
    Place kept = {0, 0, 0, 0, 0, 0, false};
    if (!helper && g0.v < NV) kept = place(g0, 0, M - 1);
    const bool has = !helper && g0.v < NV;  // else `kept` is no place to read from

    // The step's barrier; true where some entry of the new row is not small.
    auto step_sync = [&](int step, bool some) -> bool {
        if constexpr (CL) {
            int *const vote = &s_alive[step & (kAliveSlots - 1)];
            if (__any_sync(0xffffffffu, some) && lane < ncta) st_cluster(vote, lane, 1);
            chain_sync<true>(helper);
            return *vote != 0;
        } else {
            return __syncthreads_or(some ? 1 : 0) != 0;
        }
    };
    bool failed = false, alive = true, ready = false;
    const int cap = f.chainCap;
    const bool inplace = f.chainRing == 2;
    int slot = 0;  // the coming chunk's stage (floats)
    const int slotB = (int)stageFloats, slotE = NST * slotB;
    const int off0 = vB > vA ? tab[0].off : 0;
    const float *const wts = wtab[0].plain;
    constexpr int kWt = sizeof(WeightTab) / 4;
    // the steps [q0, q1) with every W row valid, in a CTA whose warps have one
    // lane group each: a loop of their own
    int q0 = nsteps, q1 = nsteps;
    if (nck == 1 && LL <= 2) {
        q0 = max(0, dir == 0 ? iin0 - i0 : i1 - 1 - iin1);
        q1 = min(nsteps, dir == 0 ? iin1 - i0 + 1 : i1 - iin0);
    }
    // every CTA of the cluster runs and has set up its shared memory
    if constexpr (CL) chain_sync<true>();
    if (mover) wait_next(-1);
    chain_sync<CL>();  // rows, first chunk ready in every CTA
    int st = 0;
    while (st < nsteps) {
        const int steps = steps0 + st;
        const bool gave_up = read_failure<CL>(&s_fail) <= st;
        // the votes' places of the four steps after this run's (four at most)
        if (CL && tid < kRunMost) s_alive[(st + kRunMost + tid) & (kAliveSlots - 1)] = 0;
        const bool due = replay || tilt_due(steps);
        const bool summed = pend > 0 && (ready || !alive);
        bool good = true;
        if (summed) {
            if (storer)
                while (qn > 0) store_row();
            if (WIDE) {
                gather_rows();
                __syncthreads();
            } else if (!ready) {
                if (!helper && has) reduce_rows(warp);
                __syncthreads();
            }
            good = sum_rows(st);
            alive = true;
        }
        if (gave_up || !good) {
            failed = true;
            break;
        }
        // tilt of the new row (the recompute sweep replays the recorded ones)
        float tn = theta;
        if (replay) {
            tn = th_next;
            mean = mc_next;
            if (st + 1 < nsteps) {
                th_next = (float)thr_[i0 + st + 2];
                mc_next = (float)mcr[i0 + st + 1];
            }
        } else if (due) {
            if (steps > 0 && lc_cnt > 0) {
                // gain = cnt / (steps + 1) within [kTiltGainMin, 1]; cnt is 4 once settled
                const float gain = steps >= 64 * lc_cnt
                                       ? kTiltGainMin
                                       : fminf(1.f, fmaxf(kTiltGainMin, (float)lc_cnt / (float)(steps + 1)));
                const float avg = lc_cnt == 4 ? lc_prev * 0.25f : (lc_cnt == 1 ? lc_prev : lc_prev / (float)lc_cnt);
                const float dt = fminf(kTiltStepMax, fmaxf(-kTiltStepMax, -gain * avg / (float)n));
                tn = fminf(kTiltMax, fmaxf(kTiltMin, theta + dt));
            }
            lc_prev = 0.f;
            lc_cnt = 0;
        }
        float dth = dir == 0 ? tn - theta : theta - tn;
        // the row's power of two, and forward its change of tilt (backward: on
        // the new row), into the next buffer: the storer writes the row as it was
        const bool pre = dir == 0 && dth != 0.f;
        int wt = vp * kWt;
        if (summed || pre) {
            const float sc = summed ? sc_last : 1.f;
            int to = cur + RS == rowE ? 0 : cur + RS;
            if (inplace) to = cur;
            for (int s = tid; s < M; s += nthr) {
                float v = rows[cur + s] * sc;
                if (inplace && summed && rank == 0) grow[st * gstep + s] = v;
                if (pre) v *= exp2f(dth * ((float)(s - xmax) - mean));
                rows[to + s] = v;
            }
            if (inplace) qn = 0;
            cur = to;
        }
        // weights 2^{(theta - 1) j}: forward of the new tilt, backward of the
        // source row's (the other table, from the next step on)
        if (tn != th_tab) {
            if (dir == 1) vp ^= 1;
            fill_weights(wtab[vp], tn);
            th_tab = tn;
        }
        if (summed || pre) __syncthreads();
        // FP64 records, while the other warps compute
        if (mover || (CL && storer)) {
            if (mover && dir == 0 && tn != theta)
                ztilt += (double)(tn - theta) * ((double)n * (i0 + st) + (double)mean);
            if (rec_row >= 0) mcr[rec_row] = (double)rec_mean;
            rec_row = -1;
        }
        theta = tn;
        // steps until the rows are summed again, at the last of them unless the
        // recompute sweep needs no sums there
        const int run = replay || steps < kTiltSettle
                            ? 1
                            : min(min(nsteps - st, cap - pend), kTiltEvery - (steps & (kTiltEvery - 1)));
        const bool sums = !replay || st + 1 == nsteps || pend + 1 == cap || th_next != tn;
        const int quick = st >= q0 ? min(run, q1 - st) : 0;
        int done = 0;
        if (quick > 0) {
            const bool fin = sums && quick == run;
            int u = 0;
            if (mover) {
                double *tr = thr_ + (dir == 0 ? i0 + st + 1 : i1 - 1 - st);
                const double tnd = (double)tn;
                for (;;) {
                    if (!CL && record && lane == 0) *tr = tnd;
                    tr += dir == 0 ? 1 : -1;
                    wait_next(st + u);
                    if (CL) cta_release();
                    alive = step_sync(st + u, false);
                    if (issued < total) issue_next();
                    if (++u == quick || !alive) break;
                }
            } else if (storer || !has) {  // (a warp without states only keeps the barriers)
                do {
                    if (storer) {
                        if (CL && record && lane == 0)
                            thr_[dir == 0 ? i0 + st + u + 1 : i1 - 1 - st - u] = (double)tn;
                        store_row();
                    }
                    alive = step_sync(st + u, false);
                } while (++u < quick && alive);
            } else {
                chain_with_dot<MNT>(kept.sel, MNS, kept.T, lane & ((1 << (kept.sel & 3)) - 1), [&](auto dot) {
                    const float m = (float)(kept.s - xmax);
                    const bool mine = kept.owner;
                    int at = cur, sl = slot;
                    const float *vw = wts + (wt + kept.voff);
                    for (;;) {
                        float acc = dot(rows + (at + kept.coff), stage0 + (sl - off0 + kept.woff), vw);
                        at = at + RS == rowE ? 0 : at + RS;
                        sl = sl + slotB == slotE ? 0 : sl + slotB;
                        if (dir == 1 && dth != 0.f) {  // the first step after an update
                            acc *= exp2f(dth * (m - mean));
                            dth = 0.f;
                            vw = wts + (vp * kWt + kept.voff);
                        }
                        if (mine) {
                            rows[at + kept.s] = acc;
                            if (CL)
                                for (int r = 0; r < ncta; ++r)
                                    if (r != rank) st_cluster(&rows[at + kept.s], r, __float_as_uint(acc));
                        }
                        const float p = mine ? 0.f + acc : 0.f;
                        if (!WIDE) {
#pragma unroll
                            for (int k = 0; k < 6; ++k) x[k] = x[k + 2];
                            x[6] = p;
                            x[7] = mine ? fmaf(acc, m, 0.f) : 0.f;
                        }
                        ++u;
                        if (!WIDE && fin && u == quick) {
                            pend += u;
                            reduce_rows(warp);
                            pend -= u;
                        }
                        alive = step_sync(st + u - 1, p >= kRowLow);
                        if (u == quick || !alive) break;
                    }
                });
            }
            ready = fin && u == quick;
            done = u;
            pend += u;
            cur += u * RS;
            if (cur >= rowE) cur -= rowE;
            slot += u * slotB;
            if (slot >= slotE) slot -= slotE;
            if (slot >= slotE) slot %= slotE;  // fewer stages than steps in a run
        }
        st += done;
        for (int u = done; u < run && alive; ++u, ++st) {
            const int i = dir == 0 ? i0 + st : i1 - 1 - st;
            if (u > 0) {
                wt = vp * kWt;
                dth = 0.f;
            }
            const bool inner = i >= iin0 && i <= iin1;
            const int nxt = cur + RS == rowE ? 0 : cur + RS;
            ++pend;
            ready = u + 1 == run && sums;
            bool some = false;
            if (mover) {
                if (!CL && record && lane == 0) thr_[dir == 0 ? i + 1 : i] = (double)tn;
                for (int k = 0; k + 1 < nck; ++k) {
                    wait_next(st);
                    __syncthreads();
                    if (issued < total) issue_next();
                }
                wait_next(st);
                if (CL) cta_release();
            } else if (storer) {
                if (CL && record && lane == 0) thr_[dir == 0 ? i + 1 : i] = (double)tn;
                store_row();
                for (int k = 0; k + 1 < nck; ++k) __syncthreads();
            } else {
                float part = 0.f, partm = 0.f;
                int t = 0, sl = slot;
                const int vlo = inner ? 0 : max(0, xmax - n * i);
                const int vhi = inner ? M - 1 : (int)min((long long)M - 1, rho - (long long)n * i + xmax);
                for (int k = 0; k < nck; ++k) {
                    if (k > 0) {
                        __syncthreads();
                        sl = sl + slotB == slotE ? 0 : sl + slotB;
                    }
                    const int buf = sl - tab[k].off, vend = min(vB, vA + (k + 1) * CK);
                    for (LaneGroup g = list[t]; g.v < vend; g = list[++t]) {
                        Place pl;
                        if (inner) {
                            const int4 q = ptab[t * 32 + lane];
                            pl.sel = g.lg >> 8;
                            pl.coff = q.x;
                            pl.woff = q.y;
                            pl.voff = q.z & 0xffff;
                            pl.T = q.z >> 16;
                            pl.s = q.w & 0x3fffffff;
                            pl.owner = q.w >> 30;
                        } else {
                            pl = place(g, vlo, vhi);
                        }
                        float acc = 0.f;
                        chain_with_dot<MNT>(pl.sel, MNS, pl.T, lane & ((1 << (pl.sel & 3)) - 1), [&](auto dot) {
                            acc = dot(rows + (cur + pl.coff), stage0 + (buf + pl.woff), wts + (wt + pl.voff));
                        });
                        if (pl.owner) {
                            const float m = (float)(pl.s - xmax);
                            if (dir == 1 && dth != 0.f) acc *= exp2f(dth * (m - mean));
                            rows[nxt + pl.s] = acc;
                            if (CL)
                                for (int r = 0; r < ncta; ++r)
                                    if (r != rank) st_cluster(&rows[nxt + pl.s], r, __float_as_uint(acc));
                            some |= acc >= kRowLow;
                            part += acc;
                            partm = fmaf(acc, m, partm);
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < 6; ++k) x[k] = x[k + 2];
                x[6] = part;
                x[7] = partm;
                if (!WIDE && ready && has) reduce_rows(warp);
            }
            alive = step_sync(st, some);
            if (mover && issued < total) issue_next();
            for (int k = 0; k < nck; ++k) slot = slot + slotB == slotE ? 0 : slot + slotB;
            cur = nxt;
        }
    }
    const bool gave_up = read_failure<CL>(&s_fail) <= st;
    if (gave_up) failed = true;
    if (!failed && pend > 0) {  // the last rows (the last step's sums are ready)
        if (storer)
            while (qn > 0) store_row();
        if (WIDE) {
            gather_rows();
            __syncthreads();
        }
        failed = !sum_rows(nsteps);
        if (storer)
            while (qn > 0) store_row();
        if (recorder && rec_row >= 0) mcr[rec_row] = (double)rec_mean;
    }
    if (failed) {
        // Copies already issued must land before the CTA's shared memory is
        // released or used again: wait for them, again with a bound.
        bool late = gave_up;
        if (mover)
            for (int h = max(0, issued - NST); h < issued; ++h)
                late |= !mbar_wait(&bar[h % NST], (uint32_t)((h / NST) & 1), wait_limit);
        late = __syncthreads_or(late ? 1 : 0) != 0;
        if (late && tid == 0) atomicMax(f.status, ST_TIMEOUT);
        if (gave_up) return;  // the same in every CTA
        if constexpr (CL) chain_sync<true>();  // the other CTAs' parts of rows that are stored again
        if (rank == 0 && !late) crowd_again(&f, dir | (replay ? 2 : 0));
        return;
    }
    const float *last = rows + cur;
    const float inv = sc_last;
    if (segm && !replay) {
        // carry the boundary row and the controller state to the next launch
        float *edge = (dir == 0) ? f.ckpt + Mp : f.bedge;
        if (rank == 0)
            for (int s = tid; s < M; s += nthr) edge[s] = last[s] * inv;
        if (record && mover && lane == 0) {
            ChainState &cs = f.cst[dir];
            cs.theta = theta;
            cs.mean = mean;
            cs.lc_sum = lc_prev;
            cs.lrow = lrow;
            cs.lc_cnt = lc_cnt;
            cs.steps = steps0 + nsteps;
            cs.zexp = zexp;
            cs.ztilt = ztilt;
        }
    }
    if (dir != 0 || replay || i1 != N || rank != 0 || !mover) return;
    const double ln2 = 0.6931471805599453;
    const double th = (double)theta;
    if (!f.phiN) {
        const float aN = last[send] * inv;
        if (lane != 0) return;
        if (!(aN > 0.f)) atomicMax(f.status, ST_ZERO);
        else *f.loglik = log((double)aN) + ((double)zexp + ztilt - th * (double)rho) * ln2;
        return;
    }
    // log P = log Z_N - theta tau log 2 + log sum_m phiN(m) alpha^_N(m) 2^{-theta m}, the sum
    // formed in FP64 relative to its largest term
    auto lterm = [&](int s) {
        const float a = last[s] * inv, w = f.phiN[s];
        return a > 0.f && w > 0.f ? log2((double)a) + log2((double)w) - th * (double)(s - xmax) : -1e300;
    };
    double lmax = -1e300, sum = 0.0;
    for (int s = lane; s < M; s += 32) lmax = fmax(lmax, lterm(s));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    if (lmax > -1e300)
        for (int s = lane; s < M; s += 32) sum += exp2(lterm(s) - lmax);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) {
        if (!(sum > 0.0)) atomicMax(f.status, ST_ZERO);
        else *f.loglik = (lmax + log2(sum) + (double)zexp + ztilt - th * (double)((long long)n * N)) * ln2;
    }
}

template <int MNT, int MODE>
cudaError_t launch_chain_one(const FrameDev *frames, const Work *work, int nwork, size_t smem, int threads,
                             cudaStream_t st) {
    // The opt-in limit is raised to the device maximum, once per device: graphs
    // hold launches of several waves with different sizes, and every one must
    // stay valid.  A size beyond it is refused by the launch.
    static std::atomic<uint64_t> attr{0};
    cudaError_t e = smem_optin_once(k_chain<MNT, MODE>, attr);
    if (e != cudaSuccess) return e;
    k_chain<MNT, MODE><<<nwork, threads, smem, st>>>(frames, work);
    return cudaGetLastError();
}
template <int MNT>
cudaError_t launch_chain_mn(const FrameDev *frames, const Work *work, int nwork, size_t smem,
                            int cluster, int threads, cudaStream_t st) {
    if (cluster == 1)
        return threads <= kChainMostThreads
                   ? launch_chain_one<MNT, kChainNarrow>(frames, work, nwork, smem, threads, st)
                   : launch_chain_one<MNT, kChainWide>(frames, work, nwork, smem, threads, st);
    static std::atomic<uint64_t> attrC{0};
    cudaError_t e = smem_optin_once(k_chain<MNT, kChainCluster>, attrC);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nwork * cluster));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_chain<MNT, kChainCluster>, frames, work);
}

}  // namespace mdk
