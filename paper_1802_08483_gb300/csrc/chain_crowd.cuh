// The recursion with every row summed and scaled at its own step: k_chain_crowd
// (chain.cu), and what k_chain falls back on.
#pragma once

#include "mapdec_dev.cuh"
#include "mapdec_kernels.h"

namespace mdk {

constexpr int kMaxStages = 8;

// Tilt controller (see k_chain).
constexpr float kTiltGainMin = 0.02f;  // long-run smoothing of the entropy-rate estimate
constexpr float kTiltStepMax = 0.02f;  // largest change of the tilt between two rows
constexpr float kTiltMin = 0.2f, kTiltMax = 1.6f;
constexpr int kTiltEvery = 4;    // steps between tilt updates once settled
constexpr int kTiltSettle = 64;  // updates every step for the first steps

// ---------------------------------------------------------------------------
// The recursions of launches with more of them than SMs (k_chain_crowd).  The same
// recursion as k_chain, and with the default block size and chunks the same sums in
// the same order, one CTA per (frame, direction), with a few registers and as little shared memory as two staged
// chunks take, so that several share an SM with each other and with the producers
// of other waves; k_chain's lower latency needs an SM to itself (256 frames N = 64,
// q = 8: 470 us a decode with this kernel, 520 to 590 with k_chain at two and
// three CTAs per SM; 512 mixed frames in waves of 64: 167 ms against 209 to 255).
// Every row is scaled when it is built; k_chain comes back to it (crowd_again) for
// rows that leave FP32's range between two sums.
constexpr int kCrowdThreads = 256;  // default block size
constexpr int kCrowdMaxThreads = 512;

// Two FP32 sums at once (row sum and first moment); every thread gets the
// same result (the warps' partials are added in one fixed order).
__device__ __forceinline__ void block_sum2(float a, float b, float &sa, float &sb, float *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) { red[warp] = a; red[32 + warp] = b; }
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    float x = 0.f, y = 0.f;
    for (int w = 0; w < nw; ++w) { x += red[w]; y += red[32 + w]; }
    sa = x;
    sb = y;
}

// Geometry of chunk k of a step: the same for every symbol, relative to the
// symbol's block of W (blocks are 16-byte aligned, so the aligned copy start,
// the shift to row r0 and the copy size do not depend on the symbol).
constexpr int kMaxChunks = 64;
struct CrowdTab {
    int d0[kMaxChunks], d1[kMaxChunks];  // owned states (alpha: destinations, beta: sources)
    int r0[kMaxChunks], r1[kMaxChunks];  // W rows staged
    int shift[kMaxChunks];               // floats between the aligned copy start and row r0
    int off[kMaxChunks];                 // aligned copy start within the symbol's block (floats)
    uint32_t bytes[kMaxChunks];          // copy size
};

__device__ __forceinline__ void crowd_geom(const FrameDev &f, int dir, int k, CrowdTab &t) {
    const int CD = f.crowdCD, M = f.M;
    const int d0 = k * CD, d1 = min(M, d0 + CD);
    int r0, r1;
    if (dir == 0) {  // destination s gets sources s - nI .. s + n
        r0 = max(0, d0 - f.n * f.I);
        r1 = min(M, d1 + f.n);
    } else {
        r0 = d0;
        r1 = d1;
    }
    const int o0 = r0 * f.MNS, o1 = r1 * f.MNS;
    const int a0 = o0 & ~3, a1 = (o1 + 3) & ~3;
    t.d0[k] = d0;
    t.d1[k] = d1;
    t.r0[k] = r0;
    t.r1[k] = r1;
    t.shift[k] = o0 - a0;
    t.off[k] = a0;
    t.bytes[k] = a1 > a0 ? (uint32_t)(a1 - a0) * 4u : 16u;
}

__device__ __forceinline__ void crowd_recursion(const FrameDev &f, int tile) {
    const int dir = tile & 1;  // 0 = forward (alpha), 1 = backward (beta); bit 1: replay
    const int M = f.M, Mp = f.Mp, MNS = f.MNS, MN = f.MN, n = f.n, N = f.N, xmax = f.xmax;
    const long long rho = f.rho;
    const int CD = f.crowdCD;
    const int nck = (M + CD - 1) / CD;
    const int NST = f.crowdStages;
    const int i0 = f.seg_i0, i1 = f.seg_i1;  // symbols of this launch (segment)
    const int send = (int)(rho - (long long)n * N) + xmax;  // state of the end drift
    const bool segm = (f.chain_flags & CH_SEGMENTED) != 0;
    const bool replay = dir == 0 && (tile & 2) != 0;
    // first launch of this direction: the frame boundary; otherwise the row carried over
    const bool fresh = dir == 0 ? (i0 == 0) : (i1 == N);

    __shared__ uint64_t bar[kMaxStages];
    __shared__ float red[64];
    __shared__ int s_fail;
    __shared__ float s_th[3];  // tilt of the current row, of the row being built, row mean
    __shared__ float vfac[kMaxMN];
    extern __shared__ float4 sm4[];
    float *cur = reinterpret_cast<float *>(sm4);
    float *nxt = cur + Mp;
    float *stage0 = nxt + Mp;
    const size_t stageFloats = ((size_t)(CD + MN + 1) * MNS + 8 + 3) & ~(size_t)3;

    for (int s = threadIdx.x; s < Mp; s += blockDim.x) {
        float v;
        if (fresh) v = (s == (dir == 0 ? xmax : send)) ? 1.f : 0.f;
        else v = (dir == 0) ? f.ckpt[s] : f.bedge[s];
        cur[s] = v;
        nxt[s] = 0.f;
    }
    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int st = 0; st < NST; ++st) mbar_init(&bar[st], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // Stream decoding: a boundary drift prior replaces the point mass
    // (alpha_0 = phi0, beta_N = phiN; Sec. II-C).  In the tilted rows the start
    // row is alpha^_0(m) = phi0(m) 2^m / Z_0 (tilt 1, received length m) and the
    // end row beta^_N(m) is proportional to phiN(m) 2^-m; both are first scaled
    // by 2^-emax (emax the largest exponent over the prior's support, exact),
    // then divided by the power of two below their sum like every row, and
    // log2 Z_0 = emax + that exponent starts the forward record.
    const float *prior = !fresh ? nullptr : (dir == 0 ? f.phi0 : f.phiN);
    __shared__ int s_emax;
    long long zexp0 = 0;  // log2 Z_0 of a prior start row (forward)
    float mean0 = (dir == 0) ? 0.f : (float)(send - xmax);
    if (prior) {
        if (threadIdx.x == 0) s_emax = -(1 << 30);
        __syncthreads();
        for (int s = threadIdx.x; s < M; s += blockDim.x)
            if (prior[s] > 0.f) atomicMax(&s_emax, dir == 0 ? s - xmax : xmax - s);
        __syncthreads();
        const int emax = s_emax;
        float part0 = 0.f, partm0 = 0.f;
        for (int s = threadIdx.x; s < M; s += blockDim.x) {
            const float w = prior[s];
            const int e = (dir == 0 ? s - xmax : xmax - s) - emax;  // <= 0
            const float v = (w > 0.f && e > -150) ? ldexpf(w, e) : 0.f;
            cur[s] = v;
            part0 += v;
            partm0 = fmaf(v, (float)(s - xmax), partm0);
        }
        float c0, cm0;
        block_sum2(part0, partm0, c0, cm0, red);
        if (!(c0 > 0.f)) {  // no mass inside the drift limits (same in every thread)
            if (threadIdx.x == 0) atomicMax(f.status, ST_ZERO);
            return;         // nothing issued yet
        }
        int ex;
        frexpf(c0, &ex);
        const float inv = ldexpf(1.f, 1 - ex);
        for (int s = threadIdx.x; s < M; s += blockDim.x) cur[s] *= inv;
        zexp0 = (long long)emax + ex - 1;
        mean0 = cm0 / c0;
        __syncthreads();
    }
    {
        float *row0 = (dir == 0) ? f.alpha + (size_t)i0 * Mp : f.beta + (size_t)i1 * Mp;
        for (int s = threadIdx.x; s < Mp; s += blockDim.x) row0[s] = cur[s];
    }
    auto symbol_of = [&](int st) { return dir == 0 ? i0 + st : i1 - 1 - st; };
    // Chunk table, and a self-check of every copy it implies: source inside
    // this launch's symbols of W (plus the 16-float tail slack), destination
    // inside its stage, 16-byte alignment and size.  A violation records
    // ST_ARG and the chain does not start.
    __shared__ CrowdTab tab;
    for (int k = threadIdx.x; k < nck && k < kMaxChunks; k += blockDim.x) {
        crowd_geom(f, dir, k, tab);
        const bool ok = tab.off[k] + (long long)tab.bytes[k] / 4 <= f.wblk + 16 &&
                        tab.bytes[k] % 16 == 0 && tab.bytes[k] / 4 <= stageFloats;
        if (!ok) atomicExch(&s_fail, ST_ARG);
    }
    if (threadIdx.x == 0 && (nck > kMaxChunks || ((uintptr_t)f.W & 15) != 0 || (f.wblk & 3) != 0 ||
                             ((uintptr_t)stage0 & 15) != 0 || (stageFloats & 3) != 0))
        atomicExch(&s_fail, ST_ARG);
    __syncthreads();
    if (s_fail) {  // same in every thread (read after the barrier); nothing issued yet
        if (threadIdx.x == 0) atomicMax(f.status, s_fail);
        return;
    }
    const long long total = (long long)(i1 - i0) * nck;
    // thread 0's issue cursor: chunks issued so far, and the next one's place
    long long issued = 0;
    int is_st = 0, is_k = 0, is_slot = 0;
    auto issue_next = [&]() {
        const float *src = f.W + (size_t)symbol_of(is_st) * f.wblk + tab.off[is_k];
        uint64_t *b = &bar[is_slot];
        if (!((f.test_flags & TEST_SKIP_COPY) && issued == 0)) {
            mbar_expect_tx(b, tab.bytes[is_k]);
            bulk_g2s(stage0 + (size_t)is_slot * stageFloats, src, tab.bytes[is_k], b);
        }
        ++issued;
        if (++is_k == nck) { is_k = 0; ++is_st; }
        if (++is_slot == NST) is_slot = 0;
    };
    if (threadIdx.x == 0)
        while (issued < NST && issued < total) issue_next();

    // controller state (thread 0); log2 Z as an integer sum of the row
    // scalings plus the FP64 sum of the tilt terms (changed rows only)
    long long zexp = zexp0;
    double ztilt = 0.0;
    float theta = 1.f;   // tilt of the current row
    float mean = mean0;  // its mean drift
    float lrow = 0.f;      // log2 of the current row's sum
    float lc_prev = 0.f;   // sum of log2 growth since the last tilt update
    int lc_cnt = 0;        // number of steps in lc_prev
    int steps = 0;         // every thread: steps taken in this direction so far
    if (!fresh && segm) {
        const ChainState &cs = f.cst[dir];
        steps = cs.steps;
        if (threadIdx.x == 0) {
            theta = cs.theta;
            mean = cs.mean;
            zexp = cs.zexp;
            ztilt = cs.ztilt;
            lc_prev = cs.lc_sum;
            lrow = cs.lrow;
            lc_cnt = cs.lc_cnt;
        }
    }
    if (replay) steps = i0;
    if (threadIdx.x == 0 && fresh && !replay) {
        if (dir == 0) { f.thf[0] = 1.0; f.mcf[0] = (double)mean0; }
        else f.thb[N] = 1.0;
    }
    // this thread's share of the row sum and of its first moment
    float part = 0.f, partm = 0.f;
    float th_cur = 1.f, th_new = 1.f, mc = 0.f;
    if (!fresh && segm && !replay) {
        // continuing a recursion: the first step here need not be an update
        // step, so restore the row's tilt and its transition weights as the
        // previous launch left them
        if (threadIdx.x == 0) {
            s_th[0] = theta;
            s_th[2] = mean;
        }
        __syncthreads();
        th_cur = th_new = s_th[0];
        mc = s_th[2];
        for (int j = threadIdx.x; j < MN; j += blockDim.x) vfac[j] = exp2f((th_cur - 1.f) * (float)j);
        __syncthreads();
    }
    bool failed = false;
    long long gfail = 0;
    int st = 0, k = 0, slot = 0;
    uint32_t ph = 0;
    for (long long g = 0; g < total; ++g) {
        const int i = symbol_of(st);
        const bool update = replay || steps < kTiltSettle || (steps & (kTiltEvery - 1)) == 0;
        if (k == 0 && update) {
            // start of an update step: choose the tilt of the rows from here on
            // (the recompute sweep replays the tilts recorded by the first sweep)
            if (threadIdx.x == 0 && replay) {
                s_th[0] = (float)f.thf[i];
                s_th[1] = (float)f.thf[i + 1];
                s_th[2] = (float)f.mcf[i];
            } else if (threadIdx.x == 0) {
                float tn = theta;
                if (steps > 0 && lc_cnt > 0) {
                    const float gain =
                        fminf(1.f, fmaxf(kTiltGainMin, (float)lc_cnt / (float)(steps + 1)));
                    const float d = fminf(kTiltStepMax,
                                          fmaxf(-kTiltStepMax, -gain * (lc_prev / (float)lc_cnt) / (float)n));
                    tn = fminf(kTiltMax, fmaxf(kTiltMin, theta + d));
                }
                s_th[0] = theta;
                s_th[1] = tn;
                s_th[2] = mean;
                lc_prev = 0.f;
                lc_cnt = 0;
            }
            __syncthreads();
            th_cur = s_th[0];
            th_new = s_th[1];
            mc = s_th[2];
            // forward: transition weight 2^{(theta_{i+1}-1) j}; backward: 2^{(theta'_{i+1}-1) j}
            const float phi = (dir == 0 ? th_new : th_cur) - 1.f;
            for (int j = threadIdx.x; j < MN; j += blockDim.x) vfac[j] = exp2f(phi * (float)j);
            if (dir == 0) {
                const float dth = th_new - th_cur;
                if (dth != 0.f)
                    for (int s = threadIdx.x; s < M; s += blockDim.x)
                        cur[s] *= exp2f(dth * ((float)(s - xmax) - mc));
            }
            __syncthreads();
        } else if (k == 0) {
            // no update: the row keeps its tilt (backward: the transition weight of
            // a step uses the source row's tilt, which is now th_new)
            if (dir == 1 && th_cur != th_new) {
                th_cur = th_new;
                const float phi = th_cur - 1.f;
                for (int j = threadIdx.x; j < MN; j += blockDim.x) vfac[j] = exp2f(phi * (float)j);
                __syncthreads();
            }
            th_cur = th_new;
        }
        const int cd0 = tab.d0[k], cd1 = tab.d1[k], cr0 = tab.r0[k], cr1 = tab.r1[k];
        const float *buf = stage0 + (size_t)slot * stageFloats + tab.shift[k];
        if (!mbar_wait(&bar[slot], ph, f.wait_limit)) atomicExch(&s_fail, ST_TIMEOUT);
        // valid source rows: window start p = n i + s - xmax inside [0, rho]
        const int vlo = max(0, xmax - n * i);
        const long long vhi_l = rho - (long long)n * i + xmax;
        const int vhi = (int)min((long long)M - 1, vhi_l);
        // JS lanes share one state, each summing every JS-th term with four
        // accumulators; the lanes combine by shuffles in a fixed order.
        const int nst = cd1 - cd0;
        int JS = 1;
        while (JS < 8 && nst * JS * 2 <= (int)blockDim.x) JS *= 2;
        const int lgJS = JS == 1 ? 0 : (JS == 2 ? 1 : (JS == 4 ? 2 : 3));
        const int lo = max(cr0, vlo), hi = min(cr1 - 1, vhi);
        for (int w0 = 0; w0 < nst * JS; w0 += blockDim.x) {
            const int w = w0 + (int)threadIdx.x;
            const int s = cd0 + (w >> lgJS), js = w & (JS - 1);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
            if (w < nst * JS) {
                if (dir == 0) {
                    // alpha'(s) = sum_j alpha(s - j + n) W[s - j + n][j] vfac[j]
                    const int jlo = max(0, s + n - hi), jhi = min(MN - 1, s + n - lo);
                    const float *cp = cur + (s + n);
                    const float *bp = buf + (size_t)(s + n - cr0) * MNS;
                    const int dm = MNS - 1;
                    int j = jlo + js;
                    for (; j + 3 * JS <= jhi; j += 4 * JS) {
                        const int j1 = j + JS, j2 = j + 2 * JS, j3 = j + 3 * JS;
                        a0 = fmaf(cp[-j], bp[-j * dm] * vfac[j], a0);
                        a1 = fmaf(cp[-j1], bp[-j1 * dm] * vfac[j1], a1);
                        a2 = fmaf(cp[-j2], bp[-j2 * dm] * vfac[j2], a2);
                        a3 = fmaf(cp[-j3], bp[-j3 * dm] * vfac[j3], a3);
                    }
                    for (; j <= jhi; j += JS) a0 = fmaf(cp[-j], bp[-j * dm] * vfac[j], a0);
                } else if (s >= vlo && s <= vhi) {
                    // beta'(s) = sum_j W[s][j] vfac[j] beta(s + j - n)
                    const int jlo = max(0, n - s), jhi = min(MN - 1, M - 1 - s + n);
                    const float *wr = buf + (size_t)(s - cr0) * MNS;
                    const float *cq = cur + (s - n);
                    int j = jlo + js;
                    for (; j + 3 * JS <= jhi; j += 4 * JS) {
                        const int j1 = j + JS, j2 = j + 2 * JS, j3 = j + 3 * JS;
                        a0 = fmaf(wr[j] * vfac[j], cq[j], a0);
                        a1 = fmaf(wr[j1] * vfac[j1], cq[j1], a1);
                        a2 = fmaf(wr[j2] * vfac[j2], cq[j2], a2);
                        a3 = fmaf(wr[j3] * vfac[j3], cq[j3], a3);
                    }
                    for (; j <= jhi; j += JS) a0 = fmaf(wr[j] * vfac[j], cq[j], a0);
                }
            }
            float acc = (a0 + a1) + (a2 + a3);
            for (int o = 1; o < JS; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (w < nst * JS && js == 0) {
                if (dir == 1) {
                    // post-scale 2^{(theta'_{i+1} - theta'_i)(m - mean)}
                    const float dth = th_cur - th_new;
                    if (dth != 0.f) acc *= exp2f(dth * ((float)(s - xmax) - mc));
                }
                nxt[s] = acc;
                part += acc;
                partm = fmaf(acc, (float)(s - xmax), partm);
            }
        }
        __syncthreads();  // stage consumed by everyone
        if (s_fail) {     // a wait gave up (written before the barrier: same in every thread)
            failed = true;
            gfail = g;    // chunks g .. issued-1 may still be in flight
            break;
        }
        if (threadIdx.x == 0 && issued < total) issue_next();
        if (k == nck - 1) {
            // end of a step: scale by a power of two, keep the exact record
            float c, cm;
            block_sum2(part, partm, c, cm, red);
            part = 0.f;
            partm = 0.f;
            const bool bad = !(c >= 1.2e-38f) || !(c <= 3.0e38f);  // same in every thread
            if (bad) {
                if (threadIdx.x == 0) s_fail = ST_ZERO;
                failed = true;
                gfail = g + 1;
                break;
            }
            int ex;
            frexpf(c, &ex);  // c = m 2^ex, m in [0.5, 1)
            const float inv = ldexpf(1.f, 1 - ex);
            if (threadIdx.x == 0) {
                const float lc = log2f(c);
                if (dir == 0 && !replay) {
                    zexp += ex - 1;
                    if (th_new != th_cur)
                        ztilt += (double)(th_new - th_cur) * ((double)n * i + (double)mc);
                    f.thf[i + 1] = (double)th_new;
                    f.mcf[i + 1] = (double)(cm / c);
                } else if (dir == 1) {
                    f.thb[i] = (double)th_new;
                }
                theta = th_new;
                mean = cm / c;
                lc_prev += lc - lrow;
                lrow = lc - (float)(ex - 1);
                ++lc_cnt;
            }
            ++steps;
            float *row = (dir == 0) ? f.alpha + (size_t)(i + 1) * Mp : f.beta + (size_t)i * Mp;
            for (int s = threadIdx.x; s < M; s += blockDim.x) {
                const float v = nxt[s] * inv;
                cur[s] = v;
                row[s] = v;
            }
            __syncthreads();
        }
        if (++k == nck) { k = 0; ++st; }
        if (++slot == NST) { slot = 0; ph ^= 1u; }
    }
    if (failed) {
        // Copies already issued (chunks gfail .. issued-1) must land before the
        // CTA's shared memory is released: wait for them, again with a bound.
        __syncthreads();
        if (threadIdx.x == 0) {
            for (long long h = gfail; h < issued; ++h)
                mbar_wait(&bar[h % NST], (uint32_t)((h / NST) & 1), f.wait_limit);
            atomicMax(f.status, s_fail);
        }
        __syncthreads();
        return;
    }
    if (segm && !replay) {
        // carry the boundary row and the controller state to the next launch
        float *edge = (dir == 0) ? f.ckpt + Mp : f.bedge;
        for (int s = threadIdx.x; s < Mp; s += blockDim.x) edge[s] = cur[s];
        if (threadIdx.x == 0) {
            ChainState &cs = f.cst[dir];
            cs.theta = theta;
            cs.mean = mean;
            cs.zexp = zexp;
            cs.ztilt = ztilt;
            cs.lc_sum = lc_prev;
            cs.lrow = lrow;
            cs.lc_cnt = lc_cnt;
            cs.steps = steps;
        }
    }
    if (dir == 0 && !replay && i1 == N && threadIdx.x == 0) {
        if (f.phiN) {
            // log P = log Z_N - theta tau log 2 + log sum_m phiN(m) alpha^_N(m) 2^{-theta m},
            // the sum formed in FP64 relative to its largest term
            const double th = (double)theta;
            double lmax = -1e300;
            for (int s = 0; s < M; ++s)
                if (f.phiN[s] > 0.f && cur[s] > 0.f)
                    lmax = fmax(lmax, log2((double)cur[s]) + log2((double)f.phiN[s]) -
                                          th * (double)(s - xmax));
            double sum = 0.0;
            if (lmax > -1e300)
                for (int s = 0; s < M; ++s)
                    if (f.phiN[s] > 0.f && cur[s] > 0.f)
                        sum += exp2(log2((double)cur[s]) + log2((double)f.phiN[s]) -
                                    th * (double)(s - xmax) - lmax);
            if (!(sum > 0.0)) {
                atomicMax(f.status, ST_ZERO);
            } else {
                *f.loglik = (lmax + log2(sum) + (double)zexp + ztilt -
                             th * (double)((long long)n * N)) * 0.6931471805599453;
            }
        } else {
            const float aN = cur[send];
            if (!(aN > 0.f)) {
                atomicMax(f.status, ST_ZERO);
            } else {
                *f.loglik = log((double)aN) +
                            ((double)zexp + ztilt - (double)theta * (double)rho) * 0.6931471805599453;
            }
        }
    }
}

// The launch's symbols once more, by one CTA of k_chain, whose copies have landed and
// whose shared memory holds nothing that is still needed: not inlined, so that k_chain
// keeps its registers.
static __device__ __noinline__ void crowd_again(const FrameDev *f, int tile) {
    uint32_t have;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(have));
    const size_t stage = ((size_t)(f->crowdCD + f->MN + 1) * f->MNS + 8 + 3) & ~(size_t)3;
    if (have < 4 * (2 * (size_t)f->Mp + (size_t)f->crowdStages * stage)) {  // (launches are sized for it)
        if (threadIdx.x == 0) atomicMax(f->status, ST_ZERO);
        return;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // bulk copies follow plain accesses
    __syncthreads();
    crowd_recursion(*f, tile);
}

}  // namespace mdk
