// Pool-bypass dispatch for BR-0 (Appendix "Pool-bypass deployment path for BR-0"): requests are
// routed one at a time, in arrival order, each to argmax_g F_g(s) = alpha s - beta (s - m_g)_+ over
// the workers whose inflight count is below its cap, with m_g = M - L_g taken from *virtual*
// loads (running requests plus those dispatched and not started yet); the chosen worker's virtual load
// and inflight count grow at once, so the next request sees them.  One warp per instance, lane g
// holds worker g (and g + 32): the chain over requests is sequential, the arg-max over workers a
// warp reduction with lowest-g tie-break.
#pragma once
#include "br_device.cuh"
#include "br_fscore.cuh"
#include "../../include/br.h"

namespace br {

struct BypassArgs {
    FscoreArgs f;             // G, H = 0, fp, aD, beta, d[0]
    int32_t n_req, first_instance;
    const int32_t *s;         // [N][n_req] prompt lengths in arrival order
    int64_t *vload;           // [N][G] virtual loads, updated
    int32_t *inflight;        // [N][G] requests running or dispatched per worker, updated
    const int32_t *cap;       // [N][G] inflight cap per worker
    int32_t *g_out;           // [N][n_req] chosen worker, -1 if every worker is at its cap
};

// The chain from one request to the next is what bounds this path (a pool has far fewer instances than
// the GPU has warps), so it carries margins m_g = M - L_g instead of loads and is as short as the
// definition allows.  Eq. 1 falls strictly beyond the margin (G >= 2; one worker needs no order), so
// argmax_g F_g(s) is the first worker with the largest min(m_g, s): one warp maximum over
// (min(m_g, s), 63 - g) gives the worker, and its upper part the growth of the envelope,
// s - min(m_g, s).  Eq. 2 scores, whose rounding may tie, lengths outside [0, 2^25), which do not fit that
// key, and margins of 2^30 and more are handled in full.  Prompt lengths are read and answers written 32 at
// a time, and the next length is fetched while the warp maximum is on its way.
// 256 instances x 200 requests at G = 32: 74 us with the envelope and a 64-bit score reduced over the warp
// for every request, 19 us with 64-bit margins, 12 this way.
// The launch overlaps the kernel ahead (launch_overlapped): a pass of two copies and the dispatch, 256 x 200, G = 32: 17.5 us,
// 16.5; 4,096 x 33, G = 64: 18.5, 17.0; 20,000 x 32: 33.1, 31.1.  Closing workers by a count kept off the chain gained
// 0.4 us more on the first and lost 1.7 on the second.
// FP: Eq. 2 scores; GW: workers per lane.
template <bool FP, int GW>
__global__ void __launch_bounds__(32) br_bypass_kernel(const BypassArgs a)
{
    stream_order_gate();
    const int lane = threadIdx.x;
    const size_t inst = (size_t)a.first_instance + blockIdx.x;
    const int G = a.f.G;
    long long L[GW], m[GW], M = (long long)0x8000000000000000ull;
    int nfl[GW], cap[GW];
#pragma unroll
    for (int w = 0; w < GW; ++w) {
        const int g = lane + 32 * w;
        L[w] = 0; nfl[w] = 0; cap[w] = 0;
        if (g < G) {
            L[w] = a.vload[inst * G + g];
            nfl[w] = a.inflight[inst * G + g];
            cap[w] = a.cap[inst * G + g];
            M = L[w] > M ? L[w] : M;
        }
    }
    // envelope M = max_g L_g over all workers (Section 3.1)
    for (int o = 16; o > 0; o >>= 1) {
        const long long v = __shfl_xor_sync(kFull, M, o);
        M = v > M ? v : M;
    }
#pragma unroll
    for (int w = 0; w < GW; ++w) m[w] = M - L[w];
    const int32_t *s = a.s + inst * a.n_req;
    int32_t *out = a.g_out + inst * a.n_req;
    // (plain loads: with an overlapping launch the kernel ahead may write the lengths while this one is resident, which
    // read-only loads do not allow)
    int next = lane < a.n_req ? s[lane] : 0;
#pragma unroll 1
    for (int i0 = 0; i0 < a.n_req; i0 += 32) {
        const int mine = next, cnt = min(32, a.n_req - i0);
        if (i0 + 32 + lane < a.n_req) next = s[i0 + 32 + lane];
        int answer = -1;
        bool packed = !FP && (unsigned)mine < (1u << 25);
#pragma unroll
        for (int w = 0; w < GW; ++w) packed = packed && (m[w] < (1ll << 30) || lane + 32 * w >= G);
        if (__all_sync(kFull, packed)) {
            // margins stay below 2^31 for 32 requests
            int mi[GW], added[GW];
#pragma unroll
            for (int w = 0; w < GW; ++w) { mi[w] = (int)m[w]; added[w] = 0; }
            int si = __shfl_sync(kFull, mine, 0);
#pragma unroll 2
            for (int i = 0; i < cnt; ++i) {
                const int after = __shfl_sync(kFull, mine, (i + 1) & 31);
                unsigned kw[GW], key = 0u;                                // 0: every worker at its cap
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    kw[w] = nfl[w] < cap[w] ? ((unsigned)min(mi[w], si) << 6) + (unsigned)(64 - lane - 32 * w) : 0u;
                    key = max(key, kw[w]);
                }
                key = __reduce_max_sync(kFull, key);
                if (key == 0u) break;                                    // ... and none opens again
                const int grow = si - (int)((key - 1u) >> 6);
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    const bool it_is = kw[w] == key;                     // (the worker is part of the key)
                    mi[w] += it_is ? grow - si : grow;
                    added[w] += it_is ? si : 0;
                    nfl[w] += it_is ? 1 : 0;
                }
                if (lane == i) answer = 63 - (int)((key - 1u) & 63u);
                si = after;
            }
#pragma unroll
            for (int w = 0; w < GW; ++w) { m[w] = mi[w]; L[w] += added[w]; }
        } else {
#pragma unroll 1
            for (int i = 0; i < cnt; ++i) {
                const int si = __shfl_sync(kFull, mine, i);
                Best b; b.key = kNoKey; b.idx = kNoIdx;
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    const int g = lane + 32 * w;
                    if (nfl[w] < cap[w]) {
                        // (the address of an array of two would put it in local memory: 4,096 x 33 requests at
                        // G = 64: 52.0 us, 46.3 this way)
                        const long long mw = m[w];
                        const long long key = fscore_key(a.f, si, GW > 1 ? &mw : &m[w]);
                        if (key > b.key) { b.key = key; b.idx = g; }       // w ascends: the lower g is kept on ties
                    }
                }
                b = warp_argmax(b);
                if (b.key == kNoKey) break;
                long long low = 0x7FFFFFFFFFFFFFFFll;                      // the largest load has margin zero
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    const bool it_is = b.idx == lane + 32 * w;
                    m[w] -= it_is ? si : 0;
                    L[w] += it_is ? si : 0;
                    nfl[w] += it_is ? 1 : 0;
                    if (lane + 32 * w < G && m[w] < low) low = m[w];
                }
                for (int o = 16; o > 0; o >>= 1) {
                    const long long v = __shfl_xor_sync(kFull, low, o);
                    low = v < low ? v : low;
                }
#pragma unroll
                for (int w = 0; w < GW; ++w) m[w] -= low;
                if (lane == i) answer = b.idx;
            }
        }
        if (i0 + lane < a.n_req) out[i0 + lane] = answer;
    }
#pragma unroll
    for (int w = 0; w < GW; ++w) {
        const int g = lane + 32 * w;
        if (g < G) { a.vload[inst * G + g] = L[w]; a.inflight[inst * G + g] = nfl[w]; }
    }
}

}  // namespace br
