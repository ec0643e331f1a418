// Batched F-score matrix: F_g({i}) for every (request, worker) pair of an instance (Eq. 1 exactly,
// Eq. 2 in fp64 term by term), and the best worker of every request.
#pragma once
#include "br_device.cuh"
#include "../../include/br.h"

namespace br {

constexpr int kFsWarps = 4;        // warps per thread block
constexpr int kFsReq = 64;         // requests per warp, two per lane
constexpr int kFsCols = 8;         // workers staged between two writes of the matrix

struct FscoreArgs {
    int32_t G, H;
    bool fp;
    double aD, beta;
    double d[BR_MAX_H + 1];
    int32_t n_req, first_instance;
    int32_t split_log2;    // log2 of the warps that share 64 requests, each with a stretch of workers (Eq. 1: of requests)
    int32_t row;           // row stride of the margins in shared memory
    const int32_t *s;      // [N][n_req]
    const int64_t *Lh;     // [N][G][H+1]
    const int32_t *cap;    // [N][G] or NULL
    double *F;             // [N][n_req][G]
    int32_t *best_g;       // [N][n_req] or NULL
};

__device__ __forceinline__ long long fscore_key(const FscoreArgs &a, int delta, const long long *m)
{
    if (!a.fp) {
        long long over = (long long)delta - m[0];
        over = over > 0 ? over : 0;
        return (long long)delta - (long long)a.G * over;
    }
    const double dl = (double)delta;
    double pen = 0.0;
    for (int h = 0; h <= a.H; ++h) {
        double over = __dsub_rn(dl, (double)m[h]);
        over = over > 0.0 ? over : 0.0;
        pen = __dadd_rn(pen, __dmul_rn(a.d[h], over));
    }
    return key_of_double(__dsub_rn(__dmul_rn(a.aD, dl), __dmul_rn(a.beta, pen)));
}

// Warps that share 64 requests: one where there are warps enough, up to four (Eq. 1: eight) where short calls would
// leave the schedulers with fewer than four each.  Eq. 2 splits the workers, Eq. 1, whose warps write whole
// runs of the matrix, the requests (16 x 100 x 64 scores: 10.9 us with one thread per element of a
// block's rows, 14.5 with 64 requests per warp, 8.3 with eight).
inline int fscore_split_log2(bool fp, int n_req, int n_instances, int G)
{
    int l = 0;
    while (l < (fp ? 2 : 3) && (!fp || (kFsCols << l) < G) &&
           ((long long)n_instances * ((n_req + kFsReq - 1) / kFsReq) << l) < 4ll * 4 * 148) ++l;
    return l;
}
// margin rows [g][h], (d_h, -2^52 d_h) pairs, one staging area per warp
inline int fscore_smem(int G, int row) { return 4 * G * row + 16 * row + kFsWarps * kFsReq * (kFsCols + 1) * 8; }

// A lane owns two requests and walks the workers: margins and discounts are read by broadcast, the best
// worker so far stays in registers, and eight scores of each request at a time go through shared memory so that
// they are written in runs.  A term of Eq. 2 is RN(d_h * over), over = max(s - m_h, 0) an integer:
// X = 2^52 + over needs no conversion, and fma(X, d_h, -2^52 d_h) rounds d_h * over once, so a term is two
// fp64 instructions and one integer one.  Eq. 2 is bound by instruction latency with five
// warps a scheduler (issue 0.59 of its peak, the fp64 pipe 0.13 busy; a warp waits for shared memory and for the instruction
// before in equal parts) and by uneven blocks (an SM is busy for 50,400 cycles on average, 57,400 at most), Eq. 1 by the writes.  200 x 1,024 x 64 scores at
// H = 8 with best workers: 224 us with five fp64 operations a term, blocks of 1,024 requests and the best
// worker found by scoring everything again; 57 with the terms above for every pair, 31 with the workers whose
// smallest margin no request of the warp exceeds left at alpha D s.
template <bool FP>
__global__ void __launch_bounds__(32 * kFsWarps) br_fscore_kernel(const FscoreArgs a)
{
    extern __shared__ __align__(16) unsigned char fs_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = a.G, H = FP ? a.H : 0, H1 = H + 1, HS = a.row;
    int *m_s = reinterpret_cast<int *>(fs_smem);                                 // [g][HS] -m_{g,h}, clipped to the range of s
    double2 *d_s = reinterpret_cast<double2 *>(fs_smem + 4 * G * HS);            // (d_h, -2^52 d_h)
    double *stage = reinterpret_cast<double *>(fs_smem + 4 * G * HS + 16 * HS) + warp * kFsReq * (kFsCols + 1);
    __shared__ int cap_s[BR_MAX_G], low_s[BR_MAX_G];                             // low_s: -min_h m_{g,h}
    const size_t inst = (size_t)a.first_instance + blockIdx.y;

    if (FP) {
        for (int g = tid; g < G; g += 32 * kFsWarps) low_s[g] = (int)0x80000000;
        __syncthreads();
    }
    // margins: one warp per four offsets, lanes over workers; the loads of the four are asked for together (one offset
    // at a time, the trips to memory of a long horizon came one after the other: 16 x 100 requests, G = 1,
    // H = 80: 8.6 us with whole rows staged at once, 12.4, 8.3 this way)
    for (int h0 = 4 * warp; h0 < H1; h0 += 4 * kFsWarps) {
        const int64_t *row = a.Lh + inst * G * (a.H + 1) + h0;
        const long long none = (long long)0x8000000000000000ull;
        long long L[2][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const int g = lane + 32 * w;
                L[w][j] = g < G && h0 + j < H1 ? row[(size_t)g * (a.H + 1) + j] : none;
            }
        long long M[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) M[j] = L[0][j] > L[1][j] ? L[0][j] : L[1][j];
        for (int o = 1; o < 32 && o < G; o <<= 1)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const long long v = __shfl_xor_sync(kFull, M[j], o);
                M[j] = v > M[j] ? v : M[j];
            }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const int g = lane + 32 * w;
                if (g >= G || h0 + j >= H1) continue;
                const int v = -(int)min(M[j] - L[w][j], 0x7FFFFFFFll);
                m_s[g * HS + h0 + j] = v;
                if (FP) atomicMax(&low_s[g], v);
            }
    }
    for (int h = tid; h < H1; h += 32 * kFsWarps) d_s[h] = make_double2(a.d[h], __dmul_rn(a.d[h], -4503599627370496.0));
    for (int g = tid; g < G; g += 32 * kFsWarps) cap_s[g] = a.cap ? a.cap[inst * G + g] : 1;
    __syncthreads();

    if (!FP) {
        // Eq. 1 is a write of the matrix: the warp's rows are one run, written 256 bytes at a time (in runs of eight
        // workers per request it reached 0.91 of the copy bandwidth at 4,096 x 1,024 x 32 scores, this way 1.0).  The best workers are
        // looked for again, two requests a lane; scoring is two integer instructions.
        int *s_w = reinterpret_cast<int *>(stage);
        const int per_warp = kFsReq >> a.split_log2;
        const int r0 = (blockIdx.x * kFsWarps + warp) * per_warp, cnt = min(per_warp, a.n_req - r0);
        if (cnt <= 0) return;
        const int32_t *s = a.s + inst * a.n_req + r0;
        for (int r = lane; r < cnt; r += 32) s_w[r] = __ldg(s + r);
        __syncwarp();
        auto score = [&](int si, int g) {                            // integers below 2^53, exact
            return (double)((long long)si - (long long)G * (long long)__viaddmax_s32(max(si, 0), m_s[g * HS], 0));
        };
        double *F = a.F + (inst * a.n_req + r0) * G;
        int r = lane / G, g = lane - r * G;
        const int step_r = 32 / G, step_g = 32 - step_r * G;
#pragma unroll 4
        for (int o = lane; o < cnt * G; o += 32) {
            F[o] = score(s_w[r], g);
            r += step_r; g += step_g;
            if (g >= G) { g -= G; ++r; }
        }
        if (a.best_g) {
            int32_t *best = a.best_g + inst * a.n_req + r0;
            for (int q = lane; q < cnt; q += 32) {
                double top = 0.0;
                int b = -1;
#pragma unroll 4
                for (int x = 0; x < G; ++x) {
                    const double f = score(s_w[q], x);
                    if (cap_s[x] > 0 && (b < 0 || f > top)) { top = f; b = x; }      // x ascends: the lower worker on ties
                }
                best[q] = b;
            }
        }
        return;
    }

    const int split = 1 << a.split_log2, sub = warp & (split - 1);
    const int r0 = (blockIdx.x * (kFsWarps >> a.split_log2) + (warp >> a.split_log2)) * kFsReq;
    const int cnt = min(kFsReq, a.n_req - r0);                        // not positive: nothing to do but the barrier
    const int span = ((G + kFsCols * split - 1) / (kFsCols * split)) * kFsCols;
    const int g_end = min(G, (sub + 1) * span);
    const int32_t *s = a.s + inst * a.n_req + r0;
    const int s0 = lane < cnt ? __ldg(s + lane) : 1, s1 = lane + 32 < cnt ? __ldg(s + lane + 32) : 1;
    const int o0 = max(s0, 0), o1 = max(s1, 0);                       // (lengths are positive; margins are never negative)
    const double aDs0 = __dmul_rn(a.aD, (double)s0), aDs1 = __dmul_rn(a.aD, (double)s1);
    // a worker whose smallest margin is not below the warp's longest request scores alpha D s: no term is positive
    const int longest = __reduce_max_sync(kFull, max(o0, o1));
    long long k0 = kNoKey, k1 = kNoKey;
    int b0 = kNoIdx, b1 = kNoIdx;
    double q0 = 0.0, q1 = 0.0;
#pragma unroll 1
    for (int gc = sub * span; gc < g_end && cnt > 0; gc += kFsCols) {
        const int cols = min(kFsCols, g_end - gc);
#pragma unroll 1
        for (int x = 0; x < cols; ++x) {
            const int g = gc + x;
            const int *mg = m_s + g * HS;
            double f0, f1;
            {
                double p0 = 0.0, p1 = 0.0;
                int h = longest + low_s[g] > 0 ? 0 : H1;
#pragma unroll 2
                for (; h + 4 <= H1; h += 4) {
                    const int4 m4 = *reinterpret_cast<const int4 *>(mg + h);
                    const int mj[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const double2 d = d_s[h + j];
                        p0 = __dadd_rn(p0, __fma_rn(__hiloint2double(0x43300000, __viaddmax_s32(o0, mj[j], 0)), d.x, d.y));
                        p1 = __dadd_rn(p1, __fma_rn(__hiloint2double(0x43300000, __viaddmax_s32(o1, mj[j], 0)), d.x, d.y));
                    }
                }
#pragma unroll 1
                for (; h < H1; ++h) {
                    const int m = mg[h];
                    const double2 d = d_s[h];
                    p0 = __dadd_rn(p0, __fma_rn(__hiloint2double(0x43300000, __viaddmax_s32(o0, m, 0)), d.x, d.y));
                    p1 = __dadd_rn(p1, __fma_rn(__hiloint2double(0x43300000, __viaddmax_s32(o1, m, 0)), d.x, d.y));
                }
                f0 = __dsub_rn(aDs0, __dmul_rn(a.beta, p0)) + 0.0;                // Eq. 2 (-0.0 -> +0.0)
                f1 = __dsub_rn(aDs1, __dmul_rn(a.beta, p1)) + 0.0;
            }
            stage[lane * (kFsCols + 1) + x] = f0;
            stage[(lane + 32) * (kFsCols + 1) + x] = f1;
            if (a.best_g && cap_s[g] > 0) {                                       // g ascends: the lower worker is kept on ties
                if (f0 > q0 || b0 == kNoIdx) { q0 = f0; b0 = g; }
                if (f1 > q1 || b1 == kNoIdx) { q1 = f1; b1 = g; }
            }
        }
        __syncwarp();
        const int x = lane & (kFsCols - 1);
        double *F = a.F + (inst * a.n_req + r0 + (lane >> 3)) * G + gc + x;
        const double *from = stage + (lane >> 3) * (kFsCols + 1) + x;
        if (x < cols) {
#pragma unroll 4
            for (int r = lane >> 3; r < cnt; r += 4) {
                *F = *from;
                F += 4 * G; from += 4 * (kFsCols + 1);
            }
        }
        __syncwarp();
    }
    if (a.best_g) {
        if (b0 != kNoIdx) k0 = key_of_double(q0);
        if (b1 != kNoIdx) k1 = key_of_double(q1);
        if (split > 1) {
            long long *ks = reinterpret_cast<long long *>(stage);
            int *is = reinterpret_cast<int *>(stage + kFsReq);
            ks[lane] = k0; ks[lane + 32] = k1; is[lane] = b0; is[lane + 32] = b1;
            __syncthreads();
            if (sub != 0) return;
            for (int w = 1; w < split; ++w) {
                const long long *kw = ks + w * kFsReq * (kFsCols + 1);
                const int *iw = is + 2 * w * kFsReq * (kFsCols + 1);
                if (kw[lane] > k0) { k0 = kw[lane]; b0 = iw[lane]; }
                if (kw[lane + 32] > k1) { k1 = kw[lane + 32]; b1 = iw[lane + 32]; }
            }
        }
        int32_t *best = a.best_g + inst * a.n_req + r0;
        if (lane < cnt) best[lane] = b0 == kNoIdx ? -1 : b0;
        if (lane + 32 < cnt) best[lane + 32] = b1 == kNoIdx ? -1 : b1;
    }
}

}  // namespace br
