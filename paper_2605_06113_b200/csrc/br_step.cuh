// The general routing-step kernel: one thread block of 32 to 256 threads per instance (BR-H, large
// fleets, optional outputs; BR-0 on small fleets runs on br_small_kernel).
//
// Phases per decode step k (Section 2.2 model; Algorithms 1 and 2):
//   ARRIVE -> PREDICT (H > 0) -> ROUTE (Stage 1, Stage 2) -> RECORD -> ADVANCE.
//
// Warp 0 is the router and walks the sequential admission loop with warp reductions only; the other
// warps meanwhile settle the requests that end at this step.  Everything else (projection, queue
// compaction, write-back) is spread over all threads.
//
// The admission loop is bound by instruction latency and instruction fetch: a pop is one chain of
// dependent warp instructions (measured: warp maximum 22 cycles, warp sum 47, shuffle or ballot 25 to
// 35, shared-memory load 34, fp64 operation 8), and a loop body of more than a few hundred
// instructions is fetched again on every pop.  So it is written to be short and straight: one loop for
// both stages; the margins m_{g,h} in shared memory, a row per worker, with the lanes spread over h;
// one lane per worker for the three selection keys (free slots, L_g(k), min_h m_{g,h}); the Stage-2
// window in registers of every lane, refilled by one warp maximum per admission; loops over h unrolled
// for H < 20; slots, snapshot edits and rare branches outside the loop.  us per call at G = 64,
// W = 1,024, H = 8, 1,024 instances / G = 21, W = 300, H = 6, 777 instances, 3 steps / G = 8, W = 512, H = 80,
// 1,024 instances, 8 steps: 110 / 672 / 503 with a copy of every part per stage and all loops over h
// unrolled, 77 / 313 / 166 with one loop, loads and envelope in shared memory and the window merged from
// the lanes' lists at every pop, 59 / 175 / 105 now.
//
// Loads are advanced incrementally: L_g(k+1) = L_g(k) - sum of the loads of the requests
// that end at k + number of survivors, so ADVANCE touches only the occupancy bit masks,
// the termination draws and the few slots whose request ends.  Only the horizon projection of BR-H
// streams the per-request state.
#pragma once
#include "br_device.cuh"
#include "br_mitm.cuh"
#include "br_plan.h"
#include "../../include/br.h"

namespace br {

// Shared memory of one instance: byte offsets, filled in by the host.
struct StepLayout {
    int32_t q_key, q_id, q_o, Lh, Ch, dn, iw, Ms, occ, occ0, fin, endm, L0, cap, sub, scal, bw, due, total;
};

// (`quads` and `b4_magic` fill gaps between pointers: with every array behind them eight bytes further on, br_small_kernel
// took 1 % longer over 16 steps, 4,096 instances of G = 32: 172.8 us, 171.7 this way.)
struct StepArgs {
    int32_t G, H, B, W, R_max, S_greedy, occ_words;
    int32_t wl;                 // log2 of the queue-position field of a packed key
    int32_t Wp;                 // W rounded up to whole groups of 128 queue positions
    int32_t HS;                 // row stride of L_g(k+h) in shared memory (>= H + 1)
    int32_t lpw_log2;           // log2 of the lanes that share a worker's row (fleets of up to 16 workers, long horizons)
    int32_t seg_log2;           // lanes per worker that turn its prediction buckets into L_g(k+h)
    int32_t delta_T;
    float gate, c_floor;
    int32_t term_mode;
    int32_t pred_mode;          // 1: c_hat = min(remaining steps, H) from act_end (term_mode 3)
    const int32_t *out_tab;     // output lengths of arrivals (term_mode 3)
    int32_t out_shift;
    int32_t quads;              // slot quads that a thread takes in PREDICT (NT * quads covers A / 4)
    const uint32_t *term_cdf;   // [B] gap thresholds of the constant hazard
    const uint32_t *arr_cdf;
    int32_t arr_len, arr_period, arr_inst_stride;
    uint32_t b4_magic;          // ceil(2^32 / (B / 4)): the worker of quad q is the upper half of q * b4_magic
    const int32_t *len_tab;
    int32_t len_shift;
    int32_t burst_every, burst_size;
    double aD, beta;
    double rel_err;             // Eq. 2: bound on the rounding error of a score, per unit of Delta
    int32_t w_below, w_above;   // Eq. 2: fixed-point weight sums up to / from which a segment clearly rises / falls
    int32_t peak_ok;            // Eq. 1: scores fall strictly beyond the margin (G >= 2)
    int32_t big_window;         // R_max > 5: Stage 2 solves its window by meeting in the middle
    double dn[2 * (BR_MAX_H + 8)];   // (d_h, -2^52 d_h), zero beyond H
    int32_t iw[BR_MAX_H + 8];        // d_h in fixed point (their sum stays below 2^31)
    int32_t N, first_instance, n_steps;
    StepLayout lay;
    br_worker_state ws;
    br_waiting_queue wq;
    const float *term_probs;
    int32_t *assign_out;
    br_load_out out;
    double fix, beta_fix, fix_err;   // scale of penalty sums in fixed point, beta / fix, and what the rounding to it adds
};

// Rows of L_g(k+h) are read by lanes that own a worker each (16-byte loads at the row stride) and by
// lanes that own an offset each (consecutive words): an odd number of 16-byte units keeps both free of
// bank conflicts.
constexpr int step_row_stride(int H)
{
    return 4 * ((step_groups(H) ? step_groups(H) : (H + 4) / 4) | 1);
}

inline StepLayout step_layout(bool fp, int G, int H, int B, int W, int occ_words, bool lifetimes, bool big_window, bool classifier)
{
    StepLayout l;
    const int Wp = (W + 127) / 128 * 128, HS = step_row_stride(H), words = 8 * G * occ_words;
    int n = 0;
    auto take = [&n](int bytes) { const int at = n; n += (bytes + 15) & ~15; return at; };
    l.q_key = take(4 * Wp);
    l.q_id = take(4 * Wp);
    l.q_o = take(lifetimes ? 4 * Wp : 0);
    l.Lh = take(fp ? 4 * (G * HS + 4) : 0);     // (Eq. 2, as the next four) PREDICT: load sums per (worker, floor(c_hat)); L_g(k+h); margins m_{g,h}
    l.Ch = take(H > 0 ? 4 * G * HS : 0);        // PREDICT: request counts
    l.dn = take(fp ? 16 * (HS + 4) : 0);        // (d_h, -2^52 d_h)
    l.iw = take(fp ? 4 * (HS + 4) : 0);         // d_h in fixed point
    l.Ms = take(fp ? 4 * HS : 0);               // envelope M_h; then its growth by an admission
    l.occ = take(words);                        // occupied slots
    l.occ0 = take(words);                       // ... at the start of the step
    l.fin = take(words);                        // constant hazard: slots whose draw says "ends"
    l.endm = take(words);                       // slots whose request ends at this step
    l.L0 = take(4 * G);
    l.cap = take(4 * G);
    l.sub = take(4 * G);                        // loads of the requests that end
    l.scal = take(4 * 32);
    l.bw = take(big_window ? 8 * (1 << 8) + 4 * 32 : 0);
    const int most = W < G * B ? W : G * B;     // admissions of a step
    l.due = take(classifier && G * B > 2 * most ? 2 * G * B : 4 * most);   // requests whose c_hat is refreshed; then the admissions
    l.total = n;
    return l;
}

// Order- and sign-preserving key of a score: Eq. 1 in integers (FP = false) or Eq. 2 in
// fp64 evaluated term by term in h (FP = true).
//
// A term of Eq. 2 is RN(d_h * over) with over = max(delta - m_h, 0) an integer.  X = 2^52 + over is
// a double that needs no conversion instruction (its low word is `over`), and one fused operation
// fma(X, d_h, -2^52 d_h) rounds d_h * over once: the same value as converting and multiplying, at
// two fp64 instructions per term instead of five.
template <bool FP>
struct Scorer {
    span_t<int> md;         // Eq. 2: row of margins m_{g,h} of the selected worker (INT_MAX beyond H)
    span_t<double> dn;      // (d_h, -2^52 d_h) pairs
    int mm;                 // min_h m_{g,h} (Eq. 1: the margin); at or below it no term is positive
    int H, G;
    double aD, beta;

    __device__ __forceinline__ long long key(int delta) const
    {
        if (!FP) {
            int over = delta - mm;
            over = over > 0 ? over : 0;
            return (long long)(delta - G * over);          // |F| < 2^31 by the create-time proof
        } else {
            const double two52 = 4503599627370496.0;
            double pen = 0.0;
#pragma unroll 1
            for (int h = 0; h <= H; h += 4) {
                const int4 m4 = *vec_at<const int4>(md, h);
                const int m[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const double2 d = *vec_at<const double2>(dn, 2 * (h + j));
                    const double x = __hiloint2double(0x43300000, max(delta - m[j], 0));
                    pen = __dadd_rn(pen, __fma_rn(x, d.x, d.y));
                }
            }
            const double dl = __dsub_rn(__hiloint2double(0x43300000, delta), two52);
            return key_of_double(__dsub_rn(__dmul_rn(aD, dl), __dmul_rn(beta, pen)));
        }
    }
    __device__ __forceinline__ static double value(long long k)
    {
        return FP ? double_of_key(k) : (double)k;
    }
};

// warp maximum of 64-bit keys; returns whether this lane holds it
__device__ __forceinline__ bool warp_max64(long long key, long long &wkey)
{
    const int hi = (int)(key >> 32);
    const int mhi = __reduce_max_sync(kFull, hi);
    const unsigned mlo = __reduce_max_sync(kFull, hi == mhi ? (unsigned)key : 0u);
    wkey = (long long)(((unsigned long long)(unsigned)mhi << 32) | mlo);
    return key == wkey;
}

// Slots of worker g that end at step k under the constant hazard, as bit masks of 64 slots each.
// Slots end independently with one probability, so the ending ones are walked by their gaps:
// cdf[j] = floor(2^32 P(gap <= j)), draw t is word t % 4 of the Philox block (k, g, TERM, t / 4),
// and a word u skips gap = #{j : u >= cdf[j]} slots (cdf ascends: the first j with u < cdf[j]).
template <typename CDF, typename OUT>
__device__ __forceinline__ void draw_ending(const CDF cdf, int B, int OW, uint32_t k,
                                            uint32_t g, uint32_t key0, uint32_t key1,
                                            const OUT out)
{
    for (int w = 0; w < OW; ++w) out[w] = 0ull;
    int pos = 0;
    uint4 r = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
    for (unsigned t = 0; t < (unsigned)B; ++t) {          // every draw moves pos forward
        if ((t & 3u) == 0u) r = philox4x32_10(k, g, kStreamTerm, t >> 2, key0, key1);
        const uint32_t u = word_of(r, t & 3u);
        const int room = B - pos;
        if (u >= cdf[room - 1]) break;                    // the gap reaches past the last slot
        int lo = 0, hi = room - 1;                        // u < cdf[hi]
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (u < cdf[mid]) hi = mid; else lo = mid + 1;
        }
        const int slot = pos + lo;
        out[slot >> 6] |= 1ull << (slot & 63);
        pos = slot + 1;
        if (pos >= B) break;
    }
}

// Loads that stay where they are written: a launch opens with one trip to memory for all it needs.
__device__ __forceinline__ int4 ld_now4(const void *p)
{
    int4 v;
    asm volatile("ld.global.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ int ld_now(const void *p)
{
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ long long ld_now8(const void *p)
{
    long long v;
    asm volatile("ld.global.s64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

// Loads of classifier output.  A row is read once, by one thread, at a scattered address; left to
// itself the L2 fetches 128 bytes around a missing sector, of which a refresh uses 32 on average,
// so the loads ask for the smallest fetch the instruction set offers (64 bytes).  Nor do they allocate in L1: where
// shared memory leaves it little, the lines that wait for rows limit how many are in flight (1,024 instances of two
// warps, a quarter of 4,096 rows each: 22.7 us, 15.9 this way; 28 KB of L1).  They are coherent loads: the
// launch overlaps the kernel ahead, which may be the one that writes the rows.
__device__ __forceinline__ float4 ld_row4(const float *p)
{
    float4 v;
    asm volatile("ld.global.L1::no_allocate.L2::64B.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
// a whole row of eight probabilities (32-byte aligned) as one 256-bit load
__device__ __forceinline__ void ld_row8(const float *p, float *o)
{
    unsigned r[8];
    asm volatile("ld.global.L1::no_allocate.L2::64B.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "l"(p));
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = __uint_as_float(r[i]);
}

// R classifier rows of H < HT probabilities, zero beyond, asked for together in the widest pieces that every row
// allows (width: 8, 4, 2 or 1 probabilities).
template <int HT, int R>
__device__ __forceinline__ void load_rows(const float *const (&row)[R], int H, int width, float (&v)[R][HT])
{
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int h = 0; h < HT; ++h) v[r][h] = 0.0f;
    if (width == 8) {
#pragma unroll
        for (int h = 0; h + 8 <= HT; h += 8)
            if (h < H)
#pragma unroll
                for (int r = 0; r < R; ++r) ld_row8(row[r] + h, &v[r][h]);
    } else if (width == 4) {
#pragma unroll
        for (int h = 0; h < HT; h += 4)
            if (h < H)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4 x = ld_row4(row[r] + h);
                    v[r][h] = x.x; v[r][h + 1] = x.y; v[r][h + 2] = x.z; v[r][h + 3] = x.w;
                }
    } else if (width == 2) {
#pragma unroll
        for (int h = 0; h < HT; h += 2)
            if (h < H)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float2 x = *reinterpret_cast<const float2 *>(row[r] + h);
                    v[r][h] = x.x; v[r][h + 1] = x.y;
                }
    } else {
#pragma unroll
        for (int h = 0; h < HT; ++h)
            if (h < H)
#pragma unroll
                for (int r = 0; r < R; ++r) v[r][h] = row[r][h];
    }
}

// Sum of the absolute probabilities of a row of a long horizon.  The order of the fp32 sum is free: it only feeds a
// bound with slack.
__device__ __forceinline__ float row_sum(const float *q, int H, int width)
{
    float s = 0.0f;
    if (width == 8) {
        for (int h = 0; h < H; h += 8) {
            float v[8];
            ld_row8(q + h, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) s += fabsf(v[j]);
        }
    } else if (width == 4) {
#pragma unroll 2
        for (int h = 0; h < H; h += 4) {
            const float4 v = ld_row4(q + h);
            s += (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
        }
    } else {
#pragma unroll 4
        for (int h = 0; h < H; ++h) s += fabsf(q[h]);
    }
    return s;
}

constexpr int kRegWin = 5;       // Stage-2 windows of up to five requests are scored one subset per lane
constexpr int kBigWinLow = 8;    // larger windows (up to BR_MAX_RMAX = 16): subsets of the low eight entries are sorted
// marks a condition as the exception, so that its block leaves the straight path of the admission loop
__device__ __forceinline__ bool rare(bool x) { return __builtin_expect(x, 0); }

// descending order of two keys
__device__ __forceinline__ void order2(int &a, int &b) { const int hi = max(a, b); b = min(a, b); a = hi; }

constexpr int kListEnd = 0x7FFFFFFF;         // head of a lane's list that ran dry although the lane may hold more keys
constexpr int kQBeyond = (int)0x8000FFFFu;   // key of a position beyond the queue (no slot index reaches 0xFFFF)

// The rarely taken branches of the router live in functions of their own: inlined, they would spread
// the admission loop over more instructions than the instruction cache of a scheduler holds.
__device__ __noinline__ uint4 philox_call(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t k0, uint32_t k1)
{
    return philox4x32_10(c0, c1, c2, 0u, k0, k1);
}

// the R largest keys of the queue: lane r gets the r-th largest
__device__ __noinline__ int largest_keys(span_t<int> q_key, int n_w, int R, int lane)
{
    int thr = 0x7FFFFFFF, mine = 0;
#pragma unroll 1
    for (int r = 0; r < R; ++r) {
        int x = 0;
#pragma unroll 1
        for (int i = lane; i < n_w; i += 32) { const int y = q_key[i]; if (y < thr) x = max(x, y); }
        thr = __reduce_max_sync(kFull, x);
        if (lane == r) mine = thr;
    }
    return mine;
}

struct WindowChoice { long long wk; unsigned chosen; int dsum; };

// Best subset of a window of 6 to 16 requests (Appendix "Bit-set subset selection"): lane r holds the
// r-th largest key in `wkey`.  m0: the margin of offset `lane` (Eq. 2).
template <bool FP>
__device__ __noinline__ WindowChoice big_window(const Scorer<FP> sc, span_t<unsigned long long> keys, span_t<int> off,
                                                span_t<int> win, int wkey, int R, int lim, int WL, int m0, int lane)
{
    if (lane < R) win[lane] = wkey >> WL;
    __syncwarp();
    const int ra = min(kBigWinLow, (R + 1) / 2), rb = R - ra, n = 1 << ra;
    // subsets of the low entries, sorted by (size, sum, mask)
#pragma unroll 1
    for (int x = lane; x < n; x += 32) {
        int sum = 0;
        for (int j = 0; j < ra; ++j) if ((x >> j) & 1) sum += win[j];
        keys[x] = ((unsigned long long)__popc(x) << 56) | ((unsigned long long)(unsigned)sum << 16) | (unsigned)x;
    }
    __syncwarp();
#pragma unroll 1
    for (int k2 = 2; k2 <= n; k2 <<= 1) {
#pragma unroll 1
        for (int j = k2 >> 1; j > 0; j >>= 1) {
#pragma unroll 1
            for (int i = lane; i < n; i += 32) {
                const int p = i ^ j;
                if (p > i) {
                    const unsigned long long x = keys[i], y = keys[p];
                    const bool up = (i & k2) == 0;
                    if ((x > y) == up) { keys[i] = y; keys[p] = x; }
                }
            }
            __syncwarp();
        }
    }
    if (lane == 0) {
        int at = 0, binom = 1;
#pragma unroll 1
        for (int c = 0; c <= ra; ++c) { off[c] = at; at += binom; binom = binom * (ra - c) / (c + 1); }
        off[ra + 1] = at;
    }
    __syncwarp();
    // the peak of the score in Delta (H <= 16 here, so one offset per lane)
    int peak = sc.mm;
    if (FP) {
        double wsum = 0.0;
#pragma unroll 1
        for (int h = 0; h <= sc.H; ++h) if (sc.md[h] <= m0) wsum = __dadd_rn(wsum, sc.dn[2 * h]);
        const bool past = lane <= sc.H && !(sc.aD > __dmul_rn(sc.beta, wsum));
        peak = (int)__reduce_min_sync(kFull, past ? (unsigned)m0 : 0x7FFFFFFFu);
    }
    MitmBest b; b.lo_sum = -1; b.lo_mask = 0xFFFFFFFFu; b.hi_sum = 0x7FFFFFFF; b.hi_mask = 0xFFFFFFFFu;
#pragma unroll 1
    for (unsigned mh = lane; mh < (1u << rb); mh += 32) {
        const int ph = __popc(mh);
        if (ph > lim) continue;
        int sh = 0;
        for (unsigned t = mh; t; t &= t - 1) sh += win[ra + __ffs(t) - 1];
        mitm_probe(keys, off, ra, lim, peak, mh, sh, ph, b);
    }
    // largest sum at or below the peak, smallest above it, lowest mask among equals
    const int ls = __reduce_max_sync(kFull, b.lo_sum);
    const unsigned lm = __reduce_min_sync(kFull, b.lo_sum == ls ? b.lo_mask : 0xFFFFFFFFu);
    const int hs = __reduce_min_sync(kFull, b.hi_sum);
    const unsigned hm = __reduce_min_sync(kFull, b.hi_sum == hs ? b.hi_mask : 0xFFFFFFFFu);
    WindowChoice r; r.wk = kNoKey; r.chosen = 1u; r.dsum = 0;
    const long long f = sc.key((lane & 1) ? (hs != 0x7FFFFFFF ? hs : 0) : max(ls, 0));
    const long long fl = __shfl_sync(kFull, f, 0), fh = __shfl_sync(kFull, f, 1);
    if (ls >= 0) { r.wk = fl; r.chosen = lm; r.dsum = ls; }
    if (hs != 0x7FFFFFFF && (fh > r.wk || (fh == r.wk && hm < r.chosen))) { r.wk = fh; r.chosen = hm; r.dsum = hs; }
    __syncwarp();
    return r;
}

// argmax_i F_g({i}) by scoring every waiting request, earliest arrival on ties; packed key, 0 if none.
// Safe requests (s <= min_h m_{g,h}) score alpha D s exactly, which grows with s, so of those only the
// largest key per lane is scored.
template <bool FP>
__device__ __noinline__ int best_of_all(const Scorer<FP> sc, span_t<int> q_key, int n_w, int WL, unsigned posmask, int lane)
{
    long long bk = kNoKey; int bkey = 0, best_safe = 0;
#pragma unroll 1
    for (int i = lane; i < n_w + 32; i += 32) {
        int x = i < n_w ? q_key[i] : 0;
        if (x > 0 && (x >> WL) <= sc.mm) { best_safe = max(best_safe, x); x = 0; }
        if (i >= n_w) x = best_safe;
        if (x > 0) {
            const long long f = sc.key(x >> WL);
            if (f > bk || (f == bk && ((unsigned)x & posmask) > ((unsigned)bkey & posmask))) { bk = f; bkey = x; }
        }
    }
    long long wk;
    const bool in = warp_max64(bk, wk);
    const unsigned mt = __reduce_max_sync(kFull, in ? (unsigned)bkey & posmask : 0u);
    const int who = (int)__reduce_min_sync(kFull, in && ((unsigned)bkey & posmask) == mt ? (unsigned)lane : 32u);
    return wk == kNoKey ? 0 : __shfl_sync(kFull, bkey, who);
}

// row g of the optional F-score matrix: F_g({i}) of every waiting request.  The margins of a short horizon stay in
// registers (read again for every request, 1,024 instances of G = 40, W = 128, H = 4: 119 us, 98
// this way).
template <bool FP, int NC>
__device__ __noinline__ void score_column(const Scorer<FP> sc, double *F, span_t<int> q_key, int n_w, int W, int G, int WL, int lane)
{
    int4 m[NC > 0 ? NC : 1];
    if (FP && NC > 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) m[c] = *vec_at<const int4>(sc.md, 4 * c);
    }
#pragma unroll 1
    for (int i = lane; i < W; i += 32) {
        double f = 0.0;
        if (i < n_w) {
            const int delta = q_key[i] >> WL;
            if (FP && NC > 0) {
                double pen = 0.0;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const int mj[4] = {m[c].x, m[c].y, m[c].z, m[c].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const double2 d = *vec_at<const double2>(sc.dn, 2 * (4 * c + j));
                        pen = __dadd_rn(pen, __fma_rn(__hiloint2double(0x43300000, max(delta - mj[j], 0)), d.x, d.y));
                    }
                }
                f = __dsub_rn(__dmul_rn(sc.aD, (double)delta), __dmul_rn(sc.beta, pen)) + 0.0;      // (-0.0 -> +0.0)
            } else {
                f = Scorer<FP>::value(sc.key(delta));
            }
        }
        F[(size_t)i * G] = f;
    }
}

// FP: Eq. 2 scores (else Eq. 1).  GW: workers per router lane.  NC: step_groups(H).  LEAN: fewer registers.
// Registers: the router's chain is the longest path, and it is shorter with more of them than with more
// warps resident (G = 64, H = 8, one instance: 22.0 us at 72 registers, 19.4 at 96; 777 instances of G = 21,
// H = 6: 194 and 181; G = 8, H = 80: 127 at 96, 119 at 128; H = 12 to 19: step_register_cap).  Batches that just miss being
// resident in one wave take the lean instantiation where there is one (step_registers, step_launch).
// EARLY: a single warp under the constant hazard (32 threads, term_mode 1), with the requests that end settled ahead of
// the router.
// (It has no output lengths to carry: with the loads of a queue that might carry them, Eq. 1 on up to 32 workers took 88
// registers instead of 75, 20 warps to an SM instead of 24.  G = 16, B = 96, W = 256, 3,256 instances: 21.5 us, 17.2 this
// way.  18 to 20 an SM, which either holds, gain 2 % in the kernel and lose 3 to 4 back to back, 2,960: 16.3, 16.9: the
// next launch's first blocks find room on some SMs only.)
template <bool FP, int GW, int NC, bool LEAN, bool EARLY>
__global__ void __maxnreg__(step_register_cap(FP, NC, LEAN)) br_step_kernel(const __grid_constant__ StepArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int NT = EARLY ? 32 : blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = EARLY ? 0 : tid >> 5, nwarps = NT >> 5;
    const int G = a.G, H = FP ? a.H : 0, B = a.B, W = a.W, A = G * B, OW = a.occ_words, WL = a.wl;
    const int H1 = H + 1, HS = NC > 0 ? 4 * (NC | 1) : a.HS;
    constexpr int HC = NC > 0 ? 1 : 3;                // horizon offsets per lane
    constexpr int HT = 4 * NC;                        // offsets of the unrolled loops
    const unsigned posmask = (1u << WL) - 1u;
    const int inst = a.first_instance + blockIdx.x;
    const bool life = !EARLY && a.term_mode == 3;     // requests carry their output lengths
    const bool classifier = FP && H > 0 && a.pred_mode == 0;
    const unsigned t_entry = (unsigned)clock64();

    // ---- shared memory ----
    const auto q_key = mk_span(reinterpret_cast<int *>(smem + a.lay.q_key), a.Wp);
    const auto q_id = mk_span(reinterpret_cast<unsigned *>(smem + a.lay.q_id), a.Wp);
    const auto q_o = mk_span(reinterpret_cast<int *>(smem + a.lay.q_o), life ? a.Wp : 0);
    const auto Lh = mk_span(reinterpret_cast<int *>(smem + a.lay.Lh), FP ? G * HS + 4 : 0);
    const auto Ch = mk_span(reinterpret_cast<int *>(smem + a.lay.Ch), H > 0 ? G * HS : 0);
    const auto dn_s = mk_span(reinterpret_cast<double *>(smem + a.lay.dn), FP ? 2 * (HS + 4) : 0);
    const auto iw_s = mk_span(reinterpret_cast<int *>(smem + a.lay.iw), FP ? HS + 4 : 0);
    const auto Ms = mk_span(reinterpret_cast<int *>(smem + a.lay.Ms), FP ? HS : 0);
    const auto occ = mk_span(reinterpret_cast<unsigned long long *>(smem + a.lay.occ), G * OW);
    const auto occ0 = mk_span(reinterpret_cast<unsigned long long *>(smem + a.lay.occ0), G * OW);
    const auto occ032 = mk_span(reinterpret_cast<unsigned *>(smem + a.lay.occ0), 2 * G * OW);
    const auto fin = mk_span(reinterpret_cast<unsigned long long *>(smem + a.lay.fin), G * OW);
    const auto endm = mk_span(reinterpret_cast<unsigned long long *>(smem + a.lay.endm), G * OW);
    const auto endm32 = mk_span(reinterpret_cast<unsigned *>(smem + a.lay.endm), 2 * G * OW);
    const auto occ32 = mk_span(reinterpret_cast<unsigned *>(smem + a.lay.occ), 2 * G * OW);
    const auto L0_s = mk_span(reinterpret_cast<int *>(smem + a.lay.L0), G);
    const auto cap_s = mk_span(reinterpret_cast<int *>(smem + a.lay.cap), G);
    const auto sub_load = mk_span(reinterpret_cast<unsigned *>(smem + a.lay.sub), G);
    const auto scal = mk_span(reinterpret_cast<int *>(smem + a.lay.scal), 32);
    const auto bw_keys = mk_span(reinterpret_cast<unsigned long long *>(smem + a.lay.bw), a.big_window ? (1 << kBigWinLow) : 0);
    const auto bw_off = mk_span(reinterpret_cast<int *>(smem + a.lay.bw + (8 << kBigWinLow)), a.big_window ? 16 : 0);
    const auto bw_win = mk_span(reinterpret_cast<int *>(smem + a.lay.bw + (8 << kBigWinLow) + 64), a.big_window ? 16 : 0);
    const auto due_list = mk_span(reinterpret_cast<unsigned short *>(smem + a.lay.due), classifier ? A : 0);
    // admissions of the step in order: queue position << 15 | worker << 9 | free slots of the worker before it; shares the
    // memory of the due list, which is not needed once the projection stands.  The key of an admitted request stays in
    // the queue, its sign bit set, until slots are given out (8 bytes an admission, the key among them, left room for
    // 19 instances of BR-0 at G = 64, W = 512 on an SM instead of 22)
    const auto adm = mk_span(reinterpret_cast<unsigned *>(smem + a.lay.due), min(W, A));
    // scal: [0] queue length after routing, [1] admitted, [2] Stage-1 iterations, [3] Stage-2 pops,
    //       [4] status bits of the step, [5] status bits of the prologue, [6] lowest admitted position,
    //       [16..31] kept entries per warp (two sets of eight, compaction)

    // what comes from the arguments alone is set up while the kernel before this one drains
    if (tid < 32) scal[tid] = 0;
    if (FP) {
#pragma unroll 1
        for (int i = 4 * tid; i < G * HS; i += 4 * NT) { *vec_at<int4>(Lh, i) = make_int4(0, 0, 0, 0); if (H > 0) *vec_at<int4>(Ch, i) = make_int4(0, 0, 0, 0); }
#pragma unroll 1
        for (int h = tid; h < HS + 4; h += NT) {
            dn_s[2 * h] = a.dn[2 * h]; dn_s[2 * h + 1] = a.dn[2 * h + 1];
            iw_s[h] = a.iw[h];
            if (h < HS) Ms[h] = h < H1 ? 0 : 0x7FFFFFFF;
        }
    }
    stream_order_gate();

    // ---- per-instance global rows ----
    const auto g_base = mk_span(a.ws.act_base + (size_t)inst * A, A);
    const auto g_aid = mk_span(a.ws.act_id ? a.ws.act_id + (size_t)inst * A : nullptr, A);
    const auto g_chat0 = mk_span(a.ws.act_chat0 ? a.ws.act_chat0 + (size_t)inst * A : nullptr, A);
    const auto g_kref = mk_span(a.ws.act_kref ? a.ws.act_kref + (size_t)inst * A : nullptr, A);
    const auto g_end = mk_span(life ? a.ws.act_end + (size_t)inst * A : nullptr, A);
    const auto g_qs = mk_span(a.wq.s + (size_t)inst * W, W);
    const auto g_qid = mk_span(a.wq.id + (size_t)inst * W, W);
    const auto g_qo = mk_span(life ? a.wq.o + (size_t)inst * W : nullptr, W);
    const auto t_len = mk_span(a.len_tab, a.len_tab ? (1ll << (32 - a.len_shift)) : 0);
    const auto t_out = mk_span(a.out_tab, a.out_tab ? (1ll << (32 - a.out_shift)) : 0);
    const auto t_term = mk_span(a.term_cdf, B);

    // ---- snapshot to shared memory: everything is asked for before the first answer is used ----
    // (one array after another, each loop waiting for its loads: 3,500 cycles for one instance of G = 64, W = 1,024;
    // 2,600 this way)
    const unsigned long long seed = (unsigned long long)ld_now8(a.ws.seed + inst);
    int k = ld_now(a.ws.step + inst);
    uint32_t next_id = (uint32_t)ld_now(a.ws.next_id + inst);
    int n_w = ld_now(a.wq.n + inst);
    unsigned long long occ_1 = 0ull;
    int nact_1 = 0, load_1 = 0;
    if (tid < G * OW) occ_1 = (unsigned long long)ld_now8(a.ws.occ + (size_t)inst * G * OW + tid);
    if (tid < G) {
        nact_1 = ld_now(a.ws.nact + (size_t)inst * G + tid);
        load_1 = (int)ld_now8(a.ws.load + (size_t)inst * G + tid);
    }
    int4 s_1 = make_int4(0, 0, 0, 0), id_1 = s_1, o_1 = s_1;
    if (4 * tid < W) {
        s_1 = ld_now4(vec_at<const int4>(g_qs, 4 * tid));
        id_1 = ld_now4(vec_at<const int4>(g_qid, 4 * tid));
        if (life) o_1 = ld_now4(vec_at<const int4>(g_qo, 4 * tid));
    }
    const uint32_t key0 = (uint32_t)seed, key1 = (uint32_t)(seed >> 32);
    int bad = 0;
    if (n_w < 0 || n_w > W) { bad = BR_ST_BAD_STATE; n_w = n_w < 0 ? 0 : W; }
#pragma unroll 1
    for (int i = tid; i < G * OW; i += NT) {
        const unsigned long long o = i == tid ? occ_1 : reinterpret_cast<const unsigned long long *>(a.ws.occ)[(size_t)inst * G * OW + i];
        occ[i] = o; occ0[i] = o; endm[i] = 0ull;
    }
#pragma unroll 1
    for (int g = tid; g < G; g += NT) {
        int na = g == tid ? nact_1 : a.ws.nact[(size_t)inst * G + g];
        const int l = g == tid ? load_1 : (int)a.ws.load[(size_t)inst * G + g];
        if (na < 0 || na > B) { bad = BR_ST_BAD_STATE; na = na < 0 ? 0 : B; }
        cap_s[g] = B - na;
        L0_s[g] = l;
        sub_load[g] = 0u;
    }
#pragma unroll 1
    for (int p0 = 4 * tid; p0 < a.Wp; p0 += 4 * NT) {
        int4 kk;
        kk.x = p0 + 0 < n_w ? (s_1.x << WL) | (int)(posmask - (unsigned)(p0 + 0)) : kQBeyond;
        kk.y = p0 + 1 < n_w ? (s_1.y << WL) | (int)(posmask - (unsigned)(p0 + 1)) : kQBeyond;
        kk.z = p0 + 2 < n_w ? (s_1.z << WL) | (int)(posmask - (unsigned)(p0 + 2)) : kQBeyond;
        kk.w = p0 + 3 < n_w ? (s_1.w << WL) | (int)(posmask - (unsigned)(p0 + 3)) : kQBeyond;
        *vec_at<int4>(q_key, p0) = kk;
        *vec_at<int4>(q_id, p0) = id_1;
        if (life) *vec_at<int4>(q_o, p0) = o_1;
        const int p1 = p0 + 4 * NT;                       // the next piece
        s_1 = id_1 = o_1 = make_int4(0, 0, 0, 0);
        if (p1 < W) {
            s_1 = ld_now4(vec_at<const int4>(g_qs, p1));
            id_1 = ld_now4(vec_at<const int4>(g_qid, p1));
            if (life) o_1 = ld_now4(vec_at<const int4>(g_qo, p1));
        }
    }
    __syncthreads();
    if (bad) atomicOr(&scal[5], bad);

#pragma unroll 1
    for (int it = 0; it < a.n_steps; ++it, ++k) {
        const size_t orow = (size_t)it * a.N + inst;
        const auto probs = mk_span(a.term_probs ? a.term_probs + orow * (size_t)A * H : nullptr, (long long)A * H);
        unsigned t_phase[7];
        const bool timing = a.out.phase_cycles != nullptr && tid == 0;
        if (timing) t_phase[0] = (unsigned)clock64();

        // ================= ARRIVE =================
        // The arrival-count row and the prompt lengths that the first arrivals would take are asked
        // for together; they are used after the projection.
        uint32_t row0 = 0xFFFFFFFFu, row1 = 0xFFFFFFFFu, u_arr = 0u;
        span_t<const uint32_t> row = mk_span((const uint32_t *)nullptr, 0);
        int s_new = 0;
        if (a.arr_cdf) {
            row = mk_span(a.arr_cdf + ((size_t)inst * a.arr_inst_stride + (size_t)(a.arr_period == 1 ? 0 : k % a.arr_period)) * a.arr_len, a.arr_len);
            if (lane < a.arr_len) row0 = row[lane];
            if (lane + 32 < a.arr_len) row1 = row[lane + 32];
            // one call serves both: lane 31 draws the count, its length word is in lane 30's block
            const bool cnt = lane == 31;
            const uint4 r = philox_call((uint32_t)k, cnt ? 0u : (uint32_t)tid >> 2, cnt ? kStreamArrCount : kStreamArrLen, key0, key1);
            u_arr = __shfl_sync(kFull, r.x, 31);
            const uint32_t last = __shfl_sync(kFull, r.w, 30);
            s_new = t_len[(cnt ? last : word_of(r, tid & 3)) >> a.len_shift];
        }
        // A single warp settles, while these loads are on their way, which of the running requests end at this step, and asks
        // for the first of every worker's: the values are used after routing.
        int pend[GW], pslot[GW];
#pragma unroll
        for (int w = 0; w < GW; ++w) { pend[w] = 0; pslot[w] = -1; }
        if (EARLY) {
#pragma unroll
            for (int w = 0; w < GW; ++w) {
                const int g = lane + 32 * w;
                if (g < G) {
                    draw_ending(t_term, B, OW, (uint32_t)k, (uint32_t)g, key0, key1, fin + (size_t)g * OW);
#pragma unroll 1
                    for (int x = 0; x < OW; ++x) {
                        const unsigned long long e = occ0[g * OW + x] & fin[g * OW + x];
                        endm[g * OW + x] = e;
                        if (e && pslot[w] < 0) pslot[w] = 64 * x + __ffsll((long long)e) - 1;
                    }
                    if (pslot[w] >= 0) pend[w] = ld_now(&g_base[g * B + pslot[w]]);
                }
            }
        }
        if (timing) t_phase[1] = (unsigned)clock64();

        // ============ PREDICT (H > 0): c_hat maintenance + horizon projection ============
        // Every running request adds (cur, 1) to the bucket (worker, floor(c_hat)); the buckets become
        // L_g(k+h) = sum_{j >= h} T_j + h * sum_{j >= h} C_j by suffix sums.  A thread takes `quads` slot quads, the next one
        // requested before this one is worked on.  The 32 lanes of a warp read eight pieces of 64 bytes a worker apart, or a
        // little more (the pieces of a run of eight workers one after another): consecutive quads in consecutive lanes are
        // one worker's, whose few buckets serialise the atomics; rows of workers several apart share banks; and
        // eight slots of one worker per thread touch 32 lines with every load.  (Look-ahead, 1,184 instances of G = 64, B = 64,
        // three steps, H = 2 / 25: 77 / 106 us with consecutive quads, 77 / 112 with pieces 4 * quads quads, here four
        // workers, apart, 63 / 99 this way.)
        int n_due = 0;                                    // requests on this warp's part of the due list
        const auto due_w = due_list + (size_t)(classifier ? 128 * warp * a.quads : 0);
        if (FP && H > 0) {
            const int A4 = A >> 2, span = (B + 15) >> 4;
            int left = a.quads, run = min(span, left), in_run = run;
            int q = (warp << 5) * left + (lane & ~3) * run + (lane & 3);
            auto next = [&]() {
                --left;
                q += 4;
                if (--in_run == 0) {
                    // the other lanes' pieces of the run, then this lane's first of the next
                    q += 28 * run - (lane & ~3) * run;
                    in_run = run = min(span, left);
                    q += (lane & ~3) * run;
                }
            };
            const bool look = a.pred_mode == 1;
            int4 b4, x4 = make_int4(0, 0, 0, 0);                              // act_base; act_end or chat0
            unsigned kr = 0u;                                                 // refresh stamps
            auto fetch = [&]() {
                b4 = make_int4(kEmpty, kEmpty, kEmpty, kEmpty);
                if (q < A4 && left > 0) {
                    b4 = *vec_at<const int4>(g_base, 4 * q);
                    if (look) {
                        x4 = *vec_at<const int4>(g_end, 4 * q);
                    } else {
                        x4 = *vec_at<const int4>(g_chat0, 4 * q);
                        kr = *vec_at<const unsigned>(g_kref, 4 * q);
                    }
                }
            };
            fetch();
            // (Adds and stores that are predicated in inline assembly instead of branched around: the compiler must not move
            // accesses across them, and its own atomics are faster, a count of one above all.  592 of G = 48, B = 96, H = 6,
            // 97 % of the slots in one bucket: 11,600 cycles a step that way, 10,400 this; 425 shapes 1.2 % on average)
            const unsigned k_4 = (unsigned)(k & 255) * 0x01010101u, lt = (1u << lane) - 1u;
            const float Hf = (float)H, dTf = (float)a.delta_T, two23 = 8388608.0f;
#pragma unroll 1
            while (left > 0) {
                const int q_now = q;
                const int g = (int)__umulhi((unsigned)q_now, a.b4_magic);
                const int bs[4] = {b4.x, b4.y, b4.z, b4.w}, xs[4] = {x4.x, x4.y, x4.z, x4.w};
                const unsigned k4 = kr;
                next();
                fetch();
                if (look) {
                    // perfect lookahead: c_hat = min(r_i(k), H) with r_i(k) = act_end - k + 1 steps still to run.
                    // A request whose last step this is (act_end == k) is settled right here.
                    unsigned fb = 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool live = bs[j] != kEmpty;
                        const int at = g * HS + min(max(xs[j] - k + 1, 0), H);
                        if (live) {
                            atomicAdd(reinterpret_cast<unsigned *>(&Lh[at]), (unsigned)(bs[j] + k));
                            atomicAdd(&Ch[at], 1);
                        }
                        fb |= live && xs[j] == k ? 1u << j : 0u;
                    }
                    if (fb) {
                        const int slot = 4 * q_now - g * B;
                        atomicOr(&endm32[2 * g * OW + (slot >> 5)], fb << (slot & 31));
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if ((fb >> j) & 1u) { atomicAdd(&sub_load[g], (unsigned)(bs[j] + k)); g_base[4 * q_now + j] = kEmpty; }
                    }
                } else {
                    // requests that are not due only age; the ones due for a refresh take c_hat = H (gate closed:
                    // the conservative anchor) and go on the warp's list, whose rows are read below.  Ages are bytes, taken
                    // from k four at a time; a byte t and floor(c) become a float and an integer through the
                    // mantissa of 2^23 + x (conversions have a quarter of the rate).
                    const unsigned t4 = ((k_4 | 0x80808080u) - (k4 & 0x7F7F7F7Fu)) ^ ((k_4 ^ ~k4) & 0x80808080u);
                    bool live[4], due[4];
                    int at[4], n = 0, to[4];
                    unsigned dues = 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float t = __int_as_float((int)__byte_perm(t4, 0x4B000000u, 0x7540u + j)) - two23;
                        const float c = __int_as_float(xs[j]) - t;
                        live[j] = bs[j] != kEmpty;
                        due[j] = live[j] & ((t >= dTf) | (c < a.c_floor));
                        const float ch = due[j] ? Hf : fminf(fmaxf(c, 0.0f), Hf);
                        at[j] = g * HS + __float_as_int(__fadd_rd(ch, two23)) - 0x4B000000;
                        to[j] = n;                                            // place among the thread's
                        n += due[j] ? 1 : 0;
                        dues |= due[j] ? 0xFFu << (8 * j) : 0u;
                    }
                    // places among the warp's: the counts of the lanes below, bit by bit
                    const unsigned n1 = __ballot_sync(kFull, n & 1), n2 = __ballot_sync(kFull, n & 2), n4 = __ballot_sync(kFull, n & 4);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (live[j]) {
                            atomicAdd(reinterpret_cast<unsigned *>(&Lh[at[j]]), (unsigned)(bs[j] + k));
                            atomicAdd(&Ch[at[j]], 1);
                        }
                    }
                    const int first = n_due + __popc(n1 & lt) + 2 * __popc(n2 & lt) + 4 * __popc(n4 & lt);
                    n_due += __popc(n1) + 2 * __popc(n2) + 4 * __popc(n4);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (due[j]) due_w[first + to[j]] = (unsigned short)(4 * q_now + j);
                    if (dues) {
                        const int anchor = __float_as_int(Hf);
                        *vec_at<int4>(g_chat0, 4 * q_now) = make_int4(due[0] ? anchor : xs[0], due[1] ? anchor : xs[1], due[2] ? anchor : xs[2], due[3] ? anchor : xs[3]);
                        *vec_at<unsigned>(g_kref, 4 * q_now) = (k4 & ~dues) | (k_4 & dues);
                    }
                }
            }
            if (classifier) {
                // The classifier row of every request on the warp's list.  p_fin = 1 - prod (1 - q_h) <= sum |q_h| while that
                // sum is below one: when the fp32 sum is clearly below the gate the fp64 product cannot reach it and is
                // not evaluated.
                __syncwarp();
                const float *rows = reinterpret_cast<const float *>(raw_of(probs));
                const int width = (H & 7) == 0 && (reinterpret_cast<size_t>(rows) & 31) == 0 ? 8 : (H & 3) == 0 ? 4 : (H & 1) == 0 ? 2 : 1;
                const float closed = fminf(a.gate, 1.0f);
                // rows in flight per thread: as many as registers hold beside their probabilities (H = 8 to 11, two instead of
                // three: one cluster of G = 32 with terminations from rows 24.9 us, 26.7; batches level.  H = 12 to 19, one
                // instead of two: 2,072 of G = 32, H = 16 131 us, 137)
                constexpr int R = NC == 2 ? 4 : NC == 3 ? 3 : 2;
#pragma unroll 1
                for (int e1 = 0; e1 < n_due; e1 += 32 * R) {
                    const int e0 = e1 + lane;
                    int sa[R];
                    const float *row[R];
                    bool open[R];
                    double c[R], surv[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        sa[r] = due_w[e0 + 32 * r < n_due ? e0 + 32 * r : e1];
                        row[r] = rows + (size_t)sa[r] * H;
                        c[r] = 0.0; surv[r] = 1.0;
                    }
                    bool any = false;
                    if (NC > 0) {
                        float v[R][NC > 0 ? 4 * NC : 1];
                        load_rows(row, H, width, v);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            float sum = 0.0f;
#pragma unroll
                            for (int h = 0; h < HT; ++h) sum += fabsf(v[r][h]);
                            open[r] = e0 + 32 * r < n_due && !(sum * 1.0001f < closed);
                            any = any || open[r];
                        }
                        if (any) {
                            // E[min(r, H)] = sum_h prod_{j<h} (1 - q_j)
#pragma unroll
                            for (int h = 0; h < HT; ++h)
                                if (h < H)
#pragma unroll
                                    for (int r = 0; r < R; ++r) {
                                        c[r] = __dadd_rn(c[r], surv[r]);
                                        surv[r] = __dmul_rn(surv[r], __dsub_rn(1.0, (double)v[r][h]));
                                    }
                        }
                    } else {
                        float sum[R];
#pragma unroll
                        for (int r = 0; r < R; ++r) sum[r] = row_sum(row[r], H, width);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            open[r] = e0 + 32 * r < n_due && !(sum[r] * 1.0001f < closed);
                            any = any || open[r];
                        }
                        if (any)
#pragma unroll 1
                            for (int h = 0; h < H; ++h)
#pragma unroll
                                for (int r = 0; r < R; ++r) {
                                    c[r] = __dadd_rn(c[r], surv[r]);
                                    surv[r] = __dmul_rn(surv[r], __dsub_rn(1.0, (double)row[r][h]));
                                }
                    }
                    if (any) {
                        unsigned cur[R];
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            open[r] = open[r] && __dsub_rn(1.0, surv[r]) >= (double)a.gate;
                            cur[r] = open[r] ? (unsigned)(g_base[sa[r]] + k) : 0u;
                        }
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            if (!open[r]) continue;
                            double cc = c[r] < (double)a.c_floor ? (double)a.c_floor : c[r];      // clipped to [floor, H]
                            cc = cc > (double)H ? (double)H : cc;
                            const float cf = (float)cc;
                            g_chat0[sa[r]] = cf;
                            const int nh = min(max((int)floorf(cf), 0), H);
                            if (nh != H) {                                      // from the anchor's bucket to its own
                                const int g = (int)__umulhi((unsigned)sa[r] >> 2, a.b4_magic);
                                atomicAdd(reinterpret_cast<unsigned *>(&Lh[g * HS + H]), 0u - cur[r]);
                                atomicAdd(&Ch[g * HS + H], -1);
                                atomicAdd(reinterpret_cast<unsigned *>(&Lh[g * HS + nh]), cur[r]);
                                atomicAdd(&Ch[g * HS + nh], 1);
                            }
                        }
                    }
                }
            }
        }
        // (This barrier is for the compiler: where it cannot tell that a warp is whole after loops of divergent length, it
        // guards every warp maximum of the admission loop, and a pop takes a fifth longer.)
        if (FP && H > 0) __syncthreads();
        // arrivals join the queue
        int n_arr = 0;
        if (a.arr_cdf) {
            n_arr = __popc(__ballot_sync(kFull, lane < a.arr_len && u_arr >= row0)) +
                    __popc(__ballot_sync(kFull, lane + 32 < a.arr_len && u_arr >= row1));
#pragma unroll 1
            for (int j0 = 64; j0 < a.arr_len; j0 += 32) {
                const int j = j0 + lane;
                n_arr += __popc(__ballot_sync(kFull, (j < a.arr_len) && (u_arr >= row[j])));
            }
            if (a.burst_every > 0 && k > 0 && (k % a.burst_every) == 0) n_arr += a.burst_size;
        }
        const int n_w_old = n_w;
#pragma unroll 1
        for (int j = tid; j < n_arr; j += NT) {
            const int pos = n_w_old + j;
            if (pos >= W) break;
            int s = s_new;
            if (j != tid) {
                const uint4 r = philox_call((uint32_t)k, (uint32_t)j >> 2, kStreamArrLen, key0, key1);
                s = t_len[word_of(r, j & 3) >> a.len_shift];
            }
            q_key[pos] = (s << WL) | (int)(posmask - (unsigned)pos);
            q_id[pos] = next_id + (unsigned)j;
            if (life) {
                const uint4 ro = philox_call((uint32_t)k, (uint32_t)j >> 2, kStreamArrOut, key0, key1);
                q_o[pos] = t_out[word_of(ro, j & 3) >> a.out_shift];
            }
        }
        const int n_drop = max(n_w + n_arr - W, 0);
        n_w = n_w + n_arr - n_drop;
        next_id += (uint32_t)n_arr;

        if (FP) {
            __syncthreads();                              // buckets complete
            // buckets -> L_g(k+h), long horizons: 2^seg_log2 lanes per worker, each with a stretch of offsets.  (The envelope
            // by a thread per offset over the workers, behind one more barrier, instead of shared-memory maxima: H = 80, four
            // steps, 1,036 of G = 8, W = 512: 71.8 us, 66.1 this way; 2,072 of G = 16: 167.6, 157.8; one cluster of G = 8 11.4, 11.2)
            if (NC == 0) {
                const int SEG = 1 << a.seg_log2, SL = (H1 + SEG - 1) >> a.seg_log2;
#pragma unroll 1
                for (int i0 = warp << 5; i0 < (G << a.seg_log2); i0 += NT) {
                    const int g = (i0 + lane) >> a.seg_log2, sg = lane & (SEG - 1);
                    const int h0 = sg * SL, h1 = g < G ? min(h0 + SL, H1) : h0;
                    int T = 0, C = 0;
#pragma unroll 2
                    for (int h = h0; h < h1; ++h) { T += Lh[g * HS + h]; C += Ch[g * HS + h]; }
                    int Ti = T, Ci = C;
#pragma unroll 1
                    for (int o = 1; o < SEG; o <<= 1) {
                        const int t = __shfl_down_sync(kFull, Ti, o), c = __shfl_down_sync(kFull, Ci, o);
                        if (sg + o < SEG) { Ti += t; Ci += c; }
                    }
                    Ti -= T; Ci -= C;                                       // the stretches above this one
#pragma unroll 2
                    for (int h = h1 - 1; h >= h0; --h) {
                        Ti += Lh[g * HS + h]; Ci += Ch[g * HS + h];
                        const int x = Ti + h * Ci;
                        Lh[g * HS + h] = x;
                        atomicMax(&Ms[h], x);                               // envelope M_h
                    }
                }
                __syncthreads();
            }
        } else {
            __syncthreads();
        }
        if (timing) t_phase[2] = (unsigned)clock64();

        // ---- requests running before this step that end at it: by warps 1.. while warp 0 routes ----
        if ((warp > 0 || nwarps == 1) && a.pred_mode != 1 && !EARLY) {
            const int t0 = nwarps == 1 ? tid : tid - 32, nt = nwarps == 1 ? NT : NT - 32;
            if (a.term_mode == 1) {
#pragma unroll 1
                for (int g = t0; g < G; g += nt) {
                    draw_ending(t_term, B, OW, (uint32_t)k, (uint32_t)g, key0, key1, fin + (size_t)g * OW);
                    unsigned sub = 0u;
#pragma unroll 1
                    for (int x = 0; x < OW; ++x) {
                        unsigned long long e = occ0[g * OW + x] & fin[g * OW + x];
                        endm[g * OW + x] = e;
#pragma unroll 1
                        for (; e; e &= e - 1ull) {
                            const int sa = g * B + 64 * x + __ffsll((long long)e) - 1;
                            sub += (unsigned)(g_base[sa] + k);
                            g_base[sa] = kEmpty;
                        }
                    }
                    sub_load[g] = sub;
                }
            } else if (a.term_mode >= 2) {
                // quads in order: the rows that a warp reads lie side by side
                const int A4 = A >> 2, B4 = B >> 2;
#pragma unroll 1
                for (int q = t0; q < A4; q += nt) {
                    const int g = (int)((unsigned)q / (unsigned)B4), slot = 4 * (q - g * B4);
                    const unsigned ob = (unsigned)(occ0[g * OW + (slot >> 6)] >> (slot & 63)) & 0xFu;
                    unsigned fb = 0u;
                    if (life) {
                        // a request ends with its o_i-th step: act_end == k
                        const int4 e = *vec_at<const int4>(g_end, 4 * q);
                        fb = (e.x == k ? 1u : 0u) | (e.y == k ? 2u : 0u) | (e.z == k ? 4u : 0u) | (e.w == k ? 8u : 0u);
                    } else if (ob) {
                        // Bernoulli(term_probs[slot][0]): 24-bit uniform below the probability
                        float p4[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) p4[j] = probs[(size_t)(4 * q + j) * H];
                        const uint4 r = philox_call((uint32_t)k, (uint32_t)q, kStreamTerm, key0, key1);
                        const uint32_t rr[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (__fmul_rn((float)(rr[j] >> 8), 5.9604644775390625e-8f) < p4[j]) fb |= 1u << j;
                    }
                    fb &= ob;
                    if (fb) {
                        atomicOr(&endm32[2 * g * OW + (slot >> 5)], fb << (slot & 31));
#pragma unroll 1
                        for (; fb; fb &= fb - 1u) {
                            const int sa = 4 * q + __ffs(fb) - 1;
                            atomicAdd(&sub_load[g], (unsigned)(g_base[sa] + k));
                            g_base[sa] = kEmpty;
                        }
                    }
                }
            }
        }

        if (warp == 0) {
            // ================= ROUTE (warp 0 only, warp-synchronous) =================
            // lane owns workers lane and lane + 32: the selection keys free slots, L_g(k) and min_h m_{g,h}.
            // Eq. 2 keeps the margins m_{g,h} = M_h - L_g(k+h) themselves in shared memory, a row per worker: an
            // admission takes Delta from one row, and only one beyond the worker's smallest margin lifts the
            // envelope, and with it every row.
            int cap[GW], L0[GW], mm[GW];
#pragma unroll
            for (int w = 0; w < GW; ++w) {
                const int g = lane + 32 * w;
                cap[w] = g < G ? cap_s[g] : -1;
                L0[w] = g < G ? (NC == 0 ? Lh[g * HS] : L0_s[g]) : 0;
                mm[w] = 0;
            }
            // rows of all workers: Ms - row (FIRST, long horizons: loads become margins) or Ms + row (the envelope grew by
            // Ms), and their minima
            auto rows = [&](const bool first) {
                if (NC == 0 && G <= 16) {
                    // long rows, few workers: 32 / G lanes share a row
                    const int q = a.lpw_log2, g = lane >> q;
                    int x = 0x7FFFFFFF;
                    if (g < G) {
#pragma unroll 2
                        for (int h = 4 * (lane & ((1 << q) - 1)); h < H1; h += 4 << q) {
                            const int4 e = *vec_at<const int4>(Ms, h);
                            int4 l = *vec_at<const int4>(Lh, g * HS + h);
                            if (first) { l.x = -l.x; l.y = -l.y; l.z = -l.z; l.w = -l.w; }
                            l.x += e.x; l.y += e.y; l.z += e.z; l.w += e.w;
                            *vec_at<int4>(Lh, g * HS + h) = l;
                            x = min(min(x, l.x), min(min(l.y, l.z), l.w));
                        }
                    }
#pragma unroll 1
                    for (int o = 1; o < (1 << q); o <<= 1) x = min(x, __shfl_xor_sync(kFull, x, o));
                    mm[0] = __shfl_sync(kFull, x, (lane << q) & 31);
                } else {
#pragma unroll
                    for (int w = 0; w < GW; ++w) {
                        const int g = lane + 32 * w;
                        int x = 0x7FFFFFFF;
                        if (g < G) {
#pragma unroll
                            for (int h = 0; h < (NC > 0 ? HT : H1); h += 4) {
                                const int4 e = *vec_at<const int4>(Ms, h);
                                int4 l = *vec_at<const int4>(Lh, g * HS + h);
                                if (first) { l.x = -l.x; l.y = -l.y; l.z = -l.z; l.w = -l.w; }
                                l.x += e.x; l.y += e.y; l.z += e.z; l.w += e.w;
                                *vec_at<int4>(Lh, g * HS + h) = l;
                                x = min(min(x, l.x), min(min(l.y, l.z), l.w));
                            }
                        }
                        mm[w] = x;
                    }
                }
                __syncwarp();
            };
            if (FP && NC > 0) {
                // buckets -> L_g(k+h) by suffix sums in registers, envelope M_h by warp maxima, margins to shared memory
                // (with a phase of all warps for the sums, and the envelope by shared-memory maxima, 2,300 to 3,200 cycles
                // a step in batches, 2,000 to 2,300 this way)
                int l[GW][HT > 0 ? HT : 1];
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    const int g = lane + 32 * w;
#pragma unroll
                    for (int h = 0; h < HT; ++h) l[w][h] = 0;
                    if (g < G) {
                        if (H > 0) {
                            int cn[HT > 0 ? HT : 1];
#pragma unroll
                            for (int h = 0; h < HT; h += 4) {
                                const int4 t = *vec_at<const int4>(Lh, g * HS + h), c = *vec_at<const int4>(Ch, g * HS + h);
                                l[w][h] = t.x; l[w][h + 1] = t.y; l[w][h + 2] = t.z; l[w][h + 3] = t.w;
                                cn[h] = c.x; cn[h + 1] = c.y; cn[h + 2] = c.z; cn[h + 3] = c.w;
                            }
#pragma unroll
                            for (int h = HT - 2; h >= 0; --h) { l[w][h] += l[w][h + 1]; cn[h] += cn[h + 1]; }
#pragma unroll
                            for (int h = 0; h < HT; ++h) l[w][h] += h * cn[h];
                            L0[w] = l[w][0];
                        } else {
                            l[w][0] = L0[w];
                        }
                        mm[w] = 0x7FFFFFFF;
                    }
                }
#pragma unroll
                for (int h = 0; h < HT; ++h) {
                    int e = l[0][h];
#pragma unroll
                    for (int w = 1; w < GW; ++w) e = max(e, l[w][h]);
                    e = __reduce_max_sync(kFull, e);                    // (lanes without a worker hold zero)
#pragma unroll
                    for (int w = 0; w < GW; ++w) {
                        l[w][h] = h < H1 ? e - l[w][h] : 0x7FFFFFFF;
                        mm[w] = min(mm[w], l[w][h]);
                    }
                }
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    const int g = lane + 32 * w;
                    if (g < G) {
#pragma unroll
                        for (int h = 0; h < HT; h += 4) *vec_at<int4>(Lh, g * HS + h) = make_int4(l[w][h], l[w][h + 1], l[w][h + 2], l[w][h + 3]);
                    }
                }
                __syncwarp();
                if (lane < HS) Ms[lane] = 0;
            } else if (FP) {
                __syncwarp();                          // every lane has read L_g(k) before rows become margins
                rows(true);
#pragma unroll
                for (int c = 0; c < HC; ++c) if (lane + 32 * c < HS) Ms[lane + 32 * c] = 0;
            } else {
                int v = L0[0];
#pragma unroll
                for (int w = 1; w < GW; ++w) v = max(v, L0[w]);
                const int M0 = __reduce_max_sync(kFull, v);
#pragma unroll
                for (int w = 0; w < GW; ++w) mm[w] = M0 - L0[w];
            }

            Scorer<FP> sc;
            sc.md = Lh; sc.dn = dn_s; sc.H = H; sc.G = G; sc.aD = a.aD; sc.beta = a.beta; sc.mm = 0;
            // the score at the sites of the loop: unrolled for short horizons, else the next four offsets are read while
            // these are added
            auto hot_key = [&](int delta) -> long long {
                if (!FP) return sc.key(delta);
                double pen = 0.0;
                if (NC > 0) {
                    int4 q[NC > 0 ? NC : 1];
#pragma unroll
                    for (int c = 0; c < NC; ++c) q[c] = *vec_at<const int4>(sc.md, 4 * c);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const int mj[4] = {q[c].x, q[c].y, q[c].z, q[c].w};
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            pen = __dadd_rn(pen, __fma_rn(__hiloint2double(0x43300000, max(delta - mj[j], 0)), a.dn[2 * (4 * c + j)], a.dn[2 * (4 * c + j) + 1]));
                    }
                } else {
                    int4 q = *vec_at<const int4>(sc.md, 0);
                    double2 d[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) d[j] = *vec_at<const double2>(dn_s, 2 * j);
#pragma unroll 2
                    for (int h = 0; h <= H; h += 4) {
                        const int mj[4] = {q.x, q.y, q.z, q.w};
                        const double2 e[4] = {d[0], d[1], d[2], d[3]};
                        q = *vec_at<const int4>(sc.md, h + 4);
#pragma unroll
                        for (int j = 0; j < 4; ++j) d[j] = *vec_at<const double2>(dn_s, 2 * (h + 4 + j));
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            pen = __dadd_rn(pen, __fma_rn(__hiloint2double(0x43300000, max(delta - mj[j], 0)), e[j].x, e[j].y));
                    }
                }
                const double dl = __dsub_rn(__hiloint2double(0x43300000, delta), 4503599627370496.0);
                return key_of_double(__dsub_rn(__dmul_rn(a.aD, dl), __dmul_rn(a.beta, pen)));
            };
            // Eq. 2 with the terms summed across the lanes: off the exact score by at most rel_err * delta + fix_err
            double w[HC];                                                   // discounts d_h of the lane's offsets
            int iw[HC];                                                     // ... in fixed point
#pragma unroll
            for (int c = 0; c < HC; ++c) {
                w[c] = FP && lane + 32 * c < H1 ? dn_s[2 * (lane + 32 * c)] : 0.0;
                iw[c] = FP && lane + 32 * c < H1 ? iw_s[lane + 32 * c] : 0;
            }
            int m[HC];                                                      // margins of the selected worker, by offset
            auto near_score = [&](int delta) -> double {
                double p = 0.0;
#pragma unroll
                for (int c = 0; c < HC; ++c) {
                    const double x = __dsub_rn(__hiloint2double(0x43300000, max(delta - m[c], 0)), 4503599627370496.0);
                    p = __fma_rn(x, w[c], p);
                }
                // 32 lanes, each rounded to 1 / fix: the sum fits 32 bits and is off by less than 32 / fix
                const unsigned q = __reduce_add_sync(kFull, __double2uint_rn(__dmul_rn(p, a.fix)));
                return __fma_rn(a.aD, (double)delta, -__dmul_rn(a.beta_fix, (double)q));
            };

            // optional F-score matrix before the first admission
            if (rare(a.out.fscore != nullptr)) {
                double *F = a.out.fscore + orow * (size_t)W * G;
#pragma unroll 1
                for (int g = 0; g < G; ++g) {
                    const int own = (GW > 1 && g >= 32) ? mm[GW - 1] : mm[0];
                    sc.mm = __shfl_sync(kFull, own, g & 31);
                    if (FP) sc.md = Lh + g * HS;
                    score_column<FP, NC>(sc, F + g, q_key, n_w, W, G, WL, lane);
                }
            }

            int S_tot = 0;
#pragma unroll
            for (int w = 0; w < GW; ++w) S_tot += cap[w] > 0 ? cap[w] : 0;
            S_tot = (int)__reduce_add_sync(kFull, (unsigned)S_tot);
            int n_left = n_w, s1_iters = 0, s2_pops = 0, status = 0, first_rm = W;
            const int n_groups = (n_w + 127) >> 7;
            // Stage-2 window: the R_max largest waiting keys, in registers of every lane, kept across the pops of
            // the step.  The largest of the rest are in lists of four per lane, sorted; an admitted entry is
            // replaced by the largest head.  A lane whose list runs dry although it may hold more keys shows kListEnd,
            // and when that is the largest head everything is built anew.
            int win[kRegWin], t0 = 0, t1 = 0, t2 = 0, t3 = 0, t_end = 0;
#pragma unroll
            for (int r = 0; r < kRegWin; ++r) win[r] = 0;
            bool valid = false;
            bool to_stage2 = true;

#pragma unroll 1
            while (n_left > 0 && S_tot > 0) {
                const bool st1 = S_tot > a.S_greedy;
                if (rare(!st1 && timing && to_stage2)) { to_stage2 = false; t_phase[3] = (unsigned)clock64(); }
                if (rare(st1 ? s1_iters >= W : s2_pops >= W + G)) { status |= BR_ST_ITER_CAP; break; }
                // most free slots; then Stage 1: smallest L_g(k), Stage 2: largest horizon-min margin; lowest g
                int bc = cap[0];
#pragma unroll
                for (int w = 1; w < GW; ++w) bc = max(bc, cap[w]);
                const int mc = __reduce_max_sync(kFull, bc);
                if (rare(mc <= 0)) break;
                int bv = kEmpty;
#pragma unroll
                for (int w = 0; w < GW; ++w) bv = max(bv, cap[w] == mc ? (st1 ? ~L0[w] : mm[w]) : kEmpty);
                const int mv = __reduce_max_sync(kFull, bv);
                int gi = 0xFF;
#pragma unroll
                for (int w = GW - 1; w >= 0; --w) gi = cap[w] == mc && (st1 ? ~L0[w] : mm[w]) == mv ? lane + 32 * w : gi;
                const int g = (int)__reduce_min_sync(kFull, (unsigned)gi);
                sc.mm = st1 ? __shfl_sync(kFull, (GW > 1 && g >= 32) ? mm[GW - 1] : mm[0], g & 31) : mv;
                if (FP) sc.md = Lh + g * HS;
#pragma unroll
                for (int c = 0; c < HC; ++c) m[c] = FP ? (lane + 32 * c < HS ? Lh[g * HS + lane + 32 * c] : 0x7FFFFFFF) : sc.mm;

                unsigned chosen = 1u;                    // window entries to admit
                int dsum = 0, wkey = 0;
                bool single = st1;
                if (st1) {
                    ++s1_iters;
                } else {
                    ++s2_pops;
                    long long wk = kNoKey;
                    // window: the R_max largest waiting requests, earliest first on ties
                    const int R = min(a.R_max, n_left), lim = min(mc, R);
                    if (rare(a.big_window != 0)) {
                        wkey = largest_keys(q_key, n_w, R, lane);
                        const WindowChoice c = big_window<FP>(sc, bw_keys, bw_off, bw_win, wkey, R, lim, WL, FP ? m[0] : 0, lane);
                        wk = c.wk; chosen = c.chosen; dsum = c.dsum;
                    } else {
                        bool none = false;
                        if (NC == 0) {
                            // The score is concave and zero at zero, so F(Delta) <= Delta / s F(s) for Delta >= s: if F(s) is
                            // negative beyond rounding for an s that no window entry is below, every subset's score is, and
                            // the starvation guard is next.  Before the window is built, the R-th largest of the lanes'
                            // maxima is such an s, and much cheaper than the window.
                            int x = 0;
                            if (valid) {
#pragma unroll
                                for (int r = 0; r < kRegWin; ++r) x = r < R ? win[r] : x;
                            } else {
                                int x0 = 0;
#pragma unroll 2
                                for (int t = 0; t < n_groups; ++t) {
                                    const int4 kk = *vec_at<const int4>(q_key, (t * 32 + lane) * 4);
                                    x0 = max(max(x0, max(kk.x, kk.y)), max(kk.z, kk.w));
                                }
#pragma unroll 1
                                for (int r = 0; r < R; ++r) { x = __reduce_max_sync(kFull, x0); x0 = x0 == x ? 0 : x0; }
                            }
                            none = near_score(x >> WL) < -__fma_rn(a.rel_err, (double)(x >> WL), a.fix_err);
                        }
                        if ((NC > 0 || !none) && !valid) {
                            t0 = t1 = t2 = t3 = 0;
#pragma unroll 2
                            for (int t = 0; t < n_groups; ++t) {
                                // a lane reads every 32nd position (long-waiting requests gather at the front of the
                                // queue), sorts its four keys and merges them into its list
                                int x0 = q_key[t * 128 + lane], x1 = q_key[t * 128 + 32 + lane];
                                int x2 = q_key[t * 128 + 64 + lane], x3 = q_key[t * 128 + 96 + lane];
                                order2(x0, x1); order2(x2, x3); order2(x0, x2); order2(x1, x3); order2(x1, x2);
                                t0 = max(t0, x3); t1 = max(t1, x2); t2 = max(t2, x1); t3 = max(t3, x0);
                                order2(t0, t2); order2(t1, t3); order2(t0, t1); order2(t2, t3);
                            }
                            t_end = t3 > 0 && n_groups > 1 ? kListEnd : 0;    // one group: four keys per lane
                            valid = true;
#pragma unroll
                            for (int r = 0; r < kRegWin; ++r) {
                                win[r] = 0;
                                if (r < a.R_max) {
                                    const int x = __reduce_max_sync(kFull, t0);
                                    win[r] = x;
                                    if (t0 == x) { t0 = t1; t1 = t2; t2 = t3; t3 = t_end; }
                                    valid = valid && x != kListEnd;
                                }
                            }
                            if (rare(!valid)) {
                                // one lane holds more of the window than its list
                                wkey = largest_keys(q_key, n_w, R, lane);
#pragma unroll
                                for (int r = 0; r < kRegWin; ++r) win[r] = __shfl_sync(kFull, wkey, r);
                            }
                        }
                        if (NC == 0 && none) {
                            wk = -1;
                        } else {
                            // subsets of the window: lane = mask, lowest mask on ties
                            int delta = 0;
#pragma unroll
                            for (int r = 0; r < kRegWin; ++r) delta += (lane >> r) & 1 ? win[r] >> WL : 0;
                            const bool cand = lane >= 1 && lane < (1 << R) && __popc(lane) <= lim;
                            const int dmax = __reduce_max_sync(kFull, cand ? delta : 0);
                            bool best = delta == dmax;
                            wk = dmax > 0 ? (long long)dmax : kNoKey;   // safe at every offset: the score alpha D Delta grows with Delta
                            if (dmax > sc.mm) {
                                if (!FP) {                          // Eq. 1 scores fit 32 bits
                                    const int fs = cand ? (int)sc.key(delta) : kEmpty;
                                    const int mf = __reduce_max_sync(kFull, fs);
                                    wk = mf;
                                    best = fs == mf;
                                } else {
                                    best = warp_max64(cand ? hot_key(delta) : kNoKey, wk);
                                }
                            }
                            chosen = __reduce_min_sync(kFull, cand && best ? (unsigned)lane : 32u);
                            dsum = 0;
#pragma unroll
                            for (int r = 0; r < kRegWin; ++r) dsum += (chosen >> r) & 1u ? win[r] >> WL : 0;
                        }
                    }
                    if (rare(wk == kNoKey)) { status |= BR_ST_ITER_CAP; break; }
                    single = wk <= 0;                           // starvation guard
                }

                int qk = 0;
                if (single) {
                    // argmax_i F_g({i}) over all waiting requests, earliest arrival on ties.
                    // The score is concave and piecewise linear in s (Eq. 2: kinks at the m_{g,h}): it rises up to
                    // s* = the smallest kink at which the slope alpha D - beta sum_{m_h <= kink} d_h is no longer
                    // positive (Eq. 1: the margin) and falls after it.  If no slope is within rounding distance of zero,
                    // the scores of integer lengths are strictly ordered on either side, and the arg-max is the
                    // largest s <= s* or the smallest s > s*: one pass of two integer minima over the queue.
                    int peak = sc.mm;
                    bool ordered = a.peak_ok != 0;
                    if (FP) {
                        if (NC > 0) {
                            int4 q[NC > 0 ? NC : 1];
                            int ws[HC];
#pragma unroll
                            for (int c = 0; c < HC; ++c) ws[c] = 0;
#pragma unroll
                            for (int c = 0; c < NC; ++c) q[c] = *vec_at<const int4>(sc.md, 4 * c);
#pragma unroll
                            for (int c = 0; c < NC; ++c) {
                                const int mj[4] = {q[c].x, q[c].y, q[c].z, q[c].w};
#pragma unroll
                                for (int j = 0; j < 4; ++j) ws[0] += mj[j] <= m[0] ? a.iw[4 * c + j] : 0;
                            }
                            peak = 0x7FFFFFFF;
                            bool flat = false;
                            if (lane < H1) {
                                flat = flat || (ws[0] > a.w_below && ws[0] < a.w_above);
                                if (ws[0] > a.w_below) peak = min(peak, m[0]);
                            }
                            peak = __reduce_min_sync(kFull, flat ? -1 : peak);
                        } else {
                            // Bisection over the kinks: the score still rises at lo, no more at hi.  The next kink to look
                            // at is the last one in the lower half of the lengths between them, or the first after.
                            int lo = -1, hi = -1;
#pragma unroll
                            for (int c = 0; c < HC; ++c) hi = max(hi, lane + 32 * c < H1 ? m[c] : -1);
                            hi = __reduce_max_sync(kFull, hi);
                            int pv = hi;                         // the last kink first: the score may rise throughout
                            peak = 0x7FFFFFFF;
#pragma unroll 1
                            while (true) {
                                unsigned ws = 0;
#pragma unroll
                                for (int c = 0; c < HC; ++c) ws += m[c] <= pv ? (unsigned)iw[c] : 0u;
                                ws = __reduce_add_sync(kFull, ws);
                                if ((int)ws > a.w_below) {
                                    peak = (int)ws < a.w_above ? -1 : pv;
                                    if (peak < 0) break;
                                    hi = pv;
                                } else {
                                    lo = pv;
                                    if (lo == hi) break;                         // rises throughout
                                }
                                const int mid = lo + ((hi - lo) >> 1);
                                int b = -1;
#pragma unroll
                                for (int c = 0; c < HC; ++c) b = max(b, lane + 32 * c < H1 && m[c] <= mid ? m[c] : -1);
                                pv = __reduce_max_sync(kFull, b);
                                if (pv <= lo) {
                                    b = 0x7FFFFFFF;
#pragma unroll
                                    for (int c = 0; c < HC; ++c) b = min(b, lane + 32 * c < H1 && m[c] > mid ? m[c] : 0x7FFFFFFF);
                                    pv = __reduce_min_sync(kFull, b);
                                    if (pv >= hi) break;                         // no kink between them
                                }
                            }
                        }
                        ordered = peak >= 0;
                    }
                    if (ordered) {
                        const int thr = peak >= (1 << (31 - WL)) ? 0x7FFFFFFF : ((peak << WL) | (int)posmask);
                        // entries that are gone or beyond the queue have negative keys: as unsigned distances they lie
                        // beyond every waiting one on the side that is searched.  A waiting one on the other side
                        // lies beyond them, and is what comes out where there is no other
                        unsigned below = 0xFFFFFFFFu, above = 0xFFFFFFFFu;
#pragma unroll 2
                        for (int t = 0; t < n_groups; ++t) {
                            const int4 kk = *vec_at<const int4>(q_key, (t * 32 + lane) * 4);
                            const unsigned ke[4] = {(unsigned)kk.x, (unsigned)kk.y, (unsigned)kk.z, (unsigned)kk.w};
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                below = min(below, (unsigned)thr - ke[j]);
                                above = min(above, (ke[j] ^ posmask) - ((unsigned)thr + 1u));
                            }
                        }
                        below = __reduce_min_sync(kFull, below);
                        above = __reduce_min_sync(kFull, above);
                        const int kl = (int)((unsigned)thr - below), ka = kl > 0 && kl <= thr ? kl : 0;
                        const int kx = (int)(above + (unsigned)thr + 1u);
                        const int kb = kx > thr ? (int)((unsigned)kx ^ posmask) : 0;
                        qk = ka | kb;
                        if (ka != 0 && kb != 0) {
                            bool take_a = false, clear = false;
                            if (FP && NC == 0) {
                                const double df = __dsub_rn(near_score(ka >> WL), near_score(kb >> WL));
                                clear = fabs(df) > __fma_rn(a.rel_err, (double)(ka >> WL) + (double)(kb >> WL), __dadd_rn(a.fix_err, a.fix_err));
                                take_a = df > 0.0;
                            }
                            if (!clear) {
                                const long long f = hot_key(((lane & 1) ? kb : ka) >> WL);
                                const long long fa = __shfl_sync(kFull, f, 0), fb = __shfl_sync(kFull, f, 1);
                                take_a = fa > fb || (fa == fb && ((unsigned)ka & posmask) > ((unsigned)kb & posmask));
                            }
                            qk = take_a ? ka : kb;
                        }
                    } else {
                        qk = best_of_all<FP>(sc, q_key, n_w, WL, posmask, lane);      // a flat segment
                    }
                    if (rare(qk <= 0)) break;
                    chosen = 1u;
                    dsum = qk >> WL;
                }

                // ---- admissions to worker g; slots are given out after routing ----
                const int n_adm = single ? 1 : __popc(chosen);
                {
                    int key = single ? qk : wkey;                // lane r: the request of bit r
                    if (!single && a.big_window == 0) {
                        key = win[0];
#pragma unroll
                        for (int x = 1; x < kRegWin; ++x) key = lane == x ? win[x] : key;
                    }
                    const int at = __popc(chosen & ((1u << lane) - 1u)), pos = (int)(posmask - ((unsigned)key & posmask));
                    if ((chosen >> lane) & 1u) {
                        adm[n_w - n_left + at] = ((unsigned)pos << 15) | ((unsigned)g << 9) | (unsigned)(mc - at);
                        q_key[pos] = key | (int)0x80000000u;
                        first_rm = min(first_rm, pos);
                    }
                }
                // the admitted requests leave the window, where the largest head moves up, or a lane's list
                unsigned out = chosen;
                if (single) {
                    out = 0u;
#pragma unroll
                    for (int x = 0; x < kRegWin; ++x) out |= win[x] == qk ? 1u << x : 0u;
                    const bool h0 = t0 == qk, h1 = h0 || t1 == qk, h2 = h1 || t2 == qk, h3 = h2 || t3 == qk;
                    t0 = h0 ? t1 : t0; t1 = h1 ? t2 : t1; t2 = h2 ? t3 : t2; t3 = h3 ? t_end : t3;
                }
                if (a.big_window == 0) {
#pragma unroll 1
                    while (out) {
                        const unsigned low = out & (0u - out);
                        const int x = __reduce_max_sync(kFull, t0);
#pragma unroll
                        for (int y = 0; y < kRegWin; ++y) {
                            win[y] = (1u << y) >= low && y + 1 < kRegWin ? win[y + 1 < kRegWin ? y + 1 : y] : win[y];
                            win[y] = y == a.R_max - 1 ? x : win[y];
                        }
                        if (t0 == x) { t0 = t1; t1 = t2; t2 = t3; t3 = t_end; }
                        valid = valid && x != kListEnd;
                        out = (out ^ low) >> 1;
                    }
                }
                // worker g grew by dsum at every offset; beyond its smallest margin it lifts the envelope
                const int up0 = dsum - sc.mm;
                if (FP) {
#pragma unroll
                    for (int c = 0; c < HC; ++c)
                        if (lane + 32 * c < H1) Lh[g * HS + lane + 32 * c] = m[c] - dsum;
                }
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    const bool it_is = g == lane + 32 * w;
                    cap[w] -= it_is ? n_adm : 0;
                    L0[w] += it_is ? dsum : 0;
                    mm[w] -= it_is ? dsum : 0;
                }
                if (up0 > 0) {
                    if (FP) {
#pragma unroll
                        for (int c = 0; c < HC; ++c)
                            if (lane + 32 * c < H1) Ms[lane + 32 * c] = max(dsum - m[c], 0);
                        __syncwarp();
                        rows(false);
                    } else {
#pragma unroll
                        for (int w = 0; w < GW; ++w) mm[w] += up0;
                    }
                }
                __syncwarp();
                S_tot -= n_adm; n_left -= n_adm;
            }
            if (timing) { t_phase[4] = (unsigned)clock64(); if (to_stage2) t_phase[3] = t_phase[4]; }

            // ================= RECORD =================
            {
                int mx = kEmpty, mn = 0x7FFFFFFF;
                long long sum = 0;
                const auto o_load = mk_span(reinterpret_cast<long long *>(a.out.load) + orow * G, G);
#pragma unroll
                for (int w = 0; w < GW; ++w) {
                    const int g = lane + 32 * w;
                    if (g < G) {
                        mx = max(mx, L0[w]); mn = min(mn, L0[w]); sum += L0[w];
                        o_load[g] = L0[w];
                        L0_s[g] = L0[w];
                    }
                }
                mx = __reduce_max_sync(kFull, mx);
                mn = __reduce_min_sync(kFull, mn);
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
                status = (int)__reduce_or_sync(kFull, (unsigned)status);
                const int fr = __reduce_min_sync(kFull, first_rm);
                if (lane == 0) {
                    const auto tr = mk_span(reinterpret_cast<long long *>(a.out.trace) + orow * 3, 3);
                    tr[0] = mx; tr[1] = mn; tr[2] = sum;
                    scal[0] = n_left; scal[1] = n_w - n_left; scal[2] = s1_iters; scal[3] = s2_pops;
                    scal[4] = status | (n_drop ? BR_ST_QUEUE_OVERFLOW : 0);
                    scal[6] = fr;
                }
            }
        }
        __syncthreads();                                          // admissions visible
        if (EARLY) {
#pragma unroll
            for (int w = 0; w < GW; ++w) {
                const int g = lane + 32 * w;
                if (pslot[w] >= 0) {
                    unsigned sub = (unsigned)(pend[w] + k);
                    g_base[g * B + pslot[w]] = kEmpty;
#pragma unroll 1
                    for (int x = pslot[w] >> 6; x < OW; ++x) {            // rare: more than one
                        unsigned long long e = endm[g * OW + x];
                        if (x == pslot[w] >> 6) e &= ~(1ull << (pslot[w] & 63));
#pragma unroll 1
                        for (; e; e &= e - 1ull) {
                            const int sa = g * B + 64 * x + __ffsll((long long)e) - 1;
                            sub += (unsigned)(g_base[sa] + k);
                            g_base[sa] = kEmpty;
                        }
                    }
                    sub_load[g] = sub;
                }
            }
            __syncwarp();
        }

        // ============ sticky admissions, one thread each ============
        // a worker's requests take its free slots in ascending order, in the order of their admission
        const int n_new = scal[0], n_adm = n_w - n_new;
#pragma unroll 1
        for (int e = tid; e < n_adm; e += NT) {
            const unsigned r = adm[e];
            const int g = (int)(r >> 9) & 63, pos = (int)(r >> 15), s = (q_key[pos] & 0x7FFFFFFF) >> WL;
            int rank = cap_s[g] - (int)(r & 511u), slot = B;
#pragma unroll 1
            for (int x = 0; x < 2 * OW; ++x) {
                unsigned fr = ~occ032[2 * g * OW + x];
                const int c = __popc(fr);
                if (rank < c) {
#pragma unroll 1
                    for (; rank > 0; --rank) fr &= fr - 1u;
                    slot = 32 * x + __ffs(fr) - 1;
                    break;
                }
                rank -= c;
            }
            if (slot >= B) {                                      // free-slot count and occupancy word disagree: gone, no slot
                atomicOr(&scal[4], BR_ST_BAD_STATE);
                q_key[pos] = kQBeyond;
                continue;
            }
            const int sa = g * B + slot;
            q_key[pos] = (int)(0x80000000u | (unsigned)sa);
            atomicOr(&occ32[2 * g * OW + (slot >> 5)], 1u << (slot & 31));
            const int o = life ? q_o[pos] : 0;
            if (H > 0 && g_chat0) {
                g_chat0[sa] = (float)(H + a.delta_T - 1);
                g_kref[sa] = (uint8_t)((k + 1 - a.delta_T) & 255);
            }
            if (life) g_end[sa] = k + o - 1;                      // runs at steps k .. k + o_i - 1
            if (g_aid) g_aid[sa] = q_id[pos];
            // it may also end at this very step
            bool ends = false;
            if (a.term_mode == 1) {
                ends = (fin[g * OW + (slot >> 6)] >> (slot & 63)) & 1ull;
            } else if (a.term_mode == 2) {
                const uint4 w = philox_call((uint32_t)k, (uint32_t)sa >> 2, kStreamTerm, key0, key1);
                ends = __fmul_rn((float)(word_of(w, sa & 3) >> 8), 5.9604644775390625e-8f) < probs[(size_t)sa * H];
            } else if (life) {
                ends = o == 1;
            }
            g_base[sa] = ends ? kEmpty : s - k;
            if (ends) {
                atomicOr(&endm32[2 * g * OW + (slot >> 5)], 1u << (slot & 31));
                atomicAdd(&sub_load[g], (unsigned)s);
            }
        }
        if (n_adm > 0) __syncthreads();

        // ============ queue compaction and assignments ============
        // A thread owns four consecutive positions of every stretch of 4 NT; an entry's new position is
        // the count of kept entries before it.  A moved entry gains the distance in its key's position field.
        const int first_rm = scal[6];
        {
            const auto assign = mk_span(a.assign_out + orow * W, W);
            int run = 0, par = 0;
#pragma unroll 1
            for (int i0 = 0; i0 < W; i0 += 4 * NT) {
                const int p0 = i0 + 4 * tid;
                if (first_rm >= min(i0 + 4 * NT, n_w)) {                       // (or beyond the queue)
                    if (p0 < W) *vec_at<int4>(assign, p0) = make_int4(-1, -1, -1, -1);
                    run += 4 * NT;                                // (beyond the queue the count is not used)
                    continue;
                }
                int4 kk = make_int4(kQBeyond, kQBeyond, kQBeyond, kQBeyond), oo = make_int4(0, 0, 0, 0);
                uint4 ii = make_uint4(0u, 0u, 0u, 0u);
                if (p0 < W) {
                    kk = *vec_at<const int4>(q_key, p0);
                    ii = *vec_at<const uint4>(q_id, p0);
                    if (life) oo = *vec_at<const int4>(q_o, p0);
                }
                const int ke[4] = {kk.x, kk.y, kk.z, kk.w};
                const unsigned idv[4] = {ii.x, ii.y, ii.z, ii.w};
                const int ov[4] = {oo.x, oo.y, oo.z, oo.w};
                int before = 0, kept = 0;                         // within the warp's 128 positions
                const unsigned lt = (1u << lane) - 1u;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const unsigned b = __ballot_sync(kFull, ke[j] > 0);
                    before += __popc(b & lt);
                    kept += __popc(b);
                }
                if (lane == 0) scal[16 + par + warp] = kept;
                int as[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int sa = ke[j] & 0x7FFFFFFF;
                    as[j] = ke[j] < 0 && sa < A ? sa : -1;
                }
                if (p0 < W) *vec_at<int4>(assign, p0) = make_int4(as[0], as[1], as[2], as[3]);
                __syncthreads();                                  // the stretch is read before any of it is overwritten
                int below = run + before, total = 0;
#pragma unroll 1
                for (int x = 0; x < nwarps; ++x) {
                    const int t = scal[16 + par + x];
                    if (x < warp) below += t;
                    total += t;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (ke[j] > 0) {
                        const int from = p0 + j;
                        if (below != from) {
                            q_key[below] = ke[j] + (from - below);
                            q_id[below] = idv[j];
                            if (life) q_o[below] = ov[j];
                        }
                        ++below;
                    }
                }
                run += total;
                par ^= 8;
            }
        }
        __syncthreads();
        // entries that moved or are new go back to the caller's rows
#pragma unroll 1
        for (int p0 = (min(first_rm, n_w_old) & ~3) + 4 * tid; p0 < n_new; p0 += 4 * NT) {
            const int4 kk = *vec_at<const int4>(q_key, p0);
            const uint4 ii = *vec_at<const uint4>(q_id, p0);
            const int4 sv = make_int4(kk.x >> WL, kk.y >> WL, kk.z >> WL, kk.w >> WL);
            if (p0 + 4 <= n_new) {
                *vec_at<int4>(g_qs, p0) = sv;
                *vec_at<uint4>(g_qid, p0) = ii;
                if (life) *vec_at<int4>(g_qo, p0) = *vec_at<const int4>(q_o, p0);
            } else {
                const int s4[4] = {sv.x, sv.y, sv.z, sv.w};
                const unsigned i4[4] = {ii.x, ii.y, ii.z, ii.w};
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if (p0 + j < n_new) {
                        g_qs[p0 + j] = s4[j]; g_qid[p0 + j] = i4[j];
                        if (life) g_qo[p0 + j] = q_o[p0 + j];
                    }
            }
        }
#pragma unroll 1
        for (int i = n_new + tid; i < n_w; i += NT) q_key[i] = kQBeyond;        // vacated tail
        n_w = n_new;
        if (timing) t_phase[5] = (unsigned)clock64();

        // ================= ADVANCE =================
        // L_g(k+1) = L_g(k) - (loads of the requests that ended) + (number of survivors)
#pragma unroll 1
        for (int g = tid; g < G; g += NT) {
            int na = 0;
            for (int x = 0; x < OW; ++x) {
                const unsigned long long o = occ[g * OW + x] & ~endm[g * OW + x];
                occ[g * OW + x] = o; occ0[g * OW + x] = o; endm[g * OW + x] = 0ull;
                na += __popcll(o);
            }
            cap_s[g] = B - na;
            L0_s[g] = L0_s[g] - (int)sub_load[g] + na;
            sub_load[g] = 0u;
        }
        // (16 bytes a store: 592 of G = 32, H = 8, four steps, 75.8 us with four, 74.0 this way; 2,072: 211.6, 208.0)
        if (FP && it + 1 < a.n_steps) {
#pragma unroll 1
            for (int i = 4 * tid; i < G * HS; i += 4 * NT) { *vec_at<int4>(Lh, i) = make_int4(0, 0, 0, 0); if (H > 0) *vec_at<int4>(Ch, i) = make_int4(0, 0, 0, 0); }
#pragma unroll 1
            for (int h = tid; h < HS; h += NT) Ms[h] = h < H1 ? 0 : 0x7FFFFFFF;
        }
        if (tid == 0) {
            if (a.out.counters) {
                uint32_t *c = a.out.counters + orow * 4;
                c[0] = (uint32_t)n_drop; c[1] = (uint32_t)scal[1]; c[2] = (uint32_t)scal[2]; c[3] = (uint32_t)scal[3];
            }
            if (a.out.status) a.out.status[orow] = scal[4] | scal[5];
            if (timing) {
                t_phase[6] = (unsigned)clock64();
                uint32_t *pc = a.out.phase_cycles + orow * 8;
#pragma unroll
                for (int p = 0; p < 6; ++p) pc[p] = (uint32_t)(t_phase[p + 1] - t_phase[p]);
                pc[6] = it == 0 ? (uint32_t)(t_phase[0] - t_entry) : 0u;
                pc[7] = 0u;
            }
        }
        __syncthreads();
    }

    // ---- write the snapshot back ----
#pragma unroll 1
    for (int g = tid; g < G; g += NT) {
        a.ws.load[(size_t)inst * G + g] = (long long)L0_s[g];
        a.ws.nact[(size_t)inst * G + g] = B - cap_s[g];
        for (int x = 0; x < OW; ++x) a.ws.occ[((size_t)inst * G + g) * OW + x] = occ[g * OW + x];
    }
    if (tid == 0) {
        a.ws.step[inst] = k;
        a.ws.next_id[inst] = next_id;
        a.wq.n[inst] = n_w;
        if (a.out.phase_cycles)      // time from kernel entry to here, for the last step's row
            a.out.phase_cycles[((size_t)(a.n_steps - 1) * a.N + inst) * 8 + 7] = (uint32_t)((unsigned)clock64() - t_entry);
    }
}

}  // namespace br
