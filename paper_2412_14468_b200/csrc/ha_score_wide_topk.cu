// SCORE + TOPK for signatures of b = 64 .. 512 bits kept as b/64 packed 64-bit integers (the widths of the paper's
// bit-width study and of its table "Latency of SCORE computation"): Eq. 1 with the bitcount(xor) identity of Section
// 4.1 at b bits, s = b - popcount(k xor q), reduced with max over the query heads of a GQA group as in the 32-bit
// layer-step, then the standard top-k of Section 4 with ties towards the lowest token index.  Scores take b + 1
// values, so the selection is again a histogram threshold plus an index-ordered compaction, never a sort.
//
// Sequences of up to 131072 tokens: ONE kernel, a thread-block cluster per (sequence, KV head) unit
// (wide_select_cluster_kernel, second half of this file).  Longer ones: three kernels over chunks of every unit, each at
// full parallelism, nothing waits:
//   1. wide_scan_kernel      streams the signatures, leaves one 16-bit score per token in the workspace and adds the
//                            chunk's level counts to the unit's (b + 1)-level histogram;
//   2. wide_count_kernel     every chunk derives the threshold T (largest level with #{S >= T} >= k) from the unit's
//                            histogram and counts its own tokens above / at T;
//   3. wide_write_kernel     every chunk adds up the counts of the chunks before it and writes its selected tokens at
//                            their final positions (ascending token index; the first r = k - #{S > T} tokens at T).
// Tokens that are always in context (the first n_sink, the most recent n_local) carry the score 0xFFFF, which is
// above every threshold, and are left out of the histogram.
#include <atomic>

#include "ha_score_dev.cuh"

namespace ha {

constexpr int kWideThreads = 256;
constexpr int kWideMaxLevels = 513;            // scores 0 .. 512
constexpr int kWideHistStride = 520;
constexpr int kWideTokensPerThread = 16;
constexpr int kWidePass = kWideThreads * kWideTokensPerThread;   // tokens of one pass of a CTA
constexpr uint32_t kWideForced = 0xFFFFu;
constexpr int kWideMaxChunks = 1024;           // chunks per unit: a single long sequence still fills the device

struct WideArgs {
    const uint64_t *q_codes, *k_codes;
    long long kc_sb, kc_sh;        // in 64-bit words
    const int32_t *seq_lens, *k_per_seq;
    int k_uniform, max_seq_len, k_max, Hq, Hkv, G, n_bits, chunk_tokens;
    Windows win;
    int32_t *idx;
    long long idx_sb, idx_sh;
    int32_t *count, *hist_out;
    int32_t *unit_hist;            // [units][kWideHistStride], zero before the scan
    int32_t *chunk_counts;         // [units][kWideMaxChunks][2]
    uint16_t *scores;              // [units][score_row]
    long long score_row;
};

struct WideUnit {
    int n, keep, keep_rest;
    WindowBounds wbd;
};
__device__ __forceinline__ WideUnit wide_unit(const WideArgs &a, int b) {
    WideUnit r;
    r.n = max(min(a.seq_lens[b], a.max_seq_len), 0);
    const int k = a.k_per_seq ? a.k_per_seq[b] : a.k_uniform;
    r.wbd = window_bounds(a.win, r.n);
    const int nf = forced_before(r.wbd, r.n);
    r.keep_rest = max(0, min(min(k, a.k_max - nf), r.n - nf));
    r.keep = nf + r.keep_rest;
    return r;
}

template <int W>
__global__ void __launch_bounds__(kWideThreads) wide_scan_kernel(const WideArgs a) {
    __shared__ int s_hist[kWideThreads / 32][kWideMaxLevels + 7];   // one table per warp
    __shared__ unsigned long long s_q[kMaxGroup][W];
    const int chunk = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, warp = tid >> 5;
    const WideUnit wu = wide_unit(a, b);
    const int start = chunk * a.chunk_tokens;
    if (start >= wu.n) return;
    const int end = min(wu.n, start + a.chunk_tokens);
    const int levels = a.n_bits + 1;
    for (int i = tid; i < (kWideThreads / 32) * (kWideMaxLevels + 7); i += kWideThreads) (&s_hist[0][0])[i] = 0;
    if (tid < a.G * W) s_q[tid / W][tid % W] = a.q_codes[((long long)b * a.Hq + (long long)g * a.G + tid / W) * W + tid % W];
    __syncthreads();
    const int unit = b * a.Hkv + g;
    const uint64_t *row = a.k_codes + (long long)b * a.kc_sb + (long long)g * a.kc_sh;
    uint16_t *srow = a.scores + (long long)unit * a.score_row;
    for (int t = start + tid; t < end; t += kWideThreads) {   // a warp reads 32 W consecutive words per step
        unsigned long long kw[W];
        if (W == 1) {
            kw[0] = __ldg(reinterpret_cast<const unsigned long long *>(row + t));
        } else {
#pragma unroll
            for (int w = 0; w < W; w += 2) {
                const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(row + (long long)t * W + w));
                kw[w] = v.x; kw[w + 1] = v.y;
            }
        }
        int best = a.n_bits + 1;   // smallest Hamming distance over the group
        for (int j = 0; j < a.G; ++j) {
            int h = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) h += __popcll(kw[w] ^ s_q[j][w]);
            best = min(best, h);
        }
        const int score = a.n_bits - best;
        const bool forced = t < wu.wbd.sink_end || t >= wu.wbd.local_begin;
        srow[t] = forced ? (uint16_t)kWideForced : (uint16_t)score;
        // unrelated signatures crowd into a few levels around b / 2: lanes with the same score add once, together
        const int key = forced ? -1 : score;
        const unsigned peers = __match_any_sync(__activemask(), key);
        if (key >= 0 && (int)(__ffs(peers) - 1) == (tid & 31)) atomicAdd(&s_hist[warp][score], __popc(peers));
    }
    __syncthreads();
    int32_t *uh = a.unit_hist + (long long)unit * kWideHistStride;
    for (int l = tid; l < levels; l += kWideThreads) {
        int c = 0;
#pragma unroll
        for (int w = 0; w < kWideThreads / 32; ++w) c += s_hist[w][l];
        if (c) atomicAdd(uh + l, c);
    }
}

// Threshold of a unit from its level counts in shared memory (levels = b + 1), by warp 0: T = largest level with
// #{S >= T} >= keep (levels if keep == 0: nothing is selected by score), gt = #{S > T}.  Result in every lane.
__device__ __forceinline__ void wide_threshold(const int *hist, int levels, int keep, int lane, int &T, int &gt) {
    const int per = (levels + 31) / 32;
    const int lo = min(levels, lane * per), hi = min(levels, lo + per);
    int seg = 0;
    for (int l = lo; l < hi; ++l) seg += hist[l];
    int above = seg;   // inclusive suffix sum over lanes: levels >= lo
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
        const int v = __shfl_down_sync(0xffffffffu, above, dd);
        if (lane + dd < 32) above += v;
    }
    T = levels; gt = 0;
    if (keep <= 0) return;
    const unsigned ok = __ballot_sync(0xffffffffu, above >= keep);   // lanes whose lowest level already has enough above it
    if (ok == 0u) { T = 0; gt = __shfl_sync(0xffffffffu, above, 0) - hist[0]; return; }   // cannot happen: #{S >= 0} = n >= keep
    const int owner = 31 - __clz(ok);
    int myT = 0, mygt = 0;
    if (lane == owner) {
        int c = above - seg;   // levels above this lane's segment
        for (int l = hi - 1; l >= lo; --l) {
            if (c + hist[l] >= keep) { myT = l; mygt = c; break; }
            c += hist[l];
        }
    }
    T = __shfl_sync(0xffffffffu, myT, owner);
    gt = __shfl_sync(0xffffffffu, mygt, owner);
}

// flags of 16 consecutive tokens from `first` on (bit i = token first + i): score > T (always-kept tokens included) / == T
__device__ __forceinline__ void wide_flags16(const uint16_t *srow, int first, int end, int T, uint32_t &gt, uint32_t &eq) {
    gt = 0u; eq = 0u;
    if (first >= end) return;
    const uint4 v0 = __ldcg(reinterpret_cast<const uint4 *>(srow + first)), v1 = __ldcg(reinterpret_cast<const uint4 *>(srow + first + 8));
    const uint32_t wv[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int s = (int)((wv[e >> 1] >> (16 * (e & 1))) & 0xffffu);
        if (first + e < end) {
            gt |= (uint32_t)(s > T) << e;
            eq |= (uint32_t)(s == T) << e;
        }
    }
}

__global__ void __launch_bounds__(kWideThreads) wide_count_kernel(const WideArgs a) {
    __shared__ int s_hist[kWideMaxLevels + 7];
    __shared__ int s_T, s_red[2][kWideThreads / 32];
    const int chunk = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const WideUnit wu = wide_unit(a, b);
    const int start = chunk * a.chunk_tokens;
    if (start >= wu.n && chunk > 0) return;
    const int end = min(wu.n, start + a.chunk_tokens);
    const int unit = b * a.Hkv + g, levels = a.n_bits + 1;
    const int32_t *uh = a.unit_hist + (long long)unit * kWideHistStride;
    for (int l = tid; l < levels; l += kWideThreads) s_hist[l] = __ldcg(uh + l);
    __syncthreads();
    if (warp == 0) {
        int T, gt;
        wide_threshold(s_hist, levels, wu.keep_rest, lane, T, gt);
        if (lane == 0) s_T = T;
    }
    __syncthreads();
    const int T = s_T;
    const uint16_t *srow = a.scores + (long long)unit * a.score_row;
    int cg = 0, ce = 0;
    for (int first = start + tid * kWideTokensPerThread; first < end; first += kWidePass) {
        uint32_t gt, eq;
        wide_flags16(srow, first, end, T, gt, eq);
        cg += __popc(gt); ce += __popc(eq);
    }
#pragma unroll
    for (int dd = 16; dd > 0; dd >>= 1) { cg += __shfl_xor_sync(0xffffffffu, cg, dd); ce += __shfl_xor_sync(0xffffffffu, ce, dd); }
    if (lane == 0) { s_red[0][warp] = cg; s_red[1][warp] = ce; }
    __syncthreads();
    if (tid < 2) {
        int s = 0;
        for (int w = 0; w < kWideThreads / 32; ++w) s += s_red[tid][w];
        a.chunk_counts[((long long)unit * kWideMaxChunks + chunk) * 2 + tid] = s;
    }
}

__global__ void __launch_bounds__(kWideThreads) wide_write_kernel(const WideArgs a) {
    __shared__ int s_hist[kWideMaxLevels + 7];
    __shared__ int s_T, s_gt, s_before[2], s_wtot[kWideThreads / 32];
    const int chunk = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const WideUnit wu = wide_unit(a, b);
    const int start = chunk * a.chunk_tokens;
    if (start >= wu.n && chunk > 0) return;
    const int end = min(wu.n, start + a.chunk_tokens);
    const int unit = b * a.Hkv + g, levels = a.n_bits + 1;
    const int32_t *uh = a.unit_hist + (long long)unit * kWideHistStride;
    for (int l = tid; l < levels; l += kWideThreads) s_hist[l] = __ldcg(uh + l);
    if (tid < 2) s_before[tid] = 0;
    __syncthreads();
    if (warp == 0) {
        int T, gt;
        wide_threshold(s_hist, levels, wu.keep_rest, lane, T, gt);
        if (lane == 0) { s_T = T; s_gt = gt; }
    } else if (warp <= 2) {   // tokens above / at the threshold in the chunks before this one
        const int which = warp - 1;
        int s = 0;
        for (int c = lane; c < chunk; c += 32) s += __ldcg(a.chunk_counts + ((long long)unit * kWideMaxChunks + c) * 2 + which);
#pragma unroll
        for (int dd = 16; dd > 0; dd >>= 1) s += __shfl_xor_sync(0xffffffffu, s, dd);
        if (lane == 0) s_before[which] = s;
    }
    __syncthreads();
    const int T = s_T, r = wu.keep_rest - s_gt;   // tokens of score exactly T that are still wanted
    int32_t *list = a.idx + (long long)b * a.idx_sb + (long long)g * a.idx_sh;
    if (chunk == 0) {
        if (tid == 0) a.count[unit] = wu.keep;
        for (int i = wu.keep + tid; i < a.k_max; i += kWideThreads) list[i] = -1;
        if (a.hist_out) for (int l = tid; l < levels; l += kWideThreads) a.hist_out[(long long)unit * levels + l] = s_hist[l];
    }
    if (wu.keep == 0) return;
    const uint16_t *srow = a.scores + (long long)unit * a.score_row;
    int run_gt = s_before[0], run_eq = s_before[1];
    for (int pass = start; pass < end; pass += kWidePass) {   // CTA-uniform
        const int first = pass + tid * kWideTokensPerThread;
        uint32_t gt, eq;
        wide_flags16(srow, first, end, T, gt, eq);
        const int packed = __popc(gt) | (__popc(eq) << 16);
        int inc = packed;
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, dd);
            if (lane >= dd) inc += v;
        }
        if (lane == 31) s_wtot[warp] = inc;
        __syncthreads();
        int wpre = 0, all = 0;
#pragma unroll
        for (int w = 0; w < kWideThreads / 32; ++w) {
            const int v = s_wtot[w];
            if (w < warp) wpre += v;
            all += v;
        }
        if (packed != 0) {
            const int excl = wpre + inc - packed;
            const int g_run = run_gt + (excl & 0xffff), q_run = run_eq + (int)((unsigned)excl >> 16);
            write_selected32(list + g_run + min(q_run, r), first, gt, eq, r - q_run);
        }
        run_gt += all & 0xffff;
        run_eq += (int)((unsigned)all >> 16);
        __syncthreads();
    }
}

// ------------------------------------------------------------------ one kernel, a cluster per unit
//
// A cluster of up to eight CTAs owns a unit: every CTA leaves the scores of its slice in shared memory (16 bits per
// token), the CTAs exchange their level counts through distributed shared memory between two cluster barriers, and each
// compacts its own slice.  Against the three kernels for long sequences there is no memset, no histogram and no score
// pass through global memory, and the signatures are asked into L2 before the programmatic-launch wait.
// Bound: the population-count unit (16 lanes per clock and SM; a token costs G popcounts per counted word), then HBM.
// Carry-save adders on the logic unit fold the xor words of a token before they are counted: 3, 4 and 5 counted words
// instead of 4, 8 and 16 for 128, 256 and 512 bits.
// Counting: counters [level][column], a lane bumps column lane % kCols (32 columns up to 128 bits, then 16 and 8: the
// table stays at 17 KB and the scores spread over more levels).
// Measured, 4 sequences of 32768 tokens with 8 KV heads and groups of 4 at 128 bits, whole decode step through the entry
// points (ENCODE of keys and of queries, this kernel, GATHER-ATT): 33.6 us, against 155 us with the three kernels above
// (19 + 5 + 6 us and a memset) and ENCODE in 128-token tiles (57 + 57 us).
constexpr int kWideSlice = kWideThreads * 8;         // tokens of one row of a CTA: eight per thread
constexpr int kWideMaxRows = 8;                      // a thread's flags fit one 64-bit word
constexpr int kWideClusterMaxSeq = 8 * kWideMaxRows * kWideSlice;

template <int W> struct WideShape;                   // tokens per thread and pass (64 to 128 bytes in flight twice), columns
template <> struct WideShape<1> { static constexpr int kTok = 8, kCols = 32; };
template <> struct WideShape<2> { static constexpr int kTok = 4, kCols = 32; };
template <> struct WideShape<4> { static constexpr int kTok = 4, kCols = 16; };
template <> struct WideShape<8> { static constexpr int kTok = 2, kCols = 8; };

// full adder on bit columns: s + 2 c = x + y + z
__device__ __forceinline__ void csa(uint32_t x, uint32_t y, uint32_t z, uint32_t &s, uint32_t &c) {
    s = x ^ y ^ z;
    c = (x & y) | (x & z) | (y & z);
}
// bits set in 2 W words
template <int W>
__device__ __forceinline__ int count_words(const uint32_t (&x)[2 * W]) {
    if constexpr (W == 1) {
        return __popc(x[0]) + __popc(x[1]);
    } else if constexpr (W == 2) {
        uint32_t s, c;
        csa(x[0], x[1], x[2], s, c);
        return __popc(s) + __popc(x[3]) + 2 * __popc(c);
    } else if constexpr (W == 4) {
        uint32_t s0, s1, s2, c0, c1, c2, t, f;
        csa(x[0], x[1], x[2], s0, c0);
        csa(x[3], x[4], x[5], s1, c1);
        csa(s0, s1, x[6], s2, c2);
        csa(c0, c1, c2, t, f);
        return __popc(s2) + __popc(x[7]) + 2 * __popc(t) + 4 * __popc(f);
    } else {
        uint32_t s[5], c[7], u0, u1, t0, t1, t2, f0, f1, f2, e, f;
#pragma unroll
        for (int i = 0; i < 5; ++i) csa(x[3 * i], x[3 * i + 1], x[3 * i + 2], s[i], c[i]);
        csa(s[0], s[1], s[2], u0, c[5]);
        csa(s[3], s[4], x[15], u1, c[6]);          // ones left: u0, u1
        csa(c[0], c[1], c[2], t0, f0);
        csa(c[3], c[4], c[5], t1, f1);
        csa(t0, t1, c[6], t2, f2);                 // twos left: t2
        csa(f0, f1, f2, f, e);                     // fours: f, eights: e
        return __popc(u0) + __popc(u1) + 2 * __popc(t2) + 4 * __popc(f) + 8 * __popc(e);
    }
}

// flags of eight consecutive 16-bit scores + 1: bit i = score > T / == T, with t2 = (T + 1) in both halves
__device__ __forceinline__ void wide_flags8(const uint4 &v, uint32_t t2, uint32_t &gt, uint32_t &eq) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    gt = 0u; eq = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t g = __vcmpgtu2(w[i], t2), q = __vcmpeq2(w[i], t2);
        gt |= ((g & 1u) | ((g >> 15) & 2u)) << (2 * i);
        eq |= ((q & 1u) | ((q >> 15) & 2u)) << (2 * i);
    }
}

template <int W>
__global__ void __launch_bounds__(kWideThreads) wide_select_cluster_kernel(const WideArgs a, int rows_max) {
    constexpr int kTok = WideShape<W>::kTok, kCols = WideShape<W>::kCols;
    extern __shared__ __align__(16) unsigned char wsm[];
    uint16_t *s_sc = reinterpret_cast<uint16_t *>(wsm);                                   // [rows_max * kWideSlice] score + 1, 0 = none
    uint32_t *c_hist = reinterpret_cast<uint32_t *>(s_sc + (size_t)rows_max * kWideSlice);    // [levels][kCols]
    const int levels = a.n_bits + 1;
    __shared__ int s_hist[kWideMaxLevels + 7], s_tot[kWideMaxLevels + 7], s_bef[kWideMaxLevels + 7];
    __shared__ __align__(16) unsigned long long s_q[kMaxGroup][W];
    __shared__ int sh_T, sh_gt, sh_gt_before, sh_eq_before, s_wcnt[kWideThreads / 32];
    const int rank = (int)cluster_rank(), cs = (int)gridDim.x;                            // the cluster spans the grid's x
    const int g = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const WideUnit wu = wide_unit(a, b);
    const int n = wu.n;
    const int Rb = (n + cs * kWideSlice - 1) / (cs * kWideSlice);                         // the sequence's own length is shared out
    const int slice = Rb * kWideSlice, base = rank * slice, unit = b * a.Hkv + g;
    const uint64_t *row = a.k_codes + (long long)b * a.kc_sb + (long long)g * a.kc_sh;

    // a pass: token base + (p kTok + i) 256 + tid for i < kTok, so that a warp reads consecutive signatures
    auto load_token = [&](unsigned long long (&kw)[W], int t) {
        if (W == 1) {
            kw[0] = __ldcg(reinterpret_cast<const unsigned long long *>(row + t));
        } else {
#pragma unroll
            for (int w = 0; w < W; w += 2) {
                const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2 *>(row + (long long)t * W + w));
                kw[w] = v.x; kw[w + 1] = v.y;
            }
        }
    };
    auto load_pass = [&](unsigned long long (&kw)[kTok][W], int p) {
#pragma unroll
        for (int i = 0; i < kTok; ++i) {
            const int l = (p * kTok + i) * kWideThreads + tid;
            if (l < slice && base + l < n) load_token(kw[i], base + l);
            else
#pragma unroll
                for (int w = 0; w < W; ++w) kw[i][w] = 0ull;
        }
    };
    // The signatures are only asked into L2 before the launch wait (one request per 128-byte line) and loaded behind it: the
    // kernel in front may still be writing one, at any slot.  The whole slice, since HBM is idle under ENCODE: 5 ragged sequences
    // of up to 65536 tokens at 256 bits 61.8 us per step, with the first four passes 65.3, with the first alone 66.9; 6 ragged ones
    // of 32768 at 512 bits 81.3 / 83.2 / 87.5.
    for (int l = tid * (16 / W); l < min(slice, n - base); l += kWideThreads * (16 / W))
        asm volatile("prefetch.global.L2 [%0];" ::"l"(row + (long long)(base + l) * W));
    unsigned long long cur[kTok][W], nxt[kTok][W];
    for (int i = tid; i < levels * kCols; i += kWideThreads) c_hist[i] = 0u;
    pdl_launch_dependents();
    pdl_wait();
    load_pass(cur, 0);
    if (tid < a.G * W)
        s_q[tid / W][tid % W] = __ldcg(reinterpret_cast<const unsigned long long *>(a.q_codes) +
                                       ((long long)b * a.Hq + (long long)g * a.G + tid / W) * W + tid % W);
    __syncthreads();

    const int n_pass = Rb * 8 / kTok;
    for (int p = 0; p < n_pass; ++p) {
        if (p + 1 < n_pass) load_pass(nxt, p + 1);
        int best[kTok];
#pragma unroll
        for (int i = 0; i < kTok; ++i) best[i] = a.n_bits;
        for (int j = 0; j < a.G; ++j) {
            unsigned long long qv[W];
#pragma unroll
            for (int w = 0; w < W; ++w) qv[w] = s_q[j][w];
#pragma unroll
            for (int i = 0; i < kTok; ++i) {
                uint32_t x[2 * W];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const unsigned long long v = cur[i][w] ^ qv[w];
                    x[2 * w] = (uint32_t)v;
                    x[2 * w + 1] = (uint32_t)(v >> 32);
                }
                best[i] = min(best[i], count_words<W>(x));
            }
        }
#pragma unroll
        for (int i = 0; i < kTok; ++i) {
            const int l = (p * kTok + i) * kWideThreads + tid, t = base + l;
            if (l < slice) {
                uint32_t v = 0u;
                if (t < n) {
                    const int score = a.n_bits - best[i];
                    if (t < wu.wbd.sink_end || t >= wu.wbd.local_begin) v = kWideForced;
                    else { v = (uint32_t)score + 1u; atomicAdd(&c_hist[score * kCols + (lane & (kCols - 1))], 1u); }
                }
                s_sc[l] = (uint16_t)v;
            }
        }
#pragma unroll
        for (int i = 0; i < kTok; ++i)
#pragma unroll
            for (int w = 0; w < W; ++w) cur[i][w] = nxt[i][w];
    }
    __syncthreads();
    for (int l = tid; l < levels; l += kWideThreads) {
        uint32_t c = 0u;
#pragma unroll
        for (int k = 0; k < kCols; ++k) c += c_hist[l * kCols + ((k + l) & (kCols - 1))];
        s_hist[l] = (int)c;
    }
    cluster_sync_all();   // every CTA's level counts are complete and visible cluster-wide
    for (int l = tid; l < levels; l += kWideThreads) {
        int tot = 0, bef = 0;
        for (int r = 0; r < cs; ++r) {
            const int v = ld_dsmem(&s_hist[l], (uint32_t)r);
            tot += v;
            if (r < rank) bef += v;
        }
        s_tot[l] = tot;
        s_bef[l] = bef;
    }
    cluster_arrive();     // done with the peers' memory; the matching wait is at the end
    __syncthreads();
    if (warp == 0) {
        int T, gt;
        wide_threshold(s_tot, levels, wu.keep_rest, lane, T, gt);
        int gb = 0;
        for (int l = T + 1 + lane; l < levels; l += 32) gb += s_bef[l];
#pragma unroll
        for (int dd = 16; dd > 0; dd >>= 1) gb += __shfl_xor_sync(0xffffffffu, gb, dd);
        if (lane == 0) { sh_T = T; sh_gt = gt; sh_gt_before = gb; sh_eq_before = T < levels ? s_bef[T] : 0; }
    }
    if (rank == 0 && a.hist_out)
        for (int l = tid; l < levels; l += kWideThreads) a.hist_out[(long long)unit * levels + l] = s_tot[l];
    __syncthreads();
    const int T = sh_T, r = wu.keep_rest - sh_gt;   // tokens of score exactly T that are still wanted
    int32_t *list = a.idx + (long long)b * a.idx_sb + (long long)g * a.idx_sh;
    if (rank == 0) {
        if (tid == 0) a.count[unit] = wu.keep;
        for (int i = wu.keep + tid; i < a.k_max; i += kWideThreads) list[i] = -1;
    }
    if (wu.keep == 0) { cluster_wait(); return; }

    // thread = the 8 Rb consecutive tokens from first_l on
    const uint32_t t2 = (uint32_t)(T + 1) * 0x00010001u;
    const int first_l = 8 * Rb * tid;
    uint32_t gt_lo = 0u, gt_hi = 0u, eq_lo = 0u, eq_hi = 0u;
#pragma unroll
    for (int j = 0; j < kWideMaxRows; ++j) {
        if (j < Rb) {
            uint32_t gf, ef;
            wide_flags8(*reinterpret_cast<const uint4 *>(s_sc + first_l + 8 * j), t2, gf, ef);
            if (j < 4) { gt_lo |= gf << (8 * j); eq_lo |= ef << (8 * j); }
            else { gt_hi |= gf << (8 * (j - 4)); eq_hi |= ef << (8 * (j - 4)); }
        }
    }
    const int packed = (__popc(gt_lo) + __popc(gt_hi)) | ((__popc(eq_lo) + __popc(eq_hi)) << 16);
    int inc = packed;
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, dd);
        if (lane >= dd) inc += v;
    }
    if (lane == 31) s_wcnt[warp] = inc;
    __syncthreads();
    int g_run = sh_gt_before + forced_before(wu.wbd, min(base, n)), q_run = sh_eq_before;
#pragma unroll
    for (int w = 0; w < kWideThreads / 32; ++w)
        if (w < warp) { g_run += s_wcnt[w] & 0xffff; q_run += (int)((unsigned)s_wcnt[w] >> 16); }
    if (packed != 0) {
        const int excl = inc - packed;
        g_run += excl & 0xffff;
        q_run += (int)((unsigned)excl >> 16);
        int32_t *dst = list + g_run + min(q_run, r);
        dst = write_selected32(dst, base + first_l, gt_lo, eq_lo, r - q_run);
        write_selected32(dst, base + first_l + 32, gt_hi, eq_hi, r - q_run - __popc(eq_lo));
    }
    cluster_wait();
}

template <int W>
static void wide_cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int Hkv, int B, int cs, int rows, cudaStream_t st) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(cs, Hkv, B);
    cfg.blockDim = dim3(kWideThreads);
    cfg.dynamicSmemBytes = (size_t)rows * kWideSlice * 2 + (size_t)(W * 64 + 1) * WideShape<W>::kCols * 4;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
}

// How many clusters of cs CTAs with `rows` rows of tokens each the device holds at once (0 on error); the answers are kept per
// device.  Registers set it up to four rows (64, 63, 121, 113 at 64, 128, 256, 512 bits: four CTAs of 256 threads per SM or two),
// shared memory beyond.
template <int W>
static int wide_resident_clusters(int cs, int rows) {
    static std::atomic<int> known[64][3][kWideMaxRows + 1];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 0;
    std::atomic<int> &k = known[dev][cs == 8 ? 2 : cs == 4 ? 1 : 0][rows];
    int n = k.load(std::memory_order_acquire);
    if (n > 0) return n;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    wide_cluster_config<W>(cfg, attr, 1, 64, cs, rows, nullptr);
    cfg.numAttrs = 1;   // the cluster shape is all the occupancy query looks at
    n = ask_resident_clusters(wide_select_cluster_kernel<W>, cfg, 64 * 1024);
    k.store(n, std::memory_order_release);
    return n;
}

// One cluster per unit: the largest of 8, 4, 2 CTAs of which all units' are resident at once, or two thirds of them where a
// second wave costs less than smaller clusters (512 bits, bound by its loads; the step from 4 to 2; CTAs of more than six rows,
// few and long); at least as many as the rows of a CTA hold.  Whole steps of 32768 tokens a sequence, 8 units each, groups of 4, us, with the chosen size and the other:
//    64, 128 bits   64 units on 8: 36.5 and 42.5, on 4: 42.7 and 53.6;  112 on 4, 128 bits: 60.9, on 2: 85.4;
//                   152 units on 4 (148 resident): 72.4 and 90.1, on 2: 77.1 and 98.4
//    256 bits       40 units on 4: 51.8, on 8 (36 resident): 54.9;  80 on 4 (74 resident): 81.3, on 2: 82.6, but 104 88.6 / 83.8
//    512 bits       40 units on 8: 91.4, on 4: 98.0;  48: 101.5 / 98.1, ragged 87.4 / 96.4;  80 on 4: 163, on 2: 174
// Sequences of 65536 (eight rows with 4): 128 bits, 80 units on 8: 87.3, on 4: 93.0, ragged 68.8 / 77.4; 256 bits, 40 units 81.7 /
// 80.4, ragged 66.9 / 76.4; of 40000 (five rows) the other way: 69.3 / 66.9 and 67.4 / 59.7.
template <int W>
static cudaError_t launch_wide_cluster(const WideArgs &a, int B, cudaStream_t st) {
    auto rows_of = [&](int cs) { return max(1, (a.max_seq_len + cs * kWideSlice - 1) / (cs * kWideSlice)); };
    int cs = 8;
    while (cs > 2 && rows_of(cs / 2) <= kWideMaxRows &&
           2LL * B * a.Hkv > (W == 8 || cs == 4 || rows_of(cs / 2) > 6 ? 3LL : 2LL) * wide_resident_clusters<W>(cs, rows_of(cs)))
        cs >>= 1;
    if (wide_resident_clusters<W>(cs, rows_of(cs)) <= 0) return cudaErrorInvalidConfiguration;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    wide_cluster_config<W>(cfg, attr, a.Hkv, B, cs, rows_of(cs), st);
    cudaError_t e = cudaLaunchKernelEx(&cfg, wide_select_cluster_kernel<W>, a, rows_of(cs));
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

// Workspace of the wide selection: header | unit histograms | chunk counts | 16-bit scores.
struct WideLayout {
    size_t off_hist, off_counts, off_scores, score_row, total;
};
WideLayout wide_layout(int B, int Hkv, int max_seq_len) {
    WideLayout L;
    const size_t units = (size_t)B * Hkv;
    size_t o = kHeaderBytes;
    L.off_hist = o;   o = align_up(o + units * kWideHistStride * 4, 256);
    L.off_counts = o; o = align_up(o + units * kWideMaxChunks * 2 * 4, 256);
    L.score_row = align_up((size_t)(max_seq_len > 0 ? max_seq_len : 0), 256);
    L.off_scores = o; o = align_up(o + units * L.score_row * 2, 256);
    L.total = o;
    return L;
}
size_t wide_workspace_bytes(int B, int Hkv, int max_seq_len) { return wide_layout(B, Hkv, max_seq_len).total; }

cudaError_t launch_score_topk_wide(int B, int Hq, int Hkv, int n_bits, const uint64_t *q_codes, const uint64_t *k_codes,
                                   long long kc_sb, long long kc_sh, const int32_t *seq_lens, const int32_t *k_per_seq,
                                   int k_uniform, int max_seq_len, int k_max, int32_t *idx, long long idx_sb, long long idx_sh,
                                   int32_t *count, int32_t *hist_out, void *workspace, cudaStream_t st, Windows win) {
    const WideLayout L = wide_layout(B, Hkv, max_seq_len);
    char *ws = reinterpret_cast<char *>(workspace);
    WideArgs a{};
    a.q_codes = q_codes; a.k_codes = k_codes; a.kc_sb = kc_sb; a.kc_sh = kc_sh; a.seq_lens = seq_lens; a.k_per_seq = k_per_seq;
    a.k_uniform = k_uniform; a.max_seq_len = max_seq_len; a.k_max = k_max; a.Hq = Hq; a.Hkv = Hkv; a.G = Hq / Hkv; a.n_bits = n_bits;
    a.win = win; a.idx = idx; a.idx_sb = idx_sb; a.idx_sh = idx_sh; a.count = count; a.hist_out = hist_out;
    a.unit_hist = reinterpret_cast<int32_t *>(ws + L.off_hist);
    a.chunk_counts = reinterpret_cast<int32_t *>(ws + L.off_counts);
    a.scores = reinterpret_cast<uint16_t *>(ws + L.off_scores);
    a.score_row = (long long)L.score_row;
    if (max_seq_len <= kWideClusterMaxSeq) {
        switch (n_bits / 64) {
            case 1: return launch_wide_cluster<1>(a, B, st);
            case 2: return launch_wide_cluster<2>(a, B, st);
            case 4: return launch_wide_cluster<4>(a, B, st);
            case 8: return launch_wide_cluster<8>(a, B, st);
            default: return cudaErrorInvalidValue;
        }
    }
    // chunks of whole passes, about eight CTAs per SM when there is that much work, at most kWideMaxChunks per unit
    const long long units = (long long)B * Hkv, n = max_seq_len > 0 ? max_seq_len : 1;
    long long per_unit = 8LL * sm_count() / (units > 0 ? units : 1);
    if (per_unit < 1) per_unit = 1;
    if (per_unit > kWideMaxChunks) per_unit = kWideMaxChunks;
    long long c = (n + per_unit - 1) / per_unit;
    const long long c_min = (n + kWideMaxChunks - 1) / kWideMaxChunks;
    if (c < c_min) c = c_min;
    if (c < kWidePass) c = kWidePass;
    a.chunk_tokens = (int)((c + kWidePass - 1) / kWidePass * kWidePass);
    const int n_chunks = (int)((n + a.chunk_tokens - 1) / a.chunk_tokens);
    cudaError_t e = cudaMemsetAsync(a.unit_hist, 0, (size_t)units * kWideHistStride * 4, st);
    if (e != cudaSuccess) return e;
    dim3 grid(n_chunks, Hkv, B);
    switch (n_bits / 64) {
        case 1: wide_scan_kernel<1><<<grid, kWideThreads, 0, st>>>(a); break;
        case 2: wide_scan_kernel<2><<<grid, kWideThreads, 0, st>>>(a); break;
        case 4: wide_scan_kernel<4><<<grid, kWideThreads, 0, st>>>(a); break;
        case 8: wide_scan_kernel<8><<<grid, kWideThreads, 0, st>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    wide_count_kernel<<<grid, kWideThreads, 0, st>>>(a);
    wide_write_kernel<<<grid, kWideThreads, 0, st>>>(a);
    count_launch(3);
    return cudaGetLastError();
}

} // namespace ha
