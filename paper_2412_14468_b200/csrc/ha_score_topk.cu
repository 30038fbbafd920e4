// SCORE + TOPK.  Scores are s = 32 - popc(k_code ^ q_code) (Eq. 1 via the bitcount-xor identity of
// Section 4.1), reduced with max over the query heads of the GQA group, so they take only 33
// values.  "Standard top-k" (Section 4) therefore needs no sort: a histogram gives the threshold
// score T and how many tokens r of score exactly T are still needed; the selection is every token
// above T plus the first r tokens at T in index order, written in ascending token order.
//
// Three implementations share the arithmetic:
//  * sequences of up to 131072 tokens: ONE kernel, a thread-block cluster per (sequence, KV head)
//    (score_select_cluster_kernel, second half of this file), over contiguous or paged signatures (24 sequences of 2000 -
//    65536 tokens in pages of 16, whole step: 61.4 us against 84.1 us with the two kernels below);
//  * many short units, many units of more than 32768 tokens with a budget each, and more than 131072 tokens from 24 units on: ONE
//    kernel whose clusters take several units each (score_select_batch_kernel; batch_cluster_size has the rule);
//  * other longer sequences: two kernels over chunks of the sequence, with the per-chunk histograms and
//    one score byte per token passed through the workspace (scan_score_kernel, select_kernel).
// No CTA ever spins on another: hand-offs are hardware cluster barriers or kernel boundaries.
// The scanning kernels request their first signatures before the programmatic-launch wait, so that
// the fetch overlaps the tail of the preceding kernel.  Every kernel that writes signatures lets its
// dependents start behind them, except the ENCODE of a layer-step (in_step): its one signature (the
// appended token, slot n-1) is re-read after the wait.  A block table is read before the wait only
// inside a layer-step, where ENCODE has waited for whatever wrote it.
#include "ha_score_dev.cuh"

namespace ha {

constexpr int kScanThreads = 256;
constexpr int kPassTokens = kScanThreads * 16;   // four uint4 per thread
constexpr int kClusterMaxSeq = 8 * 8 * 2048;     // longest sequence the cluster kernel takes (8 CTAs x 8 rows x 2048 tokens)

// Clusters of 8 CTAs of 512 threads (two per SM, 36 clusters resident at once) instead of 256: with 24 to 36 units the hardware
// stacks the small CTAs on half of the SMs.  Whole steps, groups of 4, us: 32 units of 70000 tokens 32.8 against 34.2, of 130000
// 40.9 / 45.1, of 200000 53.2 / 56.5 (there against the two kernels); 24 units of 250000 50.6 / 53.1, but of 50000 22.4 / 22.1;
// 16 units of 70000 25.3 / 24.5.  (Clusters of 16 of them for one sequence of 150000 or 250000 tokens win 5 us in back-to-back
// calls and lose 1.2 us in a step, where the kernel in front holds their SMs.)
inline bool large_clusters(long long units, int max_seq_len) {
    return units >= 24 && units <= 36 && max_seq_len > 65536 && max_seq_len <= 8 * 8 * 4096;
}

// ------------------------------------------------------------------ long-sequence path (two kernels)

// Kernel 1: one chunk per CTA.  Streams the chunk's signatures (four uint4 per thread in flight, the
// next pass requested before the current one is scored), leaves the group scores as one byte per
// token in the workspace (so that kernel 2 needs neither the signatures nor popc again) and the
// chunk's 33-bin histogram.  Counting: one 32-bit counter per (level, lane), shared by the warps and
// bumped with shared-memory reductions (a lane only meets its own column; nothing waits for a result).
template <int G>
__global__ void __launch_bounds__(kScanThreads) scan_score_kernel(const uint32_t *__restrict__ q_codes,
                                                                 const uint32_t *__restrict__ k_codes,
                                                                 long long kc_sb, long long kc_sh,
                                                                 const int32_t *__restrict__ seq_lens,
                                                                 int max_seq_len, int Hq, int Hkv,
                                                                 int chunk_tokens, long long score_row,
                                                                 unsigned char *__restrict__ ws_scores,
                                                                 int32_t *__restrict__ ws_hist, Windows win, CodePages cp,
                                                                 int row_shift, bool in_step) {
    __shared__ __align__(16) uint32_t c_hist[kBins][32];
    __shared__ int s_hist[kBins + 3];
    __shared__ uint32_t s_qc[G];
    const int chunk = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
    const int kvh = row_shift >= 0 ? (g >> row_shift) : g;   // the KV head whose signatures this unit scans
    const bool paged = cp.table != nullptr;
    const int32_t *table_b = paged ? cp.table + (long long)b * cp.bt_sb : nullptr;
    const int n = min(seq_lens[b], max_seq_len);
    const int start = chunk * chunk_tokens;
    if (start >= n) {
        if (chunk == 0) pdl_wait();   // at least one CTA of a grid waits, also when every sequence is empty
        return;
    }
    if (paged && !in_step) pdl_wait();   // a block table may come from the kernel in front
    const int tid = threadIdx.x, lane = tid & 31;
    // contiguous cache: the unit's row; paged cache: the pool from this head's offset on
    const uint32_t *row = paged ? k_codes + (long long)kvh * cp.head_stride : k_codes + (long long)b * kc_sb + (long long)kvh * kc_sh;
    uint32_t *srow = reinterpret_cast<uint32_t *>(ws_scores + ((long long)b * Hkv + g) * score_row);
    const int end = min(n, start + chunk_tokens);
    const WindowBounds wbd = window_bounds(win, n);   // always-kept tokens: byte kForcedByte, not counted

    // pass = 4096 tokens: sub-block j of 1024 tokens, one uint4 per thread (coalesced)
    auto load_pass = [&](uint4 (&c)[4], int pass) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int base = pass + j * 1024 + tid * 4;
            if (base >= end) c[j] = make_uint4(0, 0, 0, 0);
            else c[j] = paged ? load_codes4_paged(cp, row, table_b, base, end) : load_codes4(row, base, end);
        }
    };
    uint4 cur[4], nxt[4];
    load_pass(cur, start);
    for (int i = tid; i < kBins * 32 / 4; i += kScanThreads)
        reinterpret_cast<uint4 *>(&c_hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < kBins + 3) s_hist[tid] = 0;
    pdl_launch_dependents();
    pdl_wait();
    // The query signatures were written by the kernel in front of this one and must come from L2; the many
    // CTAs of a long sequence all want the same few words, so one thread per word fetches them for the CTA.
    if (tid < G) s_qc[tid] = __ldcg(q_codes + (long long)b * Hq + g * G + tid);
    __syncthreads();
    uint32_t qc[G];
#pragma unroll
    for (int j = 0; j < G; ++j) qc[j] = s_qc[j];

    // the counter of score s sits (32 - s) rows below the lane's counter of level 32
    const uint32_t top = (uint32_t)__cvta_generic_to_shared(&c_hist[kBins - 1][lane]);
    auto bump = [&](int ham) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(top - (uint32_t)ham * 128u) : "memory"); };
    auto hamming = [&](uint32_t code) {
        int h = __popc(code ^ qc[0]);
#pragma unroll
        for (int j = 1; j < G; ++j) h = min(h, __popc(code ^ qc[j]));
        return h;
    };
    for (int pass = start; pass < end; pass += kPassTokens) {
        if (pass + kPassTokens < end) load_pass(nxt, pass + kPassTokens);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int base = pass + j * 1024 + tid * 4;
            if (base < end) {
                if (paged) patch_token_paged(cur[j], base, n - 1, cp, row, table_b);   // the step's ENCODE may just have written it
                else patch_token(cur[j], base, n - 1, row);
                const int h0 = hamming(cur[j].x), h1 = hamming(cur[j].y), h2 = hamming(cur[j].z), h3 = hamming(cur[j].w);
                // bytes 33 - h = score + 1 (0 = no token); no byte borrows because h <= 32
                uint32_t s4 = 0x21212121u - ((uint32_t)h0 | ((uint32_t)h1 << 8) | ((uint32_t)h2 << 16) | ((uint32_t)h3 << 24));
                if (base + 3 < end && base >= wbd.sink_end && base + 4 <= wbd.local_begin) {
                    bump(h0); bump(h1); bump(h2); bump(h3);   // whole uint4 inside the chunk, outside the windows
                } else {
                    const int hh[4] = {h0, h1, h2, h3};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int t = base + e;
                        if (t >= end) s4 &= ~(0xffu << (8 * e));                           // zero byte: no token
                        else if (t < wbd.sink_end || t >= wbd.local_begin) s4 = (s4 & ~(0xffu << (8 * e))) | (kForcedByte << (8 * e));
                        else bump(hh[e]);
                    }
                }
                srow[base >> 2] = s4;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) cur[j] = nxt[j];
    }
    __syncthreads();
    for (int i = tid; i < kBins * 8; i += kScanThreads) {   // eight threads per level, four counters each
        const uint4 v = reinterpret_cast<const uint4 *>(&c_hist[i >> 3][0])[i & 7];
        const uint32_t ssum = (v.x + v.y) + (v.z + v.w);
        if (ssum) atomicAdd(&s_hist[i >> 3], (int)ssum);
    }
    __syncthreads();
    if (tid < kBins) ws_hist[(((long long)b * Hkv + g) * kMaxChunks + chunk) * kBins + tid] = s_hist[tid];
}

// Kernel 2: one chunk per CTA.  Sums the chunk histograms (total, and the part before its own
// chunk), derives T, r and its output offset, then walks its chunk's score bytes and writes the
// selected token indices in ascending order, visiting only those.  A thread takes 16 kQuads consecutive tokens per pass: 32, so that
// a chunk of 8192 tokens is one pass (one sequence of 524288 tokens 39.7 -> 38.3 us per step, of 300000 at 8x 53.2 -> 50.7), but 16
// of what is one pass of those anyway, where half of the threads would have nothing: the rest of a long sequence, all of a short one
// (256 units of 500 - 2000 tokens in a max_seq_len of 200000 30.1 us with 32, 29.3), and the shortest chunks, for which the kernel is
// compiled without the second half (one sequence of 200000 25.3 with it, 24.9).
template <int kQuads>
__global__ void __launch_bounds__(kScanThreads) select_kernel(const int32_t *__restrict__ seq_lens, int max_seq_len,
                                                             const int32_t *__restrict__ k_per_seq, int k_uniform,
                                                             int k_max, int Hkv, int chunk_tokens, long long score_row,
                                                             const unsigned char *__restrict__ ws_scores,
                                                             const int32_t *__restrict__ ws_hist,
                                                             int32_t *__restrict__ idx, long long idx_sb,
                                                             long long idx_sh, int32_t *__restrict__ count,
                                                             int32_t *__restrict__ hist_out, Windows win) {
    __shared__ int s_wtot[kScanThreads / 32][kBins + 3], s_wbef[kScanThreads / 32][kBins + 3];
    __shared__ int warp_tot[kScanThreads / 32];
    const int chunk = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = max(min(seq_lens[b], max_seq_len), 0);
    int k = k_per_seq ? k_per_seq[b] : k_uniform;
    const WindowBounds wbd = window_bounds(win, n);
    const int n_forced = forced_before(wbd, n);
    const int keep_rest = max(0, min(min(k, k_max - n_forced), n - n_forced));   // heavy tokens among the others
    const int keep = n_forced + keep_rest;
    const int n_chunks = (n + chunk_tokens - 1) / chunk_tokens;
    if (chunk > 0 && chunk >= n_chunks) return;
    pdl_launch_dependents();
    pdl_wait();   // histograms and score bytes come from the preceding kernel

    const uint4 *srow = reinterpret_cast<const uint4 *>(ws_scores + ((long long)b * Hkv + g) * score_row);
    const int start = chunk * chunk_tokens, end = min(n, start + chunk_tokens);
    const int quads = end - start > kPassTokens ? kQuads : 1;              // CTA-uniform
    const int per = 16 * quads, pass_tokens = kScanThreads * per;          // tokens of a thread and of the CTA per pass
    // first pass of score bytes: requested now, used after the threshold is known
    uint4 sv_next[kQuads];
#pragma unroll
    for (int h = 0; h < kQuads; ++h) {
        const int base = start + tid * per + h * 16;
        sv_next[h] = (chunk < n_chunks && base < end && h < quads) ? __ldcg(srow + (base >> 4)) : make_uint4(0u, 0u, 0u, 0u);
    }

    // totals per score level, and the part contributed by the chunks before this one.  Lane l of warp w sums
    // level l over the chunks w, w + 8, ... (coalesced rows of the counter table, every load issued before
    // the first use), lane 0 also level 32; the eight warps' sums meet in shared memory.  No atomics: a
    // hundred adds queued on one shared-memory word would stall the loads that follow them.
    {
        const int32_t *hb = ws_hist + ((long long)b * Hkv + g) * kMaxChunks * kBins;
        constexpr int kWarps = kScanThreads / 32, kPer = kMaxChunks / kWarps;
        int v[kPer], v32[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int cc = warp + i * kWarps;
            v[i] = (cc < n_chunks) ? __ldcg(hb + cc * kBins + lane) : 0;
            v32[i] = (cc < n_chunks && lane == 0) ? __ldcg(hb + cc * kBins + 32) : 0;
        }
        int tot = 0, bef = 0, tot32 = 0, bef32 = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int cc = warp + i * kWarps;
            tot += v[i];
            tot32 += v32[i];
            if (cc < chunk) { bef += v[i]; bef32 += v32[i]; }
        }
        s_wtot[warp][lane] = tot;
        s_wbef[warp][lane] = bef;
        if (lane == 0) { s_wtot[warp][32] = tot32; s_wbef[warp][32] = bef32; }
    }
    __syncthreads();
    // Every warp folds the eight partial sums and derives the threshold for itself (lane l owns level l,
    // level 32 is read by every lane): no broadcast, no further barrier.  Suffix sums over the levels give
    // #{S >= t}; T = largest level with #{S >= T} >= keep; r = keep - #{S > T}.
    int T, r, gt_before, eq_before;
    {
        int tot = 0, bef = 0, tot32 = 0, bef32 = 0;
#pragma unroll
        for (int w = 0; w < kScanThreads / 32; ++w) {
            tot += s_wtot[w][lane];
            bef += s_wbef[w][lane];
            tot32 += s_wtot[w][32];
            bef32 += s_wbef[w][32];
        }
        find_threshold(tot, bef, tot32, bef32, keep_rest, lane, T, r, gt_before, eq_before);
        if (warp == 0 && chunk == 0 && hist_out) {
            hist_out[((long long)b * Hkv + g) * kBins + lane] = tot;
            if (lane == 0) hist_out[((long long)b * Hkv + g) * kBins + 32] = tot32;
        }
    }
    int32_t *out = idx + (long long)b * idx_sb + (long long)g * idx_sh;
    if (chunk == 0) {
        if (tid == 0) count[b * Hkv + g] = keep;
        for (int i = keep + tid; i < k_max; i += kScanThreads) out[i] = -1;
    }
    if (chunk >= n_chunks || keep == 0) return;

    // Per byte b = score + 1 (0 = no token): b + 127 - (T+1) sets bit 7 iff score > T, b + 128 - (T+1) iff
    // score >= T (no byte sum reaches 256).
    const uint32_t T4 = (uint32_t)(T + 1) * 0x01010101u;
    const uint32_t c_gt = 0x7f7f7f7fu - T4, c_ge = 0x80808080u - T4;
    // tokens before this pass with S > T (always-kept tokens count as such) / S == T
    int run_gt = gt_before + forced_before(wbd, start), run_eq = eq_before;
    for (int pass = start; pass < end; pass += pass_tokens) {
        const int base = pass + tid * per;
        uint32_t gt32 = 0u, ge32 = 0u;   // bit i = token base + i
#pragma unroll
        for (int h = 0; h < kQuads; ++h) {
            const uint4 sv = sv_next[h];
            const int next = base + pass_tokens + h * 16;
            sv_next[h] = (next < end && h < quads) ? __ldcg(srow + (next >> 4)) : make_uint4(0u, 0u, 0u, 0u);   // next pass, in flight
            const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // words past the chunk were never written: drop them (end is a multiple of 4 or the sequence end)
                const uint32_t w = (base + 16 * h + 4 * j < end) ? sw[j] : 0u;
                gt32 |= high_bits_to_nibble(w + c_gt) << (16 * h + 4 * j);
                ge32 |= high_bits_to_nibble(w + c_ge) << (16 * h + 4 * j);
            }
        }
        const uint32_t eq32 = ge32 ^ gt32;   // score > T implies score >= T
        const int packed = __popc(gt32) | (__popc(eq32) << 16);
        // block-wide exclusive prefix of the packed (gt, eq) counts (a pass has at most 8192 tokens: 16-bit halves suffice)
        int inc = packed;
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, dd);
            if (lane >= dd) inc += v;
        }
        if (lane == 31) warp_tot[warp] = inc;
        __syncthreads();
        int wpre = 0, all = 0;
#pragma unroll
        for (int w = 0; w < kScanThreads / 32; ++w) {
            const int v = warp_tot[w];
            if (w < warp) wpre += v;
            all += v;
        }
        const int excl = wpre + inc - packed, q_run = run_eq + (int)((unsigned)excl >> 16);
        write_selected32(out + run_gt + (excl & 0xffff) + min(q_run, r), base, gt32, eq32, r - q_run);
        run_gt += all & 0xffff;
        run_eq += (int)((unsigned)all >> 16);
        __syncthreads();   // warp_tot is rewritten by the next pass
    }
}

// ------------------------------------------------------------------ fused single-kernel path
//
// For sequences of up to CS * 16384 tokens one thread-block cluster of CS = 8, 4 or 2 CTAs owns a
// (sequence, KV head) unit: every CTA leaves the scores of its slice in shared memory (one byte per
// token), the CTAs exchange their 33-bin histograms through distributed shared memory between two
// hardware cluster barriers, and each CTA then compacts its own slice from those bytes.  The
// signatures are read from HBM once, there is no histogram round trip through global memory and no
// second launch.
// Reading: a warp owns 256*Rb consecutive tokens and reads them in rows of 256 tokens, a lane 8
// consecutive tokens (one 32-byte sector) per row, so that every request of a warp covers 1 KB of
// contiguous memory.  Few registers are live (no per-thread score array), so six CTAs share an SM
// and hide each other's barriers and the latency of the population-count unit, which is the
// scarce resource here (one quarter-rate instruction per query head and token).
// Counting: one 32-bit counter per (level, lane), shared by the eight warps and bumped with
// shared-memory reductions: a lane only meets its own column, so an instruction never conflicts
// with itself, and nothing waits for a result.
// Writing: lane l owns the 8*Rb consecutive tokens l*8*Rb .. of its warp's range, so the prefix sums
// need one warp-shuffle scan plus one exchange of eight warp totals; only selected tokens are
// visited.

constexpr int kClusterMaxRows = 8;   // rows of 8 tokens per lane: a lane's flags fit one 64-bit word each

// kPaged: the signatures lie in a pool behind a block table.  Pages of 8 tokens or more hold a lane's 8 tokens in one piece, so
// a row costs one table entry per lane (neighbouring lanes share it) and the same two 16-byte loads.  The table entries of the
// next two rows are fetched while the current ones are scored; five CTAs per SM instead of six pay for the registers.
// kThreads: 256, or 512 (large_clusters).
template <int G, int CS, bool kPaged, int kThreads>
__global__ void __launch_bounds__(kThreads, kThreads > 256 ? 2 : kPaged ? 5 : 6) score_select_cluster_kernel(
    const uint32_t *__restrict__ q_codes, const uint32_t *__restrict__ k_codes, long long kc_sb, long long kc_sh,
    const int32_t *__restrict__ seq_lens, int max_seq_len, const int32_t *__restrict__ k_per_seq, int k_uniform,
    int k_max, int Hq, int Hkv, int32_t *__restrict__ idx, long long idx_sb, long long idx_sh,
    int32_t *__restrict__ count, int32_t *__restrict__ hist_out, Windows win, const CodePages cp, int kv_shift,
    bool in_step) {
    constexpr int kSlice = kThreads * 8;                       // tokens of one row of a CTA: eight per lane
    extern __shared__ __align__(16) unsigned char s_sc[];      // score + 1 of this CTA's tokens (0 = no token)
    __shared__ __align__(16) uint32_t c_hist[kBins][32];       // counters [level][lane]
    __shared__ int s_hist[kBins + 3];          // this CTA's histogram, read by the whole cluster
    __shared__ int s_tot[kBins], s_bef[kBins];
    __shared__ int sh_T, sh_r, sh_gt_before, sh_eq_before;
    __shared__ int s_wcnt[kThreads / 32];
    const uint32_t rank = cluster_rank();
    const int g = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = max(min(seq_lens[b], max_seq_len), 0);
    int k = k_per_seq ? k_per_seq[b] : k_uniform;
    const WindowBounds wbd = window_bounds(win, n);   // always-kept tokens: byte kForcedByte, not counted
    const int n_forced = forced_before(wbd, n);
    const int keep_rest = max(0, min(min(k, k_max - n_forced), n - n_forced));   // heavy tokens among the others
    const int keep = n_forced + keep_rest;
    const int kvh = g >> kv_shift;   // the KV head whose signatures this unit scans
    // contiguous cache: the unit's row; paged cache: the pool from this head's offset on
    const uint32_t *row = kPaged ? k_codes + (long long)kvh * cp.head_stride : k_codes + (long long)b * kc_sb + (long long)kvh * kc_sh;
    const int32_t *table_b = kPaged ? cp.table + (long long)b * cp.bt_sb : nullptr;
    // The sequence's own length is divided over the CS CTAs (ragged batches stay balanced): Rb rows per
    // lane, a warp owns the 256*Rb tokens from wb on, a CTA kSlice*Rb; row p of a lane is
    // wb + 256 p + 8 lane .. + 7.
    const int Rb = (n + CS * kSlice - 1) / (CS * kSlice);
    const int wl = warp * 256 * Rb;                    // the warp's first token inside the CTA's slice
    const int wb = (int)rank * kSlice * Rb + wl;

    // paged: the pool words from which the lane's 8 tokens of row p are addressed by token number (pages of >= 8 tokens)
    auto row_ptr = [&](int p) -> const uint32_t * {
        if (!kPaged) return row;
        const int t = wb + p * 256 + lane * 8;
        if (cp.shift < 3 || p >= Rb || t >= n) return row;
        return row + (long long)__ldcg(table_b + (t >> cp.shift)) * cp.page_stride - (t & ~((1 << cp.shift) - 1));
    };
    auto load_row = [&](int p, const uint32_t *src_row, uint4 &lo, uint4 &hi, bool early) {
        const int t = wb + p * 256 + lane * 8;
        if (kPaged && cp.shift < 3) {   // small pages: four tokens (or one) at a time
            lo = (p < Rb && t < n) ? load_codes4_paged(cp, row, table_b, t, n) : make_uint4(0, 0, 0, 0);
            hi = (p < Rb && t + 4 < n) ? load_codes4_paged(cp, row, table_b, t + 4, n) : make_uint4(0, 0, 0, 0);
        } else if (p < Rb && t + 8 <= n) {
            const uint4 *src = reinterpret_cast<const uint4 *>(src_row + t);
            if (early) { lo = __ldg(src); hi = __ldg(src + 1); }   // L1 for the halves of a sector: 115.0 / 116.7 us, 32 sequences of 8192 - 131072
            else { lo = __ldcg(src); hi = __ldcg(src + 1); }
        } else {
            lo = (p < Rb && t < n) ? load_codes4(src_row, t, n) : make_uint4(0, 0, 0, 0);
            hi = (p < Rb && t + 4 < n) ? load_codes4(src_row, t + 4, n) : make_uint4(0, 0, 0, 0);
        }
    };
    if (kPaged && !in_step) pdl_wait();   // a block table may come from the kernel in front
    uint4 c[4];   // two rows
    const uint32_t *r0 = row_ptr(0), *r1 = row_ptr(1);
    load_row(0, r0, c[0], c[1], true);
    load_row(1, r1, c[2], c[3], true);
    // the other rows of this warp start their way from HBM to L2 now (one request per 128-byte line, no registers): the
    // loads that follow turn by turn then wait for L2 only, which is what counts when few CTAs share the SM
    for (int p = 2; p < Rb; ++p) {
        const int t = wb + p * 256 + lane * 8;
        // a page of one head is a run of 4 << shift bytes: one request per 32 tokens, or per page if those are smaller
        const int every = (kPaged && cp.shift < 5) ? (1 << (max(cp.shift, 3) - 3)) - 1 : 3;
        if ((lane & every) == 0 && t < n && !(kPaged && cp.shift < 3)) asm volatile("prefetch.global.L2 [%0];" ::"l"(row_ptr(p) + t));
    }
    if (kPaged) { r0 = row_ptr(2); r1 = row_ptr(3); }
    for (int i = tid; i < kBins * 32 / 4; i += kThreads)
        reinterpret_cast<uint4 *>(&c_hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < kBins + 3) s_hist[tid] = 0;
    pdl_launch_dependents();
    pdl_wait();
    // the signature that the ENCODE of a layer-step may just have written (slot n-1): re-read by the one lane that holds it
    {
        const int e_last = (n - 1) - wb;
        if (e_last >= 0 && e_last < 512 && e_last < 256 * Rb && ((e_last & 255) >> 3) == lane) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int t = wb + j * 256 + lane * 8;
                if (kPaged) {
                    patch_token_paged(c[2 * j], t, n - 1, cp, row, table_b);
                    patch_token_paged(c[2 * j + 1], t + 4, n - 1, cp, row, table_b);
                } else {
                    patch_token(c[2 * j], t, n - 1, row);
                    patch_token(c[2 * j + 1], t + 4, n - 1, row);
                }
            }
        }
    }
    uint32_t qc[G];
#pragma unroll
    for (int j = 0; j < G; ++j) qc[j] = __ldcg(q_codes + (long long)b * Hq + g * G + j);
    __syncthreads();

    // ---- scores (four score+1 bytes per word) and this CTA's histogram.  The counter of score s sits
    // (32 - s) rows below the lane's counter of level 32, so the address comes straight from the
    // Hamming distance 32 - s.
    const uint32_t top = (uint32_t)__cvta_generic_to_shared(&c_hist[kBins - 1][lane]);
    auto bump = [&](int ham) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(top - (uint32_t)ham * 128u) : "memory"); };
    auto hamming = [&](uint32_t code) {
        int h = __popc(code ^ qc[0]);
#pragma unroll
        for (int j = 1; j < G; ++j) h = min(h, __popc(code ^ qc[j]));
        return h;
    };
    auto score_word = [&](const uint4 &cw, int t, bool whole_row) -> uint32_t {
        const int h0 = hamming(cw.x), h1 = hamming(cw.y), h2 = hamming(cw.z), h3 = hamming(cw.w);
        // bytes 33 - h = score + 1; no byte borrows because h <= 32
        uint32_t s4 = 0x21212121u - ((uint32_t)h0 | ((uint32_t)h1 << 8) | ((uint32_t)h2 << 16) | ((uint32_t)h3 << 24));
        if (whole_row) {
            bump(h0); bump(h1); bump(h2); bump(h3);
        } else {
            const int hh[4] = {h0, h1, h2, h3};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int tt = t + e;
                if (tt >= n) s4 &= ~(0xffu << (8 * e));                                // zero byte: no token
                else if (tt < wbd.sink_end || tt >= wbd.local_begin) s4 = (s4 & ~(0xffu << (8 * e))) | (kForcedByte << (8 * e));
                else bump(hh[e]);
            }
        }
        return s4;
    };
    for (int p0 = 0; p0 < Rb; p0 += 2) {   // CTA-uniform
        if (p0 > 0) {
            load_row(p0, r0, c[0], c[1], false);
            load_row(p0 + 1, r1, c[2], c[3], false);
            if (kPaged) { r0 = row_ptr(p0 + 2); r1 = row_ptr(p0 + 3); }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int p = p0 + j, t = wb + p * 256 + lane * 8;
            if (p < Rb) {
                const bool whole_row = t + 8 <= n && t >= wbd.sink_end && t + 8 <= wbd.local_begin;
                uint2 w;
                w.x = score_word(c[2 * j], t, whole_row);
                w.y = score_word(c[2 * j + 1], t + 4, whole_row);
                *reinterpret_cast<uint2 *>(s_sc + wl + p * 256 + lane * 8) = w;
            }
        }
    }
    __syncthreads();
    // fold the counters: eight threads per level, four counters each
    for (int i = tid; i < kBins * 8; i += kThreads) {
        const uint4 v = reinterpret_cast<const uint4 *>(&c_hist[i >> 3][0])[i & 7];
        const uint32_t ssum = (v.x + v.y) + (v.z + v.w);
        if (ssum) atomicAdd(&s_hist[i >> 3], (int)ssum);
    }
    cluster_sync_all();   // every CTA's histogram is complete and visible cluster-wide

    if (tid < kBins) {
        int tot = 0, bef = 0;
#pragma unroll
        for (uint32_t r = 0; r < (uint32_t)CS; ++r) {
            const int v = ld_dsmem(&s_hist[tid], r);
            tot += v;
            if (r < rank) bef += v;
        }
        s_tot[tid] = tot;
        s_bef[tid] = bef;
    }
    // this CTA is done reading its peers' shared memory; the matching wait sits at the end of the
    // kernel, so that no CTA exits while a peer may still read its histogram
    cluster_arrive();
    __syncthreads();
    if (warp == 0) {
        int tot = s_tot[lane], bef = s_bef[lane];
        const int tot32 = s_tot[32], bef32 = s_bef[32];
        int T, r, gt_before, eq_before;
        find_threshold(tot, bef, tot32, bef32, keep_rest, lane, T, r, gt_before, eq_before);
        if (lane == 0) { sh_T = T; sh_r = r; sh_gt_before = gt_before; sh_eq_before = eq_before; }
        if (rank == 0 && hist_out) {
            hist_out[((long long)b * Hkv + g) * kBins + lane] = tot;
            if (lane == 0) hist_out[((long long)b * Hkv + g) * kBins + 32] = tot32;
        }
    }
    __syncthreads();
    const int T = sh_T, r = sh_r;
    int32_t *out = idx + (long long)b * idx_sb + (long long)g * idx_sh;
    if (rank == 0) {
        if (tid == 0) count[b * Hkv + g] = keep;
        for (int i = keep + tid; i < k_max; i += kThreads) out[i] = -1;
    }
    if (keep == 0) { cluster_wait(); return; }

    // ---- flags "S > T" / "S == T" of the lane's 8*Rb consecutive tokens (bit i = token first + i)
    // Per byte b = score + 1 (0 = no token): b + 127 - (T+1) sets bit 7 iff score > T, b + 128 - (T+1) iff
    // score >= T (no byte sum reaches 256); high_bits_to_nibble gathers the four bit-7 flags of a word.
    const uint32_t T4 = (uint32_t)(T + 1) * 0x01010101u;
    const uint32_t c_gt = 0x7f7f7f7fu - T4, c_ge = 0x80808080u - T4;
    const int first_l = wl + 8 * Rb * lane;
    uint32_t gt_lo = 0u, gt_hi = 0u, ge_lo = 0u, ge_hi = 0u;
#pragma unroll
    for (int j = 0; j < kClusterMaxRows; ++j) {
        if (j < Rb) {
            const uint2 w = *reinterpret_cast<const uint2 *>(s_sc + first_l + 8 * j);
            const uint32_t gb = high_bits_to_nibble(w.x + c_gt) | (high_bits_to_nibble(w.y + c_gt) << 4);
            const uint32_t eb = high_bits_to_nibble(w.x + c_ge) | (high_bits_to_nibble(w.y + c_ge) << 4);
            if (j < 4) { gt_lo |= gb << (8 * j); ge_lo |= eb << (8 * j); }
            else { gt_hi |= gb << (8 * (j - 4)); ge_hi |= eb << (8 * (j - 4)); }
        }
    }
    const uint32_t eq_lo = ge_lo ^ gt_lo, eq_hi = ge_hi ^ gt_hi;   // score > T implies score >= T
    const int tot_packed = (__popc(gt_lo) + __popc(gt_hi)) | ((__popc(eq_lo) + __popc(eq_hi)) << 16);
    int winc = tot_packed;   // inclusive scan over the lanes of the per-lane totals
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, winc, dd);
        if (lane >= dd) winc += v;
    }
    if (lane == 31) s_wcnt[warp] = winc;
    __syncthreads();
    // tokens before this warp's range with S > T (always-kept tokens count as such) / S == T
    int run_gt = sh_gt_before + forced_before(wbd, min((int)rank * kSlice * Rb, n)), run_eq = sh_eq_before;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        if (w < warp) { run_gt += s_wcnt[w] & 0xffff; run_eq += (int)((unsigned)s_wcnt[w] >> 16); }
    }
    if (tot_packed != 0) {
        const int excl = winc - tot_packed;
        const int q_run = run_eq + (int)((unsigned)excl >> 16), first = (int)rank * kSlice * Rb + first_l;
        int32_t *dst = out + run_gt + (excl & 0xffff) + min(q_run, r);
        dst = write_selected32(dst, first, gt_lo, eq_lo, r - q_run);
        write_selected32(dst, first + 32, gt_hi, eq_hi, r - q_run - __popc(eq_lo));
    }
    cluster_wait();
}

template <int G, int CS, bool kPaged, int kThreads = kScanThreads>
static cudaError_t launch_cluster_t(int rows, int B, int Hq, int Hkv, const uint32_t *q_codes, const uint32_t *k_codes,
                                    long long kc_sb, long long kc_sh, const int32_t *seq_lens,
                                    const int32_t *k_per_seq, int k_uniform, int max_seq_len, int k_max, int32_t *idx,
                                    long long idx_sb, long long idx_sh, int32_t *count, int32_t *hist_out,
                                    cudaStream_t st, Windows win, CodePages cp, int kv_shift, bool in_step) {
    static bool opted[64] = {};   // opt in to the padded shared-memory sizes once per device
    {
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev >= 0 && dev < 64 && !opted[dev]) {
            cudaError_t e = cudaFuncSetAttribute(score_select_cluster_kernel<G, CS, kPaged, kThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
            if (e != cudaSuccess) return e;
            opted[dev] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS, Hkv, B);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = (size_t)rows * kThreads * 8;   // one score byte per token of the CTA's slice (<= 16 KB, 32 KB with 512 threads)
    {
        // Launched behind another kernel, the CTAs land wherever room appears first, and an SM that takes six of them
        // while others hold two sets the kernel's time (the population-count unit is shared by the CTAs of an SM).
        // When the grid needs fewer than six CTAs per SM, shared memory is requested as if each CTA needed a whole
        // share of the SM, so that no SM can take more than ceil(CTAs / SMs).  Clusters of 4 or 8 need some slack
        // for that (all CTAs of a cluster are placed together): without it the cap only delays their placement.
        const int n_ctas = CS * Hkv * B, n_sm = sm_count();
        const int cap = (n_ctas + n_sm - 1) / n_sm;   // CTAs per SM
        const bool slack = CS == 2 || 2 * (cap * n_sm - n_ctas) >= n_sm;
        if (kThreads == kScanThreads && n_ctas > n_sm && cap < (kPaged ? 5 : 6) && slack) {
            static size_t pad[64][6] = {};   // per device and cap: the least dynamic shared memory with which only `cap` CTAs fit
            int dev = 0;
            cudaGetDevice(&dev);
            if (dev < 0 || dev >= 64) dev = 0;
            if (!pad[dev][cap]) {
                size_t found = 0;
                for (size_t kb = 8; kb <= 100 && !found; ++kb) {
                    int occ = 0;
                    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, score_select_cluster_kernel<G, CS, kPaged, kThreads>, kThreads, kb * 1024) != cudaSuccess) {
                        cudaGetLastError();   // no cap, and no error of this query behind the launch
                        break;
                    }
                    if (occ <= cap) found = kb * 1024;
                }
                pad[dev][cap] = found ? found : 1;
            }
            if (pad[dev][cap] > cfg.dynamicSmemBytes) cfg.dynamicSmemBytes = pad[dev][cap];
        }
    }
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, score_select_cluster_kernel<G, CS, kPaged, kThreads>, q_codes, k_codes, kc_sb, kc_sh,
                                       seq_lens, max_seq_len, k_per_seq, k_uniform, k_max, Hq, Hkv, idx, idx_sb, idx_sh,
                                       count, hist_out, win, cp, kv_shift, in_step);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

// ------------------------------------------------------------------ several units per cluster
//
// As many clusters of CS = 1, 2, 4 or 8 CTAs (512 threads, two per SM) as are resident at once share the units out among them: by
// falling length, forth and back, so that ragged batches end together.  A cluster takes up to eight units at a time through every
// phase: scores of all of them, one exchange of histograms, thresholds, lists.  The fixed part (launch, first rows, barriers,
// thresholds: 7 us) is thus paid once, not in every wave of one-unit clusters, no SM is left with more CTAs than another, and the
// bytes of a sequence of up to 750000 tokens fit (96 KB of counters and score bytes per CTA), so the long ones need no second kernel.
//
// Bound: the population count (groups of 4 and 8: 14.4 us for 512 units of 32768 tokens and 4 heads, 18 - 23 us measured for the
// scoring), HBM for groups of 1.  Alone, against the one-unit clusters (us): 32 sequences of 8192 - 131072 tokens 41.6 -> 35.3, 24 of
// 2000 - 65536 18.0 -> 15.1, 64 of 2000 - 32768 24.3 -> 19.3, 48 of 8000 - 65536 in groups of 2 29.0 -> 22.0.
//  * Reading: the signatures are asked into L2 before the launch wait and read behind it, two rows of 128 tokens per warp ahead of
//    the scoring.
//  * Score bytes: 32 consecutive tokens are 8 words, and byte e of word j belongs to token 8 e + j.  Stored byte by byte in that order
//    (no packing; the 32 bytes of an instruction lie in 8 banks), eight words give the 32 flags "above / at the threshold" of their
//    tokens, in token order, with an add, a shift and one three-input operation per word.
//  * Writing: a lane takes whole groups of 32 tokens, works out which of them are selected and visits only those.
// Tried: equal shares of all rows whatever the unit boundaries (a cooperative launch, units settled by counters): balanced to the
// row, but such a launch waits for the kernel in front to drain and pays 15 us of fixed parts (16 units of 32768: 19.8 against 11.9);
// the 32 x 32 bits of products on the tensor cores (kind::mxf4, signatures spread over tensor memory): 28 us against 20 us for the
// same tokens counted with popc, the stores into tensor memory alone take 10.

// The scores (bytes of s_sc) and flags of 32 consecutive tokens, in token order: bit i = token i of the group.  gt: score above T.
__device__ __forceinline__ void group_flags(const unsigned char *group, uint32_t c_gt, uint32_t c_ge, uint32_t &gt, uint32_t &ge) {
    const uint4 lo = reinterpret_cast<const uint4 *>(group)[0], hi = reinterpret_cast<const uint4 *>(group)[1];
    const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    gt = 0u;
    ge = 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        gt = (gt >> 1) | ((w[j] + c_gt) & 0x80808080u);
        ge = (ge >> 1) | ((w[j] + c_ge) & 0x80808080u);
    }
}

// One unit of a batch, as every CTA of the cluster sees it.
struct BatchUnit {
    int b, g, n, keep, keep_rest;   // sequence, head of the unit, tokens; list length, and the heavy tokens among it
    int row0, rows;                 // this CTA's rows of 128 tokens
    int off, tab;                   // its score bytes and, where staged, its entries of the block table in the pool
    WindowBounds win;
    int T, r, gt_before, eq_before;
};

constexpr int kSelThreads = 512, kSelWarps = kSelThreads / 32;
constexpr int kSelUnits = 8;                          // units of a batch
constexpr int kSelHist = kBins * 32 * 4;              // bytes of a unit's counters [level][lane]
constexpr int kSelSort = 512;                         // sequences that are dealt out by length: at most one per thread
constexpr int kSelStepBits = 6;                       // more than 64 sequences: by this many top bits of the longest length
static_assert(kSelSort <= kSelThreads && (1 << kSelStepBits) * kSelWarps == 2 * kSelThreads, "a sequence and two counts per thread");
constexpr int kSelPool = 96 * 1024;                   // counters, score bytes and table entries of a batch: two CTAs per SM

// Bytes of a slice's entries of the block table (one more where the slice begins inside a page).
__host__ __device__ constexpr int batch_table_bytes(int rows, int shift) { return ((rows * 128 >> shift) + 5) / 4 * 16; }

// Every cluster of the grid has a unit (launch_batch_t).
// kPaged: the signatures lie in a pool behind a block table, in pages of 16 tokens or more (smaller ones lose, batch_cluster_size).
// They hold a lane's 4 tokens in one piece, so a row costs one table entry per lane (neighbouring lanes share it) and the same
// 16-byte load.
template <int G, int CS, bool kPaged>
__global__ void __launch_bounds__(kSelThreads, 2) score_select_batch_kernel(
    const uint32_t *__restrict__ q_codes, const uint32_t *__restrict__ k_codes, long long kc_sb, long long kc_sh,
    const int32_t *__restrict__ seq_lens, int max_seq_len, const int32_t *__restrict__ k_per_seq, int k_uniform,
    int k_max, int B, int Hq, int Hkv, int32_t *__restrict__ idx, long long idx_sb, long long idx_sh,
    int32_t *__restrict__ count, int32_t *__restrict__ hist_out, Windows win, const CodePages cp, int kv_shift,
    bool in_step, bool staged) {
    extern __shared__ __align__(128) unsigned char pool[];     // counters of the batch's units, then their score bytes
    __shared__ int s_all[CS][kSelUnits][kBins + 3];            // histograms of the cluster's CTAs
    __shared__ BatchUnit s_u[kSelUnits];
    __shared__ uint32_t s_nq[kSelUnits][G];
    __shared__ uint32_t s_wcnt[kSelWarps];
    __shared__ int s_len[kSelSort], s_k[kSelSort];
    __shared__ uint16_t s_perm[kSelSort];
    __shared__ int s_units;
    const int rank = CS > 1 ? (int)cluster_rank() : 0;
    if (CS > 1) cluster_arrive();                              // its wait stands in front of the first remote store
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = gridDim.x / CS, cl = blockIdx.x / CS, n_units = B * Hkv;
    auto len_of = [&](int b) -> int { return max(min(seq_lens[b], max_seq_len), 0); };
    auto budget_of = [&](int b) -> int { return k_per_seq ? k_per_seq[b] : k_uniform; };

    // ---- the cluster's units: all units by falling length, dealt out to the clusters forth and back
    const bool sorted = B <= kSelSort;
    if (B <= 64) {   // by the warp that needs them
        if (warp == 0) {
            const int l0 = lane < B ? len_of(lane) : -1, l1 = lane + 32 < B ? len_of(lane + 32) : -1;
            const int k0 = lane < B ? budget_of(lane) : 0, k1 = lane + 32 < B ? budget_of(lane + 32) : 0;
            int r0 = 0, r1 = 0;
#pragma unroll 8
            for (int j = 0; j < min(B, 32); ++j) {
                const int v = __shfl_sync(0xffffffffu, l0, j);
                r0 += (v > l0 || (v == l0 && j < lane)) ? 1 : 0;
                r1 += v >= l1 ? 1 : 0;
            }
#pragma unroll 8
            for (int j = 0; j < B - 32; ++j) {
                const int v = __shfl_sync(0xffffffffu, l1, j);
                r0 += v > l0 ? 1 : 0;
                r1 += (v > l1 || (v == l1 && j < lane)) ? 1 : 0;
            }
            if (lane < B) { s_perm[r0] = (uint16_t)lane; s_len[lane] = l0; s_k[lane] = k0; }
            if (lane + 32 < B) { s_perm[r1] = (uint16_t)(lane + 32); s_len[lane + 32] = l1; s_k[lane + 32] = k1; }
            __syncwarp();
        }
    } else if (sorted) {
        // More of them: counting sort by the top bits of the length, one sequence per thread.  The counts [step][warp] lie in the
        // pool, which nothing else uses yet.  Every CTA sorts all lengths for itself, and ranks by comparing every pair cost up to
        // 15 us (whole steps, 2 heads, 1500 tokens: 256 sequences 32.9 us, now 29.2; 512 62.8, 48.1).
        int *at = reinterpret_cast<int *>(pool);
        const int mine = tid < B ? len_of(tid) : -1;
        if (tid < B) { s_len[tid] = mine; s_k[tid] = budget_of(tid); }
        reinterpret_cast<int2 *>(at)[tid] = make_int2(0, 0);
        const int longest_here = __reduce_max_sync(0xffffffffu, mine);
        if (lane == 0) s_wcnt[warp] = (uint32_t)max(longest_here, 0);
        __syncthreads();
        uint32_t longest = 0u;
#pragma unroll
        for (int w = 0; w < kSelWarps; ++w) longest = max(longest, s_wcnt[w]);
        const int shift = max(0, 32 - kSelStepBits - __clz((int)longest));   // longest >> shift is the largest of 64 steps, or less
        const int step = tid < B ? (1 << kSelStepBits) - 1 - (mine >> shift) : 1 << kSelStepBits;   // the longest first
        const uint32_t same = __match_any_sync(0xffffffffu, step);
        const int before = __popc(same & ((1u << lane) - 1u));
        if (tid < B && before == 0) at[step * kSelWarps + warp] = __popc(same);
        __syncthreads();
        const int2 c = reinterpret_cast<const int2 *>(at)[tid];
        int sum = c.x + c.y;
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, sum, dd);
            if (lane >= dd) sum += v;
        }
        if (lane == 31) s_wcnt[warp] = (uint32_t)sum;
        __syncthreads();
        sum -= c.x + c.y;
        for (int w = 0; w < warp; ++w) sum += (int)s_wcnt[w];
        reinterpret_cast<int2 *>(at)[tid] = make_int2(sum, sum + c.x);
        __syncthreads();
        if (tid < B) s_perm[at[step * kSelWarps + warp] + before] = (uint16_t)tid;
        __syncthreads();
    }
    auto unit_of = [&](int j) -> int { return j * C + ((j & 1) ? C - 1 - cl : cl); };   // the cluster's j-th unit

    bool first_batch = true;
    for (int j0 = 0;;) {
        // ---- the batch: as many of the next units as fit the pool
        if (warp == 0) {
            BatchUnit u = {};
            const int at = lane < kSelUnits ? unit_of(j0 + lane) : n_units;
            int need = 1 << 28;
            if (at < n_units) {
                const int sb = at / Hkv;
                u.b = sorted ? s_perm[sb] : sb;
                u.g = at - sb * Hkv;
                u.n = sorted ? s_len[u.b] : len_of(u.b);
                u.win = window_bounds(win, u.n);
                const int forced = forced_before(u.win, u.n), k = sorted ? s_k[u.b] : budget_of(u.b);
                u.keep_rest = max(0, min(min(k, k_max - forced), u.n - forced));
                u.keep = forced + u.keep_rest;
                const int rows = (u.n + 127) >> 7;
                u.row0 = rows * rank / CS;
                u.rows = rows * (rank + 1) / CS - u.row0;
                need = kSelHist + (rows + CS - 1) / CS * 128;
                if (kPaged && staged) need += batch_table_bytes((rows + CS - 1) / CS, cp.shift);
                u.tab = kSelHist + (rows + CS - 1) / CS * 128;
            }
            int inc = need;
#pragma unroll
            for (int dd = 1; dd < kSelUnits; dd <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, dd);
                if (lane >= dd) inc = min(inc + v, 1 << 28);
            }
            const int U = __popc(__ballot_sync(0xffffffffu, at < n_units && inc <= kSelPool));
            u.off = inc - need - lane * kSelHist + U * kSelHist;
            u.tab += u.off - kSelHist;
            if (lane < U) s_u[lane] = u;
            if (lane == 0) s_units = U;
        }
        __syncthreads();
        const int U = s_units;
        if (U == 0) break;   // cluster-uniform
        j0 += U;

        // ---- the batch's signatures start their way from HBM to L2 (one request per 128-byte line), its part of the block table
        // into shared memory
        auto in_page = [&](const uint32_t *row, int page, int t) -> const uint32_t * {   // (the launcher sees to it that the stride fits)
            return row + (long long)page * (int)cp.page_stride + (t & ((1 << cp.shift) - 1));
        };
        auto row_of = [&](const BatchUnit &u) -> const uint32_t * {
            const int kvh = u.g >> kv_shift;   // the KV head whose signatures this unit scans
            return kPaged ? k_codes + (long long)kvh * cp.head_stride : k_codes + (long long)u.b * kc_sb + (long long)kvh * kc_sh;
        };
        if (kPaged && !in_step && first_batch) pdl_wait();   // a block table may come from the kernel in front
        for (int i = 0; i < U; ++i) {
            const BatchUnit &u = s_u[i];
            const uint32_t *row = row_of(u);
            const int first = u.row0 * 128, end = min(u.n, (u.row0 + u.rows) * 128);
            if (kPaged) {
                // a page of one head is one run of bytes: a request per page of up to 32 tokens, or per 32 tokens of a larger one
                // (a thread per page, whatever its size, left few threads with all requests of a slice: 24 sequences of 8192 - 65536 in
                // pages of 65536, whole step 66.8 us, now 60.6, 48 of 4096 - 32768 in pages of 16384 67.9, now 63.9)
                const int32_t *table = cp.table + (long long)u.b * cp.bt_sb;
                const int every = min(cp.shift, 5), e0 = first >> cp.shift;
                int32_t *tab = reinterpret_cast<int32_t *>(pool + u.tab);
                for (int t = first + (tid << every); t < end; t += kSelThreads << every) {   // first: a multiple of 128
                    const int e = t >> cp.shift, page = __ldcg(table + e);
                    if (staged && (t == first || t == e << cp.shift)) tab[e - e0] = page;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(in_page(row, page, t)));
                }
            } else {
                for (int t = first + tid * 32; t < end; t += kSelThreads * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + t));
            }
        }
        for (int i = tid; i < U * (kSelHist / 16); i += kSelThreads) reinterpret_cast<uint4 *>(pool)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (first_batch) {
            pdl_launch_dependents();
            pdl_wait();
        }
        if (tid < U * G) {   // popc(code ^ ~q) = 32 - Hamming distance
            const BatchUnit &u = s_u[tid / G];
            s_nq[tid / G][tid % G] = ~__ldcg(q_codes + (long long)u.b * Hq + u.g * G + tid % G);
        }
        __syncthreads();

        // ---- scores and this CTA's histograms.  A warp walks its rows of all the units, two at a time; the next two (of the next
        // unit if need be) are on their way while it scores
        {
            struct Rows { const uint32_t *row; const int32_t *table; int i, p, p_end, tok, n, e0; } at;   // tok: the lane's token of row 0
            at.i = -1;
            at.p = at.p_end = at.tok = at.n = at.e0 = 0;
            at.row = nullptr;
            at.table = nullptr;
            auto settle = [&]() {   // on to the next unit in which this warp has rows
                while (at.p >= at.p_end && ++at.i < U) {
                    const BatchUnit &u = s_u[at.i];
                    at.p = u.rows * warp / kSelWarps;
                    at.p_end = u.rows * (warp + 1) / kSelWarps;
                    at.tok = u.row0 * 128 + lane * 4;
                    at.n = u.n;
                    at.row = row_of(u);
                    if (kPaged) {
                        at.table = staged ? reinterpret_cast<const int32_t *>(pool + u.tab) : cp.table + (long long)u.b * cp.bt_sb;
                        at.e0 = staged ? u.row0 * 128 >> cp.shift : 0;
                    }
                }
            };
            auto load = [&](uint4 (&c)[2]) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int t = at.tok + (at.p + j) * 128;
                    c[j] = make_uint4(0u, 0u, 0u, 0u);
                    if (at.p + j < at.p_end && t < at.n) {
                        if (kPaged) {
                            const int32_t *entry = at.table + ((t >> cp.shift) - at.e0);   // in shared memory if staged
                            c[j] = load_codes4(in_page(at.row, staged ? *entry : __ldcg(entry), t) - t, t, at.n);
                        } else {
                            c[j] = load_codes4(at.row, t, at.n);
                        }
                    }
                }
            };
            uint4 c[2], nxt[2];
            settle();
            if (at.i < U) load(c);
            int cur = -1, n = 0, sink_end = 0, local_begin = 0;
            uint32_t base0 = 0u, nq[G];
            unsigned char *sc_lane = pool;
#pragma unroll
            for (int j = 0; j < G; ++j) nq[j] = 0u;
            auto bump = [&](int s) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(base0 + (uint32_t)s * 128u) : "memory"); };
            auto score = [&](uint32_t code) {
                int s = __popc(code ^ nq[0]);
#pragma unroll
                for (int j = 1; j < G; ++j) s = max(s, __popc(code ^ nq[j]));
                return s;
            };
            while (at.i < U) {   // warp-uniform
                const int i = at.i, p0 = at.p, p_end = at.p_end, tok = at.tok;
                at.p += 2;
                settle();
                if (at.i < U) load(nxt);
                if (i != cur) {
                    const BatchUnit &u = s_u[i];
                    cur = i;
                    n = u.n;
                    sink_end = u.win.sink_end;
                    local_begin = u.win.local_begin;
                    base0 = (uint32_t)__cvta_generic_to_shared(pool + i * kSelHist + lane * 4);
                    // token e of the lane's four is token 8 x + y of its group of 32 with x = (lane & 7) >> 1, y = 4 (lane & 1) + e
                    sc_lane = pool + u.off + (lane >> 3) * 32 + (lane & 1) * 16 + ((lane & 7) >> 1);
#pragma unroll
                    for (int j = 0; j < G; ++j) nq[j] = s_nq[i][j];
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int p = p0 + j, t = tok + p * 128;
                    if (p < p_end) {
                        const int s[4] = {score(c[j].x), score(c[j].y), score(c[j].z), score(c[j].w)};
                        unsigned char *dst = sc_lane + p * 128;
                        if (t + 4 <= n && t >= sink_end && t + 4 <= local_begin) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) { bump(s[e]); dst[e * 4] = (unsigned char)s[e]; }
                        } else {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const bool forced = t + e < sink_end || t + e >= local_begin;
                                if (t + e < n) {   // bytes of tokens past the end are never looked at
                                    if (!forced) bump(s[e]);
                                    dst[e * 4] = (unsigned char)(forced ? (int)kForcedByte : s[e]);
                                }
                            }
                        }
                    }
                }
                c[0] = nxt[0];
                c[1] = nxt[1];
            }
        }
        __syncthreads();
        // ---- fold the counters: one level per warp at a time; lane r < CS hands the sum to CTA r
        if (CS > 1) cluster_wait();   // every CTA of the cluster runs, and is done with the last batch's histograms
        for (int l = warp; l < U * kBins; l += kSelWarps) {
            const int sum = (int)__reduce_add_sync(0xffffffffu, reinterpret_cast<const uint32_t *>(pool)[l * 32 + lane]);
            const int i = l / kBins;
            if (CS == 1) { if (lane == 0) s_all[0][i][l - i * kBins] = sum; }
            else if (lane < CS) st_dsmem(&s_all[rank][i][l - i * kBins], (uint32_t)lane, sum);
        }
        if (CS > 1) cluster_sync_all();   // every CTA's histograms have arrived
        else __syncthreads();
        if (warp < U) {
            BatchUnit &u = s_u[warp];
            int tot = 0, bef = 0, tot32 = 0, bef32 = 0;
#pragma unroll
            for (int q = 0; q < CS; ++q) {
                const int v = s_all[q][warp][lane], v32 = s_all[q][warp][32];
                tot += v;
                tot32 += v32;
                if (q < rank) { bef += v; bef32 += v32; }
            }
            int T, r, gt_before, eq_before;
            find_threshold(tot, bef, tot32, bef32, u.keep_rest, lane, T, r, gt_before, eq_before);
            const int unit = u.b * Hkv + u.g;
            if (lane == 0) {
                u.T = T;
                u.r = r;
                u.gt_before = gt_before + forced_before(u.win, min(u.row0 * 128, u.n));   // always-kept tokens count as above
                u.eq_before = eq_before;
                if (rank == 0) count[unit] = u.keep;
            }
            if (rank == 0 && hist_out) {
                hist_out[(long long)unit * kBins + lane] = tot;
                if (lane == 0) hist_out[(long long)unit * kBins + 32] = tot32;
            }
        }
        __syncthreads();
        first_batch = false;
        const bool more = unit_of(j0) < n_units;   // cluster-uniform
        if (CS > 1 && more) cluster_arrive();      // done with the histograms

        // ---- list entries.  W warps per unit, each takes a contiguous share of the CTA's groups of 32 tokens.
        // Flags "S > T" / "S >= T", kept where the group's scores were: a byte s + 127 - T has bit 7 set iff s > T, s + 128 - T
        // iff s >= T (T <= 33, and no byte of a token before the end carries into the next).
        const int W = U > 4 ? kSelWarps / 8 : U > 2 ? kSelWarps / 4 : kSelWarps / U, i = warp / W;
        const bool busy = i < U;
        const BatchUnit &u = s_u[busy ? i : 0];
        const int part = warp - i * W, first_tok = u.row0 * 128, n = u.n, keep = u.keep, r = u.r;
        const int n_groups = busy ? max(0, min(4 * u.rows, (n - first_tok + 31) >> 5)) : 0;
        const int q_lo = n_groups * part / W, q_n = n_groups * (part + 1) / W - q_lo;   // the warp's groups
        unsigned char *sc = pool + u.off + q_lo * 32;
        uint2 *flags = reinterpret_cast<uint2 *>(sc);   // of the groups so far, where the scores of the first quarter of them were
        int32_t *out = idx + (long long)u.b * idx_sb + (long long)u.g * idx_sh;
        if (busy) {
            const uint32_t c_gt = 0x7f7f7f7fu - (uint32_t)u.T * 0x01010101u, c_ge = 0x80808080u - (uint32_t)u.T * 0x01010101u;
            uint32_t cnt = 0u;   // flags of this lane's groups: S > T in the low half, S == T in the high half
            for (int q0 = 0; q0 < q_n; q0 += 32) {   // warp-uniform
                const int q = q0 + lane;
                uint32_t gt = 0u, ge = 0u;
                if (q < q_n) {
                    group_flags(sc + q * 32, c_gt, c_ge, gt, ge);
                    const int left = n - (first_tok + (q_lo + q) * 32);
                    if (left < 32) { const uint32_t live = (1u << left) - 1u; gt &= live; ge &= live; }
                }
                __syncwarp();   // the scores are read before flags overwrite them
                if (q < q_n) flags[q] = make_uint2(gt, ge ^ gt);   // score > T implies score >= T
                cnt += (uint32_t)__popc(gt) + ((uint32_t)__popc(ge ^ gt) << 16);
            }
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            if (lane == 0) s_wcnt[warp] = cnt;
            for (int q = keep + (rank * W + part) * 32 + lane; q < k_max; q += CS * W * 32) out[q] = -1;
        }
        __syncthreads();
        if (busy && keep > 0) {
            // a lane takes `per` consecutive groups: one scan over the lanes for all of the warp's groups
            const int per = (q_n + 31) >> 5, q_first = min(lane * per, q_n), q_last = min(q_first + per, q_n);
            int n_gt = 0, n_eq = 0;
            for (int q = q_first; q < q_last; ++q) { const uint2 f = flags[q]; n_gt += __popc(f.x); n_eq += __popc(f.y); }
            int inc = n_gt | (n_eq << 16);
#pragma unroll
            for (int dd = 1; dd < 32; dd <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, dd);
                if (lane >= dd) inc += v;
            }
            // tokens before this lane's groups with S > T / S == T
            int run_gt = u.gt_before + (inc & 0xffff) - n_gt, run_eq = u.eq_before + (int)((unsigned)inc >> 16) - n_eq;
            for (int w = i * W; w < warp; ++w) { run_gt += (int)(s_wcnt[w] & 0xffffu); run_eq += (int)(s_wcnt[w] >> 16); }
            int32_t *dst = out + run_gt + min(run_eq, r);
            int room = r - run_eq;   // tokens at the threshold that are still wanted
            for (int q = q_first; q < q_last; ++q) {
                const uint2 f = flags[q];
                const int here = __popc(f.y), first = first_tok + (q_lo + q) * 32;
                dst = write_selected32(dst, first, f.x, f.y, room);
                room -= here;
            }
        }
        if (!more) break;
        __syncthreads();   // the pool and the descriptors are reused
    }
}

// The most clusters of a variant that are resident at once on the current device (0: the query failed).
template <int G, int CS, bool kPaged>
static int resident_batch_clusters() {
    static int cached[64] = {};   // 0: not asked yet
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 0;
    if (!cached[dev]) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CS);
        cfg.blockDim = dim3(kSelThreads);
        cfg.dynamicSmemBytes = kSelPool;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cached[dev] = ask_resident_clusters(score_select_batch_kernel<G, CS, kPaged>, cfg, kSelPool);
    }
    return cached[dev];
}

template <int G, int CS, bool kPaged>
static cudaError_t launch_batch_t(int B, int Hq, int Hkv, const uint32_t *q_codes, const uint32_t *k_codes,
                                    long long kc_sb, long long kc_sh, const int32_t *seq_lens,
                                    const int32_t *k_per_seq, int k_uniform, int max_seq_len, int k_max, int32_t *idx,
                                    long long idx_sb, long long idx_sh, int32_t *count, int32_t *hist_out,
                                    cudaStream_t st, Windows win, CodePages cp, int kv_shift, bool in_step) {
    const int rows = ((max_seq_len + 127) / 128 + CS - 1) / CS;   // of the longest slice
    const bool staged = kPaged && kSelHist + rows * 128 + batch_table_bytes(rows, cp.shift) <= kSelPool;
    const int most = resident_batch_clusters<G, CS, kPaged>();
    if (most <= 0) return cudaErrorInvalidConfiguration;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(CS * min((long long)most, (long long)B * Hkv)));
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = kSelPool;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CS;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CS > 1 ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, score_select_batch_kernel<G, CS, kPaged>, q_codes, k_codes, kc_sb, kc_sh,
                                       seq_lens, max_seq_len, k_per_seq, k_uniform, k_max, B, Hq, Hkv, idx, idx_sb, idx_sh,
                                       count, hist_out, win, cp, kv_shift, in_step, staged);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

// CTAs per cluster of the batch kernel, 0: one of the other kernels.  Those give every unit a cluster of its own, pay its fixed part
// of 7 us in every wave and size the cluster for max_seq_len, and beyond 131072 tokens they are two kernels with the scores in
// global memory between them; but their CTAs leave one by one and make room for GATHER-ATT, and equal units fill them evenly.  So
// this kernel wins where lengths differ, where max_seq_len is a capacity and where sequences are short.  The lengths themselves are
// on the device.  The lines are in clusters resident at once: 296 of 1, 148 of 2, 71 of 4, 33 of 8 on 148 SMs.
// Gain of this kernel over the others in a whole step in percent, with lengths from n / s to n, for four spreads s: 1, 1.1 - 1.3,
// 2 - 4, 8 - 16; 8 heads in groups of 4 where nothing else is said, "480 of 1000" = 480 units with n = 1000:
//  * up to 10240 tokens, one CTA, whatever the lengths: 480 of 1000 +5 +6 +5 +5, of 5000 +5 +3 +2 +3; 1024 of 5000 +8 +7 +5 +5;
//    2048 of 1000 +11 +13 +14 +15; but 384 of 3000 -5 -5 -5 -3.  Longer, or in larger groups, only where the CTAs are filled
//    evenly: 512 of 8000 +1 0 +2 +3, 560 of 10240 +1 +2 +5 +4, 1024 of 10240 +1 +4 +4 +4, but 464 of 8000 -2 0 +2 +1, 640 of 8192 -2 0 +4 +5;
//    in groups of 8, 512 of 4000 0 and +3 (s = 1, 4), of 8192 -3 and +2.  Lists of up to 768 entries: longer ones take GATHER-ATT
//    long enough for its early CTAs to count (n / k = 2, 4, 8, 16, 32, s = 1: 512 of 8192 -2 -1 0 0 +1, in pages of 16 -3 -6 -5 -2 0, of 1500
//    +1 +5 +8 +9 +10; 1024 of 8192 in pages -2 -5 -3 +1 +3)
//  * up to 32768, where clusters of 2 hold a unit, never: 512 of 32768 -6 -5 -1 +3, 592 of 32768 -3 -2 0 +4, 384 of 16000 -4 -3 -1 +3.
//    Except lists per query head of up to 1024 entries (append, queries, lists, attention): 464 of 16000 +2 +3 +4 +4, 512 of 32768
//    0 +3 +2 +5, but 1024 of 24000 -6 -2 0 +4, and with 2048 entries 512 of 32768 -4 and +3 (s = 1, 4)
//  * beyond, clusters of 2, and only with one budget per sequence, the one sign of unequal lengths that the host has.  Up to 65536,
//    contiguous: 256 of 50000 +2 -1 0 +3, 296 of 65536 -1 -2 0 +2, but 192 of 50000 -5 -4 0 +3, 384 of 65536 -8 -6 -2 +2; in pages of
//    16: 192 of 50000 +1 0 +2 +5, 296 of 65536 0 +1 +2 +3, 384 of 50000 -5 -3 +1 +4.  Up to 131072: 192 of 100000 -8 -3 +1 +4, 256 of
//    100000 -4 -3 +3 +8, 296 of 100000 0 0 +4 +9.  Long units of one length are given away here (256 of 131072 tokens are 17 GB of K
//    and V in a layer) for wide ranges and for capacities: n = 131072, but lengths of 500 - 2000 and of 4000 - 16000: 192 units +12
//    and +9, 256 +21 and +18, 512 +31 and +21.  In pages of 16, 128 of 100000 +4 +4 +3 -2, but 104 of 131072 -1 0 -2 -9, 160 of 100000
//    -14 -12 +2 +4.  Clusters of 4: 68 of 131072 in groups of 1, 4 and 8 +11, +8, +16 (s = 1) and +1, +3, +6 (s = 16), 64 of 100000
//    +1 +1 -3 +1, but 40 of 131072 -9 -9 -7 -8, 56 -3 -2 -3 -3
//  * beyond 131072, three spreads, 1, 1.3 and 8.  From 104 units on the smallest cluster that holds a unit, as sequences are short of
//    such a capacity: 120 of 140000 +9 +13 +16, 192 of 140000 +13 +18 +31, 136 of 300000 +11 +15 +28; lengths of 500 - 2000 in 200000
//    with clusters of 4 -21 with 128 units, -34 with 512, hence the end at 3 units a cluster.  Fewer units: the size whose fullest
//    cluster has the least to do, unless that is twice the even share (36 of 300000 -5 -3 +4; 32 +2 +5 +11, 40 +1 +3 +10, 56 +8 +10
//    +11), or 1.6 times in groups of 8 (40 of 300000 -6 -3 -1)
//  * pages of fewer than 16 tokens never: 10 sequences of 10000 - 110000 in pages of 1 75.8 us per step, 98.0 here.
template <int G>
static int batch_cluster_size(long long units, int max_seq_len, int k_max, bool budgets, bool per_head, const CodePages &cp) {
    const bool paged = cp.table != nullptr;
    if (units < 24 || units > 65536 || (paged && (cp.shift < 4 || cp.page_stride != (int)cp.page_stride))) return 0;
    const long long n = max_seq_len;
    auto resident = [&](int cs) -> long long {   // 0: the query failed, and one of the other kernels takes the call
        if (cs == 1) return paged ? resident_batch_clusters<G, 1, true>() : resident_batch_clusters<G, 1, false>();
        if (cs == 2) return paged ? resident_batch_clusters<G, 2, true>() : resident_batch_clusters<G, 2, false>();
        if (cs == 4) return paged ? resident_batch_clusters<G, 4, true>() : resident_batch_clusters<G, 4, false>();
        return paged ? resident_batch_clusters<G, 8, true>() : resident_batch_clusters<G, 8, false>();
    };
    const long long c1 = resident(1), c2 = resident(2), c4 = resident(4);
    if (c1 <= 0 || c2 <= 0 || c4 <= 0) return 0;
    const bool many = 9 * units >= 14 * c1;   // for one CTA a unit
    if (n <= 10240) {
        const long long fullest = (units + c1 - 1) / c1;
        const bool even = 6 * units >= 5 * fullest * c1;
        return many && k_max <= 768 && (n * G <= 20480 || (even && n * G <= 40960)) ? 1 : 0;
    }
    if (n <= kClusterMaxSeq) {
        if (!budgets) return 0;
        if (n <= 32768) return per_head && many && units <= 2 * c1 && k_max <= 1024 ? 1 : 0;
        if (n <= 65536) return (paged ? 5 * units >= 6 * c2 : 3 * units >= 5 * c2 && units <= 2 * c2) ? 2 : 0;
        if (5 * units >= 6 * c2 || (paged && 6 * units >= 5 * c2 && units <= c2)) return 2;
        return n > 98304 && 10 * units >= 9 * c4 && units <= c4 ? 4 : 0;
    }
    if (large_clusters(units, max_seq_len)) return 0;
    auto fits = [&](int cs) { return kSelHist + ((n + 127) / 128 + cs - 1) / cs * 128 <= kSelPool; };
    if (10 * units >= 7 * c2) {
        if (fits(2)) return 2;
        return units > 3 * c4 ? 0 : fits(4) ? 4 : fits(8) && resident(8) > 0 ? 8 : 0;
    }
    int best = 0;
    long long best_cost = 0;   // units of the fullest cluster, in eighths per CTA
    for (int cs = 2; cs <= 8; cs *= 2) {
        const long long c = fits(cs) ? resident(cs) : 0;
        if (c <= 0) continue;
        const long long cost = (units + c - 1) / c * (8 / cs);
        if (!best || cost < best_cost) { best = cs; best_cost = cost; }
    }
    return 5 * best_cost * c1 <= (G == 8 ? 64 : 80) * units ? best : 0;
}

template <int G>
static cudaError_t launch_g(int B, int Hq, int Hkv, const uint32_t *q_codes, const uint32_t *k_codes,
                            long long kc_sb, long long kc_sh, const int32_t *seq_lens, const int32_t *k_per_seq,
                            int k_uniform, int max_seq_len, int k_max, int32_t *idx, long long idx_sb,
                            long long idx_sh, int32_t *count, int32_t *hist_out, int32_t *ws_hist,
                            unsigned char *ws_scores, cudaStream_t st, Windows win, CodePages cp, int row_shift, bool in_step) {
    {
        const int kv_shift = row_shift < 0 ? 0 : row_shift;
#define HA_BATCH(CSZ) case CSZ: return cp.table ? launch_batch_t<G, CSZ, true>(HA_BATCH_ARGS) : launch_batch_t<G, CSZ, false>(HA_BATCH_ARGS)
#define HA_BATCH_ARGS B, Hq, Hkv, q_codes, k_codes, kc_sb, kc_sh, seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, \
                      idx_sb, idx_sh, count, hist_out, st, win, cp, kv_shift, in_step
        switch (batch_cluster_size<G>((long long)B * Hkv, max_seq_len, k_max, k_per_seq != nullptr, row_shift >= 0, cp)) {
            HA_BATCH(1);
            HA_BATCH(2);
            HA_BATCH(4);
            HA_BATCH(8);
            default: break;
        }
#undef HA_BATCH
#undef HA_BATCH_ARGS
    }
    if (large_clusters((long long)B * Hkv, max_seq_len)) {
        const int rows = (max_seq_len + 8 * 4096 - 1) / (8 * 4096), kv_shift = row_shift < 0 ? 0 : row_shift;
#define HA_LARGE(PAGED) launch_cluster_t<G, 8, PAGED, 512>(rows, B, Hq, Hkv, q_codes, k_codes, kc_sb, kc_sh, seq_lens, k_per_seq,   \
                                                           k_uniform, max_seq_len, k_max, idx, idx_sb, idx_sh, count, hist_out, st, \
                                                           win, cp, kv_shift, in_step)
        return cp.table ? HA_LARGE(true) : HA_LARGE(false);
#undef HA_LARGE
    }
    if (max_seq_len <= kClusterMaxSeq) {
        // Fused path: one cluster per unit.  Cluster size: the largest of 8, 4, 2 whose grid still fits
        // the GPU in one wave (about six 256-thread CTAs per SM), so that small batches get the most
        // parallelism per sequence and large batches the most work per cluster barrier; a lane then
        // holds R = ceil(n / (CS * 2048)) rows of 8 tokens (R <= 8).
        const int units = B * Hkv, one_wave = (cp.table ? 5 : 6) * sm_count();
        int cs = 8;
        while (cs > 2 && units * cs > one_wave) cs >>= 1;
        while ((max_seq_len + cs * 2048 - 1) / (cs * 2048) > kClusterMaxRows) cs <<= 1;
        const int rows = max(1, (max_seq_len + cs * 2048 - 1) / (cs * 2048));
        const int kv_shift = row_shift < 0 ? 0 : row_shift;
#define HA_CL_ARGS rows, B, Hq, Hkv, q_codes, k_codes, kc_sb, kc_sh, seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, \
                   idx_sb, idx_sh, count, hist_out, st, win, cp, kv_shift, in_step
#define HA_CL(CSZ) return cp.table ? launch_cluster_t<G, CSZ, true>(HA_CL_ARGS) : launch_cluster_t<G, CSZ, false>(HA_CL_ARGS)
        if (cs == 8) HA_CL(8);
        if (cs == 4) HA_CL(4);
        HA_CL(2);
#undef HA_CL
#undef HA_CL_ARGS
    }
    const int chunk_tokens = chunk_tokens_for(B * Hkv, max_seq_len, sm_count());
    const int n_chunks = max(1, (max_seq_len + chunk_tokens - 1) / chunk_tokens);
    const long long score_row = (long long)score_row_bytes(max_seq_len);
    dim3 grid(n_chunks, Hkv, B);
    cudaError_t e = launch_pdl(scan_score_kernel<G>, grid, dim3(kScanThreads), 0, st, q_codes, k_codes, kc_sb, kc_sh,
                               seq_lens, max_seq_len, Hq, Hkv, chunk_tokens, score_row, ws_scores, ws_hist, win, cp, row_shift, in_step);
    if (e != cudaSuccess) return e;
    e = launch_pdl(chunk_tokens > kPassTokens ? select_kernel<2> : select_kernel<1>, grid, dim3(kScanThreads), 0, st, seq_lens, max_seq_len, k_per_seq, k_uniform, k_max,
                   Hkv, chunk_tokens, score_row, (const unsigned char *)ws_scores, (const int32_t *)ws_hist, idx, idx_sb,
                   idx_sh, count, hist_out, win);
    if (e != cudaSuccess) return e;
    count_launch(2);
    return cudaGetLastError();
}

cudaError_t launch_score_topk(int B, int Hq, int Hkv, const uint32_t *q_codes, const uint32_t *k_codes,
                              long long kc_sb, long long kc_sh, const int32_t *seq_lens,
                              const int32_t *k_per_seq, int k_uniform, int max_seq_len, int k_max,
                              int32_t *idx, long long idx_sb, long long idx_sh, int32_t *count,
                              int32_t *hist_out, int32_t *ws_hist, unsigned char *ws_scores, cudaStream_t st, Windows win,
                              CodePages cp, int row_shift, bool in_step) {
    if (row_shift >= 0) {   // one unit per query head: groups of one head over Hq unit heads
        return launch_g<1>(B, Hq, Hq, q_codes, k_codes, kc_sb, kc_sh, seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, idx_sb,
                           idx_sh, count, hist_out, ws_hist, ws_scores, st, win, cp, row_shift, in_step);
    }
#define HA_ARGS B, Hq, Hkv, q_codes, k_codes, kc_sb, kc_sh, seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, \
                idx_sb, idx_sh, count, hist_out, ws_hist, ws_scores, st, win, cp, -1, in_step
    switch (Hq / Hkv) {
        case 1: return launch_g<1>(HA_ARGS);
        case 2: return launch_g<2>(HA_ARGS);
        case 4: return launch_g<4>(HA_ARGS);
        case 8: return launch_g<8>(HA_ARGS);
        default: return cudaErrorInvalidValue;
    }
#undef HA_ARGS
}

} // namespace ha
