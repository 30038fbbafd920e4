// Device-side building blocks of the SCORE + TOPK kernels (included by ha_score_topk.cu and ha_fused.cu).
#pragma once

#include "ha_common.cuh"

namespace ha {

// Loaded from L2 (.cg): a CTA may be resident while a kernel in front of it still writes signatures or table entries, and loads
// through L1 as read-only data (ld.global.nc, __ldg) are only defined for memory that nobody writes as long as the kernel lives.
// (On a B200 no such load behind griddepcontrol.wait returned an old value in 1.8 million, its line read before the wait or not.)
__device__ __forceinline__ uint4 load_codes4(const uint32_t *row, int base, int n) {
    // tokens base..base+3 of a 16-byte aligned row; tokens >= n come back as don't-care zeros
    if (base + 3 < n) return __ldcg(reinterpret_cast<const uint4 *>(row + base));
    uint4 v = make_uint4(0, 0, 0, 0);
    if (base + 0 < n) v.x = __ldcg(row + base + 0);
    if (base + 1 < n) v.y = __ldcg(row + base + 1);
    if (base + 2 < n) v.z = __ldcg(row + base + 2);
    return v;
}

// Re-read token `last` (coherently) if it lies in [base, base+4): it may have been written by the
// kernel this one was launched behind.
__device__ __forceinline__ void patch_token(uint4 &v, int base, int last, const uint32_t *row) {
    const int e = last - base;
    if (e < 0 || e > 3) return;
    const uint32_t c = __ldcg(row + last);
    if (e == 0) v.x = c; else if (e == 1) v.y = c; else if (e == 2) v.z = c; else v.w = c;
}

// The same two helpers over a paged signature cache (pool_head = pool + h * head_stride, table_b = the sequence's row of
// the block table).  Pages of at least four tokens hold an aligned group of four in one piece; smaller pages are read
// token by token.
__device__ __forceinline__ uint4 load_codes4_paged(const CodePages &cp, const uint32_t *pool_head, const int32_t *table_b,
                                                   int base, int n) {
    if (cp.shift >= 2) {
        const uint32_t *p = pool_head + (long long)__ldcg(table_b + (base >> cp.shift)) * cp.page_stride + (base & ((1 << cp.shift) - 1));
        return load_codes4(p - base, base, n);
    }
    uint32_t v[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int t = base + i;
        if (t < n) v[i] = __ldcg(pool_head + (long long)__ldcg(table_b + (t >> cp.shift)) * cp.page_stride + (t & ((1 << cp.shift) - 1)));
    }
    return make_uint4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void patch_token_paged(uint4 &v, int base, int last, const CodePages &cp, const uint32_t *pool_head,
                                                  const int32_t *table_b) {
    const int e = last - base;
    if (e < 0 || e > 3) return;
    const uint32_t c = __ldcg(pool_head + (long long)__ldcg(table_b + (last >> cp.shift)) * cp.page_stride + (last & ((1 << cp.shift) - 1)));
    if (e == 0) v.x = c; else if (e == 1) v.y = c; else if (e == 2) v.z = c; else v.w = c;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// read an int of CTA `rank`'s shared memory at the address that `local` has in this CTA
__device__ __forceinline__ int ld_dsmem(const int *local, uint32_t rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(local), ra;
    int v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(ra) : "memory");
    return v;
}
// write an int of CTA `rank`'s shared memory at the address that `local` has in this CTA
__device__ __forceinline__ void st_dsmem(int *local, uint32_t rank, int v) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(local), ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(ra), "r"(v) : "memory");
}

// Score byte of a token that is always in context (Windows): above every real score + 1 (<= 33), so the
// flag arithmetic below sees "score > T" for every threshold, and small enough that no byte sum reaches 256.
constexpr uint32_t kForcedByte = 63u;

// Bits 7, 15, 23, 31 of x gathered into a nibble (bit e = bit 7 of byte e).  The four partial products
// land on distinct bit positions, so the multiplication carries nothing into bits 28..31.
__device__ __forceinline__ uint32_t high_bits_to_nibble(uint32_t x) {
    return ((x & 0x80808080u) * 0x00204081u) >> 28;
}

// Writes the selected ones of 32 consecutive tokens from `first` on in ascending order: those with S > T (gt) and the first `room` of
// those with S == T (eq; room <= 0: none).  dst is where the first of them goes; returns dst behind the last.  The selected ones are
// worked out before any is visited: of the tokens at the threshold, often many times the wanted ones, a lane would visit all while
// the rest of its warp waits (64 sequences of 32768 tokens 92.0 -> 89.6 us per step, 5 ragged ones in one launch 18.3 -> 17.2).
__device__ __forceinline__ int32_t *write_selected32(int32_t *dst, int first, uint32_t gt, uint32_t eq, int room) {
    uint32_t sel = gt;
    if (room >= __popc(eq)) sel |= eq;
    else for (uint32_t m = eq; room > 0; --room) { sel |= m & (0u - m); m &= m - 1u; }   // the 32 in which the last one lies
    for (; sel; sel &= sel - 1u) *dst++ = first + __ffs((int)sel) - 1;
    return dst;
}

// Warp-wide threshold search over the 33 score levels.  Lane l passes the count of level l (tot) and
// the part of it that lies before the caller's own slice (bef); level 32 comes in tot32 / bef32.
// Returns T = largest level with #{S >= T} >= keep, r = keep - #{S > T}, and the numbers of tokens
// before the caller's slice with S > T and with S == T.  keep == 0 gives T = 33 (nothing selected).
__device__ __forceinline__ void find_threshold(int tot, int bef, int tot32, int bef32, int keep, int lane, int &T,
                                               int &r, int &gt_before, int &eq_before) {
    int st = tot, sb = bef;   // suffix sums over levels lane..31
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
        const int vt = __shfl_down_sync(0xffffffffu, st, dd), vb = __shfl_down_sync(0xffffffffu, sb, dd);
        if (lane + dd < 32) { st += vt; sb += vb; }
    }
    st += tot32;   // #{S >= lane}
    sb += bef32;   // same, restricted to what lies before the caller's slice
    T = kBins; r = 0; gt_before = 0; eq_before = 0;
    if (keep > 0) {
        const unsigned ge = __ballot_sync(0xffffffffu, st >= keep);
        if (tot32 >= keep) { T = 32; r = keep; gt_before = 0; eq_before = bef32; }
        else {
            T = 31 - __clz(ge);   // ge != 0 because #{S >= 0} = n >= keep
            const int above = __shfl_sync(0xffffffffu, st, min(T + 1, 31));      // #{S >= T+1}
            const int above_b = __shfl_sync(0xffffffffu, sb, min(T + 1, 31));
            const int at_b = __shfl_sync(0xffffffffu, bef, T);
            const int gt = (T == 31) ? tot32 : above;
            r = keep - gt;
            gt_before = (T == 31) ? bef32 : above_b;
            eq_before = at_b;
        }
    }
}

} // namespace ha
