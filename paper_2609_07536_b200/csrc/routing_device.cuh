// Device-side steps of the routing build that more than one kernel runs: the one-launch build and the kernels that build the
// routing of a small batch themselves.
#pragma once

#include "moe_internal.h"

namespace moe {
namespace {

__device__ __forceinline__ void routing_report(uint32_t *status, uint32_t code, uint32_t detail, uint32_t where)
{
    if (!status) return;       // (a CTA that repeats the work of another one)
    if (atomicCAS(&status[0], 0u, code) == 0u) {
        status[1] = detail;
        status[2] = where;
    }
    atomicAdd(&status[3], 1u);
}

// m-tile table entry mu: the expert is found by bisection in the tile prefix
__device__ __forceinline__ void mtile_entry(int mu, int E_tot, int tile_m, const int32_t *s_cnt, const int32_t *s_off,
                                            const int32_t *s_toff, int32_t *__restrict__ mtile_expert,
                                            int32_t *__restrict__ mtile_first_row, int32_t *__restrict__ mtile_valid)
{
    int lo = 0, hi = E_tot - 1;          // largest e with tile_offsets[e] <= mu
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_toff[mid] <= mu) lo = mid; else hi = mid - 1;
    }
    const int e = lo, i = mu - s_toff[e];
    mtile_expert[mu] = e;
    mtile_first_row[mu] = s_off[e] + i * tile_m;
    mtile_valid[mu] = min(tile_m, s_cnt[e] - i * tile_m);
}

// counter row of a warp: 16-bit (a CTA holds at most 8192 assignments), its pitch an odd number of 32-bit words,
// so that the 32 counters of one expert lie in 32 banks
__host__ __device__ constexpr int onepass_pitch(int E_tot) { return 2 * (((E_tot + 1) / 2) | 1); }

// Ranks of a warp's chunk [begin, end) of at most kRows rows of 32 assignments: e[i] the expert of this lane's assignment of row i (-1:
// none, or a bad id), rk[i] its rank among the chunk's assignments of that expert, h[x] (a row of onepass_pitch counters) how
// many the chunk has.
template <int kRows>
__device__ __forceinline__ void rank_chunk(const int32_t *__restrict__ topk_idx, int begin, int end, int rows, int k_tot, int E_tot, int pitch,
                                           uint16_t *h, int (&e)[kRows], int (&rk)[kRows], uint32_t *status)
{
    // ---- ids of the warp's chunk, and the 32 before it (a token may straddle the boundary)
    const int lane = threadIdx.x & 31;
    int before = -1;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        const int f = begin + 32 * i + lane;
        e[i] = (i < rows && f < end) ? ld_chained(topk_idx + f) : -1;
    }
    if (begin > 0 && begin < end) before = ld_chained(topk_idx + begin - 32 + lane);
    for (int x = lane; x < pitch / 2; x += 32) reinterpret_cast<uint32_t *>(h)[x] = 0u;
    __syncwarp();

    // ---- ranks inside the chunk; bad ids are reported and left out, repeated experts reported and kept
    const auto modulo_k = [&](int n) { return n - small_quotient(n, k_tot) * k_tot; };     // (begin < 2^18)
    int j = modulo_k(begin + lane), m0 = modulo_k(begin);           // slot of this lane's assignment, of the row's first
    const int step = modulo_k(32), id_bits = E_tot > 1 ? 32 - __clz(E_tot - 1) : 0;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        rk[i] = 0;
        if (i >= rows || begin + 32 * i >= end) break;              // warp-uniform
        const int f = begin + 32 * i + lane;
        const bool ok = e[i] >= 0 && e[i] < E_tot;
        if (f < end && !ok) routing_report(status, MOE_DEV_OOB, (uint32_t)f, 1u);
        // lanes with the same expert, bit by bit of the id (match_any takes ~80 cycles of the SM per row when the
        // ids differ; these votes take a quarter of that at 66 experts)
        uint32_t same = __ballot_sync(0xffffffffu, ok);
        for (int b = 0; b < id_bits; ++b) {
            const bool bit = (e[i] >> b) & 1;
            const uint32_t m = __ballot_sync(0xffffffffu, bit);
            same &= bit ? m : ~m;
        }
        const uint32_t lower = same & ((1u << lane) - 1u);
        const int base = ok ? (int)h[e[i]] : 0;
        __syncwarp();
        if (ok && lower == 0u) h[e[i]] = (uint16_t)(base + __popc(same));
        __syncwarp();
        rk[i] = base + __popc(lower);
        // the same expert twice inside one token: among the lanes of this row, then in the row before
        const int in_row = min(j, lane);
        int twice = ok ? __popc(lower & (((1u << in_row) - 1u) << (lane - in_row))) : 0;
        for (int d = 1; d <= m0; ++d) {
            const int v = __shfl_sync(0xffffffffu, before, 32 - d);
            if (ok && j - lane >= d && v == e[i]) ++twice;
        }
        for (; twice > 0; --twice) routing_report(status, MOE_DEV_DUP_EXPERT, (uint32_t)(f / k_tot), 1u);
        before = e[i];
        j += step;
        if (j >= k_tot) j -= k_tot;
        m0 += step;
        if (m0 >= k_tot) m0 -= k_tot;
        if (!ok) e[i] = -1;
    }
}

// The whole build by one CTA of kWarps warps, inside a kernel that goes on with the batch itself: at most kInlineRows rows of
// 32 assignments per warp, E_tot <= 32 kWarps.  Every CTA of the kernel builds it and writes what its own roles read (kCombines:
// pad_row too), the same values everywhere, and relies on its own writes only; the first one writes the rest and reports.
// That takes a launch and its hand-over off the step (whole step, us: DeepSeek shape T = 1 22.4 -> 20.0, T = 16 65.6 ->
// 62.2, T = 128 83.2 -> 77.5, Granite shape T = 128 26.1 -> 23.0; with GEMM1, DeepSeek shape T = 1 41.8 -> 39.8).  What it costs
// is the chain of rows in a warp, and all CTAs writing the same lines: perm, whose entries are scattered, goes through shared
// memory for that (Granite shape T = 128: 29.2 -> 23.0).  The gain shrinks from 3.3 us at 480 assignments to 2.3 at 2048,
// the four-row limit; more rows would lengthen the chain further than a cluster's hand-over takes.
// `sm`: shared memory, which bulk copies of the CTA may write afterwards.  Every thread comes here; behind it the arrays may be read.
constexpr int kInlineRows = 4;
template <int kWarps, bool kCombines>
__device__ __forceinline__ void routing_inline(const InlineRouting &p, int k_tot, int E_tot, int tile_m, uint32_t *status_dev,
                                               unsigned long long *mail, uint32_t mail_seq, int32_t *sm)
{
    const bool first = blockIdx.x == 0;
    uint32_t *status = first ? status_dev : nullptr;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, pitch = onepass_pitch(E_tot);
    uint16_t *hist = reinterpret_cast<uint16_t *>(sm);                                   // [kWarps][pitch]
    int32_t *s_cnt = sm + kWarps * pitch / 2, *s_off = s_cnt + (E_tot + 1), *s_toff = s_off + (E_tot + 1), *s_sum = s_toff + (E_tot + 1), *s_perm = s_sum + 64;
    const int rows = (p.R + 32 * kWarps - 1) / (32 * kWarps);
    const int begin = min(p.R, w * rows * 32), end = min(p.R, begin + rows * 32);
    int e[kInlineRows], rk[kInlineRows];
    uint16_t *h = hist + w * pitch;
    rank_chunk(p.topk_idx, begin, end, rows, k_tot, E_tot, pitch, h, e, rk, status);
    __syncthreads();
    // thread x, expert x: exclusive prefix of the warps' counts, then over the experts (rows and m-tiles)
    const int x = (int)threadIdx.x, n_scan = (E_tot + 31) / 32;
    int cnt = 0;
    if (x < E_tot) {
#pragma unroll
        for (int c0 = 0; c0 < kWarps; c0 += 4) {
            int v[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = hist[(c0 + c) * pitch + x];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                hist[(c0 + c) * pitch + x] = (uint16_t)cnt;
                cnt += v[c];
            }
        }
    }
    const int tl = small_quotient(cnt + tile_m - 1, tile_m);
    int ic = cnt, it = tl;
    if (w < n_scan) {
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int uc = __shfl_up_sync(0xffffffffu, ic, d), ut = __shfl_up_sync(0xffffffffu, it, d);
            if (lane >= d) { ic += uc; it += ut; }
        }
        if (lane == 31) { s_sum[w] = ic; s_sum[32 + w] = it; }
    }
    __syncthreads();
    if (w < n_scan) {
        ic += __reduce_add_sync(0xffffffffu, lane < w ? s_sum[lane] : 0);
        it += __reduce_add_sync(0xffffffffu, lane < w ? s_sum[32 + lane] : 0);
        if (x < E_tot) {
            s_cnt[x] = cnt;
            s_off[x] = ic - cnt;
            s_toff[x] = it - tl;
            if (x == E_tot - 1) { s_off[E_tot] = ic; s_toff[E_tot] = it; }
        }
    }
    __syncthreads();
    // the counts leave for the host before anything else: in a loop of the smallest steps it is what prepares the next one (tiny shape
    // T = 256: 13.6 -> 12.6 us against mailing them once the arrays are written)
    if (first && w == kWarps - 1)
        mail_counts(mail, mail_seq, E_tot, lane, [&](int y) { return y < E_tot ? s_toff[y + 1] - s_toff[y] : s_toff[E_tot]; });
#pragma unroll
    for (int i = 0; i < kInlineRows; ++i) {
        const int f = begin + 32 * i + lane;
        if (i >= rows || f >= end) break;
        int r = -1, pad = -1;
        if (e[i] >= 0) {
            const int in_expert = (int)h[e[i]] + rk[i];
            r = s_off[e[i]] + in_expert;
            pad = tile_m * s_toff[e[i]] + in_expert;
            s_perm[r] = f;
        }
        if (first) p.out.inv_perm[f] = r;
        if (first || kCombines) p.out.pad_row[f] = pad;
    }
    const int S = min(s_toff[E_tot], p.max_mtiles);
    for (int mu = x; mu < S; mu += 32 * kWarps)
        mtile_entry(mu, E_tot, tile_m, s_cnt, s_off, s_toff, p.out.mtile_expert, p.out.mtile_first_row, p.out.mtile_valid);
    if (x == 0 && s_toff[E_tot] > p.max_mtiles) routing_report(status, MOE_DEV_OOB, (uint32_t)s_toff[E_tot], 2u);
    if (x == 0) p.out.tiles[E_tot] = s_toff[E_tot];
    for (int y = x; first && y <= E_tot; y += 32 * kWarps) {
        if (y < E_tot) {
            p.out.counts[y] = s_cnt[y];
            p.out.tiles[y] = s_toff[y + 1] - s_toff[y];
        }
        p.out.offsets[y] = s_off[y];
        p.out.tile_offsets[y] = s_toff[y];
    }
    __syncthreads();
    for (int r = x; r < s_off[E_tot]; r += 32 * kWarps) p.out.perm[r] = s_perm[r];   // (coalesced: the CTAs all write here)
    // the shared memory is written by bulk copies next
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
}

}  // namespace
}  // namespace moe
