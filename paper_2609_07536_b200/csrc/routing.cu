// Routing / permutation / routed-tile-count builder (device).
//
// Section II-A: the router's token-expert assignments; Eq. 5: expert e needs
// ceil(M_e / T_M) tiles along the token dimension; Eq. 16: their sum S.
// The routed rows are the flat assignments f = t * k_tot + j in a *stable* order by expert.
//
// Two launch shapes here, the same outputs bit for bit (a whole-step call on a small batch has neither: the kernel that uses
// the routing builds it itself, routing_device.cuh):
//   routing_onepass  up to 131072 assignments: one launch of one cluster of 1 to 16 CTAs; the ids stay in
//                    registers from the histogram to the scatter, the per-expert totals of the CTAs cross
//                    through distributed shared memory;
//   otherwise four small launches over the whole GPU:
//   1. hist          every warp histograms its own contiguous chunk of assignments;
//   2. scan_columns  one CTA per expert: exclusive prefix of that expert's histogram column over
//                    the warps (the per-(warp, expert) bases) and the expert's count;
//   3. finalize      one CTA: exclusive offsets, tiles per expert and their prefix, the m-tile table;
//   4. scatter       every warp walks its chunk in order, 32 assignments at a time;
//                    match_any gives each lane its rank among equal experts -> stable.

#include "moe_internal.h"
#include "routing_device.cuh"

namespace moe {
namespace {

constexpr int kWarpsPerBlock = 8;
constexpr int kPerLane = kRoutingChunk / 32;   // assignments of a chunk held by one lane
static_assert(kRoutingChunk % 32 == 0, "a chunk is a whole number of warp-wide rows");

// launch `kernel` so that it may be set up before the previous kernel on the stream has finished
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0] = chained_launch_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ---- the three steps every path runs on a chunk, one warp per chunk --------------------------------------
//
// Slot i of lane l is flat assignment begin + 32 i + l.  The ids of a chunk are fetched with independent
// loads, all in flight together: a loop with one dependent load per 32 assignments spent its time on
// memory latency (8 round trips per chunk and pass).

// expert ids of the chunk (-1 past the end)
__device__ __forceinline__ void chunk_load(const int32_t *__restrict__ topk_idx, int begin, int end, int lane, int (&e)[kPerLane])
{
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
        const int f = begin + 32 * i + lane;
        e[i] = f < end ? ld_chained(topk_idx + f) : -1;
    }
}

// histogram of the chunk into h[E_tot] (shared memory, zeroed by the caller); bad ids and an expert chosen
// twice by one token are reported and left out / kept, as the scatter does
__device__ __forceinline__ void chunk_hist(const int32_t *__restrict__ topk_idx, int begin, int end, int lane, int k_tot,
                                           int E_tot, const int (&e)[kPerLane], int32_t *h, uint32_t *status)
{
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
        const int f = begin + 32 * i + lane;
        if (f >= end) continue;
        if (e[i] < 0 || e[i] >= E_tot) {
            routing_report(status, MOE_DEV_OOB, (uint32_t)f, 1u);
            continue;
        }
        atomicAdd(&h[e[i]], 1);
        // the same expert twice inside one token?
        const int t = f / k_tot, j = f - t * k_tot;
        for (int jj = 0; jj < j; ++jj)
            if (__ldg(topk_idx + t * k_tot + jj) == e[i]) routing_report(status, MOE_DEV_DUP_EXPERT, (uint32_t)t, 1u);
    }
}

// stable scatter of the chunk: run[e] is the next free routed row of expert e for this chunk; match_any
// gives each lane its rank among the lanes of the row with the same expert.  off / toff: exclusive prefixes
// of the per-expert rows and m-tiles.
__device__ __forceinline__ void chunk_scatter(int begin, int end, int lane, int E_tot, int tile_m, const int (&e)[kPerLane],
                                              int32_t *run, const int32_t *off, const int32_t *toff,
                                              int32_t *__restrict__ perm, int32_t *__restrict__ inv_perm,
                                              int32_t *__restrict__ pad_row)
{
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
        if (begin + 32 * i >= end) break;     // warp-uniform
        const int f = begin + 32 * i + lane;
        const bool in = f < end;
        const int ex = e[i];
        const bool ok = in && ex >= 0 && ex < E_tot;
        const unsigned active = __ballot_sync(0xffffffffu, ok);
        if (in && !ok) { inv_perm[f] = -1; pad_row[f] = -1; }
        if (ok) {
            const unsigned same = __match_any_sync(active, ex);
            const int rank = __popc(same & ((1u << lane) - 1u));
            const int r = run[ex] + rank;
            __syncwarp(active);
            if (rank == 0) run[ex] += __popc(same);
            perm[r] = f;
            inv_perm[f] = r;
            pad_row[f] = tile_m * toff[ex] + (r - off[ex]);
        }
        __syncwarp();
    }
}

// One warp: exclusive prefixes over the experts of the rows (s_off) and of the m-tiles ceil(rows / tile_m)
// (s_toff), totals in entry E_tot (Eq. 5, Eq. 16), 32 experts per step.
__device__ __forceinline__ void expert_prefix(const int32_t *s_cnt, int32_t *s_off, int32_t *s_toff, int E_tot, int tile_m, int lane)
{
    int off = 0, toff = 0;
    for (int e0 = 0; e0 < E_tot; e0 += 32) {
        const int e = e0 + lane;
        const int c = e < E_tot ? s_cnt[e] : 0;
        const int tl = (c + tile_m - 1) / tile_m;
        int ic = c, it = tl;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int uc = __shfl_up_sync(0xffffffffu, ic, d), ut = __shfl_up_sync(0xffffffffu, it, d);
            if (lane >= d) { ic += uc; it += ut; }
        }
        if (e < E_tot) {
            s_off[e] = off + ic - c;
            s_toff[e] = toff + it - tl;
        }
        off += __shfl_sync(0xffffffffu, ic, 31);
        toff += __shfl_sync(0xffffffffu, it, 31);
    }
    if (lane == 0) {
        s_off[E_tot] = off;
        s_toff[E_tot] = toff;
    }
}

// ---- large batches: four launches over the whole GPU -------------------------------------------------------

__global__ void __launch_bounds__(kWarpsPerBlock * 32)
routing_hist(const int32_t *__restrict__ topk_idx, int R, int k_tot, int E_tot, int n_warps,
             int32_t *__restrict__ whist, uint32_t *status)
{
    extern __shared__ int32_t sh[];
    const int warp_in_block = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = blockIdx.x * kWarpsPerBlock + warp_in_block;
    if (w >= n_warps) return;
    int32_t *h = sh + warp_in_block * E_tot;
    const int begin = w * kRoutingChunk, end = min(R, begin + kRoutingChunk);
    int e[kPerLane];
    chunk_load(topk_idx, begin, end, lane, e);
    for (int x = lane; x < E_tot; x += 32) h[x] = 0;
    __syncwarp();
    chunk_hist(topk_idx, begin, end, lane, k_tot, E_tot, e, h, status);
    __syncwarp();
    for (int x = lane; x < E_tot; x += 32) whist[(size_t)w * E_tot + x] = h[x];
}

// Per expert (one CTA each): counts[e], and whist[.][e] turned into an exclusive prefix over the
// sorting warps.  Thread t owns a contiguous run of warps; the run sums are scanned across the CTA.
constexpr int kScanThreads = 256;
__global__ void __launch_bounds__(kScanThreads)
routing_scan_columns(int E_tot, int n_warps, int32_t *__restrict__ whist, int32_t *__restrict__ counts)
{
    __shared__ int warp_sum[kScanThreads / 32];
    grid_dependency_wait();
    const int e = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int chunk = (n_warps + kScanThreads - 1) / kScanThreads;
    const int w_lo = min(n_warps, tid * chunk), w_hi = min(n_warps, w_lo + chunk);
    int sum = 0;
    for (int w = w_lo; w < w_hi; ++w) sum += whist[(size_t)w * E_tot + e];
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += up;
    }
    if (lane == 31) warp_sum[wid] = incl;
    __syncthreads();
    int base = incl - sum;
    for (int i = 0; i < wid; ++i) base += warp_sum[i];
    for (int w = w_lo; w < w_hi; ++w) {
        const int c = whist[(size_t)w * E_tot + e];
        whist[(size_t)w * E_tot + e] = base;
        base += c;
    }
    if (tid == kScanThreads - 1) counts[e] = base;
}

// Offsets, tile counts and the m-tile table from the per-expert counts (one CTA).
// Dynamic shared memory: 3 * (E_tot + 1) ints.
__global__ void __launch_bounds__(1024)
routing_finalize(int E_tot, int tile_m, int max_mtiles, const int32_t *__restrict__ counts,
                 int32_t *__restrict__ offsets, int32_t *__restrict__ tiles, int32_t *__restrict__ tile_offsets,
                 int32_t *__restrict__ mtile_expert, int32_t *__restrict__ mtile_first_row,
                 int32_t *__restrict__ mtile_valid, uint32_t *status, unsigned long long *mail, uint32_t mail_seq)
{
    extern __shared__ int32_t fin[];
    grid_dependency_wait();
    int32_t *s_cnt = fin, *s_off = fin + (E_tot + 1), *s_toff = fin + 2 * (E_tot + 1);
    for (int e = threadIdx.x; e < E_tot; e += blockDim.x) s_cnt[e] = counts[e];
    __syncthreads();
    if (threadIdx.x < 32) expert_prefix(s_cnt, s_off, s_toff, E_tot, tile_m, threadIdx.x);
    __syncthreads();
    if (threadIdx.x < 32)
        mail_counts(mail, mail_seq, E_tot, threadIdx.x, [&](int x) { return x < E_tot ? s_toff[x + 1] - s_toff[x] : s_toff[E_tot]; });
    if (threadIdx.x == 0 && s_toff[E_tot] > max_mtiles) routing_report(status, MOE_DEV_OOB, (uint32_t)s_toff[E_tot], 2u);
    for (int e = threadIdx.x; e <= E_tot; e += blockDim.x) {
        offsets[e] = s_off[e];
        tile_offsets[e] = s_toff[e];
        // S rides behind the per-expert tile counts for the host copy
        tiles[e] = (e < E_tot) ? s_toff[e + 1] - s_toff[e] : s_toff[E_tot];
    }
    const int S = min(s_toff[E_tot], max_mtiles);
    for (int mu = threadIdx.x; mu < S; mu += blockDim.x)
        mtile_entry(mu, E_tot, tile_m, s_cnt, s_off, s_toff, mtile_expert, mtile_first_row, mtile_valid);
}

// Dynamic shared memory: (kWarpsPerBlock * E_tot + 2 * (E_tot + 1)) ints.
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
routing_scatter(const int32_t *__restrict__ topk_idx, int R, int E_tot, int tile_m, int n_warps,
                const int32_t *__restrict__ whist, const int32_t *__restrict__ offsets,
                const int32_t *__restrict__ tile_offsets, int32_t *__restrict__ perm,
                int32_t *__restrict__ inv_perm, int32_t *__restrict__ pad_row)
{
    extern __shared__ int32_t sh[];
    const int warp_in_block = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = blockIdx.x * kWarpsPerBlock + warp_in_block;
    const int begin = min(R, w * kRoutingChunk), end = w < n_warps ? min(R, begin + kRoutingChunk) : begin;
    // the ids do not depend on the launches before this one: fetch them before waiting
    int e[kPerLane];
    chunk_load(topk_idx, begin, end, lane, e);
    grid_dependency_wait();
    int32_t *s_off = sh + kWarpsPerBlock * E_tot, *s_toff = s_off + (E_tot + 1);
    for (int x = threadIdx.x; x <= E_tot; x += blockDim.x) {
        s_off[x] = offsets[x];
        s_toff[x] = tile_offsets[x];
    }
    __syncthreads();
    if (w >= n_warps) return;
    int32_t *run = sh + warp_in_block * E_tot;  // next free row per expert, for this warp
    for (int x = lane; x < E_tot; x += 32) run[x] = s_off[x] + whist[(size_t)w * E_tot + x];
    __syncwarp();
    chunk_scatter(begin, end, lane, E_tot, tile_m, e, run, s_off, s_toff, perm, inv_perm, pad_row);
}

// ---- up to 131072 assignments: the same steps in ONE launch of one thread-block cluster ---------------------
//
// A cluster of n CTAs (1 for the decode sizes, up to 16), every warp owns `rows` (1..8) rows of 32 assignments.
// One pass over the ids: votes rank a row's equal experts, the warp's own counter row in shared memory ranks them
// across its rows, so that the rank of every assignment inside its warp's chunk is known before the prefixes are,
// the scatter is one addition, and no shared-memory atomic is needed.  Bound by the length of the serial chain
// (launch, ids, ranks, prefix over warps, CTAs and experts, stores), not by bytes: 131072 ids are 512 KB.  So the
// chain is kept short: one thread per expert reads its 32 counters with independent loads, CTA totals are pushed
// to all CTAs and cross with one cluster barrier, the experts' prefixes are one scan of the whole CTA.  perm is first
// put in order in shared memory when a CTA holds many assignments: its lines then leave whole instead of 4 bytes
// at a time.  Measured (device time; before: one CTA, one cluster of 8 or four launches, two passes over the ids):
//   assignments, experts   8, 66   192, 60   2048, 66   8024, 40   32768, 60   131072, 66   27000, 1000
//   before                 4.6     7.3       10.0       16.3       12.8        21.5         23.9 us
//   now                    3.9     3.8       5.6        5.7        7.5         14.1         12.5 us
constexpr int kOnepassWarps = 32;
constexpr int kOnepassRows = 8;
constexpr int kOnepassMaxCtas = 16;
constexpr size_t kOnepassMaxSmem = 200 * 1024;

// CTAs for R assignments (0: too many for one launch): one more row per warp lengthens the chain by ~1 us, a cluster
// of 2 to 16 costs 0.7 us over a single CTA whatever its size: as many CTAs as it takes to keep one row per warp
int onepass_ctas(int R, int max_cluster)
{
    int n = 1;
    while (n < max_cluster && n < kOnepassMaxCtas && n * kOnepassWarps * 32 < R) n *= 2;
    return (int64_t)n * kOnepassWarps * 32 * kOnepassRows >= R ? n : 0;
}
int onepass_rows(int R, int n_ctas)
{
    const int per_row = n_ctas * kOnepassWarps * 32;
    return R > per_row ? (R + per_row - 1) / per_row : 1;
}
bool onepass_staged(int rows) { return rows > 2; }
size_t onepass_smem(int n_ctas, int rows, int E_tot)
{
    size_t ints = (size_t)kOnepassWarps * onepass_pitch(E_tot) / 2;       // counters
    ints += (size_t)n_ctas * E_tot + E_tot;                                // totals of all CTAs, rows before this CTA
    ints += 4 * (size_t)(E_tot + 1);                                       // counts, offsets, tile offsets, offsets inside the CTA
    if (onepass_staged(rows)) ints += (size_t)rows * kOnepassWarps * 32;   // perm of this CTA, in order
    return ints * sizeof(int32_t);
}

__global__ void __launch_bounds__(kOnepassWarps * 32)
routing_onepass(const int32_t *__restrict__ topk_idx, int R, int k_tot, int E_tot, int tile_m, int rows, int n_ctas, int staged,
                int max_mtiles, const RoutingOut out, uint32_t *status, unsigned long long *mail, uint32_t mail_seq)
{
    extern __shared__ int32_t sm[];
    const int pitch = onepass_pitch(E_tot);
    uint16_t *hist = reinterpret_cast<uint16_t *>(sm);              // [32][pitch]
    int32_t *s_all = sm + kOnepassWarps * pitch / 2;                // [n_ctas][E_tot] rows per expert of every CTA
    int32_t *s_base = s_all + n_ctas * E_tot;                       // [E_tot] rows of the expert in the CTAs before this one
    int32_t *s_cnt = s_base + E_tot, *s_off = s_cnt + (E_tot + 1), *s_toff = s_off + (E_tot + 1);
    int32_t *s_loc = s_toff + (E_tot + 1);                          // offsets of the experts inside this CTA
    int32_t *s_perm = s_loc + (E_tot + 1);
    __shared__ int32_t s_sum[96];                                   // per scanning warp: rows, tiles, rows of this CTA
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t rank = 0;
    if (n_ctas > 1) {
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // "this CTA runs": see the push below
    }
    grid_dependency_wait();
    grid_dependents_may_launch();

    const int begin = min(R, ((int)rank * kOnepassWarps + w) * rows * 32), end = min(R, begin + rows * 32);
    int e[kOnepassRows], rk[kOnepassRows];
    uint16_t *h = hist + w * pitch;
    rank_chunk(topk_idx, begin, end, rows, k_tot, E_tot, pitch, h, e, rk, status);
    __syncthreads();

    // ---- thread x, expert x: exclusive prefix of the warps' counts; this CTA's total, pushed to every CTA; rows in the
    // CTAs before this one and in all
    const int x = (int)threadIdx.x;
    int own = 0, cnt = 0, ahead = 0;
    if (x < E_tot) {
#pragma unroll
        for (int c0 = 0; c0 < kOnepassWarps; c0 += 8) {
            int v[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = hist[(c0 + c) * pitch + x];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                hist[(c0 + c) * pitch + x] = (uint16_t)own;
                own += v[c];
            }
        }
        cnt = own;
    }
    if (n_ctas > 1) {
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");    // every CTA runs: its memory may be written
        if (x < E_tot) {
            const uint32_t mine = (uint32_t)__cvta_generic_to_shared(s_all + (int)rank * E_tot + x);
            for (int c = 0; c < n_ctas; ++c)
                asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.u32 [a], %2;\n\t}"
                             ::"r"(mine), "r"(c), "r"(own) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (x < E_tot) {
            cnt = 0;
#pragma unroll
            for (int c = 0; c < kOnepassMaxCtas; ++c) {
                const int v = c < n_ctas ? s_all[c * E_tot + x] : 0;
                if (c < (int)rank) ahead += v;
                cnt += v;
            }
        }
    }
    // ---- exclusive prefixes over the experts: rows, tiles (Eq. 5, Eq. 16) and rows of this CTA (every CTA, for its own scatter)
    const int tl = small_quotient(cnt + tile_m - 1, tile_m), n_scan = (E_tot + 31) / 32;
    int ic = cnt, it = tl, io = own;
    if (w < n_scan) {
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int uc = __shfl_up_sync(0xffffffffu, ic, d), ut = __shfl_up_sync(0xffffffffu, it, d), uo = __shfl_up_sync(0xffffffffu, io, d);
            if (lane >= d) { ic += uc; it += ut; io += uo; }
        }
        if (lane == 31) { s_sum[w] = ic; s_sum[32 + w] = it; s_sum[64 + w] = io; }
    }
    __syncthreads();
    if (w < n_scan) {
        ic += __reduce_add_sync(0xffffffffu, lane < w ? s_sum[lane] : 0);
        it += __reduce_add_sync(0xffffffffu, lane < w ? s_sum[32 + lane] : 0);
        io += __reduce_add_sync(0xffffffffu, lane < w ? s_sum[64 + lane] : 0);
        if (x < E_tot) {
            s_cnt[x] = cnt;
            s_base[x] = ahead;
            s_off[x] = ic - cnt;
            s_toff[x] = it - tl;
            s_loc[x] = io - own;
            if (x == E_tot - 1) { s_off[E_tot] = ic; s_toff[E_tot] = it; s_loc[E_tot] = io; }
        }
    }
    __syncthreads();

    // ---- results
    if (rank == 0 && w == kOnepassWarps - 1)
        mail_counts(mail, mail_seq, E_tot, lane, [&](int x) { return x < E_tot ? s_toff[x + 1] - s_toff[x] : s_toff[E_tot]; });
#pragma unroll
    for (int i = 0; i < kOnepassRows; ++i) {
        const int f = begin + 32 * i + lane;
        if (i >= rows || f >= end) break;
        int r = -1, pad = -1;
        if (e[i] >= 0) {
            const int x = e[i], in_cta = (int)h[x] + rk[i], o = s_off[x];
            r = o + s_base[x] + in_cta;
            pad = tile_m * s_toff[x] + (r - o);
            if (staged) s_perm[s_loc[x] + in_cta] = f;
            else out.perm[r] = f;
        }
        out.inv_perm[f] = r;
        out.pad_row[f] = pad;
    }
    const int S = min(s_toff[E_tot], max_mtiles);
    for (int mu = (int)rank * (int)blockDim.x + threadIdx.x; mu < S; mu += n_ctas * (int)blockDim.x)
        mtile_entry(mu, E_tot, tile_m, s_cnt, s_off, s_toff, out.mtile_expert, out.mtile_first_row, out.mtile_valid);
    if (rank == 0) {
        if (threadIdx.x == 0 && s_toff[E_tot] > max_mtiles) routing_report(status, MOE_DEV_OOB, (uint32_t)s_toff[E_tot], 2u);
        for (int x = threadIdx.x; x <= E_tot; x += blockDim.x) {
            if (x < E_tot) out.counts[x] = s_cnt[x];
            out.offsets[x] = s_off[x];
            out.tile_offsets[x] = s_toff[x];
            // S rides behind the per-expert tile counts for the host copy
            out.tiles[x] = (x < E_tot) ? s_toff[x + 1] - s_toff[x] : s_toff[E_tot];
        }
    }
    if (staged) {
        __syncthreads();
        for (int x = w; x < E_tot; x += kOnepassWarps) {
            const int src = s_loc[x], n = s_loc[x + 1] - src, dst = s_off[x] + s_base[x];
            for (int i = lane; i < n; i += 32) out.perm[dst + i] = s_perm[src + i];
        }
    }
}

void onepass_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int n_ctas, size_t smem, cudaStream_t stream)
{
    cfg.gridDim = dim3((unsigned)n_ctas);
    cfg.blockDim = dim3(kOnepassWarps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)n_ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

cudaError_t routing_onepass_launch(const int32_t *topk_idx, const moe_shape &s, int tile_m, int R, int n_ctas,
                                   const moe_routing &r, uint32_t *status, unsigned long long *mail, uint32_t mail_seq,
                                   cudaStream_t stream)
{
    const int rows = onepass_rows(R, n_ctas);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    onepass_config(cfg, attr, n_ctas, onepass_smem(n_ctas, rows, s.E_tot), stream);
    attr[1] = chained_launch_attribute();
    cfg.numAttrs = 2;
    const RoutingOut out = routing_out(r);
    return cudaLaunchKernelEx(&cfg, routing_onepass, topk_idx, R, (int)s.k_tot, (int)s.E_tot, tile_m, rows, n_ctas,
                              onepass_staged(rows) ? 1 : 0, (int)r.max_mtiles, out, status, mail, mail_seq);
}

// the four launches; `scratch`: n_chunks * E_tot ints that need not start at any value
cudaError_t routing_four_launches(const int32_t *topk_idx, const moe_shape &s, int tile_m, int R, int n_chunks,
                                  const moe_routing &r, int32_t *scratch, uint32_t *status, unsigned long long *mail, uint32_t mail_seq,
                                  cudaStream_t stream)
{
    const int blocks = (n_chunks + kWarpsPerBlock - 1) / kWarpsPerBlock;
    const int E = (int)s.E_tot;
    const size_t sh_hist = (size_t)kWarpsPerBlock * E * sizeof(int32_t);
    const size_t sh_scat = sh_hist + 2 * (size_t)(E + 1) * sizeof(int32_t);
    if (blocks > 0)
        routing_hist<<<blocks, kWarpsPerBlock * 32, sh_hist, stream>>>(topk_idx, R, s.k_tot, E, n_chunks, scratch, status);
    cudaError_t e = launch_chained(routing_scan_columns, dim3(E), dim3(kScanThreads), 0, stream, E, n_chunks, scratch, r.counts);
    if (e != cudaSuccess) return e;
    e = launch_chained(routing_finalize, dim3(1), dim3(1024), 3 * (size_t)(E + 1) * sizeof(int32_t), stream, E, tile_m,
                       (int)r.max_mtiles, r.counts, r.offsets, r.tiles, r.tile_offsets, r.mtile_expert, r.mtile_first_row,
                       r.mtile_valid, status, mail, mail_seq);
    if (e != cudaSuccess) return e;
    if (blocks > 0)
        e = launch_chained(routing_scatter, dim3(blocks), dim3(kWarpsPerBlock * 32), sh_scat, stream, topk_idx, R, E, tile_m,
                           n_chunks, scratch, r.offsets, r.tile_offsets, r.perm, r.inv_perm, r.pad_row);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace

cudaError_t routing_prepare(int *max_cluster)
{
    cudaError_t e = cudaFuncSetAttribute(routing_onepass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOnepassMaxSmem);
    if (e != cudaSuccess) return e;
    // the kernels before and behind it want all shared memory: no SM has to change its split between L1 and shared memory
    e = cudaFuncSetAttribute(routing_onepass, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(routing_onepass, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    for (*max_cluster = kOnepassMaxCtas; *max_cluster > 8; *max_cluster >>= 1) {
        onepass_config(cfg, attr, *max_cluster, kOnepassMaxSmem, nullptr);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, routing_onepass, &cfg) == cudaSuccess && n > 0) break;
    }
    (void)cudaGetLastError();
    return cudaSuccess;
}

// A copy of the counts behind the build takes 9 us of the stream for a few hundred bytes (its hand-over, then the copy); stores
// of the build's last warp take one.
int32_t *host_writable(int32_t *tile_counts_host)
{
    cudaPointerAttributes a;
    if (!tile_counts_host) return nullptr;
    if (cudaPointerGetAttributes(&a, tile_counts_host) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    return a.type == cudaMemoryTypeHost ? static_cast<int32_t *>(a.devicePointer) : nullptr;
}

cudaError_t routing_launch(const int32_t *topk_idx, const moe_shape &s, int tile_m, const moe_routing &r, int32_t *scratch,
                           int max_cluster, uint32_t *status, unsigned long long *mail, uint32_t mail_seq, cudaStream_t stream)
{
    const int R = s.T * s.k_tot;
    const int n_ctas = onepass_ctas(R, max_cluster);
    if (n_ctas > 0 && onepass_smem(n_ctas, onepass_rows(R, n_ctas), s.E_tot) <= kOnepassMaxSmem)
        return routing_onepass_launch(topk_idx, s, tile_m, R, n_ctas, r, status, mail, mail_seq, stream);
    return routing_four_launches(topk_idx, s, tile_m, R, (R + kRoutingChunk - 1) / kRoutingChunk, r, scratch, status, mail, mail_seq, stream);
}

}  // namespace moe

// ------------------------------------------------------------------------------------------
// Routing build for callers that cannot allocate device memory.
//
// Some users of this library run where cudaMalloc is off limits: inside a serving loop whose
// memory pool was sized and frozen at start-up, under a framework allocator that forbids
// foreign allocations once a model is loaded, or in a latency-critical section where an
// allocation (an implicit device synchronisation) is not acceptable.  For them the per-warp
// histograms that the builder needs as scratch live in a fixed array inside the library instead
// of in a caller-provided buffer.  Every GPU that loads the library holds the array
// (kStaticScratchInts * 4 bytes) until the process exits.
//
// `g_static_scratch` is a device symbol: in host code the name is only a host-side stand-in, not
// a device address, so the address the kernels get comes from cudaGetSymbolAddress(), looked up
// once per device with that device current.
namespace moe {
namespace {

constexpr int kStaticScratchInts = 128 * 1024;   // 512 KiB per GPU
constexpr int kMaxStaticDevices = 64;

static __device__ __align__(256) int32_t g_static_scratch[kStaticScratchInts];
int32_t *g_static_scratch_addr[kMaxStaticDevices] = {nullptr};

}  // namespace
}  // namespace moe

extern "C" int32_t moe_build_routing_static(moe_handle *h, const int32_t *topk_idx, const moe_shape *s,
                                            int32_t tile_m, const moe_routing *r,
                                            int32_t *tile_counts_host, uint32_t *status_dev, void *stream)
{
    using namespace moe;
    if (!h || !s || !r || !status_dev) return MOE_ERR_NULL;
    if (s->T < 0 || s->k_tot < 1 || s->k_tot > 32 || s->E_tot < 1 || s->E_tot > 1024 ||
        (int64_t)s->T * s->k_tot >= (int64_t)1 << 30)
        return MOE_ERR_SHAPE;
    if (tile_m != 64 && tile_m != 128 && tile_m != 256) return MOE_ERR_UNSUPPORTED;
    if (s->T > 0 && !topk_idx) return MOE_ERR_NULL;
    const int64_t R = (int64_t)s->T * s->k_tot;
    if (r->max_mtiles < (int32_t)(R / tile_m + s->E_tot)) return MOE_ERR_SHAPE;
    const int64_t n_warps = (R + kRoutingChunk - 1) / kRoutingChunk;
    if (n_warps * s->E_tot > kStaticScratchInts) {
        snprintf(h->err, sizeof h->err,
                 "moe_build_routing_static: ceil(T*k_tot/%d) * E_tot = %lld ints of scratch needed, the built-in "
                 "array holds %d; use moe_build_routing with a caller-allocated workspace",
                 kRoutingChunk, (long long)(n_warps * s->E_tot), kStaticScratchInts);
        return MOE_ERR_STATIC_LIMIT;
    }
    if (h->device < 0 || h->device >= kMaxStaticDevices) return MOE_ERR_UNSUPPORTED;
    // Every call, not only the first: the kernels below run on the CURRENT device, and the array's
    // address is only meaningful on the device it was resolved for.  A caller whose current device
    // is not the handle's gets an error instead of kernels that dereference another GPU's address.
    {
        const int32_t rc = require_handle_device(h, "moe_build_routing_static");
        if (rc != MOE_OK) return rc;
    }

    // set-up, once per device: resolve the array's device address (the handle's device is current)
    int32_t *scratch = g_static_scratch_addr[h->device];
    if (!scratch) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) return cuda_fail(h, e, "cudaGetSymbolAddress(static scratch)");
        scratch = static_cast<int32_t *>(p);
        g_static_scratch_addr[h->device] = scratch;   // every writer stores the same value
    }

    // The array keeps whatever the previous call left in it.  Nothing has to start at zero: the
    // histogram pass overwrites every (warp, expert) entry the later passes read.
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t *const direct = host_writable(tile_counts_host);
    cudaError_t e = routing_launch(topk_idx, *s, tile_m, *r, scratch, h->routing_max_cluster, status_dev,
                                   reinterpret_cast<unsigned long long *>(direct), 0u, st);
    if (e != cudaSuccess) return cuda_fail(h, e, "static routing launch");
    if (tile_counts_host && !direct) {
        e = cudaMemcpyAsync(tile_counts_host, r->tiles, (size_t)(s->E_tot + 1) * 4, cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) return cuda_fail(h, e, "tile counts copy");
    }
    return MOE_OK;
}
