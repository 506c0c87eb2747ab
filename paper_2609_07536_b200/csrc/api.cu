// Host side of the C ABI: handle, workspace layout, argument validation, tensor maps, launches.

#include <climits>
#include <cstdint>
#include <cstring>
#include <new>

#include <algorithm>

#include "moe_internal.h"

#include <chrono>

namespace moe {

int32_t cuda_fail(moe_handle *h, cudaError_t e, const char *what)
{
    if (h) snprintf(h->err, sizeof h->err, "%s: %s", what, cudaGetErrorString(e));
    return MOE_ERR_CUDA;
}

int32_t require_handle_device(moe_handle *h, const char *who)
{
    int cur = -1;
    const cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaGetDevice");
    if (cur != h->device) {
        snprintf(h->err, sizeof h->err, "%s: the current CUDA device is %d, the handle was created on device %d",
                 who, cur, h->device);
        return MOE_ERR_UNSUPPORTED;
    }
    return MOE_OK;
}

Divisor divisor_of(int32_t d)
{
    // exact below 2^31: mul exceeds 2^shift / d by less than one
    Divisor r = {0u, 31u};
    while ((1ll << (r.shift - 31u)) < (long long)d) ++r.shift;
    r.mul = (uint32_t)(((1ull << r.shift) + (uint32_t)d - 1) / (uint32_t)d);
    return r;
}

// The table's entry for these arguments, encoded if it is another one's.
static const CUtensorMap *cached_map(moe_handle *h, const void *ptr, int32_t planes, int64_t rows, int32_t cols, int32_t box_rows, int rank,
                                     const cuuint64_t *dims, const cuuint64_t *strides, const cuuint32_t *box, const char *name)
{
    if (!h->maps && !(h->maps = new (std::nothrow) MapEntry[kMapEntries]())) return nullptr;
    MapEntry &m = h->maps[map_place(ptr, box_rows)];
    if (m.ptr == ptr && m.rows == rows && m.cols == cols && m.planes == planes && m.box_rows == box_rows) return &m.map;
    typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                      const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    m.ptr = nullptr;
    const CUresult cr = reinterpret_cast<EncodeTiledFn>(h->encode_tiled)(
        &m.map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(ptr), dims, strides, box, es,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) {
        snprintf(h->err, sizeof h->err, "cuTensorMapEncodeTiled(%s) failed: %d", name, (int)cr);
        return nullptr;
    }
    m.rows = rows;
    m.cols = cols;
    m.planes = planes;
    m.box_rows = box_rows;
    m.ptr = ptr;
    return &m.map;
}

const CUtensorMap *operand_map(moe_handle *h, const void *ptr, int32_t planes, int64_t rows, int32_t cols, int32_t box_rows, const char *name)
{
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * 2 * (cuuint64_t)rows};
    const cuuint32_t box[3] = {(cuuint32_t)kBlockK, (cuuint32_t)box_rows, 1};
    return cached_map(h, ptr, planes, rows, cols, box_rows, planes ? 3 : 2, dims, strides, box, name);
}

const CUtensorMap *gate_up_map(moe_handle *h, const void *ptr, int32_t experts, int32_t inter, int32_t cols, int32_t box_inter, const char *name)
{
    const cuuint64_t row = (cuuint64_t)cols * 2, plane = row * (cuuint64_t)inter;
    const cuuint64_t dims[5] = {(cuuint64_t)cols, 16, 2, (cuuint64_t)inter / 16, (cuuint64_t)experts};
    const cuuint64_t strides[4] = {row, plane, 16 * row, 2 * plane};
    const cuuint32_t box[5] = {(cuuint32_t)kBlockK, 16, 2, (cuuint32_t)box_inter / 16, 1};
    return cached_map(h, ptr, -experts, inter, cols, box_inter, 5, dims, strides, box, name);
}

namespace {

inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

constexpr int64_t kPairTileMinRowsPerExpert = 192;   // mean routed rows per expert from which 256-row pair tiles pay
constexpr int kSplitCounterWords = 64;  // 2 parities x MOE_MAX_L split counters (32-bit), then 2 x MOE_MAX_L work queues (64-bit), padded

bool shape_ok(const moe_shape *s)
{
    return s->T >= 0 && s->H >= 8 && s->I >= 16 && s->E_tot >= 1 && s->E_tot <= 1024 && s->k_tot >= 1 &&
           s->k_tot <= 32 && s->TP >= 1 && s->TP <= 8 && s->EP >= 1 && s->EP <= MOE_MAX_EP && s->L >= 1 &&
           s->L <= MOE_MAX_L && s->H % 8 == 0 && s->I % s->TP == 0 && (s->I / s->TP) % 16 == 0 &&
           (int64_t)s->T * s->k_tot < (int64_t)1 << 30;
}
bool tile_ok(int tile_m, int tile_n)
{
    return ((tile_m == 64 || tile_m == 128) && tile_n_slot(tile_n) >= 0) || (tile_m == 256 && tile_n == 256);
}
bool tile_m_ok(int tile_m) { return tile_m == 64 || tile_m == 128 || tile_m == 256; }

int32_t max_mtiles_of(const moe_shape *s, int tile_m)
{
    return (int32_t)((int64_t)s->T * s->k_tot / tile_m + s->E_tot);
}
int32_t n_routing_warps(const moe_shape *s)
{
    return (int32_t)ceil_div((int64_t)s->T * s->k_tot, kRoutingChunk);
}

}  // namespace
}  // namespace moe

using namespace moe;

extern "C" {

int32_t moe_create(int32_t device, moe_handle **out)
{
    if (!out) return MOE_ERR_NULL;
    *out = nullptr;
    moe_handle *h = new (std::nothrow) moe_handle();
    if (!h) return MOE_ERR_CUDA;
    h->device = device;
    cudaError_t e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->G, cudaDevAttrMultiProcessorCount, device);
    int major = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
    if (e != cudaSuccess || major != 10) {
        delete h;
        return e != cudaSuccess ? MOE_ERR_CUDA : MOE_ERR_UNSUPPORTED;
    }
    cudaDriverEntryPointQueryResult q;
    e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &h->encode_tiled, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !h->encode_tiled) {
        delete h;
        return MOE_ERR_CUDA;
    }
    const int tns[3] = {64, 128, 256};
    for (int i = 0; i < 3; ++i) {
        e = fused_occupancy(tns[i], &h->o_comp[i]);
        if (e != cudaSuccess) {
            delete h;
            return MOE_ERR_CUDA;
        }
    }
    e = pair_occupancy(&h->o_pair, &h->max_pairs);
    if (e != cudaSuccess) {
        delete h;
        return MOE_ERR_CUDA;
    }
    e = routing_prepare(&h->routing_max_cluster);
    if (e == cudaSuccess) e = gemm1_prepare();
    if (e != cudaSuccess) {
        delete h;
        return MOE_ERR_CUDA;
    }
    cudaEvent_t ev = nullptr;
    e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        delete h;
        return MOE_ERR_CUDA;
    }
    h->counts_event = ev;
    // the count mailbox: a few KB of pinned host memory that the GPU addresses directly.  Without it (the
    // allocation or the mapping refused) the whole-step calls copy the counts and synchronise instead.
    constexpr size_t kMailBytes = (size_t)kMailWords * sizeof(unsigned long long);
    void *mail = nullptr, *mail_dev = nullptr;
    if (cudaHostAlloc(&mail, kMailBytes, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) {
        memset(mail, 0, kMailBytes);
        if (cudaHostGetDevicePointer(&mail_dev, mail, 0) == cudaSuccess && mail_dev) {
            h->mail_host = static_cast<unsigned long long *>(mail);
            h->mail_dev = static_cast<unsigned long long *>(mail_dev);
        } else {
            cudaFreeHost(mail);
        }
    }
    (void)cudaGetLastError();
    *out = h;
    return MOE_OK;
}

int32_t moe_destroy(moe_handle *h)
{
    if (h && h->staging) cudaFreeHost(h->staging);
    if (h && h->feed_stream) cudaStreamDestroy(h->feed_stream);
    for (int i = 0; h && i < 2; ++i)
        if (h->feed_events[i]) cudaEventDestroy(h->feed_events[i]);
    if (h && h->counts_event) cudaEventDestroy(static_cast<cudaEvent_t>(h->counts_event));
    if (h && h->mail_host) cudaFreeHost(h->mail_host);
    if (h) delete[] h->maps;
    if (h) delete[] h->plan_tables;
    delete h;
    return MOE_OK;
}

const char *moe_last_cuda_error(const moe_handle *h) { return h ? h->err : ""; }

int32_t moe_set_wait_limit_ns(moe_handle *h, uint64_t ns)
{
    if (!h) return MOE_ERR_NULL;
    h->wait_ns = ns;
    return MOE_OK;
}

int32_t moe_set_timeline(moe_handle *h, void *timeline_dev, size_t bytes)
{
    if (!h) return MOE_ERR_NULL;
    if (timeline_dev && !fused_timeline_build()) {
        snprintf(h->err, sizeof h->err, "moe_set_timeline: this library was built without -DMOE_TIMELINE=1");
        return MOE_ERR_UNSUPPORTED;
    }
    if (timeline_dev && (reinterpret_cast<uintptr_t>(timeline_dev) & 7u)) return MOE_ERR_ALIGN;
    h->timeline = static_cast<unsigned long long *>(timeline_dev);
    h->timeline_bytes = timeline_dev ? bytes : 0;
    return MOE_OK;
}

int32_t moe_set_probe(moe_handle *h, uint32_t probe_bits)
{
    if (!h) return MOE_ERR_NULL;
    if (probe_bits && !fused_timeline_build()) {
        snprintf(h->err, sizeof h->err, "moe_set_probe: this library was built without -DMOE_TIMELINE=1");
        return MOE_ERR_UNSUPPORTED;
    }
    if (probe_bits & ~63u) return MOE_ERR_SHAPE;
    h->probe = probe_bits;
    return MOE_OK;
}

int32_t moe_query_occupancy(moe_handle *h, int32_t tile_m, int32_t tile_n, moe_occupancy *occ,
                            moe_sm_limits *limits, moe_rho *rho)
{
    if (!h) return MOE_ERR_NULL;
    if (!tile_ok(tile_m, tile_n)) return MOE_ERR_UNSUPPORTED;
    if (occ) {
        occ->tile_m = tile_m;
        occ->tile_n = tile_n;
        occ->comm_tile_m = kCommTileM;
        occ->comm_tile_n = kCommTileN;
        // both roles are CTAs of the same kernel: one resident CTA per SM by shared memory
        const bool pair = (tile_m == 256);
        occ->o_comp = pair ? h->o_pair : h->o_comp[tile_n_slot(tile_n)];
        occ->o_comm = occ->o_comp;
        occ->comp_slot_sms = pair ? 2 : 1;
    }
    if (limits) {
        // a pair tile needs both CTAs of a cluster resident: count only SMs that can host one
        limits->G = (tile_m == 256) ? (2 * h->max_pairs < h->G ? 2 * h->max_pairs : h->G) : h->G;
        limits->C_max = h->G / 2;   // one-time saturation characterisation of this kernel family
        limits->force_comm_ctas = 0;
        limits->selector_off = 0;
        limits->default_C = 3;      // the fixed count of the upstream path (Section II-C)
        limits->drain_help = 1;
        limits->co_warps_max = fused_co_warps_max();
        limits->force_co_warps = -1;
        limits->C_co_max = 8;       // beside co-resident warps more dedicated CTAs than this never paid (one-time sweep)
        limits->dep_model = MOE_DEP_SPLIT;
        // Lower end of the co-resident family's legal set (one-time sweep).  One-CTA tiles: below 24 compute waves
        // co-resident warps lost 2-5 % (T = 1024: 19 waves; T = 2048: 37).  CTA-pair tiles: a co-resident warp takes
        // the shared memory of the seventh operand stage.  In a loop of equal steps w = 0 is the fastest at every size
        // (w = 0 / 1 / 2, 20 steps: T = 8192 346 / 362 / 357 us, 16384 663 / 681 / 672, 32768 1296 / 1326 / 1310; 400 steps, where
        // the power cap sets the clock: 386 / 412 / 405, 733 / 769 / 744, 1477 / 1536 / 1519); only between launches of other
        // candidates (the sweep) was w = 2 ahead, by 7 to 9 % from T = 16384 on.  The family is not offered (a forced w is
        // still honoured).
        limits->co_min_waves = (tile_m == 256) ? INT32_MAX : 24;
    }
    if (rho) {
        // One-time service-rate characterisation of this kernel family on B200 (Eq. 13), one constant per
        // GEMM tile shape (Section III-E: every kernel choice brings its own).  Reference run: DeepSeek-V2-
        // Lite shape, T = 4096, uniform routing, TP = 2, EP = 2, L = 2, K = 704; each role alone on its
        // share of the SMs at C = 32: time per communication wave (of 32-row tiles: the work is dealt out in units, so
        // that whole 128-row tiles per CTA would make the selector see waves that are not there) / time per compute wave.
        //   128x256: 19.7 us / 6.47 us ; 256x256 (CTA pair): 19.5 / 4.68 ; 128x128: 18.8 / 5.43
        // That was with a tile and a row of Y per K-shard, which the selector still counts (g = TP; k_tot * TP + 1 rows).  The launch has
        // tiles over all of I and k_tot + 1 rows whatever TP is; the same run on it: 10.0 / 5.56 ; 10.4 / 4.18 ; 10.4 / 3.12 for half
        // of a tile, that is 1.80, 2.50 and 3.35.  No constant is right for every TP, as the rows of the count grow with it.  Static
        // partition, 162 workloads of the DeepSeek shape, mean distance from the best C at TP = 1 / 2: these constants 2.9 / 1.8 %,
        // the ones measured now 4.8 / 1.9 %, the same restated for TP = 1 (9 rows, K = 1408) 1.7 / 2.4 %; with drain help 1.9 to 2.4 % for all.
        rho->K_ref = 704;
        rho->tile_m_ref = tile_m;
        rho->tile_n_ref = tile_n;
        if (tile_m == 256) rho->rho_ref = 4.17;
        else if (tile_n == 256) rho->rho_ref = 3.04;
        else if (tile_n == 128) rho->rho_ref = 3.46;
        else rho->rho_ref = 3.46 * 2.0;          // 64-wide tiles: Eq. 14 tile-area scaling from 128x128
        rho->D_ref = 2;
        rho->rows_ref = 8 * 2 + 1;
        rho->comm_cols_ref = 1024;
        rho->mode = MOE_RHO_LOCAL;
        // Warp-level capacity and bandwidth coupling, measured once on B200 (DeepSeek-V2-Lite shape):
        //   a communication CTA is 12 warps; alone it streams 68 GB/s (5.7 GB/s per warp), 148 of them together
        //   5.85 TB/s (the copy bandwidth): 5850 / 5.67 = 1030 warps saturate HBM;
        //   a co-resident warp beside a running GEMM serves 2.6-2.8 GB/s (2.2 times slower than a dedicated warp)
        //   and each one stretches the compute wave by 1.25 % (683 -> 704 -> 714 us of GEMM phase for w = 0, 1, 2,
        //   of which 2 % is the split-major tile order that w > 0 needs when L > 1: x is read once per split).
        //   the work is given out in single tokens of a communication tile (T_M^comm pieces per tile).
        rho->comm_warps_per_cta = 12;
        rho->comm_quanta_per_tile = kCommTileM;
        rho->reserved0 = 0;
        rho->n_sat_warps = 1030;
        rho->co_beta = 0.0125;
        rho->co_gamma = 2.2;
        rho->co_order = 0.02;
    }
    return MOE_OK;
}

int32_t moe_select_tile(moe_handle *h, const moe_shape *s, int32_t *tile_m, int32_t *tile_n)
{
    if (!h || !s || !tile_m || !tile_n) return MOE_ERR_NULL;
    if (!shape_ok(s)) return MOE_ERR_SHAPE;
    // Conventional kernel dispatch (Section III-E: it runs before the resource manager and hands it the tile
    // shape and residency of the kernel it chose).  Widest n-tile the split holds; rows: a tile costs the rows that it has, rounded
    // up to 16 (a pair's: 32), in both families.  The 256-row CTA-pair tile moves a third less operand traffic per FLOP, and an
    // expert of 129 to 256 rows is one tile that reads its weights once, not two; it needs two co-scheduled SMs, so that there are half as
    // many places for tiles.  Measured, whole fused step and whole layer, 128 x 256 against 256 x 256, us, skewed routing, at
    // 64 / 128 / 160 / 192 / 256 / 400 rows per expert:
    //   Granite shape  step 40/39  44/42  45/44  49/44  52/48  64/56   layer  77/78  82/82  87/85  100/85  102/88  122/114
    //   Qwen shape     step 88/95  98/99  111/104  120/108  139/118  178/157   layer  208/215  234/234  258/241  286/255  336/299  453/420
    //   DeepSeek shape step 95/103  110/112  122/117  126/120  152/132  190/157   layer  234/244  258/269  287/277  308/293  371/325  490/428
    // From 192 on the pair is ahead by 5 to 17 % in all of them, up to 128 rows 128-row tiles are, by up to 8 % (Granite shape: equal).
    // Between 129 and 191 the pair is ahead at these shapes too, by 2 to 16 %, once most experts have more than 128 rows; not where
    // experts are so few that their 128-row tiles fit one wave on narrow columns, and the line has not been drawn between the two.
    const int64_t split_w = ceil_div(s->H, s->L);
    const int32_t tn = split_w >= 256 ? 256 : split_w >= 128 ? 128 : 64;
    const int64_t rows_per_expert = (int64_t)s->T * s->k_tot / s->E_tot;
    const bool pair = tn == 256 && h->max_pairs > 0 && rows_per_expert >= kPairTileMinRowsPerExpert;
    *tile_m = pair ? 256 : 128;
    *tile_n = tn;
    return MOE_OK;
}

int32_t moe_workspace_bytes(const moe_shape *s, int32_t tile_m, int32_t tile_n, size_t *routing_bytes,
                            size_t *y_bytes, size_t *flags_bytes, size_t *status_bytes)
{
    if (!s) return MOE_ERR_NULL;
    if (!shape_ok(s)) return MOE_ERR_SHAPE;
    if (!tile_ok(tile_m, tile_n)) return MOE_ERR_UNSUPPORTED;
    const size_t R = (size_t)s->T * s->k_tot, E = (size_t)s->E_tot;
    const size_t mt = (size_t)max_mtiles_of(s, tile_m);
    if (routing_bytes) {
        size_t b = 0;
        b += align16(E * 4) + 3 * align16((E + 1) * 4);  // counts, offsets, tiles(+S), tile_offsets
        b += 3 * align16(R * 4);                          // perm, inv_perm, pad_row
        b += 3 * align16(mt * 4);                         // m-tile table
        b += align16((size_t)n_routing_warps(s) * E * 4); // per-warp histograms
        *routing_bytes = b + 16;
    }
    // (the sum over the K-shards is taken in the accumulators: neither depends on TP)
    if (y_bytes)   // token-major: [T][L][k_tot][ceil(H/L)]
        *y_bytes = align16((size_t)s->T * s->L * s->k_tot * (size_t)ceil_div(s->H, s->L) * 2) + 16;
    if (flags_bytes) {
        const size_t nts = (size_t)ceil_div(ceil_div(s->H, s->L), tile_n);
        const size_t parts = (tile_m == 256) ? 2 : 1;   // a pair tile is published in two parts
        *flags_bytes = ((size_t)kSplitCounterWords + (size_t)s->L * mt * nts * parts) * 4 + 16;
    }
    if (status_bytes) *status_bytes = 16;
    return MOE_OK;
}

int32_t moe_routing_view(void *ws, const moe_shape *s, int32_t tile_m, moe_routing *out)
{
    if (!ws || !s || !out) return MOE_ERR_NULL;
    if (!shape_ok(s)) return MOE_ERR_SHAPE;
    if (!tile_m_ok(tile_m)) return MOE_ERR_UNSUPPORTED;
    if (!aligned16(ws)) return MOE_ERR_ALIGN;
    const size_t R = (size_t)s->T * s->k_tot, E = (size_t)s->E_tot;
    const size_t mt = (size_t)max_mtiles_of(s, tile_m);
    char *p = static_cast<char *>(ws);
    auto take = [&](size_t n_ints) {
        int32_t *q = reinterpret_cast<int32_t *>(p);
        p += align16(n_ints * 4);
        return q;
    };
    out->counts = take(E);
    out->offsets = take(E + 1);
    out->tiles = take(E + 1);
    out->tile_offsets = take(E + 1);
    out->perm = take(R);
    out->inv_perm = take(R);
    out->pad_row = take(R);
    out->mtile_expert = take(mt);
    out->mtile_first_row = take(mt);
    out->mtile_valid = take(mt);
    out->scratch = take((size_t)n_routing_warps(s) * E);
    out->max_mtiles = (int32_t)mt;
    return MOE_OK;
}

int32_t moe_build_routing(moe_handle *h, const int32_t *topk_idx, const moe_shape *s, int32_t tile_m,
                          const moe_routing *r, int32_t *tile_counts_host, uint32_t *status_dev, void *stream)
{
    if (!h || !s || !r || !status_dev) return MOE_ERR_NULL;
    if (!shape_ok(s)) return MOE_ERR_SHAPE;
    if (!tile_m_ok(tile_m)) return MOE_ERR_UNSUPPORTED;
    if (s->T > 0 && !topk_idx) return MOE_ERR_NULL;
    if (r->max_mtiles < max_mtiles_of(s, tile_m)) return MOE_ERR_SHAPE;
    if (const int32_t rc = require_handle_device(h, "moe_build_routing")) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t *const direct = host_writable(tile_counts_host);
    cudaError_t e = routing_launch(topk_idx, *s, tile_m, *r, r->scratch, h->routing_max_cluster, status_dev,
                                   reinterpret_cast<unsigned long long *>(direct), 0u, st);
    if (e != cudaSuccess) return cuda_fail(h, e, "routing launch");
    if (tile_counts_host && !direct) {
        e = cudaMemcpyAsync(tile_counts_host, r->tiles, (size_t)(s->E_tot + 1) * 4, cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) return cuda_fail(h, e, "tile counts copy");
    }
    return MOE_OK;
}

}  // extern "C"

namespace {

// Routing build of the whole-step calls.  With the handle's mailbox a kernel stores the counts into host memory and
// `*seq` is the number to wait for (wait_counts): the build itself, or (`mail_later`) a launch behind it, which may also build the
// routing (`launch_builds`: nothing is launched here).  Without the mailbox, the plain build with its copy, and `*seq` = 0.
int32_t build_routing_mailed(moe_handle *h, const int32_t *topk_idx, const moe_shape *s, int32_t tile_m, const moe_routing *r,
                             int32_t *tile_counts_host, bool mail_later, bool launch_builds, uint32_t *status_dev, cudaStream_t st,
                             uint32_t *seq)
{
    *seq = 0;
    if ((!tile_counts_host || !h->mail_dev) && !launch_builds)
        return moe_build_routing(h, topk_idx, s, tile_m, r, tile_counts_host, status_dev, st);
    if (!s || !r || !status_dev) return MOE_ERR_NULL;
    if (!shape_ok(s)) return MOE_ERR_SHAPE;
    if (!tile_m_ok(tile_m)) return MOE_ERR_UNSUPPORTED;
    if (s->T > 0 && !topk_idx) return MOE_ERR_NULL;
    if (r->max_mtiles < max_mtiles_of(s, tile_m)) return MOE_ERR_SHAPE;
    if (const int32_t rc = require_handle_device(h, "moe_build_routing")) return rc;
    if (++h->mail_seq == 0u) h->mail_seq = 1u;
    if (!launch_builds) {
        const cudaError_t e = routing_launch(topk_idx, *s, tile_m, *r, r->scratch, h->routing_max_cluster, status_dev,
                                             mail_later ? nullptr : h->mail_dev, h->mail_seq, st);
        if (e != cudaSuccess) return cuda_fail(h, e, "routing launch");
    }
    *seq = tile_counts_host ? h->mail_seq : 0u;
    return MOE_OK;
}

// Waits until the counts of build `seq` are on the host and copies them to tile_counts_host (E_tot + 1 ints).
// seq = 0: they come by the stream's copy: `fallback_event` if given (recorded behind that copy), else the stream.
int32_t wait_counts(moe_handle *h, uint32_t seq, int32_t E_tot, int32_t *tile_counts_host, cudaStream_t st, cudaEvent_t fallback_event)
{
    if (seq == 0u) {
        const cudaError_t e = fallback_event ? cudaEventSynchronize(fallback_event) : cudaStreamSynchronize(st);
        return e == cudaSuccess ? MOE_OK : cuda_fail(h, e, "tile counts wait");
    }
    const volatile unsigned long long *words = h->mail_host;
    const auto t0 = std::chrono::steady_clock::now();
    uint32_t spins = 0;
    bool finished = false;
    for (int32_t x = 0; x <= E_tot; ++x) {
        unsigned long long v;
        while ((uint32_t)((v = words[x]) >> 32) != seq) {
            if ((++spins & 2047u) == 0u) {
                // the kernels finished or failed without the word arriving?
                if (finished) {
                    snprintf(h->err, sizeof h->err, "the routing build finished without delivering the tile counts");
                    return MOE_ERR_CUDA;
                }
                const cudaError_t q = cudaStreamQuery(st);
                if (q == cudaSuccess) finished = true;      // one more look at the words
                else if (q != cudaErrorNotReady) return cuda_fail(h, q, "routing build");
                const double waited = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
                if (waited > 2.0 + 2e-9 * (double)h->wait_ns) {
                    snprintf(h->err, sizeof h->err, "no tile counts from the routing build after %.1f s", waited);
                    return MOE_ERR_CUDA;
                }
            }
#if defined(__x86_64__) || defined(__i386__)
            __builtin_ia32_pause();
#endif
        }
        tile_counts_host[x] = (int32_t)(uint32_t)v;
    }
    return MOE_OK;
}

// The most m-tiles that a routing of this shape can have: an expert with rows has at most (rows - 1) / tile_m + 1.
int64_t most_mtiles(const moe_shape *s, int tile_m)
{
    const int64_t R = (int64_t)s->T * s->k_tot, used = R < s->E_tot ? R : s->E_tot;
    return (R - used) / tile_m + used;
}
// column slab of one unit: the largest power of two with k_tot * columns * 2 <= 8 KB, at most 1024
int slab_shift_of(const moe_shape *s)
{
    int sh = 10;
    while (sh > 3 && ((int64_t)s->k_tot << sh) * 2 > 8192) --sh;
    return sh;
}
// Who serves what when the compute CTAs help: a queue per split, or, up to 32 units (of 8 KB) a warp, an even share for every
// warp once the tiles are done.  Hardly any token is complete before the last tiles are, so the queue's early start is
// worth little, while its atomics and its polling cost microseconds at the end; with many units the queue's balance wins.  Whole
// step, queue / even, us, timed in turns, at 8 / 16 / 24 / 32 / 40 / 48 / 64 units a warp:
//   Granite shape, L = 1   102/91  165/152  228/217  294/286  357/353  425/421  564/567 (T = 4736 to 37888)
//   Qwen shape, L = 1      187/170  321/288  467/429  612/574  760/716  905/866  1194/1167 (T = 7104 to 56832)
//   DeepSeek shape, L = 1  178/172  297/292  427/421  560/564  699/716  838/860  1137/1175 (T = 3552 to 28416)
//   DeepSeek shape, L = 2  183/175  307/294  435/424  569/565  717/724  848/861  1139/1157
// The lines lie between 26 and 56 units; up to 32 the even shares are at most 1 % behind, above it up to 6 % ahead (Qwen shape) or 3 %
// behind (DeepSeek shape).
bool few_units(const moe_handle *h, const moe_shape *s)
{
    const int64_t split_w = ceil_div(s->H, s->L);
    return (int64_t)s->T * s->L * ceil_div(split_w, 1 << slab_shift_of(s)) <= 32ll * 12 * h->G;
}

// Whether a whole-step launch with these limits divides its CTAs by itself whatever the counts turn out to be (even shares, no C
// asked for, no co-resident warps): such a launch needs no selection, and goes out before the counts are on the host, at a
// batch size that was never seen before as well (32 sizes in turn, 15 us a step as with repeated ones; 52 when the picks for all
// counts had to be tabulated first).  The tiles are those of the launch, over all of I: counted per K-shard, as the selector does, the same
// launch at TP = 2 took co-resident warps, the queue, or the wait for the counts that it does without at TP = 1 (whole step, TP = 1 / 2, us: H = 4096,
// otherwise the DeepSeek shape, L = 2, T = 1200 196 / 203, T = 1500 215 / 226; the DeepSeek shape on 128 x 128 tiles, T = 1024 110 / 117, T = 2048 158 / 169).
bool divides_itself(const moe_handle *h, const moe_shape *s, const moe_occupancy *occ, const moe_sm_limits *lim)
{
    if (!lim->drain_help || lim->force_comm_ctas > 0 || lim->selector_off || lim->C_max < 1 || s->T < 1 || !few_units(h, s)) return false;
    const int slot = occ->comp_slot_sms;
    if (occ->o_comp != 1 || occ->o_comm != 1 || lim->G <= slot || lim->G > (slot == 2 ? 2 * h->max_pairs : h->G)) return false;   // (else: what the launch says to the plan)
    const int64_t NTs = ceil_div(ceil_div(s->H, s->L), occ->tile_n);
    if ((int64_t)max_mtiles_of(s, occ->tile_m) * NTs * s->L >= (int64_t)1 << 30) return false;     // (too many tiles: the wait knows better)
    const int32_t w_top = lim->force_co_warps >= 0 && lim->force_co_warps < lim->co_warps_max ? lim->force_co_warps : lim->co_warps_max;
    if (w_top < 1) return true;
    if (lim->force_co_warps >= 0) return false;
    // the selector tries co-resident warps from co_min_waves waves on, with C up to C_co_max
    const int32_t C_most = lim->C_co_max < lim->C_max ? lim->C_co_max : lim->C_max;
    if (C_most < 1) return true;
    const int64_t P_least = (lim->G - C_most) / slot, tiles = (int64_t)s->L * most_mtiles(s, occ->tile_m) * NTs;
    return P_least >= 1 && ceil_div(tiles, P_least) < lim->co_min_waves;
}

// What the handle knows of the selection for this shape, tile family and limits: the table where one is made (n > 0), else an
// entry to make it in (nullptr: the allocation failed).  The entry used longest ago goes first.
PlanTable *plan_table(moe_handle *h, const moe_shape *s, const moe_occupancy *occ, const moe_sm_limits *lim)
{
    if (!h->plan_tables && !(h->plan_tables = new (std::nothrow) PlanTable[kPlanTables]())) return nullptr;
    PlanTable *old = &h->plan_tables[0];
    for (int i = 0; i < kPlanTables; ++i) {
        PlanTable &t = h->plan_tables[i];
        if (t.last_use && t.tile_m == occ->tile_m && t.tile_n == occ->tile_n && memcmp(&t.shape, s, sizeof *s) == 0 &&
            memcmp(&t.limits, lim, sizeof *lim) == 0) {
            t.last_use = ++h->plan_table_uses;
            t.again = true;
            return &t;
        }
        if (t.last_use < old->last_use) old = &t;
    }
    old->shape = *s;
    old->tile_m = occ->tile_m;
    old->tile_n = occ->tile_n;
    old->limits = *lim;
    old->n = -1;
    old->again = false;
    old->last_use = ++h->plan_table_uses;
    return old;
}

// Tabulates the selection for every m-tile count of the shape (0.5 us each, 17-43 us in all); n = 0 where the launch has to wait for
// the counts: more m-tile counts than a table holds, tile-level readiness (it depends on more than the sum of the counts),
// or picks that differ in what the launch configuration fixes (grid, co-resident warps).
void tabulate(PlanTable &t, const moe_occupancy *occ, const moe_rho *rho)
{
    t.n = 0;
    const moe_shape *s = &t.shape;
    const moe_sm_limits *lim = &t.limits;
    const int64_t R = (int64_t)s->T * s->k_tot, first = ceil_div(R, occ->tile_m), last = most_mtiles(s, occ->tile_m);
    if (R < 1 || last - first + 1 > kPlanTableMax || occ->o_comp != 1 || occ->o_comm != 1 ||
        (!lim->drain_help && lim->dep_model == MOE_DEP_TILE))
        return;
    const int slot = occ->comp_slot_sms;
    for (int64_t S = first; S <= last; ++S) {
        const int32_t count = (int32_t)S;
        moe_plan p;
        if (plan_partition(&count, 1, occ, lim, s, rho, &p) != MOE_OK) return;
        if (S == first) t.plan = p;
        const int c_slots = slot == 2 ? (p.comm_ctas + 1) & ~1 : p.comm_ctas, c0 = slot == 2 ? (t.plan.comm_ctas + 1) & ~1 : t.plan.comm_ctas;
        if (p.comm_ctas < 1 || p.comm_ctas > 255 || p.co_warps != t.plan.co_warps || p.P != (lim->G - p.comm_ctas) / slot ||
            c_slots + slot * p.P != c0 + slot * t.plan.P)
            return;
        t.C[S - first] = (uint8_t)p.comm_ctas;
    }
    t.first = (int32_t)first;
    t.n = (int32_t)(last - first + 1);
}

// moe_gemm2_combine with the launch's plan, or (`table`) with the plan looked up on the device by the m-tile count;
// own_division: an even launch may divide its CTAs itself; mail_seq != 0: this launch mails the counts; topk_idx != nullptr: it builds the routing first (m-tile count on the device)
int32_t launch_gemm2_combine(moe_handle *h, const void *x_routed, const void *W2, const float *topk_w, const moe_shape *s,
                             const moe_occupancy *occ, const moe_routing *r, int32_t n_mtiles, const moe_plan *plan,
                             bool own_division, const PlanTable *table, uint32_t mail_seq, const int32_t *topk_idx, const RowFeed *feed,
                             void *const *out, void *y_ws, uint32_t *flags_ws, uint32_t *status_dev, void *stream);

}  // namespace

extern "C" {

int32_t moe_gemm2_combine(moe_handle *h, const void *x_routed, const void *W2, const int32_t *topk_idx,
                          const float *topk_w, const moe_shape *s, const moe_occupancy *occ,
                          const moe_routing *r, int32_t n_mtiles, const moe_plan *plan, void *const *out,
                          void *y_ws, uint32_t *flags_ws, uint32_t *status_dev, void *stream)
{
    (void)topk_idx;
    return launch_gemm2_combine(h, x_routed, W2, topk_w, s, occ, r, n_mtiles, plan, false, nullptr, 0u, nullptr, nullptr, out, y_ws, flags_ws, status_dev, stream);
}

}  // extern "C"

namespace {

int32_t launch_gemm2_combine(moe_handle *h, const void *x_routed, const void *W2, const float *topk_w, const moe_shape *s,
                             const moe_occupancy *occ, const moe_routing *r, int32_t n_mtiles, const moe_plan *plan,
                             bool own_division, const PlanTable *table, uint32_t mail_seq, const int32_t *topk_idx, const RowFeed *feed,
                             void *const *out, void *y_ws, uint32_t *flags_ws, uint32_t *status_dev, void *stream)
{
    if (!h || !s || !occ || !r || !plan || !out || !status_dev) return MOE_ERR_NULL;
    if (!shape_ok(s)) return MOE_ERR_SHAPE;
    if (!tile_ok(occ->tile_m, occ->tile_n)) return MOE_ERR_UNSUPPORTED;
    if (occ->comm_tile_m != kCommTileM || occ->comm_tile_n != kCommTileN) return MOE_ERR_UNSUPPORTED;
    if ((ceil_div(s->H, s->L) % 8) != 0) return MOE_ERR_SHAPE;   // 16-byte column chunks per split
    if (s->T == 0) return MOE_OK;
    if (!x_routed || !W2 || !topk_w || !y_ws || !flags_ws) return MOE_ERR_NULL;
    const bool counts_on_device = (n_mtiles == MOE_MTILES_ON_DEVICE);
    if (counts_on_device) n_mtiles = r->max_mtiles;   // bound for the sizes checked on the host
    if (n_mtiles < 0 || n_mtiles > r->max_mtiles) return MOE_ERR_SHAPE;
    if (!aligned16(x_routed) || !aligned16(W2) || !aligned16(y_ws) || !aligned16(flags_ws) ||
        !aligned16(status_dev))
        return MOE_ERR_ALIGN;
    for (int d = 0; d < s->EP; ++d) {
        if (!out[d]) return MOE_ERR_NULL;
        if (!aligned16(out[d])) return MOE_ERR_ALIGN;
    }
    const int mode = plan->mode;
    if (mode != MOE_MODE_FUSED && mode != MOE_MODE_GEMM_ONLY && mode != MOE_MODE_COMBINE_ONLY)
        return MOE_ERR_SHAPE;
    const int C = (mode == MOE_MODE_GEMM_ONLY) ? 0 : plan->comm_ctas;
    const int Pc = (mode == MOE_MODE_COMBINE_ONLY) ? 0 : plan->P;
    const int o_comp = occ->o_comp > 0 ? occ->o_comp : 1, o_comm = occ->o_comm > 0 ? occ->o_comm : 1;
    const bool pair = (occ->tile_m == 256);
    const int slot_sms = pair ? 2 : 1;
    if (occ->comp_slot_sms != slot_sms) return MOE_ERR_UNSUPPORTED;
    // without a communication CTA somebody else has to serve the communication work: the compute CTAs, once
    // their GEMM tiles are done (drain help)
    if (mode != MOE_MODE_GEMM_ONLY && (C < 0 || (C < 1 && !(mode == MOE_MODE_FUSED && plan->drain_help))))
        return MOE_ERR_PLAN_INFEASIBLE;
    if (plan->co_warps < 0 || plan->co_warps > kCoWarpsMax) return MOE_ERR_PLAN_INFEASIBLE;
    if (mode != MOE_MODE_COMBINE_ONLY && Pc < 1) return MOE_ERR_PLAN_INFEASIBLE;
    if (mode == MOE_MODE_FUSED && (int64_t)plan->R * o_comm < C) return MOE_ERR_PLAN_INFEASIBLE;
    // every CTA must be resident at once: spinning communication CTAs may never keep a compute
    // CTA off the GPU (Section II-C: the legal set keeps positive compute capacity)
    if (ceil_div(C, o_comm) + ceil_div(Pc, o_comp) * slot_sms > h->G) return MOE_ERR_PLAN_INFEASIBLE;
    if (pair && (((C + 1) & ~1) + 2 * Pc > 2 * h->max_pairs)) return MOE_ERR_PLAN_INFEASIBLE;
    if (const int32_t rc = require_handle_device(h, "moe_gemm2_combine")) return rc;

    FusedParams p;
    memset(&p, 0, sizeof p);
    // the sum over the K-shards is taken in the accumulators: a tile runs over all of I, whatever TP is
    p.T = s->T; p.H = s->H; p.EP = s->EP; p.L = s->L; p.k_tot = s->k_tot;
    p.S = n_mtiles;
    p.tile_m = occ->tile_m;
    p.flag_parts = pair ? 2 : 1;
    p.split_w = (int32_t)ceil_div(s->H, s->L);
    p.NTs = (int32_t)ceil_div(p.split_w, occ->tile_n);
    const int64_t Wc = (int64_t)n_mtiles * p.NTs;
    if (Wc * s->TP * s->L * 2 >= (int64_t)1 << 31) return MOE_ERR_SHAPE;   // (the plan's count, a tile per K-shard)
    p.W_comp = (int32_t)Wc;
    p.S_dev = counts_on_device ? r->tiles + s->E_tot : nullptr;
    p.C = C; p.P = Pc; p.mode = mode;
    // (the plan counts a tile per K-shard: split, m-tile, shard, n-tile)
    p.withhold = plan->debug_withhold_tile < 0 ? -1 : plan->debug_withhold_tile / (s->TP * p.NTs) * p.NTs + plan->debug_withhold_tile % p.NTs;
    p.G = h->G;
    p.slot_sms = slot_sms;
    p.E_tot = s->E_tot;
    if (topk_idx) p.routing = {topk_idx, routing_out(*r), s->T * s->k_tot, r->max_mtiles};
    if (table) {
        p.G = table->limits.G;
        p.c_table_first = table->first;
        p.c_table_n = table->n;
        memcpy(p.c_table, table->C, (size_t)table->n);
    }
    if (mail_seq != 0u) {
        p.mail = h->mail_dev;
        p.mail_seq = mail_seq;
    }
    p.drain_help = (mode == MOE_MODE_FUSED && plan->drain_help) ? 1 : 0;
    p.tok_blk = (int32_t)ceil_div(s->T, s->EP);
    p.by_k = divisor_of(s->k_tot);
    p.comm_cols = (int32_t)ceil_div(p.split_w, kCommTileN);
    p.num_kb = (int32_t)ceil_div(s->I, kBlockK);
    p.last_ksteps = (s->I - (p.num_kb - 1) * kBlockK) / kUmmaK;
    p.R_pad = (long long)occ->tile_m * n_mtiles;
    p.wait_ns = h->wait_ns;
    p.mtile_expert = r->mtile_expert;
    p.mtile_first_row = r->mtile_first_row;
    p.mtile_valid = r->mtile_valid;
    p.pad_row = r->pad_row;
    p.perm = r->perm;
    p.slab_shift = slab_shift_of(s);
    p.slab_cols = 1 << p.slab_shift;
    p.topk_w = topk_w;
    p.Y = y_ws;
    p.status = status_dev;
    for (int d = 0; d < s->EP; ++d) p.out[d] = out[d];
    if (feed) {
        p.x_ready = feed->ready;
        p.wait_ns += feed->extra_wait_ns;
    }
    // Co-resident communication warps need the dynamic hand-out (they pull from the queues) and units of at most 16
    // rows; where one of these does not hold the launch runs without them (same result, bit for bit).
    p.co_warps = plan->co_warps < fused_co_warps_max() ? plan->co_warps : fused_co_warps_max();
    if (!p.drain_help || s->k_tot > 16) p.co_warps = 0;
    // warps 16-19 of a compute CTA: co-resident communication warps, or -- when none is asked for -- a fourth
    // epilogue column group (a third less epilogue work per warp: what bounds tiles with a short K)
    p.epi_warps = p.co_warps == 0 ? 16 : 12;
    // Tile sequence: split-major (the paper's) whenever something consumes a split while the next one is
    // computed; m-tile-major across the splits (x is read from DRAM once) when nothing does
    p.tile_order = (plan->drain_help && p.co_warps == 0) ? 1 : 0;
    const int64_t R = (int64_t)s->T * s->k_tot;
    p.dry_rows = (int32_t)(R / s->E_tot < occ->tile_m ? R / s->E_tot + 1 : occ->tile_m);
    p.w2_once = R <= (int64_t)s->E_tot * kMmaM;    // at most one 128-row tile per expert on average
    // Even shares or the queue (few_units).  Co-resident warps draw on the queue; a launch with a withheld tile is about that
    // tile's flag.
    p.even = p.drain_help && p.co_warps == 0 && plan->debug_withhold_tile < 0 && few_units(h, s);
    int TN = occ->tile_n, ctas_c = C, ctas_p = Pc;
    // In a whole-step call with no C asked for, such a launch divides its CTAs by itself, from the m-tile count that it reads
    // (launch_part): the plan's C is taken for communication beside the GEMM, of which there is none, and on counts left on
    // the device it comes from an estimate, which costs up to a wave.
    p.balance = p.even && own_division;
    if (p.balance) {
        p.C = ctas_c = 0;                                        // slots to divide: all of the plan's
        p.P = ctas_p = pair ? Pc + (C + 1) / 2 : Pc + C;
        p.c_table_n = 0;
    }
    if (p.even && !pair) {
        // One wave: where every tile that this routing can have finds an SM of its own among the plan's, all of them compute (a
        // communication CTA would have nothing to do until the only wave ends), on the narrowest tiles for which that holds
        // (the time of a wave is the time to stream and store one tile: DeepSeek shape, T = 1, 19 -> 16 us).
        const int64_t bound = most_mtiles(s, occ->tile_m), S_max = counts_on_device && bound < n_mtiles ? bound : n_mtiles;
        for (int tn = 64; tn <= occ->tile_n; tn *= 2) {
            if (S_max * s->L * ceil_div(p.split_w, tn) > C + Pc) continue;
            TN = tn;
            p.NTs = (int32_t)ceil_div(p.split_w, TN);
            p.W_comp = n_mtiles * p.NTs;
            p.C = ctas_c = 0;
            p.P = ctas_p = C + Pc;
            p.c_table_n = 0;
            break;
        }
    }

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    // launch epoch of this workspace: a flag equal to the epoch means "ready in this launch"
    uint32_t &ep = h->epochs[flags_ws];
    ep += 1u;
    if (ep == 0u) {  // wrapped: start over from a clean workspace
        size_t fb = 0;
        moe_workspace_bytes(s, occ->tile_m, occ->tile_n, nullptr, nullptr, &fb, nullptr);
        e = cudaMemsetAsync(flags_ws, 0, fb - 16, st);
        if (e != cudaSuccess) return cuda_fail(h, e, "flags reset");
        ep = 1u;
    }
    p.epoch = ep;
    p.split_done = flags_ws + (ep & 1u) * MOE_MAX_L;
    p.split_done_next = flags_ws + ((ep + 1u) & 1u) * MOE_MAX_L;
    p.queue = reinterpret_cast<unsigned long long *>(flags_ws + 2 * MOE_MAX_L) + (ep & 1u) * MOE_MAX_L;
    p.queue_next = reinterpret_cast<unsigned long long *>(flags_ws + 2 * MOE_MAX_L) + ((ep + 1u) & 1u) * MOE_MAX_L;
    p.flags = flags_ws + kSplitCounterWords;

    // operands (Section II-A): x_routed [R, I] and W2 [E_tot, H, I], k contiguous; a pair CTA loads half the n-tile's rows
    // (no m-tile has more rows than there are assignments, whatever the routing; a CTA of a pair holds half of them)
    const int64_t most_rows = R < occ->tile_m ? R : occ->tile_m, cta_rows = pair ? ((most_rows + 31) & ~31ll) / 2 : most_rows;
    p.x_rows = cta_rows <= 32 && !pair ? 32 : cta_rows <= 64 ? 64 : kMmaM;
    CUtensorMap *const mA[3] = {&p.tmA, &p.tmA64, &p.tmA32};
    for (int i = 0, first = p.x_rows == kMmaM ? 0 : p.x_rows == 64 ? 1 : 2; i < (pair ? 2 : 3); ++i) {
        // the boxes that the launch can need; in the place of a wider one a map that it does not use stands for the prefetch of the first
        const CUtensorMap *m = operand_map(h, x_routed, 0, R, s->I, 128 >> (i < first ? first : i), "x_routed");
        if (!m) return MOE_ERR_CUDA;
        *mA[i] = *m;
    }
    const CUtensorMap *mB = operand_map(h, W2, s->E_tot, s->H, s->I, pair ? TN / 2 : TN, "W2");
    if (!mB) return MOE_ERR_CUDA;
    p.tmB = *mB;
    p.stages = fused_stages(pair, TN, p.x_rows, p.co_warps == 0, &p.stage_bytes);
    const int grid = pair ? ((ctas_c + 1) & ~1) + 2 * ctas_p : ctas_c + ctas_p;
    p.timeline = nullptr;
    if (h->timeline && h->timeline_bytes >= ((size_t)grid * kTimelineSlots + MOE_MAX_L) * sizeof(unsigned long long))
        p.timeline = h->timeline;
    p.probe = h->probe;
    e = pair ? pair_launch(p, grid, st) : fused_launch(TN, p, grid, st);
    if (e != cudaSuccess) return cuda_fail(h, e, "fused launch");
    return MOE_OK;
}

// What a whole-step call selects with.
struct Selection {
    moe_occupancy occ;
    moe_sm_limits lim;
    moe_rho rho;
    bool alone;            // divides_itself
    bool divides;          // ... with the counts on the host wanted
    PlanTable *table;      // else, with the counts on the host wanted: plan_table
    // whether the fused launch goes out before the counts are on the host
    bool launch_first() const { return divides || (table && table->n > 0); }
};
int32_t selection_of(moe_handle *h, const moe_shape *s, int32_t tile_m, int32_t tile_n, const moe_sm_limits *limits_or_null,
                     bool host_counts, Selection *sel)
{
    if (!shape_ok(s)) return MOE_ERR_SHAPE;
    const int32_t rc = moe_query_occupancy(h, tile_m, tile_n, &sel->occ, &sel->lim, &sel->rho);
    if (rc != MOE_OK) return rc;
    if (limits_or_null) sel->lim = *limits_or_null;
    const bool mailed = host_counts && h->mail_dev;
    sel->alone = divides_itself(h, s, &sel->occ, &sel->lim);
    sel->divides = mailed && sel->alone;
    sel->table = mailed && !sel->divides ? plan_table(h, s, &sel->occ, &sel->lim) : nullptr;
    return MOE_OK;
}

// What the whole-step calls do after the routing build (and GEMM1): select, launch, and have the counts on the host.
// Where the launch divides its CTAs by itself, or the selection is tabulated, it goes out at once, queued behind its
// predecessor without a gap, and the host waits for the counts and plans afterwards, beside the running kernel (step of the
// tiny configuration 20.5 -> 16 us, of the DeepSeek shape at T = 16 76.7 -> 71); otherwise it waits first, and from a
// selection's second call on makes the table behind the launch.  `mail_seq` != 0: a launch that goes out first mails the counts.  `counts_event`: recorded behind the counts' copy, for a build without the mailbox
// (seq = 0).
int32_t select_and_launch(moe_handle *h, const void *x_routed, const void *W2, const float *topk_w, const moe_shape *s,
                          const Selection &sel, const moe_routing *routing, uint32_t seq, uint32_t mail_seq,
                          const int32_t *topk_idx, const RowFeed *feed, cudaEvent_t counts_event, int32_t *tile_counts,
                          void *const *out, void *y_ws, uint32_t *flags_ws, uint32_t *status_dev, moe_plan *plan_out, void *ev_before, void *ev_after, cudaStream_t st)
{
    moe_plan plan;
    int32_t rc = MOE_OK, n_mtiles = MOE_MTILES_ON_DEVICE;
    auto counts_and_plan = [&]() -> int32_t {
        const int32_t r = wait_counts(h, seq, s->E_tot, tile_counts, st, counts_event);
        return r != MOE_OK ? r : plan_partition(tile_counts, s->E_tot, &sel.occ, &sel.lim, s, &sel.rho, &plan);
    };
    const bool first = sel.launch_first();
    const PlanTable *table = first && !sel.divides ? sel.table : nullptr;
    if (sel.divides) {
        const int slot = sel.occ.comp_slot_sms;         // (the launch divides all of G, whatever C is)
        memset(&plan, 0, sizeof plan);
        plan.comm_ctas = plan.R = 1;
        plan.P = (sel.lim.G - 1) / slot;
        plan.mode = MOE_MODE_FUSED;
        plan.debug_withhold_tile = -1;
        plan.drain_help = 1;
    } else if (table) {
        plan = table->plan;
    } else if (tile_counts) {
        if ((rc = counts_and_plan()) != MOE_OK) return rc;
        n_mtiles = tile_counts[s->E_tot];
    } else {
        if ((rc = plan_partition_estimate(&sel.occ, &sel.lim, s, &sel.rho, &plan)) != MOE_OK) return rc;   // counts stay on the device
    }
    if (ev_before) cudaEventRecord(static_cast<cudaEvent_t>(ev_before), st);
    const bool own_division = sel.lim.force_comm_ctas <= 0 && !sel.lim.selector_off;
    moe_plan launched = plan;
    if (sel.alone) launched.co_warps = 0;               // (the selector counts a tile per K-shard, and may have found waves enough for them)
    rc = launch_gemm2_combine(h, x_routed, W2, topk_w, s, &sel.occ, routing, n_mtiles, &launched, own_division, table, first ? mail_seq : 0u, topk_idx, feed, out, y_ws,
                              flags_ws, status_dev, st);
    if (ev_after) cudaEventRecord(static_cast<cudaEvent_t>(ev_after), st);
    if (rc == MOE_OK && first) rc = counts_and_plan();
    else if (rc == MOE_OK && sel.table && sel.table->again && sel.table->n < 0) tabulate(*sel.table, &sel.occ, &sel.rho);
    if (plan_out && rc == MOE_OK) *plan_out = plan;
    return rc;
}

}  // namespace

extern "C" {

int32_t moe_release_workspace(moe_handle *h, const uint32_t *flags_ws)
{
    if (!h) return MOE_ERR_NULL;
    if (flags_ws) h->epochs.erase(flags_ws);
    else h->epochs.clear();
    return MOE_OK;
}

int32_t moe_get_status(moe_handle *h, const uint32_t *status_dev, moe_status *host, void *stream)
{
    if (!h || !status_dev || !host) return MOE_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // (through the mailbox's spare words: a copy to pageable memory is staged by the driver)
    uint32_t on_stack[4], *w = h->mail_host ? reinterpret_cast<uint32_t *>(h->mail_host + kMailWords - 2) : on_stack;
    cudaError_t e = cudaMemcpyAsync(w, status_dev, sizeof on_stack, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(h, e, "status copy");
    host->code = w[0]; host->detail = w[1]; host->where = w[2]; host->count = w[3];
    return w[0] == 0 ? MOE_OK : MOE_ERR_DEVICE_STATUS;
}

int32_t moe_clear_status(moe_handle *h, uint32_t *status_dev, void *stream)
{
    if (!h || !status_dev) return MOE_ERR_NULL;
    cudaError_t e = cudaMemsetAsync(status_dev, 0, 16, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? MOE_OK : cuda_fail(h, e, "status clear");
}

// ---- whole step on device-resident inputs -----------------------------------------------------

int32_t moe_layer(moe_handle *h, const void *x_routed, const void *W2, const int32_t *topk_idx,
                  const float *topk_w, const moe_shape *s, int32_t tile_m, int32_t tile_n,
                  const moe_sm_limits *limits_or_null, const moe_routing *routing,
                  int32_t *tile_counts_pinned, void *const *out, void *y_ws, uint32_t *flags_ws,
                  uint32_t *status_dev, moe_plan *plan_out, void *ev_before, void *ev_after, void *stream)
{
    if (!h || !s || !routing) return MOE_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Selection sel;
    int32_t rc = selection_of(h, s, tile_m, tile_n, limits_or_null, tile_counts_pinned != nullptr, &sel);
    if (rc != MOE_OK) return rc;
    uint32_t seq = 0;
    const bool inlined = routing_inline_ok(*s, tile_m, kFusedThreads) && (sel.launch_first() || !tile_counts_pinned);
    rc = build_routing_mailed(h, topk_idx, s, tile_m, routing, tile_counts_pinned, sel.launch_first(), inlined, status_dev, st, &seq);
    if (rc != MOE_OK) return rc;
    return select_and_launch(h, x_routed, W2, topk_w, s, sel, routing, seq, seq, inlined ? topk_idx : nullptr, nullptr, nullptr, tile_counts_pinned, out, y_ws,
                             flags_ws, status_dev, plan_out, ev_before, ev_after, st);
}

// ---- the post-router MoE layer on device-resident inputs (Section II-A: steps 1-3) -------------

int32_t moe_post_router_layer(moe_handle *h, const void *hidden, const void *W1, const void *W2,
                              const int32_t *topk_idx, const float *topk_w, const moe_shape *s, int32_t tile_m,
                              int32_t tile_n, const moe_sm_limits *limits_or_null, const moe_routing *routing,
                              int32_t *tile_counts_pinned, void *h_routed_ws, void *x_routed_ws, void *const *out,
                              void *y_ws, uint32_t *flags_ws, uint32_t *status_dev, moe_plan *plan_out, void *stream)
{
    if (!h || !s || !routing) return MOE_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Selection sel;
    int32_t rc = selection_of(h, s, tile_m, tile_n, limits_or_null, tile_counts_pinned != nullptr, &sel);
    if (rc != MOE_OK) return rc;
    const bool gemm1_mails = s->T > 0;
    const bool inlined = routing_inline_ok(*s, tile_m, kThreads) && (h->mail_dev || !tile_counts_pinned);
    uint32_t seq = 0;
    rc = build_routing_mailed(h, topk_idx, s, tile_m, routing, tile_counts_pinned, gemm1_mails, inlined, status_dev, st, &seq);
    if (rc != MOE_OK) return rc;
    // GEMM1 reads the m-tile count on the device, so it is launched before the host waits for the counts: the wait
    // and the planning are hidden behind it.  Without the mailbox (seq = 0) the copy of the counts was queued right
    // behind the routing kernels, before GEMM1: an event marks it.
    cudaEvent_t counts_event = static_cast<cudaEvent_t>(h->counts_event);
    if (tile_counts_pinned && seq == 0u && counts_event) cudaEventRecord(counts_event, st);
    rc = launch_gemm1_act(h, hidden, W1, inlined ? topk_idx : nullptr, s, tile_m, routing, MOE_MTILES_ON_DEVICE, h_routed_ws, x_routed_ws,
                          status_dev, seq, st);
    if (rc != MOE_OK) return rc;
    if (tile_counts_pinned && seq == 0u && !counts_event) return MOE_ERR_CUDA;
    return select_and_launch(h, x_routed_ws, W2, topk_w, s, sel, routing, seq, 0u, nullptr, nullptr, counts_event, tile_counts_pinned, out, y_ws,
                             flags_ws, status_dev, plan_out, nullptr, nullptr, st);
}

// ---- one-time service-rate characterisation (Eq. 13) ---------------------------------------

int32_t moe_calibrate_rho(moe_handle *h, const void *x_routed, const void *W2, const int32_t *topk_idx,
                          const float *topk_w, const moe_shape *s, int32_t tile_m, int32_t tile_n,
                          int32_t C_ref, int32_t n_samples, const moe_routing *routing,
                          int32_t *tile_counts_pinned, void *const *out, void *y_ws, uint32_t *flags_ws,
                          uint32_t *status_dev, moe_rho *rho_out, double *wave_us_out, void *stream)
{
    if (!h || !s || !routing || !tile_counts_pinned || !rho_out) return MOE_ERR_NULL;
    if (C_ref < 1 || n_samples < 1 || n_samples > 64) return MOE_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t rc = moe_build_routing(h, topk_idx, s, tile_m, routing, tile_counts_pinned, status_dev, st);
    if (rc != MOE_OK) return rc;
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(h, e, "tile counts sync");
    moe_occupancy occ;
    moe_sm_limits lim;
    moe_rho rho;
    rc = moe_query_occupancy(h, tile_m, tile_n, &occ, &lim, &rho);
    if (rc != MOE_OK) return rc;
    lim.force_comm_ctas = C_ref;
    lim.drain_help = 0;                       // each role alone on its share of the SMs
    moe_plan plan;
    rc = plan_partition(tile_counts_pinned, s->E_tot, &occ, &lim, s, &rho, &plan);
    if (rc != MOE_OK) return rc;
    if (plan.W_comp < 1 || plan.W_comm < 1) return MOE_ERR_SHAPE;
    const int32_t S = tile_counts_pinned[s->E_tot];

    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if ((e = cudaEventCreate(&ev0)) != cudaSuccess) return cuda_fail(h, e, "event");
    if ((e = cudaEventCreate(&ev1)) != cudaSuccess) { cudaEventDestroy(ev0); return cuda_fail(h, e, "event"); }
    double med[2] = {0.0, 0.0};
    for (int role = 0; role < 2 && rc == MOE_OK; ++role) {
        moe_plan p = plan;
        p.mode = role == 0 ? MOE_MODE_GEMM_ONLY : MOE_MODE_COMBINE_ONLY;   // GEMM first: it also fills Y
        float t[64];
        for (int i = -2; i < n_samples && rc == MOE_OK; ++i) {              // two warm-up launches
            cudaEventRecord(ev0, st);
            rc = moe_gemm2_combine(h, x_routed, W2, topk_idx, topk_w, s, &occ, routing, S, &p, out, y_ws,
                                   flags_ws, status_dev, st);
            cudaEventRecord(ev1, st);
            if ((e = cudaEventSynchronize(ev1)) != cudaSuccess) rc = cuda_fail(h, e, "calibration launch");
            if (rc == MOE_OK && i >= 0) cudaEventElapsedTime(&t[i], ev0, ev1);
        }
        if (rc == MOE_OK) {
            std::sort(t, t + n_samples);
            med[role] = 1e3 * (double)t[n_samples / 2];
        }
    }
    cudaEventDestroy(ev0);
    cudaEventDestroy(ev1);
    if (rc != MOE_OK) return rc;
    // Eq. 13: time per wave of each role; a launch runs L splits of V waves each
    const double comp_waves = (double)ceil_div(plan.W_comp, plan.P) * s->L;
    const double comm_waves = (double)ceil_div(plan.W_comm, C_ref) * s->L;
    const double wave_comp = med[0] / comp_waves, wave_comm = med[1] / comm_waves;
    if (!(wave_comp > 0.0)) return MOE_ERR_SHAPE;
    if (wave_us_out) { wave_us_out[0] = wave_comp; wave_us_out[1] = wave_comm; }
    *rho_out = rho;
    rho_out->rho_ref = wave_comm / wave_comp;
    rho_out->K_ref = s->I / s->TP;
    rho_out->tile_m_ref = tile_m;
    rho_out->tile_n_ref = tile_n;
    rho_out->D_ref = s->EP;
    rho_out->rows_ref = s->k_tot * s->TP + 1;
    const int64_t split_w = ceil_div(s->H, s->L);
    rho_out->comm_cols_ref = (int32_t)(split_w < kCommTileN ? split_w : kCommTileN);
    return MOE_OK;
}

// ---- whole step from host buffers ----------------------------------------------------------

namespace {
struct ArenaLayout {
    size_t x, idx, w, routing, y, flags, status, out, total;
    size_t routing_b, y_b, flags_b;
};
int32_t arena_layout(const moe_shape *s, int tile_m, int tile_n, ArenaLayout *a)
{
    size_t sb = 0;
    int32_t rc = moe_workspace_bytes(s, tile_m, tile_n, &a->routing_b, &a->y_b, &a->flags_b, &sb);
    if (rc != MOE_OK) return rc;
    const size_t R = (size_t)s->T * s->k_tot;
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    // idx, w, status and flags lie together: one copy brings the small inputs and the zeros (moe_layer_host)
    size_t off = 0;
    a->x = off; off += up(R * s->I * 2);
    a->idx = off; off += up(R * 4);
    a->w = off; off += up(R * 4);
    a->status = off; off += up(16);
    a->flags = off; off += up(a->flags_b);
    a->routing = off; off += up(a->routing_b);
    a->y = off; off += up(a->y_b);
    a->out = off; off += up((size_t)ceil_div(s->T, s->EP) * s->EP * s->H * 2);
    a->total = off;
    return MOE_OK;
}
constexpr size_t kFeedMinBytes = 2 << 20;    // x_routed from which the copies overlap the GEMM
constexpr size_t kFeedLastBytes = 1 << 20;   // the last chunk holds this much or less
typedef CUresult (*WriteValueFn)(CUstream, CUdeviceptr, cuuint32_t, unsigned int);
// The stream and events of the overlapped copies, made on first use; false: not to be had, copy first instead.
bool feed_ready(moe_handle *h)
{
    if (h->feed_stream) return true;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuStreamWriteValue32", &h->write_value, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !h->write_value) {
        (void)cudaGetLastError();
        return false;
    }
    for (cudaEvent_t &ev : h->feed_events)
        if (!ev && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return false;
    return cudaStreamCreateWithFlags(&h->feed_stream, cudaStreamNonBlocking) == cudaSuccess;
}
constexpr size_t kStagingBytes = 64 << 10;
// The pinned buffer through which the small inputs go as one copy, made on first use.
bool staging_ready(moe_handle *h)
{
    if (!h->staging && cudaHostAlloc(reinterpret_cast<void **>(&h->staging), kStagingBytes, cudaHostAllocPortable) != cudaSuccess) {
        (void)cudaGetLastError();
        h->staging = nullptr;
    }
    return h->staging != nullptr;
}
}  // namespace

int32_t moe_host_arena_bytes(const moe_shape *s, int32_t tile_m, int32_t tile_n, size_t *bytes)
{
    if (!s || !bytes) return MOE_ERR_NULL;
    ArenaLayout a;
    int32_t rc = arena_layout(s, tile_m, tile_n, &a);
    if (rc != MOE_OK) return rc;
    *bytes = a.total;
    return MOE_OK;
}

int32_t moe_layer_host(moe_handle *h, const void *x_routed_host, const int32_t *topk_idx_host,
                       const float *topk_w_host, const void *W2_dev, const moe_shape *s, int32_t tile_m,
                       int32_t tile_n, const moe_sm_limits *limits_or_null, void *arena, size_t arena_bytes,
                       int32_t *tile_counts_pinned, void *out_host, moe_plan *plan_out, void *stream)
{
    if (!h || !s || !arena || !tile_counts_pinned || !out_host || !W2_dev) return MOE_ERR_NULL;
    if (s->T > 0 && (!x_routed_host || !topk_idx_host || !topk_w_host)) return MOE_ERR_NULL;
    ArenaLayout a;
    int32_t rc = arena_layout(s, tile_m, tile_n, &a);
    if (rc != MOE_OK) return rc;
    if (arena_bytes < a.total) return MOE_ERR_ARENA;
    if ((reinterpret_cast<uintptr_t>(arena) & 255u) != 0) return MOE_ERR_ALIGN;
    if (s->T == 0) return MOE_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *base = static_cast<char *>(arena);
    const size_t R = (size_t)s->T * s->k_tot;
    Selection sel;
    rc = selection_of(h, s, tile_m, tile_n, limits_or_null, true, &sel);
    if (rc != MOE_OK) return rc;
    if ((rc = require_handle_device(h, "moe_layer_host")) != MOE_OK) return rc;
    moe_routing rt;
    rc = moe_routing_view(base + a.routing, s, tile_m, &rt);
    if (rc != MOE_OK) return rc;
    uint32_t *status = reinterpret_cast<uint32_t *>(base + a.status), *ready = status + 16;   // (256 bytes lie there)
    cudaError_t e;
    const size_t small_b = a.flags + a.flags_b - a.idx;
    if (small_b <= kStagingBytes && staging_ready(h)) {
        // (the previous call on this handle has waited for its copy out of the staging buffer)
        memset(h->staging, 0, small_b);
        memcpy(h->staging, topk_idx_host, R * 4);
        memcpy(h->staging + (a.w - a.idx), topk_w_host, R * 4);
        e = cudaMemcpyAsync(base + a.idx, h->staging, small_b, cudaMemcpyHostToDevice, st);
    } else {
        e = cudaMemcpyAsync(base + a.idx, topk_idx_host, R * 4, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(base + a.w, topk_w_host, R * 4, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, a.flags + a.flags_b - a.status, st);
    }
    if (e != cudaSuccess) return cuda_fail(h, e, "idx copy");
    h->epochs.erase(base + a.flags);  // the workspace was just cleared
    // The rows of x_routed are most of the copies, and the GEMM takes them in order: from 2 MB on they come in chunks on a
    // stream of the handle's, each with the rows so far written behind it, which the kernel's x producers wait for, so that the
    // GEMM runs beside the copies.  A chunk costs the copy engine 7 us, so there are few: each brings 60 % of what is left,
    // the last one 1 MB or less.
    RowFeed feed = {nullptr, 0};
    const size_t row_b = (size_t)s->I * 2, x_b = R * row_b;
    const bool fed = x_b >= kFeedMinBytes && feed_ready(h);
    // (nothing is left in flight on the way out: the caller's buffers and the handle's staging buffer are free again)
    const auto fail = [&](int32_t code) {
        cudaStreamSynchronize(st);
        if (fed) cudaStreamSynchronize(h->feed_stream);
        return code;
    };
    if (fed) {
        feed.ready = ready;
        feed.extra_wait_ns = x_b / 10;               // 10 GB/s: far below what a host link moves
        e = cudaEventRecord(h->feed_events[0], st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(h->feed_stream, h->feed_events[0], 0);
    } else {
        e = cudaMemcpyAsync(base + a.x, x_routed_host, x_b, cudaMemcpyHostToDevice, st);
    }
    if (e != cudaSuccess) return fail(cuda_fail(h, e, "input copies"));
    uint32_t seq = 0;
    int32_t *const idx = reinterpret_cast<int32_t *>(base + a.idx);
    const bool inlined = routing_inline_ok(*s, tile_m, kFusedThreads) && (sel.launch_first() || !tile_counts_pinned);
    rc = build_routing_mailed(h, idx, s, tile_m, &rt, tile_counts_pinned, sel.launch_first(), inlined, status, st, &seq);
    if (rc != MOE_OK) return fail(rc);
    for (size_t r = 0; fed && r < R && e == cudaSuccess;) {
        size_t rows = R - r;
        if (rows * row_b > kFeedLastBytes) rows = (rows * 3 + 4) / 5;
        e = cudaMemcpyAsync(base + a.x + r * row_b, static_cast<const char *>(x_routed_host) + r * row_b, rows * row_b,
                            cudaMemcpyHostToDevice, h->feed_stream);
        r += rows;
        if (e == cudaSuccess && reinterpret_cast<WriteValueFn>(h->write_value)(h->feed_stream, (CUdeviceptr)(uintptr_t)ready, (cuuint32_t)r, 0) != CUDA_SUCCESS)
            e = cudaErrorUnknown;
    }
    if (fed && e == cudaSuccess) e = cudaEventRecord(h->feed_events[1], h->feed_stream);
    if (e != cudaSuccess) return fail(cuda_fail(h, e, "input copies"));
    void *outs[MOE_MAX_EP];
    const size_t blk = (size_t)ceil_div(s->T, s->EP);
    for (int d = 0; d < s->EP; ++d) outs[d] = base + a.out + (size_t)d * blk * s->H * 2;
    rc = select_and_launch(h, base + a.x, W2_dev, reinterpret_cast<float *>(base + a.w), s, sel, &rt, seq, seq,
                           inlined ? idx : nullptr, fed ? &feed : nullptr, nullptr, tile_counts_pinned, outs, base + a.y,
                           reinterpret_cast<uint32_t *>(base + a.flags), status, plan_out, nullptr, nullptr, st);
    if (rc != MOE_OK) return fail(rc);
    // whatever the kernel needed of the rows, their copies are over before the caller has its buffers back
    if (fed) e = cudaStreamWaitEvent(st, h->feed_events[1], 0);
    // rank d owns tokens [d*blk, (d+1)*blk): the EP blocks are contiguous in token order
    if (e == cudaSuccess) e = cudaMemcpyAsync(out_host, base + a.out, (size_t)s->T * s->H * 2, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return fail(cuda_fail(h, e, "output copy"));
    moe_status hs;
    return moe_get_status(h, status, &hs, st);
}

}  // extern "C"
