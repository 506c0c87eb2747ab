// Fused grouped GEMM2 + GatherRS combine for sm_100a: one persistent launch, one CTA per SM,
// role by blockIdx.
//
//   blockIdx <  C : communication CTA c (Section II-B: consumes published results; the same
//                   C CTAs serve all splits in sequence, its warps an even share of every split's
//                   units -- or, with drain help, all CTAs serve once their tiles are done, by even
//                   shares, or from a queue of token ranges per split).
//   blockIdx >= C : compute CTA b = blockIdx - C (Section III-C: takes global tiles
//                   b, b+P, b+2P, ... of the split-major sequence in which the expert
//                   problems of one split are contiguous; m-tile-major across the splits when
//                   the communication work is handed out dynamically).
//
// Compute CTA (warp-specialised; tile_m x tile_n with tile_m in {64, 128}):
//   warps 0, 2  TMA producers (one thread each): warp 0 the x_routed tile (up to 128 rows x 64 k), warp 2 the
//               W2 tile (tile_n rows x 64 k) of every k-block, into a ring of 128B-swizzled stages;
//   warp 1      MMA issuer (the warp runs the loop converged, an elected lane issues; all operands warp-uniform):
//               tcgen05.mma (M = 128 output columns, N = the tile's rows, K = 16, bf16 -> fp32; two of them for 256 columns) into one
//               of two TMEM accumulator buffers; tcgen05.commit frees stages / publishes the tile;
//   warps 4-15  epilogue: tcgen05.ld -> bf16, transposed -> Y (three groups of four warps, one per TMEM lane quarter; warps 16-19
//               are a fourth group when the launch carries no co-resident communication warp);
//   warp 3      publisher (one thread): once the epilogue warps have stored a tile, release fence, then the
//               tile's readiness flag and the split counter (one fence for all tiles stored by then).
// Compute CTA pair (256 x 256 tiles): the same roles in both CTAs of a cluster of two; one
//   tcgen05.mma.cta_group::2 (M = 256) spans both SMs, each CTA loads only its own operand halves; six operand
//   stages, seven when the aux region of shared memory is free while the GEMM runs.
// Y is token-major: the epilogue scatters each routed row to its (token, slot) place, so
//   that the k_tot rows of one (token, split, column slab) form one contiguous block.  The sum over the tensor-parallel
//   K-shards (Section II-A: each rank's partial product, here all on one GPU) is taken in the accumulator, in fp32: a tile runs over
//   all of I.  With a tile and a bf16 row of Y per shard, each partial was rounded, stored, read back and added by the combine:
//   TP times the Y traffic and the epilogue stores.  Whole step at TP = 2, us, a tile per shard -> now: Granite shape T = 4096
//   130 -> 96, Qwen shape T = 8192 287 -> 249, DeepSeek shape T = 256 88 -> 82 and T = 16384 943 -> 836; three calls with the static
//   partition, DeepSeek shape T = 2048 207 -> 178.  Y holds a row per assignment, rounded once instead of once per shard.
// Communication CTA (12 independent warps): a warp fetches such a block with one bulk asynchronous
//   copy into its own double-buffered shared-memory stage (the readiness of the producing tiles is
//   checked first: split counter, else per-tile flags with ld.acquire.gpu; bounded), sums the rows in
//   fp32 in slot order with the token's weights and stores bf16 into the owning rank's buffer.
// Co-resident communication warps (Section III-B with o_comm > 1 in spirit: communication work that
//   shares an SM with a compute CTA instead of reserving one): a compute CTA may carry extra warps
//   (of 16-19; two have stages) that run the same per-unit pipeline on stages of their own, take work from
//   the front of the per-split queues and serve split s while the CTA's other warps compute split
//   s + 1.  They wait for a whole split (no token of a split is complete before the last expert's
//   tiles of that split are), not for single tiles.
//
// Every wait is bounded: after `wait_ns` the waiter records MOE_DEV_TIMEOUT and the CTA winds
// down (pending bulk copies are drained, TMEM is released).

#include <cuda_bf16.h>

#include <type_traits>

#include "moe_internal.h"
#include "routing_device.cuh"
#include "sm100_device.cuh"

// Timeline build (-DMOE_TIMELINE=1, a separate library): the kernels record per-CTA time stamps and cycle
// counters into a caller-provided buffer (moe_set_timeline), kTimelineSlots 64-bit words per CTA followed by
// one completion stamp per split.  In the normal build every TL(...) statement compiles to nothing.
#ifndef MOE_TIMELINE
#define MOE_TIMELINE 0
#endif
#if MOE_TIMELINE
#define TL(...) do { __VA_ARGS__; } while (0)
#define TL_DECL(...) __VA_ARGS__
#else
#define TL(...) do { } while (0)
#define TL_DECL(...)
#endif

namespace moe {
namespace {

// slots of a CTA's timeline record (see bench.py --timeline for the reader)
enum {
    kTlBegin = 0, kTlRole = 1, kTlFirstAcc = 2, kTlMmaEnd = 3, kTlTiles = 4, kTlWaitOperand = 5, kTlIssue = 6,
    kTlWaitTmem = 7, kTlMmaCycles = 8, kTlComputeEnd = 9, kTlCtaEnd = 10, kTlEpiWait = 11, kTlEpiWork = 12,
    kTlProducerWait = 13, kTlCommUnits = 14, kTlCommWaitNs = 15, kTlCoWarp = 16,  // 8 slots per co-resident warp (16..31)
    kTlPubWait = 32, kTlPubFence = 33, kTlEpiPubWait = 34,
    kTlStageLate = 35   // pair tiles: k-blocks whose operand stage was not complete when the MMA issuer first looked
};
#if MOE_TIMELINE
__device__ __forceinline__ void tl_put(const FusedParams &P, int slot, unsigned long long v)
{
    if (P.timeline) P.timeline[(size_t)blockIdx.x * kTimelineSlots + slot] = v;
}
// Probes of the timeline build (moe_set_probe): parts of the launch's data movement are left out so that their
// cost shows in the launch time.  The results of a probed launch are garbage by construction.
#define MOE_PROBE(bit) ((P.probe & (bit)) != 0)
#else
#define MOE_PROBE(bit) false
#endif
enum { kProbeSkipOddW2 = 1, kProbeSkipAllW2 = 2, kProbeSkipYStores = 4, kProbeSkipX = 8, kProbeFreeRunMma = 16, kProbeSlowIssuer = 32 };

// --------------------------------------------------------------------------- shared memory

// Weights on the M side of the MMA, tokens on the N side: an accumulator lane is a column of the output, an accumulator column a
// routed row, and N is the tile's row count rounded up to 16 (a pair: 32).  (With the rows on the M side every tile was computed for
// 128 or 256 rows.  Whole calls, us, rows on M -> on N: DeepSeek shape T = 16 58.9 -> 53.5, T = 256 81 -> 72, Qwen shape T = 8192
// 239 -> 229, its whole layer T = 48 187 -> 170, T = 3000 126 -> 116; where hardly a row is padding, Granite shape T = 13784, equal.)
template <int TN>
struct Cfg {
    static constexpr int kWBytes = TN * kBlockK * 2;             // 8 / 16 / 32 KB: the tile's rows of W2, one k-block
    static constexpr int kStageKb = TN == 256 ? 1 : 2;           // k-blocks of a stage
    static constexpr int kThinKb = TN == 64 ? 4 : kStageKb;      // ... where no m-tile has more than 32 rows
    static constexpr int kBlocks = TN > kMmaM ? 2 : 1;           // blocks of 128 output columns, an MMA each (TN = 64: half of one is used)
    static constexpr int kAccCols = kBlocks * kMmaM;             // TMEM columns of an accumulator buffer
    static constexpr int kTmemCols = 2 * kAccCols;               // two of them
};

// Tiles a CTA may have stored but not yet published: the publisher's release fence takes thousands of cycles,
// and one fence covers every tile whose epilogue is over by then.
constexpr int kPubSlots = 4;

// A stage of a one-CTA tile: the W2 rows of its k-blocks one after the other, then their routed rows, with room for as many as an m-tile
// of the launch can have (FusedParams::x_rows: 32, 64 or 128).  Narrow tiles are bound by the instructions of the issuer's loop: about
// 290 cycles of waiting, branching and the commit for a stage and 45 to 53 for an MMA (fitted to 500, 355 and 250 cycles for every 64
// columns of I with one, two and four k-blocks a stage).  So a stage holds as many k-blocks as leave a ring of three or four.  That
// counts where tiles are few and their chain of k-blocks is long: a tile over all of I has TP times the chain of one per K-shard.
// Whole step, us, a tile per K-shard (TP as given) / over all of I, stages of one k-block and 128 rows / now:
//   one token        Qwen shape, TP = 2, 15.4 / 17.0 / 15.9; DeepSeek shape, TP = 2, 18.8 / 18.2 / 17.5; 8 experts, k = 2, I = 14336,
//                    TP = 8: H = 4096 46.5 / 69.3 / 53.4, H = 512 18.9 / 68.3 / 39.1 (16 tiles; the other SMs have none)
//   T = 4096         DeepSeek shape, TP = 2, tiles of 64 x 64 974 / 732 / 556, 64 x 128 529 / 390 / 320, 128 x 128 369 / 268 / 258
// (256 columns take two MMAs for every K = 16; one k-block a stage there.  More stages of one k-block instead, 16 in place of 8: 0.  The
// issuer looking at the next stage's barrier ahead of its MMAs: +10 % on the long chains.)
constexpr int kMaxStages = 8;

struct Control {
    unsigned long long full[kMaxStages];
    unsigned long long empty[kMaxStages];
    unsigned long long tmem_full[2];
    unsigned long long tmem_empty[2];
    unsigned long long epi_done[kPubSlots];   // every epilogue warp has stored its rows of the tile (tile number mod kPubSlots)
    unsigned long long pub_done[kPubSlots];   // the publisher warp has raised that tile's flag
    uint32_t tmem_base;
    volatile uint32_t abort;
    volatile uint32_t tile_n[kMaxStages];   // N of a tile's MMAs (tile number mod kMaxStages), from the x producer to the MMA issuer
    unsigned long long comm_full[24];   // communication CTA: one barrier per warp and stage
    unsigned long long co_full[8];      // co-resident communication warps: one barrier per warp and stage
};

// 33 KB after the control block: per-row weights of the unit each communication warp reduces (12 warps x 256 floats), or the stages
// and weights of co-resident communication warps
constexpr int kAuxBytes = 33 * 1024;
static_assert(12 * 256 * 4 <= kAuxBytes, "communication weights exceed the aux region");

// Bounded mbarrier wait, warp-collective: lane 0 polls (32 lanes polling the same barrier would
// each occupy the shared-memory pipe), the result is broadcast.  Returns false on timeout or when
// another warp of the CTA gave up.
__device__ __forceinline__ bool wait_barrier(uint32_t bar, uint32_t parity, Control *ctl,
                                             unsigned long long deadline, uint32_t *status,
                                             uint32_t detail, uint32_t where)
{
    uint32_t ok = 1u;
    if ((threadIdx.x & 31u) == 0u) {
        uint32_t spins = 0;
        while (!mbar_try_wait(bar, parity)) {
            if ((++spins & 63u) == 0u) {
                if (ctl->abort) { ok = 0u; break; }
                if (globaltimer_ns() > deadline) {
                    ctl->abort = 1u;
                    report(status, MOE_DEV_TIMEOUT, detail, where);
                    ok = 0u;
                    break;
                }
            }
        }
    }
    return __shfl_sync(0xffffffffu, ok, 0) != 0u;
}

// The same wait for a loop that a single thread runs on its own (no broadcast).
__device__ __forceinline__ bool wait_barrier_1t(uint32_t bar, uint32_t parity, Control *ctl,
                                                unsigned long long deadline, uint32_t *status,
                                                uint32_t detail, uint32_t where)
{
    uint32_t spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 63u) == 0u) {
            if (ctl->abort) return false;
            if (globaltimer_ns() > deadline) {
                ctl->abort = 1u;
                report(status, MOE_DEV_TIMEOUT, detail, where);
                return false;
            }
        }
    }
    return true;
}

// Barrier of the warps that compute: 16, or all 20 when warps 16-19 serve as a fourth epilogue column group
// (co-resident communication warps never join it).
__device__ __forceinline__ void sync_compute_warps(const FusedParams &P)
{
    asm volatile("bar.sync 1, %0;" ::"r"(kThreads + 32 * (P.epi_warps - 12)) : "memory");
}
// N of a tile's MMAs: its rows, rounded up to what the instruction takes (M = 128: 16, M = 256 over a pair: 32)
template <bool kPair>
__device__ __forceinline__ int mma_n_of(int valid) { return kPair ? (valid + 31) & ~31 : (valid + 15) & ~15; }

// The MMA issuer's N of its tile `it`, behind the tile's first full barrier.  The producer knows the tile's rows; looked up by the issuer
// itself, the table entry is a load in the issuer's way.  (A place is written again kMaxStages tiles later, each of
// at least one stage, behind the wait for the later tile's first stage: in a ring of kMaxStages or fewer that stage, or one that came
// after it, was freed by MMAs of the earlier tile, so that the issuer is past the look.)
template <typename Ctl>
__device__ __forceinline__ int tile_n(const Ctl *ctl, int it) { return (int)__reduce_max_sync(0xffffffffu, ctl->tile_n[it & (kMaxStages - 1)]); }   // (warp-uniform)

// What a launch's roles are divided by: compute tiles per split (Eq. 5), communication CTAs, compute slots.
struct Part {
    int W_comp, S, C, P;     // S: m-tiles
};

struct Tile {
    int s, mu, i_n;
    int id;   // canonical tile number s * W_comp + mu * NTs + i_n: indexes the readiness flags
};
// The tiles of the processing sequence that a compute slot takes: b, b + P, b + 2 P, ...  Split-major (Section III-C: all tiles of
// split s precede those of s + 1; inside a split the expert problems are contiguous), or, when the work is handed out dynamically
// and nothing waits for an early split (drain help), m-tile-major: the n-tiles of ALL splits of one
// m-tile are adjacent, so that the x rows are read from DRAM once instead of once per split.
// A position is a number of three digits (split, m-tile, n-tile), the step another one: no division per tile (with two for every
// look-up the epilogue warps spent 2500 cycles of a tile's 6200 between tiles at the Granite shape, and paced it).  Made once, for all
// roles: a copy in each of them is code that has to be fetched, on the way to the first tile.
struct TileWalk {
    int W_comp, NTs, n_mid, last_mu;     // n_mid: values of the middle digit
    bool m_major;
    int top, mid, low, d_top, d_mid, d_low;
    __device__ __forceinline__ TileWalk(const FusedParams &P, const Part &pt, int b)
    {
        W_comp = pt.W_comp;
        NTs = P.NTs;
        m_major = P.tile_order != 0;
        n_mid = m_major ? P.L : pt.S;
        last_mu = pt.S - 1;
        split(b, top, mid, low);
        split(pt.P, d_top, d_mid, d_low);
    }
    __device__ __forceinline__ void split(int g, int &t, int &m, int &l) const
    {
        const int r = small_quotient(g, NTs);      // (g: a compute slot, or how many there are)
        l = g - r * NTs;
        t = small_quotient(r, n_mid);
        m = r - t * n_mid;
    }
    __device__ __forceinline__ void next()
    {
        low += d_low;
        mid += d_mid;
        top += d_top;
        if (low >= NTs) { low -= NTs; ++mid; }
        if (mid >= n_mid) { mid -= n_mid; ++top; }
    }
    // (past the end of the sequence: some tile of the table, for look-ups that nobody uses)
    __device__ __forceinline__ Tile tile() const
    {
        Tile t;
        t.s = m_major ? mid : top;
        t.mu = m_major ? min(top, last_mu) : mid;
        t.i_n = low;
        t.id = t.s * W_comp + t.mu * NTs + low;
        return t;
    }
};

// x_routed that is still being copied in (FusedParams::x_ready): waits until the rows up to `last_row` have arrived.  One
// thread; `seen`: rows known to have arrived.  The copies were issued before this launch, so the wait ends on its own.
__device__ __forceinline__ bool wait_rows(const FusedParams &P, int last_row, uint32_t &seen, Control *ctl, unsigned long long deadline)
{
    const uint32_t need = (uint32_t)last_row + 1u;
    if (seen >= need) return true;
    uint32_t spins = 0;
    while ((seen = ld_acquire_sys_u32(P.x_ready)) < need) {
        __nanosleep(200);
        if ((++spins & 15u) == 0u) {
            if (ctl->abort) return false;
            if (globaltimer_ns() > deadline) {
                ctl->abort = 1u;
                report(P.status, MOE_DEV_TIMEOUT, (uint32_t)last_row, 46u);
                return false;
            }
        }
    }
    asm volatile("fence.proxy.async;" ::: "memory");   // read next by TMA
    return true;
}

// --------------------------------------------------------------------------- epilogue helper

// 32 rows x 32 columns of the accumulator at `taddr` -> bf16 -> Y, one warp.  The accumulator has the columns in its lanes, Y has
// them contiguous: 8 x 8 blocks are transposed in registers, then the four lanes that hold a row's 32 columns in pairs deal them
// out in eights, so that one store instruction covers 64 contiguous bytes of eight rows.  (By way of shared memory, 256 contiguous
// bytes a row: the staging buffers take an operand stage, and the GEMM phase grows by it, DeepSeek shape T = 16384 578 -> 696 us.)
// `dst`: lane i, where the first of the 32 columns of row i goes (nullptr: nowhere); `cols`: columns that exist.
__device__ __forceinline__ void store_rows(const FusedParams &P, const uint32_t (&lo)[16], const uint32_t (&hi)[16], __nv_bfloat16 *dst, int cols)
{
    const int lane = threadIdx.x & 31, c = lane & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) {                // rows 8j..8j+7; this lane: row 8j + lane / 4
        uint32_t v[4] = {transpose_8x8(pack_bf16(lo[4 * j], lo[4 * j + 1])), transpose_8x8(pack_bf16(lo[4 * j + 2], lo[4 * j + 3])),
                         transpose_8x8(pack_bf16(hi[4 * j], hi[4 * j + 1])), transpose_8x8(pack_bf16(hi[4 * j + 2], hi[4 * j + 3]))};
        // v[m]: columns 8m + 2c and the next one -> v[k]: columns 8c + 2k and the next one
#pragma unroll
        for (int d = 1; d < 4; d *= 2)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                if (m & d) continue;
                const bool up = (c & d) != 0;
                const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? v[m] : v[m + d], d);
                if (up) v[m] = got;
                else v[m + d] = got;
            }
        __nv_bfloat16 *row = reinterpret_cast<__nv_bfloat16 *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst), 8 * j + (lane >> 2)));
        if (row != nullptr && c * 8 < cols && !MOE_PROBE(kProbeSkipYStores)) *reinterpret_cast<uint4 *>(row + c * 8) = make_uint4(v[0], v[1], v[2], v[3]);
    }
}

// --------------------------------------------------------------------------- epilogue and publisher roles
//
// Shared by the one-CTA and the CTA-pair compute roles (kPair: this CTA is rank `rank` of a pair and owns columns
// rank * 128 ... of the tile; the accumulator buffer is handed back on the leader's barrier; the tile is
// published in two parts, one flag per CTA).

// Epilogue, one warp: TMEM -> bf16 -> Y of every tile of this CTA: its TMEM lane quarter (32 of 128 columns) of every third or fourth
// piece of 32 rows x 128 columns, then the hand-over to the publisher warp.
template <int TN, bool kPair>
__device__ __forceinline__ void epilogue_role(const FusedParams &P, const Part &pt, Control *ctl, int b,
                                              uint32_t tmem_base, unsigned long long deadline, int rank, TileWalk walk)
{
    constexpr int kBlocks = kPair ? 1 : Cfg<TN>::kBlocks, kAccCols = kPair ? TN : Cfg<TN>::kAccCols;
    constexpr int kPieces = 3;                 // pieces of a tile that a warp may have: 8, over at least three groups of warps
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total_tiles = P.L * pt.W_comp;
    const int q4 = warp & 3;                   // TMEM lane quarter this warp may read
    const int grp = (warp - 4) >> 2, groups = P.epi_warps >> 2;
    __nv_bfloat16 *Y = reinterpret_cast<__nv_bfloat16 *>(P.Y);
    // Row bookkeeping runs ahead of the accumulators: the m-tile table entries are fetched two tiles
    // ahead and the rows' flat assignments one tile ahead, so that these dependent global loads are
    // not in the way between an accumulator becoming ready and its first store.
    int valid = 0, valid_n = 0, first_n = 0;
    int f[kPieces];                            // piece i: assignment of row `lane` of it
    const int max_pieces = groups == 3 ? 3 : 2;
    const auto load_rows = [&](int first, int n, int (&fr)[kPieces]) {
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
            const int row = (grp + i * groups) / kBlocks * 32 + lane;
            fr[i] = i < max_pieces && row < n ? ld_chained(&P.perm[first + row]) : -1;
        }
    };
    TL_DECL(long long tl_ew = 0, tl_ek = 0, tl_ep = 0, tl_q;)
    Tile t = walk.tile(), t_n = t;
    if (b < total_tiles) {
        walk.next();
        t_n = walk.tile();
        valid = ld_chained(&P.mtile_valid[t.mu]);
        const int first0 = ld_chained(&P.mtile_first_row[t.mu]);
        valid_n = ld_chained(&P.mtile_valid[t_n.mu]);
        first_n = ld_chained(&P.mtile_first_row[t_n.mu]);
        load_rows(first0, valid, f);
    }
    // Round -1 (one-CTA tiles: small launches, whose tail counts) is dry: the store path runs once without a tile while the first operands are on their way, on whatever the
    // second accumulator buffer holds, so that its instructions are at hand when the first tile is done.
    int it = (!kPair && P.even) ? -1 : 0;
#pragma unroll 1
    for (int g = b; g < total_tiles;) {
        const bool dry = !kPair && it < 0;
        const int a = it & 1;
        const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
        Tile t_nn = t_n;
        int valid_nn = valid_n, first_nn = first_n, f_n[kPieces];
        bool ok = true;
        if (!dry) {
            walk.next();
            t_nn = walk.tile();
            valid_nn = ld_chained(&P.mtile_valid[t_nn.mu]);
            first_nn = ld_chained(&P.mtile_first_row[t_nn.mu]);
            load_rows(first_n, valid_n, f_n);
        }
        const int n_pieces = (dry ? 1 : (valid + 31) >> 5) * kBlocks;
        const int mine = dry ? 1 : n_pieces > grp ? (n_pieces - grp + groups - 1) / groups : 0;
        // destinations of this lane's rows: a routed row belongs to flat assignment f = (token, slot); Y is token-major so that the
        // combine reads one contiguous block
        __nv_bfloat16 *dst[kPieces];
        int cols[kPieces];
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
            const int block = (grp + i * groups) % kBlocks;
            const int cis = t.i_n * TN + (kPair ? rank : block) * kMmaM + q4 * 32;       // first column, inside the split
            cols[i] = min(min(P.H, (t.s + 1) * P.split_w) - t.s * P.split_w, t.i_n * TN + TN) - cis;
            dst[i] = nullptr;
            if (!dry && f[i] >= 0 && cols[i] > 0) {
                const int tok = quotient(P.by_k, f[i]), q = f[i] - tok * P.k_tot;
                const int slab = cis >> P.slab_shift, wslab = min(P.slab_cols, P.split_w - (slab << P.slab_shift));
                dst[i] = Y + y_unit(tok, t.s, slab << P.slab_shift, P.L, P.split_w, P.k_tot) + (uint32_t)(q * wslab + (cis & (P.slab_cols - 1)));
            }
        }
        TL(tl_q = clock64());
        if (!dry) ok = wait_barrier(smem_u32(&ctl->tmem_full[a]), acc_phase, ctl, deadline, P.status, (uint32_t)g, 30u);
        TL(tl_ew += clock64() - tl_q; tl_q = clock64());
        if (ok) {
            tc_fence_after();
            const auto release = [&]() {
                // the accumulator buffer (this CTA's half of it) may be overwritten by the MMA of the tile after next
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (kPair) mbar_arrive_cluster_relaxed(mapa_u32(smem_u32(&ctl->tmem_empty[a]), 0u));   // the leader's barrier
                    else mbar_arrive(smem_u32(&ctl->tmem_empty[a]));
                }
            };
#pragma unroll
            for (int i = 0; i < kPieces; ++i) {
                if (i >= mine) break;
                const int piece = grp + i * groups, chunk = piece / kBlocks, block = piece - chunk * kBlocks;
                if (dry || cols[i] > 0) {
                    const uint32_t taddr = tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(a * kAccCols + (dry ? 0 : block * kMmaM + chunk * 32));
                    uint32_t lo[16], hi[16];
                    tmem_ld_16x256_x4(taddr, lo);
                    tmem_ld_16x256_x4(taddr + (16u << 16), hi);
                    tmem_ld_wait(lo);
                    tmem_ld_wait(hi);
                    if (!dry && i == mine - 1) release();
                    store_rows(P, lo, hi, dst[i], cols[i]);
                } else if (i == mine - 1) {
                    release();
                }
            }
            if (dry) {
                ++it;
                continue;
            }
            if (mine == 0) release();
            TL(tl_ek += clock64() - tl_q);
        }
        // hand the tile to the publisher warp.  Its barrier is reused every kPubSlots tiles, so the warp first
        // makes sure that the tile kPubSlots back has been published (it normally has, long ago).
        const int slot = it & (kPubSlots - 1);
        TL(tl_q = clock64());
        if (ok && it >= kPubSlots)
            ok = wait_barrier(smem_u32(&ctl->pub_done[slot]), (uint32_t)((it - kPubSlots) / kPubSlots) & 1u, ctl, deadline,
                              P.status, (uint32_t)g, 31u);
        TL(tl_ep += clock64() - tl_q);
        if (!ok) break;
        __syncwarp();   // the lanes' stores are ordered before lane 0's arrival
        if (lane == 0) mbar_arrive(smem_u32(&ctl->epi_done[slot]));
        valid = valid_n;
#pragma unroll
        for (int i = 0; i < kPieces; ++i) f[i] = f_n[i];
        t = t_n;
        t_n = t_nn;
        valid_n = valid_nn;
        first_n = first_nn;
        g += pt.P;
        ++it;
    }
    TL(if (warp == 4 && lane == 0) { tl_put(P, kTlEpiWait, (unsigned long long)tl_ew); tl_put(P, kTlEpiWork, (unsigned long long)tl_ek);
                                      tl_put(P, kTlEpiPubWait, (unsigned long long)tl_ep); });
}

// Publisher, one thread of warp 3: raises the readiness flag of every finished tile.  The release costs
// microseconds (the fence waits until the CTA's stores to Y have been performed: 2800 cycles per tile at the
// DeepSeek shape, 4900 at the Granite shape, where a tile's four k-blocks take less than that); here it is off
// the path of the epilogue warps, which go straight on to the next accumulator, and one fence covers every tile
// whose epilogue has finished by then (up to kPubSlots).
template <bool kPair>
__device__ __forceinline__ void publisher_role(const FusedParams &P, const Part &pt, Control *ctl, int b,
                                               unsigned long long deadline, int rank, TileWalk walk)
{
    const int total_tiles = P.L * pt.W_comp;
    if ((threadIdx.x & 31) == 0) {
        int it = 0;
        TL_DECL(long long tl_pw = 0, tl_pf = 0, tl_q;)
        for (int g = b; g < total_tiles;) {
            TL(tl_q = clock64());
            if (!wait_barrier_1t(smem_u32(&ctl->epi_done[it & (kPubSlots - 1)]), (uint32_t)(it / kPubSlots) & 1u, ctl,
                                 deadline, P.status, (uint32_t)g, 32u))
                break;
            TL(tl_pw += clock64() - tl_q; tl_q = clock64());
            // the following tiles too, as far as their epilogues are already over (waiting for more of them before
            // the fence was measured: no gain)
            int n = 1;
            while (n < kPubSlots && g + n * pt.P < total_tiles &&
                   mbar_test_wait(smem_u32(&ctl->epi_done[(it + n) & (kPubSlots - 1)]), (uint32_t)((it + n) / kPubSlots) & 1u))
                ++n;
            fence_acq_rel_gpu();   // release: the epilogue warps' stores (observed through epi_done) come first
            for (int j = 0; j < n; ++j, ++it, g += pt.P, walk.next()) {
                const Tile t = walk.tile();
                if (t.id != P.withhold) {
                    if (!P.even) st_relaxed_u32(&P.flags[kPair ? 2 * t.id + rank : t.id], P.epoch);
#if MOE_TIMELINE
                    if (atomicAdd(&P.split_done[t.s], 1u) + 1u == (uint32_t)(pt.W_comp * P.flag_parts) && P.timeline)
                        P.timeline[(size_t)gridDim.x * kTimelineSlots + t.s] = globaltimer_ns();
#else
                    red_relaxed_add_u32(&P.split_done[t.s], 1u);
#endif
                }
                mbar_arrive(smem_u32(&ctl->pub_done[it & (kPubSlots - 1)]));
            }
            TL(tl_pf += clock64() - tl_q);
        }
        TL(tl_put(P, kTlPubWait, (unsigned long long)tl_pw); tl_put(P, kTlPubFence, (unsigned long long)tl_pf));
    }
    __syncwarp();
}

struct PairCfg {
    static constexpr int kTileN = 256;
    static constexpr int kWBytes = kMmaM * kBlockK * 2;                 // 16 KB: this CTA's 128 W2 rows
    static constexpr int kXBytes = (kTileN / 2) * kBlockK * 2;          // 16 KB: this CTA's half of the tile's rows
    static constexpr int kStageBytes = kWBytes + kXBytes;               // 32 KB
    static constexpr int kStageKb = 1, kThinKb = 1;                     // k-blocks of a stage
    static constexpr int kTmemCols = 2 * kTileN;                        // two accumulator buffers
};
// (a one-CTA ring: fused_stages)
static_assert(kStageBytesTotal / PairCfg::kStageBytes + 1 <= kMaxStages && (kMaxStages & (kMaxStages - 1)) == 0, "barriers and tile_n of a ring");

// --------------------------------------------------------------------------- TMA producers
//
// One thread: kX the x_routed rows, else the W2 rows of every k-block of this CTA's tiles; both complete on the same full barrier
// (two issuing threads halve the serial issue latency per k-block).  The way from a freed stage to its next copies is the longest
// of the ring, so the loop over the k-blocks holds nothing but the wait, the copy and constants to add: a k-block of the rows is ONE
// copy, of 128 rows or, where they suffice, 64 or 32 (two copies of 64 rows lengthen the GEMM phase of the DeepSeek shape T = 16384 from
// 609 to 690 us, a number of copies and bytes that it looks up by 30), and the next tile is looked up between two k-blocks.
template <int TN, bool kPair, bool kX>
__device__ __forceinline__ void producer_role(const FusedParams &P, const Part &pt, uint8_t *ring, Control *ctl, int b, unsigned long long deadline, uint32_t rank,
                                              bool dry, TileWalk walk)
{
    using C = typename std::conditional<kPair, PairCfg, Cfg<TN>>::type;
    const int total_tiles = P.L * pt.W_comp, n_stages = P.stages;
    const uint32_t stage_bytes = kPair ? (uint32_t)PairCfg::kStageBytes : (uint32_t)P.stage_bytes;
    const bool thin = !kPair && P.x_rows == 32;
    const int stage_kb = thin ? C::kThinKb : C::kStageKb;
    // pair: the leader's full barriers, which lie at the same offsets in CTA 0
    const uint32_t dst0 = smem_u32(ring) + (kX ? (uint32_t)(C::kWBytes * stage_kb) : 0u), empty0 = smem_u32(&ctl->empty[0]);
    const uint32_t full0 = kPair ? smem_u32(&ctl->full[0]) & 0xFEFFFFFFu : smem_u32(&ctl->full[0]);
    uint32_t dst = dst0, full_bar = full0, empty_bar = empty0;
    int stage = 0, it = 0;
    uint32_t phase = 0, seen = 0;
    uint32_t armed = 0;  // bit s: stage s was handed to the TMA unit at least once
    bool ok = true;
    const unsigned long long w_policy = P.w2_once ? l2_evict_first_policy() : l2_evict_normal_policy();
    TL_DECL(long long tl_pw = 0, tl_q;)
    Tile t = walk.tile(), t_next = t;
    int e = 0, e_next = 0, row0 = 0, valid = P.dry_rows, row0_next = 0, valid_next = 0;
    if (!dry) {
        if (kX) {
            row0 = ld_chained(&P.mtile_first_row[t.mu]);
            valid = ld_chained(&P.mtile_valid[t.mu]);
        } else {
            e = ld_chained(&P.mtile_expert[t.mu]);
        }
    }
    const int ahead_at = min(2, P.num_kb - 1) / stage_kb * stage_kb;
    for (int g = b; g < total_tiles && ok; g += pt.P, ++it) {
        const int n0 = t.s * P.split_w + t.i_n * TN + (kPair ? (int)rank * (TN / 2) : 0);
        const int n = mma_n_of<kPair>(min(valid, kPair ? 2 * P.x_rows : P.x_rows)), my_rows = kPair ? n >> 1 : n, my_row0 = row0 + (kPair ? (int)rank * my_rows : 0);
        if (kX && P.x_ready && !dry && !(ok = wait_rows(P, row0 + valid - 1, seen, ctl, deadline))) break;
        const auto kloop = [&](auto box_rows, auto kbs) {
            constexpr int kKb = decltype(kbs)::value;
            constexpr int kRows = decltype(box_rows)::value;
            constexpr uint32_t kXCopy = (uint32_t)(kRows * kBlockK * 2);
            const CUtensorMap *const map = !kX ? &P.tmB : kRows == 128 ? &P.tmA : kRows == 64 ? &P.tmA64 : &P.tmA32;
            int kx = 0;
            for (int kb = 0; kb < P.num_kb; kb += kKb, kx += kBlockK * kKb) {
                const bool whole = kKb == 1 || kb + kKb <= P.num_kb;
                const uint32_t n_kb = whole ? (uint32_t)kKb : (uint32_t)(P.num_kb - kb);
                TL(tl_q = clock64());
                ok = wait_barrier_1t(empty_bar, phase ^ 1u, ctl, deadline, P.status, (uint32_t)g, 10u);
                if (!ok) break;
                TL(tl_pw += clock64() - tl_q);
                // (a probe that leaves a copy out completes its bytes by hand: every producer stays in the
                // barrier's dependency chain, or the one that arms it could lap the others)
                if (dry) {
                } else if (kX) {
                    if (kb == 0) ctl->tile_n[it & (kMaxStages - 1)] = (uint32_t)n;
                    if (!kPair) mbar_arrive_expect_tx(full_bar, ((uint32_t)C::kWBytes + kXCopy) * n_kb);
                    else if (rank == 0) mbar_arrive_expect_tx(full_bar, 2u * ((uint32_t)C::kWBytes + kXCopy));
                    if (MOE_PROBE(kProbeSkipX)) mbar_complete_tx_cluster(mapa_u32(smem_u32(&ctl->full[stage]), kPair ? 0u : cluster_ctarank()), kXCopy * n_kb);
                    else if (kPair) tma_load_2d_pair(dst, map, full_bar, kx, my_row0);
                    else tma_load_2d(dst, map, full_bar, kx, my_row0);
#pragma unroll
                    for (int j = 1; j < kKb; ++j)
                        if ((whole || kb + j < P.num_kb) && !MOE_PROBE(kProbeSkipX)) tma_load_2d(dst + (uint32_t)(j * P.x_rows * kBlockK * 2), map, full_bar, kx + j * kBlockK, my_row0);
                } else if (MOE_PROBE(kProbeSkipAllW2) || (MOE_PROBE(kProbeSkipOddW2) && (kb / kKb & 1))) {   // (whole stages)
                    mbar_complete_tx_cluster(mapa_u32(smem_u32(&ctl->full[stage]), kPair ? 0u : cluster_ctarank()), (uint32_t)C::kWBytes * n_kb);
                } else {
                    if (kPair) tma_load_3d_pair(dst, map, full_bar, kx, n0, e);
                    else tma_load_3d_hint(dst, map, full_bar, kx, n0, e, w_policy);
#pragma unroll
                    for (int j = 1; j < kKb; ++j)
                        if (whole || kb + j < P.num_kb) tma_load_3d_hint(dst + (uint32_t)(j * C::kWBytes), map, full_bar, kx + j * kBlockK, n0, e, w_policy);
                }
                armed |= 1u << stage;
                dst += stage_bytes;
                full_bar += 8u;
                empty_bar += 8u;
                if (++stage == n_stages) {
                    stage = 0;
                    phase ^= 1u;
                    dst = dst0;
                    full_bar = full0;
                    empty_bar = empty0;
                }
                if (dry) break;
                if (kb == ahead_at) {
                    walk.next();
                    t_next = walk.tile();
                    if (kX) {
                        row0_next = ld_chained(&P.mtile_first_row[t_next.mu]);
                        valid_next = ld_chained(&P.mtile_valid[t_next.mu]);
                    } else {
                        e_next = ld_chained(&P.mtile_expert[t_next.mu]);
                    }
                }
            }
        };
        const std::integral_constant<int, C::kStageKb> kbs;
        if (C::kThinKb != C::kStageKb && thin) kloop(std::integral_constant<int, 32>{}, std::integral_constant<int, C::kThinKb>{});
        else if (!kX || my_rows > 64) kloop(std::integral_constant<int, 128>{}, kbs);
        else if (kPair || my_rows > 32) kloop(std::integral_constant<int, 64>{}, kbs);
        else kloop(std::integral_constant<int, 32>{}, kbs);
        if (dry) return;
        t = t_next;
        e = e_next;
        row0 = row0_next;
        valid = valid_next;
    }
    TL(if (kX) tl_put(P, kTlProducerWait, (unsigned long long)tl_pw));
    if (!ok && rank == 0) {
        // wind-down: let the copies already issued land before shared memory is released
        // (bounded; a stage consumed meanwhile has completed its phase and passes at once)
        const unsigned long long drain = globaltimer_ns() + 2000000ull;
        for (int sidx = 0; sidx < n_stages; ++sidx) {
            if (!(armed & (1u << sidx))) continue;
            const uint32_t par = (sidx < stage) ? phase : (phase ^ 1u);
            while (!mbar_try_wait(smem_u32(&ctl->full[sidx]), par) && globaltimer_ns() < drain) {}
        }
    }
}

// --------------------------------------------------------------------------- compute CTA

// Barriers (thread 0) and TMEM (warp 1) of a compute CTA, before it is known that this CTA computes; a CTA-wide barrier of the
// kernel makes them visible.
template <int TN>
__device__ __forceinline__ void compute_setup(const FusedParams &P, Control *ctl)
{
    using C = Cfg<TN>;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int i = 0; i < P.stages; ++i) {
            mbar_init(smem_u32(&ctl->full[i]), 1);
            mbar_init(smem_u32(&ctl->empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&ctl->tmem_full[i]), 1);
            mbar_init(smem_u32(&ctl->tmem_empty[i]), (uint32_t)P.epi_warps);
        }
        for (int i = 0; i < kPubSlots; ++i) {
            mbar_init(smem_u32(&ctl->epi_done[i]), (uint32_t)P.epi_warps);
            mbar_init(smem_u32(&ctl->pub_done[i]), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), C::kTmemCols);
}

template <int TN>
__device__ void compute_cta(const FusedParams &P, const Part &pt, uint8_t *ring, Control *ctl, int b)
{
    using C = Cfg<TN>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total_tiles = P.L * pt.W_comp;
    const int n_stages = P.stages;
    const unsigned long long deadline = globaltimer_ns() + P.wait_ns;
    const uint32_t tmem_base = ctl->tmem_base;
    const TileWalk walk(P, pt, b);

    if (warp == 0 || warp == 2) {
        // ---------------- TMA producers: warp 0 loads the x_routed tile, warp 2 the W2 tile of every k-block
        if (lane == 0 && b < total_tiles) {
            if (warp == 0) producer_role<TN, false, true>(P, pt, ring, ctl, b, deadline, 0u, false, walk);
            else producer_role<TN, false, false>(P, pt, ring, ctl, b, deadline, 0u, false, walk);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer: the whole warp runs the loop, converged, one elected lane issues; the loop
        // is as short as it can be and its operands are warp-uniform (both for the reasons given in
        // compute_cta_pair): the four MMAs of a k-block (and the commit) are one statement with 32-bit descriptor
        // arithmetic, addresses advance by additions, the barrier's first look is the non-suspending test.
        {
            const uint32_t lo_stage = (uint32_t)P.stage_bytes >> 4;
            constexpr uint32_t kLoW = (uint32_t)(C::kWBytes >> 4);                   // the stage's next k-block
            const uint32_t lo_x = (uint32_t)(P.x_rows * kBlockK * 2 >> 4);
            const int all_ksteps = (P.num_kb - 1) * (kBlockK / kUmmaK) + P.last_ksteps;
            constexpr uint32_t kLoBlock = (uint32_t)(kMmaM * kBlockK * 2 >> 4);      // the next 128 rows of W2
            const uint32_t lo0 = smem_desc_lo(smem_u32(ring));
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            uint32_t w_lo = lo0, full_bar = full0, empty_bar = empty0;
            int stage = 0;
            uint32_t phase = 0;
            int it = 0;
            bool ok = true;
            TL_DECL(const long long tl_c0 = clock64(); long long tl_wf = 0, tl_wt = 0, tl_is = 0, tl_q;)
            for (int g = b; g < total_tiles && ok; g += pt.P, ++it) {
                const int a = it & 1;
                const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
                uint32_t idesc = 0;
                TL(tl_q = clock64());
                if (!__all_sync(0xffffffffu, mbar_test_wait(smem_u32(&ctl->tmem_empty[a]), acc_phase ^ 1u))) {
                    // (every lane polls; the vote keeps `ok`, and with it the loop, provably warp-uniform)
                    ok = __all_sync(0xffffffffu, wait_barrier_1t(smem_u32(&ctl->tmem_empty[a]), acc_phase ^ 1u, ctl, deadline, P.status, (uint32_t)g, 20u));
                    if (!ok) break;
                }
                TL(tl_wt += clock64() - tl_q);
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(a * C::kAccCols);
                const auto kloop = [&](auto kbs) {
                    constexpr int kKb = decltype(kbs)::value, kKsteps = kKb * (kBlockK / kUmmaK);
                    for (int ks = 0; ks < all_ksteps; ks += kKsteps) {
                        TL(tl_q = clock64());
                        if (!__all_sync(0xffffffffu, mbar_test_wait(full_bar, phase))) {
                            ok = __all_sync(0xffffffffu, wait_barrier_1t(full_bar, phase, ctl, deadline, P.status, (uint32_t)g, 21u));
                            if (!ok) break;
                        }
                        TL(tl_wf += clock64() - tl_q; tl_q = clock64());
                        if (ks == 0) idesc = make_idesc(kMmaM, tile_n(ctl, it));
                        tc_fence_after();
                        // advancing K by 16 bf16 = 32 bytes inside the swizzle row: +2 in the address field
                        if (elect_one_sync()) {
                            if (ks + kKsteps <= all_ksteps) {
                                uint32_t wl = w_lo, xl = w_lo + kKb * kLoW, acc = ks > 0 ? 1u : 0u;
                                if (C::kBlocks == 2) tc_ksteps_bf16(d_tmem + kMmaM, wl + kLoBlock, xl, idesc, acc);
#pragma unroll
                                for (int j = 1; j < kKb; ++j, wl += kLoW, xl += lo_x, acc = 1u) tc_ksteps_bf16(d_tmem, wl, xl, idesc, acc);
                                tc_kblock_bf16(d_tmem, wl, xl, idesc, acc, empty_bar);
                            } else {
                                for (int k = 0; k < all_ksteps - ks; ++k) {
                                    const uint32_t j = (uint32_t)k / (kBlockK / kUmmaK), in_row = 2u * ((uint32_t)k % (kBlockK / kUmmaK));
                                    const uint64_t w_desc = ((uint64_t)kSmemDescHi << 32) | (w_lo + j * kLoW + in_row),
                                                   x_desc = ((uint64_t)kSmemDescHi << 32) | (w_lo + kKb * kLoW + j * lo_x + in_row);
                                    for (int i = 0; i < C::kBlocks; ++i)
                                        tc_mma_bf16(d_tmem + (uint32_t)(i * kMmaM), w_desc + (uint64_t)(i * (int)kLoBlock), x_desc, idesc, (k > 0 || ks > 0) ? 1u : 0u);
                                }
                                tc_commit(empty_bar);   // stage reusable once these MMAs have read it
                            }
                        }
                        TL(tl_is += clock64() - tl_q);
                        w_lo += lo_stage;
                        full_bar += 8u;
                        empty_bar += 8u;
                        if (++stage == n_stages) {
                            stage = 0;
                            phase ^= 1u;
                            w_lo = lo0;
                            full_bar = full0;
                            empty_bar = empty0;
                        }
                    }
                };
                if (C::kThinKb != C::kStageKb && P.x_rows == 32) kloop(std::integral_constant<int, C::kThinKb>{});
                else kloop(std::integral_constant<int, C::kStageKb>{});
                __syncwarp();
                if (ok && elect_one_sync()) tc_commit(smem_u32(&ctl->tmem_full[a]));  // accumulator complete
                TL(if (it == 0 && lane == 0) tl_put(P, kTlFirstAcc, globaltimer_ns()));
            }
            TL(if (lane == 0) {
                   tl_put(P, kTlMmaEnd, globaltimer_ns()); tl_put(P, kTlTiles, (unsigned long long)it);
                   tl_put(P, kTlWaitOperand, (unsigned long long)tl_wf); tl_put(P, kTlIssue, (unsigned long long)tl_is);
                   tl_put(P, kTlWaitTmem, (unsigned long long)tl_wt); tl_put(P, kTlMmaCycles, (unsigned long long)(clock64() - tl_c0)); });
        }
        __syncwarp();
    } else if (warp >= 4 && warp < 4 + P.epi_warps) {
        epilogue_role<TN, false>(P, pt, ctl, b, tmem_base, deadline, 0, walk);
    } else if (warp == 3) {
        publisher_role<false>(P, pt, ctl, b, deadline, 0, walk);
    }
    // ---------------- teardown
    tc_fence_before();
    sync_compute_warps(P);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
}


// --------------------------------------------------------------------------- compute CTA pair
//
// 256 x 256 pair tile: two CTAs of a cluster (two SMs) compute one tile with tcgen05.mma.cta_group::2, M = 256 columns of the
// output, N = the tile's rows, rounded up to 32.  CTA `rank` loads its own half of those rows of x_routed and its own 128 of the
// 256 W2 rows of every k-block (no multicast: each CTA issues its own loads), so a k-block costs 32 KB per SM instead of 48 KB.
// Rank 0 (the leader) issues the MMAs; tcgen05.commit arrives on the barriers of both CTAs.
//   full[stage]       only the leader's is used: armed by the leader for the bytes of both CTAs
//   empty[stage]      one per CTA (its producer waits on it), signalled by the leader's commit
//   tmem_full[a]      one per CTA (its epilogue waits on it), signalled by the leader's commit
//   tmem_empty[a]     only the leader's is used: the epilogue warps of both CTAs arrive, 16 each (12 beside co-resident warps)

// Barriers (thread 0) and TMEM (warp 1) of a CTA of a pair, before it is known that the pair computes; the cluster barrier behind it
// makes the peer's barriers exist before anything arrives on them.
__device__ __forceinline__ void pair_setup(const FusedParams &P, Control *ctl)
{
    if (threadIdx.x == 0) {
        for (int i = 0; i < P.stages; ++i) {
            mbar_init(smem_u32(&ctl->full[i]), 1);
            mbar_init(smem_u32(&ctl->empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&ctl->tmem_full[i]), 1);
            mbar_init(smem_u32(&ctl->tmem_empty[i]), 2u * (uint32_t)P.epi_warps);
        }
        for (int i = 0; i < kPubSlots; ++i) {
            mbar_init(smem_u32(&ctl->epi_done[i]), (uint32_t)P.epi_warps);
            mbar_init(smem_u32(&ctl->pub_done[i]), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if ((threadIdx.x >> 5) == 1) tmem_alloc_pair(smem_u32(&ctl->tmem_base), PairCfg::kTmemCols);
}

__device__ __forceinline__ void compute_cta_pair(const FusedParams &P, const Part &pt, uint8_t *ring, Control *ctl, int b, bool dry)
{
    using C = PairCfg;
    constexpr int TN = C::kTileN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const bool leader_cta = (rank == 0);
    const int total_tiles = P.L * pt.W_comp;
    const int n_stages = P.stages;
    const unsigned long long deadline = globaltimer_ns() + P.wait_ns;
    const uint32_t tmem_base = ctl->tmem_base;
    const TileWalk walk(P, pt, b);

    if (warp == 0 || warp == 2) {
        // ---------------- TMA producers (both CTAs): warp 0 loads this CTA's x_routed rows, warp 2 its W2
        // rows; both complete on the leader's full barrier.
        if (lane == 0 && b < total_tiles && !MOE_PROBE(kProbeFreeRunMma)) {
            if (warp == 0) producer_role<TN, true, true>(P, pt, ring, ctl, b, deadline, rank, dry, walk);
            else producer_role<TN, true, false>(P, pt, ring, ctl, b, deadline, rank, dry, walk);
        }
        __syncwarp();
    } else if (warp == 1 && leader_cta) {
        // ---------------- MMA issuer (leader CTA only).  The whole warp runs the loop, converged, and one elected
        // lane issues.  Two measured facts shape it.  (1) The tensor pipe buffers little ahead of the MMA it
        // executes: 200 idle cycles of the issuer per k-block cost a launch 130 cycles per k-block
        // (bench.py --timeline --probe 32), so the loop is as short as it can be: a whole k-block (four MMAs and
        // the commit) is one statement with 32-bit descriptor arithmetic, addresses advance by additions, the
        // barrier's first look is the non-suspending test.  (2) tcgen05.mma takes its descriptors and addresses
        // from uniform registers: when a single thread ran this loop inside `if (lane == 0)` every operand was
        // moved over from ordinary registers, MMA by MMA; with warp-uniform values in warp-uniform control flow
        // and elect.sync around the issue the GEMM phase is 6 % faster.
        {
            constexpr uint32_t kLoStage = (uint32_t)(C::kStageBytes >> 4), kLoX = (uint32_t)(C::kWBytes >> 4);
            const uint32_t lo0 = smem_desc_lo(smem_u32(ring));
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            uint32_t w_lo = lo0, full_bar = full0, empty_bar = empty0;
            int stage = 0;
            uint32_t phase = 0;
            int it = 0;
            bool ok = true;
            TL_DECL(const long long tl_c0 = clock64(); long long tl_wf = 0, tl_wt = 0, tl_is = 0, tl_q; unsigned long long tl_late = 0;)
            for (int g = b; g < total_tiles && ok; g += pt.P, ++it) {
                const int a = it & 1;
                const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
                TL(tl_q = clock64());
                if (!__all_sync(0xffffffffu, mbar_test_wait(smem_u32(&ctl->tmem_empty[a]), acc_phase ^ 1u))) {
                    // (every lane polls; the vote keeps `ok`, and with it the loop, provably warp-uniform)
                    ok = __all_sync(0xffffffffu, wait_barrier_1t(smem_u32(&ctl->tmem_empty[a]), acc_phase ^ 1u, ctl, deadline, P.status, (uint32_t)g, 20u));
                    if (!ok) break;
                }
                TL(tl_wt += clock64() - tl_q);
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(a * TN);
                const auto wait_stage = [&]() {
                    if (MOE_PROBE(kProbeFreeRunMma) || __all_sync(0xffffffffu, mbar_test_wait(full_bar, phase) || dry)) return;
                    TL(++tl_late);
                    ok = __all_sync(0xffffffffu, wait_barrier_1t(full_bar, phase, ctl, deadline, P.status, (uint32_t)g, 21u));
                };
                const auto kloop = [&](auto full, uint32_t n) {
                    const uint32_t idesc = make_idesc(2 * kMmaM, decltype(full)::value ? TN : (int)n);
                    for (int kb = 0; kb < P.num_kb; ++kb) {
                        TL(tl_q = clock64());
                        wait_stage();
                        if (!ok) break;
                        TL(tl_wf += clock64() - tl_q; tl_q = clock64());
                        tc_fence_after();
                        if (MOE_PROBE(kProbeSlowIssuer)) {   // 200 cycles in which nothing is issued
                            const long long until = clock64() + 200;
                            while (clock64() < until) {}
                        }
                        if (dry) break;
                        if (elect_one_sync()) {
                            if ((kb < P.num_kb - 1 || P.last_ksteps == kBlockK / kUmmaK) && !MOE_PROBE(kProbeFreeRunMma)) {
                                tc_kblock_bf16_pair(d_tmem, w_lo, w_lo + kLoX, idesc, kb > 0 ? 1u : 0u, empty_bar);
                            } else {
                                const uint64_t w_desc = ((uint64_t)kSmemDescHi << 32) | w_lo, x_desc = w_desc + kLoX;
                                const int ksteps = (kb == P.num_kb - 1) ? P.last_ksteps : (kBlockK / kUmmaK);
                                for (int k = 0; k < ksteps; ++k)
                                    tc_mma_bf16_pair(d_tmem, w_desc + (uint64_t)(2 * k), x_desc + (uint64_t)(2 * k), idesc,
                                                     (k > 0 || kb > 0) ? 1u : 0u);
                                if (!MOE_PROBE(kProbeFreeRunMma)) tc_commit_pair(empty_bar);      // both CTAs may refill the stage
                            }
                        }
                        TL(tl_is += clock64() - tl_q);
                        w_lo += kLoStage;
                        full_bar += 8u;
                        empty_bar += 8u;
                        if (++stage == n_stages) {
                            stage = 0;
                            phase ^= 1u;
                            w_lo = lo0;
                            full_bar = full0;
                            empty_bar = empty0;
                        }
                    }
                };
                // full tiles in a loop of their own: with a constant N the issuer needs 27 cycles a k-block less
                wait_stage();
                if (!ok) break;
                const uint32_t n = MOE_PROBE(kProbeFreeRunMma) || dry ? 256u : ctl->tile_n[it & (kMaxStages - 1)];
                if (__all_sync(0xffffffffu, n == (uint32_t)TN)) kloop(std::true_type{}, 0u);
                else kloop(std::false_type{}, __reduce_max_sync(0xffffffffu, n));
                if (dry) break;
                __syncwarp();
                if (ok && elect_one_sync()) tc_commit_pair(smem_u32(&ctl->tmem_full[a]));   // both epilogues may start
                TL(if (it == 0 && lane == 0) tl_put(P, kTlFirstAcc, globaltimer_ns()));
            }
            TL(if (lane == 0) {
                   tl_put(P, kTlMmaEnd, globaltimer_ns()); tl_put(P, kTlTiles, (unsigned long long)it);
                   tl_put(P, kTlWaitOperand, (unsigned long long)tl_wf); tl_put(P, kTlIssue, (unsigned long long)tl_is);
                   tl_put(P, kTlWaitTmem, (unsigned long long)tl_wt); tl_put(P, kTlMmaCycles, (unsigned long long)(clock64() - tl_c0));
                   tl_put(P, kTlStageLate, tl_late); });
        }
        __syncwarp();
    } else if (warp >= 4 && warp < 4 + P.epi_warps) {
        if (!dry) epilogue_role<TN, true>(P, pt, ctl, b, tmem_base, deadline, (int)rank, walk);
    } else if (warp == 3) {
        if (!dry) publisher_role<true>(P, pt, ctl, b, deadline, (int)rank, walk);
    }
    if (dry) return;
    // ---------------- teardown: nobody leaves while its peer may still touch its memory (the co-resident
    // communication warps arrived on this cluster barrier at once)
    tc_fence_before();
    sync_compute_warps(P);
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, C::kTmemCols);
    }
}

// --------------------------------------------------------------------------- communication CTA

// two fp32 FMAs in one instruction (sm_100): acc = x * w + acc on packed pairs
__device__ __forceinline__ unsigned long long ffma2(unsigned long long x, unsigned long long w, unsigned long long acc)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x), "l"(w), "l"(acc));
    return d;
}
__device__ __forceinline__ unsigned long long pack_f32x2(uint32_t lo, uint32_t hi)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
    return d;
}
__device__ __forceinline__ void unpack_f32x2(unsigned long long v, float &lo, float &hi)
{
    uint32_t a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
    lo = __uint_as_float(a);
    hi = __uint_as_float(b);
}
// acc[i] (a pair of fp32) += w * (the two bf16 of word i), for the four words of v
__device__ __forceinline__ void fma2_bf16x8(unsigned long long (&acc)[4], const uint4 &v, unsigned long long ww)
{
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = ffma2(pack_f32x2(u[i] << 16, u[i] & 0xFFFF0000u), ww, acc[i]);
}

// The weights of a unit's rows, read back as shared-memory broadcasts.  `w`: lane j holds the weight of slot j (0: the slot has
// no source row); `wq`: room for k_tot floats, rounded up to the rows that reduce_unit takes together.
__device__ __forceinline__ void put_row_weights(const FusedParams &P, float w, float *wq)
{
    const int lane = threadIdx.x & 31;
    if (lane < P.k_tot) wq[lane] = w;
}
// Reduces one unit that sits in shared memory at `stage_s`: the weighted sum of its k_tot rows in slot order, one warp.  all_valid:
// every slot has a source row; `orow`: where the unit's columns of the token go; kAhead: rows fetched from shared memory together.
template <int kAhead>
__device__ __forceinline__ void reduce_unit(const FusedParams &P, bool all_valid, int n16, int row_bytes, const float *wq, uint32_t stage_s,
                                            __nv_bfloat16 *orow)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();   // the weights
    const uint32_t wq_s = smem_u32(wq);
#pragma unroll 1
    for (int c16 = lane; c16 < n16; c16 += 32) {
        unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
        uint32_t src = stage_s + (uint32_t)c16 * 16u, wsrc = wq_s;
        const auto add_rows = [&](int q, auto whole_group) {
            constexpr bool whole = decltype(whole_group)::value;
            uint4 v[kAhead];
            float wr[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i, src += (uint32_t)row_bytes)
                v[i] = whole || q + i < P.k_tot ? lds_v4(src) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int i = 0; i < kAhead; i += 4) {
                const uint4 w4 = lds_v4(wsrc + 4u * i);
                wr[i] = __uint_as_float(w4.x);
                wr[i + 1] = __uint_as_float(w4.y);
                wr[i + 2] = __uint_as_float(w4.z);
                wr[i + 3] = __uint_as_float(w4.w);
            }
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                // a slot without a source row holds bytes nobody wrote, and there is no row past the last slot: nothing is added
                if (!whole && ((!all_valid && wr[i] == 0.f) || q + i >= P.k_tot)) v[i] = make_uint4(0u, 0u, 0u, 0u), wr[i] = 0.f;
                fma2_bf16x8(acc, v[i], pack_f32x2(__float_as_uint(wr[i]), __float_as_uint(wr[i])));
            }
        };
#pragma unroll 1
        for (int q = 0; q < P.k_tot; q += kAhead, wsrc += 4u * kAhead) {
            // (long launches spare the checks of whole groups; short ones the second instance of the code)
            if (kAhead == 8 && all_valid && q + kAhead <= P.k_tot) add_rows(q, std::true_type{});
            else add_rows(q, std::false_type{});
        }
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float lo, hi;
            unpack_f32x2(acc[i], lo, hi);
            __nv_bfloat162 hh = __floats2bfloat162_rn(lo, hi);
            o[i] = *reinterpret_cast<uint32_t *>(&hh);
        }
        __stcs(reinterpret_cast<uint4 *>(orow + c16 * 8), make_uint4(o[0], o[1], o[2], o[3]));
    }
    __syncwarp();   // all lanes are done with the stage (and with wq) before either is reused
}

// Communication warp.  Y is token-major: the k_tot rows of one (token, split, column
// slab) are one contiguous block (a "unit", at most 8 KB).  Every communication warp works on its own:
// it owns two 8 KB stages of shared memory and one mbarrier per stage, fetches a unit with ONE bulk
// asynchronous copy (global -> shared), and while that copy is in flight it reduces the previous unit
// in fp32 in slot order with the token's weights and stores the bf16 result into the owning rank's
// buffer.  No warp waits on another one: the issue latency of the copies and the memory latency
// overlap across the warps of an SM.
//
// Who runs it (role):
//   kRoleFront       warp of a communication CTA, dynamic hand-out: ranges from the front of the
//                    per-split queues, split 0 first; a unit waits for the tiles under it (flags);
//   kRoleBack        warp of a compute CTA whose GEMM tiles are done (drain help): ranges from the back,
//                    last split first;
//   kRoleCoResident  extra warp of a compute CTA that is still computing: from the front, split 0
//                    first, but only from splits that are complete (it sleeps on the split counter
//                    instead of polling single tiles, so that it costs the computing warps nothing
//                    while it has nothing to do).
constexpr int kCommWarps = 12;
constexpr int kCommUnitBytes = 8192;
constexpr int kCommWarpBytes = 2 * kCommUnitBytes;
static_assert(kCommWarps * kCommWarpBytes <= kStageBytesTotal, "communication stages exceed the ring");
// Co-resident communication warps live in the aux region: two warps' stages (32 KB), then the per-row weights in compact
// 16-float slots -- four for co-resident warps, twelve for the CTA's own warps once they turn to
// communication (their usual 256-float slots would overlap the co-resident stages).  Needs k_tot <= 16.
constexpr int kCoWarpsAux = 2;          // co-resident warps whose stages fit the aux region
constexpr int kCoWeightFloats = 16;
constexpr int kCoWeightsOffset = kCoWarpsAux * kCommWarpBytes;
static_assert(PairCfg::kStageBytes <= kAuxBytes && 12 * 256 * 4 <= PairCfg::kStageBytes, "a seventh pair stage exceeds the allocation");
static_assert(kCoWeightsOffset + (kCoWarpsMax + kCommWarps) * kCoWeightFloats * 4 <= kAuxBytes,
              "co-resident stages and weights exceed the aux region");

enum { kRoleFront = 1, kRoleBack = 2, kRoleCoResident = 3 };

// what one communication warp owns
struct CommWarpRes {
    uint8_t *stages;              // 2 x kCommUnitBytes
    unsigned long long *full;     // 2 mbarriers (initialised with count 1 at kernel start)
    float *wq;                    // room for k_tot floats
};

struct CommUnit {
    int t, d, s, slab, wslab, ucols;
    float w;          // lane j: weight of slot j (0 when the slot has no source row)
    bool live;
    bool all_valid;   // every slot of the token has a source row
};

template <int TN>
__device__ void comm_warp(const FusedParams &P, const Part &pt, Control *ctl, const CommWarpRes res, int role, int tl_slot)
{
    (void)tl_slot;   // index of the warp's record in a timeline build
    const int lane = threadIdx.x & 31;
    const bool wait_needed = (P.mode != MOE_MODE_COMBINE_ONLY);
    const bool helper = (role == kRoleBack);
    const unsigned long long deadline = globaltimer_ns() + P.wait_ns;
    // the wait for a copy only follows a readiness wait: it gets a later deadline so that the first
    // report names the wait that really ran out
    const unsigned long long deadline2 = deadline + P.wait_ns / 4 + 1000000ull;

    TL_DECL(unsigned long long tl_first = 0, tl_last = 0, tl_sleep = 0; uint32_t tl_units = 0, tl_by_split[4] = {0u, 0u, 0u, 0u};)
    uint8_t *my_ring = res.stages;
    float *wq = res.wq;
    const unsigned long long y_policy = l2_evict_first_policy();
    const uint32_t full_s = smem_u32(res.full);
    const __nv_bfloat16 *Y = reinterpret_cast<const __nv_bfloat16 *>(P.Y);

    // reduce the unit sitting in stage `st` (its copy was issued one unit ago)
    auto consume = [&](const CommUnit &u, int st, uint32_t parity) -> bool {
        bool ok = wait_barrier(full_s + 8u * (uint32_t)st, parity, ctl, deadline2, P.status, (uint32_t)u.t, 43u);
        if (!ok) return false;
        __nv_bfloat16 *orow = reinterpret_cast<__nv_bfloat16 *>(P.out[u.d]) +
                              (size_t)(u.t - u.d * P.tok_blk) * (size_t)P.H + u.s * P.split_w + (u.slab << P.slab_shift);
        put_row_weights(P, u.w, wq);
        reduce_unit<8>(P, u.all_valid, u.ucols >> 3, u.wslab * 2, wq, smem_u32(my_ring + st * kCommUnitBytes), orow);
        TL(tl_last = globaltimer_ns(); if (tl_units == 0) tl_first = tl_last; ++tl_units; if (u.s < 4) ++tl_by_split[u.s]);
        return true;
    };

    int n_mine = 0;          // units this warp has issued so far: stage n_mine & 1, parity (n_mine >> 1) & 1
    CommUnit prev;
    prev.live = false;
    uint32_t ready_mask = wait_needed ? 0u : 0xffffffffu;   // bit s: split s is known to be complete

    // One unit: wait until the GEMM tiles under it are published (unless its split is known to be
    // complete), start its copy, then reduce the previous unit of this warp while the copy is in flight.
    // False when the warp had to give up (reported); nothing of this warp is in flight then.
    auto unit_step = [&](CommUnit &u) -> bool {
        // ---- readiness of the producing tiles
        if (!((ready_mask >> u.s) & 1u)) {
            uint32_t done = 0;
            if (lane == 0) done = ld_acquire_u32(&P.split_done[u.s]);
            done = __shfl_sync(0xffffffffu, done, 0);
            if (done >= (uint32_t)(pt.W_comp * P.flag_parts)) {
                ready_mask |= 1u << u.s;
            } else {
                // per tile: every (slot j, n-tile under this slab); a pair tile is published in two parts, one per CTA: its
                // column halves
                const int cs0 = u.slab << P.slab_shift, flag_cols = P.flag_parts == 2 ? TN / 2 : TN;
                const int in0 = cs0 / flag_cols;
                const int nt = (cs0 + u.ucols - 1) / flag_cols - in0 + 1;
                bool failed = false;
                for (int chk = lane; chk < P.k_tot * nt && !failed; chk += 32) {
                    const int j = chk / nt;
                    const int tn = chk - j * nt;
                    const int row = ld_chained(&P.pad_row[(size_t)u.t * P.k_tot + j]);
                    if (row < 0 || row >= P.R_pad) continue;
                    const int mu = row / P.tile_m;
                    const int g = (u.s * pt.W_comp + mu * P.NTs) * P.flag_parts + in0 + tn;
                    uint32_t spins = 0;
                    TL_DECL(const unsigned long long tl_f0 = globaltimer_ns();)
                    while (ld_acquire_u32(&P.flags[g]) != P.epoch) {
                        if ((++spins & 31u) == 0u && (ctl->abort || globaltimer_ns() > deadline)) {
                            report(P.status, MOE_DEV_TIMEOUT, (uint32_t)g, 40u);
                            failed = true;
                            break;
                        }
                        __nanosleep(64);
                    }
                    TL(tl_sleep += globaltimer_ns() - tl_f0);
                }
                if (__any_sync(0xffffffffu, failed)) {
                    // this warp gives up; the copy it still has in flight must land first
                    if (prev.live) consume(prev, (n_mine - 1) & 1, (uint32_t)((n_mine - 1) >> 1) & 1u);
                    prev.live = false;
                    return false;
                }
            }
            __syncwarp();
            // rows published through ordinary stores are read by the copy engine next
            asm volatile("fence.proxy.async;" ::: "memory");
        }
        // ---- issue this unit's copy, then reduce the previous unit while it is in flight
        const int st = n_mine & 1;
        if (lane == 0) {
            const uint32_t full = full_s + 8u * (uint32_t)st;
            const uint32_t bytes = (uint32_t)(P.k_tot * u.wslab) * 2u;
            const __nv_bfloat16 *src = Y + y_unit(u.t, u.s, u.slab << P.slab_shift, P.L, P.split_w, P.k_tot);
            mbar_arrive_expect_tx(full, bytes);
            bulk_load_once(smem_u32(my_ring + st * kCommUnitBytes), src, bytes, full, y_policy);   // Y is read once
        }
        __syncwarp();
        ++n_mine;
        if (prev.live && !consume(prev, (n_mine - 2) & 1, (uint32_t)((n_mine - 2) >> 1) & 1u)) {
            // the previous copy never landed (reported); wait for the one just issued, then leave
            const unsigned long long drain = globaltimer_ns() + 2000000ull;
            while (!mbar_try_wait(full_s + 8u * (uint32_t)st, (uint32_t)((n_mine - 1) >> 1) & 1u) && globaltimer_ns() < drain) {}
            prev.live = false;
            return false;
        }
        prev = u;
        return true;
    };

    // serve items [i0, i1) of split s on this warp alone.  An item is one token x one communication
    // column tile (token-major numbering); its units are the column slabs of that tile.
    auto serve_items = [&](int s, uint32_t i0, uint32_t i1) -> bool {
        const int split_c0 = s * P.split_w;
        const int split_c1 = min(P.H, split_c0 + P.split_w);
        int nxt_row = -1;
        float nxt_w = 0.f;
        if (lane < P.k_tot) {
            const int tn = (int)(i0 / (uint32_t)P.comm_cols);
            nxt_row = ld_chained(&P.pad_row[(size_t)tn * P.k_tot + lane]);
            nxt_w = ld_chained(&P.topk_w[(size_t)tn * P.k_tot + lane]);
        }
        for (uint32_t item = i0; item < i1; ++item) {
            const int tok = (int)(item / (uint32_t)P.comm_cols);
            const int col_tile = (int)(item - (uint32_t)tok * (uint32_t)P.comm_cols);
            int my_row = nxt_row;
            float my_w = nxt_w;
            if (item + 1 < i1 && lane < P.k_tot) {
                const int tn = (int)((item + 1) / (uint32_t)P.comm_cols);
                nxt_row = ld_chained(&P.pad_row[(size_t)tn * P.k_tot + lane]);
                nxt_w = ld_chained(&P.topk_w[(size_t)tn * P.k_tot + lane]);
            }
            if (lane < P.k_tot) {
                if (my_row >= P.R_pad) {
                    report(P.status, MOE_DEV_OOB, (uint32_t)my_row, 42u);
                    my_row = -1;
                }
                if (my_row < 0) my_w = 0.f;
            }
            const bool all_valid = __all_sync(0xffffffffu, lane >= P.k_tot || my_row >= 0);
            const int c0 = split_c0 + col_tile * kCommTileN;
            const int c1 = min(split_c1, c0 + kCommTileN);
            if (c0 >= c1) continue;
            const int slab0 = (c0 - split_c0) >> P.slab_shift;
            const int slab1 = (c1 - split_c0 + P.slab_cols - 1) >> P.slab_shift;
            for (int slab = slab0; slab < slab1; ++slab) {
                CommUnit u;
                u.t = tok;
                u.d = tok / P.tok_blk;
                u.s = s;
                u.slab = slab;
                u.wslab = min(P.slab_cols, P.split_w - (slab << P.slab_shift));
                u.ucols = min(u.wslab, split_c1 - split_c0 - (slab << P.slab_shift));
                u.w = my_w;
                u.live = true;
                u.all_valid = all_valid;
                if (!unit_step(u)) return false;
            }
        }
        return true;
    };

    {
        // Dynamic hand-out, to warps.  Every split has a two-ended queue of its items in one 64-bit word
        // (low half: items taken from the front, high half: from the back).  Warps of the communication
        // CTAs and co-resident warps take from the front, split 0 first; warps of compute CTAs that have
        // run out of GEMM tiles take from the back, last split first.  One atomic add claims a range;
        // ranges shrink towards the end so that the last ones finish together.  The next claim is issued
        // before the current range is served, which hides the latency of the atomic.
        const uint32_t n_items = (uint32_t)P.T * (uint32_t)P.comm_cols;
        int s = helper ? P.L - 1 : 0;
        unsigned long long old = 0;
        uint32_t chunk = 0;
        auto claim = [&](int split) {   // lane 0 issues the atomic; the result is picked up later
            if (lane == 0) {
                const unsigned long long q = *reinterpret_cast<volatile unsigned long long *>(&P.queue[split]);
                const uint32_t taken = (uint32_t)q + (uint32_t)(q >> 32);
                const uint32_t rem = taken < n_items ? n_items - taken : 0u;
                chunk = min(8u, max(1u, rem >> 12));
                old = atomicAdd(&P.queue[split], helper ? ((unsigned long long)chunk << 32) : (unsigned long long)chunk);
            }
        };
        bool claimed = false;      // a claim on split s is outstanding
        while (s >= 0 && s < P.L) {
            if (!claimed) {
                if (role == kRoleCoResident && !((ready_mask >> s) & 1u)) {
                    // A co-resident warp only takes work that can be served at once.  Inside a split the
                    // tiles run expert by expert and a token needs tiles of all its experts, so hardly any
                    // token is complete before the split is: wait for the whole split, asleep most of the time.
                    uint32_t state = 0;   // 1: split complete, 2: split handed out already, 3: give up
                    if (lane == 0) {
                        if (ld_acquire_u32(&P.split_done[s]) >= (uint32_t)(pt.W_comp * P.flag_parts)) state = 1;
                        else {
                            const unsigned long long q = *reinterpret_cast<volatile unsigned long long *>(&P.queue[s]);
                            if ((uint32_t)q + (uint32_t)(q >> 32) >= n_items) state = 2;
                            else if (ctl->abort) state = 3;
                            else if (globaltimer_ns() > deadline) {
                                report(P.status, MOE_DEV_TIMEOUT, (uint32_t)s, 44u);
                                state = 3;
                            }
                        }
                    }
                    state = __shfl_sync(0xffffffffu, state, 0);
                    if (state == 0) {
                        TL_DECL(const unsigned long long tl_s0 = globaltimer_ns();)
                        __nanosleep(2000);
                        TL(tl_sleep += globaltimer_ns() - tl_s0);
                        continue;
                    }
                    if (state == 2) {
                        ++s;
                        continue;
                    }
                    if (state == 3) {
                        ctl->abort = 1u;
                        break;
                    }
                    ready_mask |= 1u << s;
                    // rows published through ordinary stores are read by the copy engine next
                    asm volatile("fence.proxy.async;" ::: "memory");
                }
                claim(s);
                claimed = true;
            }
            const unsigned long long o = __shfl_sync(0xffffffffu, old, 0);
            const uint32_t ch = __shfl_sync(0xffffffffu, chunk, 0);
            const uint32_t f = (uint32_t)o, bk = (uint32_t)(o >> 32);
            const uint32_t hi = bk < n_items ? n_items - bk : 0u;    // items [hi, n) are taken from the back
            uint32_t i0, i1;
            if (!helper) {
                i0 = f;
                i1 = min(f + ch, hi);
            } else {
                i1 = hi;
                i0 = max(f, hi > ch ? hi - ch : 0u);
            }
            const int cur = s;
            if (i0 >= i1) {                      // this split is handed out: go on to the next one
                s += helper ? -1 : 1;
                claimed = false;
                continue;
            }
            claim(s);
            // warp-uniform exit: the loop body holds full-mask collectives
            if (__any_sync(0xffffffffu, ctl->abort != 0u)) break;
            if (!serve_items(cur, i0, i1)) {
                ctl->abort = 1u;
                return;
            }
        }
    }
    if (prev.live) consume(prev, (n_mine - 1) & 1, (uint32_t)((n_mine - 1) >> 1) & 1u);
#if MOE_TIMELINE
    if (lane == 0) {
        if (role == kRoleCoResident) {
            const int base = kTlCoWarp + 8 * tl_slot;
            tl_put(P, base + 0, tl_first); tl_put(P, base + 1, tl_last); tl_put(P, base + 2, tl_units); tl_put(P, base + 3, tl_sleep);
            for (int i = 0; i < 4; ++i) tl_put(P, base + 4 + i, tl_by_split[i]);
        } else if (tl_slot == 0) {
            tl_put(P, kTlCommUnits, tl_units);
            tl_put(P, kTlCommWaitNs, tl_sleep);
        }
    }
#endif
}

// The communication warps of a CTA whose only role is communication (dedicated communication CTA, or a
// compute CTA that has run out of GEMM tiles): warps 0-11, stages in the operand ring.
template <int TN>
__device__ __forceinline__ void comm_cta(const FusedParams &P, const Part &pt, uint8_t *ring, Control *ctl, uint8_t *aux, int role)
{
    const int warp = threadIdx.x >> 5;
    if (warp >= kCommWarps) return;
    CommWarpRes res;
    res.stages = ring + warp * kCommWarpBytes;
    res.full = &ctl->comm_full[2 * warp];
    res.wq = (role == kRoleBack && P.co_warps > 0)
                 ? reinterpret_cast<float *>(aux + kCoWeightsOffset) + (kCoWarpsMax + warp) * kCoWeightFloats
                 : reinterpret_cast<float *>(aux) + warp * 256;
    comm_warp<TN>(P, pt, ctl, res, role, warp);
}

// Communication work by shares: the units of a split, dealt one by one over the serving CTAs first, then over their warps
// 0-11, once the tiles under them are done: all CTAs when the compute CTAs help (FusedParams::even: once for all splits), the
// communication CTAs under the static partition (split after split).  Nothing is handed out and one thread of the CTA waits:
// the queues' atomics and the polling of all warps on one word took longer than the work of a small launch; and with whole
// communication tiles per CTA (the paper's map) CTAs have no work where tiles are few (DeepSeek shape, T = 2048, EP = 4, static:
// 16 tiles a split, so that 32 CTAs took as long as 16, 218 us; 167 us by units).  What is left of a small launch's tail is
// mostly latency, instruction fetches among it (it runs this code once, from L2 at best): so the loop is short, one instance of
// every step.  (Rows read straight into registers by 20 warps, eight loads ahead, instead of by one bulk copy per unit into
// shared memory: 46 GB/s a CTA instead of 56.)
// `c` of `n_ctas` serving CTAs.
constexpr int kRowsAhead = 4;   // rows of a unit fetched from shared memory together
__device__ __forceinline__ void serve_shares(const FusedParams &P, const Part &pt, uint8_t *ring, Control *ctl, uint8_t *aux, int c, int n_ctas)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= kCommWarps) return;
    uint8_t *stages = ring + warp * kCommWarpBytes;
    float *wq = reinterpret_cast<float *>(aux) + warp * 256;      // weights of the unit's rows
    const uint32_t full = smem_u32(&ctl->comm_full[2 * warp]);
    const unsigned long long deadline = globaltimer_ns() + P.wait_ns, deadline2 = deadline + P.wait_ns / 4 + 1000000ull;
    const unsigned long long y_policy = l2_evict_first_policy();
    const __nv_bfloat16 *Y = reinterpret_cast<const __nv_bfloat16 *>(P.Y);
    // unit n of a split: token n / n_slabs, column slab n % n_slabs; this warp's next one is `workers` on
    const int n_slabs = (P.split_w + P.slab_cols - 1) >> P.slab_shift, workers = kCommWarps * n_ctas;
    const int step_tok = small_quotient(workers, n_slabs), step_slab = workers - step_tok * n_slabs;
    int k = 0;                // copies issued so far: stage k & 1, parity (k >> 1) & 1
    int n = warp * n_ctas + c, past = 0;      // this warp's first unit of the split; even: units of a split, modulo `workers`
#pragma unroll 1
    for (int s = 0; s < P.L; ++s) {
        if (P.even && s > 0) {     // the deal goes on where the split before ended
            if (s == 1) past = P.T * n_slabs - small_quotient(P.T * n_slabs, workers) * workers;
            n -= past;
            if (n < 0) n += workers;
        }
        int tok = small_quotient(n, n_slabs), slab = n - tok * n_slabs, d = 0;
        // routing of a unit's token, fetched one unit ahead: lane j, row and weight of slot j
        int row = -1;
        float w = 0.f;
        const auto fetch_routing = [&]() {
            row = -1;
            w = 0.f;
            if (tok < P.T && lane < P.k_tot) {
                row = ld_chained(&P.pad_row[(size_t)tok * P.k_tot + lane]);
                w = ld_chained(&P.topk_w[(size_t)tok * P.k_tot + lane]);
            }
        };
        fetch_routing();
        if (P.mode != MOE_MODE_COMBINE_ONLY && (s == 0 || !P.even)) {
            if (threadIdx.x == 0) {
                for (int sw = s; sw < (P.even ? P.L : s + 1) && !ctl->abort; ++sw) {
                    uint32_t spins = 0;
                    while (ld_acquire_u32(&P.split_done[sw]) < (uint32_t)(pt.W_comp * P.flag_parts)) {
                        if ((++spins & 31u) == 0u && globaltimer_ns() > deadline) {
                            report(P.status, MOE_DEV_TIMEOUT, (uint32_t)sw, 45u);
                            ctl->abort = 1u;
                            break;
                        }
                        __nanosleep(64);
                    }
                }
            }
            asm volatile("bar.sync 2, %0;" ::"r"(32 * kCommWarps) : "memory");
            // rows published through ordinary stores are read by the copy engine next
            asm volatile("fence.proxy.async;" ::: "memory");
        }
        // (a warp that gives up keeps coming to the barriers)
        if (__any_sync(0xffffffffu, ctl->abort != 0u)) continue;
        // the unit in flight: issued one round ago
        bool flying = false, all_valid = false;
        int n16 = 0, row_bytes = 0;
        float w_f = 0.f;
        __nv_bfloat16 *orow = nullptr;
#pragma unroll 1
        while (true) {
            const bool have = tok < P.T;
            bool valid_n = false;
            int n16_n = 0, row_bytes_n = 0;
            float w_n = 0.f;
            __nv_bfloat16 *orow_n = nullptr;
            if (have) {
                const int c0 = slab << P.slab_shift, split_cols = min(P.H, (s + 1) * P.split_w) - s * P.split_w;
                const int wslab = min(P.slab_cols, P.split_w - c0);            // layout pitch
                n16_n = max(0, min(wslab, split_cols - c0)) >> 3;              // 16-byte chunks of real columns
                row_bytes_n = wslab * 2;
                while (tok >= (d + 1) * P.tok_blk) ++d;                        // owning rank
                if (lane < P.k_tot) {
                    if (row >= P.R_pad) {
                        report(P.status, MOE_DEV_OOB, (uint32_t)row, 42u);
                        row = -1;
                    }
                    if (row < 0) w = 0.f;
                }
                orow_n = reinterpret_cast<__nv_bfloat16 *>(P.out[d]) + (size_t)(tok - d * P.tok_blk) * (size_t)P.H + s * P.split_w + c0;
                if (lane == 0) {
                    const uint32_t bytes = (uint32_t)(P.k_tot * row_bytes_n), bar = full + 8u * (uint32_t)(k & 1);
                    const __nv_bfloat16 *src = Y + y_unit(tok, s, c0, P.L, P.split_w, P.k_tot);
                    mbar_arrive_expect_tx(bar, bytes);
                    bulk_load_once(smem_u32(stages + (k & 1) * kCommUnitBytes), src, bytes, bar, y_policy);   // Y is read once
                }
                w_n = w;
                valid_n = __all_sync(0xffffffffu, lane >= P.k_tot || row >= 0);
                ++k;
                tok += step_tok;
                slab += step_slab;
                if (slab >= n_slabs) {
                    slab -= n_slabs;
                    ++tok;
                }
                fetch_routing();
            }
            if (flying) {
                const int prev = k - 1 - (have ? 1 : 0), st = prev & 1;
                put_row_weights(P, w_f, wq);
                if (!wait_barrier(full + 8u * (uint32_t)st, (uint32_t)(prev >> 1) & 1u, ctl, deadline2, P.status, (uint32_t)tok, 43u)) {
                    // (reported) the copy just issued must land before shared memory is released
                    const unsigned long long drain = globaltimer_ns() + 2000000ull;
                    while (have && !mbar_try_wait(full + 8u * (uint32_t)((k - 1) & 1), (uint32_t)((k - 1) >> 1) & 1u) && globaltimer_ns() < drain) {}
                    break;
                }
                reduce_unit<kRowsAhead>(P, all_valid, n16, row_bytes, wq, smem_u32(stages + st * kCommUnitBytes), orow);
            }
            if (!have) break;
            flying = true;
            all_valid = valid_n;
            n16 = n16_n;
            row_bytes = row_bytes_n;
            w_f = w_n;
            orow = orow_n;
        }
    }
}

// Co-resident communication warp `cw` of a compute CTA: stages and weights in the aux region.
template <int TN>
__device__ __forceinline__ void co_resident_warp(const FusedParams &P, const Part &pt, Control *ctl, uint8_t *aux, int cw)
{
    CommWarpRes res;
    res.stages = aux + cw * kCommWarpBytes;
    res.full = &ctl->co_full[2 * cw];
    res.wq = reinterpret_cast<float *>(aux + kCoWeightsOffset) + cw * kCoWeightFloats;
    comm_warp<TN>(P, pt, ctl, res, kRoleCoResident, cw);
}

// Co-resident warp number of warp 16..19.  The four warp schedulers of an SM take warps by number modulo
// four, and scheduler 1 holds the thread that issues the MMAs, which has to stay ahead of the tensor pipe:
// warps 18 and 19 are used first, then 16, and 17 (scheduler 1) last.
__device__ __forceinline__ int co_warp_number(int warp)
{
    return warp == 18 ? 0 : warp == 19 ? 1 : warp == 16 ? 2 : 3;
}

// Barriers of every communication stage the CTA may use, and the abort flag; before the first CTA-wide
// barrier of the kernel.
__device__ __forceinline__ void init_comm_barriers(Control *ctl)
{
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * kCommWarps; ++i) mbar_init(smem_u32(&ctl->comm_full[i]), 1);
        for (int i = 0; i < 2 * kCoWarpsMax; ++i) mbar_init(smem_u32(&ctl->co_full[i]), 1);
        ctl->abort = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
}

// --------------------------------------------------------------------------- kernel

// The launch's partition.  With the routed counts left on the device the m-tile count S is read from the routing
// workspace (the routing kernel ran earlier on the same stream); with the selector's picks tabulated over S
// (FusedParams::c_table) the communication-CTA count is looked up by it, so that no host wait lies between the
// routing build and this launch.
__device__ __forceinline__ Part launch_part(const FusedParams &P)
{
    Part pt = {P.W_comp, P.S, P.C, P.P};
    if (P.S_dev) {
        const int S = ld_chained_uniform(P.S_dev);
        pt.S = min(S, P.S);
        pt.W_comp = pt.S * P.NTs;
        if (P.c_table_n > 0) {
            pt.C = P.c_table[max(0, min(S - P.c_table_first, P.c_table_n - 1))];
            pt.P = (P.G - pt.C) >> (P.slot_sms - 1);
        }
    }
    if (P.balance) {
        // As many waves as all slots need, over as few slots as then suffice: the same number of tiles on each but the last
        // few.  The CTAs left over only serve their share of the combine; with them computing too the same waves take longer
        // (DeepSeek shape T = 128: 78.5 -> 74.6 us whole step, Qwen shape T = 512 74.3 -> 70.7).  Against the plan's C, with counts
        // on the device: DeepSeek shape T = 16 63.1 -> 57.2, T = 300 85.2 -> 77.1, T = 1024 120.9 -> 116.3; with counts on the
        // host: Granite shape T = 4096 89.1 -> 85.4, Qwen shape T = 8192 235.4 -> 233.1, others equal.
        const int tiles = pt.W_comp * P.L, waves = max(1, small_quotient(tiles + P.P - 1, P.P));     // (few_units bounds the tiles)
        pt.P = max(1, small_quotient(tiles + waves - 1, waves));
        pt.C = (P.P - pt.P) * P.slot_sms;
    }
    return pt;
}

template <int TN>
__global__ void __launch_bounds__(kFusedThreads, 1)
moe_gemm2_combine_kernel(const __grid_constant__ FusedParams P)
{
    extern __shared__ uint8_t smem_raw[];
    // 128B-swizzled tiles need 1024-byte aligned bases
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    Control *ctl = reinterpret_cast<Control *>(ring + kStageBytesTotal);
    uint8_t *aux = reinterpret_cast<uint8_t *>(ring + kStageBytesTotal + ((sizeof(Control) + 127) & ~(size_t)127));
    const int warp = threadIdx.x >> 5;

    // what does not depend on the predecessor is done before the wait for it: barriers, TMEM, tensor maps
    init_comm_barriers(ctl);
    if (P.P > 0) compute_setup<TN>(P, ctl);
    if (threadIdx.x == 96) {
        prefetch_tensormap(&P.tmA);
        prefetch_tensormap(&P.tmB);
    }
    grid_dependency_wait();
    if (P.routing.topk_idx)
        routing_inline<kFusedThreads / 32, true>(P.routing, P.k_tot, P.E_tot, P.tile_m, P.status, P.mail, P.mail_seq, reinterpret_cast<int32_t *>(ring));
    if (blockIdx.x == 0 && threadIdx.x < (unsigned)P.L) {
        P.split_done_next[threadIdx.x] = 0u;
        P.queue_next[threadIdx.x] = 0ull;
    }
    const Part pt = launch_part(P);
    tc_fence_before();
    __syncthreads();          // the only barrier all 20 warps share
    tc_fence_after();
    TL(if (threadIdx.x == 0) { tl_put(P, kTlBegin, globaltimer_ns()); tl_put(P, kTlRole, (int)blockIdx.x < pt.C ? 0u : 1u); });

    const bool queued = P.drain_help && !P.even;           // (drain help is a matter of fused launches)
    if (P.mail && !P.routing.topk_idx && blockIdx.x == 0 && warp == kCommWarps)
        mail_counts(P.mail, P.mail_seq, P.E_tot, threadIdx.x & 31, [&](int x) { return ld_chained(P.S_dev - P.E_tot + x); });
    if ((int)blockIdx.x < pt.C) {
        if (warp == 1 && P.P > 0) tmem_dealloc(ctl->tmem_base, Cfg<TN>::kTmemCols);
        if (queued) comm_cta<TN>(P, pt, ring, ctl, aux, kRoleFront);
    } else if (warp >= kThreads / 32 && P.epi_warps == 12) {
        if (co_warp_number(warp) < P.co_warps) co_resident_warp<TN>(P, pt, ctl, aux, co_warp_number(warp));
        return;
    } else {
        compute_cta<TN>(P, pt, ring, ctl, (int)blockIdx.x - pt.C);
        TL(if (threadIdx.x == 0) tl_put(P, kTlComputeEnd, globaltimer_ns()));
        // out of GEMM tiles: help with the communication that is left (all TMA and TMEM traffic is over)
        if (queued && !ctl->abort) comm_cta<TN>(P, pt, ring, ctl, aux, kRoleBack);
    }
    if (P.even || (!queued && (int)blockIdx.x < pt.C)) serve_shares(P, pt, ring, ctl, aux, (int)blockIdx.x, P.even ? (int)gridDim.x : pt.C);
    TL(if (threadIdx.x == 0) tl_put(P, kTlCtaEnd, globaltimer_ns()));
}

// Pair kernel: launched with clusters of two CTAs.  Communication CTAs are single CTAs (blockIdx < C);
// with an odd C the cluster-mate of the last one has no role; compute pairs start at the next even index.
__global__ void __launch_bounds__(kFusedThreads, 1)
moe_gemm2_combine_pair_kernel(const __grid_constant__ FusedParams P)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    // Layout: six operand stages, the control block, the aux region -- or, when no co-resident communication warp needs the aux region
    // while the GEMM runs, seven stages and the control block; the seventh stage then serves as the aux region of the
    // communication role, which only starts after the CTA's last MMA (drain help) or never computes (communication CTA).
    const bool seven = P.stages == 7;
    Control *ctl = reinterpret_cast<Control *>(ring + kStageBytesTotal + (seven ? PairCfg::kStageBytes : 0));
    uint8_t *aux = seven ? ring + kStageBytesTotal
                         : reinterpret_cast<uint8_t *>(ring + kStageBytesTotal + ((sizeof(Control) + 127) & ~(size_t)127));
    const int warp = threadIdx.x >> 5;

    // what does not depend on the predecessor is done before the wait for it
    init_comm_barriers(ctl);
    if (P.P > 0) pair_setup(P, ctl);
    if (threadIdx.x == 96) {
        prefetch_tensormap(&P.tmA);
        prefetch_tensormap(&P.tmB);
    }
    tc_fence_before();
    cluster_sync_all();       // the only barrier all 20 warps share
    tc_fence_after();
    // Twice through the code of the producers and the issuer: dry, before the predecessor is waited for, then in earnest.  A launch runs
    // cold: from the end of the wait to the first copy a producer took 8000 cycles, almost all of them misses of its instruction and constant
    // caches, one after the other.  Behind a routing build this CTA has 10000 cycles to itself before the wait ends; with the dry round
    // (4800 cycles) in them it is 3700 from there to the first copy (whole calls, with the set-up moved in front of the wait, us:
    // Granite shape T = 4096 91.6 -> 89.1, its whole layer T = 1003 81.9 -> 80.7, Qwen shape T = 8192 236 -> 232).  The dry round
    // touches neither barriers' phases nor memory, and reads nothing that the predecessor writes.  (With the combine's code in
    // it as well it takes 12000 cycles, which is longer than the wait: whole layer T = 1003 +2 %.  In GEMM1: 0 to +1 %.)
    const bool queued = P.drain_help && !P.even;           // (drain help is a matter of fused launches)
    const bool co_resident = warp >= kThreads / 32 && P.epi_warps == 12;
    Part pt = {1, 1, 0, 1};
    int c_even = 0;
#pragma unroll 1
    for (int round = P.P > 0 ? 0 : 1; round < 2; ++round) {
        const bool dry = round == 0;
        if (!dry) {
            grid_dependency_wait();
            if (blockIdx.x == 0 && threadIdx.x < (unsigned)P.L) {
                P.split_done_next[threadIdx.x] = 0u;
                P.queue_next[threadIdx.x] = 0ull;
            }
            pt = launch_part(P);
            c_even = (pt.C + 1) & ~1;
            TL(if (threadIdx.x == 0) { tl_put(P, kTlBegin, globaltimer_ns()); tl_put(P, kTlRole, (int)blockIdx.x < c_even ? 0u : 1u); });
            if (P.mail && blockIdx.x == 0 && warp == kCommWarps)
                mail_counts(P.mail, P.mail_seq, P.E_tot, threadIdx.x & 31, [&](int x) { return ld_chained(P.S_dev - P.E_tot + x); });
            if ((int)blockIdx.x < c_even) {
                if (warp == 1 && P.P > 0) tmem_dealloc_pair(ctl->tmem_base, PairCfg::kTmemCols);
                break;
            }
        }
        if (!co_resident) compute_cta_pair(P, pt, ring, ctl, dry ? 0 : ((int)blockIdx.x - c_even) >> 1, dry);
    }
    if ((int)blockIdx.x < c_even) {
        // odd C: the last communication CTA's cluster-mate cannot compute (no partner).  With dynamic work
        // distribution it serves communication work as well; under the static map it has no tile list.
        if (queued) comm_cta<256>(P, pt, ring, ctl, aux, kRoleFront);
    } else if (co_resident) {
        // The compute warps of both CTAs meet at a cluster barrier at the end, and a cluster barrier counts every thread: these
        // warps arrive at once (they hold nothing a peer could touch) and pick its completion up when their own work is done.
        cluster_arrive();
        if (co_warp_number(warp) < P.co_warps) co_resident_warp<256>(P, pt, ctl, aux, co_warp_number(warp));
        cluster_wait();
        return;
    } else {
        TL(if (threadIdx.x == 0) tl_put(P, kTlComputeEnd, globaltimer_ns()));
        if (queued && !ctl->abort) comm_cta<256>(P, pt, ring, ctl, aux, kRoleBack);
    }
    // The next kernel on the stream may be placed while the shares are served: a following step's routing build, and GEMM1 behind
    // it, then start 2-3 us earlier (whole layer, Granite shape T = 1003 86.5 -> 84.1 us).  (One-CTA tiles: 0 to +0.4 us, not done.)
    if (P.even) grid_dependents_may_launch();
    if (P.even || (!queued && (int)blockIdx.x < pt.C)) serve_shares(P, pt, ring, ctl, aux, (int)blockIdx.x, P.even ? (int)gridDim.x : pt.C);
    TL(if (threadIdx.x == 0) tl_put(P, kTlCtaEnd, globaltimer_ns()));
}

}  // namespace

int fused_co_warps_max() { return kCoWarpsAux; }
int fused_stages(bool pair, int tile_n, int x_rows, bool aux_free, int *stage_bytes)
{
    const int kbs = tile_n == 64 ? (x_rows == 32 ? Cfg<64>::kThinKb : Cfg<64>::kStageKb) : tile_n == 128 ? Cfg<128>::kStageKb : 1;
    *stage_bytes = pair ? PairCfg::kStageBytes : (tile_n + x_rows) * kBlockK * 2 * kbs;
    const int n = kStageBytesTotal / *stage_bytes + (pair && aux_free ? 1 : 0);
    return n < kMaxStages ? n : kMaxStages;
}
bool fused_timeline_build() { return MOE_TIMELINE != 0; }

size_t fused_smem_bytes(int) { return (size_t)kStageBytesTotal + 1024 + ((sizeof(Control) + 127) & ~(size_t)127) + kAuxBytes; }

template <int TN>
static cudaError_t prepare()
{
    return cudaFuncSetAttribute(moe_gemm2_combine_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)fused_smem_bytes(TN));
}

cudaError_t fused_occupancy(int tile_n, int *blocks_per_sm)
{
    cudaError_t e;
    const size_t sm = fused_smem_bytes(tile_n);
    switch (tile_n) {
    case 64:
        if ((e = prepare<64>()) != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, moe_gemm2_combine_kernel<64>, kFusedThreads, sm);
    case 128:
        if ((e = prepare<128>()) != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, moe_gemm2_combine_kernel<128>, kFusedThreads, sm);
    case 256:
        if ((e = prepare<256>()) != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, moe_gemm2_combine_kernel<256>, kFusedThreads, sm);
    }
    return cudaErrorInvalidValue;
}

cudaError_t pair_occupancy(int *blocks_per_sm, int *max_clusters)
{
    const size_t sm = fused_smem_bytes(256);
    cudaError_t e = cudaFuncSetAttribute(moe_gemm2_combine_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, moe_gemm2_combine_pair_kernel, kFusedThreads, sm);
    if (e != cudaSuccess) return e;
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_sm & ~1));
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = sm;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(max_clusters, moe_gemm2_combine_pair_kernel, &cfg);
}

cudaError_t pair_launch(const FusedParams &p, int grid, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = fused_smem_bytes(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0] = chained_launch_attribute();
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, moe_gemm2_combine_pair_kernel, p);
}

cudaError_t fused_launch(int tile_n, const FusedParams &p, int grid, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = fused_smem_bytes(tile_n);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1] = {chained_launch_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    switch (tile_n) {
    case 64: return cudaLaunchKernelEx(&cfg, moe_gemm2_combine_kernel<64>, p);
    case 128: return cudaLaunchKernelEx(&cfg, moe_gemm2_combine_kernel<128>, p);
    case 256: return cudaLaunchKernelEx(&cfg, moe_gemm2_combine_kernel<256>, p);
    }
    return cudaErrorInvalidValue;
}

}  // namespace moe
