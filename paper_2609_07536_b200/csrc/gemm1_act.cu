// Up-stream stage of the post-router MoE layer on one GPU (Section II-A, steps 1 and 2): the rows of the
// hidden states are collected in routed order (the paper's AllGather; here all tokens are local, so it
// is a gather by the routing permutation), grouped GEMM1 computes the gate and the up projection of
// every routed row with its expert's weights, and the gated activation silu(gate) * up forms x_routed,
// the input of GEMM2 + GatherRS.  The paper leaves this stage unchanged and does not name the
// activation; SiLU gating is the reading taken.
//
// One persistent kernel, one 512-thread CTA per SM.  The gather is part of the operand loads: four loader warps know
// the token of every row of the tile and copy each k-block of those rows straight from the hidden states into the
// 128B-swizzled stage (16-byte cp.async, eight lanes per row).  A gather launch in front wrote and re-read the routed
// rows, k_tot times the hidden states: 142 us and 1 GB of a 1280 us stage at 131072 rows of 2048 (now 1260 in all; Granite
// shape, T = 4096: 120 -> 98 us).  (One TMA tile::gather4 copy per four rows does not keep up: 80 cycles each on an SM, 3660 us
// for the stage.)  Rows past the end
// of an expert's last tile are not fetched at all: nothing stored depends on them.
// The weights are on the M side of the MMA, the rows on its N side, as in the fused kernel: N is the tile's row count rounded up to 16
// (a pair: 32), so that a tile costs what its rows cost.  The rows of W1 come in groups of 32, 16 gate rows and the 16 up rows of the
// same columns: then the gate and the up projection of an output lie in one TMEM lane quarter, 16 lanes apart, and the 16-lane loads of
// the epilogue put them into the same register of the same thread.
// (Rows on the M side, every tile computed for 128 or 256 of them -> now, whole layer, us: DeepSeek shape T = 1 40.4 -> 39.0,
// Qwen shape T = 48 179 -> 165, Granite shape T = 1003 84.3 -> 82.1, DeepSeek shape T = 16384, 6 % padding, 2106 -> 2091; same bits.)
//   tile_m <= 128: tile = up to 128 routed rows x 128 intermediate columns per CTA (two MMAs of 64), four 48 KB stages;
//   tile_m = 256 : tile = up to 256 rows x 128 columns per pair of CTAs (tcgen05 cta_group::2), seven 32 KB stages: each CTA
//                  holds half of the rows and loads the gate and up rows of 64 columns, so that a k-block costs an SM 32 KB
//                  instead of 48.
//   warp 0      TMA producer (one thread): the expert's rows of W1 for the tile's columns (64 k), one copy;
//   warps 12-15 loaders of the gathered rows; their copies arrive by themselves on the stage's `rows` barrier;
//   warp 2      relay (one thread): waits for that barrier, makes the rows visible to the tensor core's proxy and
//               arrives on the stage's full barrier (a fence in the issuing warp would cost every k-block its cycles).  Pair: the
//               other CTA's relay arrives on the leader's barrier;
//   warp 1      issues tcgen05.mma (converged warp, elected lane; K = 16, bf16 -> fp32) into one of two accumulator buffers in TMEM;
//   warps 4-11  epilogue: tcgen05.ld of the gate and the up values of 16 columns x 32 rows, silu(g) * u in fp32,
//               bf16, transposed, one 32-byte store per row (x_routed rows are contiguous: no scatter here).
// The n-tile index runs fastest in the tile sequence, so the CTAs of a wave share the gathered rows.
// Every wait is bounded like in the fused kernel (status word, no trap).

#include <cuda_bf16.h>

#include <cstring>
#include <type_traits>

#include "moe_internal.h"
#include "routing_device.cuh"
#include "sm100_device.cuh"

namespace moe {
namespace {

constexpr int kG1TileN = 128;                                   // intermediate columns per tile; 64 or 96 for the smallest batches
constexpr int kG1EpiWarps = 8;          // warps 4..11: two column groups x four TMEM lane quarters
constexpr int kG1LoadWarps = 4;         // warps 12..15
constexpr int kG1RowsPerStep = 4 * kG1LoadWarps;   // rows that one copy instruction of all loader warps covers
constexpr int kG1MaxStages = 7;

// TN: intermediate columns per tile (a pair: 128)
template <bool kPair, int TN>
struct G1Cfg {
    static constexpr int kCols = kPair ? TN / 2 : TN;                                // intermediate columns whose weights this CTA loads
    static constexpr int kWBytes = 2 * kCols * kBlockK * 2;                          // their gate and up rows
    static constexpr int kXBytes = kMmaM * kBlockK * 2;                              // 16 KB: up to 128 rows of the hidden states
    static constexpr int kStageBytes = kWBytes + kXBytes;                            // (TN = 96: the second MMA reads 64 rows past the weights, for lanes nobody reads)
    static constexpr int kStages = kPair || TN == 64 ? kG1MaxStages : TN == 96 ? 5 : 4;
    static constexpr int kBlocks = kPair || TN == 64 ? 1 : 2;                        // MMAs per K = 16, of 64 intermediate columns (a pair: 128)
    static constexpr int kAccCols = kPair ? 2 * kMmaM : kBlocks * kMmaM;             // TMEM columns of an accumulator buffer
    static constexpr int kTmemCols = 2 * kAccCols;
    static constexpr int kRingBytes = kStages * kStageBytes;
};

struct alignas(64) G1Params {
    CUtensorMap tmW;   // W1 [E_tot][2][I][H] as [E_tot][I / 16][2][16][H]    box: a CTA's columns / 16 groups of 32 rows x 64
    const int32_t *mtile_expert;
    const int32_t *mtile_first_row;
    const int32_t *mtile_valid;
    const __nv_bfloat16 *hidden;   // [T, H]
    const int32_t *perm;           // flat assignment of every routed row
    const int32_t *S_dev;          // != nullptr: the m-tile count is read here
    InlineRouting routing;         // topk_idx != nullptr: this launch builds the routing first (one-CTA tiles)
    int32_t tile_m;
    __nv_bfloat16 *x_routed;       // [R, I]
    uint32_t *status;
    unsigned long long wait_ns;
    int32_t S;                     // m-tiles of the routing workspace (or their bound with S_dev)
    int32_t T, k_tot, H;
    Divisor by_k, by_NT, by_slots;   // k_tot, NT, CTAs (pairs) of the launch
    int32_t I, NT;                 // intermediate size, n-tiles = ceil(I / tile columns)
    int32_t num_kb, last_ksteps;
    int32_t w1_once;               // W1 is read (about) once: its lines go first when L2 needs room
    unsigned long long *mail;      // != nullptr: the tile counts (S_dev - E_tot) are mailed to the host by this launch
    uint32_t mail_seq;
    int32_t E_tot;
};

struct G1Control {
    unsigned long long full[kG1MaxStages];
    unsigned long long empty[kG1MaxStages];
    unsigned long long rows[kG1MaxStages];    // every loader thread's copies of the stage have landed
    unsigned long long tmem_full[2];
    unsigned long long tmem_empty[2];
    uint32_t tmem_base;
    volatile uint32_t abort;
    volatile uint32_t tile_n[8];              // N of a tile's MMAs (tile number mod 8), from the W1 producer to the MMA issuer
};
static_assert(kG1MaxStages < 8, "a place in tile_n may be written again while its tile is still to be issued");

template <bool kCluster = false>   // kCluster: what the other CTA of the pair released
__device__ __forceinline__ bool g1_wait(uint32_t bar, uint32_t parity, G1Control *ctl, unsigned long long deadline,
                                        uint32_t *status, uint32_t detail, uint32_t where)
{
    uint32_t spins = 0;
    while (!(kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity))) {
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
__device__ __forceinline__ bool g1_wait_warp(uint32_t bar, uint32_t parity, G1Control *ctl, unsigned long long deadline,
                                             uint32_t *status, uint32_t detail, uint32_t where)
{
    uint32_t ok = 1u;
    if ((threadIdx.x & 31u) == 0u) ok = g1_wait(bar, parity, ctl, deadline, status, detail, where) ? 1u : 0u;
    return __shfl_sync(0xffffffffu, ok, 0) != 0u;
}

// silu(z) = z / silu_divisor(z).  The quotient is the division operator's, correctly rounded: what is left of the error is __expf's.
__device__ __forceinline__ float silu_divisor(float z) { return 1.0f + __expf(-z); }

struct G1Tile {
    int e, row0, valid, n0;   // valid: rows of the whole m-tile (up to 256 for a pair tile)
};
// tile g of the sequence: m-tile outer, n-tile inner
template <int TN>
__device__ __forceinline__ G1Tile g1_decode(int g, const G1Params &P)
{
    const int mu = quotient(P.by_NT, g);
    G1Tile t;
    t.e = ld_chained(&P.mtile_expert[mu]);
    t.row0 = ld_chained(&P.mtile_first_row[mu]);
    t.valid = ld_chained(&P.mtile_valid[mu]);
    t.n0 = (g - mu * P.NT) * TN;
    return t;
}
// N of a tile's MMAs: its rows, rounded up to what the instruction takes (M = 128: 16, M = 256 over a pair: 32)
template <bool kPair>
__device__ __forceinline__ int g1_mma_n(int valid) { return kPair ? (valid + 31) & ~31 : (valid + 15) & ~15; }
// flat assignments of the rows this loader thread copies (step i of the stage: row 16 i + `first` of this CTA's)
template <bool kPair>
__device__ __forceinline__ void g1_load_perm(const G1Params &P, const G1Tile &t, uint32_t rank, int first, int (&f)[kMmaM / kG1RowsPerStep])
{
    const int held = kPair ? g1_mma_n<kPair>(t.valid) >> 1 : kMmaM, row0 = (int)rank * held, rows = min(held, t.valid - row0);
#pragma unroll
    for (int i = 0; i < kMmaM / kG1RowsPerStep; ++i) {
        const int r = kG1RowsPerStep * i + first;
        f[i] = r < rows ? ld_chained(&P.perm[t.row0 + row0 + r]) : -1;
    }
}

// --------------------------------------------------------------------------- GEMM1 + activation

template <bool kPair, int TN>
__global__ void __launch_bounds__(kThreads, 1)
moe_gemm1_act_kernel(const __grid_constant__ G1Params P)
{
    using C = G1Cfg<kPair, TN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    G1Control *ctl = reinterpret_cast<G1Control *>(ring + C::kRingBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = kPair ? cluster_ctarank() : 0u;
    // tiles are dealt to the CTAs, or to the pairs
    int b = kPair ? (int)blockIdx.x >> 1 : (int)blockIdx.x, stride = kPair ? (int)gridDim.x >> 1 : (int)gridDim.x;

    if (threadIdx.x == 0) {
        for (int i = 0; i < C::kStages; ++i) {
            mbar_init(smem_u32(&ctl->full[i]), kPair ? 3 : 2);   // the W1 producer and the relay of every CTA
            mbar_init(smem_u32(&ctl->empty[i]), 1);
            mbar_init(smem_u32(&ctl->rows[i]), 32 * kG1LoadWarps);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&ctl->tmem_full[i]), 1);
            mbar_init(smem_u32(&ctl->tmem_empty[i]), (kPair ? 2 : 1) * kG1EpiWarps);
        }
        ctl->abort = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        prefetch_tensormap(&P.tmW);
    }
    if (warp == 1) {
        if (kPair) tmem_alloc_pair(smem_u32(&ctl->tmem_base), C::kTmemCols);
        else tmem_alloc(smem_u32(&ctl->tmem_base), C::kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    if (kPair) cluster_sync_all();     // the peer's barriers exist before anything arrives on them
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    grid_dependency_wait();
    if (!kPair && P.routing.topk_idx)
        routing_inline<kThreads / 32, false>(P.routing, P.k_tot, P.E_tot, P.tile_m, P.status, P.mail, P.mail_seq, reinterpret_cast<int32_t *>(ring));
    const int S = P.S_dev ? min(ld_chained_uniform(P.S_dev), P.S) : P.S;
    const int total_tiles = S * P.NT;
    {
        // as many waves as all CTAs need, over as few CTAs as then suffice: with all of them the same waves take longer, each
        // tile's share of the memory bandwidth being smaller (stage alone: Granite shape T = 16 30.7 -> 28.0 us, T = 400 32.5 -> 30.6,
        // DeepSeek shape T = 300 145.9 -> 140.8, Qwen shape T = 512 122.3 -> 118.1; large batches equal)
        const int waves = max(1, quotient(P.by_slots, total_tiles + stride - 1));
        stride = max(1, small_quotient(total_tiles + waves - 1, waves));
        if (b >= stride) b = total_tiles;
    }
    const unsigned long long deadline = globaltimer_ns() + P.wait_ns;

    if (P.mail && (kPair || !P.routing.topk_idx) && blockIdx.x == 0 && warp == 3)
        mail_counts(P.mail, P.mail_seq, P.E_tot, lane, [&](int x) { return ld_chained(P.S_dev - P.E_tot + x); });
    if (warp == 0) {
        // ---------------- W1 producer.  Pair: everything completes on the leader's full barrier, armed by the leader for both
        // CTAs.
        if (lane == 0 && b < total_tiles) {
            int stage = 0;
            uint32_t phase = 0, armed = 0;
            bool ok = true;
            const unsigned long long w_policy = P.w1_once ? l2_evict_first_policy() : l2_evict_normal_policy();
            G1Tile t = g1_decode<TN>(b, P);
            int it = 0;
            for (int g = b; g < total_tiles && ok; g += stride, ++it) {
                const G1Tile t_next = g1_decode<TN>(min(g + stride, total_tiles - 1), P);   // fetched one tile ahead
                const int group = t.n0 / 16 + (kPair ? (int)rank * (TN / 32) : 0);
                int kx = 0;
                for (int kb = 0; kb < P.num_kb; ++kb, kx += kBlockK) {
                    ok = g1_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, ctl, deadline, P.status, (uint32_t)g, 50u);
                    if (!ok) break;
                    const uint32_t own_full = smem_u32(&ctl->full[stage]);
                    const uint32_t w_dst = smem_u32(ring + stage * C::kStageBytes);
                    if (kb == 0 && rank == 0) ctl->tile_n[it & 7] = (uint32_t)g1_mma_n<kPair>(t.valid);
                    if (rank == 0) mbar_arrive_expect_tx(own_full, (kPair ? 2u : 1u) * (uint32_t)C::kWBytes);
                    // (pair: the barrier lies at the same offset in the leader CTA, rank 0)
                    if (kPair) tma_load_5d_pair(w_dst, &P.tmW, own_full & 0xFEFFFFFFu, kx, 0, 0, group, t.e);
                    else tma_load_5d_hint(w_dst, &P.tmW, own_full, kx, 0, 0, group, t.e, w_policy);
                    armed |= 1u << stage;
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                }
                t = t_next;
            }
            if (!ok && rank == 0) {
                // wind-down: let the copies already issued land before shared memory is released
                const unsigned long long drain = globaltimer_ns() + 2000000ull;
                for (int sidx = 0; sidx < C::kStages; ++sidx) {
                    if (!(armed & (1u << sidx))) continue;
                    const uint32_t par = (sidx < stage) ? phase : (phase ^ 1u);
                    while (!mbar_try_wait(smem_u32(&ctl->full[sidx]), par) && globaltimer_ns() < drain) {}
                }
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------- relay: rows landed -> visible to the tensor core's (async) proxy -> full barrier.  Pair: the other CTA's
        // relay hands its rows to the leader's MMA issuer, release to acquire at cluster scope.  (With an unrestricted
        // release: 1500-1900 cycles later per stage, stage alone, Granite shape T = 1003 46 -> 57 us, Qwen shape T = 2880
        // 159 -> 190.  By way of the leader's relay, one barrier more: whole layer, DeepSeek shape T = 16384, +0.5 %.)
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int g = b; g < total_tiles && ok; g += stride) {
                for (int kb = 0; kb < P.num_kb; ++kb) {
                    ok = g1_wait(smem_u32(&ctl->rows[stage]), phase, ctl, deadline, P.status, (uint32_t)g, 54u);
                    if (!ok) break;
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    if (rank != 0) mbar_arrive_cluster_release_shared(mapa_u32(smem_u32(&ctl->full[stage]), 0u));
                    else mbar_arrive(smem_u32(&ctl->full[stage]));
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else if (warp >= 4 + kG1EpiWarps) {
        // ---------------- loaders: thread = one 16-byte column chunk of every 16th row
        constexpr int kSteps = kMmaM / kG1RowsPerStep;
        const int chunk = lane & 7, first = (warp - 4 - kG1EpiWarps) * 4 + (lane >> 3);
        const uint32_t dst0 = (uint32_t)first * 128u + (uint32_t)((chunk ^ (first & 7)) << 4);   // 128B swizzle; 16 rows on: + 2048
        if (b < total_tiles) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            // where this thread's chunk of its rows begins (nullptr: the tile has no such row)
            const auto rows_of = [&](const int (&f)[kSteps], const __nv_bfloat16 *(&src)[kSteps]) {
#pragma unroll
                for (int i = 0; i < kSteps; ++i)
                    src[i] = f[i] >= 0 ? P.hidden + (size_t)min(quotient(P.by_k, f[i]), P.T - 1) * (size_t)P.H + chunk * 8 : nullptr;
            };
            G1Tile t_next = g1_decode<TN>(min(b + stride, total_tiles - 1), P);
            int f_next[kSteps];
            const __nv_bfloat16 *src[kSteps], *src_next[kSteps];
            g1_load_perm<kPair>(P, g1_decode<TN>(b, P), rank, first, f_next);
            rows_of(f_next, src);
            for (int g = b; g < total_tiles && ok; g += stride) {
                // Fetched ahead: the table entries two tiles, the rows' assignments one tile; their addresses (a division each) are
                // worked out between two k-blocks, so that nothing but copies stands between the last k-block of a tile and
                // the first of the next.  The way from a freed stage to its next rows is the longest of the ring: with the
                // divisions at the head of the tile and a test per row in every k-block the stage took 1270 us at the DeepSeek
                // shape T = 16384, now 1177 (20 more instructions a k-block for something else: 1400).
                const G1Tile t_nn = g1_decode<TN>(min(g + 2 * stride, total_tiles - 1), P);
                g1_load_perm<kPair>(P, t_next, rank, first, f_next);
                bool whole = true;               // the tile has all rows of this warp
#pragma unroll
                for (int i = 0; i < kSteps; ++i) whole = whole && src[i] != nullptr;
                whole = __all_sync(0xffffffffu, whole);
                const int ahead_at = min(4, P.num_kb - 1);
                int left = P.H - chunk * 8;      // columns from this chunk on
                for (int kb = 0; kb < P.num_kb; ++kb, left -= kBlockK) {
                    if (!mbar_test_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u))
                        ok = g1_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, ctl, deadline, P.status, (uint32_t)g, 55u);
                    if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                    const uint32_t dst = smem_u32(ring + stage * C::kStageBytes) + (uint32_t)C::kWBytes + dst0;
                    if (left > 0) {              // (past the last column: no MMA reads it)
                        if (whole) {
#pragma unroll
                            for (int i = 0; i < kSteps; ++i) cp_async_16(dst + (uint32_t)(i * kG1RowsPerStep * 128), src[i] + kb * kBlockK);
                        } else {
#pragma unroll
                            for (int i = 0; i < kSteps; ++i)
                                if (src[i]) cp_async_16(dst + (uint32_t)(i * kG1RowsPerStep * 128), src[i] + kb * kBlockK);
                        }
                    }
                    cp_async_arrive(smem_u32(&ctl->rows[stage]));
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                    if (kb == ahead_at) rows_of(f_next, src_next);
                }
                t_next = t_nn;
#pragma unroll
                for (int i = 0; i < kSteps; ++i) src[i] = src_next[i];
            }
            cp_async_wait_all();
        }
        __syncwarp();
    } else if (warp == 1 && rank == 0) {
        // ---------------- MMA issuer (pair: the leader CTA): the whole warp runs the loop, converged, and one elected lane
        // issues.  tcgen05.mma takes its descriptors and addresses from uniform registers, and the tensor pipe buffers
        // little ahead of the MMA it executes: warp-uniform values in warp-uniform control flow spare a move per
        // operand and MMA, a whole k-block (four MMAs and the commit) is one statement with 32-bit descriptor
        // arithmetic, addresses advance by additions, the barrier's first look is the non-suspending test.
        {
            constexpr uint32_t kLoStage = (uint32_t)(C::kStageBytes >> 4), kLoX = (uint32_t)(C::kWBytes >> 4);
            constexpr uint32_t kLoBlock = (uint32_t)(kMmaM * kBlockK * 2 >> 4);      // the next 128 rows of W1: 64 columns
            constexpr int kFullN = kPair ? 2 * kMmaM : kMmaM;
            const uint32_t lo0 = smem_desc_lo(smem_u32(ring));
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            uint32_t w_lo = lo0, full_bar = full0, empty_bar = empty0;
            int stage = 0, it = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int g = b; g < total_tiles && ok; g += stride, ++it) {
                const int a = it & 1;
                const uint32_t acc_parity = ((uint32_t)(it >> 1) & 1u) ^ 1u;
                if (!__all_sync(0xffffffffu, mbar_test_wait(smem_u32(&ctl->tmem_empty[a]), acc_parity))) {
                    // (every lane polls; the vote keeps `ok`, and with it the loop, provably warp-uniform)
                    ok = __all_sync(0xffffffffu, g1_wait(smem_u32(&ctl->tmem_empty[a]), acc_parity, ctl, deadline, P.status, (uint32_t)g, 51u));
                    if (!ok) break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(a * C::kAccCols);
                const auto wait_stage = [&]() {
                    if (__all_sync(0xffffffffu, kPair ? mbar_test_wait_cluster(full_bar, phase) : mbar_test_wait(full_bar, phase))) return;
                    ok = __all_sync(0xffffffffu, g1_wait<kPair>(full_bar, phase, ctl, deadline, P.status, (uint32_t)g, 52u));
                };
                const auto kloop = [&](auto full, uint32_t n) {
                    const uint32_t idesc = make_idesc(kPair ? 2 * kMmaM : kMmaM, decltype(full)::value ? kFullN : (int)n);
                    for (int kb = 0; kb < P.num_kb; ++kb) {
                        wait_stage();
                        if (!ok) break;
                        tc_fence_after();
                        if (elect_one_sync()) {
                            if (kb < P.num_kb - 1 || P.last_ksteps == kBlockK / kUmmaK) {
                                if (C::kBlocks == 2) tc_ksteps_bf16(d_tmem + kMmaM, w_lo + kLoBlock, w_lo + kLoX, idesc, kb > 0 ? 1u : 0u);
                                if (kPair) tc_kblock_bf16_pair(d_tmem, w_lo, w_lo + kLoX, idesc, kb > 0 ? 1u : 0u, empty_bar);
                                else tc_kblock_bf16(d_tmem, w_lo, w_lo + kLoX, idesc, kb > 0 ? 1u : 0u, empty_bar);
                            } else {
                                const uint64_t w_desc = ((uint64_t)kSmemDescHi << 32) | w_lo, x_desc = w_desc + kLoX;
                                for (int k = 0; k < P.last_ksteps; ++k) {
                                    const uint32_t acc = (k > 0 || kb > 0) ? 1u : 0u;
                                    for (int i = 0; i < C::kBlocks; ++i) {
                                        const uint64_t wd = w_desc + (uint64_t)(2 * k + i * (int)kLoBlock), xd = x_desc + (uint64_t)(2 * k);
                                        if (kPair) tc_mma_bf16_pair(d_tmem, wd, xd, idesc, acc);
                                        else tc_mma_bf16(d_tmem + (uint32_t)(i * kMmaM), wd, xd, idesc, acc);
                                    }
                                }
                                if (kPair) tc_commit_pair(empty_bar);
                                else tc_commit(empty_bar);
                            }
                        }
                        w_lo += kLoStage;
                        full_bar += 8u;
                        empty_bar += 8u;
                        if (++stage == C::kStages) {
                            stage = 0;
                            phase ^= 1u;
                            w_lo = lo0;
                            full_bar = full0;
                            empty_bar = empty0;
                        }
                    }
                };
                // the producer knows the tile's rows; looked up here, the table entry is a load in the issuer's way.  Full tiles of a
                // pair in a loop of their own, with a constant N, as in the fused kernel.
                wait_stage();
                if (!ok) break;
                const uint32_t n = ctl->tile_n[it & 7];
                if (kPair && __all_sync(0xffffffffu, n == (uint32_t)kFullN)) kloop(std::true_type{}, 0u);
                else kloop(std::false_type{}, __reduce_max_sync(0xffffffffu, n));
                __syncwarp();
                if (ok && elect_one_sync()) {
                    if (kPair) tc_commit_pair(smem_u32(&ctl->tmem_full[a]));
                    else tc_commit(smem_u32(&ctl->tmem_full[a]));
                }
            }
        }
        __syncwarp();
    } else if (warp >= 4 && warp < 4 + kG1EpiWarps) {
        // ---------------- epilogue: pieces of 32 rows x 16 columns (this warp's lane quarter), dealt over the two groups of warps.
        // Every division is a branch (its slow path), so a lane's divisions run one after the other: where a launch is
        // one wave, that chain is its tail.  It holds nothing but the divisions, and those of eights of rows that the tile has.
        const int q4 = warp & 3, grp = (warp - 4) >> 2, c = lane & 3;
        int it = 0;
        for (int g = b; g < total_tiles; g += stride, ++it) {
            const G1Tile t = g1_decode<TN>(g, P);
            const int a = it & 1, pieces = ((t.valid + 31) >> 5) * C::kBlocks;
            const bool ok = g1_wait_warp(smem_u32(&ctl->tmem_full[a]), (uint32_t)(it >> 1) & 1u, ctl, deadline, P.status,
                                         (uint32_t)g, 53u);
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(a * C::kAccCols);
            const auto release = [&]() {
                // everything this warp needs of the accumulator is in registers: hand the buffer back
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (kPair) mbar_arrive_cluster_relaxed(mapa_u32(smem_u32(&ctl->tmem_empty[a]), 0u));   // the leader's barrier
                    else mbar_arrive(smem_u32(&ctl->tmem_empty[a]));
                }
            };
            if (grp >= pieces) release();
#pragma unroll 1
            for (int piece = grp; piece < pieces; piece += kG1EpiWarps / 4) {
                const int chunk = piece / C::kBlocks, block = piece % C::kBlocks;
                const int col = (kPair ? (int)rank : block) * (kMmaM / 2) + q4 * 16;      // first column, inside the tile
                const bool live = col < TN && t.n0 + col < P.I;
                uint32_t gt[16], up[16];
                if (live) {
                    tmem_ld_16x256_x4(taddr + (uint32_t)(block * kMmaM + chunk * 32), gt);
                    tmem_ld_16x256_x4(taddr + (16u << 16) + (uint32_t)(block * kMmaM + chunk * 32), up);
                    tmem_ld_wait(gt);
                    tmem_ld_wait(up);
                }
                if (piece + kG1EpiWarps / 4 >= pieces) release();
                if (!live) continue;
                const int rows = t.valid - chunk * 32;
                // registers 4j..4j+3: rows 8j + 2c and the next one, of columns lane / 4 (4j, 4j + 1) and 8 + lane / 4
                float d[16];
                uint32_t w[8];
#pragma unroll
                for (int i = 0; i < 16; ++i) d[i] = silu_divisor(__uint_as_float(gt[i]));
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    w[j] = w[4 + j] = 0u;
                    if (8 * j >= rows) continue;
                    float y[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) y[i] = __uint_as_float(gt[4 * j + i]) / d[4 * j + i] * __uint_as_float(up[4 * j + i]);
                    w[j] = transpose_8x8(pack_bf16(__float_as_uint(y[0]), __float_as_uint(y[1])));
                    w[4 + j] = transpose_8x8(pack_bf16(__float_as_uint(y[2]), __float_as_uint(y[3])));
                }
                // w[j], w[4 + j]: columns 2c and 8 + 2c and the next ones of row 8j + lane / 4 -> all 16 columns of row 8c + lane / 4
#pragma unroll
                for (int x = 1; x < 4; x *= 2)
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        if (m & x) continue;
                        const bool hi = (c & x) != 0;
                        const uint32_t got = __shfl_xor_sync(0xffffffffu, hi ? w[m] : w[m + x], x);
                        if (hi) w[m] = got;
                        else w[m + x] = got;
                    }
                const int row = 8 * c + (lane >> 2);
                if (row < rows) st_global_v8(P.x_routed + (size_t)(t.row0 + chunk * 32 + row) * (size_t)P.I + t.n0 + col, w);
            }
        }
    }
    // ---------------- teardown (pair: nobody leaves while its peer may still touch its memory)
    tc_fence_before();
    __syncthreads();
    if (kPair) cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        if (kPair) tmem_dealloc_pair(tmem_base, C::kTmemCols);
        else tmem_dealloc(tmem_base, C::kTmemCols);
    }
}

template <bool kPair, int TN>
constexpr size_t g1_smem_bytes() { return (size_t)G1Cfg<kPair, TN>::kRingBytes + 1024 + ((sizeof(G1Control) + 127) & ~(size_t)127); }
static_assert(g1_smem_bytes<true, 128>() <= 227 * 1024 && g1_smem_bytes<false, 64>() <= 227 * 1024 && g1_smem_bytes<false, 96>() <= 227 * 1024, "GEMM1 stages exceed the shared memory of an SM");

inline bool aligned(const void *p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

}  // namespace
}  // namespace moe

using namespace moe;

cudaError_t moe::gemm1_prepare()
{
    cudaError_t e = cudaFuncSetAttribute(moe_gemm1_act_kernel<false, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g1_smem_bytes<false, 64>());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(moe_gemm1_act_kernel<false, 96>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g1_smem_bytes<false, 96>());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(moe_gemm1_act_kernel<false, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g1_smem_bytes<false, 128>());
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(moe_gemm1_act_kernel<true, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g1_smem_bytes<true, 128>());
}

extern "C" int32_t moe_gemm1_workspace_bytes(const moe_shape *s, size_t *h_routed_bytes)
{
    if (!s || !h_routed_bytes) return MOE_ERR_NULL;
    if (s->T < 0 || s->k_tot < 1 || s->H < 1) return MOE_ERR_SHAPE;
    *h_routed_bytes = (((size_t)s->T * s->k_tot * s->H * 2) + 15) / 16 * 16 + 16;
    return MOE_OK;
}

extern "C" int32_t moe_gemm1_act(moe_handle *h, const void *hidden, const void *W1, const moe_shape *s,
                                 int32_t tile_m, const moe_routing *r, int32_t n_mtiles, void *h_routed_ws,
                                 void *x_routed, uint32_t *status_dev, void *stream)
{
    return launch_gemm1_act(h, hidden, W1, nullptr, s, tile_m, r, n_mtiles, h_routed_ws, x_routed, status_dev, 0u, stream);
}

int32_t moe::launch_gemm1_act(moe_handle *h, const void *hidden, const void *W1, const int32_t *topk_idx, const moe_shape *s,
                              int32_t tile_m, const moe_routing *r, int32_t n_mtiles, void *h_routed_ws, void *x_routed, uint32_t *status_dev,
                              uint32_t mail_seq, void *stream)
{
    if (!h || !s || !r || !status_dev) return MOE_ERR_NULL;
    if (s->T < 0 || s->H < 64 || s->H % 16 != 0 || s->I < 16 || s->I % 16 != 0 || s->E_tot < 1 || s->k_tot < 1 ||
        (int64_t)s->T * s->k_tot >= (int64_t)1 << 30)
        return MOE_ERR_SHAPE;
    if (tile_m != 64 && tile_m != 128 && tile_m != 256) return MOE_ERR_UNSUPPORTED;
    if (s->T == 0) return MOE_OK;
    if (!hidden || !W1 || !h_routed_ws || !x_routed) return MOE_ERR_NULL;
    if (!aligned(hidden, 16) || !aligned(W1, 16) || !aligned(h_routed_ws, 16) || !aligned(x_routed, 32) ||
        !aligned(status_dev, 16))
        return MOE_ERR_ALIGN;
    const bool counts_on_device = (n_mtiles == MOE_MTILES_ON_DEVICE);
    if (counts_on_device) n_mtiles = r->max_mtiles;
    if (n_mtiles < 0 || n_mtiles > r->max_mtiles) return MOE_ERR_SHAPE;
    if (const int32_t rc = moe::require_handle_device(h, "moe_gemm1_act")) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    G1Params p;
    memset(&p, 0, sizeof p);
    p.mtile_expert = r->mtile_expert;
    p.mtile_first_row = r->mtile_first_row;
    p.mtile_valid = r->mtile_valid;
    p.S_dev = counts_on_device ? r->tiles + s->E_tot : nullptr;
    p.x_routed = static_cast<__nv_bfloat16 *>(x_routed);
    p.status = status_dev;
    p.wait_ns = h->wait_ns;
    p.S = n_mtiles;
    if (mail_seq != 0u && counts_on_device) {
        p.mail = h->mail_dev;
        p.mail_seq = mail_seq;
    }
    p.E_tot = s->E_tot;
    p.tile_m = tile_m;
    if (topk_idx) p.routing = {topk_idx, routing_out(*r), s->T * s->k_tot, r->max_mtiles};
    p.perm = r->perm;
    p.hidden = static_cast<const __nv_bfloat16 *>(hidden);
    p.T = s->T;
    p.H = s->H;
    p.k_tot = s->k_tot;
    p.I = s->I;
    const bool pair = tile_m == 256;
    // Narrow tiles where every one that this routing can have then still finds an SM of its own: the time of the only wave is the
    // time to stream one tile's weights (Granite shape, T = 2, 64 columns: 14.6 -> 12.7 us; DeepSeek shape, T = 1, 96 columns: 20.4
    // -> 18.8).  With more tiles than SMs the wide ones are faster at every size (64 columns: +1 to +8 % over a layer).
    int TN = kG1TileN;
    if (!pair) {
        const int64_t R = (int64_t)s->T * s->k_tot, used = R < s->E_tot ? R : s->E_tot, bound = (R - used) / tile_m + used;
        const int64_t S_max = counts_on_device && bound < n_mtiles ? bound : n_mtiles;
        for (int tn = 64; tn < kG1TileN && TN == kG1TileN; tn += 32)
            if (S_max * ((s->I + tn - 1) / tn) <= h->G) TN = tn;
    }
    p.NT = (s->I + TN - 1) / TN;
    p.num_kb = (s->H + kBlockK - 1) / kBlockK;
    p.w1_once = (int64_t)s->T * s->k_tot <= (int64_t)s->E_tot * kMmaM;   // at most one 128-row tile per expert on average
    p.last_ksteps = (s->H - (p.num_kb - 1) * kBlockK) / kUmmaK;
    if ((int64_t)n_mtiles * p.NT >= (int64_t)1 << 31) return MOE_ERR_SHAPE;

    // columns past I read zeros
    const CUtensorMap *mW = gate_up_map(h, W1, s->E_tot, s->I, s->H, pair ? TN / 2 : TN, "W1");
    if (!mW) return MOE_ERR_CUDA;
    p.tmW = *mW;

    const int64_t tiles_bound = (int64_t)n_mtiles * p.NT;
    const int slots = pair ? h->max_pairs : h->G;
    const int used = (int)(tiles_bound < slots ? (tiles_bound > 0 ? tiles_bound : 1) : slots);
    p.by_k = divisor_of(s->k_tot);
    p.by_NT = divisor_of(p.NT);
    p.by_slots = divisor_of(used);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2] = {chained_launch_attribute()};
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pair ? 2 : 1;
    cfg.stream = st;
    cfg.gridDim = dim3((unsigned)(pair ? 2 * used : used));
    cfg.blockDim = dim3(kThreads);
    cudaError_t e;
    if (pair) {
        cfg.dynamicSmemBytes = g1_smem_bytes<true, 128>();
        e = cudaLaunchKernelEx(&cfg, moe_gemm1_act_kernel<true, 128>, p);
    } else if (TN == 64) {
        cfg.dynamicSmemBytes = g1_smem_bytes<false, 64>();
        e = cudaLaunchKernelEx(&cfg, moe_gemm1_act_kernel<false, 64>, p);
    } else if (TN == 96) {
        cfg.dynamicSmemBytes = g1_smem_bytes<false, 96>();
        e = cudaLaunchKernelEx(&cfg, moe_gemm1_act_kernel<false, 96>, p);
    } else {
        cfg.dynamicSmemBytes = g1_smem_bytes<false, 128>();
        e = cudaLaunchKernelEx(&cfg, moe_gemm1_act_kernel<false, 128>, p);
    }
    if (e != cudaSuccess) return cuda_fail(h, e, "gemm1 launch");
    return MOE_OK;
}
