// Internal declarations shared by the translation units of libmoe_b200.so.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <cstring>
#include <unordered_map>

#include "../../include/moe_b200.h"

namespace moe {

constexpr int kThreads = 512;          // threads of a CTA's compute (or dedicated communication) role: 16 warps
constexpr int kCoWarpsMax = 4;         // co-resident communication warps a compute CTA of the fused kernel may carry
constexpr int kFusedThreads = kThreads + 32 * kCoWarpsMax;   // block size of the fused kernel
constexpr int kBlockK = 64;            // bf16 elements per k-block: one 128-byte swizzle row
constexpr int kUmmaK = 16;             // K of one tcgen05.mma.kind::f16 instruction
constexpr int kMmaM = 128;             // M of a one-CTA MMA: output columns (a pair's: twice that); also the rows of a one-CTA tile
constexpr int kStageBytesTotal = 192 * 1024;  // operand ring, all stages together
constexpr int kCommTileM = 32;         // T_M^comm: the piece in which the selector counts communication work (a CTA's units are 8 KB)
constexpr int kCommTileN = 1024;       // T_N^comm
constexpr int kMailWords = 1024 + 1 + 31;   // the handle's count mailbox: one (count, sequence number) word per expert, then S
constexpr int kPlanTableMax = 256;     // m-tile counts a tabulated selection may span (a shape has E_tot + 1 or fewer)
constexpr int kRoutingChunk = 256;     // flat assignments handled by one warp while sorting
constexpr uint64_t kDefaultWaitNs = 2000000000ull;
constexpr int kTimelineSlots = 40;     // 64-bit words per CTA in a timeline buffer (timeline build only)

// the routing arrays as the kernels write them
struct RoutingOut {
    int32_t *counts, *offsets, *tiles, *tile_offsets, *mtile_expert, *mtile_first_row, *mtile_valid, *perm, *inv_perm, *pad_row;
};

// division by a number that the host knows, as a multiplication (quotient())
struct Divisor {
    uint32_t mul, shift;
};
// routing build inside a kernel that uses it (topk_idx = nullptr: the arrays are there already)
struct InlineRouting {
    const int32_t *topk_idx;
    RoutingOut out;
    int32_t R, max_mtiles;
};
constexpr int kInlineMaxR = 2048;      // assignments up to which a kernel builds the routing itself: four rows of 32 per warp of 16 warps

// Parameters of one fused launch.  Passed by value (__grid_constant__): the tensor maps
// must sit in kernel parameter space, 64-byte aligned.
struct alignas(64) FusedParams {
    CUtensorMap tmA, tmA64, tmA32;   // x_routed [R, I]   boxes 64 x 128, 64 and (one-CTA tiles) 32 rows, 128B swizzle
    CUtensorMap tmB;   // W2 [E_tot, H, I]     box 64 x tile_n rows (a pair's CTA: half of them) x 1, 128B swizzle
    const int32_t *mtile_expert;
    const int32_t *mtile_first_row;
    const int32_t *mtile_valid;
    InlineRouting routing;         // topk_idx != nullptr: this launch builds the routing first
    const int32_t *S_dev;          // != nullptr: the m-tile count is read here by the kernel (S and W_comp below are unset)
    const int32_t *pad_row;
    const int32_t *perm;
    const float *topk_w;
    void *Y;                       // bf16 [T][L][slabs][k_tot][slab cols], token-major
    uint32_t *flags;               // [L * W_comp] readiness per global tile (== epoch when ready)
    uint32_t *split_done;          // [L] tiles finished per split (this launch)
    uint32_t *split_done_next;     // [L] counters of the next launch, zeroed by this one
    unsigned long long *queue;     // [L] drain help: items of the split handed out so far, front | back << 32
    unsigned long long *queue_next;  // [L] ... of the next launch, zeroed by this one
    uint32_t *status;              // 4 words
    unsigned long long *timeline;  // timeline build: per-CTA records, then one stamp per split; else nullptr
    uint32_t probe;                // timeline build: parts of the data movement left out (moe_set_probe); else 0
    void *out[MOE_MAX_EP];
    unsigned long long wait_ns;
    long long R_pad;
    int32_t T, H, EP, L, k_tot;
    int32_t S, tile_m, NTs, split_w, W_comp;
    int32_t C, P, mode, withhold;
    unsigned long long *mail;           // != nullptr: the tile counts (S_dev - E_tot) are mailed to the host by this launch
    uint32_t mail_seq;
    int32_t E_tot;
    int32_t G, slot_sms;                // c_table: SMs the partition is made of, SMs of one compute slot
    int32_t c_table_first, c_table_n;   // c_table[i]: communication CTAs when S = c_table_first + i (0 entries: C and P above hold)
    uint8_t c_table[kPlanTableMax];
    int32_t tok_blk, comm_cols;
    Divisor by_k;                       // k_tot: flat assignment -> token
    int32_t even;                       // the communication work is dealt evenly to all warps once all tiles are done (no per-tile
                                        // flags, no queue)
    int32_t balance;                    // (even) P counts all compute slots; the kernel divides them by whole waves of its tiles
    const uint32_t *x_ready;            // != nullptr: x_routed is still being copied in; the rows that have arrived
    int32_t w2_once;                    // W2 is read (about) once: its lines go first when L2 needs room
    int32_t num_kb, last_ksteps;
    int32_t dry_rows;                   // rows of a tile as they are to be expected, for the dry round (pair kernel)
    int32_t drain_help;                 // compute CTAs serve communication tiles once their GEMM tiles are done
    int32_t co_warps;                   // co-resident communication warps per compute CTA (0..2)
    int32_t x_rows;                     // the most rows that a CTA can hold of an m-tile of the launch, rounded up to a copy's 32 (one-CTA tiles), 64 or 128
    int32_t stages, stage_bytes;        // operand stages of a compute CTA: as many as fit the ring; a pair's has one more where the aux
                                        // region of shared memory is free during the GEMM (no co-resident warp)
    int32_t epi_warps;                  // epilogue warps of a compute CTA: 12 (warps 4-15), or 16 (warps 4-19) when no
                                        // co-resident warp is asked for
    int32_t tile_order;                 // 0: split-major tile sequence (the paper's); 1: m-tile-major across splits
    int32_t flag_parts;                 // readiness flags per tile: 1, or 2 for a CTA-pair tile
    int32_t slab_cols, slab_shift;      // slab_cols = 1 << slab_shift; a unit is k_tot rows of a slab
    uint32_t epoch;
};

}  // namespace moe

namespace moe {
// An operand tensor map (bf16, k contiguous, 64 x box_rows boxes, 128B swizzle) and what it was encoded for: [rows, cols], or
// [planes, rows, cols], or gate and up planes of `-planes` experts.  The handle keeps the maps of the operands that it has
// seen (a model's layers, the buffers of a loop of steps) in a small direct-mapped table: encoding one takes 0.07 us of a call's 5 on the host.
struct alignas(64) MapEntry {
    CUtensorMap map;
    const void *ptr;
    int64_t rows;
    int32_t cols, planes, box_rows;
};
constexpr int kMapEntries = 128;
// The place of an operand's map.  The maps of one operand for different boxes (32 to 256 rows: steps of 32) lie in places of their own, and
// so do those of two operands that are a power of two of bytes apart, as buffers out of one allocation are (with the rows added to the
// address instead, the 128-row box of one buffer and the 64-row box of another 16 KB behind it pushed each other out on every call).
inline uint32_t map_place(const void *ptr, int32_t box_rows)
{
    const uint64_t mixed = (uint64_t)(reinterpret_cast<uintptr_t>(ptr) >> 8) * 0x9E3779B97F4A7C15ull;
    return ((uint32_t)(mixed >> 57) + (uint32_t)box_rows / 32u) & (uint32_t)(kMapEntries - 1);
}
static_assert(kMapEntries == 1 << (64 - 57), "the hash's upper bits index the table");
// x_routed of a launch that starts while the rows are still being copied in (host-buffer entry point)
struct RowFeed {
    const uint32_t *ready;         // [device] rows that have arrived, written behind each copy
    uint64_t extra_wait_ns;        // what the copies may add to the kernel's wait limit
};
// The selector's pick for every m-tile count S that a routing of one shape can have: plan_partition depends on the
// routed counts through their sum alone (but for tile-level readiness, which is not tabulated).
struct PlanTable {
    moe_shape shape;
    int32_t tile_m, tile_n;
    moe_sm_limits limits;
    int32_t first, n;              // S = first .. first + n - 1; n = 0: not to be tabulated; n < 0: not made yet
    bool again;                    // not the first call with this selection: worth tabulating
    uint64_t last_use;             // number of the last call with it (0: entry unused)
    moe_plan plan;                 // what all picks have in common, and the pick for `first`
    uint8_t C[kPlanTableMax];
};
constexpr int kPlanTables = 8;     // selections a handle keeps tabulated; the one used longest ago goes first
}  // namespace moe

struct moe_handle {
    int device = 0;
    int G = 0;
    unsigned long long wait_ns = moe::kDefaultWaitNs;
    char err[512] = {0};
    std::unordered_map<const void *, uint32_t> epochs;  // per flags workspace
    void *encode_tiled = nullptr;                       // cuTensorMapEncodeTiled
    int o_comp[3] = {0, 0, 0};                          // tile_n = 64, 128, 256
    int o_pair = 0;                                     // CTA-pair kernel: resident CTAs per SM
    int max_pairs = 0;                                  // ... and co-resident clusters of two
    int routing_max_cluster = 8;                        // CTAs of the largest cluster the one-launch routing build may use
    // Mailbox for the routed-tile counts (Section III-E: the manager reads them on the host): pinned host
    // memory the GPU writes directly.  The routing kernel stores tiles[0..E_tot) and S, each as one 64-bit word
    // with the call's sequence number in its upper half; the whole-step calls poll the words instead of queueing
    // a copy and synchronising the stream.
    unsigned long long *mail_host = nullptr;
    unsigned long long *mail_dev = nullptr;             // the same memory as the GPU addresses it
    uint32_t mail_seq = 0;
    char *staging = nullptr;                            // host-buffer entry point: pinned, the small inputs on their way to the GPU
    cudaStream_t feed_stream = nullptr;                 // host-buffer entry point: copies x_routed in beside the caller's stream ...
    cudaEvent_t feed_events[2] = {nullptr, nullptr};    // ... from the first event on, up to the second
    void *write_value = nullptr;                        // cuStreamWriteValue32
    void *counts_event = nullptr;                       // cudaEvent_t: "the tile counts have reached the host"
    unsigned long long *timeline = nullptr;             // timeline build: where the next fused launch records
    size_t timeline_bytes = 0;
    uint32_t probe = 0;                                 // timeline build: moe_set_probe bits for the next launches
    moe::MapEntry *maps = nullptr;                      // [kMapEntries], by a hash of the operand's address
    moe::PlanTable *plan_tables = nullptr;              // [kPlanTables]
    uint64_t plan_table_uses = 0;
};

namespace moe {

// Every kernel of this library may be launched before its predecessor on the stream has finished: each waits for the
// predecessor's writes (griddepcontrol.wait) before it touches global memory, so that the launch latencies and
// prologues of a step's kernels lie beside the end of the kernel before.  The routing kernels let their successor start
// early, and the pair kernel does once it serves its shares of the combine; behind the other long ones it starts as they
// end.  CTAs that sit and wait on the SMs that a long kernel leaves idle cost more than they save: whole step at T = 1 / 16 /
// 256 on the DeepSeek shape 73.2 / 72.4 / 102.7 us with early starts everywhere, 68.2 / 69.7 / 99.1 from the short kernels
// alone, 77.2 / 74.1 / 103.5 without chained launches (measured when the routing build was a launch of its own at these sizes).
inline cudaLaunchAttribute chained_launch_attribute()
{
    cudaLaunchAttribute a = {};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    return a;
}
#ifdef __CUDACC__
// Y [T][L][split_w columns in slabs][k_tot][slab's columns]: where the rows of (token, split, slab from column c0 of the split on) begin.
// 64 bits from the first product on: T * L alone passes 2^32 at sizes that fit the card (T = 2^29 tokens of one expert each, L = 8).
__host__ __device__ __forceinline__ size_t y_unit(int tok, int s, int c0, int L, int split_w, int k_tot)
{
    return (((size_t)tok * (size_t)L + (size_t)s) * (size_t)split_w + (size_t)c0) * (size_t)k_tot;
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// (after the wait, so that everything before this kernel is complete when a successor starts)
__device__ __forceinline__ void grid_dependents_may_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// n / d for a quotient below 2^20, n >= 0, d > 0.  A launch runs cold: what its critical path costs is the bytes of the instructions on it,
// fetched one line after the other, and a division of integers is 25 of them at every place.
// (Divisions out of the kernels' preambles, and the tile sequence set up once instead of in every role, whole calls, us: DeepSeek shape
// T = 1 39.2 -> 37.7, T = 16 53.7 -> 53.1, Granite shape T = 1003 81.3 -> 78.7, tiny shape 13.4 -> 13.0.  Warming more code ahead
// of time instead, by warps that wait, delays the code that is needed: +1 to +3 us.)
__device__ __forceinline__ int small_quotient(int n, int d)
{
    int q = (int)__fdividef((float)n, (float)d);        // off by one at most
    const int r = n - q * d;
    if (r < 0) --q;
    if (r >= d) ++q;
    return q;
}
// n / d for 0 <= n < 2^31
__device__ __forceinline__ int quotient(const Divisor &d, int n) { return (int)((unsigned long long)(uint32_t)n * d.mul >> d.shift); }
// Load of what a predecessor may have written: an ordinary load that stays behind the wait (a read-only __ldg may be moved)
template <typename T>
__device__ __forceinline__ T ld_chained(const T *p)
{
    static_assert(sizeof(T) == 4, "32-bit values");
    uint32_t v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    T t;
    memcpy(&t, &v, 4);
    return t;
}
// The same for a count that every thread of a converged warp reads: the reduction makes the value warp-uniform for the
// compiler as well, so that the loops it bounds keep their operands in uniform registers (the loop that issues the
// MMAs is 5 % slower over a whole GEMM1 launch when it cannot)
__device__ __forceinline__ int ld_chained_uniform(const int32_t *p)
{
    return (int)__reduce_max_sync(0xffffffffu, (unsigned)ld_chained(p));
}

// The tile counts for the host, written straight into host memory the GPU can address (`mail`, or nullptr), by one
// warp: word x is the pair (count x, seq), x = 0..E_tot, the last one S.  A 64-bit store arrives whole, so every
// word says by itself whether it belongs to this call: no fence orders anything here.  (Plain counts followed by a
// sequence number needed system-scope fences of the whole CTA, 4-5 us of a small build's 12.)  A kernel is complete
// only when these stores have crossed the bus, so they are left to the kernel behind the routing build where one
// follows without waiting for the host.  seq = 0: `mail` is a plain array of E_tot + 1 counts, for a caller that synchronises
// with the stream.
template <class Count>
__device__ __forceinline__ void mail_counts(unsigned long long *mail, uint32_t seq, int E_tot, int lane, Count count)
{
    if (!mail) return;
    if (seq == 0u) {
        for (int x = lane; x <= E_tot; x += 32) reinterpret_cast<volatile int32_t *>(mail)[x] = count(x);
        return;
    }
    for (int x = lane; x <= E_tot; x += 32)
        *reinterpret_cast<volatile unsigned long long *>(mail + x) = ((unsigned long long)seq << 32) | (uint32_t)count(x);
}
#endif

inline int tile_n_slot(int tile_n) { return tile_n == 64 ? 0 : tile_n == 128 ? 1 : tile_n == 256 ? 2 : -1; }

int32_t cuda_fail(moe_handle *h, cudaError_t e, const char *what);
// MOE_OK when the calling thread's current CUDA device is the handle's; MOE_ERR_UNSUPPORTED (with a
// message in the handle) otherwise.  Every launching entry point checks it: kernels run on the
// current device, the buffers and the cached residency belong to the handle's.
int32_t require_handle_device(moe_handle *h, const char *who);
Divisor divisor_of(int32_t d);     // d > 0
// the tensor map of an operand (planes = 0: two dimensions); nullptr, with a message in the handle, when it cannot be encoded
const CUtensorMap *operand_map(moe_handle *h, const void *ptr, int32_t planes, int64_t rows, int32_t cols, int32_t box_rows, const char *name);
// ... of the gate and up weights [experts][2][inter][cols]: boxes of box_inter intermediate columns (a multiple of 16), in groups of 16
// gate rows followed by the 16 up rows of the same columns; inter % 16 == 0
const CUtensorMap *gate_up_map(moe_handle *h, const void *ptr, int32_t experts, int32_t inter, int32_t cols, int32_t box_inter, const char *name);
// fused kernel (gemm2_combine.cu)
size_t fused_smem_bytes(int tile_n);
cudaError_t fused_occupancy(int tile_n, int *blocks_per_sm);
cudaError_t fused_launch(int tile_n, const FusedParams &p, int grid, cudaStream_t stream);
int fused_co_warps_max();      // co-resident communication warps a compute CTA has shared memory for
// operand stages of a compute CTA, and their size; x_rows: see FusedParams; aux_free: no co-resident warps
int fused_stages(bool pair, int tile_n, int x_rows, bool aux_free, int *stage_bytes);
bool fused_timeline_build();   // the library was compiled with -DMOE_TIMELINE=1
// CTA-pair kernel (256 x 256 tiles, clusters of two)
cudaError_t pair_occupancy(int *blocks_per_sm, int *max_clusters);
cudaError_t pair_launch(const FusedParams &p, int grid, cudaStream_t stream);
// GEMM1 (gemm1_act.cu): once per device, kernel attributes
cudaError_t gemm1_prepare();
// moe_gemm1_act; mail_seq != 0: this launch mails the tile counts (with MOE_MTILES_ON_DEVICE); topk_idx != nullptr: it builds the
// routing first
int32_t launch_gemm1_act(moe_handle *h, const void *hidden, const void *W1, const int32_t *topk_idx, const moe_shape *s, int32_t tile_m,
                         const moe_routing *r, int32_t n_mtiles, void *h_routed_ws, void *x_routed, uint32_t *status_dev, uint32_t mail_seq, void *stream);
inline RoutingOut routing_out(const moe_routing &r)
{
    return {r.counts, r.offsets, r.tiles, r.tile_offsets, r.mtile_expert, r.mtile_first_row, r.mtile_valid, r.perm, r.inv_perm, r.pad_row};
}
// whether a kernel of `threads` threads on one-CTA tiles may build this batch's routing itself
inline bool routing_inline_ok(const moe_shape &s, int tile_m, int threads)
{
    return s.T > 0 && tile_m <= 128 && (int64_t)s.T * s.k_tot <= kInlineMaxR && s.E_tot <= threads;
}
// routing kernels (routing.cu)
// the address under which a kernel can write the caller's tile_counts_host itself (pinned memory), nullptr: it takes a copy
int32_t *host_writable(int32_t *tile_counts_host);
// once per device: kernel attributes, and the largest cluster the one-launch build can run with
cudaError_t routing_prepare(int *max_cluster);
// mail / mail_seq: see mail_counts (nullptr: the counts are not mailed); `scratch`: ceil(R / 256) * E_tot ints
// for the sizes that take more than one launch, any contents
cudaError_t routing_launch(const int32_t *topk_idx, const moe_shape &s, int tile_m, const moe_routing &r, int32_t *scratch,
                           int max_cluster, uint32_t *status, unsigned long long *mail, uint32_t mail_seq, cudaStream_t stream);

}  // namespace moe
