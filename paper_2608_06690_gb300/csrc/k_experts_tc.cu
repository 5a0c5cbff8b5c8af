// Stages 3 and 4 of the layer on the 5th-generation tensor cores: grouped
// BF16 expert GEMMs with tcgen05.mma accumulating in tensor memory (TMEM),
// operands staged into 128-byte-swizzled shared memory.
//
//   gate/up:  act = bf16(silu(A_e W_gate,e^T) * (A_e W_up,e^T))    (SwiGLU fused)
//   down:     y   = bf16(w_row * (act_e W_down,e^T))
//
// Groups are the routed experts (rows of the dispatch order) plus, with
// shared experts, one dense group over all T tokens (gate/up weights of the
// E_sh experts side by side; the down projection sums the E_sh experts in
// one accumulator).
//
// The grid is persistent, one CTA per SM in CTA pairs (cta_group::2,
// tc_ptx.cuh).  The weights are the MMA's M and the tokens its N: a pair's
// tile is 256 weight rows (gate/up: each CTA 64 gate and the same 64 up
// columns; down: 128 output columns each) x N tokens of one expert, N any
// multiple of 32 up to 256, half of them staged by each CTA.  N follows the
// expert's rows, so a tile computes at most 31 padding rows (128-row M tiles
// computed 31 % padding at Qwen3 prefill), and a full tile stages 32 KB per CTA
// and 64-wide K step for what a single CTA's 128 x 256 tile stages 48 KB.
// The ring's stages are as large as the launch's largest N needs: 6 of 32 KB
// at N = 256, 10 of 18 KB at N = 32 (decode), so that a batch of few rows per
// expert keeps 160 KB of weights in flight per SM.
//
// What bounds it: HBM (the weights) up to a few thousand tokens, then the rate
// at which L2 delivers the operands (32 KB a stage and CTA in 512 clocks at the
// full MMA rate).  Whole forward, against single-CTA tiles of 128 tokens x 256
// weight rows with the roles' loops in single threads (both on one GPU; the
// figures hold the other steps described here too): Qwen3 shape T = 4096 432 -> 369
// us, T = 16384 1248 -> 1060 us, T = 777 275 -> 266 us, T = 64 215 -> 207 us;
// DeepSeek shape T = 8192 1037 -> 884 us.  Half of that is the roles' own time a
// stage (tc_ptx.cuh: the waits' timer, the elected lane) and a tile (the queue
// below).
//
// The pairs walk a tile list built on the device from the dispatch offsets:
// no host sync, and empty experts contribute no tile.  The list holds every
// gate/up tile, then every down tile, expert by expert with the pools
// interleaved where it pays (pool_place), weight-block major inside
// a group, so that the tiles sharing weights are next to each other.  Each pair
// takes the next tile when its loader is ready for one (an atomic counter);
// the leader hands it to the roles of both CTAs through a small queue in
// shared memory.  A down tile waits (bounded) until the gate/up tiles of its
// activation rows have stored them; every one of those was handed out earlier
// to a running pair, and no gate/up tile ever waits, so the wait ends.
//
// The routed gate/up tiles read their token rows straight from the hidden
// states: the row of dispatch slot r is hidden[tok_of_slot[r]], gathered into
// shared memory by eight warps with 16-byte cp.async copies (the hidden states,
// read by every expert a token routes to, stay in L2), so the dispatched rows
// are never written out.  The gather warps never wait for their own copies:
// each thread's copies of a stage arrive on a barrier when they complete
// (cp.async.mbarrier.arrive): the leader's on the stage's full barrier; the
// other CTA's on one of its own, where its warp 0 waits, fences the async proxy
// and arrives on the leader's.  With in-launch routing (at most 128 tokens) TMA
// gather4 copies of four rows take their place, which complete on the leader's
// full barrier like any other (see kGatherGroups).
//
// CTA roles (480 threads; 384 with in-launch routing):
//   warp 0       hands out the tiles (leader) and loads the token rows that
//                come through TMA (activations or, for the shared group, hidden
//                states; with in-launch routing half of the gathered ones)
//   warp 1       allocates 512 TMEM columns (two accumulators of 256 columns,
//                so the epilogue of one tile overlaps the MMAs of the next);
//                the leader's issues tcgen05.mma M = 256, K = 16
//   warps 2..5   epilogue: tcgen05.ld of the warp's 32 TMEM lanes (= 32 weight
//                columns).  Gate/up: the gate columns sit in warps 0-1's lanes
//                and the up columns in warps 2-3's; the two warps of a column
//                swap half of each 32-token chunk through shared memory, so
//                each computes the SwiGLU of 16 tokens.  Results are transposed
//                through shared memory into row-major 64-byte runs.  In gate/up
//                mode the tiles of weight block 0 also write the execution audit,
//                each row checked against the route log of its token
//   warps 6..13  the row gather of the routed gate/up tiles (cp.async), two
//                groups of four warps taking turns; with in-launch routing
//                warp 6 alone, the other half of the rows by gather4
//   next         the weights through TMA
// The issuing warps run their loops as whole warps and issue TMA and MMA
// instructions from one elected lane.
// Expert weights that only one tile reads stream through L2 (evict first);
// the hidden states and activations, read again by other tiles of the launch,
// are kept (evict last).
// Every wait is bounded in time: on expiry the CTA records
// PMPE_STATUS_PIPELINE_TIMEOUT, stops issuing work, waits (bounded) for its
// own copies and MMAs in flight, frees its TMEM and exits.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "pmpe_internal.cuh"
#include "tc_ptx.cuh"

namespace pmpe {
namespace {

constexpr int kMaxN = 256;                    // tokens per tile at most (MMA N; a multiple of 32)
constexpr int kRowBlock = 128;                // rows per block of the execution audit's tile count
constexpr int BK = 64;                        // K per stage: one 128-byte swizzle row
constexpr int kWBytes = 128 * BK * 2;         // a CTA's weight rows of a stage: 16 KB
constexpr int kRingBytes = 6 * 2 * kWBytes;   // 6 stages at N = 256
constexpr int kMaxStages = 10;                // at N = 32: 18 KB each
constexpr int kAccCols = kMaxN;               // FP32 TMEM columns per accumulator
constexpr int kTmemCols = 2 * kAccCols;
// The row gather of the routed gate/up tiles: with in-launch routing (at most
// 128 tokens) TMA gather4 copies of four rows, issued by warp 0 and one more;
// else groups of four warps with cp.async, every other stage each.  (gather4
// takes about 43 clocks for four rows: one token's step 48 -> 44.5 us and a
// decode step of 96 tokens 224 -> 220 us with it, but 32 of them a stage
// took the gate/up GEMM at T = 16384 from 527 to 1,037 us.)
constexpr int kGatherGroups = 2;
constexpr int kGatherWarp = 6;                // the first of the gather's warps
template <bool kRoute> constexpr int kGatherWarps = kRoute ? 1 : 4 * kGatherGroups;
// (In-launch routing: four more warps, which only take part in the routing and
// the combine; 207.9 -> 207.0 us at T = 64.)
template <bool kRoute> constexpr int kTcThreads = 192 + 32 * kGatherWarps<kRoute> + (kRoute ? 160 : 32);
constexpr int kGatherThreads = 128;           // of a cp.async group: the arrivals of a gathered stage
// Arrivals of a ring stage: the leader's token and weight loaders; with cp.async
// the leader's gather and the other CTA's.
template <bool kRoute> constexpr int kFullArrivals = kRoute ? 2 : 3 + kGatherThreads;
constexpr int kMaxGroups = 2 * kMaxPool + 1;
constexpr int kPrefetchTiles = 76;            // gate/up tiles (1 MB of weights each) prefetched into L2 at small batches
// Large batches, the launch following the router: the gate and up weights of
// the list's first experts (at most 96 MiB, at most 16 experts) prefetched
// into L2 while the router runs, by the CTAs that start early, after a delay
// that lets the router's own reads of the token rows go first.
constexpr size_t kPrefillPrefetchBytes = 96ull << 20;
constexpr int kPrefillPrefetchExperts = 16;
constexpr unsigned long long kPrefillPrefetchDelayNs = 14000;
constexpr int kTQ = 8;                        // tile queue entries (tile indices handed to the pair's roles)
constexpr int kHandOutStages = 8;             // K steps before a tile's last at which the next tile is handed out
// Readers of a queue entry (one lane each): the leader's MMA, weight, epilogue
// and gather warps; the other CTA's token, weight, epilogue and gather warps.
template <bool kRoute> constexpr int kTQConsumers = 2 * (2 + 4 + kGatherWarps<kRoute>);
constexpr int kStageOutBytes = 4096;          // per epilogue warp: two 2 KB exchange / transpose buffers
constexpr int kRowWBytes = kMaxN * 4;         // per epilogue warp: the tile's routing weights
constexpr int kDynSmem = kRingBytes + 4 * (kStageOutBytes + kRowWBytes) + 1024 /* alignment slack */;
constexpr int kTokBoxes = 4;                  // token row boxes: 128, 64, 32, 16 rows

enum { kGateUp = 0, kDown = 1 };

struct TcPhase {
    bf16 *C_routed, *C_shared;
};

struct TcParams {
    // which GEMMs this launch runs: the gate/up tiles, the down tiles
    int has_gu, has_down;
    TcPhase ph[2];    // [kGateUp], [kDown]
    uint32_t idesc;   // tcgen05 instruction descriptor (BF16 x BF16 -> FP32, M = 256, N added per tile)
    int E, E_pub, E_sh, T, H, I, R, k;
    const uint32_t *offsets;
    const float *w_of_slot;
    const int32_t *tok_of_slot;
    const int32_t *topk_idx;  // [T, k] the route log, read back by the execution audit
    const bf16 *hidden;       // the gather source of the routed gate/up tiles
    // has_gu && has_down: per (group, row tile), the gate/up epilogue warps
    // whose activations are stored (zeroed before the launch)
    uint32_t *ready;
    // the next tile of the list to hand out (zeroed before the launch): pairs
    // take tiles in list order, each when it is ready for one
    uint32_t *tile_ctr;
    uint32_t *exec_rows, *exec_tiles, *exec_priv_rows, *shared_rows, *status;
    // fused dispatch (the launch follows the router directly): the CTAs first
    // derive the dispatch order from the router's per-tile counts and route
    // log, write the slot maps, clear the counters above, and meet at a grid
    // barrier (grid_bar, zeroed by the router) before the first tile
    int fuse_dispatch;
    const int32_t *ticket;      // [T, k] 128 * router tile + position among the tile's rows of its expert
    const float *w_route;       // [T, k] routing weights
    const uint32_t *tile_counts;  // [E][slots4] rows of each expert per router tile
    int slots, slots4;
    uint32_t *counts_w, *offsets_w;  // written: rows and first slot of each expert
    int32_t *slot_of_w, *tok_of_slot_w;
    float *w_of_slot_w;
    uint32_t *grid_bar;
    int clear_words;            // readiness counters and the tile counter, from `ready`
    // routing in the launch (T <= 128, nothing launched before this kernel
    // but the clearing of `ready`, the tile counter and the barriers): the
    // CTAs compute the masked router's logits, the top k, the routing weights
    // and the route log, then the dispatch order (route_in_launch)
    int fuse_route;
    int renorm;
    const uint8_t *policy;           // [T] policy bytes, or NULL (every token DENY)
    const bf16 *router_w[2];         // [E_pub, H] public, [E_priv, H] private router
    float *z;                        // [T][zpitch] logits of each token's pool (scratch)
    int zpitch;
    int32_t *idx_w, *ticket_w;       // [T, k] route log written
    float *w_w;                      // [T, k] routing weights written
    uint8_t *tau_w;                  // [T]
    uint32_t *tile_counts_w;         // [E][slots4]
    uint32_t *route_count, *route_priv_rows;
    uint32_t *bar_a, *bar_b;         // grid barriers after the logits and after the selection
    // with fuse_route: the weighted combine too, after a last grid barrier
    // (bar_d) once every CTA's down tiles are stored
    int fuse_combine;
    uint32_t *bar_d;
    bf16 *out;                       // [T, H]
    // small batches (at most 128 tokens: every expert one row tile): the first
    // `prefetch_tiles` gate/up tiles of the list of all experts have their
    // weights prefetched into L2 by the CTA of the same index, before the
    // launch waits for the routing (the weights are inputs, not results of
    // the kernels before); 0 = off
    int prefetch_tiles;
    int prefetch_experts;      // large batches: CTA e < this prefetches expert e's gate and up rows
    uint8_t up_first[3];      // the box holds the up rows before the gate rows
    uint8_t gu_two_boxes[3];
    const bf16 *gate_w[2], *up_w[2];  // [E_pool * I, H] public / private
    // optional FP32: the gate and up accumulators saved for the backward,
    // [R][2I] G | U of the routed rows, then [T][2 E_sh I] of the shared
    // experts
    float *saved_gu;
};

struct TcMaps {
    // per pool [pub, priv, shared]: the gate and up rows of 64 columns as one
    // 3-D box of both tensors (one dimension steps from one to the other), or
    // (p.gu_two_boxes) 64-row boxes of each; down, 128-row boxes
    CUtensorMap gu[3], gate[3], up[3], down[3];
    CUtensorMap hidden;        // the hidden states, one-row boxes (gather4)
    CUtensorMap tok[2][kTokBoxes];     // per GEMM, by box rows: the shared group's hidden states; the activations
    CUtensorMap tok_sh[kTokBoxes];     // the shared group's activations
};

// ------------------------------------------------------------- tile list

// A tile as the queue carries it: two 16-byte words of shared memory.
enum { kTileDown = 1, kTileShared = 2, kTileManyRows = 4, kTileEnd = 8 };
struct __align__(16) Tile {
    int flags;      // kTile...: the GEMM, the shared group, several row tiles read its weights, the list's end
    int g, m_tile, m0, n0, rows, row_base, nkb;
    __device__ __forceinline__ bool down() const { return flags & kTileDown; }
    __device__ __forceinline__ bool shared() const { return flags & kTileShared; }
    __device__ __forceinline__ bool gather() const { return (flags & (kTileDown | kTileShared)) == 0; }
    __device__ __forceinline__ int n() const { return (rows + 31) & ~31; }
};

struct TileTable {
    int prefix[2][kMaxGroups + 1];  // tiles of the places before L, per GEMM
    uint16_t order[2 * kMaxPool];   // the expert at place L (pool_place, or L)
    int mpre[kMaxGroups + 1];       // row tiles of the groups before g
    int rows[kMaxGroups];
    int base[kMaxGroups];
};

// Row tiles of a group of n rows: the fewest that hold 256 rows, of equal size
// up to a multiple of 32 (equal tiles cost the same MMA time as full ones and a
// remainder, and end together).
__device__ __forceinline__ int row_tiles(int n) { return (n + kMaxN - 1) / kMaxN; }
__device__ __forceinline__ int round32(int n) { return (n + 31) & ~31; }
__device__ __forceinline__ int row_tile_size(int n, int mt) { return round32((n + mt - 1) / mt); }

// Weight blocks of a group: 128 activation columns (gate and up rows) or 256
// output columns (the last block of an H of 128 mod 256 half empty).
__device__ __forceinline__ int group_blocks(const TcParams &p, int mode, bool shared)
{
    return mode == kGateUp ? (shared ? p.E_sh * p.I : p.I) / 128 : (p.H + 255) / 256;
}
__device__ __forceinline__ int group_k(const TcParams &p, int mode, bool shared)
{
    return mode == kGateUp ? p.H : (shared ? p.E_sh * p.I : p.I);
}

__device__ __forceinline__ int total_tiles(const TcParams &p, const TileTable &tt, int G)
{
    return (p.has_gu ? tt.prefix[kGateUp][G] : 0) + (p.has_down ? tt.prefix[kDown][G] : 0);
}

// The down GEMM's order of the places: with shared experts their group sits
// after the first half of the routed experts, so that the list ends with
// routed down tiles (K = I) instead of the shared group's (K = E_sh I, the
// launch's longest tiles), which otherwise made the last wave uneven; there
// the shared group's gate/up tiles, the last of the gate/up list, are long
// finished.  The gate/up GEMM's list ends with the shared group: its token rows
// come through TMA, and the gather warps fill no stage after such a tile.
// down_place inverts it.
__device__ __forceinline__ int down_group(const TcParams &p, int L)
{
    if (p.E_sh == 0) return L;
    const int h = p.E / 2;
    return L < h ? L : (L == h ? p.E : L - 1);
}
__device__ __forceinline__ int down_place(const TcParams &p, int g)
{
    if (p.E_sh == 0) return g;
    const int h = p.E / 2;
    return g < h ? g : (g == p.E ? h : g + 1);
}

// Tile `tile` of the list (the end at `total`): the gate/up tiles (when this
// launch runs them), then the down tiles; inside a GEMM, place by place (the
// down GEMM in down_group order), weight-block major.  By a whole warp.
template <bool kRoute>
__device__ __forceinline__ Tile decode_tile(const TcParams &p, const TileTable &tt, int G, int tile, int total, int lane)
{
    Tile t;
    if (tile >= total) {
        t.flags = kTileEnd;
        t.g = t.m_tile = t.m0 = t.n0 = t.rows = t.row_base = t.nkb = 0;
        return t;
    }
    const int n_gu = p.has_gu ? tt.prefix[kGateUp][G] : 0;
    const int ph = tile < n_gu ? kGateUp : kDown;
    const int local_all = tile - (ph == kDown ? n_gu : 0);
    const int *pre = tt.prefix[ph];
    int n = 0;  // places with prefix <= local_all; the last of them holds the tile
    for (int b = 0; b < G; b += 32) n += __popc(__ballot_sync(~0u, b + lane < G && pre[b + lane] <= local_all));
    const int lo = n - 1;
    const int L = ph == kDown ? down_group(p, lo) : lo;
    const bool shared = L >= p.E;
    const int g = shared ? p.E : kRoute ? L : tt.order[L];
    const int rows = tt.rows[g], mt = row_tiles(rows);
    const int local = local_all - pre[lo];
    const int block = local / mt;
    const int bm = row_tile_size(rows, mt);
    t.flags = (ph == kDown ? kTileDown : 0) | (shared ? kTileShared : 0) | (mt > 1 ? kTileManyRows : 0);
    t.g = g;
    t.m_tile = local - block * mt;
    t.m0 = t.m_tile * bm;
    t.n0 = block * (ph == kGateUp ? 128 : 256);
    t.rows = min(bm, rows - t.m0);
    t.row_base = tt.base[g];
    t.nkb = group_k(p, ph, shared) / BK;
    return t;
}

// ---------------------------------------------------------------- kernel

// Weights of gate/up tile blockIdx.x of the list of all experts (the first
// wave when every expert has one row tile): 128 gate rows and
// 128 up rows, each block contiguous, prefetched into L2 by one thread.
__device__ __forceinline__ void prefetch_first_wave(const TcParams &p, bool by_place)
{
    const int nt = p.I / 128;
    const int L = (int)blockIdx.x / nt, n = (int)blockIdx.x - L * nt;
    if (L < p.E) {
        const int e = by_place ? pool_at(L, p.E_pub, p.E - p.E_pub) : L;
        const int q = e < p.E_pub ? 0 : 1;
        const size_t row0 = (size_t)(q ? e - p.E_pub : e) * p.I + (size_t)n * 128;
        const uint32_t bytes = (uint32_t)(128u * (uint32_t)p.H * 2u);
        bulk_prefetch_l2(p.gate_w[q] + row0 * p.H, bytes);
        bulk_prefetch_l2(p.up_w[q] + row0 * p.H, bytes);
    }
}

// Arrival at a grid barrier (or on a readiness counter): a release add, so that
// the writes the barrier before it ordered (of every thread of the CTA, or of the
// warp) are visible to whoever acquires the count.
__device__ __forceinline__ void grid_arrive(uint32_t *ctr)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(ctr) : "memory");
}

// Every CTA of the grid arrives (after all of its threads' writes), then
// waits, bounded, until `target` arrivals are counted (acquire loads; the CTA
// barrier after them orders the other threads); writes before the barrier,
// by any thread of any CTA, are visible after it.  The grid is resident all
// at once (checked before the launch).  False after a timeout or an abort.
// (A release add and a tight acquire spin measured 0.5 us faster a decode
// step than a full fence, a relaxed add and a spin with back-off.)
__device__ bool grid_barrier(uint32_t *ctr, uint32_t target, volatile int *abort_flag, uint32_t *status)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        grid_arrive(ctr);
        const unsigned long long t0 = globaltimer_ns();
        while (ld_acquire_gpu(ctr) < target) {
            if (*abort_flag) { ok = 0; break; }
            if (globaltimer_ns() - t0 > kWaitLimitNs) {
                *abort_flag = 1;
                if (status) atomicOr(status, PMPE_STATUS_PIPELINE_TIMEOUT);
                ok = 0;
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

constexpr int kRouteMaxTokens = 128;   // routing in the launch: one selection CTA per token
constexpr int kRouteMaxH = 2048;       // the logits hold a row's 16-byte pieces in registers, 8 a lane at most
constexpr int kRouteXChunks = kRouteMaxH / 256;  // 16-byte pieces of the token row per lane

__device__ __forceinline__ float dot8_bf16(const uint4 &a, const uint4 &b, float acc)
{
    const __nv_bfloat162 *x = reinterpret_cast<const __nv_bfloat162 *>(&a);
    const __nv_bfloat162 *y = reinterpret_cast<const __nv_bfloat162 *>(&b);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 u = __bfloat1622float2(x[i]), v = __bfloat1622float2(y[i]);
        acc = fmaf(u.x, v.x, acc);
        acc = fmaf(u.y, v.y, acc);
    }
    return acc;
}

// Exact ranking of two candidates (logit, pool-local id): the larger logit,
// at equal logits the lower id (NaN was cleaned to -inf before).
__device__ __forceinline__ bool route_above(float x, int e, float bx, int be)
{
    return (x > bx) | ((x == bx) & (e < be));
}

// Routing inside the persistent launch, for T <= 128 tokens (Sec. 3.1 Eq. 4
// and App. B.1), in three steps separated by grid barriers:
//   1. logits: work items (token t, block c of t's pool), spread over the
//      CTAs, at most one each; each warp of a CTA forms the dot products of its
//      experts with the token row (FP32: a lane's 16-byte pieces in order,
//      then a butterfly), into z[t][e].  A token meets only its own pool's
//      router rows.
//   2. selection: CTA t < T, one warp: the top k of z[t] by k passes of an
//      exact (logit, id) maximum, ties to the lower id; the weights (softmax
//      over the k, or over the pool); the route log.
//   3. dispatch: every CTA forms per expert the mask of the tokens that
//      picked it, the counts and first slots (experts in id order, tokens in
//      order), and resolves its share of the routed rows (slot = first slot
//      + rank of the token among the expert's tokens).  The tile table takes
//      the counts and first slots; the caller then arrives at grid_bar.
// Returns false after an abort (a barrier timed out).
__device__ bool route_in_launch(const TcParams &p, uint8_t *ring, TileTable &tt, volatile int *s_abort)
{
    __shared__ int s_item[kRouteMaxTokens + 1];  // items of the tokens before t
    __shared__ uint8_t s_tau[kRouteMaxTokens];
    __shared__ int s_nd;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kThreads = kTcThreads<true>, kWarps = kThreads / 32;
    const int T = p.T, K = p.k, E = p.E, E_priv = p.E - p.E_pub, R = p.R;
    // ---- tau per token (Sec. 2.1) and the logit work items: (token, block
    // of bs experts of its pool), bs the least size from 16 up that gives
    // every CTA at most one item (a CTA's item is a chain of dependent load
    // rounds, so two items on one CTA would double the step)
    __shared__ int s_bs;
    if (warp == 0) {
        int nd = 0;
        for (int b0 = 0; b0 < T; b0 += 32) {
            const int t = b0 + lane;
            const int tau = (t < T && p.policy) ? (p.policy[t] == 0x01 ? 1 : 0) : 0;
            if (t < T) s_tau[t] = (uint8_t)tau;
            nd += __popc(__ballot_sync(~0u, t < T && tau == 0));
        }
        const int na = T - nd;
        int bs = 256;  // one item per token always fits (T <= the grid)
        for (int b1 = 16; b1 < 256; b1 += 32) {  // the lanes test 32 sizes at a time
            const int c = b1 + lane;
            const bool fits = nd * ((p.E_pub + c - 1) / c) + na * ((E_priv + c - 1) / c) <= (int)gridDim.x;
            const unsigned m = __ballot_sync(~0u, fits);
            if (m) {
                bs = b1 + __ffs(m) - 1;
                break;
            }
        }
        int carry = 0;
        for (int b0 = 0; b0 < T; b0 += 32) {
            const int t = b0 + lane;
            const int v0 = t < T ? ((s_tau[t] ? E_priv : p.E_pub) + bs - 1) / bs : 0;
            int v = v0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(~0u, v, off);
                if (lane >= off) v += y;
            }
            if (t < T) s_item[t] = carry + v - v0;
            carry += __shfl_sync(~0u, v, 31);
        }
        if (lane == 0) {
            s_item[T] = carry;
            s_nd = nd;
            s_bs = bs;
        }
    }
    __syncthreads();
    const int nitems = s_item[T], nd = s_nd, bs = s_bs;
    const int nch = p.H / 8;  // 16-byte pieces of a row
    // ---- 1. logits (loads straight into registers: each warp takes its
    // experts two at a time, so that a lane has 16 loads of 16 bytes in
    // flight; bulk copies of the block into shared memory were slower)
    for (int i = (int)blockIdx.x; i < nitems; i += (int)gridDim.x) {
        int lo = 0, hi = T - 1;  // the token of item i: the last t with s_item[t] <= i
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_item[mid] <= i) lo = mid; else hi = mid - 1;
        }
        const int t = lo, tau = s_tau[t];
        const int e0 = (i - s_item[t]) * bs;
        const int ne = min(bs, (tau ? E_priv : p.E_pub) - e0);
        const uint4 *xrow = reinterpret_cast<const uint4 *>(p.hidden + (size_t)t * p.H);
        const uint4 *wblk = reinterpret_cast<const uint4 *>(p.router_w[tau] + (size_t)e0 * p.H);
        uint4 xr[kRouteXChunks];
#pragma unroll
        for (int q = 0; q < kRouteXChunks; ++q) {
            const int ch = lane + 32 * q;
            xr[q] = ch < nch ? __ldg(xrow + ch) : make_uint4(0u, 0u, 0u, 0u);
        }
        for (int e = warp; e < ne; e += 2 * kWarps) {
            const int e2 = e + kWarps;  // the second expert of the pair (absent past the block)
            uint4 wa[kRouteXChunks], wb[kRouteXChunks];
#pragma unroll
            for (int q = 0; q < kRouteXChunks; ++q) {
                const int ch = lane + 32 * q;
                wa[q] = ch < nch ? __ldg(wblk + (size_t)e * nch + ch) : make_uint4(0u, 0u, 0u, 0u);
                wb[q] = (ch < nch && e2 < ne) ? __ldg(wblk + (size_t)e2 * nch + ch) : make_uint4(0u, 0u, 0u, 0u);
            }
            float acc_a = 0.f, acc_b = 0.f;
#pragma unroll
            for (int q = 0; q < kRouteXChunks; ++q) {
                if (lane + 32 * q < nch) {
                    acc_a = dot8_bf16(wa[q], xr[q], acc_a);
                    acc_b = dot8_bf16(wb[q], xr[q], acc_b);
                }
            }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) {
                acc_a += __shfl_xor_sync(~0u, acc_a, off);
                acc_b += __shfl_xor_sync(~0u, acc_b, off);
            }
            if (lane == 0) {
                p.z[(size_t)t * p.zpitch + e0 + e] = acc_a;
                if (e2 < ne) p.z[(size_t)t * p.zpitch + e0 + e2] = acc_b;
            }
        }
    }
    if (!grid_barrier(p.bar_a, gridDim.x, s_abort, p.status)) return false;
    // the first wave's weights into L2 while the selection and the dispatch
    // run (not earlier: the prefetch would delay the router rows)
    if (warp == 2 && lane == 0 && (int)blockIdx.x < p.prefetch_tiles) prefetch_first_wave(p, false);
    // ---- 2. selection, one warp per token
    if ((int)blockIdx.x < T && warp == 0) {
        const int t = (int)blockIdx.x, tau = s_tau[t];
        const int P = tau ? E_priv : p.E_pub, base = tau ? p.E_pub : 0;
        const float *zt = p.z + (size_t)t * p.zpitch;
        float v[8], vo[8];
        int id[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = lane + 32 * q;
            const float x = e < P ? zt[e] : -INFINITY;
            vo[q] = v[q] = x != x ? -INFINITY : x;  // NaN never outranks a number
            id[q] = e < P ? e : 0x7fffffff;
        }
        float my_v = 0.f, top = 0.f;
        int my_e = 0;
        for (int j = 0; j < K; ++j) {
            float bv = v[0];
            int be = id[0];
#pragma unroll
            for (int q = 1; q < 8; ++q)
                if (route_above(v[q], id[q], bv, be)) {
                    bv = v[q];
                    be = id[q];
                }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) {
                const float ov = __shfl_xor_sync(~0u, bv, off);
                const int oe = __shfl_xor_sync(~0u, be, off);
                if (route_above(ov, oe, bv, be)) {
                    bv = ov;
                    be = oe;
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (id[q] == be) {
                    v[q] = -INFINITY;
                    id[q] = 0x7fffffff;
                }
            if (lane == j) {
                my_v = bv;
                my_e = be;
            }
            if (j == 0) top = bv;
        }
        float den = 0.f;
        if (p.renorm) {  // softmax over the k selected logits, in rank order
            for (int j = 0; j < K; ++j) den += expf(__shfl_sync(~0u, my_v, j) - top);
        } else {         // softmax over the pool
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (lane + 32 * q < P) den += expf(vo[q] - top);
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) den += __shfl_xor_sync(~0u, den, off);
        }
        if (lane < K) {
            p.idx_w[(size_t)t * K + lane] = base + my_e;
            p.w_w[(size_t)t * K + lane] = expf(my_v - top) / den;
            if (p.route_count) atomicAdd(&p.route_count[base + my_e], 1u);
        }
        if (lane == 0) {
            p.tau_w[t] = (uint8_t)tau;
            if (p.route_priv_rows) atomicAdd(&p.route_priv_rows[t], tau ? (unsigned)K : 0u);
        }
    }
    if (!grid_barrier(p.bar_b, gridDim.x, s_abort, p.status)) return false;
    // ---- 3. dispatch order: per expert the mask of its tokens (4 x 32 bits)
    uint32_t *smask = reinterpret_cast<uint32_t *>(ring);
    int *sfirst = reinterpret_cast<int *>(smask + (size_t)E * 4);
    int *scount = sfirst + E;
    for (int i = tid; i < E * 4; i += kThreads) smask[i] = 0u;
    __syncthreads();
    for (int r = tid; r < R; r += kThreads) {
        const int e = p.idx_w[r], t = r / K;
        if ((unsigned)e < (unsigned)E) atomicOr(&smask[e * 4 + (t >> 5)], 1u << (t & 31));
    }
    __syncthreads();
    if (warp == 0) {  // rows per expert and their exclusive prefix: the first slots
        int carry = 0;
        for (int b0 = 0; b0 < E; b0 += 32) {
            const int g = b0 + lane;
            const int v0 = g < E ? __popc(smask[g * 4]) + __popc(smask[g * 4 + 1]) + __popc(smask[g * 4 + 2]) +
                                       __popc(smask[g * 4 + 3])
                                 : 0;
            int v = v0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(~0u, v, off);
                if (lane >= off) v += y;
            }
            if (g < E) {
                sfirst[g] = carry + v - v0;
                scount[g] = v0;
            }
            carry += __shfl_sync(~0u, v, 31);
        }
    }
    __syncthreads();
    // the router tile of a pool's tokens (the cluster router's numbering:
    // the DENY tile first when there are DENY tokens)
    auto tile_of = [&](int g) { return g < p.E_pub ? 0 : (nd > 0 ? 1 : 0); };
    if (blockIdx.x == 0) {
        for (int g = tid; g < E; g += kThreads) {
            p.offsets_w[g] = (uint32_t)sfirst[g];
            p.counts_w[g] = (uint32_t)scount[g];
            for (int sl = 0; sl < p.slots; ++sl)
                p.tile_counts_w[(size_t)g * p.slots4 + sl] = sl == tile_of(g) ? (uint32_t)scount[g] : 0u;
        }
        if (tid == 0) p.offsets_w[E] = (uint32_t)R;
    }
    for (int r = (int)blockIdx.x * kThreads + tid; r < R; r += (int)gridDim.x * kThreads) {
        const int e = p.idx_w[r], t = r / K;
        if ((unsigned)e >= (unsigned)E) {  // never produced by the selection
            if (p.status) atomicOr(p.status, PMPE_STATUS_BAD_EXPERT_ID);
            continue;
        }
        const int wd = t >> 5;
        int rank = __popc(smask[e * 4 + wd] & ((1u << (t & 31)) - 1u));
        for (int w2 = 0; w2 < wd; ++w2) rank += __popc(smask[e * 4 + w2]);
        const int slot = sfirst[e] + rank;
        if ((unsigned)slot >= (unsigned)R) continue;
        p.slot_of_w[r] = slot;
        p.tok_of_slot_w[slot] = t;
        p.w_of_slot_w[slot] = p.w_w[r];
        p.ticket_w[r] = tile_of(e) * 128 + rank;
    }
    for (int g = tid; g < E; g += kThreads) {
        tt.rows[g] = scount[g];
        tt.base[g] = sfirst[g];
    }
    fence_proxy_async_smem();  // this thread's use of the ring, before the GEMM's copies land there
    return true;
}

// Shared-memory bytes the fused dispatch needs for its per-expert prefix of
// the router tiles' counts ([E][slots + 1] words, inside the ring).
constexpr size_t fused_dispatch_smem(int E, int slots) { return (size_t)E * (size_t)(slots + 1) * 4u; }

// kRoute: the instantiation that can route the tokens itself (p.fuse_route);
// the other one carries none of that code (fewer registers, a smaller body).
template <bool kRoute>
__global__ void __launch_bounds__(kTcThreads<kRoute>, 1) expert_gemm_tc_kernel(const TcParams p, const __grid_constant__ TcMaps maps)
{
    constexpr int kThreads = kTcThreads<kRoute>, kWeightWarp = kGatherWarp + kGatherWarps<kRoute>;
    extern __shared__ uint8_t dsmem[];
    __shared__ TileTable tt;
    __shared__ __align__(8) uint64_t bars[3 * kMaxStages + 5 + 2 * kTQ];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ Tile s_tq[kTQ];
    __shared__ volatile int s_pdl_done;  // thread 0 has passed griddepcontrol.wait

    const int tid = threadIdx.x, warp = __shfl_sync(~0u, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)cluster_ctarank();  // 0: the pair's leader, whose thread issues the MMAs
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const uint32_t sbase = (smem_u32(dsmem) + 1023u) & ~1023u;
    const uint32_t bar0 = smem_u32(bars);
    // The leader's: full (a stage's TMA bytes and gathered rows of both CTAs),
    // tempty (both CTAs' epilogues), tq_empty.  The other CTA's: gfull (its
    // gathered rows, which it reports to full).  Each CTA's own: empty, tfull (the commits' arrivals) and
    // tq_full, which the leader signals in both.
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
    auto gfull_bar = [&](int s) { return bar0 + 8u * (2 * kMaxStages + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (3 * kMaxStages + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (3 * kMaxStages + 2 + b); };
    const uint32_t done_bar = bar0 + 8u * (3 * kMaxStages + 4);
    auto tq_full_bar = [&](int i) { return bar0 + 8u * (3 * kMaxStages + 5 + i); };
    auto tq_empty_bar = [&](int i) { return bar0 + 8u * (3 * kMaxStages + 5 + kTQ + i); };
    // Entry i of the pair's tile sequence, for a consumer role (a whole warp).
    // False at the end of the list or after an abort.
    // With gather_only (the gather warps) also at the first tile that is not
    // gathered, after which none is: the warp then leaves the entries' barriers,
    // so that it no longer polls beside the down tiles.  It leaves slot by slot,
    // at this entry and the kTQ - 1 after it, once each is published: only then is
    // its arrival on that slot due.  (A drop is also an arrival; on the slot of an
    // earlier entry that a slower role has yet to read it would be this warp's
    // second, and hand the slot back in that role's place.)
    auto next_tile = [&](int i, Tile &t, bool gather_only = false) -> bool {
        const int slot = i % kTQ;
        int ok = 1;
        if (lane == 0) ok = mbar_wait(tq_full_bar(slot), (uint32_t)(i / kTQ) & 1u, &s_abort, p.status) ? 1 : 0;
        if (!__shfl_sync(~0u, ok, 0)) return false;
        const uint32_t a = smem_u32(&s_tq[slot]);
        const uint4 x = ld_shared_v4(a), y = ld_shared_v4(a + 16);
        t.flags = (int)x.x; t.g = (int)x.y; t.m_tile = (int)x.z; t.m0 = (int)x.w;
        t.n0 = (int)y.x; t.rows = (int)y.y; t.row_base = (int)y.z; t.nkb = (int)y.w;
        // (the vote needs every lane's entry: it is read before its slot is handed back)
        const bool live = !__any_sync(~0u, t.flags & kTileEnd) && __all_sync(~0u, t.rows > 0 && t.nkb > 0);
        if (gather_only && !t.gather()) {
            if (lane == 0) {
                int flags = t.flags;
                for (int e = i;;) {
                    mbar_arrive_drop(dsmem_addr(tq_empty_bar(e % kTQ), 0));
                    if (++e == i + kTQ || (flags & kTileEnd)) break;
                    if (!mbar_wait(tq_full_bar(e % kTQ), (uint32_t)(e / kTQ) & 1u, &s_abort, p.status)) break;
                    flags = (int)ld_shared_v4(smem_u32(&s_tq[e % kTQ])).x;
                }
            }
            return false;
        }
        if (lane == 0) {
            if (rank == 0) mbar_arrive(tq_empty_bar(slot));
            else mbar_arrive_remote(dsmem_addr(tq_empty_bar(slot), 0));
        }
        return live;
    };

    const int G = p.E + (p.E_sh > 0 ? 1 : 0);
    // (in-launch routing: few rows an expert, id order)
    const bool by_place = !kRoute && interleave_pools(p.R, p.E);
    // expert weights that one tile reads stream through L2 (evict first); the
    // hidden states, activations and per-row outputs are read again by other
    // tiles of this launch (evict last)
    const uint64_t pol_stream = l2_policy_evict_first(), pol_keep = l2_policy_evict_last();
    const uint64_t pol_normal = l2_policy_evict_normal();
    if (warp == 0 && lane < 2) {  // the weight maps of this launch's GEMMs, ahead of their first loads
        if (lane == 0 ? p.has_gu : p.has_down)
            for (int q = 0; q < (p.E_sh > 0 ? 3 : 2); ++q) prefetch_tmap(lane == 0 ? &maps.gu[q] : &maps.down[q]);
    }
    pdl_trigger();

    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(full_bar(s), kFullArrivals<kRoute>);
            mbar_init(empty_bar(s), 1);
            mbar_init(gfull_bar(s), kGatherThreads);
        }
        for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 8); }
        mbar_init(done_bar, 1);
        for (int i = 0; i < kTQ; ++i) { mbar_init(tq_full_bar(i), 1); mbar_init(tq_empty_bar(i), kTQConsumers<kRoute>); }
        s_abort = 0;
        s_pdl_done = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 1) tmem_alloc_pair(smem_u32(&s_tmem), kTmemCols);
    __syncthreads();  // s_pdl_done and s_abort are initialised
    // weights of the first wave into L2 while the routing is computed (in
    // this launch: after this CTA's router rows have landed, which the
    // prefetch would otherwise delay)
    if (warp == 2 && lane == 0 && (int)blockIdx.x < p.prefetch_tiles && !p.fuse_route) prefetch_first_wave(p, by_place);
    if (warp == 2 && lane == 0 && (int)blockIdx.x < p.prefetch_experts) {
        // the list starts with the first places' tiles: the first wave's weights, after the delay, or at once when the router
        // has already finished (thread 0 passed its wait; bounded spin)
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < kPrefillPrefetchDelayNs && !s_pdl_done) {
        }
        const int e = by_place ? pool_at((int)blockIdx.x, p.E_pub, p.E - p.E_pub) : (int)blockIdx.x;
        const int q = e < p.E_pub ? 0 : 1;
        const size_t row0 = (size_t)(q ? e - p.E_pub : e) * p.I;
        for (int r = 0; r < p.I; r += 128) {
            const uint32_t bytes = (uint32_t)min(128, p.I - r) * (uint32_t)p.H * 2u;
            bulk_prefetch_l2(p.gate_w[q] + (row0 + r) * p.H, bytes);
            bulk_prefetch_l2(p.up_w[q] + (row0 + r) * p.H, bytes);
        }
    }
    pdl_wait();  // the dispatch offsets and slot maps (or the route log, or cleared counters) come from the previous kernel
    if (tid == 0) s_pdl_done = 1;
    if (kRoute && p.fuse_route) {
        const bool ok = route_in_launch(p, dsmem + (sbase - smem_u32(dsmem)), tt, &s_abort);
        if (!ok && tid == 0) s_abort = 1;
        __syncthreads();
        if (tid == 0) grid_arrive(p.grid_bar);  // the roles wait for it (wait_dispatch)
    }
    if (p.fuse_dispatch) {
        // ---- the dispatch order, as dispatch_kernel derives it.  pre[e][s]:
        // rows of expert e in the router tiles before tile s (in the ring,
        // which no load has touched yet), its total = the expert's rows
        uint32_t *pre = reinterpret_cast<uint32_t *>(dsmem + (sbase - smem_u32(dsmem)));
        const int sp = p.slots + 1;
        for (int g = tid; g < p.E; g += kThreads) {
            const uint32_t *tc = p.tile_counts + (size_t)g * p.slots4;
            uint32_t acc = 0;
            int s2 = 0;
            for (; s2 + 4 <= p.slots; s2 += 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(tc + s2);  // slots4: rows 16-byte aligned
                pre[g * sp + s2] = acc; acc += v.x;
                pre[g * sp + s2 + 1] = acc; acc += v.y;
                pre[g * sp + s2 + 2] = acc; acc += v.z;
                pre[g * sp + s2 + 3] = acc; acc += v.w;
            }
            for (; s2 < p.slots; ++s2) { pre[g * sp + s2] = acc; acc += tc[s2]; }
            pre[g * sp + p.slots] = acc;
            tt.rows[g] = (int)acc;
        }
        __syncthreads();
        if (warp == 0) {  // exclusive prefix over the experts: their first slots
            int carry = 0;
            for (int b = 0; b < p.E; b += 32) {
                const int v0 = b + lane < p.E ? tt.rows[b + lane] : 0;
                int v = v0;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int y = __shfl_up_sync(~0u, v, off);
                    if (lane >= off) v += y;
                }
                if (b + lane < p.E) tt.base[b + lane] = carry + v - v0;
                carry += __shfl_sync(~0u, v, 31);
            }
        }
        __syncthreads();
        if (blockIdx.x == 0) {
            for (int g = tid; g < p.E; g += kThreads) {
                p.offsets_w[g] = (uint32_t)tt.base[g];
                p.counts_w[g] = (uint32_t)tt.rows[g];
            }
            if (tid == 0) p.offsets_w[p.E] = (uint32_t)(tt.base[p.E - 1] + tt.rows[p.E - 1]);
            for (int i = tid; i < p.clear_words; i += kThreads) p.ready[i] = 0u;
        }
        // this CTA's share of the routed rows r = (t, j): slot = first slot of
        // its expert + the expert's rows in earlier router tiles + its
        // position in its tile (ticket = 128 * tile + position)
        for (int r = blockIdx.x * kThreads + tid; r < p.R; r += gridDim.x * kThreads) {
            const int e = p.topk_idx[r];
            if ((unsigned)e >= (unsigned)p.E) {  // never produced by the router
                if (p.status) atomicOr(p.status, PMPE_STATUS_BAD_EXPERT_ID);
                continue;
            }
            const int tk = p.ticket[r];
            const int ts = min(tk >> 7, p.slots);
            const int slot = tt.base[e] + (int)pre[e * sp + ts] + (tk & 127);
            if ((unsigned)slot >= (unsigned)p.R) continue;  // only a corrupt ticket could fail this
            p.slot_of_w[r] = slot;
            p.tok_of_slot_w[slot] = r / p.k;
            p.w_of_slot_w[slot] = p.w_route[r];
        }
        // arrive at the grid barrier (an arrival counter the router zeroed);
        // each role waits for every CTA's arrival (wait_dispatch) only before
        // it first reads what other CTAs wrote here, so that the tile table,
        // the first weight loads and the other CTAs' arrivals overlap
        fence_proxy_async_smem();  // this thread's use of the ring, before the GEMM's copies land there
        __syncthreads();
        if (tid == 0) grid_arrive(p.grid_bar);
    }
    // Until every CTA has arrived: the slot maps (tok_of_slot, w_of_slot) and
    // the readiness and tile counters (cleared by CTA 0) are not yet final.
    // Every lane that calls this acquires the arrivals itself (bounded wait;
    // the grid is resident all at once, checked before the launch).
    auto wait_dispatch = [&]() -> bool {
        if (!p.fuse_dispatch && !p.fuse_route) return true;
        const unsigned long long t0 = globaltimer_ns();
        while (ld_acquire_gpu(p.grid_bar) < gridDim.x) {
            if (s_abort) return false;
            if (globaltimer_ns() - t0 > kWaitLimitNs) {
                s_abort = 1;
                if (p.status) atomicOr(p.status, PMPE_STATUS_PIPELINE_TIMEOUT);
                return false;
            }
            __nanosleep(32);
        }
        return true;
    };
    // tile list: rows and tiles per group, prefixes over groups
    int nmax = 0;  // bit b: some row tile has N = 32 (b + 1)
    for (int g = tid; g < G; g += kThreads) {
        const bool shared = g >= p.E;
        int rows, base;
        if (shared) {
            rows = p.T;
            base = 0;
        } else if (p.fuse_dispatch || p.fuse_route) {  // derived above
            rows = min(tt.rows[g], p.R);
            base = min(tt.base[g], p.R - rows);
        } else {  // clamped to [0, R): only a corrupt workspace could make this matter
            const int b = min((int)p.offsets[g], p.R), e = min(max((int)p.offsets[g + 1], b), p.R);
            rows = e - b;
            base = b;
        }
        const int mt = row_tiles(rows);
        if (mt > 0) nmax |= 1 << (row_tile_size(rows, mt) / 32 - 1);
        tt.rows[g] = rows;
        tt.base[g] = base;
        tt.mpre[g + 1] = mt;
        const int L = shared ? p.E : by_place ? pool_place(g, p.E_pub, p.E - p.E_pub) : g;
        if (!kRoute && !shared) tt.order[L] = (uint16_t)g;
        tt.prefix[kGateUp][L + 1] = mt * group_blocks(p, kGateUp, shared);
        tt.prefix[kDown][down_place(p, L) + 1] = mt * group_blocks(p, kDown, shared);
    }
    // the same value in every thread of every CTA (all read the same offsets)
    nmax = __reduce_or_sync(~0u, nmax);
    __shared__ int s_nmax[kThreads / 32];
    if (lane == 0) s_nmax[warp] = nmax;
    __syncthreads();
    if (warp < 3) {  // three inclusive scans, one per warp: tiles of each GEMM, row blocks
        int *arr = warp == 2 ? tt.mpre : tt.prefix[warp];
        int carry = 0;
        for (int b = 0; b < G; b += 32) {
            int v = b + lane < G ? arr[b + lane + 1] : 0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(~0u, v, off);
                if (lane >= off) v += y;
            }
            __syncwarp();
            if (b + lane < G) arr[b + lane + 1] = carry + v;
            carry += __shfl_sync(~0u, v, 31);
        }
        if (lane == 0) arr[0] = 0;
    }
    __syncwarp();
    for (int w = 0; w < kThreads / 32; ++w) nmax |= s_nmax[w];
    tc_fence_before();
    cluster_sync_all();  // both CTAs' barriers, TMEM and tables are ready
    tc_fence_after();
    const uint32_t tmem_base = s_tmem;
    const int total = total_tiles(p, tt, G);
    // the ring: stages of 16 KB of weights and half of the launch's largest
    // N of token rows
    const int stage_bytes = kWBytes + (nmax ? 32 - __clz(nmax) : 1) * (16 * BK * 2);
    const int nst = min(kMaxStages, kRingBytes / stage_bytes);

    // A barrier wait by a whole warp: every lane waits, and the vote keeps the
    // warp together (a lane left behind could be lapped) and gives one answer.
    auto warp_wait = [&](uint32_t bar, uint32_t parity) -> bool {
        return __all_sync(~0u, mbar_wait(bar, parity, &s_abort, p.status));
    };

    // gather4 (kRoute): this CTA's half of a gathered tile's token rows, half
    // `part` of that by warp 0 (0) and by the gather warp (1).  load_rows keeps the
    // rows' token ids (rows past the tile's read token 0, whose columns are not
    // stored).
    __shared__ __align__(16) int s_rows[kRoute ? 2 : 1][kRoute ? kMaxN / 4 : 4];
    auto load_rows = [&](const Tile &t, int part) {
        const int n4 = t.n() / 4, first = rank * (t.n() / 2) + part * n4;
        __syncwarp();
        for (int i = lane; i < n4; i += 32) {
            const int tok = first + i < t.rows ? p.tok_of_slot[t.row_base + t.m0 + first + i] : 0;
            s_rows[part][i] = (unsigned)tok < (unsigned)p.T ? tok : 0;
        }
        __syncwarp();
    };
    auto gather_stage = [&](int stage, int kb, int ng, int part) {
        const uint32_t dst = sbase + stage * stage_bytes + kWBytes + part * ng * 512;
        const uint32_t fb = dsmem_addr(full_bar(stage), 0), ids = smem_u32(s_rows[part]);
#pragma unroll 4
        for (int g = 0; g < ng; ++g) {
            const uint4 r = ld_shared_v4(ids + g * 16);
            tma_gather4_pair(dst + g * 512, &maps.hidden, fb, kb * BK, (int)r.x, (int)r.y, (int)r.z, (int)r.w, pol_keep);
        }
    };

    if (warp == 0) {
        // ------------------------------------------------ tile hand-out, token rows through TMA
        // This CTA's half of the tile's token rows when they come through TMA
        // (the activations, or the hidden states of the shared group; at most
        // three boxes, of 128 to 16 rows); every copy completes on the leader's
        // barrier, where the leader announces both CTAs' bytes.  In a gathered
        // tile the other CTA's warp waits for its CTA's rows, fences the async
        // proxy and arrives there for them.  (Each of these warps holds up
        // every stage until it has passed it: a warp that only followed the
        // ring could be lapped, which a parity wait cannot see.)  The leader
        // picks the tiles (the first one by the pair's index, so that its
        // weights load before the dispatch is final) and hands each to both
        // CTAs' other roles.
        int stage = 0;
        uint32_t phase = 0;
        int issued = 0;       // stages passed, for the drain below
        uint32_t ahead = 0u;  // leader, lane 0: the next tile
        bool synced = false;  // lane 0: wait_dispatch has returned
        // Leader: the next tile is taken when a tile starts and handed out
        // kHandOutStages before its last stage (handed out after the last stage,
        // every tile began with 1.4 us in which nothing was loaded; taken a tile
        // earlier, the CTAs ended less evenly, 212 -> 216 us a decode step).
        Tile t, next;
        auto push = [&](int i, Tile &e) {
            const int slot = i % kTQ;
            if (lane == 0) {
                if (!mbar_wait(tq_empty_bar(slot), ((uint32_t)(i / kTQ) & 1u) ^ 1u, &s_abort, p.status) || s_abort)
                    e.flags |= kTileEnd;
                const uint4 x = make_uint4((uint32_t)e.flags, (uint32_t)e.g, (uint32_t)e.m_tile, (uint32_t)e.m0);
                const uint4 y = make_uint4((uint32_t)e.n0, (uint32_t)e.rows, (uint32_t)e.row_base, (uint32_t)e.nkb);
                const uint32_t a = smem_u32(&s_tq[slot]);
                st_shared_v4(a, x);
                st_shared_v4(a + 16, y);
                mbar_arrive(tq_full_bar(slot));
                st_async_32(dsmem_addr(a, 1), x, y, dsmem_addr(tq_full_bar(slot), 1));
            }
            e.flags = __shfl_sync(~0u, e.flags, 0);
        };
        if (rank == 0) {
            t = decode_tile<kRoute>(p, tt, G, pair, total, lane);
            push(0, t);
        }
        for (int qi = 0;; ++qi) {
            if (rank == 0) {
                if (t.flags & kTileEnd) break;
                if (lane == 0) {
                    if (!synced) synced = wait_dispatch();
                    ahead = synced ? (uint32_t)pairs + atomicAdd(p.tile_ctr, 1u) : (uint32_t)total;
                }
            } else if (!next_tile(qi, t)) {
                break;
            }
            const bool gather = t.gather();
            const CUtensorMap *tmap = !t.down() ? maps.tok[kGateUp] : (t.shared() ? maps.tok_sh : maps.tok[kDown]);
            const int tn = t.n(), trows = tn / 2;  // this CTA's token rows
            const int trow = t.row_base + t.m0 + rank * trows;
            int ok = 1;
            if (kRoute && gather && lane == 0) {  // the slot maps are read here
                if (!synced) synced = wait_dispatch();
                ok = synced;
            }
            if (t.down() && p.has_gu && lane == 0) {
                // a down tile after the gate/up tiles of the same launch: its
                // activation rows are complete once every gate/up epilogue
                // warp of their row tile has stored its part (bounded wait;
                // the weights are loaded meanwhile)
                const uint32_t need = 8u * (uint32_t)group_blocks(p, kGateUp, t.shared());
                const uint32_t *rp = p.ready + tt.mpre[t.g] + t.m_tile;
                if (!synced) synced = wait_dispatch();
                if (!synced) ok = 0;
                const unsigned long long t0 = globaltimer_ns();
                while (ok && ld_acquire_gpu(rp) < need) {
                    if (s_abort) { ok = 0; break; }
                    if (globaltimer_ns() - t0 > kWaitLimitNs) {
                        s_abort = 1;
                        if (p.status) atomicOr(p.status, PMPE_STATUS_PIPELINE_TIMEOUT);
                        ok = 0;
                        break;
                    }
                    __nanosleep(128);
                }
            }
            ok = __all_sync(~0u, ok);
            if (!ok) break;
            if (t.down() && p.has_gu) {
                // the async proxy reads what lane 0's acquire observed: the fence in
                // every lane, since any may be the one elected to issue the copies
                __syncwarp();
                asm volatile("fence.proxy.async.global;\n" ::: "memory");
            }
            auto advance = [&]() {
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            };
            // the boxes of this CTA's rows, largest first (1 to 3)
            const int b0 = __clz(trows) - 24, r0 = 128 >> b0;  // trows is 16 .. 128
            const int b1 = trows > r0 ? __clz(trows - r0) - 24 : -1, r1 = b1 < 0 ? 0 : r0 + (128 >> b1);
            const int b2 = b1 >= 0 && trows > r1 ? __clz(trows - r1) - 24 : -1;
            const int hand_out = max(t.nkb - kHandOutStages, 1);
            if (kRoute && gather) load_rows(t, 0);
            int kb = 0;
#pragma unroll 1
            for (int part = 0; part < 2 && ok; ++part) {
                const int end = part == 0 ? hand_out : t.nkb;
                if (part == 1 && rank == 0) {
                    next = decode_tile<kRoute>(p, tt, G, (int)min(__shfl_sync(~0u, ahead, 0), (uint32_t)total), total, lane);
                    push(qi + 1, next);
                }
                if (kRoute && gather) {
                    for (; kb < end; ++kb, advance()) {
                        if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = 0; break; }
                        if (elect_one()) {
                            if (rank == 0) mbar_expect_tx(full_bar(stage), (uint32_t)(tn * BK * 2));
                            gather_stage(stage, kb, tn / 16, 0);
                        }
                    }
                } else if (gather && rank == 1) {
                    for (; kb < end; ++kb, advance()) {
                        if (!warp_wait(gfull_bar(stage), phase)) { ok = 0; break; }
                        if (elect_one()) {
                            fence_proxy_async_smem();
                            mbar_arrive_remote(dsmem_addr(full_bar(stage), 0));
                        }
                    }
                } else if (gather) {
                    for (; kb < end; ++kb, advance()) {
                        if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = 0; break; }
                        if (elect_one()) mbar_arrive(full_bar(stage));
                    }
                } else {
                    for (; kb < end; ++kb, advance()) {
                        if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = 0; break; }
                        if (elect_one()) {
                            const uint32_t sT = sbase + stage * stage_bytes + kWBytes;
                            const uint32_t fb = dsmem_addr(full_bar(stage), 0);
                            if (rank == 0) {
                                mbar_expect_tx(full_bar(stage), (uint32_t)(tn * BK * 2));
                                if (!kRoute) mbar_arrive_count(full_bar(stage), 1 + kGatherThreads);  // nothing is gathered
                            }
                            tma_load_2d_pair_hint(sT, &tmap[b0], fb, kb * BK, trow, pol_keep);
                            if (b1 >= 0) tma_load_2d_pair_hint(sT + r0 * 128, &tmap[b1], fb, kb * BK, trow + r0, pol_keep);
                            if (b2 >= 0) tma_load_2d_pair_hint(sT + r1 * 128, &tmap[b2], fb, kb * BK, trow + r1, pol_keep);
                        }
                    }
                }
            }
            issued += t.nkb;
            if (!ok) break;
            if (rank == 0) t = next;
        }
        // drain: every copy of the pair has landed before its CTAs exit (the
        // last use of each stage).  No lane polls before the elected one has
        // issued its last copies.
        __syncwarp();
        for (int s = 0; s < nst && rank == 0 && issued > 0; ++s) {
            if (issued < nst && s >= stage) break;
            const uint32_t last = s < stage ? phase : phase ^ 1u;
            const unsigned long long t0 = globaltimer_ns();
            while (!mbar_try_wait(full_bar(s), last))
                if (globaltimer_ns() - t0 > kWaitLimitNs) break;
        }
    } else if (warp == kWeightWarp) {
        // ------------------------------------------------ weights through TMA
        // One 16 KB box a stage: 64 gate and 64 up rows, or 128 output columns'
        // rows.  (The drain above covers these copies.)
        int stage = 0;
        uint32_t phase = 0;
        int ok = 1;
        Tile t;
        for (int qi = 0; next_tile(qi, t); ++qi) {
            const int q = t.shared() ? 2 : (t.g < p.E_pub ? 0 : 1);
            const int ei = t.shared() ? 0 : (q == 0 ? t.g : t.g - p.E_pub);
            const bool gu = !t.down(), two = p.gu_two_boxes[q];
            const uint64_t wpol = (t.flags & kTileManyRows) ? pol_normal : pol_stream;
            // shared gate/up: n0 spans E_sh * I rows; shared down: the experts
            // one after another along K
            int y = gu ? ei * p.I + t.n0 + rank * 64 : ei * p.H + t.n0 + rank * 128;
            const int kend = gu ? p.H : p.I;
            int x = 0;
            for (int kb = 0; kb < t.nkb; ++kb) {
                if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = 0; break; }
                if (elect_one()) {
                    const uint32_t sW = sbase + stage * stage_bytes;
                    const uint32_t fb = dsmem_addr(full_bar(stage), 0);
                    if (rank == 0) mbar_expect_tx(full_bar(stage), 2u * kWBytes);
                    if (!gu) {
                        tma_load_2d_pair_hint(sW, &maps.down[q], fb, x, y, wpol);
                    } else if (!two) {
                        tma_load_3d_pair_hint(sW, &maps.gu[q], fb, x, y, 0, wpol);
                    } else {
                        tma_load_2d_pair_hint(sW, &maps.gate[q], fb, x, y, wpol);
                        tma_load_2d_pair_hint(sW + kWBytes / 2, &maps.up[q], fb, x, y, wpol);
                    }
                }
                x += BK;
                if (x == kend) { x = 0; y += p.H; }
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            }
            if (!ok) break;
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        int stage = 0, it = 0;
        uint32_t phase = 0;
        Tile t;
        for (int qi = 0; rank == 0 && next_tile(qi, t); ++qi) {
            const bool gather = t.gather();
            const uint32_t idesc = p.idesc | ((uint32_t)(t.n() >> 3) << 17);
            const int buf = it & 1;
            const uint32_t use = (uint32_t)(it >> 1) & 1u;
            ++it;
            if (!warp_wait(tempty_bar(buf), use ^ 1u)) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * kAccCols);
            // The warp's own work per stage must stay below the 512 clocks of
            // four full MMAs: the next stage's barrier is tested (without
            // waiting) before this stage's MMAs are issued.
            int ok = 1;
            bool ready = false;
            for (int kb = 0; kb < t.nkb; ++kb) {
                if (!__all_sync(~0u, ready || mbar_wait(full_bar(stage), phase, &s_abort, p.status))) { ok = 0; break; }
                // rows this CTA's gather warps copied (generic proxy, complete
                // when the barrier's phase completed) are read by the tensor
                // cores through the async proxy
                if (!kRoute && gather) fence_proxy_async_smem();
                tc_fence_after();
                const uint32_t eb = empty_bar(stage);
                const uint32_t sW = sbase + stage * stage_bytes;
                const uint64_t ad = sw128_desc(sW), bd = sw128_desc(sW + kWBytes);
                if (++stage == nst) { stage = 0; phase ^= 1u; }
                ready = mbar_test_wait(full_bar(stage), phase);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)  // +32 bytes of K per step inside the swizzle row
                        tc_mma_pair(d_tmem, ad + 2 * k, bd + 2 * k, idesc, (kb | k) != 0);
                    tc_commit_pair(eb);
                    if (kb == t.nkb - 1) tc_commit_pair(tfull_bar(buf));
                }
                __syncwarp();
            }
            if (!ok) break;
        }
        // the leader's last commit: its MMAs and every commit before (whose
        // arrivals reach both CTAs) are done before either CTA exits
        if (elect_one()) {
            if (rank == 0) tc_commit_pair(done_bar);
            const unsigned long long t0 = globaltimer_ns();
            while (!mbar_try_wait(done_bar, 0))
                if (globaltimer_ns() - t0 > kWaitLimitNs) break;
        }
    } else if (warp >= 2 && warp < 6) {
        // ------------------------------------------------ epilogue
        const int quarter = warp & 3;  // TMEM lanes this warp may access
        const uint32_t stage0 = sbase + kRingBytes;
        const uint32_t own = stage0 + quarter * kStageOutBytes;            // this warp's two 2 KB buffers
        const uint32_t partner = stage0 + (quarter ^ 2) * kStageOutBytes;  // those of the warp of the same columns
        const uint32_t roww = stage0 + 4 * kStageOutBytes + quarter * kRowWBytes;
        int it = 0;
        bool synced = false;  // wait_dispatch has returned (every lane acquires)
        for (int qi = 0;; ++qi) {
            Tile t;
            int ok = next_tile(qi, t);
            const int buf = it & 1;
            const uint32_t use = (uint32_t)(it >> 1) & 1u;
            ++it;
            if (ok && !synced) ok = synced = __all_sync(~0u, wait_dispatch());
            if (ok) {
                if (t.down() && !t.shared()) {  // the rows' routing weights, ahead of the accumulator
                    float w[kMaxN / 32];
#pragma unroll
                    for (int c = 0; c < kMaxN / 32; ++c) {
                        const int r = c * 32 + lane;
                        w[c] = r < t.rows ? p.w_of_slot[t.row_base + t.m0 + r] : 0.f;
                    }
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < kMaxN / 32; ++c) st_shared_f32(roww + (c * 32 + lane) * 4, w[c]);
                    __syncwarp();
                }
                // one lane waits, the warp follows: tcgen05.ld below is warp-collective
                if (lane == 0) ok = mbar_wait(tfull_bar(buf), use, &s_abort, p.status) ? 1 : 0;
                ok = __shfl_sync(~0u, ok, 0);
            }
            // the four warps go on together (they meet at barriers inside a tile) or stop together
            if (!named_barrier_all(3, 128, ok)) break;
            tc_fence_after();
            const bool gu = !t.down(), shared = t.shared();
            const TcPhase &ph = p.ph[gu ? kGateUp : kDown];
            const int nch = t.n() / 32;
            const int row0 = t.row_base + t.m0;  // slot (shared: token) of the tile's first token row
            const uint32_t taddr = tmem_base + (uint32_t)(buf * kAccCols) + ((uint32_t)(quarter * 32) << 16);
            // Each chunk of 32 tokens is read as two 16-lane fragments (tmem_frag16):
            // v[h][4 j + q] is column 16 h + 8 (q / 2) + lane / 4, token
            // 8 j + 2 (lane & 3) + (q & 1).  stmatrix.trans turns packed pairs of
            // tokens into rows of columns: half the shared-memory instructions of a
            // transpose by 32-bit stores from one column per thread.
            const int srow = lane & 7, scol = lane >> 3;  // stmatrix: this lane's row of matrix scol
            if (gu) {
                const bool first = quarter < 2;  // this warp computes tokens 0-15 of a chunk, its partner 16-31
                const bool gate = first != (p.up_first[shared ? 2 : (t.g < p.E_pub ? 0 : 1)] != 0);
                const int col = t.n0 + rank * 64 + (quarter & 1) * 32;  // this warp's columns
                const int ldc = shared ? p.E_sh * p.I : p.I;
                bf16 *crow = (shared ? ph.C_shared : ph.C_routed) + (size_t)row0 * ldc + col + (lane & 3) * 8;
                const int ld2 = 2 * ldc;  // saved G | U: floats per row
                float *saved = p.saved_gu ? p.saved_gu + (shared ? (size_t)p.R * 2 * p.I : 0) + (size_t)row0 * ld2 +
                                                (gate ? 0 : ldc) + col + (lane & 7) * 4
                                          : nullptr;
#pragma unroll 1
                for (int c = 0; c < nch; ++c) {
                    const uint32_t xo = own + (uint32_t)((c & 1) * 2048), xp = partner + (uint32_t)((c & 1) * 2048);
                    float v[2][16];
                    tmem_frag16(taddr + c * 32, v[0]);
                    tmem_frag16(taddr + c * 32 + (16u << 16), v[1]);
                    tmem_ld_wait();
                    if (saved) {  // the FP32 accumulators for the backward, 16 tokens at a time
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) {  // h = i / 8, j = 2 hh + (i / 4) % 2, q = i % 4
                                const int tok = 8 * ((i >> 2) & 1) + 2 * (lane & 3) + (i & 1);
                                const int cc = 16 * (i >> 3) + 8 * ((i >> 1) & 1) + (lane >> 2);
                                st_shared_f32(xo + (tok * 32 + (cc ^ ((lane & 3) << 3))) * 4,
                                              v[i >> 3][8 * hh + (i & 7)]);
                            }
                            __syncwarp();
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int r = j * 4 + (lane >> 3), tok = c * 32 + hh * 16 + r;
                                const uint4 f = ld_shared_v4(xo + r * 128 + ((((lane & 7) * 4) ^ (((r >> 1) & 3) << 3)) * 4));
                                if (tok < t.rows) *reinterpret_cast<uint4 *>(saved + (size_t)tok * ld2) = f;
                            }
                            __syncwarp();
                        }
                    }
                    // each warp of the pair gives the other its values of the
                    // tokens that the other computes
                    float mine[16], other[16];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float *s = &v[i >> 1][(i & 1) * 4];  // tokens 0-15; + 8: tokens 16-31
#pragma unroll
                        for (int q = 0; q < 4; ++q) mine[4 * i + q] = first ? s[q] : s[8 + q];
                        st_shared_v4(xo + i * 512 + lane * 16,
                                     make_uint4(__float_as_uint(first ? s[8] : s[0]), __float_as_uint(first ? s[9] : s[1]),
                                                __float_as_uint(first ? s[10] : s[2]), __float_as_uint(first ? s[11] : s[3])));
                    }
                    named_barrier_sync(1 + (quarter & 1), 64);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint4 f = ld_shared_v4(xp + i * 512 + lane * 16);
                        other[4 * i] = __uint_as_float(f.x); other[4 * i + 1] = __uint_as_float(f.y);
                        other[4 * i + 2] = __uint_as_float(f.z); other[4 * i + 3] = __uint_as_float(f.w);
                    }
                    uint32_t pk[8];  // [h][j][q / 2]
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float a0 = silu_mul(gate ? mine[2 * i] : other[2 * i], gate ? other[2 * i] : mine[2 * i]);
                        const float a1 = silu_mul(gate ? mine[2 * i + 1] : other[2 * i + 1],
                                                  gate ? other[2 * i + 1] : mine[2 * i + 1]);
                        pk[i] = pack_bf16x2(a0, a1);
                    }
                    __syncwarp();
                    // transposed through the partner's buffer, which this warp has read
                    // and the partner fills again only after their next barrier
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int r = 8 * j + srow;
                        stmatrix_x4_trans(xp + r * 64 + ((scol ^ ((r >> 1) & 3)) << 4), pk[2 * j], pk[2 * j + 1], pk[4 + 2 * j],
                                          pk[5 + 2 * j]);
                    }
                    __syncwarp();
                    uint4 f[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int r = 8 * h + (lane >> 2);
                        f[h] = ld_shared_v4(xp + r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4));
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int tok = c * 32 + (first ? 0 : 16) + 8 * h + (lane >> 2);
                        if (tok < t.rows) st_global_hint(crow + (size_t)tok * ldc, f[h], pol_keep);
                    }
                }
            } else {
                // ---- down: y = w * (act W_down^T), BF16
                const int col = t.n0 + rank * 128 + quarter * 32;
                bf16 *crow = (shared ? ph.C_shared : ph.C_routed) + (size_t)row0 * p.H + col + (lane & 3) * 8;
#pragma unroll 1
                for (int c = 0; c < nch && col < p.H; ++c) {  // (a last block's second half may lie past H)
                    const uint32_t xo = own + (uint32_t)((c & 1) * 2048);
                    float v[2][16];
                    tmem_frag16(taddr + c * 32, v[0]);
                    tmem_frag16(taddr + c * 32 + (16u << 16), v[1]);
                    float2 w[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        w[j] = shared ? make_float2(1.f, 1.f) : ld_shared_f32x2(roww + (c * 32 + 8 * j + 2 * (lane & 3)) * 4);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int r = 8 * j + srow;
                        stmatrix_x4_trans(xo + r * 64 + ((scol ^ ((r >> 1) & 3)) << 4),
                                          pack_bf16x2(v[0][4 * j] * w[j].x, v[0][4 * j + 1] * w[j].y),
                                          pack_bf16x2(v[0][4 * j + 2] * w[j].x, v[0][4 * j + 3] * w[j].y),
                                          pack_bf16x2(v[1][4 * j] * w[j].x, v[1][4 * j + 1] * w[j].y),
                                          pack_bf16x2(v[1][4 * j + 2] * w[j].x, v[1][4 * j + 3] * w[j].y));
                    }
                    __syncwarp();
                    uint4 f[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int r = 8 * h + (lane >> 2);
                        f[h] = ld_shared_v4(xo + r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4));
                    }
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int tok = c * 32 + 8 * h + (lane >> 2);
                        if (tok < t.rows) *reinterpret_cast<uint4 *>(crow + (size_t)tok * p.H) = f[h];
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (rank == 0) mbar_arrive(tempty_bar(buf));
                else mbar_arrive_remote(dsmem_addr(tempty_bar(buf), 0));
            }
            // execution audit: rows this tile processed, counted where they
            // ran (by the leader of the pair, which runs them in weight block 0).
            // A row counts for its expert only if its token's route names this
            // expert (the route log is read back and checked, row by row); a
            // row that fails the check is a dispatch mismatch.  The per-token
            // private count follows the rows physically run.
            if (gu && rank == 0 && p.status) {
                if (!shared && t.n0 == 0) {
                    for (int c = quarter; c < nch; c += 4) {
                        const bool valid = c * 32 + lane < t.rows;
                        const int tok = valid ? p.tok_of_slot[row0 + c * 32 + lane] : -1;
                        bool routed = false;
                        if ((unsigned)tok < (unsigned)p.T) {
                            const int32_t *ti = p.topk_idx + (size_t)tok * p.k;
                            for (int j = 0; j < p.k; ++j) routed |= ti[j] == t.g;
                        }
                        if (valid && !routed) atomicOr(p.status, PMPE_STATUS_DISPATCH_MISMATCH);
                        const unsigned ok_rows = __ballot_sync(~0u, valid && routed);
                        if (lane == 0 && ok_rows) atomicAdd(&p.exec_rows[t.g], (unsigned)__popc(ok_rows));
                        if ((unsigned)tok < (unsigned)p.T && t.g >= p.E_pub) atomicAdd(&p.exec_priv_rows[tok], 1u);
                    }
                    // 128-row blocks of the expert that start in this row tile
                    if (lane == 0 && quarter == 0)
                        atomicAdd(&p.exec_tiles[t.g], (unsigned)((t.m0 + t.rows + kRowBlock - 1) / kRowBlock -
                                                                 (t.m0 + kRowBlock - 1) / kRowBlock));
                }
                if (shared && lane == 0 && quarter == 0 && (t.n0 % p.I) == 0)
                    atomicAdd(p.shared_rows, (unsigned)t.rows);
            }
            if (gu && p.has_down) {
                // release this warp's activation columns to the down tiles that read
                // them (through TMA, after an acquire and a proxy fence): the release
                // add follows the warp barrier, so it covers every lane's stores
                __syncwarp();
                if (lane == 0) {
                    asm volatile("fence.proxy.async.global;\n" ::: "memory");
                    grid_arrive(p.ready + tt.mpre[t.g] + t.m_tile);
                }
                __syncwarp();
            }
        }
    } else if (kRoute && warp == kGatherWarp) {
        // ------------------------------------------------ gather4 of the second half of the rows
        int stage = 0;
        uint32_t phase = 0;
        int ok = 1;
        bool synced = false;  // wait_dispatch has returned (every lane acquires)
        Tile t;
        for (int qi = 0; ok && next_tile(qi, t, true); ++qi) {
            if (!synced && !(synced = __all_sync(~0u, wait_dispatch()))) break;
            load_rows(t, 1);
            for (int kb = 0; kb < t.nkb; ++kb) {
                if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = 0; break; }
                if (elect_one()) gather_stage(stage, kb, t.n() / 16, 1);
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp >= kGatherWarp && warp < kWeightWarp) {
        // ------------------------------------------------ token row gather
        // This CTA's half of a routed gate/up tile's token rows: thread i of
        // a group's 128 copies 16-byte chunk (i & 7) of rows (i >> 3) + 16 j of
        // the group's stages (every other one: a stage costs a thread about
        // 600 clocks whatever its rows, more than its MMAs) into the 128-byte-swizzled token slot of the stage (chunk c of
        // row r at chunk c ^ (r & 7)); a warp instruction covers four whole
        // 128-byte rows.  Rows past the tile's rows are zero-filled.  Each
        // thread's copies of a stage arrive on the leader's full barrier, or the
        // other CTA's gfull barrier, when they complete (cp.async.mbarrier.arrive), so the threads never wait for
        // their own copies: up to the whole ring is in flight.
        const int gi = (tid - 192) & 127, group = (warp - kGatherWarp) >> 2;
        const int chunk = gi & 7, row0 = gi >> 3;
        int stage = 0;
        uint32_t phase = 0;
        int turn = 0;                        // the group whose stage is next
        auto gbar = [&](int s) { return rank == 0 ? full_bar(s) : gfull_bar(s); };
        bool ok = true;
        bool synced = false;                 // wait_dispatch has returned (every lane acquires)
        Tile t;
        for (int qi = 0; ok && next_tile(qi, t, true); ++qi) {
            if (!synced && !(synced = __all_sync(~0u, wait_dispatch()))) break;
            // this thread's rows: their token rows in the hidden states
            const int nj = t.n() / 32, first = rank * (t.n() / 2);
            const bf16 *src[8];
            uint32_t nbytes[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int r = first + row0 + 16 * j;
                const int tok = j < nj && r < t.rows ? p.tok_of_slot[t.row_base + t.m0 + r] : -1;
                const bool in = (unsigned)tok < (unsigned)p.T;
                src[j] = p.hidden + (in ? (size_t)tok * p.H : 0) + chunk * 8;
                nbytes[j] = in ? 16u : 0u;
            }
            for (int kb = 0; kb < t.nkb; ++kb) {
                if (turn == group) {
                    int free_ = 1;
                    if (lane == 0) free_ = mbar_wait(empty_bar(stage), phase ^ 1u, &s_abort, p.status) ? 1 : 0;
                    free_ = __shfl_sync(~0u, free_, 0);
                    if (!free_) { ok = false; break; }
                    const uint32_t sT = sbase + stage * stage_bytes + kWBytes;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int r = row0 + 16 * j;
                        if (j < nj)
                            cp_async16_zfill(sT + r * 128 + ((chunk ^ (r & 7)) << 4), src[j] + kb * BK, nbytes[j],
                                             pol_keep);
                    }
                    cp_async_arrive_noinc(gbar(stage));
                }
                turn = turn == kGatherGroups - 1 ? 0 : turn + 1;
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            }
        }
        cp_async_wait<0>();
    }

    // every warp reconverges before the cluster barrier (a warp-aligned
    // barrier; the single-thread roles above diverge from their warps): the
    // pair's MMAs, copies, barrier arrivals and TMEM reads are done
    __syncwarp();
    tc_fence_before();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
    if (kRoute && p.fuse_combine) {
        // ---- the weighted combine (Sec. 3.1), as combine_kernel sums it:
        // j ascending, then the shared experts, in FP32, once every CTA has met
        // at the last grid barrier (whose release covers the epilogues' stores).
        if (grid_barrier(p.bar_d, gridDim.x, &s_abort, p.status)) {
            const bf16 *y = p.ph[kDown].C_routed;
            const bf16 *y_sh = p.E_sh > 0 ? p.ph[kDown].C_shared : nullptr;
            const int nv = p.H / 8;
            for (int t = (int)blockIdx.x; t < p.T; t += (int)gridDim.x) {
                for (int c = tid; c < nv; c += kThreads) {
                    float acc[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) acc[q] = 0.f;
                    for (int j = 0; j < p.k; ++j) {
                        int slot = p.slot_of_w[(size_t)t * p.k + j];
                        if ((unsigned)slot >= (unsigned)p.R) slot = 0;  // only after a dispatch mismatch (status set)
                        const uint4 v = *reinterpret_cast<const uint4 *>(y + (size_t)slot * p.H + (size_t)c * 8);
                        const __nv_bfloat162 *b = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 f = __bfloat1622float2(b[q]);
                            acc[2 * q] += f.x;
                            acc[2 * q + 1] += f.y;
                        }
                    }
                    if (y_sh) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(y_sh + (size_t)t * p.H + (size_t)c * 8);
                        const __nv_bfloat162 *b = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 f = __bfloat1622float2(b[q]);
                            acc[2 * q] += f.x;
                            acc[2 * q + 1] += f.y;
                        }
                    }
                    uint4 o;
                    o.x = pack_bf16x2(acc[0], acc[1]);
                    o.y = pack_bf16x2(acc[2], acc[3]);
                    o.z = pack_bf16x2(acc[4], acc[5]);
                    o.w = pack_bf16x2(acc[6], acc[7]);
                    reinterpret_cast<uint4 *>(p.out + (size_t)t * p.H)[c] = o;
                }
            }
        }
    }
}

// ------------------------------------------------------------ host side

// Tensor maps of the token rows at `ptr` [rows, cols], by box rows.
bool encode_tokens(CUtensorMap *m, const bf16 *ptr, int cols, uint64_t rows)
{
    bool ok = true;
    for (int b = 0; b < kTokBoxes; ++b) ok &= encode_2d(&m[b], ptr, cols, rows, 128u >> b);
    return ok;
}

// Outputs and tensor maps of one GEMM (`mode`) of a launch.
bool fill_phase(const Ctx &c, int mode, TcParams &p, TcMaps &maps)
{
    const Shape &s = c.s;
    const uint64_t R = (uint64_t)s.T * s.k, T = (uint64_t)s.T;
    const bool gu = mode == kGateUp;
    bool ok = true;
    p.ph[mode].C_routed = gu ? c.act : c.y;
    p.ph[mode].C_shared = gu ? c.act_sh : c.y_sh;
    for (int q = 0; q < (s.E_sh > 0 ? 3 : 2); ++q) {
        const uint64_t n = (uint64_t)(q == 0 ? s.E_pub : q == 1 ? s.E_priv : s.E_sh);
        if (!gu) {
            ok &= encode_2d(&maps.down[q], c.down[q], s.I, n * s.H, 128);
            continue;
        }
        bool up_first;
        p.gu_two_boxes[q] = !encode_gate_up(&maps.gu[q], c.gate[q], c.up[q], s.H, n * s.I, &up_first);
        p.up_first[q] = up_first;
        if (p.gu_two_boxes[q]) {
            p.up_first[q] = 0;
            ok &= encode_2d(&maps.gate[q], c.gate[q], s.H, n * s.I, 64);
            ok &= encode_2d(&maps.up[q], c.up[q], s.H, n * s.I, 64);
        }
    }
    if (gu) ok &= encode_2d(&maps.hidden, c.hidden, s.H, T, 1);
    if (gu && s.E_sh > 0) ok &= encode_tokens(maps.tok[kGateUp], c.hidden, s.H, T);
    if (!gu) ok &= encode_tokens(maps.tok[kDown], c.act, s.I, R);
    if (!gu && s.E_sh > 0) ok &= encode_tokens(maps.tok_sh, c.act_sh, s.E_sh * s.I, T);
    return ok;
}

// The dynamic shared-memory limit of one instantiation, raised once per device.
template <bool kRoute>
cudaError_t ensure_tc_smem()
{
    static std::atomic<int> smem_limit[64];
    return ensure_dynamic_smem(expert_gemm_tc_kernel<kRoute>, kDynSmem, smem_limit);
}

// CTAs of the launch: one pair for every two SMs.
int tc_grid(const Ctx &c) { return c.num_sms / 2 * 2; }

// One persistent launch of the gate/up tiles, the down tiles, or both (and,
// with fuse_dispatch, the dispatch before them).
cudaError_t launch_tc(const Ctx &c, bool gu, bool down, bool fuse_dispatch = false, bool fuse_route = false,
                      bool fuse_combine = false)
{
    const Shape &s = c.s;
    TcParams p;
    TcMaps maps;
    memset(&p, 0, sizeof(p));
    memset(&maps, 0, sizeof(maps));
    p.has_gu = gu;
    p.has_down = down;
    p.E = s.E(); p.E_pub = s.E_pub; p.E_sh = s.E_sh; p.T = s.T; p.H = s.H; p.I = s.I; p.R = s.T * s.k; p.k = s.k;
    p.idesc = make_idesc(256, 0);
    p.offsets = c.offsets;
    p.w_of_slot = c.w_of_slot;
    p.tok_of_slot = c.tok_of_slot;
    p.topk_idx = c.idx;
    p.hidden = c.hidden;
    p.ready = c.gemm_ready;
    if (gu && s.T <= kRouteMaxTokens && (long long)s.H * s.I >= (1ll << 20)) {
        // at most T rows per expert: one row tile each.  (Not for small experts,
        // as in the tiny layer: the launch is too short to gain from it; and not
        // below a pick for every five experts, when most of the prefetched weights
        // would not be used.  Qwen3 shape: T = 1 42.8 us with it, 41.9 without;
        // T = 4 63.2 both; T = 8 89.8 and 90.4; T = 64 211.3 and 213.8.)
        p.prefetch_tiles = 5 * s.T * s.k >= s.E() ? std::min(s.E() * (s.I / 128), kPrefetchTiles) : 0;
        for (int q = 0; q < 2; ++q) {
            p.gate_w[q] = c.gate[q];
            p.up_w[q] = c.up[q];
        }
    }
    p.tile_ctr = c.gemm_ready + gemm_ready_words(s) - 2;
    p.exec_rows = c.audit.exec_rows;
    p.exec_tiles = c.audit.exec_tiles;
    p.exec_priv_rows = c.audit.exec_priv_rows;
    p.shared_rows = c.audit.shared_rows;
    p.status = c.audit.status;
    if (fuse_dispatch) {
        p.fuse_dispatch = 1;
        const size_t gu_bytes = (size_t)2 * s.I * s.H * 2;  // one expert's gate and up rows
        p.prefetch_experts = (int)std::min<size_t>(std::min<size_t>(kPrefillPrefetchBytes / gu_bytes,
                                                                    (size_t)kPrefillPrefetchExperts),
                                                   (size_t)s.E());
        for (int q = 0; q < 2; ++q) {
            p.gate_w[q] = c.gate[q];
            p.up_w[q] = c.up[q];
        }
        p.ticket = c.ticket;
        p.w_route = c.w;
        p.tile_counts = c.tile_counts;
        p.slots = router_slots(s.T);
        p.slots4 = router_slots4(s.T);
        p.counts_w = c.counts;
        p.offsets_w = c.offsets;
        p.slot_of_w = c.slot_of;
        p.tok_of_slot_w = c.tok_of_slot;
        p.w_of_slot_w = c.w_of_slot;
        p.grid_bar = c.gemm_ready + gemm_ready_words(s) - 1;
        p.clear_words = (int)gemm_ready_words(s) - 1;
    }
    if (fuse_route) {  // every counter cleared by clear_counters_kernel before this launch
        p.fuse_route = 1;
        p.renorm = s.renorm;
        p.policy = c.policy;
        p.router_w[0] = c.router_pub;
        p.router_w[1] = c.router_priv;
        p.z = reinterpret_cast<float *>(c.router_rows);  // the chunked router's scratch, unused here
        p.zpitch = std::max(s.E_pub, s.E_priv);
        p.idx_w = c.idx;
        p.ticket_w = c.ticket;
        p.w_w = c.w;
        p.tau_w = c.tau;
        p.tile_counts_w = c.tile_counts;
        p.route_count = c.audit.route_count;
        p.route_priv_rows = c.audit.route_priv_rows;
        p.slots = router_slots(s.T);
        p.slots4 = router_slots4(s.T);
        p.counts_w = c.counts;
        p.offsets_w = c.offsets;
        p.slot_of_w = c.slot_of;
        p.tok_of_slot_w = c.tok_of_slot;
        p.w_of_slot_w = c.w_of_slot;
        p.bar_a = c.gemm_ready + gemm_ready_words(s) - 4;
        p.bar_b = c.gemm_ready + gemm_ready_words(s) - 3;
        p.grid_bar = c.gemm_ready + gemm_ready_words(s) - 1;
        if (fuse_combine) {
            p.fuse_combine = 1;
            p.bar_d = c.gemm_ready + gemm_ready_words(s) - 5;
            p.out = c.out;
        }
    }
    bool ok = true;
    if (gu) ok &= fill_phase(c, kGateUp, p, maps);
    if (down) ok &= fill_phase(c, kDown, p, maps);
    if (gu) p.saved_gu = c.saved_gu;
    if (!ok) return cudaErrorInvalidValue;
    const cudaError_t err = fuse_route ? ensure_tc_smem<true>() : ensure_tc_smem<false>();
    if (err != cudaSuccess) return err;
    if (fuse_route)
        return launch_cluster_pdl(expert_gemm_tc_kernel<true>, 2, dim3(tc_grid(c)), dim3(kTcThreads<true>), kDynSmem, c.stream, p,
                                  maps);
    return launch_cluster_pdl(expert_gemm_tc_kernel<false>, 2, dim3(tc_grid(c)), dim3(kTcThreads<false>), kDynSmem, c.stream, p,
                              maps);
}

// Whether the persistent grid (one CTA per SM, in pairs) can be resident all
// at once: the down tiles of the gate/up + down launch wait for gate/up tiles
// that other pairs own, so every pair must run concurrently.  Cached per device.
template <bool kRoute>
bool pairs_fit(const Ctx &c)
{
    if (ensure_tc_smem<kRoute>() != cudaSuccess) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tc_grid(c));
    cfg.blockDim = dim3(kTcThreads<kRoute>);
    cfg.dynamicSmemBytes = kDynSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, expert_gemm_tc_kernel<kRoute>, &cfg) == cudaSuccess && 2 * n >= tc_grid(c);
}

static bool grid_fits(const Ctx &c)
{
    static std::atomic<int> fits[64];  // 0 unknown, 1 yes, 2 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    if (dev >= 0 && dev < 64 && fits[dev].load() != 0) return fits[dev].load() == 1;
    const bool ok = pairs_fit<false>(c) && pairs_fit<true>(c);
    if (dev >= 0 && dev < 64) fits[dev].store(ok ? 1 : 2);
    return ok;
}

}  // namespace

// The two GEMMs in separate launches (diagnostics, and the fallback when the
// persistent grid cannot be resident at once): each starts from tile 0.
cudaError_t launch_gateup(const Ctx &c)
{
    const cudaError_t err = cudaMemsetAsync(c.gemm_ready + gemm_ready_words(c.s) - 2, 0, sizeof(uint32_t), c.stream);
    return err == cudaSuccess ? launch_tc(c, true, false) : err;
}

cudaError_t launch_down(const Ctx &c)
{
    const cudaError_t err = cudaMemsetAsync(c.gemm_ready + gemm_ready_words(c.s) - 2, 0, sizeof(uint32_t), c.stream);
    return err == cudaSuccess ? launch_tc(c, false, true) : err;
}

// The dispatch can run inside the persistent launch when that launch's grid
// is resident at once (its grid barrier) and the prefix table of the router
// tiles' counts fits its ring.  For small experts (fewer than 2^20 weights a
// projection: the tiny test layer) the launch is short and the grid barrier
// costs more than the dispatch kernel it saves (40.1 vs 38.2 us a step).
bool experts_fuse_dispatch(const Ctx &c)
{
    return (long long)c.s.H * c.s.I >= (1ll << 20) && grid_fits(c) &&
           fused_dispatch_smem(c.s.E(), router_slots(c.s.T)) <= (size_t)kRingBytes;
}

// Routing in the expert launch: at most 128 tokens (one selection CTA each,
// all resident with the persistent grid), the masked router of the method
// (not the unmasked control), pools of at most 256 experts (8 logits a lane
// in the selection), H <= 2048 (a lane holds at most 8 16-byte pieces of a
// row in registers for the logits), and the dispatch's per-expert masks fit
// the ring.
bool experts_fuse_route(const Ctx &c)
{
    const Shape &s = c.s;
    return s.T >= 1 && s.T <= kRouteMaxTokens && s.T <= tc_grid(c) && !c.unmasked && s.H <= kRouteMaxH &&
           s.E_pub <= 256 && s.E_priv <= 256 && (size_t)s.E() * 24u <= (size_t)kRingBytes &&
           grid_fits(c);
}

__global__ void clear_counters_kernel(uint32_t *w, int n)
{
    pdl_trigger();
    pdl_wait();  // the previous forward on this workspace has finished with them
    for (int i = threadIdx.x; i < n; i += blockDim.x) w[i] = 0u;
}

// The forward's launches when the expert launch routes: the counters
// (readiness, tile, barriers) cleared by a one-block kernel, then the
// persistent launch (routing, dispatch order, gate/up and down).
cudaError_t launch_experts_routed(const Ctx &c, bool combine)
{
    const cudaError_t err =
        launch_pdl(clear_counters_kernel, dim3(1), dim3(256), 0, c.stream, c.gemm_ready, (int)gemm_ready_words(c.s));
    return err == cudaSuccess ? launch_tc(c, true, true, false, true, combine) : err;
}

cudaError_t launch_experts(const Ctx &c, bool zero_ready, bool fuse_dispatch)
{
    if (!grid_fits(c)) {  // the two GEMMs one after the other: no cross-CTA wait
        const cudaError_t err = launch_gateup(c);
        return err == cudaSuccess ? launch_down(c) : err;
    }
    if (zero_ready && !fuse_dispatch) {
        const cudaError_t err = cudaMemsetAsync(c.gemm_ready, 0, sizeof(uint32_t) * gemm_ready_words(c.s), c.stream);
        if (err != cudaSuccess) return err;
    }
    return launch_tc(c, true, true, fuse_dispatch);
}

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    });
    return fn;
}

// 2-D tensor map over a row-major [rows, cols] matrix of `type` elements of
// `elem_bytes` bytes, box = box_cols x box_rows, zero fill out of bounds.
static bool encode_2d_typed(CUtensorMap *m, CUtensorMapDataType type, uint32_t elem_bytes, const void *ptr,
                            uint64_t cols, uint64_t rows, uint32_t box_cols, uint32_t box_rows,
                            CUtensorMapSwizzle swizzle)
{
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * elem_bytes};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, type, 2, const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_3d_blocks(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_rows, uint32_t nblocks)
{
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {64, rows, cols / 64};
    const cuuint64_t strides[2] = {cols * 2, 128};  // row pitch; 64-column blocks 128 bytes apart
    const cuuint32_t box[3] = {64, box_rows, nblocks};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_gate_up(CUtensorMap *m, const bf16 *gate, const bf16 *up, uint64_t cols, uint64_t rows, bool *up_first)
{
    *up_first = up < gate;
    const bf16 *lo = *up_first ? up : gate, *hi = *up_first ? gate : up;
    const uint64_t apart = (uint64_t)((uintptr_t)hi - (uintptr_t)lo);
    auto fn = encode_fn();
    if (!fn || apart == 0 || apart >= (1ull << 40)) return false;  // a map's strides are below 2^40 bytes
    const cuuint64_t dims[3] = {cols, rows, 2};
    const cuuint64_t strides[2] = {cols * 2, apart};
    const cuuint32_t box[3] = {64, 64, 2};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16 *>(lo), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_2d_box(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_cols,
                   uint32_t box_rows, CUtensorMapSwizzle swizzle)
{
    return encode_2d_typed(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ptr, cols, rows, box_cols, box_rows, swizzle);
}

bool encode_2d_f32(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_cols,
                   uint32_t box_rows, CUtensorMapSwizzle swizzle)
{
    return encode_2d_typed(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ptr, cols, rows, box_cols, box_rows, swizzle);
}

bool encode_2d(CUtensorMap *m, const void *ptr, uint64_t cols, uint64_t rows, uint32_t box_rows)
{
    return encode_2d_box(m, ptr, cols, rows, 64u, box_rows, CU_TENSOR_MAP_SWIZZLE_128B);
}

uint32_t make_idesc(int M, int N)
{
    return (1u << 4)                    // D: FP32
           | (1u << 7)                  // A: BF16
           | (1u << 10)                 // B: BF16
           | ((uint32_t)(N >> 3) << 17) // N / 8
           | ((uint32_t)(M >> 4) << 24);// M / 16   (A and B K-major: transpose bits 15, 16 = 0)
}

uint32_t make_idesc_major(int M, int N, bool a_mn_major, bool b_mn_major)
{
    return make_idesc(M, N) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16);
}


}  // namespace pmpe
