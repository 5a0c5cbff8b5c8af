// Backward of the private branch on the 5th-generation tensor cores (G2,
// Sec. 2.2; Sec. 3.2 trains the private experts and the private router only).
// Three persistent grouped GEMM launches over the private experts, each in the
// TMA -> shared memory -> tcgen05.mma -> TMEM -> epilogue pipeline of the
// forward's expert GEMMs:
//
//   bwd_rows_pair_kernel<C = A B>   K = H (weights as M, an expert's rows as N):
//     Z = D W_down                  (D: the rows' upstream gradients; W_down read
//                                    MN-major; so dL/da = w Z) -> BF16
//   bwd_rows_pair_kernel<gate/up>   the same form, K = H:
//     G = A W_gate^T, U = A W_up^T  (A: the expert's dispatched rows; recomputed)
//   and in the epilogue, with Z read back, per row and column:
//     act = bf16(silu(G) U) (the forward's activation), dL/dw partial = sum Z act,
//     dG = w Z U silu'(G), dU = w Z silu(G)  -> BF16 [dG | dU];  w act -> BF16
//   Z, [dG | dU] and w act use a padded row layout: expert q's rows start at a
//   multiple of 128, and the rows past its count of the last two are zeros.
//
//   bwd_wgrad_tc_kernel   rows of an expert as the contracted K:
//     [dW_gate; dW_up]_q = [dG | dU]^T A     (M = 2I, N = H)
//     dW_down_q          = D^T (w act)        (M = H,  N = I)
//   both operands MN-major, read as stored (no transpose in memory); the zero
//   rows of the padded operand cancel what the other operand holds past the
//   expert's rows.  FP32 outputs.
//
// The same two row kernels, over all routed experts and the shared experts,
// and the pair launch dA = [dG | dU] [W_gate; W_up] give the gradient of
// the layer's input (launch_rows_z, launch_rows_gu, launch_rows_da).
//
// Every launch keeps 160 to 192 KB of operand stages in flight and two FP32
// accumulators, so the epilogue of one tile overlaps the MMAs of the next.  CTA roles (224 threads): warps 0 and 6 issue
// the TMA loads of the first and the second operand, warp 1 allocates TMEM and
// issues the MMAs, warps 2-5 drain TMEM (a warp's 32 lanes are 32 output columns
// in the row launches, 32 rows of a gradient in the weight gradients).  Warps 0, 1
// and 6 run their loops as whole warps, with one elected lane issuing (elect_one).  Every wait
// is bounded in time; on expiry the CTA records PMPE_STATUS_PIPELINE_TIMEOUT,
// stops, waits (bounded) for its copies and MMAs in flight, frees TMEM and exits.
#include <cuda.h>

#include <algorithm>
#include <cstring>

#include "pmpe_internal.cuh"
#include "tc_ptx.cuh"

namespace pmpe {
namespace {

constexpr int BM = 128;                        // MMA M (rows of a tile)
constexpr int BK = 64;                         // K per stage
constexpr int kABytes = BM * BK * 2;           // 16 KB
constexpr int kMnBlockBytes = 64 * BK * 2;     // one 64-element MN block of an MN-major operand: 8 KB
constexpr int kThreads = 224;
constexpr int kLoaders = 2;                    // loader warps 0 and 6: one operand each
constexpr int kPad = 128;                      // padded row layout: each expert starts at a multiple of 128

constexpr int kAccCols = 256;
constexpr int kTmemCols = 2 * kAccCols;

// Groups of a launch: the routed experts g0 .. g0 + G - 1 (rows = their
// dispatch slots), or G shared experts that each run every one of shared_T
// tokens.  Per group q: its rows, its first row relative to the first slot of
// expert g0 (0 for shared groups), its first row of the padded layout; and the
// tiles of the groups before q.
constexpr int kMaxGroups = 2 * kMaxPool;
struct GroupTable {
    int tiles[kMaxGroups + 1];
    int rows[kMaxGroups];
    int off[kMaxGroups];
    int pad[kMaxGroups];
};

// All threads: fill the table (routed groups from the forward's dispatch
// offsets).  tiles_per_row_block: tiles of a group per 128-row block (0 where the
// tiles are not read).
__device__ void build_groups(GroupTable &gt, const uint32_t *offsets, int g0, int G, int R, int shared_T,
                             int tiles_per_row_block)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int p0 = shared_T ? 0 : (int)min(offsets[g0], (uint32_t)R);
    for (int q = tid; q < G; q += blockDim.x) {
        int b = 0, e = shared_T;
        if (!shared_T) {
            b = min(max((int)offsets[g0 + q], p0), R);
            e = min(max((int)offsets[g0 + q + 1], b), R);
        }
        const int rows = e - b;
        gt.rows[q] = rows;
        gt.off[q] = b - p0;
        gt.tiles[q + 1] = ((rows + BM - 1) / BM) * tiles_per_row_block;
        gt.pad[q] = (rows + kPad - 1) / kPad * kPad;  // made exclusive prefix below
    }
    __syncthreads();
    if (warp < 2) {  // warp 0: inclusive scan of tiles; warp 1: exclusive scan of padded rows
        int carry = 0;
        for (int b = 0; b < G; b += 32) {
            const int q = b + lane;
            const int v = q < G ? (warp == 0 ? gt.tiles[q + 1] : gt.pad[q]) : 0;
            int x = v;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(~0u, x, off);
                if (lane >= off) x += y;
            }
            if (q < G) {
                if (warp == 0) gt.tiles[q + 1] = carry + x;
                else gt.pad[q] = carry + x - v;
            }
            carry += __shfl_sync(~0u, x, 31);
        }
        if (warp == 0 && lane == 0) gt.tiles[0] = 0;
    }
    __syncthreads();
}

// Bounded wait for the drain at exit, by a whole warp: every copy a loader issued
// has landed (the last use of each stage, after `issued` stages up to `stage` in
// `phase`).  The lanes meet first: lanes already polling can keep the elected lane
// from issuing the last copies that they wait for.
__device__ __forceinline__ void drain_stages(uint32_t bar0, int stages, int issued, int stage, uint32_t phase)
{
    __syncwarp();
    for (int s = 0; s < stages && issued > 0; ++s) {
        if (issued < stages && s >= stage) break;
        const unsigned long long t0 = globaltimer_ns();
        while (!mbar_try_wait(bar0 + 8u * s, s < stage ? phase : phase ^ 1u))
            if (globaltimer_ns() - t0 > kWaitLimitNs) break;
    }
}

// ------------------------------------------------------------- rows

enum { kArowsTight = 0, kArowsSlot = 1, kArowsPad = 2 };

// One launch of the row GEMMs: C = A B on CTA pairs (A K-major rows of K, B
// read MN-major from a weight tensor of the group's expert: K blocks below
// k_split from w0, the rest from w1; kb_rows rows of K per expert in those
// tensors; C BF16 [padded rows][N]), or the gate/up recompute (K = H) with the
// SwiGLU backward epilogue.
struct RowsParams {
    int E_pub, H, I, R;
    int g0, G, shared_T;  // the groups (see build_groups)
    int K, N;             // contracted size, output columns
    int kb_rows, k_split; // C = A B: K rows of B per expert; first K block taken from w1
    int a_rows;           // A row of a tile row: kArowsTight (relative to expert g0's first slot),
                          // kArowsSlot (the dispatch slot; the token for shared groups), kArowsPad
    const uint32_t *offsets;
    const float *w_of_slot;  // gate/up: routing weights per slot (shared groups: weight 1)
    const bf16 *zpad;     // gate/up: Z in the padded row layout [RP][I]
    float *gw_part;       // gate/up (routed, may be null): [R][I / 32] dL/dw partial per 32 columns
    int wact;             // saved gate/up: 1 to write w act for the private experts' rows
    int gemm_next;        // 1: another of these launches follows (see pdl_trigger's use)
    uint32_t *status;
    uint32_t idesc;
};

struct RowsTile {
    int q, m0, n0, n_tile, rows;
};

// Tile `tile` of the list, given its group lo.
__device__ __forceinline__ RowsTile rows_tile(const GroupTable &gt, int lo, int bn, int tile)
{
    RowsTile t;
    t.q = lo;
    const int mt = (gt.rows[lo] + BM - 1) / BM;
    const int local = tile - gt.tiles[lo];
    t.n_tile = local / mt;  // n-tile major inside a group: its m tiles share the weight slice
    const int m_tile = local - t.n_tile * mt;
    t.m0 = m_tile * BM;
    t.n0 = t.n_tile * bn;
    t.rows = min(BM, gt.rows[lo] - t.m0);
    return t;
}

__device__ __forceinline__ RowsTile decode_rows_thread(const GroupTable &gt, int G, int bn, int tile)
{
    int lo = 0, hi = G - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (gt.tiles[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    return rows_tile(gt, lo, bn, tile);
}

// Weight pool (0 public or shared, 1 private) and index inside it of group q.
__device__ __forceinline__ int2 group_weights(const RowsParams &p, int q)
{
    if (p.shared_T) return make_int2(0, q);
    const int e = p.g0 + q;
    return e >= p.E_pub ? make_int2(1, e - p.E_pub) : make_int2(0, e);
}

// SwiGLU backward of one element, from the gate and up accumulators g, u,
// the row's Z value z and routing weight w: a = bf16(silu(g) u) with the
// forward's arithmetic, dG = w z u silu'(g), dU = w z silu(g), and w a.
__device__ __forceinline__ void swiglu_bwd(float g, float u, float z, float w, float &a, float &dg, float &du,
                                           float &wa)
{
    const float den = 1.f + __expf(-g);
    const float silu = __fdividef(g, den);
    a = __bfloat162float(__float2bfloat16_rn(silu * u));
    const float sg = __fdividef(1.f, den);
    const float wz = w * z;
    dg = wz * u * sg * (1.f + g * (1.f - sg));
    du = wz * silu;
    wa = w * a;
}

// ------------------------------------------------------------- rows, CTA pairs

// Z and dA on CTA pairs with the weights as M and the tokens as N, as the
// forward's expert GEMMs: a tile is 256 output columns (128 a CTA) x up to 256
// rows of an expert (N a multiple of 32, half staged by each CTA), so that a
// K step stages 32 KB a CTA for what a single CTA's 128 x 256 tile stages 48 KB,
// and an expert's rows are padded to 32 instead of 128: Z 145 -> 101 us and dA
// 201 -> 180 us at the DeepSeek shape, T = 3000 (its shared experts 45 -> 28 and
// 53 -> 47), 119 -> 112 and 222 -> 199 us at Qwen3 T = 4096, where the weights'
// DRAM reads bound them.  The weights are read
// MN-major as stored.  Pair i takes tiles i, i + pairs, ...: tiles of all sizes,
// and the row tiles of a weight block at the same time.  (Contiguous runs split
// by the tiles' N took 318 us for dA at Qwen3 T = 4096: a tile of few tokens
// costs its weights' DRAM time, as much as a full one.)
constexpr int kPairMaxN = 256;
constexpr int kPairRing = 6 * 2 * kABytes;      // 6 stages at N = 256
constexpr int kPairMaxStages = 10;              // at N = 32
constexpr int kPairOutBytes = 4096;             // per epilogue warp: two 2 KB transpose buffers
constexpr int kPairRowWBytes = kPairMaxN * 4;   // per epilogue warp: the tile's routing weights
constexpr int kPairDynSmem = kPairRing + 4 * (kPairOutBytes + kPairRowWBytes) + 1024;
constexpr int kTokBoxes = 4;                    // token row boxes: 128, 64, 32, 16 rows

struct PairMaps {
    CUtensorMap tok[kTokBoxes];  // the contracted rows' operand (K-major), by box rows
    CUtensorMap w0[2], w1[2];    // per weight pool, 64 x 64 x 2 3-D boxes (MN-major); gate/up: 64-row boxes of
                                 // the gate and the up rows, where one box cannot hold both
    CUtensorMap gu[2];           // gate/up: 64 gate and 64 up rows (encode_gate_up)
};

// The gate/up recompute's outputs (GuOut) or C.
struct PairOut {
    bf16 *c;              // C [padded rows][N], or [dG | dU] [padded rows][2I]
    bf16 *wact;           // gate/up: w act [padded rows][I] (private experts' rows), or NULL
    uint8_t up_first[2], two_boxes[2];  // gate/up, per weight pool: the box's order; two boxes
};

struct PairTable {
    int tiles[kMaxGroups + 1];   // tiles of the places before L
    uint16_t order[kMaxGroups];  // the group at place L (all routed experts: pool_place; else L)
    int rows[kMaxGroups], off[kMaxGroups], pad[kMaxGroups];  // as GroupTable
    int nmax;                    // bit b: some tile has N = 32 (b + 1)
};

struct PairTile {
    int q, m0, n0, n, rows;
};

__device__ __forceinline__ int pair_row_tiles(int rows) { return (rows + kPairMaxN - 1) / kPairMaxN; }
__device__ __forceinline__ int pair_row_size(int rows, int mt) { return ((rows + mt - 1) / mt + 31) & ~31; }

// The last entry of a nondecreasing prefix that is <= x, by a whole warp.
__device__ __forceinline__ int prefix_find(const int *pre, int G, int x, int lane)
{
    int n = 0;
    for (int b = 0; b < G; b += 32) n += __popc(__ballot_sync(~0u, b + lane < G && pre[b + lane] <= x));
    return n - 1;
}

__device__ __forceinline__ PairTile decode_pair(const PairTable &pt, int G, int width, int tile, int lane)
{
    PairTile t;
    const int L = prefix_find(pt.tiles, G, tile, lane);
    t.q = pt.order[L];
    const int rows = pt.rows[t.q], mt = pair_row_tiles(rows), bm = pair_row_size(rows, mt);
    const int local = tile - pt.tiles[L], block = local / mt;  // block major: its row tiles share the weights
    t.m0 = (local - block * mt) * bm;
    t.n0 = block * width;
    t.rows = min(bm, rows - t.m0);
    t.n = (t.rows + 31) & ~31;
    return t;
}

// All threads: the table of a launch over `blocks` column blocks a group.
__device__ void build_pairs(PairTable &pt, const uint32_t *offsets, int g0, int G, int E_pub, int R, int shared_T, int blocks)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int p0 = shared_T ? 0 : (int)min(offsets[g0], (uint32_t)R);
    if (tid == 0) pt.nmax = 0;
    __syncthreads();
    int nmax = 0;
    for (int q = tid; q < G; q += blockDim.x) {
        int b = 0, e = shared_T;
        if (!shared_T) {
            b = min(max((int)offsets[g0 + q], p0), R);
            e = min(max((int)offsets[g0 + q + 1], b), R);
        }
        const int rows = e - b, mt = pair_row_tiles(rows), bm = mt ? pair_row_size(rows, mt) : 0;
        if (mt) nmax |= 1 << (bm / 32 - 1);
        pt.rows[q] = rows;
        pt.off[q] = b - p0;
        const int L = !shared_T && g0 == 0 && interleave_pools(R, G) ? pool_place(q, E_pub, G - E_pub) : q;
        pt.order[L] = (uint16_t)q;
        pt.tiles[L + 1] = mt * blocks;
        pt.pad[q] = (rows + kPad - 1) / kPad * kPad;  // made exclusive prefix below
    }
    if (nmax) atomicOr(&pt.nmax, nmax);
    __syncthreads();
    if (warp < 2) {  // inclusive scan of tiles, exclusive scan of padded rows
        int *arr = warp == 0 ? pt.tiles + 1 : pt.pad;
        int carry = 0;
        for (int b = 0; b < G; b += 32) {
            const int q = b + lane;
            const int v = q < G ? arr[q] : 0;
            int x = v;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(~0u, x, off);
                if (lane >= off) x += y;
            }
            if (q < G) arr[q] = carry + (warp == 1 ? x - v : x);
            carry += __shfl_sync(~0u, x, 31);
        }
        if (warp == 0 && lane == 0) arr[-1] = 0;
    }
    __syncthreads();
}

// The rows of a 16-token x 32-column tile of BF16 pairs (pk[4 h + 2 j + q]:
// tokens 8 j + 2 (lane & 3), + 1 of column 16 h + 8 q + lane / 4) through 1 KB
// of shared memory: f[i] is this lane's 8 columns 8 (lane & 3) of token 8 i + lane / 4.
__device__ __forceinline__ void rows16(uint32_t buf, int lane, const uint32_t *pk, uint4 *f)
{
    const int srow = lane & 7, scol = lane >> 3;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = 8 * j + srow;
        stmatrix_x4_trans(buf + r * 64 + ((scol ^ ((r >> 1) & 3)) << 4), pk[2 * j], pk[2 * j + 1], pk[4 + 2 * j],
                          pk[5 + 2 * j]);
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = 8 * h + (lane >> 2);
        f[h] = ld_shared_v4(buf + r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4));
    }
}

// The SwiGLU backward of a gate/up tile by one epilogue warp: per chunk of 32
// tokens it computes 16 (first 16: warps 0-1) of its 32 columns, from its own
// accumulators and its partner's (exchanged as in the forward), with Z read
// row by row and turned into the accumulators' layout by ldmatrix.  dL/dw is
// summed over the 32 columns in the order of bwd_swiglu_saved_kernel (pairs of
// neighbouring columns, then pairs of pairs, ...), by a butterfly that halves
// the values it carries.  Rows past the expert's, to the end of its padded
// rows, are written as zeros.
__device__ __forceinline__ void gu_epilogue(const RowsParams &p, const PairOut &out, const PairTable &pt, const PairTile &t,
                                            uint32_t tb, uint32_t own, uint32_t partner, uint32_t roww, int rank,
                                            int quarter, int lane, int prow, int p0)
{
    const bool first = quarter < 2;
    const int2 wq = group_weights(p, t.q);
    const bool gate = first != (out.up_first[wq.x] != 0);
    const int col = t.n0 + rank * 64 + (quarter & 1) * 32, half = first ? 0 : 16;
    const int I = p.I, ch8 = (lane & 3) * 8, r4 = lane >> 2;
    const bool wa_out = out.wact != nullptr && !p.shared_T && p.g0 + t.q >= p.E_pub;
    bf16 *drow = out.c + (size_t)prow * 2 * I + col + ch8;
    bf16 *arow = wa_out ? out.wact + (size_t)prow * I + col + ch8 : nullptr;
    const bf16 *zrow = p.zpad + (size_t)prow * I + col + ch8;
    const int nch = t.n / 32;
    uint4 z[2];
    auto load_z = [&](int c) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int tok = c * 32 + half + 8 * h + r4;
            z[h] = c < nch && tok < t.rows ? *reinterpret_cast<const uint4 *>(zrow + (size_t)tok * I)
                                           : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    load_z(0);
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
        const uint32_t xo = own + (uint32_t)((c & 1) * 2048), xp = partner + (uint32_t)((c & 1) * 2048);
        float v[2][16];
        tmem_frag16(tb + c * 32, v[0]);
        tmem_frag16(tb + c * 32 + (16u << 16), v[1]);
        tmem_ld_wait();
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
        __syncwarp();
        // Z through the partner's buffer, which this warp has read (and the
        // partner fills again only after their next barrier)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = 8 * h + r4;
            st_shared_v4(xp + r * 64 + (((lane & 3) ^ ((r >> 1) & 3)) << 4), z[h]);
        }
        __syncwarp();
        uint32_t zf[2][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = 8 * j + (lane & 7);
            ldmatrix_x4_trans(zf[j][0], zf[j][1], zf[j][2], zf[j][3], xp + r * 64 + (((lane >> 3) ^ ((r >> 1) & 3)) << 4));
        }
        load_z(c + 1);
        uint32_t pg[8], pu[8], pa[8];  // [4 h + 2 j + q / 2]
        float s[16];                   // z a: [8 j + 4 (token parity) + 2 h + q / 2]
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 w2 = ld_shared_f32x2(roww + (c * 32 + half + 8 * j + 2 * (lane & 3)) * 4);
            const int tok = c * 32 + half + 8 * j + 2 * (lane & 3);
            const bool v0 = tok < t.rows, v1 = tok + 1 < t.rows;
#pragma unroll
            for (int a = 0; a < 4; ++a) {  // column group 8 a: h = a / 2, q / 2 = a & 1
                const int i = 4 * (2 * (a >> 1) + j) + 2 * (a & 1);
                const float2 zz = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&zf[j][a]));
                float act, dg[2], du[2], wa[2];
                swiglu_bwd(gate ? mine[i] : other[i], gate ? other[i] : mine[i], zz.x, w2.x, act, dg[0], du[0], wa[0]);
                s[8 * j + a] = __fmul_rn(zz.x, act);
                swiglu_bwd(gate ? mine[i + 1] : other[i + 1], gate ? other[i + 1] : mine[i + 1], zz.y, w2.y, act, dg[1],
                           du[1], wa[1]);
                s[8 * j + 4 + a] = __fmul_rn(zz.y, act);
                if (!v0) dg[0] = du[0] = wa[0] = 0.f;
                if (!v1) dg[1] = du[1] = wa[1] = 0.f;
                const int o = 4 * (a >> 1) + 2 * j + (a & 1);
                pg[o] = pack_bf16x2(dg[0], dg[1]);
                pu[o] = pack_bf16x2(du[0], du[1]);
                pa[o] = pack_bf16x2(wa[0], wa[1]);
            }
        }
        __syncwarp();  // Z has been read
        uint4 f[2], f2[2];
        rows16(xp, lane, pg, f);
        rows16(xp + 1024, lane, pu, f2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            bf16 *d = drow + (size_t)(c * 32 + half + 8 * h + r4) * 2 * I;
            *reinterpret_cast<uint4 *>(d) = f[h];
            *reinterpret_cast<uint4 *>(d + I) = f2[h];
        }
        if (wa_out) {
            __syncwarp();
            rows16(xp, lane, pa, f);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<uint4 *>(arow + (size_t)(c * 32 + half + 8 * h + r4) * I) = f[h];
        }
        if (p.gw_part) {
            // over the 8 columns of each group (lane / 4): at each level a lane
            // keeps the half of its values that its bit names
            float a8[8], a4[4], a2[2];
#pragma unroll
            for (int i = 0; i < 8; ++i) {  // keep token octet j = bit 2
                const float keep = (lane & 4) ? s[8 + i] : s[i], give = (lane & 4) ? s[i] : s[8 + i];
                a8[i] = __fadd_rn(keep, __shfl_xor_sync(~0u, give, 4));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {  // keep token parity = bit 3
                const float keep = (lane & 8) ? a8[4 + i] : a8[i], give = (lane & 8) ? a8[i] : a8[4 + i];
                a4[i] = __fadd_rn(keep, __shfl_xor_sync(~0u, give, 8));
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {  // keep column groups 0-1 or 2-3 = bit 4
                const float keep = (lane & 16) ? a4[2 + i] : a4[i], give = (lane & 16) ? a4[i] : a4[2 + i];
                a2[i] = __fadd_rn(keep, __shfl_xor_sync(~0u, give, 16));
            }
            const float b = __fadd_rn(a2[0], a2[1]);
            const float gw = __fadd_rn(b, __shfl_xor_sync(~0u, b, 16));
            const int tok = c * 32 + half + ((lane & 4) ? 8 : 0) + 2 * (lane & 3) + ((lane & 8) ? 1 : 0);
            if (lane < 16 && tok < t.rows)
                p.gw_part[(size_t)(p0 + pt.off[t.q] + t.m0 + tok) * (I / 32) + col / 32] = gw;
        }
    }
    if (t.m0 + t.rows == pt.rows[t.q]) {  // the expert's last rows: zeros to the end of its padded rows
        const int end = (pt.rows[t.q] + kPad - 1) / kPad * kPad - t.m0;
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        for (int r = t.n + r4 + (first ? 0 : 8); r < end; r += 16) {
            *reinterpret_cast<uint4 *>(drow + (size_t)r * 2 * I) = zero;
            *reinterpret_cast<uint4 *>(drow + (size_t)r * 2 * I + I) = zero;
            if (wa_out) *reinterpret_cast<uint4 *>(arow + (size_t)r * I) = zero;
        }
    }
}

// kGU: the gate/up recompute with the SwiGLU backward (tiles of 128 columns: each
// CTA 64 gate and the same 64 up columns, as the forward's); else C = A B.
template <bool kGU>
__global__ void __launch_bounds__(kThreads, 1) bwd_rows_pair_kernel(const RowsParams p, const PairOut out,
                                                                    const __grid_constant__ PairMaps maps)
{
    extern __shared__ uint8_t dsmem[];
    __shared__ PairTable pt;
    __shared__ __align__(8) uint64_t bars[2 * kPairMaxStages + 5];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;

    const int tid = threadIdx.x, warp = __shfl_sync(~0u, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)cluster_ctarank();  // 0: the leader, whose warp 1 issues the pair's MMAs
    const uint32_t sbase = (smem_u32(dsmem) + 1023u) & ~1023u;
    const uint32_t bar0 = smem_u32(bars);
    // full (both CTAs' copies) and tempty (both CTAs' epilogues) are the
    // leader's; empty and tfull are signalled in both CTAs by the commits
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kPairMaxStages + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * kPairMaxStages + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * kPairMaxStages + 2 + b); };
    const uint32_t done_bar = bar0 + 8u * (2 * kPairMaxStages + 4);

    if (tid == 0) {
        for (int s = 0; s < kPairMaxStages; ++s) { mbar_init(full_bar(s), kLoaders); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 8); }
        mbar_init(done_bar, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    // An early start of the next launch pays when it is another of these GEMMs
    // (private gradients at T = 1000 437 -> 429 us) and costs when it is not: a small
    // kernel's CTAs that started beside a GEMM's ran with the L1 its shared memory
    // left over (the T = 4096 step 1086 -> 1110 us with every launch triggering).
    // The recompute triggers always: dA follows it, but in the private gradients,
    // where the router's small kernels do and it makes no difference (425.3 us with
    // the trigger, 425.3 without).
    if (kGU || p.gemm_next) pdl_trigger();
    if (warp == 1) tmem_alloc_pair(smem_u32(&s_tmem), kTmemCols);
    pdl_wait();
    const int width = kGU ? 128 : 256;  // output columns of a tile
    build_pairs(pt, p.offsets, p.g0, p.G, p.E_pub, p.R, p.shared_T, (p.N + width - 1) / width);
    tc_fence_before();
    cluster_sync_all();  // both CTAs' barriers and TMEM are ready
    tc_fence_after();
    const uint32_t tmem_base = s_tmem;
    const int first = blockIdx.x >> 1, pairs = gridDim.x >> 1, last = pt.tiles[p.G];
    const int nkb = p.K / BK;
    const int p0 = p.shared_T ? 0 : (int)min(p.offsets[p.g0], (uint32_t)p.R);
    const int stage_bytes = kABytes + (pt.nmax ? 32 - __clz(pt.nmax) : 1) * (16 * BK * 2);
    const int nst = min(kPairMaxStages, kPairRing / stage_bytes);
    // A barrier wait by a whole warp, with one answer.
    auto warp_wait = [&](uint32_t bar, uint32_t parity) -> bool {
        return __all_sync(~0u, mbar_wait(bar, parity, &s_abort, p.status));
    };

    if (warp == 0 || warp == 6) {
        // ------------------------------------------------ TMA producers
        // warp 0: this CTA's half of the tile's token rows (at most three boxes
        // of 128 to 16 rows); warp 6: its 128 columns of the weights (16 KB).
        // Every copy completes on the leader's barrier, where the leader's
        // warps announce both CTAs' bytes.
        int stage = 0, issued = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = first; tile < last && ok; tile += pairs) {
            const PairTile t = decode_pair(pt, p.G, width, tile, lane);
            if (warp == 0) {
                const int trows = t.n / 2;
                const int y = (p.a_rows == kArowsPad ? pt.pad[t.q] : (p.a_rows == kArowsSlot ? p0 : 0) + pt.off[t.q]) +
                              t.m0 + rank * trows;
                const int b0 = __clz(trows) - 24, r0 = 128 >> b0;  // the boxes, largest first (trows is 16 .. 128)
                const int b1 = trows > r0 ? __clz(trows - r0) - 24 : -1, r1 = b1 < 0 ? 0 : r0 + (128 >> b1);
                const int b2 = b1 >= 0 && trows > r1 ? __clz(trows - r1) - 24 : -1;
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = false; break; }
                    if (elect_one()) {
                        const uint32_t sT = sbase + stage * stage_bytes + kABytes;
                        const uint32_t fb = dsmem_addr(full_bar(stage), 0);
                        if (rank == 0) mbar_expect_tx(full_bar(stage), (uint32_t)(t.n * BK * 2));
                        tma_load_2d_pair(sT, &maps.tok[b0], fb, kb * BK, y);
                        if (b1 >= 0) tma_load_2d_pair(sT + r0 * 128, &maps.tok[b1], fb, kb * BK, y + r0);
                        if (b2 >= 0) tma_load_2d_pair(sT + r1 * 128, &maps.tok[b2], fb, kb * BK, y + r1);
                    }
                    ++issued;
                    if (++stage == nst) { stage = 0; phase ^= 1u; }
                }
            } else {
                const int2 wq = group_weights(p, t.q);
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = false; break; }
                    const uint32_t sW = sbase + stage * stage_bytes, fb = dsmem_addr(full_bar(stage), 0);
                    if (kGU) {
                        const int y = wq.y * p.I + t.n0 + rank * 64;
                        if (elect_one()) {
                            if (rank == 0) mbar_expect_tx(full_bar(stage), 2u * kABytes);
                            if (!out.two_boxes[wq.x]) {
                                tma_load_3d_pair(sW, &maps.gu[wq.x], fb, kb * BK, y, 0);
                            } else {
                                tma_load_2d_pair(sW, &maps.w0[wq.x], fb, kb * BK, y);
                                tma_load_2d_pair(sW + kABytes / 2, &maps.w1[wq.x], fb, kb * BK, y);
                            }
                        }
                    } else {
                        const bool second = kb >= p.k_split;
                        const int krow = wq.y * p.kb_rows + (second ? kb - p.k_split : kb) * BK;
                        if (elect_one()) {
                            if (rank == 0) mbar_expect_tx(full_bar(stage), 2u * kABytes);
                            tma_load_3d_pair(sW, second ? &maps.w1[wq.x] : &maps.w0[wq.x], fb, 0, krow,
                                             (t.n0 + rank * 128) / 64);
                        }
                    }
                    ++issued;
                    if (++stage == nst) { stage = 0; phase ^= 1u; }
                }
            }
        }
        if (rank == 0) drain_stages(bar0, nst, issued, stage, phase);  // both CTAs' copies
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        int stage = 0, it = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = first; rank == 0 && tile < last && ok; tile += pairs, ++it) {
            const PairTile t = decode_pair(pt, p.G, width, tile, lane);
            const uint32_t idesc = p.idesc | ((uint32_t)(t.n >> 3) << 17);
            const int buf = it & 1;
            const uint32_t use = (uint32_t)(it >> 1) & 1u;
            if (!warp_wait(tempty_bar(buf), use ^ 1u)) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * kAccCols);
            bool ready = false;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!__all_sync(~0u, ready || mbar_wait(full_bar(stage), phase, &s_abort, p.status))) { ok = false; break; }
                tc_fence_after();
                const uint32_t eb = empty_bar(stage);
                const uint32_t sW = sbase + stage * stage_bytes;
                const uint64_t bd = sw128_desc(sW + kABytes);
                if (++stage == nst) { stage = 0; phase ^= 1u; }
                ready = mbar_test_wait(full_bar(stage), phase);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        tc_mma_pair(d_tmem, kGU ? sw128_desc(sW) + 2 * k : mn_sw128_desc(sW + k * 2048, kMnBlockBytes),
                                    bd + 2 * k, idesc, (kb | k) != 0);
                    tc_commit_pair(eb);
                    if (kb == nkb - 1) tc_commit_pair(tfull_bar(buf));
                }
                __syncwarp();
            }
        }
        // the leader's last commit: its MMAs and every commit before (whose
        // arrivals reach both CTAs) are done before either CTA exits
        if (elect_one()) {
            if (rank == 0) tc_commit_pair(done_bar);
            const unsigned long long t0 = globaltimer_ns();
            while (!mbar_try_wait(done_bar, 0))
                if (globaltimer_ns() - t0 > kWaitLimitNs) break;
        }
    } else {
        // ------------------------------------------------ epilogue
        // A warp's 32 TMEM lanes are 32 output columns; chunks of 32 tokens are
        // turned into rows of 64 bytes through shared memory (see the forward's
        // epilogues, whose exchange of gate and up values this one shares).
        const int quarter = warp & 3;
        const uint32_t stage0 = sbase + kPairRing;
        const uint32_t own = stage0 + quarter * kPairOutBytes, partner = stage0 + (quarter ^ 2) * kPairOutBytes;
        const uint32_t roww = stage0 + 4 * kPairOutBytes + quarter * kPairRowWBytes;
        const int srow = lane & 7, scol = lane >> 3;
        int it = 0;
        for (int tile = first; tile < last; tile += pairs, ++it) {
            const PairTile t = decode_pair(pt, p.G, width, tile, lane);
            const int buf = it & 1;
            const int prow = pt.pad[t.q] + t.m0;  // the tile's first row of the padded layout
            if (kGU) {  // the rows' routing weights, ahead of the accumulator
                const int slot0 = p0 + pt.off[t.q] + t.m0;
                float w[kPairMaxN / 32];
#pragma unroll
                for (int c = 0; c < kPairMaxN / 32; ++c) {
                    const int r = c * 32 + lane;
                    w[c] = r < t.rows ? (p.shared_T ? 1.f : p.w_of_slot[slot0 + r]) : 0.f;
                }
                __syncwarp();
#pragma unroll
                for (int c = 0; c < kPairMaxN / 32; ++c) st_shared_f32(roww + (c * 32 + lane) * 4, w[c]);
                __syncwarp();
            }
            const bool ok = warp_wait(tfull_bar(buf), (uint32_t)(it >> 1) & 1u);
            // (gate/up: the four warps, which meet at barriers inside a tile, go on or stop together)
            if (kGU ? !named_barrier_all(3, 128, ok) : !ok) break;
            tc_fence_after();
            const uint32_t tb = tmem_base + (uint32_t)(buf * kAccCols) + ((uint32_t)(quarter * 32) << 16);
            if (kGU) {
                gu_epilogue(p, out, pt, t, tb, own, partner, roww, rank, quarter, lane, prow, p0);
            } else {
                const int col = t.n0 + rank * 128 + quarter * 32;
                bf16 *orow = out.c + (size_t)prow * p.N + col + (lane & 3) * 8;
#pragma unroll 1
                for (int c = 0; c < t.n / 32 && col < p.N; ++c) {  // (a last block's second half may lie past N)
                    const uint32_t xo = own + (uint32_t)((c & 1) * 2048);
                    float v[2][16];
                    tmem_frag16(tb + c * 32, v[0]);
                    tmem_frag16(tb + c * 32 + (16u << 16), v[1]);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int r = 8 * j + srow;
                        stmatrix_x4_trans(xo + r * 64 + ((scol ^ ((r >> 1) & 3)) << 4), pack_bf16x2(v[0][4 * j], v[0][4 * j + 1]),
                                          pack_bf16x2(v[0][4 * j + 2], v[0][4 * j + 3]),
                                          pack_bf16x2(v[1][4 * j], v[1][4 * j + 1]),
                                          pack_bf16x2(v[1][4 * j + 2], v[1][4 * j + 3]));
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
                        if (tok < t.rows) *reinterpret_cast<uint4 *>(orow + (size_t)tok * p.N) = f[h];
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (rank == 0) mbar_arrive(tempty_bar(buf));
                else mbar_arrive_remote(dsmem_addr(tempty_bar(buf), 0));
            }
        }
    }

    __syncwarp();
    tc_fence_before();
    cluster_sync_all();  // the pair's MMAs, copies and barrier arrivals are done
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------- saved G | U

// The gate/up launch's outputs from the forward's saved accumulators G | U
// ([R][2I] FP32) instead of a recomputing GEMM: one warp per routed row and
// 128-column tile, four columns per lane (coalesced rows), with the
// epilogue's per-element arithmetic and its order of summing dL/dw over 32
// columns, so [dG | dU], w act and the dL/dw partials are bitwise those of
// bwd_rows_pair_kernel, in the same padded layout; padded tail rows are written as
// zeros.
__global__ void __launch_bounds__(256) bwd_swiglu_saved_kernel(const RowsParams p, const float *saved_gu, bf16 *dgu,
                                                               bf16 *wact)
{
    __shared__ GroupTable gt;
    pdl_trigger();
    pdl_wait();
    const int nt = p.I / 128;
    build_groups(gt, p.offsets, p.g0, p.G, p.R, p.shared_T, nt);
    const int total = gt.tiles[p.G];
    const int p0 = p.shared_T ? 0 : (int)min(p.offsets[p.g0], (uint32_t)p.R);
    // saved rows: routed [R][2I] (G | U), then shared [T][2 G I] (all G, then all U)
    const int ld2 = p.shared_T ? 2 * p.G * p.I : 2 * p.I;
    const float *sbase = p.shared_T ? saved_gu + (size_t)p.R * 2 * p.I : saved_gu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x) {
        const RowsTile t = decode_rows_thread(gt, p.G, 128, tile);
        const bool wa_out = p.wact && !p.shared_T && p.g0 + t.q >= p.E_pub;
        const int gcol = p.shared_T ? t.q * p.I : 0;  // the group's G columns in its saved row
        for (int r = warp; r < BM; r += nwarps) {
            const bool valid = r < t.rows;  // warp-uniform
            const int prow = gt.off[t.q] + t.m0 + r;
            const int orow = gt.pad[t.q] + t.m0 + r;
            const int col = t.n0 + 4 * lane;
            float g[4] = {0.f, 0.f, 0.f, 0.f}, u[4] = {0.f, 0.f, 0.f, 0.f}, z[4] = {0.f, 0.f, 0.f, 0.f};
            float w = 0.f;
            if (valid) {
                const float *grow = sbase + (size_t)(p0 + prow) * ld2 + gcol;
                const float4 gv = *reinterpret_cast<const float4 *>(grow + col);
                const float4 uv = *reinterpret_cast<const float4 *>(grow + ld2 / 2 + col);
                const uint2 zv = *reinterpret_cast<const uint2 *>(p.zpad + (size_t)orow * p.I + col);
                g[0] = gv.x; g[1] = gv.y; g[2] = gv.z; g[3] = gv.w;
                u[0] = uv.x; u[1] = uv.y; u[2] = uv.z; u[3] = uv.w;
                const float2 z01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&zv.x));
                const float2 z23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&zv.y));
                z[0] = z01.x; z[1] = z01.y; z[2] = z23.x; z[3] = z23.y;
                w = p.shared_T ? 1.f : p.w_of_slot[p0 + prow];
            }
            float dg[4], du[4], wa[4], q[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                float a;
                swiglu_bwd(g[h], u[h], z[h], w, a, dg[h], du[h], wa[h]);
                q[h] = __fmul_rn(z[h], a);
                if (!valid) dg[h] = du[h] = wa[h] = 0.f;
            }
            bf16 *dst = dgu + (size_t)orow * 2 * p.I + col;
            *reinterpret_cast<uint2 *>(dst) = make_uint2(pack_bf16x2(dg[0], dg[1]), pack_bf16x2(dg[2], dg[3]));
            *reinterpret_cast<uint2 *>(dst + p.I) = make_uint2(pack_bf16x2(du[0], du[1]), pack_bf16x2(du[2], du[3]));
            if (wa_out)
                *reinterpret_cast<uint2 *>(wact + (size_t)orow * p.I + col) =
                    make_uint2(pack_bf16x2(wa[0], wa[1]), pack_bf16x2(wa[2], wa[3]));
            // the 32-column chunk sums: pairs of neighbouring columns, then pairs of
            // those, and so on (four columns in the lane, then a butterfly over
            // the chunk's eight lanes)
            float sum = __fadd_rn(__fadd_rn(q[0], q[1]), __fadd_rn(q[2], q[3]));
            sum = __fadd_rn(sum, __shfl_xor_sync(~0u, sum, 1));
            sum = __fadd_rn(sum, __shfl_xor_sync(~0u, sum, 2));
            sum = __fadd_rn(sum, __shfl_xor_sync(~0u, sum, 4));
            const float c0 = __shfl_sync(~0u, sum, 0), c1 = __shfl_sync(~0u, sum, 8);
            const float c2 = __shfl_sync(~0u, sum, 16), c3 = __shfl_sync(~0u, sum, 24);
            if (lane == 0 && valid && p.gw_part)
                *reinterpret_cast<float4 *>(p.gw_part + (size_t)(p0 + prow) * (p.I / 32) + t.n0 / 32) =
                    make_float4(c0, c1, c2, c3);
        }
    }
}

// ------------------------------------------------------------- wgrad

// On CTA pairs (tc_ptx.cuh): a tile is 256 rows of M (2I or H) x up to 256
// columns of N; each CTA stages its 128 rows of A and its half of B's columns
// (32 KB a stage at N = 256) and drains its own 128 rows.  What bounds it is
// the FP32 gradients: 604 MB written and 210 MB of operands read at Qwen3
// prefill (16,384 private rows) are 120 us at the measured copy rate.  The
// epilogue must keep up with short K loops (8 steps, about 4,300 clocks, at
// 512 rows an expert): boxes of 4 KB, three in flight a warp, take it out of
// the way (2 KB boxes, two in flight: 5,600 clocks a tile).  Training step at
// Qwen3 T = 4096 1184 -> 1177 us, at the DeepSeek shape T = 3000 1559 -> 1542
// us against single-CTA 128 x 256 tiles.
constexpr int kWgStages = 5;
constexpr int kWgStageBytes = 2 * kABytes;
constexpr int kWgLoaders = 2;               // loader warps 0 and 6
constexpr int kWgOutBufs = 3;              // per epilogue warp, boxes of 32 rows x 32 FP32 columns
constexpr int kWgOutBoxBytes = 32 * 128;
constexpr int kWgDynSmem = kWgStages * kWgStageBytes + 4 * kWgOutBufs * kWgOutBoxBytes + 1024;

struct WgParams {
    int E_pub, E_priv, H, I, R;
    // the group table's groups (the private experts alone, g0 = E_pub, or all
    // routed experts, g0 = 0, whose padded layout the operands then use) and
    // the table index of private expert 0
    int g0, G, q_off;
    const uint32_t *offsets;
    uint32_t *status;
    uint32_t idesc;  // M = 256, both operands MN-major, N = 0 (added per tile)
};

struct WgMaps {
    // 3-D maps, boxes of 64 rows (K) x 64-element MN blocks (encode_3d_blocks):
    // A: a CTA's 128 rows of M, 2 blocks; B [0]: its half of 256 columns, 2
    // blocks, [1]: of a last tile of 128 columns, 1 block
    CUtensorMap dgu;         // [padded rows][2I] (A)
    CUtensorMap a_perm[2];   // [R][H] (B)
    CUtensorMap dout_rows;   // [R + 64][H] (A)
    CUtensorMap wact[2];     // [padded rows][I] (B)
    CUtensorMap d_gate, d_up, d_down;  // FP32 outputs, 32 x 32 boxes, 128-byte swizzle
};

struct WgTile {
    int prob, q, m0, n0, bn, nkb;
};

// M blocks of 256 and N blocks of at most 256 (H and I are multiples of 128;
// 2I is one of 256).
__device__ __forceinline__ int wg_blocks(int n) { return (n + 255) / 256; }

__device__ __forceinline__ int wg_total(const WgParams &p)
{
    return p.E_priv * (p.I / 128 * wg_blocks(p.H) + wg_blocks(p.H) * wg_blocks(p.I));
}

__device__ __forceinline__ WgTile decode_wg(const WgParams &p, const GroupTable &gt, int tile)
{
    WgTile t;
    const int na = wg_blocks(p.H), nta = p.I / 128 * na;
    const int nb = wg_blocks(p.I), ntb = wg_blocks(p.H) * nb;
    int local;
    if (tile < p.E_priv * nta) {
        t.prob = 0;
        t.q = tile / nta;
        local = tile - t.q * nta;
        t.m0 = (local / na) * 256;
        t.n0 = (local % na) * 256;
        t.bn = min(256, p.H - t.n0);
    } else {
        tile -= p.E_priv * nta;
        t.prob = 1;
        t.q = tile / ntb;
        local = tile - t.q * ntb;
        t.m0 = (local / nb) * 256;
        t.n0 = (local % nb) * 256;
        t.bn = min(256, p.I - t.n0);
    }
    t.nkb = (gt.rows[t.q + p.q_off] + BK - 1) / BK;
    return t;
}

__global__ void __launch_bounds__(kThreads, 1) bwd_wgrad_tc_kernel(const WgParams p, const __grid_constant__ WgMaps maps)
{
    extern __shared__ uint8_t dsmem[];
    __shared__ GroupTable gt;
    __shared__ __align__(8) uint64_t bars[2 * kWgStages + 5];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;

    const int tid = threadIdx.x, warp = __shfl_sync(~0u, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)cluster_ctarank();  // 0: the leader, whose thread issues the pair's MMAs
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const uint32_t sbase = (smem_u32(dsmem) + 1023u) & ~1023u;
    const uint32_t bar0 = smem_u32(bars);
    // full (both CTAs' copies) and tempty (both CTAs' epilogues) are the
    // leader's; empty and tfull are signalled in both CTAs by the commits
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kWgStages + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * kWgStages + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * kWgStages + 2 + b); };
    const uint32_t done_bar = bar0 + 8u * (2 * kWgStages + 4);

    if (tid == 0) {
        for (int s = 0; s < kWgStages; ++s) { mbar_init(full_bar(s), kWgLoaders); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 8); }
        mbar_init(done_bar, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 1) tmem_alloc_pair(smem_u32(&s_tmem), kTmemCols);
    pdl_wait();
    build_groups(gt, p.offsets, p.g0, p.G, p.R, 0, 0);
    tc_fence_before();
    cluster_sync_all();  // both CTAs' barriers and TMEM are ready
    tc_fence_after();
    const uint32_t tmem_base = s_tmem;
    const int total = wg_total(p);
    const int p0 = (int)min(p.offsets[p.g0], (uint32_t)p.R);

    auto warp_wait = [&](uint32_t bar, uint32_t parity) -> bool {
        return __all_sync(~0u, mbar_wait(bar, parity, &s_abort, p.status));
    };

    if (warp == 0 || warp == 6) {
        // ------------------------------------------------ TMA producers
        // warp 0: this CTA's two 64-element MN blocks of A; warp 6: its half of
        // B's bn / 64 blocks; one 3-D box each (64 MN elements x 64 rows of
        // K per block).  Every copy completes on the leader's barrier, where
        // the leader's warps announce both CTAs' bytes.
        int stage = 0, issued = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = pair; tile < total && ok; tile += pairs) {
            const WgTile t = decode_wg(p, gt, tile);
            const int half = t.bn / 128;  // MN blocks of B per CTA
            const int gq = t.q + p.q_off;  // the expert's entry in the group table
            const int rowA = t.prob == 0 ? gt.pad[gq] : gt.off[gq];
            const int rowB = t.prob == 0 ? p0 + gt.off[gq] : gt.pad[gq];
            const CUtensorMap *map = warp == 0 ? (t.prob == 0 ? &maps.dgu : &maps.dout_rows)
                                               : (t.prob == 0 ? &maps.a_perm[2 - half] : &maps.wact[2 - half]);
            const int row = warp == 0 ? rowA : rowB;
            const int block = warp == 0 ? t.m0 / 64 + 2 * rank : t.n0 / 64 + half * rank;
            const uint32_t bytes = 2u * (warp == 0 ? (uint32_t)kABytes : (uint32_t)(half * kMnBlockBytes));
            for (int kb = 0; kb < t.nkb; ++kb) {
                if (!warp_wait(empty_bar(stage), phase ^ 1u)) { ok = false; break; }
                if (elect_one()) {
                    const uint32_t dst = sbase + stage * kWgStageBytes + (warp == 0 ? 0 : kABytes);
                    const uint32_t fb = dsmem_addr(full_bar(stage), 0);
                    if (rank == 0) mbar_expect_tx(full_bar(stage), bytes);
                    tma_load_3d_pair(dst, map, fb, 0, row + kb * BK, block);
                }
                ++issued;
                if (++stage == kWgStages) { stage = 0; phase ^= 1u; }
            }
        }
        if (rank == 0) drain_stages(bar0, kWgStages, issued, stage, phase);  // both CTAs' copies
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        // two 256-column FP32 accumulators: the epilogue of one tile overlaps the
        // MMAs of the next.  A tile of an expert without rows issues no MMA;
        // its epilogue writes zeros.
        int stage = 0, it = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = pair; rank == 0 && tile < total && ok; tile += pairs, ++it) {
            const WgTile t = decode_wg(p, gt, tile);
            const uint32_t idesc = p.idesc | ((uint32_t)(t.bn >> 3) << 17);
            const int buf = it & 1;
            const uint32_t use = (uint32_t)(it >> 1) & 1u;
            if (!warp_wait(tempty_bar(buf), use ^ 1u)) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256);
            bool ready = false;
            for (int kb = 0; kb < t.nkb; ++kb) {
                if (!__all_sync(~0u, ready || mbar_wait(full_bar(stage), phase, &s_abort, p.status))) { ok = false; break; }
                tc_fence_after();
                const uint32_t eb = empty_bar(stage);
                const uint32_t sA = sbase + stage * kWgStageBytes, sB = sA + kABytes;
                if (++stage == kWgStages) { stage = 0; phase ^= 1u; }
                ready = mbar_test_wait(full_bar(stage), phase);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        tc_mma_pair(d_tmem, mn_sw128_desc(sA + k * 2048, kMnBlockBytes),
                                    mn_sw128_desc(sB + k * 2048, kMnBlockBytes), idesc, (kb | k) != 0);
                    tc_commit_pair(eb);
                }
                __syncwarp();
            }
            if (ok && elect_one()) tc_commit_pair(tfull_bar(buf));
            __syncwarp();
        }
        // the leader's last commit: its MMAs and every commit before (whose
        // arrivals reach both CTAs) are done before either CTA exits
        if (elect_one()) {
            if (rank == 0) tc_commit_pair(done_bar);
            const unsigned long long t0 = globaltimer_ns();
            while (!mbar_try_wait(done_bar, 0))
                if (globaltimer_ns() - t0 > kWaitLimitNs) break;
        }
    } else {
        // ------------------------------------------------ epilogue
        const int quarter = warp & 3;
        const uint32_t out0 = sbase + kWgStages * kWgStageBytes + (uint32_t)((warp - 2) * kWgOutBufs * kWgOutBoxBytes);
        int it = 0, ob = 0;
        for (int tile = pair; tile < total; tile += pairs, ++it) {
            const WgTile t = decode_wg(p, gt, tile);
            const int buf = it & 1;
            const uint32_t use = (uint32_t)(it >> 1) & 1u;
            int ok = 1;
            if (lane == 0) ok = mbar_wait(tfull_bar(buf), use, &s_abort, p.status) ? 1 : 0;
            ok = __shfl_sync(~0u, ok, 0);
            if (!ok) break;
            __syncwarp();
            tc_fence_after();
            const int m0 = t.m0 + rank * BM;  // this CTA's 128 rows
            const bool inside = m0 < (t.prob == 0 ? 2 * p.I : p.H);  // (H may end inside the pair's 256 rows)
            const CUtensorMap *omap;
            int orow;
            if (t.prob == 0) {
                omap = m0 < p.I ? &maps.d_gate : &maps.d_up;
                orow = t.q * p.I + (m0 < p.I ? m0 : m0 - p.I);
            } else {
                omap = &maps.d_down;
                orow = t.q * p.H + m0;
            }
            orow += quarter * 32;
            const uint32_t tb = tmem_base + (uint32_t)(buf * 256) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
            for (int c = 0; inside && c < t.bn / 32; ++c) {
                float v[32];
                if (t.nkb > 0) {
                    tmem_ld32(tb + c * 32, v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = 0.f;
                }
                // a box of 32 rows of 128 bytes, 16-byte chunk j of row r at chunk
                // j ^ (r & 7): the TMA 128-byte swizzle, conflict-free here
                const uint32_t sbuf = out0 + (uint32_t)(ob * kWgOutBoxBytes);
                if (lane == 0) bulk_wait_read<kWgOutBufs - 1>();  // the store that used this buffer has read it
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(sbuf + lane * 128 + ((j ^ (lane & 7)) << 4)),
                                 "f"(v[4 * j]), "f"(v[4 * j + 1]), "f"(v[4 * j + 2]), "f"(v[4 * j + 3])
                                 : "memory");
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(omap, sbuf, t.n0 + c * 32, orow);
                    bulk_commit();
                }
                ob = ob == kWgOutBufs - 1 ? 0 : ob + 1;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (rank == 0) mbar_arrive(tempty_bar(buf));
                else mbar_arrive_remote(dsmem_addr(tempty_bar(buf), 0));
            }
        }
        if (lane == 0) bulk_wait_all();
    }

    __syncwarp();
    tc_fence_before();
    cluster_sync_all();  // the pair's MMAs, copies and barrier arrivals are done
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

}  // namespace

// Rows of the padded layout (an upper bound over all routings).
size_t backward_padded_rows(const Shape &s) { return (size_t)s.T * s.k + (size_t)kPad * s.E_priv; }

namespace {

// Fields shared by every row launch over the groups `g`.
RowsParams rows_params(const Ctx &c, const RowsGroups &g)
{
    const Shape &s = c.s;
    RowsParams p;
    memset(&p, 0, sizeof(p));
    p.E_pub = s.E_pub; p.H = s.H; p.I = s.I; p.R = s.T * s.k;
    p.g0 = g.g0; p.G = g.G; p.shared_T = g.shared_T;
    p.offsets = c.offsets;
    p.w_of_slot = c.w_of_slot;
    p.status = c.audit.status;
    return p;
}

// The weight tensor of pool q (0 public, 1 private) for routed groups, or the
// shared one, with its rows: experts x rows_per_expert.
const bf16 *pool_tensor(const Ctx &c, const RowsGroups &g, const bf16 *const *w, int q, int rows_per_expert,
                        uint64_t *rows)
{
    const Shape &s = c.s;
    const int n = g.shared_T ? s.E_sh : (q ? s.E_priv : s.E_pub);
    *rows = (uint64_t)n * rows_per_expert;
    return g.shared_T ? w[2] : w[q];
}

// A launch on CTA pairs: the rows' operand A [a_rows][K] K-major, the
// weights' maps filled in.
template <bool kGU>
cudaError_t run_pairs(const Ctx &c, RowsParams &p, PairMaps &maps, const bf16 *a, uint64_t a_rows, const PairOut &out)
{
    for (int b = 0; b < kTokBoxes; ++b)
        if (!encode_2d(&maps.tok[b], a, p.K, a_rows, 128u >> b)) return cudaErrorInvalidValue;
    p.idesc = kGU ? make_idesc(2 * BM, 0) : make_idesc_major(2 * BM, 0, true, false);  // N added per tile
    static std::atomic<int> smem_limit[64];
    cudaError_t err = ensure_dynamic_smem(bwd_rows_pair_kernel<kGU>, kPairDynSmem, smem_limit);
    if (err != cudaSuccess) return err;
    return launch_cluster_pdl(bwd_rows_pair_kernel<kGU>, 2, dim3(c.num_sms / 2 * 2), dim3(kThreads), kPairDynSmem, c.stream,
                              p, out, maps);
}

}  // namespace

cudaError_t launch_rows_z(const Ctx &c, const RowsGroups &g, const bf16 *d, uint64_t d_rows, int tight, bf16 *zpad)
{
    const Shape &s = c.s;
    RowsParams p = rows_params(c, g);
    PairMaps maps;
    memset(&maps, 0, sizeof(maps));
    p.K = s.H; p.N = s.I;
    p.kb_rows = s.H; p.k_split = s.H / BK;
    p.a_rows = tight ? kArowsTight : kArowsSlot;
    p.gemm_next = c.saved_gu == nullptr;
    bool ok = true;
    for (int q = 0; q < (g.shared_T ? 1 : 2); ++q) {
        uint64_t rows;
        const bf16 *w = pool_tensor(c, g, c.down, q, s.H, &rows);
        ok &= encode_3d_blocks(&maps.w0[q], w, s.I, rows, 64, 2);
    }
    return ok ? run_pairs<false>(c, p, maps, d, d_rows, PairOut{zpad, nullptr, {}, {}}) : cudaErrorInvalidValue;
}

cudaError_t launch_rows_gu(const Ctx &c, const RowsGroups &g, const bf16 *a, uint64_t a_rows, const bf16 *zpad,
                           bf16 *dgu, bf16 *wact, float *gw_part)
{
    const Shape &s = c.s;
    RowsParams p = rows_params(c, g);
    p.K = s.H; p.N = s.I;
    p.zpad = zpad;
    p.gw_part = gw_part;
    p.wact = wact ? 1 : 0;
    if (c.saved_gu)  // the forward saved the G | U accumulators of these rows
        return launch_pdl(bwd_swiglu_saved_kernel, dim3(c.num_sms * 8), dim3(256), 0, c.stream, p,
                          (const float *)c.saved_gu, dgu, wact);
    PairMaps maps;
    memset(&maps, 0, sizeof(maps));
    p.a_rows = kArowsSlot;
    PairOut out{dgu, wact, {}, {}};
    bool ok = true;
    for (int q = 0; q < (g.shared_T ? 1 : 2); ++q) {
        uint64_t rows;
        const bf16 *wg = pool_tensor(c, g, c.gate, q, s.I, &rows);
        const bf16 *wu = pool_tensor(c, g, c.up, q, s.I, &rows);
        bool up_first;
        if (encode_gate_up(&maps.gu[q], wg, wu, s.H, rows, &up_first)) {
            out.up_first[q] = up_first;
        } else {
            out.two_boxes[q] = 1;
            ok &= encode_2d(&maps.w0[q], wg, s.H, rows, 64);
            ok &= encode_2d(&maps.w1[q], wu, s.H, rows, 64);
        }
    }
    return ok ? run_pairs<true>(c, p, maps, a, a_rows, out) : cudaErrorInvalidValue;
}

cudaError_t launch_rows_da(const Ctx &c, const RowsGroups &g, const bf16 *dgu, bf16 *da)
{
    const Shape &s = c.s;
    RowsParams p = rows_params(c, g);
    PairMaps maps;
    memset(&maps, 0, sizeof(maps));
    p.K = 2 * s.I; p.N = s.H;
    p.kb_rows = s.I; p.k_split = s.I / BK;  // K blocks of dG take W_gate, those of dU take W_up
    p.a_rows = kArowsPad;
    bool ok = true;
    for (int q = 0; q < (g.shared_T ? 1 : 2); ++q) {
        uint64_t rows;
        const bf16 *wg = pool_tensor(c, g, c.gate, q, s.I, &rows);
        const bf16 *wu = pool_tensor(c, g, c.up, q, s.I, &rows);
        ok &= encode_3d_blocks(&maps.w0[q], wg, s.H, rows, 64, 2);
        ok &= encode_3d_blocks(&maps.w1[q], wu, s.H, rows, 64, 2);
    }
    return ok ? run_pairs<false>(c, p, maps, dgu, g.padded_rows, PairOut{da, nullptr, {}, {}}) : cudaErrorInvalidValue;
}

cudaError_t launch_backward_rows(const Ctx &c, const bf16 *dout_rows, bf16 *zpad, bf16 *dgu, bf16 *wact,
                                 float *gw_part)
{
    const Shape &s = c.s;
    const RowsGroups g{s.E_pub, s.E_priv, 0, backward_padded_rows(s)};
    cudaError_t err = launch_rows_z(c, g, dout_rows, (uint64_t)s.T * s.k + 64, 1, zpad);
    if (err != cudaSuccess) return err;
    return launch_rows_gu(c, g, c.a_perm, (uint64_t)s.T * s.k, zpad, dgu, wact, gw_part);
}

cudaError_t launch_backward_wgrad(const Ctx &c, const bf16 *dout_rows, const bf16 *dgu, const bf16 *wact,
                                  float *d_gate, float *d_up, float *d_down, const RowsGroups *all)
{
    const Shape &s = c.s;
    const uint64_t R = (uint64_t)s.T * s.k, RP = all ? all->padded_rows : backward_padded_rows(s);
    WgParams p;
    WgMaps maps;
    memset(&p, 0, sizeof(p));
    memset(&maps, 0, sizeof(maps));
    p.E_pub = s.E_pub; p.E_priv = s.E_priv; p.H = s.H; p.I = s.I; p.R = (int)R;
    p.g0 = all ? 0 : s.E_pub;
    p.G = all ? s.E() : s.E_priv;
    p.q_off = all ? s.E_pub : 0;
    p.offsets = c.offsets;
    p.status = c.audit.status;
    p.idesc = make_idesc_major(2 * BM, 0, true, true);
    bool ok = encode_3d_blocks(&maps.dgu, dgu, 2 * (uint64_t)s.I, RP, 64, 2);
    ok &= encode_3d_blocks(&maps.dout_rows, dout_rows, s.H, R + 64, 64, 2);
    for (int h = 0; h < 2; ++h) {  // full tiles of 256 columns; a last one of 128
        ok &= encode_3d_blocks(&maps.a_perm[h], c.a_perm, s.H, R, 64, 2 - h);
        ok &= encode_3d_blocks(&maps.wact[h], wact, s.I, RP, 64, 2 - h);
    }
    const CUtensorMapSwizzle osw = CU_TENSOR_MAP_SWIZZLE_128B;
    ok &= encode_2d_f32(&maps.d_gate, d_gate, s.H, (uint64_t)s.E_priv * s.I, 32, 32, osw);
    ok &= encode_2d_f32(&maps.d_up, d_up, s.H, (uint64_t)s.E_priv * s.I, 32, 32, osw);
    ok &= encode_2d_f32(&maps.d_down, d_down, s.I, (uint64_t)s.E_priv * s.H, 32, 32, osw);
    if (!ok) return cudaErrorInvalidValue;
    static std::atomic<int> smem_limit[64];
    cudaError_t err = ensure_dynamic_smem(bwd_wgrad_tc_kernel, kWgDynSmem, smem_limit);
    if (err != cudaSuccess) return err;
    return launch_cluster_pdl(bwd_wgrad_tc_kernel, 2, dim3(c.num_sms / 2 * 2), dim3(kThreads), kWgDynSmem, c.stream, p,
                              maps);
}

}  // namespace pmpe
