// Internal declarations shared by the libpmpe translation units: the launch
// context, the workspace carve-up and small device helpers.  Nothing here is
// part of the C ABI (include/pmpe.h is).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>

#include "../../include/pmpe.h"

namespace pmpe {

typedef __nv_bfloat16 bf16;

// Limits checked on the host before any launch.
constexpr int kMaxPool = 256;   // experts per pool (router smem tiles)
constexpr int kMaxTopK = 32;    // one warp lane per selected expert
constexpr int kDimAlign = 128;  // H and I granularity

struct Shape {
    int T, H, I, E_pub, E_priv, E_sh, k, renorm;
    int E() const { return E_pub + E_priv; }
};

// Pointers into the audit buffer (all NULL when the caller passed none).
struct Audit {
    uint32_t *status, *shared_rows, *route_count, *exec_rows, *exec_tiles, *route_priv_rows, *exec_priv_rows;
};

Audit audit_ptrs(uint32_t *base, int T, int E);

// Everything one forward call needs, resolved from the descriptor.
struct Ctx {
    Shape s;
    const bf16 *hidden;
    const uint8_t *policy;
    const bf16 *router_pub, *router_priv;
    // [0] public, [1] private, [2] shared
    const bf16 *gate[3], *up[3], *down[3];
    bf16 *out;
    int32_t *idx;
    float *w;
    Audit audit;
    // workspace regions
    uint8_t *tau;
    uint32_t *counts, *offsets;
    int32_t *slot_of, *tok_of_slot;
    int32_t *ticket;    // [T, k] 128 * router tile + position among the tile's rows of its expert
    float *w_of_slot;
    uint32_t *tile_done;  // [router slots] chunk CTAs finished per router tile
    uint32_t *tile_counts; // [E][router_slots4] rows of each expert per router tile
    uint32_t *gemm_ready; // [gemm_ready_words] gate/up warps done per (group, row tile)
    float2 *router_lists; // [router CTAs * 128, k] per-chunk sorted (score, id)
    float4 *router_meta;  // [router CTAs * 128] per-chunk softmax partials
    bf16 *router_rows;  // [router CTAs * 128, H] copied token rows of non-contiguous router tiles
    bf16 *a_perm;  // [T*k, H] dispatched rows: filled only by the backward (the forward gathers on the fly)
    bf16 *act, *y, *act_sh, *y_sh;
    cudaStream_t stream;
    int num_sms;
    int unmasked;  // the soft-router control: no hard mask (a negative control, not the method)
    float *saved_gu;  // optional [T*k][2I] FP32 G | U written by the forward, read by the backward
};

int compute_layout(const Shape &s, pmpe_workspace_layout *L);
// Router geometry: 32-expert chunks of a pool, 128-token tile slots for T tokens.
int router_chunks(int pool_size);
int router_slots(int T);
// router_slots rounded up to a multiple of 4 (the row pitch of tile_counts).
int router_slots4(int T);
// Readiness counters of the persistent expert GEMMs: one per (group, row
// tile of at most 256 rows); sized for 128-row blocks, an upper bound over all
// routings.
size_t gemm_ready_words(const Shape &s);

// Launchers (one per stage); each returns the launch's cudaError_t.
// The router; with write_dispatch (only where route_writes_dispatch holds)
// it also writes the dispatch order and clears the expert launch's
// readiness counters, in place of the dispatch step.
cudaError_t launch_route(const Ctx &c, bool write_dispatch);
// Whether the router can write the dispatch order itself: T <= 128 (each
// pool fills at most one router tile) and the cluster router runs.
bool route_writes_dispatch(const Ctx &c);
// Whether launch_route takes the cluster router (no memset before it; the
// dispatch derives the per-expert counts from tile_counts) or the chunked one.
bool route_uses_cluster_kernel(const Shape &s, int unmasked, int num_sms);
cudaError_t launch_permute(const Ctx &c);
cudaError_t launch_gateup(const Ctx &c);
cudaError_t launch_down(const Ctx &c);
// Backward of the private branch (k_backward.cu): scratch bytes and launch.
size_t backward_workspace_bytes(const Shape &s);
cudaError_t launch_backward_private(const Ctx &c, const bf16 *dout, float *d_router, float *d_gate, float *d_up,
                                    float *d_down, uint8_t *bws);
// Its pieces shared with the input gradient: the upstream gradients of the
// dispatch rows of experts g0 .. g1 - 1 (and 64 zero rows after them); the
// router's softmax gradient from the dL/dw partials per slot (both_pools = 0:
// the private pool, zero for DENY tokens; 1: each token's own pool), dz [T][ld]
// (pool softmax: the pools' token lists go to pool_tok [T] and pool_n [2]).
cudaError_t launch_gather_rows(const bf16 *dout, const int32_t *tok_of_slot, const uint32_t *offsets, int g0, int g1, int R,
                        int H, bf16 *rows, int num_sms, cudaStream_t st);
cudaError_t launch_router_dz(const Ctx &c, const float *gw_part, int both_pools, int ld, float *dz, int32_t *pool_tok,
                             int *pool_n, float *logit_part);
// Ranges of h the pool-softmax logits are split over: logit_part holds
// router_logit_splits(s) * T * ld floats.
int router_logit_splits(const Shape &s);
// The pool-softmax router term of the input gradient, added to d_hidden
// (pool lists from launch_router_dz).
cudaError_t launch_router_term(const Ctx &c, const float *dz, int ld, const int32_t *pool_tok, const int *pool_n,
                               float *d_hidden);
constexpr int kMaxRouterSplits = 64;  // token ranges of the router weight gradient
// The private router's weight gradient from dz (rows ld apart; DENY rows read
// as zeros): token-range partials (part, router_wgrad_part_bytes) and their
// fixed-order sum into d_router [E_priv, H]; active: kMaxRouterSplits words.
size_t router_wgrad_part_bytes(const Shape &s);
cudaError_t launch_router_wgrad(const Ctx &c, const float *dz, int ld, float *part, int *active, float *d_router);
// Gradient of the layer's input (k_backward_input.cu): scratch bytes and launch.
size_t backward_input_workspace_bytes(const Shape &s);
cudaError_t launch_backward_input(const Ctx &c, const bf16 *dout, float *d_hidden, uint8_t *bws);
// Both in one pass (k_backward_input.cu): the private gradients and the input
// gradient from one set of row launches over all routed experts.
size_t backward_step_workspace_bytes(const Shape &s);
cudaError_t launch_backward_step(const Ctx &c, const bf16 *dout, float *d_router, float *d_gate, float *d_up,
                                 float *d_down, float *d_hidden, uint8_t *bws);
// Its tensor-core GEMMs (k_backward_tc.cu): rows of the padded layout, the
// dL/da and gate/up recompute launches, and the weight-gradient launch.
size_t backward_padded_rows(const Shape &s);
cudaError_t launch_backward_rows(const Ctx &c, const bf16 *dout_rows, bf16 *zpad, bf16 *dgu, bf16 *wact,
                                 float *gw_part);
// The groups of one row launch: routed experts g0 .. g0 + G - 1 (shared_T = 0)
// or the G = E_sh shared experts over shared_T tokens; padded_rows bounds the
// padded row layout of their outputs (each group's rows rounded up to 128).
struct RowsGroups {
    int g0, G, shared_T;
    uint64_t padded_rows;
};
// Z = D W_down (D rows: tight = relative to expert g0's first slot, else the
// slot or token) -> zpad; the gate/up recompute with the SwiGLU backward ->
// [dG | dU] (and w act, dL/dw partials when non-null); dA = [dG | dU] [W_gate; W_up].
cudaError_t launch_rows_z(const Ctx &c, const RowsGroups &g, const bf16 *d, uint64_t d_rows, int tight, bf16 *zpad);
cudaError_t launch_rows_gu(const Ctx &c, const RowsGroups &g, const bf16 *a, uint64_t a_rows, const bf16 *zpad,
                           bf16 *dgu, bf16 *wact, float *gw_part);
cudaError_t launch_rows_da(const Ctx &c, const RowsGroups &g, const bf16 *dgu, bf16 *da);
// all == null: the operands use the private experts' own padded layout and
// dout_rows starts at the first private slot; otherwise the padded layout of
// all routed experts (`all`) and dout_rows indexed by dispatch slot.
cudaError_t launch_backward_wgrad(const Ctx &c, const bf16 *dout_rows, const bf16 *dgu, const bf16 *wact,
                                  float *d_gate, float *d_up, float *d_down, const RowsGroups *all = nullptr);
// Gate/up and down in one persistent launch (down tiles wait for their
// activation rows); zero_ready clears the readiness counters first.  When the
// device cannot host one CTA per SM at once, the two GEMMs run as two launches.
// The persistent gate/up + down launch.  With fuse_dispatch (the router ran
// just before in the same call, and experts_fuse_dispatch holds) the launch
// also derives the dispatch order itself, in place of launch_permute.
cudaError_t launch_experts(const Ctx &c, bool zero_ready, bool fuse_dispatch);
bool experts_fuse_dispatch(const Ctx &c);
// Whether the expert launch can route the tokens itself (T <= 128, the
// masked router, pools of at most 256 experts, H <= 2048, a resident grid),
// and that form of the forward: a kernel clearing the counters, then the
// persistent launch (routing, dispatch, both GEMMs and, with `combine`, the
// weighted combine).
bool experts_fuse_route(const Ctx &c);
cudaError_t launch_experts_routed(const Ctx &c, bool combine);
cudaError_t launch_combine(const Ctx &c);
// The token rows of the dispatch slots of groups g0 .. g1 - 1 copied from the
// hidden states into the workspace's dispatched-row matrix (a_perm), which the
// backward's GEMMs read.
cudaError_t launch_gather_dispatch_rows(const Ctx &c, int g0, int g1);
cudaError_t launch_resolve(const uint8_t *policy, int T, uint8_t *tau, cudaStream_t stream);
cudaError_t launch_policy_from_requests(const uint8_t *req_policy, const int32_t *cu_seqlens, int n_req, int T,
                                        uint8_t *policy_out, cudaStream_t stream);

// Raise `kernel`'s dynamic shared-memory limit on the current device to at
// least `bytes`, calling the runtime only when the limit must grow (the
// setting persists for the process; `limit` caches it per device, 64 devices).
template <typename Kernel>
cudaError_t ensure_dynamic_smem(Kernel kernel, int bytes, std::atomic<int> *limit)
{
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (limit[dev].load() >= bytes) return cudaSuccess;
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (err == cudaSuccess) {
        int cur = limit[dev].load();
        while (cur < bytes && !limit[dev].compare_exchange_weak(cur, bytes)) {
        }
    }
    return err;
}

// Launch with programmatic dependent launch: the kernel may start (and run
// its prologue) while the previous kernel in the stream finishes; it must
// execute pdl_wait() before touching anything that kernel wrote, or writing
// anything a previous kernel might still read.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                       Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// launch_pdl with clusters of `cluster` CTAs (the grid is a multiple of it).
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster_pdl(void (*kernel)(KArgs...), int cluster, dim3 grid, dim3 block, size_t smem,
                               cudaStream_t stream, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// ------------------------------------------------------------ device helpers

// Wait until the previous kernel in the stream has completed and its memory
// operations are visible (programmatic dependent launch).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// Allow the next kernel in the stream to launch now (it still waits for this
// one to complete before touching its results).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte async copy global -> shared; src_bytes = 0 zero-fills the 16 bytes.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, int src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes));
}
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// The grouped GEMMs take the experts in an order that spreads the private pool
// evenly among the public one.  The pools differ in rows per expert (a policy
// that allows half the tokens gives a quarter as many private experts four
// times the rows), so a run of one pool's tiles waits for the weights' DRAM
// reads and a run of the other's for the tensor cores; interleaved, the two
// overlap: Qwen3 T = 4096 374 -> 368 us, its training step 1058 -> 1036 us.  From
// 64 rows an expert on average, where below both pools' tiles wait for DRAM
// alike (T = 777, 39 rows: 264.3 us in id order, 265.3 interleaved), to 512,
// where above both wait for the tensor cores (T = 16384, 819 rows: 1057 and 1063 us).
// pool_place: the place of expert g; pool_at: the expert at place L (a walk,
// for small L); public experts first where both are due.
__host__ __device__ __forceinline__ bool interleave_pools(int R, int E) 
{
    return R >= 64 * E && R < 512 * E;
}
__device__ __forceinline__ int pool_place(int g, int E_pub, int E_priv)
{
    if (g < E_pub) return g + (E_priv > 0 ? min(E_priv, (((2 * g + 1) * E_priv - 1) / E_pub + 1) / 2) : 0);
    const int j = g - E_pub;
    return j + min(E_pub, ((2 * j + 1) * E_pub / E_priv + 1) / 2);
}
__device__ __forceinline__ int pool_at(int L, int E_pub, int E_priv)
{
    int i = 0, j = 0, g = 0;
    for (int s = 0; s <= L; ++s)
        g = j >= E_priv || (i < E_pub && (2 * i + 1) * E_priv <= (2 * j + 1) * E_pub) ? i++ : E_pub + j++;
    return g;
}

// silu(g) * u with the fast reciprocal-based division (for g -> -inf the
// denominator overflows to +inf and the quotient is 0, the correct limit).
__device__ __forceinline__ float silu_mul(float g, float u) { return __fdividef(g, 1.0f + __expf(-g)) * u; }

}  // namespace pmpe
