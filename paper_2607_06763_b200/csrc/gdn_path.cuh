// What the kernels that advance a state along an accepted path have in common: their arguments, the fetch of the path's rows
// and the check of the path with its per-step scalars.
#pragma once

#include "gdn_fragments.cuh"
#include "gdn_internal.cuh"

namespace gdn {

struct CommitParams {
    int h_qk, h_v, d_k, d_v, max_depth;
    float *S;
    const void *k, *v, *g, *beta;
    const int32_t *parent, *node_offsets, *path, *path_offsets;
    int32_t *status_dev;
    // padded layout (d_k = d_v = 128, bf16 only; t_pad = 0: ragged packing): slot b keeps its rows at b * t_pad and carries
    // tree b % n_trees, whose parent[] row, node count and accepted path are shared by its slots
    int t_pad, n_trees, path_stride, raw_gates;
    const int32_t *n_nodes, *path_len;
};

// The commit kernels and that of small trees are launched with programmatic stream serialization: a grid may become resident under
// the tail of the kernel in front of it and waits here before it reads or writes anything; the kernel behind it (a verification that
// waits for this grid in turn) may be made resident as the last CTAs run.  48 layers of two calls each (121 nodes, 32
// heads): 994 -> 850 us; verification and commit of 48 slots as two calls: 95.7 -> 92.3 us.
__device__ __forceinline__ void wait_for_previous_kernel()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
}

constexpr int CF_THREADS = 256;
constexpr int CF_MD = 16;

__device__ __forceinline__ void cf_cp_async_16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cf_cp_async_4(uint32_t dst, const void *src, bool valid)   // zero-fills where not valid
{
    const int n = valid ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// Rows of a path of 1 .. 16 steps on their way to shared memory (cp.async).
// Every thread reads the path entry whose row piece it fetches (no hand-over through shared memory in front of the
// row fetch); an entry outside the tree is skipped here and reported by the check below.  k rows word by word into the
// fragment order, zero up to the next multiple of eight rows.
__device__ __forceinline__ void path_rows_fetch(const CommitParams &p, int pp0, int len, int pb, int pT, int h, int hk, uint32_t pk,
                                                uint16_t *pv_s, int tid)
{
    const __nv_bfloat16 *k = static_cast<const __nv_bfloat16 *>(p.k), *v = static_cast<const __nv_bfloat16 *>(p.v);
#pragma unroll 2
    for (int idx = tid; idx < ((len + 7) & ~7) * 64; idx += CF_THREADS) {
        const int t = idx >> 6, w = idx & 63;
        int nt = t < len ? p.path[pp0 + t] : 0;
        const bool valid = t < len && nt >= 0 && nt < pT;
        if (!valid) nt = 0;
        cf_cp_async_4(pk + t * GDN_PK_STRIDE + path_row_word(w), k + ((size_t)(pb + nt) * p.h_qk + hk) * GDN_TILE_D + w * 2, valid);
    }
    if (tid < len * 16) {
        const int t = tid >> 4, c16 = tid & 15, nt = p.path[pp0 + t];
        if (nt >= 0 && nt < pT)
            cf_cp_async_16((uint32_t)__cvta_generic_to_shared(pv_s + t * GDN_TILE_D + c16 * 8),
                           v + ((size_t)(pb + nt) * p.h_v + h) * GDN_TILE_D + c16 * 8);
    }
}

// By one warp.  Lane t: entry t of the path and that node's parent; the path must be a chain from a root inside the tree
// (len 0: a path of an impossible length).  Writes the per-step scalars and the decay of the whole path, leaves g and beta
// of step `lane` in gt, be.  Returns the length, 0 if the path was rejected (and reported).
__device__ __forceinline__ int path_check_and_scalars(const CommitParams &p, int pp0, int len, int pb, int pT, int ppar, int h, int lane,
                                                      float &gt, float &be, float4 *scal_s, float &decay_s)
{
    const bool mine = lane < len;
    int n = -1, parent_n = -2;
    if (mine) {
        n = p.path[pp0 + lane];
        if (n >= 0 && n < pT) {
            if (p.parent) parent_n = p.parent[ppar + n];
            const size_t i = (size_t)(pb + n) * p.h_v + h;
            gt = gate_log_decay(static_cast<const unsigned short *>(p.g)[i], p.raw_gates != 0);
            be = gate_beta(static_cast<const unsigned short *>(p.beta)[i], p.raw_gates != 0);
        }
    }
    const int n_up = __shfl_up_sync(0xffffffffu, n, 1);
    bool bad = false;
    if (mine) {
        if (n < 0 || n >= pT) bad = true;
        else if (p.parent) bad = parent_n != (lane ? n_up : -1);
        else if (lane && n <= n_up) bad = true;   // without parent[] only the topological order can be checked
    }
    if (__any_sync(0xffffffffu, bad) || len == 0) {
        if (lane == 0) report_status(p.status_dev, GDN_ERR_PATH);
        len = 0;
    }
    // sums of g along the path over the lanes (up to and including step t, and behind it), and the per-step scalars
    float G = gt;
#pragma unroll
    for (int off = 1; off < CF_MD; off <<= 1) {
        const float up = __shfl_up_sync(0xffffffffu, G, off);
        if (lane >= off) G += up;
    }
    const float G_L = __shfl_sync(0xffffffffu, G, max(len - 1, 0));
    const float behind = DecayWindows(gt).sum(max(len - 1, 0), max(len - 1 - lane, 0));
    if (lane < len) scal_s[lane] = make_float4(be, be * expf(G), expf(behind), 0.f);
    if (lane == 0) decay_s = expf(G_L);
    return len;
}

// Trees of at most SS_MAX_NODES nodes on the shapes of the tensor-core path (gdn_step_small.cu): the verification, behind the commit of
// `prev` in the same pass over the state if with_commit, else on prev.S as it is (of prev only the sizes, raw_gates, S and
// status_dev count then).  node_offsets == nullptr: padded layout.
// plan: the padded layout with node counts and root paths out of a plan (no parent, n_nodes), verification alone.
constexpr int SS_MAX_NODES = 32;
struct SmallTreePlan {
    const uint4 *unit_list = nullptr;
    const int32_t *unit_count = nullptr;   // [0] records in the list, [1] what plan_magic says of the plan's shape
    const uint8_t *anc8 = nullptr;
    int capacity = 0, magic = 0;
};
bool step_small_supported(const gdn_shape_t &s);
cudaError_t launch_step_small(const gdn_shape_t &s, const CommitParams &prev, bool with_commit, const void *q, const void *k, const void *v,
                              const void *g, const void *beta, const int32_t *parent, const int32_t *node_offsets, int n_trees,
                              const int32_t *n_nodes, void *o, cudaStream_t stream, const SmallTreePlan &plan = {});

}  // namespace gdn
