// The tree-plan computation for one tree (Section 3.4.2, "computed once per decode step"): depth and root-path list of
// every node, and for trees of more than 64 nodes the depth-first numbering cut into ancestor-closed groups, with one
// record per group appended to the unit list that the tensor-core verify kernel walks (see gdn_internal.cuh for the
// layouts).  A device function, so that it can run as a kernel of its own (gdn_plan.cu) or as extra CTAs in front of
// the commit kernel's (gdn_commit.cu: the fused call on trees of more than 64 nodes).  One CTA per tree, the more threads the
// shorter: bound by latency (a chain of shared-memory walks and barriers).  Root paths are walked in shared memory wherever
// they are needed, and the subtree sizes are counted on the way, one shared-memory atomic per node and ancestor: they return
// nothing and do not stand in the chain of the walk, while a vote on which lanes have met, to add as one, does (this grid on one
// tree of 512 nodes, geometric / best-first: 7.9 / 12.9 us with the vote, 6.4 / 8.9 so; within the commit's grid, 256 threads,
// three trees of 123 nodes: 7.4 / 10.0 and 6.4 / 7.6).
#pragma once

#include "gdn_internal.cuh"

namespace gdn {

constexpr int PLAN_THREADS = 512;   // of the plan kernel

struct PlanArgs {
    int n_seq, total_nodes, max_tree_nodes, max_depth;
    const int32_t *parent, *node_offsets, *n_nodes;   // node_offsets == nullptr: padded layout, node counts in n_nodes
    int32_t *tree_ok;
    uint8_t *depth;
    uint16_t *anc;
    uint8_t *anc8;
    uint16_t *dfs_node;
    uint8_t *dfs_depth, *dfs_anc8;
    uint16_t *group_start;
    int32_t *unit_count;
    uint4 *unit_list;
    int32_t *status_dev;
};

inline PlanArgs plan_args(const gdn_shape_t &s, const int32_t *parent, const int32_t *node_offsets,
                          const int32_t *n_nodes, const PlanPtrs &plan, int32_t *status_dev)
{
    return {s.n_seq, s.total_nodes, s.max_tree_nodes, s.max_depth, parent, node_offsets, n_nodes, plan.tree_ok,
            plan.depth, plan.anc, plan.anc8, plan.dfs_node, plan.dfs_depth, plan.dfs_anc8, plan.group_start,
            plan.unit_count, plan.unit_list, status_dev};
}

#ifdef __CUDACC__
template <int THREADS> __device__ __forceinline__ void plan_tree(const PlanArgs &a, const int b)
{
    const int n_seq = a.n_seq, total_nodes = a.total_nodes, max_tree_nodes = a.max_tree_nodes, max_depth = a.max_depth;
    const int32_t *__restrict__ parent = a.parent;
    const int32_t *__restrict__ node_offsets = a.node_offsets;
    const int32_t *__restrict__ n_nodes = a.n_nodes;
    int32_t *__restrict__ tree_ok = a.tree_ok;
    uint8_t *__restrict__ depth = a.depth;
    uint16_t *__restrict__ anc = a.anc;
    uint8_t *__restrict__ anc8 = a.anc8;
    uint16_t *__restrict__ dfs_node = a.dfs_node;
    uint8_t *__restrict__ dfs_depth = a.dfs_depth;
    uint8_t *__restrict__ dfs_anc8 = a.dfs_anc8;
    uint16_t *__restrict__ group_start = a.group_start;
    int32_t *unit_count = a.unit_count;
    uint4 *__restrict__ unit_list = a.unit_list;
    int32_t *status_dev = a.status_dev;

    __shared__ int size_s[GDN_GROUPED_MAX_NODES];        // subtree sizes
    __shared__ uint16_t left_s[GDN_GROUPED_MAX_NODES];   // nodes in the subtrees of earlier siblings
    __shared__ uint16_t pos_s[GDN_GROUPED_MAX_NODES];    // pre-order position of node i
    __shared__ uint8_t depth_at_s[GDN_GROUPED_MAX_NODES];   // depth of the node at pre-order position r
    __shared__ uint16_t node_at_s[GDN_GROUPED_MAX_NODES];   // the node itself
    __shared__ uint8_t depth_s[GDN_GROUPED_MAX_NODES];      // depth of node i
    __shared__ uint16_t gstart_s[GDN_MAX_GROUPS + 1];        // first position of each group (then the tree's size)
    // parent[] of this tree, staged once so that the root-path walks below run out of shared memory
    __shared__ int32_t par_s[GDN_MAX_TREE_NODES];
    if (b == 0 && threadIdx.x == 0) unit_count[1] = plan_magic(n_seq, max_tree_nodes, max_depth);
    // ragged packing: the tree's rows by node_offsets[]; padded layout: max_tree_nodes rows per tree, n_nodes[b] used
    const int lo = node_offsets ? node_offsets[b] : b * max_tree_nodes;
    const int hi = node_offsets ? node_offsets[b + 1] : lo + n_nodes[b];
    const int T = hi - lo;
    bool offsets_ok = lo >= 0 && T >= 0 && T <= max_tree_nodes && hi <= total_nodes;
    if (node_offsets && b == 0) offsets_ok = offsets_ok && lo == 0;
    if (node_offsets && b == n_seq - 1) offsets_ok = offsets_ok && hi == total_nodes;
    if (!offsets_ok) {
        if (threadIdx.x == 0) {
            report_status(status_dev, GDN_ERR_TREE);
            tree_ok[b] = 0;
            if (n_seq == 1) *unit_count = 0;
        }
        return;   // no record in the unit list: nothing of this tree is verified
    }
    const bool grouped = max_depth <= 16 && T > 64 && T <= GDN_GROUPED_MAX_NODES;
    for (int i = threadIdx.x; i < T; i += THREADS) {
        par_s[i] = parent[lo + i];
        if (grouped) size_s[i] = 0;
    }
    __syncthreads();
    int err = 0;
    for (int i = threadIdx.x; i < T; i += THREADS) {
        // up to the root, checking parent[]; each id is shifted into the list from below (the root ends up first)
        int d = 0, cur = i;
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = 0xFFFFFFFFu;
        while (cur >= 0) {
            if (grouped) atomicAdd(&size_s[cur], 1);   // node i lies in the subtrees of the nodes on its path
            const int p = par_s[cur];
            if (++d > max_depth) err = GDN_ERR_DEPTH;
            else if (p < -1 || p >= cur) err = GDN_ERR_TREE;
#pragma unroll
            for (int e = 7; e > 0; --e) w[e] = __funnelshift_l(w[e - 1], w[e], 16);
            w[0] = (w[0] << 16) | (uint32_t)cur;
            cur = err ? -1 : p;
        }
        if (err) continue;
        depth[lo + i] = (uint8_t)d;
        if (grouped) depth_s[i] = (uint8_t)d;
        uint16_t *row = anc + (size_t)(lo + i) * max_depth;
        if (max_depth == 16) {
            reinterpret_cast<uint4 *>(row)[0] = make_uint4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<uint4 *>(row)[1] = make_uint4(w[4], w[5], w[6], w[7]);
        } else {
            cur = i;
            for (int t = d - 1; t >= 0; --t) {
                row[t] = (uint16_t)cur;
                cur = par_s[cur];
            }
        }
        // the same list as bytes, one 16-byte row per node
        if (max_depth <= 16 && T <= 256)
            *reinterpret_cast<uint4 *>(anc8 + (size_t)(lo + i) * 16) =
                make_uint4(__byte_perm(w[0], w[1], 0x6420), __byte_perm(w[2], w[3], 0x6420), __byte_perm(w[4], w[5], 0x6420),
                           __byte_perm(w[6], w[7], 0x6420));
    }
    const int any_err = __syncthreads_or(err != 0);
    if (err) report_status(status_dev, err);
    if (threadIdx.x == 0) tree_ok[b] = any_err ? 0 : 1;
    if (any_err || !grouped) {
        // a tree that fits one tile is its own single group with the identity numbering, marked by n_prefix =
        // 0xFF (no group at all if the tree was rejected or is empty)
        // (a call with a single tree keeps the count itself; otherwise the counter was zeroed in front of this grid)
        const bool one = !any_err && T > 0 && T <= GDN_GROUP_TILE;
        if (threadIdx.x == 0 && n_seq == 1) *unit_count = one ? 1 : 0;
        if (threadIdx.x == 0 && one)
            unit_list[n_seq == 1 ? 0 : atomicAdd(unit_count, 1)] =
                make_uint4((uint32_t)b, (uint32_t)lo, (uint32_t)T << 16, 0xFFu | (1u << 8));
        return;
    }

    // Pre-order position = (#proper ancestors) + sum over the root path of the sizes of the subtrees
    // hanging off earlier siblings (roots count as siblings of one another; siblings by increasing id).
    // With a breadth-first numbering (parent[] non-decreasing, what tree builders emit) the siblings of a node are
    // its neighbours: the earlier ones are the run in front of it; any other topological numbering is searched.
    bool sorted_here = true;
    for (int i = threadIdx.x + 1; i < T; i += THREADS) sorted_here = sorted_here && par_s[i] >= par_s[i - 1];
    const bool sorted = __syncthreads_and(sorted_here);
    for (int i = threadIdx.x; i < T; i += THREADS) {
        const int p = par_s[i];
        int acc = 0;
        if (sorted) {
            for (int j = i - 1; j > p && par_s[j] == p; --j) acc += size_s[j];
        } else {
            for (int j = p + 1; j < i; ++j)
                if (par_s[j] == p) acc += size_s[j];
        }
        left_s[i] = (uint16_t)acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < T; i += THREADS) {
        const int d = depth_s[i];
        int pos = d - 1;
        for (int cur = i; cur >= 0; cur = par_s[cur]) pos += left_s[cur];
        pos_s[i] = (uint16_t)pos;
        dfs_node[lo + pos] = (uint16_t)i;
        node_at_s[pos] = (uint16_t)i;
        dfs_depth[lo + pos] = (uint8_t)d;
        depth_at_s[pos] = (uint8_t)d;
    }
    __syncthreads();
    // Groups: each takes as many positions as the tile leaves after the proper ancestors of its first node; their records
    // stand next to one another in the unit list
    __shared__ int list_base_s, n_groups_s;
    if (threadIdx.x == 0) {
        int start = 0, k = 0;
        while (start < T && k < GDN_MAX_GROUPS) {
            gstart_s[k++] = (uint16_t)start;
            start += GDN_GROUP_TILE - (depth_at_s[start] - 1);
        }
        n_groups_s = k;
        if (n_seq == 1) {
            *unit_count = k;
            list_base_s = 0;
        } else {
            list_base_s = atomicAdd(unit_count, k);
        }
        for (; k <= GDN_MAX_GROUPS; ++k) gstart_s[k] = (uint16_t)T;
    }
    __syncthreads();
    for (int k = threadIdx.x; k <= GDN_MAX_GROUPS; k += THREADS)
        group_start[(size_t)b * (GDN_MAX_GROUPS + 1) + k] = gstart_s[k];
    for (int k = threadIdx.x; k < GDN_MAX_GROUPS; k += THREADS) {
        const int g0 = gstart_s[k], own = gstart_s[k + 1] - g0;
        if (own > 0)   // (first position, own nodes, k), (n_prefix, groups of the tree, node at the first position)
            unit_list[list_base_s + k] =
                make_uint4((uint32_t)b, (uint32_t)lo, (uint32_t)g0 | ((uint32_t)own << 16) | ((uint32_t)k << 24),
                           (uint32_t)(depth_at_s[g0] - 1) | ((uint32_t)n_groups_s << 8) | ((uint32_t)node_at_s[g0] << 16));
    }
    // Root path of every node in the virtual indices of its group: an ancestor before the group's first
    // position is an ancestor of the group's first node and gets index depth-1; one inside the group gets
    // n_prefix + its offset in the group, n_prefix = depth(first node) - 1.
    for (int i = threadIdx.x; i < T; i += THREADS) {
        const int pos = pos_s[i];
        int k = 0;
        while (gstart_s[k + 1] <= pos) ++k;   // the group of this position (at most GDN_MAX_GROUPS steps)
        const int g0 = gstart_s[k];
        const int n_prefix = depth_at_s[g0] - 1;
        uint32_t w[4] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
        for (int t = depth_s[i] - 1, cur = i; t >= 0; --t, cur = par_s[cur]) {
            const int pa = pos_s[cur];
            const uint32_t v = pa < g0 ? (uint32_t)t : (uint32_t)(n_prefix + pa - g0);
            w[3] = __funnelshift_l(w[2], w[3], 8);
            w[2] = __funnelshift_l(w[1], w[2], 8);
            w[1] = __funnelshift_l(w[0], w[1], 8);
            w[0] = (w[0] << 8) | v;
        }
        *reinterpret_cast<uint4 *>(dfs_anc8 + (size_t)(lo + pos) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
#endif

}  // namespace gdn
