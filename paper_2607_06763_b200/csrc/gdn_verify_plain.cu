// Tree verification alone on the sm_100a tensor cores: d_k = d_v = 128, bf16 inputs, root paths of at most 16 nodes, at
// most 64 nodes per unit of work (larger trees are cut into ancestor-closed groups, each a unit of its own).
//
// It evaluates the triangular form of Section 3.4.1 (Eq. 9-11) restricted to real ancestors, with the W S0 term folded
// into the right-hand side as in Section 3.4.2, rearranged so that everything but one contraction is independent of the
// state.  Along the root path of node i, with kappa_jt = k_j.k_t and gamma_it = q_i.k_t, the decays factor out of the
// back-substitution: the weights
//     w_it = beta_t (gamma_it - sum_{l > t} w_il kappa_lt)                 (t, l on the root path of i)
// are those of the undecayed delta rule, and Eq. 11 reads
//     o_i = S0^T [ sa_i (q_i - sum_t w_it k_t) ] + sum_t [ scale exp(G_i - G_t) w_it ] v_t,    sa_i = scale exp(G_i),
// G_i = sum of g along the root path.  The bracket next to S0 is a modified query q'_i, so a node costs one product with
// the state instead of two (S0^T k and S0^T q), and no right-hand side has to be formed per node and component:
//     coefficients:  Gram = [k;q].k^T -> w -> C = -sa w.K -> q' = sa q + C
//     output:        O [d_v x nodes] = V^T.z' + S0.q'^T                            z'_it = scale exp(G_i - G_t) w_it
// Contractions run on the 5th-generation tensor cores (tcgen05.mma, bf16 operands, fp32 accumulators in tensor memory);
// k, q and v are exact bf16 operands, fp32 quantities are split into two bf16 terms (x = hi + lo, |x - hi - lo| <=
// 2^-17 |x|): w, z', q' and S0; the lo.lo term of q'.S0^T is dropped.  The state operand is the one that lives in tensor
// memory: the tile goes there from registers without passing through shared memory.
//
// Measured against the kernel that formed S0^T k and S0^T q and a right-hand side per node (same two CTAs per SM): 48
// slots x 32 heads, 64-node tree, verification then commit as two calls 110 -> 84 us (the commit from 48 to 43 of it);
// 256-node trees, fused call (commit kernel + this one) 324 -> 263 us; 32 ragged trees of 16..256 nodes 132 -> 121 us; one
// layer of 512 nodes, plan included, 29.7 -> 24.7 us.
//
// What bounds it: the chain of a unit (Gram -> lists -> back-substitution -> C -> q' -> output product -> rows), not memory
// and not the tensor pipe; so the unit has as few instructions and barriers as could be found, two CTAs share an SM and
// fill each other's waits, and a CTA takes neighbouring units, which have much in common.
#include "gdn_internal.cuh"
#include "gdn_path.cuh"
#include "gdn_replay.cuh"
#include "gdn_tc.cuh"

namespace gdn {

namespace {

constexpr int VP_THREADS = 256;
constexpr int VP_D = 128;           // d_k = d_v
constexpr int VP_T = 64;            // max nodes per unit
constexpr int VP_MD = 16;           // max nodes on a root path

// tensor memory columns.  C has its 64 rows (nodes) on 16 of the 32 lanes of a warp's quarter: the two 64-column halves
// of its 128 columns go to lane offsets 0 and 16 of the same tensor-memory columns, so that a 32-lane load returns 32
// useful rows: lanes 0-15 = nodes 16 w + l, components 0..63; lanes 16-31 = the same nodes, components 64..127.
constexpr int TM_GC = 0;            // 64: Gram block of the unit to come (lanes: k rows then q rows), then C
constexpr int TM_O = 64;            // 64: outputs, value components on the lanes, nodes on the columns
constexpr int TM_S = 128;           // 2 x 64: state operand hi, lo: value components on the lanes, bf16 pairs of the key dimension
constexpr int TM_COLS = 256;

// shared memory map (bytes from a 1024-byte aligned base); tiles are 128-byte swizzled, [64-column half][rows][128 B]
constexpr int SP_KQ = 0;                         // [2][128 rows: k 0..63, q 64..127][128 B]
constexpr int SP_V = 32768;                      // v rows: [2][64 rows][128 B]
constexpr int SP_WZ = 49152;                     // -sa w hi, lo, z' hi, lo: 8 KB each, [64 rows = nodes i][64 nodes j];
                                                 // then q' hi, lo: 16 KB each, [2][64 rows = nodes][128 B];
                                                 // then the output rows [64][128] TOut
constexpr int SP_KAPPA = 81920;                  // fp32 [64][16] kappa(i, t): t-th proper ancestor of i (root first); the
                                                 // four-entry piece p of row i sits at place p ^ ((i >> 1) & 3)
constexpr int SP_GAMMA = 86016;                  // fp32 [64][16] gamma(i, t), i itself included; same places
constexpr int SP_ANC = 90112;                    // u8 [64][16] root path, root first, node itself last (0xFF = unused)
constexpr int SP_AMASK = 91136;                  // u64 [64]: ancestors of i and i itself as bits (0 beyond the tree)
constexpr int SP_BETA = 91648;                   // float [64]: beta_i
constexpr int SP_SA = 92160;                     // float [64]: scale exp(G_i)
constexpr int SP_G = 92416;                      // float [64]: g_i; from step (6) on of the next unit
constexpr int SP_PAR = 92672;                    // s8 [64]: its parents
constexpr int SP_VN = 92736;                     // u16 [64]: grouped mode, node id of virtual index u
constexpr int SP_BAD = 92864;                    // int: the unit's tree was rejected (nothing of it is stored)
constexpr int SP_FLAG = 92868;                   // u32: a bounded wait expired
constexpr int SP_TMEM = 92872;                   // u32: tensor memory base
constexpr int SP_MBAR = 92880;                   // u64 [5]: Gram, C, O done; k/q, v rows landed
constexpr int SP_BYTES = SP_MBAR + 40;
constexpr int SP_ALLOC = SP_BYTES + 1024;        // slack for the 1024-byte alignment of the base

struct VerifyPlainParams {
    // TMA descriptors of the packed k, q, v tensors viewed as [N][heads][128] bf16 (not used by the grouped mode)
    alignas(64) CUtensorMap tm_k;
    alignas(64) CUtensorMap tm_q;
    alignas(64) CUtensorMap tm_v;
    int h_qk, h_v;
    int n_units;        // n_seq * h_v (grouped mode: an upper bound that only sizes the grid)
    int box_rows;       // rows of a TMA box: the largest tree rounded up to 16
    float scale;
    const float *S0;
    const __nv_bfloat16 *q, *k, *v, *g, *beta;
    const int32_t *node_offsets;
    const int32_t *parent;                             // trees of at most 64 nodes: the kernel builds the metadata itself
    int n_seq, total_nodes, max_tree_nodes, max_depth;
    void *o;
    int32_t *status_dev;
    // Padded layout of Section 3.4.2 (t_pad = 0: ragged packing by node_offsets[]): slot b keeps its nodes in rows
    // b * t_pad .. and carries tree b % n_trees, whose parent[] row and node count are shared by all the slots (layers).
    int t_pad, n_trees;
    const int32_t *n_nodes;
    int raw_gates;                                     // g / beta arrive as raw gate inputs ("scalars" stage on chip)
    int state_late;                                    // the kernel in front writes the state alone (see the wait)
    // grouped verification of trees with more than 64 nodes (only read by the GROUPED instantiation)
    int groups_per_tree, anc_stride;                   // upper bound of the groups of a tree (sizes the grid); entries
                                                       // per row of anc16
    const uint8_t *anc8, *dfs_anc8;
    const uint16_t *anc16, *dfs_node;
    const uint4 *unit_list;                            // one record per group (see the workspace layout)
    const int32_t *unit_count;                         // [0] records in the list, [1] plan_magic of the plan's shape
    int unit_capacity, plan_magic;                     // what the list can hold; what [1] has to read
};

// PADDED: dense layout (rows and tree of a slot by arithmetic, trees shared by slots, raw gate inputs).
// GROUPED (trees of more than 64 nodes, cut into ancestor-closed groups by the plan kernel): a unit is (tree, value
// head, group); it is verified as a virtual tree of the <= 15 proper ancestors of the group's first node followed by the
// group's own nodes, its rows are gathered with cp.async, its tables come from the plan, and outputs are stored for the
// group's own nodes only.
//
// A CTA takes a contiguous run of the units in the order (slot, head) -- GROUPED: (layer, tree, head, group) -- so that
// what neighbouring units have in common is made once: k/q rows, Gram block and lists for the value heads of a key head,
// the state operand for the groups of a tree.  Nothing a unit can know in advance is waited for inside it: the next unit's
// rows stream in as soon as this one's are dead, its Gram block is issued at the end of this one, and its tables are
// fetched in stages, each global load issued one phase before its value is used.
template <typename TOut, bool PADDED, bool GROUPED>
__global__ void __launch_bounds__(VP_THREADS, 2) verify_plain_kernel(const __grid_constant__ VerifyPlainParams p)
{
    extern __shared__ uint8_t vp_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(vp_smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    volatile uint32_t *flag = reinterpret_cast<volatile uint32_t *>(smem + SP_FLAG);
    const uint32_t mbar_g = sbase + SP_MBAR, mbar_c = mbar_g + 8, mbar_o = mbar_g + 16;
    const uint32_t mbar_kq = mbar_g + 24, mbar_v = mbar_g + 32;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    // The asynchronous work is issued by one elected lane each of four warps: warp 0 C, warp 1 V^T.z' and the last product,
    // warp 2 the Gram block of the unit to come, warp 3 the TMA loads; warps 2 and 3 also keep the tree tables (thread
    // 64 + i: node i).
    constexpr int W_MMA_C = 0, W_MMA_O = 1, W_MMA_G = 2, W_TMA = 3;
    const int tnode = tid - 64;
    const bool tbl_thread = tid >= 64 && tid < 64 + VP_T;
    // neighbouring CTAs of the unit order share an SM (CTA i and i + grid / 2 do, as far as the hardware deals them out in
    // order), so that the SMs differ by one unit at most
    const int half_grid = (int)gridDim.x >> 1;
    const int cta = p.n_units <= (int)gridDim.x || (gridDim.x & 1) ? (int)blockIdx.x
                    : (int)blockIdx.x < half_grid ? 2 * (int)blockIdx.x : 2 * ((int)blockIdx.x - half_grid) + 1;

    if (warp == 0) tmem_alloc(sbase + SP_TMEM, TM_COLS);
    if (tid == 32) {
        mbar_init(mbar_g, 1);
        mbar_init(mbar_c, 2);   // C and V^T.z'
        mbar_init(mbar_o, 1);
        mbar_init(mbar_kq, GROUPED ? VP_THREADS : 1);   // gathered rows: every thread arrives once its copies have landed
        mbar_init(mbar_v, GROUPED ? VP_THREADS : 1);
        *flag = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(smem + SP_TMEM), 0);
    // Launched with programmatic stream serialization: everything above overlaps the tail of the kernel in front (the
    // previous call, or the plan kernel); nothing that is computed from memory may run before that kernel's writes are
    // visible.  L2 can be asked for the first unit's state tile and rows meanwhile (a prefetch consumes nothing): where
    // the rows are may depend on node_offsets[], which the kernel in front may still be writing, so the value read here
    // only steers prefetches (clamped to the tensors), and comes from L2: nothing of it stays in L1 for the read that counts.
    const int u_first = (int)((long long)p.n_units * cta / (int)gridDim.x);   // (not GROUPED)
    if constexpr (!GROUPED) {
        if (tid < 4) prefetch_l2_bulk(p.S0 + (size_t)u_first * VP_D * VP_D + (size_t)tid * 4096, 16384);
        if (!p.state_late && tid >= 128 && tid < 128 + VP_T && tid - 128 < p.max_tree_nodes) {
            const int ub = u_first / p.h_v, uh = u_first % p.h_v, uhk = uh / (p.h_v / p.h_qk);
            const int row = (PADDED ? ub * p.t_pad : __ldcg(p.node_offsets + ub)) + tid - 128;
            if (row >= 0 && row < p.total_nodes) {
                prefetch_l2_bulk(p.v + ((size_t)row * p.h_v + uh) * VP_D, 256);
                prefetch_l2_bulk(p.k + ((size_t)row * p.h_qk + uhk) * VP_D, 256);
                prefetch_l2_bulk(p.q + ((size_t)row * p.h_qk + uhk) * VP_D, 256);
                asm volatile("prefetch.global.L2 [%0];" ::"l"(p.g + (size_t)row * p.h_v + uh));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(p.beta + (size_t)row * p.h_v + uh));
            }
        }
    }
    // state_late: the kernel in front is the commit of the same call, which itself has waited for everything before it and
    // writes nothing but the state; only the first use of a state tile waits for it (and the rows are loaded right away:
    // prefetches would only stand in front of the loads, one layer 9.4 -> 11.7 us).
    bool state_late = !GROUPED && p.state_late;
    auto wait_for_previous_kernel = [&]() {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // ... and whatever is launched behind this grid with the same attribute (the next call's kernel, which itself waits
        // for this grid to complete before it reads or writes anything) may be made resident as CTAs leave.
        asm volatile("griddepcontrol.launch_dependents;");
    };
    if (!state_late) wait_for_previous_kernel();

    // ------------------------------------------------------------------------------------ the units of this CTA
    // Unit = slot b * h_v + head h; GROUPED: E = records in the plan's list (the groups of a tree next to one another),
    // E * h_v * layers units in the order (layer, tree, head, group).
    int u_end, n_records = 1;
    const int ratio = p.h_v / p.h_qk;
    const int ratio_shift = (ratio & (ratio - 1)) == 0 ? 31 - __clz(ratio) : -1;
    auto hk_of = [&](int h_) -> int { return ratio_shift >= 0 ? h_ >> ratio_shift : h_ / ratio; };
    auto tree_of = [&](int b_) -> int { return p.n_trees == 1 ? 0 : b_ % p.n_trees; };   // padded layout only
    struct Cursor { int u, b, h, rec; };        // GROUPED: b = layer, rec = index of the group's record
    struct Raw { int lo, hi; uint4 rec; };
    // A unit: slot, head, first row, nodes; par0 = first entry of the tree in parent[].  GROUPED: pb = first row of the
    // tree in the plan's tables, g0 = first depth-first position of the group, n_prefix = proper ancestors of its first
    // node (virtual indices 0 .. n_prefix - 1), first = node at position g0; ident: a tree of at most 64 nodes inside a
    // grouped call (identity numbering); fresh: first unit of this CTA on its state tile.
    struct Unit { int b, h, base, T, par0, pb, g0, n_prefix, first; bool ident, fresh; };
    Cursor cur{0, 0, 0, 0};
    if constexpr (GROUPED) {
        // the plan kernel has counted the groups of all trees
        int n_rec = reinterpret_cast<const volatile int32_t *>(p.unit_count)[0];
        if (reinterpret_cast<const volatile int32_t *>(p.unit_count)[1] != p.plan_magic || n_rec < 0 ||
            n_rec > p.unit_capacity) {   // not a plan of this shape (never built, or built for other sizes)
            if (tid == 0) report_status(p.status_dev, GDN_ERR_WORKSPACE);
            n_rec = 0;
        }
        const int n_layers = PADDED ? p.n_seq / p.n_trees : 1;
        n_records = n_rec > 0 ? n_rec : 1;
        const long long total = (long long)n_rec * p.h_v * n_layers;
        // (the grid is sized by an upper bound: when every CTA has one unit at most, the first ones have it, which stand on
        // SMs of their own as far as those go -- 110 units on a grid of 168: 14.3 us spread over the grid, 11.9 so)
        const bool one_each = total <= (int)gridDim.x;
        cur.u = one_each ? min((int)blockIdx.x, (int)total) : (int)(total * cta / (int)gridDim.x);
        u_end = one_each ? min((int)blockIdx.x + 1, (int)total) : (int)(total * (cta + 1) / (int)gridDim.x);
        if (cur.u < u_end) {
            cur.b = cur.u / (n_records * p.h_v);
            const int r = cur.u - cur.b * n_records * p.h_v, pos = r / p.h_v;
            const uint4 rec = p.unit_list[pos];   // written by the plan kernel in front of this grid: no read-only path
            const int n_groups = (int)((rec.w >> 8) & 0xFFu), head_rec = pos - (int)(rec.z >> 24);
            const int local = r - head_rec * p.h_v;
            cur.h = local / n_groups;
            cur.rec = head_rec + local - cur.h * n_groups;
        }
    } else {
        cur.u = u_first;
        u_end = (int)((long long)p.n_units * (cta + 1) / (int)gridDim.x);
        cur.b = cur.u / p.h_v;
        cur.h = cur.u - cur.b * p.h_v;
    }
    // The loads a decode needs are issued one unit ahead.
    auto load_raw = [&](const Cursor &c) -> Raw {
        Raw r{0, 0, make_uint4(0u, 0u, 0u, 0u)};
        if (c.u >= u_end) return r;
        if constexpr (GROUPED) {
            r.rec = p.unit_list[c.rec];
        } else if (PADDED) {
            r.lo = p.n_nodes[tree_of(c.b)];
        } else {
            r.lo = p.node_offsets[c.b];
            r.hi = p.node_offsets[c.b + 1];
        }
        return r;
    };
    Raw raw = load_raw(cur);
    bool first_unit = true;
    // The next unit that has work (false: none left).  A tree with inconsistent node_offsets[] (reported) or no nodes is
    // skipped.
    auto pull = [&](Unit &un) -> bool {
        while (cur.u < u_end) {
            bool ok;
            un.h = cur.h;
            if constexpr (GROUPED) {
                const int tree = (int)raw.rec.x, grp = (int)(raw.rec.z >> 24), n_groups = (int)((raw.rec.w >> 8) & 0xFFu);
                if (PADDED) {   // slot = layer * n_trees + tree
                    un.b = cur.b * p.n_trees + tree;
                    un.base = un.b * p.t_pad;
                    un.pb = tree * p.t_pad;
                } else {
                    un.b = tree;
                    un.base = (int)raw.rec.y;   // checked by the plan kernel (a tree with bad offsets has no record)
                    un.pb = un.base;
                }
                un.g0 = (int)(raw.rec.z & 0xFFFFu);
                un.ident = (raw.rec.w & 0xFFu) == 0xFFu;
                un.n_prefix = un.ident ? 0 : (int)(raw.rec.w & 0xFFu);
                un.first = (int)(raw.rec.w >> 16);
                un.T = un.n_prefix + (int)((raw.rec.z >> 16) & 0xFFu);
                un.par0 = 0;
                un.fresh = first_unit || grp == 0;
                ++cur.u;
                if (grp + 1 < n_groups) {
                    ++cur.rec;
                } else if (++cur.h < p.h_v) {
                    cur.rec -= grp;
                } else {
                    cur.h = 0;
                    if (++cur.rec >= n_records) {
                        cur.rec = 0;
                        ++cur.b;
                    }
                }
                ok = true;
            } else {
                un.b = cur.b;
                bool off_ok;
                if (PADDED) {   // padded layout: rows of the slot, node count and parent[] row of its tree
                    un.base = un.b * p.t_pad;
                    un.T = raw.lo;
                    un.par0 = tree_of(un.b) * p.t_pad;
                    off_ok = un.T >= 0 && un.T <= VP_T && un.T <= p.t_pad;
                } else {
                    un.base = raw.lo;
                    un.T = raw.hi - raw.lo;
                    un.par0 = un.base;
                    off_ok = un.base >= 0 && un.T >= 0 && un.T <= VP_T && un.T <= p.max_tree_nodes && raw.hi <= p.total_nodes;
                    if (un.b == 0) off_ok = off_ok && un.base == 0;
                    if (un.b == p.n_seq - 1) off_ok = off_ok && raw.hi == p.total_nodes;
                }
                if (!off_ok && tid == 0) report_status(p.status_dev, GDN_ERR_TREE);
                ok = off_ok && un.T > 0;
                un.fresh = true;
                ++cur.u;
                if (++cur.h == p.h_v) {
                    cur.h = 0;
                    ++cur.b;
                }
            }
            first_unit = false;
            raw = load_raw(cur);
            if (ok) return true;
        }
        return false;
    };

    // ------------------------------------------------------------------------------------ rows
    // node id of virtual index u (< T) of a group, from the plan (written by the kernel in front: no read-only path)
    auto vnode_of = [&](const Unit &un, int u) -> int {
        if (un.ident) return u;
        if (u < un.n_prefix) return (int)p.anc16[(size_t)(un.pb + un.first) * p.anc_stride + u];
        return (int)p.dfs_node[un.pb + un.g0 + u - un.n_prefix];
    };
    uint16_t *vnode_s = reinterpret_cast<uint16_t *>(smem + SP_VN);   // node ids of the unit whose rows are asked for next
    // k/q rows (rows 0..63 = k, 64..127 = q) by TMA: four boxes, 128-byte swizzled.  A box always spans box_rows rows: rows
    // beyond the tree belong to the next tree (or are zero past the end of the tensor), every use of them is masked.
    // GROUPED: gathered row by row with cp.async (zero-filled beyond the unit).
    auto issue_kq = [&](const Unit &un) {
        const int hk = hk_of(un.h);
        if constexpr (GROUPED) {
            const int r16 = tid >> 4, c16 = tid & 15;
#pragma unroll 2
            for (int u = r16; u < VP_T; u += 16) {
                const size_t off = ((size_t)(un.base + vnode_s[u]) * p.h_qk + hk) * VP_D + c16 * 8;
                cp_async_16(sbase + SP_KQ + sw128_offset(u, c16), p.k + off, u < un.T);
                cp_async_16(sbase + SP_KQ + sw128_offset(VP_T + u, c16), p.q + off, u < un.T);
            }
            cp_async_arrive_on(mbar_kq);
        } else if (warp == W_TMA && elect_one()) {
            mbar_expect_tx(mbar_kq, (uint32_t)p.box_rows * 512u);
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {
                tma_load_3d(sbase + SP_KQ + kh * 16384, &p.tm_k, kh * 64, hk, un.base, mbar_kq);
                tma_load_3d(sbase + SP_KQ + kh * 16384 + 8192, &p.tm_q, kh * 64, hk, un.base, mbar_kq);
            }
        }
    };
    auto issue_v = [&](const Unit &un) {
        if constexpr (GROUPED) {
            const int r16 = tid >> 4, c16 = tid & 15;
#pragma unroll 2
            for (int u = r16; u < VP_T; u += 16)
                cp_async_16(sbase + SP_V + (c16 >> 3) * 8192 + sw128_row_offset(u, c16 & 7),
                            p.v + ((size_t)(un.base + vnode_s[u]) * p.h_v + un.h) * VP_D + c16 * 8, u < un.T);
            cp_async_arrive_on(mbar_v);
        } else if (warp == W_TMA && elect_one()) {
            mbar_expect_tx(mbar_v, (uint32_t)p.box_rows * 256u);
            tma_load_3d(sbase + SP_V, &p.tm_v, 0, un.h, un.base, mbar_v);
            tma_load_3d(sbase + SP_V + 8192, &p.tm_v, 64, un.h, un.base, mbar_v);
        }
    };
    // Gram = [k;q].k^T of the rows that are landing, into the columns that C has left.
    auto issue_gram = [&](int T, uint32_t kq_parity) {
        if (warp == W_MMA_G && elect_one()) {
            if (!mbar_wait_bounded(mbar_kq, kq_parity)) *flag = 1;
            if constexpr (GROUPED) fence_proxy_async();   // rows written by cp.async become visible to the tensor core
            tc_fence_after();
            const uint64_t b_kq = smem_desc_sw128(sbase + SP_KQ);
            const uint32_t id = idesc_bf16(128, 0) | (uint32_t)(max(1, (T + 15) >> 4) * 2) << 17;   // as many k rows as there are
#pragma unroll 2
            for (int ks = 0; ks < 8; ++ks) {
                const uint64_t adv = (uint64_t)((ks >> 2) * 1024 + (ks & 3) * 2);
                umma_bf16(tmem + TM_GC, b_kq + adv, b_kq + adv, id, ks > 0);
            }
            umma_commit(mbar_g);
        }
    };

    // ------------------------------------------------------------------------------------ tree tables
    // Thread 64 + i keeps node i.  tables_load() asks for its parent and gates (registers), tables_put() stages parent and
    // log decay in shared memory, and behind a barrier tables_build() climbs from the node to its root, shifting each id
    // into a 16-byte row from below (the root ends up in byte 0), collecting the ancestor mask and the path sum of g.  A
    // tree with a bad parent[] or a root path of more than max_depth nodes is reported and runs as a tree of no nodes.  A
    // climb is a chain of shared-memory loads: the units of a tree share the rows (and the verdict) of its first one, and
    // GROUPED takes them, in virtual indices, from the plan; what is left is the sum of g over the row.
    signed char *par_s = reinterpret_cast<signed char *>(smem + SP_PAR);
    float *g_s = reinterpret_cast<float *>(smem + SP_G);
    volatile int *bad_s = reinterpret_cast<volatile int *>(smem + SP_BAD);
    struct NodeRaw { int par, node; uint32_t g, beta; };
    auto gates_load = [&](const Unit &un, NodeRaw &nr) {
        if (tbl_thread && tnode < un.T) {
            const size_t n = (size_t)(un.base + nr.node) * p.h_v + un.h;
            nr.g = __ldg(reinterpret_cast<const unsigned short *>(p.g) + n);
            nr.beta = __ldg(reinterpret_cast<const unsigned short *>(p.beta) + n);
        }
    };
    auto tables_load = [&](const Unit &un, NodeRaw &nr, const bool same_tree) {
        nr.par = -1;
        nr.node = 0;
        nr.g = nr.beta = 0;
        if (tbl_thread && tnode < un.T) {
            nr.node = tnode;
            if constexpr (GROUPED) {
                nr.node = vnode_of(un, tnode);
                if (!un.ident && tnode < un.n_prefix) {   // an ancestor of the group's first node: its path is 0..tnode
                    const uint32_t ids[4] = {0x03020100u, 0x07060504u, 0x0B0A0908u, 0x0F0E0D0Cu};
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int n = min(max(tnode + 1 - 4 * e, 0), 4);
                        w[e] = n == 4 ? ids[e] : ids[e] | 0xFFFFFFFFu << (8 * n);
                    }
                    *reinterpret_cast<uint4 *>(smem + SP_ANC + tnode * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                } else {   // (the rows of the unit before have been read)
                    cp_async_16(sbase + SP_ANC + tnode * 16, un.ident ? p.anc8 + (size_t)(un.pb + tnode) * 16
                                                                      : p.dfs_anc8 + (size_t)(un.pb + un.g0 + tnode - un.n_prefix) * 16, true);
                    asm volatile("cp.async.commit_group;" ::: "memory");
                }
            } else {
                if (!same_tree) nr.par = __ldg(p.parent + un.par0 + tnode);
                gates_load(un, nr);
            }
        }
    };
    bool my_bad = false;
    auto tables_put = [&](const Unit &un, const NodeRaw &nr, const bool same_tree) {
        if (tbl_thread) {
            if (!GROUPED && !same_tree) {
                int pv = nr.par;
                my_bad = tnode < un.T && (pv < -1 || pv >= tnode);
                if (my_bad) pv = -1;
                par_s[tnode] = (signed char)pv;
            }
            g_s[tnode] = gate_log_decay(nr.g, PADDED && p.raw_gates);
            if constexpr (GROUPED) vnode_s[tnode] = (uint16_t)nr.node;
        }
        if (tid == 0 && !same_tree) *bad_s = 0;
    };
    auto tables_build = [&](const Unit &un, const NodeRaw &nr, const bool same_tree) {
        if (!tbl_thread) return;
        float G = 0.f;
        if (GROUPED || same_tree) {
            if constexpr (GROUPED) asm volatile("cp.async.wait_group 0;" ::: "memory");   // (the row copies are in no group)
            uint4 path = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
            if (tnode < un.T) path = *reinterpret_cast<const uint4 *>(smem + SP_ANC + tnode * 16);
            const uint32_t w[4] = {path.x, path.y, path.z, path.w};
            uint32_t mlo = 0, mhi = 0;
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (!__any_sync(0xffffffffu, w[e] != 0xFFFFFFFFu)) break;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint32_t id = (w[e] >> (8 * c)) & 0xFFu;
                    const float gv = g_s[id & 63u];
                    if (id != 0xFFu) sum[c] += gv;
                    if constexpr (GROUPED) {
                        if (id < 32u) mlo |= 1u << id;
                        else if (id < 64u) mhi |= 1u << (id - 32u);
                    }
                }
            }
            G = (sum[0] + sum[1]) + (sum[2] + sum[3]);
            if constexpr (GROUPED) {
                if (tnode >= un.T) *reinterpret_cast<uint4 *>(smem + SP_ANC + tnode * 16) = path;
                *reinterpret_cast<uint2 *>(smem + SP_AMASK + tnode * 8) = make_uint2(mlo, mhi);
            }
        } else {
            int d = 0, err = my_bad ? GDN_ERR_TREE : 0, c = tnode < un.T && !err ? tnode : -1;
            uint32_t w0 = 0xFFFFFFFFu, w1 = 0xFFFFFFFFu, w2 = 0xFFFFFFFFu, w3 = 0xFFFFFFFFu, mlo = 0, mhi = 0;
#pragma unroll 1
            while (c >= 0) {
                if (++d > p.max_depth) { err = GDN_ERR_DEPTH; break; }
                const int up = par_s[c];
                w3 = __funnelshift_l(w2, w3, 8);
                w2 = __funnelshift_l(w1, w2, 8);
                w1 = __funnelshift_l(w0, w1, 8);
                w0 = (w0 << 8) | (uint32_t)c;
                if (c < 32) mlo |= 1u << c;
                else mhi |= 1u << (c - 32);
                G += g_s[c];
                c = up;
            }
            if (err) {
                mlo = mhi = 0;
                report_status(p.status_dev, err);
                *bad_s = 1;
            }
            *reinterpret_cast<uint4 *>(smem + SP_ANC + tnode * 16) = make_uint4(w0, w1, w2, w3);
            *reinterpret_cast<uint2 *>(smem + SP_AMASK + tnode * 8) = make_uint2(mlo, mhi);
        }
        reinterpret_cast<float *>(smem + SP_BETA)[tnode] = gate_beta(nr.beta, PADDED && p.raw_gates);
        reinterpret_cast<float *>(smem + SP_SA)[tnode] = p.scale * __expf(G);
    };

    // ------------------------------------------------------------------------------------ first unit
    Unit un{}, nx{};
    NodeRaw nr{-1, 0, 0u, 0u};
    bool have = pull(un);
    uint32_t rows_parity = 0, gram_parity = 0, par = 0;   // phases of the barriers
    if (have) {
        if constexpr (!GROUPED) {
            issue_kq(un);
            issue_v(un);
        }
        tables_load(un, nr, false);
        if constexpr (GROUPED) gates_load(un, nr);
        tables_put(un, nr, false);
    }
    __syncthreads();
    if (have) {
        if constexpr (GROUPED) {
            issue_kq(un);
            issue_v(un);
        }
        tables_build(un, nr, false);
        issue_gram(un.T, 0);
        rows_parity = 1;
    }
    bool new_rows = true;

    const int quarter = warp & 3, hh = warp >> 2;   // tensor-memory lanes 32 * quarter .. of this warp
    const int row0 = 32 * quarter + 16 * hh;        // value components of this warp: state rows, output lanes
    const uint32_t t_lane = tmem + ((uint32_t)(32 * quarter) << 16);
#pragma unroll 1
    while (have) {
        // State tile, as 16 x 8 fragments in a permuted column order: lane = 4 g + l4 holds rows g and g + 8 of the warp's
        // sixteen, and of each the key positions 32 jj + 8 l4 + e (e = 0..7) as x[4 jj + (e >> 1)][2 r + (e & 1)], i.e. 32
        // contiguous bytes per lane and load.  Asked for at the top, needed behind the coefficients; in two pieces, or, beside
        // the row copies of the grouped mode, in four (256-node trees, fused call: 278.5 -> 275.5 us; plain trees are 2 % slower
        // that way).
        float x[16][4];
        const size_t tile = (size_t)(un.b * p.h_v + un.h) * VP_D * VP_D + (size_t)(row0 + (lane >> 2)) * VP_D + (lane & 3) * 8;
        auto load_state = [&](int j0, int j1) {
            if (!GROUPED || un.fresh) {
#pragma unroll
                for (int jj = j0; jj < j1; ++jj)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        float4 a, b;
                        ldg_v8(p.S0 + tile + r * 8 * VP_D + jj * 32, a, b);
                        x[4 * jj + 0][2 * r] = a.x; x[4 * jj + 0][2 * r + 1] = a.y; x[4 * jj + 1][2 * r] = a.z; x[4 * jj + 1][2 * r + 1] = a.w;
                        x[4 * jj + 2][2 * r] = b.x; x[4 * jj + 2][2 * r + 1] = b.y; x[4 * jj + 3][2 * r] = b.z; x[4 * jj + 3][2 * r + 1] = b.w;
                    }
            }
        };
        if (!state_late) load_state(0, GROUPED ? 1 : 2);
        if (new_rows) {
            if (!mbar_wait_bounded(mbar_kq, gram_parity)) *flag = 1;
            if (!mbar_wait_bounded(mbar_g, gram_parity)) *flag = 1;
            tc_fence_after();
            gram_parity ^= 1;
        }
        __syncthreads();   // tables; the output stage has been read
        if (!state_late) load_state(GROUPED ? 1 : 2, GROUPED ? 2 : 4);
        // a tree whose parent[] was rejected while its tables were built runs as a tree of no nodes
        const bool bad = *bad_s != 0;
        const int T = bad ? 0 : un.T;
        if (new_rows) {
            // (1) entries of the Gram rows that belong to ancestors -> lists by path position (an ancestor has a smaller index
            // than its descendants, so that ascending columns are ascending positions): kappa (k rows, proper ancestors),
            // gamma (q rows).  The value heads of a key head share the lists.
            const int node = (quarter & 1) * 32 + lane;
            const bool is_q = quarter >= 2;
            const uint2 em = *reinterpret_cast<const uint2 *>(smem + SP_AMASK + node * 8);
            uint32_t m = hh ? em.y : em.x;
            uint32_t t4 = hh ? __popc(em.x) * 4 : 0;
            if (!is_q && (node >> 5) == hh) m &= ~(1u << (node & 31));
            const uint32_t list = sbase + (is_q ? SP_GAMMA : SP_KAPPA) + node * 64 + ((node >> 1) & 3) * 16;   // xor 4 t = entry t
#pragma unroll 1
            for (int part = 0; part < 4; ++part, m >>= 8) {
                if (!__any_sync(0xffffffffu, m & 0xFFu)) continue;
                uint32_t r[8];
                GDN_TMEM_LD8(t_lane + TM_GC + hh * 32 + part * 8, r);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 a;\n\tsetp.ne.u32 p, %2, 0;\n\txor.b32 a, %1, %0;\n\t"
                                 "@p st.shared.b32 [a], %3;\n\t@p add.u32 %0, %0, 4;\n\t}"
                                 : "+r"(t4) : "r"(list), "r"(m & (1u << c)), "r"(r[c]) : "memory");
            }
            tc_fence_before();
            __syncthreads();
        }
        if constexpr (GROUPED) load_state(2, 3);
        // (2) w by back-substitution over the root path (column-oriented: once w_l is final, subtract w_l kappa(n_l, t) from
        // every entry t < l); four threads per node, thread sq of the quad owning path positions 4 sq .. 4 sq + 3
        const int zi = tid >> 2, sq = tid & 3;
        if (warp * 8 < T) {
            const uint2 zm = *reinterpret_cast<const uint2 *>(smem + SP_AMASK + zi * 8);
            const int d = __popc(zm.x) + __popc(zm.y);
            const uint4 path = *reinterpret_cast<const uint4 *>(smem + SP_ANC + zi * 16);
            const uint32_t idw[4] = {path.x, path.y, path.z, path.w};
            const uint32_t mine = *reinterpret_cast<const uint32_t *>(smem + SP_ANC + zi * 16 + sq * 4);
            const float *kappa = reinterpret_cast<const float *>(smem + SP_KAPPA);
            const float *beta_s = reinterpret_cast<const float *>(smem + SP_BETA);
            float z[4], bt[4], et[4];   // of this lane's path nodes: beta, scale exp(sum of g behind the node, down to node i)
            float gl[4];
            {
                const float4 g4 = *reinterpret_cast<const float4 *>(smem + SP_GAMMA + zi * 64 + ((sq ^ ((zi >> 1) & 3)) << 4));
                const float gv[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t id = (mine >> (8 * e)) & 63u;
                    const bool on = sq * 4 + e < d;
                    z[e] = on ? gv[e] : 0.f;
                    bt[e] = on ? beta_s[id] : 0.f;
                    gl[e] = on ? g_s[id] : 0.f;
                }
            }
            const int dmax = __reduce_max_sync(0xffffffffu, d);
#pragma unroll
            for (int l = VP_MD - 1; l >= 1; --l) {
                if (l < dmax) {   // warp-uniform
                    const float wl = __shfl_sync(0xffffffffu, z[l & 3] * bt[l & 3], (lane & ~3) | (l >> 2));
                    if (l < d && sq * 4 < l) {
                        const int nl = (int)((idw[l >> 2] >> ((l & 3) * 8)) & 63u);
                        const float4 x4 = *reinterpret_cast<const float4 *>(kappa + nl * VP_MD + ((sq ^ ((nl >> 1) & 3)) << 2));
                        const float xv[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (sq * 4 + e < l) z[e] = fmaf(-wl, xv[e], z[e]);
                    }
                }
            }
            // (sums over just those nodes: G_i - G would lose the weak decays behind a strong one, and alpha = 0)
            {
                const float all = (gl[0] + gl[1]) + (gl[2] + gl[3]), next = __shfl_xor_sync(0xffffffffu, all, 1);
                const float other = __shfl_xor_sync(0xffffffffu, all + next, 2);
                float behind = ((sq & 1) ? 0.f : next) + ((sq & 2) ? 0.f : other);
#pragma unroll
                for (int e = 3; e >= 0; --e) {
                    et[e] = p.scale * __expf(behind);
                    behind += gl[e];
                }
            }
            // (3) -sa w and z' into their operand tiles (zero off the root path)
            const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    *reinterpret_cast<uint4 *>(smem + SP_WZ + t * 8192 + sw128_row_offset(zi, 2 * sq + e)) = zero4;
            const float neg_sa = -reinterpret_cast<const float *>(smem + SP_SA)[zi];
            __syncwarp();   // the quad's zero fill precedes the scattered stores below
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (sq * 4 + e < d) {
                    const int j = (int)((mine >> (e * 8)) & 63u);
                    const float w = bt[e] * z[e];
                    uint32_t hi, lo;
                    split_pack_bf16(neg_sa * w, et[e] * w, hi, lo);
                    uint8_t *dst = smem + SP_WZ + sw128_row_offset(zi, j >> 3) + (j & 7) * 2;
                    *reinterpret_cast<uint16_t *>(dst) = (uint16_t)hi;
                    *reinterpret_cast<uint16_t *>(dst + 8192) = (uint16_t)lo;
                    *reinterpret_cast<uint16_t *>(dst + 16384) = (uint16_t)(hi >> 16);
                    *reinterpret_cast<uint16_t *>(dst + 24576) = (uint16_t)(lo >> 16);
                }
            }
        }
        if constexpr (GROUPED) load_state(3, 4);
        if (!mbar_wait_bounded(mbar_v, par)) *flag = 1;
        // k and v rows between the tree and the next multiple of 16 belong to another tree (or are padding): they meet zero
        // weights in the products, which have to be zero whatever they hold
        const int nk = max(1, (T + 15) >> 4);   // 16-node pieces of the unit
        if (!GROUPED && T < nk * 16) {
            for (int idx = tid; idx < (nk * 16 - T) * 32; idx += VP_THREADS) {
                const int r = T + (idx >> 5), c = idx & 15;
                uint8_t *dst = (idx & 16) ? smem + SP_V + (c >> 3) * 8192 + sw128_row_offset(r, c & 7) : smem + SP_KQ + sw128_offset(r, c);
                *reinterpret_cast<uint4 *>(dst) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        fence_proxy_async();   // generic-proxy writes of the operands become visible to the tensor core
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        // (4) C = -sa w.K (nodes on the lanes) and O = V^T.z' (value components on the lanes)
        if (warp == W_MMA_C && elect_one()) {
            constexpr uint32_t id_c = idesc_bf16(64, 64) | (1u << 16);   // B: rows along K (nodes)
            const uint64_t w_hi = smem_desc_sw128(sbase + SP_WZ), k0 = smem_desc_sw128(sbase + SP_KQ);
#pragma unroll 1
            for (int ks = 0; ks < nk; ++ks) {
#pragma unroll
                for (int part = 0; part < 2; ++part) {   // hi, lo
                    const uint32_t acc = (ks | part) != 0;
                    umma_bf16(tmem + TM_GC, w_hi + (uint64_t)(part * 512 + ks * 2), k0 + (uint64_t)(ks * 128), id_c, acc);
                    umma_bf16(tmem + TM_GC + (16u << 16), w_hi + (uint64_t)(part * 512 + ks * 2), k0 + (uint64_t)(1024 + ks * 128), id_c, acc);
                }
            }
            umma_commit(mbar_c);
        } else if (warp == W_MMA_O && elect_one()) {
            const uint32_t id_v = idesc_bf16(128, 0) | (1u << 15) | (uint32_t)(nk * 2) << 17;   // A: rows along K (nodes)
            const uint64_t z_hi = smem_desc_sw128(sbase + SP_WZ) + 1024;
            const uint64_t v0 = smem_desc_sw128(sbase + SP_V) + (511ull << 16);   // halves 8 KB apart
#pragma unroll 1
            for (int ks = 0; ks < nk; ++ks)
#pragma unroll
                for (int part = 0; part < 2; ++part)
                    umma_bf16(tmem + TM_O, v0 + (uint64_t)(ks * 128), z_hi + (uint64_t)(part * 512 + ks * 2), id_v, (ks | part) != 0);
            umma_commit(mbar_c);
        }
        // the next unit: its place and its tables (registers)
        const bool have_n = pull(nx);
        const bool next_rows = have_n && (GROUPED || nx.b != un.b || hk_of(nx.h) != hk_of(un.h));
        const bool same_tree = !GROUPED && have_n && (PADDED ? tree_of(nx.b) == tree_of(un.b) : nx.b == un.b);
        if (have_n) {
            tables_load(nx, nr, same_tree);
            if (tid < 4 && (!GROUPED || nx.fresh))   // ... and its state tile and, not gathered, its rows into L2
                prefetch_l2_bulk(p.S0 + (size_t)(nx.b * p.h_v + nx.h) * VP_D * VP_D + (size_t)tid * 4096, 16384);
            if (!GROUPED && tbl_thread && tnode < nx.T) {
                const size_t n = (size_t)(nx.base + tnode);
                auto prefetch_row = [](const __nv_bfloat16 *r) {
                    asm volatile("prefetch.global.L2 [%0];\n\tprefetch.global.L2 [%0 + 128];" ::"l"(r));
                };
                prefetch_row(p.v + (n * p.h_v + nx.h) * VP_D);
                if (next_rows) {
                    const size_t hk = (size_t)hk_of(nx.h);
                    prefetch_row(p.k + (n * p.h_qk + hk) * VP_D);
                    prefetch_row(p.q + (n * p.h_qk + hk) * VP_D);
                }
            }
        }
        if (state_late) {
            wait_for_previous_kernel();
            state_late = false;
            load_state(0, 4);
        }
        // (5) the state tile as bf16 hi + lo, the operand of the last product; a warp writes the lanes it can reach
        if (!GROUPED || un.fresh) {
            const uint32_t ts = tmem + ((uint32_t)row0 << 16) + TM_S;
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                uint32_t hi[8], lo[8];
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const int to = 4 * (n >> 1) + 2 * r + (n & 1);
                        split_pack_bf16(x[4 * jj + n][2 * r], x[4 * jj + n][2 * r + 1], hi[to], lo[to]);
                    }
                tmem_st_16x256_x2(ts + jj * 16, hi);
                tmem_st_16x256_x2(ts + 64 + jj * 16, lo);
            }
            tmem_wait_st();
        }
        if (GROUPED && have_n) gates_load(nx, nr);
        // (6) q' = sa q + C -> operand tiles over w and z', which C and V^T.z' have left.  In the state operand the key
        // positions are permuted within blocks of 32 (see the load): groups of four go from place 2 l4 + j to 4 j + l4.
        if (!mbar_wait_bounded(mbar_c, par)) *flag = 1;
        tc_fence_after();
        if (quarter * 16 < T) {
            const int row = quarter * 16 + (lane & 15), half = lane >> 4;   // node, half of the components
            const float sa = reinterpret_cast<const float *>(smem + SP_SA)[row];
            const float2 sa2 = make_float2(sa, sa);
            const uint8_t *q_s = smem + SP_KQ + half * 16384 + 8192;
            uint8_t *dst = smem + SP_WZ + half * 8192;
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {   // 16 components each
                uint32_t r[16], hi[8], lo[8];
                GDN_TMEM_LD16(t_lane + TM_GC + hh * 32 + c * 16, r);
                tmem_wait_ld();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint4 q4 = *reinterpret_cast<const uint4 *>(q_s + sw128_row_offset(row, hh * 4 + 2 * c + h));
                    const uint32_t qw[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int i = h * 8 + 2 * e, to = 4 * (e >> 1) + 2 * h + (e & 1);
                        const float2 v = __ffma2_rn(sa2, make_float2(__uint_as_float(qw[e] << 16), __uint_as_float(qw[e] & 0xFFFF0000u)),
                                                    make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])));
                        split_pack_bf16(v.x, v.y, hi[to], lo[to]);
                    }
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const uint32_t at = sw128_row_offset(row, hh * 4 + 2 * j + c);
                    *reinterpret_cast<uint4 *>(dst + at) = make_uint4(hi[4 * j], hi[4 * j + 1], hi[4 * j + 2], hi[4 * j + 3]);
                    *reinterpret_cast<uint4 *>(dst + 16384 + at) = make_uint4(lo[4 * j], lo[4 * j + 1], lo[4 * j + 2], lo[4 * j + 3]);
                }
            }
        }
        // output rows of this thread (GROUPED: vnode_s is about to take the next unit's ids)
        constexpr int CHUNKS = VP_D * (int)sizeof(TOut) / 16;   // 16-byte pieces of an output row
        constexpr int ROWS_STEP = VP_THREADS / CHUNKS;          // rows per pass of the CTA
        uint32_t out_ids[GROUPED ? VP_T / ROWS_STEP : 1];
        if constexpr (GROUPED) {
#pragma unroll
            for (int e = 0; e < VP_T / ROWS_STEP; ++e) out_ids[e] = vnode_s[tid / CHUNKS + e * ROWS_STEP];
            __syncthreads();
        }
        if (have_n) tables_put(nx, nr, same_tree);
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        // (7) O += S0.q'^T: hi.hi, lo.hi, hi.lo; lo.lo is below 2^-18 of the result
        if (warp == W_MMA_O && elect_one()) {
            const uint32_t id = idesc_bf16(128, 0) | (uint32_t)(nk * 2) << 17;
            const uint64_t q_hi = smem_desc_sw128(sbase + SP_WZ), q_lo = q_hi + 1024;
#pragma unroll 2
            for (int ks = 0; ks < 8; ++ks) {
                const uint64_t adv = (uint64_t)((ks >> 2) * 512 + (ks & 3) * 2);
                umma_bf16_ts(tmem + TM_O, tmem + TM_S + ks * 8, q_hi + adv, id);
                umma_bf16_ts(tmem + TM_O, tmem + TM_S + 64 + ks * 8, q_hi + adv, id);
                umma_bf16_ts(tmem + TM_O, tmem + TM_S + ks * 8, q_lo + adv, id);
            }
            umma_commit(mbar_o);
        }
        // meanwhile the next unit's rows (these are dead) and tables
        if (have_n) {
            if (next_rows) issue_kq(nx);
            issue_v(nx);
            tables_build(nx, nr, same_tree);
        }
        if (!mbar_wait_bounded(mbar_o, par)) *flag = 1;
        tc_fence_after();
        // (8) outputs through shared memory (over q', which is dead) so that global memory sees 16-byte stores of whole rows.
        // A fragment holds components g, g + 8 of nodes 2 l4, 2 l4 + 1.
        {
            const uint32_t src = tmem + ((uint32_t)row0 << 16) + TM_O;
            const int g = lane >> 2, l4 = lane & 3;
#pragma unroll 1
            for (int n0 = 0; n0 < T; n0 += 32) {
                uint32_t r[16];
                GDN_TMEM_LD_16x256_X4(src + n0, r);
                tmem_wait_ld();
                if constexpr (sizeof(TOut) == 2) {
                    // 8 x 8 blocks transposed by stmatrix into [node][256 B], piece c of node i at place c ^ (i & 7)
#pragma unroll
                    for (int j = 0; j < 4; j += 2) {
                        const int node = n0 + 8 * (j + (lane >> 4)) + (lane & 7), c = (row0 >> 3) + ((lane >> 3) & 1);
                        stmatrix_x4_trans(sbase + SP_WZ + node * 256 + ((c ^ (node & 7)) << 4),
                                          pack_bf16(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1])),
                                          pack_bf16(__uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3])),
                                          pack_bf16(__uint_as_float(r[4 * j + 4]), __uint_as_float(r[4 * j + 5])),
                                          pack_bf16(__uint_as_float(r[4 * j + 6]), __uint_as_float(r[4 * j + 7])));
                    }
                } else {
                    // [node][512 B], 32-byte piece c of node i at place c ^ ((i >> 1) & 3)
                    uint32_t *stage = reinterpret_cast<uint32_t *>(smem + SP_WZ);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int node = n0 + 8 * j + 2 * l4 + (e & 1), c = (row0 >> 3) + (e >> 1);
                            stage[node * 128 + ((c ^ l4) << 3) + g] = r[4 * j + e];
                        }
                }
            }
        }
        tc_fence_before();
        __syncthreads();
        const bool done_ok = *flag == 0;
        if (!done_ok) break;   // a bounded wait expired: stop, report, release
        {
            uint8_t *const o = static_cast<uint8_t *>(p.o);
            const int ck = tid % CHUNKS;
#pragma unroll
            for (int e = 0; e < VP_T / ROWS_STEP; ++e) {
                const int i = tid / CHUNKS + e * ROWS_STEP;
                if (i < T && (!GROUPED || i >= un.n_prefix)) {   // the ancestors in front of a group belong to other groups
                    const int at = sizeof(TOut) == 2 ? ck ^ (i & 7) : ck ^ (i & 6);
                    const uint4 val = *reinterpret_cast<const uint4 *>(smem + SP_WZ + i * (VP_D * (int)sizeof(TOut)) + at * 16);
                    const int node = GROUPED ? (int)out_ids[GROUPED ? e : 0] : i;
                    *reinterpret_cast<uint4 *>(o + ((size_t)(un.base + node) * p.h_v + un.h) * VP_D * sizeof(TOut) + ck * 16) = val;
                }
            }
        }
        if (next_rows) {
            issue_gram(nx.T, rows_parity);   // as soon as its rows are there
            rows_parity ^= 1;
        }
        par ^= 1;
        new_rows = next_rows;
        un = nx;
        have = have_n;
    }

    if (state_late) wait_for_previous_kernel();   // (no unit had work: this grid must not end before the one in front)
    if (*flag != 0 && tid == 0) report_status(p.status_dev, GDN_ERR_TIMEOUT);
    cp_async_wait_all();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TM_COLS);
}

template <typename TOut, bool PADDED, bool GROUPED> cudaError_t launch_kernel(const VerifyPlainParams &p, LaunchInFront commit, cudaStream_t stream)
{
    static PerContext seen;
    int sms = 0;
    cudaError_t e = device_sms(seen, reinterpret_cast<const void *>(verify_plain_kernel<TOut, PADDED, GROUPED>), SP_ALLOC, &sms);
    if (e == cudaSuccess && commit) e = commit();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(p.n_units < 2 * sms ? p.n_units : 2 * sms));   // persistent CTAs, two per SM
    cfg.blockDim = dim3(VP_THREADS);
    cfg.dynamicSmemBytes = SP_ALLOC;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, verify_plain_kernel<TOut, PADDED, GROUPED>, p);
}

template <bool GROUPED> cudaError_t launch_plain(const gdn_shape_t &s, VerifyPlainParams &p, LaunchInFront commit, cudaStream_t stream)
{
    p.state_late = !GROUPED && commit ? 1 : 0;   // (grouped: the kernel in front writes the plan as well)
    if constexpr (GROUPED) {
        // trees of more than 64 nodes: a unit is one ancestor-closed group of a (tree, head), taken from the plan's
        // unit list (its length is read on the device; this bound only sizes the grid); rows are gathered
        p.n_units *= p.groups_per_tree;
    } else {
        p.box_rows = (s.max_tree_nodes + 15) / 16 * 16;
        if (!make_row_tensor_map(&p.tm_k, p.k, s.total_nodes, s.h_qk, 64, p.box_rows, true) ||
            !make_row_tensor_map(&p.tm_q, p.q, s.total_nodes, s.h_qk, 64, p.box_rows, true) ||
            !make_row_tensor_map(&p.tm_v, p.v, s.total_nodes, s.h_v, 64, p.box_rows, true))
            return cudaErrorNotSupported;
    }
    // the padded layout and the on-chip gate activations share an instantiation
    if (s.out_dtype == GDN_BF16)
        return p.t_pad != 0 ? launch_kernel<__nv_bfloat16, true, GROUPED>(p, commit, stream) : launch_kernel<__nv_bfloat16, false, GROUPED>(p, commit, stream);
    return p.t_pad != 0 ? launch_kernel<float, true, GROUPED>(p, commit, stream) : launch_kernel<float, false, GROUPED>(p, commit, stream);
}

VerifyPlainParams make_params(const gdn_shape_t &s, const float *S0, const void *q, const void *k, const void *v,
                              const void *g, const void *beta, const int32_t *node_offsets, void *o,
                              const PlanPtrs &plan, int32_t *status_dev)
{
    VerifyPlainParams p{};
    p.h_qk = s.h_qk; p.h_v = s.h_v; p.n_units = s.n_seq * s.h_v; p.scale = s.scale;
    p.S0 = S0;
    p.q = static_cast<const __nv_bfloat16 *>(q); p.k = static_cast<const __nv_bfloat16 *>(k);
    p.v = static_cast<const __nv_bfloat16 *>(v); p.g = static_cast<const __nv_bfloat16 *>(g);
    p.beta = static_cast<const __nv_bfloat16 *>(beta);
    p.node_offsets = node_offsets; p.o = o;
    p.n_seq = s.n_seq; p.total_nodes = s.total_nodes; p.max_tree_nodes = s.max_tree_nodes; p.max_depth = s.max_depth;
    p.status_dev = status_dev;
    // upper bound of the groups of a tree (the real ones are in the plan's unit list)
    p.groups_per_tree = s.max_tree_nodes <= VP_T ? 1 : (s.max_tree_nodes + GDN_GROUP_MIN_NODES - 1) / GDN_GROUP_MIN_NODES;
    p.anc_stride = s.max_depth;
    p.anc8 = plan.anc8; p.dfs_anc8 = plan.dfs_anc8;
    p.anc16 = plan.anc; p.dfs_node = plan.dfs_node;
    p.unit_list = plan.unit_list;
    p.unit_count = plan.unit_count;
    p.unit_capacity = (int)unit_list_capacity(s);
    p.plan_magic = plan_magic(s.n_seq, s.max_tree_nodes, s.max_depth);
    return p;
}

// The state of a verification alone, for the kernel of small trees (which writes it behind a commit only).
CommitParams state_only(const gdn_shape_t &s, const float *S0, bool raw_gates, int32_t *status_dev)
{
    CommitParams c{};
    c.h_qk = s.h_qk; c.h_v = s.h_v; c.d_k = s.d_k; c.d_v = s.d_v; c.max_depth = s.max_depth;
    c.S = const_cast<float *>(S0);
    c.status_dev = status_dev;
    c.raw_gates = raw_gates ? 1 : 0;
    return c;
}

}  // namespace

// Padded layout, trees of at most 64 nodes.
cudaError_t launch_verify_sm100_padded(const gdn_shape_t &s, int n_trees, bool raw_gates, const float *S0,
                                       const void *q, const void *k, const void *v, const void *g, const void *beta,
                                       const int32_t *parent, const int32_t *n_nodes, void *o, int32_t *status_dev,
                                       cudaStream_t stream, LaunchInFront commit)
{
    if (s.n_seq == 0 || s.total_nodes == 0) return cudaSuccess;
    if (!commit && step_small_supported(s))
        return launch_step_small(s, state_only(s, S0, raw_gates, status_dev), false, q, k, v, g, beta, parent, nullptr, n_trees, n_nodes, o,
                                 stream);
    VerifyPlainParams p = make_params(s, S0, q, k, v, g, beta, nullptr, o, PlanPtrs{}, status_dev);
    p.parent = parent;
    p.t_pad = s.max_tree_nodes; p.n_trees = n_trees; p.n_nodes = n_nodes; p.raw_gates = raw_gates ? 1 : 0;
    return launch_plain<false>(s, p, commit, stream);
}

cudaError_t launch_verify_sm100_planned(const gdn_shape_t &s, int n_trees, bool raw_gates, const float *S0,
                                        const void *q, const void *k, const void *v, const void *g, const void *beta,
                                        const PlanPtrs &plan, void *o, int32_t *status_dev, cudaStream_t stream)
{
    if (s.n_seq == 0 || s.total_nodes == 0) return cudaSuccess;
    gdn_shape_t ps = s;   // the shape the plan was built for: n_trees trees of t_pad rows
    ps.n_seq = n_trees;
    ps.total_nodes = n_trees * s.max_tree_nodes;
    const int capacity = (int)unit_list_capacity(ps), magic = plan_magic(n_trees, s.max_tree_nodes, s.max_depth);
    if (step_small_supported(s))
        return launch_step_small(s, state_only(s, S0, raw_gates, status_dev), false, q, k, v, g, beta, nullptr, nullptr, n_trees, nullptr, o,
                                 stream, {plan.unit_list, plan.unit_count, plan.anc8, capacity, magic});
    VerifyPlainParams p = make_params(s, S0, q, k, v, g, beta, nullptr, o, plan, status_dev);
    p.t_pad = s.max_tree_nodes; p.n_trees = n_trees; p.raw_gates = raw_gates ? 1 : 0;
    p.unit_capacity = capacity;
    p.plan_magic = magic;
    return launch_plain<true>(s, p, {}, stream);
}

bool verify_sm100_supported(const gdn_shape_t &s)
{
    return s.d_k == VP_D && s.d_v == VP_D && s.in_dtype == GDN_BF16 && s.max_tree_nodes <= GDN_GROUPED_MAX_NODES &&
           s.max_depth <= VP_MD;
}

bool verify_sm100_single_group(const gdn_shape_t &s) { return verify_sm100_supported(s) && s.max_tree_nodes <= VP_T; }

cudaError_t launch_verify_sm100(const gdn_shape_t &s, const float *S0, const void *q, const void *k,
                                const void *v, const void *g, const void *beta, const int32_t *parent,
                                const int32_t *node_offsets, void *o, const PlanPtrs &plan,
                                int32_t *status_dev, cudaStream_t stream, LaunchInFront commit)
{
    if (s.n_seq == 0 || s.total_nodes == 0) return cudaSuccess;
    if (!commit && step_small_supported(s))
        return launch_step_small(s, state_only(s, S0, false, status_dev), false, q, k, v, g, beta, parent, node_offsets, 1, nullptr, o,
                                 stream);
    VerifyPlainParams p = make_params(s, S0, q, k, v, g, beta, node_offsets, o, plan, status_dev);
    p.parent = parent;
    if (!verify_sm100_single_group(s)) return launch_plain<true>(s, p, commit, stream);
    return launch_plain<false>(s, p, commit, stream);
}

}  // namespace gdn
