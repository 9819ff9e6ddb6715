// Commit of the previous step's paths and tree verification in one kernel (gdn_verify_plain.cu: verification alone) for
// sm_100a: d_k = d_v = 128, bf16 inputs, root paths of at most 16 nodes, trees of at most 64 nodes.  It evaluates the
// triangular form of Section 3.4.1 (Eq. 9-11) restricted to real ancestors, with the W S0 term folded into the
// right-hand side as in Section 3.4.2, and turns all of the per-component work into dense contractions on the
// 5th-generation tensor cores (tcgen05.mma, bf16 operands, fp32 accumulators in tensor memory):
//
//   (1) P  [d_v x 2T] = S0 [d_v x d_k] . [k rows; q rows]^T          the S0 projections of Eq. 11 / Eq. 13
//       Gr [2T x T]   = [k rows; q rows] . [k rows]^T                k_i.k_j and q_i.k_j of Eq. 9
//   (2) D  [d_v x T]  = R^T [d_v x T] . Z^T [T x T]                  the whole masked solve + output
//
// where r_j = beta_j (v_j - a_j S0^T k_j) is the folded right-hand side and row i of Z is
// z_i^T = y_i^T (I + X_path(i))^-1: because the ancestors of a node form a chain, the inverse restricted to one
// root path is a back-substitution with at most 16 unknowns that each node can run on its own (four threads per
// node, no dependence between nodes).  Then
//   o_i = scale (a_i S0^T q_i + sum_{j on the root path of i} Z_ij r_j),
// which is Eq. 11 with U - W S0 eliminated; no per-component sequential substitution is left.
// fp32 quantities that feed the tensor cores are split into two bf16 terms (x = hi + lo, |x - hi - lo| <= 2^-16 |x|):
// S0 for (1), R and Z for (2); the lo.lo term of (2) is dropped.
//
// Operand orientation: d_v on the TMEM lanes, nodes on the TMEM columns, so every thread of a warp owns one value
// component.  256 threads, about 112 KB of shared memory and 256 TMEM columns per CTA, so two CTAs share an SM.
// One persistent kernel: a software pipeline across the units of a CTA, TMA tiles on mbarriers, the commit of the previous
// step in front of each unit's verification, on the same registers.
//
// What bounds it: the chain of a unit together with the FMA of the replay (about 364 cycles per step and SM), not memory;
// the state crosses HBM once each way.  48 slots x 32 heads, 64 nodes, path of 7: 84.5 us (43 of memory traffic).  Of the
// forms tried for it -- one CTA per SM with specialised warps, the replay as matrix products on the fragments, the commit
// and verify kernels back to back (86.6 us; 72 against 84 at a path of 1) -- none is faster over the path lengths.
#include "gdn_internal.cuh"
#include "gdn_path.cuh"
#include "gdn_replay.cuh"
#include "gdn_tc.cuh"

namespace gdn {

namespace {

constexpr int FV_THREADS = 256;
constexpr int FV_D = 128;           // d_k = d_v
constexpr int FV_T = 64;            // max nodes per tree
constexpr int FV_MD = 16;           // max nodes on a root path
constexpr int FV_TMEM_COLS = 256;   // P: columns [0,128); D: [128,192); Gram block of the unit to come: [192,256)

// shared memory map (bytes from a 1024-byte aligned base)
constexpr int SM_A_HI = 0;                       // S0 hi: [2][128 rows][128 B], 128B-swizzled, K-major
constexpr int SM_A_LO = 32768;                   // S0 lo
constexpr int SM_B_KQ = 65536;                   // k and q rows, same layout: rows 0..63 = k, 64..127 = q
// after the first MMA group the operand tiles are dead and are reused:
constexpr int SM_GRAM = 0;                       // fp32 [128][64]: four-column piece c of row r at position c ^ (r & 15)
constexpr int SM_RT_HI = 0;                      // then R^T hi: [128 rows = components][64 nodes] bf16, swizzled
constexpr int SM_RT_LO = 16384;                  //      R^T lo
constexpr int SM_VE = 40960;                     // v rows of the tree, bf16 [64][128]: they land here at the top of a unit (free
                                                 // until the state operand is written) and move into registers before that
constexpr int SM_Z_HI = 49152;                   // Z hi: [64 rows = nodes i][64 nodes j] bf16, swizzled
constexpr int SM_Z_LO = 57344;                   // Z lo
constexpr int SM_X = 98304;                      // fp32 [64][16]  X(i, t-th path node)
constexpr int SM_Y = SM_X + 4096;                // fp32 [64][16]  Y(i, t-th path node), node itself included
constexpr int SM_ANC = SM_Y + 4096;              // u8   [64][16]  root-path node ids (0xFF = unused)
constexpr int SM_GAB = SM_ANC + 1024;            // float4 [64]: (., a_i, beta_i, g_i)
constexpr int SM_DEPTH = SM_GAB + 1024;          // u8 [64] (0 beyond T)
constexpr int SM_PATH = SM_DEPTH + FV_T;         // fused commit, two slots of 384 B: int [16] path node ids, int length (0 = no
                                                 // replay), int first node of the tree; at +128 float4 [16] (A_t = decay of the
                                                 // path up to and including step t, beta_t, alpha_t, 1 / A_t)
constexpr int SM_PATH_SLOT = 384;
constexpr int SM_PK = 32768;                     // fused commit: k rows of the accepted path, bf16 [16][128], parked in the
constexpr int SM_PV = 36864;                     // state-operand area until the replay is over; v rows likewise
constexpr int SM_TABLE2 = SM_PATH + 2 * SM_PATH_SLOT;   // second copy of ANC / GAB / DEPTH (2112 B)
constexpr int SM_TABLE_STRIDE = SM_TABLE2 - SM_ANC;   // table buffer tb lives SM_TABLE_STRIDE * tb further on
constexpr int SM_MBAR = SM_TABLE2 + 2176;        // 5 x u64: Gram done, P done, D done, k/q tile landed, v tile landed
constexpr int SM_TMEM = SM_MBAR + 40;            // u32
constexpr int SM_FLAG = SM_TMEM + 4;             // u32 (timeout flag)
constexpr int SM_PAR = SM_FLAG + 4;              // s8 [64] parent[] of the tree whose tables are being built
constexpr int SM_BAD = SM_PAR + FV_T;            // int [2], tree of table buffer tb was rejected
constexpr int SM_BYTES = SM_BAD + 8;
constexpr int SM_ALLOC = SM_BYTES + 1024;        // slack for the 1024-byte alignment of the base

struct VerifyFastParams {
    // TMA descriptors of the packed k, q, v tensors viewed as [N][heads][128] bf16
    alignas(64) CUtensorMap tm_k;
    alignas(64) CUtensorMap tm_q;
    alignas(64) CUtensorMap tm_v;
    int h_qk, h_v;
    int n_units;        // n_seq * h_v
    float scale;
    const float *S0;
    const __nv_bfloat16 *q, *k, *v, *g, *beta;
    const int32_t *node_offsets;
    const int32_t *parent;                             // trees of at most 64 nodes: the kernel builds the metadata itself
    int n_seq, total_nodes, max_tree_nodes, max_depth;
    void *o;
    int32_t *status_dev;
    // commit of the previous step's accepted paths
    float *S_rw;                                       // same tensor as S0, written in place
    const __nv_bfloat16 *pk, *pv, *pg, *pbeta;         // the previous tree's k, v, g, beta
    const int32_t *pparent, *pnode_offsets, *path, *path_offsets;
    // Padded layout of Section 3.4.2 (persistent kernel; t_pad = 0: ragged packing by node_offsets[]): slot b keeps
    // its nodes in rows b * t_pad .. and carries tree b % n_trees, whose parent[] row and node count are shared by
    // all the slots (layers) of that tree; the accepted paths are per tree as well.
    int t_pad, n_trees, pt_pad, path_stride;
    const int32_t *n_nodes, *pn_nodes, *path_len;
    int raw_gates;                                     // g / beta arrive as raw gate inputs ("scalars" stage on chip)
};

// ---------------------------------------------------------------------------------------- kernel
// The k/q tile holds the k rows first and the q rows second (rows i and 64 + i), so P has p^k in columns 0..63 and
// p^q in columns 64..127, and the Gram block needs only N = 64.
// Eq. 7 is replayed along the previous step's accepted path on the state tile while it sits in registers
// -- per row c, s_c <- alpha s_c + k beta (v_c - alpha k.s_c), the eight lanes that share a row reducing k.s_c with
// three shuffles -- the tile is written back as the only state write of the step, and the new tree is verified
// against it.
// A CTA keeps its tensor memory and walks over the units blockIdx.x, blockIdx.x + gridDim.x, ...  Nothing a unit
// can know in advance is waited for inside it: the next unit's k/q tile streams into the operand tile as soon as the
// first MMA group has released it, its Gram block is issued at the end of the current unit into spare TMEM columns,
// and its per-node tables, decay tables and accepted path are fetched in stages, each global load one phase before
// its value is used.  The state tile is asked for at the top of the unit and is needed only after the Gram /
// coefficient phases; the v rows land by TMA in an area that is free until the state operand is written.
// SMALL (every tree of the call has at most 32 nodes, the largest more than 16: gdn_step_small.cu has the others): the R and output
// phases skip the 16-node pieces beyond the tree.
template <typename TOut, bool SMALL, bool PADDED>
__global__ void __launch_bounds__(FV_THREADS, 2) commit_verify_kernel(const __grid_constant__ VerifyFastParams p)
{
    extern __shared__ uint8_t fv_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(fv_smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    float *xs = reinterpret_cast<float *>(smem + SM_X);
    float *ys = reinterpret_cast<float *>(smem + SM_Y);
    float *gram = reinterpret_cast<float *>(smem + SM_GRAM);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + SM_TMEM);
    volatile uint32_t *flag = reinterpret_cast<volatile uint32_t *>(smem + SM_FLAG);
    const uint32_t mbar_g = sbase + SM_MBAR, mbar_p = mbar_g + 8, mbar_d = mbar_g + 16;
    const uint32_t mbar_kq = mbar_g + 24, mbar_v = mbar_g + 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r4 = lane >> 3, l8 = lane & 7;
    // The asynchronous work of a unit is issued by one elected lane each of four warps, so that no single warp
    // carries all of it: warp 0 the projection MMA group, warp 1 the D group, warp 2 the Gram block of the unit to
    // come, warp 3 the TMA loads.  Every issuer commits its own MMAs to an mbarrier.
    constexpr int W_MMA_P = 0, W_MMA_D = 1, W_MMA_G = 2, W_TMA = 3;

    if (warp == 0) tmem_alloc(sbase + SM_TMEM, FV_TMEM_COLS);
    if (tid == 32) {
        mbar_init(mbar_g, 1);
        mbar_init(mbar_p, 1);
        mbar_init(mbar_d, 1);
        mbar_init(mbar_kq, 1);
        mbar_init(mbar_v, 1);
        *flag = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);   // warp-uniform by construction
    // Launched with programmatic stream serialization: everything above overlaps the tail of the kernel in front
    // (the previous call, or the plan kernel); nothing that is computed from memory may run before that kernel's
    // writes are visible.  L2 can be asked for the first unit's state tile meanwhile (a prefetch consumes nothing).
    if (tid < 4 && (int)blockIdx.x < p.n_units)
        prefetch_l2_bulk(p.S0 + (size_t)blockIdx.x * FV_D * FV_D + (size_t)tid * 4096, 16384);
    // ... and for the rows of the first unit's tree.  Their place may depend on node_offsets[], which the kernel in
    // front may still be writing: the value read here only steers prefetches (clamped to the tensors) and comes from
    // L2, so that nothing of it stays in L1; it is read again behind the dependency wait before anything is computed
    // from it.
    if ((int)blockIdx.x < p.n_units && tid >= 128 && tid < 128 + FV_T) {
        const int ub = (int)blockIdx.x / p.h_v, uh = (int)blockIdx.x % p.h_v, uhk = uh / (p.h_v / p.h_qk);
        const int row = ((PADDED) ? ub * p.t_pad : __ldcg(p.node_offsets + ub)) + tid - 128;
        if (row >= 0 && row < p.total_nodes) {
            prefetch_l2_bulk(p.v + ((size_t)row * p.h_v + uh) * FV_D, 256);
            prefetch_l2_bulk(p.k + ((size_t)row * p.h_qk + uhk) * FV_D, 256);
            prefetch_l2_bulk(p.q + ((size_t)row * p.h_qk + uhk) * FV_D, 256);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.g + (size_t)row * p.h_v + uh));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.beta + (size_t)row * p.h_v + uh));
        }
    }
    signed char *par_s = reinterpret_cast<signed char *>(smem + SM_PAR);
    volatile int *bad_s = reinterpret_cast<volatile int *>(smem + SM_BAD);

    // unit -> (tree, head, first node, size); a unit whose node_offsets[] are inconsistent (reported) or whose tree
    // is empty is skipped.  parent[] itself is checked when the unit's tables are built.
    // A CTA walks the units blockIdx.x, blockIdx.x + gridDim.x, ...: the indices of a unit follow from those of the
    // unit before by additions and carries, so that the integer divisions by the head and group counts (a few dozen
    // instructions each, for every thread) are paid once per CTA and not once per unit.
    // Unit = slot b * h_v + head h.
    struct Cursor { int u, b, h; };
    const int n_units = p.n_units;
    const int ratio = p.h_v / p.h_qk;
    const int ratio_shift = (ratio & (ratio - 1)) == 0 ? 31 - __clz(ratio) : -1;
    auto hk_of = [&](int h_) -> int { return ratio_shift >= 0 ? h_ >> ratio_shift : h_ / ratio; };
    auto tree_of = [&](int b_) -> int { return p.n_trees == 1 ? 0 : b_ % p.n_trees; };   // padded layout only
    const int step_h = (int)gridDim.x % p.h_v, step_b = (int)gridDim.x / p.h_v;
    auto cursor_at = [&](int u) -> Cursor {
        Cursor c;
        c.u = u;
        c.h = u % p.h_v;
        c.b = u / p.h_v;
        return c;
    };
    auto advance = [&](Cursor &c) {
        c.u += (int)gridDim.x;
        c.h += step_h;
        const int carry_h = c.h >= p.h_v ? 1 : 0;
        c.h -= carry_h ? p.h_v : 0;
        c.b += step_b + carry_h;
    };
    // The loads a decode needs are issued by decode_load() and looked at by decode() later (the unit after
    // next is asked for at the top of a unit and decoded in its middle), so that no thread waits for them.
    struct DecodeRaw { int lo, hi; };
    auto decode_load = [&](const Cursor &c) -> DecodeRaw {
        DecodeRaw r{0, 0};
        if (c.u >= n_units) return r;
        const int ub = c.b;
        if (PADDED) {
            r.lo = p.n_nodes[tree_of(ub)];
        } else {
            r.lo = p.node_offsets[ub];
            r.hi = p.node_offsets[ub + 1];
        }
        return r;
    };
    auto decode = [&](const Cursor &c, const DecodeRaw &raw, int &ub, int &uh, int &uhk, int &ubase, int &uT, int &upar) -> bool {
        if (c.u >= n_units) return false;
        ub = c.b;
        uh = c.h;
        uhk = hk_of(uh);
        bool off_ok;
        if (PADDED) {   // padded layout: rows of the slot, node count and parent[] row of its tree
            const int tree = tree_of(ub);
            ubase = ub * p.t_pad;
            uT = raw.lo;
            upar = tree * p.t_pad;
            off_ok = uT >= 0 && uT <= FV_T && uT <= p.t_pad;
        } else {
            ubase = raw.lo;
            const int uend = raw.hi;
            uT = uend - ubase;
            upar = ubase;
            off_ok = ubase >= 0 && uT >= 0 && uT <= FV_T && uT <= p.max_tree_nodes && uend <= p.total_nodes;
            if (ub == 0) off_ok = off_ok && ubase == 0;
            if (ub == p.n_seq - 1) off_ok = off_ok && uend == p.total_nodes;
        }
        if (!off_ok && tid == 0) report_status(p.status_dev, GDN_ERR_TREE);
        const bool tree_good = off_ok && uT > 0;
        if (!tree_good) {
            // the commit of the previous step does not depend on the new tree: the unit runs as a tree of no
            // nodes (every node masked, nothing stored), so that its accepted path is still replayed
            ubase = 0;
            uT = 0;
            upar = 0;
            return true;
        }
        return tree_good;
    };
    // k and q rows -> B operand tile by TMA: four 64-row x 64-column boxes (k and q, either K half), 128-byte
    // swizzled, completing on mbar_kq.  A box always spans 64 nodes: rows beyond the tree belong to the next tree
    // (or are zero past the end of the tensor); every use of them is masked further down.
    auto issue_kq = [&](int ub, int uhk, int ubase, int uT) {
        (void)ub; (void)uT;
        if (warp == W_TMA && elect_one()) {
            mbar_expect_tx(mbar_kq, 32768);
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {
                tma_load_3d(sbase + SM_B_KQ + kh * 16384, &p.tm_k, kh * 64, uhk, ubase, mbar_kq);
                tma_load_3d(sbase + SM_B_KQ + kh * 16384 + 8192, &p.tm_q, kh * 64, uhk, ubase, mbar_kq);
            }
        }
    };
    // Tree metadata of Section 3.4.2 for one tree of at most 64 nodes, built by the CTA itself one unit ahead of
    // its use: depth and root-path list (root first, node last, 0xFF beyond) of every node.  put_parent() stages
    // parent[] in shared memory (entries outside [-1, i) are reported and cut); after a CTA barrier walk_tables()
    // lets thread i climb from node i to its root, shifting each id into a 16-byte row from below, so that the
    // root ends up in byte 0.  A tree with a bad parent[] or a root path of more than max_depth nodes is flagged in
    // bad_s[tb]; the unit then runs as a tree of no nodes.
    // Node i is handled by thread FV_T + i (warps 2 and 3; warps 0 and 1 issue MMAs at the same time).  In the padded layout
    // the slots of a tree share its parent[]: a unit with the tree of the one before copies its rows and verdict (48 slots of one
    // 61-node tree, path of 12: 104.6 -> 102.3 us).
    const int tnode = tid - FV_T;
    const bool tbl_thread = tid >= FV_T && tid < 2 * FV_T;
    auto put_parent = [&](int uT, int par, int tb, bool same_tree) -> bool {
        bool bad = false;
        if (tbl_thread && !same_tree) {
            int pv = -1;
            if (tnode < uT) {
                pv = par;
                if (pv < -1 || pv >= tnode) { bad = true; pv = -1; }
            }
            par_s[tnode] = (signed char)pv;
        }
        if (tid == 0) bad_s[tb] = same_tree ? bad_s[tb ^ 1] : 0;
        return bad;
    };
    auto walk_tables = [&](int uT, int tb, uint32_t g_bits, uint32_t be_bits, bool my_bad, bool same_tree) {
        if (tbl_thread) {
            int d = 0, err = my_bad ? GDN_ERR_TREE : 0;
            uint32_t w0 = 0xFFFFFFFFu, w1 = 0xFFFFFFFFu, w2 = 0xFFFFFFFFu, w3 = 0xFFFFFFFFu;
            if (same_tree) {   // rows of the unit before
                d = (smem + SM_DEPTH + (tb ^ 1) * SM_TABLE_STRIDE)[tnode];
                const uint4 row = *reinterpret_cast<const uint4 *>(smem + SM_ANC + (tb ^ 1) * SM_TABLE_STRIDE + tnode * 16);
                w0 = row.x; w1 = row.y; w2 = row.z; w3 = row.w;
            } else if (tnode < uT && !err) {
                int cur = tnode;
                while (cur >= 0) {
                    if (++d > p.max_depth) { err = GDN_ERR_DEPTH; break; }
                    w3 = __funnelshift_l(w2, w3, 8);
                    w2 = __funnelshift_l(w1, w2, 8);
                    w1 = __funnelshift_l(w0, w1, 8);
                    w0 = (w0 << 8) | (uint32_t)cur;
                    cur = par_s[cur];
                }
            }
            if (err) {
                d = 0;
                report_status(p.status_dev, err);
                bad_s[tb] = 1;
            }
            (smem + SM_DEPTH + tb * SM_TABLE_STRIDE)[tnode] = (uint8_t)d;
            *reinterpret_cast<uint4 *>(smem + SM_ANC + tb * SM_TABLE_STRIDE + tnode * 16) = make_uint4(w0, w1, w2, w3);
            reinterpret_cast<float4 *>(smem + SM_GAB + tb * SM_TABLE_STRIDE)[tnode] =
                make_float4(0.f, 0.f, gate_beta(be_bits, PADDED && p.raw_gates), gate_log_decay(g_bits, PADDED && p.raw_gates));
        }
    };
    // the same two steps with the loads issued on the spot (first unit of a CTA, and behind a skipped unit)
    auto load_parent = [&](int upar, int uT, int tb) -> bool {
        return put_parent(uT, tbl_thread && tnode < uT ? p.parent[upar + tnode] : -1, tb, false);
    };
    auto load_tables = [&](int uh, int ubase, int uT, int tb, bool my_bad) {
        uint32_t gb = 0, bb = 0;
        if (tbl_thread && tnode < uT) {
            const size_t n = (size_t)(ubase + tnode);
            gb = __ldg(reinterpret_cast<const unsigned short *>(p.g) + n * p.h_v + uh);
            bb = __ldg(reinterpret_cast<const unsigned short *>(p.beta) + n * p.h_v + uh);
        }
        walk_tables(uT, tb, gb, bb, my_bad, false);
    };

    // Fused commit: the accepted path of tree `ub` in the previous step goes to path slot `ps`.  One warp
    // fetches it (lane t: entry t and that node's parent) and checks with shuffles that it is a chain from a
    // root inside the previous tree; a bad path is reported and its length stored as 0, so that this state
    // stays as it was.  Readable by the other warps after the next CTA barrier.
    auto fetch_path = [&](int ub, int ps) {
        if (warp == 4) {
            int *slot = reinterpret_cast<int *>(smem + SM_PATH + ps * SM_PATH_SLOT);
            int pp0, len, pb = 0, pT = 0, ppar = 0;   // len 0 leaves the state alone
            if (PADDED) {
                const int tree = tree_of(ub);
                pp0 = tree * p.path_stride;
                len = p.path_len[tree];
                pb = ub * p.pt_pad;
                pT = min(p.pn_nodes[tree], p.pt_pad);
                ppar = tree * p.pt_pad;
            } else {
                pp0 = p.path_offsets[ub];
                len = p.path_offsets[ub + 1] - pp0;
                if (len != 0) {
                    pb = p.pnode_offsets[ub];
                    pT = p.pnode_offsets[ub + 1] - pb;
                    ppar = pb;
                }
            }
            if (len != 0) {
                const bool shape_ok = len > 0 && len <= FV_MD && len <= p.max_depth && pT > 0 && pp0 >= 0;
                const bool mine = shape_ok && lane < len;
                int n = -1, parent_n = -2;
                if (mine) {
                    n = p.path[pp0 + lane];
                    if (p.pparent && n >= 0 && n < pT) parent_n = p.pparent[ppar + n];
                    slot[lane] = n;
                }
                const int n_up = __shfl_up_sync(0xffffffffu, n, 1);
                bool bad = false;
                if (mine) {
                    if (n < 0 || n >= pT) bad = true;
                    else if (p.pparent) bad = parent_n != (lane ? n_up : -1);
                    else if (lane && n <= n_up) bad = true;   // without parent[] only the topological order can be checked
                }
                if (__any_sync(0xffffffffu, bad) || !shape_ok) {
                    if (lane == 0) report_status(p.status_dev, GDN_ERR_PATH);
                    len = 0;
                }
            }
            if (lane == 0) {
                slot[16] = len;
                slot[17] = pb;
                slot[18] = len;
            }
        }
    };
    // k and v rows of that path (bf16, 256 B each) into their parking area: issued by everybody once the slot is
    // readable and the parking area is free.  Only node ids that have been range-checked are used (slot[18] =
    // length of the path as far as it has been checked when the rows are asked for).
    auto fetch_path_kv = [&](int uh, int uhk, int ps) {
        const int *slot = reinterpret_cast<const int *>(smem + SM_PATH + ps * SM_PATH_SLOT);
        const int len = slot[18], pb = slot[17];
        for (int idx = tid; idx < len * 32; idx += FV_THREADS) {
            const int t = idx >> 5, c16 = idx & 15;
            const size_t n = (size_t)pb + slot[t];
            if (idx & 16)
                cp_async_16(sbase + SM_PV + t * 256 + c16 * 16, p.pv + (n * p.h_v + uh) * FV_D + c16 * 8, true);
            else
                cp_async_16(sbase + SM_PK + t * 256 + c16 * 16, p.pk + (n * p.h_qk + uhk) * FV_D + c16 * 8, true);
        }
    };
    // per-step scalars of the path, computed on the spot (first unit of a CTA, and behind a skipped unit)
    auto path_scalars_direct = [&](int uh, int ps) {
        const int *slot = reinterpret_cast<const int *>(smem + SM_PATH + ps * SM_PATH_SLOT);
        float4 *ab = reinterpret_cast<float4 *>(smem + SM_PATH + ps * SM_PATH_SLOT + 128);
        const int len = slot[16], pb = slot[17];
        if (tid < len) {
            float gsum = 0.f, gt = 0.f;
            const unsigned short *pg = reinterpret_cast<const unsigned short *>(p.pg);
            const unsigned short *pbe = reinterpret_cast<const unsigned short *>(p.pbeta);
            for (int t = 0; t <= tid; ++t) {
                gt = gate_log_decay(pg[((size_t)pb + slot[t]) * p.h_v + uh], PADDED && p.raw_gates);
                gsum += gt;
            }
            const size_t n = (size_t)pb + slot[tid];
            const float A = expf(gsum);
            ab[tid] = make_float4(A, gate_beta(pbe[n * p.h_v + uh], PADDED && p.raw_gates), expf(gt), 1.f / A);
        }
    };
    // a_i = exp(sum of g along the root path), and for every path node the sum of g behind it, down to node i, in the place of
    // its Y (free by now; a difference of two sums from the root would lose the weak decays behind a strong one, and alpha = 0),
    // for the tables in buffer `tb`
    auto path_decay = [&](int tb) {   // four threads per node, four path positions each
        float4 *gab_t = reinterpret_cast<float4 *>(smem + SM_GAB + tb * SM_TABLE_STRIDE);
        const int i = tid >> 2, s4 = tid & 3;
        const int d = (smem + SM_DEPTH + tb * SM_TABLE_STRIDE)[i];
        const uint32_t ids = *reinterpret_cast<const uint32_t *>(smem + SM_ANC + tb * SM_TABLE_STRIDE + i * FV_MD + s4 * 4);
        float gl[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) gl[e] = s4 * 4 + e < d ? gab_t[(ids >> (8 * e)) & 0xFFu].w : 0.f;
        const float all = (gl[0] + gl[1]) + (gl[2] + gl[3]), next = __shfl_xor_sync(0xffffffffu, all, 1);
        const float other = __shfl_xor_sync(0xffffffffu, all + next, 2);
        const float b3 = ((s4 & 1) ? 0.f : next) + ((s4 & 2) ? 0.f : other), b2 = b3 + gl[3], b1 = b2 + gl[2], b0 = b1 + gl[1];
        *reinterpret_cast<float4 *>(ys + i * FV_MD + s4 * 4) = make_float4(b0, b1, b2, b3);
        if (s4 == 0) gab_t[i].y = d ? __expf(all + next + other) : 0.f;
    };
    // Gram = [k;q].k^T of the tile in the k/q operand area, into TMEM columns 192..255, which nothing else uses:
    // issued by one thread as soon as the tile has landed, one unit ahead of its use.
    auto issue_gram = [&](uint32_t kq_parity) {
        if (warp == W_MMA_G && elect_one()) {
            if (!mbar_wait_bounded(mbar_kq, kq_parity)) *flag = 1;
            tc_fence_after();
            const uint64_t b_kq = smem_desc_sw128(sbase + SM_B_KQ);
            constexpr uint32_t id = idesc_bf16(128, 64);   // B = the 64 k rows
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                const uint64_t adv = (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4);
                umma_bf16(tmem + 192, b_kq + adv, b_kq + adv, id, ks > 0);
            }
            umma_commit(mbar_g);
        }
    };

    int b = 0, h = 0, hk = 0, base = 0, T = 0, par0 = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ... and whatever is launched behind this grid with the same attribute (the next call's kernel, which itself
    // waits for this grid to complete before it reads or writes anything) may be made resident now.
    asm volatile("griddepcontrol.launch_dependents;");
    Cursor ucur = cursor_at((int)blockIdx.x);
    bool cur_ok;
    cur_ok = decode(ucur, decode_load(ucur), b, h, hk, base, T, par0);
    bool par_bad = false;
    if (cur_ok) {
        issue_kq(b, hk, base, T);
        fetch_path(b, 0);
        par_bad = load_parent(par0, T, 0);
    }
    __syncthreads();
    if (cur_ok) load_tables(h, base, T, 0, par_bad);
    __syncthreads();
    if (cur_ok) {
        path_decay(0);
        fetch_path_kv(h, hk, 0);
        path_scalars_direct(h, 0);
        issue_gram(0);
    }
    int done_units = 0;
#pragma unroll 1
    for (int iter = 0; ucur.u < n_units; ++iter) {
    const uint32_t par = (uint32_t)(done_units & 1);   // every barrier completes once per processed unit
    int nb = 0, nh = 0, nhk = 0, nbase = 0, nT = 0, npar0 = 0;
    Cursor ncur = ucur;
    advance(ncur);
    bool next_ok = false;
    const DecodeRaw next_raw = decode_load(ncur);   // looked at in the middle of the unit (stage 1)
    auto decode_next = [&]() {
        next_ok = decode(ncur, next_raw, nb, nh, nhk, nbase, nT, npar0);
    };
    float4 *gab = reinterpret_cast<float4 *>(smem + SM_GAB + (iter & 1) * SM_TABLE_STRIDE);
    uint8_t *anc_s = smem + SM_ANC + (iter & 1) * SM_TABLE_STRIDE;
    uint8_t *depth_s = smem + SM_DEPTH + (iter & 1) * SM_TABLE_STRIDE;
    // L2 warming for this CTA's next unit, in slices at phase boundaries
    auto warm_l2_state = [&](int slice) {
        if (tid == 96 && ncur.u < n_units)
            prefetch_l2_bulk(p.S0 + (size_t)(ncur.b * p.h_v + ncur.h) * FV_D * FV_D + (size_t)slice * 4096, 16384);
    };

    // a tree whose parent[] was rejected while its tables were built runs as a tree of no nodes: nothing of it
    // is stored (fused form: its accepted path of the previous step is committed all the same)
    if (bad_s[iter & 1]) {
        T = 0;
        if (tid < FV_T) depth_s[tid] = 0;
    }
    // (1) state tile loads: a warp instruction covers four rows; the eight lanes of a row each own one
    // 16-byte bf16 piece of either K half.  Needed only after the Gram / coefficient phases.
    float4 x[4][4];   // [row i][kh*2 + half]
    // The load/store unit takes a while to accept 64 KB of requests: the tile is asked for in pieces -- a half at the
    // top and a half behind the Gram copy when the commit needs the tile right after the coefficients; a quarter at
    // the top, a quarter behind the Gram wait and a half behind the Gram copy otherwise -- so that the threads are
    // not held at the top of the unit for all of it.
    auto load_state_rows = [&](int i0, int i1) {
        const float *S = p.S0 + (size_t)(b * p.h_v + h) * FV_D * FV_D;
#pragma unroll
        for (int i = i0; i < i1; ++i) {
            const float *src = S + (size_t)(warp * 16 + i * 4 + r4) * FV_D + l8 * 8;
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) ldg_v8(src + kh * 64, x[i][kh * 2 + 0], x[i][kh * 2 + 1]);
        }
    };
    load_state_rows(0, 2);
    // this tree's v rows: one TMA box into an area that stays free until the state operand is written
    if (warp == W_TMA && elect_one()) {
        mbar_expect_tx(mbar_v, FV_T * FV_D * 2);
        tma_load_3d(sbase + SM_VE, &p.tm_v, 0, h, base, mbar_v);
    }
    // fused commit: this tree's accepted path of the previous step was fetched one unit ahead
    const float4 *ab_path = reinterpret_cast<const float4 *>(smem + SM_PATH + (iter & 1) * SM_PATH_SLOT + 128);
    int path_len = 0;
    path_len = reinterpret_cast<const int *>(smem + SM_PATH + (iter & 1) * SM_PATH_SLOT)[16];

    // Everything that depends only on q, k, g, beta runs now, under the latency of the state loads.  The Gram
    // block of this unit was issued one unit ahead; every thread waits for it on its own (bounded: on expiry it
    // flags the error and everybody falls through to the clean-up).
    if (!mbar_wait_bounded(mbar_g, par)) *flag = 1;
    tc_fence_after();
    __syncthreads();
    warm_l2_state(0);
    if (*flag == 0) {
        // k-columns of the Gram block out of tensor memory, into the (still unused) state-operand area
        {
            const int row = (warp & 3) * 32 + lane;
            const int half = warp >> 2;   // TMEM columns 192 + 32*half .. : k_j for j = 32*half ..
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 192 + half * 32;
            // SMALL: only rows k_0..k_31, q_0..q_31 against columns k_0..k_31 can belong to the tree
            if (!SMALL || (half == 0 && (warp & 1) == 0)) {
                uint32_t ra[32];
                GDN_TMEM_LD32(taddr, ra);
                tmem_wait_ld();
                // row r of the copy: 16 pieces of four columns, piece c stored at position c ^ (r & 15), so that the
                // 16-byte stores of a quarter-warp (eight consecutive rows, same piece) hit all the banks once
#pragma unroll
                for (int c4 = 0; c4 < 8; ++c4)
                    *reinterpret_cast<uint4 *>(gram + row * 64 + (((half * 8 + c4) ^ (row & 15)) << 2)) =
                        make_uint4(ra[4 * c4], ra[4 * c4 + 1], ra[4 * c4 + 2], ra[4 * c4 + 3]);
            }
        }
        load_state_rows(2, 4);
        tc_fence_before();
        __syncthreads();
        warm_l2_state(1);
        // X and Y for real ancestors only; the decay from node j down to node i is the exponential of what stands in Y's place
        // (SMALL: nodes 32.. do not exist; their rows of X and Y are never looked at)
        {
            constexpr int NU = SMALL ? 2 : 4;
            float gdiff[4], gk[4], gq[4], bi[4];
            bool on[4], onx[4];
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                const int idx = u * FV_THREADS + tid;
                const int i = idx >> 4, t = idx & 15;
                const int d = depth_s[i];
                on[u] = t < d;
                onx[u] = t < d - 1;
                const int j = on[u] ? anc_s[idx] : 0;
                gdiff[u] = ys[idx];
                bi[u] = gab[i].z;
                const int jpos = (((j >> 2) ^ (i & 15)) << 2) | (j & 3);   // rows i and 64 + i share i & 15
                gq[u] = gram[(64 + i) * 64 + jpos];   // row 64 + i: q_i
                gk[u] = gram[i * 64 + jpos];          // row i: k_i
            }
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                const int idx = u * FV_THREADS + tid;
                const float dec = __expf(gdiff[u]);
                ys[idx] = on[u] ? dec * gq[u] : 0.f;
                xs[idx] = onx[u] ? bi[u] * dec * gk[u] : 0.f;
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();   // X and Y complete; the Gram copy is dead and its area can take the state operand

    // (3') fused commit: replay Eq. 7 along the previous step's accepted path on the state tile while it
    // sits in registers, write it back, and let everything below verify the new tree against it.
    // Per row c (one value component): s_c <- alpha s_c + k beta (v_c - alpha k.s_c); the eight lanes that
    // share a row reduce k.s_c with three shuffles.  The path's k/v rows were fetched above.
    const bool healthy = *flag == 0;   // uniform: every write of the flag so far lies before the barrier above
    if (!healthy) path_len = 0;    // a wait expired: this state is left as it was
    if (path_len > 0) {
        replay_path_on_tile(x, path_len, reinterpret_cast<const uint16_t *>(smem + SM_PK),
                            reinterpret_cast<const uint16_t *>(smem + SM_PV), ab_path, warp * 16, r4, l8);
    }
    // The v rows move into registers in the orientation of the R phase (component c = TMEM lane of this
    // thread, its 32 nodes, two bf16 per register): they are about to be overwritten by the state operand.
    uint32_t vreg[16];
    {
        if (!mbar_wait_bounded(mbar_v, par)) *flag = 1;
        const uint16_t *ve = reinterpret_cast<const uint16_t *>(smem + SM_VE) + ((warp >> 2) * 32) * FV_D +
                             (warp & 3) * 32 + lane;
#pragma unroll
        for (int m = 0; m < 16; ++m)
            vreg[m] = (uint32_t)ve[(2 * m) * FV_D] | ((uint32_t)ve[(2 * m + 1) * FV_D] << 16);
    }
    __syncthreads();   // the v rows and the path rows sit where the state operand is about to be written

    // (4) fp32 -> bf16 hi + lo, written as the A operand.  The committed state -- the only state write of
    // the step -- goes out from the same registers, one 32-byte store in front of each piece's conversion so
    // that the stores drain while the arithmetic runs.
    float *S_out = nullptr;
    if (path_len > 0) S_out = p.S_rw + (size_t)(b * p.h_v + h) * FV_D * FV_D;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = warp * 16 + i * 4 + r4;
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) {
            if (S_out) stg_v8(S_out + (size_t)row * FV_D + l8 * 8 + kh * 64, x[i][kh * 2 + 0], x[i][kh * 2 + 1]);
            const float4 u = x[i][kh * 2 + 0], w = x[i][kh * 2 + 1];
            const float f[8] = {u.x, u.y, u.z, u.w, w.x, w.y, w.z, w.w};
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) split_pack_bf16(f[2 * e], f[2 * e + 1], hi[e], lo[e]);
            const uint32_t off = sw128_offset(row, kh * 8 + l8);
            *reinterpret_cast<uint4 *>(smem + SM_A_HI + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4 *>(smem + SM_A_LO + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
    fence_proxy_async();   // generic-proxy writes of the operand become visible to the tensor core
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    warm_l2_state(2);
    // (5) P = S0.[k;q]^T (hi then lo) on the tensor core, issued before anything else; meanwhile the loads of stage 1
    // and the back-substitution below
    if (warp == W_MMA_P && elect_one()) {
        const uint64_t a_hi = smem_desc_sw128(sbase + SM_A_HI), a_lo = smem_desc_sw128(sbase + SM_A_LO);
        const uint64_t b_kq = smem_desc_sw128(sbase + SM_B_KQ);
        constexpr uint32_t id = idesc_bf16(128, 128);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const uint64_t adv = (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4);
            umma_bf16(tmem, a_hi + adv, b_kq + adv, id, ks > 0);
        }
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const uint64_t adv = (uint64_t)(((ks >> 2) * 16384 + (ks & 3) * 32) >> 4);
            umma_bf16(tmem, a_lo + adv, b_kq + adv, id, 1);
        }
        umma_commit(mbar_p);
    }
    // The next unit's tables and accepted path are fetched in stages, each load issued one phase before its
    // value is used, so that no global-memory latency is paid in front of a barrier.
    // stage 1: table entries of node `tid` and the path bounds (registers only)
    int t_par = -1;
    bool t_bad = false;
    unsigned short t_g = 0, t_be = 0;
    int q_pp0 = 0, q_len = 0, q_pb = 0, q_pT = 0, q_ppar = 0, q_n = -1, q_par = -2;
    unsigned short q_g = 0, q_be = 0;
    bool q_shape_ok = false, q_mine = false;
    decode_next();
    const bool same_tree = PADDED && next_ok && tree_of(nb) == tree_of(b);
    if (next_ok) {
        if (tbl_thread && tnode < nT) {
            const int n = nbase + tnode;
            if (!same_tree) t_par = __ldg(p.parent + npar0 + tnode);
            t_g = __ldg(reinterpret_cast<const unsigned short *>(p.g) + (size_t)n * p.h_v + nh);
            t_be = __ldg(reinterpret_cast<const unsigned short *>(p.beta) + (size_t)n * p.h_v + nh);
        }
        if (warp == 4) {
            if (PADDED) {   // (stage 2 takes differences: hand it begin / end pairs)
                const int tree = tree_of(nb);
                q_pp0 = tree * p.path_stride;
                q_len = q_pp0 + p.path_len[tree];
                q_pb = nb * p.pt_pad;
                q_pT = q_pb + min(p.pn_nodes[tree], p.pt_pad);
                q_ppar = tree * p.pt_pad;
            } else {
                q_pp0 = p.path_offsets[nb];
                q_len = p.path_offsets[nb + 1];
                q_pb = p.pnode_offsets[nb];
                q_pT = p.pnode_offsets[nb + 1];
                q_ppar = q_pb;
            }
        }
    }

    // (6) z^T = y^T (I + X_path)^-1 by back-substitution over the root path (column-oriented: once z_l is
    // final, subtract z_l X(n_l, n_t) from every z_t, t < l).  Four threads per node, thread sq of the quad
    // owning path positions 4 sq .. 4 sq + 3; z stays in registers until the k/q tile can be overwritten.
    const int zi = tid >> 2, sq = tid & 3;
        const int d = depth_s[zi];
        const int dmax = __reduce_max_sync(0xffffffffu, d);
        const uint4 row = *reinterpret_cast<const uint4 *>(anc_s + zi * 16);
        const uint32_t idw[4] = {row.x, row.y, row.z, row.w};
        const float4 y4 = *reinterpret_cast<const float4 *>(ys + zi * FV_MD + sq * 4);
        float z[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
        for (int l = FV_MD - 1; l >= 1; --l) {
            if (l < dmax) {   // warp-uniform
                const float zl = __shfl_sync(0xffffffffu, z[l & 3], (lane & ~3) | (l >> 2));
                if (l < d && sq * 4 < l) {
                    const int nl = (int)((idw[l >> 2] >> ((l & 3) * 8)) & 0xFFu);
                    const float4 x4 = *reinterpret_cast<const float4 *>(xs + nl * FV_MD + sq * 4);
                    const float xv[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (sq * 4 + e < l) z[e] = fmaf(-zl, xv[e], z[e]);
                }
            }
        }
    // stage 2: the path entries
    if (next_ok && warp == 4) {
        q_len -= q_pp0;
        q_pT -= q_pb;
        q_shape_ok = q_len > 0 && q_len <= FV_MD && q_len <= p.max_depth && q_pT > 0 && q_pp0 >= 0;
        q_mine = q_shape_ok && lane < q_len;
        if (q_mine) q_n = p.path[q_pp0 + lane];
    }
    bool unit_done_ok = false;
    // From here to the output staging every thread waits on the barriers of the tensor core and of TMA itself;
    // an expired wait only raises the flag, which is looked at behind the next CTA barrier (uniform decision).
    if (!mbar_wait_bounded(mbar_p, par)) *flag = 1;
    tc_fence_after();
    warm_l2_state(3);

    {
        // (7) both operand tiles are dead now: z is scattered into the dense bf16 hi/lo tiles Z[i][j] (zero off
        // the root path) over the state operand
        // the k/q tile is dead: start on the next unit of this CTA (its k/q tile, its tables), to be
        // consumed after the loop comes round
        if (next_ok) {
            issue_kq(nb, nhk, nbase, nT);
            // stage 3: parent[] of the next tree is staged for the walk behind the next CTA barrier; the parents of
            // the path entries are asked for
            t_bad = put_parent(nT, t_par, (iter + 1) & 1, same_tree);
            if (warp == 4) {
                // the entries are published as far as they are checked (inside the previous tree), so that
                // their rows can be asked for behind the next barrier; whether they form a chain is decided then
                int *slot = reinterpret_cast<int *>(smem + SM_PATH + ((iter + 1) & 1) * SM_PATH_SLOT);
                const bool in_range = q_mine && q_n >= 0 && q_n < q_pT;
                const bool all_in = __all_sync(0xffffffffu, !q_mine || in_range);
                if (lane < FV_MD) slot[lane] = in_range ? q_n : 0;
                if (lane == 0) {
                    slot[17] = q_pb;
                    slot[18] = q_shape_ok && all_in ? q_len : 0;
                }
                if (in_range && p.pparent) q_par = p.pparent[q_ppar + q_n];
            }
        }
        {
            const int i = zi;
            const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4 *>(smem + SM_Z_HI + sw128_row_offset(i, 2 * sq)) = zero4;
            *reinterpret_cast<uint4 *>(smem + SM_Z_HI + sw128_row_offset(i, 2 * sq + 1)) = zero4;
            *reinterpret_cast<uint4 *>(smem + SM_Z_LO + sw128_row_offset(i, 2 * sq)) = zero4;
            *reinterpret_cast<uint4 *>(smem + SM_Z_LO + sw128_row_offset(i, 2 * sq + 1)) = zero4;
            __syncwarp();   // the quad's zero fill precedes the scattered stores below
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int t = sq * 4 + e;
                if (t < d) {
                    const int j = (int)((idw[sq] >> (e * 8)) & 0xFFu);
                    float hi, lo;
                    split_bf16(z[e], hi, lo);
                    const uint32_t off = sw128_row_offset(i, j >> 3) + (j & 7) * 2;
                    *reinterpret_cast<__nv_bfloat16 *>(smem + SM_Z_HI + off) = __float2bfloat16_rn(hi);
                    *reinterpret_cast<__nv_bfloat16 *>(smem + SM_Z_LO + off) = __float2bfloat16_rn(lo);
                }
            }
        }

        // (8) all warps: r_j[c] = beta_j (v_j[c] - a_j p^k_j[c]) for component c = TMEM lane and 32 nodes,
        // split into bf16 hi/lo and stored as the K-major A operand R^T[c][j]
        {
            const int c = (warp & 3) * 32 + lane;
            const int half = warp >> 2;
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
            for (int part = 0; part < 2; ++part) {
                const int j0 = half * 32 + part * 16;
                if (SMALL && j0 >= T) {   // no node of the tree in this 16-column piece: exact zeros for the D GEMM
                    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                    for (int oct = 0; oct < 2; ++oct) {
                        const uint32_t off = sw128_row_offset(c, half * 4 + part * 2 + oct);
                        *reinterpret_cast<uint4 *>(smem + SM_RT_HI + off) = zero4;
                        *reinterpret_cast<uint4 *>(smem + SM_RT_LO + off) = zero4;
                    }
                    continue;
                }
                uint32_t rr[16];
                GDN_TMEM_LD16(taddr + j0, rr);   // columns j0 .. j0+15: p^k of 16 nodes
                float vv[16], aj[16], bj[16];
                uint32_t vpart[8];
#pragma unroll
                for (int m = 0; m < 8; ++m) vpart[m] = part ? vreg[8 + m] : vreg[m];
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) {
                    const uint32_t vw = vpart[jj >> 1];
                    vv[jj] = __uint_as_float((jj & 1) ? (vw & 0xFFFF0000u) : (vw << 16));
                    const float4 gj = gab[j0 + jj];
                    aj[jj] = gj.y;
                    bj[jj] = gj.z;
                }
                tmem_wait_ld();
                uint32_t hi[8], lo[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    // nodes beyond the tree hold another tree's rows: their r is forced to an exact zero
                    const float r0 = j0 + 2 * e < T ? bj[2 * e] * (vv[2 * e] - aj[2 * e] * __uint_as_float(rr[2 * e])) : 0.f;
                    const float r1 = j0 + 2 * e + 1 < T
                                         ? bj[2 * e + 1] * (vv[2 * e + 1] - aj[2 * e + 1] * __uint_as_float(rr[2 * e + 1]))
                                         : 0.f;
                    split_pack_bf16(r0, r1, hi[e], lo[e]);
                }
#pragma unroll
                for (int oct = 0; oct < 2; ++oct) {
                    const uint32_t off = sw128_row_offset(c, half * 4 + part * 2 + oct);
                    *reinterpret_cast<uint4 *>(smem + SM_RT_HI + off) = make_uint4(hi[4 * oct], hi[4 * oct + 1], hi[4 * oct + 2], hi[4 * oct + 3]);
                    *reinterpret_cast<uint4 *>(smem + SM_RT_LO + off) = make_uint4(lo[4 * oct], lo[4 * oct + 1], lo[4 * oct + 2], lo[4 * oct + 3]);
                }
            }
        }
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();

        // (9) second MMA group: D[c][i] = sum_j R^T[c][j] Z[i][j] with the hi/lo cross terms
        if (warp == W_MMA_D && elect_one()) {
            constexpr uint32_t id2 = idesc_bf16(128, 64);
            const uint64_t a2[2] = {smem_desc_sw128(sbase + SM_RT_HI), smem_desc_sw128(sbase + SM_RT_LO)};
            const uint64_t b2[2] = {smem_desc_sw128(sbase + SM_Z_HI), smem_desc_sw128(sbase + SM_Z_LO)};
#pragma unroll
            for (int combo = 0; combo < 3; ++combo) {   // hi.hi, lo.hi, hi.lo; lo.lo is below 2^-18 of the result
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_bf16(tmem + 128, a2[combo & 1] + (uint64_t)(ks * 2), b2[combo >> 1] + (uint64_t)(ks * 2), id2,
                              (combo | ks) != 0);
            }
            umma_commit(mbar_d);
        }
        // stage 4: the path is checked (a chain from a root inside the previous tree) and published; the
        // per-step scalars of its nodes are asked for
        if (next_ok && warp == 4) {
            int *slot = reinterpret_cast<int *>(smem + SM_PATH + ((iter + 1) & 1) * SM_PATH_SLOT);
            const int n_up = __shfl_up_sync(0xffffffffu, q_n, 1);
            bool bad = false;
            if (q_mine) {
                if (q_n < 0 || q_n >= q_pT) bad = true;
                else if (p.pparent) bad = q_par != (lane ? n_up : -1);
                else if (lane && q_n <= n_up) bad = true;
            }
            if (q_len != 0 && (__any_sync(0xffffffffu, bad) || !q_shape_ok)) {
                if (lane == 0) report_status(p.status_dev, GDN_ERR_PATH);
                q_len = 0;
            }
            if (lane == 0) {
                slot[16] = q_len;
                slot[17] = q_pb;
            }
            if (lane < q_len) {
                const size_t n = (size_t)q_pb + q_n;
                q_g = __ldg(reinterpret_cast<const unsigned short *>(p.pg) + n * p.h_v + nh);
                q_be = __ldg(reinterpret_cast<const unsigned short *>(p.pbeta) + n * p.h_v + nh);
            }
        }

        // stage 5, while the tensor core works: the next unit's tables (depth, root paths) from the staged parent[]
        if (next_ok) walk_tables(nT, (iter + 1) & 1, t_g, t_be, t_bad, same_tree);
        if (!mbar_wait_bounded(mbar_d, par)) *flag = 1;
        tc_fence_after();

        // (10) outputs: o_i[c] = scale (a_i p^q_i[c] + D[c][i]), staged through shared memory (over the
        // dead R^T tiles) so that global memory sees 16-byte stores of whole rows
        {
            const int c = (warp & 3) * 32 + lane;
            const int half = warp >> 2;
            const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
            TOut *o_s = reinterpret_cast<TOut *>(smem + SM_RT_HI);   // [64][128] TOut: 16 or 32 KB
#pragma unroll 1
            for (int part = 0; part < 2; ++part) {
                const int i0 = half * 32 + part * 16;
                if constexpr (SMALL) {
                    if (i0 >= T) continue;   // rows beyond the tree are never stored
                }
                uint32_t pp[16], dd[16];
                GDN_TMEM_LD16(trow + 64 + i0, pp);    // p^q of 16 nodes
                GDN_TMEM_LD16(trow + 128 + i0, dd);
                float ai[16];
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) ai[jj] = gab[i0 + jj].y;
                tmem_wait_ld();
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) {
                    const float out = p.scale * fmaf(ai[jj], __uint_as_float(pp[jj]), __uint_as_float(dd[jj]));
                    store_from_float(o_s + (i0 + jj) * FV_D + c, out);
                }
            }
        }
        __syncthreads();
        // stage 6: the next unit's decay tables, and its path rows (published above, behind a barrier now; the area
        // they land in is free)
        if (next_ok) path_decay((iter + 1) & 1);
        if (next_ok) fetch_path_kv(nh, nhk, (iter + 1) & 1);
        // ... and the scalars of that path (asked for a phase ago)
        if (next_ok && warp == 4) {   // lane t: decay of the path up to and including step t by a prefix sum
            const float gt = lane < q_len ? gate_log_decay(q_g, PADDED && p.raw_gates) : 0.f;
            float gsum = gt;
#pragma unroll
            for (int off = 1; off < FV_MD; off <<= 1) {
                const float up = __shfl_up_sync(0xffffffffu, gsum, off);
                if (lane >= off) gsum += up;
            }
            if (lane < q_len) {
                const float A = expf(gsum);
                reinterpret_cast<float4 *>(smem + SM_PATH + ((iter + 1) & 1) * SM_PATH_SLOT + 128)[lane] =
                    make_float4(A, gate_beta(q_be, PADDED && p.raw_gates), expf(gt), 1.f / A);
            }
        }
        unit_done_ok = *flag == 0;
        if (unit_done_ok) {
            constexpr int ROW_CHUNKS = FV_D * (int)sizeof(TOut) / 16;   // 16-byte pieces per output row
            uint8_t *o = static_cast<uint8_t *>(p.o);
            for (int idx = tid; idx < T * ROW_CHUNKS; idx += FV_THREADS) {
                const int i = idx / ROW_CHUNKS, ck = idx % ROW_CHUNKS;
                const uint4 val = *reinterpret_cast<const uint4 *>(smem + SM_RT_HI + (size_t)i * FV_D * sizeof(TOut) + ck * 16);
                *reinterpret_cast<uint4 *>(o + (((size_t)(base + i) * p.h_v + h) * FV_D) * sizeof(TOut) + ck * 16) = val;
            }
        }
    }
    ++done_units;
    if (!unit_done_ok) break;   // a bounded wait expired: stop, report, release
    if (next_ok) issue_gram((uint32_t)(done_units & 1));   // the next unit's Gram block, as soon as its tile is there
    b = nb; h = nh; hk = nhk; base = nbase; T = nT; cur_ok = next_ok;
    ucur = ncur;
    }   // unit loop

    if (*flag != 0 && tid == 0) report_status(p.status_dev, GDN_ERR_TIMEOUT);
    cp_async_wait_all();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, FV_TMEM_COLS);
}

template <typename TOut> cudaError_t launch_typed(const gdn_shape_t &s, const VerifyFastParams &p, cudaStream_t stream)
{
    // persistent CTAs, two per SM, pipelined across units
    VerifyFastParams pt = p;
    const bool padded = p.t_pad != 0, small = s.max_tree_nodes <= 32;
    if (!make_row_tensor_map(&pt.tm_k, p.k, s.total_nodes, s.h_qk, 64, FV_T, true) ||
        !make_row_tensor_map(&pt.tm_q, p.q, s.total_nodes, s.h_qk, 64, FV_T, true) ||
        !make_row_tensor_map(&pt.tm_v, p.v, s.total_nodes, s.h_v, FV_D, FV_T, false))
        return cudaErrorNotSupported;
    // the padded layout and the on-chip gate activations share an instantiation
    void (*kernel)(const VerifyFastParams) = small ? padded ? commit_verify_kernel<TOut, true, true> : commit_verify_kernel<TOut, true, false>
                                                   : padded ? commit_verify_kernel<TOut, false, true> : commit_verify_kernel<TOut, false, false>;
    static PerContext seen[4];
    int sms = 0;
    const cudaError_t e = device_sms(seen[2 * padded + small], reinterpret_cast<const void *>(kernel),
                                     SM_ALLOC, &sms);
    if (e != cudaSuccess) return e;
    const int grid = pt.n_units < 2 * sms ? pt.n_units : 2 * sms;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(FV_THREADS);
    cfg.dynamicSmemBytes = SM_ALLOC;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, pt);
}

VerifyFastParams make_params(const gdn_shape_t &s, const float *S0, const void *q, const void *k, const void *v,
                             const void *g, const void *beta, const int32_t *node_offsets, void *o,
                             int32_t *status_dev)
{
    VerifyFastParams p{};
    p.h_qk = s.h_qk; p.h_v = s.h_v; p.n_units = s.n_seq * s.h_v; p.scale = s.scale;
    p.S0 = S0;
    p.q = static_cast<const __nv_bfloat16 *>(q); p.k = static_cast<const __nv_bfloat16 *>(k);
    p.v = static_cast<const __nv_bfloat16 *>(v); p.g = static_cast<const __nv_bfloat16 *>(g);
    p.beta = static_cast<const __nv_bfloat16 *>(beta);
    p.node_offsets = node_offsets; p.o = o;
    p.n_seq = s.n_seq; p.total_nodes = s.total_nodes; p.max_tree_nodes = s.max_tree_nodes; p.max_depth = s.max_depth;
    p.status_dev = status_dev;
    return p;
}

}  // namespace

// Few units: the commit kernel and, behind it, the verification, which works out everything but the product with the state
// meanwhile -- the two run side by side on SMs of their own as long as there are enough of them.  Measured (us, 64 nodes;
// this kernel / two kernels), path of 7: 32 units 13.3 / 9.5, 64 units 13.5 / 9.7, 128 units 13.9 / 13.0; path of 1: 64 units
// 11.3 / 9.9, 128 units 11.6 / 12.3 (the path lengths are on the device, so the line lies where both gain).
static bool as_two_kernels(const gdn_shape_t &s)
{
    static PerContext seen;
    int sms = 0;
    return device_sms(seen, nullptr, 0, &sms) == cudaSuccess && s.n_seq * s.h_v <= sms / 2;
}

cudaError_t launch_commit_verify_sm100_padded(const gdn_shape_t &s, int n_trees, bool raw_gates, float *S,
                                              int prev_t_pad, const void *k_prev, const void *v_prev,
                                              const void *g_prev, const void *beta_prev, const int32_t *parent_prev,
                                              const int32_t *n_nodes_prev, const int32_t *path,
                                              const int32_t *path_len, const void *q, const void *k, const void *v,
                                              const void *g, const void *beta, const int32_t *parent,
                                              const int32_t *n_nodes, void *o, int32_t *status_dev,
                                              cudaStream_t stream)
{
    if (s.n_seq == 0 || s.total_nodes == 0) return cudaSuccess;
    if (step_small_supported(s)) {
        const CommitParams prev{s.h_qk, s.h_v, s.d_k, s.d_v, s.max_depth, S, k_prev, v_prev, g_prev, beta_prev, parent_prev, nullptr,
                                path, nullptr, status_dev, prev_t_pad, n_trees, s.max_depth, raw_gates ? 1 : 0, n_nodes_prev, path_len};
        return launch_step_small(s, prev, true, q, k, v, g, beta, parent, nullptr, n_trees, n_nodes, o, stream);
    }
    if (as_two_kernels(s)) {
        gdn_shape_t ps = s;   // the commit reads the slots of the previous step
        ps.max_tree_nodes = prev_t_pad;
        const auto commit = [&] {
            return launch_commit_padded(ps, n_trees, raw_gates, S, k_prev, v_prev, g_prev, beta_prev, parent_prev, n_nodes_prev,
                                        path, path_len, status_dev, stream);
        };
        return launch_verify_sm100_padded(s, n_trees, raw_gates, S, q, k, v, g, beta, parent, n_nodes, o, status_dev, stream,
                                          in_front(commit));
    }
    VerifyFastParams p = make_params(s, S, q, k, v, g, beta, nullptr, o, status_dev);
    p.parent = parent;
    p.t_pad = s.max_tree_nodes; p.n_trees = n_trees; p.n_nodes = n_nodes; p.raw_gates = raw_gates ? 1 : 0;
    p.S_rw = S;
    p.pk = static_cast<const __nv_bfloat16 *>(k_prev); p.pv = static_cast<const __nv_bfloat16 *>(v_prev);
    p.pg = static_cast<const __nv_bfloat16 *>(g_prev); p.pbeta = static_cast<const __nv_bfloat16 *>(beta_prev);
    p.pparent = parent_prev; p.path = path;
    p.pt_pad = prev_t_pad; p.pn_nodes = n_nodes_prev; p.path_len = path_len; p.path_stride = s.max_depth;
    if (s.out_dtype == GDN_BF16) return launch_typed<__nv_bfloat16>(s, p, stream);
    return launch_typed<float>(s, p, stream);
}

cudaError_t launch_commit_verify_sm100(const gdn_shape_t &s, float *S, const void *k_prev, const void *v_prev,
                                       const void *g_prev, const void *beta_prev, const int32_t *parent_prev,
                                       const int32_t *node_offsets_prev, const int32_t *path,
                                       const int32_t *path_offsets, const void *q, const void *k, const void *v,
                                       const void *g, const void *beta, const int32_t *parent,
                                       const int32_t *node_offsets, void *o, int32_t *status_dev,
                                       cudaStream_t stream)
{
    if (s.n_seq == 0 || s.total_nodes == 0) return cudaSuccess;
    if (step_small_supported(s)) {
        const CommitParams prev{s.h_qk, s.h_v, s.d_k, s.d_v, s.max_depth, S, k_prev, v_prev, g_prev, beta_prev, parent_prev, node_offsets_prev,
                                path, path_offsets, status_dev, 0, 0, 0, 0, nullptr, nullptr};
        return launch_step_small(s, prev, true, q, k, v, g, beta, parent, node_offsets, 1, nullptr, o, stream);
    }
    if (as_two_kernels(s)) {
        const auto commit = [&] {
            return launch_commit_generic(s, S, k_prev, v_prev, g_prev, beta_prev, parent_prev, node_offsets_prev, path,
                                         path_offsets, status_dev, stream);
        };
        return launch_verify_sm100(s, S, q, k, v, g, beta, parent, node_offsets, o, PlanPtrs{}, status_dev, stream, in_front(commit));
    }
    VerifyFastParams p = make_params(s, S, q, k, v, g, beta, node_offsets, o, status_dev);
    p.parent = parent;
    p.S_rw = S;
    p.pk = static_cast<const __nv_bfloat16 *>(k_prev); p.pv = static_cast<const __nv_bfloat16 *>(v_prev);
    p.pg = static_cast<const __nv_bfloat16 *>(g_prev); p.pbeta = static_cast<const __nv_bfloat16 *>(beta_prev);
    p.pparent = parent_prev; p.pnode_offsets = node_offsets_prev; p.path = path; p.path_offsets = path_offsets;
    if (s.out_dtype == GDN_BF16) return launch_typed<__nv_bfloat16>(s, p, stream);
    return launch_typed<float>(s, p, stream);
}


}  // namespace gdn
