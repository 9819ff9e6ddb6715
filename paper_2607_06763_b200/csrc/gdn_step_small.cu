// Verification of trees of at most SS_MAX_NODES nodes, alone or behind the commit of the previous step's accepted path in the
// same pass over the state: d_k = d_v = 128, bf16 inputs, root paths of at most 16 nodes.
//
// The mathematics is that of gdn_verify_plain.cu (the solve on the query side, one product with the state per node):
//     coefficients:  Gram = [k;q].k^T -> w by back-substitution -> q' = sa q - sa w.K,  z' = scale dec w
//     output:        O [d_v x nodes] = V^T.z' + S.q'^T
// and that of the commit gdn_fragments.cuh; both take the state tile through registers as fragments of m16n8k16, so that a chunk
// that the commit has just advanced is split (hi + lo) and multiplied with q' before it leaves the registers.  Contractions run
// on warp-level tensor-core instructions: with so few nodes they are small, and what a unit costs is its chain of dependent
// steps and the state's way through the SM.  There is no tensor memory to hand out and no 64-row tile to fill, so that up to four
// CTAs of one unit each share an SM, and the loads of one run under the arithmetic of the others.
//
// Measured (us, 32 heads; the kernels of 64-node tiles / this one), trees of 16 nodes: 64 chains, accepted paths of 0 / 1 / 7 / 16
// nodes 66.5 / 82.2 / 100.6 / 132.5 -> 44.4 / 75.7 / 80.7 / 91.2 (the state read and written once at the copy bandwidth: 41), verification
// alone 44.6 -> 35.0; 48 geometric trees, paths of 0 / 1 / 7 47.8 / 60.2 / 67.6 -> 33.1 / 59.1 / 62.2; one layer, path of 7 11.4 -> 8.2.
// Error of fp32 outputs against 64 bits, in the norm, 40 trees of 16 nodes: verification 2.9e-6 -> 2.8e-6, step 4.3e-6 -> 2.6e-6 (its
// state 5.9e-8 -> 5.1e-8).  Bound by HBM latency and the chain of a unit.
#include "gdn_path.cuh"
#include "gdn_tc.cuh"

namespace gdn {

namespace {

constexpr int SS_THREADS = CF_THREADS;
constexpr int SS_D = GDN_TILE_D;
constexpr int SS_ROW = GDN_PK_STRIDE;   // bytes from one row of an operand to the next

struct StepSmallParams {
    CommitParams c;   // the previous step (COMMIT); c.S: the state, of either form
    int n_seq, total_nodes, max_tree_nodes;
    int rows_early;   // L2 is asked for the rows before the kernel in front has completed
    float scale;
    const __nv_bfloat16 *q, *k, *v, *g, *beta;
    const int32_t *parent, *node_offsets;
    void *o;
    int t_pad, n_trees;   // padded layout (0: ragged packing): slot b keeps its rows at b * t_pad and carries tree b % n_trees
    const int32_t *n_nodes;
    // PLANNED: padded layout, node counts and root paths out of a plan of the n_trees trees (unit list, its count and shape mark, paths)
    SmallTreePlan plan;
};

// CTAs per SM: what the registers give without spilling more than a few words (N = 16 alone at three instead of four: 36.2 us for
// 64 chains of 16 nodes instead of 35.0; N = 32 alone at three instead of two: 12.7 us for 8 trees instead of 9.8).
// A commit at four spills 64 words' worth, which paths of more than 8 nodes pay for (step of 64 chains of 16 nodes, paths of 16 / 7: 91.3 /
// 80.9 at three, 96.8 / 75.5 at four), so that it runs at four where such paths are not to be expected (trees of at most 8 nodes: 48 of
// them, path of 7, 61.0 / 57.6) or where that makes one wave of what would be two (16 trees of 16 nodes 27.9 / 23.4), but not where
// three are enough (12 trees 17.0 / 21.3).
inline bool commit_at_four(int max_tree_nodes, long long units, int sms)
{
    return units > 3LL * sms && (units <= 4LL * sms || max_tree_nodes <= 8);
}

// CTAs of a unit behind a commit (PARTS): one, or, while every one of them has an SM of its own, four or two that take 32 or 64 value
// components each, every warp on the key positions of one or two chunks of its rows, which then stay in its registers.  With the whole
// tile on one CTA the passes over it are 5300 of a unit's 11300 cycles (path of 1; 7500 behind one of 16), and its second half and both
// halves once more are waited for; the coefficients, which every CTA makes for itself, are done in less time than the rows take to
// come.  Calls in a row, us, paths of 1 / 8 / 9 / 16 nodes, 32 heads ("two kernels": commit, then the verification of 64-node tiles):
//                                                   two kernels             one CTA a unit         four or two parts
//   in a graph, in L2:      1 sequence, 16 nodes     8.3  8.3  8.3  9.5      7.9  8.7 10.2 10.6     5.4  6.1  6.9  7.3
//                           1 sequence, 32 nodes     8.5  8.5  8.5  9.6      9.4  9.8 10.8 11.2     7.6  7.9  8.7  9.1
//                           2 sequences, 16 nodes    8.6  9.3  9.9 11.9      8.0  8.8 10.3 10.8     6.3  6.9  7.6  8.1   (four: 6.7  7.5  8.6  9.2)
//                           2 sequences, 32 nodes    9.0  9.4 10.0 11.9      9.7 10.1 11.0 11.4     9.2  9.5 10.3 10.7   (four: 9.9 10.6 11.8 12.3)
//   in a graph, not in L2:  1 sequence, 16 nodes     9.0  9.0  9.6 11.0      9.3 10.2 12.0 12.4     6.5  7.3  8.4  8.7
//                           1 sequence, 32 nodes     9.3  9.3  9.7 11.1     10.9 11.3 12.6 13.0     8.5  8.9 10.0 10.4
//                           2 sequences, 16 nodes    9.2 10.6 11.4 13.5      9.7 10.6 12.3 12.8     7.7  8.4  9.4  9.8
//                           2 sequences, 32 nodes    9.5 10.6 11.5 13.5     11.4 11.8 13.0 13.4    10.4 10.7 11.7 12.2
//   by the host, not in L2: 2 sequences, 32 nodes   11.5 11.6 12.3 14.4     11.8 12.2 13.4 13.9    11.4 11.7 12.7 13.3
// (Two kernels stay faster for two sequences of 32 nodes and short paths in a graph; their commit goes step by step for so few tiles,
// which leaves the state up to 1.6e-7 off in the norm with raw gates, this one below 7e-8.)  Three sequences in two parts, two on some
// SMs: 16 nodes 7.9 8.9 9.8 10.4 instead of 8.0 8.8 10.4 10.8, 32 nodes 12.2 12.9 14.2 14.4 instead of 9.7 10.1 11.1 11.5.
inline int commit_parts(long long units, int sms) { return units <= sms / 4 ? 4 : units <= sms / 2 ? 2 : 1; }

// N: nodes a tree may have here (16 or 32).
template <int N, int PARTS> struct StepSmallSmem {
    static constexpr int W_ROW = 2 * N + 16;   // bytes from one row of w, z' to the next
    static constexpr int G_ROW = N + 4;        // floats from one row of the Gram block to the next
    // k, q, v rows (zero beyond the tree); over k and q, once q' is there, the outputs on their way out (PARTS > 1: the warps' shares of them)
    alignas(16) uint8_t rows[3][N * SS_ROW];
    alignas(16) uint8_t qp[2][N * SS_ROW];     // q' as bf16 hi, lo; before that the Gram block [k;q].k^T
    alignas(16) uint8_t wz[4][N * W_ROW];      // -sa w hi, lo; z' hi, lo
    alignas(16) uint8_t pk[CF_MD * SS_ROW];
    alignas(16) uint16_t pv[CF_MD * SS_D];
    alignas(16) float couple[CF_MD * 16];
    alignas(16) float products[PARTS == 1 ? 4 : 8 * 8 * 32];   // the warps' shares of the path's products with the old state
    float4 scal[CF_MD];
    uint32_t mask[N];                          // nodes on the root path
    float g[N], beta[N], sa[N];
    int len, bad;
    float decay;
    static_assert(2 * N * G_ROW * 4 <= 2 * N * SS_ROW, "the Gram block fits q'");
    static_assert(8 * N / 2 * 32 * 4 <= 2 * N * SS_ROW, "so do the shares of the outputs k and q");
};

// The sum of what the PARTS warps on the same rows have of an entry (s: the first one's, stride: from one warp to the next).
template <int PARTS> __device__ __forceinline__ float sum_shares(const float *s, int stride)
{
    constexpr int GROUPS = 8 / PARTS;
    if constexpr (PARTS == 2) return s[0] + s[GROUPS * stride];
    else return (s[0] + s[GROUPS * stride]) + (s[2 * GROUPS * stride] + s[3 * GROUPS * stride]);
}

// Acc[nodes] += S.q'^T of one chunk of 32 key positions: hi.hi, lo.hi, hi.lo (lo.lo is below 2^-18 of the result).
template <int N>
__device__ __forceinline__ void output_chunk(const float (&x)[4][4], int jj, uint32_t q_hi, float (&acc)[N / 8][4])
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) split_pack_bf16(x[2 * h + (i >> 1)][2 * (i & 1)], x[2 * h + (i >> 1)][2 * (i & 1) + 1], hi[i], lo[i]);
#pragma unroll
        for (int n = 0; n < N / 8; n += 2) {
            // b: of two 8-node tiles, this half's two 8-position matrices of q'
            uint32_t b[4];
            const uint32_t at = q_hi + n * 8 * SS_ROW + jj * 64 + h * 32;
            ldmatrix_x4(at, b);
            mma_16816(acc[n], hi, b[0], b[1]);
            mma_16816(acc[n + 1], hi, b[2], b[3]);
            mma_16816(acc[n], lo, b[0], b[1]);
            mma_16816(acc[n + 1], lo, b[2], b[3]);
            ldmatrix_x4(at + N * SS_ROW, b);
            mma_16816(acc[n], hi, b[0], b[1]);
            mma_16816(acc[n + 1], hi, b[2], b[3]);
        }
    }
}

// The passes of the state through the registers (x: chunks 0, 1): with a path (of at most 8 TILES steps) the products of the old state
// with its keys and then, chunk by chunk, the update, the write and the product with q' (nodes: there are any); without
// (TILES = 0) that product alone.
template <int N, int TILES>
__device__ __forceinline__ void state_passes(float *S, float (&x)[2][4][4], int len, uint32_t operand, const PathTile &path, int row, int lane,
                                             float A_L, uint32_t q_hi, float (&acc)[N / 8][4], bool nodes)
{
    PathUpdate<TILES ? TILES : 1> up;
    if constexpr (TILES != 0) {
        PathProducts<TILES> a;
#pragma unroll
        for (int i = 0; i < TILES; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) a.z[i][e] = a.rest[i][e] = 0.f;
#pragma unroll 1
        for (int j = 0; j < 4; j += 2)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                path_products_chunk(x[i], j + i, operand, a);
                load_chunk(S, (j + i + 2) & 3, x[i]);   // (the first two again, for the update)
            }
        path_solve(a, len, path, row, lane, up);
    }
#pragma unroll 1
    for (int j = 0; j < 4; j += 2)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if constexpr (TILES != 0) {
                path_update_chunk(x[i], j + i, operand, A_L, up);
                store_chunk(S, j + i, x[i]);
            }
            if (nodes) output_chunk<N>(x[i], j + i, q_hi, acc);
            if (j == 0) load_chunk(S, i + 2, x[i]);
        }
}

// The same of one of PARTS CTAs: PARTS warps share 16 rows, each with 4 / PARTS chunks of them (jj and on) that stay in its registers
// (x).  Of the products with the old state and of those with q' a warp has a share; the first are summed here, by every warp for
// itself, acc is left as it is.  share: this lane's place in products[], sum: its place in that of the first warp on the same rows.
template <int N, int TILES, int PARTS>
__device__ __forceinline__ void state_share(float *S, float (&x)[4 / PARTS][4][4], int jj, int len, uint32_t operand, const PathTile &path, int row,
                                            int lane, float *share, const float *sum, float A_L, uint32_t q_hi, float (&acc)[N / 8][4], bool nodes)
{
    PathUpdate<TILES ? TILES : 1> up;
    if constexpr (TILES != 0) {
        PathProducts<TILES> a;
#pragma unroll
        for (int i = 0; i < TILES; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) a.z[i][e] = a.rest[i][e] = 0.f;
#pragma unroll
        for (int j = 0; j < 4 / PARTS; ++j) path_products_chunk(x[j], jj + j, operand, a);
#pragma unroll
        for (int i = 0; i < TILES; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) share[(i * 4 + e) * 32] = a.z[i][e] + a.rest[i][e];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < TILES; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                a.z[i][e] = sum_shares<PARTS>(sum + (i * 4 + e) * 32, 8 * 32);
                a.rest[i][e] = 0.f;
            }
        path_solve(a, len, path, row, lane, up);
    }
#pragma unroll
    for (int j = 0; j < 4 / PARTS; ++j) {
        if constexpr (TILES != 0) {
            path_update_chunk(x[j], jj + j, operand, A_L, up);
            store_chunk(S, jj + j, x[j]);
        }
        if (nodes) output_chunk<N>(x[j], jj + j, q_hi, acc);
    }
}

// CTAS: per SM.  PLANNED: the trees come from a plan.
template <int N, typename TOut, bool COMMIT, int CTAS, bool PLANNED, int PARTS>
__global__ void __launch_bounds__(SS_THREADS, CTAS) verify_step_small_kernel(const StepSmallParams p)
{
    extern __shared__ __align__(16) uint8_t ss_smem[];
    using Smem = StepSmallSmem<N, PARTS>;
    Smem &sm = *reinterpret_cast<Smem *>(ss_smem);
    const CommitParams &c = p.c;
    const int unit = blockIdx.x / PARTS, part = blockIdx.x % PARTS, b = unit / c.h_v, h = unit - b * c.h_v, hk = h / (c.h_v / c.h_qk);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < 4 / PARTS)   // L2 may be asked for the tile meanwhile (a prefetch consumes nothing)
        prefetch_l2_bulk(c.S + (size_t)unit * SS_D * SS_D + (size_t)(part * (4 / PARTS) + tid) * 4096, 16384);
    if ((!COMMIT || CTAS <= 2) && p.rows_early && tid >= SS_THREADS - N && tid - (SS_THREADS - N) < p.max_tree_nodes) {
        // ... and for the rows; node_offsets[] only steers here: clamped to the tensors, and by way
        // of L2, so that nothing stays in L1 for the read that counts.  Over buffers that L2 does not hold (us, in a graph, 64-node kernels
        // / without / with): verification of 1 / 4 / 6 trees of 32 nodes 6.6 7.3 9.6 / 6.8 7.9 10.1 / 6.1 6.8 9.3, of 16 nodes 6.4 7.0 8.4 /
        // 5.3 6.2 7.8 / 4.7 5.2 6.5; planned layer of one tree of 32 nodes, commit included, 12.8 / 13.5 / 13.2.  (A commit at three or four
        // CTAs per SM: 12 trees of 16 nodes, path of 8, 18.1 without, 18.5 with.)
        const int row = (p.t_pad ? b * p.t_pad : __ldcg(p.node_offsets + b)) + tid - (SS_THREADS - N);
        if (row >= 0 && row < p.total_nodes) {
            prefetch_l2_bulk(p.k + ((size_t)row * c.h_qk + hk) * SS_D, 256);
            prefetch_l2_bulk(p.q + ((size_t)row * c.h_qk + hk) * SS_D, 256);
            prefetch_l2_bulk(p.v + ((size_t)row * c.h_v + h) * SS_D, 256);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.g + (size_t)row * c.h_v + h));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.beta + (size_t)row * c.h_v + h));
        }
    }
    wait_for_previous_kernel();

    // the new tree; one with inconsistent node_offsets[] is reported and runs as a tree of no nodes
    const int tree = p.t_pad ? b % p.n_trees : b;
    int base, T;
    bool off_ok;
    if (PLANNED) {
        // a tree of at most 64 nodes has one record, anywhere in the list; a rejected or empty one has none
        // (48 layers, commit and planned verification each, a tree of 8 / 16 / 32 nodes: 609 / 625 / 646 us with the kernel of grouped
        // trees, 489 / 497 / 589 so).  The trees' CTAs claimed their places about in their order, so that the search begins at the tree's own
        // place and goes on to both sides of it, 32 records at a time (1024 trees of 16 nodes, one layer: 545 us from the head of the list on, 471 so;
        // units in the order of the list, which need no search, find the tile that they had L2 fetch in another unit: 588)
        base = b * p.t_pad;
        T = 0;
        const int n_rec = p.plan.unit_count[0];
        if (p.plan.unit_count[1] != p.plan.magic || n_rec < 0 || n_rec > p.plan.capacity) {   // not a plan of this shape
            if (tid == 0) report_status(c.status_dev, GDN_ERR_WORKSPACE);
            return;
        }
        const int n_win = (n_rec + 31) >> 5, w0 = min(tree >> 5, n_win - 1);
        for (int i = 0; i < 2 * n_win; ++i) {   // windows w0, w0 + 1, w0 - 1, w0 + 2, ...
            const int w = w0 + (i & 1 ? (i + 1) >> 1 : -(i >> 1)), r = w * 32 + lane;
            if (w < 0 || w >= n_win) continue;
            const uint4 rec = r < n_rec ? p.plan.unit_list[r] : make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
            const uint32_t found = __ballot_sync(0xffffffffu, rec.x == (uint32_t)tree);
            if (found) {
                T = (int)((__shfl_sync(0xffffffffu, rec.z, __ffs(found) - 1) >> 16) & 0xFFu);
                break;
            }
        }
        off_ok = T <= p.t_pad;
    } else if (p.t_pad) {
        base = b * p.t_pad;
        T = p.n_nodes[tree];
        off_ok = T >= 0 && T <= p.t_pad;
    } else {
        base = p.node_offsets[b];
        const int end = p.node_offsets[b + 1];
        T = end - base;
        off_ok = base >= 0 && T >= 0 && T <= p.max_tree_nodes && end <= p.total_nodes;
        if (b == 0) off_ok = off_ok && base == 0;
        if (b == p.n_seq - 1) off_ok = off_ok && end == p.total_nodes;
    }
    if (!off_ok || T > N) {
        if (tid == 0) report_status(c.status_dev, GDN_ERR_TREE);
        T = 0;
    }
    int pp0 = 0, len = 0;
    if constexpr (COMMIT) {
        const int ptree = c.t_pad ? b % c.n_trees : b;
        pp0 = c.t_pad ? ptree * c.path_stride : c.path_offsets[b];
        len = c.t_pad ? c.path_len[ptree] : c.path_offsets[b + 1] - pp0;
    }
    if (len == 0 && T == 0) return;

    // the state first: its latency covers what is fetched and worked out below
    // a warp's 16 rows and its chunks (PARTS == 1: all four, two at a time)
    constexpr int GROUPS = 8 / PARTS, COMPS = SS_D / PARTS, CHUNKS = PARTS == 1 ? 2 : 4 / PARTS;
    const int rg = PARTS == 1 ? warp : warp % GROUPS, jj = PARTS == 1 ? 0 : warp / GROUPS * CHUNKS;
    const int comp0 = part * COMPS + rg * 16, row = comp0 + (lane >> 2);
    float *S = c.S + (size_t)unit * SS_D * SS_D + (size_t)row * SS_D + (lane & 3) * 8;
    float x[CHUNKS][4][4];
#pragma unroll
    for (int j = 0; j < CHUNKS; ++j) load_chunk(S, jj + j, x[j]);

    const uint32_t rows = smem_u32(sm.rows[0]), pk = smem_u32(sm.pk);
    if (T > 0) {
#pragma unroll
        for (int e = 0; e < 3 * N * 16 / SS_THREADS; ++e) {
            const int idx = tid + e * SS_THREADS, what = idx / (N * 16), i = (idx >> 4) % N, c16 = idx & 15;
            if (PARTS > 1 && what == 2 && c16 / (16 / PARTS) != part) continue;   // (of v its own components only)
            const bool on = i < T;
            const size_t n = (size_t)(base + (on ? i : 0));
            const __nv_bfloat16 *src = what == 2 ? p.v + (n * c.h_v + h) * SS_D : (what ? p.q : p.k) + (n * c.h_qk + hk) * SS_D;
            cp_async_16(rows + what * N * SS_ROW + i * SS_ROW + c16 * 16, src + c16 * 8, on);
        }
    }
    float gt = 0.f, be = 0.f;   // of path step `lane` (warp 0)
    if constexpr (COMMIT) {
        if (len != 0) {
            const int ptree = c.t_pad ? b % c.n_trees : b;
            const int pb = c.t_pad ? b * c.t_pad : c.node_offsets[b];
            const int pT = c.t_pad ? min(c.n_nodes[ptree], c.t_pad) : c.node_offsets[b + 1] - pb;
            const bool shape_ok = len > 0 && len <= CF_MD && len <= c.max_depth && pT > 0 && pp0 >= 0;
            if (shape_ok) path_rows_fetch(c, pp0, len, pb, pT, h, hk, pk, sm.pv, tid);
            if (warp == 0) {
                const int n = path_check_and_scalars(c, pp0, shape_ok ? len : 0, pb, pT, c.t_pad ? ptree * c.t_pad : pb, h, lane, gt, be,
                                                     sm.scal, sm.decay);
                if (lane == 0) sm.len = n;
            }
        }
    }
    if (warp == 1 && T > 0) {
        // lane i: node i.  Ancestor masks by pointer doubling (five rounds cover 32 nodes).
        const bool mine = lane < T;
        const size_t n = (size_t)(base + lane) * c.h_v + h;
        const uint32_t g16 = mine ? reinterpret_cast<const unsigned short *>(p.g)[n] : 0u;
        const uint32_t b16 = mine ? reinterpret_cast<const unsigned short *>(p.beta)[n] : 0u;
        uint32_t m = 1u << lane;
        bool bad = false;
        if constexpr (PLANNED) {
            if (mine) {   // the root path as bytes, 0xFF behind its end
                const uint4 path = *reinterpret_cast<const uint4 *>(p.plan.anc8 + ((size_t)tree * p.t_pad + lane) * 16);
                const uint32_t w[4] = {path.x, path.y, path.z, path.w};
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const uint32_t id = (w[e >> 2] >> (8 * (e & 3))) & 0xFFu;
                    if (id != 0xFFu) m |= 1u << (id & 31u);
                }
            }
        } else {
            int up = mine ? p.parent[(p.t_pad ? tree * p.t_pad : base) + lane] : -1;
            int err = up < -1 || (mine && up >= lane) ? GDN_ERR_TREE : 0;
            if (err) up = -1;
#pragma unroll
            for (int r = 1; r < N; r *= 2) {
                const uint32_t above = __shfl_sync(0xffffffffu, m, max(up, 0));
                const int next = __shfl_sync(0xffffffffu, up, max(up, 0));
                if (up >= 0) {
                    m |= above;
                    up = next;
                }
            }
            if (mine && !err && __popc(m) > c.max_depth) err = GDN_ERR_DEPTH;
            if (err) report_status(c.status_dev, err);
            bad = __any_sync(0xffffffffu, err != 0);
        }
        if (lane < N) {
            sm.mask[lane] = mine ? m : 0u;
            sm.g[lane] = gate_log_decay(g16, c.raw_gates != 0);
            sm.beta[lane] = gate_beta(b16, c.raw_gates != 0);
        }
        if (lane == 0) sm.bad = bad;
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (T > 0 && sm.bad) T = 0;           // a rejected tree runs as one of no nodes
    if (COMMIT && len != 0) len = sm.len;   // (a rejected path: the state stays as it was)
    if (len == 0 && T == 0) return;

    const uint32_t qp = smem_u32(sm.qp[0]), wz = smem_u32(sm.wz[0]);
    float *const gram = reinterpret_cast<float *>(sm.qp[0]);
    const int l4 = lane & 3, g8 = lane >> 2;
    if (COMMIT && warp == 0 && len > 1) path_coupling(pk, len, gt, be, sm.couple, lane);
    // (1) Gram = [k;q].k^T, a warp per 16 x 16 block (16 x N / 2 blocks right of the diagonal belong to no ancestor)
    {
        constexpr int BLOCKS = N / 16;
        const int job = warp - 1, mt = job / BLOCKS, nt = job % BLOCKS;   // rows 16 mt .. of [k;q], columns 16 nt ..
        for (int j = job; T > 0 && j >= 0 && j < 2 * BLOCKS * BLOCKS; j += 7) {
            const int m_ = j == job ? mt : j / BLOCKS, n_ = j == job ? nt : j % BLOCKS;
            if (n_ > m_ % BLOCKS) continue;
            float d[2][4] = {};
            const uint32_t a_at = rows + (m_ * 16 + (lane & 15)) * SS_ROW + (lane >> 4) * 16;
            const uint32_t b_at = rows + (n_ * 16 + (lane & 7) + 8 * (lane >> 4)) * SS_ROW + ((lane >> 3) & 1) * 16;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                uint32_t a[4], bb[4];
                ldmatrix_x4(a_at + ks * 32, a);
                ldmatrix_x4(b_at + ks * 32, bb);
                mma_16816(d[0], a, bb[0], bb[1]);
                mma_16816(d[1], a, bb[2], bb[3]);
            }
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    *reinterpret_cast<float2 *>(gram + (m_ * 16 + g8 + 8 * r) * Smem::G_ROW + n_ * 16 + n * 8 + 2 * l4) =
                        make_float2(d[n][2 * r], d[n][2 * r + 1]);
        }
    }
    __syncthreads();
    // (2) w by back-substitution over the root path in node order (an ancestor has a smaller index): N lanes per node, lane j
    // owning ancestor j; once w_l is final, w_l kappa(l, j) is subtracted from every ancestor j of node l.  Decays are sums of g over just
    // the nodes they span.
    if (T > 0) {
        constexpr int NE = N * N / SS_THREADS;   // nodes per lane group
        const int j = lane & (N - 1);
        const float bj = sm.beta[j], gj = sm.g[j];
        float z[NE];
        uint32_t m[NE], any = 0;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int i = N == 16 ? warp * 2 + (lane >> 4) : warp * 4 + e;
            m[e] = sm.mask[i];
            z[e] = (m[e] >> j) & 1 ? gram[(N + i) * Smem::G_ROW + j] : 0.f;
            any |= m[e];
        }
        any = __reduce_or_sync(0xffffffffu, any);
        for (any &= ~1u; any; ) {
            const int l = 31 - __clz(any);
            any ^= 1u << l;
            const float kap = gram[l * Smem::G_ROW + j];
#pragma unroll
            for (int e = 0; e < NE; ++e) {
                const float wl = __shfl_sync(0xffffffffu, z[e] * bj, (lane & ~(N - 1)) | l);
                if (j < l && (m[e] >> l) & (m[e] >> j) & 1) z[e] = fmaf(-wl, kap, z[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int i = N == 16 ? warp * 2 + (lane >> 4) : warp * 4 + e;
            const bool on = (m[e] >> j) & 1;
            float sum = on ? gj : 0.f;   // of g over the path nodes from j on down
#pragma unroll
            for (int off = 1; off < N; off *= 2) {
                const float below = __shfl_down_sync(0xffffffffu, sum, off, N);
                if (j + off < N) sum += below;
            }
            float behind = __shfl_down_sync(0xffffffffu, sum, 1, N);
            if (j == N - 1) behind = 0.f;
            const float sa = p.scale * __expf(__shfl_sync(0xffffffffu, sum, 0, N));
            const float w = on ? bj * z[e] : 0.f;
            uint32_t hi, lo;
            split_pack_bf16(on ? -sa * w : 0.f, on ? p.scale * __expf(behind) * w : 0.f, hi, lo);
            uint16_t *dst = reinterpret_cast<uint16_t *>(sm.wz[0] + i * Smem::W_ROW + 2 * j);
            constexpr int PLANE = N * Smem::W_ROW / 2;
            dst[0] = (uint16_t)hi;
            dst[PLANE] = (uint16_t)lo;
            dst[2 * PLANE] = (uint16_t)(hi >> 16);
            dst[3 * PLANE] = (uint16_t)(lo >> 16);
            if (j == 0) sm.sa[i] = sa;
        }
    }
    __syncthreads();
    // (3) q' = sa q - sa w.K: a warp per 16 key positions
    if (T > 0) {
        const uint32_t w_at = wz + (lane & 15) * Smem::W_ROW + (lane >> 4) * 16;
        const uint32_t k_at = rows + ((lane & 7) + 8 * ((lane >> 3) & 1)) * SS_ROW + warp * 32 + (lane >> 4) * 16;
#pragma unroll
        for (int mt = 0; mt < N / 16; ++mt) {
            float d[2][4] = {};
#pragma unroll
            for (int ks = 0; ks <= mt; ++ks) {   // (ancestors have smaller indices)
                uint32_t kb[4], a[4];
                ldmatrix_x4_trans(k_at + ks * 16 * SS_ROW, kb);
#pragma unroll
                for (int part = 0; part < 2; ++part) {   // hi, lo
                    ldmatrix_x4(w_at + part * N * Smem::W_ROW + mt * 16 * Smem::W_ROW + ks * 32, a);
                    mma_16816(d[0], a, kb[0], kb[1]);
                    mma_16816(d[1], a, kb[2], kb[3]);
                }
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int i = mt * 16 + g8 + 8 * r;
                const float sa = sm.sa[i];
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    const int word = warp * 8 + n * 4 + l4;   // of the row: key positions 2 word, 2 word + 1
                    const uint32_t qw = *reinterpret_cast<const uint32_t *>(sm.rows[1] + i * SS_ROW + word * 4);
                    uint32_t hi, lo;
                    split_pack_bf16(fmaf(sa, __uint_as_float(qw << 16), d[n][2 * r]), fmaf(sa, __uint_as_float(qw & 0xFFFF0000u), d[n][2 * r + 1]),
                                    hi, lo);
                    uint8_t *dst = sm.qp[0] + i * SS_ROW + path_row_word(word);
                    *reinterpret_cast<uint32_t *>(dst) = hi;
                    *reinterpret_cast<uint32_t *>(dst + N * SS_ROW) = lo;
                }
            }
        }
    }
    __syncthreads();
    // (4) the state: advanced along the path and written, and its product with q'
    // of q': lanes 0..15 the two 8-position matrices of nodes 0..7, lanes 16..31 those of nodes 8..15
    const uint32_t q_hi = qp + (uint32_t)((lane & 7) + 8 * (lane >> 4)) * SS_ROW + (uint32_t)((lane >> 3) & 1) * 16;
    float acc[N / 8][4];
#pragma unroll
    for (int n = 0; n < N / 8; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
    const PathTile path{sm.pv, sm.scal, sm.couple};
    if constexpr (PARTS > 1) {
        const uint32_t operand = path_operand(pk, lane);
        float *const share = sm.products + warp * 256 + lane;
        const float *const sum = sm.products + rg * 256 + lane;
        if (len > 8) state_share<N, 2, PARTS>(S, x, jj, len, operand, path, row, lane, share, sum, sm.decay, q_hi, acc, T > 0);
        else if (len > 0) state_share<N, 1, PARTS>(S, x, jj, len, operand, path, row, lane, share, sum, sm.decay, q_hi, acc, T > 0);
        else state_share<N, 0, PARTS>(S, x, jj, 0, 0, path, row, lane, share, sum, 1.f, q_hi, acc, true);
    } else if (COMMIT && len > 8) state_passes<N, 2>(S, x, len, path_operand(pk, lane), path, row, lane, sm.decay, q_hi, acc, T > 0);
    else if (COMMIT && len > 0) state_passes<N, 1>(S, x, len, path_operand(pk, lane), path, row, lane, sm.decay, q_hi, acc, T > 0);
    else state_passes<N, 0>(S, x, 0, 0, path, row, lane, 1.f, q_hi, acc, true);
    // (5) the v rows' part of the outputs, then a warp's sixteen components of every node through its own piece of shared memory, then 16-byte stores
    if (T > 0) {
        const uint32_t v_at = rows + 2 * N * SS_ROW + ((lane & 7) + 8 * (lane >> 4)) * SS_ROW + comp0 * 2 + ((lane >> 3) & 1) * 16;
        const uint32_t z_at = wz + 2 * N * Smem::W_ROW + ((lane & 7) + 8 * (lane >> 4)) * Smem::W_ROW + ((lane >> 3) & 1) * 16;
#pragma unroll
        for (int ks = 0; ks < N / 16; ++ks) {
            if (PARTS > 1 && warp / GROUPS != ks) continue;
            uint32_t a[4], zb[4];
            ldmatrix_x4_trans(v_at + ks * 16 * SS_ROW, a);
#pragma unroll
            for (int n = 2 * ks; n < N / 8; n += 2)
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    ldmatrix_x4(z_at + part * N * Smem::W_ROW + n * 8 * Smem::W_ROW + ks * 32, zb);
                    mma_16816(acc[n], a, zb[0], zb[1]);
                    mma_16816(acc[n + 1], a, zb[2], zb[3]);
                }
        }
        if constexpr (PARTS > 1) {   // the warps' shares, summed a component of a node per thread
            float *const shares = reinterpret_cast<float *>(sm.rows[0]);
            constexpr int SHARE = N / 2 * 32;   // of a warp
#pragma unroll
            for (int n = 0; n < N / 8; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) shares[warp * SHARE + (n * 4 + e) * 32 + lane] = acc[n][e];
            __syncthreads();
            TOut *const o = static_cast<TOut *>(p.o) + ((size_t)base * c.h_v + h) * SS_D + part * COMPS;
            for (int idx = tid; idx < T * COMPS; idx += SS_THREADS) {
                const int i = idx / COMPS, cc = idx % COMPS;   // held by lane 4 (cc mod 8) + (i mod 8) / 2 of the warps of row group cc / 16
                const float *s = shares + cc / 16 * SHARE + (i / 8 * 4 + 2 * (cc / 8 % 2) + i % 2) * 32 + cc % 8 * 4 + i % 8 / 2;
                store_from_float(o + (size_t)i * c.h_v * SS_D + cc, sum_shares<PARTS>(s, SHARE));
            }
        } else {
            uint8_t *const stage = sm.rows[0] + warp * (N * 64);
            constexpr int ROW_BYTES = 16 * (int)sizeof(TOut), PIECES = ROW_BYTES / 16;
            if constexpr (sizeof(TOut) == 2) {
                const uint32_t at = smem_u32(stage) + ((lane & 7) + 8 * (lane >> 4)) * ROW_BYTES + ((lane >> 3) & 1) * 16;
#pragma unroll
                for (int n = 0; n < N / 8; n += 2)
                    stmatrix_x4_trans(at + n * 8 * ROW_BYTES, pack_bf16(acc[n][0], acc[n][1]), pack_bf16(acc[n][2], acc[n][3]),
                                      pack_bf16(acc[n + 1][0], acc[n + 1][1]), pack_bf16(acc[n + 1][2], acc[n + 1][3]));
            } else {
                float *const st = reinterpret_cast<float *>(stage);   // component c of node i at place c ^ 8 (i / 2 mod 2)
#pragma unroll
                for (int n = 0; n < N / 8; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int i = n * 8 + 2 * l4 + (e & 1);
                        st[i * 16 + ((g8 + 8 * (e >> 1)) ^ (8 * (l4 & 1)))] = acc[n][e];
                    }
            }
            __syncwarp();
            uint8_t *const o = static_cast<uint8_t *>(p.o) + (((size_t)base * c.h_v + h) * SS_D + warp * 16) * sizeof(TOut);
#pragma unroll
            for (int e = 0; e < N * PIECES / 32; ++e) {
                const int i = (e * 32 + lane) / PIECES, piece = (e * 32 + lane) % PIECES;
                const int at = sizeof(TOut) == 2 ? piece : piece ^ (2 * ((i >> 1) & 1));
                if (i < T)
                    *reinterpret_cast<uint4 *>(o + (size_t)i * c.h_v * SS_D * sizeof(TOut) + piece * 16) =
                        *reinterpret_cast<const uint4 *>(stage + i * ROW_BYTES + at * 16);
            }
        }
    }
}

template <int N, typename TOut, bool COMMIT, int CTAS, bool PLANNED = false, int PARTS = 1>
cudaError_t launch_kernel(StepSmallParams p, cudaStream_t stream)
{
    static PerContext seen;
    int sms = 0;
    const auto kernel = verify_step_small_kernel<N, TOut, COMMIT, CTAS, PLANNED, PARTS>;
    cudaError_t e = device_sms(seen, reinterpret_cast<const void *>(kernel), sizeof(StepSmallSmem<N, PARTS>), &sms);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(p.n_seq * p.c.h_v * PARTS));
    // (up to three quarters of what is resident at once: 9 trees of 32 nodes take 10.7 us without and 10.2 with, but 9.4 and 9.6 out of L2)
    p.rows_early = cfg.gridDim.x <= (unsigned)(CTAS * sms * 3 / 4);
    cfg.blockDim = dim3(SS_THREADS);
    cfg.dynamicSmemBytes = sizeof(StepSmallSmem<N, PARTS>);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <typename TOut> cudaError_t launch_typed(const StepSmallParams &p, bool with_commit, cudaStream_t stream)
{
    if (p.plan.unit_list)
        return p.max_tree_nodes > 16 ? launch_kernel<32, TOut, false, 2, true>(p, stream) : launch_kernel<16, TOut, false, 4, true>(p, stream);
    if (!with_commit)
        return p.max_tree_nodes > 16 ? launch_kernel<32, TOut, false, 2>(p, stream) : launch_kernel<16, TOut, false, 4>(p, stream);
    static PerContext seen;
    int sms = 0;
    const cudaError_t e = device_sms(seen, nullptr, 0, &sms);
    if (e != cudaSuccess) return e;
    const long long units = (long long)p.n_seq * p.c.h_v;
    const int parts = commit_parts(units, sms);
    if (p.max_tree_nodes > 16)
        return parts == 4   ? launch_kernel<32, TOut, true, 2, false, 4>(p, stream)
               : parts == 2 ? launch_kernel<32, TOut, true, 2, false, 2>(p, stream)
                            : launch_kernel<32, TOut, true, 2>(p, stream);
    if (parts == 4) return launch_kernel<16, TOut, true, 2, false, 4>(p, stream);
    if (parts == 2) return launch_kernel<16, TOut, true, 2, false, 2>(p, stream);
    return commit_at_four(p.max_tree_nodes, units, sms) ? launch_kernel<16, TOut, true, 4>(p, stream)
                                                        : launch_kernel<16, TOut, true, 3>(p, stream);
}

}  // namespace

// Trees of at most 16 nodes, always; of up to 32 only while all units are resident at once.  Measured (us; the kernels of 64-node
// tiles / this one), trees of 32 nodes, 32 heads, path of 7 and verification alone: 1 tree 11.1 / 8.5 and 8.4 / 7.9, 4 trees 13.7 / 10.8
// and 8.4 / 7.8, 8 trees 18.8 / 14.9 and 10.6 / 9.8, 9 trees 19.6 / 15.5 and 11.0 / 10.0; beyond that the 64-node tiles share the
// coefficients of a key head's value heads: 12 trees 32.2 / 26.3 and 15.5 / 15.7, 16 trees 32.3 / 31.4 and 16.3 / 18.8, 48 trees 74.7 / 78.3
// and 35.6 / 47.5.
bool step_small_supported(const gdn_shape_t &s)
{
    if (!verify_sm100_supported(s) || s.max_tree_nodes > SS_MAX_NODES) return false;
    if (s.max_tree_nodes <= 16) return true;
    static PerContext seen;
    int sms = 0;
    return device_sms(seen, nullptr, 0, &sms) == cudaSuccess && (long long)s.n_seq * s.h_v <= 2LL * sms;
}

cudaError_t launch_step_small(const gdn_shape_t &s, const CommitParams &prev, bool with_commit, const void *q, const void *k, const void *v,
                              const void *g, const void *beta, const int32_t *parent, const int32_t *node_offsets, int n_trees,
                              const int32_t *n_nodes, void *o, cudaStream_t stream, const SmallTreePlan &plan)
{
    if (s.n_seq == 0 || s.total_nodes == 0) return cudaSuccess;
    StepSmallParams p{};
    p.c = prev;
    p.n_seq = s.n_seq; p.total_nodes = s.total_nodes; p.max_tree_nodes = s.max_tree_nodes; p.scale = s.scale;
    p.q = static_cast<const __nv_bfloat16 *>(q); p.k = static_cast<const __nv_bfloat16 *>(k);
    p.v = static_cast<const __nv_bfloat16 *>(v); p.g = static_cast<const __nv_bfloat16 *>(g);
    p.beta = static_cast<const __nv_bfloat16 *>(beta);
    p.parent = parent; p.node_offsets = node_offsets; p.o = o;
    p.t_pad = node_offsets ? 0 : s.max_tree_nodes; p.n_trees = n_trees; p.n_nodes = n_nodes;
    p.plan = plan;
    return s.out_dtype == GDN_BF16 ? launch_typed<__nv_bfloat16>(p, with_commit, stream) : launch_typed<float>(p, with_commit, stream);
}

}  // namespace gdn
