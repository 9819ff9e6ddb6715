// Commit kernel: replay Eq. 7 along the accepted root path and write the state in place
// (Section 3.4: the commit is delayed until the accepted branch is known and is "a short
// recurrence"; Section 3.4.2: it is the only state write of a decode step).
//
// With S' = alpha S (decay first), Eq. 7 reads S <- S' - beta k (k^T S') + beta k v^T, i.e. per
// value component c (one contiguous row of the [d_v][d_k] tile):
//     s_c <- alpha s_c + k * beta (v_c - alpha (k . s_c)).
// General form: one CTA per (tree, value head); eight lanes hold four rows, an eighth of the key dimension each (16-byte
// pieces, 128 contiguous bytes per row and load), and k . s_c of the four is reduced over them with shuffles.  The path
// nodes' k and v rows are fetched once into shared memory; the state is read once and written once.  The state loads are
// issued before anything else so that the path checks and the row staging run under their latency.  With four lanes per
// row and one row per thread each k piece served one row only and shared memory bounded the steps: 8 trees, 32 heads of
// 128 x 128, path of 5, fp32: 14.3 -> 8.6 us.
#include "gdn_path.cuh"
#include "gdn_plan.cuh"

namespace gdn {

namespace {

constexpr int CM_THREADS = 256;
constexpr int CM_SPLIT = 8;
constexpr int CM_ROWS = 4;
constexpr int CM_DK = GDN_MAX_HEAD_DIM;
static_assert(CM_THREADS / CM_SPLIT * CM_ROWS == GDN_MAX_HEAD_DIM, "a row of the state for every value component");

// max_shared: on SMs set up for the most shared memory, so that a verification launched behind can move in beside the grid.
template <typename... KernelArgs, typename... Args>
cudaError_t launch_overlapped(void (*kernel)(KernelArgs...), int grid, int threads, size_t smem, bool max_shared, cudaStream_t stream,
                              Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    cfg.attrs = attr;
    cfg.numAttrs = max_shared ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

constexpr size_t commit_generic_smem(int max_depth) { return sizeof(float) * (2 * (size_t)CM_DK + 2) * max_depth; }

template <typename TIn>
__global__ void __launch_bounds__(CM_THREADS, 2) commit_generic_kernel(const CommitParams p)
{
    extern __shared__ __align__(16) float cm_smem[];
    float (*ks)[CM_DK] = reinterpret_cast<float (*)[CM_DK]>(cm_smem);   // [L][CM_DK]
    float (*vs)[CM_DK] = ks + p.max_depth;                              // [L][CM_DK]
    float *alpha_s = cm_smem + 2 * (size_t)p.max_depth * CM_DK;         // [L]
    float *beta_s = alpha_s + p.max_depth;                              // [L]

    wait_for_previous_kernel();
    const int b = blockIdx.x / p.h_v, h = blockIdx.x % p.h_v;
    const int p0 = p.path_offsets[b];
    const int L = p.path_offsets[b + 1] - p0;
    if (L == 0) return;   // nothing accepted from this tree: state untouched
    const int base = p.node_offsets[b];
    const int T = p.node_offsets[b + 1] - base;
    const int tid = threadIdx.x, lane = tid & 31;
    const int d_k = p.d_k, d_v = p.d_v;
    const bool shape_ok = L > 0 && L <= p.max_depth && T > 0 && p0 >= 0;

    const int hk = h / (p.h_v / p.h_qk);
    const int s = tid % CM_SPLIT, c = tid / CM_SPLIT * CM_ROWS;
    const TIn *k = static_cast<const TIn *>(p.k), *v = static_cast<const TIn *>(p.v);
    const TIn *g = static_cast<const TIn *>(p.g), *beta = static_cast<const TIn *>(p.beta);

    // The state goes first: its latency covers the path checks and the row staging below.
    float *rows = p.S + ((size_t)(b * p.h_v + h) * d_v + c) * d_k;
    float2 x[CM_ROWS][8];   // row c + r, key positions 32 j + 4 s + e (zero beyond d_k / d_v)
#pragma unroll
    for (int r = 0; r < CM_ROWS; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int at = 32 * j + 4 * s;
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
            if (shape_ok && c + r < d_v && at < d_k) y = *reinterpret_cast<const float4 *>(rows + (size_t)r * d_k + at);
            x[r][2 * j] = make_float2(y.x, y.y);
            x[r][2 * j + 1] = make_float2(y.z, y.w);
        }

    // The path's rows (fp32, zero padded to CM_DK) and per-step scalars: every thread reads the path entry whose row piece
    // it fetches, an entry outside the tree is skipped here and reported by the check.
    bool bad = !shape_ok;
    if (shape_ok) {
#pragma unroll 2
        for (int idx = tid; idx < L * CM_DK; idx += CM_THREADS) {
            const int t = idx / CM_DK, r = idx % CM_DK, nt = p.path[p0 + t];
            if (nt < 0 || nt >= T) continue;
            const size_t n = (size_t)base + nt;
            ks[t][r] = r < d_k ? load_as_float(k + (n * p.h_qk + hk) * d_k + r) : 0.f;
            vs[t][r] = r < d_v ? load_as_float(v + (n * p.h_v + h) * d_v + r) : 0.f;
        }
        if (tid < L) {
            // thread t: entry t must be the child of entry t - 1 (entry 0: a root)
            const int nt = p.path[p0 + tid], up = tid ? p.path[p0 + tid - 1] : -1;
            if (nt < 0 || nt >= T) bad = true;
            else {
                // (without parent[] only the topological order can be checked)
                bad = p.parent ? p.parent[base + nt] != up : tid && nt <= up;
                alpha_s[tid] = expf(load_as_float(g + ((size_t)base + nt) * p.h_v + h));
                beta_s[tid] = load_as_float(beta + ((size_t)base + nt) * p.h_v + h);
            }
        }
    }
    if (__syncthreads_or(bad)) {
        if (tid == 0) report_status(p.status_dev, GDN_ERR_PATH);
        return;
    }

    const bool b2 = (s & 4) != 0, b1 = (s & 2) != 0;
    const int mine = (b2 ? 2 : 0) + (b1 ? 1 : 0);   // the row whose k.s this lane ends up with
#pragma unroll 1
    for (int t = 0; t < L; ++t) {
        float2 kf[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 kx = *reinterpret_cast<const float4 *>(&ks[t][32 * j + 4 * s]);
            kf[2 * j] = make_float2(kx.x, kx.y);
            kf[2 * j + 1] = make_float2(kx.z, kx.w);
        }
        float dot[CM_ROWS];
#pragma unroll
        for (int r = 0; r < CM_ROWS; ++r) {
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 8; ++j) acc = __ffma2_rn(kf[j], x[r][j], acc);
            dot[r] = acc.x + acc.y;
        }
        // the four rows folded into one another over the eight lanes; lanes 0, 2, 4, 6 of them end up with rows 0, 1, 2, 3
        const float e0 = (b2 ? dot[2] : dot[0]) + __shfl_xor_sync(0xffffffffu, b2 ? dot[0] : dot[2], 4);
        const float e1 = (b2 ? dot[3] : dot[1]) + __shfl_xor_sync(0xffffffffu, b2 ? dot[1] : dot[3], 4);
        float d = (b1 ? e1 : e0) + __shfl_xor_sync(0xffffffffu, b1 ? e0 : e1, 2);
        d += __shfl_xor_sync(0xffffffffu, d, 1);
        const float alpha = alpha_s[t];
        const float w_mine = beta_s[t] * (vs[t][c + mine] - alpha * d);
        const float2 a2 = make_float2(alpha, alpha);
#pragma unroll
        for (int r = 0; r < CM_ROWS; ++r) {
            const float w = __shfl_sync(0xffffffffu, w_mine, (lane & ~7) | (2 * r));
            const float2 w2 = make_float2(w, w);
#pragma unroll
            for (int j = 0; j < 8; ++j) x[r][j] = __ffma2_rn(kf[j], w2, __fmul2_rn(a2, x[r][j]));
        }
    }

#pragma unroll
    for (int r = 0; r < CM_ROWS; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int at = 32 * j + 4 * s;
            if (c + r < d_v && at < d_k)
                *reinterpret_cast<float4 *>(rows + (size_t)r * d_k + at) =
                    make_float4(x[r][2 * j].x, x[r][2 * j].y, x[r][2 * j + 1].x, x[r][2 * j + 1].y);
        }
}

// Fast forms for d_k = d_v = 128, bf16 inputs, paths of at most 16 nodes: CTAs of 256 threads, one per (tree, value head);
// the state loads go first, the path is fetched and checked by one warp with shuffles, its k/v rows arrive by cp.async.
// Two forms of the arithmetic and, for few tiles, a split of the tile, chosen by how many tiles the call has for how many SMs
// (commit_form):
//   step by step (commit_replay_unit): 64 state registers per thread, two CTAs per SM; the shortest chain, the better one
//     while all CTAs of the call are resident at once that way;
//   step by step with 32 rows of the tile per CTA, one per thread: a step is as short as its reduction then.  32 tiles, path of
//     1 / 7 / 12: 4.1 / 5.7 / 6.8 -> 3.1 / 3.9 / 4.6 us, followed by a verification 11.5 / 13.0 / 14.4 -> 11.6 / 11.7 / 12.9 us (only
//     with the carve-out of launch_overlapped: 14.5 without); at 64 tiles the pair gets slower (11.7 / 13.2 -> 12.7 / 13.4);
//   as matrix products (commit_fragment_unit, gdn_fragments.cuh): 32 state registers, the tile read twice, the second time
//     out of L2; three or four CTAs per SM, so that the loads of some run under the arithmetic of others.
// Measured (us; 32 heads per slot, path of 7; two by two / three / four per SM): 4 slots 6.5 / 6.9 / 7.2, 8 slots 9.8 / 11.4 /
// 10.3, 12 slots 15.4 / 12.9 / 14.7, 14 slots 17.2 / 17.9 / 16.0, 32 slots 33.2 / 31.2 / 29.5, 48 slots 46.9 / 43.1 / 40.6 (path of
// 1: 37.7 / 39.9 / 38.0, of 12: 57.4 / 52.2 / 54.3, of 16: 64.2 / 54.0 / 55.7; HBM alone: 31).
// Error of the state against 64 bits, in the norm, step by step / as matrix products: path of 1 5.5e-8 / 4.5e-8, of 7 6.7e-8 /
// 6.2e-8, of 16 6.6e-8 / 6.3e-8.
// PARTS: the tile's rows split over that many CTAs.
template <int PARTS> __device__ __forceinline__ void commit_replay_unit(const CommitParams &p, const int unit, const int part)
{
    constexpr int ROWS = 4 / PARTS;   // per thread
    __shared__ __align__(16) uint16_t pk_s[CF_MD * GDN_TILE_D];
    __shared__ __align__(16) uint16_t pv_s[CF_MD * GDN_TILE_D];
    __shared__ __align__(16) float4 ab_s[CF_MD];
    __shared__ int len_s;

    const int b = unit / p.h_v, h = unit % p.h_v;
    const int hk = h / (p.h_v / p.h_qk);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = part * (GDN_TILE_D / PARTS) + warp * 4 * ROWS;   // of this warp
    if (tid < ROWS)   // L2 may be asked for the tile meanwhile (a prefetch consumes nothing)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                     ::"l"(p.S + (size_t)unit * GDN_TILE_D * GDN_TILE_D + (size_t)(part * ROWS + tid) * 4096), "r"(16384) : "memory");
    wait_for_previous_kernel();
    const int r4 = lane >> 3, l8 = lane & 7;
    const int tree = p.t_pad ? b % p.n_trees : b;
    const int pp0 = p.t_pad ? tree * p.path_stride : p.path_offsets[b];
    int len = p.t_pad ? p.path_len[tree] : p.path_offsets[b + 1] - pp0;
    if (len == 0) return;   // nothing accepted from this tree: state untouched

    // the state tile first: its latency covers the path fetch below
    float *S = p.S + (size_t)(b * p.h_v + h) * GDN_TILE_D * GDN_TILE_D;
    float4 x[ROWS][4];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        const float *src = S + (size_t)(row0 + i * 4 + r4) * GDN_TILE_D + l8 * 8;
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) ldg_v8(src + kh * 64, x[i][kh * 2 + 0], x[i][kh * 2 + 1]);
    }

    const int pb = p.t_pad ? b * p.t_pad : p.node_offsets[b];
    const int pT = p.t_pad ? min(p.n_nodes[tree], p.t_pad) : p.node_offsets[b + 1] - pb;
    const int ppar = p.t_pad ? tree * p.t_pad : pb;   // first entry of the tree in parent[]
    const __nv_bfloat16 *k = static_cast<const __nv_bfloat16 *>(p.k), *v = static_cast<const __nv_bfloat16 *>(p.v);
    const __nv_bfloat16 *g = static_cast<const __nv_bfloat16 *>(p.g), *beta = static_cast<const __nv_bfloat16 *>(p.beta);
    const bool shape_ok = len > 0 && len <= CF_MD && len <= p.max_depth && pT > 0 && pp0 >= 0;
    // Every thread reads the path entry whose row piece it fetches (no hand-over through shared memory in front of
    // the row fetch); an entry outside the tree is skipped here and reported by the check below.
    if (shape_ok) {
        for (int idx = tid; idx < len * 32; idx += CF_THREADS) {
            const int t = idx >> 5, c16 = idx & 15;
            const int nt = p.path[pp0 + t];
            if (nt < 0 || nt >= pT) continue;
            const size_t n = (size_t)pb + nt;
            if (idx & 16)
                cf_cp_async_16((uint32_t)__cvta_generic_to_shared(pv_s + t * GDN_TILE_D + c16 * 8),
                               v + (n * p.h_v + h) * GDN_TILE_D + c16 * 8);
            else
                cf_cp_async_16((uint32_t)__cvta_generic_to_shared(pk_s + t * GDN_TILE_D + c16 * 8),
                               k + (n * p.h_qk + hk) * GDN_TILE_D + c16 * 8);
        }
    }
    if (warp == 0) {
        // lane t: entry t of the path and that node's parent; the path must be a chain from a root inside the tree
        const bool mine = shape_ok && lane < len;
        int n = -1, parent_n = -2;
        if (mine) {
            n = p.path[pp0 + lane];
            if (p.parent && n >= 0 && n < pT) parent_n = p.parent[ppar + n];
        }
        const int n_up = __shfl_up_sync(0xffffffffu, n, 1);
        bool bad = false;
        if (mine) {
            if (n < 0 || n >= pT) bad = true;
            else if (p.parent) bad = parent_n != (lane ? n_up : -1);
            else if (lane && n <= n_up) bad = true;   // without parent[] only the topological order can be checked
        }
        if (__any_sync(0xffffffffu, bad) || !shape_ok) {
            if (lane == 0) report_status(p.status_dev, GDN_ERR_PATH);
            len = 0;
        }
        // per-step scalars: decay of the path up to and including step t by a prefix sum over the lanes
        float gt = 0.f, be = 0.f;
        if (lane < len) {
            const unsigned short *g16 = reinterpret_cast<const unsigned short *>(g);
            const unsigned short *b16 = reinterpret_cast<const unsigned short *>(beta);
            gt = gate_log_decay(g16[((size_t)pb + n) * p.h_v + h], p.raw_gates != 0);
            be = gate_beta(b16[((size_t)pb + n) * p.h_v + h], p.raw_gates != 0);
        }
        float gsum = gt;
#pragma unroll
        for (int off = 1; off < CF_MD; off <<= 1) {
            const float up = __shfl_up_sync(0xffffffffu, gsum, off);
            if (lane >= off) gsum += up;
        }
        if (lane < len) {
            const float A = expf(gsum);
            ab_s[lane] = make_float4(A, be, expf(gt), 1.f / A);
        }
        if (lane == 0) len_s = len;
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    len = len_s;
    if (len == 0) return;   // rejected path: this state stays as it was

    replay_path_on_tile(x, len, pk_s, pv_s, ab_s, row0, r4, l8);

#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        float *dst = S + (size_t)(row0 + i * 4 + r4) * GDN_TILE_D + l8 * 8;
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) stg_v8(dst + kh * 64, x[i][kh * 2 + 0], x[i][kh * 2 + 1]);
    }
}

// The two passes of the tile through the registers (all threads; a barrier in between, for the coupling table).  x: chunks 0, 1.
template <int TILES>
__device__ __forceinline__ void commit_tile_passes(float *S, float (&x)[2][4][4], int len, uint32_t operand, const PathTile &path, int row,
                                                   int lane, const float &decay_s)
{
    PathUpdate<TILES> up;
    {
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
        __syncthreads();   // the coupling table
        path_solve(a, len, path, row, lane, up);
    }
    const float A_L = decay_s;
#pragma unroll 1
    for (int j = 0; j < 4; j += 2)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            path_update_chunk(x[i], j + i, operand, A_L, up);
            store_chunk(S, j + i, x[i]);
            if (j == 0) load_chunk(S, i + 2, x[i]);
        }
}

__device__ __forceinline__ void commit_fragment_unit(const CommitParams &p, const int unit)
{
    __shared__ __align__(16) uint8_t pk_s[CF_MD * GDN_PK_STRIDE];
    __shared__ __align__(16) uint16_t pv_s[CF_MD * GDN_TILE_D];
    __shared__ __align__(16) float couple_s[CF_MD * 16];
    __shared__ __align__(16) float4 scal_s[CF_MD];
    __shared__ int len_s;
    __shared__ float decay_s;

    const int b = unit / p.h_v, h = unit % p.h_v;
    const int hk = h / (p.h_v / p.h_qk);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < 4)   // L2 may be asked for the tile meanwhile (a prefetch consumes nothing)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                     ::"l"(p.S + (size_t)unit * GDN_TILE_D * GDN_TILE_D + (size_t)tid * 4096), "r"(16384) : "memory");
    wait_for_previous_kernel();
    const int tree = p.t_pad ? b % p.n_trees : b;
    const int pp0 = p.t_pad ? tree * p.path_stride : p.path_offsets[b];
    int len = p.t_pad ? p.path_len[tree] : p.path_offsets[b + 1] - pp0;
    if (len == 0) return;   // nothing accepted from this tree: state untouched

    // the state first: its latency covers the path fetch below
    const int row = warp * 16 + (lane >> 2);
    float *S = p.S + (size_t)unit * GDN_TILE_D * GDN_TILE_D + (size_t)row * GDN_TILE_D + (lane & 3) * 8;
    float x[2][4][4];
    load_chunk(S, 0, x[0]);
    load_chunk(S, 1, x[1]);

    const int pb = p.t_pad ? b * p.t_pad : p.node_offsets[b];
    const int pT = p.t_pad ? min(p.n_nodes[tree], p.t_pad) : p.node_offsets[b + 1] - pb;
    const bool shape_ok = len > 0 && len <= CF_MD && len <= p.max_depth && pT > 0 && pp0 >= 0;
    const uint32_t pk = (uint32_t)__cvta_generic_to_shared(pk_s);
    if (shape_ok) path_rows_fetch(p, pp0, len, pb, pT, h, hk, pk, pv_s, tid);
    float gt = 0.f, be = 0.f;   // of step `lane` (warp 0)
    if (warp == 0) {
        len = path_check_and_scalars(p, pp0, shape_ok ? len : 0, pb, pT, p.t_pad ? tree * p.t_pad : pb, h, lane, gt, be, scal_s, decay_s);
        if (lane == 0) len_s = len;
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    len = len_s;
    if (len == 0) return;   // rejected path: this state stays as it was
    if (warp == 0 && len > 1) path_coupling(pk, len, gt, be, couple_s, lane);
    const PathTile path{pv_s, scal_s, couple_s};
    if (len <= 8) commit_tile_passes<1>(S, x, len, path_operand(pk, lane), path, row, lane, decay_s);
    else commit_tile_passes<2>(S, x, len, path_operand(pk, lane), path, row, lane, decay_s);
}

// CTAS: CTAs per SM (1, 2: step by step, 1: a quarter of a tile per CTA; otherwise as matrix products)
template <int CTAS> __device__ __forceinline__ void commit_unit(const CommitParams &p, const int i)
{
    if constexpr (CTAS == 1) commit_replay_unit<4>(p, i >> 2, i & 3);
    else if constexpr (CTAS == 2) commit_replay_unit<1>(p, i, 0);
    else commit_fragment_unit(p, i);
}

template <int CTAS> __global__ void __launch_bounds__(CF_THREADS, CTAS == 1 ? 4 : CTAS) commit_tile128_kernel(const CommitParams p)
{
    commit_unit<CTAS>(p, (int)blockIdx.x);
}

// The fused call on trees of more than 64 nodes: the plans of the NEW trees do not depend on the commit of the previous
// step's paths, so they are built by the first n_seq CTAs of the same grid instead of by a launch of their own in
// between (one launch and one dependency hop less in front of the verify kernel).
template <int CTAS> __global__ void __launch_bounds__(CF_THREADS, CTAS == 1 ? 2 : CTAS) commit_plan_kernel(const CommitParams p, const PlanArgs a)
{
    if ((int)blockIdx.x < a.n_seq) {
        wait_for_previous_kernel();
        plan_tree<CF_THREADS>(a, (int)blockIdx.x);
    } else
        commit_unit<CTAS>(p, (int)blockIdx.x - a.n_seq);
}

// Form for a call of `units` tiles: a quarter of a tile per CTA while those have SMs of their own, otherwise the fewest CTAs
// per SM with which they are all resident at once.
int commit_form(int units)
{
    static PerContext seen;
    int sms = 0;
    if (device_sms(seen, nullptr, 0, &sms) != cudaSuccess) return 2;
    return 4 * units <= sms ? 1 : units <= 2 * sms ? 2 : units <= 3 * sms ? 3 : 4;
}

cudaError_t launch_tile128(const CommitParams &p, int units, cudaStream_t stream)
{
    const int form = commit_form(units);
    return launch_overlapped(form == 1   ? commit_tile128_kernel<1>
                             : form == 2 ? commit_tile128_kernel<2>
                             : form == 3 ? commit_tile128_kernel<3>
                                         : commit_tile128_kernel<4>,
                             form == 1 ? 4 * units : units, CF_THREADS, 0, form == 1, stream, p);
}

}  // namespace

cudaError_t launch_commit_generic(const gdn_shape_t &s, float *S, const void *k, const void *v,
                                  const void *g, const void *beta, const int32_t *parent,
                                  const int32_t *node_offsets, const int32_t *path,
                                  const int32_t *path_offsets, int32_t *status_dev, cudaStream_t stream)
{
    const int grid = s.n_seq * s.h_v;
    if (grid == 0) return cudaSuccess;
    CommitParams p{s.h_qk, s.h_v, s.d_k, s.d_v, s.max_depth, S, k, v, g, beta,
                   parent, node_offsets, path, path_offsets, status_dev, 0, 0, 0, 0, nullptr, nullptr};
    if (commit_tile128_supported(s) && (reinterpret_cast<uintptr_t>(S) & 31u) == 0)   // 32-byte accesses of the state
        return launch_tile128(p, grid, stream);
    static PerContext seen[2];
    const auto kernel = s.in_dtype == GDN_BF16 ? commit_generic_kernel<__nv_bfloat16> : commit_generic_kernel<float>;
    int sms = 0;
    const cudaError_t e = device_sms(seen[s.in_dtype == GDN_BF16], reinterpret_cast<const void *>(kernel),
                                     commit_generic_smem(GDN_MAX_DEPTH_CAP), &sms);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kernel, grid, CM_THREADS, commit_generic_smem(s.max_depth), false, stream, p);
}

bool commit_tile128_supported(const gdn_shape_t &s) { return commit_padded_supported(s); }

// Commit of the previous step's paths (ragged packing, tile kernel) and the plan of the new trees in one grid.
cudaError_t launch_commit_plan(const gdn_shape_t &s, float *S, const void *k, const void *v, const void *g,
                               const void *beta, const int32_t *parent_prev, const int32_t *node_offsets_prev,
                               const int32_t *path, const int32_t *path_offsets, const int32_t *parent,
                               const int32_t *node_offsets, const PlanPtrs &plan, int32_t *status_dev,
                               cudaStream_t stream)
{
    if (s.n_seq == 0) return cudaSuccess;
    if (s.n_seq > 1) {   // the trees' CTAs claim their places in the unit list from a counter
        cudaError_t e0 = cudaMemsetAsync(plan.unit_count, 0, sizeof(int32_t), stream);
        if (e0 != cudaSuccess) return e0;
    }
    CommitParams p{s.h_qk, s.h_v, s.d_k, s.d_v, s.max_depth, S, k, v, g, beta, parent_prev, node_offsets_prev, path,
                   path_offsets, status_dev, 0, 0, 0, 0, nullptr, nullptr};
    const int units = s.n_seq * s.h_v, form = commit_form(units);
    return launch_overlapped(form == 1   ? commit_plan_kernel<1>
                             : form == 2 ? commit_plan_kernel<2>
                             : form == 3 ? commit_plan_kernel<3>
                                         : commit_plan_kernel<4>,
                             s.n_seq + (form == 1 ? 4 * units : units), CF_THREADS, 0, form == 1, stream, p,
                             plan_args(s, parent, node_offsets, nullptr, plan, status_dev));
}

bool commit_padded_supported(const gdn_shape_t &s)
{
    return s.d_k == GDN_TILE_D && s.d_v == GDN_TILE_D && s.in_dtype == GDN_BF16 && s.max_depth <= CF_MD;
}

cudaError_t launch_commit_padded(const gdn_shape_t &s, int n_trees, bool raw_gates, float *S, const void *k,
                                 const void *v, const void *g, const void *beta, const int32_t *parent,
                                 const int32_t *n_nodes, const int32_t *path, const int32_t *path_len,
                                 int32_t *status_dev, cudaStream_t stream)
{
    const int grid = s.n_seq * s.h_v;
    if (grid == 0) return cudaSuccess;
    CommitParams p{s.h_qk, s.h_v, s.d_k, s.d_v, s.max_depth, S, k, v, g, beta, parent, nullptr, path, nullptr,
                   status_dev, s.max_tree_nodes, n_trees, s.max_depth, raw_gates ? 1 : 0, n_nodes, path_len};
    return launch_tile128(p, grid, stream);
}

}  // namespace gdn
