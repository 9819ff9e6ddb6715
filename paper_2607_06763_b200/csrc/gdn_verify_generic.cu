// Generic tree-verify kernel: any d_k, d_v <= 128, fp32 or bf16 inputs, CUDA cores only.
//
// It evaluates the triangular form of Section 3.4.1 restricted to real ancestors.  With
// dec(i,j) = exp(sum of g over the nodes after j up to and including i on i's root path)
// (= a_i / a_j of Eq. 9, formed as a suffix sum so that no large exponents cancel):
//     p^k_i = S0^T k_i,  p^q_i = S0^T q_i                          (the S0 terms of Eq. 11 / 13)
//     u~_i  = beta_i (v_i - a_i p^k_i) - sum_{j < i on path} dec(i,j) beta_i (k_i.k_j) u~_j   (Eq. 10, 13)
//     o_i   = scale (a_i p^q_i + sum_{j <= i on path} dec(i,j) (q_i.k_j) u~_j)              (Eq. 11)
// u~_i = u_i - w_i^T S0 is the quantity the substitution returns once the W S0 term is folded
// into the right-hand side (Section 3.4.2), so W is never formed.
//
// One CTA per (tree, value head).  Thread (c, s): value component c, quarter s of the key
// dimension; the [d_v][d_k] state tile lives in registers (32 floats per thread) and the two
// projections are reduced over the four s-lanes with warp shuffles.  Nodes are visited in index
// order (parents first); u~ is kept in the workspace (L2) because a tree may be larger than
// shared memory allows.
#include "gdn_internal.cuh"

namespace gdn {

namespace {

constexpr int VG_THREADS = 512;
constexpr int VG_SPLIT = 4;                      // lanes sharing one value component
constexpr int VG_CHUNK = 32;                     // nodes whose coefficients are prepared together
constexpr int VG_DK = GDN_MAX_HEAD_DIM;          // padded key dim in shared memory
constexpr int VG_REGS = VG_DK / VG_SPLIT;        // state floats per thread
constexpr int VG_WARPS = VG_THREADS / 32;

struct VerifyGenericParams {
    int h_qk, h_v, d_k, d_v, max_depth;
    float scale;
    const float *S0;
    const void *q, *k, *v, *g, *beta;
    const int32_t *node_offsets;
    void *o;
    const int32_t *tree_ok;
    const uint8_t *depth;
    const uint16_t *anc;
    float *utilde;
};

template <typename TIn, typename TOut>
__global__ void __launch_bounds__(VG_THREADS, 1) verify_generic_kernel(const VerifyGenericParams p)
{
    extern __shared__ __align__(16) float vg_smem[];
    float (*ks)[VG_DK] = reinterpret_cast<float (*)[VG_DK]>(vg_smem);
    float (*qs)[VG_DK] = ks + VG_CHUNK;
    float *xc = &qs[VG_CHUNK][0];                 // [VG_CHUNK][max_depth]: dec, then X coefficients
    float *yc = xc + VG_CHUNK * p.max_depth;      // [VG_CHUNK][max_depth]: Y coefficients (self included)
    float *a_s = yc + VG_CHUNK * p.max_depth;     // [VG_CHUNK]
    float *beta_s = a_s + VG_CHUNK;               // [VG_CHUNK]

    const int b = blockIdx.x / p.h_v, h = blockIdx.x % p.h_v;
    if (!p.tree_ok[b]) return;
    const int base = p.node_offsets[b];
    const int T = p.node_offsets[b + 1] - base;
    if (T <= 0) return;
    const int hk = h / (p.h_v / p.h_qk);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = tid / VG_SPLIT, s = tid % VG_SPLIT;
    const bool comp_on = c < p.d_v;
    const int d_k = p.d_k, d_v = p.d_v, md = p.max_depth;

    const TIn *q = static_cast<const TIn *>(p.q), *k = static_cast<const TIn *>(p.k);
    const TIn *v = static_cast<const TIn *>(p.v), *g = static_cast<const TIn *>(p.g);
    const TIn *beta = static_cast<const TIn *>(p.beta);
    TOut *o = static_cast<TOut *>(p.o);

    // State slice: register 4*j+e holds S0[c][16*j + 4*s + e] (zero beyond d_k / d_v).
    float sreg[VG_REGS];
    {
        const float *row = p.S0 + ((size_t)(b * p.h_v + h) * d_v + (comp_on ? c : 0)) * d_k;
#pragma unroll
        for (int j = 0; j < VG_REGS / 4; ++j) {
            const int r = 16 * j + 4 * s;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (comp_on && r < d_k) x = __ldg(reinterpret_cast<const float4 *>(row + r));
            sreg[4 * j + 0] = x.x; sreg[4 * j + 1] = x.y; sreg[4 * j + 2] = x.z; sreg[4 * j + 3] = x.w;
        }
    }
    for (int idx = tid; idx < VG_CHUNK * VG_DK; idx += VG_THREADS) {
        (&ks[0][0])[idx] = 0.f;
        (&qs[0][0])[idx] = 0.f;
    }

    for (int i0 = 0; i0 < T; i0 += VG_CHUNK) {
        const int cn = min(VG_CHUNK, T - i0);
        __syncthreads();   // previous chunk fully consumed (and the zero fill done)
        // (a) stage this chunk's k and q rows as fp32
        for (int idx = tid; idx < cn * d_k; idx += VG_THREADS) {
            const int t = idx / d_k, r = idx % d_k;
            const size_t src = ((size_t)(base + i0 + t) * p.h_qk + hk) * d_k + r;
            ks[t][r] = load_as_float(k + src);
            qs[t][r] = load_as_float(q + src);
        }
        // (b0) per node: decay from each path position to the node, total decay a_i, beta_i
        if (tid < cn) {
            const int n = base + i0 + tid;
            const int d = p.depth[n];
            const uint16_t *path = p.anc + (size_t)n * md;
            float sfx = 0.f;
            for (int a = d - 1; a >= 0; --a) {
                xc[tid * md + a] = expf(sfx);
                sfx += load_as_float(g + (size_t)(base + path[a]) * p.h_v + h);
            }
            a_s[tid] = expf(sfx);
            beta_s[tid] = load_as_float(beta + (size_t)n * p.h_v + h);
        }
        __syncthreads();
        // (b) one warp per (node, path position): k_i.k_j and q_i.k_j, scaled into X and Y of Eq. 9
        for (int idx = warp; idx < cn * md; idx += VG_WARPS) {
            const int t = idx / md, a = idx % md;
            const int n = base + i0 + t;
            const int d = p.depth[n];
            if (a >= d) continue;
            const int j = p.anc[(size_t)n * md + a];
            const TIn *kj = k + ((size_t)(base + j) * p.h_qk + hk) * d_k;
            float kk = 0.f, qk = 0.f;
            for (int r = lane; r < d_k; r += 32) {
                const float x = load_as_float(kj + r);
                kk = fmaf(ks[t][r], x, kk);
                qk = fmaf(qs[t][r], x, qk);
            }
#pragma unroll
            for (int m = 16; m > 0; m >>= 1) {
                kk += __shfl_xor_sync(0xffffffffu, kk, m);
                qk += __shfl_xor_sync(0xffffffffu, qk, m);
            }
            if (lane == 0) {
                const float dec = xc[t * md + a];
                yc[t * md + a] = dec * qk;
                xc[t * md + a] = beta_s[t] * dec * kk;   // entry a = d-1 (the node itself) is never read
            }
        }
        __syncthreads();
        // (c) nodes in order: projections, forward substitution step, output
        for (int t = 0; t < cn; ++t) {
            const int n = base + i0 + t;
            float pk = 0.f, pq = 0.f;
#pragma unroll
            for (int j = 0; j < VG_REGS / 4; ++j) {
                const float4 kx = *reinterpret_cast<const float4 *>(&ks[t][16 * j + 4 * s]);
                const float4 qx = *reinterpret_cast<const float4 *>(&qs[t][16 * j + 4 * s]);
                pk = fmaf(sreg[4 * j + 0], kx.x, pk); pk = fmaf(sreg[4 * j + 1], kx.y, pk);
                pk = fmaf(sreg[4 * j + 2], kx.z, pk); pk = fmaf(sreg[4 * j + 3], kx.w, pk);
                pq = fmaf(sreg[4 * j + 0], qx.x, pq); pq = fmaf(sreg[4 * j + 1], qx.y, pq);
                pq = fmaf(sreg[4 * j + 2], qx.z, pq); pq = fmaf(sreg[4 * j + 3], qx.w, pq);
            }
            pk += __shfl_xor_sync(0xffffffffu, pk, 1); pk += __shfl_xor_sync(0xffffffffu, pk, 2);
            pq += __shfl_xor_sync(0xffffffffu, pq, 1); pq += __shfl_xor_sync(0xffffffffu, pq, 2);

            const int d = p.depth[n];
            const uint16_t *path = p.anc + (size_t)n * md;
            float sx = 0.f, sy = 0.f;   // partial sums over this lane's share of the ancestors
            if (comp_on) {
                for (int a = s; a < d - 1; a += VG_SPLIT) {
                    const float uj = __ldcg(p.utilde + ((size_t)(base + path[a]) * p.h_v + h) * d_v + c);
                    sx = fmaf(xc[t * md + a], uj, sx);
                    sy = fmaf(yc[t * md + a], uj, sy);
                }
            }
            sx += __shfl_xor_sync(0xffffffffu, sx, 1); sx += __shfl_xor_sync(0xffffffffu, sx, 2);
            sy += __shfl_xor_sync(0xffffffffu, sy, 1); sy += __shfl_xor_sync(0xffffffffu, sy, 2);
            if (comp_on) {
                const float vi = load_as_float(v + ((size_t)n * p.h_v + h) * d_v + c);
                const float ui = beta_s[t] * (vi - a_s[t] * pk) - sx;
                const float out = p.scale * (fmaf(a_s[t], pq, sy) + yc[t * md + d - 1] * ui);
                if (s == 0) {
                    __stcg(p.utilde + ((size_t)n * p.h_v + h) * d_v + c, ui);
                    store_from_float(o + ((size_t)n * p.h_v + h) * d_v + c, out);
                }
            }
            __syncwarp();   // lane s==0's u~ store is ordered before the other lanes' later loads
        }
    }
}

// ---------------------------------------------------------------------------------------- trees of at most 64 nodes
// The same triangular form with the solve moved to the query side, so that no node waits for another one.  With
// X(l, t) = beta_l dec(l, t) (k_l.k_t) and y_it = dec(i, t) (q_i.k_t) along the root path of node i, row i of
// Z = Y (I + X)^-1 is a back-substitution over that path alone, and
//     o_i = S0^T q'_i + sum_t scale z_it beta_t v_t,      q'_i = scale (a_i q_i - sum_t z_it beta_t a_t k_t).
// One CTA per (tree, value head, run of blocks of VS_NODES nodes); the tree metadata is derived from parent[] by every CTA
// (64 nodes: a walk of at most max_depth steps per thread), so no plan kernel runs in front.  Bound by shared memory
// bandwidth (16-byte loads: the k rows in the dots, k and v rows in q' and outputs, q' in the state product, where eight
// lanes hold four state rows so that a piece of q' serves four of them) and by latency for small batches.  Against the
// kernel above, which visits the nodes of a tree one after the other: 8 trees of 9..64 nodes, 32 heads of 128 components,
// fp32, verification alone: 61 us with one block per CTA, one dot per warp at a time, two rows per thread and v rows read
// where they are used, 29 us in this form; verification and commit 230 -> 42 us; one tree of 8 nodes, 4 heads of 32
// components 27.0 -> 10.4 us.
constexpr int VS_THREADS = 256;
constexpr int VS_TREE = 64;      // largest tree
constexpr int VS_NODES = 16;     // nodes per block
constexpr int VS_SPLIT = 8;      // lanes sharing four value components
constexpr int VS_VROW = VG_DK + 4;   // floats of a staged v row: the eight lanes read one piece of eight different rows

struct VerifySmallParams {
    int h_qk, h_v, d_k, d_v, max_depth, max_tree_nodes, total_nodes, n_seq;
    int n_parts, part_nodes;   // CTAs per (tree, head); nodes of each, a multiple of VS_NODES
    float scale;
    const float *S0;
    const void *q, *k, *v, *g, *beta;
    const int32_t *parent, *node_offsets;
    void *o;
    int32_t *status_dev;
};

__device__ __forceinline__ float4 load4_as_float(const __nv_bfloat16 *p)
{
    const uint2 w = __ldg(reinterpret_cast<const uint2 *>(p));
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                       __uint_as_float(w.y & 0xFFFF0000u));
}

// Rows 0 .. rows - 1 of one head (d components, `stride` apart in memory) as fp32 into dst; fp32 rows by cp.async.
template <typename T, int ROW>
__device__ __forceinline__ void stage_rows(float (*dst)[ROW], const T *src, size_t stride, int rows, int d, int tid)
{
    if (d % 4 == 0) {
#pragma unroll 4
        for (int idx = tid; idx < rows * 32; idx += VS_THREADS) {
            const int t = idx >> 5, r = (idx & 31) * 4;
            if (r >= d) continue;
            if constexpr (sizeof(T) == 4)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             ::"r"((uint32_t)__cvta_generic_to_shared(&dst[t][r])), "l"(src + t * stride + r) : "memory");
            else
                *reinterpret_cast<float4 *>(&dst[t][r]) = load4_as_float(src + t * stride + r);
        }
    } else {
#pragma unroll 4
        for (int idx = tid; idx < rows * VG_DK; idx += VS_THREADS) {
            const int t = idx / VG_DK, r = idx % VG_DK;
            if (r >= d) continue;
            if constexpr (sizeof(T) == 4)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                             ::"r"((uint32_t)__cvta_generic_to_shared(&dst[t][r])), "l"(src + t * stride + r) : "memory");
            else
                dst[t][r] = load_as_float(src + t * stride + r);
        }
    }
}

struct VerifySmallSmem {
    float ks[VS_TREE][VG_DK];              // k rows of the nodes up to the CTA's last
    float vs[VS_TREE][VS_VROW];            // their v rows
    float qp[2][VS_NODES][VG_DK];          // q rows of a block, then its q'
    float x[VS_TREE][VS_TREE];             // decays, then X(l, .): entry j belongs to the j-th node up the root path of l
    float y[VS_NODES][2 * VS_TREE];        // y, then the weights of the k rows, same order; from VS_TREE on those of the v
                                           // rows; then the v rows' part of the outputs
    float a[VS_TREE], beta[VS_TREE], g[VS_TREE];
    unsigned long long mask[VS_TREE];      // nodes on the root path
    int par[VS_TREE];
    uint8_t up[VS_TREE][VS_TREE];          // j-th node up the root path (0 = the node itself)
    uint8_t depth[VS_TREE];
};

template <typename TIn, typename TOut>
__global__ void __launch_bounds__(VS_THREADS, 2) verify_generic_small_kernel(const VerifySmallParams p)
{
    extern __shared__ __align__(16) uint8_t vs_smem[];
    VerifySmallSmem &sm = *reinterpret_cast<VerifySmallSmem *>(vs_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int part = blockIdx.x % p.n_parts, bh = blockIdx.x / p.n_parts, b = bh / p.h_v, h = bh % p.h_v;
    const int hk = h / (p.h_v / p.h_qk), i_lo = part * p.part_nodes;
    const int d_k = p.d_k, d_v = p.d_v;
    const TIn *q = static_cast<const TIn *>(p.q), *k = static_cast<const TIn *>(p.k);
    const TIn *v = static_cast<const TIn *>(p.v), *g = static_cast<const TIn *>(p.g), *beta = static_cast<const TIn *>(p.beta);
    TOut *o = static_cast<TOut *>(p.o);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");

    const int base = p.node_offsets[b], end = p.node_offsets[b + 1], T = end - base;
    bool offsets_ok = base >= 0 && T >= 0 && T <= p.max_tree_nodes && T <= VS_TREE && end <= p.total_nodes;
    if (b == 0) offsets_ok = offsets_ok && base == 0;
    if (b == p.n_seq - 1) offsets_ok = offsets_ok && end == p.total_nodes;
    if (!offsets_ok) {
        if (tid == 0) report_status(p.status_dev, GDN_ERR_TREE);
        return;
    }
    if (i_lo >= T) return;
    const int i_hi = min(i_lo + p.part_nodes, T);
    if (tid < T) {
        sm.par[tid] = p.parent[base + tid];
        sm.g[tid] = load_as_float(g + (size_t)(base + tid) * p.h_v + h);
        sm.beta[tid] = load_as_float(beta + (size_t)(base + tid) * p.h_v + h);
    }
    // Rows of the nodes up to the CTA's last (an ancestor has a smaller index) and the first block's q rows, then the state:
    // all of it is under way while the root paths are walked.
    const TIn *q_head = q + ((size_t)base * p.h_qk + hk) * d_k;
    const size_t q_stride = (size_t)p.h_qk * d_k;
    stage_rows(sm.ks, k + ((size_t)base * p.h_qk + hk) * d_k, q_stride, i_hi, d_k, tid);
    stage_rows(sm.qp[0], q_head + i_lo * q_stride, q_stride, min(VS_NODES, i_hi - i_lo), d_k, tid);
    stage_rows(sm.vs, v + ((size_t)base * p.h_v + h) * d_v, (size_t)p.h_v * d_v, i_hi, d_v, tid);
    // State: rows c .. c + 3; sreg[r][2 j], [2 j + 1] hold key positions 32 j + 4 s + e (zero beyond d_k / d_v).  Not through the
    // read-only path: the commit in front may still be writing the state while this grid moves in.
    const int c = (tid / VS_SPLIT) * 4, s = tid % VS_SPLIT;
    float2 sreg[4][8];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float *row = p.S0 + ((size_t)(b * p.h_v + h) * d_v + (c + r < d_v ? c + r : 0)) * d_k;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int at = 32 * j + 4 * s;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c + r < d_v && at < d_k) x = *reinterpret_cast<const float4 *>(row + at);
            sreg[r][2 * j] = make_float2(x.x, x.y);
            sreg[r][2 * j + 1] = make_float2(x.z, x.w);
        }
    }
    __syncthreads();

    // Root paths, by one thread per node; decays as sums of g from the ancestor's child down to the node, so that no large
    // exponents cancel.  A bad parent[] or a path of more than max_depth nodes rejects the tree.
    int err = 0;
    if (tid < T) {
        int d = 0, cur = tid;
        float sfx = 0.f;
        unsigned long long m = 0;
        while (cur >= 0) {
            if (d == p.max_depth) { err = GDN_ERR_DEPTH; break; }
            sm.up[tid][d] = (uint8_t)cur;
            sm.x[tid][d] = expf(sfx);
            m |= 1ull << cur;
            sfx += sm.g[cur];
            ++d;
            const int up = sm.par[cur];
            if (up < -1 || up >= cur) { err = GDN_ERR_TREE; break; }
            cur = up;
        }
        sm.depth[tid] = (uint8_t)d;
        sm.mask[tid] = m;
        sm.a[tid] = expf(sfx);
    }
    if (err) report_status(p.status_dev, err);
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (__syncthreads_or(err != 0)) return;
    unsigned long long need = 0;   // the CTA's nodes and their ancestors
    for (int i = i_lo; i < i_hi; ++i) need |= sm.mask[i];
    const int vecs = d_k / 4;

    const int l8 = lane & 7;
    // Block by block in ascending order, so that an ancestor's X is there; the buffer of the block after the next barrier
    // takes the q rows of the block to come.
#pragma unroll 1
    for (int i0 = i_lo, buf = 0; i0 < i_hi; i0 += VS_NODES, buf ^= 1) {
        const int nn = min(VS_NODES, i_hi - i0);
        // X and y: a warp per node, eight lanes per path entry, four entries at a time; the first block also takes the
        // ancestors in front of the CTA's nodes
        for (int l = (i0 == i_lo ? 0 : i0) + warp; l < i0 + nn; l += VS_THREADS / 32) {
            if (!((need >> l) & 1)) continue;
            const bool own = l >= i0;
            float4 kl[4], ql[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int r = l8 + 8 * m;
                kl[m] = ql[m] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (r < vecs) {
                    kl[m] = *reinterpret_cast<const float4 *>(&sm.ks[l][4 * r]);
                    if (own) ql[m] = *reinterpret_cast<const float4 *>(&sm.qp[buf][l - i0][4 * r]);
                }
            }
            const int d = sm.depth[l];
            const float be = sm.beta[l];
            for (int j0 = own ? 0 : 1; j0 < d; j0 += 8) {
                float w[2], dec[2];
                int j[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    j[e] = j0 + 4 * e + (lane >> 3);
                    w[e] = dec[e] = 0.f;
                    if (j0 + 4 * e >= d) break;
                    const float *kr = sm.ks[j[e] < d ? sm.up[l][j[e]] : l];
                    dec[e] = j[e] < d ? sm.x[l][j[e]] : 0.f;
                    float4 k4 = make_float4(0.f, 0.f, 0.f, 0.f), q4 = k4;
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const int r = l8 + 8 * m;
                        float4 kt = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (r < vecs) kt = *reinterpret_cast<const float4 *>(kr + 4 * r);
                        k4 = make_float4(fmaf(kl[m].x, kt.x, k4.x), fmaf(kl[m].y, kt.y, k4.y), fmaf(kl[m].z, kt.z, k4.z),
                                         fmaf(kl[m].w, kt.w, k4.w));
                        q4 = make_float4(fmaf(ql[m].x, kt.x, q4.x), fmaf(ql[m].y, kt.y, q4.y), fmaf(ql[m].z, kt.z, q4.z),
                                         fmaf(ql[m].w, kt.w, q4.w));
                    }
                    // lanes 0..3 of the eight end up with k.k, lanes 4..7 with q.k
                    const float kk = (k4.x + k4.y) + (k4.z + k4.w), qk = (q4.x + q4.y) + (q4.z + q4.w);
                    w[e] = (lane & 4 ? qk : kk) + __shfl_xor_sync(0xffffffffu, lane & 4 ? kk : qk, 4);
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) w[e] += __shfl_xor_sync(0xffffffffu, w[e], 2);
#pragma unroll
                for (int e = 0; e < 2; ++e) w[e] += __shfl_xor_sync(0xffffffffu, w[e], 1);
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (j[e] < d && l8 == 0) sm.x[l][j[e]] = be * dec[e] * w[e];   // (entry 0, the node itself, is never read)
                    if (j[e] < d && l8 == 4 && own) sm.y[l - i0][j[e]] = dec[e] * w[e];
                }
            }
        }
        __syncthreads();
        if (i0 + VS_NODES < i_hi)
            stage_rows(sm.qp[buf ^ 1], q_head + (i0 + VS_NODES) * q_stride, q_stride, min(VS_NODES, i_hi - i0 - VS_NODES), d_k, tid);

        // z by back-substitution: 16 lanes per node, lane ln owning the entries ln, ln + 16, ... ; once z_j is final it is
        // added, times X(up_j, .), to what the entries further up subtract (sums of their own: they are smaller than z, and are
        // rounded as such)
        {
            const int i = tid >> 4, ln = tid & 15, n = i0 + i;
            const int d = i < nn ? sm.depth[n] : 0;
            const int d_warp = __reduce_max_sync(0xffffffffu, d);
            float z[VS_TREE / 16], sub[VS_TREE / 16];
#pragma unroll
            for (int e = 0; e < VS_TREE / 16; ++e) {
                z[e] = ln + 16 * e < d ? sm.y[i][ln + 16 * e] : 0.f;
                sub[e] = 0.f;
            }
#pragma unroll
            for (int e = 0; e < VS_TREE / 16; ++e) {
                if (16 * e >= d_warp - 1) break;
#pragma unroll 1
                for (int l = 0; l < 16; ++l) {
                    const int j = 16 * e + l;
                    if (j >= d_warp - 1) break;
                    const float zj = __shfl_sync(0xffffffffu, z[e] - sub[e], (lane & 16) | l);
                    if (j < d - 1) {
                        const float *xr = sm.x[sm.up[n][j]];
#pragma unroll
                        for (int f = e; f < VS_TREE / 16; ++f) {
                            const int t = ln + 16 * f;
                            if (t > j && t < d) sub[f] = fmaf(zj, xr[t - j], sub[f]);
                        }
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < VS_TREE / 16; ++e) {
                const int t = ln + 16 * e;
                if (t < d) {
                    const int m = sm.up[n][t];
                    const float w = p.scale * (z[e] - sub[e]) * sm.beta[m];
                    sm.y[i][VS_TREE + t] = w;
                    sm.y[i][t] = w * sm.a[m];
                }
            }
        }
        __syncthreads();

        // q' over the q rows, and the v rows' part of the outputs over the weights: 16 lanes per node, eight key positions and
        // eight components each
        {
            const int i = tid >> 4, ln = tid & 15, n = i0 + i;
            if (i < nn) {
                const int d = sm.depth[n];
                const float sa = p.scale * sm.a[n];
                float4 w[2], ov[2], x[2];
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int r = half * 64 + ln * 4;
                    w[half] = ov[half] = x[half] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r < d_k) x[half] = *reinterpret_cast<const float4 *>(&sm.qp[buf][i][r]);
                }
                // (from the root down, q last: the large terms come last)
#pragma unroll 2
                for (int t = d - 1; t >= 0; --t) {
                    const float cf = -sm.y[i][t], cv = sm.y[i][VS_TREE + t];
                    const int m = sm.up[n][t];
                    const float *kr = sm.ks[m], *vr = sm.vs[m];
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const int r = half * 64 + ln * 4;
                        if (r < d_k) {
                            const float4 kt = *reinterpret_cast<const float4 *>(&kr[r]);
                            w[half] = make_float4(fmaf(cf, kt.x, w[half].x), fmaf(cf, kt.y, w[half].y), fmaf(cf, kt.z, w[half].z),
                                                  fmaf(cf, kt.w, w[half].w));
                        }
                        const float4 vt = *reinterpret_cast<const float4 *>(&vr[r]);   // (components beyond d_v are not stored)
                        ov[half] = make_float4(fmaf(cv, vt.x, ov[half].x), fmaf(cv, vt.y, ov[half].y), fmaf(cv, vt.z, ov[half].z),
                                               fmaf(cv, vt.w, ov[half].w));
                    }
                }
#pragma unroll
                for (int half = 0; half < 2; ++half)
                    w[half] = make_float4(fmaf(sa, x[half].x, w[half].x), fmaf(sa, x[half].y, w[half].y), fmaf(sa, x[half].z, w[half].z),
                                          fmaf(sa, x[half].w, w[half].w));
                __syncwarp(0xffffu << (lane & 16));   // the node's weights have been read
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    *reinterpret_cast<float4 *>(&sm.qp[buf][i][half * 64 + ln * 4]) = w[half];
                    *reinterpret_cast<float4 *>(&sm.y[i][half * 64 + ln * 4]) = ov[half];
                }
            }
        }
        __syncthreads();

        // outputs, four nodes at a time: the eight lanes of four rows share key positions and path entries; the sixteen sums
        // (four nodes x four rows) are folded into one another so that lane s ends up with two rows of node s >> 1
#pragma unroll 1
        for (int ib = 0; ib < nn; ib += 4) {
            float acc[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float2 sum[4];   // (of no use from node nn on)
#pragma unroll
                for (int r = 0; r < 4; ++r) sum[r] = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 x = *reinterpret_cast<const float4 *>(&sm.qp[buf][ib + u][32 * j + 4 * s]);
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        sum[r] = __ffma2_rn(sreg[r][2 * j], make_float2(x.x, x.y), sum[r]);
                        sum[r] = __ffma2_rn(sreg[r][2 * j + 1], make_float2(x.z, x.w), sum[r]);
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[u][r] = sum[r].x + sum[r].y;
            }
            const bool b2 = (s & 4) != 0, b1 = (s & 2) != 0, b0 = (s & 1) != 0;
            float f2[2][4], f1[4], out[2];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int r = 0; r < 4; ++r)   // keep nodes 2 (s >> 2) + u
                    f2[u][r] = (b2 ? acc[2 + u][r] : acc[u][r]) + __shfl_xor_sync(0xffffffffu, b2 ? acc[u][r] : acc[2 + u][r], 4);
#pragma unroll
            for (int r = 0; r < 4; ++r) f1[r] = (b1 ? f2[1][r] : f2[0][r]) + __shfl_xor_sync(0xffffffffu, b1 ? f2[0][r] : f2[1][r], 2);
#pragma unroll
            for (int r = 0; r < 2; ++r) out[r] = (b0 ? f1[2 + r] : f1[r]) + __shfl_xor_sync(0xffffffffu, b0 ? f1[r] : f1[2 + r], 1);
            const int i = ib + (s >> 1), c2 = c + 2 * (s & 1);
            if (i < nn) {
                TOut *dst = o + ((size_t)(base + i0 + i) * p.h_v + h) * d_v + c2;
                const float2 ov = *reinterpret_cast<const float2 *>(&sm.y[i][c2]);
                if (c2 < d_v) store_from_float(dst, out[0] + ov.x);
                if (c2 + 1 < d_v) store_from_float(dst + 1, out[1] + ov.y);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();   // the next block's q rows are there; y, zv and this block's q' have been read
    }
}

template <typename TIn, typename TOut>
cudaError_t launch_small_typed(VerifySmallParams p, cudaStream_t stream, LaunchInFront commit)
{
    static PerContext seen;
    int sms = 0;
    cudaError_t e = device_sms(seen, reinterpret_cast<const void *>(verify_generic_small_kernel<TIn, TOut>),
                               sizeof(VerifySmallSmem), &sms);
    if (e == cudaSuccess && commit) e = commit();
    if (e != cudaSuccess) return e;
    // Blocks per CTA: as few as let all CTAs be resident at once, so that small calls spread over the SMs; a CTA reads rows
    // and state once for all of its blocks.  A batch of mixed sizes (mean below two thirds of the largest) stops at three: the last
    // blocks of its few large trees, as CTAs of their own, fill in behind the small trees.  32 heads of 128 components, fp32, 3 / 4
    // blocks per CTA (us): 8 trees of 10..54 nodes 29.1 / 33.5, of 28..61 28.6 / 32.3, 8 more of 9..64 28.4 / 34.7, 12 of 9..64 43.0 /
    // 41.3, 32 of 16..64 111.9 / 104.1; but 8 trees of 64 nodes 49.6 / 38.4, of 50..64 49.5 / 37.1, 9 of 64 53.0 / 38.5, 16 of 64
    // 85.1 / 76.1.
    const int blocks = (p.max_tree_nodes + VS_NODES - 1) / VS_NODES;
    const long long heads = (long long)p.n_seq * p.h_v;
    const bool mixed = 3LL * p.total_nodes < 2LL * p.max_tree_nodes * p.n_seq;
    const int most = mixed ? min(blocks, 3) : blocks;
    int per = 1;
    while (per < most && heads * ((blocks + per - 1) / per) > 2 * sms) ++per;
    p.part_nodes = per * VS_NODES;
    p.n_parts = (blocks + per - 1) / per;
    const long long grid = heads * p.n_parts;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(VS_THREADS);
    cfg.dynamicSmemBytes = sizeof(VerifySmallSmem);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, verify_generic_small_kernel<TIn, TOut>, p);
}

template <typename TIn, typename TOut>
cudaError_t launch_typed(const gdn_shape_t &s, const VerifyGenericParams &p, cudaStream_t stream, LaunchInFront commit)
{
    const int grid = s.n_seq * s.h_v;
    if (grid == 0 || s.total_nodes == 0) return cudaSuccess;
    const size_t smem = sizeof(float) * (2 * VG_CHUNK * VG_DK + 2 * VG_CHUNK * (size_t)s.max_depth + 2 * VG_CHUNK);
    cudaError_t e = cudaFuncSetAttribute(verify_generic_kernel<TIn, TOut>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && commit) e = commit();
    if (e != cudaSuccess) return e;
    verify_generic_kernel<TIn, TOut><<<grid, VG_THREADS, smem, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace

// The grid has (tree, head, block) CTAs whatever the tree sizes: blocks beyond a tree return at once.
bool verify_generic_small_supported(const gdn_shape_t &s)
{
    return s.max_tree_nodes <= VS_TREE &&
           (long long)s.n_seq * s.h_v * ((s.max_tree_nodes + VS_NODES - 1) / VS_NODES) <= 0x7fffffffLL;
}

cudaError_t launch_verify_generic_small(const gdn_shape_t &s, const float *S0, const void *q, const void *k,
                                        const void *v, const void *g, const void *beta, const int32_t *parent,
                                        const int32_t *node_offsets, void *o, int32_t *status_dev, cudaStream_t stream,
                                        LaunchInFront commit)
{
    if (s.n_seq == 0 || s.total_nodes == 0) return cudaSuccess;
    const VerifySmallParams p{s.h_qk, s.h_v, s.d_k, s.d_v, s.max_depth, s.max_tree_nodes, s.total_nodes, s.n_seq,
                              0, 0, s.scale, S0, q, k, v, g, beta, parent,
                              node_offsets, o, status_dev};
    const bool in_bf = s.in_dtype == GDN_BF16, out_bf = s.out_dtype == GDN_BF16;
    if (in_bf && out_bf) return launch_small_typed<__nv_bfloat16, __nv_bfloat16>(p, stream, commit);
    if (in_bf) return launch_small_typed<__nv_bfloat16, float>(p, stream, commit);
    if (out_bf) return launch_small_typed<float, __nv_bfloat16>(p, stream, commit);
    return launch_small_typed<float, float>(p, stream, commit);
}

cudaError_t launch_verify_generic(const gdn_shape_t &s, const float *S0, const void *q, const void *k,
                                  const void *v, const void *g, const void *beta,
                                  const int32_t *node_offsets, void *o, const PlanPtrs &plan,
                                  cudaStream_t stream, LaunchInFront commit)
{
    VerifyGenericParams p{s.h_qk, s.h_v, s.d_k, s.d_v, s.max_depth, s.scale, S0, q, k, v, g, beta,
                          node_offsets, o, plan.tree_ok, plan.depth, plan.anc, plan.utilde};
    const bool in_bf = s.in_dtype == GDN_BF16, out_bf = s.out_dtype == GDN_BF16;
    if (in_bf && out_bf) return launch_typed<__nv_bfloat16, __nv_bfloat16>(s, p, stream, commit);
    if (in_bf) return launch_typed<__nv_bfloat16, float>(s, p, stream, commit);
    if (out_bf) return launch_typed<float, __nv_bfloat16>(s, p, stream, commit);
    return launch_typed<float, float>(s, p, stream, commit);
}

}  // namespace gdn
