// The commit (Eq. 7 along an accepted path, the delayed commit of Section 3.4) on a 128 x 128 fp32 state tile taken
// through registers as accumulator fragments of the warp-level tensor-core instruction m16n8k16, so that both halves of
// the work -- the products k_t.s of every step with the old state, and the rank-L update -- are matrix products on the
// registers as they are.  Against the step-by-step replay (gdn_replay.cuh) the work per tile grows little with the length of
// the path, and a tile needs 32 registers per thread instead of 64, so that four share an SM instead of two: 1536 tiles, path of
// 1 / 7 / 12 / 16: 38.0 / 40.6 / 54.3 / 55.7 us against 37.7 / 46.9 / 57.4 / 64.2.
//
// Thread layout: a warp owns 16 rows (rows = value components, contiguous in memory along the key dimension), taken in
// four chunks of 32 key positions; lane = 4 g + l4 holds of rows g and g + 8 the key positions 32 jj + 8 l4 + e (e = 0..7)
// of chunk jj: x[e >> 1][2 r + (e & 1)] for row g + 8 r, i.e. 32 contiguous bytes per lane and row.  As a fragment, x[n]
// is the n-th 16 x 8 tile of the chunk in a permuted column order (column 2 l4 + (e & 1) of tile e >> 1); the other operand
// of every product, the path's k rows in shared memory, is stored in that order (path_row_word).
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "gdn_replay.cuh"

namespace gdn {

constexpr int GDN_PK_STRIDE = 272;   // bytes from one path row to the next: eight rows of a 16-byte column hit all banks once

// Byte place of 4-byte word `w` (0..63) of a k row in the permuted order.
__device__ __forceinline__ uint32_t path_row_word(int w) { return (uint32_t)((w & ~15) + (w & 3) * 4 + ((w >> 2) & 3)) * 4u; }

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_1688(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ uint32_t pack_bf16_pair(float2 x)
{
    __nv_bfloat162 t = __floats2bfloat162_rn(x.x, x.y);
    return *reinterpret_cast<uint32_t *>(&t);
}
// x minus the bf16 pair h, two values at a time (exact)
__device__ __forceinline__ float2 bf16_rest(float2 x, uint32_t h)
{
    return make_float2(x.x - __uint_as_float(h << 16), x.y - __uint_as_float(h & 0xFFFF0000u));
}
// x = hi + mid + lo in three bf16 terms (|x - hi - mid - lo| <= 2^-26 |x|: fp32 precision), two values at a time
__device__ __forceinline__ void split3_bf16(float x0, float x1, uint32_t &hi, uint32_t &mid, uint32_t &lo)
{
    float2 x = make_float2(x0, x1);
    hi = pack_bf16_pair(x);
    x = bf16_rest(x, hi);
    mid = pack_bf16_pair(x);
    lo = pack_bf16_pair(bf16_rest(x, mid));
}

// One chunk of a warp's 16 rows: global memory <-> fragments.  src: this lane's first row at its first key position.
__device__ __forceinline__ void load_chunk(const float *src, int jj, float (&x)[4][4])
{
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        float4 a, b;
        ldg_v8(src + r * 8 * GDN_TILE_D + jj * 32, a, b);
        x[0][2 * r] = a.x; x[0][2 * r + 1] = a.y; x[1][2 * r] = a.z; x[1][2 * r + 1] = a.w;
        x[2][2 * r] = b.x; x[2][2 * r + 1] = b.y; x[3][2 * r] = b.z; x[3][2 * r + 1] = b.w;
    }
}
__device__ __forceinline__ void store_chunk(float *dst, int jj, const float (&x)[4][4])
{
#pragma unroll
    for (int r = 0; r < 2; ++r)
        stg_v8(dst + r * 8 * GDN_TILE_D + jj * 32, make_float4(x[0][2 * r], x[0][2 * r + 1], x[1][2 * r], x[1][2 * r + 1]),
               make_float4(x[2][2 * r], x[2][2 * r + 1], x[3][2 * r], x[3][2 * r + 1]));
}

// An accepted path in shared memory: k rows in the permuted order (zero up to the next multiple of eight rows), v rows
// bf16 [..][128], and per step t: scal (beta_t, beta_t A_t, E_t, .) with A_t = exp(sum of g up to and including step t), E_t =
// exp(sum of g behind step t); coupling[u][t] = beta_t exp(sum of g behind step u up to and including t) k_t.k_u for t > u, 0
// otherwise (row stride 16).  Every sum runs over just the steps it names: as a difference of two sums from the root it would
// lose the weak decays behind a strong one (-3000 on the path: 1.2e-4 off), and be no number behind g = -inf (alpha = 0).
struct PathTile {
    const uint16_t *pv;
    const float4 *scal;
    const float *coupling;
};

// S <- S after L steps (1 <= L <= 16).  With u_t = beta_t (v_t - A_t k_t.S) - sum_{u < t} coupling_ut u_u (the triangular
// form of Section 3.4.1 on the path alone), S_L = A_L S + sum_t E_t u_t k_t^T; every decay factor is in 0..1 whatever the
// decays.  The products run on bf16 operands that are exact (k) or three-term splits (S, E u), i.e.
// at fp32 precision; what is left of an error comes from the tensor core, which cuts off what it adds to an accumulator, and is
// kept below that of the replay by short sums that meet one another with ordinary roundings (gdn_commit.cu has both errors).
// The tile passes through the registers twice: once for the products, once for the update.
// TILES: 8-step tiles of the path, 1 for L <= 8, 2 otherwise (code of their own: 64 registers are few).
template <int TILES> struct PathProducts {     // steps 2 l4, 2 l4 + 1 (+ 8 in the second entry) of rows g (entries 0, 1) and g + 8 (2, 3)
    float z[TILES][4], rest[TILES][4];   // the mid and lo terms go to accumulators of their own (shorter chains)
};
__device__ __forceinline__ uint32_t path_operand(uint32_t pk, int lane)
{
    return pk + (uint32_t)(lane & 7) * GDN_PK_STRIDE + (uint32_t)(lane >> 3) * 16;
}
template <int TILES>
__device__ __forceinline__ void path_products_chunk(const float (&x)[4][4], int jj, uint32_t operand, PathProducts<TILES> &a)
{
    uint32_t b[TILES][4];
#pragma unroll
    for (int i = 0; i < TILES; ++i) ldmatrix_x4(operand + i * 8 * GDN_PK_STRIDE + jj * 64, b[i]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t hi[4], mid[4], lo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) split3_bf16(x[2 * h + (i >> 1)][2 * (i & 1)], x[2 * h + (i >> 1)][2 * (i & 1) + 1], hi[i], mid[i], lo[i]);
#pragma unroll
        for (int i = 0; i < TILES; ++i) {
            mma_16816(a.z[i], hi, b[i][2 * h], b[i][2 * h + 1]);
            mma_16816(a.rest[i], mid, b[i][2 * h], b[i][2 * h + 1]);
            mma_16816(a.rest[i], lo, b[i][2 * h], b[i][2 * h + 1]);
        }
    }
}
// products -> E_t u_t in three bf16 terms, the other operand of the update.  row: this lane's first row
template <int TILES> struct PathUpdate { uint32_t hi[2 * TILES], mid[2 * TILES], lo[2 * TILES]; };
template <int TILES>
__device__ __forceinline__ void path_solve(PathProducts<TILES> &a, int L, const PathTile &p, int row, int lane, PathUpdate<TILES> &u)
{
    const int l4 = lane & 3;
    float (&z)[TILES][4] = a.z, (&sum)[TILES][4] = a.rest;
#pragma unroll
    for (int i = 0; i < TILES; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int t = 8 * i + 2 * l4 + e;
            const bool on = t < L;
            const float4 sc = on ? p.scal[t] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float v = on ? __uint_as_float((uint32_t)p.pv[t * GDN_TILE_D + row + 8 * r] << 16) : 0.f;
                z[i][2 * r + e] = on ? fmaf(-sc.y, z[i][2 * r + e] + a.rest[i][2 * r + e], sc.x * v) : 0.f;
                sum[i][2 * r + e] = 0.f;
            }
        }
    // forward substitution: once u_t is final its four lanes add its share to the sums that the later steps subtract (coupling
    // is zero for the others); the sums are much smaller than u, and are rounded as such
#pragma unroll
    for (int k = 0; k < TILES; ++k)   // steps of tile k, which later ones of it and of the tiles behind it depend on
#pragma unroll 1
        for (int t = 8 * k; t < min(L - 1, 8 * k + 8); ++t) {
            const int src = (lane & ~3) | ((t & 7) >> 1);
            const bool odd = (t & 1) != 0;
            const float u0 = __shfl_sync(0xffffffffu, odd ? z[k][1] - sum[k][1] : z[k][0] - sum[k][0], src);
            const float u1 = __shfl_sync(0xffffffffu, odd ? z[k][3] - sum[k][3] : z[k][2] - sum[k][2], src);
#pragma unroll
            for (int i = k; i < TILES; ++i) {
                const float2 c = *reinterpret_cast<const float2 *>(p.coupling + t * 16 + 8 * i + 2 * l4);
                sum[i][0] = fmaf(c.x, u0, sum[i][0]); sum[i][1] = fmaf(c.y, u0, sum[i][1]);
                sum[i][2] = fmaf(c.x, u1, sum[i][2]); sum[i][3] = fmaf(c.y, u1, sum[i][3]);
            }
        }
#pragma unroll
    for (int i = 0; i < TILES; ++i) {
        const int t = 8 * i + 2 * l4;
        const float e0 = t < L ? p.scal[t].z : 0.f, e1 = t + 1 < L ? p.scal[t + 1].z : 0.f;
#pragma unroll
        for (int r = 0; r < 2; ++r)
            split3_bf16(t < L ? e0 * (z[i][2 * r] - sum[i][2 * r]) : 0.f, t + 1 < L ? e1 * (z[i][2 * r + 1] - sum[i][2 * r + 1]) : 0.f,
                        u.hi[2 * i + r], u.mid[2 * i + r], u.lo[2 * i + r]);
    }
}
// x <- A_L x + sum_t (E_t u_t) k_t^T, eight steps at a time.  The products of the hi terms have an accumulator of their own, those
// of the mid and lo terms another; both meet the state with ordinary roundings, the large one last (the tensor core cuts off
// what it adds).
template <int TILES>
__device__ __forceinline__ void path_update_chunk(float (&x)[4][4], int jj, uint32_t operand, float A_L, const PathUpdate<TILES> &u)
{
#pragma unroll
    for (int i = 0; i < TILES; ++i) {
        uint32_t b[4];
        ldmatrix_x4_trans(operand + i * 8 * GDN_PK_STRIDE + jj * 64, b);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float hi[4], rest[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) hi[e] = rest[e] = 0.f;
            mma_1688(rest, u.lo[2 * i], u.lo[2 * i + 1], b[q]);
            mma_1688(hi, u.hi[2 * i], u.hi[2 * i + 1], b[q]);
            mma_1688(rest, u.mid[2 * i], u.mid[2 * i + 1], b[q]);
#pragma unroll
            for (int e = 0; e < 4; ++e) x[q][e] = hi[e] + (i == 0 ? fmaf(A_L, x[q][e], rest[e]) : x[q][e] + rest[e]);
        }
    }
}

// Sums of g over runs of steps, by one warp whose lane t holds g of step t (0 beyond the path): w[j] is the sum of the 2^j
// steps up to and including step t.
struct DecayWindows {
    float w[4];
    __device__ __forceinline__ explicit DecayWindows(float g)
    {
        w[0] = g;
#pragma unroll
        for (int j = 1; j < 4; ++j) w[j] = w[j - 1] + __shfl_up_sync(0xffffffffu, w[j - 1], 1 << (j - 1));
    }
    // the n steps up to and including step t (0 <= n <= 15, n <= t + 1; all lanes call)
    __device__ __forceinline__ float sum(int t, int n) const
    {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float x = __shfl_sync(0xffffffffu, w[j], t);
            if ((n >> j) & 1) {
                s += x;
                t -= 1 << j;
            }
        }
        return s;
    }
};

// The coupling table of a path whose k rows are in shared memory, by one warp (lane t: g_t, beta_t of step t; rows beyond
// L up to the next multiple of eight are zero).
__device__ __forceinline__ void path_coupling(uint32_t pk, int L, float g_t, float beta, float *coupling, int lane)
{
    const int g = lane >> 2, l4 = lane & 3;
    const bool two = L > 8;
    float k[2][2][4];   // [parity of the chunk][tile of u]: k_t.k_u, rows t = g (entries 0, 1) and g + 8 (2, 3)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) k[0][i][e] = k[1][i][e] = 0.f;
    const int half = (lane >> 3) & 1;   // ldmatrix: matrices (rows 0-7, chunk c), (rows 8-15, c), (rows 0-7, c + 1), (rows 8-15, c + 1)
    const uint32_t addr = pk + (uint32_t)((lane & 7) + (two ? 8 * half : 0)) * GDN_PK_STRIDE + (uint32_t)(lane >> 4) * 16;
#pragma unroll 2
    for (int c = 0; c < 8; ++c) {
        uint32_t a[4];
        ldmatrix_x4(addr + c * 32, a);
        mma_16816(k[c & 1][0], a, a[0], a[2]);
        if (two) mma_16816(k[c & 1][1], a, a[1], a[3]);
    }
    const DecayWindows windows(g_t);
#pragma unroll
    for (int r = 0; r < 2; ++r) {   // t = g + 8 r
        if (r == 1 && !two) break;
        const int t = g + 8 * r;
        const float bt = __shfl_sync(0xffffffffu, beta, t);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int u = 8 * i + 2 * l4;   // ... and u + 1
            float d0 = 0.f, d1 = 0.f;   // decays behind u, behind u + 1
            if (i <= r) {               // (otherwise t < u)
                const float near = windows.sum(t, max(t - u - 1, 0));
                d0 = expf(near + __shfl_sync(0xffffffffu, g_t, u + 1));
                d1 = expf(near);
            }
            if (!two && i == 1) continue;
            if (u < L) coupling[u * 16 + t] = t > u && t < L ? bt * d0 * (k[0][i][2 * r] + k[1][i][2 * r]) : 0.f;
            if (u + 1 < L) coupling[(u + 1) * 16 + t] = t > u + 1 && t < L ? bt * d1 * (k[0][i][2 * r + 1] + k[1][i][2 * r + 1]) : 0.f;
        }
    }
}

}  // namespace gdn
