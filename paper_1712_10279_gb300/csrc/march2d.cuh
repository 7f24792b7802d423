// Streaming engine, marching form: S iterations of Section 7.2 (vector OMT) in one pass
// over the grid.
//
// A warp owns a strip of 32 columns, one per lane, and marches up a chunk of rows.  Per
// row-step it takes in one row of the state (phi, u_x, u_y, w) and of b, and every stage
// s = 1 .. S advances one row by one iteration: with rows y - s and y - s + 1 of the
// iterate after s - 1 iterations at hand, stage s forms row y - s of the next one.  All
// of it stays in registers: the row above is what the previous stage has just produced,
// 2u' - u of the row below is carried from the previous row-step, and the neighbours
// along x are the neighbouring lanes' (shuffles).  u' is computed once per point and
// stage, and there is no barrier.
//
// The neighbours that a strip and a chunk lack cost redundant work: each stage loses one
// column on either side and one row at either end, so a warp writes 32 - 2 S columns and
// reads S more rows on either side of its chunk.  In return one pass over memory serves S
// iterations: at 2048^2 with three channels a pass of S = 4 moves 0.47 GB in 107 us, 65% of
// the measured copy rate, with three quarters of the issue slots busy (190 instructions per
// point and iteration); with a check every 100 iterations and the layout conversions a
// solve takes 29.4 us per iteration, where one iteration per pass with TMA tiles takes 79
// us and is bound by HBM alone.  1024^2 with one channel 3.9 us (was 9.2), 512^2 with eight
// channels 22 us (118 us: the recomputed shrinks of the one-iteration kernel spill).
//
// Every value is rounded as the one-iteration kernels (or, RES, the resident kernels) round
// it, operation by operation (edges listed in the order of the pairs), so that the
// iterates are theirs bit for bit: after hundreds of iterations w, which is zero except where a difference of phi passes its threshold,
// differs by 1e-5 and more of its norm between two roundings of phi.  The sums over
// channels of the graph gradient reduce to the two channels of a pair (the other terms are
// exact zeros), which keeps its matrix out of the registers.
//
// Rows and columns outside the grid hold finite values that never reach a stored point:
// the differences across the grid's edge are multiplied by 0.
#pragma once

#include <stdint.h>

#include "internal.h"
#include "march2d.h"
#include "pdhg_device.cuh"

namespace vomt {
namespace march {

constexpr int WARPS = 4, NTHR = 32 * WARPS;      // warps per block, each on its own strip and chunk

// Rows in flight per warp (a power of two).  Four cover the latency of HBM (at 2048^2, three
// channels, S = 3, eight rows were no faster); from six channels on a row is 5 KB and more
// and two leave room for a second block on the SM.
__host__ __device__ constexpr int depth(int K) { return K <= 5 ? 4 : 2; }
// Blocks per SM the registers are limited for.
__host__ __device__ constexpr int min_blocks(int K, int S)
{
    return K == 1 ? 6 : (K == 2 ? 4 : (K == 3 ? (S == 4 ? 3 : (S == 2 ? 4 : 5)) : (S == 1 && K <= 5 ? 3 : 2)));
}

__host__ __device__ constexpr int pairs(int K) { return K * (K - 1) / 2; }
__host__ __device__ constexpr int slots(int K) { return pairs(K) > 0 ? pairs(K) : 1; }
// Number of the pair lo < hi of K channels in the order (0,1), (0,2), ..., (1,2), ...
__host__ __device__ constexpr int pair_at(int K, int lo, int hi) { return lo * (2 * K - lo - 1) / 2 + hi - lo - 1; }

// State layout: the groups of four values of a point (phi, u_x, u_y, w, padded with zeros),
// interleaved in blocks of 32 columns, float4 [y][x / 32][group][x % 32]; b likewise.  A
// lane moves four values per access, rows of any length are aligned, and all groups of a
// point sit at fixed distances from one address.  w holds one value per pair of channels
// (pairs without an edge stay zero).
template <int K>
struct Quads {
    static constexpr int NQ = (3 * K + pairs(K) + 3) / 4, NB = (K + 3) / 4;
};
__host__ __device__ inline size_t quad_at(int n, int groups, int y, int x)
{
    return ((size_t)y * ((n + 31) >> 5) + (x >> 5)) * groups * 32 + (x & 31);
}

__device__ __forceinline__ float rsq(float s2)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s2));
    return r;
}

// shrink_2 factor of Appendix B (dev::shrink2_factor) where sums of squares that flush to
// zero are below the squared threshold
__device__ __forceinline__ float factor(float s2, float t) { return fmaxf(1.0f - t * rsq(s2), 0.0f); }

// x x + y y in the two roundings the one-iteration kernels have
__device__ __forceinline__ float sq2(float x, float y) { return __fmaf_rn(x, x, __fmul_rn(y, y)); }

// shrink_u and shrink_w of Section 7.2 on one point, threshold t
template <int K, int UN>
__device__ __forceinline__ void shrink_u(float (&vx)[K], float (&vy)[K], float t)
{
    if (UN == VOMT_U_L12) {
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const float f = factor(sq2(vx[c], vy[c]), t);
            vx[c] *= f;
            vy[c] *= f;
        }
    } else if (UN == VOMT_U_L2) {
        float s2 = 0.0f;
#pragma unroll
        for (int c = 0; c < K; ++c) s2 += sq2(vx[c], vy[c]);
        const float f = factor(s2, t);
#pragma unroll
        for (int c = 0; c < K; ++c) { vx[c] *= f; vy[c] *= f; }
    } else {
#pragma unroll
        for (int c = 0; c < K; ++c) { vx[c] = dev::soft(vx[c], t); vy[c] = dev::soft(vy[c], t); }
    }
}
template <int L, int WN>
__device__ __forceinline__ void shrink_w(float (&x)[L], float t)
{
    if (WN == VOMT_W_L1) {
#pragma unroll
        for (int e = 0; e < L; ++e) x[e] = dev::soft(x[e], t);
    } else {
        float s2 = 0.0f;
#pragma unroll
        for (int e = 0; e < L; ++e) s2 = __fmaf_rn(x[e], x[e], s2);
        const float f = factor(s2, t);
#pragma unroll
        for (int e = 0; e < L; ++e) x[e] *= f;
    }
}

// 16-byte asynchronous copy to shared memory; bytes = 0 writes zeros and reads nothing
__device__ __forceinline__ void copy16(float4 *dst, const float4 *src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One point's values of a row.
template <int K>
struct Row {
    float p[K], x[K], y[K], w[slots(K)], b[K];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int c = 0; c < K; ++c) p[c] = x[c] = y[c] = b[c] = 0.0f;
#pragma unroll
        for (int e = 0; e < slots(K); ++e) w[e] = 0.0f;
    }
    __device__ __forceinline__ void state_from(const float4 *src)      // groups 32 apart
    {
        constexpr int NQ = Quads<K>::NQ;
        float v[4 * NQ];
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const float4 z = src[i * 32];
            v[4 * i] = z.x; v[4 * i + 1] = z.y; v[4 * i + 2] = z.z; v[4 * i + 3] = z.w;
        }
#pragma unroll
        for (int c = 0; c < K; ++c) {
            p[c] = v[c];
            x[c] = v[K + c];
            y[c] = v[2 * K + c];
        }
        w[0] = 0.0f;
#pragma unroll
        for (int e = 0; e < pairs(K); ++e) w[e] = v[3 * K + e];
    }
    __device__ __forceinline__ void b_from(const float4 *src)
    {
        constexpr int NB = Quads<K>::NB;
        float v[4 * NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const float4 z = src[i * 32];
            v[4 * i] = z.x; v[4 * i + 1] = z.y; v[4 * i + 2] = z.z; v[4 * i + 3] = z.w;
        }
#pragma unroll
        for (int c = 0; c < K; ++c) b[c] = v[c];
    }
    __device__ __forceinline__ void state_to(float4 *dst) const
    {
        constexpr int NQ = Quads<K>::NQ;
        float v[4 * NQ];
#pragma unroll
        for (int i = 0; i < 4 * NQ; ++i) v[i] = 0.0f;
#pragma unroll
        for (int c = 0; c < K; ++c) {
            v[c] = p[c];
            v[K + c] = x[c];
            v[2 * K + c] = y[c];
        }
#pragma unroll
        for (int e = 0; e < pairs(K); ++e) v[3 * K + e] = w[e];
#pragma unroll
        for (int i = 0; i < NQ; ++i) dst[i * 32] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
};

// ------------------------------------------------------------------ S iterations
// What warp wi of a pass does.
template <int K, int UN, int WN, int S, bool REG, bool RES>
__device__ __forceinline__ void march_warp(const MarchArgs &a, const MarchOp &g, const int wi)
{
    constexpr int L = slots(K), W = 32 - 2 * S, NQ = Quads<K>::NQ, NB = Quads<K>::NB, D = depth(K);
    constexpr int ROW = (NQ + NB) * 32;
    const int lane = threadIdx.x & 31;
    const int n = g.n;
    const int strip = wi % a.strips, chunk = wi / a.strips;
    const int x = strip * W - S + lane;
    const int y0 = chunk * a.rows, y1 = min(n, y0 + a.rows);
    const int ya = max(y0 - S, 0), yb = y1 + S;          // rows taken in: [ya, yb), zeros from n on
    const bool in = x >= 0 && x < n;
    const bool wr = in && lane >= S && lane < S + W;
    const float g1x = x < n - 1 ? g.g1 : 0.0f, mL = x > 0 ? 1.0f : 0.0f;
    const int xc = min(max(x, 0), n - 1), blk = (n + 31) >> 5;
    const float4 *pin = a.in + quad_at(n, NQ, ya, xc), *pb = a.b + quad_at(n, NB, ya, xc);
    const ptrdiff_t dy = (ptrdiff_t)blk * NQ * 32, dyb = (ptrdiff_t)blk * NB * 32;
    const ptrdiff_t to_out = a.out - a.in, to_prev = a.prev ? a.prev - a.in : 0;

    // Rows arrive by asynchronous copies into a ring of D rows in shared memory, D - 1 rows
    // ahead of their use; a lane reads back only what it copied itself, so waiting for its
    // own copies is all the synchronisation there is.
    extern __shared__ __align__(16) float4 ring_all[];
    float4 *const ring = ring_all + (threadIdx.x >> 5) * (D * ROW) + lane;
    auto fetch = [&](int y) {             // row y, the one pin and pb point at, into its slot
        float4 *dst = ring + (y & (D - 1)) * ROW;
        const uint32_t bytes = y < n && in ? 16u : 0u;
#pragma unroll
        for (int i = 0; i < NQ; ++i) copy16(dst + i * 32, pin + i * 32, bytes);
#pragma unroll
        for (int i = 0; i < NB; ++i) copy16(dst + (NQ + i) * 32, pb + i * 32, bytes);
        copies_commit();
        pin += dy;
        pb += dyb;
    };
#pragma unroll
    for (int q = 0; q < D - 1; ++q) fetch(ya + q);
    if (a.st->stop) {
        copies_wait<0>();
        return;
    }

    Row<K> d[S];                          // row y - s of stage s, waiting for the row above it
    float cy[S][K];                       // 2u'_y - u_y of the row below it
#pragma unroll
    for (int q = 0; q < S; ++q) {
        d[q].zero();
#pragma unroll
        for (int c = 0; c < K; ++c) cy[q][c] = 0.0f;
    }
    // unrolled by two: a row's registers move from stage to stage, and the moves that the
    // rotation costs are paid once per turn of the loop
#pragma unroll 2
    for (int y = ya; y < yb; ++y) {
        fetch(y + D - 1);
        copies_wait<D - 1>();
        Row<K> cur;
        cur.state_from(ring + (y & (D - 1)) * ROW);
        cur.b_from(ring + (y & (D - 1)) * ROW + NQ * 32);
#pragma unroll
        for (int q = 0; q < S; ++q) {
            if (q == S - 1 && S > 1 && a.prev) {
                const int yp = y - (S - 1);
                if (yp >= y0 && yp < y1 && wr) cur.state_to(const_cast<float4 *>(pin) + (to_prev - (D + S - 1) * dy));
            }
            // stage q + 1: row r = y - q - 1 from its values dq and the row above, cur
            Row<K> &dq = d[q];
            const int r = y - q - 1;
            const float g1y = r < n - 1 ? g.g1 : 0.0f, mD = r > 0 ? 1.0f : 0.0f;
            Row<K> o;
            float vx[K], vy[K], ubx[K], div[K];
#pragma unroll
            for (int c = 0; c < K; ++c) {
                const float right = __shfl_down_sync(0xffffffffu, dq.p[c], 1);
                const float sx = g1x * (right - dq.p[c]), sy = g1y * (cur.p[c] - dq.p[c]);
                vx[c] = RES ? fmaf(g.g2, sx, dq.x[c]) : __fadd_rn(dq.x[c], __fmul_rn(g.g2, sx));
                vy[c] = RES ? fmaf(g.g2, sy, dq.y[c]) : __fadd_rn(dq.y[c], __fmul_rn(g.g2, sy));
                if (REG) { vx[c] *= g.su; vy[c] *= g.su; }
            }
            shrink_u<K, UN>(vx, vy, g.tu);
#pragma unroll
            for (int c = 0; c < K; ++c) {
                ubx[c] = 2.0f * vx[c] - dq.x[c];
                const float uby = 2.0f * vy[c] - dq.y[c];
                div[c] = uby - mD * cy[q][c];
                cy[q][c] = uby;
                o.x[c] = vx[c];
                o.y[c] = vy[c];
            }
            float wx[L], rr[K];
            wx[0] = 0.0f;
#pragma unroll
            for (int lo = 0; lo < K; ++lo)
#pragma unroll
                for (int hi = lo + 1; hi < K; ++hi) {
                    const int e = pair_at(K, lo, hi);
                    const float ge = __fmaf_rn(-g.inv[e], dq.p[hi], __fmul_rn(g.inv[e], dq.p[lo]));
                    wx[e] = dq.w[e] + g.nu * ge;
                    if (REG) wx[e] *= g.sw;
                }
            if (K > 1) shrink_w<L, WN>(wx, g.tw);
            float dx[K];
#pragma unroll
            for (int c = 0; c < K; ++c) {
                const float left = __shfl_up_sync(0xffffffffu, ubx[c], 1);
                dx[c] = (ubx[c] - mL * left) + div[c];
                rr[c] = RES ? 0.0f : g.ih * dx[c] + dq.b[c];
            }
#pragma unroll
            for (int lo = 0; lo < K; ++lo)
#pragma unroll
                for (int hi = lo + 1; hi < K; ++hi) {
                    const int e = pair_at(K, lo, hi);
                    const float v = 2.0f * wx[e] - dq.w[e];
                    rr[lo] -= g.inv[e] * v;
                    rr[hi] += g.inv[e] * v;
                }
#pragma unroll
            for (int c = 0; c < K; ++c) {
                if (RES) rr[c] = g.ih * dx[c] + (rr[c] + dq.b[c]);
                o.p[c] = dq.p[c] + g.tau * rr[c];
                o.b[c] = dq.b[c];
            }
#pragma unroll
            for (int e = 0; e < L; ++e) o.w[e] = wx[e];
            dq = cur;
            cur = o;
        }
        const int yo = y - S;
        if (yo >= y0 && yo < y1 && wr) cur.state_to(const_cast<float4 *>(pin) + (to_out - (D + S) * dy));
    }
    copies_wait<0>();
}

template <int K, int UN, int WN, int S, bool REG, bool RES>
__global__ void __launch_bounds__(NTHR, min_blocks(K, S)) k_march(const __grid_constant__ MarchArgs a,
                                                                  const __grid_constant__ MarchOp g)
{
    const int wi = blockIdx.x * WARPS + (threadIdx.x >> 5);
    cudaGridDependencySynchronize();      // after the previous kernel (no-op for a normal launch)
    // the next pass may be scheduled from here on; it waits for this one to finish
    cudaTriggerProgrammaticLaunchCompletion();
    if (wi < a.warps) march_warp<K, UN, WN, S, REG, RES>(a, g, wi);       // whole warps
}

// The same pass over many problems of K channels and any sides (default norms): block q
// works on problem map[q].  state 0 or 1 holds the iterates; prev: state 2 takes the
// iterate before the last.
template <int K, int S>
__global__ void __launch_bounds__(NTHR, min_blocks(K, S)) k_march_many(const BatchItem *__restrict__ items,
                                                                       const int *__restrict__ map, int state, int prev)
{
    const BatchItem &d = items[map[blockIdx.x]];
    constexpr int q = S == 4 ? 2 : S - 1;
    const int wi = ((int)blockIdx.x - d.pass[q].first) * WARPS + (threadIdx.x >> 5);
    MarchArgs a;
    a.in = d.S[state];
    a.out = d.S[state ^ 1];
    a.prev = prev ? d.S[2] : nullptr;
    a.b = d.b;
    a.st = d.st;
    a.rows = d.pass[q].rows;
    a.strips = d.pass[q].strips;
    a.warps = d.pass[q].warps;
    const MarchOp g = d.g;
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    if (wi < a.warps) march_warp<K, VOMT_U_L12, VOMT_W_L1, S, false, true>(a, g, wi);
}

// ------------------------------------------------------------------ one check
// The terms of a convergence check (the sums RED_*) of the iterate cur and its
// predecessor prv.  The same march: both states' rows once, neighbours along x by
// shuffles, the row below carried; strips write no columns, so a strip covers 30.  Sums
// per thread and warp in pairs of FP32 numbers (CheckAcc), per block and grid in FP64; the
// constraint residual, which cancels several digits, as a pair too (residual_pair), where the
// one-iteration kernels form it in FP64.
// About 15 us at 1024^2 with one channel, bound by the latency of a row's loads; loading
// a row ahead costs more in resident warps than it hides (19 us).
template <int K, int UN, int WN>
__device__ __forceinline__ void check_block(const CheckArgs &a, const MarchOp &g, const int block, const int blocks)
{
    constexpr int NQ = Quads<K>::NQ, NB = Quads<K>::NB;
    const int lane = threadIdx.x & 31, n = g.n;
    const float ih = g.ih, alpha = g.alpha;
    dev::CheckAcc acc;
    acc.zero();
    for (int wi = block * WARPS + (threadIdx.x >> 5); wi < a.items; wi += blocks * WARPS) {
        const int strip = wi % a.strips, chunk = wi / a.strips;
        const int x = strip * 30 - 1 + lane;
        const int y0 = chunk * a.rows, y1 = min(n, y0 + a.rows);
        const bool in = x >= 0 && x < n, own = in && lane >= 1 && lane < 31;
        const float ihx = x < n - 1 ? ih : 0.0f, mL = x > 0 ? 1.0f : 0.0f;
        const int xc = min(max(x, 0), n - 1);
        Row<K> c0, p0;                    // row y of cur and prv
        float dn[K], un_[K];              // u_y and u_y - its predecessor of the row below
        const int yl = max(y0 - 1, 0);
        c0.state_from(a.cur + quad_at(n, NQ, yl, xc));
        p0.state_from(a.prv + quad_at(n, NQ, yl, xc));
#pragma unroll
        for (int c = 0; c < K; ++c) {
            un_[c] = y0 > 0 ? c0.y[c] : 0.0f;
            dn[c] = y0 > 0 ? c0.y[c] - p0.y[c] : 0.0f;
        }
        if (y0 > 0) {
            c0.state_from(a.cur + quad_at(n, NQ, y0, xc));
            p0.state_from(a.prv + quad_at(n, NQ, y0, xc));
        }
        for (int y = y0; y < y1; ++y) {
            Row<K> c1, p1;                // the row above
            const int yu = min(y + 1, n - 1);
            c1.state_from(a.cur + quad_at(n, NQ, yu, xc));
            p1.state_from(a.prv + quad_at(n, NQ, yu, xc));
            c0.b_from(a.b + quad_at(n, NB, y, xc));
            const float ihy = y < n - 1 ? ih : 0.0f;
            float dph[K], ddiv[K], gwb[K], uxs[K], uxl[K], dnn[K], unn[K];
            float nu_pt = 0.0f, dn_u = 0.0f, fdu = 0.0f, fdp = 0.0f, fd = 0.0f, fbb = 0.0f, fdw = 0.0f, fx = 0.0f;
            float q2 = 0.0f, dist = 0.0f;
#pragma unroll
            for (int c = 0; c < K; ++c) {
                const float uxc = c0.x[c], uyc = c0.y[c], bc = c0.b[c], ph = c0.p[c];
                const float dux = uxc - p0.x[c], duy = uyc - p0.y[c];
                uxs[c] = uxc;
                uxl[c] = mL * __shfl_up_sync(0xffffffffu, uxc, 1);
                const float dxl = mL * __shfl_up_sync(0xffffffffu, dux, 1);
                const float pr = __shfl_down_sync(0xffffffffu, ph, 1);
                ddiv[c] = ih * ((dux - dxl) + (duy - dn[c]));
                dnn[c] = duy;
                unn[c] = uyc;
                dph[c] = ph - p0.p[c];
                gwb[c] = bc;
                fdu += dux * dux + duy * duy;
                fdp += dph[c] * dph[c];
                fd += ph * bc;
                fbb += bc * bc;
                q2 += uxc * uxc + uyc * uyc;
                const float gx = ihx > 0.0f ? ih * (pr - ph) : 0.0f, gy = ihy > 0.0f ? ih * (c1.p[c] - ph) : 0.0f;
                if (UN == VOMT_U_L12) {
                    nu_pt += sqrtf(uxc * uxc + uyc * uyc);
                    const float gn = sqrtf(gx * gx + gy * gy), o = fmaxf(gn - 1.0f, 0.0f);
                    dn_u = fmaxf(dn_u, gn);
                    dist += o * o;
                } else if (UN == VOMT_U_L2) {
                    nu_pt += uxc * uxc + uyc * uyc;
                    dn_u += gx * gx + gy * gy;
                } else {
                    nu_pt += fabsf(uxc) + fabsf(uyc);
                    dn_u = fmaxf(dn_u, fmaxf(fabsf(gx), fabsf(gy)));
                    const float ox = fmaxf(fabsf(gx) - 1.0f, 0.0f), oy = fmaxf(fabsf(gy) - 1.0f, 0.0f);
                    dist += ox * ox + oy * oy;
                }
            }
            if (UN == VOMT_U_L2) {
                nu_pt = sqrtf(nu_pt);
                dn_u = sqrtf(dn_u);
                const float o = fmaxf(dn_u - 1.0f, 0.0f);
                dist += o * o;
            }
            float nw_pt = 0.0f, dn_w = 0.0f;
#pragma unroll
            for (int lo = 0; lo < K; ++lo)
#pragma unroll
                for (int hi = lo + 1; hi < K; ++hi) {
                    const int e = pair_at(K, lo, hi);
                    const float we = c0.w[e], dwe = we - p0.w[e], ge = g.inv[e] * (c0.p[lo] - c0.p[hi]);
                    fdw += dwe * dwe;
                    q2 += we * we;
                    gwb[lo] -= g.inv[e] * we;
                    gwb[hi] += g.inv[e] * we;
                    ddiv[lo] -= g.inv[e] * dwe;
                    ddiv[hi] += g.inv[e] * dwe;
                    if (WN == VOMT_W_L1) {
                        nw_pt += fabsf(we);
                        dn_w = fmaxf(dn_w, fabsf(ge));
                        const float o = fmaxf(fabsf(ge) - alpha, 0.0f);
                        dist += o * o;
                    } else {
                        nw_pt += we * we;
                        dn_w += ge * ge;
                    }
                }
            if (WN == VOMT_W_L2) {
                nw_pt = sqrtf(nw_pt);
                dn_w = sqrtf(dn_w);
                const float o = fmaxf(dn_w - alpha, 0.0f);
                if (g.l > 0) dist += o * o;
            }
#pragma unroll
            for (int c = 0; c < K; ++c) {
                float lo;
                const float rc = dev::residual_pair(ih, uxs[c], uxl[c], unn[c], un_[c], gwb[c], lo);
                if (own) acc.add_square(RED_RR, rc, lo);
                fx += dph[c] * ddiv[c];
                un_[c] = unn[c];
                dn[c] = dnn[c];
            }
            if (own) {
                acc.add(RED_P, nu_pt + alpha * nw_pt);
                if (g.reg) {
                    acc.add(RED_P, g.eps * q2);
                    acc.add(RED_DIST, dist);
                }
                acc.add(RED_D, fd);
                acc.add(RED_BB, fbb);
                acc.add(RED_DU, fdu);
                acc.add(RED_DW, fdw);
                acc.add(RED_DP, fdp);
                acc.add(RED_X, fx);
                float di = fmaxf(dn_u - 1.0f, 0.0f);
                if (g.l > 0) di = fmaxf(di, dn_w - alpha);
                acc.max(RED_MAX, di);
            }
            c0 = c1;
            p0 = p1;
        }
    }
    dev::block_sum_store<NTHR>(acc, a.partials + (size_t)block * NRED);
}

template <int K, int UN, int WN>
__global__ void __launch_bounds__(NTHR) k_march_check(const __grid_constant__ CheckArgs a,
                                                      const __grid_constant__ MarchOp g)
{
    cudaGridDependencySynchronize();
    if (a.st->stop) return;
    check_block<K, UN, WN>(a, g, (int)blockIdx.x, (int)gridDim.x);
}

// many problems: map[block] is the block's problem; cur, prv: which states
template <int K>
__global__ void __launch_bounds__(NTHR) k_check_many(const BatchItem *__restrict__ items, const int *__restrict__ map,
                                                     int cur, int prv)
{
    const BatchItem &d = items[map[blockIdx.x]];
    CheckArgs a;
    a.cur = d.S[cur];
    a.prv = d.S[prv];
    a.b = d.b;
    a.partials = d.partials;
    a.rows = d.check_rows;
    a.strips = d.check_strips;
    a.items = d.check_items;
    const MarchOp g = d.g;
    const int block = (int)blockIdx.x - d.check_first, blocks = d.check_blocks;
    cudaGridDependencySynchronize();
    if (d.st->stop) return;
    check_block<K, VOMT_U_L12, VOMT_W_L1>(a, g, block, blocks);
}

// ------------------------------------------------------------------ layouts
// Planar fields <-> the engine's layout; b = rho1 - rho0.
template <int K>
__device__ __forceinline__ void layout_in(const PlanarArgs &a, const MarchOp &g, float4 *state, float4 *bq)
{
    const int n = g.n;
    const size_t nn = (size_t)n * n;
    for (int y = blockIdx.y; y < n; y += gridDim.y) {
        const int x = blockIdx.x * blockDim.x + threadIdx.x;
        if (x >= n) continue;
        const size_t q = (size_t)y * n + x;
        Row<K> r;
        r.zero();
#pragma unroll
        for (int c = 0; c < K; ++c) {
            r.b[c] = a.rho1[c * nn + q] - a.rho0[c * nn + q];
            if (a.warm) {
                r.p[c] = a.phi[c * nn + q];
                r.x[c] = x < n - 1 ? a.u[c * nn + q] : 0.0f;
                r.y[c] = y < n - 1 ? a.u[(K + c) * nn + q] : 0.0f;
            }
        }
        if (a.warm)
#pragma unroll
            for (int e = 0; e < pairs(K); ++e)
                if (g.edge[e] >= 0) r.w[e] = a.w[g.edge[e] * nn + q];
        r.state_to(state + quad_at(n, Quads<K>::NQ, y, x));
        float v[4 * Quads<K>::NB];
#pragma unroll
        for (int c = 0; c < 4 * Quads<K>::NB; ++c) v[c] = c < K ? r.b[c < K ? c : 0] : 0.0f;
        float4 *dst = bq + quad_at(n, Quads<K>::NB, y, x);
#pragma unroll
        for (int i = 0; i < Quads<K>::NB; ++i)
            dst[i * 32] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
}

template <int K>
__global__ void k_march_in(const __grid_constant__ PlanarArgs a, const __grid_constant__ MarchOp g, float4 *state,
                           float4 *bq)
{
    layout_in<K>(a, g, state, bq);
}
template <int K>
__global__ void k_in_many(const BatchItem *__restrict__ items)
{
    const BatchItem &d = items[blockIdx.z];
    layout_in<K>(d.planar, d.g, d.S[0], d.b);
}

template <int K>
__device__ __forceinline__ void layout_out(const PlanarArgs &a, const MarchOp &g, const float4 *state)
{
    const int n = g.n;
    const size_t nn = (size_t)n * n;
    for (int y = blockIdx.y; y < n; y += gridDim.y) {
        const int x = blockIdx.x * blockDim.x + threadIdx.x;
        if (x >= n) continue;
        const size_t q = (size_t)y * n + x;
        Row<K> r;
        r.state_from(state + quad_at(n, Quads<K>::NQ, y, x));
#pragma unroll
        for (int c = 0; c < K; ++c) {
            a.phi[c * nn + q] = r.p[c];
            a.u[c * nn + q] = r.x[c];
            a.u[(K + c) * nn + q] = r.y[c];
        }
#pragma unroll
        for (int e = 0; e < pairs(K); ++e)
            if (g.edge[e] >= 0) a.w[g.edge[e] * nn + q] = r.w[e];
    }
}

template <int K>
__global__ void k_march_out(const __grid_constant__ PlanarArgs a, const __grid_constant__ MarchOp g,
                            const float4 *s0, const float4 *s1, const DevStatus *st)
{
    layout_out<K>(a, g, st->slot ? s1 : s0);
}
template <int K>
__global__ void k_out_many(const BatchItem *__restrict__ items)
{
    const BatchItem &d = items[blockIdx.z];
    layout_out<K>(d.planar, d.g, d.S[d.st->slot ? 1 : 0]);
}

// ------------------------------------------------------------------ dispatch
template <int K, int UN, int WN, bool REG, bool RES = false>
Kernels kernels_of()
{
    Kernels q = {};
    q.step[0] = k_march<K, UN, WN, 1, REG, RES>;
    if constexpr (K <= 6) q.step[1] = k_march<K, UN, WN, 2, REG, RES>;
    if constexpr (K <= 3) q.step[2] = k_march<K, UN, WN, 4, REG, RES>;
    if constexpr (RES && K <= 5) {
        q.many[0] = k_march_many<K, 1>;
        q.many[1] = k_march_many<K, 2>;
        if constexpr (K <= 3) q.many[2] = k_march_many<K, 4>;
        q.check_many = k_check_many<K>;
        q.in_many = k_in_many<K>;
        q.out_many = k_out_many<K>;
    }
    q.check = k_march_check<K, UN, WN>;
    q.in = k_march_in<K>;
    q.out = k_march_out<K>;
    q.groups = Quads<K>::NQ;
    q.bgroups = Quads<K>::NB;
    q.smem = depth(K) * (Quads<K>::NQ + Quads<K>::NB) * 512 * WARPS;
    return q;
}

// The plain problem with the default norms has its own kernels; every other one takes
// those with the regularisation's factors (1 without it).
template <int K>
Kernels pick_norms(int un, int wn, bool reg, bool res)
{
    if (K == 1) wn = VOMT_W_L1;           // no edges
    if (res) return kernels_of<K, 0, 0, false, true>();      // default norms, eps = 0 only (run_engine)
    if (un == VOMT_U_L12 && wn == VOMT_W_L1) return reg ? kernels_of<K, 0, 0, true>() : kernels_of<K, 0, 0, false>();
    if constexpr (K > 1) {
        if (wn == VOMT_W_L2)
            return un == VOMT_U_L12 ? kernels_of<K, 0, 1, true>()
                                    : (un == VOMT_U_L2 ? kernels_of<K, 1, 1, true>() : kernels_of<K, 2, 1, true>());
    }
    return un == VOMT_U_L2 ? kernels_of<K, 1, 0, true>() : kernels_of<K, 2, 0, true>();
}

}  // namespace march
}  // namespace vomt
