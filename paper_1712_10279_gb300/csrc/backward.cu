// Gradients of the vector-OMT cost.
//
// Envelope gradient.  V(rho0, rho1) is the value of the dual problem (eq.
// vomt-dual): a maximum over a feasible set that does not depend on the
// densities of the linear function <phi, rho1 - rho0>.  At a solution phi*,
// dV/drho1 = phi* and dV/drho0 = -phi*, up to the constant the dual leaves free
// (grad and grad_G vanish on a constant shared by all channels), fixed here by
// making phi* zero-mean.  V is also the value of the primal (eq. vomt), linear
// in alpha for fixed (u, w), so dV/dalpha = sum_ij ||w*_ij||_w.  A cluster of
// blocks per problem: the mean, then the scaled, centred copy.
//
// Unrolled gradient.  J_T = P(u^T, w^T), the primal objective after T
// iterations of Section 7.2 from the zero iterate, is differentiated by reverse
// mode through the T iterations.  The forward pass keeps every iterate where that
// takes no more than the context's memory limit, else one every `ckpt` iterations, from
// which the reverse pass recomputes a segment at a time; the reverse pass applies the transposed Jacobian of
// one iteration per step (k_adj_step; at 256^2, three channels, 4.6 us a step, 15 us
// marching two rows per warp, and 2.9 us a forward step): the chain rule through phi' = phi + tau(div_x ubar + div_G wbar +
// rho1 - rho0), through u' = shrink(u + mu grad phi; mu) and through
// w' = shrink_w(w + nu grad_G phi; alpha nu), with div_x^T = -grad_x
// (Appendix A) and div_G = -grad_G^* (Section 3.1).
#include <math.h>
#include <string.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "internal.h"
#include "march2d.h"
#include "pdhg_device.cuh"

namespace vomt {
namespace {

constexpr int AX = 32, AY = 8, AT = AX * AY;

// Most blocks of a problem's cluster; a warp takes whole rows.  The sums meet through
// distributed shared memory, so the call needs no scratch and calls on several streams do not
// disturb each other.
constexpr int kEnvCluster = 8;

// This block's sums of phi and of ||w|| (L1; Sum: TripleSum, or WideSum where that overflows),
// then the cluster's: totals[0], totals[1], the same in every thread.  The squares of the
// joint norm and their root are FP64.
template <typename Sum>
__device__ __forceinline__ void envelope_totals(cooperative_groups::cluster_group &cluster, int n, int pitch, int k, int l,
                                                int wn, const float *P, const float *Wb, int first, int step,
                                                double (&totals)[2])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const size_t pw = (size_t)n * pitch;
    Sum s, sw;
    double joint = 0.0;
    for (int r = first; r < k * n; r += step) {
        const float *row = P + (size_t)r * pitch;
#pragma unroll 4
        for (int i = lane; i < n; i += 32) s.add(row[i]);
    }
    if (l > 0) {
        for (int r = first; r < n; r += step) {
            const float *row = Wb + (size_t)r * pitch;
            if (wn == VOMT_W_L1) {
                for (int e = 0; e < l; ++e)
#pragma unroll 4
                    for (int i = lane; i < n; i += 32) sw.add(fabsf(row[e * pw + i]));
            } else {
                for (int i = lane; i < n; i += 32) {
                    double a = 0.0;
                    for (int e = 0; e < l; ++e) {
                        const double x = row[e * pw + i];
                        a += x * x;
                    }
                    joint += sqrt(a);
                }
            }
        }
    }
    // warps, blocks, cluster: kept in Sum's form all the way
    __shared__ uint32_t sh[32][2][3], block[2][3];
    __shared__ double joints[32], block_joint, out[2];
    s.warp();
    sw.warp();
    if (wn != VOMT_W_L1)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) joint += __shfl_down_sync(0xffffffffu, joint, off);
    if (lane == 0) {
        s.save(sh[wid][0]);
        sw.save(sh[wid][1]);
        joints[wid] = joint;
    }
    __syncthreads();
    if (wid < 2) {                        // warp 0: phi, warp 1: w
        Sum t;
        if (lane < warps) t.merge(sh[lane][wid]);
        t.warp();
        if (lane == 0) t.save(block[wid]);
    } else if (threadIdx.x == 64) {
        double t = 0.0;
        for (int q = 0; q < warps; ++q) t += joints[q];
        block_joint = t;
    }
    cluster.sync();
    if (threadIdx.x < 2) {
        Sum t;
        double j = 0.0;
        for (int q = 0; q < (int)cluster.num_blocks(); ++q) {
            t.merge(cluster.map_shared_rank(&block[threadIdx.x][0], q));
            if (threadIdx.x == 1) j += *cluster.map_shared_rank(&block_joint, q);
        }
        out[threadIdx.x] = t.value() + j;
    }
    __syncthreads();
    totals[0] = out[0];
    totals[1] = out[1];
    cluster.sync();                       // no block leaves, or sums again, while another reads its sums
}

// A cluster of one to kEnvCluster blocks per problem (vomt_backward).  Bound by the latency of
// two passes over a problem.
__global__ void __launch_bounds__(1024) k_envelope(int n, int pitch, int k, int l, int wn, const float *__restrict__ phi,
                                                   const float *__restrict__ w, const float *__restrict__ gscale,
                                                   float *__restrict__ d_rho0, float *__restrict__ d_rho1,
                                                   float *__restrict__ d_alpha)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int blocks = (int)cluster.num_blocks(), problem = blockIdx.x / blocks, rank = blockIdx.x % blocks;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int first = rank * warps + wid, step = blocks * warps;      // this warp's rows
    const size_t pw = (size_t)n * pitch, pcnt = (size_t)k * pw;
    const float *P = phi + problem * pcnt, *Wb = w + problem * (size_t)l * pw;
    double totals[2];
    envelope_totals<dev::TripleSum>(cluster, n, pitch, k, l, wn, P, Wb, first, step, totals);
    if (!isfinite(totals[0]) || !isfinite(totals[1]))
        envelope_totals<dev::WideSum>(cluster, n, pitch, k, l, wn, P, Wb, first, step, totals);
    // phi - mean, the mean in three FP32 numbers and the rounding errors carried to one final
    // addition: the FP64 difference rounded to FP32, at FP32's rate
    const double mean = totals[0] / ((double)k * n * n);
    const float mh = (float)mean, mm = (float)(mean - (double)mh), ml = (float)(mean - (double)mh - (double)mm);
    const float g = gscale ? gscale[problem] : 1.0f;
    for (int r = first; r < k * n; r += step) {
        const size_t o = (size_t)r * pitch;
#pragma unroll 4
        for (int i = lane; i < n; i += 32) {
            float e, f, h;
            const float d = dev::two_sum(P[o + i], -mh, e), t = dev::two_sum(e, -mm, f);
            const float c = dev::two_sum(d, t, h);
            const float v = g * (c + (h + (f - ml)));
            if (d_rho1) d_rho1[problem * pcnt + o + i] = v;
            if (d_rho0) d_rho0[problem * pcnt + o + i] = -v;
        }
    }
    if (threadIdx.x == 0 && rank == 0 && d_alpha) d_alpha[problem] = (float)(g * totals[1]);
}

// The reverse step's sums, each rounded in a fixed way: the shrink's derivative jumps where
// |v| crosses the threshold, so at a point that lies on it another rounding moves the
// gradient (one such point of 256^2 moved dJ/dalpha by 1.7e-5).
__device__ __forceinline__ float dot2(float a, float b, float c, float d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); }
__device__ __forceinline__ float madd(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float mul_add(float a, float b, float c) { return __fadd_rn(__fmul_rn(a, b), c); }

// transpose of the Jacobian of shrink_2(.; t) at v (a 2-vector), applied to H:
// (1 - t/s) H + t (v.H) v / s^3 for s = |v| > t, else 0
__device__ __forceinline__ void vjp_shrink2(float vx, float vy, float t, float hx, float hy, float &ox, float &oy)
{
    const float s2 = dot2(vx, vx, vy, vy);
    if (s2 > t * t) {
        const float r = rsqrtf(s2);
        const float a = madd(-t, r, 1.0f), c = t * dot2(vx, hx, vy, hy) * r * r * r;
        ox = dot2(a, hx, c, vx);
        oy = dot2(a, hy, c, vy);
    } else {
        ox = 0.0f;
        oy = 0.0f;
    }
}

template <int K>
struct ALK {
    static constexpr int v = K * (K - 1) / 2 > 0 ? K * (K - 1) / 2 : 1;
};

// Adjoint of J_T = P(u^T, w^T) with respect to the final iterate (||u||_{1,2},
// ||w||_1 or ||w||_2); per-block partial sums of J_T and of sum ||w^T|| go to
// part[blk][0..1].
template <int K>
__global__ void __launch_bounds__(AT) k_adj_init(int n, int l, int wn, float alpha, const float *__restrict__ S,
                                                  float *__restrict__ A, double *__restrict__ part)
{
    const int i = blockIdx.x * AX + threadIdx.x, j = blockIdx.y * AY + threadIdx.y;
    const size_t nn = (size_t)n * n;
    double jp = 0.0, wp = 0.0;
    if (i < n && j < n) {
        const size_t p = (size_t)j * n + i;
        for (int c = 0; c < K; ++c) {
            const float x = S[(K + c) * nn + p], y = S[(2 * K + c) * nn + p];
            const float s = sqrtf(x * x + y * y);
            jp += s;
            A[c * nn + p] = 0.0f;                                  // adjoint of phi^T
            A[(K + c) * nn + p] = s > 0.0f ? x / s : 0.0f;         // adjoint of u^T
            A[(2 * K + c) * nn + p] = s > 0.0f ? y / s : 0.0f;
        }
        float ws = 0.0f;
        for (int e = 0; e < l; ++e) {
            const float x = S[(3 * K + e) * nn + p];
            ws += (wn == VOMT_W_L1) ? fabsf(x) : x * x;
        }
        if (wn == VOMT_W_L2) ws = sqrtf(ws);
        for (int e = 0; e < l; ++e) {
            const float x = S[(3 * K + e) * nn + p];
            float gdir = (wn == VOMT_W_L1) ? (x > 0.0f ? 1.0f : (x < 0.0f ? -1.0f : 0.0f)) : (ws > 0.0f ? x / ws : 0.0f);
            A[(3 * K + e) * nn + p] = alpha * gdir;
        }
        jp += (double)alpha * ws;
        wp = ws;
    }
    __shared__ double sh[2][AT];
    const int t = threadIdx.y * AX + threadIdx.x;
    sh[0][t] = jp;
    sh[1][t] = wp;
    __syncthreads();
    for (int off = AT / 2; off > 0; off >>= 1) {
        if (t < off) { sh[0][t] += sh[0][t + off]; sh[1][t] += sh[1][t + off]; }
        __syncthreads();
    }
    if (t == 0) {
        const int blk = blockIdx.y * gridDim.x + blockIdx.x;
        part[blk * 2 + 0] = sh[0][0];
        part[blk * 2 + 1] = sh[1][0];
    }
}

// One reverse step: given the iterate s^t (S) and the adjoint of s^{t+1} (A1),
// write the adjoint of s^t (A0), add tau * (adjoint of phi^{t+1}) to grho (the
// derivative with respect to rho1; rho0 gets its negative) and add this block's
// contribution to dJ/dalpha to apart[blk].  ||u||_{1,2} (per channel shrink_2).
//
// A warp takes a row of a strip of 30 columns, one column per lane, and reads everything it
// needs at once: the shrink's adjoint is formed in the row (its x component reaches the
// right neighbour by a shuffle) and once more in the row below, whose y component enters.
// At the sizes that are unrolled in practice a step is bound by latency (256^2, three
// channels: 27 planes, 7 MB, all in L2): one round trip to L2 and the launch, which
// overlaps the previous step's end (launch_pdl).
template <int K>
__global__ void __launch_bounds__(AT) k_adj_step(const __grid_constant__ march::MarchOp g, int wn,
                                                 const float *__restrict__ S, const float *__restrict__ A1,
                                                 float *__restrict__ A0, float *__restrict__ grho,
                                                 double *__restrict__ apart)
{
    cudaGridDependencySynchronize();      // after the previous kernel (no-op for a normal launch)
    constexpr int LK = ALK<K>::v;
    const int n = g.n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = blockIdx.x * 30 - 1 + lane, j = blockIdx.y * AY + wid;
    dev::TripleSum sum;                   // this thread's share of -dJ/dalpha / nu
    if (j < n) {                          // whole warps
        const bool in = i >= 0 && i < n, own = in && lane >= 1 && lane < 31;
        const bool hR = i < n - 1, hL = i > 0, hU = j < n - 1, hD = j > 0;
        const size_t nn = (size_t)n * n, p = (size_t)j * n + (in ? i : 0);
        const float mu = g.mu, nu = g.nu, tau = g.tau, ih = g.ih, muih = mu * ih;
        const float *ux = S + (size_t)K * nn, *uy = S + (size_t)2 * K * nn, *w = S + (size_t)3 * K * nn;
        const float *Gx = A1 + (size_t)K * nn, *Gy = A1 + (size_t)2 * K * nn, *Gw = A1 + (size_t)3 * K * nn;
        const bool iu = in && hU, id = in && hD;
        float pc[K], qc[K], pu[K], qu[K], pd[K], qd[K], x[K], y[K], hx[K], hy[K], xd[K], yd[K], hxd[K], hyd[K], gr[K];
        float w0[LK], hw[LK];
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const size_t o = c * nn + p;
            pc[c] = in ? S[o] : 0.0f;
            qc[c] = in ? A1[o] : 0.0f;
            pu[c] = iu ? S[o + n] : 0.0f;
            qu[c] = iu ? A1[o + n] : 0.0f;
            pd[c] = id ? S[o - n] : 0.0f;
            qd[c] = id ? A1[o - n] : 0.0f;
            x[c] = in ? ux[o] : 0.0f;
            y[c] = in ? uy[o] : 0.0f;
            hx[c] = in ? Gx[o] : 0.0f;
            hy[c] = in ? Gy[o] : 0.0f;
            xd[c] = id ? ux[o - n] : 0.0f;
            yd[c] = id ? uy[o - n] : 0.0f;
            hxd[c] = id ? Gx[o - n] : 0.0f;
            hyd[c] = id ? Gy[o - n] : 0.0f;
            gr[c] = own ? grho[o] : 0.0f;
        }
#pragma unroll
        for (int e = 0; e < K * (K - 1) / 2; ++e) {
            const int ed = g.edge[e];
            w0[e] = ed >= 0 && own ? w[ed * nn + p] : 0.0f;
            hw[e] = ed >= 0 && own ? Gw[ed * nn + p] : 0.0f;
        }
        float dvg[K];
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const float pr = __shfl_down_sync(0xffffffffu, pc[c], 1), qr = __shfl_down_sync(0xffffffffu, qc[c], 1);
            const float prd = __shfl_down_sync(0xffffffffu, pd[c], 1), qrd = __shfl_down_sync(0xffffffffu, qd[c], 1);
            const float ax = hR ? ih * (qr - qc[c]) : 0.0f, ay = hU ? ih * (qu[c] - qc[c]) : 0.0f;
            const float ex = hR ? pr - pc[c] : 0.0f, ey = hU ? pu[c] - pc[c] : 0.0f;
            const float kx = madd(-2.0f * tau, ax, hx[c]), ky = madd(-2.0f * tau, ay, hy[c]);
            float gvx, gvy, glx, gdy = 0.0f, t_;
            vjp_shrink2(mul_add(muih, ex, x[c]), mul_add(muih, ey, y[c]), mu, kx, ky, gvx, gvy);
            // its x component as the right neighbour has it
            vjp_shrink2(madd(muih, ex, x[c]), mul_add(muih, ey, y[c]), mu, kx, ky, glx, t_);
            if (hD) {                     // the y component in the row below
                const float dax = hR ? ih * (qrd - qd[c]) : 0.0f, day = ih * (qc[c] - qd[c]);
                const float edx = hR ? prd - pd[c] : 0.0f;
                vjp_shrink2(mul_add(muih, edx, xd[c]), madd(muih, pc[c] - pd[c], yd[c]), mu,
                            madd(-2.0f * tau, dax, hxd[c]), madd(-2.0f * tau, day, hyd[c]), t_, gdy);
            }
            const float left = __shfl_up_sync(0xffffffffu, glx, 1);
            dvg[c] = ih * ((gvx - (hL ? left : 0.0f)) + (gvy - gdy));      // div of the shrink adjoint
            if (own) {
                A0[(K + c) * nn + p] = madd(tau, ax, gvx);
                A0[(2 * K + c) * nn + p] = madd(tau, ay, gvy);
            }
        }
        if (own) {
            // graph part
            float xw[LK], dq[LK], gxw[LK];
            const float th = g.alpha * nu;
            float s2 = 0.0f, xh = 0.0f;
#pragma unroll
            for (int lo = 0; lo < K; ++lo)
#pragma unroll
                for (int hi = lo + 1; hi < K; ++hi) {
                    const int e = lo * (2 * K - lo - 1) / 2 + hi - lo - 1;
                    dq[e] = dot2(-g.inv[e], qc[hi], g.inv[e], qc[lo]);
                    xw[e] = madd(nu, dot2(-g.inv[e], pc[hi], g.inv[e], pc[lo]), w0[e]);    // 0 where there is no edge
                    hw[e] = madd(-2.0f * tau, dq[e], hw[e]);
                    gxw[e] = 0.0f;
                    s2 = madd(xw[e], xw[e], s2);
                    xh = madd(xw[e], hw[e], xh);
                }
            if (wn == VOMT_W_L1) {
#pragma unroll
                for (int e = 0; e < K * (K - 1) / 2; ++e)
                    if (fabsf(xw[e]) > th) {
                        gxw[e] = hw[e];
                        sum.add(xw[e] > 0.0f ? hw[e] : -hw[e]);
                    }
            } else if (s2 > th * th) {
                const float r = rsqrtf(s2), a = madd(-th, r, 1.0f), c3 = th * xh * r * r * r;
#pragma unroll
                for (int e = 0; e < K * (K - 1) / 2; ++e) gxw[e] = dot2(a, hw[e], c3, xw[e]);
                sum.add(xh * r);
            }
            float gg[K];
#pragma unroll
            for (int c = 0; c < K; ++c) gg[c] = 0.0f;
#pragma unroll
            for (int lo = 0; lo < K; ++lo)
#pragma unroll
                for (int hi = lo + 1; hi < K; ++hi) {
                    const int e = lo * (2 * K - lo - 1) / 2 + hi - lo - 1, ed = g.edge[e];
                    if (ed >= 0) A0[(3 * K + ed) * nn + p] = mul_add(tau, dq[e], gxw[e]);
                    gg[lo] = madd(g.inv[e], gxw[e], gg[lo]);
                    gg[hi] = madd(-g.inv[e], gxw[e], gg[hi]);
                }
#pragma unroll
            for (int c = 0; c < K; ++c) {
                A0[c * nn + p] = madd(nu, gg[c], madd(-mu, dvg[c], qc[c]));
                grho[c * nn + p] = madd(tau, qc[c], gr[c]);
            }
        }
    }
    // the block's sum: three FP32 numbers over a warp that has terms, FP64 over the warps; the
    // terms cancel, so each enters unrounded and nu multiplies the sum
    __shared__ double sh[AY];
    if (__any_sync(0xffffffffu, sum.hi != 0.0f || sum.mid != 0.0f || sum.lo != 0.0f)) sum.warp();
    if (lane == 0) sh[wid] = sum.value();
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int q = 0; q < AY; ++q) t += sh[q];
        apart[blockIdx.y * gridDim.x + blockIdx.x] -= (double)g.nu * t;
    }
}

__global__ void k_sub(size_t cnt, const float *__restrict__ r0, const float *__restrict__ r1, float *__restrict__ b)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < cnt; q += (size_t)gridDim.x * blockDim.x)
        b[q] = r1[q] - r0[q];
}

__global__ void k_finish_grad(size_t cnt, float scale, const float *__restrict__ grho, float *__restrict__ d_rho0,
                              float *__restrict__ d_rho1)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < cnt; q += (size_t)gridDim.x * blockDim.x) {
        if (d_rho1) d_rho1[q] = scale * grho[q];
        if (d_rho0) d_rho0[q] = -scale * grho[q];
    }
}

using AdjInit = void (*)(int, int, int, float, const float *, float *, double *);
using AdjStep = void (*)(const march::MarchOp, int, const float *, const float *, float *, float *, double *);

template <int K>
void pick_adj_k(AdjInit *ai, AdjStep *as)
{
    *ai = k_adj_init<K>;
    *as = k_adj_step<K>;
}

void pick_adj(int k, AdjInit *ai, AdjStep *as)
{
    switch (k) {
        case 1: pick_adj_k<1>(ai, as); break;
        case 2: pick_adj_k<2>(ai, as); break;
        case 3: pick_adj_k<3>(ai, as); break;
        case 4: pick_adj_k<4>(ai, as); break;
        case 5: pick_adj_k<5>(ai, as); break;
        case 6: pick_adj_k<6>(ai, as); break;
        case 7: pick_adj_k<7>(ai, as); break;
        default: pick_adj_k<8>(ai, as); break;
    }
}

}  // namespace
}  // namespace vomt

using namespace vomt;

extern "C" int vomt_backward(vomt_ctx *ctx, int batch, int n, int pitch, int k, int n_edges, int w_norm,
                             const float *phi, const float *w, const float *grad_scale, float *d_rho0, float *d_rho1,
                             float *d_alpha, void *stream)
{
    if (!ctx) return VOMT_ERR_BAD_ARG;
    ctx->err.clear();
    if (batch < 1 || n < 2 || k < 1 || k > KVEC || n_edges < 0 || n_edges > LVEC || w_norm < 0 || w_norm > 1)
        return fail(ctx, VOMT_ERR_BAD_ARG, "backward: bad sizes");
    if (pitch == 0) pitch = n;
    if (pitch < n) return fail(ctx, VOMT_ERR_BAD_ARG, "backward: pitch must be 0 or >= n");
    if (!phi || (n_edges > 0 && !w)) return fail(ctx, VOMT_ERR_BAD_ARG, "backward: null array");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "cudaSetDevice");
    // Blocks of 16384 values and more, no more of them than two per SM, and threads with sixteen
    // values and more.  A block too many costs more than it saves: with eight blocks of 1024
    // threads for every problem, 2048 of 16^2 took 1430 us (now 23) and 512 of 32^2, three
    // channels, 370 (now 32), while eight of 256^2 want all 64 blocks (23 us, 677 with one block
    // each, FP64 sums per value and a division per index).
    const double values = (double)(k + n_edges) * n * n;
    unsigned blocks = 1, threads = 128;
    while (blocks < kEnvCluster && values >= 16384.0 * 2 * blocks && (double)batch * 2 * blocks <= 2.0 * ctx->sm_count)
        blocks *= 2;
    while (threads < 1024 && values > 16.0 * blocks * threads) threads *= 2;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)batch * blocks);
    cfg.blockDim = dim3(threads);
    cfg.stream = (cudaStream_t)stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_envelope, n, pitch, k, n_edges, w_norm, phi, w, grad_scale, d_rho0, d_rho1, d_alpha);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "backward launch");
    return VOMT_OK;
}

extern "C" int vomt_unrolled_grad(vomt_ctx *ctx, int n, const float *rho0, const float *rho1, const vomt_graph *graph,
                                  double alpha, const vomt_params *pin, int T, int ckpt, double scale, float *d_rho0,
                                  float *d_rho1, double *d_alpha, double *J, void *stream)
{
    try {
        if (!ctx) return VOMT_ERR_BAD_ARG;
        OpDev op;
        StepDev s;
        SolveCfg cfg;
        vomt_params p;
        int rc = prepare_vector(ctx, n, graph, alpha, pin, &op, &s, &cfg, &p);
        if (rc) return rc;
        if (p.eps != 0.0) return fail(ctx, VOMT_ERR_BAD_ARG, "the unrolled gradient takes eps = 0");
        if (p.u_norm != VOMT_U_L12) return fail(ctx, VOMT_ERR_BAD_ARG, "unrolled gradient: u_norm must be VOMT_U_L12");
        if (T < 1 || ckpt < 1) return fail(ctx, VOMT_ERR_BAD_ARG, "unrolled gradient: T >= 1 and ckpt >= 1");
        if (!rho0 || !rho1) return fail(ctx, VOMT_ERR_BAD_ARG, "null array");
        cudaStream_t st = (cudaStream_t)stream;
        cudaError_t e = cudaSetDevice(ctx->device);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "cudaSetDevice");
        ctx->launches = 0;
        rc = check_vector_densities(ctx, op.k, n, rho0, rho1, st);
        if (rc) return rc;
        const int K = op.k, l = op.l;
        march::MarchOp mop;
        if (!march_op(op, s, &mop)) return fail(ctx, VOMT_ERR_BAD_ARG, "unrolled gradient: not a channel graph");
        const size_t nn = (size_t)n * n, SZ = (size_t)(3 * K + l) * nn;
        // Every iterate is kept where that takes no more than the context's memory limit:
        // nothing is computed twice then (256^2, three channels, 200 iterations: 0.6 GB and 190
        // launches fewer).  Beyond, or where the memory is not to be had, checkpoints every `ckpt`
        // iterations.
        bool keep = ((size_t)T + 1) * SZ * sizeof(float) <= ctx->spare_bytes;
        const int nck = T / ckpt + 1, slots = std::min(ckpt, T) + 1;      // checkpoints, recompute slots
        auto floats = [&]() {
            return (size_t)2 * K * nn + 2 * SZ + (keep ? (size_t)T + 1 : (size_t)nck + slots) * SZ;
        };
        rc = ensure_buffer(ctx, (void **)&ctx->gbuf, &ctx->gbuf_bytes, floats() * sizeof(float), "gradient scratch");
        if (rc && keep) {
            keep = false;
            rc = ensure_buffer(ctx, (void **)&ctx->gbuf, &ctx->gbuf_bytes, floats() * sizeof(float), "gradient scratch");
            if (!rc) ctx->err.clear();
        }
        if (rc) return rc;
        const dim3 blk(AX, AY), grd((n + AX - 1) / AX, (n + AY - 1) / AY);
        const int nb = (int)(grd.x * grd.y);
        const dim3 rgrd((n + 29) / 30, (n + AY - 1) / AY);        // reverse steps: strips of 30 columns
        const int rb = (int)(rgrd.x * rgrd.y);
        rc = ensure_buffer(ctx, (void **)&ctx->gpart, &ctx->gpart_bytes, sizeof(double) * (2 * (size_t)nb + rb), "gradient sums");
        if (rc) return rc;
        float *b = ctx->gbuf, *grho = b + (size_t)K * nn;
        float *adj = grho + (size_t)K * nn;                 // 2 adjoint states
        float *ck = adj + 2 * SZ;                           // the iterates kept (all, or nck checkpoints)
        float *seg = ck + (size_t)nck * SZ;                 // `slots` recompute slots
        double *part = ctx->gpart, *apart = part + 2 * (size_t)nb;
        const int pb = (int)(((size_t)K * nn + 255) / 256 < 2048 ? ((size_t)K * nn + 255) / 256 : 2048);
        e = cudaMemsetAsync(ctx->dstatus, 0, sizeof(DevStatus), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(ck, 0, SZ * sizeof(float), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(grho, 0, (size_t)K * nn * sizeof(float), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(apart, 0, sizeof(double) * rb, st);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "gradient reset");
        k_sub<<<pb, 256, 0, st>>>((size_t)K * nn, rho0, rho1, b);
        ++ctx->launches;
        // forward, keeping every iterate or every ckpt-th
        const float *cur = ck;
        for (int t = 1; t <= T; ++t) {
            float *out = keep ? ck + (size_t)t * SZ
                              : (t % ckpt == 0 ? ck + (size_t)(t / ckpt) * SZ : seg + (size_t)(t & 1) * SZ);
            launch_step(op, s, p.u_norm, p.w_norm, cur, out, b, ctx->dstatus, st);
            ++ctx->launches;
            cur = out;
        }
        AdjInit ai;
        AdjStep as;
        pick_adj(K, &ai, &as);
        ai<<<grd, blk, 0, st>>>(n, l, p.w_norm, s.alpha, cur, adj, part);
        ++ctx->launches;
        int a_in = 0;
        auto reverse = [&](const float *St) {
            launch_pdl(as, rgrd, dim3(AT), 0, st, mop, p.w_norm, St, (const float *)(adj + (size_t)a_in * SZ),
                       adj + (size_t)(1 - a_in) * SZ, grho, apart);
            ++ctx->launches;
            a_in = 1 - a_in;
        };
        if (keep) {
            for (int t = T - 1; t >= 0; --t) reverse(ck + (size_t)t * SZ);
        } else {
            // one checkpoint segment at a time
            for (int sg = (T - 1) / ckpt; sg >= 0; --sg) {
                const int t0 = sg * ckpt, t1 = (t0 + ckpt < T) ? t0 + ckpt : T;
                const float *base = ck + (size_t)sg * SZ;
                for (int m = 1; m < t1 - t0; ++m) {
                    const float *in = (m == 1) ? base : seg + (size_t)(m - 1) * SZ;
                    launch_step(op, s, p.u_norm, p.w_norm, in, seg + (size_t)m * SZ, b, ctx->dstatus, st);
                    ++ctx->launches;
                }
                for (int t = t1 - 1; t >= t0; --t) reverse(t == t0 ? base : seg + (size_t)(t - t0) * SZ);
            }
        }
        k_finish_grad<<<pb, 256, 0, st>>>((size_t)K * nn, (float)scale, grho, d_rho0, d_rho1);
        ++ctx->launches;
        std::vector<double> hp((size_t)2 * nb + rb);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(hp.data(), part, sizeof(double) * hp.size(), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "unrolled gradient");
        double jv = 0.0, ws = 0.0, ga = 0.0;
        for (int q = 0; q < nb; ++q) {
            jv += hp[2 * q];
            ws += hp[2 * q + 1];
        }
        for (int q = 0; q < rb; ++q) ga += hp[2 * (size_t)nb + q];
        ctx->last_form = keep ? VOMT_FORM_UNROLLED_KEPT : VOMT_FORM_UNROLLED_CKPT;
        if (J) *J = jv;
        if (d_alpha) *d_alpha = scale * (ws + ga);
        if (!isfinite(jv)) return fail(ctx, VOMT_ERR_NONFINITE, "unrolled objective is not finite");
        return VOMT_OK;
    } catch (...) {
        return fail(ctx, VOMT_ERR_BAD_ARG, "internal exception");
    }
}
