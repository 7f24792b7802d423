// Batched engine: many independent vector-OMT problems of mixed grid size,
// channel count and channel graph in one persistent launch.
//
// Each thread block takes whole problems ("instances") from a device-side
// queue, largest first, and runs the PDHG iteration of Section 7.2 on each one
// to its own stopping point (per-instance tolerance and iteration cap) before
// taking the next.  Instances are independent, so a block needs no exchange
// with other blocks: one block barrier per iteration (the fused stencil
// recomputes the neighbouring shrinks, as the streaming engine does) and a
// block-level FP64 reduction per convergence check.  Iterates ping-pong between
// two buffers of a scratch arena in HBM; L1 and L2 keep the working set of an
// instance close.  The queue order balances the load: the longest instances
// start first and the small ones fill in at the end.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "internal.h"
#include "march2d.h"
#include "pdhg_device.cuh"
#include "resident_kernel.cuh"

namespace vomt {
namespace {

using namespace dev;

constexpr int BK = KVEC;                   // channels per instance (vector OMT, k <= 8)
constexpr int BL = BK * (BK - 1) / 2;

struct InstDev {
    int n, k, l, pad;
    float mu, nu, tau, alpha, ih;
    float wc[BK], we[BL];
    float G[BL][BK];
    float Dv[BK][BL];
    size_t o_rho0, o_rho1, o_u, o_w, o_phi;   // offsets (floats) into the caller's arena
    size_t o_b, o_s[2];                       // offsets (floats) into the scratch arena
    double mu_d, nu_d, tau_d;
    int reg;                                  // quadratic regularisation (see StepDev)
    float eps, su, sw;
    double eps_d;
};

struct InstStatus {
    int iter, checks, error, stop;
    double met[NMET];
};

struct BatchArgs {
    const InstDev *inst;
    const int *order;          // queue order (largest first)
    int count;
    int un, wn, max_iters, check_every, warm;
    double tol_gap, tol_res;
    float *arena;
    float *scratch;
    InstStatus *status;
    int *queue;                // next queue position
};

template <int K>
struct BLK {
    static constexpr int v = K * (K - 1) / 2 > 0 ? K * (K - 1) / 2 : 1;
};

// One fused iteration at point (i, j) of one instance (the streaming engine's
// formulation): u' at (i,j), (i-1,j), (i,j-1), w' at (i,j), phi' at (i,j).
template <int K>
__device__ __forceinline__ void step_point(const InstDev &I, int i, int j, const float *__restrict__ S0,
                                           float *__restrict__ S1, const float *__restrict__ b, int un, int wn)
{
    constexpr int LK = BLK<K>::v;
    const int n = I.n, l = I.l;
    const size_t nn = (size_t)n * n, p = (size_t)j * n + i;
    const float *phi = S0, *ux = S0 + (size_t)K * nn, *uy = S0 + (size_t)2 * K * nn, *w = S0 + (size_t)3 * K * nn;
    const bool hR = i < n - 1, hU = j < n - 1, hL = i > 0, hD = j > 0;
    const float mu = I.mu, muih = I.mu * I.ih, ih = I.ih;
    const float su = I.reg ? I.su : 1.0f, tu = I.reg ? mu * I.su : mu;
    float pc[K], vx[K], vy[K], ux0[K], uy0[K], lx[K], ly[K], lx0[K], dx[K], dy[K], dy0[K];
#pragma unroll
    for (int c = 0; c < K; ++c) {
        const float *P = phi + c * nn + p;
        pc[c] = P[0];
        const float pr = hR ? P[1] : 0.0f, pu = hU ? P[n] : 0.0f;
        const float pl = hL ? P[-1] : 0.0f, plu = (hL && hU) ? P[n - 1] : 0.0f;
        const float pd = hD ? P[-n] : 0.0f, prd = (hR && hD) ? P[1 - n] : 0.0f;
        ux0[c] = ux[c * nn + p];
        uy0[c] = uy[c * nn + p];
        vx[c] = ux0[c] + (hR ? muih * (pr - pc[c]) : 0.0f);
        vy[c] = uy0[c] + (hU ? muih * (pu - pc[c]) : 0.0f);
        lx0[c] = hL ? ux[c * nn + p - 1] : 0.0f;
        const float ly0 = hL ? uy[c * nn + p - 1] : 0.0f;
        lx[c] = lx0[c] + (hL ? muih * (pc[c] - pl) : 0.0f);
        ly[c] = ly0 + ((hL && hU) ? muih * (plu - pl) : 0.0f);
        const float dx0 = hD ? ux[c * nn + p - n] : 0.0f;
        dy0[c] = hD ? uy[c * nn + p - n] : 0.0f;
        dx[c] = dx0 + ((hR && hD) ? muih * (prd - pd) : 0.0f);
        dy[c] = dy0[c] + (hD ? muih * (pc[c] - pd) : 0.0f);
        if (I.reg) {
            vx[c] *= su; vy[c] *= su; lx[c] *= su; ly[c] *= su; dx[c] *= su; dy[c] *= su;
        }
    }
    shrink_u<K>(vx, vy, tu, un, I.wc);
    shrink_u<K>(lx, ly, tu, un, I.wc);
    shrink_u<K>(dx, dy, tu, un, I.wc);
    float w0[LK], wx[LK];
#pragma unroll
    for (int e = 0; e < LK; ++e) {
        float ge = 0.0f;
#pragma unroll
        for (int c = 0; c < K; ++c) ge += I.G[e][c] * pc[c];
        w0[e] = (e < l) ? w[e * nn + p] : 0.0f;
        wx[e] = (e < l) ? w0[e] + I.nu * ge : 0.0f;
        if (I.reg) wx[e] *= I.sw;
    }
    shrink_w<LK>(wx, l, I.reg ? I.alpha * I.nu * I.sw : I.alpha * I.nu, wn, I.we);
    float *ophi = S1, *oux = S1 + (size_t)K * nn, *ouy = S1 + (size_t)2 * K * nn, *ow = S1 + (size_t)3 * K * nn;
#pragma unroll
    for (int c = 0; c < K; ++c) {
        const float bxl = hL ? 2.0f * lx[c] - lx0[c] : 0.0f;
        const float byd = hD ? 2.0f * dy[c] - dy0[c] : 0.0f;
        float r = ih * (((2.0f * vx[c] - ux0[c]) - bxl) + ((2.0f * vy[c] - uy0[c]) - byd)) + b[c * nn + p];
#pragma unroll
        for (int e = 0; e < LK; ++e) r -= I.Dv[c][e] * (2.0f * wx[e] - w0[e]);
        ophi[c * nn + p] = pc[c] + I.tau * r;
        oux[c * nn + p] = vx[c];
        ouy[c * nn + p] = vy[c];
    }
#pragma unroll
    for (int e = 0; e < LK; ++e)
        if (e < l) ow[e * nn + p] = wx[e];
}

// FP64 metric terms of point (i, j) for state S1 (after the iteration) and S0
// (before), accumulated into v (see RED_*).
template <int K>
__device__ __forceinline__ void metric_point(const InstDev &I, int i, int j, const float *__restrict__ S1,
                                             const float *__restrict__ S0, const float *__restrict__ b, int un,
                                             int wn, double (&v)[NRED])
{
    constexpr int LK = BLK<K>::v;
    const int n = I.n, l = I.l;
    const size_t nn = (size_t)n * n, p = (size_t)j * n + i;
    const bool hR = i < n - 1, hU = j < n - 1, hL = i > 0, hD = j > 0;
    const float ih = I.ih;
    const double dih = (double)(n - 1);
    float ph[K], dph[K], ddiv[K];
    double rdiv[K];
    float nu_pt = 0.0f, dn_u = 0.0f, q2 = 0.0f, dist = 0.0f;
#pragma unroll
    for (int c = 0; c < K; ++c) {
        const size_t q = c * nn + p;
        const float *cux = S1 + (size_t)K * nn, *cuy = S1 + (size_t)2 * K * nn;
        const float *pux = S0 + (size_t)K * nn, *puy = S0 + (size_t)2 * K * nn;
        const float uxc = cux[q], uyc = cuy[q], bc = b[q], wgt = I.wc[c];
        ph[c] = S1[q];
        dph[c] = ph[c] - S0[q];
        const float xl = hL ? cux[q - 1] : 0.0f, yd = hD ? cuy[q - n] : 0.0f;
        rdiv[c] = dih * (((double)uxc - (double)xl) + ((double)uyc - (double)yd)) + (double)bc;
        const float dux = uxc - pux[q], duy = uyc - puy[q];
        const float dxl = hL ? cux[q - 1] - pux[q - 1] : 0.0f;
        const float dyd = hD ? cuy[q - n] - puy[q - n] : 0.0f;
        ddiv[c] = ih * ((dux - dxl) + (duy - dyd));
        v[RED_DU] += (double)(wgt * (dux * dux + duy * duy));
        v[RED_DP] += (double)(wgt * dph[c] * dph[c]);
        v[RED_D] += (double)wgt * (double)ph[c] * (double)bc;
        v[RED_BB] += (double)(wgt * bc * bc);
        const float gx = hR ? ih * (S1[q + 1] - ph[c]) : 0.0f;
        const float gy = hU ? ih * (S1[q + n] - ph[c]) : 0.0f;
        q2 += wgt * (uxc * uxc + uyc * uyc);
        if (un == VOMT_U_L12) {
            nu_pt += sqrtf(uxc * uxc + uyc * uyc);
            const float gn = sqrtf(gx * gx + gy * gy);
            dn_u = fmaxf(dn_u, gn);
            const float o = fmaxf(gn - 1.0f, 0.0f);
            dist += o * o;
        } else if (un == VOMT_U_L2) {
            nu_pt += wgt * (uxc * uxc + uyc * uyc);
            dn_u += wgt * (gx * gx + gy * gy);
        } else {
            nu_pt += wgt * (fabsf(uxc) + fabsf(uyc));
            dn_u = fmaxf(dn_u, fmaxf(fabsf(gx), fabsf(gy)));
            const float ox = fmaxf(fabsf(gx) - 1.0f, 0.0f), oy = fmaxf(fabsf(gy) - 1.0f, 0.0f);
            dist += wgt * (ox * ox + oy * oy);
        }
    }
    if (un == VOMT_U_L2) {
        nu_pt = sqrtf(nu_pt);
        dn_u = sqrtf(dn_u);
        const float o = fmaxf(dn_u - 1.0f, 0.0f);
        dist += o * o;
    }
    float nw_pt = 0.0f, dn_w = 0.0f;
    const float *cw = S1 + (size_t)3 * K * nn, *pw = S0 + (size_t)3 * K * nn;
#pragma unroll
    for (int e = 0; e < LK; ++e) {
        if (e < l) {
            const size_t q = e * nn + p;
            const float we = cw[q], dwe = we - pw[q], wgt = I.we[e];
            v[RED_DW] += (double)(wgt * dwe * dwe);
            q2 += wgt * we * we;
            float ge = 0.0f;
#pragma unroll
            for (int c = 0; c < K; ++c) {
                ge += I.G[e][c] * ph[c];
                rdiv[c] -= (double)I.Dv[c][e] * (double)we;
                ddiv[c] -= I.Dv[c][e] * dwe;
            }
            if (wn == VOMT_W_L1) {
                nw_pt += wgt * fabsf(we);
                dn_w = fmaxf(dn_w, fabsf(ge));
                const float o = fmaxf(fabsf(ge) - I.alpha, 0.0f);
                dist += wgt * o * o;
            } else {
                nw_pt += wgt * we * we;
                dn_w += wgt * ge * ge;
            }
        }
    }
    if (wn == VOMT_W_L2) {
        nw_pt = sqrtf(nw_pt);
        dn_w = sqrtf(dn_w);
        const float o = fmaxf(dn_w - I.alpha, 0.0f);
        if (l > 0) dist += o * o;
    }
    v[RED_P] += (double)nu_pt + (double)I.alpha * (double)nw_pt;
    if (I.reg) {
        v[RED_P] += (double)(I.eps * q2);
        v[RED_DIST] += (double)dist;
    }
#pragma unroll
    for (int c = 0; c < K; ++c) {
        v[RED_RR] += (double)I.wc[c] * rdiv[c] * rdiv[c];
        v[RED_X] += (double)(I.wc[c] * dph[c] * ddiv[c]);
    }
    float di = fmaxf(dn_u - 1.0f, 0.0f);
    if (l > 0) di = fmaxf(di, dn_w - I.alpha);
    v[RED_MAX] = fmax(v[RED_MAX], (double)di);
}

// block-wide fixed-order reduction of v; the result is valid in thread 0
__device__ __forceinline__ void block_reduce(double (&v)[NRED], double *red)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int q = 0; q < NRED; ++q) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const double o = __shfl_down_sync(0xffffffffu, v[q], off);
            v[q] = (q == RED_MAX) ? fmax(v[q], o) : v[q] + o;
        }
    }
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NRED; ++q) red[wid * NRED + q] = v[q];
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < nw; ++w)
#pragma unroll
            for (int q = 0; q < NRED; ++q) v[q] = (q == RED_MAX) ? fmax(v[q], red[w * NRED + q]) : v[q] + red[w * NRED + q];
}

// Solve one instance with the whole block.  I lives in shared memory.
template <int K>
__device__ void solve_one(const InstDev &I, const BatchArgs &a, InstStatus *st, double *red, int *flag)
{
    const int n = I.n, l = I.l;
    const int np = n * n;
    const size_t nn = (size_t)np;
    float *b = a.scratch + I.o_b;
    float *S[2] = {a.scratch + I.o_s[0], a.scratch + I.o_s[1]};
    const float *r0 = a.arena + I.o_rho0, *r1 = a.arena + I.o_rho1;
    float *u = a.arena + I.o_u, *w = a.arena + I.o_w, *phi = a.arena + I.o_phi;
    // b = rho1 - rho0; iterate 0 from zero or from the caller's arrays (ghost cells zeroed)
    for (int q = threadIdx.x; q < np; q += blockDim.x) {
        const int i = q % n, j = q / n;
        for (int c = 0; c < K; ++c) {
            b[c * nn + q] = r1[c * nn + q] - r0[c * nn + q];
            S[0][c * nn + q] = a.warm ? phi[c * nn + q] : 0.0f;
            S[0][(K + c) * nn + q] = (a.warm && i < n - 1) ? u[c * nn + q] : 0.0f;
            S[0][(2 * K + c) * nn + q] = (a.warm && j < n - 1) ? u[(K + c) * nn + q] : 0.0f;
        }
        for (int e = 0; e < l; ++e) S[0][(3 * K + e) * nn + q] = a.warm ? w[e * nn + q] : 0.0f;
    }
    __syncthreads();
    const int T = a.max_iters, CE = a.check_every;
    int t = 0, checks = 0;
    bool stop = false;
    while (!stop) {
        const bool do_step = t < T;
        if (do_step) {
            ++t;
            const float *in = S[(t - 1) & 1];
            float *out = S[t & 1];
            for (int q = threadIdx.x; q < np; q += blockDim.x) step_point<K>(I, q % n, q / n, in, out, b, a.un, a.wn);
            __syncthreads();
        }
        if (!do_step || t % CE == 0 || t == T) {
            // convergence check on the iterate after iteration t
            double v[NRED];
#pragma unroll
            for (int q = 0; q < NRED; ++q) v[q] = 0.0;
            const float *cur = S[t & 1], *prv = t > 0 ? S[(t - 1) & 1] : S[t & 1];
            for (int q = threadIdx.x; q < np; q += blockDim.x) metric_point<K>(I, q % n, q / n, cur, prv, b, a.un, a.wn, v);
            block_reduce(v, red);
            if (threadIdx.x == 0) {
                double m[NMET];
                m[0] = v[RED_P];
                m[1] = v[RED_D] - (I.reg ? v[RED_DIST] / (4.0 * I.eps_d) : 0.0);
                m[2] = fabs(m[0] - m[1]) / fmax(fabs(m[0]), 1e-300);
                m[3] = sqrt(v[RED_RR]) / (v[RED_BB] > 0.0 ? sqrt(v[RED_BB]) : 1.0);
                m[4] = v[RED_DU] / I.mu_d + (l > 0 ? v[RED_DW] / I.nu_d : 0.0) + v[RED_DP] / I.tau_d - 2.0 * v[RED_X];
                m[5] = v[RED_MAX];
                m[6] = (double)t;
                bool finite = true;
                for (int q = 0; q < 6; ++q) finite = finite && isfinite(m[q]);
                const bool conv = a.tol_gap > 0.0 && m[2] <= a.tol_gap && m[3] <= a.tol_res;
                m[7] = conv ? 1.0 : 0.0;
                for (int q = 0; q < NMET; ++q) st->met[q] = m[q];
                st->iter = t;
                st->checks = ++checks;
                if (!finite) st->error = VOMT_ERR_NONFINITE;
                const bool s_ = conv || !finite || t >= T;
                st->stop = s_ ? 1 : 0;
                *flag = s_ ? 1 : 0;
            }
            __syncthreads();
            stop = *flag != 0;
            __syncthreads();
        }
    }
    // final iterate to the caller's arrays
    const float *fin = S[t & 1];
    for (int q = threadIdx.x; q < np; q += blockDim.x) {
        for (int c = 0; c < K; ++c) {
            phi[c * nn + q] = fin[c * nn + q];
            u[c * nn + q] = fin[(K + c) * nn + q];
            u[(K + c) * nn + q] = fin[(2 * K + c) * nn + q];
        }
        for (int e = 0; e < l; ++e) w[e * nn + q] = fin[(3 * K + e) * nn + q];
    }
    __syncthreads();
}

__global__ void __launch_bounds__(512) k_batch(BatchArgs a)
{
    __shared__ InstDev I;
    __shared__ double red[32 * NRED];
    __shared__ int slot, flag;
    for (;;) {
        if (threadIdx.x == 0) slot = atomicAdd(a.queue, 1);
        __syncthreads();
        const int s = slot;
        if (s >= a.count) break;
        const int idx = a.order[s];
        // copy the instance record to shared memory (uniform, read by every point)
        const int words = (int)(sizeof(InstDev) / 4);
        for (int q = threadIdx.x; q < words; q += blockDim.x) ((int *)&I)[q] = ((const int *)&a.inst[idx])[q];
        __syncthreads();
        InstStatus *st = a.status + idx;
        switch (I.k) {
            case 1: solve_one<1>(I, a, st, red, &flag); break;
            case 2: solve_one<2>(I, a, st, red, &flag); break;
            case 3: solve_one<3>(I, a, st, red, &flag); break;
            case 4: solve_one<4>(I, a, st, red, &flag); break;
            case 5: solve_one<5>(I, a, st, red, &flag); break;
            case 6: solve_one<6>(I, a, st, red, &flag); break;
            case 7: solve_one<7>(I, a, st, red, &flag); break;
            default: solve_one<8>(I, a, st, red, &flag); break;
        }
        __syncthreads();
    }
}

}  // namespace
}  // namespace vomt

namespace vomt {
namespace {

// Blocks per instance of the density checks, one per 16384 values of the largest instance: one
// of 256^2 with five channels is 2.6 MB, 0.6 ms for one block, while 16 blocks for each of 64
// instances of 32^2 cost 20 us, most of it the host's look at their results.
constexpr int kValChunks = 16;
int val_chunks(const std::vector<InstDev> &h)
{
    size_t most = 0;
    for (const InstDev &I : h) most = std::max(most, (size_t)I.k * I.n * I.n);
    return (int)std::min<size_t>(std::max<size_t>((most + 16383) / 16384, 1), kValChunks);
}

// per instance and chunk (a block each): sum rho0, sum rho1, min rho0, min rho1, non-finite count
template <typename Sum>
__global__ void __launch_bounds__(256) k_batch_validate(const InstDev *inst, const float *arena, int chunks, double *out)
{
    const InstDev &I = inst[blockIdx.x / chunks];
    const size_t cnt = (size_t)I.k * I.n * I.n, chunk = blockIdx.x % chunks;
    const float *r0 = arena + I.o_rho0, *r1 = arena + I.o_rho1;
    const size_t q0 = cnt * chunk / chunks, q1 = cnt * (chunk + 1) / chunks;
    DensityCheck<Sum> c;
#pragma unroll 4
    for (size_t q = q0 + threadIdx.x; q < q1; q += 256) c.add(r0[q], r1[q]);
    c.store(out + (size_t)blockIdx.x * 5);
}

}  // namespace

// Per-context state of the batched engine (device tables, scratch, captured graph).
struct BatchState {
    InstDev *dinst = nullptr;
    int *dorder = nullptr, *dqueue = nullptr;
    InstStatus *dstatus = nullptr, *hstatus = nullptr;
    double *dval = nullptr;
    int cap = 0;
    float *scratch = nullptr;
    size_t scratch_floats = 0;
    cudaGraphExec_t exec = nullptr;
    // what the captured graph was built for
    int g_count = -1, g_threads = 0, g_blocks = 0;
    const float *g_arena = nullptr;
    cudaStream_t g_stream = nullptr;
    BatchArgs g_args;
    int tuned_threads = 0;
    int tuned_engine = 0;      // set by vomt_batch_tune: the faster path for AUTO solves (0: by estimate)
    // whether the marching form was faster still, for batches of the tuned one's sides, channels
    // and edges: 1 or 0 (-1: not timed); trying: the tuner is timing it
    int tuned_march = -1;
    bool trying_march = false;
    std::vector<int> tuned_shapes;
    // grouped path: job tables, exchange scratch, control word, per-problem status
    void *gjobs = nullptr;
    size_t gjobs_bytes = 0;
    void *gvalid = nullptr;
    size_t gvalid_bytes = 0;
    void *gscratch = nullptr;
    size_t gscratch_bytes = 0;
    void *gstat = nullptr;
    size_t gstat_bytes = 0;
    DevStatus *hgstat = nullptr;
    int hgstat_cap = 0;
    BatchMarchScratch march;         // marching form
    // grouped path: the waves captured as one CUDA graph, and what it was built for
    cudaGraphExec_t gexec = nullptr;
    std::vector<unsigned char> gkey;
    long long graph_replays = 0;     // grouped solves that ran as one graph launch
};

void batch_state_free(BatchState *b)
{
    if (!b) return;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->gexec) cudaGraphExecDestroy(b->gexec);
    cudaFree(b->dinst);
    cudaFree(b->dorder);
    cudaFree(b->dqueue);
    cudaFree(b->dstatus);
    cudaFree(b->dval);
    cudaFree(b->scratch);
    if (b->hstatus) cudaFreeHost(b->hstatus);
    cudaFree(b->gjobs);
    cudaFree(b->gvalid);
    cudaFree(b->gscratch);
    cudaFree(b->gstat);
    if (b->hgstat) cudaFreeHost(b->hgstat);
    march_scratch_free(&b->march);
    delete b;
}

void batch_state_trim(BatchState *b, size_t bytes)
{
    if (!b || b->march.data_cap <= bytes) return;
    cudaFree(b->march.data);
    b->march.data = nullptr;
    b->march.data_cap = 0;
}

static int batch_reserve(vomt_ctx *ctx, BatchState *b, int count)
{
    if (b->cap >= count) return VOMT_OK;
    cudaFree(b->dinst); cudaFree(b->dorder); cudaFree(b->dqueue); cudaFree(b->dstatus); cudaFree(b->dval);
    if (b->hstatus) cudaFreeHost(b->hstatus);
    b->dinst = nullptr; b->dorder = b->dqueue = nullptr; b->dstatus = b->hstatus = nullptr; b->dval = nullptr;
    b->cap = 0;
    cudaError_t e = cudaMalloc(&b->dinst, sizeof(InstDev) * count);
    if (e == cudaSuccess) e = cudaMalloc(&b->dorder, sizeof(int) * count);
    if (e == cudaSuccess) e = cudaMalloc(&b->dqueue, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->dstatus, sizeof(InstStatus) * count);
    if (e == cudaSuccess) e = cudaMalloc(&b->dval, sizeof(double) * 5 * kValChunks * count);
    if (e == cudaSuccess) e = cudaMallocHost(&b->hstatus, sizeof(InstStatus) * count);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch tables");
    b->cap = count;
    if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
    b->g_count = -1;
    return VOMT_OK;
}

}  // namespace vomt

using namespace vomt;

static double table1_tau(int n) { return n <= 64 ? 1.0 : 3.0; }

extern "C" int vomt_batch_layout(int count, vomt_instance *inst, size_t *total_floats)
{
    if (count < 0 || (count > 0 && !inst)) return VOMT_ERR_BAD_ARG;
    size_t off = 0;
    for (int q = 0; q < count; ++q) {
        const int n = inst[q].n, k = inst[q].graph.k, l = inst[q].graph.n_edges;
        if (n < 2 || k < 1 || k > KVEC || l < 0 || l > LVEC) return VOMT_ERR_BAD_ARG;
        inst[q].offset = off;
        off += (size_t)(5 * k + l) * n * n;
        off = (off + 15) & ~(size_t)15;
    }
    if (total_floats) *total_floats = off;
    return VOMT_OK;
}

static int batch_prepare(vomt_ctx *ctx, int count, const vomt_instance *inst, const vomt_params &p,
                         std::vector<InstDev> &hinst, std::vector<int> &order, size_t *scratch_floats, int *bad_index)
{
    hinst.assign(count, InstDev());
    order.resize(count);
    size_t soff = 0;
    std::vector<double> cost(count);
    for (int q = 0; q < count; ++q) {
        *bad_index = q;
        const vomt_instance &in = inst[q];
        const int n = in.n;
        if (n < 2 || n > 32768) return fail(ctx, VOMT_ERR_BAD_ARG, "instance: n must be in [2, 32768]");
        if (!(in.alpha > 0.0) || !isfinite(in.alpha)) return fail(ctx, VOMT_ERR_BAD_ARG, "instance: alpha must be positive");
        GraphDev gd;
        int rc = graph_to_dev(&in.graph, &gd, &ctx->err);
        if (rc) return rc;
        OpDev op;
        graph_to_op(gd, &op);
        InstDev &I = hinst[q];
        memset(&I, 0, sizeof I);
        const int k = gd.k, l = gd.l;
        const size_t nn = (size_t)n * n;
        const double tau = in.tau > 0.0 ? in.tau : (p.tau > 0.0 ? p.tau : table1_tau(n));
        const double n1 = (double)(n - 1), lmax = graph_lmax(gd, in.graph.cost);
        const double mu = l > 0 ? 1.0 / (32.0 * tau * n1 * n1) : 1.0 / (16.0 * tau * n1 * n1);
        const double nu = l > 0 ? 1.0 / (4.0 * tau * lmax) : 1.0;
        I.n = n; I.k = k; I.l = l;
        I.mu = (float)mu; I.nu = (float)nu; I.tau = (float)tau; I.alpha = (float)in.alpha; I.ih = (float)n1;
        I.mu_d = mu; I.nu_d = nu; I.tau_d = tau;
        I.reg = p.eps > 0.0 ? 1 : 0;
        I.eps = (float)p.eps;
        I.eps_d = p.eps;
        I.su = (float)(1.0 / (1.0 + 2.0 * mu * p.eps));
        I.sw = (float)(1.0 / (1.0 + 2.0 * nu * p.eps));
        // the instance table holds vector-OMT operators (k <= 8): copy entry by entry
        for (int c = 0; c < BK; ++c) I.wc[c] = op.wc[c];
        for (int e = 0; e < BL; ++e) I.we[e] = op.we[e];
        for (int e = 0; e < BL; ++e)
            for (int c = 0; c < BK; ++c) {
                I.G[e][c] = op.G[e][c];
                I.Dv[c][e] = op.Dv[c][e];
            }
        I.o_rho0 = in.offset;
        I.o_rho1 = in.offset + (size_t)k * nn;
        I.o_u = in.offset + (size_t)2 * k * nn;
        I.o_w = in.offset + (size_t)4 * k * nn;
        I.o_phi = in.offset + (size_t)(4 * k + l) * nn;
        I.o_b = soff;
        I.o_s[0] = soff + (size_t)k * nn;
        I.o_s[1] = I.o_s[0] + (size_t)(3 * k + l) * nn;
        soff += (size_t)(7 * k + 2 * l) * nn;
        soff = (soff + 15) & ~(size_t)15;
        cost[q] = (double)nn * (7 * k + 2 * l);
        order[q] = q;
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    *scratch_floats = soff;
    *bad_index = -1;
    return VOMT_OK;
}

// ------------------------------------------------------------- grouped path
// Problems with the same channel count and grid side form a wave.  In one
// cooperative launch per wave the SMs split into groups of T blocks (T tiles of
// one problem, resident_plan_wave); each group runs the resident algorithm on
// its share of the wave's problems one after the other, the groups side by
// side.  A large problem is thus spread over many SMs instead of one, and
// small problems still fill the GPU.
struct Wave {
    int k, n;
    std::vector<int> insts;
    ResidentPlan plan;
    int groups, per;
};

// The problems the grouped path can take: K <= 5 (grouped kernels exist), a tile
// plan exists, and tags stay unique (iterations below 2^20 per problem).
static bool grouped_plan(vomt_ctx *ctx, int count, const std::vector<InstDev> &h, const vomt_params &p,
                         std::vector<Wave> &waves)
{
    waves.clear();
    if (p.max_iters >= (1 << 20) - 2) return false;
    std::vector<int> idx(count);
    for (int q = 0; q < count; ++q) idx[q] = q;
    std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) {
        return h[a].k != h[b].k ? h[a].k < h[b].k : h[a].n > h[b].n;
    });
    for (int q : idx) {
        if (h[q].k > 5) return false;
        if (waves.empty() || waves.back().k != h[q].k || waves.back().n != h[q].n) {
            Wave w;
            w.k = h[q].k;
            w.n = h[q].n;
            waves.push_back(w);
        }
        waves.back().insts.push_back(q);
    }
    for (Wave &w : waves) {
        if (!resident_plan_wave(w.n, w.k, (int)w.insts.size(), ctx->sm_count, &w.plan)) return false;
        const int T = w.plan.Gx * w.plan.Gy;
        w.groups = std::min((int)w.insts.size(), ctx->sm_count / T);
        w.per = ((int)w.insts.size() + w.groups - 1) / w.groups;
        const int nm = (p.u_norm == VOMT_U_L12 && p.w_norm == VOMT_W_L1) ? 1 : 0;
        if (!res::res_multi_kernel(w.k, w.plan.P, nm, w.plan.lb)) return false;
    }
    return true;
}

// Estimated time (ns) of the two paths at the iteration cap: the grouped waves
// by their tile plans; one block per problem by the measured cost of its fused
// step on one SM (about 14 ns per point and iteration at k = 3, scaled by the
// bytes per point), limited by the largest problem or the total over the SMs.
static double grouped_estimate(const std::vector<Wave> &waves, int iters)
{
    double t = 0.0;
    for (const Wave &w : waves)      // est_ns of a wave plan already covers its rounds
        t += w.plan.est_ns * (double)iters * (double)(7 * w.k + w.k * (w.k - 1)) / 27.0 + 20000.0;
    return t;
}

static double queue_estimate(const std::vector<InstDev> &h, int iters, int sms)
{
    double total = 0.0, longest = 0.0;
    for (const InstDev &I : h) {
        const double c = 14.0 * (double)I.n * I.n * (double)(7 * I.k + 2 * I.l) / 27.0 * (double)iters;
        total += c;
        longest = std::max(longest, c);
    }
    return std::max(longest, total / sms);
}

// the problems as the marching form takes them; false where it does not
static bool march_problems(const std::vector<InstDev> &h, float *arena, const vomt_params &p,
                           std::vector<BatchProblem> *out)
{
    for (const InstDev &I : h) {
        OpDev op;
        memset(&op, 0, sizeof op);
        op.k = I.k;
        op.l = I.l;
        for (int c = 0; c < BK; ++c) op.wc[c] = I.wc[c];
        for (int e = 0; e < BL; ++e) {
            op.we[e] = I.we[e];
            for (int c = 0; c < BK; ++c) {
                op.G[e][c] = I.G[e][c];
                op.Dv[c][e] = I.Dv[c][e];
            }
        }
        StepDev s{I.n, I.ih, I.mu, I.nu, I.tau, I.alpha};
        BatchProblem b;
        b.k = I.k;
        if (!march_op(op, s, &b.g) || !edges_in_order(b.g) || b.g.tu < 2e-19f || (I.l > 0 && b.g.tw < 2e-19f)) return false;
        b.cfg = SolveCfg{p.tol_gap, p.tol_res, I.mu_d, I.nu_d, I.tau_d, I.l > 0 ? 1 : 0};
        b.planar = march::PlanarArgs{arena + I.o_rho0, arena + I.o_rho1, arena + I.o_u, arena + I.o_w, arena + I.o_phi,
                                     p.warm_start};
        out->push_back(b);
    }
    return true;
}

static std::vector<int> batch_shapes(const std::vector<InstDev> &h)
{
    std::vector<int> s;
    for (const InstDev &I : h) s.insert(s.end(), {I.n, I.k, I.l});
    return s;
}

static int grouped_solve(vomt_ctx *ctx, BatchState *b, int count, const std::vector<InstDev> &h, float *arena,
                         const vomt_params &p, std::vector<Wave> &waves, cudaStream_t st, bool *as_graph)
{
    *as_graph = false;
    const int nm = (p.u_norm == VOMT_U_L12 && p.w_norm == VOMT_W_L1) ? 1 : 0;
    // scratch: per wave, per group two job slots of exchange words and check rows
    size_t jobs_total = 0, scratch_words = 0;
    for (const Wave &w : waves) {
        const int T = w.plan.Gx * w.plan.Gy;
        const int F2 = (3 * w.k + w.k * (w.k - 1) / 2 + 1) / 2;
        const size_t xw = (size_t)T * 2 * F2 * w.plan.TXm * w.plan.TYm * 2;
        const size_t rw = (size_t)2 * T * NRED * 2;
        scratch_words = std::max(scratch_words, (size_t)w.groups * 2 * (xw + rw));
        jobs_total += (size_t)w.groups * w.per;
    }
    const size_t ctl_bytes = 256;
    int rc = ensure_buffer(ctx, &b->gjobs, &b->gjobs_bytes, sizeof(res::ResArgs) * jobs_total, "grouped jobs");
    if (!rc) rc = ensure_buffer(ctx, &b->gvalid, &b->gvalid_bytes, sizeof(int) * jobs_total, "grouped jobs");
    if (!rc) rc = ensure_buffer(ctx, &b->gscratch, &b->gscratch_bytes, scratch_words * 8 + ctl_bytes, "grouped scratch");
    if (!rc) rc = ensure_buffer(ctx, &b->gstat, &b->gstat_bytes, sizeof(DevStatus) * count, "grouped status");
    if (rc) return rc;
    if (b->hgstat_cap < count) {
        if (b->hgstat) cudaFreeHost(b->hgstat);
        b->hgstat = nullptr;
        b->hgstat_cap = 0;
        cudaError_t e = cudaMallocHost(&b->hgstat, sizeof(DevStatus) * count);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "grouped status");
        b->hgstat_cap = count;
    }
    unsigned long long *xbase = (unsigned long long *)b->gscratch;
    dev::ResCtl *ctl = (dev::ResCtl *)((unsigned char *)b->gscratch + scratch_words * 8);
    DevStatus *dstat = (DevStatus *)b->gstat;
    std::vector<res::ResArgs> jobs(jobs_total);
    std::vector<int> valid(jobs_total, 0);
    size_t jbase = 0;
    std::vector<size_t> wave_job0(waves.size());
    for (size_t wi = 0; wi < waves.size(); ++wi) {
        const Wave &w = waves[wi];
        wave_job0[wi] = jbase;
        const ResidentPlan &pl = w.plan;
        const int T = pl.Gx * pl.Gy;
        const int F2 = (3 * w.k + w.k * (w.k - 1) / 2 + 1) / 2;
        const size_t xw = (size_t)T * 2 * F2 * pl.TXm * pl.TYm * 2;
        const size_t rw = (size_t)2 * T * NRED * 2;
        const int EWm = pl.TXm + 2 * pl.H, EHm = pl.TYm + 2 * pl.H;
        for (size_t i = 0; i < w.insts.size(); ++i) {
            const int q = w.insts[i];
            const InstDev &I = h[q];
            const int g = (int)(i % w.groups), j = (int)(i / w.groups);
            res::ResArgs &a = jobs[jbase + (size_t)g * w.per + j];
            memset(&a, 0, sizeof a);
            a.geo = res::ResGeom{I.n, pl.Gx, pl.Gy, pl.TXm, pl.TYm, T == 1 ? (1 << 30) : pl.H, T == 1 ? 0 : pl.H,
                                 res::row_stride(EWm), EHm};
            a.g.k = I.k;
            a.g.l = I.l;
            for (int c = 0; c < BK; ++c) a.g.wc[c] = I.wc[c];
            for (int e = 0; e < BL; ++e) a.g.we[e] = I.we[e];
            for (int e = 0; e < BL; ++e)
                for (int c = 0; c < BK; ++c) {
                    a.g.G[e][c] = I.G[e][c];
                    a.g.Dv[c][e] = I.Dv[c][e];
                }
            a.s = StepDev{I.n, I.ih, I.mu, I.nu, I.tau, I.alpha};
            a.cfg = SolveCfg{p.tol_gap, p.tol_res, I.mu_d, I.nu_d, I.tau_d, I.l > 0 ? 1 : 0};
            set_regularisation(&a.s, &a.cfg, p.eps, I.mu_d, I.nu_d);
            a.un = p.u_norm;
            a.wn = p.w_norm;
            a.max_iters = p.max_iters;
            a.check_every = p.check_every;
            a.warm = p.warm_start;
            a.rho0 = arena + I.o_rho0;
            a.rho1 = arena + I.o_rho1;
            a.u = arena + I.o_u;
            a.w = arena + I.o_w;
            a.phi = arena + I.o_phi;
            unsigned long long *slot = xbase + ((size_t)g * 2 + (j & 1)) * (xw + rw);
            a.xch = slot;
            a.rows = slot + xw;
            a.ctl = ctl;
            a.st = dstat + q;
            a.hist = nullptr;
            a.hist_cap = 0;
            a.wait_ns = ctx->wait_ns ? ctx->wait_ns : dev::kWaitBudgetNs;
            a.drop_exch = ctx->drop_exchange;
            a.tag_hi = (uint32_t)(q % 4095 + 1) << 20;
            valid[jbase + (size_t)g * w.per + j] = 1;
        }
        jbase += (size_t)w.groups * w.per;
    }
    cudaError_t e = cudaMemcpyAsync(b->gjobs, jobs.data(), sizeof(res::ResArgs) * jobs_total, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b->gvalid, valid.data(), sizeof(int) * jobs_total, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "grouped setup");
    // launch shape of every wave (attributes and occupancy are set outside any capture)
    // A wave whose problems each take every tile of the GPU (one group) runs them one after
    // the other as launches of the single-problem kernel, whose arguments sit in the constant
    // bank (the grouped kernel reads each problem's operator from shared memory).
    struct WaveLaunch {
        res::MultiKernel kern;
        res::ResKernel single;
        int blocks, threads, smem, jobs;
        size_t job0;
        size_t reset_bytes;
        res::MultiArgs m;
    };
    std::vector<WaveLaunch> wl(waves.size());
    // waves that share a kernel may need different shared memory: the kernel's limit is
    // set to the largest of its waves, once, before any launch
    std::vector<std::pair<res::MultiKernel, int>> limits;
    for (const Wave &w : waves) {
        const ResidentPlan &pl = w.plan;
        const int EWm = pl.TXm + 2 * pl.H, EHm = pl.TYm + 2 * pl.H;
        const int smem = res::smem_layout(w.k, res::row_stride(EWm), EHm, pl.Gx * pl.Gy).total;
        res::MultiKernel kern = res::res_multi_kernel(w.k, pl.P, nm, pl.lb);
        bool found = false;
        for (auto &lim : limits)
            if (lim.first == kern) { lim.second = std::max(lim.second, smem); found = true; }
        if (!found) limits.push_back({kern, smem});
    }
    for (const auto &lim : limits) {
        e = cudaFuncSetAttribute((const void *)lim.first, cudaFuncAttributeMaxDynamicSharedMemorySize, lim.second);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "grouped smem attribute");
    }
    std::vector<std::pair<res::ResKernel, int>> single_limits;
    for (const Wave &w : waves) {
        if (w.groups != 1) continue;
        const ResidentPlan &pl = w.plan;
        const int EWm = pl.TXm + 2 * pl.H, EHm = pl.TYm + 2 * pl.H;
        const int smem = res::smem_layout(w.k, res::row_stride(EWm), EHm, pl.Gx * pl.Gy).total;
        res::ResKernel kern = res::res_kernel(w.k, pl.P, nm, pl.lb > 0 ? pl.lb : res::res_threads(w.k), 0);
        if (!kern) continue;
        bool found = false;
        for (auto &lim : single_limits)
            if (lim.first == kern) { lim.second = std::max(lim.second, smem); found = true; }
        if (!found) single_limits.push_back({kern, smem});
    }
    for (const auto &lim : single_limits) {
        e = cudaFuncSetAttribute((const void *)lim.first, cudaFuncAttributeMaxDynamicSharedMemorySize, lim.second);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "grouped smem attribute");
    }
    for (size_t wi = 0; wi < waves.size(); ++wi) {
        const Wave &w = waves[wi];
        const ResidentPlan &pl = w.plan;
        const int T = pl.Gx * pl.Gy;
        const int EWm = pl.TXm + 2 * pl.H, EHm = pl.TYm + 2 * pl.H;
        const res::SmemLayout SL = res::smem_layout(w.k, res::row_stride(EWm), EHm, T);
        res::MultiKernel kern = res::res_multi_kernel(w.k, pl.P, nm, pl.lb);
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)kern, pl.threads, SL.total);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "grouped occupancy");
        const int blocks = w.groups * T;
        if (per_sm < 1 || blocks > per_sm * ctx->sm_count) {
            ctx->err = "grouped wave does not fit on the device";
            return VOMT_ERR_TOO_LARGE;
        }
        WaveLaunch &L = wl[wi];
        L.kern = kern;
        L.single = nullptr;
        L.blocks = blocks;
        L.threads = pl.threads;
        L.smem = SL.total;
        L.jobs = (int)w.insts.size();
        L.job0 = wave_job0[wi];
        if (w.groups == 1) {
            res::ResKernel sk = res::res_kernel(w.k, pl.P, nm, pl.lb > 0 ? pl.lb : res::res_threads(w.k), 0);
            int per_sm1 = 0;
            if (sk && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm1, (const void *)sk, pl.threads, SL.total) ==
                          cudaSuccess &&
                per_sm1 >= 1 && blocks <= per_sm1 * ctx->sm_count)
                L.single = sk;
            (void)cudaGetLastError();
        }
        // exchange words of an earlier wave must not match this wave's tags
        L.reset_bytes = (size_t)w.groups * 2 *
                        ((size_t)T * 2 * ((3 * w.k + w.k * (w.k - 1) / 2 + 1) / 2) * pl.TXm * pl.TYm * 2 +
                         (size_t)2 * T * NRED * 2) * 8;
        memset(&L.m, 0, sizeof L.m);
        L.m.jobs = (const res::ResArgs *)b->gjobs + wave_job0[wi];
        L.m.valid = (const int *)b->gvalid + wave_job0[wi];
        L.m.per = w.per;
        L.m.T = T;
        L.m.ctl = ctl;
    }
    auto enqueue = [&](cudaStream_t q) -> cudaError_t {
        cudaError_t r = cudaMemsetAsync(dstat, 0, sizeof(DevStatus) * count, q);
        if (r == cudaSuccess) r = cudaMemsetAsync(ctl, 0, ctl_bytes, q);
        for (size_t wi = 0; wi < wl.size() && r == cudaSuccess; ++wi) {
            WaveLaunch &L = wl[wi];
            r = cudaMemsetAsync(b->gscratch, 0, L.reset_bytes, q);
            if (r != cudaSuccess) break;
            if (L.single) {
                // one problem at a time on every tile; consecutive problems alternate exchange
                // slots and carry their own tag prefixes, as in the grouped kernel
                for (int j = 0; j < L.jobs && r == cudaSuccess; ++j) {
                    void *args[] = {&jobs[L.job0 + (size_t)j]};
                    r = cudaLaunchCooperativeKernel((const void *)L.single, dim3(L.blocks), dim3(L.threads), args,
                                                    L.smem, q);
                }
                continue;
            }
            void *args[] = {&L.m};
            r = cudaLaunchCooperativeKernel((const void *)L.kern, dim3(L.blocks), dim3(L.threads), args, L.smem, q);
        }
        if (r == cudaSuccess) r = cudaMemcpyAsync(b->hgstat, dstat, sizeof(DevStatus) * count, cudaMemcpyDeviceToHost, q);
        return r;
    };
    for (const WaveLaunch &L : wl) ctx->launches += L.single ? L.jobs : 1;
    // One CUDA graph holds every wave's launch; it is replayed on `st` while the job tables
    // and the launch shapes repeat (the tables are uploaded before each replay).  Capture
    // runs on `st`, or on the context's private stream when `st` is the legacy stream.
    std::vector<unsigned char> key;
    auto put = [&key](const void *p, size_t n) {
        const unsigned char *c = (const unsigned char *)p;
        key.insert(key.end(), c, c + n);
    };
    put(&count, sizeof count);
    put(jobs.data(), sizeof(res::ResArgs) * jobs_total);
    put(valid.data(), sizeof(int) * jobs_total);
    for (const WaveLaunch &L : wl) put(&L, sizeof L);
    if (!(b->gexec && key == b->gkey)) {
        if (b->gexec) { cudaGraphExecDestroy(b->gexec); b->gexec = nullptr; }
        b->gkey.clear();
        if (!st && !ctx->cap_stream) cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking);
        cudaStream_t cs = st ? st : ctx->cap_stream;
        cudaGraph_t graph = nullptr;
        e = cs ? cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) : cudaErrorInvalidResourceHandle;
        if (e == cudaSuccess) {
            cudaError_t r = enqueue(cs);
            e = cudaStreamEndCapture(cs, &graph);
            if (r != cudaSuccess) e = r;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&b->gexec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            // capture not available: launch the waves directly
            if (b->gexec) { cudaGraphExecDestroy(b->gexec); b->gexec = nullptr; }
            (void)cudaGetLastError();
            e = enqueue(st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) return set_cuda_error(ctx, e, "grouped solve");
            return VOMT_OK;
        }
        b->gkey.swap(key);
    }
    e = cudaGraphLaunch(b->gexec, st);
    ++b->graph_replays;
    *as_graph = e == cudaSuccess;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "grouped solve");
    return VOMT_OK;
}

extern "C" int vomt_solve_batched(vomt_ctx *ctx, int count, const vomt_instance *inst, float *arena,
                                  const vomt_params *pin, vomt_result *results, void *stream)
{
    try {
        if (!ctx) return VOMT_ERR_BAD_ARG;
        ctx->err.clear();
        if (count < 1 || !inst || !arena) return fail(ctx, VOMT_ERR_BAD_ARG, "need count >= 1, instances and an arena");
        vomt_params p;
        vomt_default_params(&p);
        if (pin) p = *pin;
        if (p.max_iters < 0 || p.check_every < 1) return fail(ctx, VOMT_ERR_BAD_ARG, "max_iters >= 0, check_every >= 1");
        if (p.u_norm < 0 || p.u_norm > 2 || p.w_norm < 0 || p.w_norm > 1) return fail(ctx, VOMT_ERR_BAD_ARG, "bad norm code");
        if (!(p.eps >= 0.0) || !isfinite(p.eps)) return fail(ctx, VOMT_ERR_BAD_ARG, "eps must be finite and >= 0");
        cudaStream_t st = (cudaStream_t)stream;
        cudaError_t e = cudaSetDevice(ctx->device);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "cudaSetDevice");
        if (!ctx->batch) ctx->batch = new BatchState();
        BatchState *b = ctx->batch;
        ctx->launches = 0;
        std::vector<InstDev> hinst;
        std::vector<int> order;
        size_t sfl = 0;
        int bad = -1;
        int rc = batch_prepare(ctx, count, inst, p, hinst, order, &sfl, &bad);
        if (rc) {
            char buf[64];
            snprintf(buf, sizeof buf, " (instance %d)", bad);
            ctx->err += buf;
            return rc;
        }
        rc = batch_reserve(ctx, b, count);
        if (rc) return rc;
        if (b->scratch_floats < sfl) {
            cudaFree(b->scratch);
            b->scratch = nullptr;
            b->scratch_floats = 0;
            e = cudaMalloc(&b->scratch, sizeof(float) * sfl);
            if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch scratch");
            b->scratch_floats = sfl;
            if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
        }
        e = cudaMemcpyAsync(b->dinst, hinst.data(), sizeof(InstDev) * count, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(b->dorder, order.data(), sizeof(int) * count, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch table upload");
        // density checks, several blocks per instance
        const int chunks = val_chunks(hinst);
        std::vector<double> hv((size_t)5 * chunks * count);
        for (int wide = 0; wide < 2; ++wide) {
            if (wide)
                k_batch_validate<WideSum><<<count * chunks, 256, 0, st>>>(b->dinst, arena, chunks, b->dval);
            else
                k_batch_validate<TripleSum><<<count * chunks, 256, 0, st>>>(b->dinst, arena, chunks, b->dval);
            ++ctx->launches;
            e = cudaMemcpyAsync(hv.data(), b->dval, sizeof(double) * hv.size(), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch validate");
            bool fits = true;
            for (double v : hv) fits = fits && !isnan(v);      // (the minimum of no entries is +inf)
            if (fits) break;
        }
        for (int q = 0; q < count; ++q) {
            double h[5] = {0.0, 0.0, INFINITY, INFINITY, 0.0};
            for (int c = 0; c < chunks; ++c) {
                const double *v = &hv[(size_t)5 * ((size_t)q * chunks + c)];
                h[0] += v[0];
                h[1] += v[1];
                h[2] = fmin(h[2], v[2]);
                h[3] = fmin(h[3], v[3]);
                h[4] += v[4];
            }
            char buf[96];
            int code = 0;
            if (h[4] > 0.0) { code = VOMT_ERR_NONFINITE; snprintf(buf, sizeof buf, "instance %d: NaN or Inf density", q); }
            else if (h[2] < 0.0 || h[3] < 0.0) { code = VOMT_ERR_NEGATIVE_DENSITY; snprintf(buf, sizeof buf, "instance %d: negative density", q); }
            else if (fabs(h[0] - h[1]) > kMassRelTol * fmax(fabs(h[0]), fabs(h[1]))) { code = VOMT_ERR_MASS_MISMATCH; snprintf(buf, sizeof buf, "instance %d: different total mass", q); }
            if (code) return fail(ctx, code, buf);
        }
        // path: grouped resident waves, or one block per problem from a queue
        std::vector<Wave> waves;
        bool grouped = false;
        const bool may_march = (p.engine == VOMT_ENGINE_AUTO || p.engine == VOMT_ENGINE_BATCHED) && p.u_norm == VOMT_U_L12 &&
                               p.w_norm == VOMT_W_L1 && p.eps == 0.0 && !ctx->drop_exchange &&
                               std::min(p.check_every, p.max_iters) >= 4;
        int march = -1;            // 1, 0: by the tuner's timing of such a batch
        if (may_march && b->trying_march) march = 1;
        else if (may_march && b->tuned_march >= 0 && b->tuned_shapes == batch_shapes(hinst)) march = b->tuned_march;
        if (p.engine == VOMT_ENGINE_RESIDENT) {
            if (!grouped_plan(ctx, count, hinst, p, waves))
                return fail(ctx, VOMT_ERR_TOO_LARGE,
                            "grouped batch path needs k <= 5, a resident tile plan and max_iters < 2^20 - 2");
            grouped = true;
        } else if (p.engine == VOMT_ENGINE_AUTO || p.engine == VOMT_ENGINE_BATCHED) {
            if (b->tuned_engine == VOMT_ENGINE_RESIDENT || march > 0)
                grouped = grouped_plan(ctx, count, hinst, p, waves);
            else if (b->tuned_engine == 0)
                grouped = grouped_plan(ctx, count, hinst, p, waves) &&
                          grouped_estimate(waves, std::max(p.max_iters, 1)) <
                              queue_estimate(hinst, std::max(p.max_iters, 1), ctx->sm_count);
        }
        // The marching form takes a grouped batch (same results, bit for bit) where the tuner
        // timed it faster or, for batches it has not seen, where it is estimated faster.  The
        // estimate of a wave is about twice what it takes (256^2, three channels: 3.06 us per
        // iteration against 1.57); of 22 batches of 2 to 300 problems the choice was the faster
        // one at every interval between checks, by 2% (2 x 256^2, a check every 4 iterations) to
        // 3.2 times (32 of 64^2 and 128^2 with five channels).
        std::vector<DevStatus> mstat;
        std::vector<int> mblocks;
        bool marched = false;
        if (grouped && may_march && march != 0) {
            const int iters = std::max(p.max_iters, 1);
            std::vector<int> sides, ks;
            for (const InstDev &I : hinst) {
                sides.push_back(I.n);
                ks.push_back(I.k);
            }
            std::vector<BatchProblem> probs;
            if ((march > 0 ||
                 march_batch_estimate(ctx, &b->march, sides, ks, p) < 0.5e-3 * grouped_estimate(waves, iters) / iters) &&
                march_problems(hinst, arena, p, &probs)) {
                rc = march_batch(ctx, &b->march, probs, p, st, &mstat, &mblocks, &marched);
                if (rc) return rc;
            }
        }
        if (grouped) {
            bool as_graph = false;
            if (!marched) {
                rc = grouped_solve(ctx, b, count, hinst, arena, p, waves, st, &as_graph);
                if (rc) return rc;
            }
            ctx->last_form = marched ? VOMT_FORM_BATCH_MARCH : VOMT_FORM_BATCH_GROUPED;
            std::vector<int> tiles(count, 1), halo(count, 0);
            for (const Wave &w : waves)
                for (int q : w.insts) {
                    tiles[q] = marched ? mblocks[q] : w.plan.Gx * w.plan.Gy;
                    halo[q] = !marched && tiles[q] > 1 ? w.plan.H : 0;
                }
            int status = VOMT_OK;
            for (int q = 0; q < count; ++q) {
                const DevStatus &h = marched ? mstat[q] : b->hgstat[q];
                int s_ = VOMT_OK;
                if (h.error) s_ = h.error;
                else if (h.checks == 0) s_ = VOMT_ERR_BARRIER_TIMEOUT;       // never started: the launch aborted
                else if (p.tol_gap > 0.0 && h.met[7] == 0.0) s_ = VOMT_NOT_CONVERGED;
                if (s_ < 0 && status >= 0) status = s_;
                else if (s_ == VOMT_NOT_CONVERGED && status == VOMT_OK) status = s_;
                if (results) {
                    vomt_result &r = results[q];
                    double met[NMET];
                    for (int m = 0; m < NMET; ++m) met[m] = h.met[m];
                    if (h.raw) finish_raw_row(met);
                    r.primal = met[0]; r.dual = met[1]; r.rel_gap = met[2]; r.rel_res = met[3];
                    r.fp_resid = met[4]; r.dual_infeas = met[5];
                    r.mu = hinst[q].mu_d; r.nu = hinst[q].nu_d; r.tau = hinst[q].tau_d;
                    r.iters = h.iter; r.status = s_; r.engine = VOMT_ENGINE_BATCHED; r.checks = h.checks;
                    r.launches = ctx->launches; r.blocks = tiles[q]; r.halo = halo[q];
                    r.variant = as_graph ? 1 : 0;
                }
            }
            if (status < 0) ctx->err = status == VOMT_ERR_BARRIER_TIMEOUT ? "device wait timed out"
                                                                          : "a problem produced a non-finite iterate";
            return status;
        }
        // launch shape: the tuned block size (untuned: 512, which the tuner picked for every
        // mix measured on GB300, twice as fast as 256 on the 512-problem mix), as many
        // resident blocks as fit, at most one per instance
        const int threads = b->tuned_threads > 0 ? b->tuned_threads : 512;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch, threads, 0);
        if (e != cudaSuccess || per_sm < 1) return set_cuda_error(ctx, e == cudaSuccess ? cudaErrorInvalidConfiguration : e, "batch occupancy");
        const int blocks = std::min(count, per_sm * ctx->sm_count);
        BatchArgs a;
        memset(&a, 0, sizeof a);
        a.inst = b->dinst;
        a.order = b->dorder;
        a.count = count;
        a.un = p.u_norm;
        a.wn = p.w_norm;
        a.max_iters = p.max_iters;
        a.check_every = p.check_every;
        a.warm = p.warm_start;
        a.tol_gap = p.tol_gap;
        a.tol_res = p.tol_res;
        a.arena = arena;
        a.scratch = b->scratch;
        a.status = b->dstatus;
        a.queue = b->dqueue;
        auto enqueue = [&]() -> cudaError_t {
            cudaError_t r = cudaMemsetAsync(b->dqueue, 0, sizeof(int), st);
            if (r == cudaSuccess) r = cudaMemsetAsync(b->dstatus, 0, sizeof(InstStatus) * count, st);
            if (r != cudaSuccess) return r;
            k_batch<<<blocks, threads, 0, st>>>(a);
            r = cudaGetLastError();
            if (r == cudaSuccess) r = cudaMemcpyAsync(b->hstatus, b->dstatus, sizeof(InstStatus) * count, cudaMemcpyDeviceToHost, st);
            return r;
        };
        if (st != nullptr) {
            // one captured graph per (tables, arena, launch shape, parameters); replayed while they repeat
            const bool same = b->exec && b->g_count == count && b->g_threads == threads && b->g_blocks == blocks &&
                              b->g_arena == arena && b->g_stream == st && memcmp(&b->g_args, &a, sizeof a) == 0;
            if (!same) {
                if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
                cudaGraph_t graph = nullptr;
                e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
                if (e == cudaSuccess) {
                    cudaError_t r = enqueue();
                    e = cudaStreamEndCapture(st, &graph);
                    if (r != cudaSuccess) e = r;
                }
                if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, graph, 0);
                if (graph) cudaGraphDestroy(graph);
                if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch graph capture");
                b->g_count = count; b->g_threads = threads; b->g_blocks = blocks; b->g_arena = arena; b->g_stream = st;
                b->g_args = a;
            }
            e = cudaGraphLaunch(b->exec, st);
        } else {
            e = enqueue();
        }
        ++ctx->launches;
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch solve");
        ctx->last_form = VOMT_FORM_BATCH_QUEUE;
        int status = VOMT_OK;
        for (int q = 0; q < count; ++q) {
            const InstStatus &h = b->hstatus[q];
            int s_ = VOMT_OK;
            if (h.error) s_ = h.error;
            else if (p.tol_gap > 0.0 && h.met[7] == 0.0) s_ = VOMT_NOT_CONVERGED;
            if (s_ < 0 && status >= 0) status = s_;
            else if (s_ == VOMT_NOT_CONVERGED && status == VOMT_OK) status = s_;
            if (results) {
                vomt_result &r = results[q];
                r.primal = h.met[0]; r.dual = h.met[1]; r.rel_gap = h.met[2]; r.rel_res = h.met[3];
                r.fp_resid = h.met[4]; r.dual_infeas = h.met[5];
                r.mu = hinst[q].mu_d; r.nu = hinst[q].nu_d; r.tau = hinst[q].tau_d;
                r.iters = h.iter; r.status = s_; r.engine = VOMT_ENGINE_BATCHED; r.checks = h.checks;
                r.launches = ctx->launches; r.blocks = 1; r.halo = 0;
                r.variant = st != nullptr ? 1 : 0;
            }
        }
        if (status < 0) ctx->err = "an instance produced a non-finite iterate";
        return status;
    } catch (...) {
        return fail(ctx, VOMT_ERR_BAD_ARG, "internal exception");
    }
}

static int batch_tune(vomt_ctx *ctx, int count, const vomt_instance *inst, float *arena, const vomt_params *pin,
                      int sample_iters, int *best_threads, double *ms)
{
    vomt_params p;
    vomt_default_params(&p);
    if (pin) p = *pin;
    p.max_iters = sample_iters;
    p.check_every = sample_iters;
    p.tol_gap = p.tol_res = 0.0;
    p.warm_start = 0;
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "cudaSetDevice");
    if (!ctx->batch) ctx->batch = new BatchState();
    BatchState *b = ctx->batch;
    // time one pass of each candidate (after an untimed pass: table upload, graph capture)
    auto timed = [&](vomt_params q, double *out) -> int {
        int rc = vomt_solve_batched(ctx, count, inst, arena, &q, nullptr, nullptr);
        if (rc < 0) return rc;
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        cudaEventRecord(e0, nullptr);
        rc = vomt_solve_batched(ctx, count, inst, arena, &q, nullptr, nullptr);
        cudaEventRecord(e1, nullptr);
        cudaEventSynchronize(e1);
        float t = 0.0f;
        cudaEventElapsedTime(&t, e0, e1);
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        *out = t;
        return rc < 0 ? rc : VOMT_OK;
    };
    const int cands[3] = {128, 256, 512};
    double best = 1e300;
    int pick = 256;
    vomt_params q = p;
    q.engine = VOMT_ENGINE_STREAM;          // one block per problem
    for (int c = 0; c < 3; ++c) {
        b->tuned_threads = cands[c];
        double t = 0.0;
        int rc = timed(q, &t);
        if (rc < 0) return rc;
        if (ms) ms[c] = t;
        if (t < best) { best = t; pick = cands[c]; }
    }
    b->tuned_threads = pick;
    if (best_threads) *best_threads = pick;
    // the grouped resident path, where it can take the problems
    b->tuned_engine = VOMT_ENGINE_STREAM;
    b->tuned_march = -1;
    if (ms) ms[3] = -1.0;
    std::vector<InstDev> hinst;
    std::vector<int> order;
    size_t sfl = 0;
    int bad = -1;
    std::vector<Wave> waves;
    if (batch_prepare(ctx, count, inst, p, hinst, order, &sfl, &bad) == VOMT_OK &&
        grouped_plan(ctx, count, hinst, p, waves)) {
        q.engine = VOMT_ENGINE_RESIDENT;
        double t = 0.0;
        int rc = timed(q, &t);
        if (rc < 0) return rc;
        if (ms) ms[3] = t;
        if (t < best) b->tuned_engine = VOMT_ENGINE_RESIDENT;
        best = std::min(best, t);
        // the marching form, where it takes them
        b->trying_march = true;
        q.engine = VOMT_ENGINE_AUTO;
        double tm = 0.0;
        rc = timed(q, &tm);
        b->trying_march = false;
        if (rc < 0) return rc;
        if (ctx->last_form == VOMT_FORM_BATCH_MARCH) {
            b->tuned_march = tm < best ? 1 : 0;
            b->tuned_shapes = batch_shapes(hinst);
        }
    }
    ctx->err.clear();
    return VOMT_OK;
}

extern "C" int vomt_batch_tune(vomt_ctx *ctx, int count, const vomt_instance *inst, float *arena,
                               const vomt_params *pin, int sample_iters, int *best_threads, double *ms)
{
    if (!ctx || sample_iters < 1) return VOMT_ERR_BAD_ARG;
    try {
        return batch_tune(ctx, count, inst, arena, pin, sample_iters, best_threads, ms);
    } catch (...) {
        return fail(ctx, VOMT_ERR_BAD_ARG, "internal exception");
    }
}

extern "C" int vomt_batch_set_threads(vomt_ctx *ctx, int threads)
{
    if (!ctx || !(threads == 0 || threads == 128 || threads == 256 || threads == 512)) return VOMT_ERR_BAD_ARG;
    if (!ctx->batch) ctx->batch = new BatchState();
    ctx->batch->tuned_threads = threads;
    return VOMT_OK;
}
