// Device helpers shared by the resident engines: the shrink operators of
// Appendix B with the norm picked at run time (the branch is uniform across a
// launch), tagged 64-bit exchange words and bounded waits.
#pragma once

#include <stdint.h>

#include "internal.h"
#include "matrix_norms.cuh"

namespace vomt {
namespace dev {

// factor of shrink_2 (Appendix B): 1 - t/s for s = sqrt(s2) > t, else 0, as
// max(1 - t / s, 0): the factor is positive exactly when s > t, and at s2 = 0 the
// reciprocal square root is +inf, so 1 - t/s is -inf (or NaN for t = 0, which
// fmaxf also maps to 0)
__device__ __forceinline__ float shrink2_factor(float s2, float t)
{
    return fmaxf(1.0f - t * rsqrtf(s2), 0.0f);
}

// shrink_1 (Appendix B): soft threshold sign(x) max(|x| - t, 0), as x minus x
// clamped to [-t, t] (the same single rounding of x -+ t where |x| > t, exactly 0
// elsewhere)
__device__ __forceinline__ float soft(float x, float t)
{
    return x - fminf(fmaxf(x, -t), t);
}

template <int K>
__device__ __forceinline__ float pick(const float (&a)[K], int idx)
{
    float r = 0.0f;
#pragma unroll
    for (int c = 0; c < K; ++c) r = (c == idx) ? a[c] : r;
    return r;
}

// shrink_u on one point (all channels), in place; un = VOMT_U_*; channel weights wc
// enter the joint norm (2 for an off-diagonal matrix entry)
// Is coordinate c the real part of a complex entry (bit c of `pairs`)?  The
// imaginary part is coordinate c + 1.
__device__ __forceinline__ bool pair_first(uint32_t pairs, int c) { return (pairs >> c) & 1u; }
__device__ __forceinline__ bool pair_second(uint32_t pairs, int c) { return c > 0 && ((pairs >> (c - 1)) & 1u); }
__device__ __forceinline__ bool wpair_first(const uint32_t (&wp)[2], int e) { return (wp[e >> 5] >> (e & 31)) & 1u; }
__device__ __forceinline__ bool wpair_second(const uint32_t (&wp)[2], int e)
{
    return e > 0 && ((wp[(e - 1) >> 5] >> ((e - 1) & 31)) & 1u);
}

template <int K>
__device__ __forceinline__ void shrink_u(float (&vx)[K], float (&vy)[K], float t, int un, const float *wc,
                                         uint32_t pairs = 0u)
{
    if (un == VOMT_U_L12) {
#pragma unroll
        for (int c = 0; c < K; ++c) {
            float f = shrink2_factor(vx[c] * vx[c] + vy[c] * vy[c], t);
            vx[c] *= f;
            vy[c] *= f;
        }
    } else if (un == VOMT_U_L2) {
        float s2 = 0.0f;
#pragma unroll
        for (int c = 0; c < K; ++c) s2 += wc[c] * (vx[c] * vx[c] + vy[c] * vy[c]);
        float f = shrink2_factor(s2, t);
#pragma unroll
        for (int c = 0; c < K; ++c) { vx[c] *= f; vy[c] *= f; }
    } else if (un == VOMT_U_NUC) {
        // ||U_x||_nuc + ||U_y||_nuc: each direction's symmetric matrix on its own
        mat::sym_shrink_nuc<K>(vx, t);
        mat::sym_shrink_nuc<K>(vy, t);
    } else if (un == U_CL1) {
        // complex entrywise ||.||_1 (sum of moduli) in each direction: the prox of t |z|
        // scales an (Re, Im) pair by its modulus (in the compact inner product the pair's
        // weight 2 multiplies both the norm and the distance, so the threshold stays t);
        // real coordinates (Hermitian diagonals) take the soft threshold
#pragma unroll
        for (int c = 0; c < K; ++c) {
            if (pair_first(pairs, c) && c + 1 < K) {
                const float fx = shrink2_factor(vx[c] * vx[c] + vx[c + 1] * vx[c + 1], t);
                const float fy = shrink2_factor(vy[c] * vy[c] + vy[c + 1] * vy[c + 1], t);
                vx[c] *= fx;
                vx[c + 1] *= fx;
                vy[c] *= fy;
                vy[c + 1] *= fy;
            } else if (!pair_second(pairs, c)) {
                vx[c] = soft(vx[c], t);
                vy[c] = soft(vy[c], t);
            }
        }
    } else {
#pragma unroll
        for (int c = 0; c < K; ++c) { vx[c] = soft(vx[c], t); vy[c] = soft(vy[c], t); }
    }
}

// shrink_w on one point, l <= LK flux entries with weights we; wn = VOMT_W_*
template <int LK>
__device__ __forceinline__ void shrink_w(float (&x)[LK], int l, float t, int wn, const float *we,
                                         const uint32_t *wpairs = nullptr)
{
    if (wn == W_CL1) {
        // complex entrywise ||.||_1 of the skew-Hermitian components, as in shrink_u
        const uint32_t wp[2] = {wpairs ? wpairs[0] : 0u, wpairs ? wpairs[1] : 0u};
#pragma unroll
        for (int e = 0; e < LK; ++e) {
            if (e >= l) continue;
            if (wpair_first(wp, e) && e + 1 < LK) {
                const float f = shrink2_factor(x[e] * x[e] + x[e + 1] * x[e + 1], t);
                x[e] *= f;
                x[e + 1] *= f;
            } else if (!wpair_second(wp, e)) {
                x[e] = soft(x[e], t);
            }
        }
    } else if (wn == VOMT_W_L1) {
#pragma unroll
        for (int e = 0; e < LK; ++e)
            if (e < l) x[e] = soft(x[e], t);
    } else if (wn == VOMT_W_NUC) {
        // 3 x 3 skew components, entries (a, b, c) consecutive: Euclidean group shrink
        if constexpr (LK % 3 == 0) {
#pragma unroll
            for (int g = 0; g < LK; g += 3) {
                if (g < l) {
                    const float f = shrink2_factor(x[g] * x[g] + x[g + 1] * x[g + 1] + x[g + 2] * x[g + 2], t);
                    x[g] *= f;
                    x[g + 1] *= f;
                    x[g + 2] *= f;
                }
            }
        }
    } else {
        float s2 = 0.0f;
#pragma unroll
        for (int e = 0; e < LK; ++e)
            if (e < l) s2 += we[e] * x[e] * x[e];
        float f = shrink2_factor(s2, t);
#pragma unroll
        for (int e = 0; e < LK; ++e) x[e] *= f;
    }
}

// ---------------------------------------------------------------- check sums
// Error-free sum (Knuth's TwoSum): s + e == a + b exactly.
__device__ __forceinline__ float two_sum(float a, float b, float &e)
{
    const float s = a + b;
    const float bv = s - a;
    e = (a - (s - bv)) + (b - bv);
    return s;
}

// ih * ((ux - xl) + (uy - yd)) + gb with the rounding errors of the
// differences, their sum, the product and the final sum carried along (the
// compensated evaluation of Ogita, Rump and Oishi, "Accurate sum and dot
// product", 2005): about twice FP32 precision for the constraint residual,
// whose terms cancel as the iteration converges.
__device__ __forceinline__ float residual_c(float ih, float ux, float xl, float uy, float yd, float gb)
{
    float e1, e2, e3, e4;
    const float d1 = two_sum(ux, -xl, e1);
    const float d2 = two_sum(uy, -yd, e2);
    const float s = two_sum(d1, d2, e3);
    const float p = ih * s;
    const float pe = fmaf(ih, s, -p);
    const float r = two_sum(p, gb, e4);
    return r + (e4 + (pe + ih * ((e1 + e2) + e3)));
}

// The same with nothing dropped but the rounding of the smallest terms: the residual as a
// normalised pair hi + lo, correct to about 2^-48 of hi.
__device__ __forceinline__ float residual_pair(float ih, float ux, float xl, float uy, float yd, float gb, float &lo)
{
    float e1, e2, e3, e4, f1, f2, g1, g2, h;
    const float d1 = two_sum(ux, -xl, e1);
    const float d2 = two_sum(uy, -yd, e2);
    const float s = two_sum(d1, d2, e3);
    const float p = ih * s;
    const float pe = fmaf(ih, s, -p);
    const float r = two_sum(p, gb, e4);
    const float t = two_sum(two_sum(e1, e2, f1), e3, f2);
    const float q = ih * t;
    const float c = two_sum(two_sum(pe, q, g1), e4, g2);
    const float hi = two_sum(r, c, h);
    lo = h + ((g1 + g2) + (fmaf(ih, t, -q) + ih * (f1 + f2)));
    return hi;
}

// A running sum kept as three FP32 numbers by TwoSum, what the first addition rounds off
// going to the second number and what that rounds off to the third: no less accurate than an
// FP64 sum at FP32's rate (FP64 additions run at a sixty-fourth of it on this GPU, so a pass
// that adds every value it reads in FP64 is bound by them).  Over 96 x 2048 values summed per
// thread and warp and then in FP64, the error against exact sums, over the sum of the
// magnitudes, is (root mean square) 6.6e-17 for densities (FP64 8.2e-17, pairs 3.1e-16), 2.2e-19
// for potentials (2.2e-19, 5.5e-19) and 0 for terms that cancel to 1e-6 (0, 1.9e-18).  A sum
// beyond FP32's range becomes NaN.
struct TripleSum {
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        float e, f;
        hi = two_sum(hi, x, e);
        mid = two_sum(mid, e, f);
        lo += f;
    }
    __device__ __forceinline__ void merge(float oh, float om, float ol)
    {
        float f;
        add(oh);
        mid = two_sum(mid, om, f);
        lo += ol + f;
    }
    __device__ __forceinline__ void warp()          // lane 0 ends with the warp's sum
    {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            merge(__shfl_down_sync(0xffffffffu, hi, off), __shfl_down_sync(0xffffffffu, mid, off),
                  __shfl_down_sync(0xffffffffu, lo, off));
    }
    __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
    __device__ __forceinline__ void save(uint32_t *w) const
    {
        w[0] = __float_as_uint(hi);
        w[1] = __float_as_uint(mid);
        w[2] = __float_as_uint(lo);
    }
    __device__ __forceinline__ void merge(const uint32_t *w)
    {
        merge(__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]));
    }
};

// The same in FP64, for sums beyond FP32's range.
struct WideSum {
    double v = 0.0;
    __device__ __forceinline__ void add(float x) { v += x; }
    __device__ __forceinline__ void warp()
    {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    }
    __device__ __forceinline__ double value() const { return v; }
    __device__ __forceinline__ void save(uint32_t *w) const
    {
        w[0] = (uint32_t)__double2loint(v);
        w[1] = (uint32_t)__double2hiint(v);
        w[2] = 0;
    }
    __device__ __forceinline__ void merge(const uint32_t *w) { v += __hiloint2double((int)w[1], (int)w[0]); }
};

// Input checks of densities: what a block of 256 threads has seen, stored as five FP64
// values (sum rho0, sum rho1, min rho0, min rho1, count of non-finite entries).  Where a
// TripleSum comes back non-finite, the caller runs the check again with WideSum.
template <typename Sum>
struct DensityCheck {
    Sum s0, s1;
    float m0 = INFINITY, m1 = INFINITY;
    int bad = 0;
    __device__ __forceinline__ void add(float a, float c)
    {
        if (!(fabsf(a) < INFINITY) || !(fabsf(c) < INFINITY)) {
            ++bad;
            return;
        }
        s0.add(a);
        s1.add(c);
        m0 = fminf(m0, a);
        m1 = fminf(m1, c);
    }
    __device__ __forceinline__ void store(double *out)
    {
        __shared__ double sh[8][5];
        s0.warp();
        s1.warp();
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            m0 = fminf(m0, __shfl_down_sync(0xffffffffu, m0, off));
            m1 = fminf(m1, __shfl_down_sync(0xffffffffu, m1, off));
            bad += __shfl_down_sync(0xffffffffu, bad, off);
        }
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        if (lane == 0) {
            sh[wid][0] = s0.value();
            sh[wid][1] = s1.value();
            sh[wid][2] = m0;
            sh[wid][3] = m1;
            sh[wid][4] = bad;
        }
        __syncthreads();
        if (threadIdx.x < 5) {
            double t = sh[0][threadIdx.x];
            for (int w = 1; w < 8; ++w) {
                const double x = sh[w][threadIdx.x];
                t = threadIdx.x == 2 || threadIdx.x == 3 ? fmin(t, x) : t + x;
            }
            out[threadIdx.x] = t;
        }
    }
};

// One thread's share of a convergence check: each sum slot is a pair of FP32
// numbers (hi, lo) that TwoSum keeps equal to the exact running sum up to the
// rounding of lo (about twice FP32 precision); the maximum slot is a plain FP32
// maximum (exact).  FP64 arithmetic runs at a small fraction of the FP32 rate on
// this GPU, so FP64 is kept for the sums across warps and blocks.
struct CheckAcc {
    float hi[NRED], lo[NRED];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int q = 0; q < NRED; ++q) hi[q] = lo[q] = 0.0f;
    }
    __device__ __forceinline__ void add(int q, float x)
    {
        float e;
        hi[q] = two_sum(hi[q], x, e);
        lo[q] += e;
    }
    // an FP64 term: its FP32 head through TwoSum, the remainder into lo
    __device__ __forceinline__ void add_d(int q, double x)
    {
        const float h = __double2float_rn(x);
        add(q, h);
        lo[q] += __double2float_rn(x - (double)h);
    }
    // (x + y)^2, y below the rounding of x
    __device__ __forceinline__ void add_square(int q, float x, float y)
    {
        const float s = x * x;
        add(q, s);
        lo[q] += fmaf(x, x, -s) + 2.0f * x * y;
    }
    __device__ __forceinline__ void max(int q, float x) { hi[q] = fmaxf(hi[q], x); }
};

// The block's FP64 row of a check (NRED slots) from every thread's CheckAcc: warp
// sums of the (hi, lo) pairs in FP32 with TwoSum (fixed order), then the warps'
// pairs summed in FP64 by one thread per slot, in warp order.  NTH threads per
// block, numbered x fastest; every thread must call it.
template <int NTH>
__device__ __forceinline__ void block_sum_store(CheckAcc &a, double *dst)
{
    constexpr int NW = NTH / 32;
    __shared__ float sh[NW][NRED][2];
    const int tid = (int)(threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z));
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int q = 0; q < NRED; ++q) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float oh = __shfl_down_sync(0xffffffffu, a.hi[q], off);
            const float ol = __shfl_down_sync(0xffffffffu, a.lo[q], off);
            if (q == RED_MAX) {
                a.hi[q] = fmaxf(a.hi[q], oh);
            } else {
                float e;
                a.hi[q] = two_sum(a.hi[q], oh, e);
                a.lo[q] = a.lo[q] + (ol + e);
            }
        }
    }
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NRED; ++q) {
            sh[wid][q][0] = a.hi[q];
            sh[wid][q][1] = a.lo[q];
        }
    __syncthreads();
    if (tid < NRED) {
        double s = 0.0;
        for (int w = 0; w < NW; ++w)
            s = (tid == RED_MAX) ? fmax(s, (double)sh[w][tid][0]) : s + ((double)sh[w][tid][0] + (double)sh[w][tid][1]);
        dst[tid] = s;
    }
}

// ---------------------------------------------------------------- exchange words
// A 64-bit word carries one FP32 value in its low half and a 32-bit tag (the
// iteration it belongs to, plus one) in its high half.  Aligned 64-bit stores
// and loads are single-copy atomic, so a reader that sees the expected tag also
// sees the value written with it: no separate flag, no fence.
__device__ __forceinline__ void st_tagged(unsigned long long *p, float v, uint32_t tag)
{
    unsigned long long w = ((unsigned long long)tag << 32) | (unsigned long long)__float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long *p)
{
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
}

__device__ __forceinline__ uint32_t ld_relaxed32(const uint32_t *p)
{
    uint32_t w;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
    return w;
}

__device__ __forceinline__ uint32_t ld_acquire32(const uint32_t *p)
{
    uint32_t w;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
    return w;
}

__device__ __forceinline__ void st_release32(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ double ld_relaxed_f64(const double *p)
{
    double w;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(w) : "l"(p) : "memory");
    return w;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Control words of a resident launch (device memory, zeroed before the launch).
struct ResCtl {
    uint32_t abort;     // set by the first wait that runs out of time
    uint32_t where;     // which wait gave up (diagnostics)
};

constexpr uint64_t kWaitBudgetNs = 2000000000ull;   // default limit of one wait: 2 s


}  // namespace dev
}  // namespace vomt
