// Marching form of the streaming engine (march2d.cuh, march2d.cu): interface of its units.
#pragma once

#include "internal.h"

namespace vomt {
namespace march {

// A vector problem as the kernels see it: step constants and one entry per pair of channels.
struct MarchOp {
    int n, l, reg;
    float ih, mu, nu, tau, alpha;
    float g1, g2;                     // the primal step takes g2 (g1 (difference)): (ih, mu) or (1, mu ih)
    float tu, tw;                     // thresholds of the shrinks
    float eps, su, sw;
    float inv[LVEC];                  // 1 / c_e (0: no edge)
    int edge[LVEC];                   // the caller's edge number (-1: no edge)
};

struct MarchArgs {
    const float4 *in;                 // state
    float4 *out;                      // state after S iterations
    float4 *prev;                     // state after S - 1 iterations (nullptr: not wanted)
    const float4 *b;                  // rho1 - rho0
    const DevStatus *st;
    int rows, strips, warps;          // rows of a chunk, strips across the grid, warps in all
};

struct CheckArgs {
    const float4 *cur, *prv, *b;
    double *partials;
    const DevStatus *st;
    int rows, strips, items;
};

struct PlanarArgs {
    const float *rho0, *rho1;
    float *u, *w, *phi;
    int warm;
};

constexpr int kStages[3] = {1, 2, 4};   // iterations per pass of Kernels::step

struct Kernels {
    void (*step[3])(const MarchArgs, const MarchOp);
    void (*check)(const CheckArgs, const MarchOp);
    void (*in)(const PlanarArgs, const MarchOp, float4 *, float4 *);
    void (*out)(const PlanarArgs, const MarchOp, const float4 *, const float4 *, const DevStatus *);
    int groups, bgroups;              // groups of four values of a point: state, b
    int smem;                         // shared memory of a step
};

Kernels pick_k12(int k, int un, int wn, bool reg, bool res);
Kernels pick_k3(int k, int un, int wn, bool reg, bool res);
Kernels pick_k4(int k, int un, int wn, bool reg, bool res);
Kernels pick_k5(int k, int un, int wn, bool reg, bool res);
Kernels pick_k6(int k, int un, int wn, bool reg, bool res);
Kernels pick_k7(int k, int un, int wn, bool reg, bool res);
Kernels pick_k8(int k, int un, int wn, bool reg, bool res);

}  // namespace march

bool march_op(const OpDev &g, const StepDev &s, march::MarchOp *out);

}  // namespace vomt
