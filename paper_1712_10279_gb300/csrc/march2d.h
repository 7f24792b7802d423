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

// One problem of a batch.
struct BatchItem {
    MarchOp g;
    float4 *S[3], *b;                 // two states, the state before a check, rho1 - rho0
    double *partials;
    DevStatus *st;
    SolveCfg cfg;
    PlanarArgs planar;
    struct {
        int rows, strips, warps, first;      // of a pass of 1, 2, 4 iterations; its first block
    } pass[3];
    int check_rows, check_strips, check_items, check_first, check_blocks;
};

constexpr int kStages[3] = {1, 2, 4};   // iterations per pass of Kernels::step

struct Kernels {
    void (*step[3])(const MarchArgs, const MarchOp);
    void (*check)(const CheckArgs, const MarchOp);
    void (*in)(const PlanarArgs, const MarchOp, float4 *, float4 *);
    void (*out)(const PlanarArgs, const MarchOp, const float4 *, const float4 *, const DevStatus *);
    // many problems at once (default norms, up to five channels, resident engine's order)
    void (*many[3])(const BatchItem *, const int *, int, int);
    void (*check_many)(const BatchItem *, const int *, int, int);
    void (*in_many)(const BatchItem *);
    void (*out_many)(const BatchItem *);
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
// whether its edges are listed in the order of the pairs: the marching form sums over the
// edges at a channel in that order, the other kernels in the listed one
bool edges_in_order(const march::MarchOp &m);

// A batch of vector problems (default norms, eps = 0, k <= 5) in the marching form, in the
// resident engine's order of operations (march2d.cu).
struct BatchProblem {
    march::MarchOp g;
    int k;
    SolveCfg cfg;
    march::PlanarArgs planar;
};
struct BatchMarchScratch {            // what march_batch keeps on its context
    void *items = nullptr, *maps = nullptr, *data = nullptr, *stat = nullptr, *hstat = nullptr;
    size_t items_cap = 0, maps_cap = 0, data_cap = 0, stat_cap = 0, hstat_cap = 0;
    // blocks per SM of each pass kernel (-1: its launch attributes are still to be set)
    int per_sm[5][3] = {{-1, -1, -1}, {-1, -1, -1}, {-1, -1, -1}, {-1, -1, -1}, {-1, -1, -1}};
};
void march_scratch_free(BatchMarchScratch *s);
// microseconds an iteration of problems with these sides and channel counts takes by estimate
double march_batch_estimate(vomt_ctx *ctx, BatchMarchScratch *scr, const std::vector<int> &n,
                            const std::vector<int> &k, const vomt_params &p);
// *taken = false where the memory is not to be had; status[q]: the host copy of each problem's
// final status block, blocks[q]: the blocks of its main pass
int march_batch(vomt_ctx *ctx, BatchMarchScratch *scr, const std::vector<BatchProblem> &probs, const vomt_params &p,
                cudaStream_t st, std::vector<DevStatus> *status, std::vector<int> *blocks, bool *taken);

}  // namespace vomt
