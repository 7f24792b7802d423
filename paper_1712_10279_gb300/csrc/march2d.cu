// Marching form of the streaming engine: host side (kernels in march2d.cuh).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "march2d.h"

namespace vomt {

// The pairwise form of a channel graph's operator: every row of G is +1/c_e at one channel
// and -1/c_e at a later one, Dv its transpose, all weights 1.  False for any other operator
// (matrix fields).
bool march_op(const OpDev &g, const StepDev &s, march::MarchOp *out)
{
    if (g.k < 1 || g.k > KVEC || g.l > LVEC) return false;
    march::MarchOp m;
    memset(&m, 0, sizeof m);
    for (int e = 0; e < LVEC; ++e) m.edge[e] = -1;
    for (int c = 0; c < g.k; ++c)
        if (g.wc[c] != 1.0f) return false;
    for (int e = 0; e < g.l; ++e) {
        int lo = -1, hi = -1;
        for (int c = 0; c < g.k; ++c) {
            if (g.Dv[c][e] != g.G[e][c]) return false;
            if (g.G[e][c] == 0.0f) continue;
            if (lo < 0) lo = c;
            else if (hi < 0) hi = c;
            else return false;
        }
        if (lo < 0) continue;                     // 1 / cost is 0 in FP32: any free pair, below
        if (hi < 0 || g.we[e] != 1.0f || !(g.G[e][lo] > 0.0f) || g.G[e][hi] != -g.G[e][lo]) return false;
        const int q = lo * (2 * g.k - lo - 1) / 2 + hi - lo - 1;
        if (m.edge[q] >= 0) return false;
        m.edge[q] = e;
        m.inv[q] = g.G[e][lo];
    }
    for (int e = 0; e < g.l; ++e) {
        bool set = false;
        for (int q = 0; q < LVEC; ++q) set = set || m.edge[q] == e;
        for (int q = 0; !set && q < g.k * (g.k - 1) / 2; ++q)
            if (m.edge[q] < 0) {
                m.edge[q] = e;
                set = true;
            }
        if (!set) return false;
    }
    m.n = s.n;
    m.l = g.l;
    m.reg = s.reg;
    m.ih = s.ih;
    m.mu = s.mu;
    m.nu = s.nu;
    m.tau = s.tau;
    m.alpha = s.alpha;
    m.eps = s.eps;
    m.g1 = s.ih;
    m.g2 = s.mu;
    m.tu = s.reg ? s.mu * s.su : s.mu;
    m.tw = s.reg ? s.alpha * s.nu * s.sw : s.alpha * s.nu;
    m.su = s.reg ? s.su : 1.0f;
    m.sw = s.reg ? s.sw : 1.0f;
    *out = m;
    return true;
}

bool edges_in_order(const march::MarchOp &m)
{
    int last = -1;
    for (int q = 0; q < LVEC; ++q)
        if (m.edge[q] >= 0) {
            if (m.edge[q] < last) return false;
            last = m.edge[q];
        }
    return true;
}

namespace {

using namespace march;

constexpr int kWarps = 4;             // warps per block (march2d.cuh)
constexpr int kSmemBlock = 227 * 1024;    // most shared memory of a block
constexpr int kSmemSM = 228 * 1024;   // shared memory of an SM (each block takes 1 KB besides its own)

Kernels pick(int k, int un, int wn, bool reg, bool res)
{
    switch (k) {
        case 1:
        case 2: return pick_k12(k, un, wn, reg, res);
        case 3: return pick_k3(k, un, wn, reg, res);
        case 4: return pick_k4(k, un, wn, reg, res);
        case 5: return pick_k5(k, un, wn, reg, res);
        case 6: return pick_k6(k, un, wn, reg, res);
        case 7: return pick_k7(k, un, wn, reg, res);
        default: return pick_k8(k, un, wn, reg, res);
    }
}

// One kind of pass: its stages, chunks and estimated time.
struct Pass {
    int stages = 0, rows = 0, strips = 0, warps = 0, blocks = 0;
    double us = 0.0;
    int smem = 0;
};

// Chunk rows of a pass with S stages: those of the least arithmetic time.  A warp takes
// rows + 2 S row-steps of S stages; a stage of a row costs a scheduler `issue` cycles when
// enough warps share it and `lat` cycles when a warp is alone (the chain through two
// shuffles and a reciprocal square root).  The estimate adds what every pass costs besides
// (launch, first rows, last stores) and is no shorter than the pass's bytes take: 6.3 TB/s
// from HBM, 12 TB/s where the states stay in L2.  Against every chunk length on a GB300 its
// choice was within 5% of the fastest for k = 1, 2, 3, 5, 6, 8 and n = 32 .. 2048.
Pass plan_pass(int n, int k, int groups, int S, int blocks_per_sm, int sms)
{
    const double issue = 20.0 + 40.0 * k + 4.0 * k * (k - 1), lat = 180.0, ghz = 1.95;
    const int W = 32 - 2 * S, strips = (n + W - 1) / W;
    const long cap = (long)blocks_per_sm * sms;
    Pass best;
    for (int chunks = 1; chunks <= n; ++chunks) {
        const int rows = (n + chunks - 1) / chunks;
        if (chunks > 1 && (n + rows - 1) / rows != chunks) continue;       // the same rows again
        const long warps = (long)strips * chunks, blocks = (warps + kWarps - 1) / kWarps;
        if (blocks > (1l << 30)) break;
        const long full = blocks / cap, rest = blocks % cap;
        const double per_sched = (double)kWarps / 4.0;                    // warps a block puts on a scheduler
        double cycles = (double)full * std::max(lat, issue * per_sched * blocks_per_sm);
        if (rest) cycles += std::max(lat, issue * per_sched * ceil((double)rest / sms));
        const double us = cycles * S * (rows + 2 * S) / (ghz * 1e3);
        if (best.stages == 0 || us < best.us) best = Pass{S, rows, strips, (int)warps, (int)blocks, us};
    }
    const double mb = 16e-6 * n * n * (2 * groups + (k + 3) / 4);
    best.us = 3.5 + std::max(best.us, mb / (mb > 110.0 ? 6.3 : 12.0));
    return best;
}

// How the host learns that a solve with a tolerance has stopped.  After a check it queues a
// copy of the status blocks, goes on queueing work, and reads the copy once another kLead
// microseconds of work (by the passes' estimates) are queued behind it, so that the GPU has
// work while the host waits; after the deciding check no more than that runs, as empty
// passes of under 2 us.  A copy takes the GPU a few microseconds between two kernels: one
// after the first check, then at growing distances, kGap at most.
struct StopPoll {
    static constexpr double kLead = 80.0, kGap = 150.0;
    const bool on;
    const cudaStream_t st;
    const DevStatus *const dev;
    DevStatus *const host;               // pinned, `count` blocks
    const int count;
    cudaEvent_t ev = nullptr;
    bool pending = false;
    double clock = 0.0, collect_at = 0.0, due = 0.0, gap = 10.0;
    cudaError_t error = cudaSuccess;
    StopPoll(bool on_, cudaStream_t s, const DevStatus *d, DevStatus *h, int n) : on(on_), st(s), dev(d), host(h), count(n)
    {
        if (on) error = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    }
    ~StopPoll()
    {
        if (ev) cudaEventDestroy(ev);
    }
    void queued(double us) { clock += us; }
    void checked()                       // a check has been queued
    {
        clock += kCheckUs;
        if (!on || pending || clock < due || error != cudaSuccess) return;
        error = cudaMemcpyAsync(host, dev, sizeof(DevStatus) * count, cudaMemcpyDeviceToHost, st);
        if (error == cudaSuccess) error = cudaEventRecord(ev, st);
        pending = error == cudaSuccess;
        collect_at = clock + kLead;
        due = clock + gap;
        gap = std::min(2.0 * gap, kGap);
    }
    const DevStatus *arrived()           // the status of the last copy, once it is time to read it
    {
        if (!pending || clock < collect_at) return nullptr;
        pending = false;
        error = cudaEventSynchronize(ev);
        return error == cudaSuccess ? host : nullptr;
    }
    static constexpr double kCheckUs = 12.0;
};

// The pass to launch next, m iterations before a check: fewer-stage passes first.
int next_pass(const Pass (&pass)[3], int main_pass, int m)
{
    const int odd = m % kStages[main_pass];
    if (odd == 0) return main_pass;
    int r = main_pass - 1;
    while (r > 0 && (!pass[r].stages || odd < kStages[r])) --r;
    return r;
}

}  // namespace

// The solve of stream_solve for vector problems.  *taken = false (and VOMT_OK) where this
// form does not apply: operators other than a channel graph's, state that does not fit the
// device's memory, and up to four channels with fewer than four iterations between checks,
// where the one-iteration kernels need no second layout and are as fast (2048^2, three
// channels: 79 us against 84 with one stage).
int march_solve(vomt_ctx *ctx, const OpDev &g, const StepDev &s, const SolveCfg &cfg, const vomt_params &p, bool res,
                const float *rho0, const float *rho1, float *u, float *w, float *phi, cudaStream_t st, bool *taken)
{
    *taken = false;
    MarchOp op;
    if (p.u_norm > VOMT_U_L1 || p.w_norm > VOMT_W_L2 || !march_op(g, s, &op) || !edges_in_order(op)) return VOMT_OK;
    const int n = s.n, k = g.k;
    const int interval = std::min(p.check_every, std::max(p.max_iters, 0));
    if (k <= 4 && interval < 4) return VOMT_OK;
    // the kernels' reciprocal square root takes sums of squares below 1.2e-38 for zero, which
    // is right where the threshold is above their root
    if (op.tu < 2e-19f || (g.l > 0 && op.tw < 2e-19f)) return VOMT_OK;
    if (res) {
        op.g1 = 1.0f;
        op.g2 = s.mu * s.ih;
    }
    const Kernels K = pick(k, p.u_norm, p.w_norm, s.reg != 0, res);

    Pass pass[3];
    int main_pass = 0;
    for (int q = 0; q < 3; ++q) {
        if (!K.step[q]) continue;
        cudaError_t e = cudaFuncSetAttribute((const void *)K.step[q], cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBlock);
        int per_sm = 0;
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)K.step[q], 32 * kWarps, K.smem);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "marching kernel");
        if (per_sm < 1) continue;
        pass[q] = plan_pass(n, k, K.groups, kStages[q], per_sm, ctx->sm_count);
        if (kStages[q] <= std::max(interval, 1) &&
            (pass[main_pass].stages == 0 || pass[q].us / kStages[q] < pass[main_pass].us / kStages[main_pass]))
            main_pass = q;
    }
    if (pass[0].stages == 0) return VOMT_OK;
    // A pass starts while the one before it drains, and would fill whatever slots are free
    // by then, three blocks on some SMs and one on others (2048^2, three channels, two blocks
    // per SM: 140 us a pass instead of 100).  So each pass asks for the shared memory that
    // leaves room for just its share of blocks per SM.
    for (int q = 0; q < 3; ++q) {
        if (!pass[q].stages) continue;
        const int share = (pass[q].blocks + ctx->sm_count - 1) / ctx->sm_count;
        pass[q].smem = std::max(K.smem, kSmemSM / (share + 1));
    }

    // b, two states, and the state one iteration before a check where a pass of several
    // iterations ends on it
    const int states = main_pass > 0 ? 3 : 2;
    const size_t state4 = (size_t)n * ((n + 31) / 32) * K.groups * 32, b4 = (size_t)n * ((n + 31) / 32) * K.bgroups * 32;
    int rc = ensure_buffer(ctx, (void **)&ctx->ws, &ctx->ws_floats, sizeof(float4) * (b4 + states * state4), "workspace");
    if (rc) {
        ctx->err.clear();
        return VOMT_OK;
    }
    float4 *b = (float4 *)ctx->ws, *S[3] = {b + b4, b + b4 + state4, b + b4 + 2 * state4};

    // the check: strips of 30 columns, chunks that give every SM work, at most kMetricBlocks
    // blocks (k_finalize adds a row per block: with 998 blocks at 1024^2 it took 14.7 us, with
    // 604 9.2)
    CheckArgs ca;
    memset(&ca, 0, sizeof ca);
    ca.strips = (n + 29) / 30;
    ca.rows = std::max(4, (int)(((long)ca.strips * n + (long)kMetricBlocks * kWarps - 1) / ((long)kMetricBlocks * kWarps)));
    ca.items = ca.strips * ((n + ca.rows - 1) / ca.rows);
    const int mblocks = std::min((ca.items + kWarps - 1) / kWarps, kMetricBlocks);
    rc = ensure_buffer(ctx, (void **)&ctx->partials, &ctx->partials_cap, sizeof(double) * (size_t)mblocks * NRED, "partials");
    if (rc) return rc;
    ca.partials = ctx->partials;
    ca.b = b;
    ca.st = ctx->dstatus;
    rc = ensure_history(ctx, p.max_iters / p.check_every + 2);
    if (rc) return rc;
    cudaError_t e = cudaMemsetAsync(ctx->dstatus, 0, sizeof(DevStatus), st);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "status reset");
    *taken = true;
    ctx->last_form = VOMT_FORM_MARCH;
    ctx->hist_raw = false;           // k_finalize writes finished rows
    ctx->last_blocks = pass[main_pass].blocks;

    const PlanarArgs planar{rho0, rho1, u, w, phi, p.warm_start};
    const dim3 lgrid((n + 127) / 128, std::min(n, 2048));
    K.in<<<lgrid, 128, 0, st>>>(planar, op, S[0], b);
    ctx->launches += 1;

    int cur = 0;                     // the state that holds the iterate
    const float4 *before = S[0];     // its predecessor, after `run` with `last`
    auto one = [&](int q, bool last) {
        const Pass &ps = pass[q];
        MarchArgs a;
        a.in = S[cur];
        a.out = S[cur ^ 1];
        a.prev = last && ps.stages > 1 ? S[2] : nullptr;
        a.b = b;
        a.st = ctx->dstatus;
        a.rows = ps.rows;
        a.strips = ps.strips;
        a.warps = ps.warps;
        launch_pdl(K.step[q], dim3(ps.blocks), dim3(32 * kWarps), (size_t)ps.smem, st, a, op);
        ctx->launches += 1;
        before = a.prev ? a.prev : a.in;
        cur ^= 1;
    };
    auto check = [&](int t) {
        CheckArgs c = ca;
        c.cur = S[cur];
        c.prv = before;
        launch_pdl(K.check, dim3(mblocks), dim3(32 * kWarps), 0, st, c, op);
        launch_pdl(k_finalize, dim3(1), dim3(kFinThreads), 0, st, (const double *)ctx->partials, mblocks, cfg, t,
                   ctx->dstatus, ctx->dhist, ctx->hist_cap, cur);
        ctx->launches += 2;
    };
    if (p.max_iters == 0) check(0);
    StopPoll poll(cfg.tol_gap > 0.0, st, ctx->dstatus, ctx->hstatus, 1);
    auto stopped = [&]() {
        const DevStatus *h = poll.arrived();
        return poll.error != cudaSuccess || (h && h->stop);
    };
    bool stop = false;
    for (int t = 0; t < p.max_iters && !stop;) {
        for (int m = std::min(p.check_every, p.max_iters - t); m > 0 && !stop;) {
            const int q = next_pass(pass, main_pass, m);
            one(q, m == kStages[q]);
            m -= kStages[q];
            t += kStages[q];
            poll.queued(pass[q].us);
            stop = stopped();
        }
        if (stop) break;
        check(t);
        poll.checked();
        stop = stopped();
    }
    K.out<<<lgrid, 128, 0, st>>>(planar, op, S[0], S[1], ctx->dstatus);
    ctx->launches += 1;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = poll.error;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&ctx->hstatus[0], ctx->dstatus, sizeof(DevStatus), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "solve");
    return VOMT_OK;
}

// ------------------------------------------------------------------ batches
__global__ void k_finalize_many(const march::BatchItem *__restrict__ items, int t, int slot);

void march_scratch_free(BatchMarchScratch *s)
{
    cudaFree(s->items);
    cudaFree(s->maps);
    cudaFree(s->data);
    cudaFree(s->stat);
    if (s->hstat) cudaFreeHost(s->hstat);
    *s = BatchMarchScratch();
}

namespace {

// A check's chunk of rows for `strip_rows` rows of strips: 16 warps per SM, enough to hide
// the loads of a row (8 x 256^2, three channels: 140 us with 8 blocks a problem, 30 so).
int check_chunk(long strip_rows, int sms) { return (int)std::max(2l, (strip_rows + 16l * sms - 1) / (16l * sms)); }

// The problems of one channel count: passes over those still running at once, with chunks of
// the same number of rows in every problem.
struct Group {
    int k = 0, main_pass = 0;
    std::vector<int> probs, live;     // all its problems; those the passes below are planned for
    std::vector<std::pair<int, int>> sides;       // of the live ones: side, how many
    double points = 0.0;              // of the live ones
    Kernels K;
    int per_sm[3] = {0, 0, 0};
    Pass pass[3];                     // blocks: of the whole group
    int check_rows = 2, check_blocks = 0;
    int first_live = 0;               // its first item of the pass tables
    size_t map_at[4] = {0, 0, 0, 0};  // block maps of its three passes and its check
    int cur = 0, before = 0;          // states that hold the iterates and their predecessors
};

// plan_pass for a group: the chunk length of the least arithmetic time
Pass plan_group(const Group &gr, int S, int blocks_per_sm, int sms)
{
    const int k = gr.k, W = 32 - 2 * S;
    const double issue = 20.0 + 40.0 * k + 4.0 * k * (k - 1), lat = 180.0, ghz = 1.95;
    const long cap = (long)blocks_per_sm * sms;
    const int top = gr.sides.back().first;
    Pass best;
    for (int rows = 1; rows <= top; rows += rows < 32 ? 1 : rows / 16) {
        long blocks = 0, warps = 0;
        for (const auto &side : gr.sides) {
            const int n = side.first;
            const long w = (long)((n + W - 1) / W) * ((n + rows - 1) / rows);
            warps += w * side.second;
            blocks += (w + kWarps - 1) / kWarps * side.second;
        }
        if (blocks > (1l << 30)) continue;
        const long full = blocks / cap, rest = blocks % cap;
        double cycles = (double)full * std::max(lat, issue * blocks_per_sm);
        if (rest) cycles += std::max(lat, issue * ceil((double)rest / sms));
        const double us = cycles * S * (rows + 2 * S) / (ghz * 1e3);
        if (best.stages == 0 || us < best.us) best = Pass{S, rows, 0, (int)warps, (int)blocks, us};
    }
    const double mb = 16e-6 * gr.points * (2 * gr.K.groups + (k + 3) / 4);
    best.us = 3.5 + std::max(best.us, mb / (mb > 110.0 ? 6.3 : 12.0));
    return best;
}

// The passes and the check of a group's live problems; n: the problems' sides.
void plan_live(const std::vector<int> &n, Group &g, int interval, int sms)
{
    std::vector<int> s;
    for (int q : g.live) s.push_back(n[q]);
    std::sort(s.begin(), s.end());
    g.sides.clear();
    g.points = 0.0;
    long strip_rows = 0;
    for (int side : s) {
        if (g.sides.empty() || g.sides.back().first != side) g.sides.push_back({side, 0});
        g.sides.back().second += 1;
        g.points += (double)side * side;
        strip_rows += (long)((side + 29) / 30) * side;
    }
    g.check_rows = check_chunk(strip_rows, sms);
    g.main_pass = 0;
    for (int q = 0; q < 3 && !s.empty(); ++q) {
        if (g.per_sm[q] < 1) continue;
        Pass &ps = g.pass[q];
        ps = plan_group(g, kStages[q], g.per_sm[q], sms);
        const int share = (ps.blocks + sms - 1) / sms;      // see march_solve
        ps.smem = std::max(g.K.smem, kSmemSM / (share + 1));
        if (kStages[q] <= interval && (g.pass[g.main_pass].stages == 0 ||
                                       ps.us / kStages[q] < g.pass[g.main_pass].us / kStages[g.main_pass]))
            g.main_pass = q;
    }
}

// A problem's side and channel count are all that its passes are planned from.
int plan_groups(vomt_ctx *ctx, BatchMarchScratch *scr, const std::vector<int> &n, const std::vector<int> &ks,
                const vomt_params &p, std::vector<Group> *out)
{
    out->clear();
    const int interval = std::max(1, std::min(p.check_every, p.max_iters));
    for (int k = 1; k <= 5; ++k) {
        Group g;
        g.k = k;
        for (int q = 0; q < (int)n.size(); ++q)
            if (ks[q] == k) g.probs.push_back(q);
        if (g.probs.empty()) continue;
        g.live = g.probs;
        g.K = pick(k, VOMT_U_L12, VOMT_W_L1, false, true);
        for (int q = 0; q < 3; ++q) {
            if (!g.K.many[q]) continue;
            int &per_sm = scr->per_sm[k - 1][q];
            if (per_sm < 0) {
                int got = 0;
                cudaError_t e = cudaFuncSetAttribute((const void *)g.K.many[q],
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBlock);
                if (e == cudaSuccess)
                    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, (const void *)g.K.many[q], 32 * kWarps,
                                                                      g.K.smem);
                if (e != cudaSuccess) return set_cuda_error(ctx, e, "marching kernel");
                per_sm = got;
            }
            g.per_sm[q] = per_sm;
        }
        if (g.per_sm[0] < 1) return VOMT_ERR_TOO_LARGE;
        plan_live(n, g, interval, ctx->sm_count);
        if (g.pass[0].stages == 0) return VOMT_ERR_TOO_LARGE;
        out->push_back(g);
    }
    return VOMT_OK;
}

// Pass tables of the live problems, group by group: an item each and, per pass and check,
// the problem of every block.  Fills the groups' places in them.
struct Tables {
    std::vector<BatchItem> items;
    std::vector<int> maps;
    size_t sum_rows = 0;
};
Tables build_tables(const std::vector<BatchProblem> &probs, std::vector<Group> &groups,
                    const std::vector<BatchItem> &base, const std::vector<int> &slot_of, double *sums,
                    std::vector<int> *blocks)
{
    Tables t;
    for (Group &g : groups) {
        int next[4] = {0, 0, 0, 0};
        std::vector<int> gm[4];
        g.first_live = (int)t.items.size();
        for (size_t i = 0; i < g.live.size(); ++i) {
            const int q = g.live[i], n = probs[q].g.n;
            BatchItem d = base[slot_of[q]];
            for (int c = 0; c < 3; ++c) {
                if (!g.pass[c].stages) continue;
                const int W = 32 - 2 * kStages[c];
                d.pass[c].rows = std::min(g.pass[c].rows, n);
                d.pass[c].strips = (n + W - 1) / W;
                d.pass[c].warps = d.pass[c].strips * ((n + d.pass[c].rows - 1) / d.pass[c].rows);
                d.pass[c].first = next[c];
                const int nb = (d.pass[c].warps + kWarps - 1) / kWarps;
                gm[c].insert(gm[c].end(), nb, (int)i);
                next[c] += nb;
                if (c == g.main_pass) (*blocks)[q] = nb;
            }
            d.check_strips = (n + 29) / 30;
            d.check_rows = g.check_rows;
            d.check_items = d.check_strips * ((n + d.check_rows - 1) / d.check_rows);
            d.check_blocks = (d.check_items + kWarps - 1) / kWarps;
            d.check_first = next[3];
            d.partials = sums + (t.sum_rows + next[3]) * NRED;
            gm[3].insert(gm[3].end(), d.check_blocks, (int)i);
            next[3] += d.check_blocks;
            t.items.push_back(d);
        }
        for (int c = 0; c < 4; ++c) {
            g.map_at[c] = t.maps.size();
            t.maps.insert(t.maps.end(), gm[c].begin(), gm[c].end());
            if (c < 3) g.pass[c].blocks = next[c];
        }
        g.check_blocks = next[3];
        t.sum_rows += next[3];
    }
    return t;
}

}  // namespace

namespace {

constexpr int kMaxPart = 65535;      // problems of a part: a launch's third dimension

// Bytes of a problem's three states and b.
size_t state_bytes(int n, int k)
{
    const size_t l = (size_t)k * (k - 1) / 2, tile = (size_t)n * ((n + 31) / 32) * 32;
    return sizeof(float4) * tile * (3 * ((3 * k + l + 3) / 4) + (k + 3) / 4);
}

// Runs of problems that are advanced together: as many as fit the context's memory limit and
// a launch's third dimension.  The first problem of each, and the end; empty where one problem
// alone does not fit.
std::vector<int> batch_parts(const vomt_ctx *ctx, const std::vector<int> &n, const std::vector<int> &k)
{
    std::vector<int> first;
    size_t bytes = 0;
    for (int q = 0; q < (int)n.size(); ++q) {
        const size_t need = state_bytes(n[q], k[q]);
        if (need > ctx->spare_bytes) return {};
        if (q == 0 || bytes + need > ctx->spare_bytes || q - first.back() == kMaxPart) {
            first.push_back(q);
            bytes = 0;
        }
        bytes += need;
    }
    first.push_back((int)n.size());
    return first;
}

}  // namespace

double march_batch_estimate(vomt_ctx *ctx, BatchMarchScratch *scr, const std::vector<int> &n,
                            const std::vector<int> &k, const vomt_params &p)
{
    const std::vector<int> first = batch_parts(ctx, n, k);
    double us = first.empty() ? 1e30 : 0.0;
    for (size_t i = 0; i + 1 < first.size(); ++i) {
        std::vector<Group> groups;
        if (plan_groups(ctx, scr, {n.begin() + first[i], n.begin() + first[i + 1]},
                        {k.begin() + first[i], k.begin() + first[i + 1]}, p, &groups))
            return 1e30;
        for (const Group &g : groups) us += g.pass[g.main_pass].us / kStages[g.main_pass];
    }
    return us;
}

// The problems of a channel count advance together, a pass over all of them per launch.
// Eight pairs at 256^2 with three channels take 5.6 us per iteration together, where one
// after another on every SM (the grouped resident form) they take 8 x 1.6.  A problem that
// has stopped still costs its blocks the copies of a chunk's first rows, and the chunks of
// the others stay as long as they were planned with it, so when a quarter of a group's points
// has stopped, its passes are planned again for the problems left.
static int march_part(vomt_ctx *ctx, BatchMarchScratch *scr, const std::vector<BatchProblem> &probs, const vomt_params &p,
                      cudaStream_t st, std::vector<DevStatus> *status, std::vector<int> *blocks, bool *taken)
{
    *taken = false;
    const int count = (int)probs.size(), sms = ctx->sm_count;
    std::vector<int> side(count), ks(count);
    for (int q = 0; q < count; ++q) {
        side[q] = probs[q].g.n;
        ks[q] = probs[q].k;
    }
    std::vector<Group> groups;
    int rc = plan_groups(ctx, scr, side, ks, p, &groups);
    if (rc) return rc == VOMT_ERR_TOO_LARGE ? VOMT_OK : rc;
    // scratch: per problem b, two states, the state before a check; check sums (rows for any
    // subset of the problems: check_chunk gives 16 warps per SM, a partly filled chunk per
    // strip and a partly filled block per problem); tables
    size_t floats4 = 0, sum_rows = 0;
    std::vector<size_t> off(count);
    for (const Group &g : groups) {
        size_t strips = 0;
        for (int q : g.probs) {
            const size_t n = probs[q].g.n, tile = n * ((n + 31) / 32) * 32;
            off[q] = floats4;
            floats4 += tile * (3 * (size_t)g.K.groups + g.K.bgroups);
            strips += (n + 29) / 30;
        }
        sum_rows += (16 * (size_t)sms + strips) / kWarps + g.probs.size() + 1;
    }
    const size_t sums = sizeof(double) * NRED * sum_rows;
    rc = ensure_buffer(ctx, &scr->data, &scr->data_cap, sizeof(float4) * floats4 + sums, "batch states");
    if (rc) {
        ctx->err.clear();
        return VOMT_OK;
    }
    rc = ensure_buffer(ctx, &scr->items, &scr->items_cap, 2 * sizeof(BatchItem) * count, "batch tables");
    if (!rc) rc = ensure_buffer(ctx, &scr->stat, &scr->stat_cap, sizeof(DevStatus) * count, "batch status");
    if (rc) return rc;
    if (scr->hstat_cap < 2 * sizeof(DevStatus) * count) {
        if (scr->hstat) cudaFreeHost(scr->hstat);
        scr->hstat = nullptr;
        scr->hstat_cap = 0;
        cudaError_t e = cudaMallocHost(&scr->hstat, 2 * sizeof(DevStatus) * count);
        if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch status");
        scr->hstat_cap = 2 * sizeof(DevStatus) * count;
    }
    float4 *data = (float4 *)scr->data;
    double *dsums = (double *)(data + floats4);
    DevStatus *dstat = (DevStatus *)scr->stat, *hstat = (DevStatus *)scr->hstat;
    // what does not depend on the passes, all problems group by group
    std::vector<BatchItem> base(count);
    std::vector<int> slot_of(count), first_item(groups.size()), top(groups.size(), 0);
    int at = 0;
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        const Group &g = groups[gi];
        first_item[gi] = at;
        for (int q : g.probs) {
            const int n = probs[q].g.n;
            const size_t tile = (size_t)n * ((n + 31) / 32) * 32;
            BatchItem &d = base[at];
            memset(&d, 0, sizeof d);
            d.g = probs[q].g;
            d.g.g1 = 1.0f;
            d.g.g2 = d.g.mu * d.g.ih;
            d.cfg = probs[q].cfg;
            d.planar = probs[q].planar;
            d.b = data + off[q];
            for (int c = 0; c < 3; ++c) d.S[c] = d.b + tile * (g.K.bgroups + (size_t)c * g.K.groups);
            d.st = dstat + at;
            slot_of[q] = at++;
            top[gi] = std::max(top[gi], n);
        }
    }
    blocks->assign(count, 1);
    std::vector<Tables> plans;           // kept until the copies from them are done
    plans.push_back(build_tables(probs, groups, base, slot_of, dsums, blocks));
    // (room for the maps of a later plan: blocks of up to a wave more per pass and check)
    rc = ensure_buffer(ctx, &scr->maps, &scr->maps_cap,
                       sizeof(int) * (plans[0].maps.size() + 4 * 8 * (size_t)sms * groups.size()), "batch tables");
    if (rc) return rc;
    BatchItem *const ditems = (BatchItem *)scr->items, *const dlive = ditems + count;
    int *const dmaps = (int *)scr->maps;
    // The kernels read the tables before they wait for the kernel before them, so the first one
    // after a copy of new tables is launched as an ordinary kernel, after the copy.
    bool fresh = true;
    auto launch = [&](auto kern, unsigned grid, unsigned block, size_t smem, auto... args) {
        if (fresh)
            kern<<<grid, block, smem, st>>>(args...);
        else
            launch_pdl(kern, dim3(grid), dim3(block), smem, st, args...);
        fresh = false;
        ctx->launches += 1;
    };
    auto upload = [&]() {
        fresh = true;
        const Tables &t = plans.back();
        cudaError_t r = cudaMemcpyAsync(dlive, t.items.data(), sizeof(BatchItem) * t.items.size(), cudaMemcpyHostToDevice, st);
        return r != cudaSuccess ? r : cudaMemcpyAsync(dmaps, t.maps.data(), sizeof(int) * t.maps.size(),
                                                      cudaMemcpyHostToDevice, st);
    };
    cudaError_t e = cudaMemcpyAsync(ditems, base.data(), sizeof(BatchItem) * count, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = upload();
    if (e == cudaSuccess) e = cudaMemsetAsync(dstat, 0, sizeof(DevStatus) * count, st);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch tables");
    *taken = true;
    auto layout_grid = [&](size_t gi) {
        return dim3((top[gi] + 127) / 128, std::min(top[gi], 256), (unsigned)groups[gi].probs.size());
    };
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        groups[gi].K.in_many<<<layout_grid(gi), 128, 0, st>>>(ditems + first_item[gi]);
        ctx->launches += 1;
    }
    auto one = [&](Group &g, int q, bool last) {
        const int prev = last && kStages[q] > 1 ? 1 : 0;
        launch(g.K.many[q], g.pass[q].blocks, 32 * kWarps, (size_t)g.pass[q].smem, (const BatchItem *)dlive + g.first_live,
               (const int *)dmaps + g.map_at[q], g.cur, prev);
        g.before = prev ? 2 : g.cur;
        g.cur ^= 1;
    };
    auto check = [&](Group &g, int t) {
        launch(g.K.check_many, g.check_blocks, 32 * kWarps, 0, (const BatchItem *)dlive + g.first_live,
               (const int *)dmaps + g.map_at[3], g.cur, g.before);
        launch(k_finalize_many, (unsigned)g.live.size(), kFinThreads, 0, (const BatchItem *)dlive + g.first_live, t, g.cur);
    };
    if (p.max_iters == 0)
        for (Group &g : groups) check(g, 0);
    StopPoll poll(p.tol_gap > 0.0, st, dstat, hstat, count);
    const int interval = std::max(1, std::min(p.check_every, p.max_iters));
    // plan the passes again for the problems that run on, where enough have stopped
    auto thin_out = [&](const DevStatus *h) -> cudaError_t {
        std::vector<std::vector<int>> live(groups.size());
        bool again = false;
        for (size_t gi = 0; gi < groups.size(); ++gi) {
            double left = 0.0;
            for (int q : groups[gi].live)
                if (!h[slot_of[q]].stop) {
                    live[gi].push_back(q);
                    left += (double)side[q] * side[q];
                }
            again = again || left < 0.75 * groups[gi].points;
        }
        if (!again) return cudaSuccess;
        std::vector<Group> next = groups;
        std::vector<int> nblocks = *blocks;
        for (size_t gi = 0; gi < groups.size(); ++gi) {
            next[gi].live = live[gi];
            plan_live(side, next[gi], interval, sms);
        }
        Tables t = build_tables(probs, next, base, slot_of, dsums, &nblocks);
        if (t.sum_rows > sum_rows || sizeof(int) * t.maps.size() > scr->maps_cap) return cudaSuccess;
        groups.swap(next);
        blocks->swap(nblocks);
        plans.push_back(std::move(t));
        return upload();
    };
    // whether the solve is over: all problems have stopped, or an error (in e or the poll's)
    auto stopped = [&]() {
        const DevStatus *h = poll.arrived();
        if (poll.error != cudaSuccess) return true;
        if (!h) return false;
        bool all = true;
        for (int q = 0; q < count; ++q) all = all && h[q].stop;
        if (!all) e = thin_out(h);
        return all || e != cudaSuccess;
    };
    bool stop = false;
    for (int t = 0; t < p.max_iters && !stop;) {
        const int m = std::min(p.check_every, p.max_iters - t);
        t += m;
        for (size_t gi = 0; gi < groups.size() && !stop; ++gi) {
            for (int left = m; left > 0 && !stop && !groups[gi].live.empty();) {
                Group &g = groups[gi];                // (planned anew at any poll)
                const int q = next_pass(g.pass, g.main_pass, left);
                one(g, q, left == kStages[q]);
                left -= kStages[q];
                poll.queued(g.pass[q].us);
                stop = stopped();
            }
            if (stop || groups[gi].live.empty()) continue;
            check(groups[gi], t);
            if (gi + 1 < groups.size()) poll.queued(StopPoll::kCheckUs);
        }
        if (stop) break;
        poll.checked();
        stop = stopped();
    }
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        groups[gi].K.out_many<<<layout_grid(gi), 128, 0, st>>>(ditems + first_item[gi]);
        ctx->launches += 1;
    }
    if (e == cudaSuccess) e = poll.error;
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(hstat, dstat, sizeof(DevStatus) * count, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch solve");
    status->resize(count);
    for (int q = 0; q < count; ++q) (*status)[q] = hstat[slot_of[q]];
    return VOMT_OK;
}

// The parts of a batch one after the other, in the same scratch.
int march_batch(vomt_ctx *ctx, BatchMarchScratch *scr, const std::vector<BatchProblem> &probs, const vomt_params &p,
                cudaStream_t st, std::vector<DevStatus> *status, std::vector<int> *blocks, bool *taken)
{
    *taken = false;
    std::vector<int> n, k;
    for (const BatchProblem &b : probs) {
        n.push_back(b.g.n);
        k.push_back(b.k);
    }
    const std::vector<int> first = batch_parts(ctx, n, k);
    if (first.empty()) return VOMT_OK;
    // the largest part's scratch before the first part runs: a part that has run cannot be
    // left to another path (check sums: march_part's bound, of up to five groups)
    size_t most = 0;
    for (size_t i = 0; i + 1 < first.size(); ++i) {
        size_t bytes = 0, rows = 5 * (4 * (size_t)ctx->sm_count + 2);
        for (int q = first[i]; q < first[i + 1]; ++q) {
            bytes += state_bytes(n[q], k[q]);
            rows += (size_t)(n[q] + 29) / 30 + 1;
        }
        most = std::max(most, bytes + sizeof(double) * NRED * rows);
    }
    if (ensure_buffer(ctx, &scr->data, &scr->data_cap, most, "batch states")) {
        ctx->err.clear();
        return VOMT_OK;
    }
    status->clear();
    blocks->clear();
    for (size_t i = 0; i + 1 < first.size(); ++i) {
        std::vector<DevStatus> s;
        std::vector<int> b;
        const int rc = march_part(ctx, scr, {probs.begin() + first[i], probs.begin() + first[i + 1]}, p, st, &s, &b, taken);
        if (rc) return rc;
        if (!*taken) return i == 0 ? VOMT_OK : fail(ctx, VOMT_ERR_CUDA, "batch states");
        status->insert(status->end(), s.begin(), s.end());
        blocks->insert(blocks->end(), b.begin(), b.end());
    }
    return VOMT_OK;
}

}  // namespace vomt
