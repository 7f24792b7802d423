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

// How the host learns that a solve with a tolerance has stopped: each next() queues a copy of
// the status blocks and returns the copy before it once that has arrived (nullptr: none yet,
// or no tolerance), so the GPU always has the work queued since then to go on with.
struct StopPoll {
    const bool on;
    const cudaStream_t st;
    const DevStatus *const dev;
    DevStatus *const host;               // pinned, 2 * count blocks
    const int count;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    int calls = 0;
    cudaError_t error = cudaSuccess;
    StopPoll(bool on_, cudaStream_t s, const DevStatus *d, DevStatus *h, int n) : on(on_), st(s), dev(d), host(h), count(n)
    {
        for (int q = 0; q < 2 && on; ++q)
            if (error == cudaSuccess) error = cudaEventCreateWithFlags(&ev[q], cudaEventDisableTiming);
    }
    ~StopPoll()
    {
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
    }
    const DevStatus *next()
    {
        if (!on || error != cudaSuccess) return nullptr;
        const int slot = calls++ & 1;
        error = cudaMemcpyAsync(host + (size_t)slot * count, dev, sizeof(DevStatus) * count, cudaMemcpyDeviceToHost, st);
        if (error == cudaSuccess) error = cudaEventRecord(ev[slot], st);
        if (error != cudaSuccess || calls < 2) return nullptr;
        error = cudaEventSynchronize(ev[slot ^ 1]);
        return error == cudaSuccess ? host + (size_t)(slot ^ 1) * count : nullptr;
    }
};

// Estimated microseconds from one check to the next, `interval` iterations and the check.
double interval_us(const Pass (&pass)[3], int main_pass, int interval)
{
    const double us = pass[main_pass].stages ? pass[main_pass].us / pass[main_pass].stages : 0.0;
    return us * interval + 8.0;
}

// Checks from one poll to the next: about 150 us of work.  A poll costs the GPU a few
// microseconds between two kernels, and after the deciding check the work up to the second
// next poll still runs, as empty passes of about 2 us each.
int poll_every(double check_us) { return (int)std::min(std::max(150.0 / check_us, 1.0), 1024.0); }

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
    // m iterations, fewer-stage passes first
    auto run = [&](int m) {
        int q = main_pass, odd = m % kStages[q];
        for (int r = q - 1; r >= 0; --r)
            for (; pass[r].stages && odd >= kStages[r]; odd -= kStages[r], m -= kStages[r]) one(r, m == kStages[r]);
        for (; m > 0; m -= kStages[q]) one(q, m == kStages[q]);
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
    const int every = poll_every(interval_us(pass, main_pass, interval));
    int since = 0;
    bool stopped = false;
    for (int t = 0; t < p.max_iters && !stopped;) {
        const int m = std::min(p.check_every, p.max_iters - t);
        run(m);
        t += m;
        check(t);
        if (++since < every) continue;
        since = 0;
        const DevStatus *h = poll.next();
        stopped = poll.error != cudaSuccess || (h && h->stop);
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

// The problems of one channel count: passes over all of them at once, with chunks of the
// same number of rows in every problem.
struct Group {
    int k = 0, main_pass = 0;
    std::vector<int> probs;
    Kernels K;
    Pass pass[3];                     // blocks: of the whole group
    int check_rows = 2, check_blocks = 0;
};

// plan_pass for a group: the chunk length of the least arithmetic time
Pass plan_group(const std::vector<BatchProblem> &probs, const Group &gr, int S, int blocks_per_sm, int sms)
{
    const int k = gr.k, W = 32 - 2 * S;
    const double issue = 20.0 + 40.0 * k + 4.0 * k * (k - 1), lat = 180.0, ghz = 1.95;
    const long cap = (long)blocks_per_sm * sms;
    int top = 0;
    double pts = 0.0;
    for (int q : gr.probs) {
        top = std::max(top, probs[q].g.n);
        pts += (double)probs[q].g.n * probs[q].g.n;
    }
    Pass best;
    for (int rows = 1; rows <= top; rows += rows < 32 ? 1 : rows / 16) {
        long blocks = 0, warps = 0;
        for (int q : gr.probs) {
            const int n = probs[q].g.n;
            const long w = (long)((n + W - 1) / W) * ((n + rows - 1) / rows);
            warps += w;
            blocks += (w + kWarps - 1) / kWarps;
        }
        if (blocks > (1l << 30)) continue;
        const long full = blocks / cap, rest = blocks % cap;
        double cycles = (double)full * std::max(lat, issue * blocks_per_sm);
        if (rest) cycles += std::max(lat, issue * ceil((double)rest / sms));
        const double us = cycles * S * (rows + 2 * S) / (ghz * 1e3);
        if (best.stages == 0 || us < best.us) best = Pass{S, rows, 0, (int)warps, (int)blocks, us};
    }
    const double mb = 16e-6 * pts * (2 * gr.K.groups + (k + 3) / 4);
    best.us = 3.5 + std::max(best.us, mb / (mb > 110.0 ? 6.3 : 12.0));
    return best;
}

int plan_groups(vomt_ctx *ctx, const std::vector<BatchProblem> &probs, const vomt_params &p, std::vector<Group> *out)
{
    out->clear();
    const int interval = std::max(1, std::min(p.check_every, p.max_iters));
    for (int k = 1; k <= 5; ++k) {
        Group g;
        g.k = k;
        for (int q = 0; q < (int)probs.size(); ++q)
            if (probs[q].k == k) g.probs.push_back(q);
        if (g.probs.empty()) continue;
        g.K = pick(k, VOMT_U_L12, VOMT_W_L1, false, true);
        for (int q = 0; q < 3; ++q) {
            if (!g.K.many[q]) continue;
            int per_sm = 0;
            cudaError_t e = cudaFuncSetAttribute((const void *)g.K.many[q], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 kSmemBlock);
            if (e == cudaSuccess)
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)g.K.many[q], 32 * kWarps,
                                                                  g.K.smem);
            if (e != cudaSuccess) return set_cuda_error(ctx, e, "marching kernel");
            if (per_sm < 1) continue;
            Pass &ps = g.pass[q];
            ps = plan_group(probs, g, kStages[q], per_sm, ctx->sm_count);
            const int share = (ps.blocks + ctx->sm_count - 1) / ctx->sm_count;      // see march_solve
            ps.smem = std::max(g.K.smem, kSmemSM / (share + 1));
            if (kStages[q] <= interval && (g.pass[g.main_pass].stages == 0 ||
                                           ps.us / kStages[q] < g.pass[g.main_pass].us / kStages[g.main_pass]))
                g.main_pass = q;
        }
        if (g.pass[0].stages == 0) return VOMT_ERR_TOO_LARGE;
        out->push_back(g);
    }
    return VOMT_OK;
}

}  // namespace

double march_batch_estimate(vomt_ctx *ctx, const std::vector<BatchProblem> &probs, const vomt_params &p)
{
    std::vector<Group> groups;
    if (plan_groups(ctx, probs, p, &groups)) return 1e30;
    double us = 0.0;
    for (const Group &g : groups) us += g.pass[g.main_pass].us / kStages[g.main_pass];
    return us;
}

// The problems of a channel count advance together, a pass over all of them per launch; a
// problem that has stopped costs its blocks a look at its status.  Eight pairs at 256^2
// with three channels take 5.6 us per iteration together, where one after another on
// every SM (the grouped resident form) they take 8 x 1.6.
int march_batch(vomt_ctx *ctx, BatchMarchScratch *scr, const std::vector<BatchProblem> &probs, const vomt_params &p,
                cudaStream_t st, std::vector<DevStatus> *status, std::vector<int> *blocks, bool *taken)
{
    *taken = false;
    const int count = (int)probs.size();
    if (count > 65535) return VOMT_OK;                // a launch's third dimension
    std::vector<Group> groups;
    int rc = plan_groups(ctx, probs, p, &groups);
    if (rc) return rc == VOMT_ERR_TOO_LARGE ? VOMT_OK : rc;
    // scratch: per problem b, two states, the state before a check; check sums; tables
    std::vector<BatchItem> items(count);
    std::vector<int> maps, slot_of(count);            // items are stored group by group
    size_t floats4 = 0;
    std::vector<size_t> off(count);
    for (const Group &g : groups)
        for (int q : g.probs) {
            const size_t tile = (size_t)probs[q].g.n * ((probs[q].g.n + 31) / 32) * 32;
            off[q] = floats4;
            floats4 += tile * (3 * (size_t)g.K.groups + g.K.bgroups);
        }
    size_t sum_rows = 0;
    for (Group &g : groups) {
        long strip_rows = 0;
        for (int q : g.probs) strip_rows += (long)((probs[q].g.n + 29) / 30) * probs[q].g.n;
        g.check_rows = check_chunk(strip_rows, ctx->sm_count);
        g.check_blocks = 0;
        for (int q : g.probs) {
            const int n = probs[q].g.n, items = (n + 29) / 30 * ((n + g.check_rows - 1) / g.check_rows);
            g.check_blocks += (items + kWarps - 1) / kWarps;
        }
        sum_rows += g.check_blocks;
    }
    const size_t sums = sizeof(double) * NRED * sum_rows;
    rc = ensure_buffer(ctx, &scr->data, &scr->data_cap, sizeof(float4) * floats4 + sums, "batch states");
    if (rc) {
        ctx->err.clear();
        return VOMT_OK;
    }
    rc = ensure_buffer(ctx, &scr->items, &scr->items_cap, sizeof(BatchItem) * count, "batch tables");
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
    blocks->assign(count, 1);
    int at = 0;
    size_t sum_at = 0;
    std::vector<size_t> map_at(groups.size() * 4, 0);      // of its three passes and its check
    std::vector<int> first_item(groups.size()), top(groups.size(), 0);
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        const Group &g = groups[gi];
        first_item[gi] = at;
        int next[4] = {0, 0, 0, 0};
        std::vector<int> gm[4];
        for (size_t i = 0; i < g.probs.size(); ++i, ++at) {
            const int q = g.probs[i], n = probs[q].g.n;
            const size_t tile = (size_t)n * ((n + 31) / 32) * 32;
            BatchItem &d = items[at];
            memset(&d, 0, sizeof d);
            d.g = probs[q].g;
            d.g.g1 = 1.0f;
            d.g.g2 = d.g.mu * d.g.ih;
            d.cfg = probs[q].cfg;
            d.planar = probs[q].planar;
            d.b = data + off[q];
            for (int c = 0; c < 3; ++c) d.S[c] = d.b + tile * (g.K.bgroups + (size_t)c * g.K.groups);
            d.st = dstat + at;
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
            d.partials = dsums + (sum_at + next[3]) * NRED;
            gm[3].insert(gm[3].end(), d.check_blocks, (int)i);
            next[3] += d.check_blocks;
            slot_of[q] = at;
            top[gi] = std::max(top[gi], n);
        }
        for (int c = 0; c < 4; ++c) {
            map_at[gi * 4 + c] = maps.size();
            maps.insert(maps.end(), gm[c].begin(), gm[c].end());
            if (c < 3) groups[gi].pass[c].blocks = next[c];
        }
        sum_at += next[3];
    }
    rc = ensure_buffer(ctx, &scr->maps, &scr->maps_cap, sizeof(int) * maps.size(), "batch tables");
    if (rc) return rc;
    cudaError_t e = cudaMemcpyAsync(scr->items, items.data(), sizeof(BatchItem) * count, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(scr->maps, maps.data(), sizeof(int) * maps.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dstat, 0, sizeof(DevStatus) * count, st);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch tables");
    *taken = true;
    const BatchItem *ditems = (const BatchItem *)scr->items;
    const int *dmaps = (const int *)scr->maps;
    auto layout_grid = [&](size_t gi) {
        return dim3((top[gi] + 127) / 128, std::min(top[gi], 256), (unsigned)groups[gi].probs.size());
    };
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        groups[gi].K.in_many<<<layout_grid(gi), 128, 0, st>>>(ditems + first_item[gi]);
        ctx->launches += 1;
    }
    std::vector<int> cur(groups.size(), 0), before(groups.size(), 0);
    auto one = [&](size_t gi, int q, bool last) {
        const Group &g = groups[gi];
        const int prev = last && kStages[q] > 1 ? 1 : 0;
        launch_pdl(g.K.many[q], dim3(g.pass[q].blocks), dim3(32 * kWarps), (size_t)g.pass[q].smem, st,
                   ditems + first_item[gi], dmaps + map_at[gi * 4 + q], cur[gi], prev);
        ctx->launches += 1;
        before[gi] = prev ? 2 : cur[gi];
        cur[gi] ^= 1;
    };
    auto advance = [&](size_t gi, int m) {        // m iterations, fewer-stage passes first
        const Group &g = groups[gi];
        const int q = g.main_pass;
        int odd = m % kStages[q];
        for (int r = q - 1; r >= 0; --r)
            for (; g.pass[r].stages && odd >= kStages[r]; odd -= kStages[r], m -= kStages[r]) one(gi, r, m == kStages[r]);
        for (; m > 0; m -= kStages[q]) one(gi, q, m == kStages[q]);
    };
    auto check = [&](size_t gi, int t) {
        const Group &g = groups[gi];
        const unsigned np = (unsigned)g.probs.size();
        launch_pdl(g.K.check_many, dim3(g.check_blocks), dim3(32 * kWarps), 0, st, ditems + first_item[gi],
                   dmaps + map_at[gi * 4 + 3], cur[gi], before[gi]);
        launch_pdl(k_finalize_many, dim3(np), dim3(kFinThreads), 0, st, ditems + first_item[gi], t, cur[gi]);
        ctx->launches += 2;
    };
    if (p.max_iters == 0)
        for (size_t gi = 0; gi < groups.size(); ++gi) check(gi, 0);
    const bool tol_mode = p.tol_gap > 0.0;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (tol_mode)
        for (int q = 0; q < 2; ++q) cudaEventCreateWithFlags(&ev[q], cudaEventDisableTiming);
    const int chunk = p.check_every * ((2048 + p.check_every - 1) / p.check_every);
    int t = 0, nchunk = 0;
    bool stopped = false;
    while (t < p.max_iters && !stopped) {
        const int end = p.max_iters - t > chunk ? t + chunk : p.max_iters;
        while (t < end) {
            const int m = std::min(p.check_every, p.max_iters - t);
            t += m;
            for (size_t gi = 0; gi < groups.size(); ++gi) {
                advance(gi, m);
                check(gi, t);
            }
        }
        if (tol_mode) {
            const int slot = nchunk & 1;
            cudaMemcpyAsync(hstat + (size_t)slot * count, dstat, sizeof(DevStatus) * count, cudaMemcpyDeviceToHost, st);
            cudaEventRecord(ev[slot], st);
            if (nchunk >= 1) {
                // the previous chunk's flags: the GPU keeps running the chunk just queued
                cudaEventSynchronize(ev[slot ^ 1]);
                stopped = true;
                for (int q = 0; q < count; ++q) stopped = stopped && hstat[(size_t)(slot ^ 1) * count + q].stop;
            }
            ++nchunk;
        }
    }
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        groups[gi].K.out_many<<<layout_grid(gi), 128, 0, st>>>(ditems + first_item[gi]);
        ctx->launches += 1;
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(hstat, dstat, sizeof(DevStatus) * count, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    for (int q = 0; q < 2; ++q)
        if (ev[q]) cudaEventDestroy(ev[q]);
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "batch solve");
    status->resize(count);
    for (int q = 0; q < count; ++q) (*status)[q] = hstat[slot_of[q]];
    return VOMT_OK;
}

}  // namespace vomt
