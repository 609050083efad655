// rlb_batch_api.cpp -- host side of the batched-tube ABI (include/rlb.h):
// validation, tube storage, the job plan of the persistent launch, the CUDA
// graph that replays it, and the autotuner.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <functional>
#include <mutex>
#include <new>
#include <queue>
#include <string>
#include <vector>

#include "../../include/rlb.h"
#include "rlb_consts.h"
#include "rlb_internal.h"

using rlb::StepParams;
using rlb::batch::Job;
using rlb::batch::Tube;

struct rlb_batch {
    int B = 0;
    int limiter = 0;
    rlb_options opt{};
    int device = 0;
    int sms = 0;
    int l2_bytes = 0;
    std::vector<int> nx;
    std::vector<long long> pack;     // B + 1 packed offsets
    std::vector<Tube> tubes;
    long long total = 0;             // sum of nx
    long long ps = 0;                // plane stride (elements)
    int max_nx = 0;
    int max_clusters = 0;            // capacity of the cluster table
    void *block = nullptr;
    float *f0 = nullptr, *f1 = nullptr, *prev = nullptr;   // blocks of 32 cells, 38 populations (f, h) or 5 values each
    size_t state_bytes = 0;          // f0 .. prev, contiguous from f0
    double *stage = nullptr;         // 6 x total doubles
    Tube *d_tubes = nullptr;
    long long *d_pack = nullptr;
    int *d_par = nullptr, *d_steps = nullptr, *d_order = nullptr, *d_cl = nullptr;
    Job *d_jobs = nullptr;
    unsigned *d_status = nullptr;
    double *d_tot = nullptr;
    void *host = nullptr;            // pinned staging
    unsigned *h_status = nullptr;
    int *h_steps = nullptr, *h_order = nullptr, *h_cl = nullptr;
    Job *h_jobs = nullptr;
    double *h_tot = nullptr;
    rlb_batch_tuning tune{};
    int nclusters = 0;               // clusters resident at once for `tune`
    bool shape_set = false;          // the launch shape was set or tuned (else choose_shape's)
    bool plan_ok = false;
    std::vector<long long> plan_steps;
    cudaStream_t stream = nullptr, cap_stream = nullptr;
    cudaGraphExec_t graph = nullptr;
    long long launches = 0;
    StepParams sp{};
    std::string err = "no error";
};

namespace {

thread_local std::string g_berr = "no error";

rlb_status bfail(rlb_batch *b, rlb_status st, const std::string &msg)
{
    if (b) b->err = msg;
    else {
        g_berr = msg;
        rlb::set_thread_error(msg.c_str());
    }
    return st;
}

rlb_status bcuda(rlb_batch *b, cudaError_t e, const char *where)
{
    return bfail(b, RLB_E_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define RLB_BCUDA(b, call)                                      \
    do {                                                        \
        cudaError_t e_ = (call);                                \
        if (e_ != cudaSuccess) return bcuda((b), e_, #call);    \
    } while (0)

size_t aup(size_t v, size_t a) { return (v + a - 1) / a * a; }

bool valid_tuning(const rlb_batch_tuning &t, std::string &why)
{
    if (t.bound != 256 && t.bound != 384 && t.bound != 512) {
        why = "tuning.bound must be 256, 384 or 512";
        return false;
    }
    if (t.threads < 32 || t.threads > t.bound || t.threads % 32 != 0) {
        why = "tuning.threads must be a multiple of 32 in [32, bound]";
        return false;
    }
    if (t.cluster != 1 && t.cluster != 2 && t.cluster != 4 && t.cluster != 8) {
        why = "tuning.cluster must be 1, 2, 4 or 8";
        return false;
    }
    if (t.pairs_per_thread < 1 || t.pairs_per_thread > 64) {
        why = "tuning.pairs_per_thread must be in [1, 64]";
        return false;
    }
    return true;
}

// the job plan (see rlb_batch_plan in rlb.h)
struct Plan {
    std::vector<int> order;
    std::vector<Job> jobs;       // grouped by cluster
    std::vector<int> cl_start;   // nclusters + 1
    long long critical = 0;
};

// longest-running first: steps, then length, then id
std::vector<int> tube_order(int B, const int *nx, const long long *steps)
{
    std::vector<int> ids(B);
    for (int i = 0; i < B; ++i) ids[i] = i;
    std::stable_sort(ids.begin(), ids.end(), [&](int a, int b) {
        if (steps[a] != steps[b]) return steps[a] > steps[b];
        return nx[a] > nx[b];
    });
    return ids;
}

// consecutive tubes of that order in jobs of at most cluster x threads x
// pairs_per_thread pairs
void group_tubes(const std::vector<int> &ids, const int *nx, const long long *steps, const rlb_batch_tuning &t,
                 std::vector<Job> &jobs)
{
    const long long cap = (long long)t.cluster * t.threads * t.pairs_per_thread;
    jobs.clear();
    for (size_t k = 0; k < ids.size(); ++k) {
        const int id = ids[k];
        if (steps[id] == 0) break;
        const int pairs = (nx[id] + 1) / 2;
        if (!jobs.empty()) {
            Job &J = jobs.back();
            if (J.count < rlb::batch::kMaxJobTubes && (long long)J.pairs + pairs <= cap) {
                J.count += 1;
                J.pairs += pairs;
                continue;
            }
        }
        jobs.push_back(Job{int(k), 1, int(steps[id]), pairs});
    }
}

long long passes(const Job &J, const rlb_batch_tuning &t)
{
    const long long per_pass = (long long)t.cluster * t.threads;
    return (J.pairs + per_pass - 1) / per_pass;
}

rlb_status make_plan(int B, const int *nx, const long long *steps, const rlb_batch_tuning &t, int nclusters,
                     Plan &pl, std::string &why)
{
    if (B < 1 || !nx || !steps) {
        why = "B < 1 or a NULL array";
        return RLB_E_INVALID;
    }
    if (!valid_tuning(t, why)) return RLB_E_INVALID;
    if (nclusters < 1) {
        why = "nclusters must be >= 1";
        return RLB_E_INVALID;
    }
    for (int i = 0; i < B; ++i) {
        if (nx[i] < 1) {
            why = "every tube needs nx >= 1";
            return RLB_E_INVALID;
        }
        if (steps[i] < 0 || steps[i] > INT_MAX) {
            why = "step counts must be in [0, 2^31 - 1]";
            return RLB_E_INVALID;
        }
    }
    pl.order = tube_order(B, nx, steps);
    std::vector<Job> jobs;
    group_tubes(pl.order, nx, steps, t, jobs);
    // longest processing time first, each job to the least loaded cluster
    auto cost = [&](const Job &J) { return J.steps * passes(J, t); };
    std::vector<int> jorder(jobs.size());
    for (size_t i = 0; i < jobs.size(); ++i) jorder[i] = int(i);
    std::stable_sort(jorder.begin(), jorder.end(), [&](int a, int b) { return cost(jobs[a]) > cost(jobs[b]); });
    using Slot = std::pair<long long, int>;   // (load, cluster)
    std::priority_queue<Slot, std::vector<Slot>, std::greater<Slot>> heap;
    for (int c = 0; c < nclusters; ++c) heap.push({0, c});
    std::vector<int> owner(jobs.size());
    std::vector<long long> load(nclusters, 0);
    for (int j : jorder) {
        Slot s = heap.top();
        heap.pop();
        owner[j] = s.second;
        s.first += cost(jobs[j]);
        load[s.second] = s.first;
        heap.push(s);
    }
    pl.cl_start.assign(nclusters + 1, 0);
    for (size_t j = 0; j < jobs.size(); ++j) pl.cl_start[owner[j] + 1] += 1;
    for (int c = 0; c < nclusters; ++c) pl.cl_start[c + 1] += pl.cl_start[c];
    std::vector<int> fill(pl.cl_start.begin(), pl.cl_start.end() - 1);
    pl.jobs.assign(jobs.size(), Job{});
    for (int j : jorder) pl.jobs[fill[owner[j]]++] = jobs[j];
    pl.critical = 0;
    for (long long v : load) pl.critical = std::max(pl.critical, v);
    return RLB_OK;
}

// us of a job under a launch shape: passes in which w warps of a cluster's first
// block have pairs take us[w] each, a step `step` more
struct Price {
    rlb_batch_tuning t;
    double us[17], step;
    double operator()(const Job &J) const
    {
        const int per_pass = t.cluster * t.threads, full = J.pairs / per_pass, rest = J.pairs - full * per_pass;
        return J.steps * (full * us[t.threads / 32] + us[(std::min(rest, t.threads) + 31) / 32] + step);
    }
};

// the longest load when the jobs, longest first, each go to the least loaded cluster
double critical_path(const std::vector<Job> &jobs, const Price &price, int nclusters)
{
    std::vector<double> cost(jobs.size());
    for (size_t j = 0; j < jobs.size(); ++j) cost[j] = price(jobs[j]);
    std::sort(cost.begin(), cost.end(), std::greater<double>());
    double longest = cost[0];
    if (cost.size() <= size_t(nclusters)) return longest;
    std::priority_queue<double, std::vector<double>, std::greater<double>> load(
        std::greater<double>(), std::vector<double>(cost.begin(), cost.begin() + nclusters));
    for (size_t j = nclusters; j < cost.size(); ++j) {
        const double l = load.top() + cost[j];
        load.pop();
        load.push(l);
        longest = std::max(longest, l);
    }
    return longest;
}

rlb_status check_status(rlb_batch *b)
{
    RLB_BCUDA(b, cudaMemcpyAsync(b->h_status, b->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, b->stream));
    RLB_BCUDA(b, cudaStreamSynchronize(b->stream));
    if (*b->h_status != 0u) {
        RLB_BCUDA(b, cudaMemsetAsync(b->d_status, 0, sizeof(unsigned), b->stream));
        RLB_BCUDA(b, cudaStreamSynchronize(b->stream));
        return bfail(b, RLB_E_NONPHYSICAL, "a cell was non-physical (E <= |M|, n <= 0, |u| >= 1 or non-finite)");
    }
    return RLB_OK;
}

rlb::batch::Args make_args(rlb_batch *b)
{
    rlb::batch::Args a;
    a.p = b->sp;
    a.tubes = b->d_tubes;
    a.order = b->d_order;
    a.steps = b->d_steps;
    a.par = b->d_par;
    a.jobs = b->d_jobs;
    a.cl_start = b->d_cl;
    a.nclusters = b->nclusters;
    a.cluster = b->tune.cluster;
    a.np = b->opt.symmetry_1d ? 7 : 19;
    a.f0 = b->f0;
    a.f1 = b->f1;
    a.prev = b->prev;
    return a;
}

// clusters of tuning t resident at once (0: does not fit)
rlb_status resident_clusters(rlb_batch *b, const rlb_batch_tuning &t, int &n)
{
    rlb::batch::Args a = make_args(b);
    a.cluster = t.cluster;
    n = 0;
    cudaError_t e = rlb::batch::launch_tubes(a, t.threads, t.bound, t.cluster, b->stream, &n);
    if (e != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    if (n > b->max_clusters) n = b->max_clusters;
    return RLB_OK;
}

// The same for the shapes choose_shape looks at, asked once per process for
// each device and form: it depends on the kernels alone.
int resident_shape(rlb_batch *b, const rlb_batch_tuning &t)
{
    constexpr int kMaxDevices = 64;
    static std::mutex lock;
    static int known[kMaxDevices][2][4][4];   // 0: not asked yet, else clusters + 1
    int n = 0;
    if (b->device >= kMaxDevices) {
        resident_clusters(b, t, n);
        return n;
    }
    const std::lock_guard<std::mutex> hold(lock);
    const int j = t.cluster == 8 ? 3 : t.cluster / 2;
    int &k = known[b->device][b->opt.symmetry_1d != 0][t.threads / 128 - 1][j];
    if (k == 0) {
        resident_clusters(b, t, n);
        k = n + 1;
    }
    return std::min(k - 1, b->max_clusters);
}

rlb_status upload_plan(rlb_batch *b, const long long *steps, const Plan &pl)
{
    for (int i = 0; i < b->B; ++i) b->h_steps[i] = int(steps[i]);
    std::memcpy(b->h_order, pl.order.data(), sizeof(int) * b->B);
    if (!pl.jobs.empty()) std::memcpy(b->h_jobs, pl.jobs.data(), sizeof(Job) * pl.jobs.size());
    std::memcpy(b->h_cl, pl.cl_start.data(), sizeof(int) * pl.cl_start.size());
    RLB_BCUDA(b, cudaMemcpyAsync(b->d_steps, b->h_steps, sizeof(int) * b->B, cudaMemcpyHostToDevice, b->stream));
    RLB_BCUDA(b, cudaMemcpyAsync(b->d_order, b->h_order, sizeof(int) * b->B, cudaMemcpyHostToDevice, b->stream));
    if (!pl.jobs.empty())
        RLB_BCUDA(b, cudaMemcpyAsync(b->d_jobs, b->h_jobs, sizeof(Job) * pl.jobs.size(), cudaMemcpyHostToDevice,
                                     b->stream));
    RLB_BCUDA(b, cudaMemcpyAsync(b->d_cl, b->h_cl, sizeof(int) * pl.cl_start.size(), cudaMemcpyHostToDevice,
                                 b->stream));
    return RLB_OK;
}

bool planned(const rlb_batch *b, const long long *steps)
{
    return b->plan_ok && std::equal(b->plan_steps.begin(), b->plan_steps.end(), steps);
}

// plan for `steps` under the current tuning, uploaded (the host staging is
// reused only after the previous call synchronised)
rlb_status prepare(rlb_batch *b, const long long *steps)
{
    if (planned(b, steps)) return RLB_OK;
    Plan pl;
    std::string why;
    rlb_status st = make_plan(b->B, b->nx.data(), steps, b->tune, b->nclusters, pl, why);
    if (st != RLB_OK) return bfail(b, st, why);
    st = upload_plan(b, steps, pl);
    if (st != RLB_OK) return st;
    b->plan_steps.assign(steps, steps + b->B);
    b->plan_ok = true;
    return RLB_OK;
}

void drop_graph(rlb_batch *b)
{
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
}

rlb_status apply_tuning(rlb_batch *b, const rlb_batch_tuning &t)
{
    std::string why;
    if (!valid_tuning(t, why)) return bfail(b, RLB_E_INVALID, why);
    int n = 0;
    rlb_status st = resident_clusters(b, t, n);
    if (st != RLB_OK) return st;
    if (n < 1) return bfail(b, RLB_E_INVALID, "this tuning does not fit on the device");
    b->tune = t;
    b->tune.ms = 0.0;
    b->nclusters = n;
    b->plan_ok = false;
    drop_graph(b);
    return RLB_OK;
}

// The launch shape of a batch that nobody tuned, chosen with each new plan (one
// kept from a call that advanced a single tube made 512 tubes take twice as
// long): the one with the shortest critical path when jobs are priced in us.  A
// pass takes the time of the busiest scheduler's warps (GB300, us with 1 / 2 / 3
// / 4 warps: 4.4, 5.4, 7.1, 9.1; with 7 classes 2.15, 2.9, 3.75, 4.7), up to a
// third more when the tubes in progress do not fit in the L2 cache, and a step
// in a cluster 1.2 us more (0.9).  The warps that count are those that have
// pairs, in the blocks that have jobs (and a little for blocks that may meet on
// an SM while others idle): pricing every block that fits took four blocks of
// 128 for as dear as one of 512, and 64 tubes of 256 cells 1.9 times as long as
// their best shape.  Blocks of 128 and 256 threads run the kernel of bound 256:
// with bound 512 more of them fit, and few jobs then share SMs.  Over 246 batches
// of 1 to 2048 tubes of 20 to 8192 cells the choice takes 1.03 times the
// autotuner's best time (1.38 before), at most 1.46 times (2.64).
//
// The tubes are sorted once, and a shape's jobs are laid out only while its lower
// bound (the longest job, or all work over all clusters) is below the best
// critical path so far.
rlb_status choose_shape(rlb_batch *b, const long long *steps)
{
    const bool sym = b->opt.symmetry_1d != 0;
    const double pass[2][4] = {{4.4, 5.4, 7.1, 9.1}, {2.15, 2.9, 3.75, 4.7}}, join[2] = {1.2, 0.9};
    const double pair_bytes = 2.0 * sizeof(float) * (2 * (sym ? 14 : 38) + 5);
    struct Shape {
        Price price;
        int n;
        double bound;   // of the critical path
    };
    std::vector<Shape> shapes;
    std::vector<Job> jobs;
    const std::vector<int> order = tube_order(b->B, b->nx.data(), steps);
    for (int threads : {128, 256, 384, 512}) {
        for (int cluster : {1, 2, 4, 8}) {
            const rlb_batch_tuning t{threads, std::max(threads, 256), cluster, 1, 0.0};
            const int n = resident_shape(b, t);
            if (n < 1) continue;
            group_tubes(order, b->nx.data(), steps, t, jobs);
            double work = 0.0, pairs = 0.0;   // pairs of a job, mean over the work
            for (const Job &J : jobs) {
                const double w = double(J.steps) * double(passes(J, t));
                work += w;
                pairs += w * double(J.pairs);
            }
            const int busy = int(std::min<size_t>(jobs.size(), size_t(n)));
            const int fit = std::max(1, (n * cluster + b->sms / 2) / b->sms), used = (busy * cluster + b->sms - 1) / b->sms;
            const double on_sm = used < fit ? used + 0.25 : fit;
            const double in_l2 = busy * (pairs / work) * pair_bytes / b->l2_bytes;
            const double far = 1.0 + 0.35 * std::max(0.0, 1.0 - 0.8 / in_l2);
            Price price{t, {0.0}, cluster > 1 ? join[sym] : 0.0};
            for (int w = 1; w <= threads / 32; ++w) {
                const double warps = on_sm * w / 4.0;   // of one scheduler
                const int q = std::min(3, std::max(1, int(warps)));
                const double *p = pass[sym];
                price.us[w] = far * (warps <= 1.0 ? p[0] : p[q - 1] + (p[q] - p[q - 1]) * (warps - q));
            }
            double longest = 0.0, total = 0.0;
            for (const Job &J : jobs) {
                const double c = price(J);
                total += c;
                longest = std::max(longest, c);
            }
            shapes.push_back(Shape{price, n, std::max(longest, total / n)});
        }
    }
    std::stable_sort(shapes.begin(), shapes.end(), [](const Shape &x, const Shape &y) { return x.bound < y.bound; });
    const Shape *best = nullptr;
    double best_cost = 0.0;
    for (const Shape &s : shapes) {
        if (best && s.bound >= best_cost) break;
        group_tubes(order, b->nx.data(), steps, s.price.t, jobs);
        const double c = critical_path(jobs, s.price, s.n);
        if (!best || c < best_cost) {
            best_cost = c;
            best = &s;
        }
    }
    if (!best) return RLB_OK;
    const rlb_batch_tuning &t = best->price.t, &now = b->tune;
    if (t.threads == now.threads && t.bound == now.bound && t.cluster == now.cluster &&
        t.pairs_per_thread == now.pairs_per_thread)
        return RLB_OK;
    return apply_tuning(b, t);
}

rlb_status ensure_graph(rlb_batch *b)
{
    if (b->graph) return RLB_OK;
    const rlb::batch::Args a = make_args(b);
    RLB_BCUDA(b, cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = rlb::batch::launch_tubes(a, b->tune.threads, b->tune.bound, b->tune.cluster, b->cap_stream,
                                             nullptr);
    cudaGraph_t g = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(b->cap_stream, &g);
    if (e != cudaSuccess || e2 != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return bcuda(b, e != cudaSuccess ? e : e2, "capture of the tube kernel");
    }
    e = cudaGraphInstantiate(&b->graph, g, 0ULL);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        b->graph = nullptr;
        return bcuda(b, e, "cudaGraphInstantiate");
    }
    return RLB_OK;
}

rlb_status check_steps(rlb_batch *b, const long long *nsteps)
{
    if (!nsteps) return bfail(b, RLB_E_INVALID, "nsteps is NULL");
    for (int i = 0; i < b->B; ++i)
        if (nsteps[i] < 0 || nsteps[i] > INT_MAX)
            return bfail(b, RLB_E_INVALID, "step counts must be in [0, 2^31 - 1]");
    return RLB_OK;
}

// under the 1-D symmetry reduction only the class representatives' planes
// are current: copy them to the other populations of their classes
rlb_status expand(rlb_batch *b)
{
    if (!b->opt.symmetry_1d) return RLB_OK;
    RLB_BCUDA(b, rlb::batch::launch_tubes_expand(b->B, b->max_nx, b->d_tubes, b->d_par, b->f0, b->f1,
                                                 b->stream));
    b->launches += 1;
    return RLB_OK;
}

}  // namespace

extern "C" {

rlb_status rlb_batch_plan(int B, const int *nx, const long long *nsteps, const rlb_batch_tuning *t,
                          int nclusters, int *order, int *jobs, int *njobs, int *cl_start, long long *critical)
{
    if (!t || !order || !jobs || !njobs || !cl_start) return bfail(nullptr, RLB_E_INVALID, "a NULL argument");
    Plan pl;
    std::string why;
    const rlb_status st = make_plan(B, nx, nsteps, *t, nclusters, pl, why);
    if (st != RLB_OK) return bfail(nullptr, st, why);
    std::memcpy(order, pl.order.data(), sizeof(int) * B);
    for (size_t j = 0; j < pl.jobs.size(); ++j) {
        jobs[4 * j + 0] = pl.jobs[j].first;
        jobs[4 * j + 1] = pl.jobs[j].count;
        jobs[4 * j + 2] = pl.jobs[j].steps;
        jobs[4 * j + 3] = pl.jobs[j].pairs;
    }
    *njobs = int(pl.jobs.size());
    std::memcpy(cl_start, pl.cl_start.data(), sizeof(int) * pl.cl_start.size());
    if (critical) *critical = pl.critical;
    return RLB_OK;
}

rlb_status rlb_batch_create(int B, const int *nx, const double *eta_over_s, const double *zeta_over_s,
                            int limiter, const rlb_options *opts, rlb_batch **out)
{
    if (!out) return bfail(nullptr, RLB_E_INVALID, "out is NULL");
    *out = nullptr;
    if (B < 1 || B > 65535) return bfail(nullptr, RLB_E_INVALID, "B must be in [1, 65535]");
    if (!nx || !eta_over_s || !zeta_over_s) return bfail(nullptr, RLB_E_INVALID, "a per-tube array is NULL");
    rlb_options o;
    rlb_default_options(&o);
    o.precision = RLB_FP32_STORAGE;
    if (opts) o = *opts;
    if (o.precision != RLB_FP32_STORAGE)
        return bfail(nullptr, RLB_E_INVALID, "the batched path stores populations in FP32 (RLB_FP32_STORAGE)");
    if (o.euler_mode != 0) return bfail(nullptr, RLB_E_INVALID, "the batched path runs the viscous step only");
    if (o.symmetry_1d != 0 && o.symmetry_1d != 1) return bfail(nullptr, RLB_E_INVALID, "symmetry_1d must be 0 or 1");
    if (o.model != 0) return bfail(nullptr, RLB_E_INVALID, "the batched path runs the extended lattice (model 0)");
    if (o.recovery_fp64 != 0)
        return bfail(nullptr, RLB_E_INVALID, "the batched path runs the double-float recovery (recovery_fp64 = 0)");
    if (o.slab_rows != 0) return bfail(nullptr, RLB_E_INVALID, "slab_rows is an option of grids (0 for batches)");
    if (limiter != RLB_LIMITER_MINMOD && limiter != RLB_LIMITER_NONE)
        return bfail(nullptr, RLB_E_INVALID, "unknown limiter");
    if (!(o.dt_over_dx > 0.0) || !std::isfinite(o.dt_over_dx))
        return bfail(nullptr, RLB_E_INVALID, "dt_over_dx must be finite and > 0");
    if (!std::isfinite(o.tau_override) || !std::isfinite(o.alpha_override))
        return bfail(nullptr, RLB_E_INVALID, "overrides must be finite");
    if (o.dt_over_dx * 2.0 * rlb::kC0Ct > 1.0)
        return bfail(nullptr, RLB_E_UNSTABLE, "dt/dx exceeds the Courant bound of the extended lattice");
    long long cells = 0, stored = 0;
    int max_nx = 0;
    for (int i = 0; i < B; ++i) {
        if (nx[i] < 1) return bfail(nullptr, RLB_E_INVALID, "every tube needs nx >= 1");
        if (!(eta_over_s[i] >= 0.0) || !std::isfinite(eta_over_s[i]) || !(zeta_over_s[i] >= 0.0) ||
            !std::isfinite(zeta_over_s[i]))
            return bfail(nullptr, RLB_E_INVALID, "eta_over_s and zeta_over_s must be finite and >= 0");
        const double alpha = o.alpha_override >= 0.0 ? o.alpha_override : rlb::alpha_of_zeta(zeta_over_s[i]);
        if (2.0 * rlb::kOmegaC * o.dt_over_dx * alpha > 1.0)
            return bfail(nullptr, RLB_E_UNSTABLE, "alpha dt exceeds the explicit diffusion bound");
        cells += nx[i];
        stored += (long long)aup(size_t(nx[i]), rlb::batch::kAlignCells);
        max_nx = std::max(max_nx, nx[i]);
    }
    if (stored > (1LL << 30)) return bfail(nullptr, RLB_E_INVALID, "more than 2^30 cells in the batch");

    rlb_batch *b = new (std::nothrow) rlb_batch();
    if (!b) return bfail(nullptr, RLB_E_NOMEM, "host allocation failed");
    b->B = B;
    b->limiter = limiter;
    b->opt = o;
    b->nx.assign(nx, nx + B);
    b->total = cells;
    b->max_nx = max_nx;
    b->stream = (cudaStream_t)o.cuda_stream;
    b->pack.assign(B + 1, 0);
    b->tubes.resize(B);
    long long off = 0;
    for (int i = 0; i < B; ++i) {
        b->pack[i + 1] = b->pack[i] + nx[i];
        const double alpha = o.alpha_override >= 0.0 ? o.alpha_override : rlb::alpha_of_zeta(zeta_over_s[i]);
        b->tubes[i] = Tube{int(off), nx[i], float(eta_over_s[i]), float(rlb::kOmegaC * o.dt_over_dx * alpha)};
        off += (long long)aup(size_t(nx[i]), rlb::batch::kAlignCells);
    }
    b->ps = (long long)aup(size_t(off), 64);
    cudaError_t e = cudaGetDevice(&b->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->l2_bytes, cudaDevAttrL2CacheSize, b->device);
    if (e != cudaSuccess) {
        delete b;
        return bcuda(nullptr, e, "cudaGetDevice");
    }
    b->max_clusters = b->sms * 32;

    const size_t plane = size_t(b->ps) * sizeof(float);
    size_t offs[14], o2 = 0;
    offs[0] = o2; o2 += 38 * plane;                                   // f0, h0
    offs[2] = o2; o2 += 38 * plane;                                   // f1, h1
    offs[4] = o2; o2 += 5 * plane;                                    // prev
    b->state_bytes = o2;
    o2 = aup(o2, 256);
    offs[5] = o2; o2 = aup(o2 + sizeof(int) * B, 256);                // par (kept with the state)
    offs[6] = o2; o2 = aup(o2 + 6 * sizeof(double) * size_t(cells), 256);   // stage
    offs[7] = o2; o2 = aup(o2 + sizeof(Tube) * B, 256);
    offs[8] = o2; o2 = aup(o2 + sizeof(long long) * (B + 1), 256);
    offs[9] = o2; o2 = aup(o2 + sizeof(int) * B, 256);                // steps
    offs[10] = o2; o2 = aup(o2 + sizeof(int) * B, 256);               // order
    offs[11] = o2; o2 = aup(o2 + sizeof(Job) * B, 256);               // jobs
    offs[12] = o2; o2 = aup(o2 + sizeof(int) * (b->max_clusters + 1), 256);   // cluster table
    offs[13] = o2; o2 = aup(o2 + 256 + 5 * sizeof(double) * B, 256);  // status, totals
    e = cudaMalloc(&b->block, o2);
    if (e != cudaSuccess) {
        delete b;
        return bfail(nullptr, RLB_E_NOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    }
    char *base = (char *)b->block;
    b->f0 = (float *)(base + offs[0]);
    b->f1 = (float *)(base + offs[2]);
    b->prev = (float *)(base + offs[4]);
    b->d_par = (int *)(base + offs[5]);
    b->stage = (double *)(base + offs[6]);
    b->d_tubes = (Tube *)(base + offs[7]);
    b->d_pack = (long long *)(base + offs[8]);
    b->d_steps = (int *)(base + offs[9]);
    b->d_order = (int *)(base + offs[10]);
    b->d_jobs = (Job *)(base + offs[11]);
    b->d_cl = (int *)(base + offs[12]);
    b->d_status = (unsigned *)(base + offs[13]);
    b->d_tot = (double *)(base + offs[13] + 256);

    const size_t hbytes = 256 + sizeof(int) * 2 * B + sizeof(Job) * B + sizeof(int) * (b->max_clusters + 1) +
                          5 * sizeof(double) * B + 64;
    e = cudaMallocHost(&b->host, hbytes);
    if (e != cudaSuccess) {
        cudaFree(b->block);
        delete b;
        return bfail(nullptr, RLB_E_NOMEM, std::string("cudaMallocHost: ") + cudaGetErrorString(e));
    }
    char *hp = (char *)b->host;
    b->h_status = (unsigned *)hp;
    b->h_tot = (double *)(hp + 64);
    b->h_jobs = (Job *)(hp + 64 + 5 * sizeof(double) * B);
    b->h_steps = (int *)((char *)b->h_jobs + sizeof(Job) * B);
    b->h_order = b->h_steps + B;
    b->h_cl = b->h_order + B;

    e = cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->block, 0, o2, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_tubes, b->tubes.data(), sizeof(Tube) * B, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_pack, b->pack.data(), sizeof(long long) * (B + 1), cudaMemcpyHostToDevice,
                            b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) {
        rlb_batch_destroy(b);
        return bcuda(nullptr, e, "batch setup");
    }

    StepParams &sp = b->sp;
    std::memset(&sp, 0, sizeof(sp));
    sp.nx = max_nx;
    sp.ny = sp.nz = 1;
    sp.ps = b->ps;
    for (int a = 0; a < 3; ++a) sp.bc_lo[a] = sp.bc_hi[a] = RLB_BC_OUTFLOW;
    sp.half_lim = limiter == RLB_LIMITER_MINMOD ? 0.5 : 0.0;
    sp.k1 = rlb::kC0Ct * o.dt_over_dx;
    sp.k2 = 2.0 * rlb::kC0Ct * o.dt_over_dx;
    sp.kw = rlb::kOmegaC * o.dt_over_dx;
    sp.tau_override = o.tau_override;
    sp.status = b->d_status;
    sp.f_k1 = float(sp.k1);
    sp.f_k2 = float(sp.k2);
    sp.f_half_lim = float(sp.half_lim);
    sp.f_kw = float(sp.kw);
    sp.f_tau_override = float(sp.tau_override);

    // a shape that fits every GB300 configuration, until a step call chooses one
    // for its step counts; rlb_batch_autotune measures them
    rlb_batch_tuning t{256, 256, 1, 1, 0.0};
    const rlb_status st = apply_tuning(b, t);
    if (st != RLB_OK) {
        const std::string msg = b->err;
        rlb_batch_destroy(b);
        return bfail(nullptr, st, msg);
    }
    *out = b;
    return RLB_OK;
}

rlb_status rlb_batch_init(rlb_batch *b, const double *n, const double *T, const double *ux, int on_device)
{
    if (!b) return bfail(nullptr, RLB_E_INVALID, "batch is NULL");
    if (!n || !T || !ux) return bfail(b, RLB_E_INVALID, "a field pointer is NULL");
    RLB_BCUDA(b, cudaSetDevice(b->device));
    const double *dev[3] = {n, T, ux};
    if (!on_device) {
        const size_t bytes = sizeof(double) * size_t(b->total);
        for (int k = 0; k < 3; ++k) {
            RLB_BCUDA(b, cudaMemcpyAsync(b->stage + size_t(k) * b->total, dev[k], bytes, cudaMemcpyHostToDevice,
                                         b->stream));
            dev[k] = b->stage + size_t(k) * b->total;
        }
    }
    RLB_BCUDA(b, cudaMemsetAsync(b->d_par, 0, sizeof(int) * b->B, b->stream));
    RLB_BCUDA(b, rlb::batch::launch_tubes_init(b->B, b->max_nx, b->d_tubes, b->d_pack, dev[0], dev[1], dev[2], b->f0,
                                               b->prev, b->d_status, b->stream));
    b->launches += 1;
    const rlb_status st = check_status(b);
    return st == RLB_E_NONPHYSICAL ? bfail(b, RLB_E_INVALID, "initial state has n <= 0, T <= 0 or |u| >= 1") : st;
}

rlb_status rlb_batch_step(rlb_batch *b, const long long *nsteps)
{
    if (!b) return bfail(nullptr, RLB_E_INVALID, "batch is NULL");
    rlb_status st = check_steps(b, nsteps);
    if (st != RLB_OK) return st;
    bool any = false;
    for (int i = 0; i < b->B; ++i) any = any || nsteps[i] > 0;
    if (!any) return RLB_OK;
    RLB_BCUDA(b, cudaSetDevice(b->device));
    if (!b->shape_set && !planned(b, nsteps) && (st = choose_shape(b, nsteps)) != RLB_OK) return st;
    if ((st = prepare(b, nsteps)) != RLB_OK) return st;
    if ((st = ensure_graph(b)) != RLB_OK) return st;
    RLB_BCUDA(b, cudaGraphLaunch(b->graph, b->stream));
    b->launches += 1;
    return check_status(b);
}

rlb_status rlb_batch_macroscopic(rlb_batch *b, double *out, int on_device)
{
    if (!b) return bfail(nullptr, RLB_E_INVALID, "batch is NULL");
    if (!out) return bfail(b, RLB_E_INVALID, "out is NULL");
    RLB_BCUDA(b, cudaSetDevice(b->device));
    if (rlb_status st = expand(b); st != RLB_OK) return st;
    double *dst = on_device ? out : b->stage;
    RLB_BCUDA(b, rlb::batch::launch_tubes_macro(b->B, b->max_nx, b->d_tubes, b->d_pack, b->d_par, b->total, b->f0,
                                                b->f1, dst, b->d_status, b->stream));
    b->launches += 1;
    if (!on_device)
        RLB_BCUDA(b, cudaMemcpyAsync(out, b->stage, 6 * sizeof(double) * size_t(b->total), cudaMemcpyDeviceToHost,
                                     b->stream));
    return check_status(b);
}

rlb_status rlb_batch_totals(rlb_batch *b, double *out)
{
    if (!b) return bfail(nullptr, RLB_E_INVALID, "batch is NULL");
    if (!out) return bfail(b, RLB_E_INVALID, "out is NULL");
    RLB_BCUDA(b, cudaSetDevice(b->device));
    if (rlb_status st = expand(b); st != RLB_OK) return st;
    RLB_BCUDA(b, rlb::batch::launch_tubes_totals(b->B, b->d_tubes, b->d_par, b->f0, b->f1,
                                                 b->d_tot, b->stream));
    b->launches += 1;
    RLB_BCUDA(b, cudaMemcpyAsync(b->h_tot, b->d_tot, 5 * sizeof(double) * b->B, cudaMemcpyDeviceToHost, b->stream));
    RLB_BCUDA(b, cudaStreamSynchronize(b->stream));
    std::memcpy(out, b->h_tot, 5 * sizeof(double) * b->B);
    return RLB_OK;
}

rlb_status rlb_batch_set_tuning(rlb_batch *b, const rlb_batch_tuning *t)
{
    if (!b) return bfail(nullptr, RLB_E_INVALID, "batch is NULL");
    if (!t) return bfail(b, RLB_E_INVALID, "tuning is NULL");
    RLB_BCUDA(b, cudaSetDevice(b->device));
    const rlb_status st = apply_tuning(b, *t);
    if (st == RLB_OK) b->shape_set = true;
    return st;
}

rlb_status rlb_batch_get_tuning(const rlb_batch *b, rlb_batch_tuning *t, int *resident_clusters)
{
    if (!b || !t) return bfail(nullptr, RLB_E_INVALID, "a NULL argument");
    *t = b->tune;
    if (resident_clusters) *resident_clusters = b->nclusters;
    return RLB_OK;
}

rlb_status rlb_batch_autotune(rlb_batch *b, const long long *nsteps, int divisor, rlb_batch_tuning *trials,
                              int max_trials, int *n_trials, rlb_batch_tuning *best)
{
    if (!b) return bfail(nullptr, RLB_E_INVALID, "batch is NULL");
    rlb_status st = check_steps(b, nsteps);
    if (st != RLB_OK) return st;
    if (divisor < 1) return bfail(b, RLB_E_INVALID, "divisor must be >= 1");
    if (max_trials > 0 && !trials) return bfail(b, RLB_E_INVALID, "trials is NULL");
    RLB_BCUDA(b, cudaSetDevice(b->device));
    std::vector<long long> ts(b->B);
    for (int i = 0; i < b->B; ++i) ts[i] = (nsteps[i] + divisor - 1) / divisor;

    // snapshot of the state (populations, previous level, buffer parities)
    const size_t snap_bytes = (size_t)((char *)b->d_par - (char *)b->f0) + sizeof(int) * b->B;
    void *snap = nullptr;
    cudaError_t e = cudaMalloc(&snap, snap_bytes);
    if (e != cudaSuccess) return bfail(b, RLB_E_NOMEM, std::string("autotune snapshot: ") + cudaGetErrorString(e));
    RLB_BCUDA(b, cudaMemcpyAsync(snap, b->f0, snap_bytes, cudaMemcpyDeviceToDevice, b->stream));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);

    const rlb_batch_tuning saved = b->tune;
    std::vector<rlb_batch_tuning> done;
    rlb_status fail_st = RLB_OK;
    std::string fail_msg;
    auto run = [&](rlb_batch_tuning t) {
        if (fail_st != RLB_OK) return;
        t.ms = -1.0;
        if (apply_tuning(b, t) == RLB_OK) {
            cudaMemcpyAsync(b->f0, snap, snap_bytes, cudaMemcpyDeviceToDevice, b->stream);
            if (prepare(b, ts.data()) == RLB_OK) {
                const rlb::batch::Args a = make_args(b);
                cudaEventRecord(e0, b->stream);
                cudaError_t le = rlb::batch::launch_tubes(a, t.threads, t.bound, t.cluster, b->stream, nullptr);
                cudaEventRecord(e1, b->stream);
                cudaError_t se = cudaStreamSynchronize(b->stream);
                if (le == cudaSuccess && se == cudaSuccess) {
                    float ms = 0.0f;
                    cudaEventElapsedTime(&ms, e0, e1);
                    t.ms = ms;
                } else if (se != cudaSuccess) {
                    fail_st = RLB_E_CUDA;
                    fail_msg = std::string("autotune trial: ") + cudaGetErrorString(se);
                } else {
                    cudaGetLastError();
                }
                b->launches += 1;
                if (check_status(b) != RLB_OK) t.ms = -1.0;
            }
        }
        done.push_back(t);
    };
    for (int bound : {512, 384, 256})
        for (int threads : {128, 256, 384, 512})
            if (threads <= bound)
                for (int cluster : {1, 2, 4, 8}) run(rlb_batch_tuning{threads, bound, cluster, 1, 0.0});
    auto pick = [&]() {
        int k = -1;
        for (size_t i = 0; i < done.size(); ++i)
            if (done[i].ms > 0.0 && (k < 0 || done[i].ms < done[k].ms)) k = int(i);
        return k;
    };
    int k = pick();
    if (k >= 0) {
        const rlb_batch_tuning t1 = done[k];
        for (int ppt : {2, 4}) run(rlb_batch_tuning{t1.threads, t1.bound, t1.cluster, ppt, 0.0});
        k = pick();
    }
    cudaMemcpyAsync(b->f0, snap, snap_bytes, cudaMemcpyDeviceToDevice, b->stream);
    cudaStreamSynchronize(b->stream);
    cudaFree(snap);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (fail_st != RLB_OK) return bfail(b, fail_st, fail_msg);
    if (k < 0) {
        apply_tuning(b, saved);
        return bfail(b, RLB_E_CUDA, "no tuning candidate ran");
    }
    const rlb_batch_tuning chosen = done[k];
    st = apply_tuning(b, chosen);
    if (st != RLB_OK) return st;
    b->shape_set = true;
    b->tune.ms = chosen.ms;
    if (n_trials) *n_trials = int(done.size());
    for (int i = 0; i < max_trials && i < int(done.size()); ++i) trials[i] = done[i];
    if (best) *best = chosen;
    return RLB_OK;
}

rlb_status rlb_batch_set_stream(rlb_batch *b, void *cuda_stream)
{
    if (!b) return bfail(nullptr, RLB_E_INVALID, "batch is NULL");
    b->stream = (cudaStream_t)cuda_stream;
    return RLB_OK;
}

long long rlb_batch_total_cells(const rlb_batch *b) { return b ? b->total : 0; }

long long rlb_batch_launch_count(const rlb_batch *b) { return b ? b->launches : 0; }

void rlb_batch_destroy(rlb_batch *b)
{
    if (!b) return;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
    if (b->host) cudaFreeHost(b->host);
    if (b->block) cudaFree(b->block);
    delete b;
}

const char *rlb_batch_last_error(const rlb_batch *b) { return b ? b->err.c_str() : g_berr.c_str(); }

}  // extern "C"
