// api.cu -- the C ABI declared in include/fp.h.
//
// Host side of the hot path: per-pair depth draws, plan cache (one plan per
// depth for fixed-topology ensembles, one per pair for local circuits),
// batching under a device-memory budget, the launches (sampler -> merge ->
// tables -> sweep+meet), the FP32->FP64 recontraction policy and the
// Monte Carlo driver.  Every step of the path runs in the kernels; the host
// only plans, marshals and orders work.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <numeric>
#include <tuple>
#include <string>
#include <thread>
#include <vector>

#include "fp.h"
#include "kernels.h"
#include "brick.h"
#include "planner.h"
#include "side_stream.h"
#include "tune.h"

using namespace fpk;

namespace {

thread_local std::string g_err;

fp_status fail(fp_status s, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return s;
}

#define CK(call)                                                                         \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess)                                                           \
            return fail(e_ == cudaErrorMemoryAllocation ? FP_ERR_OOM : FP_ERR_CUDA,      \
                        "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

// Host-side fault injection (fp_inject_alloc_failures): the next N device
// allocations of ensemble buffers fail as if the device were out of memory.
std::atomic<int> g_alloc_failures{0};
// Time limit of every bounded device wait (fp_set_wait_limit_ns).
std::atomic<uint64_t> g_wait_ns{1000000000ull};

// Device buffer that grows on demand.
struct DBuf {
    void *p = nullptr;
    size_t bytes = 0;
    ~DBuf() { if (p) cudaFree(p); }
    cudaError_t reserve(size_t b) {
        if (b <= bytes) return cudaSuccess;
        if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
        for (int f = g_alloc_failures.load(); f > 0;)
            if (g_alloc_failures.compare_exchange_weak(f, f - 1)) return cudaErrorMemoryAllocation;
        cudaError_t e = cudaMalloc(&p, b);
        if (e == cudaSuccess) bytes = b;
        return e;
    }
    template <typename T> T *as() const { return (T *)p; }
};

bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

namespace fpk {
void set_last_error(const char *msg) { g_err = msg; }
uint64_t wait_limit_ns() { return g_wait_ns.load(); }
}  // namespace fpk

struct GraphKey {
    int key;
    uint64_t nb;
    const void *pairs, *raw, *maps, *states, *tr, *kappa, *err;
    bool operator<(const GraphKey &o) const {
        return std::tie(key, nb, pairs, raw, maps, states, tr, kappa, err) <
               std::tie(o.key, o.nb, o.pairs, o.raw, o.maps, o.states, o.tr, o.kappa, o.err);
    }
};

struct BrickCache {
    BrickHostPlan hp;
    DBuf d_gates, d_rpasses, d_rgates, d_tcwins, d_tcxa;
    BrickDevPlan dp;
    size_t extra_per_pair = 0;   // tensor-core window matrices (bytes per pair, after the boundaries)
    int variant[4] = {0, 0, 0, 0};   // tile bits, window bits, threads, pass kind (fp_brick_variant)
    double mma_flops_pair = 0;       // tensor-core flops issued per pair (tensor-core passes)
};

struct SpiralCache {        // one depth of the paper's HEA on the spiral sweep
    SpiralPlan sp;
    DBuf d_maps, d_items, d_refs, d_plan;
    // variants: FP64 over 2^p CTAs (p <= kSpiralMaxSplit; R = 0: not for this size, but
    // `base`, the smallest), then FP32
    static constexpr int kFp32 = kSpiralMaxSplit + 1;
    SpiralConfig cfg[kFp32 + 1];
    DBuf d_wins[kFp32 + 1];   // register windows of cfg[p]
    int nwins[kFp32 + 1] = {}, base = 0;
    int resident[kFp32] = {};        // FP64 clusters of variant p on the device at a time
    SpiralCut cut[kFp32 + 1];
};

struct fp_ensemble {
    static constexpr size_t kSideStreams = 8;
    fp_ensemble_desc d;
    cudaStream_t st = nullptr;
    int device = 0;
    int sms = 0;
    int raw_kind = RAW_HAAR4;
    int n_groups = 0;
    size_t ws_budget = 0;
    // fixed-topology plan cache
    std::map<int, int> plan_of_depth;
    std::vector<HostPlan> plans;
    bool dev_plans_dirty = true;
    // device plan pools (fixed topology) and per-batch pools (local)
    DBuf d_plans, d_ops, d_recipes, d_items, d_refs;
    // batch buffers
    DBuf d_pairs, d_order, d_raw, d_merged, d_tables, d_ws, d_ticket, d_tr, d_kappa, d_err, d_group;
    DBuf d_partials, d_moments;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    cudaEvent_t kev[2 * FP_K_CLASSES] = {};
    fp_kernel_stats kst{};
    uint64_t kst_requeued = 0;
    bool timing = false;
    // brickwork fast path
    std::map<int, std::unique_ptr<BrickCache>> brick_plans;   // key brick_key(l, prec)
    // spiral sweep (the paper's HEA), per depth; null: the depth is not spiral-shaped
    std::map<int, std::unique_ptr<SpiralCache>> spiral_plans;
    DBuf d_spiral_scratch;
    std::vector<SideStream> side;
    DBuf d_maps, d_states;
    DBuf d_step_items, d_step_which, d_step_pairs, d_step_meet, d_step_part;   // lock-step sweep
    DBuf d_flag;               // device error flag of kernels with bounded waits (zero when clear)
    std::atomic<int> cancel{0};   // fp_cancel: checked by the Monte Carlo driver between batches
    std::string gpu_name;
    // CUDA graphs of the brickwork sub-batch pipeline
    cudaStream_t gst = nullptr;
    cudaEvent_t gev[2] = {};
    std::map<GraphKey, cudaGraphExec_t> graphs;
    uint64_t graph_replays = 0;
    // FP_FLAG_SKIP_INFEASIBLE: slots (relative to the current call's first pair)
    // left uncontracted because their boundary exceeds FP_MAX_STATE_BITS
    std::vector<uint64_t> skipped;
    DBuf d_skip;
    // bootstrap buffers
    DBuf d_boot_tr, d_boot_group, d_boot_xs, d_boot_out;
    // resident clusters of the generic sweep per cluster size (index log2 cs) and precision; -1 unknown
    int sweep_slots[5][2] = {{-1, -1}, {-1, -1}, {-1, -1}, {-1, -1}, {-1, -1}};
};

namespace {

int depth_of_pair(const fp_ensemble_desc &d, uint64_t pair) {
    U64x4 x = philox(d.seed, 0, 0, pair, 4);
    if (d.kind == FP_LOCAL) {
        uint32_t choices = (uint32_t)((d.T_max - d.T_min) / d.T_step + 1);
        return d.T_min + (int)pick(x.x[0], choices) * d.T_step;
    }
    uint32_t choices = (uint32_t)(d.depth_max - d.depth_min + 1);
    return d.depth_min + (int)pick(x.x[0], choices);
}

int group_of_depth(const fp_ensemble_desc &d, int depth) {
    return d.kind == FP_LOCAL ? (depth - d.T_min) / d.T_step : depth - d.depth_min;
}

std::vector<int> local_bonds(const fp_ensemble_desc &d, uint64_t pair, int which, int T) {
    int w = (d.flags & FP_FLAG_SELF_PAIR) ? 0 : which;
    std::vector<int> b(T);
    for (int g = 0; g < T; ++g) {
        U64x4 x = philox(d.seed, 0, (uint64_t)g, pair, (uint64_t)(2 + w));
        b[g] = (int)pick(x.x[0], (uint32_t)(d.n - 1));
    }
    return b;
}

// f(i) for i in [0, count) on the host cores (at most 64 threads; serial for
// small counts).  f must be safe to run concurrently for different i.
template <typename F>
void parallel_for(uint64_t count, F f, unsigned most = 64) {
    unsigned nt = std::max(1u, std::min(most, std::thread::hardware_concurrency()));
    if (count < 64 || nt == 1) {
        for (uint64_t i = 0; i < count; ++i) f(i);
        return;
    }
    nt = (unsigned)std::min<uint64_t>(nt, count / 16);
    std::atomic<uint64_t> next{0};
    auto work = [&]() {
        for (;;) {
            const uint64_t i0 = next.fetch_add(16);
            if (i0 >= count) return;
            for (uint64_t i = i0; i < std::min(count, i0 + 16); ++i) f(i);
        }
    };
    std::vector<std::thread> th;
    for (unsigned t = 1; t < nt; ++t) th.emplace_back(work);
    work();
    for (auto &t : th) t.join();
}

// Gate layout of circuit `which` of a pair and the number of raw gates per circuit.
std::vector<GateSlot> circuit_layout(const fp_ensemble_desc &d, uint64_t pair, int which, int depth, int *n_raw) {
    switch (d.kind) {
        case FP_PARALLEL: {
            std::vector<GateSlot> g = layout_brickwork(d.n, depth);
            *n_raw = (int)g.size();
            return g;
        }
        case FP_HEA:
            *n_raw = depth * d.n;
            return layout_hea(d.n, depth);
        case FP_HEA_PAULI:
            *n_raw = 1 + d.n + depth * d.n;
            return layout_hea_pauli(d.n, depth, (d.flags & FP_FLAG_HEA_CZ) != 0);
        default:
            *n_raw = depth;
            return layout_local(d.n, local_bonds(d, pair, which, depth));
    }
}

HostPlan build_plan(const fp_ensemble_desc &d, int raw_kind, int depth, uint64_t pair) {
    int n_raw = 0;
    std::vector<GateSlot> U = circuit_layout(d, pair, 0, depth, &n_raw);
    std::vector<GateSlot> V = circuit_layout(d, pair, 1, depth, &n_raw);
    return make_plan(d.n, U, V, raw_kind, n_raw, d.n / 2, FP_MAX_STATE_BITS);
}

// Flatten host plans into device pools.
struct PlanPools {
    std::vector<DevPlan> plans;
    std::vector<DevOp> ops;
    std::vector<DevRecipe> recipes;
    std::vector<MergeItem> items;
    std::vector<MergeRef> refs;
    // plan(i), i in [0, count): sizes first, then the copies on the host cores, a thread (20 to 30 us to
    // start) per 8,192 operations (about 0.2 ms)
    template <typename F>
    void fill(size_t count, F plan) {
        plans.resize(count);
        size_t no = 0, ni = 0, nr = 0;
        for (size_t i = 0; i < count; ++i) {
            const HostPlan &h = plan(i);
            DevPlan &p = plans[i];
            std::memset(&p, 0, sizeof p);
            p.ops_off = p.rec_off = (int)no;
            p.merge_off = (int)ni;
            p.ref_off = (int)nr;
            no += h.ops.size();
            ni += h.merges.size();
            nr += h.refs.size();
        }
        ops.resize(no);
        recipes.resize(no);
        items.resize(ni);
        refs.resize(nr);
        parallel_for(count, [&](uint64_t i) {
            const HostPlan &h = plan(i);
            DevPlan &p = plans[i];
            p.n_left = h.n_left;
            p.n_right = h.n_right;
            p.n_merged = (int)h.merges.size();
            p.n_raw = h.n_raw;
            p.raw_kind = h.raw_kind;
            p.bits_max = h.bits_max;
            p.bits_final = h.bits_final;
            p.left_final_buf = h.left_final_buf;
            for (int k = 0; k < FP_MAX_STATE_BITS && k < (int)h.dot_perm.size(); ++k) p.dot_perm[k] = h.dot_perm[k];
            p.prefactor = h.prefactor;
            p.cost = h.cost;
            p.sqrt_ops = std::sqrt((double)std::max(1, std::max(h.n_left, h.n_right)));
            std::copy(h.ops.begin(), h.ops.end(), ops.begin() + p.ops_off);
            std::copy(h.recipes.begin(), h.recipes.end(), recipes.begin() + p.rec_off);
            std::copy(h.merges.begin(), h.merges.end(), items.begin() + p.merge_off);
            std::copy(h.refs.begin(), h.refs.end(), refs.begin() + p.ref_off);
        }, (unsigned)std::min<size_t>(64, 1 + no / 8192));
    }
};

template <typename T>
cudaError_t upload(DBuf &b, const std::vector<T> &v, cudaStream_t st) {
    size_t bytes = std::max<size_t>(sizeof(T), v.size() * sizeof(T));
    cudaError_t e = b.reserve(bytes);
    if (e != cudaSuccess || v.empty()) return e;
    return cudaMemcpyAsync(b.p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, st);
}

fp_status upload_pools(fp_ensemble *E, const PlanPools &pp) {
    CK(upload(E->d_plans, pp.plans, E->st));
    CK(upload(E->d_ops, pp.ops, E->st));
    CK(upload(E->d_recipes, pp.recipes, E->st));
    CK(upload(E->d_items, pp.items, E->st));
    CK(upload(E->d_refs, pp.refs, E->st));
    return FP_OK;
}

// Optional per-launch CUDA-event timing (FP_FLAG_TIMING).
struct KTimer {
    fp_ensemble *E;
    int cls;
    KTimer(fp_ensemble *e, int c) : E(e), cls(c) {
        if (E->timing) cudaEventRecord(E->kev[2 * cls], E->st);
    }
    cudaError_t stop(double work, int launches = 1) {
        if (!E->timing) return cudaSuccess;
        cudaError_t e = cudaEventRecord(E->kev[2 * cls + 1], E->st);
        if (e != cudaSuccess) return e;
        if ((e = cudaEventSynchronize(E->kev[2 * cls + 1])) != cudaSuccess) return e;
        float ms = 0;
        if ((e = cudaEventElapsedTime(&ms, E->kev[2 * cls], E->kev[2 * cls + 1])) != cudaSuccess) return e;
        E->kst.ms[cls] += ms;
        E->kst.launches[cls] += (uint64_t)launches;
        E->kst.work[cls] += work;
        return cudaSuccess;
    }
};

// Lock-step sweep (kernels_step.cu): pairs of at least 2^kStepBits amplitudes.  Below it a
// pair's boundary fits an SM's caches and one CTA per pair keeps it there: the 2,205 smaller
// pairs of 4,000 at n = 20, T = 20..100 take 0.6 ms.
constexpr int kStepBits = 14;
// amplitudes of one buffer of each side (whole 16-byte words)
void step_sides(const HostPlan &h, size_t *left, size_t *right) {
    int b[2] = {0, 0};
    for (size_t k = 0; k < h.ops.size(); ++k) {
        int &m = b[(int)k < h.n_left ? 0 : 1];
        m = std::max(m, (int)h.ops[k].b_out);
    }
    *left = std::max<size_t>(16, (size_t)1 << b[0]);
    *right = std::max<size_t>(16, (size_t)1 << b[1]);
}

// log2 of a block's units in a step of `items` operations and about `total` units: 10, or fewer (down to 6,
// two warps) until the step has two blocks per SM.  A batch of a few pairs is as fast as the number of
// SM quarters that share it, in FP64 above all (an instruction per 77 cycles and quarter): 2 pairs of n = 14,
// T = 70 take 0.93 ms in FP64; 1.55 with 10 throughout, 1.30 on clusters of 16 CTAs.
int step_log_units(uint64_t items, uint64_t total, int sms) {
    int lg = 10;
    while (lg > 6 && items + (total >> lg) < 2 * (uint64_t)sms) --lg;
    return lg;
}

// Work lists of a lock-step batch, uploaded; plans: the uploaded DevPlans by pinfo[i].plan.
template <typename F>
fp_status build_steps(fp_ensemble *E, uint64_t nb, F plan, const std::vector<PairInfo> &pinfo,
                      const std::vector<DevPlan> &plans, StepBatch &out) {
    std::vector<StepPair> sp(nb);
    size_t n_steps = 0, at = 0, n_items = 0;
    for (uint64_t i = 0; i < nb; ++i) n_steps = std::max(n_steps, (size_t)std::max(plan(i).n_left, plan(i).n_right));
    std::vector<uint32_t> count(n_steps + 1, 0), blocks(n_steps, 0);
    const bool few = nb < 2 * (uint64_t)E->sms;   // else the operations alone make two blocks per SM
    std::vector<uint64_t> quads(n_steps, 0);   // amplitudes first
    for (uint64_t i = 0; i < nb; ++i)
        for (int s = 0; s < 2; ++s)
            for (int k = 0; k < (s ? plan(i).n_right : plan(i).n_left); ++k) {
                ++count[k + 1];
                if (!few) continue;
                const DevOp &op = plan(i).ops[s ? plan(i).n_left + k : k];
                quads[k] += 1ull << std::max<int>(op.b_in, op.b_out);
            }
    for (size_t k = 0; k < n_steps; ++k) count[k + 1] += count[k];   // first item of each step
    n_items = count[n_steps];
    std::vector<uint8_t> log_units(n_steps);
    for (size_t k = 0; k < n_steps; ++k)
        log_units[k] = few ? (uint8_t)step_log_units(count[k + 1] - count[k], quads[k] >> 2, E->sms) : 10;
    std::vector<uint32_t> fill(count.begin(), count.end() - 1);
    std::vector<StepItem> items(n_items);
    uint32_t meet = 0;
    std::vector<uint32_t> meet_which;
    for (uint64_t r = nb; r-- > 0;) {   // largest boundaries first: the small ones fill the launch's tail
        const HostPlan &h = plan(r);
        size_t side[2];
        step_sides(h, &side[0], &side[1]);
        for (int s = 0; s < 2; ++s) {
            const uint64_t buf[2] = {at, at + side[s]};
            at += 2 * side[s];
            sp[r].base[s] = buf[0];
            int cur = 0;
            for (int k = 0; k < (s ? h.n_right : h.n_left); ++k) {
                const int local = s ? h.n_left + k : k;
                const DevOp &op = h.ops[local];
                StepItem &it = items[fill[k]++];
                std::memset(&it, 0, sizeof it);
                const bool flat = op.nk == 0;
                it.form = op.inplace2 ? STEP_IN_PLACE
                        : flat && op.nc == 1 && op.nn == 3 ? STEP_1_3
                        : flat && op.nc == 3 && op.nn == 1 ? STEP_3_1
                        : flat && op.nc == 0 && op.nn == 4 ? STEP_0_4
                        : flat && op.nc == 4 && op.nn == 0 ? STEP_4_0 : STEP_ANY;
                it.units = it.form == STEP_IN_PLACE ? 1u << (op.b_out - 2)
                         : it.form == STEP_ANY ? 1u << op.b_out : 1u << (op.b_in - op.nc);
                it.log_units = it.units >= (1u << 16) ? 12 : log_units[k];
                it.in = buf[cur];
                if (it.form != STEP_IN_PLACE) cur ^= 1;
                it.out = buf[cur];
                it.op = plans[pinfo[r].plan].ops_off + local;
                it.table = pinfo[r].table_off + local;
                it.first = blocks[k];
                blocks[k] += std::max(1u, it.units >> it.log_units);
            }
            sp[r].final[s] = buf[cur];
        }
        sp[r].first = meet;
        const uint32_t mb = h.bits_final > kMeetChunk ? 1u << (h.bits_final - kMeetChunk) : 1u;
        meet_which.insert(meet_which.end(), mb, (uint32_t)r);
        meet += mb;
    }
    out.step_first.assign(n_steps + 1, 0);
    for (size_t k = 0; k < n_steps; ++k) out.step_first[k + 1] = out.step_first[k] + blocks[k];
    std::vector<uint32_t> which(out.step_first[n_steps]);
    for (size_t k = 0; k < n_steps; ++k)
        for (uint32_t j = count[k]; j < count[k + 1]; ++j) {
            const uint32_t first = out.step_first[k] + items[j].first;
            std::fill_n(which.begin() + first, std::max(1u, items[j].units >> items[j].log_units), j);
        }
    CK(upload(E->d_step_items, items, E->st));
    CK(upload(E->d_step_which, which, E->st));
    CK(upload(E->d_step_pairs, sp, E->st));
    CK(upload(E->d_step_meet, meet_which, E->st));
    CK(E->d_step_part.reserve((size_t)meet * 4 * sizeof(double)));
    CK(cudaStreamSynchronize(E->st));   // the host lists end here
    out.items = E->d_step_items.as<StepItem>();
    out.which = E->d_step_which.as<uint32_t>();
    out.pairs = E->d_step_pairs.as<StepPair>();
    out.meet_which = E->d_step_meet.as<uint32_t>();
    out.partials = E->d_step_part.p;
    out.meet_blocks = meet;
    return FP_OK;
}

// Generic path over a subset of pairs: outputs go to slots idx[i] of the
// device arrays (pairs first + idx[i]).
fp_status run_generic(fp_ensemble *E, uint64_t first, const std::vector<uint64_t> &idx_in,
                      const std::vector<int> &depth, int prec, double *tr, double *kappa, double *err,
                      float *gpu_ms) {
    const fp_ensemble_desc &d = E->d;
    const bool local = d.kind == FP_LOCAL;
    const bool skip = (d.flags & FP_FLAG_SKIP_INFEASIBLE) != 0;
    if (idx_in.empty()) return FP_OK;
    std::vector<int> plan_idx;
    std::vector<HostPlan> local_plans;
    std::vector<uint64_t> kept;   // output slots contracted here, in batch order
    PlanPools pools;
    if (!local) {
        for (uint64_t slot : idx_in) {
            const int dep = depth[slot];
            auto it = E->plan_of_depth.find(dep);
            if (it == E->plan_of_depth.end()) {
                HostPlan h = build_plan(d, E->raw_kind, dep, first + slot);
                if (!h.error.empty() && !h.infeasible) return fail(FP_ERR_ARG, "planner: %s", h.error.c_str());
                if (h.infeasible && !skip) return fail(FP_ERR_INFEASIBLE, "depth %d: %s", dep, h.error.c_str());
                E->plans.push_back(std::move(h));
                it = E->plan_of_depth.emplace(dep, (int)E->plans.size() - 1).first;
                E->dev_plans_dirty = true;
            }
            const HostPlan &h = E->plans[it->second];
            if (h.infeasible) {
                if (!skip) return fail(FP_ERR_INFEASIBLE, "depth %d: %s", dep, h.error.c_str());
                E->skipped.push_back(slot);
                continue;
            }
            plan_idx.push_back(it->second);
            kept.push_back(slot);
        }
        if (E->dev_plans_dirty) {
            pools.fill(E->plans.size(), [&](size_t i) -> const HostPlan & { return E->plans[i]; });
            fp_status s = upload_pools(E, pools);
            if (s != FP_OK) return s;
            E->dev_plans_dirty = false;
        }
    } else {
        // every local-circuit pair has its own topology: plan them on the host
        // cores in parallel, then order the batch by boundary size so that the
        // memory-budgeted sub-batches below group pairs of similar workspace
        const uint64_t n_in = idx_in.size();
        std::vector<HostPlan> all(n_in);
        parallel_for(n_in, [&](uint64_t i) {
            all[i] = build_plan(d, E->raw_kind, depth[idx_in[i]], first + idx_in[i]);
        });
        std::vector<uint64_t> feas;
        for (uint64_t i = 0; i < n_in; ++i) {
            const HostPlan &h = all[i];
            if (h.infeasible) {
                if (!skip)
                    return fail(FP_ERR_INFEASIBLE, "pair %llu (T=%d): %s", (unsigned long long)(first + idx_in[i]),
                                depth[idx_in[i]], h.error.c_str());
                E->skipped.push_back(idx_in[i]);
                continue;
            }
            if (!h.error.empty()) return fail(FP_ERR_ARG, "planner: %s", h.error.c_str());
            feas.push_back(i);
        }
        std::stable_sort(feas.begin(), feas.end(),
                         [&](uint64_t a, uint64_t b) { return all[a].bits_max < all[b].bits_max; });
        for (uint64_t i : feas) {
            local_plans.push_back(std::move(all[i]));
            kept.push_back(idx_in[i]);
        }
        for (uint64_t i = 0; i < local_plans.size(); ++i) plan_idx.push_back((int)i);
        pools.fill(local_plans.size(), [&](size_t i) -> const HostPlan & { return local_plans[i]; });
        if (!local_plans.empty()) {
            fp_status s = upload_pools(E, pools);
            if (s != FP_OK) return s;
            E->dev_plans_dirty = true;   // the fixed-topology pool was overwritten
        }
    }
    const uint64_t count = kept.size();
    if (count == 0) return FP_OK;
    const std::vector<DevPlan> &dev_plans = pools.plans;   // (local circuits: filled above)
    const std::vector<uint64_t> &idx = kept;
    auto hp = [&](uint64_t i) -> const HostPlan & { return local ? local_plans[i] : E->plans[plan_idx[i]]; };
    const bool fp32 = prec != FP_PREC_FP64;
    const size_t celem = fp32 ? sizeof(float2) : sizeof(double2);
    // pairs with large boundaries get a cluster of CTAs each (see sweep_cluster_size)
    auto cluster_of = [&](int bits) {
        int cs = sweep_cluster_size(bits);
        while (cs > 1) {
            int lg = cs == 4 ? 2 : (cs == 8 ? 3 : 4);
            int &slots = E->sweep_slots[lg][fp32 ? 1 : 0];
            if (slots < 0) slots = sweep_max_clusters(cs, fp32);
            if (slots > 0) return std::make_pair(cs, slots);
            cs /= 2;   // clusters of this size cannot launch here: smaller ones
            if (cs == 2) cs = 1;
        }
        return std::make_pair(1, E->sms * 2);
    };
    // local-circuit pairs of 2^14 amplitudes and more go in lock-step (kernels_step.cu), each with
    // its own boundaries; they are the last ones in the order by size.  A batch of fewer pairs than SMs with a large
    // one among them goes in lock-step as a whole: apart, the small ones, a CTA each, take their time before
    // the large ones (5 pairs of n = 18, T = 60 in FP64: 0.69 ms together, 1.20 apart).
    const bool lockstep = local && !sweep_cluster_forced();
    const int step_bits = lockstep && count < (uint64_t)E->sms && hp(count - 1).bits_max >= kStepBits ? 0 : kStepBits;
    auto in_steps = [&](uint64_t i) { return lockstep && hp(i).bits_max >= step_bits; };
    uint64_t done = 0;
    while (done < count) {
        uint64_t nb = 0;
        size_t raw_b = 0, mer_b = 0, tab_b = 0, step_b = 0;
        int bits_max = 0, max_raw = 0, max_mer = 0, max_ops = 0;
        const bool steps = in_steps(done);
        while (done + nb < count && nb < 65535) {
            const HostPlan &h = hp(done + nb);
            if (in_steps(done + nb) != steps) break;
            size_t r = (size_t)2 * h.n_raw * 16 * sizeof(double2);
            size_t m = h.merges.size() * 16 * sizeof(double2);
            size_t t = h.ops.size() * 16 * sizeof(double2);
            int bm = std::max(bits_max, h.bits_max);
            const int slots_full = cluster_of(bm).second;
            size_t ws = (size_t)std::min<uint64_t>(slots_full, nb + 1) * 3 * ((size_t)1 << bm) * sizeof(double2);
            size_t own = 0;
            if (steps) {
                size_t sl, sr;
                step_sides(h, &sl, &sr);
                own = 2 * (sl + sr) * celem;
            }
            if (nb > 0 && raw_b + r + mer_b + m + tab_b + t + (steps ? step_b + own : ws) > E->ws_budget) break;
            raw_b += r; mer_b += m; tab_b += t; step_b += own; bits_max = bm;
            max_raw = std::max(max_raw, h.n_raw);
            max_mer = std::max<int>(max_mer, (int)h.merges.size());
            max_ops = std::max<int>(max_ops, (int)h.ops.size());
            ++nb;
        }
        std::vector<PairInfo> pinfo(nb);
        int64_t ro = 0, mo = 0, to = 0;
        double cmacs = 0;
        for (uint64_t i = 0; i < nb; ++i) {
            const HostPlan &h = hp(done + i);
            pinfo[i].pair = first + idx[done + i];
            pinfo[i].plan = plan_idx[done + i];
            pinfo[i].n_raw = h.n_raw;
            pinfo[i].raw_off = ro;
            pinfo[i].merged_off = mo;
            pinfo[i].table_off = to;
            pinfo[i].out = (int64_t)idx[done + i];
            ro += 2 * h.n_raw;
            mo += (int64_t)h.merges.size();
            to += (int64_t)h.ops.size();
            cmacs += h.cost;
        }
        std::vector<int32_t> order(nb);
        std::iota(order.begin(), order.end(), 0);
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return hp(done + a).cost > hp(done + b).cost; });
        const auto cl = cluster_of(bits_max);
        const int slots = (int)std::min<uint64_t>(nb, (uint64_t)cl.second);
        const int ctas = slots * cl.first;
        size_t ws_elems = (size_t)1 << bits_max;
        CK(upload(E->d_pairs, pinfo, E->st));
        StepBatch sb;
        if (steps) {
            fp_status bs = build_steps(E, nb, [&](uint64_t i) -> const HostPlan & { return hp(done + i); }, pinfo, dev_plans, sb);
            if (bs != FP_OK) return bs;
        } else {
            CK(upload(E->d_order, order, E->st));
        }
        CK(E->d_raw.reserve(std::max<size_t>(16, ro * 16 * sizeof(double2))));
        CK(E->d_merged.reserve(std::max<size_t>(16, mo * 16 * sizeof(double2))));
        CK(E->d_tables.reserve(std::max<size_t>(16, to * 16 * sizeof(double2))));
        CK(E->d_ws.reserve(steps ? step_b : (size_t)slots * 3 * ws_elems * celem));
        SampleParams sp;
        sp.seed = d.seed;
        sp.n = d.n;
        sp.raw_kind = E->raw_kind;
        sp.self_pair = (d.flags & FP_FLAG_SELF_PAIR) ? 1 : 0;
        CK(cudaEventRecord(E->ev0, E->st));
        {
            KTimer t(E, FP_K_SAMPLE);
            CK(launch_sample(sp, E->d_pairs.as<PairInfo>(), (int)nb, max_raw, E->d_raw.as<double2>(), E->st));
            CK(t.stop((double)nb));
        }
        {
            KTimer t(E, FP_K_MERGE);
            CK(launch_merge(E->d_pairs.as<PairInfo>(), (int)nb, max_mer, E->d_plans.as<DevPlan>(),
                            E->d_items.as<MergeItem>(), E->d_refs.as<MergeRef>(), E->d_raw.as<double2>(),
                            E->d_merged.as<double2>(), E->st));
            CK(t.stop((double)nb));
        }
        {
            KTimer t(E, FP_K_TABLES);
            CK(launch_tables(E->d_pairs.as<PairInfo>(), (int)nb, max_ops, E->d_plans.as<DevPlan>(),
                             E->d_recipes.as<DevRecipe>(), E->d_merged.as<double2>(), E->d_tables.p, fp32, E->st));
            CK(t.stop((double)nb));
        }
        {
            KTimer t(E, FP_K_SWEEP);
            if (steps) {
                CK(launch_steps(sb, E->d_pairs.as<PairInfo>(), (int)nb, E->d_plans.as<DevPlan>(), E->d_ops.as<DevOp>(),
                                E->d_tables.p, fp32, E->d_ws.p, FP_ERR_SAFETY * (fp32 ? 0x1.0p-24 : 0x1.0p-53), tr,
                                kappa, err, E->st));
                CK(t.stop(cmacs, (int)sb.step_first.size() + 2));
            } else {
            CK(launch_sweep_generic(E->d_pairs.as<PairInfo>(), E->d_order.as<int32_t>(), (int)nb, E->d_plans.as<DevPlan>(),
                                    E->d_ops.as<DevOp>(), E->d_tables.p, fp32, E->d_ws.p, ws_elems, ctas,
                                    cl.first, E->d_ticket.as<int>(), FP_ERR_SAFETY * (fp32 ? 0x1.0p-24 : 0x1.0p-53), tr,
                                    kappa, err, E->st));
            CK(t.stop(cmacs));
            }
        }
        CK(cudaEventRecord(E->ev1, E->st));
        CK(cudaEventSynchronize(E->ev1));
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, E->ev0, E->ev1));
        if (gpu_ms) *gpu_ms += ms;
        E->kst.pairs += nb;
        done += nb;
    }
    return FP_OK;
}

// Build and upload one brickwork plan variant.
// The device error flag of kernels with bounded waits: a raised flag is
// reported as FP_ERR_TIMEOUT and cleared, so that the ensemble stays usable.
fp_status check_flag(fp_ensemble *E) {
    int h = 0;
    CK(cudaMemcpyAsync(&h, E->d_flag.p, sizeof h, cudaMemcpyDeviceToHost, E->st));
    CK(cudaStreamSynchronize(E->st));
    if (!h) return FP_OK;
    CK(cudaMemsetAsync(E->d_flag.p, 0, sizeof h, E->st));
    return fail(FP_ERR_TIMEOUT, "a bounded device wait ran out in the tensor-core tile pass (results discarded)");
}

// The brickwork plan cache's key: depth and precision class (FP64; FP32 with the
// autotuner's free choice; FP32 restricted to the tensor-core passes).
int brick_key(int l, int prec) {
    return 4 * l + (prec == FP_PREC_FP64 ? 0 : prec == FP_PREC_TF32X3 ? 2 : 1);
}

fp_status make_brick_cache(fp_ensemble *E, int l, int prec, int K, int R, int TH, int persist,
                           std::unique_ptr<BrickCache> &out) {
    const bool fp32 = prec != FP_PREC_FP64;
    auto bc = std::make_unique<BrickCache>();
    if (persist == 5) {   // the HEA sweep: its shape follows from the boundary
        K = 99;
        if (E->d.kind != FP_HEA || !hea_shape(2 * (l - 1), fp32, &R, &TH))
            return fail(FP_ERR_ARG, "the HEA sweep needs an HEA boundary of at most 14 bits");
    }
    bc->variant[0] = K; bc->variant[1] = R; bc->variant[2] = TH; bc->variant[3] = persist;
    // K > N: shared-memory sweep, K == N: one tile
    // arcs hold the 5 (FP32) or 4 (FP64) lowest bits, so that tile loads read contiguous runs;
    // the tensor-core pass (12-bit tiles) holds 3: at l = 10 a 12-bit arc through the 5
    // lowest bits would need 49 passes instead of 20.  FP_PREC_TF32X3 from 20 bits up: 2 (27 passes
    // at l = 11 instead of 49, a run of 4 amplitudes is one 32-byte sector; 2 % at 22 and 24 bits).
    // FP_PREC_FP32 keeps 3, with which the FFMA passes are the faster ones at 20 bits (n = 50, 96
    // pairs: 34.8 ms against 35.7): with 2 the tensor cores would win there (26.6 ms) with 9
    // times the error (1.1e-5 of a trace against 1.3e-6, their accumulators truncate).
    const int low = persist >= 3 ? (prec == FP_PREC_TF32X3 && 2 * (l - 1) >= 20 ? 2 : 3) : (fp32 ? 5 : 4);
    bc->hp = make_brick_plan(E->d.n, l, K, low, R, E->d.kind == FP_HEA ? 1 : 0);
    for (const auto &ps : bc->hp.passes) {
        if (ps.n_gates > 255) return fail(FP_ERR_ARG, "tile pass with %d gates exceeds 255", ps.n_gates);
        if (ps.n_rp > 160) return fail(FP_ERR_ARG, "tile pass with %d register passes exceeds 160", ps.n_rp);
    }
    if (persist == 3 || persist == 4) {   // tensor-core windows: FP32, 12-bit tiles, 5-bit windows only
        if (!fp32 || !tc_plan_ok(bc->hp.dev, bc->hp.passes.data(), bc->hp.rpasses.data()))
            return fail(FP_ERR_ARG, "the tensor-core tile pass needs FP32, %d-bit tiles, %d-bit windows and l >= 8",
                        kTcTile, kMaxWin);
        const std::vector<TcWin> wins = make_tc_windows(bc->hp, persist == 3);
        CK(upload(bc->d_tcwins, wins, E->st));
        CK(upload(bc->d_tcxa, make_tc_xaddr(bc->hp, wins), E->st));
        bc->dp.tcwins = bc->d_tcwins.as<TcWin>();
        bc->dp.tcxa = bc->d_tcxa.as<TcXa>();
        bc->extra_per_pair = tc_wmat_bytes_per_pair(bc->hp.dev, bc->hp.passes.data());
        // per window and tile: 3 products x 8 K steps of a 128 x 64 x 8 MMA
        double windows = 0;
        for (const BrickPass &ps : bc->hp.passes) windows += ps.n_rp;
        bc->mma_flops_pair = windows * (double)(1u << (bc->hp.dev.N - kTcTile)) * 3.0 * 2.0 * 128.0 * 64.0 * 64.0;
        if (!E->d_flag.p) {
            CK(E->d_flag.reserve(16));
            CK(cudaMemsetAsync(E->d_flag.p, 0, 16, E->st));
        }
        bc->dp.err_flag = E->d_flag.as<int>();
    }
    CK(upload(bc->d_gates, bc->hp.gates, E->st));
    CK(upload(bc->d_rpasses, bc->hp.rpasses, E->st));
    CK(upload(bc->d_rgates, bc->hp.rgates, E->st));
    bc->dp.gates = bc->d_gates.as<BrickGate>();
    bc->dp.rpasses = bc->d_rpasses.as<RegPass>();
    bc->dp.rgates = bc->d_rgates.as<RegGate>();
    bc->dp.win_bits = R;
    bc->dp.threads = TH;
    bc->dp.persist = persist;
    out = std::move(bc);
    return FP_OK;
}

// Autotuner: time every (tile bits, window bits) variant of the tiled
// brickwork sweep on a trial batch of this depth (sampler and maps once, then
// each variant's init + passes + meet), keep the fastest.  Results persist in
// the file named by FP_AUTOTUNE_CACHE (if set), keyed by GPU name, n, l and
// precision.
fp_status tune_brick(fp_ensemble *E, uint64_t first, const std::vector<uint64_t> &idx, int l, int prec) {
    const fp_ensemble_desc &d = E->d;
    const int N = 2 * (l - 1);
    const bool fp32 = prec != FP_PREC_FP64;
    const int key = brick_key(l, prec);
    struct Cand { int K, R, TH, P; };
    // K = 99: whole boundary in one CTA's shared memory (brick_smem_kernel);
    // P = 1: persistent double-buffered tile passes (brick_pass_db_kernel)
    std::vector<Cand> cands = fp32 ? std::vector<Cand>{{14, 4, 512, 0}, {14, 5, 256, 0}, {13, 4, 512, 0},
                                                       {13, 4, 256, 0}, {13, 5, 256, 0}, {13, 4, 512, 1},
                                                       {13, 5, 256, 1}, {12, 4, 256, 0}, {12, 5, 128, 0}}
                                   : std::vector<Cand>{{13, 3, 512, 0}, {13, 4, 256, 0}};
    if (((size_t)1 << N) * (fp32 ? sizeof(float2) : sizeof(double2)) <= (size_t)200 * 1024) cands.push_back({99, 0, 0, 0});
    // P = 4: tensor-core windows (TF32 x 3 tcgen05 MMAs) with the tile's operand in tensor memory,
    // boundaries of more than two 12-bit tiles.  P = 3 (the operand in shared memory) runs when the
    // cache file asks for it; it was 20-25 % slower at every depth, and planning it took seconds.
    if (fp32 && N >= kTcTile + 2) cands.push_back({kTcTile, kMaxWin, 256, 4});
    // P = 5: the HEA's own sweep, the fastest of all wherever it applies (kernels_hea.cu), so
    // there is nothing to time; FP_PREC_TF32X3 keeps to the tensor cores where they apply
    int heaR = 0, heaT = 0;
    if (d.kind == FP_HEA && !(prec == FP_PREC_TF32X3 && N >= kTcTile + 2) && hea_shape(N, fp32, &heaR, &heaT))
        cands.assign(1, {99, heaR, heaT, 5});
    const int kmin = 10;   // boundaries up to 2^10: shared-memory sweep, nothing to tune
    char ckey[256];
    // the HEA's ring has its own plans: its entries carry the kind after the precision
    snprintf(ckey, sizeof ckey, "%s n=%d l=%d %s%s", E->gpu_name.c_str(), d.n, l,
             !fp32 ? "fp64" : (prec == FP_PREC_TF32X3 && N >= kTcTile + 2) ? "tf32x3" : "fp32",
             d.kind == FP_HEA ? " hea" : "");
    int bestK = cands[0].K, bestR = cands[0].R, bestT = cands[0].TH, bestP = cands[0].P;
    bool have = false;
    const char *cache = getenv("FP_AUTOTUNE_CACHE");
    if (N <= kmin) {
        have = true;            // whole boundary in one CTA: nothing to tune
        bestK = 99;
    } else if (cache) {
        FILE *f = fopen(cache, "r");
        if (f) {
            char line[512];
            while (fgets(line, sizeof line, f)) {
                int K, R, T, Pp = 0;
                char k2[256];
                if (sscanf(line, "%255[^|]|%d %d %d %d", k2, &K, &R, &T, &Pp) >= 4 && strcmp(k2, ckey) == 0) {
                    bestK = K; bestR = R; bestT = T; bestP = Pp; have = true;
                }
            }
            fclose(f);
        }
    }
    // where one variant alone is in question, the file's word does not count: entries of before
    // the HEA sweep would keep a boundary on passes some 7 times slower
    if (have && N > kmin && cands.size() == 1 && bestP != cands[0].P) have = false;
    std::unique_ptr<BrickCache> cached;
    if (have && N > kmin && make_brick_cache(E, l, prec, bestK, bestR, bestT, bestP, cached) != FP_OK) {
        have = false;   // a cache entry this depth cannot run (another build's file): tune instead
        cached.reset();
    }
    if (!have && cands.size() == 1) {
        bestK = cands[0].K; bestR = cands[0].R; bestT = cands[0].TH; bestP = cands[0].P;
        if (cache) {
            FILE *f = fopen(cache, "a");
            if (f) { fprintf(f, "%s|%d %d %d %d\n", ckey, bestK, bestR, bestT, bestP); fclose(f); }
        }
    } else if (!have && !idx.empty()) {
        const uint64_t nt = std::min<uint64_t>(idx.size(), 192);   // several waves of tiles per variant
        const int n_raw = d.kind == FP_HEA ? l * d.n : (int)layout_brickwork(d.n, l).size();
        const int n_maps = (d.kind == FP_HEA ? 2 * d.n : d.n - 1) * (l - 1);
        const size_t celem = fp32 ? sizeof(float2) : sizeof(double2);
        std::vector<PairInfo> pinfo(nt);
        for (uint64_t i = 0; i < nt; ++i) {
            std::memset(&pinfo[i], 0, sizeof(PairInfo));
            pinfo[i].pair = first + idx[i];
            pinfo[i].n_raw = n_raw;
            pinfo[i].raw_off = (int64_t)i * 2 * n_raw;
            pinfo[i].out = (int64_t)idx[i];
        }
        CK(upload(E->d_pairs, pinfo, E->st));
        const bool haar = E->raw_kind == RAW_HAAR4;   // maps straight from the sampler
        if (!haar) CK(E->d_raw.reserve(nt * 2 * n_raw * 16 * sizeof(double2)));
        CK(E->d_maps.reserve(nt * n_maps * 16 * celem));
        CK(E->d_states.reserve(nt * 2 * ((size_t)1 << N) * celem));
        SampleParams sp;
        sp.seed = d.seed; sp.n = d.n; sp.raw_kind = E->raw_kind; sp.self_pair = (d.flags & FP_FLAG_SELF_PAIR) ? 1 : 0;
        if (haar)
            CK(launch_brick_haar_maps(make_brick_plan(d.n, l, 0, 0, 0).dev, sp, E->d_pairs.as<PairInfo>(), (int)nt,
                                      E->d_maps.p, fp32, E->st));
        else
            CK(launch_sample(sp, E->d_pairs.as<PairInfo>(), (int)nt, n_raw, E->d_raw.as<double2>(), E->st));
        std::unique_ptr<BrickCache> bc;
        // (the uncounted run: a few pairs, which load the code)
        auto run = [&](int i, bool counted, float &ms) -> int {
            const int np = counted ? (int)nt : (int)std::min<uint64_t>(nt, 4);
            const Cand &c = cands[(size_t)i];
            if (c.K != 99 && c.K > N) return 1;   // tiles larger than the boundary
            const int want[4] = {c.K, c.R, c.TH, c.P};
            if (!bc || std::memcmp(bc->variant, want, sizeof want) != 0) {
                if (make_brick_cache(E, l, prec, c.K, c.R, c.TH, c.P, bc) != FP_OK) return 1;
                if (bc->extra_per_pair) CK(E->d_states.reserve(nt * (2 * ((size_t)1 << N) * celem + bc->extra_per_pair)));
            }
            CK(cudaEventRecord(E->ev0, E->st));
            int nl = 0;
            if (launch_brick(bc->hp.dev, bc->hp.passes.data(), bc->dp, E->d_pairs.as<PairInfo>(), np,
                             haar ? nullptr : E->d_raw.as<double2>(), E->d_maps.p, E->d_states.p, fp32, 0.0, E->d_tr.as<double>(),
                             nullptr, nullptr, E->st, &nl) != cudaSuccess) {
                cudaGetLastError();   // a variant this device cannot launch: skip it
                return 1;
            }
            CK(cudaEventRecord(E->ev1, E->st));
            CK(cudaEventSynchronize(E->ev1));
            CK(cudaEventElapsedTime(&ms, E->ev0, E->ev1));
            return bc->dp.err_flag ? check_flag(E) : FP_OK;
        };
        std::vector<float> ms;
        const int ts = time_variants((int)cands.size(), ms, run);
        if (ts < 0) return (fp_status)ts;
        // FP_PREC_TF32X3: the fastest tensor-core variant when one runs, else the fastest of all
        // The others take the tensor cores where they gain 2 %: their traces have 7 to 11 times the
        // error, which noise in the timing (half a percent) should not decide.  (n = 50, fastest FFMA
        // variant over tensor cores in a trial of up to 192 pairs: l = 8 1.04, 9 1.35, 10 1.48,
        // 11 0.89 to 0.98, 12 1.29, 13 1.21.)
        float best_ms = kNoTime, best_tc_ms = kNoTime;
        Cand best_tc{0, 0, 0, 0};
        for (size_t i = 0; i < cands.size(); ++i) {
            const Cand &c = cands[i];
            if (c.P >= 3 && prec != FP_PREC_TF32X3) ms[i] *= 1.02f;
            if (ms[i] < best_ms) { best_ms = ms[i]; bestK = c.K; bestR = c.R; bestT = c.TH; bestP = c.P; }
            if (c.P >= 3 && ms[i] < best_tc_ms) { best_tc_ms = ms[i]; best_tc = c; }
        }
        if (prec == FP_PREC_TF32X3 && best_tc_ms < kNoTime) {
            bestK = best_tc.K; bestR = best_tc.R; bestT = best_tc.TH; bestP = best_tc.P;
        }
        if (cache) {
            FILE *f = fopen(cache, "a");
            if (f) { fprintf(f, "%s|%d %d %d %d\n", ckey, bestK, bestR, bestT, bestP); fclose(f); }
        }
    }
    std::unique_ptr<BrickCache> bc = std::move(cached);
    if (!bc) {
        fp_status s = make_brick_cache(E, l, prec, bestK, bestR, bestT, bestP, bc);
        if (s != FP_OK) return s;
    }
    E->brick_plans.emplace(key, std::move(bc));
    return FP_OK;
}

// Brickwork fast path for pairs of one depth l >= 2.
fp_status run_brick(fp_ensemble *E, uint64_t first, const std::vector<uint64_t> &idx, int l, int prec,
                    double *tr, double *kappa, double *err, float *gpu_ms) {
    const fp_ensemble_desc &d = E->d;
    const uint64_t count = idx.size();
    if (count == 0) return FP_OK;
    const bool fp32 = prec != FP_PREC_FP64;
    const int N = 2 * (l - 1);
    if (N > FP_MAX_STATE_BITS)
        return fail(FP_ERR_INFEASIBLE, "depth %d: boundary of %d bits exceeds the limit of %d", l, N, FP_MAX_STATE_BITS);
    const int key = brick_key(l, prec);
    auto it = E->brick_plans.find(key);
    if (it == E->brick_plans.end()) {
        fp_status s = tune_brick(E, first, idx, l, prec);
        if (s != FP_OK) return s;
        it = E->brick_plans.find(key);
    }
    const BrickHostPlan &bp = it->second->hp;
    const BrickDev &bd = bp.dev;
    const size_t celem = fp32 ? sizeof(float2) : sizeof(double2);
    const size_t S = (size_t)1 << N;
    const int n_raw = d.kind == FP_HEA ? l * d.n : (int)layout_brickwork(d.n, l).size();
    const bool hea = it->second->dp.persist == 5;   // slot factors in place of raw gates and maps
    const bool haar = E->raw_kind == RAW_HAAR4;     // maps straight from the sampler
    const size_t per_raw = hea || haar ? 0 : (size_t)2 * n_raw * 16 * sizeof(double2);
    const size_t per_map = hea ? (size_t)d.n * N * 4 * celem : (size_t)maps_per_pair(bd) * 16 * celem;
    bool both = false;
    if (bd.tile_bits == 0 && !hea) brick_smem_bytes(bd, fp32, &both);
    const size_t per_state = bd.tile_bits ? 2 * S * celem + it->second->extra_per_pair : (both ? 0 : S * celem);
    const size_t per_pair = per_raw + per_map + per_state;
    uint64_t cap = std::max<uint64_t>(1, std::min<uint64_t>(65535, E->ws_budget / per_pair));
    // work of the sweep (complex multiply-adds): 4 per amplitude per gate; the HEA's own sweep, per qubit
    // and amplitude: a product per register window (per factor up to 4 bits) and N Hadamards, 2 real
    // additions of an 8-flop multiply-add each
    double cmac_pair = 4.0 * (double)S * (double)maps_per_pair(bd);
    if (hea) {
        const int R = it->second->variant[1];
        cmac_pair = (double)S * d.n * ((N <= 4 ? N : (N + R - 1) / R) + N / 4.0);
    }
    SampleParams sp;
    sp.seed = d.seed;
    sp.n = d.n;
    sp.raw_kind = E->raw_kind;
    sp.self_pair = (d.flags & FP_FLAG_SELF_PAIR) ? 1 : 0;
    for (uint64_t done = 0; done < count;) {
        const uint64_t nb = std::min<uint64_t>(cap, count - done);
        std::vector<PairInfo> pinfo(nb);
        for (uint64_t i = 0; i < nb; ++i) {
            std::memset(&pinfo[i], 0, sizeof(PairInfo));
            pinfo[i].pair = first + idx[done + i];
            pinfo[i].n_raw = n_raw;
            pinfo[i].raw_off = (int64_t)i * 2 * n_raw;
            pinfo[i].out = (int64_t)idx[done + i];
        }
        CK(upload(E->d_pairs, pinfo, E->st));
        CK(E->d_raw.reserve(std::max<size_t>(16, nb * per_raw)));
        CK(E->d_maps.reserve(nb * per_map));
        CK(E->d_states.reserve(std::max<size_t>(16, nb * per_state)));
        const double G = (double)std::max(bd.n_layers[0], bd.n_layers[1]) * bd.m;
        // (FP64 in 64-bit integers, fixed.h: alignment, product and settling each round a component within
        // half a unit, 2^-58 to 2^-57 of its block's largest: together rms 2^-54.5 of the norm of a block of 16
        // amplitudes at most, 2^-55.5 of a quad's, where the estimate takes 2^-53 an operation)
        const double err_scale = FP_ERR_SAFETY * (fp32 ? 0x1.0p-24 : 0x1.0p-53) * std::sqrt(G);
        // CUDA graph replay: the launch sequence of a sub-batch (sampler, maps,
        // init, passes, meet) is captured once per (depth, precision, size,
        // buffers) on the ensemble's internal stream and replayed with fresh
        // pair records; the first sub-batch of a shape runs directly (it also
        // sets the kernels' shared-memory attributes outside any capture).
        const bool use_graph = !E->timing && !(d.flags & FP_FLAG_NO_GRAPHS);
        auto sample = [&](cudaStream_t st) {
            return hea  ? launch_hea_slots(sp, E->d_pairs.as<PairInfo>(), (int)nb, l, E->d_maps.p, fp32, st)
                   : haar ? launch_brick_haar_maps(bd, sp, E->d_pairs.as<PairInfo>(), (int)nb, E->d_maps.p, fp32, st)
                       : launch_sample(sp, E->d_pairs.as<PairInfo>(), (int)nb, n_raw, E->d_raw.as<double2>(), st);
        };
        auto sweep = [&](cudaStream_t st, int *nl) {
            if (!hea)
                return launch_brick(bd, bp.passes.data(), it->second->dp, E->d_pairs.as<PairInfo>(), (int)nb,
                                    haar ? nullptr : E->d_raw.as<double2>(), E->d_maps.p, E->d_states.p, fp32,
                                    err_scale, tr, kappa, err, st, nl);
            *nl = 1;
            return launch_hea_sweep(bd, E->d_pairs.as<PairInfo>(), (int)nb, E->d_maps.p, E->d_states.p, fp32, err_scale,
                                    tr, kappa, err, st);
        };
        GraphKey gk{key, nb, E->d_pairs.p, E->d_raw.p, E->d_maps.p, E->d_states.p, tr, kappa, err};
        auto git = use_graph ? E->graphs.find(gk) : E->graphs.end();
        CK(cudaEventRecord(E->ev0, E->st));
        if (use_graph && git != E->graphs.end() && git->second) {
            CK(cudaEventRecord(E->gev[0], E->st));
            CK(cudaStreamWaitEvent(E->gst, E->gev[0], 0));
            CK(cudaGraphLaunch(git->second, E->gst));
            CK(cudaEventRecord(E->gev[1], E->gst));
            CK(cudaStreamWaitEvent(E->st, E->gev[1], 0));
            E->graph_replays++;
        } else {
            {
                KTimer t(E, FP_K_SAMPLE);
                CK(sample(E->st));
                CK(t.stop((double)nb));
            }
            {
                KTimer t(E, FP_K_BRICK);
                int nl = 0;
                CK(sweep(E->st, &nl));
                CK(t.stop(cmac_pair * (double)nb));
                if (E->timing) {
                    E->kst.launches[FP_K_BRICK] += (uint64_t)(nl - 1);
                    E->kst.mma_flops += it->second->mma_flops_pair * (double)nb;
                }
            }
            if (use_graph) {
                if (E->graphs.size() > 64) {
                    for (auto &kv : E->graphs) if (kv.second) cudaGraphExecDestroy(kv.second);
                    E->graphs.clear();
                }
                cudaGraph_t graph = nullptr;
                cudaGraphExec_t exec = nullptr;
                CK(cudaStreamBeginCapture(E->gst, cudaStreamCaptureModeThreadLocal));
                cudaError_t ce = sample(E->gst);
                int nl = 0;
                if (ce == cudaSuccess) ce = sweep(E->gst, &nl);
                cudaError_t ee = cudaStreamEndCapture(E->gst, &graph);
                if (ce == cudaSuccess && ee == cudaSuccess && graph) {
                    ce = cudaGraphInstantiate(&exec, graph, 0);
                    if (ce != cudaSuccess) exec = nullptr;
                }
                if (graph) cudaGraphDestroy(graph);
                cudaGetLastError();           // a failed capture leaves the direct path in use
                E->graphs[gk] = exec;
            }
        }
        CK(cudaEventRecord(E->ev1, E->st));
        CK(cudaEventSynchronize(E->ev1));
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, E->ev0, E->ev1));
        if (gpu_ms) *gpu_ms += ms;
        if (it->second->dp.err_flag) {
            fp_status fs = check_flag(E);
            if (fs != FP_OK) return fs;
        }
        E->kst.pairs += nb;
        done += nb;
    }
    return FP_OK;
}

// The spiral program of depth L (built and uploaded once); null when the
// circuit is not spiral-shaped (the generic sweep takes it then).
SpiralCache *spiral_plan(fp_ensemble *E, int L) {
    auto it = E->spiral_plans.find(L);
    if (it != E->spiral_plans.end()) return it->second.get();
    std::unique_ptr<SpiralCache> sc;
    int n_raw = 0;
    const std::vector<GateSlot> lay = circuit_layout(E->d, 0, 0, L, &n_raw);
    SpiralPlan sp = make_spiral_plan(E->d.n, lay, lay, E->raw_kind);
    if (sp.ok) {
        sc = std::make_unique<SpiralCache>();
        sc->sp = std::move(sp);
        DevPlan pl;
        std::memset(&pl, 0, sizeof pl);
        pl.n_merged = (int)sc->sp.merges.size();
        pl.n_raw = n_raw;
        pl.raw_kind = E->raw_kind;
        if (upload(sc->d_maps, sc->sp.maps, E->st) != cudaSuccess || upload(sc->d_items, sc->sp.merges, E->st) != cudaSuccess ||
            upload(sc->d_refs, sc->sp.refs, E->st) != cudaSuccess ||
            upload(sc->d_plan, std::vector<DevPlan>{pl}, E->st) != cudaSuccess)
            sc.reset();
        if (sc) sc->base = spiral_config(sc->sp.bits, false).split;
        for (int p = 0; sc && p <= SpiralCache::kFp32; ++p) {
            const bool fp32 = p == SpiralCache::kFp32;
            if (!fp32 && p < sc->base) continue;
            sc->cfg[p] = spiral_config(sc->sp.bits, fp32, fp32 ? 0 : p);
            if (sc->cfg[p].R == 0) continue;
            std::vector<SpiralWin> wins;
            std::vector<uint8_t> ij;
            spiral_windows(sc->sp, sc->cfg[p].R, sc->cfg[p].split, wins, ij, sc->cut[p].h);
            sc->nwins[p] = (int)wins.size();
            if (!fp32) sc->resident[p] = spiral_resident(sc->sp.bits, sc->cfg[p]);
            if (upload(sc->d_wins[p], wins, E->st) != cudaSuccess) sc.reset();
        }
    }
    SpiralCache *out = sc.get();
    E->spiral_plans.emplace(L, std::move(sc));
    return out;
}

// FP64 variant for nb pairs: the fewest microseconds per window over the waves of clusters
// that nb pairs take (16 CTAs per pair for the few pairs that a recontraction usually has).
int spiral_variant(const SpiralCache *sc, uint64_t nb, bool fp32) {
    if (fp32) return SpiralCache::kFp32;
    int best = sc->base;
    double best_us = 1e300;
    for (int p = sc->base; p < SpiralCache::kFp32; ++p) {
        if (sc->cfg[p].R == 0 || sc->cfg[p].split != p || sc->resident[p] <= 0) continue;
        const double us = std::ceil((double)nb / sc->resident[p]) * spiral_wave_us(sc->sp.bits, p);
        if (us < best_us) { best_us = us; best = p; }
    }
    return best;
}

struct SpiralJob {   // pairs of one depth L
    int L;
    const std::vector<uint64_t> *idx;
    SpiralCache *sc;
    int variant, n_raw, n_merged, n_maps;
    size_t scr, per_pair;         // amplitudes of global state and bytes per pair
    uint64_t pair0 = 0;           // a batch's first pair, raw gate, merged item, map and state of the buffers
    size_t raw0 = 0, merged0 = 0, map0 = 0, scr0 = 0;
};

// The batch [done, done + nb) of a job's pairs, from the host's descriptors to the traces, on `st`.
fp_status spiral_batch(fp_ensemble *E, const SpiralJob &j, uint64_t nb, bool fp32, double *tr, double *kappa, double *err,
                       cudaStream_t st) {
    const SpiralCache *sc = j.sc;
    const size_t celem = fp32 ? sizeof(float2) : sizeof(double2);
    const PairInfo *pairs = E->d_pairs.as<PairInfo>() + j.pair0;
    SampleParams smp;
    smp.seed = E->d.seed;
    smp.n = E->d.n;
    smp.raw_kind = E->raw_kind;
    smp.self_pair = (E->d.flags & FP_FLAG_SELF_PAIR) ? 1 : 0;
    const double err_scale = FP_ERR_SAFETY * (fp32 ? 0x1.0p-24 : 0x1.0p-53) * std::sqrt((double)j.n_maps);
    {
        KTimer t(E, FP_K_SAMPLE);
        CK(launch_sample(smp, pairs, (int)nb, j.n_raw, E->d_raw.as<double2>(), st));
        CK(t.stop((double)nb));
    }
    {
        KTimer t(E, FP_K_MERGE);
        CK(launch_merge(pairs, (int)nb, j.n_merged, sc->d_plan.as<DevPlan>(), sc->d_items.as<MergeItem>(),
                        sc->d_refs.as<MergeRef>(), E->d_raw.as<double2>(), E->d_merged.as<double2>(), st));
        CK(t.stop((double)nb));
    }
    {
        KTimer t(E, FP_K_SPIRAL);
        const int p = j.variant;
        const SpiralConfig &cf = sc->cfg[p];
        const bool use_win = cf.R > 0;
        char *maps = E->d_maps.as<char>() + j.map0 * spiral_map_elems(fp32) * celem;
        CK(launch_spiral(pairs, (int)nb, sc->d_maps.as<SpiralMap>(), j.n_maps, sc->sp.bits, sc->sp.first_bit, cf,
                         use_win ? sc->d_wins[p].as<SpiralWin>() : nullptr, use_win ? sc->nwins[p] : 0, sc->cut[p],
                         E->d_merged.as<double2>(), maps, E->d_spiral_scratch.as<char>() + j.scr0 * celem, fp32,
                         err_scale, tr, kappa, err, st));
        CK(t.stop(4.0 * (double)j.n_maps * (double)((size_t)1 << sc->sp.bits) * (double)nb));
        if (E->timing) E->kst.launches[FP_K_SPIRAL] += 1;   // maps + sweep
    }
    return FP_OK;
}

// Spiral sweep for pairs of the depths in `by_depth` (FP_HEA_PAULI with CNOT walls):
// sampler, merged 1-qubit operators, maps, a CTA or cluster per pair.  Depths that fit the
// workspace budget together run side by side on a stream each, deepest first: the
// recontracted pairs of one depth alone leave most SMs idle (n = 50, L = 2..8: their FP64
// sweeps take 14.9 ms one after another, 5 side by side).  Otherwise (or to time the kernels) depth by depth, in sub-batches under the budget.
fp_status run_spiral(fp_ensemble *E, uint64_t first, const std::map<int, std::vector<uint64_t>> &by_depth, int prec,
                     double *tr, double *kappa, double *err, float *gpu_ms) {
    const fp_ensemble_desc &d = E->d;
    const bool fp32 = prec != FP_PREC_FP64;
    const size_t celem = fp32 ? sizeof(float2) : sizeof(double2);
    constexpr uint64_t kMaxBatch = 65535;   // the sampler and merge grids index pairs by grid.y
    std::vector<SpiralJob> jobs;
    size_t all = 0;
    bool together = !E->timing;
    for (auto it = by_depth.rbegin(); it != by_depth.rend(); ++it) {
        SpiralJob j;
        j.L = it->first;
        j.idx = &it->second;
        j.sc = E->spiral_plans[j.L].get();
        j.n_raw = 1 + d.n + j.L * d.n;
        j.n_merged = (int)j.sc->sp.merges.size();
        j.n_maps = (int)j.sc->sp.maps.size();
        j.scr = j.sc->cfg[fp32 ? SpiralCache::kFp32 : j.sc->base].scratch_elems;
        j.per_pair = (size_t)2 * j.n_raw * 16 * sizeof(double2) + (size_t)j.n_merged * 16 * sizeof(double2) +
                     (size_t)j.n_maps * spiral_map_elems(fp32) * celem + j.scr * celem;
        all += j.idx->size() * j.per_pair;
        together = together && j.idx->size() <= kMaxBatch;
        jobs.push_back(j);
    }
    together = together && jobs.size() > 1 && all <= E->ws_budget;
    // a launch set: one batch of one job, or every job's only batch
    std::vector<PairInfo> pinfo;
    auto place = [&](SpiralJob &j, uint64_t done, uint64_t nb, const SpiralJob *after, uint64_t nb_after) {
        if (after) {
            j.pair0 = after->pair0 + nb_after;
            j.raw0 = after->raw0 + nb_after * 2 * after->n_raw;
            j.merged0 = after->merged0 + nb_after * after->n_merged;
            j.map0 = after->map0 + nb_after * after->n_maps;
            j.scr0 = after->scr0 + nb_after * after->scr;
        }
        j.variant = spiral_variant(j.sc, nb, fp32);
        for (uint64_t i = 0; i < nb; ++i) {
            PairInfo pi;
            std::memset(&pi, 0, sizeof pi);
            pi.pair = first + (*j.idx)[done + i];
            pi.n_raw = j.n_raw;
            pi.raw_off = (int64_t)(j.raw0 + i * 2 * j.n_raw);
            pi.merged_off = (int64_t)(j.merged0 + i * j.n_merged);
            pi.out = (int64_t)(*j.idx)[done + i];
            pinfo.push_back(pi);
        }
    };
    auto reserve = [&](const SpiralJob &j, uint64_t nb) -> fp_status {   // up to the end of j's batch of nb
        CK(upload(E->d_pairs, pinfo, E->st));
        CK(E->d_raw.reserve((j.raw0 + nb * 2 * j.n_raw) * 16 * sizeof(double2)));
        CK(E->d_merged.reserve(std::max<size_t>(16, (j.merged0 + nb * j.n_merged) * 16 * sizeof(double2))));
        CK(E->d_maps.reserve((j.map0 + nb * j.n_maps) * spiral_map_elems(fp32) * celem));
        CK(E->d_spiral_scratch.reserve(std::max<size_t>(16, (j.scr0 + nb * j.scr) * celem)));
        return FP_OK;
    };
    auto finish = [&](uint64_t pairs) -> fp_status {
        CK(cudaEventRecord(E->ev1, E->st));
        CK(cudaEventSynchronize(E->ev1));
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, E->ev0, E->ev1));
        if (gpu_ms) *gpu_ms += ms;
        E->kst.pairs += pairs;
        return FP_OK;
    };
    if (together) {
        uint64_t total = 0;
        for (size_t k = 0; k < jobs.size(); ++k) {
            place(jobs[k], 0, jobs[k].idx->size(), k ? &jobs[k - 1] : nullptr, k ? jobs[k - 1].idx->size() : 0);
            total += jobs[k].idx->size();
        }
        fp_status s = reserve(jobs.back(), jobs.back().idx->size());
        if (s != FP_OK) return s;
        while (E->side.size() < std::min(jobs.size(), fp_ensemble::kSideStreams)) CK(add_side_stream(E->side));
        CK(cudaEventRecord(E->ev0, E->st));
        for (SideStream &x : E->side) CK(cudaStreamWaitEvent(x.st, E->ev0, 0));
        for (size_t k = 0; k < jobs.size() && s == FP_OK; ++k)
            s = spiral_batch(E, jobs[k], jobs[k].idx->size(), fp32, tr, kappa, err, E->side[k % E->side.size()].st);
        cudaError_t joined = cudaSuccess;   // (after a failed launch too: what runs still uses the buffers)
        for (SideStream &x : E->side) {
            cudaError_t e = cudaEventRecord(x.ev, x.st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(E->st, x.ev, 0);
            if (e != cudaSuccess) joined = e;
        }
        if (s != FP_OK || joined != cudaSuccess)
            for (SideStream &x : E->side) cudaStreamSynchronize(x.st);
        if (s != FP_OK) return s;
        CK(joined);
        return finish(total);
    }
    for (SpiralJob &j : jobs) {
        const uint64_t cap = std::max<uint64_t>(1, std::min<uint64_t>(kMaxBatch, E->ws_budget / j.per_pair));
        for (uint64_t done = 0; done < j.idx->size();) {
            const uint64_t nb = std::min<uint64_t>(cap, j.idx->size() - done);
            pinfo.clear();
            place(j, done, nb, nullptr, 0);
            fp_status s = reserve(j, nb);
            if (s != FP_OK) return s;
            CK(cudaEventRecord(E->ev0, E->st));
            s = spiral_batch(E, j, nb, fp32, tr, kappa, err, E->st);
            if (s != FP_OK) return s;
            s = finish(nb);
            if (s != FP_OK) return s;
            done += nb;
        }
    }
    return FP_OK;
}

// Route pairs first + idx[i] to the brickwork or generic path.
__global__ void mark_skipped_kernel(const uint64_t *slots, uint64_t n, double *tr, double *kappa, double *err) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t s = slots[i];
    tr[2 * s] = tr[2 * s + 1] = NAN;
    kappa[s] = NAN;
    err[s] = NAN;
}

// Qudit brickwork pairs of one depth l: sampler, maps, sweep and meet
// (kernels_qudit.cu), in sub-batches under the workspace budget.
fp_status run_qudit(fp_ensemble *E, uint64_t first, const std::vector<uint64_t> &idx, int l, int prec, double *tr,
                    double *kappa, double *err, float *gpu_ms) {
    const fp_ensemble_desc &d = E->d;
    const uint64_t count = idx.size();
    if (count == 0) return FP_OK;
    const bool fp32 = prec != FP_PREC_FP64;
    const BrickDev bd = make_brick_plan(d.n, l, 0, 0, 0, 0).dev;
    double S = 1;
    for (int i = 0; i < bd.N; ++i) S *= d.q;
    if (S > (double)(1u << FP_MAX_STATE_BITS))
        return fail(FP_ERR_INFEASIBLE, "qudit depth %d: boundary of %d^%d amplitudes exceeds 2^%d", l, d.q, bd.N,
                    FP_MAX_STATE_BITS);
    const int n_raw = (int)layout_brickwork(d.n, l).size();
    const size_t per_pair = qudit_workspace_per_pair(d.q, bd, fp32);
    const uint64_t cap = std::max<uint64_t>(1, std::min<uint64_t>(65535, E->ws_budget / per_pair));
    const double G = (double)std::max(bd.n_layers[0], bd.n_layers[1]) * bd.m;
    const double err_scale = FP_ERR_SAFETY * (fp32 ? 0x1.0p-24 : 0x1.0p-53) * std::sqrt(G);
    const double cmac_pair = (double)maps_per_pair(bd) * S * d.q * d.q;   // each map: S/q^2 groups of q^4
    for (uint64_t done = 0; done < count;) {
        const uint64_t nb = std::min<uint64_t>(cap, count - done);
        std::vector<PairInfo> pinfo(nb);
        for (uint64_t i = 0; i < nb; ++i) {
            std::memset(&pinfo[i], 0, sizeof(PairInfo));
            pinfo[i].pair = first + idx[done + i];
            pinfo[i].n_raw = n_raw;
            pinfo[i].out = (int64_t)idx[done + i];
        }
        CK(upload(E->d_pairs, pinfo, E->st));
        CK(E->d_states.reserve(nb * per_pair));
        CK(cudaEventRecord(E->ev0, E->st));
        {
            KTimer t(E, FP_K_BRICK);
            CK(launch_qudit(d.q, bd, d.seed, E->d_pairs.as<PairInfo>(), (int)nb,
                            (d.flags & FP_FLAG_SELF_PAIR) ? 1 : 0, fp32, E->d_states.p, err_scale, tr, kappa, err,
                            E->st));
            CK(t.stop(cmac_pair * (double)nb, 2));
        }
        CK(cudaEventRecord(E->ev1, E->st));
        CK(cudaEventSynchronize(E->ev1));
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, E->ev0, E->ev1));
        if (gpu_ms) *gpu_ms += ms;
        E->kst.pairs += nb;
        done += nb;
    }
    return FP_OK;
}

fp_status route(fp_ensemble *E, uint64_t first, const std::vector<uint64_t> &idx, const std::vector<int> &depth,
                int prec, double *tr, double *kappa, double *err, float *gpu_ms) {
    const fp_ensemble_desc &d = E->d;
    if (d.q > 2) {   // qudit brickwork: its own sweep, per depth
        std::map<int, std::vector<uint64_t>> qd;
        for (uint64_t i : idx) qd[depth[i]].push_back(i);
        for (auto it = qd.rbegin(); it != qd.rend(); ++it) {
            fp_status s = run_qudit(E, first, it->second, it->first, prec, tr, kappa, err, gpu_ms);
            if (s != FP_OK) return s;
        }
        return FP_OK;
    }
    const bool brick = (d.kind == FP_PARALLEL || d.kind == FP_HEA) && !(d.flags & FP_FLAG_GENERIC_ONLY);
    const bool spiral = d.kind == FP_HEA_PAULI && !(d.flags & (FP_FLAG_GENERIC_ONLY | FP_FLAG_HEA_CZ));
    const bool skip = (d.flags & FP_FLAG_SKIP_INFEASIBLE) != 0;
    std::map<int, std::vector<uint64_t>> by_depth, spiral_depth;
    std::vector<uint64_t> generic;
    for (uint64_t i : idx) {
        if (spiral && depth[i] >= 2 && spiral_plan(E, depth[i])) {
            spiral_depth[depth[i]].push_back(i);
            continue;
        }
        if (brick && depth[i] >= 2) {
            if (skip && 2 * (depth[i] - 1) > FP_MAX_STATE_BITS) {   // boundary of 2(l-1) segment bits
                E->skipped.push_back(i);
                continue;
            }
            by_depth[depth[i]].push_back(i);
        } else {
            generic.push_back(i);
        }
    }
    // deepest first: the largest working sets get the memory while it is free
    for (auto it = by_depth.rbegin(); it != by_depth.rend(); ++it) {
        fp_status s = run_brick(E, first, it->second, it->first, prec, tr, kappa, err, gpu_ms);
        if (s != FP_OK) return s;
    }
    if (!spiral_depth.empty()) {
        fp_status s = run_spiral(E, first, spiral_depth, prec, tr, kappa, err, gpu_ms);
        if (s != FP_OK) return s;
    }
    return run_generic(E, first, generic, depth, prec, tr, kappa, err, gpu_ms);
}

// Contract pairs [first, first+count) into device arrays E->d_tr / E->d_kappa
// / E->d_err (indices relative to `first`), groups into E->d_group.
fp_status trace_device(fp_ensemble *E, uint64_t first, uint64_t count, int prec, float *gpu_ms,
                       uint64_t *requeued, double *max_kappa) {
    const fp_ensemble_desc &d = E->d;
    std::vector<int> depth(count), grp(count);
    for (uint64_t i = 0; i < count; ++i) {
        depth[i] = depth_of_pair(d, first + i);
        grp[i] = group_of_depth(d, depth[i]);
    }
    CK(E->d_tr.reserve(count * 2 * sizeof(double)));
    CK(E->d_kappa.reserve(count * sizeof(double)));
    CK(E->d_err.reserve(count * sizeof(double)));
    CK(E->d_group.reserve(count * sizeof(int32_t)));
    CK(E->d_ticket.reserve(sizeof(int) * 4));
    CK(cudaMemcpyAsync(E->d_group.p, grp.data(), count * sizeof(int32_t), cudaMemcpyHostToDevice, E->st));
    if (gpu_ms) *gpu_ms = 0;
    std::vector<uint64_t> all(count);
    std::iota(all.begin(), all.end(), 0);
    double *tr = E->d_tr.as<double>(), *kap = E->d_kappa.as<double>(), *err = E->d_err.as<double>();
    E->skipped.clear();
    fp_status s = route(E, first, all, depth, prec, tr, kap, err, gpu_ms);
    if (s != FP_OK) return s;
    std::vector<char> skipped(count, 0);
    if (!E->skipped.empty()) {
        // uncontracted pairs: NaN results, group -1 (left out of every moment)
        for (uint64_t i : E->skipped) {
            skipped[i] = 1;
            grp[i] = -1;
        }
        CK(cudaMemcpyAsync(E->d_group.p, grp.data(), count * sizeof(int32_t), cudaMemcpyHostToDevice, E->st));
        CK(upload(E->d_skip, E->skipped, E->st));
        mark_skipped_kernel<<<(unsigned)((E->skipped.size() + 255) / 256), 256, 0, E->st>>>(
            E->d_skip.as<uint64_t>(), E->skipped.size(), tr, kap, err);
        CK(cudaGetLastError());
    }
    const bool policy = prec == FP_PREC_FP32 || prec == FP_PREC_TF32X3;   // FP64 recontraction of flagged pairs
    if (policy || max_kappa) {
        std::vector<double> k(count), e(count);
        CK(cudaMemcpyAsync(k.data(), kap, count * sizeof(double), cudaMemcpyDeviceToHost, E->st));
        CK(cudaMemcpyAsync(e.data(), err, count * sizeof(double), cudaMemcpyDeviceToHost, E->st));
        CK(cudaStreamSynchronize(E->st));
        const double tol = d.fp32_tol > 0 ? d.fp32_tol : 1e-4;
        std::vector<uint64_t> redo;
        for (uint64_t i = 0; i < count; ++i) {
            if (max_kappa && std::isfinite(k[i])) *max_kappa = std::max(*max_kappa, k[i]);
            const bool over = !(e[i] <= tol) || (d.kappa_max > 0 && !(k[i] <= d.kappa_max));
            if (policy && over && !skipped[i]) redo.push_back(i);
        }
        if (!redo.empty()) {
            if (requeued) *requeued += redo.size();
            s = route(E, first, redo, depth, FP_PREC_FP64, tr, kap, err, gpu_ms);
            if (s != FP_OK) return s;
        }
    }
    return FP_OK;
}

}  // namespace

namespace fpk {
fp_status api_fail(fp_status s, const char *msg) { return fail(s, "%s", msg); }
fp_ensemble_desc ens_desc(const fp_ensemble *E) { return E->d; }
cudaStream_t ens_stream(const fp_ensemble *E) { return E->st; }
fp_status cv_trace(fp_ensemble *E, uint64_t first, uint64_t count, double **tr_dev, float *gpu_ms) {
    fp_status s = trace_device(E, first, count, FP_PREC_FP32, gpu_ms, nullptr, nullptr);
    if (s != FP_OK) return s;
    *tr_dev = E->d_tr.as<double>();
    return FP_OK;
}
}  // namespace fpk

namespace {

fp_status copy_out(fp_ensemble *E, void *dst, const void *src, size_t bytes) {
    if (!dst) return FP_OK;
    cudaMemcpyKind k = is_device_ptr(dst) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    CK(cudaMemcpyAsync(dst, src, bytes, k, E->st));
    return FP_OK;
}

}  // namespace

extern "C" {

const char *fp_last_error(void) { return g_err.c_str(); }

fp_status fp_ensemble_create(const fp_ensemble_desc *desc, void *cuda_stream, fp_ensemble **out) {
    if (!desc || !out) return fail(FP_ERR_ARG, "null argument");
    *out = nullptr;
    const fp_ensemble_desc &d = *desc;
    if (d.kind < FP_PARALLEL || d.kind > FP_HEA_PAULI) return fail(FP_ERR_ARG, "unknown ensemble kind %d", d.kind);
    if (d.n < 2 || d.n > 64) return fail(FP_ERR_ARG, "n = %d outside [2, 64]", d.n);
    if (d.kind == FP_LOCAL) {
        if (d.T_min < 1 || d.T_max < d.T_min || d.T_step < 1)
            return fail(FP_ERR_ARG, "bad local-circuit gate counts [%d, %d] step %d", d.T_min, d.T_max, d.T_step);
    } else if (d.depth_min < 1 || d.depth_max < d.depth_min) {
        return fail(FP_ERR_ARG, "bad depth range [%d, %d]", d.depth_min, d.depth_max);
    }
    if ((d.flags & FP_FLAG_DIAGONAL_GATES) && (d.kind == FP_HEA || d.kind == FP_HEA_PAULI))
        return fail(FP_ERR_ARG, "FP_FLAG_DIAGONAL_GATES applies to Haar-gate ensembles only");
    if ((d.flags & FP_FLAG_HEA_CZ) && d.kind != FP_HEA_PAULI)
        return fail(FP_ERR_ARG, "FP_FLAG_HEA_CZ applies to FP_HEA_PAULI only");
    if (d.q != 0 && d.q != 2 && !(d.kind == FP_PARALLEL && (d.q == 3 || d.q == 4)))
        return fail(FP_ERR_ARG, "local dimension q = %d: qudits (q = 3, 4) are supported for FP_PARALLEL only", d.q);
    if (d.q > 2 && (d.flags & (FP_FLAG_DIAGONAL_GATES | FP_FLAG_GENERIC_ONLY)))
        return fail(FP_ERR_ARG, "FP_FLAG_DIAGONAL_GATES and FP_FLAG_GENERIC_ONLY apply to qubits only");
    if (d.q > 2 && d.depth_min < 2)
        return fail(FP_ERR_ARG, "qudit brickwork needs depth >= 2 (at depth 1 the trace is the product of the gates' traces)");
    std::unique_ptr<fp_ensemble> E(new fp_ensemble());
    E->d = d;
    E->st = (cudaStream_t)cuda_stream;
    CK(cudaGetDevice(&E->device));
    CK(cudaDeviceGetAttribute(&E->sms, cudaDevAttrMultiProcessorCount, E->device));
    {
        cudaDeviceProp prop;
        CK(cudaGetDeviceProperties(&prop, E->device));
        E->gpu_name = prop.name;
    }
    E->raw_kind = d.kind == FP_HEA ? RAW_ROT2
                : d.kind == FP_HEA_PAULI ? RAW_PAULI
                : ((d.flags & FP_FLAG_DIAGONAL_GATES) ? RAW_DIAG4 : RAW_HAAR4);
    E->n_groups = d.kind == FP_LOCAL ? (d.T_max - d.T_min) / d.T_step + 1 : d.depth_max - d.depth_min + 1;
    size_t freeb = 0, totb = 0;
    CK(cudaMemGetInfo(&freeb, &totb));
    // default: 32 GB (room for as many 2^24-amplitude generic-sweep slots as 16-CTA
    // clusters can be resident), at most half the free memory
    size_t cap = d.workspace_bytes ? (size_t)d.workspace_bytes : ((size_t)32 << 30);
    E->ws_budget = std::min(cap, freeb / 2);
    CK(cudaEventCreate(&E->ev0));
    CK(cudaEventCreate(&E->ev1));
    E->timing = (d.flags & FP_FLAG_TIMING) != 0;
    CK(cudaStreamCreateWithFlags(&E->gst, cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&E->gev[0], cudaEventDisableTiming));
    CK(cudaEventCreateWithFlags(&E->gev[1], cudaEventDisableTiming));
    for (int k = 0; k < 2 * FP_K_CLASSES; ++k) CK(cudaEventCreate(&E->kev[k]));
    *out = E.release();
    return FP_OK;
}

void fp_ensemble_destroy(fp_ensemble *ens) {
    if (!ens) return;
    if (ens->st) cudaStreamSynchronize(ens->st);
    else cudaDeviceSynchronize();
    if (ens->ev0) cudaEventDestroy(ens->ev0);
    if (ens->ev1) cudaEventDestroy(ens->ev1);
    for (int k = 0; k < 2 * FP_K_CLASSES; ++k)
        if (ens->kev[k]) cudaEventDestroy(ens->kev[k]);
    if (ens->gst) cudaStreamSynchronize(ens->gst);
    for (auto &kv : ens->graphs) if (kv.second) cudaGraphExecDestroy(kv.second);
    for (int k = 0; k < 2; ++k) if (ens->gev[k]) cudaEventDestroy(ens->gev[k]);
    if (ens->gst) cudaStreamDestroy(ens->gst);
    for (SideStream &x : ens->side) {
        if (x.ev) cudaEventDestroy(x.ev);
        cudaStreamDestroy(x.st);
    }
    delete ens;
}

fp_status fp_groups(const fp_ensemble *ens, int32_t *n_groups, int32_t *values) {
    if (!ens || !n_groups) return fail(FP_ERR_ARG, "null argument");
    *n_groups = ens->n_groups;
    if (values)
        for (int g = 0; g < ens->n_groups; ++g)
            values[g] = ens->d.kind == FP_LOCAL ? ens->d.T_min + g * ens->d.T_step : ens->d.depth_min + g;
    return FP_OK;
}

fp_status fp_pair_groups(const fp_ensemble *ens, uint64_t first, uint64_t count, int32_t *group) {
    if (!ens || (!group && count)) return fail(FP_ERR_ARG, "null argument");
    for (uint64_t i = 0; i < count; ++i) group[i] = group_of_depth(ens->d, depth_of_pair(ens->d, first + i));
    return FP_OK;
}

fp_status fp_export_gates(fp_ensemble *ens, uint64_t pair, int32_t which, void *host_buf, size_t *bytes) {
    if (!ens || !bytes || (which != 0 && which != 1)) return fail(FP_ERR_ARG, "bad argument");
    const fp_ensemble_desc &d = ens->d;
    if (d.q > 2) return fail(FP_ERR_ARG, "gates of qudit ensembles are not exported (records hold 4x4 matrices)");
    int depth = depth_of_pair(d, pair);
    int n_raw = 0;
    std::vector<GateSlot> lay = circuit_layout(d, pair, which, depth, &n_raw);
    struct Rec { int32_t kind, q; double m[32]; };
    size_t need = lay.size() * sizeof(Rec);
    if (!host_buf) { *bytes = need; return FP_OK; }
    if (*bytes < need) { *bytes = need; return fail(FP_ERR_ARG, "buffer too small: need %zu bytes", need); }
    *bytes = need;
    PairInfo pi;
    pi.pair = pair; pi.plan = 0; pi.n_raw = n_raw; pi.raw_off = 0; pi.merged_off = 0; pi.table_off = 0;
    CK(upload(ens->d_pairs, std::vector<PairInfo>{pi}, ens->st));
    CK(ens->d_raw.reserve((size_t)2 * n_raw * 16 * sizeof(double2)));
    SampleParams sp;
    sp.seed = d.seed; sp.n = d.n; sp.raw_kind = ens->raw_kind; sp.self_pair = (d.flags & FP_FLAG_SELF_PAIR) ? 1 : 0;
    CK(launch_sample(sp, ens->d_pairs.as<PairInfo>(), 1, n_raw, ens->d_raw.as<double2>(), ens->st));
    std::vector<double2> raw((size_t)2 * n_raw * 16);
    CK(cudaMemcpyAsync(raw.data(), ens->d_raw.p, raw.size() * sizeof(double2), cudaMemcpyDeviceToHost, ens->st));
    CK(cudaStreamSynchronize(ens->st));
    Rec *out = (Rec *)host_buf;
    for (size_t i = 0; i < lay.size(); ++i) {
        std::memset(&out[i], 0, sizeof(Rec));
        out[i].q = lay[i].q;
        if (lay[i].kind == 2) {
            out[i].kind = 2;
            double dg[4] = {1, 1, 1, -1};
            for (int k = 0; k < 4; ++k) out[i].m[2 * k] = dg[k];
            continue;
        }
        out[i].kind = lay[i].kind == 3 ? 1 : lay[i].kind;
        const double2 *g = &raw[((size_t)which * n_raw + lay[i].raw) * 16];
        for (int k = 0; k < 16; ++k) { out[i].m[2 * k] = g[k].x; out[i].m[2 * k + 1] = g[k].y; }
    }
    return FP_OK;
}

fp_status fp_trace_batch(fp_ensemble *ens, uint64_t first, uint64_t count, int32_t prec, double *tr,
                         double *kappa, double *err, int32_t *group) {
    if (!ens || (!tr && count)) return fail(FP_ERR_ARG, "null argument");
    if (prec < FP_PREC_FP64 || prec > FP_PREC_TF32X3) return fail(FP_ERR_ARG, "unknown precision %d", prec);
    if (count == 0) return FP_OK;
    fp_status s = trace_device(ens, first, count, prec, nullptr, nullptr, nullptr);
    if (s != FP_OK) return s;
    if ((s = copy_out(ens, tr, ens->d_tr.p, count * 2 * sizeof(double))) != FP_OK) return s;
    if ((s = copy_out(ens, kappa, ens->d_kappa.p, count * sizeof(double))) != FP_OK) return s;
    if ((s = copy_out(ens, err, ens->d_err.p, count * sizeof(double))) != FP_OK) return s;
    if ((s = copy_out(ens, group, ens->d_group.p, count * sizeof(int32_t))) != FP_OK) return s;
    CK(cudaStreamSynchronize(ens->st));
    return FP_OK;
}

fp_status fp_reduce_moments(fp_ensemble *ens, const double *tr, const int32_t *group, uint64_t count,
                            int32_t k_max, double *moments) {
    if (!ens || !tr || !moments) return fail(FP_ERR_ARG, "null argument");
    if (k_max < 1 || k_max > FP_MAX_KMAX) return fail(FP_ERR_ARG, "k_max = %d outside [1, %d]", k_max, FP_MAX_KMAX);
    if (!is_device_ptr(tr) || (group && !is_device_ptr(group)))
        return fail(FP_ERR_ARG, "tr and group must be device pointers");
    int ng = group ? ens->n_groups : 1, nb = moments_blocks(count), nv = 2 * k_max + 1;
    CK(ens->d_partials.reserve((size_t)nb * ng * nv * sizeof(double)));
    CK(ens->d_moments.reserve((size_t)ng * nv * sizeof(double)));
    {
        KTimer t(ens, FP_K_MOMENTS);
        CK(launch_moments(tr, group, count, k_max, ng, ens->d_partials.as<double>(), nb, ens->d_moments.as<double>(), ens->st));
        CK(t.stop((double)count));
    }
    fp_status s = copy_out(ens, moments, ens->d_moments.p, (size_t)ng * nv * sizeof(double));
    if (s != FP_OK) return s;
    CK(cudaStreamSynchronize(ens->st));
    return FP_OK;
}

fp_status fp_bootstrap(fp_ensemble *ens, const double *tr, const int32_t *group, uint64_t count, int32_t k_max,
                       int32_t n_resamples, uint64_t seed, double *F_boot) {
    if (!ens || !tr || !group || !F_boot) return fail(FP_ERR_ARG, "null argument");
    if (k_max < 1 || k_max > FP_MAX_KMAX) return fail(FP_ERR_ARG, "k_max = %d outside [1, %d]", k_max, FP_MAX_KMAX);
    if (n_resamples < 1) return fail(FP_ERR_ARG, "n_resamples = %d must be positive", n_resamples);
    if (count >= (1ull << 32)) return fail(FP_ERR_ARG, "count must be below 2^32");
    const int ng = ens->n_groups;
    const double *dtr = tr;
    if (!is_device_ptr(tr)) {
        CK(ens->d_boot_tr.reserve(std::max<uint64_t>(count, 1) * 2 * sizeof(double)));
        if (count) CK(cudaMemcpyAsync(ens->d_boot_tr.p, tr, count * 2 * sizeof(double), cudaMemcpyHostToDevice, ens->st));
        dtr = ens->d_boot_tr.as<double>();
    }
    const int32_t *dgroup = group;
    if (!is_device_ptr(group)) {
        CK(ens->d_boot_group.reserve(std::max<uint64_t>(count, 1) * sizeof(int32_t)));
        if (count) CK(cudaMemcpyAsync(ens->d_boot_group.p, group, count * sizeof(int32_t), cudaMemcpyHostToDevice, ens->st));
        dgroup = ens->d_boot_group.as<int32_t>();
    }
    CK(ens->d_boot_xs.reserve(bootstrap_scratch(count, ng, k_max, n_resamples)));
    const size_t nout = (size_t)ng * k_max * n_resamples;
    CK(ens->d_boot_out.reserve(nout * sizeof(double)));
    {
        KTimer t(ens, FP_K_BOOTSTRAP);
        CK(launch_bootstrap(dtr, dgroup, count, ng, k_max, n_resamples, seed, ens->d_boot_xs.p,
                            ens->d_boot_out.as<double>(), ens->st));
        CK(t.stop((double)count * n_resamples));
    }
    fp_status s = copy_out(ens, F_boot, ens->d_boot_out.p, nout * sizeof(double));
    if (s != FP_OK) return s;
    CK(cudaStreamSynchronize(ens->st));
    return FP_OK;
}

fp_status fp_frame_potential_resume(fp_ensemble *ens, fp_checkpoint *ck, uint64_t max_pairs, uint64_t max_batches,
                                    int32_t k_max, double target_rel_stderr, int32_t prec, double *F,
                                    double *stderr_) {
    if (!ens || !ck || !ck->sums || !F || !stderr_) return fail(FP_ERR_ARG, "null argument");
    if (k_max < 1 || k_max > FP_MAX_KMAX) return fail(FP_ERR_ARG, "k_max = %d outside [1, %d]", k_max, FP_MAX_KMAX);
    if (prec < FP_PREC_FP64 || prec > FP_PREC_TF32X3) return fail(FP_ERR_ARG, "unknown precision %d", prec);
    const int ng = ens->n_groups, nv = 2 * k_max + 1;
    if (ck->next_batch == 0) {   // first call of a run
        ck->k_max = k_max;
        ck->n_groups = ng;
        ck->pairs_done = 0;
        std::memset(&ck->stats, 0, sizeof ck->stats);
        // with a target: batches from 4096 pairs, doubling, so the stop can come early;
        // without one: batches as large as the workspace allows
        ck->next_batch = target_rel_stderr > 0 ? 4096 : (1u << 20);
    } else if (ck->k_max != k_max || ck->n_groups != ng) {
        return fail(FP_ERR_ARG, "checkpoint of k_max = %d, %d groups resumed with k_max = %d, %d groups", ck->k_max,
                    ck->n_groups, k_max, ng);
    }
    double *acc = ck->sums, *comp = ck->sums + (size_t)ng * nv;
    std::vector<double> part((size_t)ng * nv);
    fp_run_stats &st = ck->stats;
    st.n_groups = ng;
    const int kt = k_max >= 2 ? 2 : 1;
    auto estimate = [&]() {   // F, stderr from the sums; whether every group met the target
        bool ok = target_rel_stderr > 0;
        for (int g = 0; g < ng; ++g) {
            double N = acc[g * nv] + comp[g * nv];
            for (int k = 1; k <= k_max; ++k) {
                double S = acc[g * nv + k] + comp[g * nv + k];
                double Q = acc[g * nv + k_max + k] + comp[g * nv + k_max + k];
                double mean = N > 0 ? S / N : NAN;
                double var = N > 1 ? std::max(0.0, (Q - S * S / N) / (N - 1)) : NAN;
                F[g * k_max + k - 1] = mean;
                stderr_[g * k_max + k - 1] = N > 1 ? std::sqrt(var / N) : NAN;
            }
            double f = F[g * k_max + kt - 1], e = stderr_[g * k_max + kt - 1];
            if (!(N > 1 && f > 0 && e / f <= target_rel_stderr)) ok = false;
        }
        return ok;
    };
    bool reached = ck->pairs_done > 0 && estimate();
    for (uint64_t nbatches = 0; ck->pairs_done < max_pairs && !reached && (max_batches == 0 || nbatches < max_batches);
         ++nbatches) {
        if (ens->cancel.exchange(0)) {
            estimate();
            return fail(FP_ERR_CANCELLED, "cancelled before the batch at pair %llu (the checkpoint can be resumed)",
                        (unsigned long long)ck->next_pair);
        }
        uint64_t nb = std::min<uint64_t>(ck->next_batch, max_pairs - ck->pairs_done);
        float ms = 0;
        uint64_t recon = 0;
        double mk = 0;
        fp_status s = trace_device(ens, ck->next_pair, nb, prec, &ms, &recon, &mk);
        if (s != FP_OK) return s;
        int nb_blocks = moments_blocks(nb);
        CK(ens->d_partials.reserve((size_t)nb_blocks * ng * nv * sizeof(double)));
        CK(ens->d_moments.reserve((size_t)ng * nv * sizeof(double)));
        {
            KTimer t(ens, FP_K_MOMENTS);
            CK(launch_moments(ens->d_tr.as<double>(), ens->d_group.as<int32_t>(), nb, k_max, ng,
                              ens->d_partials.as<double>(), nb_blocks, ens->d_moments.as<double>(), ens->st));
            CK(t.stop((double)nb));
        }
        CK(cudaMemcpyAsync(part.data(), ens->d_moments.p, part.size() * sizeof(double), cudaMemcpyDeviceToHost, ens->st));
        CK(cudaStreamSynchronize(ens->st));
        // the batch is complete: fold it into the checkpoint
        for (size_t i = 0; i < part.size(); ++i) {   // Neumaier accumulation across batches
            double y = acc[i] + part[i];
            comp[i] += std::fabs(acc[i]) >= std::fabs(part[i]) ? (acc[i] - y) + part[i] : (part[i] - y) + acc[i];
            acc[i] = y;
        }
        st.fp64_recontracted += recon;
        st.max_kappa = std::max(st.max_kappa, mk);
        st.infeasible += ens->skipped.size();
        st.gpu_seconds += ms * 1e-3;
        ck->pairs_done += nb;
        ck->next_pair += nb;
        st.pairs = ck->pairs_done - st.infeasible;
        if (ck->next_batch < (1u << 20)) ck->next_batch *= 2;
        reached = estimate();
    }
    if (ck->pairs_done == 0) estimate();
    st.reached_target = reached ? 1 : 0;
    return FP_OK;
}

fp_status fp_frame_potential(fp_ensemble *ens, uint64_t first, uint64_t max_pairs, int32_t k_max,
                             double target_rel_stderr, int32_t prec, double *F, double *stderr_,
                             fp_run_stats *stats) {
    if (!ens || !F || !stderr_) return fail(FP_ERR_ARG, "null argument");
    if (k_max < 1 || k_max > FP_MAX_KMAX) return fail(FP_ERR_ARG, "k_max = %d outside [1, %d]", k_max, FP_MAX_KMAX);
    std::vector<double> sums((size_t)2 * ens->n_groups * (2 * k_max + 1), 0.0);
    fp_checkpoint ck;
    std::memset(&ck, 0, sizeof ck);
    ck.next_pair = first;
    ck.sums = sums.data();
    fp_status s = fp_frame_potential_resume(ens, &ck, max_pairs, 0, k_max, target_rel_stderr, prec, F, stderr_);
    if (s == FP_OK && stats) *stats = ck.stats;
    return s;
}

fp_status fp_cancel(fp_ensemble *ens) {
    if (!ens) return fail(FP_ERR_ARG, "null argument");
    ens->cancel.store(1);
    return FP_OK;
}

fp_status fp_inject_alloc_failures(int32_t count) {
    if (count < 0) return fail(FP_ERR_ARG, "count < 0");
    g_alloc_failures.store(count);
    return FP_OK;
}

fp_status fp_set_wait_limit_ns(uint64_t ns) {
    g_wait_ns.store(ns ? ns : 1000000000ull);
    return FP_OK;
}

fp_status fp_brick_variant(const fp_ensemble *ens, int32_t depth, int32_t precision, int32_t *out) {
    if (!ens || !out) return fail(FP_ERR_ARG, "null argument");
    if (precision < FP_PREC_FP64 || precision > FP_PREC_TF32X3) return fail(FP_ERR_ARG, "unknown precision %d", precision);
    auto it = ens->brick_plans.find(brick_key(depth, precision));
    if (it == ens->brick_plans.end())
        return fail(FP_ERR_ARG, "no brickwork sweep of depth %d at this precision has run on this ensemble", depth);
    for (int i = 0; i < 4; ++i) out[i] = it->second->variant[i];
    return FP_OK;
}

fp_status fp_kernel_stats_get(fp_ensemble *ens, fp_kernel_stats *out, int32_t reset) {
    if (!ens || !out) return fail(FP_ERR_ARG, "null argument");
    *out = ens->kst;
    out->graph_replays = ens->graph_replays;
    if (reset) {
        std::memset(&ens->kst, 0, sizeof ens->kst);
        ens->graph_replays = 0;
    }
    return FP_OK;
}

}  // extern "C"
