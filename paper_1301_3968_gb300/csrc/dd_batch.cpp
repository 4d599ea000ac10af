// Many beams in one dedispersion launch, its CUDA graph, and the schedule autotuner.
//
// A batch holds one plan per beam (uneven trial counts, DM ranges and lengths).  Its
// work list has one item per CTA tile of every beam -- (beam, trial block, time tile) --
// and the launch one CTA per item, in list order: beams by decreasing cost (the small
// ones fill the last wave), each beam's tiles in the plain launch's grouped order.  The
// graph captures the launch and, when bound, every beam's channel statistics and boxcar
// S/N, so one graph launch processes a block of all beams.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <new>
#include <sstream>
#include <string>

#include "dd_internal.h"
#include "dd_trace.h"

struct dd_batch_s {
    std::vector<dd_plan_s*> plans;    // the caller's
    // per beam the plan whose schedule the launch takes: the caller's, or the batch's own of it
    // (twin, of the profiles and schedule twin_id)
    std::vector<dd_plan_s*> sched, twin;
    std::vector<uint64_t> twin_id;
    bool u8 = false, pair = true;
    bool rl = false;         // run-length beams (per-channel prefix sums, then differences)
    bool short_taps = true;  // every plan's tap runs fit one register window (run-length
                             // beams: every plan shares difference rows in the CTA)
    std::vector<uint32_t*> d_prefix;  // beams that read prefix sums: theirs (else null)
    std::vector<int64_t> ldp;
    std::vector<dd::BatchItem> items;
    // one launch per kernel: row kernels with 16 and 8 warps per CTA, then the tap kernels
    struct Group {
        int warps;  // of the row kernel; 0: tap kernel
        size_t first, count, smem;
    };
    std::vector<Group> groups;
    std::vector<uint64_t> gen;         // the uploads that the bound arguments point into
    int grid = 0;
    int device = -1;
    int64_t units = 0;  // sum over beams of trials x outputs
    dd::DedispArgs* d_args = nullptr;
    dd::BatchItem* d_items = nullptr;
    bool bound = false;
    // per-beam buffers bound for the boxcar stage of the graph
    std::vector<const void*> in;
    std::vector<int64_t> in_ld;
    std::vector<void*> out;
    std::vector<int64_t> out_ld;
    std::vector<int32_t> widths;
    std::vector<double*> mean, sd;
    std::vector<float*> peak;
    std::vector<int32_t*> arg;
    bool box_bound = false;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

namespace {

int64_t plan_t_out(const dd_plan_s* p) { return p->band.nsamp - p->dmax; }

void free_batch_dev(dd_batch_s* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (uint32_t* q : b->d_prefix) cudaFree(q);
    b->d_prefix.clear();
    b->ldp.clear();
    cudaFree(b->d_args);
    cudaFree(b->d_items);
    b->exec = nullptr;
    b->graph = nullptr;
    b->d_args = nullptr;
    b->d_items = nullptr;
}

// Work list: one item per CTA tile, with the tile's FMA count (run-length beams: its
// trial-channel pairs, each costing the same per output whatever its taps) plus a fixed
// per-stage cost as the estimate; sorted largest first.
// The work list: beams in decreasing order of estimated cost (so that the small ones fill
// the last wave), and within a beam the plain launch's tile order: trial blocks taken
// kGroupBlocks at a time, blocks fastest within a group and then time tiles, so that the
// CTAs working together share the beam's input columns and stage records in L2.
void build_items(dd_batch_s* b) {
    constexpr int kGroupBlocks = 16;
    struct Beam {
        int warps;  // of the beam's row kernel, or 0
        double cost;
        int beam;
    };
    std::vector<Beam> order;
    b->units = 0;
    for (int beam = 0; beam < (int)b->plans.size(); ++beam) {
        const dd_plan_s* p = b->sched[beam];
        const int64_t t_out = plan_t_out(p);
        const int nst = (p->nchan + p->cs - 1) / p->cs;
        const int64_t tile = dd::plan_tile_t(p);
        const int64_t ntile = (t_out + tile - 1) / tile;
        double taps = 0;
        for (int64_t i = 0; i < (int64_t)p->ndm * p->nchan; ++i) taps += p->rl || p->rk ? 1.0 : p->taps[(size_t)i];
        b->units += (int64_t)p->ndm * t_out;
        order.push_back({p->rk ? p->row_warps : 0, taps * (double)t_out + 2.0e4 * nst * ntile * p->nblk, beam});
    }
    std::stable_sort(order.begin(), order.end(), [](const Beam& x, const Beam& y) {
        return x.warps != y.warps ? x.warps > y.warps : x.cost > y.cost;
    });
    b->items.clear();
    b->groups.clear();
    for (const Beam& bm : order) {
        const dd_plan_s* p = b->sched[bm.beam];
        const int64_t t_out = plan_t_out(p);
        const int64_t tile = dd::plan_tile_t(p);
        if (b->groups.empty() || b->groups.back().warps != bm.warps)
            b->groups.push_back({bm.warps, b->items.size(), 0, 0});
        const int ntile = (int)((t_out + tile - 1) / tile);
        for (int g0 = 0; g0 < p->nblk; g0 += kGroupBlocks)
            for (int tx = 0; tx < ntile; ++tx)
                for (int blk = g0; blk < std::min(p->nblk, g0 + kGroupBlocks); ++blk) {
                    dd::BatchItem it;
                    it.beam = bm.beam;
                    it.blk = blk;
                    it.tx = tx;
                    it.pad = 0;
                    b->items.push_back(it);
                }
        // shared memory: the most that any beam of the launch needs
        dd_batch_s::Group& g = b->groups.back();
        g.count = b->items.size() - g.first;
        g.smem = std::max(g.smem, dd::dedisp_smem_for(p));
    }
}

// The schedules of the launch.  Beams of one wave each have stages for an SM of their own; where
// their CTAs together are more than the SMs, two should fit (6 beams of some 110 trials x 336
// channels x 7400 outputs, block with statistics and boxcar: 945 us, with two 827).  Those are
// twins, which the batch keeps: the plans stay as they are.
void choose_schedules(dd_batch_s* b) {
    auto small = [](const dd_plan_s* p) { return p->rk && p->row_warps == dd::kWarps && p->own_schedule; };
    int64_t ctas = 0;
    for (const dd_plan_s* p : b->plans)
        if (p->rk && p->row_warps == dd::kWarps)
            ctas += (plan_t_out(p) + dd::plan_tile_t(p) - 1) / dd::plan_tile_t(p) * p->nblk;
    for (size_t i = 0; i < b->plans.size(); ++i) {
        dd_plan_s* p = b->plans[i];
        const bool want = ctas > 152 && small(p);
        if (b->twin_id[i] != p->sched_id || !want) {
            if (b->twin[i]) dd::destroy_plan(b->twin[i]);
            b->twin[i] = want ? dd::twin_of(p, dd::Twin::kSharesSm) : nullptr;
            b->twin_id[i] = want ? p->sched_id : 0;
        }
        b->sched[i] = b->twin[i] ? b->twin[i] : p;
    }
}

// The row kernels' kind for the batch's beams.
int row_kind(const dd_batch_s* b) { return b->pair ? dd::kRowsFir : dd::kRowsPk; }

bool aligned16(const void* ptr) { return ((uintptr_t)ptr & 15u) == 0; }

}  // namespace

extern "C" {

dd_status dd_batch_create(dd_batch_t* out, const dd_plan_t* plans, int32_t nbeams) {
    if (!out || !plans || nbeams < 1) return DD_ERR_ARG;
    *out = nullptr;
    for (int i = 0; i < nbeams; ++i) {
        if (!plans[i]) return DD_ERR_ARG;
        if (plans[i]->band.in_type != plans[0]->band.in_type || plans[i]->pair != plans[0]->pair)
            return DD_ERR_ARG;
        if (plan_t_out(plans[i]) < 1) return DD_ERR_ARG;
        // one kernel serves the batch: every beam on the same tap-sum path
        if (plans[i]->rl != plans[0]->rl || plans[i]->rl_b != plans[0]->rl_b) return DD_ERR_UNSUPPORTED;
        if (plans[i]->rl && plans[i]->band.nsamp > ((int64_t)1 << 24)) return DD_ERR_UNSUPPORTED;
    }
    dd_batch_s* b = new (std::nothrow) dd_batch_s;
    if (!b) return DD_ERR_OOM;
    b->plans.assign(plans, plans + nbeams);
    b->u8 = plans[0]->band.in_type == DD_U8;
    b->pair = plans[0]->pair;
    b->rl = plans[0]->rl;
    b->sched = b->plans;
    b->twin.assign(nbeams, nullptr);
    b->twin_id.assign(nbeams, 0);
    choose_schedules(b);
    build_items(b);
    *out = b;
    return DD_OK;
}

dd_status dd_batch_bind(dd_batch_t b, const void* const* d_in, const int64_t* in_ld,
                        void* const* d_out, const int64_t* out_ld) {
    if (!b || !d_in || !in_ld || !d_out || !out_ld) return DD_ERR_ARG;
    const int nb = (int)b->plans.size();
    std::vector<dd::DedispArgs> args(nb);
    for (int i = 0; i < nb; ++i) {
        dd_plan_s* p = b->plans[i];
        if (p->rl != b->rl || p->pair != b->pair || (b->rl && p->rl_b != b->plans[0]->rl_b))
            return DD_ERR_UNSUPPORTED;  // a plan changed path since dd_batch_create
        const int64_t esz = p->band.in_type == DD_U8 ? 1 : 4;
        const int64_t t_out = plan_t_out(p);
        if (!d_in[i] || !d_out[i] || !aligned16(d_in[i]) || (in_ld[i] * esz) % 16 != 0 ||
            in_ld[i] < p->band.nsamp || out_ld[i] < t_out)
            return DD_ERR_ARG;
        dd_status st = dd::upload_tables(p);
        if (st != DD_OK) return st;
    }
    // plans may have been retuned since dd_batch_create: schedules and work list again
    b->bound = false;
    free_batch_dev(b);
    choose_schedules(b);
    for (int i = 0; i < nb; ++i)
        if (b->twin[i]) {
            const dd_status st = dd::upload_tables(b->twin[i]);
            if (st != DD_OK) return st;
        }
    for (int i = 0; i < nb; ++i) {
        dd_plan_s* p = b->sched[i];
        // beams that read prefix sums have their own, which the batch owns
        const int64_t ldp = (p->band.nsamp + 1 + 3) & ~(int64_t)3;
        const size_t bytes = (size_t)ldp * p->nchan * sizeof(uint32_t);
        uint32_t* q = nullptr;
        if (dd::reads_prefix(p)) {
            const int64_t limit = b->plans[i]->scratch_limit;
            cudaError_t e = limit > 0 && (int64_t)bytes > limit ? cudaErrorMemoryAllocation : cudaMalloc((void**)&q, bytes);
            if (e == cudaErrorMemoryAllocation && !p->rl) {  // direct sums do without, tap by tap
                cudaGetLastError();
                q = nullptr;
                if (b->twin[i]) dd::destroy_plan(b->twin[i]);
                b->twin[i] = dd::twin_of(b->plans[i], dd::Twin::kTaps);
                b->twin_id[i] = 0;  // (chosen anew at the next bind)
                b->sched[i] = b->twin[i] ? b->twin[i] : b->plans[i];
                if (b->twin[i] && dd::upload_tables(b->twin[i]) == DD_OK) e = cudaSuccess;
            }
            if (e != cudaSuccess) {
                free_batch_dev(b);
                return dd::cuda_status(e);
            }
        }
        b->d_prefix.push_back(q);
        b->ldp.push_back(ldp);
        p = b->sched[i];
        dd::fill_dedisp_args(p, q ? q : d_in[i], q ? ldp : in_ld[i], 0, plan_t_out(p), d_out[i], out_ld[i], &args[i]);
    }
    build_items(b);
    int dev = -1, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return dd::cuda_status(e);
    b->short_taps = true;
    for (auto* p : b->sched)
        if (!p->rk) b->short_taps = b->short_taps && (p->rl ? p->rl_b : p->pair ? p->umax <= dd::kRPair : p->kmax <= dd::kRInt);
    int per_sm = 32;
    for (const auto& g : b->groups)
        per_sm = std::min(per_sm, g.warps ? dd::rows_batched_blocks_per_sm(row_kind(b), b->u8, g.warps, g.smem)
                                          : dd::dedisp_batched_blocks_per_sm(b->u8, b->pair, b->short_taps, g.smem, b->rl));
    if (per_sm < 1) return DD_ERR_UNSUPPORTED;
    if (b->items.size() >= (size_t)INT32_MAX) return DD_ERR_UNSUPPORTED;
    b->grid = (int)b->items.size();  // one CTA per work item
    b->device = dev;
    e = cudaMalloc((void**)&b->d_args, nb * sizeof(dd::DedispArgs));
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_items, b->items.size() * sizeof(dd::BatchItem));
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_args, args.data(), nb * sizeof(dd::DedispArgs), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_items, b->items.data(), b->items.size() * sizeof(dd::BatchItem),
                       cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        free_batch_dev(b);
        return dd::cuda_status(e);
    }
    b->in.assign(d_in, d_in + nb);
    b->in_ld.assign(in_ld, in_ld + nb);
    b->out.assign(d_out, d_out + nb);
    b->out_ld.assign(out_ld, out_ld + nb);
    size_t smem = 0;
    for (const auto& g : b->groups) smem = std::max(smem, g.smem);
    b->gen.clear();
    for (auto* p : b->plans) b->gen.push_back(p->dev_gen);
    b->bound = true;
    b->box_bound = false;
    dd::log_msg(1, "batch of %d beams (%s): %zu work items (one CTA each, %d resident per SM on %d SMs), "
             "%zu launches, up to %zu bytes of shared memory", nb, b->rl ? "run-length sums" : (b->pair ? "fp32 pair units" : "exact integer sums"),
             b->items.size(), per_sm, sms, b->groups.size(), smem);
    return DD_OK;
}

// Whether a bound plan's device tables have been replaced since (new profiles or weights).
static bool batch_stale(const dd_batch_s* b) {
    for (size_t i = 0; i < b->plans.size(); ++i)
        if (b->plans[i]->dev_dirty || b->plans[i]->dev_gen != b->gen[i]) return true;
    return false;
}

// Binds the same buffers again, keeping the boxcar stage's.
static dd_status batch_rebind(dd_batch_s* b) {
    const std::vector<const void*> in = b->in;
    const std::vector<int64_t> in_ld = b->in_ld, out_ld = b->out_ld;
    const std::vector<void*> out = b->out;
    const bool box = b->box_bound;
    for (auto* p : b->plans)
        if (plan_t_out(p) < 1) return DD_ERR_ARG;
    const dd_status st = dd_batch_bind(b, in.data(), in_ld.data(), out.data(), out_ld.data());
    if (st != DD_OK) return st;
    b->box_bound = box;
    return DD_OK;
}

dd_status dd_batch_dedisperse(dd_batch_t b, void* stream) {
    DD_TRACE("dd_batch_dedisperse");
    if (!b) return DD_ERR_ARG;
    if (!b->bound) return DD_ERR_STATE;
    if (batch_stale(b)) {
        const dd_status st = batch_rebind(b);
        if (st != DD_OK) return st;
    }
    for (size_t i = 0; i < b->plans.size(); ++i)  // the prefix sums of the beams that read them
        if (b->d_prefix[i]) {
            const dd_status st = dd::launch_prefix_into(b->sched[i], b->in[i], b->in_ld[i], 0,
                                                        b->sched[i]->band.nsamp, b->d_prefix[i], b->ldp[i],
                                                        (cudaStream_t)stream);
            if (st != DD_OK) return st;
        }
    for (const auto& g : b->groups) {
        const dd_status st =
            g.warps ? dd::launch_rows_batched(row_kind(b), b->u8, g.warps, b->d_args, b->d_items + g.first,
                                              (int32_t)g.count, g.smem, (cudaStream_t)stream)
                    : dd::launch_dedisperse_batched(b->u8, b->pair, b->short_taps, b->d_args, b->d_items + g.first,
                                                    (int32_t)g.count, g.smem, (cudaStream_t)stream, b->rl);
        if (st != DD_OK) return st;
    }
    return DD_OK;
}

dd_status dd_batch_bind_boxcar(dd_batch_t b, const int32_t* widths, int32_t nw, double* const* d_mean,
                               double* const* d_std, float* const* d_peak, int32_t* const* d_arg) {
    if (!b || !widths || nw < 1 || !d_mean || !d_std || !d_peak || !d_arg) return DD_ERR_ARG;
    if (!b->bound) return DD_ERR_STATE;
    const int nb = (int)b->plans.size();
    for (int i = 0; i < nb; ++i) {
        if (!d_mean[i] || !d_std[i] || !d_peak[i] || !d_arg[i]) return DD_ERR_ARG;
        if (widths[nw - 1] > plan_t_out(b->plans[i])) return DD_ERR_ARG;
    }
    for (int i = 1; i < nw; ++i)
        if (widths[i] <= widths[i - 1] || widths[0] < 1) return DD_ERR_ARG;
    b->widths.assign(widths, widths + nw);
    b->mean.assign(d_mean, d_mean + nb);
    b->sd.assign(d_std, d_std + nb);
    b->peak.assign(d_peak, d_peak + nb);
    b->arg.assign(d_arg, d_arg + nb);
    b->box_bound = true;
    return DD_OK;
}

// Runs one block of every beam: the batched dedispersion launch and, when bound,
// every beam's channel statistics and boxcar S/N.
static dd_status batch_run(dd_batch_s* b, cudaStream_t s) {
    dd_status st = dd_batch_dedisperse(b, s);
    if (st != DD_OK || !b->box_bound) return st;
    for (size_t i = 0; i < b->plans.size(); ++i) {
        dd_plan_s* p = b->plans[i];
        st = dd_channel_stats(p, b->in[i], b->in_ld[i], 0, p->band.nsamp, b->mean[i], b->sd[i], s);
        if (st != DD_OK) return st;
        st = dd_boxcar_snr(p, b->out[i], b->out_ld[i], plan_t_out(p), b->widths.data(),
                           (int32_t)b->widths.size(), b->mean[i], b->sd[i], b->peak[i], b->arg[i],
                           INFINITY, nullptr, 0, nullptr, s);
        if (st != DD_OK) return st;
    }
    return DD_OK;
}

dd_status dd_batch_run(dd_batch_t b, void* stream) {
    DD_TRACE("dd_batch_run");
    if (!b) return DD_ERR_ARG;
    if (!b->bound) return DD_ERR_STATE;
    return batch_run(b, (cudaStream_t)stream);
}

// Captures one block on `s` (every workspace exists) into the batch's graph.
static dd_status capture_run(dd_batch_s* b, cudaStream_t s) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return dd::cuda_status(e);
    const dd_status st = batch_run(b, s);
    cudaGraph_t g = nullptr;
    e = cudaStreamEndCapture(s, &g);
    if (st != DD_OK) {
        if (g) cudaGraphDestroy(g);
        return st;
    }
    if (e != cudaSuccess) return dd::cuda_status(e);
    b->graph = g;
    e = cudaGraphInstantiate(&b->exec, g, 0);
    return dd::cuda_status(e);
}

dd_status dd_batch_capture(dd_batch_t b, void* stream) {
    if (!b || !stream) return DD_ERR_ARG;
    if (!b->bound) return DD_ERR_STATE;
    cudaStream_t s = (cudaStream_t)stream;
    // one eager pass first: it creates every plan's workspace, which a capture may not
    dd_status st = batch_run(b, s);
    if (st != DD_OK) return st;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return dd::cuda_status(e);
    return capture_run(b, s);
}

dd_status dd_batch_replay(dd_batch_t b, void* stream) {
    DD_TRACE("dd_batch_replay");
    if (!b) return DD_ERR_ARG;
    if (!b->exec) return DD_ERR_STATE;
    if (batch_stale(b)) {
        // a plan's tables have moved: this block eagerly, and a new graph for the next
        dd_status st = batch_run(b, (cudaStream_t)stream);
        if (st != DD_OK) return st;
        cudaStream_t s = nullptr;
        const cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        if (e != cudaSuccess) return dd::cuda_status(e);
        st = capture_run(b, s);
        cudaStreamDestroy(s);
        return st;
    }
    return dd::cuda_status(cudaGraphLaunch(b->exec, (cudaStream_t)stream));
}

dd_status dd_batch_info(dd_batch_t b, int32_t* nitems, int32_t* grid, int64_t* units) {
    if (!b) return DD_ERR_ARG;
    if (nitems) *nitems = (int32_t)b->items.size();
    if (grid) *grid = b->grid;
    if (units) *units = b->units;
    return DD_OK;
}

dd_status dd_batch_destroy(dd_batch_t b) {
    if (!b) return DD_ERR_ARG;
    free_batch_dev(b);
    for (dd_plan_s* t : b->twin)
        if (t) dd::destroy_plan(t);
    delete b;
    return DD_OK;
}

}  // extern "C"
