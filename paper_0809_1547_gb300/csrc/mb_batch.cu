// C ABI of the batched ensemble: B realizations (ordinary contexts sharing
// the batch's stream) advanced together, either by one persistent launch per
// call or by their own launches on concurrent streams.
#include "mb_ctx.h"

#include <algorithm>
#include <cmath>
#include <map>
#include <string>
#include <tuple>
#include <vector>

struct mb_batch {
    std::vector<mb_ctx*> inst;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int sms = 0;
    // device copies of the instances' step arguments, probes and work lists
    mb::StepArgs* d_inst = nullptr;
    mb::DevPointProbes* d_probes = nullptr;
    int4* d_items1 = nullptr;
    int4* d_items2 = nullptr;
    int* d_tiles = nullptr;
    unsigned* d_bar = nullptr;
    unsigned long long* d_tick = nullptr;
    int* d_err = nullptr;
    long long* d_ctr = nullptr;
    // the copy of its state that each instance's device arguments point at
    // (its own single-pass or small-grid steps change copies)
    std::vector<const float*> at;
    int n1 = 0, n2 = 0;
    dim3 block{32, 4, 1};
    int kz = 16;
    int blocks = 0;
    bool dirty = true;
    cudaGraphExec_t graph_chunk = nullptr;
    int graph_steps = 32;
    bool graph_ok = true;
    int64_t n = 0;
    // MB_BATCH_CONCURRENT: instance q steps on lanes[q % lanes.size()] (its
    // own stream pointed there for the call); fork_ev / lane_ev join the
    // lanes to the batch's stream
    int mode = MB_BATCH_PERSISTENT;
    std::vector<cudaStream_t> lanes;
    std::vector<cudaEvent_t> lane_ev;
    cudaEvent_t fork_ev = nullptr;
    std::string err;
};

namespace {

int bfail(mb_batch* b, int code, const std::string& msg) {
    if (b) b->err = msg;
    mb::set_thread_error(msg);
    return code;
}

#define MB_BCUDA(b, call)                                                                  \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess)                                                             \
            return bfail((b), e_ == cudaErrorMemoryAllocation ? MB_ERR_OOM : MB_ERR_CUDA, \
                         std::string(#call) + ": " + cudaGetErrorString(e_));              \
    } while (0)

void free_arrays(mb_batch* b) {
    void* bufs[] = {b->d_inst, b->d_probes, b->d_items1, b->d_items2, b->d_tiles};
    for (void* p : bufs)
        if (p) cudaFree(p);
    b->d_inst = nullptr;
    b->d_probes = nullptr;
    b->d_items1 = b->d_items2 = nullptr;
    b->d_tiles = nullptr;
    if (b->graph_chunk) cudaGraphExecDestroy(b->graph_chunk);
    b->graph_chunk = nullptr;
}

mb::BatchArgs batch_args(mb_batch* b, int nsteps) {
    mb::BatchArgs a{};
    a.inst = b->d_inst;
    a.probes = b->d_probes;
    a.ninst = (int)b->inst.size();
    a.items1 = b->d_items1;
    a.n1 = b->n1;
    a.items2 = b->d_items2;
    a.n2 = b->n2;
    a.tiles = b->d_tiles;
    a.kz = b->kz;
    a.gq = (int)(b->block.x * b->block.y) * mb::kBatchGainPerThread;
    a.bar = b->d_bar;
    a.tick = b->d_tick;
    a.err = b->d_err;
    a.ctr = b->d_ctr;
    a.nsteps = nsteps;
    a.dt = b->inst[0]->dt;
    return a;
}

// Device copies of the instances' arguments and the two work lists.
int rebuild(mb_batch* b) {
    free_arrays(b);
    const int B = (int)b->inst.size();
    std::vector<mb::StepArgs> args;
    std::vector<mb::DevPointProbes> probes;
    std::vector<int> tiles;
    std::vector<int4> items1, items2;
    b->at.clear();
    const int threads = (int)(b->block.x * b->block.y);
    const int gq = threads * mb::kBatchGainPerThread;
    for (int q = 0; q < B; ++q) {
        mb_ctx* c = b->inst[q];
        if (!c->have_material) return bfail(b, MB_ERR_STATE, "batch member without material");
        if (c->face.on || !c->planes.empty())
            return bfail(b, MB_ERR_STATE, "face and plane probes are not advanced inside a batch");
        args.push_back(c->args);
        b->at.push_back(c->args.f.ex);
        probes.push_back({(int)c->probes.size(), c->probe_nfreq, c->d_probe_cell, c->d_probe_omega,
                          c->d_probe_acc});
        const int gx = (c->nx + b->block.x - 1) / b->block.x;
        const int gy = (c->ny + b->block.y - 1) / b->block.y;
        const int gz = (c->nz + b->kz - 1) / b->kz;
        tiles.push_back(gx);
        tiles.push_back(gy);
        const long long nH = (long long)gx * gy * gz;
        // a gain item takes kBatchGainSub consecutive blocks of gq list entries
        const long long gi = (long long)gq * mb::kBatchGainSub;
        const long long nG = (c->args.gain.on && c->glist_count) ? (c->glist_count + gi - 1) / gi : 0;
        // H tiles and gain chunks interleaved by progress through the
        // instance (a gain chunk re-reads E^n where the H tiles next to it in
        // the list read it, so the line is still in L2); E tiles in tile order
        // (neighbouring tiles share halo lines).
        for (long long t = 0; t < nH + nG; ++t) {
            const long long g0 = t * nG / (nH + nG), g1 = (t + 1) * nG / (nH + nG);
            if (g1 > g0) items1.push_back(make_int4(q, 1, (int)g0, 0));
            else items1.push_back(make_int4(q, 0, (int)(t - g0), 0));
        }
        for (long long t = 0; t < nH; ++t) items2.push_back(make_int4(q, 2, (int)t, 0));
    }
    MB_BCUDA(b, cudaMalloc((void**)&b->d_inst, sizeof(mb::StepArgs) * B));
    MB_BCUDA(b, cudaMalloc((void**)&b->d_probes, sizeof(mb::DevPointProbes) * B));
    MB_BCUDA(b, cudaMalloc((void**)&b->d_tiles, sizeof(int) * tiles.size()));
    MB_BCUDA(b, cudaMalloc((void**)&b->d_items1, sizeof(int4) * items1.size()));
    MB_BCUDA(b, cudaMalloc((void**)&b->d_items2, sizeof(int4) * items2.size()));
    MB_BCUDA(b, cudaMemcpyAsync(b->d_inst, args.data(), sizeof(mb::StepArgs) * B, cudaMemcpyHostToDevice, b->stream));
    MB_BCUDA(b, cudaMemcpyAsync(b->d_probes, probes.data(), sizeof(mb::DevPointProbes) * B, cudaMemcpyHostToDevice, b->stream));
    MB_BCUDA(b, cudaMemcpyAsync(b->d_tiles, tiles.data(), sizeof(int) * tiles.size(), cudaMemcpyHostToDevice, b->stream));
    MB_BCUDA(b, cudaMemcpyAsync(b->d_items1, items1.data(), sizeof(int4) * items1.size(), cudaMemcpyHostToDevice, b->stream));
    MB_BCUDA(b, cudaMemcpyAsync(b->d_items2, items2.data(), sizeof(int4) * items2.size(), cudaMemcpyHostToDevice, b->stream));
    MB_BCUDA(b, cudaStreamSynchronize(b->stream));
    b->n1 = (int)items1.size();
    b->n2 = (int)items2.size();
    const int per_sm = mb::batch_blocks_per_sm(b->block);
    if (per_sm < 1) return bfail(b, MB_ERR_CUDA, "persistent kernel does not fit on an SM with this block");
    b->blocks = per_sm * b->sms;
    b->dirty = false;
    return MB_OK;
}

// Streams of the concurrent mode (created on first use).
constexpr int kLanes = 8;

int ensure_lanes(mb_batch* b) {
    if (!b->lanes.empty()) return MB_OK;
    MB_BCUDA(b, cudaEventCreateWithFlags(&b->fork_ev, cudaEventDisableTiming));
    for (int l = 0; l < kLanes; ++l) {
        cudaStream_t st = nullptr;
        cudaEvent_t ev = nullptr;
        MB_BCUDA(b, cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
        b->lanes.push_back(st);
        MB_BCUDA(b, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        b->lane_ev.push_back(ev);
    }
    return MB_OK;
}

// n steps of every instance by its own launches (as mb_step), the instances
// spread over the lanes; the lanes start after the work already queued on
// the batch's stream and the batch's stream waits for all of them (the
// probes an instance leaves on its second stream included).
int step_concurrent(mb_batch* b, int n) {
    if (int rc = ensure_lanes(b)) return rc;
    const int L = (int)b->lanes.size();
    MB_BCUDA(b, cudaEventRecord(b->fork_ev, b->stream));
    for (cudaStream_t st : b->lanes) MB_BCUDA(b, cudaStreamWaitEvent(st, b->fork_ev, 0));
    int rc = MB_OK;
    for (size_t q = 0; q < b->inst.size() && rc == MB_OK; ++q) {
        mb_ctx* c = b->inst[q];
        c->stream = b->lanes[q % L];
        rc = mb_step(c, n);
        if (rc == MB_OK) mb::join_probes(c);
        c->stream = b->stream;
        if (rc) rc = bfail(b, rc, mb_last_error(c));
    }
    for (int l = 0; l < L; ++l) {
        cudaEventRecord(b->lane_ev[l], b->lanes[l]);
        cudaStreamWaitEvent(b->stream, b->lane_ev[l], 0);
    }
    if (rc) return rc;
    MB_BCUDA(b, cudaGetLastError());
    return MB_OK;
}

int check_lockstep(mb_batch* b) {
    for (mb_ctx* c : b->inst)
        if (c->n != b->n)
            return bfail(b, MB_ERR_STATE, "an instance was stepped outside the batch");
    return MB_OK;
}

int launch_steps(mb_batch* b, int nsteps) {
    const mb::BatchArgs a = batch_args(b, nsteps);
    cudaError_t e = mb::launch_batch(a, b->block, b->blocks, b->stream);
    if (e != cudaSuccess) return bfail(b, MB_ERR_CUDA, std::string("batch launch: ") + cudaGetErrorString(e));
    return MB_OK;
}

}  // namespace

extern "C" {

int mb_batch_create(mb_batch** out, int B, const int* grids, double dx, double dt, const mb_params* p,
                    void* cuda_stream) {
    if (!out || !grids || B < 1) return bfail(nullptr, MB_ERR_ARG, "bad batch arguments");
    *out = nullptr;
    mb_batch* b = new mb_batch();
    auto bail = [&](int rc) {
        mb_batch_destroy(b);
        return rc;
    };
    if (cuda_stream) {
        b->stream = (cudaStream_t)cuda_stream;
    } else {
        cudaError_t e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) return bail(bfail(nullptr, MB_ERR_CUDA, cudaGetErrorString(e)));
        b->own_stream = true;
    }
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev);
    for (int q = 0; q < B; ++q) {
        mb_ctx* c = nullptr;
        int rc = mb_create(&c, grids + 3 * q, dx, dt, p, b->stream);
        if (rc) return bail(rc);
        // a launch of many steps that a lone context of this grid was tuned to
        // fills the GPU by itself: not beside other members untried
        if (c->tune_f.variant == mb::kVariantSmall) c->use_fused = false;
        b->inst.push_back(c);
    }
    int64_t largest = 0;
    for (mb_ctx* c : b->inst) largest = std::max(largest, c->ncell);
    if (largest < mb::kSmallPassCells) b->kz = mb::kSmallPassPlanes;
    cudaError_t e = cudaMalloc((void**)&b->d_bar, sizeof(unsigned) * 2);
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_err, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_tick, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemset(b->d_tick, 0, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_ctr, sizeof(long long));
    if (e == cudaSuccess) e = cudaMemset(b->d_bar, 0, sizeof(unsigned) * 2);
    if (e == cudaSuccess) e = cudaMemset(b->d_err, 0, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(b->d_ctr, 0, sizeof(long long));
    if (e != cudaSuccess) return bail(bfail(nullptr, MB_ERR_OOM, cudaGetErrorString(e)));
    *out = b;
    return MB_OK;
}

int mb_batch_destroy(mb_batch* b) {
    if (!b) return MB_OK;
    if (b->stream) cudaStreamSynchronize(b->stream);
    for (cudaStream_t st : b->lanes) {
        cudaStreamSynchronize(st);
        cudaStreamDestroy(st);
    }
    for (cudaEvent_t ev : b->lane_ev) cudaEventDestroy(ev);
    if (b->fork_ev) cudaEventDestroy(b->fork_ev);
    free_arrays(b);
    for (mb_ctx* c : b->inst) mb_destroy(c);
    void* bufs[] = {b->d_bar, b->d_err, b->d_ctr, b->d_tick};
    for (void* p : bufs)
        if (p) cudaFree(p);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
    return MB_OK;
}

int mb_batch_set_instance(mb_batch* b, int q, const float* eps_map, const uint8_t* gain_mask, double N_a,
                          double pump, uint64_t seed) {
    if (!b || q < 0 || q >= (int)b->inst.size()) return bfail(b, MB_ERR_ARG, "bad instance index");
    int rc = mb_set_material(b->inst[q], eps_map, gain_mask, N_a, pump);
    if (rc) return bfail(b, rc, mb_last_error(b->inst[q]));
    rc = mb_set_seed(b->inst[q], seed);
    if (rc) return bfail(b, rc, mb_last_error(b->inst[q]));
    b->dirty = true;
    return MB_OK;
}

int mb_batch_instance(mb_batch* b, int q, mb_ctx** ctx) {
    if (!b || !ctx || q < 0 || q >= (int)b->inst.size()) return bfail(b, MB_ERR_ARG, "bad instance index");
    *ctx = b->inst[q];
    b->dirty = true;   // the caller may add probes or a source
    return MB_OK;
}

int mb_batch_step(mb_batch* b, int n) {
    if (!b || n < 0) return bfail(b, MB_ERR_ARG, "bad batch step arguments");
    if (n == 0) return MB_OK;
    if (int rc = check_lockstep(b)) return rc;
    if (b->mode == MB_BATCH_PERSISTENT && !b->dirty)
        for (size_t q = 0; q < b->inst.size(); ++q) b->dirty = b->dirty || b->at[q] != b->inst[q]->args.f.ex;
    if (b->dirty)
        if (int rc = rebuild(b)) return rc;
    if (b->mode == MB_BATCH_CONCURRENT) {
        const int rc = step_concurrent(b, n);   // advances each instance's count
        if (rc == MB_OK) b->n += n;
        return rc;
    }
    // the batch counter follows the instances' own step count
    const long long n0 = (long long)b->n;
    MB_BCUDA(b, cudaMemcpyAsync(b->d_ctr, &n0, sizeof(long long), cudaMemcpyHostToDevice, b->stream));
    int left = n;
    if (b->graph_ok && left >= b->graph_steps) {
        if (!b->graph_chunk) {
            cudaGraph_t g = nullptr;
            bool ok = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
            if (ok) {
                const mb::BatchArgs a = batch_args(b, b->graph_steps);
                cudaError_t le = mb::launch_batch(a, b->block, b->blocks, b->stream);
                cudaError_t ce = cudaStreamEndCapture(b->stream, &g);
                ok = le == cudaSuccess && ce == cudaSuccess &&
                     cudaGraphInstantiate(&b->graph_chunk, g, 0) == cudaSuccess;
                if (g) cudaGraphDestroy(g);
            }
            if (!ok) {   // cooperative launches not capturable here: launch directly
                cudaGetLastError();
                b->graph_ok = false;
                b->graph_chunk = nullptr;
            }
        }
        while (b->graph_chunk && left >= b->graph_steps) {
            MB_BCUDA(b, cudaGraphLaunch(b->graph_chunk, b->stream));
            left -= b->graph_steps;
        }
    }
    if (left > 0)
        if (int rc = launch_steps(b, left)) return rc;
    b->n += n;
    for (mb_ctx* c : b->inst) {
        c->n += n;
        c->launches += 1;
    }
    return MB_OK;
}

int mb_batch_synchronize(mb_batch* b) {
    if (!b) return bfail(nullptr, MB_ERR_ARG, "null batch");
    MB_BCUDA(b, cudaStreamSynchronize(b->stream));
    for (mb_ctx* c : b->inst)   // bounded waits of the instances' own launches
        if (int rc = mbi::check_device_error(c)) return bfail(b, rc, mb_last_error(c));
    int e = 0;
    MB_BCUDA(b, cudaMemcpy(&e, b->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (e) {
        cudaMemset(b->d_err, 0, sizeof(int));
        cudaMemset(b->d_bar, 0, sizeof(unsigned) * 2);
        cudaMemset(b->d_tick, 0, sizeof(unsigned long long));
        return bfail(b, MB_ERR_TIMEOUT, "a grid barrier of the batched launch gave up");
    }
    return MB_OK;
}

int mb_batch_autotune(mb_batch* b) {
    if (!b) return bfail(nullptr, MB_ERR_ARG, "null batch");
    if (int rc = check_lockstep(b)) return rc;
    MB_BCUDA(b, cudaStreamSynchronize(b->stream));
    size_t total = 0;
    for (mb_ctx* c : b->inst) total += mb::state_device_bytes(c);
    char* backup = nullptr;
    MB_BCUDA(b, cudaMalloc((void**)&backup, total));
    {
        char* o = backup;
        for (mb_ctx* c : b->inst) {
            mb::state_snapshot(c, o);
            o += mb::state_device_bytes(c);
        }
    }
    struct Cand { dim3 block; int kz; };
    const Cand cands[] = {{dim3(32, 4, 1), 16}, {dim3(32, 4, 1), 8}, {dim3(32, 8, 1), 8},
                          {dim3(64, 2, 1), 16}, {dim3(32, 2, 1), 16}, {dim3(64, 4, 1), 8},
                          {dim3(32, 8, 1), 16}, {dim3(32, 4, 1), 32}, {dim3(64, 4, 1), 16}};
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    Cand pick{b->block, b->kz};
    const long long n0 = (long long)b->n;
    for (const Cand& cd : cands) {
        b->block = cd.block;
        b->kz = cd.kz;
        if (rebuild(b)) continue;
        cudaMemcpyAsync(b->d_ctr, &n0, sizeof(long long), cudaMemcpyHostToDevice, b->stream);
        if (launch_steps(b, 1)) continue;
        cudaEventRecord(e0, b->stream);
        if (launch_steps(b, 2)) continue;
        cudaEventRecord(e1, b->stream);
        cudaEventSynchronize(e1);
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) {
            best = ms;
            pick = cd;
        }
    }
    auto restore_all = [&]() {
        const char* o = backup;
        for (mb_ctx* c : b->inst) {
            mb::state_restore(c, o);
            o += mb::state_device_bytes(c);
        }
    };
    b->block = pick.block;
    b->kz = pick.kz;
    // The instances' own launch shapes (tuned once per grid shape and CPML
    // depth in the process), then each mode from the same state: a warm-up
    // of 2 steps (graph captures) and the timed steps; even counts, so a
    // single-pass instance ends in the copy it started from.
    int rc = MB_OK;
    {
        std::map<std::tuple<int, int, int, int>, mb_ctx*> tuned;   // one trial set per grid shape and row length
        for (mb_ctx* c : b->inst) {
            if (rc) break;
            auto it = tuned.find({c->nx, c->ny, c->nz, c->px});
            if (it == tuned.end()) {
                if ((rc = mb_autotune(c))) rc = bfail(b, rc, mb_last_error(c));
                tuned[{c->nx, c->ny, c->nz, c->px}] = c;
            } else {
                const mb_ctx* t = it->second;
                c->tune_h = t->tune_h;
                c->tune_e = t->tune_e;
                c->tune_f = t->tune_f;
                c->use_fused = t->use_fused;
                c->fused_ratio = t->fused_ratio;
                mbi::drop_graphs(c);
            }
        }
    }
    std::vector<int64_t> n_keep, l_keep;
    for (mb_ctx* c : b->inst) {
        n_keep.push_back(c->n);
        l_keep.push_back(c->launches);
    }
    // ms of a call of n steps of the members' own launches, after one untimed
    auto concurrent_ms = [&](int n) -> float {
        float ms = 1e30f;
        restore_all();
        if (step_concurrent(b, n) == MB_OK && cudaEventRecord(e0, b->stream) == cudaSuccess &&
            step_concurrent(b, n) == MB_OK && cudaEventRecord(e1, b->stream) == cudaSuccess &&
            cudaEventSynchronize(e1) == cudaSuccess)
            cudaEventElapsedTime(&ms, e0, e1);
        return ms;
    };
    // Members tuned (alone) to many steps a launch: such a launch holds most of
    // the GPU's shared memory, so that two members' launches run one after the
    // other, where their two passes run beside each other (sides 48, 52 and 60:
    // 26.7 us a step against 22.4; 24, 28 and 30: 4.7 against 10.1).  Both are
    // timed with all members running, in calls of 4 and of 32 steps; the launch
    // stays where a step of it is the shorter, for calls long enough to repay
    // the members' loading and storing of their states.
    std::vector<mb_ctx*> many;
    for (mb_ctx* c : b->inst)
        if (rc == MB_OK && c->use_fused && c->tune_f.variant == mb::kVariantSmall) many.push_back(c);
    bool kept = false;
    if (!many.empty()) {
        float t[2][2];   // [launch of many steps][calls of 4, of 32 steps]
        for (int on = 1; on >= 0; --on) {
            for (mb_ctx* c : many) {
                c->use_fused = on != 0;
                mbi::drop_graphs(c);
            }
            for (int q = 0; q < 2; ++q) t[on][q] = std::min(concurrent_ms(q ? 32 : 4), concurrent_ms(q ? 32 : 4));
        }
        const float step1 = (t[1][1] - t[1][0]) / 28.0f, step0 = (t[0][1] - t[0][0]) / 28.0f;
        if (step1 < 0.97f * step0) {
            const float fixed = (t[1][0] - 4.0f * step1) - (t[0][0] - 4.0f * step0);
            const int least = (int)std::ceil(std::max(fixed, 0.0f) / (step0 - step1));
            kept = least <= mb::kSmallMaxSteps;
            for (mb_ctx* c : many) {
                c->use_fused = kept;
                c->tune_f.kz = std::max(c->tune_f.kz, std::max(least, 1));
                mbi::drop_graphs(c);
            }
        }
    }
    // Members tuned (alone) to the two passes by a little: beside others, whose
    // launches fill the gaps of either, the single-pass step's fewer bytes count
    // (sides 97, 126 and 148, four of each: 26.1 ms with the smallest on two
    // passes, 24.1 without; alone both take 27.5 us).
    std::vector<mb_ctx*> close;
    for (mb_ctx* c : b->inst)
        if (rc == MB_OK && !c->use_fused && c->tune_f.variant == mb::kVariantTma && c->fused_ratio < 1.1f &&
            mb::fused_supported(c->args))
            close.push_back(c);
    if (!close.empty() && b->inst.size() > 1) {
        float t[2];
        for (int on = 1; on >= 0; --on) {
            for (mb_ctx* c : close) {
                c->use_fused = on != 0;
                mbi::drop_graphs(c);
            }
            t[on] = concurrent_ms(4);
        }
        if (t[1] < t[0])
            for (mb_ctx* c : close) {
                c->use_fused = true;
                mbi::drop_graphs(c);
            }
    }
    // each mode over calls of 4 steps, of 32 where the members take the launch
    // of many (a few microseconds a step)
    const int n_mode = kept ? 32 : 4;
    float t_mode[2] = {1e30f, 1e30f};
    for (int m = 0; m < 2 && rc == MB_OK; ++m) {
        restore_all();
        bool ok;
        if (m == MB_BATCH_PERSISTENT) {
            ok = rebuild(b) == MB_OK &&
                 cudaMemcpyAsync(b->d_ctr, &n0, sizeof(long long), cudaMemcpyHostToDevice, b->stream) ==
                     cudaSuccess &&
                 launch_steps(b, 2) == MB_OK && cudaEventRecord(e0, b->stream) == cudaSuccess &&
                 launch_steps(b, n_mode) == MB_OK;
        } else {
            ok = step_concurrent(b, 2) == MB_OK && cudaEventRecord(e0, b->stream) == cudaSuccess &&
                 step_concurrent(b, n_mode) == MB_OK;
        }
        if (ok && cudaEventRecord(e1, b->stream) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess)
            cudaEventElapsedTime(&t_mode[m], e0, e1);
    }
    for (size_t q = 0; q < b->inst.size(); ++q) {
        b->inst[q]->n = n_keep[q];
        b->inst[q]->launches = l_keep[q];
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    restore_all();
    cudaStreamSynchronize(b->stream);
    cudaFree(backup);
    if (rc) return rc;
    b->mode = t_mode[MB_BATCH_CONCURRENT] < t_mode[MB_BATCH_PERSISTENT] ? MB_BATCH_CONCURRENT
                                                                         : MB_BATCH_PERSISTENT;
    b->dirty = true;
    MB_BCUDA(b, cudaGetLastError());
    return MB_OK;
}

int mb_batch_set_mode(mb_batch* b, int mode) {
    if (!b) return bfail(nullptr, MB_ERR_ARG, "null batch");
    if (mode != MB_BATCH_PERSISTENT && mode != MB_BATCH_CONCURRENT)
        return bfail(b, MB_ERR_ARG, "mode must be MB_BATCH_PERSISTENT or MB_BATCH_CONCURRENT");
    b->mode = mode;
    return MB_OK;
}

int mb_batch_get_mode(mb_batch* b, int* mode) {
    if (!b || !mode) return bfail(b, MB_ERR_ARG, "null argument");
    *mode = b->mode;
    return MB_OK;
}

int mb_selftest_bounded_waits(int which, int limit, int* gave_up) {
    if ((which != 0 && which != 1) || limit < 1 || limit > mb::kBarrierSpinLimit || !gave_up)
        return bfail(nullptr, MB_ERR_ARG, "which must be 0 or 1, 1 <= limit <= 2^22, gave_up non-null");
    unsigned* bar = nullptr;
    int* d = nullptr;
    int blocks = 1;
    cudaError_t e = cudaMalloc((void**)&bar, sizeof(unsigned) * 2);
    if (e == cudaSuccess) e = cudaMalloc((void**)&d, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(bar, 0, sizeof(unsigned) * 2);
    if (e == cudaSuccess) e = cudaMemset(d, 0, sizeof(int));
    if (e == cudaSuccess) {
        if (which == 0) {
            int dev = 0, sms = 1;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            blocks = std::min(sms, 8);
            e = mb::launch_selftest_barrier(bar, blocks, limit, d, nullptr);
        } else {
            e = mb::launch_selftest_mbarrier(limit, d, nullptr);
        }
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    int n = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&n, d, sizeof(int), cudaMemcpyDeviceToHost);
    if (bar) cudaFree(bar);
    if (d) cudaFree(d);
    if (e != cudaSuccess) return bfail(nullptr, MB_ERR_CUDA, cudaGetErrorString(e));
    *gave_up = n;
    return MB_OK;
}

int mb_batch_get_tuning(mb_batch* b, int* out3) {
    if (!b || !out3) return bfail(b, MB_ERR_ARG, "null argument");
    out3[0] = (int)b->block.x;
    out3[1] = (int)b->block.y;
    out3[2] = b->kz;
    return MB_OK;
}

}  // extern "C"
