// Several scatterers marched together (the uneven batch).  Two forms, chosen at creation:
//
//  * Persistent (every member FP32, one incident wave, direct solve: the uneven-batch workload):
//    ONE cooperative kernel runs the phases of up to B_STEPS steps of every member -- where a chunk
//    starts, the envelopes, tests and pre-sums of its steps; the history rows inside the chunk and the
//    T_0^-1 rows of every step; where a chunk or the call ends, the post-processing of its steps
//    together -- with grid-wide barriers in between.  The units of a phase (rows, edges, triangles of all members) are dealt to the warps in
//    turn, so that every member spreads over the whole grid; no unit waits for a counter.  The
//    arithmetic is that of the per-handle step (simt.h), so every member's currents equal those of
//    tdcfie_step bit for bit.  Units per turn, warps per block and blocks per SM come from a
//    measuring autotuner (tdcfie_batch_tune).
//  * Graph branches (any other mix of precisions, waves or solvers): one CUDA graph holds one step
//    of every handle, each on its own forked stream.
// Either way a single launch advances all members; the handles keep their own blocks,
// rings and step counters.  Every grid-wide wait is bounded (%globaltimer, 2 s) and reports
// TDCFIE_E_TIMEOUT.
#include <algorithm>
#include <string>
#include <vector>

#include "internal.h"
#include "plan.h"
#include "simt.h"

using namespace tdc;

namespace tdc {

enum { PH_ENV = 0, PH_GATHER, PH_PRE, PH_HIST, PH_SOLVE, PH_PIN, PH_PINV, PH_POUT, NPH };
constexpr int64_t B_STEPS = 32;      // steps per kernel

struct BArgs {
    const SimtDev<float>* mem;
    int nmem;
    const int* first[NPH];   // first unit of every member in a phase, [nmem + 1]
    unsigned long long* sync;      // arrivals so far, timeout flag
};

// units of a phase for one member (one warp works on a unit)
static int phase_units(const StepPlan* p, int ph) {
    const auto up = [](int64_t a, int b) { return (int)((a + b - 1) / b); };
    switch (ph) {
        case PH_ENV: return up((int64_t)p->npts * p->C, 32);
        case PH_GATHER: return p->ne;
        case PH_PRE: return up(p->ne, pre_rows<float>()) * p->ngroups * up(p->C, PRE_COLS);
        // post-processing: all columns of a chunk
        case PH_PIN: return up(p->nc, 32) * p->C;
        case PH_PINV: return up(p->nc, pre_rows<float>()) * up(p->C, PRE_COLS);
        case PH_POUT: return up(p->ne, 32) * p->C;
        // rows of the history, of every lag that may be pushed, and of the solve
        case PH_HIST: return up(p->ne, step_rows<1>()) * (1 + std::max(0, std::min(p->C - 1, p->K - 1) - 1));
        default: return p->ne;
    }
}

// u: the unit; t: steps since the kernel's first (the step counters stay until its end), left: steps from
// this one on; np: steps to post-process, the last of them this one
__device__ __forceinline__ void batch_unit(int ph, const SimtDev<float>& d, int t, int left, int np, int u, int lane) {
    const Ctl* c = d.ctl;
    StepPos pos{c->n + t, (c->slot + t) % d.ring, (c->col + t) % d.C};
    const Cols cs = ph <= PH_PRE ? new_cols(d.ctl, d.C, pos.n, pos.col, left) : Cols{};
    if (ph == PH_ENV) {
        const int idx = 32 * u + lane, nc = cs.hi - cs.lo;
        if (idx < d.npts * nc) {
            const int i = cs.lo + idx % nc, pt = idx / nc;
            d.env[pt * d.C + i] = env_point<float>(d.exc, pos.n - pos.col + i, d.dt, d.pts[3 * pt], d.pts[3 * pt + 1], d.pts[3 * pt + 2]);
        }
    } else if (ph == PH_GATHER) {
        gather_edge<float>(d, cs, u, 0, lane);
    } else if (ph == PH_PRE) {
        const int ctiles = (d.C + PRE_COLS - 1) / PRE_COLS, q = u % ctiles, g = u / ctiles % d.ngroups;
        pre_item<float>(d, cs, ring_at(pos.slot, -pos.col, d.ring), u / ctiles / d.ngroups * pre_rows<float>(), g, q, lane);
    } else if (ph == PH_HIST) {
        hist_unit<float, 1>(d, pos, u, lane, true, Nothing());
    } else if (ph == PH_SOLVE) {
        solve_unit<float, 1>(d, pos, u, lane, Nothing());
    } else if (ph == PH_PINV) {
        const int ctiles = (d.C + PRE_COLS - 1) / PRE_COLS, col0 = u % ctiles * PRE_COLS;
        if (col0 < np) pinv_item<float>(d, np, u / ctiles * pre_rows<float>(), col0, lane);
    } else {
        const int len = ph == PH_PIN ? d.nc : d.ne, per = (len + 31) / 32, q = u / per, i = (u - q * per) * 32 + lane;
        if (q >= np || i >= len) return;
        const int back = np - 1 - q, slot = ring_at(pos.slot, -back, d.ring);
        if (ph == PH_PIN) pin_value<float>(d, pos.n - back, slot, q, 0, i);
        else pout_value<float>(d, pos.n - back, slot, q, 0, i);
    }
}

// `steps` MOT steps of every member; rows: consecutive units per turn of a warp.  Launches and barriers
// bound it: five members of uneven size took 44 us a step with a kernel per step and the post-processing
// in each (six barriers), 28 us with two phases a step.
__global__ void __launch_bounds__(256) k_batch_step(const __grid_constant__ BArgs a, int rows, int steps) {
    extern __shared__ int2 mcol[];      // every member's column of the kernel's first step, and C (negative: its march's first chunk)
    __shared__ int failed;
    if (threadIdx.x == 0) failed = (int)a.sync[1];      // an earlier kernel's wait ran out
    for (int s = threadIdx.x; s < a.nmem; s += blockDim.x) {
        const Ctl* c = a.mem[s].ctl;
        mcol[s] = make_int2(c->col, c->n - c->col == 1 ? -a.mem[s].C : a.mem[s].C);
    }
    __syncthreads();
    if (failed) return;
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int t = 0; t < steps; ++t) {
        bool starts = false, ends = t == steps - 1;      // some member starts, ends a chunk
        for (int s = threadIdx.x; s < a.nmem; s += blockDim.x) {
            const int C = abs(mcol[s].y), col = (mcol[s].x + t) % C;
            starts |= col == 0 || (t == 0 && mcol[s].y < 0);      // (new_cols)
            ends |= col == C - 1;
        }
        starts = __syncthreads_or(starts);
        ends = __syncthreads_or(ends);
        for (int ph = starts ? PH_ENV : PH_HIST; ph < (ends ? NPH : PH_PIN); ++ph) {
            const int* first = a.first[ph];
            const int total = first[a.nmem];
            int s = 0;
            for (int64_t u0 = warp * rows; u0 < total; u0 += nwarps * rows)
                for (int64_t u = u0; u < min(u0 + rows, (int64_t)total); ++u) {
                    while (u >= first[s + 1]) ++s;
                    const int C = abs(mcol[s].y), col = (mcol[s].x + t) % C;
                    if (ph <= PH_PRE && col != 0 && (t != 0 || mcol[s].y > 0)) continue;
                    if (ph >= PH_PIN && col != C - 1 && t != steps - 1) continue;
                    batch_unit(ph, a.mem[s], t, steps - t, min(t, col) + 1, (int)(u - first[s]), lane);
                }
            if (!group_barrier(a.sync, gridDim.x, a.sync + 1, &failed)) return;
        }
    }
    // every block has passed the last barrier: advance the members
    if (blockIdx.x == 0)
        for (int s = threadIdx.x; s < a.nmem; s += blockDim.x) {
            const SimtDev<float>& d = a.mem[s];
            d.ctl->n += steps;
            d.ctl->slot = (d.ctl->slot + steps) % d.ring;
            d.ctl->col = (d.ctl->col + steps) % d.C;
            d.ctl->p0 = d.ctl->n;
        }
}

// output base of the next steps of every member
__global__ void k_batch_outputs(const __grid_constant__ BArgs a, void* const* outs) {
    for (int s = threadIdx.x; s < a.nmem; s += blockDim.x) {
        Ctl* c = a.mem[s].ctl;
        c->n0 = c->n;
        c->out = outs ? outs[s] : nullptr;
        c->yout = nullptr;
    }
}
__global__ void k_batch_status(const __grid_constant__ BArgs a, Ctl* out) {
    for (int s = threadIdx.x; s < a.nmem; s += blockDim.x) out[s] = *a.mem[s].ctl;
}

}  // namespace tdc

struct tdcfie_batch_s {
    std::vector<tdcfie_t> hs;
    cudaStream_t main = nullptr;
    std::vector<cudaStream_t> branch;
    std::vector<cudaEvent_t> joined;
    cudaEvent_t fork = nullptr, t0 = nullptr, t1 = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    double last_step_ms = 0.0;
    int64_t launches_per_step = 0;
    // persistent form
    bool persistent = false;
    SimtDev<float>* dmem = nullptr;
    int* dfirst = nullptr;
    unsigned long long* dsync = nullptr;
    void** douts = nullptr;       // the members' output pointers of a call
    Ctl* dstat = nullptr;         // the members' step states after a call
    BArgs args{};
    int rows = 1, threads = 256, blocks_per_sm = 1, grid = 0, sms = 0;
    double hist_bytes = 0.0;
};

static void destroy_batch(tdcfie_batch_t b) {
    if (!b) return;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    for (auto s : b->branch) cudaStreamDestroy(s);
    for (auto e : b->joined) cudaEventDestroy(e);
    for (cudaEvent_t e : {b->fork, b->t0, b->t1})
        if (e) cudaEventDestroy(e);
    if (b->main) cudaStreamDestroy(b->main);
    for (void* p : {(void*)b->dmem, (void*)b->dfirst, (void*)b->dsync, (void*)b->douts, (void*)b->dstat})
        if (p) cudaFree(p);
    delete b;
}

namespace tdc {
// The batch's stream starts after what is queued on the members' streams (a handle's device work is
// ordered with its opts.stream; for a stream of the library's own, with the legacy default stream, as in
// plan_step): fills and last readers of the output buffers above all.
static cudaError_t wait_members(tdcfie_batch_t b) {
    cudaError_t e = cudaSuccess;
    bool legacy = false;
    for (size_t i = 0; i < b->hs.size() && e == cudaSuccess; ++i) {
        tdcfie_t h = b->hs[i];
        if (h->own_stream && legacy) continue;
        legacy = legacy || h->own_stream;
        e = cudaEventRecord(h->ev_in, h->own_stream ? cudaStreamLegacy : h->stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(b->main, h->ev_in, 0);
    }
    return e;
}

// a handle the persistent kernel can step: FP32, one wave, direct solve
static bool persistent_member(tdcfie_t h) {
    return h->plan && h->plan->prec == TDCFIE_FP32 && h->plan->R == 1 && !h->plan->gmres_on && h->plan->blocks;
}

// nsteps steps of the members with the batch's configuration
static cudaError_t launch_persistent(tdcfie_batch_t b, int64_t nsteps, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b->grid);
    cfg.blockDim = dim3(b->threads);
    cfg.dynamicSmemBytes = b->hs.size() * sizeof(int2);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaSuccess;
    for (; nsteps > 0 && e == cudaSuccess; nsteps -= B_STEPS)
        e = cudaLaunchKernelEx(&cfg, k_batch_step, b->args, b->rows, (int)std::min(nsteps, B_STEPS));
    return e;
}

static int max_blocks_per_sm(tdcfie_batch_t b, int threads) {
    int nb = 0;
    const size_t smem = b->hs.size() * sizeof(int2);
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch_step, threads, smem) == cudaSuccess ? nb : 0;
}

// the kernel's launch shape; the barrier's count starts again, it is a multiple of the grid
static cudaError_t set_shape(tdcfie_batch_t b, int rows, int threads, int blocks_per_sm) {
    b->rows = rows;
    b->threads = threads;
    b->blocks_per_sm = blocks_per_sm;
    b->grid = b->sms * blocks_per_sm;
    return cudaMemsetAsync(b->dsync, 0, sizeof(unsigned long long), b->main);
}

// members' views and the units of every phase
static cudaError_t build_persistent(tdcfie_batch_t b) {
    const int n = (int)b->hs.size();
    std::vector<SimtDev<float>> mem(n);
    std::vector<int> first((size_t)NPH * (n + 1), 0);
    b->hist_bytes = 0.0;
    for (int s = 0; s < n; ++s) {
        const StepPlan* p = b->hs[s]->plan;
        mem[s] = simt_view<float>(b->hs[s], *p);
        b->hist_bytes += (double)p->nblk * p->ne * p->ne * 4.0;
        for (int ph = 0; ph < NPH; ++ph) first[ph * (n + 1) + s + 1] = first[ph * (n + 1) + s] + phase_units(p, ph);
    }
    cudaError_t e;
    if ((e = cudaMalloc(&b->dmem, sizeof(SimtDev<float>) * n)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->dfirst, sizeof(int) * first.size())) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->dsync, sizeof(unsigned long long) * 2)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->douts, sizeof(void*) * n)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&b->dstat, sizeof(Ctl) * n)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(b->dmem, mem.data(), sizeof(SimtDev<float>) * n, cudaMemcpyHostToDevice, b->main)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(b->dfirst, first.data(), sizeof(int) * first.size(), cudaMemcpyHostToDevice, b->main)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(b->dsync, 0, sizeof(unsigned long long) * 2, b->main)) != cudaSuccess) return e;
    b->args.mem = b->dmem;
    b->args.nmem = n;
    for (int ph = 0; ph < NPH; ++ph) b->args.first[ph] = b->dfirst + ph * (n + 1);
    b->args.sync = b->dsync;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    return set_shape(b, 1, 256, 1);
}
}  // namespace tdc

#define BK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { destroy_batch(b); return cuda_fail(nullptr, e_, #x); } } while (0)

extern "C" tdcfie_status tdcfie_batch_create(const tdcfie_t* handles, int64_t n, tdcfie_batch_t* out) {
    if (!handles || !out || n < 1) return fail(nullptr, TDCFIE_E_ARG, "need n >= 1 handles and an output pointer");
    if (n > 4096) return fail(nullptr, TDCFIE_E_ARG, "at most 4096 handles in a batch");
    for (int64_t i = 0; i < n; ++i) {
        if (!handles[i]) return fail(nullptr, TDCFIE_E_ARG, "NULL handle in the batch");
        if (!handles[i]->assembled || !handles[i]->plan)
            return fail(nullptr, TDCFIE_E_STATE, "every handle must be assembled before tdcfie_batch_create");
        if (handles[i]->opts.device != handles[0]->opts.device)
            return fail(nullptr, TDCFIE_E_ARG, "all handles of a batch must use the same device");
        for (int64_t j = 0; j < i; ++j)
            if (handles[j] == handles[i]) return fail(nullptr, TDCFIE_E_ARG, "a handle appears twice in the batch");
    }
    auto* b = new tdcfie_batch_s();
    b->hs.assign(handles, handles + n);
    BK(cudaSetDevice(handles[0]->opts.device));
    BK(cudaStreamCreateWithFlags(&b->main, cudaStreamNonBlocking));
    BK(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming));
    BK(cudaEventCreate(&b->t0));
    BK(cudaEventCreate(&b->t1));
    for (int64_t i = 0; i < n; ++i) {
        cudaStream_t s;
        cudaEvent_t e;
        BK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
        b->branch.push_back(s);
        BK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        b->joined.push_back(e);
    }
    b->persistent = true;
    for (int64_t i = 0; i < n; ++i) b->persistent = b->persistent && persistent_member(handles[i]);
    if (b->persistent) BK(build_persistent(b));
    *out = b;
    return TDCFIE_OK;
}

extern "C" tdcfie_status tdcfie_batch_step(tdcfie_batch_t b, int64_t nsteps, void* const* currents_out) {
    if (!b) return fail(nullptr, TDCFIE_E_ARG, "batch is NULL");
    if (nsteps < 0) return fail(nullptr, TDCFIE_E_ARG, "nsteps < 0");
    const int64_t n = (int64_t)b->hs.size();
    for (tdcfie_t h : b->hs)
        if (!h->excited || !h->plan)
            return fail(nullptr, TDCFIE_E_STATE, "set the excitation of every handle of the batch first");
    if (nsteps == 0) return TDCFIE_OK;
    cudaError_t e = cudaSetDevice(b->hs[0]->opts.device);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaSetDevice");
    e = wait_members(b);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "waiting for the members' streams");
    if (b->persistent) {
        // one kernel sets every member's output base
        if (currents_out) e = cudaMemcpyAsync(b->douts, currents_out, sizeof(void*) * n, cudaMemcpyHostToDevice, b->main);
        if (e == cudaSuccess) {
            k_batch_outputs<<<1, 256, 0, b->main>>>(b->args, currents_out ? b->douts : nullptr);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return cuda_fail(nullptr, e, "batch outputs");
    } else {
        for (int64_t i = 0; i < n; ++i) {
            const tdcfie_status st = plan_set_outputs(b->hs[i], currents_out ? currents_out[i] : nullptr, nullptr);
            if (st != TDCFIE_OK) return fail(nullptr, st, "batch handle " + std::to_string(i) + ": " + b->hs[i]->err);
        }
    }
    if (b->persistent) {
        b->launches_per_step = 1;      // one launch steps every member, and up to B_STEPS steps
    } else if (!b->exec) {
        e = cudaStreamBeginCapture(b->main, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaStreamBeginCapture");
        cudaError_t ce = cudaSuccess;
        // one step of every handle, each on its own branch of the graph
        ce = cudaEventRecord(b->fork, b->main);
        b->launches_per_step = 0;
        for (int64_t i = 0; i < n && ce == cudaSuccess; ++i) {
            ce = cudaStreamWaitEvent(b->branch[i], b->fork, 0);
            if (ce == cudaSuccess) ce = capture_step(b->hs[i], b->branch[i]);
            if (ce == cudaSuccess) ce = cudaEventRecord(b->joined[i], b->branch[i]);
            if (ce == cudaSuccess) ce = cudaStreamWaitEvent(b->main, b->joined[i], 0);
            b->launches_per_step += plan_launches_per_step(b->hs[i]);
        }
        const cudaError_t ee = cudaStreamEndCapture(b->main, &b->graph);
        if (ce != cudaSuccess || ee != cudaSuccess) {
            if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
            return cuda_fail(nullptr, ce != cudaSuccess ? ce : ee, "capturing the batch step graph");
        }
        e = cudaGraphInstantiate(&b->exec, b->graph, 0);
        if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaGraphInstantiate (batch)");
    }
    std::vector<Ctl> ctl(n);
    unsigned long long timeout = 0;
    e = cudaEventRecord(b->t0, b->main);
    if (b->persistent && e == cudaSuccess) e = launch_persistent(b, nsteps, b->main);
    for (int64_t i = 0; !b->persistent && i < nsteps && e == cudaSuccess; ++i) e = cudaGraphLaunch(b->exec, b->main);
    if (e == cudaSuccess) e = cudaEventRecord(b->t1, b->main);
    if (e == cudaSuccess && b->persistent) {
        k_batch_status<<<1, 256, 0, b->main>>>(b->args, b->dstat);
        e = cudaMemcpyAsync(ctl.data(), b->dstat, sizeof(Ctl) * n, cudaMemcpyDeviceToHost, b->main);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&timeout, b->dsync + 1, sizeof timeout, cudaMemcpyDeviceToHost, b->main);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->main);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "batch step");
    float ms = 0.f;
    cudaEventElapsedTime(&ms, b->t0, b->t1);
    b->last_step_ms = ms / (double)nsteps;
    if (timeout) return fail(nullptr, TDCFIE_E_TIMEOUT, "a bounded grid-wide wait of the batch kernel ran out");
    for (int64_t i = 0; i < n; ++i) {
        const tdcfie_status st = b->persistent ? plan_status(b->hs[i], ctl[i]) : plan_check(b->hs[i]);
        if (st != TDCFIE_OK) return fail(nullptr, st, "batch handle " + std::to_string(i) + ": " + b->hs[i]->err);
    }
    return TDCFIE_OK;
}

extern "C" tdcfie_status tdcfie_batch_tune(tdcfie_batch_t b, int64_t steps_per_candidate, int32_t* config) {
    if (!b) return fail(nullptr, TDCFIE_E_ARG, "batch is NULL");
    if (steps_per_candidate < 1) return fail(nullptr, TDCFIE_E_ARG, "steps_per_candidate < 1");
    for (tdcfie_t h : b->hs)
        if (!h->excited || !h->plan)
            return fail(nullptr, TDCFIE_E_STATE, "set the excitation of every handle of the batch first");
    if (b->persistent) {
        cudaError_t e = cudaSetDevice(b->hs[0]->opts.device);
        if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaSetDevice");
        for (tdcfie_t h : b->hs) {
            const tdcfie_status st = plan_set_outputs(h, nullptr, nullptr);
            if (st != TDCFIE_OK) return st;
        }
        // whole chunks of every member, so that each candidate sees as many chunk starts
        steps_per_candidate = (steps_per_candidate + 15) / 16 * 16;
        double best = 1e300;
        int br = b->rows, bt = b->threads, bb = b->blocks_per_sm;
        for (int rows : {1, 2, 4})
            for (int threads : {64, 128, 256}) {
                const int maxb = max_blocks_per_sm(b, threads);
                for (int bps : {1, 2, 4}) {
                    if (bps > maxb) continue;
                    e = set_shape(b, rows, threads, bps);
                    if (e == cudaSuccess) e = launch_persistent(b, 1, b->main);                        // warm-up
                    if (e == cudaSuccess) e = cudaEventRecord(b->t0, b->main);
                    if (e == cudaSuccess) e = launch_persistent(b, steps_per_candidate, b->main);
                    if (e == cudaSuccess) e = cudaEventRecord(b->t1, b->main);
                    if (e == cudaSuccess) e = cudaStreamSynchronize(b->main);
                    if (e != cudaSuccess) return cuda_fail(nullptr, e, "batch autotuner");
                    float ms = 0.f;
                    cudaEventElapsedTime(&ms, b->t0, b->t1);
                    if (ms < best) { best = ms; br = rows; bt = threads; bb = bps; }
                }
            }
        e = set_shape(b, br, bt, bb);
        if (e != cudaSuccess) return cuda_fail(nullptr, e, "batch autotuner");
        unsigned long long timeout = 0;
        e = cudaMemcpyAsync(&timeout, b->dsync + 1, sizeof timeout, cudaMemcpyDeviceToHost, b->main);
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->main);
        if (e != cudaSuccess) return cuda_fail(nullptr, e, "batch status");
        if (timeout) return fail(nullptr, TDCFIE_E_TIMEOUT, "a bounded grid-wide wait of the batch kernel ran out");
        // the candidates marched the members: back to the start of the march
        for (tdcfie_t h : b->hs) {
            const tdcfie_status st = plan_reset(h);
            if (st != TDCFIE_OK) return st;
        }
    }
    if (config) {
        config[0] = b->persistent ? 1 : 0;
        config[1] = b->rows;
        config[2] = b->threads;
        config[3] = b->blocks_per_sm;
    }
    return TDCFIE_OK;
}

extern "C" tdcfie_status tdcfie_batch_timing(tdcfie_batch_t b, double* step_ms, int64_t* launches_per_step) {
    if (!b) return fail(nullptr, TDCFIE_E_ARG, "batch is NULL");
    if (step_ms) *step_ms = b->last_step_ms;
    if (launches_per_step) *launches_per_step = b->launches_per_step;
    return TDCFIE_OK;
}

extern "C" tdcfie_status tdcfie_batch_destroy(tdcfie_batch_t b) {
    destroy_batch(b);
    return TDCFIE_OK;
}
