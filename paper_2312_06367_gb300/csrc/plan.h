// Per-handle step plan shared by the SIMT (march.cu) and tensor-core (umma.cu) paths.
#pragma once
#include "internal.h"

namespace tdc {
struct TcStep;
struct GmresPlan;
struct MlpState;
struct FactPlan;

struct StepPlan {
    int prec = TDCFIE_FP64;
    int R = 1, ne = 0, nc = 0, K = 0, nblk = 0, ring = 0;
    size_t esz = 8;
    int C = 1;                   // steps per chunk (simt.h)
    int ld = 0, ldc = 0;         // SIMT paths: row lengths of matrices and vectors (16-byte multiples)
    int ngroups = 0, npts = 0;   // SIMT paths: groups of the pre-sums, distinct quadrature points
    void* blocks = nullptr;      // nblk x ne x ld (path precision): -A, alpha L2, -T_1 .. -T_{K-1}
    void* t0inv = nullptr;       // ne x ld
    void* t0mat = nullptr;       // ne x ne, T_0 itself (GMRES matvec)
    void* guessbuf = nullptr;    // R x ld learned initial guess
    GmresPlan* gm = nullptr;
    MlpState* mlp = nullptr;     // learned-guess network (GMRES with TDCFIE_GUESS_MLP)
    bool gmres_on = false;       // per-step solve by GMRES (else the explicit T_0^-1)
    bool mlp_on = false;         // learned guess evaluated each step
    bool guess_extrap = false;   // learned guess on top of the cubic extrapolation (else y_{n-1})
    void* pinv = nullptr;        // nc x ldc
    void* E = nullptr;           // C x R x ld  (e of the chunk's steps)
    void* Hv = nullptr;          // C x R x ld  (h)
    void* ringbuf = nullptr;     // ring x R x ld, then R x ld zeros
    void* b = nullptr;           // R x ld
    void* partial = nullptr;     // ngroups x C x R x ld pre-sums (8 bytes each: FP64, or an FP32 pair)
    void* inner = nullptr;       // C x C x R x ld products of the lags inside a chunk
    void* z = nullptr;           // C x R x ldc
    void* u = nullptr;           // C x R x ldc
    int* done = nullptr;
    Ctl* ctl = nullptr;
    // plane-wave tests: distinct points, and per edge (e-points first) point index and weighted basis
    // vector (tensor paths: as {c, index}); env: envelopes of a chunk (SIMT paths)
    void* env = nullptr; void* pts = nullptr; void* ecoef = nullptr;
    int* eptr = nullptr; int* enE = nullptr; int* eidx = nullptr;
    // factored history form (factored.cu); blocks and t0inv are then unused
    FactPlan* fact = nullptr;
    // tensor-core path
    TcStep* gemm = nullptr;
    // graphs: G_PRE the tests (and, SIMT paths, pre-sums) of a chunk, G_STEP one step's history and
    // solve, G_LAST the same and the post-processing of the finished steps (tensor paths: of k steps in
    // G_LAST + k - 1), G_CHUNK a whole chunk
    enum { G_STEP = 0, G_PRE, G_CHUNK, G_LAST, NGRAPH = G_LAST + 3 };
    cudaGraph_t graph[NGRAPH] = {};
    cudaGraphExec_t exec[NGRAPH] = {};
    int nodes[NGRAPH] = {};                              // kernels per graph
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    int launches_per_step = 0;
};

template <typename T>
struct SimtDev;
// device view of the plan (march.cu)
template <typename T>
SimtDev<T> simt_view(tdcfie_t h, const StepPlan& p);
// plane-wave tests into p.E, p.Hv, of the columns that new_cols gives (march.cu); returns the number of
// kernels
template <typename T>
int launch_tests(tdcfie_t h, StepPlan& p, int most, cudaStream_t s);
// factored history form (factored.cu)
tdcfie_status build_fact(tdcfie_t h, StepPlan* p);
tdcfie_status reset_fact(tdcfie_t h, StepPlan* p);
void destroy_fact(FactPlan* f);
double fact_step_bytes(const StepPlan* p);
int64_t fact_nnz(const StepPlan* p, bool stored);
// history, solve and post-processing of one step (the factored form needs j_n in its own history)
template <typename T>
int launch_step_fact(tdcfie_t h, StepPlan& p, cudaStream_t s);

}  // namespace tdc
