// Interfaces of the projection adjoint (projection_adj.cu).
#pragma once
#include <mutex>
#include <vector>

#include "likelihood.cuh"

namespace gpuns {

// Where a gradient call's results go: a device slot that its set-up kernel writes,
// so that the launches behind it hold no pointer of the caller's.
struct OutPtr {
    double* const* slot;
    __device__ __forceinline__ double* get() const { return *slot; }
};

// Those launches (some twenty, with a fork and a join) as CUDA graphs, one per row
// bucket, made at a bucket's third call: a lockstep NUTS step or a training step
// of 64 rows is bound by the host (359 -> 304 us per call through autograd).  At most
// kMost graphs per problem; other buckets, and calls on a stream that is being
// captured, are launched one by one.  (Log-likelihood calls have half the launches
// and their host keeps ahead of the GPU: replaying them cost 2 - 8 us per call.)
struct CallGraphs {
    static constexpr int kMost = 8;
    struct Entry { int rows, seen; cudaGraphExec_t exec; };
    // Held by a call from its set-up kernel to its last launch: the launches read the row
    // count, the parameters and the result slots that this kernel writes.  Calls on
    // different streams follow one another by `done` (1 us of host time), so that none of
    // them can write through the slots of another, whose buffers may be gone.
    std::mutex mu;
    cudaEvent_t done = nullptr;
    std::vector<Entry> entries;
    cudaStream_t cap = nullptr;
    double** d_out = nullptr;     // device slots: log L, gradient
    int create(std::vector<void*>& owned);
    void release();
    // set-up, then the launches of `body`, alone or as a graph (mu is taken)
    template <typename S, typename F>
    int call(int rows, cudaStream_t st, S&& setup, F&& body);
    template <typename F>
    int run(int rows, cudaStream_t st, F&& body);
};
// Rows a call's grids are sized for: powers of two up to 16, then multiples of 16.
inline int call_rows(int B, int max_batch) {
    int r = 1;
    if (B > 16) r = (B + 15) & ~15;
    else while (r < B) r *= 2;
    return r < max_batch ? r : max_batch;
}

template <typename S, typename F>
int CallGraphs::call(int rows, cudaStream_t st, S&& setup, F&& body) {
    std::lock_guard<std::mutex> lk(mu);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        NS_TRY(setup());                          // the caller orders the replays of its own graph
        return body(st);
    }
    NS_CUDA_TRY(cudaStreamWaitEvent(st, done, 0));
    NS_TRY(setup());
    const int s = run(rows, st, body);
    NS_CUDA_TRY(cudaEventRecord(done, st));       // after a failed launch too: what was queued still runs
    return s;
}

template <typename F>
int CallGraphs::run(int rows, cudaStream_t st, F&& body) {
    Entry* e = nullptr;
    for (Entry& x : entries)
        if (x.rows == rows) e = &x;
    if (!e) {
        if ((int)entries.size() >= kMost) return body(st);
        entries.push_back(Entry{rows, 0, nullptr});
        e = &entries.back();
    }
    if (!e->exec && ++e->seen == 3) {
        cudaGraph_t g = nullptr;
        if (!cap) NS_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
        NS_CUDA_TRY(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal));
        const int s = body(cap);
        const cudaError_t c = cudaStreamEndCapture(cap, &g);
        if (s != NS_OK) {
            if (c == cudaSuccess) cudaGraphDestroy(g);
            return s;
        }
        NS_CUDA_TRY(c);
        const cudaError_t i = cudaGraphInstantiate(&e->exec, g, 0);
        cudaGraphDestroy(g);
        NS_CUDA_TRY(i);
    }
    if (!e->exec) return body(st);
    NS_CUDA_TRY(cudaGraphLaunch(e->exec, st));
    return NS_OK;
}

constexpr int kAdjWarps = 4;                            // warps per CTA of the Limber adjoint
constexpr size_t kAdjSmemMax = 227 * 1024 - 8 * 1024;   // dynamic shared memory beside the kernels' static arrays

// Per-problem buffers of the projection adjoint for `cap` rows, in the problem's
// arithmetic type.
struct ProjectionAdj {
    void *win = nullptr, *resid = nullptr, *C = nullptr, *gC = nullptr, *gV = nullptr, *glnc = nullptr, *gv = nullptr;
    void* win_nodes = nullptr;         // FP64: the windows' node-local functions
    void* part = nullptr;              // partial rows of the table gradient
    void* scratch = nullptr;           // arrays of k_windows_adj where shared memory does not hold them
    size_t win_smem = 0;
    int sorted = 0;                    // ascending multipoles
    int4* ranges[3] = {};              // node ranges for 8, 16, 32 warps per evaluation
    int *ptr[3] = {}, *idx[3] = {}, part_rows[3] = {};
    cudaStream_t side = nullptr;       // the windows run beside the emulator
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    std::vector<void*> owned;
};

// Where d log L / d table goes: rows x (n_z n_k) in FP64 or FP32, or (px = 2, 3)
// scaled into px bf16 planes.
struct TableGrad {
    void* table = nullptr;
    int px = 0;
    __nv_bfloat16* planes = nullptr;
    long long stride = 0;
    int pitch = 0;
    float scale = 1.f;
};

int projection_adj_create(const ShearParams& sp, int elt, int cap, ProjectionAdj* a);
void projection_adj_free(ProjectionAdj* a);

// Windows stage on the adjoint's side stream, forked from st; then, after the
// emulator on st, the rest (joins the windows first).
template <typename T>
int launch_projection_adj_windows(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const int* nrows,
                                  int grid_rows, cudaStream_t st);
template <typename T>
int launch_projection_adj(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const T* table,
                          const T* LinvT, const T* Linv, double c0, const TableGrad& out, double* gfull, OutPtr logL,
                          const int* nrows, int grid_rows, int* err, cudaStream_t st);

}  // namespace gpuns
