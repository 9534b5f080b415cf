// Interfaces of the projection adjoint (projection_adj.cu).
#pragma once
#include <vector>

#include "likelihood.cuh"

namespace gpuns {

constexpr int kAdjWarps = 4;                            // warps per CTA of the Limber adjoint
constexpr size_t kAdjSmemMax = 227 * 1024 - 8 * 1024;   // dynamic shared memory beside the kernels' static arrays

// Per-problem buffers of the projection adjoint for `cap` rows, in the problem's
// arithmetic type.
struct ProjectionAdj {
    void *win = nullptr, *resid = nullptr, *C = nullptr, *gC = nullptr, *gV = nullptr, *glnc = nullptr;
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
                          const T* LinvT, const T* Linv, double c0, const TableGrad& out, double* gfull, double* logL,
                          const int* nrows, int grid_rows, int* err, cudaStream_t st);

}  // namespace gpuns
