// Hand-written adjoint of the shear likelihood: d log L / d theta.
//
// The emulator forward with stored activations, the projection and its reverse
// (projection_adj.cu: log L, the table gradient and the gradient of the
// parameters that enter the projection), the emulator backward (transposed
// GEMMs, tanh' from the stored activations), and the emulator inputs' share
// added to the parameter gradient in k_finish_grad.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "likelihood.cuh"
#include "projection_adj.cuh"
#include "tcgen05.cuh"

namespace gpuns {

// ------------------------------------------------------------------ emulator backward
namespace adj {

// FP64 backward layer: share z of the contraction C = A W (A: rows x K, W: K x N
// row-major), k in [z kc, (z + 1) kc).  Bound by the FP64 pipe (2 FMA per cycle and
// SM): the output layer of the 39-d problem contracts 10000 outputs into 16 tiles of
// 64 units, so that without shares 16 of 152 SMs worked (24 gradients 21.6 ms, 2.1
// with them and the forward pass on the tensor cores).
constexpr int kBackN = 64, kBackK = 8, kBackThreads = 256;
template <int BM>
__global__ void __launch_bounds__(kBackThreads)
k_back(const double* __restrict__ A, const double* __restrict__ W, double* __restrict__ part, int cap,
       const int* __restrict__ nrows, int N, int K, int kc) {
    constexpr int TN = 4, TX = kBackN / TN, TY = kBackThreads / TX, TM = BM / TY;
    const int M = *nrows;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * kBackN;
    if (m0 >= M) return;
    __shared__ double As[kBackK][BM + 1];
    __shared__ double Bs[kBackK][kBackN + 1];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int k_end = min(K, ((int)blockIdx.z + 1) * kc);
    double acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;
    for (int k0 = blockIdx.z * kc; k0 < k_end; k0 += kBackK) {
        for (int i = tid; i < BM * kBackK; i += kBackThreads) {
            const int rr = i / kBackK, c = i % kBackK;
            As[c][rr] = (m0 + rr < M && k0 + c < k_end) ? A[(size_t)(m0 + rr) * K + k0 + c] : 0.0;
        }
        for (int i = tid; i < kBackN * kBackK; i += kBackThreads) {
            const int c = i / kBackN, nn = i % kBackN;
            Bs[c][nn] = (n0 + nn < N && k0 + c < k_end) ? W[(size_t)(k0 + c) * N + n0 + nn] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kBackK; ++kk) {
            double a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + i * TY];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + j * TX];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int gm = m0 + ty + i * TY;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int gn = n0 + tx + j * TX;
            if (gn < N) part[((size_t)blockIdx.z * cap + gm) * N + gn] = acc[i][j];
        }
    }
}

// the shares added in order, times tanh' from the stored activations
__global__ void k_back_sum(const double* __restrict__ part, int cap, int shares, const double* __restrict__ h, int N,
                           double* __restrict__ out, const int* __restrict__ nrows) {
    const int row = blockIdx.y, n = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= *nrows || n >= N) return;
    double s = 0.0;
    for (int z = 0; z < shares; ++z) s += part[((size_t)z * cap + row) * N + n];
    const double hh = h[(size_t)row * N + n];
    out[(size_t)row * N + n] = s * (1.0 - hh * hh);
}

// Shares of a backward contraction: enough for one block per SM at one row tile,
// at least 64 terms each, by shape only.  (The table gradient's partial sums go by the
// rows of a call, projection_adj.cu, as do the K splits of the backward plane GEMMs: a
// gradient has the same bits in every call of its row bucket, log L in every call.)
static int back_shares(int N, int K) {
    const int tiles = (N + kBackN - 1) / kBackN;
    return std::max(1, std::min((K + 63) / 64, 152 / tiles));
}

// FP64 input layer
__global__ void k_emu_in_store(const double* __restrict__ theta_full, int P, const int* __restrict__ inputs,
                               const double* __restrict__ center, const double* __restrict__ scale, int K0,
                               const double* __restrict__ W0, const double* __restrict__ b0, int N,
                               double* __restrict__ out, const int* __restrict__ nrows) {
    const int row = blockIdx.y;
    if (row >= *nrows) return;
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    double acc = b0[n];
    for (int j = 0; j < K0; ++j)
        acc += W0[(size_t)n * K0 + j] * ((theta_full[(size_t)row * P + inputs[j]] - center[j]) / scale[j]);
    out[(size_t)row * N + n] = tanh(acc);
}

// The emulator inputs' share g_x = g_pre_1 W0 (rows x K0, K0 <= KMAX) added to
// the projection's parameter gradient, free parameters only.  One block per
// row; the K0 sums are formed in one pass over the row and reduced together
// (a block reduction per input took 42 us at 4096 rows of 7 inputs).
template <typename T, int KMAX>
__global__ void __launch_bounds__(256)
k_finish_grad(const T* __restrict__ gpre, const T* __restrict__ W0, int N1, int K0, const int* __restrict__ inputs,
              const double* __restrict__ scale, const double* __restrict__ gfull, int P,
              const int* __restrict__ free_of_full, const OutPtr grad, int d, const int* __restrict__ nrows) {
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    __shared__ T part[8][KMAX];
    __shared__ double gx[KMAX];
    T s[KMAX];
#pragma unroll
    for (int j = 0; j < KMAX; ++j) s[j] = T(0);
    for (int n = threadIdx.x; n < N1; n += 256) {
        const T g = gpre[(size_t)row * N1 + n];
#pragma unroll
        for (int j = 0; j < KMAX; ++j)
            if (j < K0) s[j] = fma(g, W0[(size_t)n * K0 + j], s[j]);
    }
#pragma unroll
    for (int j = 0; j < KMAX; ++j) {
        if (j >= K0) break;
        const T t = warp_sum(s[j]);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5][j] = t;
    }
    __syncthreads();
    if (threadIdx.x < K0) {
        T t = T(0);
        for (int w = 0; w < 8; ++w) t += part[w][threadIdx.x];
        gx[threadIdx.x] = (double)t / scale[threadIdx.x];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < P; i += 256) {
        const int f = free_of_full[i];
        if (f < 0) continue;
        double v = gfull[(size_t)row * P + i];
        for (int j = 0; j < K0; ++j)
            if (inputs[j] == i) v += gx[j];
        grad.get()[(size_t)row * d + f] = v;
    }
}

template <typename T>
__global__ void k_scale(const T* __restrict__ in, T* __restrict__ out, T s, int n_per_row, const int* __restrict__ nrows) {
    const int row = blockIdx.y;
    if (row >= *nrows) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_per_row; i += gridDim.x * blockDim.x)
        out[(size_t)row * n_per_row + i] = s * in[(size_t)row * n_per_row + i];
}

// Transpose of the coarse -> fine Catmull-Rom z interpolation:
// g_coarse[j][k] = sum_{jz, q: zr[jz][q] = j} w[jz][q] g_fine[jz][k].
template <typename T>
__global__ void k_zinterp_adj(const T* __restrict__ gfine, int nz, const int* __restrict__ zr,
                              const double* __restrict__ zw, T* __restrict__ gcoarse, int nzc, int nk,
                              const int* __restrict__ nrows) {
    const int row = blockIdx.y;
    if (row >= *nrows) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nzc * nk; i += gridDim.x * blockDim.x) {
        const int j = i / nk, k = i % nk;
        T s = T(0);
        for (int jz = 0; jz < nz; ++jz)
            for (int q = 0; q < 4; ++q)
                if (zr[jz * 4 + q] == j) s += (T)zw[jz * 4 + q] * gfine[(size_t)row * nz * nk + jz * nk + k];
        gcoarse[(size_t)row * nzc * nk + i] = s;
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_transpose(const T* __restrict__ A, T* __restrict__ B, int D) {
    __shared__ T t[32][33];
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32, x = threadIdx.x & 31;
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (y0 + y < D && x0 + x < D) t[y][x] = A[(size_t)(y0 + y) * D + x0 + x];
    __syncthreads();
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (x0 + y < D && y0 + x < D) B[(size_t)(x0 + y) * D + y0 + x] = t[x][y];
}

// T[p][k][n] = W[p][n][k] for bf16 planes: W N rows of pitch wp, T K rows of pitch tp.
__global__ void __launch_bounds__(256) k_transpose_planes(const __nv_bfloat16* __restrict__ W, int N, int K, int wp,
                                                          __nv_bfloat16* __restrict__ T, int tp) {
    __shared__ __nv_bfloat16 t[32][33];
    const __nv_bfloat16* w = W + (size_t)blockIdx.z * N * wp;
    __nv_bfloat16* o = T + (size_t)blockIdx.z * K * tp;
    const int n0 = blockIdx.y * 32, k0 = blockIdx.x * 32, x = threadIdx.x & 31;
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (n0 + y < N && k0 + x < K) t[y][x] = w[(size_t)(n0 + y) * wp + k0 + x];
    __syncthreads();
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (k0 + y < K && n0 + x < N) o[(size_t)(k0 + y) * tp + n0 + x] = t[x][y];
}

// g_pre_l = (g_pre_{l+1} W_l) * (1 - h_l^2)
static int back_layer(const double* A, const double* W, const double* h, double* part, int cap, double* out,
                      const int* nrows, int grid_rows, int N, int K, cudaStream_t st) {
    const int S = back_shares(N, K), kc = ((K + S - 1) / S + kBackK - 1) / kBackK * kBackK;
    // 24 rows fill three quarters of a 32-row tile and three eighths of a 64-row one
    const int bm = grid_rows <= 16 ? 16 : grid_rows <= 32 ? 32 : 64;
    const dim3 g((N + kBackN - 1) / kBackN, (grid_rows + bm - 1) / bm, S);
    if (bm == 16) k_back<16><<<g, kBackThreads, 0, st>>>(A, W, part, cap, nrows, N, K, kc);
    else if (bm == 32) k_back<32><<<g, kBackThreads, 0, st>>>(A, W, part, cap, nrows, N, K, kc);
    else k_back<64><<<g, kBackThreads, 0, st>>>(A, W, part, cap, nrows, N, K, kc);
    NS_CUDA_TRY(cudaGetLastError());
    k_back_sum<<<dim3((N + 255) / 256, grid_rows), 256, 0, st>>>(part, cap, S, h, N, out, nrows);
    NS_CUDA_TRY(cudaGetLastError());
    return NS_OK;
}

}  // namespace adj

// One problem's gradient state.  Its kernels report to the problem's status word
// (Workspace::d_err), which ns_problem_status reads.
struct GradState {
    const ns_problem* p = nullptr;
    int* d_nrows = nullptr;
    double* theta_full = nullptr;
    void* table = nullptr;     // cap x n_out (emulator output)
    void* table_fine = nullptr;
    void* gtab = nullptr;      // cap x n_z n_k
    void* gcoarse = nullptr;   // cap x n_out, coarse-z emulators
    void* Linv = nullptr;      // D x D, L^-1 row-major in the arithmetic type
    ProjectionAdj proj;
    double* gfull = nullptr;   // cap x P
    // FP64: stored activations per hidden layer, the slices of one, adjoints
    // (ping-pong) and the shares of a backward contraction
    SliceInput xs;
    double* part = nullptr;
    int cap = 0;
    std::vector<double*> H;
    double* g64[2] = {nullptr, nullptr};
    // FP32 and BF16: activations and adjoints in px bf16 planes (3: FP32; 2: the
    // leading 16 bits beside exact bf16 weights), weights in pw planes.  Layer l
    // (1 .. L-1) maps dims[l] -> dims[l+1].
    int px = 0, pw = 0;
    long long rows_pad = 0;
    std::vector<__nv_bfloat16*> Hp;          // input activations of layer l: px x rows_pad x pitch
    __nv_bfloat16* Gp[2] = {nullptr, nullptr};
    float* G1 = nullptr;                     // gradient of layer 1's input pre-activations (rows x dims[1])
    std::vector<CUtensorMap> tmW, tmWT;      // W_l and its transpose
    std::vector<PlaneMapX> tmH, tmG;         // layer l's forward and backward operands
    CallGraphs graphs;
    std::vector<void*> owned;
};

static std::mutex g_grad_mu;

int CallGraphs::create(std::vector<void*>& owned) {
    void* v;
    if (cudaMalloc(&v, 2 * sizeof(double*)) != cudaSuccess) return NS_ENOMEM;
    owned.push_back(v);
    d_out = (double**)v;
    NS_CUDA_TRY(cudaEventCreateWithFlags(&done, cudaEventDisableTiming));
    return NS_OK;
}

void CallGraphs::release() {
    for (Entry& e : entries)
        if (e.exec) cudaGraphExecDestroy(e.exec);
    entries.clear();
    if (cap) cudaStreamDestroy(cap);
    if (done) cudaEventDestroy(done);
    cap = nullptr;
    done = nullptr;
}

static int grad_alloc(GradState* g, size_t bytes, void** out) {
    if (cudaMalloc(out, bytes) != cudaSuccess) return NS_ENOMEM;
    g->owned.push_back(*out);
    return NS_OK;
}

static int grad_state_create(const ns_problem* p, GradState* g) {
    const int L = p->n_layers, cap = p->max_batch, n_out = p->dims.back(), nzk = p->sp.n_z * p->sp.n_k;
    const bool f64 = p->precision == NS_PREC_FP64, coarse = p->n_z_emu != p->sp.n_z;
    const size_t T = f64 ? 8 : 4;
    void* v;
    g->p = p;
    NS_TRY(g->graphs.create(g->owned));
    NS_TRY(grad_alloc(g, sizeof(int), (void**)&g->d_nrows));
    NS_TRY(grad_alloc(g, sizeof(double) * (size_t)cap * p->P, (void**)&g->theta_full));
    NS_TRY(grad_alloc(g, sizeof(double) * (size_t)cap * p->P, (void**)&g->gfull));
    NS_TRY(grad_alloc(g, T * (size_t)cap * n_out, &g->table));
    NS_TRY(grad_alloc(g, T * (size_t)cap * nzk, &g->gtab));
    if (coarse) {
        NS_TRY(grad_alloc(g, T * (size_t)cap * nzk, &g->table_fine));
        NS_TRY(grad_alloc(g, T * (size_t)cap * n_out, &g->gcoarse));
    }
    NS_TRY(projection_adj_create(p->sp, (int)T, cap, &g->proj));
    NS_TRY(grad_alloc(g, T * (size_t)p->D * p->D, &g->Linv));
    {
        const dim3 b((p->D + 31) / 32, (p->D + 31) / 32);
        if (f64) adj::k_transpose<double><<<b, 256>>>(p->d_LinvT64, (double*)g->Linv, p->D);
        else adj::k_transpose<float><<<b, 256>>>(p->d_LinvT32, (float*)g->Linv, p->D);
        NS_CUDA_TRY(cudaGetLastError());
    }
    int wmax = 0;
    for (int l = 1; l <= L; ++l) wmax = std::max(wmax, p->dims[l]);
    if (f64) {
        g->H.assign(L, nullptr);
        for (int l = 1; l < L; ++l) NS_TRY(grad_alloc(g, 8 * (size_t)cap * p->dims[l], (void**)&g->H[l]));
        for (int i = 0; i < 2; ++i) NS_TRY(grad_alloc(g, 8 * (size_t)cap * wmax, (void**)&g->g64[i]));
        g->cap = cap;
        size_t part = 0;
        for (int l = 1; l < L; ++l)
            part = std::max(part, (size_t)adj::back_shares(p->dims[l], p->dims[l + 1]) * p->dims[l]);
        NS_TRY(grad_alloc(g, 8 * part * cap, (void**)&g->part));
        if (takes_slices(p)) {
            const size_t n = slice_input_bytes(p, cap);
            NS_TRY(grad_alloc(g, n, (void**)&g->xs.slices));
            NS_CUDA_TRY(cudaMemsetAsync(g->xs.slices, 0, n, nullptr));
            NS_TRY(grad_alloc(g, sizeof(double) * cap, (void**)&g->xs.scale));
            NS_TRY(slice_input_maps(p, cap, &g->xs));
        }
        NS_CUDA_TRY(cudaStreamSynchronize(nullptr));   // calls may come on any stream
        return NS_OK;
    }
    const bool f32 = p->precision == NS_PREC_FP32;
    g->px = f32 ? 3 : 2;
    g->pw = f32 ? 3 : 1;
    g->rows_pad = ((cap + 127) / 128) * 128;
    g->Hp.assign(L, nullptr);
    g->tmH.resize(L); g->tmG.resize(L); g->tmW.resize(L); g->tmWT.resize(L);
    for (int i = 0; i < 2; ++i) {
        // the first holds the widest operand (the output layer's), the second hidden layers only
        const size_t n = (size_t)g->px * g->rows_pad * plane_pitch(i == 0 ? wmax : p->hidden_max);
        NS_TRY(grad_alloc(g, 2 * n, &v));
        g->Gp[i] = (__nv_bfloat16*)v;
        NS_CUDA_TRY(cudaMemset(v, 0, 2 * n));
    }
    NS_TRY(grad_alloc(g, 4 * (size_t)g->rows_pad * p->dims[1], (void**)&g->G1));
    for (int l = 1; l < L; ++l) {
        const int K = p->dims[l], N = p->dims[l + 1], kp = plane_pitch(K), np = plane_pitch(N);
        const long long hs = g->rows_pad * kp;
        NS_TRY(grad_alloc(g, 2 * (size_t)g->px * hs, &v));
        NS_CUDA_TRY(cudaMemset(v, 0, 2 * (size_t)g->px * hs));
        g->Hp[l] = (__nv_bfloat16*)v;
        NS_TRY(make_plane_maps_x(&g->tmH[l], v, (int)g->rows_pad, K, hs, g->px));
        // backward step l reads G_{l+1} from buffer (L - l - 1) % 2
        NS_TRY(make_plane_maps_x(&g->tmG[l], g->Gp[(L - l - 1) & 1], (int)g->rows_pad, N, g->rows_pad * np, g->px));
        const __nv_bfloat16* W = f32 ? p->d_Wp[l] : (const __nv_bfloat16*)p->d_W[l];
        NS_TRY(make_tensor_map_planes(&g->tmW[l], W, N, K, (long long)N * kp, g->pw, 128));
        NS_TRY(grad_alloc(g, 2 * (size_t)g->pw * K * np, &v));
        adj::k_transpose_planes<<<dim3((K + 31) / 32, (N + 31) / 32, g->pw), 256>>>(W, N, K, kp, (__nv_bfloat16*)v, np);
        NS_CUDA_TRY(cudaGetLastError());
        NS_TRY(make_tensor_map_planes(&g->tmWT[l], v, K, N, (long long)K * np, g->pw, 128));
    }
    NS_CUDA_TRY(cudaStreamSynchronize(nullptr));   // calls may come on any stream
    return NS_OK;
}

static void grad_state_free(GradState* g) {
    g->graphs.release();
    projection_adj_free(&g->proj);
    for (void* q : g->owned) cudaFree(q);
    delete g;
}

template <typename T>
static int launch_finish_grad(const ns_problem* p, GradState* g, const T* gpre, int B, OutPtr grad, cudaStream_t st) {
    auto kern = p->dims[0] <= 8 ? adj::k_finish_grad<T, 8> : adj::k_finish_grad<T, 32>;
    NS_CUDA_TRY(launch_pdl(kern, dim3(B), dim3(256), 0, st, gpre, (const T*)p->d_W[0], p->dims[1], p->dims[0],
                           (const int*)p->d_inputs, (const double*)p->d_in_scale, (const double*)g->gfull, p->P,
                           (const int*)p->d_free_of_full, grad, p->d, (const int*)g->d_nrows));
    return NS_OK;
}

// FP64 problems: the emulator forward as fixed-point slices on the tensor cores (as the
// likelihood's), backward on the FP64 pipe.
static int run_grad_f64(const ns_problem* p, GradState* g, int B, OutPtr logL, OutPtr grad, cudaStream_t st) {
    const int L = p->n_layers, n_out = p->dims.back();
    const ShearParams& sp = p->sp;
    NS_TRY(launch_projection_adj_windows<double>(sp, &g->proj, g->theta_full, g->d_nrows, B, st));
    const dim3 g0((p->dims[1] + 255) / 256, B);
    adj::k_emu_in_store<<<g0, 256, 0, st>>>(g->theta_full, p->P, p->d_inputs, p->d_in_center, p->d_in_scale,
                                            p->dims[0], (const double*)p->d_W[0], (const double*)p->d_b[0],
                                            p->dims[1], g->H[1], g->d_nrows);
    NS_CUDA_TRY(cudaGetLastError());
    for (int l = 1; l < L; ++l)
        NS_TRY(launch_layer_f64(p, l, g->xs, g->H[l], l == L - 1 ? (double*)g->table : g->H[l + 1], g->d_nrows, B,
                                p->ws.d_err, st));
    const double* tab = (const double*)g->table;
    const bool coarse = p->n_z_emu != sp.n_z;
    if (coarse) {
        NS_TRY(launch_zinterp_generic(p, g->table, g->table_fine, g->d_nrows, B, 8, st));
        tab = (const double*)g->table_fine;
    }
    NS_TRY(launch_projection_adj<double>(sp, &g->proj, g->theta_full, tab, p->d_LinvT64, (const double*)g->Linv, p->c0,
                                         TableGrad{g->gtab}, g->gfull, logL, g->d_nrows, B, p->ws.d_err, st));
    // table adjoint -> emulator output adjoint (transpose of the z interpolation) -> g_pre_L
    const double* gt = (const double*)g->gtab;
    if (coarse) {
        const dim3 gz((n_out + 255) / 256, B);
        adj::k_zinterp_adj<double><<<gz, 256, 0, st>>>(gt, sp.n_z, p->d_zi_row, p->d_zi_w, (double*)g->gcoarse,
                                                       p->n_z_emu, sp.n_k, g->d_nrows);
        gt = (const double*)g->gcoarse;
    }
    const dim3 gs((n_out + 255) / 256, B);
    adj::k_scale<double><<<gs, 256, 0, st>>>(gt, g->g64[0], p->out_sigma, n_out, g->d_nrows);
    NS_CUDA_TRY(cudaGetLastError());
    // g_pre_{l} = (g_pre_{l+1} W_l) * (1 - h_l^2), l = L-1 .. 1
    int cur = 0;
    for (int l = L - 1; l >= 1; --l) {
        NS_TRY(adj::back_layer(g->g64[cur], (const double*)p->d_W[l], g->H[l], g->part, g->cap, g->g64[cur ^ 1],
                               g->d_nrows, B, p->dims[l], p->dims[l + 1], st));
        cur ^= 1;
    }
    return launch_finish_grad<double>(p, g, g->g64[cur], B, grad, st);
}

// FP32 and BF16 problems: the emulator forward and backward as plane GEMMs
// (gemm_planes.cu), the projection adjoint in FP32.
static int run_grad_planes(const ns_problem* p, GradState* g, int B, OutPtr logL, OutPtr grad, cudaStream_t st) {
    const int L = p->n_layers, n_out = p->dims.back(), px = g->px, pw = g->pw;
    const ShearParams& sp = p->sp;
    auto planes_out = [&](PlaneEpi& e, __nv_bfloat16* buf, int width) {
        e.planes = buf;
        e.pitch = plane_pitch(width);
        e.plane_stride = g->rows_pad * e.pitch;
    };
    NS_TRY(launch_projection_adj_windows<float>(sp, &g->proj, g->theta_full, g->d_nrows, B, st));
    NS_TRY(launch_emu_input_planes(p, g->theta_full, g->d_nrows, B, px, g->Hp[1],
                                   g->rows_pad * plane_pitch(p->dims[1]), st));
    for (int l = 1; l < L; ++l) {
        const bool last = (l == L - 1);
        PlaneEpi e;
        e.mode = last ? PLN_OUT : PLN_TANH;
        e.bias = (const float*)p->d_b[l];
        if (last) {
            e.mu = (const float*)p->d_out_mu;
            e.sigma = (float)p->out_sigma;
            e.out = (float*)g->table;
        } else {
            planes_out(e, g->Hp[l + 1], p->dims[l + 1]);
        }
        // by shape alone, so that log L does not depend on the batch; BF16: no K split, so
        // that every activation has the bits of the one chain
        NS_TRY(launch_gemm_planes(px, pw, &g->tmW[l], &g->tmH[l], e, g->d_nrows, B, p->dims[l + 1], p->dims[l],
                                  pw == 1 ? 1 : plane_split(p->dims[l + 1], p->dims[l]), p->ws.d_err, st));
    }
    const float* tab = (const float*)g->table;
    const bool coarse = p->n_z_emu != sp.n_z;
    if (coarse) {
        NS_TRY(launch_zinterp_generic(p, g->table, g->table_fine, g->d_nrows, B, 4, st));
        tab = (const float*)g->table_fine;
    }
    // d log L / d (output pre-scaling) = sigma * d log L / d table, in planes
    TableGrad tg;
    if (coarse) {
        tg.table = g->gtab;
    } else {
        tg.px = px;
        tg.planes = g->Gp[0];
        tg.pitch = plane_pitch(n_out);
        tg.stride = g->rows_pad * tg.pitch;
        tg.scale = (float)p->out_sigma;
    }
    NS_TRY(launch_projection_adj<float>(sp, &g->proj, g->theta_full, tab, p->d_LinvT32, (const float*)g->Linv, p->c0, tg,
                                        g->gfull, logL, g->d_nrows, B, p->ws.d_err, st));
    if (coarse) {
        const dim3 gz((n_out + 255) / 256, B);
        adj::k_zinterp_adj<float><<<gz, 256, 0, st>>>((const float*)g->gtab, sp.n_z, p->d_zi_row, p->d_zi_w,
                                                      (float*)g->gcoarse, p->n_z_emu, sp.n_k, g->d_nrows);
        NS_CUDA_TRY(cudaGetLastError());
        NS_TRY(launch_split_planes(px, (const float*)g->gcoarse, (float)p->out_sigma, B, n_out, g->Gp[0],
                                   g->rows_pad * plane_pitch(n_out), plane_pitch(n_out), g->d_nrows, st));
    }
    // backward: G_l = (G_{l+1} W_l) (1 - h_l^2), l = L-1 .. 1 (the last in FP32)
    for (int l = L - 1; l >= 1; --l) {
        PlaneEpi e;
        e.mode = l == 1 ? PLN_DTANH32 : PLN_DTANH;
        e.aux = g->Hp[l];
        e.aux_pitch = plane_pitch(p->dims[l]);
        e.aux_stride = g->rows_pad * e.aux_pitch;
        if (l == 1) e.out = g->G1;
        else planes_out(e, g->Gp[(L - l) & 1], p->dims[l]);
        NS_TRY(launch_gemm_planes(px, pw, &g->tmWT[l], &g->tmG[l], e, g->d_nrows, B, p->dims[l], p->dims[l + 1], 0,
                                  p->ws.d_err, st));
    }
    return launch_finish_grad<float>(p, g, g->G1, B, grad, st);
}

}  // namespace gpuns

using namespace gpuns;

namespace {
std::vector<GradState*> g_grad_states;
}  // namespace

// Isotropic Gaussian test likelihood and its gradient at free parameters
// (every parameter of that kind is free).
__global__ void k_gauss_grad(const double* __restrict__ theta, int d, double mu, double sigma,
                             double* __restrict__ logL, double* __restrict__ grad, int B) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= B) return;
    double s = 0.0;
    for (int i = 0; i < d; ++i) {
        const double r = (theta[(size_t)row * d + i] - mu) / sigma;
        s += r * r;
        grad[(size_t)row * d + i] = -r / sigma;
    }
    logL[row] = -0.5 * s - d * log(sigma * 2.5066282746310005024);
}

extern "C" int loglike_grad_batch(const ns_problem* p, const double* theta_dev, int B, double* logL_dev,
                                  double* grad_dev, void* stream) {
    if (!p || B < 0 || B > p->max_batch || (B > 0 && (!theta_dev || !logL_dev || !grad_dev))) return NS_EINVAL;
    if (p->kind != NS_KIND_SHEAR && p->kind != NS_KIND_GAUSS) return NS_ENOTSUP;
    if (B == 0) return NS_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if (p->kind == NS_KIND_GAUSS) {
        if (p->d != p->P) return NS_ENOTSUP;
        k_gauss_grad<<<(B + 127) / 128, 128, 0, st>>>(theta_dev, p->d, p->g_mu, p->g_sigma, logL_dev, grad_dev, B);
        NS_CUDA_TRY(cudaGetLastError());
        return NS_OK;
    }
    GradState* gs = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_grad_mu);
        for (GradState* s : g_grad_states) if (s->p == p) gs = s;
        if (!gs) {
            gs = new GradState();
            const int rc = grad_state_create(p, gs);
            if (rc != NS_OK) {
                grad_state_free(gs);
                return rc;
            }
            g_grad_states.push_back(gs);
        }
    }
    double** out = gs->graphs.d_out;
    const int rows = call_rows(B, p->max_batch);
    return gs->graphs.call(
        rows, st,
        [&] { return launch_free_to_full(p, theta_dev, B, gs->theta_full, gs->d_nrows, out, logL_dev, grad_dev, st); },
        [&](cudaStream_t s) {
            return p->precision == NS_PREC_FP64 ? run_grad_f64(p, gs, rows, OutPtr{out}, OutPtr{out + 1}, s)
                                                : run_grad_planes(p, gs, rows, OutPtr{out}, OutPtr{out + 1}, s);
        });
}

// Called by ns_problem_free: release the gradient state of a problem.
void gpuns_release_grad_state(const ns_problem* p) {
    std::lock_guard<std::mutex> lk(g_grad_mu);
    for (size_t i = 0; i < g_grad_states.size(); ++i) {
        GradState* s = g_grad_states[i];
        if (s->p != p) continue;
        grad_state_free(s);
        g_grad_states.erase(g_grad_states.begin() + i);
        return;
    }
}
