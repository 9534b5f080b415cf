// Likelihood stages on CUDA cores (FP64 / FP32) and the pipeline driver.
//
//   prior transform   Table 1 (uniform, Gaussian via Phi^-1, fixed)
//   emulator          MLP stand-in for CosmoPower (Sec. 2.5): input layer on
//                     CUDA cores, hidden/output layers as tcgen05 GEMMs: BF16
//                     (gemm_tc.cu), FP32 as three bf16 planes (gemm_planes.cu),
//                     FP64 with tanh as six fp16 slices (gemm_slices.cu); FP64
//                     with other activations on CUDA cores here
//   projection.cu     App. A projection (distances, windows, P lookup, Limber,
//                     data vector) and the whitened chi^2.
#include <algorithm>
#include <type_traits>

#include "likelihood.cuh"
#include "tcgen05.cuh"

namespace gpuns {

__global__ void k_set_int(int* p, int v) {
    pdl_begin();
    *p = v;
}

__constant__ double c_glx[4] = {-0.86113631159405257522, -0.33998104358485626480,
                                 0.33998104358485626480, 0.86113631159405257522};
__constant__ double c_glw[4] = {0.34785484513745385737, 0.65214515486254614263,
                                 0.65214515486254614263, 0.34785484513745385737};

// ------------------------------------------------------------ prior transform
__global__ void k_cube_to_theta(const double* __restrict__ cube, int d, int P,
                                const int* __restrict__ kind, const double* __restrict__ pa,
                                const double* __restrict__ pb, const int* __restrict__ free_of_full,
                                double* __restrict__ theta_full, const int* __restrict__ nrows) {
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int f = free_of_full[i];
        double v;
        if (f < 0) {
            v = pa[i];
        } else {
            const double c = cube[(size_t)row * d + f];
            if (kind[i] == NS_PRIOR_UNIFORM) v = pa[i] + (pb[i] - pa[i]) * c;
            else v = pa[i] + pb[i] * normcdfinv(c);
        }
        theta_full[(size_t)row * P + i] = v;
    }
}

__global__ void k_cube_to_free(const double* __restrict__ cube, int d, int P,
                               const int* __restrict__ kind, const double* __restrict__ pa,
                               const double* __restrict__ pb, const int* __restrict__ free_of_full,
                               double* __restrict__ theta, int B, int f32) {
    const int row = blockIdx.x;
    if (row >= B) return;
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int f = free_of_full[i];
        if (f < 0) continue;
        const double c = cube[(size_t)row * d + f];
        theta[(size_t)row * d + f] = (kind[i] == NS_PRIOR_UNIFORM) ? pa[i] + (pb[i] - pa[i]) * c
                                                                   : pa[i] + pb[i] * gauss_quantile(c, f32 != 0);
    }
}

__global__ void k_free_to_full(const double* __restrict__ theta, int d, int P,
                               const double* __restrict__ pa, const int* __restrict__ free_of_full,
                               double* __restrict__ theta_full, int B, int* __restrict__ nrows,
                               double** __restrict__ slots, double* out0, double* out1) {
    const int row = blockIdx.x;
    if (row >= B) return;
    if (row == 0 && threadIdx.x == 0) {
        *nrows = B;
        if (slots) {
            slots[0] = out0;
            slots[1] = out1;
        }
    }
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int f = free_of_full[i];
        theta_full[(size_t)row * P + i] = (f < 0) ? pa[i] : theta[(size_t)row * d + f];
    }
}

// ------------------------------------------------------------ gauss test
__global__ void k_gauss_loglike(const double* __restrict__ theta_full, int P, double mu, double sigma,
                                double* __restrict__ logL, const int* __restrict__ nrows) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= *nrows) return;
    double s = 0.0;
    for (int i = 0; i < P; ++i) {
        const double r = (theta_full[(size_t)row * P + i] - mu) / sigma;
        s += r * r;
    }
    logL[row] = -0.5 * s - P * log(sigma * 2.5066282746310005024);
}

// ------------------------------------------------------------ emulator
// Hidden-layer activation: tanh, or CosmoPower's sigmoid-linear
// f(x) = [g + (1 - g) sigmoid(beta x)] x with one (g, beta) per unit.
template <typename T> __device__ inline T act_tanh(T x);
template <> __device__ inline double act_tanh<double>(double x) { return tanh(x); }
template <> __device__ inline float act_tanh<float>(float x) { return tanhf(x); }
template <typename T> __device__ inline T ex_acc(T x);
template <> __device__ inline double ex_acc<double>(double x) { return exp(x); }
template <> __device__ inline float ex_acc<float>(float x) { return expf(x); }

template <typename T>
struct ActDev {
    int kind;
    const T* g;
    const T* beta;
};

template <typename T>
__device__ __forceinline__ T act_apply(const ActDev<T>& a, int n, T x) {
    if (a.kind == NS_ACT_TANH) return act_tanh<T>(x);
    const T g = a.g[n];
    return (g + (T(1) - g) / (T(1) + ex_acc<T>(-a.beta[n] * x))) * x;
}

// Where the input layer puts h[row][n]: a plain matrix in the next layer's
// type, or the three bf16 planes that hold an FP32 value (gemm_planes.cu).
struct OutF64 {
    double* p;
    __device__ __forceinline__ void put(int row, int n, int N, double v) const { p[(size_t)row * N + n] = v; }
};
struct OutBf16 {
    __nv_bfloat16* p;
    __device__ __forceinline__ void put(int row, int n, int N, float v) const {
        p[(size_t)row * N + n] = __float2bfloat16_rn(v);
    }
};
template <int P>
struct OutPlanes {
    __nv_bfloat16* p;
    long long stride;
    int pitch;
    __device__ __forceinline__ void put(int row, int n, int, float v) const {
        tc::plane_store<P>(v, p + (size_t)row * pitch + n, stride);
    }
};

// Input layer: h = act(W0 x + b0), x = (theta[inputs] - center) / scale.  A
// CTA takes kInRows consecutive rows; thread t owns units t, t + blockDim, ...
// and keeps a unit's bias and K0 (<= KMAX) weights in registers over the CTA's
// rows, so the weights are read once per CTA and the launch has
// ceil(rows / kInRows) CTAs rather than one per (row, 256 units).
constexpr int kInRows = 2;
template <typename T, typename OUT, int KMAX>
__global__ void __launch_bounds__(256)
k_emu_input(const double* __restrict__ theta_full, int P, const int* __restrict__ inputs,
            const double* __restrict__ center, const double* __restrict__ scale,
            const double* __restrict__ inv_scale, int K0,
            const T* __restrict__ W0, const T* __restrict__ b0, ActDev<T> act, int N,
            const OUT out, const int* __restrict__ nrows) {
    // the weights of a thread's first UP units are problem constants: in
    // registers before the dependency wait
    constexpr int UP = sizeof(T) == 4 && KMAX <= 8 ? 4 : 1;
    // FP64 (tanh is ~50 operations on a pipe of two per cycle and SM): the units
    // are spread over gridDim.y CTAs too
    const int n0 = sizeof(T) == 8 ? 256 * blockIdx.y : 0, nstep = sizeof(T) == 8 ? 256 * gridDim.y : blockDim.x;
    T wp[UP][KMAX], bp[UP];
#pragma unroll
    for (int u = 0; u < UP; ++u) {
        const int n = n0 + threadIdx.x + u * blockDim.x;
#pragma unroll
        for (int j = 0; j < KMAX; ++j) wp[u][j] = (n < N && j < K0) ? W0[(size_t)n * K0 + j] : T(0);
        bp[u] = n < N ? b0[n] : T(0);
    }
    pdl_begin();
    const int M = *nrows;
    const int r0 = blockIdx.x * kInRows;
    if (r0 >= M) return;
    const int nr = min(kInRows, M - r0);
    __shared__ T x[kInRows][KMAX];
    for (int i = threadIdx.x; i < nr * K0; i += blockDim.x) {
        const int r = i / K0, j = i - r * K0;
        // FP64 standardisation; reduced-precision emulators multiply by the
        // reciprocal scale (an FP64 divide is a long sequence on GB300's FP64 pipe)
        const double v = theta_full[(size_t)(r0 + r) * P + inputs[j]] - center[j];
        x[r][j] = sizeof(T) == 8 ? (T)(v / scale[j]) : (T)(v * inv_scale[j]);
    }
    __syncthreads();
    auto unit = [&](int n, const T (&w)[KMAX], T bn) {
        for (int r = 0; r < nr; ++r) {
            T acc = bn;
#pragma unroll
            for (int j = 0; j < KMAX; ++j)
                if (j < K0) acc = fma(w[j], x[r][j], acc);
            out.put(r0 + r, n, N, act_apply<T>(act, n, acc));
        }
    };
#pragma unroll
    for (int u = 0; u < UP; ++u) {
        const int n = n0 + threadIdx.x + u * blockDim.x;
        if (n < N) unit(n, wp[u], bp[u]);
    }
    for (int n = n0 + threadIdx.x + UP * nstep; n < N; n += nstep) {
        T w[KMAX];
#pragma unroll
        for (int j = 0; j < KMAX; ++j) w[j] = j < K0 ? W0[(size_t)n * K0 + j] : T(0);
        unit(n, w, b0[n]);
    }
}

// C[M x N] = epi(A[M x K] W[N x K]^T + b).  Threads own an interleaved
// TM x TN sub-tile (rows ty + i*BM/TM, cols tx + j*BN/TN) so shared-memory
// reads and global stores are conflict-free / coalesced.  FP64 problems and
// set-up work (FP32 layers run on the tensor cores, gemm_planes.cu).
//   EPI_ACT: act(acc + b);  EPI_OUT: mu + s (acc + b), s = sig_vec[n] or sigma.
enum { EPI_ACT = 0, EPI_OUT = 1 };

template <typename T, int BM, int BN, int BK, int TM, int TN, int EPI>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
k_gemm_simt(const T* __restrict__ A, const T* __restrict__ W, const T* __restrict__ bias, ActDev<T> act,
            const T* __restrict__ out_mu, const T* __restrict__ sig_vec, T out_sigma, T* __restrict__ C,
            const int* __restrict__ nrows, int N, int K) {
    constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
    const int M = *nrows;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    if (m0 >= M) return;
    __shared__ T As[BK][BM + 1];
    __shared__ T Bs[BK][BN + 1];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
        for (int i = tid; i < BM * BK; i += NT) {
            const int r = i / BK, c = i % BK;
            const int gm = m0 + r, gk = k0 + c;
            As[c][r] = (gm < M && gk < K) ? A[(size_t)gm * K + gk] : T(0);
        }
        for (int i = tid; i < BN * BK; i += NT) {
            const int r = i / BK, c = i % BK;
            const int gn = n0 + r, gk = k0 + c;
            Bs[c][r] = (gn < N && gk < K) ? W[(size_t)gn * K + gk] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[TM], b[TN];
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
            if (gn >= N) continue;
            T v = acc[i][j] + (bias ? bias[gn] : T(0));
            if (EPI == EPI_ACT) v = act_apply<T>(act, gn, v);
            else v = out_mu[gn] + (sig_vec ? sig_vec[gn] : out_sigma) * v;
            C[(size_t)gm * N + gn] = v;
        }
    }
}

// Coarse-z emulator table -> n_z table: out[jz][ik] = sum_q w[jz][q] in[row[jz][q]][ik]
// (Catmull-Rom in z with folded ghosts).  A block takes a share of an
// evaluation's z nodes, threads V columns each (16-byte accesses where rows
// allow); the taps and weights, converted once, sit in shared memory.  375 rows of
// 10 -> 50 nodes: 29 us with a division and four FP64 conversions per entry.
template <typename T, int V>
__global__ void __launch_bounds__(256) k_zinterp(const T* __restrict__ coarse, int nzc, const int* __restrict__ zr,
                                                 const double* __restrict__ zwt, T* __restrict__ fine, int nz, int nk,
                                                 const int* __restrict__ nrows) {
    struct alignas(sizeof(T) * V) Vec { T v[V]; };
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* w = reinterpret_cast<T*>(smem_raw);
    int* tap = reinterpret_cast<int*>(w + 4 * nz);
    for (int i = threadIdx.x; i < 4 * nz; i += 256) {
        w[i] = (T)zwt[i];
        tap[i] = zr[i] * nk;
    }
    pdl_begin();
    const int row = blockIdx.y;
    if (row >= *nrows) return;
    __syncthreads();
    const T* c = coarse + (size_t)row * nzc * nk;
    T* f = fine + (size_t)row * nz * nk;
    const int cols = nk / V, per = min(cols, 256), lines = 256 / per;
    if (threadIdx.x >= per * lines) return;
    const int k0 = threadIdx.x % per;
    for (int jz = blockIdx.x * lines + threadIdx.x / per; jz < nz; jz += gridDim.x * lines)
        for (int k = k0; k < cols; k += per) {
            Vec o;
#pragma unroll
            for (int e = 0; e < V; ++e) o.v[e] = T(0);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const Vec x = *reinterpret_cast<const Vec*>(c + tap[jz * 4 + q] + k * V);
#pragma unroll
                for (int e = 0; e < V; ++e) o.v[e] += w[jz * 4 + q] * x.v[e];
            }
            *reinterpret_cast<Vec*>(f + (size_t)jz * nk + k * V) = o;
        }
}

template <typename T>
static int launch_zinterp(const ns_problem* p, const T* coarse, T* fine, const int* nrows, int grid_rows,
                          cudaStream_t st) {
    constexpr int V = 16 / sizeof(T);
    const ShearParams& sp = p->sp;
    const bool vec = sp.n_k % V == 0;          // rows of 16-byte multiples in cudaMalloc'ed buffers
    const size_t smem = 4 * (size_t)sp.n_z * (sizeof(T) + sizeof(int));
    if (smem > 48 * 1024) {
        auto k = vec ? k_zinterp<T, V> : k_zinterp<T, 1>;
        NS_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    }
    NS_CUDA_TRY(launch_pdl(vec ? k_zinterp<T, V> : k_zinterp<T, 1>, dim3(grid_rows < 304 ? 4 : 2, grid_rows), dim3(256),
                           smem, st, coarse, p->n_z_emu, (const int*)p->d_zi_row, (const double*)p->d_zi_w, fine, sp.n_z,
                           sp.n_k, nrows));
    return NS_OK;
}

static int launch_gemm_simt(const double* A, const double* W, const double* bias, ActDev<double> act, const double* mu,
                            const double* sig_vec, double sigma, double* C, const int* nrows, int grid_rows, int N,
                            int K, int epi, cudaStream_t st) {
    constexpr int BM = 64, BN = 64, BK = 8, TM = 4, TN = 4, NT = (BM / TM) * (BN / TN);
    const dim3 grid((N + BN - 1) / BN, (grid_rows + BM - 1) / BM);
    auto kern = epi == EPI_ACT ? k_gemm_simt<double, BM, BN, BK, TM, TN, EPI_ACT>
                               : k_gemm_simt<double, BM, BN, BK, TM, TN, EPI_OUT>;
    kern<<<grid, NT, 0, st>>>(A, W, bias, act, mu, sig_vec, sigma, C, nrows, N, K);
    NS_CUDA_TRY(cudaGetLastError());
    return NS_OK;
}

// Plain FP64 GEMM C = A W^T (M x N, K inner) on the device, for set-up work
// (the CMB whitening fold); nrows_dev holds M.
int gemm_f64_plain(const double* A, const double* W, double* C, const int* nrows_dev, int M, int N, int K,
                   const double* zeros_n, cudaStream_t st) {
    return launch_gemm_simt(A, W, zeros_n, ActDev<double>{0, nullptr, nullptr}, zeros_n, nullptr,
                                            1.0, C, nrows_dev, M, N, K, EPI_OUT, st);
}

int launch_cube_to_theta(const ns_problem* p, Workspace* ws, const double* cube, int grid_rows,
                         cudaStream_t st) {
    if (grid_rows <= 0) return NS_OK;
    NS_CUDA_TRY(launch_pdl(k_cube_to_theta, dim3(grid_rows), dim3(64), 0, st, cube, p->d, p->P,
                           (const int*)p->d_pkind, (const double*)p->d_pa, (const double*)p->d_pb,
                           (const int*)p->d_free_of_full, ws->theta_full, (const int*)ws->d_nrows));
    return NS_OK;
}

template <typename T>
static ActDev<T> layer_act(const ns_problem* p, int l) {
    ActDev<T> a{p->act, nullptr, nullptr};
    if (p->act == NS_ACT_SIGMOID_LINEAR) {
        a.g = (const T*)p->d_act_g[l];
        a.beta = (const T*)p->d_act_beta[l];
    }
    return a;
}

template <typename T, typename OUT>
static int launch_emu_input(const ns_problem* p, const double* theta_full, const int* nrows, int grid_rows,
                            const ActDev<T>& act, const OUT& out, cudaStream_t st) {
    const int K0 = p->dims[0], H1 = p->dims[1];
    const dim3 g((grid_rows + kInRows - 1) / kInRows, sizeof(T) == 8 ? std::min(8, (H1 + 255) / 256) : 1);
    auto kern = K0 <= 8 ? k_emu_input<T, OUT, 8> : k_emu_input<T, OUT, 32>;
    NS_CUDA_TRY(launch_pdl(kern, g, dim3(256), 0, st, theta_full, p->P, (const int*)p->d_inputs,
                           (const double*)p->d_in_center, (const double*)p->d_in_scale,
                           (const double*)p->d_in_inv_scale, K0, (const T*)p->d_W[0], (const T*)p->d_b[0], act, H1,
                           out, nrows));
    return NS_OK;
}

int launch_emu_input_planes(const ns_problem* p, const double* theta_full, const int* nrows, int grid_rows, int px,
                            __nv_bfloat16* out, long long stride, cudaStream_t st) {
    const ActDev<float> tanh_act{NS_ACT_TANH, nullptr, nullptr};
    const int pitch = plane_pitch(p->dims[1]);
    if (px == 3) return launch_emu_input<float>(p, theta_full, nrows, grid_rows, tanh_act, OutPlanes<3>{out, stride, pitch}, st);
    if (px == 2) return launch_emu_input<float>(p, theta_full, nrows, grid_rows, tanh_act, OutPlanes<2>{out, stride, pitch}, st);
    return NS_EINVAL;
}

// The emulator's last layer: W h + b, de-standardised as mu + s * (.), written to out.
struct Head {
    const void* W;           // FP64 problems
    const CUtensorMap* tmW;  // FP32 heads: three bf16 planes
    const void* bias;
    const void* mu;
    const void* sig_vec;
    double sigma;
    void* out;
    int n_out = 0;           // outputs computed (the first rows of W); 0: all
};

static Head model_head(const ns_problem* p, void* out) {
    const int L = p->n_layers;
    return Head{p->d_W[L - 1], p->tmWp.empty() ? nullptr : &p->tmWp[L - 1], p->d_b[L - 1], p->d_out_mu, p->d_out_sig,
                p->out_sigma, out};
}

bool takes_slices(const ns_problem* p) {
    return std::any_of(p->d_wscale.begin(), p->d_wscale.end(), [](const double* s) { return s != nullptr; });
}

size_t slice_input_bytes(const ns_problem* p, int cap) {
    const size_t rows_pad = ((size_t)cap + 127) / 128 * 128;
    return sizeof(__half) * tc::kSlices * rows_pad * plane_pitch(p->hidden_max);
}

int slice_input_maps(const ns_problem* p, int cap, SliceInput* x) {
    const int rows_pad = ((cap + 127) / 128) * 128;
    x->stride = (long long)rows_pad * plane_pitch(p->hidden_max);
    x->tm.resize(p->n_layers);
    for (int l = 1; l < p->n_layers; ++l)
        for (int i = 0; i < 3; ++i)
            NS_TRY(make_tensor_map_slices(&x->tm[l].m[i], x->slices, rows_pad, p->dims[l], x->stride, 16 << i));
    return NS_OK;
}

int launch_layer_f64(const ns_problem* p, int l, const SliceInput& xs, const double* x, double* out, const int* nrows,
                     int grid_rows, int* err, cudaStream_t st) {
    const bool last = l == p->n_layers - 1;
    const int K = p->dims[l], N = p->dims[l + 1];
    const double *mu = last ? (const double*)p->d_out_mu : nullptr, sigma = last ? p->out_sigma : 0.0;
    if (l >= (int)p->d_wscale.size() || !p->d_wscale[l])
        return launch_gemm_simt(x, (const double*)p->d_W[l], (const double*)p->d_b[l],
                                ActDev<double>{NS_ACT_TANH, nullptr, nullptr}, mu, nullptr, sigma, out, nrows, grid_rows,
                                N, K, last ? EPI_OUT : EPI_ACT, st);
    NS_TRY(launch_slice_rows(x, grid_rows, K, xs.slices, xs.stride, plane_pitch(K), xs.scale, nrows, st));
    SliceEpi e;
    e.tanh = !last;
    e.bias = (const double*)p->d_b[l];
    e.wscale = p->d_wscale[l];
    e.xscale = xs.scale;
    e.mu = mu;
    e.sigma = sigma;
    e.out = out;
    return launch_gemm_slices(&p->tmWs[l], &xs.tm[l], e, nrows, grid_rows, N, K, err, st);
}

// FP64: tanh emulators mostly on the tensor cores, others (CMB: unbounded activations, folded
// heads) on CUDA cores.
static int run_emulator_f64(const ns_problem* p, Workspace* ws, int grid_rows, cudaStream_t st, const Head& hd) {
    const int L = p->n_layers;
    NS_TRY(launch_emu_input<double>(p, ws->theta_full, ws->d_nrows, grid_rows, layer_act<double>(p, 0),
                                    OutF64{(double*)ws->act[0]}, st));
    int cur = 0;
    for (int l = 1; l < L; ++l) {
        const int K = p->dims[l], N = p->dims[l + 1];
        const double* x = (const double*)ws->act[cur];
        if (!p->d_wscale.empty()) {
            NS_TRY(launch_layer_f64(p, l, ws->xs, x, l == L - 1 ? (double*)hd.out : (double*)ws->act[cur ^ 1],
                                    ws->d_nrows, grid_rows, ws->d_err, st));
        } else if (l == L - 1) {
            NS_TRY(launch_gemm_simt(x, (const double*)hd.W, (const double*)hd.bias, ActDev<double>{0, nullptr, nullptr},
                                    (const double*)hd.mu, (const double*)hd.sig_vec, hd.sigma, (double*)hd.out,
                                    ws->d_nrows, grid_rows, hd.n_out ? hd.n_out : N, K, EPI_OUT, st));
        } else {
            NS_TRY(launch_gemm_simt(x, (const double*)p->d_W[l], (const double*)p->d_b[l], layer_act<double>(p, l),
                                    nullptr, nullptr, 0.0, (double*)ws->act[cur ^ 1], ws->d_nrows, grid_rows, N, K,
                                    EPI_ACT, st));
        }
        cur ^= 1;
    }
    return NS_OK;
}

// An FP32 head (FP32 problems: px = 3 planes of activations; BF16 CMB: px = 1).
static int launch_head_f32(const ns_problem* p, Workspace* ws, int grid_rows, int px, const Head& hd, cudaStream_t st) {
    const int L = p->n_layers;
    PlaneEpi e;
    e.mode = PLN_OUT;
    e.bias = (const float*)hd.bias;
    e.mu = (const float*)hd.mu;
    e.sig_vec = (const float*)hd.sig_vec;
    e.sigma = (float)hd.sigma;
    e.out = (float*)hd.out;
    const int N = hd.n_out ? hd.n_out : p->dims[L], K = p->dims[L - 1];
    return launch_gemm_planes(px, 3, hd.tmW, &ws->tmXp[L - 1], e, ws->d_nrows, grid_rows, N, K, plane_split(N, K),
                              ws->d_err, st);
}

// FP32: the input layer on CUDA cores, every further layer as an FP32-accurate
// GEMM on the tensor cores; activations travel as three bf16 planes.
static int run_emulator_f32(const ns_problem* p, Workspace* ws, int grid_rows, cudaStream_t st, const Head& hd) {
    const int L = p->n_layers;
    NS_TRY(launch_emu_input<float>(
        p, ws->theta_full, ws->d_nrows, grid_rows, layer_act<float>(p, 0),
        OutPlanes<3>{(__nv_bfloat16*)ws->act[0], ws->plane_stride, plane_pitch(p->dims[1])}, st));
    int cur = 0;
    for (int l = 1; l + 1 < L; ++l) {
        const ActDev<float> a = layer_act<float>(p, l);
        PlaneEpi e;
        e.mode = p->act == NS_ACT_SIGMOID_LINEAR ? PLN_SIGLIN : PLN_TANH;
        e.bias = (const float*)p->d_b[l];
        e.g = a.g;
        e.beta = a.beta;
        e.planes = (__nv_bfloat16*)ws->act[cur ^ 1];
        e.plane_stride = ws->plane_stride;
        e.pitch = plane_pitch(p->dims[l + 1]);
        NS_TRY(launch_gemm_planes(3, 3, &p->tmWp[l], &ws->tmXp[l], e, ws->d_nrows, grid_rows, p->dims[l + 1],
                                  p->dims[l], plane_split(p->dims[l + 1], p->dims[l]), ws->d_err, st));
        cur ^= 1;
    }
    return launch_head_f32(p, ws, grid_rows, 3, hd, st);
}

static int probe_begin(const StageProbe* pr, int stage, Workspace* ws, cudaStream_t st) {
    if (!pr || pr->stage != stage) return NS_OK;
    NS_CUDA_TRY(cudaMemcpyAsync(pr->h_rows, ws->d_nrows, sizeof(int), cudaMemcpyDeviceToHost, st));
    NS_CUDA_TRY(cudaEventRecordWithFlags(pr->ev0, st, cudaEventRecordExternal));
    return NS_OK;
}
static int probe_end(const StageProbe* pr, int stage, cudaStream_t st) {
    if (!pr || pr->stage != stage) return NS_OK;
    NS_CUDA_TRY(cudaEventRecordWithFlags(pr->ev1, st, cudaEventRecordExternal));
    return NS_OK;
}

// BF16: input layer on CUDA cores, hidden layers as tcgen05 GEMMs with the
// activation in the epilogue.  The last layer: for the shear kind a tcgen05
// GEMM with the de-standardising epilogue into the FP32 table; for the CMB
// kind `hd` with FP32 weights as three bf16 planes (gemm_planes.cu).
static int run_emulator_bf16(const ns_problem* p, Workspace* ws, int grid_rows, cudaStream_t st,
                             const StageProbe* probe, const Head* hd) {
    const int L = p->n_layers;
    int cur = 0, l1 = 1;
    if (p->fused_cs) {
        // input and hidden layers in one clustered kernel; its output is the
        // buffer the per-layer path would leave the last hidden layer in
        NS_TRY(probe_begin(probe, PROBE_EMU_HIDDEN, ws, st));
        NS_TRY(launch_emu_fused(p, ws, grid_rows, st));
        NS_TRY(probe_end(probe, PROBE_EMU_HIDDEN, st));
        cur = (L - 2) & 1;
        l1 = L - 1;
    } else {
        NS_TRY(launch_emu_input<float>(p, ws->theta_full, ws->d_nrows, grid_rows, layer_act<float>(p, 0),
                                       OutBf16{(__nv_bfloat16*)ws->act[0]}, st));
    }
    for (int l = l1; l < L; ++l) {
        const int K = p->dims[l], N = p->dims[l + 1];
        const bool last = (l == L - 1);
        const int stage = last ? PROBE_EMU_OUT : (l == 1 ? PROBE_EMU_HIDDEN : PROBE_NONE);
        NS_TRY(probe_begin(probe, stage, ws, st));
        if (last && hd) {
            NS_TRY(launch_head_f32(p, ws, grid_rows, 1, *hd, st));
        } else if (last && p->tile_n[l] == 128) {
            // the output layer with few rows: features as the MMA's M (one wave of CTAs)
            NS_TRY(launch_gemm_tc_out_swap(&p->tmB[l], &ws->tmX_out, (const float*)p->d_b[l],
                                           (const float*)p->d_out_mu, (float)p->out_sigma, (float*)ws->table,
                                           ws->d_nrows, grid_rows, N, K, ws->d_err, st));
        } else {
            const ActDev<float> a = layer_act<float>(p, l);
            const int epi = last ? TC_EPI_OUT : (p->act == NS_ACT_SIGMOID_LINEAR ? TC_EPI_SIGLIN : TC_EPI_TANH);
            // Hidden tiles are autotuned for at most 384 rows; from 64 CTAs of 64-wide tiles
            // on (four row tiles of a 1024-wide layer) these are the faster ones, reading
            // the activations fewer times (same bits): log-likelihoods of 500 rows
            // 122.5 -> 121.3 us, of 4096 rows 614 -> 591 (128-wide: 589), nested-sampling
            // calls 9.12 -> 8.99 ms; at 375 rows they cost 1 %.
            int tn = p->tile_n[l];
            const CUtensorMap* tmB = &p->tmB[l];
            if (!last && !p->tmB64.empty() && tn < 64 &&
                (long long)((N + 63) / 64) * ((grid_rows + 127) / 128) >= 64) {
                tn = 64;
                tmB = &p->tmB64[l];
            }
            NS_TRY(launch_gemm_tc(&ws->tmA[l], tmB, tn, (const float*)p->d_b[l],
                                  last ? (const float*)p->d_out_mu : a.g, last ? (float)p->out_sigma : 0.f,
                                  last ? ws->table : ws->act[cur ^ 1], ws->d_nrows, grid_rows, N, K, epi,
                                  last ? nullptr : a.beta, ws->d_err, st));
        }
        NS_TRY(probe_end(probe, stage, st));
        cur ^= 1;
    }
    return NS_OK;
}

template <typename T>
__global__ void k_to_double(const T* __restrict__ in, double* __restrict__ out, int n_per_row,
                            const int* __restrict__ nrows) {
    const int row = blockIdx.y;
    if (row >= *nrows) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_per_row; i += gridDim.x * blockDim.x)
        out[(size_t)row * n_per_row + i] = (double)in[(size_t)row * n_per_row + i];
}

// chi^2 = sum_a y_a^2 per row (fixed-order block tree, partials widened to
// FP64), log L = c0 - chi^2 / 2 in FP64.
template <typename T>
__global__ void __launch_bounds__(256) k_rowsq(const T* __restrict__ y, int D, double c0, double* __restrict__ logL,
                                               const int* __restrict__ nrows) {
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    __shared__ double part[256];
    const T* yr = y + (size_t)row * D;
    T s = T(0);
    for (int a = threadIdx.x; a < D; a += 256) s = fma(yr[a], yr[a], s);
    part[threadIdx.x] = (double)s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) logL[row] = c0 - 0.5 * part[0];
}

// Cosmic-variance TT log L per row: c0 - sum_ell (k/2) g(C_ell / d_ell) with
// g(r) = ln r + 1/r - 1 = log1p(u) - u / (1 + u), u = r - 1 (no cancellation
// near the peak); partial sums widened to FP64 in a fixed-order block tree.
template <typename T>
__global__ void __launch_bounds__(256) k_cmb_tt(const T* __restrict__ C, int n_tt, int ld, const T* __restrict__ dobs,
                                                const T* __restrict__ halfk, double c0, double* __restrict__ logL,
                                                const int* __restrict__ nrows) {
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    __shared__ double part[256];
    const T* c = C + (size_t)row * ld;
    T s = T(0);
    for (int i = threadIdx.x; i < n_tt; i += 256) {
        const T u = c[i] / dobs[i] - T(1);
        s += halfk[i] * (log1p(u) - u / (T(1) + u));
    }
    part[threadIdx.x] = (double)s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) logL[row] = c0 - part[0];
}

int run_emulator_only(const ns_problem* p, Workspace* ws, int grid_rows, double* out, cudaStream_t st) {
    if (grid_rows <= 0) return NS_OK;
    const int n_out = p->dims.back();
    dim3 g((n_out + 255) / 256, grid_rows);
    const Head hd = model_head(p, ws->table);
    if (p->precision == NS_PREC_FP64) {
        NS_TRY(run_emulator_f64(p, ws, grid_rows, st, hd));
        k_to_double<double><<<g, 256, 0, st>>>((const double*)ws->table, out, n_out, ws->d_nrows);
    } else {
        if (p->precision == NS_PREC_FP32) NS_TRY(run_emulator_f32(p, ws, grid_rows, st, hd));
        else NS_TRY(run_emulator_bf16(p, ws, grid_rows, st, nullptr, p->kind == NS_KIND_CMB ? &hd : nullptr));
        k_to_double<float><<<g, 256, 0, st>>>((const float*)ws->table, out, n_out, ws->d_nrows);
    }
    NS_CUDA_TRY(cudaGetLastError());
    return NS_OK;
}

// CMB kind (Sec. 3.1 problem, dense covariance): FOLD runs the hidden layers
// and the folded head y = c' - W' h, then chi^2 = |y|^2; LITERAL (FP64) forms
// r = (d - mu) - sigma (W h + b) with the same head kernel and whitens it by
// L^-1; model_out gets the de-standardised emulator output.
static int run_cmb(const ns_problem* p, Workspace* ws, int grid_rows, double* logL_out, double* model_out,
                   cudaStream_t st, const StageProbe* probe) {
    const int D = p->D;
    if (model_out) return run_emulator_only(p, ws, grid_rows, model_out, st);
    const bool f64 = p->precision == NS_PREC_FP64;
    if (p->cmb_form == NS_CMB_TT_CV) {
        // the TT block of the head only (the first n_tt outputs), then the sums
        Head hd = model_head(p, ws->table);
        hd.n_out = p->n_tt;
        if (f64) NS_TRY(run_emulator_f64(p, ws, grid_rows, st, hd));
        else if (p->precision == NS_PREC_FP32) NS_TRY(run_emulator_f32(p, ws, grid_rows, st, hd));
        else NS_TRY(run_emulator_bf16(p, ws, grid_rows, st, probe, &hd));
        NS_TRY(probe_begin(probe, PROBE_CHI2, ws, st));
        auto tt = [&](auto kern, auto* tab) -> int {
            using T = std::remove_pointer_t<decltype(tab)>;
            NS_CUDA_TRY(launch_pdl(kern, dim3(grid_rows), dim3(256), 0, st, (const T*)tab, p->n_tt, p->n_tt,
                                   (const T*)p->d_tt_obs, (const T*)p->d_tt_halfk, p->c0, logL_out,
                                   (const int*)ws->d_nrows));
            return NS_OK;
        };
        if (f64) NS_TRY(tt(k_cmb_tt<double>, (double*)ws->table));
        else NS_TRY(tt(k_cmb_tt<float>, (float*)ws->table));
        return probe_end(probe, PROBE_CHI2, st);
    }
    if (p->cmb_solve == NS_SOLVE_LITERAL) {
        const int L = p->n_layers;
        const Head hd{p->d_W[L - 1], nullptr, p->d_b[L - 1], p->d_lit_mu, p->d_lit_sig, 0.0, ws->resid};
        NS_TRY(run_emulator_f64(p, ws, grid_rows, st, hd));
        NS_TRY(probe_begin(probe, PROBE_CHI2, ws, st));
        NS_TRY((launch_chi2<double, double>((const double*)ws->resid, D, p->d_LinvT64, p->c0, logL_out,
                                            ws->d_nrows, grid_rows, st)));
        return probe_end(probe, PROBE_CHI2, st);
    }
    const Head hd{p->d_Wfold, &p->tmWfold, p->d_zeroD, p->d_cfold, nullptr, -1.0, ws->table};
    if (f64) NS_TRY(run_emulator_f64(p, ws, grid_rows, st, hd));
    else if (p->precision == NS_PREC_FP32) NS_TRY(run_emulator_f32(p, ws, grid_rows, st, hd));
    else NS_TRY(run_emulator_bf16(p, ws, grid_rows, st, probe, &hd));
    NS_TRY(probe_begin(probe, PROBE_CHI2, ws, st));
    if (f64)
        NS_CUDA_TRY(launch_pdl(k_rowsq<double>, dim3(grid_rows), dim3(256), 0, st, (const double*)ws->table, D, p->c0,
                               logL_out, (const int*)ws->d_nrows));
    else
        NS_CUDA_TRY(launch_pdl(k_rowsq<float>, dim3(grid_rows), dim3(256), 0, st, (const float*)ws->table, D, p->c0,
                               logL_out, (const int*)ws->d_nrows));
    return probe_end(probe, PROBE_CHI2, st);
}

int run_likelihood(const ns_problem* p, Workspace* ws, int grid_rows, double* logL_out, double* model_out,
                   cudaStream_t st, const StageProbe* probe) {
    if (grid_rows <= 0) return NS_OK;
    if (p->kind == NS_KIND_GAUSS) {
        k_gauss_loglike<<<(grid_rows + 127) / 128, 128, 0, st>>>(ws->theta_full, p->P, p->g_mu, p->g_sigma,
                                                                 logL_out, ws->d_nrows);
        NS_CUDA_TRY(cudaGetLastError());
        return NS_OK;
    }
    if (p->kind == NS_KIND_CMB) return run_cmb(p, ws, grid_rows, logL_out, model_out, st, probe);
    const ShearParams& sp = p->sp;
    const bool coarse = p->n_z_emu != sp.n_z;
    const bool f64 = p->precision == NS_PREC_FP64;
    // fork: the windows stage needs only theta, so it runs on the side stream
    // while the emulator runs on `st`; the Limber stage joins both.
    NS_CUDA_TRY(cudaEventRecord(ws->ev_fork, st));
    NS_CUDA_TRY(cudaStreamWaitEvent(ws->side, ws->ev_fork, 0));
    NS_TRY(probe_begin(probe, PROBE_WINDOWS, ws, ws->side));
    if (f64) NS_TRY(launch_windows<double, false>(sp, ws->theta_full, (double*)ws->win, ws->d_nrows, grid_rows, ws->side, (double*)ws->win_nodes));
    else if (p->precision == NS_PREC_FP32)
        NS_TRY(launch_windows<float, false>(sp, ws->theta_full, (float*)ws->win, ws->d_nrows, grid_rows, ws->side));
    else NS_TRY(launch_windows<float, true>(sp, ws->theta_full, (float*)ws->win, ws->d_nrows, grid_rows, ws->side));
    NS_TRY(probe_end(probe, PROBE_WINDOWS, ws->side));
    NS_CUDA_TRY(cudaEventRecord(ws->ev_join, ws->side));
    if (f64) {
        NS_TRY(run_emulator_f64(p, ws, grid_rows, st, model_head(p, ws->table)));
        const double* tab = (const double*)ws->table;
        if (coarse) {
            NS_TRY(launch_zinterp<double>(p, tab, (double*)ws->table_fine, ws->d_nrows, grid_rows, st));
            tab = (const double*)ws->table_fine;
        }
        NS_CUDA_TRY(cudaStreamWaitEvent(st, ws->ev_join, 0));
        NS_TRY(launch_limber<double, false>(sp, ws->theta_full, tab, (const double*)ws->win, (double*)ws->resid,
                                            model_out, ws->d_nrows, grid_rows, ws->d_err, st));
        if (model_out) return NS_OK;
        return launch_chi2<double, double>((const double*)ws->resid, sp.D, p->d_LinvT64, p->c0, logL_out,
                                           ws->d_nrows, grid_rows, st, true);
    }
    // FP32 stages (FP32 / BF16 / BF16_F64CHI2)
    if (p->precision == NS_PREC_FP32) NS_TRY(run_emulator_f32(p, ws, grid_rows, st, model_head(p, ws->table)));
    else NS_TRY(run_emulator_bf16(p, ws, grid_rows, st, probe, nullptr));
    const float* tab = (const float*)ws->table;
    if (coarse) {
        NS_TRY(launch_zinterp<float>(p, tab, (float*)ws->table_fine, ws->d_nrows, grid_rows, st));
        tab = (const float*)ws->table_fine;
    }
    NS_CUDA_TRY(cudaStreamWaitEvent(st, ws->ev_join, 0));
    NS_TRY(probe_begin(probe, PROBE_PROJECTION, ws, st));
    if (p->precision == NS_PREC_FP32)
        NS_TRY(launch_limber<float, false>(sp, ws->theta_full, tab, (const float*)ws->win, (float*)ws->resid,
                                           model_out, ws->d_nrows, grid_rows, ws->d_err, st));
    else
        NS_TRY(launch_limber<float, true>(sp, ws->theta_full, tab, (const float*)ws->win, (float*)ws->resid,
                                          model_out, ws->d_nrows, grid_rows, ws->d_err, st));
    NS_TRY(probe_end(probe, PROBE_PROJECTION, st));
    if (model_out) return NS_OK;
    NS_TRY(probe_begin(probe, PROBE_CHI2, ws, st));
    if (p->precision == NS_PREC_BF16_F64CHI2)
        NS_TRY(launch_chi2<float, double>((const float*)ws->resid, sp.D, p->d_LinvT64, p->c0, logL_out,
                                          ws->d_nrows, grid_rows, st, true));
    else
        NS_TRY(launch_chi2<float, float>((const float*)ws->resid, sp.D, p->d_LinvT32, p->c0, logL_out,
                                         ws->d_nrows, grid_rows, st, true));
    return probe_end(probe, PROBE_CHI2, st);
}

}  // namespace gpuns

// host helpers used by the C API in problem.cu
namespace gpuns {
int launch_cube_to_free(const ns_problem* p, const double* cube, int B, double* theta, cudaStream_t st) {
    // the sampler's prior transform: FP32 quantile for reduced-precision problems
    k_cube_to_free<<<B, 64, 0, st>>>(cube, p->d, p->P, p->d_pkind, p->d_pa, p->d_pb, p->d_free_of_full, theta, B,
                                     p->precision != NS_PREC_FP64 ? 1 : 0);
    NS_CUDA_TRY(cudaGetLastError());
    return NS_OK;
}
int launch_free_to_full(const ns_problem* p, const double* theta, int B, double* theta_full, int* nrows,
                        double** slots, double* out0, double* out1, cudaStream_t st) {
    k_free_to_full<<<B, 64, 0, st>>>(theta, p->d, p->P, p->d_pa, p->d_free_of_full, theta_full, B, nrows, slots, out0,
                                     out1);
    NS_CUDA_TRY(cudaGetLastError());
    return NS_OK;
}
}  // namespace gpuns

namespace gpuns {
int launch_zinterp_generic(const ns_problem* p, const void* coarse, void* fine, const int* nrows, int grid_rows, int elt,
                           cudaStream_t st) {
    if (elt == 8) return launch_zinterp<double>(p, (const double*)coarse, (double*)fine, nrows, grid_rows, st);
    return launch_zinterp<float>(p, (const float*)coarse, (float*)fine, nrows, grid_rows, st);
}
}  // namespace gpuns
