// FP64 GEMMs on the fp16 tensor path (tcgen05), for the layers of FP64 tanh
// emulators:  out[r][f] = epi( sum_k X[r][k] W[f][k] ).
//
// GB300 runs FP64 at two FMAs per cycle and SM (1.26 TFLOP/s), a thousandth of
// its fp16 tensor rate.  An operand is therefore held in fixed point, every row of W and
// every row of activations scaled to |v| <= 1 by a power of two of its own, as
// six 9-bit slices:  v = sum_i q_i 2^-(8 + 9 i),  |q_i| <= 256 an integer, the
// rest at most 2^-54.  Products q_i q_j are integers of at most 2^16; the 26 slice pairs
// with i + j <= 6 are kept, one FP32 accumulator in TMEM for each sum i + j, whose
// i + j + 1 pairs over 64 k stay within FP32's 24 bits up to i + j = 3: the tensor core
// adds them exactly.  (Those of i + j = 4, 5 and 6 could leave the 24 bits if every slice of
// every operand were near its largest value with equal signs, in a total near 64; a unit of
// theirs is 2^-52 and less.)  Every 64 k the epilogue warps add the seven accumulators to two
// 64-bit integers per element (in registers, while the next MMAs run in the second TMEM
// buffer), and one FP64 expression at the end joins them.
//
// Error, of sum |w| |h|, in an emulation of the digits (rms, normal weights): K = 1024,
// activations of order 1 6.9e-18, of order 1e-3 or 1e-6 1.1e-17, spread over four decades
// 1.5e-17; K = 64 2.6e-17, 3.9e-17, 5.5e-17; an FP64 FMA chain 4.7e-17 to 8.9e-17 throughout.  Without
// the activations' scale order 1e-6 gave 7.7e-12; without the pairs of i + j = 6 (2^-54 of the
// scale each) K = 64 1.5e-16 where the chain has 5.5e-17.
//
// Layers whose weights do not suit that (k_unfit_rows) keep the FP64 FMA kernel.
//
// The ranks of a cluster take whole groups of 64 k, so that every group is added
// alike in every split: a row's bits do not depend on its batch.
//
// Tiles: 128 features (the MMA's M) x 16, 32 or 64 rows, seven accumulators each
// (twice in TMEM for up to 32 rows).  Slots of 32 k hold every slice of both
// operands (60 KB for 32 rows, 64-byte swizzle, three slots).  Few tiles are spread over clusters of S CTAs along k,
// whose integer partial tiles are added exactly through cluster shared memory.
// A NaN operand (its leading slice is NaN) and a timeout give NaN.
//
// Measured on the 39-d emulator: 64 rows 5.80 ms of FP64 FMA tiles -> 0.22 ms (a
// hidden layer 27 us, its slices 7, the output layer 107), beside the windows' 130; the call
// 6367 -> 571 us.  With 21 pairs, 128 k per sum and activations sliced in the epilogues,
// which lost bits, it took 559.  Error of its standardised outputs against 113-bit
// arithmetic rms 2.34e-15, largest 9.2e-15 (FMA chain 2.41e-15 and 1.04e-14: the mean
// table's own rounding is most of both).
//
// Warps 0-7 (0-15 for 64 rows): drain and epilogue; then one warp for the copies
// and one for TMEM and MMAs.  Waits are bounded as in gemm_planes.cu.
#include <algorithm>

#include "likelihood.cuh"
#include "tcgen05.cuh"

namespace gpuns {
namespace slc {

using namespace tc;

constexpr int NS = kSlices;                      // slices of an operand
constexpr int NSUM = NS + 1;                     // sums i + j kept
constexpr int SBK = 32;                          // k per slot: 64 bytes of fp16
constexpr int W_SUB = 128 * SBK * 2;
constexpr int STAGES = 3;
constexpr int CHUNK = 2;                         // slots per TMEM accumulation: 64 k
// Stands for NaN in a rank's sum: ordinary sums, of either sign, stay below 2^50, so a
// total of one to eight markers and ordinary sums lies above kNaN / 2, any other below.
constexpr long long kNaN = 1ll << 58;

template <int BR>                                // rows per tile
struct CfgL {
    static constexpr int X_SUB = BR * SBK * 2;
    static constexpr int STAGE_BYTES = NS * (W_SUB + X_SUB);
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 + 256;
    static constexpr int NBUF = BR <= 32 ? 2 : 1;    // sets of accumulators that fit TMEM
    static constexpr uint32_t TMEM_COLS = BR == 16 ? 256 : 512;
    static constexpr int EPI_WARPS = BR == 64 ? 16 : 8, THREADS = 32 * (EPI_WARPS + 2);
    static constexpr int HC = BR / (EPI_WARPS / 4);  // rows per epilogue warp
    static_assert(STAGES * STAGE_BYTES >= 128 * BR * 16, "the partial tile reuses the ring");
    static_assert(NBUF * NSUM * BR <= (int)TMEM_COLS, "accumulators in TMEM");
};

// K-major tile of 64-byte rows, 64-byte swizzle (8-row groups of 512 bytes).
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | (uint64_t)1 << 16 | (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)4 << 61;
}

// kind::f16, D = F32, A = B = F16, K-major, M = 128, N = BR
template <int BR>
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(BR >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

template <int BR>
__global__ void __launch_bounds__(CfgL<BR>::THREADS, 1)
k_gemm_slices(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const SliceEpi e,
              const int* __restrict__ nrows, int N, int K, int* __restrict__ err) {
    using C = CfgL<BR>;
    constexpr int STAGE_BYTES = C::STAGE_BYTES, X_SUB = C::X_SUB, EPI_WARPS = C::EPI_WARPS, HC = C::HC, NBUF = C::NBUF;
    constexpr int W_LOAD = EPI_WARPS, W_MMA = EPI_WARPS + 1;   // the other two warps
    pdl_begin();
    const int M = *nrows;
    const int S = gridDim.x, rank = blockIdx.x;
    const int f0 = blockIdx.y * 128, r0 = blockIdx.z * BR;
    if (r0 >= M) return;                         // every CTA of the cluster has these rows

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - raw);
    const uint32_t bar0 = base + STAGES * STAGE_BYTES;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto acc_full = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + STAGES * STAGE_BYTES + 8 * (2 * STAGES + 4));
    __shared__ int s_fail;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        s_fail = 0;
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), EPI_WARPS); }
        mbar_init_fence();
    }
    if (warp == W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tmem_slot)), "r"(C::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const int nk = (K + SBK - 1) / SBK;
    const int nc = (nk + CHUNK - 1) / CHUNK;     // at least one for every rank (launch_gemm_slices)
    const int kb0 = nc * rank / S * CHUNK, n_it = min(nk, nc * (rank + 1) / S * CHUNK) - kb0;
    const int n_chunk = (n_it + CHUNK - 1) / CHUNK;

    uint32_t nan = 0;                            // elements whose leading accumulator is NaN
    long long hi[HC], lo[HC];                    // sums of i + j = 0..2 and 3..6, in units of the last of each
#pragma unroll
    for (int j = 0; j < HC; ++j) { hi[j] = 0; lo[j] = 0; }
    if (warp == W_LOAD) {
        if (lane == 0) {
            int issued = 0;
            for (int it = 0; it < n_it; ++it) {
                const int s = it % STAGES;
                if (it >= STAGES && !mbar_wait(empty_bar(s), ((it / STAGES) & 1) ^ 1)) { s_fail = 1; break; }
                const uint32_t sa = base + s * STAGE_BYTES;
                mbar_expect_tx(full_bar(s), STAGE_BYTES);
                tma_load_3d(sa, &tmW, full_bar(s), (kb0 + it) * SBK, f0, 0);
                tma_load_3d(sa + NS * W_SUB, &tmX, full_bar(s), (kb0 + it) * SBK, r0, 0);
                ++issued;
            }
            // no copy may still be in flight when the CTA leaves
            for (int it = max(0, issued - STAGES); it < issued; ++it)
                if (!mbar_wait(full_bar(it % STAGES), (it / STAGES) & 1)) s_fail = 1;
        }
        __syncwarp();
    } else if (warp == W_MMA) {
        if (lane == 0) {
            bool ok = true;
            for (int it = 0; it < n_it && ok; ++it) {
                const int s = it % STAGES, c = it / CHUNK, b = c % NBUF, in = it % CHUNK;
                if (in == 0 && c >= NBUF) ok = mbar_wait(acc_empty(b), ((c / NBUF) & 1) ^ 1);
                ok = ok && mbar_wait(full_bar(s), (it / STAGES) & 1);
                if (!ok) { s_fail = 1; break; }
                fence_after();
                const uint32_t sw = base + s * STAGE_BYTES, sx = sw + NS * W_SUB;
#pragma unroll
                for (int i = 0; i < NS; ++i)
#pragma unroll
                    for (int j = 0; j < NS && i + j < NSUM; ++j) {
                        const uint64_t dw = desc64(sw + i * W_SUB), dx = desc64(sx + j * X_SUB);
#pragma unroll
                        for (int kk = 0; kk < SBK / 16; ++kk)
                            mma_bf16(tmem + (uint32_t)((b * NSUM + i + j) * BR), dw + 2 * kk, dx + 2 * kk, kIdesc<BR>,
                                     in != 0 || !(i == 0 || j == NS - 1) || kk != 0);
                    }
                mma_commit(empty_bar(s));
                if (in == CHUNK - 1 || it == n_it - 1) mma_commit(acc_full(b));
            }
        }
        __syncwarp();
    } else {
        const uint32_t addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * HC);
        for (int c = 0; c < n_chunk; ++c) {
            const int b = c % NBUF;
            if (!mbar_wait(acc_full(b), (c / NBUF) & 1)) { s_fail = 1; break; }
            fence_after();
            __syncwarp();
#pragma unroll
            for (int s = 0; s < NSUM; ++s) {
                float v[HC];
                tmem_ld<HC>(addr + (uint32_t)((b * NSUM + s) * BR), v);
                if (s == 0) {
#pragma unroll
                    for (int j = 0; j < HC; ++j) nan |= (uint32_t)(v[j] != v[j]) << j;
                }
                const long long unit = 1ll << (9 * (s < 3 ? 2 - s : NSUM - 1 - s));
#pragma unroll
                for (int j = 0; j < HC; ++j) (s < 3 ? hi[j] : lo[j]) += (long long)__float2int_rn(v[j]) * unit;
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty(b));
        }
        __syncwarp();
    }

    const int f = f0 + (tid & 127);
    const bool fv = tid < 32 * EPI_WARPS && f < N;
    double bias = 0, mu = 0, ws = 0;
    if (fv) {
        bias = e.bias[f];
        ws = e.wscale[f];
        if (!e.tanh) mu = e.mu[f];
    }
    auto finish = [&](int rl, long long h, long long l) {
        const int row = r0 + rl;
        if (!fv || row >= M) return;
        double v = fma((double)l, 0x1p-70, (double)h * 0x1p-34) * ws * e.xscale[row] + bias;
        if (h >= kNaN / 2) v = NAN;
        e.out[(size_t)row * N + f] = e.tanh ? tanh(v) : mu + e.sigma * v;
    };
    __syncthreads();                             // the ring's last copies have landed
    const bool failed = s_fail != 0;
    if (failed) nan = 0xffffffffu;
    long long* red = reinterpret_cast<long long*>(gbase);       // hi, then lo: BR x 128 each
    if (warp < EPI_WARPS) {
#pragma unroll
        for (int j = 0; j < HC; ++j) {
            const int at = ((warp >> 2) * HC + j) * 128 + (tid & 127);
            red[at] = (nan >> j) & 1 ? kNaN : hi[j];
            red[BR * 128 + at] = lo[j];
        }
    }
    if (S == 1) __syncthreads();
    else cluster_sync_all();
    if (warp < EPI_WARPS) {
        const int end = min(BR * (rank + 1) / S, M - r0);
#pragma unroll 1
        for (int rl = BR * rank / S + (tid >> 7); rl < end; rl += EPI_WARPS / 4) {
            const int at = rl * 128 + (tid & 127);
            long long h = red[at], l = red[BR * 128 + at];
            for (int q = 1; q < S; ++q) {        // integers: any order
                const uint32_t peer = (uint32_t)((rank + q) % S);
                h += ld_cluster_s64(mapa_u32(base + 8u * (uint32_t)at, peer));
                l += ld_cluster_s64(mapa_u32(base + 8u * (uint32_t)(BR * 128 + at), peer));
            }
            finish(rl, h, l);
        }
    }
    if (S > 1) cluster_sync_all();               // peers have read this CTA's partial tile
    if (failed && tid == 0 && err) atomicOr(err, NS_BIT_TIMEOUT);
    fence_before();
    __syncthreads();
    if (warp == W_MMA) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(C::TMEM_COLS) : "memory");
    }
}

// Slices and power-of-two scale of every row of a matrix (rows x K): the weights once, the
// activations before each layer.  A block per row, bound by its two dependent passes (64
// rows of 1024: 7 us); the row's maximum takes all of a layer's CTAs, so that the layer's
// epilogue cannot slice.
__global__ void __launch_bounds__(256) k_slice_rows(const double* __restrict__ W, int K, __half* __restrict__ out,
                                                    long long stride, int pitch, double* __restrict__ scale,
                                                    const int* __restrict__ nrows) {
    pdl_begin();
    if (nrows && (int)blockIdx.x >= *nrows) return;
    __shared__ double red[8];
    const double* w = W + (size_t)blockIdx.x * K;
    double m = 0;
    for (int k = threadIdx.x; k < K; k += 256) m = fmax(m, fabs(w[k]));
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int i = 0; i < 8; ++i) m = fmax(m, red[i]);
    // the least power of two that is no smaller than the row's largest |v|
    int ex = 0;
    if (m > 0 && frexp(m, &ex) == 0.5) --ex;
    ex = max(ex, -900);                          // 1 / scale stays finite
    const double s = scalbn(1.0, -ex);
    for (int k = threadIdx.x; k < K; k += 256) slice_store(w[k] * s, out + (size_t)blockIdx.x * pitch + k, stride);
    if (threadIdx.x == 0) scale[blockIdx.x] = scalbn(1.0, ex);
}

// Whether a row's largest |w| is infinite, beyond the exponents that the scales are made
// for, or more than sqrt(K) / 2 times the row's mean |w|.  The digits' error is near
// 0.45 max |w| / mean |w| max |h| / mean |h| / sqrt(K) of an FMA chain's (emulated for K = 64
// to 2048), so that with the activations of a normal distribution, max |h| near 4 mean |h|, it
// stays below the chain's up to here; a weight of 10^6 times the others against a tiny
// activation made it 10^5 times as large.  Normal weights reach 4 to 5 times their mean: K of
// some hundred and more takes the slices.  A NaN does not count: it marks its sums.
__global__ void __launch_bounds__(256) k_unfit_rows(const double* __restrict__ W, int K, int* __restrict__ unfit) {
    __shared__ double red[2][8];
    const double* w = W + (size_t)blockIdx.x * K;
    double m = 0, s = 0;
    for (int k = threadIdx.x; k < K; k += 256) {
        const double a = fmax(0.0, fabs(w[k]));
        m = fmax(m, a);
        s += a;
    }
    m = warp_max(m);
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = m; red[1][threadIdx.x >> 5] = s; }
    __syncthreads();
    if (threadIdx.x) return;
    for (int i = 1; i < 8; ++i) { m = fmax(m, red[0][i]); s += red[1][i]; }
    if (m > 0 && !(m > 0x1p-400 && m < 0x1p400 && m * sqrt((double)K) <= 0.5 * s)) atomicOr(unfit, 1);
}

}  // namespace slc

template <int BR>
static int launch_slices_t(const CUtensorMap* tmW, const CUtensorMap* tmX, const SliceEpi& e, const int* nrows,
                           int grid_rows, int N, int K, int S, int* err, cudaStream_t st) {
    using C = slc::CfgL<BR>;
    static bool attr = false;
    if (!attr) {
        NS_CUDA_TRY(cudaFuncSetAttribute(slc::k_gemm_slices<BR>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
        attr = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, (N + 127) / 128, (grid_rows + BR - 1) / BR);
    cfg.blockDim = dim3(C::THREADS);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute a[2];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    a[1].id = cudaLaunchAttributeClusterDimension;
    a[1].val.clusterDim.x = S;
    a[1].val.clusterDim.y = 1;
    a[1].val.clusterDim.z = 1;
    cfg.attrs = a;
    cfg.numAttrs = 2;
    NS_CUDA_TRY(cudaLaunchKernelEx(&cfg, slc::k_gemm_slices<BR>, *tmW, *tmX, e, nrows, N, K, err));
    return NS_OK;
}

int launch_gemm_slices(const CUtensorMap* tmW, const SliceMapX* tmX, const SliceEpi& e, const int* nrows,
                       int grid_rows, int N, int K, int* err, cudaStream_t st) {
    if (grid_rows <= 0) return NS_OK;
    // Rows per tile and K split by the cycles of the SM that ends last (every group of
    // 64 k is added alike in each, so the choice does not change a bit).  A slot is 52 MMAs of ~65 cycles
    // each up to N = 64; the epilogue's FP64 runs at two operations per cycle (tanh
    // ~75 per element, the output 6); 64-row tiles have one set of accumulators and
    // wait for each drain; clusters of 8 (4) find room on about 96 (128) SMs.  Timed
    // against all twelve (rows per tile, split) at 1 to 256 rows of 1024 -> 1024,
    // 1024 -> 2000 and 1024 -> 10000: the choice is the fastest or within 3 % (64 rows,
    // whole emulator: 242 us with 16 / 4 hidden and 64 / 4 output tiles; 64 / 1 output 251,
    // 32 / 1 267; 16 / 2 hidden 285, 64 / 4 312).
    const int nk = (K + slc::SBK - 1) / slc::SBK, mt = (N + 127) / 128;
    int best_br = 32, best_s = 1;
    double best = 1e300;
    for (int br : {16, 32, 64})
        for (int s : {1, 2, 4, 8}) {
            if (s > 1 && nk < slc::CHUNK * s) continue;
            const int sms = s == 8 ? 96 : s == 4 ? 128 : 152, slots = (nk + s - 1) / s;
            const long long ctas = (long long)mt * ((grid_rows + br - 1) / br) * s;
            const double t = (double)((ctas + sms - 1) / sms) *
                             (3000.0 + 3400.0 * slots + (br == 64 ? 3000.0 * (slots / slc::CHUNK) : 0.0) +
                              64.0 * br / s * (e.tanh ? 75 : 6) + (s > 1 ? 2500.0 : 0.0));
            if (t < 0.97 * best) { best = t; best_br = br; best_s = s; }
        }
    switch (best_br) {
        case 16: return launch_slices_t<16>(tmW, &tmX->m[0], e, nrows, grid_rows, N, K, best_s, err, st);
        case 32: return launch_slices_t<32>(tmW, &tmX->m[1], e, nrows, grid_rows, N, K, best_s, err, st);
        default: return launch_slices_t<64>(tmW, &tmX->m[2], e, nrows, grid_rows, N, K, best_s, err, st);
    }
}

int slices_fit(const double* W, int rows, int K, int* d_flag, bool* fit) {
    int unfit = K > 65536;                       // 64-bit sums hold K < 2^17
    if (!unfit) {
        NS_CUDA_TRY(cudaMemset(d_flag, 0, sizeof(int)));
        slc::k_unfit_rows<<<rows, 256>>>(W, K, d_flag);
        NS_CUDA_TRY(cudaGetLastError());
        NS_CUDA_TRY(cudaMemcpy(&unfit, d_flag, sizeof(int), cudaMemcpyDeviceToHost));
    }
    *fit = !unfit;
    return NS_OK;
}

int launch_slice_rows(const double* in, int rows, int K, __half* out, long long stride, int pitch, double* scale,
                      const int* nrows, cudaStream_t st) {
    NS_CUDA_TRY(launch_pdl(slc::k_slice_rows, dim3(rows), dim3(256), 0, st, in, K, out, stride, pitch, scale, nrows));
    return NS_OK;
}

}  // namespace gpuns
