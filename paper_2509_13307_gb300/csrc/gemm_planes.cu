// GEMMs of FP32 accuracy on the bf16 tensor path (tcgen05), for the FP32
// emulators, the FP32 heads of the CMB problem and the adjoint.
//
//   out[r][f] = epi( sum_k X[r][k] W[f][k] ),   X, W given as bf16 planes
//
// An FP32 value is the exact sum of three bf16 values (8 significant bits
// each): hi = bf16(v), mid = bf16(v - hi), lo = v - hi - mid.  (An infinite operand makes
// NaN, not the infinity of an FP32 sum.)  X comes in PX
// planes and W in PW planes (3: an FP32 operand, 2: the leading 16 bits, 1: a
// bf16 operand), and the products of plane pairs with p + q <= 2 are summed;
// the three pairs left out of 3 x 3 are below 2^-25 of the full product.
//
// Accumulation.  The tensor core adds the products of one instruction to the
// FP32 accumulator with less than round-to-nearest care, so long chains lose
// accuracy.  Each 64-deep k-block is therefore summed in TMEM by itself,
// small plane products first, and the epilogue warps add the block sums in
// FP32 registers (round to nearest) while the next block's MMAs run in the
// second TMEM buffer.  (BF16 gradients, two planes of 16 bits on bf16 weights,
// are far from that limit: one accumulator for all of K, leading plane first.)
//
// Tiles.  The MMA's M is 128 features (rows of W), its N is BR rows of X, so
// few rows waste no tensor work; BR = 32, 64, 128, or 256 where two ring slots
// of that size fit (two planes of X beside one of W: 4096-row gradients).  When the (feature, row)
// tiles are fewer than the SMs the k-blocks are split over a cluster of S
// CTAs; each leaves its FP32 partial tile in shared memory and rank q adds
// the S partials of its share of the rows in rank order (deterministic) and
// applies the epilogue.  plane_tiling picks BR and S.
//
// Warps 0-7 drain TMEM and run the epilogue (warp w: features 32 (w % 4) ..,
// half w / 4 of the tile's rows), warp 8 loads (one TMA copy per operand and
// slot brings every plane), warp 9 owns TMEM and issues the MMAs.  Every wait
// is bounded: a timeout records NS_BIT_TIMEOUT and the CTA still meets its
// cluster, waits for its own copies in flight and frees TMEM.
//
// Bound: the tensor core (six MMAs per plane block: 80 GFLOP for 500 rows of
// the 39-d emulator, 42 us at the measured peak) for many rows, the copies and
// the fixed cost of a launch for few.  Against the FP32 FMA GEMM it replaced
// (128 x 128 tiles, 32 CTAs per hidden layer at 500 rows): log-likelihoods of
// 500 rows of the 39-d problem 2082 -> 247 us (221 with the stages around the
// layers of today), of 250 rows of the dense CMB problem 814 -> 65 us, of 333
// rows of its TT form with BF16 hidden layers 200 -> 48 us.  500 FP32 rows: a
// hidden layer 17 us, the output layer 87 us with the tensor pipe active 44 % of
// its cycles; 4096 rows of a BF16 gradient: 43 and 280 us forward, 57 and 191
// backward.  Sending the tile through shared memory to one rolled epilogue loop,
// instead of an epilogue unrolled over the registers, took the 500-row call from
// 275 to 247 us.  Error of the 39-d emulator's table against FP64 over 500 rows:
// rms 8.90e-8 dex, largest 4.8e-7 (FMA chain: 9.01e-8 and 5.2e-7).
#include <algorithm>

#include "likelihood.cuh"
#include "tcgen05.cuh"

namespace gpuns {
namespace tc {

template <int PX, int PW, int BR>
struct CfgP {
    static constexpr int W_SUB = 128 * BK * 2, X_SUB = BR * BK * 2;   // one plane's k-block
    static constexpr int W_BYTES = PW * W_SUB;
    static constexpr int STAGE_BYTES = W_BYTES + PX * X_SUB;
    static constexpr int FIT = (192 * 1024) / STAGE_BYTES;
    static constexpr int STAGES = FIT > 4 ? 4 : FIT;
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/;
    static constexpr uint32_t TMEM_COLS = 2 * BR;
    static_assert(STAGES >= 2, "two slots");
    static_assert(STAGES * STAGE_BYTES >= 128 * BR * 4, "the partial tile reuses the ring");
};

// 256-row tiles where two slots of them fit
template <int PX, int PW> constexpr bool kPlaneRows256 = 2 * 128 * (128 * PW + 256 * PX) <= 192 * 1024;

constexpr int kPlaneEpiWarps = 8, kPlaneThreads = 32 * (kPlaneEpiWarps + 2);

template <int PX, int PW, int BR>
__global__ void __launch_bounds__(kPlaneThreads, 1)
k_gemm_planes(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const PlaneEpi e,
              const int* __restrict__ nrows, int N, int K, int* __restrict__ err) {
    using C = CfgP<PX, PW, BR>;
    constexpr bool CHAIN = PX == 2;                  // all of K in one accumulator
    constexpr int HC = BR / 2;                       // rows per epilogue warp
    pdl_begin();
    const int M = *nrows;
    const int S = gridDim.x, rank = blockIdx.x;      // the cluster is the whole x extent
    const int f0 = blockIdx.y * 128, r0 = blockIdx.z * BR;
    if (r0 >= M) return;                             // every CTA of the cluster has these rows

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - raw);
    const uint32_t bar0 = base + C::STAGES * C::STAGE_BYTES;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (C::STAGES + s); };
    auto acc_full = [&](int b) { return bar0 + 8u * (2 * C::STAGES + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (2 * C::STAGES + 2 + b); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + C::STAGES * C::STAGE_BYTES + 8 * (2 * C::STAGES + 4));
    __shared__ int s_fail;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        s_fail = 0;
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), kPlaneEpiWarps); }
        mbar_init_fence();
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tmem_slot)), "r"(C::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const int nk = (K + BK - 1) / BK;
    const int kb0 = (int)((long long)nk * rank / S), n_it = (int)((long long)nk * (rank + 1) / S) - kb0;

    float acc[HC];
#pragma unroll
    for (int j = 0; j < HC; ++j) acc[j] = 0.f;
    if (warp == 8) {
        if (lane == 0) {
            int issued = 0;
            for (int it = 0; it < n_it; ++it) {
                const int s = it % C::STAGES;
                if (it >= C::STAGES && !mbar_wait(empty_bar(s), ((it / C::STAGES) & 1) ^ 1)) { s_fail = 1; break; }
                const uint32_t sa = base + s * C::STAGE_BYTES;
                mbar_expect_tx(full_bar(s), C::STAGE_BYTES);
                tma_load_3d(sa, &tmW, full_bar(s), (kb0 + it) * BK, f0, 0);
                tma_load_3d(sa + C::W_BYTES, &tmX, full_bar(s), (kb0 + it) * BK, r0, 0);
                ++issued;
            }
            // no copy may still be in flight when the CTA leaves
            for (int it = max(0, issued - C::STAGES); it < issued; ++it)
                if (!mbar_wait(full_bar(it % C::STAGES), (it / C::STAGES) & 1)) s_fail = 1;
        }
        __syncwarp();
    } else if (warp == 9) {
        if (lane == 0) {
            constexpr uint32_t idesc = instr_desc<BR>();
            for (int it = 0; it < n_it; ++it) {
                const int s = it % C::STAGES, b = it & 1;
                if (!CHAIN && it >= 2 && !mbar_wait(acc_empty(b), ((it >> 1) & 1) ^ 1)) { s_fail = 1; break; }
                if (!mbar_wait(full_bar(s), (it / C::STAGES) & 1)) { s_fail = 1; break; }
                fence_after();
                const uint32_t sa = base + s * C::STAGE_BYTES, sx = sa + C::W_BYTES;
                if constexpr (CHAIN) {
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
#pragma unroll
                        for (int q = 0; q < PX; ++q)
                            mma_bf16(tmem, smem_desc(sa) + 2 * kk, smem_desc(sx + q * C::X_SUB) + 2 * kk, idesc,
                                     (it | kk | q) != 0);
                    mma_commit(empty_bar(s));
                    if (it == n_it - 1) mma_commit(acc_full(0));
                    continue;
                }
                const uint32_t d = tmem + (uint32_t)(b * BR);
                uint32_t accumulate = 0;
                // plane pairs in ascending order of size: p + q = 2, 1, 0
#pragma unroll
                for (int sum = 2; sum >= 0; --sum)
#pragma unroll
                    for (int q = PX - 1; q >= 0; --q) {
                        const int p = sum - q;
                        if (p < 0 || p >= PW) continue;
                        const uint64_t dw = smem_desc(sa + p * C::W_SUB);
                        const uint64_t dx = smem_desc(sx + q * C::X_SUB);
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            mma_bf16(d, dw + 2 * kk, dx + 2 * kk, idesc, accumulate);
                            accumulate = 1;
                        }
                    }
                mma_commit(empty_bar(s));
                mma_commit(acc_full(b));
            }
        }
        __syncwarp();
    } else {
        const uint32_t addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * HC);
        constexpr int CW = HC < 32 ? HC : 32;
        for (int it = 0; it < (CHAIN ? 1 : n_it); ++it) {
            const int b = it & 1;
            if (!mbar_wait(acc_full(b), (it >> 1) & 1)) { s_fail = 1; break; }
            fence_after();
            __syncwarp();
#pragma unroll
            for (int c = 0; c < HC / CW; ++c) {
                float v[CW];
                tmem_ld<CW>(addr + b * BR + c * CW, v);
#pragma unroll
                for (int j = 0; j < CW; ++j) acc[c * CW + j] += v[j];
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty(b));
        }
        __syncwarp();
    }

    // epilogue of one element; a thread's feature is fixed
    const int f = f0 + (tid & 127);
    const bool fv = tid < 256 && f < N;
    float bias = 0.f, mu = 0.f, sg = 0.f, g = 0.f, beta = 0.f;
    if (fv) {
        if (e.bias) bias = __ldg(e.bias + f);
        if (e.mode == PLN_OUT) {
            mu = __ldg(e.mu + f);
            sg = e.sig_vec ? __ldg(e.sig_vec + f) : e.sigma;
        } else if (e.mode == PLN_SIGLIN) {
            g = __ldg(e.g + f);
            beta = __ldg(e.beta + f);
        }
    }
    // h of row rl for the backward epilogues (loaded ahead of their use)
    const bool dtanh = e.mode == PLN_DTANH || e.mode == PLN_DTANH32;
    auto h_of = [&](int rl) {
        float h = 0.f;
        if (dtanh && fv && r0 + rl < M) {
#pragma unroll
            for (int p = PX - 1; p >= 0; --p)
                h += __bfloat162float(e.aux[p * e.aux_stride + (size_t)(r0 + rl) * e.aux_pitch + f]);
        }
        return h;
    };
    auto finish = [&](int rl, float v, float h) {
        const int row = r0 + rl;
        if (!fv || row >= M) return;
        if (e.mode == PLN_OUT) {
            e.out[(size_t)row * N + f] = mu + sg * (v + bias);
            return;
        }
        if (e.mode == PLN_TANH) v = tanhf(v + bias);
        else if (e.mode == PLN_SIGLIN) {
            v += bias;
            v = (g + (1.f - g) / (1.f + expf(-beta * v))) * v;
        } else {
            v *= 1.f - h * h;
            if (e.mode == PLN_DTANH32) {
                e.out[(size_t)row * N + f] = v;
                return;
            }
        }
        if constexpr (PX > 1) plane_store<PX>(v, e.planes + (size_t)row * e.pitch + f, e.plane_stride);
    };
    __syncthreads();                                 // the ring's last copies have landed
    const bool failed = s_fail != 0;
    if (failed) {
#pragma unroll
        for (int j = 0; j < HC; ++j) acc[j] = NAN;
    }
    // the (partial) tile goes through shared memory, so that one rolled loop
    // applies the epilogue: rows of all 128 features, 256 threads to two rows
    float* red = reinterpret_cast<float*>(gbase);
    if (warp < kPlaneEpiWarps) {
#pragma unroll
        for (int j = 0; j < HC; ++j) red[((warp >> 2) * HC + j) * 128 + (tid & 127)] = acc[j];
    }
    if (S == 1) {
        __syncthreads();
        if (warp < kPlaneEpiWarps) {
            // four rows at a time: the backward epilogues' loads of h overlap
            const int hi = min(BR, M - r0);
#pragma unroll 1
            for (int rl = tid >> 7; rl < hi; rl += 8) {
                float h[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) h[q] = h_of(rl + 2 * q);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (rl + 2 * q < hi) finish(rl + 2 * q, red[(rl + 2 * q) * 128 + (tid & 127)], h[q]);
            }
        }
    } else {
        cluster_sync_all();
        if (warp < kPlaneEpiWarps) {
            const int hi = min(BR * (rank + 1) / S, M - r0);
            const uint32_t off = base + 4u * (uint32_t)(tid & 127);
#pragma unroll 1
            for (int rl = BR * rank / S + (tid >> 7); rl < hi; rl += 2) {
                float v = 0.f;
#pragma unroll 4
                for (int q = 0; q < S; ++q) v += ld_cluster_f32(mapa_u32(off + 512u * (uint32_t)rl, (uint32_t)q));
                finish(rl, v, h_of(rl));
            }
        }
        cluster_sync_all();                          // peers have read this CTA's partial tile
    }
    if (failed && tid == 0 && err) atomicOr(err, NS_BIT_TIMEOUT);
    fence_before();
    __syncthreads();
    if (warp == 9) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(C::TMEM_COLS) : "memory");
    }
}

template <int PX, int PW, int BR>
static int launch_planes_t(const CUtensorMap* tmW, const CUtensorMap* tmX, const PlaneEpi& e, const int* nrows,
                           int grid_rows, int N, int K, int S, int* err, cudaStream_t st) {
    using CF = CfgP<PX, PW, BR>;
    static bool attr = false;
    if (!attr) {
        NS_CUDA_TRY(cudaFuncSetAttribute(k_gemm_planes<PX, PW, BR>, cudaFuncAttributeMaxDynamicSharedMemorySize, CF::SMEM));
        attr = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, (N + 127) / 128, (grid_rows + BR - 1) / BR);
    cfg.blockDim = dim3(kPlaneThreads);
    cfg.dynamicSmemBytes = CF::SMEM;
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
    NS_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_gemm_planes<PX, PW, BR>, *tmW, *tmX, e, nrows, N, K, err));
    return NS_OK;
}

template <int PX, int PW>
static int launch_planes_p(const CUtensorMap* tmW, const PlaneMapX* tmX, const PlaneEpi& e, const int* nrows,
                           int grid_rows, int N, int K, PlaneTiling t, int* err, cudaStream_t st) {
    switch (t.br) {
        case 32: return launch_planes_t<PX, PW, 32>(tmW, &tmX->m[0], e, nrows, grid_rows, N, K, t.split, err, st);
        case 64: return launch_planes_t<PX, PW, 64>(tmW, &tmX->m[1], e, nrows, grid_rows, N, K, t.split, err, st);
        case 128: return launch_planes_t<PX, PW, 128>(tmW, &tmX->m[2], e, nrows, grid_rows, N, K, t.split, err, st);
        case 256:
            if constexpr (kPlaneRows256<PX, PW>)
                return launch_planes_t<PX, PW, 256>(tmW, &tmX->m[3], e, nrows, grid_rows, N, K, t.split, err, st);
            return NS_EINVAL;
        default: return NS_EINVAL;
    }
}

// planes[p][r][c] = plane p of s * in[r][c] (row pitch `pitch`).  A thread takes
// four columns when rows and pitch keep 16-byte loads and 8-byte stores aligned.
template <int P, int V>
__global__ void __launch_bounds__(256) k_split_planes(const float* __restrict__ in, float s, int rows, int cols,
                                                      __nv_bfloat16* __restrict__ planes, long long stride, int pitch,
                                                      const int* __restrict__ nrows) {
    pdl_begin();
    const int n = nrows ? min(rows, *nrows) : rows;
    const int c = (blockIdx.x * 256 + threadIdx.x) * V;
    if (c >= cols) return;
    for (int r = blockIdx.y; r < n; r += gridDim.y) {
        __align__(16) float v[V];
        if constexpr (V == 4) *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(in + (size_t)r * cols + c);
        else v[0] = in[(size_t)r * cols + c];
#pragma unroll
        for (int j = 0; j < V; ++j) v[j] *= s;
        __nv_bfloat16* o = planes + (size_t)r * pitch + c;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            __align__(8) __nv_bfloat16 q[V];
#pragma unroll
            for (int j = 0; j < V; ++j) q[j] = plane_take(p, v[j]);
            if constexpr (V == 4) *reinterpret_cast<uint2*>(o + p * stride) = *reinterpret_cast<const uint2*>(q);
            else o[p * stride] = q[0];
        }
    }
}

}  // namespace tc

// Rows per tile and K split (unless given) of one launch, by the cycles of the SM that ends
// last.  A k-block costs its MMAs (N / 2 cycles each, or the shared-memory
// reads of both operands) or its copies (54 B per cycle and SM with every SM
// loading, 450 cycles at least); a CTA adds 2500 for set-up and the first
// copies and 25 per row of epilogue; a split adds the exchange of the partial
// tiles.  One CTA fits an SM; clusters of 8 (4) find room on about 96 (128) of
// the 152 SMs, as GPCs do not hold whole multiples.  The constants are fitted
// to timed sweeps of every (BR, S) for 1 to 1000 rows of the 1024 -> 1024 ->
// 10000 and 512 -> 512 -> 2507 layers: the choice is the fastest of the 12 or
// within 7 % of it everywhere (1024 -> 1024, emulator at 64 rows: 90 us with
// the chosen 64 / 8, 101 with 32 / 8, 130 with 64 / 1, 181 with 128 / 1).
PlaneTiling plane_tiling(int rows, int N, int K, int px, int pw, int split) {
    int prod = 0;
    for (int p = 0; p < pw; ++p)
        for (int q = 0; q < px; ++q) prod += p + q <= 2;
    const int nk = (K + tc::BK - 1) / tc::BK, mt = (N + 127) / 128;
    PlaneTiling best{128, std::max(split, 1)};
    double best_t = 1e300;
    for (int br : {32, 64, 128, 256})
        for (int s : {1, 2, 4, 8}) {
            if (s > nk || (split && s != split) || (br == 256 && 256 * (128 * pw + 256 * px) > 192 * 1024)) continue;
            const double mma = prod * 4.0 * std::max(br / 2.0, (128 + br) / 4.0);
            const double load = std::max(450.0, 128.0 * (128 * pw + br * px) / 54.0);
            const int sms = s == 8 ? 96 : s == 4 ? 128 : 152;
            const long long ctas = (long long)mt * ((rows + br - 1) / br) * s;
            const double waves = (double)((ctas + sms - 1) / sms);
            const double t = waves * (2500.0 + ((nk + s - 1) / s) * std::max(mma, load) + 25.0 * br / s +
                                      (s > 1 ? 2500.0 + 10.0 * br : 0.0));
            if (t < 0.97 * best_t) { best_t = t; best = PlaneTiling{br, s}; }
        }
    return best;
}

// The K split of a likelihood's layer, by its shape alone: a row's log L must not
// depend on the batch it comes in (the shards of a run evaluate their own
// chains), and the split fixes the order of the sums.  Four ways while that
// leaves a chip of SMs to the row tiles: on 1024 -> 1024 within 5 % of the best split
// at 1 to 1000 rows.
int plane_split(int N, int K) {
    const int mt = (N + 127) / 128, nk = (K + tc::BK - 1) / tc::BK;
    return mt <= 8 && nk >= 4 ? 4 : mt <= 16 && nk >= 2 ? 2 : 1;
}

int launch_gemm_planes(int px, int pw, const CUtensorMap* tmW, const PlaneMapX* tmX, const PlaneEpi& e,
                       const int* nrows, int grid_rows, int N, int K, int split, int* err, cudaStream_t st) {
    if (grid_rows <= 0) return NS_OK;
    const PlaneTiling t = plane_tiling(grid_rows, N, K, px, pw, split);
    if (px == 3 && pw == 3) return tc::launch_planes_p<3, 3>(tmW, tmX, e, nrows, grid_rows, N, K, t, err, st);
    if (px == 2 && pw == 1) return tc::launch_planes_p<2, 1>(tmW, tmX, e, nrows, grid_rows, N, K, t, err, st);
    if (px == 1 && pw == 3) return tc::launch_planes_p<1, 3>(tmW, tmX, e, nrows, grid_rows, N, K, t, err, st);
    return NS_EINVAL;
}

int launch_split_planes(int planes, const float* in, float s, int rows, int cols, __nv_bfloat16* out, long long stride,
                        int pitch, const int* nrows, cudaStream_t st) {
    if (rows <= 0 || cols <= 0) return NS_OK;
    const bool vec = cols % 4 == 0 && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0 &&
                     pitch % 4 == 0 && stride % 4 == 0;
    const int per = vec ? 1024 : 256;
    const dim3 g((cols + per - 1) / per, std::min(rows, 16384));
    auto kern = planes == 3 ? (vec ? tc::k_split_planes<3, 4> : tc::k_split_planes<3, 1>)
                            : (vec ? tc::k_split_planes<2, 4> : tc::k_split_planes<2, 1>);
    if (planes != 2 && planes != 3) return NS_EINVAL;
    NS_CUDA_TRY(launch_pdl(kern, g, dim3(256), 0, st, in, s, rows, cols, out, stride, pitch, nrows));
    return NS_OK;
}

}  // namespace gpuns
