// Adjoint of the shear projection: from the emulator table and theta
// to log L, d log L / d table and d log L / d theta (emulator inputs' share
// through the emulator excluded).  The forward stages are the likelihood's own
// kernels (projection.cu), with the Limber sums kept; the reverse stages are
//
//   k_chi2_adj     y = L^-1 r, log L, g_m = L^-T y; g_C = g_m (1+m_i)(1+m_j);
//                  gradients of the biases and the noise templates
//   k_limber_nodes per node and multipole: g_P = sum_p g_C V_i V_j;
//                  g_V_i += g_C V_j P; g_v = ln 10 P g_P; d v / d ln k (Catmull-Rom
//                  derivative) gives g_ln chi
//   k_limber_adj   g_v spread over the 16 table taps of each node and multipole
//   k_table_adj    the table gradient: the warps' partial rows summed in order,
//                  ghost rows and columns folded back
//   k_windows_adj  windows (Eq. 5-6: the exclusive suffix sums transpose to
//                  exclusive prefix sums of their adjoints), n(z) normalisation
//                  and D_z shifts, growth (suffix sums of g_ln D through the
//                  trapezoid segments), distances (suffix sums of g_chi onto
//                  each Gauss-Legendre interval, then d E^2 / d(Omega_m, w0,
//                  wa) at every quadrature point), and the scalars Omega_m =
//                  (omega_b + omega_cdm)/h^2, c/H0 = c/(100 h), gamma(w0, wa)
//
// No stage uses atomics, so gradients repeat bit for bit.
//
// Bound: FP32 instruction issue and the latencies behind it (16 to 28 warps per
// SM).  The one-kernel form it replaced kept 250 KB of intermediates per evaluation
// in global memory and added 16 atomics per (node, multipole) to the table
// gradient.  Whole BF16 gradient calls of the 39-d problem: 4096 rows 9978 -> 3290
// us, 64 rows 608 -> 300 us.  Per 4096 evaluations (BF16 problem): k_limber_adj 705
// us, k_limber_nodes 539, k_windows_adj 521, k_chi2_adj 150, k_table_adj 155.
#include <algorithm>
#include <vector>

#include "likelihood.cuh"
#include "projection_adj.cuh"
#include "tcgen05.cuh"

namespace gpuns {
namespace adj {

// 4-point Gauss-Legendre weights as compile-time constants of the kernel's type
// (no double -> float conversions at run time).
template <typename T> __device__ __forceinline__ T glw(int g) {
    return (g == 0 || g == 3) ? T(0.34785484513745385737) : T(0.65214515486254614263);
}

template <typename T> __device__ __forceinline__ const T* pick(const double* d, const float* f);
template <> __device__ __forceinline__ const double* pick<double>(const double* d, const float*) { return d; }
template <> __device__ __forceinline__ const float* pick<float>(const double*, const float* f) { return f; }
template <typename T> __device__ __forceinline__ T pick_s(double d, float f);
template <> __device__ __forceinline__ double pick_s<double>(double d, float) { return d; }
template <> __device__ __forceinline__ float pick_s<float>(double, float f) { return f; }

template <typename T> __device__ __forceinline__ T ex(T x);
template <> __device__ __forceinline__ double ex<double>(double x) { return exp(x); }
template <> __device__ __forceinline__ float ex<float>(float x) { return expf(x); }
template <typename T> __device__ __forceinline__ T lg(T x);
template <> __device__ __forceinline__ double lg<double>(double x) { return log(x); }
template <> __device__ __forceinline__ float lg<float>(float x) { return logf(x); }
// 1 / sqrt: FP32 takes one Newton step on the SFU value
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }
__device__ __forceinline__ float rsq(float x) {
    const float y = rsqrtf(x);
    return fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);
}
// 10^v and its FP32 form on exp2
__device__ __forceinline__ double p10(double v) { return exp(v * kLn10); }
__device__ __forceinline__ float p10(float v) { return exp2f(v * 3.32192809488736234787f); }

// ------------------------------------------------------------------ chi^2
// RB rows per block: each entry of L^-1 read serves RB rows, whose values lie
// beside one another in shared memory.  A thread takes V neighbouring columns (one
// 16-byte load) of one of `parts` shares of the reduction range, a short chain of
// L2 latencies (64 rows, D = 300: one thread per column 119 us, so 23 us with a cold L2).
constexpr int kChiThreads = 960, kChiSeg = 16;
template <typename T> constexpr int kChiV = 16 / sizeof(T);

// Shares of the reduction range: what the threads allow, whatever the rows per block, so
// that a row's sums have one order in every batch.
__host__ __device__ inline int chi2_adj_parts(int D, int v) {
    const int p = kChiThreads / ((D + v - 1) / v);
    return p < 1 ? 1 : p;
}
__host__ __device__ inline size_t chi2_adj_elems(int D, int v, int nb, int np, int nt, int rb) {
    return (size_t)rb * ((2 + chi2_adj_parts(D, v)) * (size_t)((D + v - 1) / v * v) + nb + np + kChiSeg * (size_t)nt);
}

template <typename T, int RB>
__global__ void __launch_bounds__(kChiThreads)
k_chi2_adj(const ShearParams sp, const double* __restrict__ theta_full, const T* __restrict__ resid,
           const T* __restrict__ C, const T* __restrict__ LinvT, const T* __restrict__ Linv, double c0,
           T* __restrict__ gC, double* __restrict__ gfull, const OutPtr logL, const int* __restrict__ nrows) {
    pdl_begin();
    const int M = *nrows, r0 = blockIdx.x * RB;
    if (r0 >= M) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int V = kChiV<T>;
    const int D = sp.D, P = sp.n_params, nb = sp.nb, n_ell = sp.n_ell, nt = sp.n_tmpl, np = sp.n_pairs;
    const int groups = (D + V - 1) / V, Dv = groups * V, parts = chi2_adj_parts(D, V);
    T* r = reinterpret_cast<T*>(smem_raw);     // Dv x RB, later g_m
    T* y = r + Dv * RB;                        // Dv x RB
    T* part = y + Dv * RB;                     // parts x Dv x RB
    T* th = part + (size_t)parts * Dv * RB;    // RB x nb: 1 + m_i
    T* S = th + RB * nb;                       // np x RB: sum_ell g_m C
    T* tp = S + np * RB;                       // kChiSeg x RB x nt partial template sums
    __shared__ int pi[16], pj[16];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid < np) { pi[tid] = sp.pi[tid]; pj[tid] = sp.pj[tid]; }
    for (int i = tid; i < RB * D; i += kChiThreads) {
        const int j = i / D, a = i - j * D;
        r[a * RB + j] = r0 + j < M ? resid[(size_t)(r0 + j) * D + a] : T(0);
    }
    for (int i = tid; i < RB * nb; i += kChiThreads) {
        const int j = i / nb;
        th[i] = r0 + j < M ? T(1) + (T)theta_full[(size_t)(r0 + j) * P + 11 + nb + i % nb] : T(0);
    }
    __syncthreads();
    // part[seg][a][j] = share seg of sum_b A[b][a] x[b][j]; lower: b <= a, else b >= a (A is zero elsewhere)
    const bool vec = D % V == 0;
    auto columns = [&](const T* A, const T* x, bool lower) {
        for (int i = tid; i < groups * parts; i += kChiThreads) {
            const int seg = i / groups, a = V * (i - seg * groups);
            const int lo = lower ? 0 : a, hi = lower ? min(D, a + V) : D;
            const int b0 = lo + (hi - lo) * seg / parts, b1 = lo + (hi - lo) * (seg + 1) / parts;
            T acc[V][RB];
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int j = 0; j < RB; ++j) acc[v][j] = T(0);
#pragma unroll 8
            for (int b = b0; b < b1; ++b) {
                struct alignas(16) { T v[V]; } l;
                if (vec) l = *reinterpret_cast<const decltype(l)*>(A + (size_t)b * D + a);
                else
#pragma unroll
                    for (int v = 0; v < V; ++v) l.v[v] = a + v < D ? A[(size_t)b * D + a + v] : T(0);
#pragma unroll
                for (int v = 0; v < V; ++v)
#pragma unroll
                    for (int j = 0; j < RB; ++j) acc[v][j] = fma(l.v[v], x[b * RB + j], acc[v][j]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int j = 0; j < RB; ++j) part[((size_t)seg * Dv + a + v) * RB + j] = acc[v][j];
        }
        __syncthreads();
    };
    auto join = [&](int i) {                   // i = a * RB + j
        T s = T(0);
        for (int q = 0; q < parts; ++q) s += part[(size_t)q * Dv * RB + i];
        return s;
    };
    columns(LinvT, r, true);
    for (int i = tid; i < D * RB; i += kChiThreads) y[i] = join(i);
    __syncthreads();
    static_assert(kChiThreads / 32 >= RB, "a warp per row");
    if (wid < RB && r0 + wid < M) {            // chi^2 of a row by one warp
        T sq = T(0);
        for (int a = lane; a < D; a += 32) sq = fma(y[a * RB + wid], y[a * RB + wid], sq);
        sq = warp_sum(sq);
        if (lane == 0) logL.get()[r0 + wid] = c0 - 0.5 * (double)sq;
    }
    // g_m = L^-T y: (g_m)_a = sum_{b >= a} (L^-1)[b][a] y_b
    columns(Linv, y, false);
    for (int i = tid; i < D * RB; i += kChiThreads) {
        const int a = i / RB, j = i % RB, p = a / n_ell;
        const T g = join(i);
        r[i] = g;
        if (r0 + j < M) gC[(size_t)(r0 + j) * D + a] = g * th[j * nb + pi[p]] * th[j * nb + pj[p]];
    }
    __syncthreads();
    for (int q = tid; q < np * RB; q += kChiThreads) {
        const int p = q / RB, j = q % RB;
        T s = T(0);
        if (r0 + j < M)
#pragma unroll 4
            for (int e = 0; e < n_ell; ++e) s = fma(r[(p * n_ell + e) * RB + j], C[(size_t)(r0 + j) * D + p * n_ell + e], s);
        S[q] = s;
    }
    if (wid < kChiSeg) {   // templates: warp w sums its share of the data vector, lanes over templates
        const T* tm = pick<T>(sp.tmpl, sp.tmpl_f);
        const int lo = D * wid / kChiSeg, hi = D * (wid + 1) / kChiSeg;
        for (int t = lane; t < nt; t += 32) {
            T acc[RB];
#pragma unroll
            for (int j = 0; j < RB; ++j) acc[j] = T(0);
#pragma unroll 8
            for (int a = lo; a < hi; ++a) {
                const T g = tm[(size_t)a * nt + t];
#pragma unroll
                for (int j = 0; j < RB; ++j) acc[j] = fma(g, r[a * RB + j], acc[j]);
            }
#pragma unroll
            for (int j = 0; j < RB; ++j) tp[(wid * RB + j) * nt + t] = acc[j];
        }
    }
    __syncthreads();
    for (int q = tid; q < RB * P; q += kChiThreads) {
        const int j = q / P, i = q % P - (11 + nb);
        if (r0 + j >= M) continue;
        T v = T(0);
        if (i >= 0 && i < nb) {
            for (int p = 0; p < np; ++p) {
                if (pi[p] == i) v = fma(S[p * RB + j], th[j * nb + pj[p]], v);
                if (pj[p] == i) v = fma(S[p * RB + j], th[j * nb + pi[p]], v);
            }
        } else if (i >= nb) {
            for (int w = 0; w < kChiSeg; ++w) v += tp[(w * RB + j) * nt + i - nb];
        }
        gfull[(size_t)(r0 + j) * P + q % P] = (double)v;
    }
}

// ------------------------------------------------------------------ Limber
// Entry (r, c) of the table padded by one ghost row and column on every side
// (linear extrapolation), rows 0 .. n_z + 1, columns 0 .. n_k + 1.
template <typename T>
__device__ __forceinline__ T padded_row(const T* t, int n_k, int c) {
    if (c == 0) return T(2) * t[0] - t[1];
    if (c == n_k + 1) return T(2) * t[n_k - 1] - t[n_k - 2];
    return t[c - 1];
}
template <typename T>
__device__ __forceinline__ T padded(const T* t, int n_z, int n_k, int r, int c) {
    if (r >= 1 && r <= n_z && c >= 1 && c <= n_k) return t[(size_t)(r - 1) * n_k + c - 1];
    if (r == 0) return T(2) * padded_row(t, n_k, c) - padded_row(t + n_k, n_k, c);
    if (r == n_z + 1)
        return T(2) * padded_row(t + (size_t)(n_z - 1) * n_k, n_k, c) - padded_row(t + (size_t)(n_z - 2) * n_k, n_k, c);
    return padded_row(t + (size_t)(r - 1) * n_k, n_k, c);
}

// Pairs of values: packed FP32x2 instructions for float, two FMAs for double.
template <typename T> struct P2;
template <> struct P2<float> {
    float2 v;
    __device__ __forceinline__ P2() {}
    __device__ __forceinline__ P2(float x, float y) : v(make_float2(x, y)) {}
    static __device__ __forceinline__ P2 mul(P2 a, P2 b) { P2 r; r.v = __fmul2_rn(a.v, b.v); return r; }
    static __device__ __forceinline__ P2 fma(P2 a, P2 b, P2 c) { P2 r; r.v = __ffma2_rn(a.v, b.v, c.v); return r; }
    static __device__ __forceinline__ P2 add(P2 a, P2 b) { P2 r; r.v = __fadd2_rn(a.v, b.v); return r; }
};
template <> struct P2<double> {
    double2 v;
    __device__ __forceinline__ P2() {}
    __device__ __forceinline__ P2(double x, double y) : v(make_double2(x, y)) {}
    static __device__ __forceinline__ P2 mul(P2 a, P2 b) { return P2(a.v.x * b.v.x, a.v.y * b.v.y); }
    static __device__ __forceinline__ P2 fma(P2 a, P2 b, P2 c) {
        return P2(::fma(a.v.x, b.v.x, c.v.x), ::fma(a.v.y, b.v.y, c.v.y));
    }
    static __device__ __forceinline__ P2 add(P2 a, P2 b) { return P2(a.v.x + b.v.x, a.v.y + b.v.y); }
};
// four z-taps of a table column
template <typename T> struct alignas(16) Z4 {
    P2<T> a, b;
    __device__ __forceinline__ T operator[](int i) const { return i == 0 ? a.v.x : i == 1 ? a.v.y : i == 2 ? b.v.x : b.v.y; }
};

// Reverse of the Limber sums, node by node: one lane per chi node, its windows and
// their gradients in registers, two multipoles at a time as the halves of packed
// values; g_C, the same for every lane, and the padded table come from shared
// memory.  Sums over multipoles stay in the lane.  The gradient of the
// interpolated table value (doubled-weight sum), g_v, goes to global memory for
// k_limber_adj, whose lanes are multipoles.  With both halves in one kernel and one
// multipole per lane, 20 of 32 lanes worked and each node took a warp reduction of
// six values and the loads of its windows: 460 k warp instructions per evaluation,
// 2560 us for 4096 evaluations of the 39-d problem; the two kernels: 66 k and
// 140 k instructions, 539 + 705 us.
template <typename T, int NB> constexpr int kGQuads = (NB * (NB + 1) / 2 + 1) / 2;   // pairs of g_C entries
constexpr int kNodeThreads = 256;

template <typename T, int NB, bool STAGE>
__global__ void __launch_bounds__(kNodeThreads, sizeof(T) == 4 ? 2 : 1)
k_limber_nodes(const ShearParams sp, const T* __restrict__ table, const T* __restrict__ win, const T* __restrict__ gC,
               T* __restrict__ gv_out, T* __restrict__ gV, T* __restrict__ glnc, const int* __restrict__ nrows) {
    using Q = P2<T>;
    constexpr int NP = NB * (NB + 1) / 2, NG = kGQuads<T, NB>;
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    const int N = sp.N, n_k = sp.n_k, n_z = sp.n_z, n_ell = sp.n_ell, D = sp.D, PK = n_k + 2, Np = (N + 3) & ~3;
    const int n_lp = (n_ell + 1) / 2, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Z4<T>* Gs = reinterpret_cast<Z4<T>*>(smem_raw);
    Q* Ls = reinterpret_cast<Q*>(Gs + n_lp * NG);          // ln(ell + 1/2) of the pairs
    T* U = reinterpret_cast<T*>(Ls + n_lp + (n_lp & 1));
    const T* src = table + (size_t)row * n_z * n_k;
    const T* lnchi = win + (size_t)row * (NB + 1) * Np;
    const T* V = lnchi + Np;
    const Z4<T>* zwp = reinterpret_cast<const Z4<T>*>(pick<T>(sp.zw4d, sp.zw4f));
    const T* lnell = pick<T>(sp.lnell, sp.lnell_f);
    const T lkmin = pick_s<T>(sp.lnk_min, sp.lnk_min_f), lkmax = pick_s<T>(sp.lnk_max, sp.lnk_max_f);
    const T inv_dk = pick_s<T>(1.0 / sp.dlnk, sp.inv_dlnk_f);
    if (STAGE)
        for (int r = wid; r < n_z; r += kNodeThreads / 32)
#pragma unroll 8
            for (int c = lane; c < n_k; c += 32) U[(r + 1) * PK + c + 1] = src[(size_t)r * n_k + c];
    for (int x = tid; x < n_lp; x += kNodeThreads) Ls[x] = Q(lnell[2 * x], lnell[min(2 * x + 1, n_ell - 1)]);
    // symmetric g_C with a doubled diagonal: h_i = sum_j G_ij V_j is the derivative of
    // g_P = 1/2 sum_ij G_ij V_i V_j by V_i
    for (int x = tid; x < n_lp * 2 * NG; x += kNodeThreads) {
        const int lp = x / (2 * NG), p = x % (2 * NG);
        T g0 = T(0), g1 = T(0);
        if (p < NP) {
            const T f = sp.pi[p] == sp.pj[p] ? T(2) : T(1);
            const T* g = gC + (size_t)row * D + p * n_ell + 2 * lp;
            g0 = f * g[0];
            if (2 * lp + 1 < n_ell) g1 = f * g[1];
        }
        reinterpret_cast<Q*>(Gs)[x] = Q(g0, g1);
    }
    __syncthreads();
    if (STAGE) {                               // ghost rows, then ghost columns (linear extrapolation)
        for (int c = 1 + tid; c <= n_k; c += kNodeThreads) {
            U[c] = T(2) * U[PK + c] - U[2 * PK + c];
            U[(n_z + 1) * PK + c] = T(2) * U[n_z * PK + c] - U[(n_z - 1) * PK + c];
        }
        __syncthreads();
        for (int r = tid; r < n_z + 2; r += kNodeThreads) {
            U[r * PK] = T(2) * U[r * PK + 1] - U[r * PK + 2];
            U[r * PK + n_k + 1] = T(2) * U[r * PK + n_k] - U[r * PK + n_k - 1];
        }
        __syncthreads();
    }
    auto two = [](T x) { return Q(x, x); };
    for (int n = 1 + blockIdx.y * kNodeThreads + tid; n < N; n += kNodeThreads * gridDim.y) {
        const T lc = lnchi[n];
        const Z4<T> wz = zwp[n];
        const Q w[4] = {two(wz.a.v.x), two(wz.a.v.y), two(wz.b.v.x), two(wz.b.v.y)};
        const int zr = sp.zrp[n];
        const T* rz = U + zr * PK;
        Q v[NB], sV[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            v[i] = two(V[i * Np + n]);
            sV[i] = two(T(0));
        }
        T sl = T(0);
        T* gvp = gv_out + (size_t)row * n_ell * Np + n;
#pragma unroll 1
        for (int lp = 0; lp < n_lp; ++lp) {
            const bool both = 2 * lp + 1 < n_ell;
            const Q le = Ls[lp];
            const T s0 = le.v.x - lc, s1 = le.v.y - lc;
            const T c0 = fmin(fmax(s0, lkmin), lkmax), c1 = fmin(fmax(s1, lkmin), lkmax);
            const T u0 = (c0 - lkmin) * inv_dk, u1 = (c1 - lkmin) * inv_dk;
            const int k0 = min((int)u0, n_k - 2), k1 = min((int)u1, n_k - 2);
            // taps folded over z
            Q col[4];
            if (STAGE) {
                const T *p0 = rz + k0, *p1 = rz + k1;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    col[q] = Q::mul(w[0], Q(p0[q], p1[q]));
#pragma unroll
                    for (int r = 1; r < 4; ++r) col[q] = Q::fma(w[r], Q(p0[r * PK + q], p1[r * PK + q]), col[q]);
                }
            } else {
#pragma unroll 1
                for (int q = 0; q < 4; ++q) {
                    Q x = two(T(0));
                    for (int r = 0; r < 4; ++r)
                        x = Q::fma(two(r == 0 ? wz.a.v.x : r == 1 ? wz.a.v.y : r == 2 ? wz.b.v.x : wz.b.v.y),
                                   Q(padded(src, n_z, n_k, zr + r, k0 + q), padded(src, n_z, n_k, zr + r, k1 + q)), x);
#pragma unroll
                    for (int y = 0; y < 4; ++y)
                        if (y == q) col[y] = x;
                }
            }
            // doubled Catmull-Rom weights in ln k and their derivatives (the z-weights are doubled too)
            const Q t(u0 - (T)k0, u1 - (T)k1), t2 = Q::mul(t, t);
            const Q m = Q::mul(t, Q::fma(two(T(-3)), t, two(T(4))));
            const Q one = two(T(1)), neg = two(T(-1));
            const Q w0 = Q::mul(t, Q::fma(t, Q::fma(t, neg, two(T(2))), neg));
            const Q w1 = Q::fma(t2, Q::fma(two(T(3)), t, two(T(-5))), two(T(2)));
            const Q w2 = Q::fma(t, m, t), w3 = Q::mul(t2, Q::add(t, neg));
            const Q d0 = Q::add(m, neg), d1 = Q::mul(t, Q::fma(two(T(9)), t, two(T(-10))));
            const Q d2 = Q::fma(t, Q::fma(two(T(-9)), t, two(T(8))), one);
            const Q d3 = Q::mul(t, Q::fma(two(T(3)), t, two(T(-2))));
            const Q f = Q::fma(w3, col[3], Q::fma(w2, col[2], Q::fma(w1, col[1], Q::mul(w0, col[0]))));
            const Q df = Q::fma(d3, col[3], Q::fma(d2, col[2], Q::fma(d1, col[1], Q::mul(d0, col[0]))));
            const Q P(p10(T(0.25) * f.v.x), p10(T(0.25) * f.v.y));
            Q h[NB];
#pragma unroll
            for (int i = 0; i < NB; ++i) h[i] = two(T(0));
            {
                const Z4<T>* G = Gs + lp * NG;
                int p = 0;
                Z4<T> g;
#pragma unroll
                for (int i = 0; i < NB; ++i)
#pragma unroll
                    for (int j = i; j < NB; ++j) {
                        if ((p & 1) == 0) g = G[p / 2];
                        const Q e = (p & 1) ? g.b : g.a;
                        h[i] = Q::fma(e, v[j], h[i]);
                        if (j != i) h[j] = Q::fma(e, v[i], h[j]);
                        ++p;
                    }
            }
            Q gP = Q::mul(v[0], h[0]);
#pragma unroll
            for (int i = 1; i < NB; ++i) gP = Q::fma(v[i], h[i], gP);
#pragma unroll
            for (int i = 0; i < NB; ++i) sV[i] = Q::fma(h[i], P, sV[i]);
            // d log L / d (doubled-weight sum); gP is twice g_P; s = ln(ell + 1/2) - ln chi
            const Q gv = Q::mul(Q::mul(gP, P), two((T)(kLn10 * 0.125)));
            const Q gs = Q::mul(gv, df);
            if (s0 == c0) sl = fma(-inv_dk, gs.v.x, sl);
            if (s1 == c1) sl = fma(-inv_dk, gs.v.y, sl);
            gvp[(size_t)(2 * lp) * Np] = gv.v.x;
            if (both) gvp[(size_t)(2 * lp + 1) * Np] = gv.v.y;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) gV[((size_t)row * NB + i) * N + n] = sV[i].v.x + sV[i].v.y;
        glnc[(size_t)row * N + n] = sl;
    }
}

// Table gradient of g_v.  Bound by instruction issue (140 k warp instructions per
// evaluation, 2.4 per cycle); node constants are read where they are used, which
// leaves registers for 28 warps per SM (held for four nodes at a time: 870 us against
// 714 for 4096 evaluations).  One warp walks a contiguous range of chi nodes, one
// multipole per lane.  Neighbouring nodes fall into the same z cell, and at most
// distances into the same ln k cell (u moves by ~0.05 cells per node), so a lane
// keeps the 16 gradients of its cell's taps in registers.  A step to the
// next cell down adds the one column that leaves to the warp's own columns in shared
// memory (four z-taps of a column side by side), any other step all four; when the
// warp enters the next z cell the rows it has left go to the warp's partial
// rows in global memory.  No two lanes add to one column at a time: with
// ascending multipoles the lanes' cells ascend too, so only neighbours can share one
// (clamped ln k); lanes with equal cells take turns.
template <typename T>
__global__ void __launch_bounds__(32 * kAdjWarps, sizeof(T) == 4 ? 7 : 3)
k_limber_adj(const ShearParams sp, const T* __restrict__ win, const T* __restrict__ gv_in,
             const int4* __restrict__ ranges, int W, int part_rows, T* __restrict__ part, int sorted,
             const int* __restrict__ nrows) {
    using Q = P2<T>;
    constexpr unsigned ALL = 0xffffffffu;
    pdl_begin();
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per_row = W / nw, row = blockIdx.x / per_row;
    if (row >= *nrows) return;
    const int4 rg = ranges[(blockIdx.x % per_row) * nw + wid];
    const int lo = rg.x, hi = rg.y;
    if (lo >= hi) return;                      // warps work alone: no block barrier below
    const int N = sp.N, n_k = sp.n_k, n_ell = sp.n_ell, PK = n_k + 2, Np = (N + 3) & ~3;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Z4<T>* acc = reinterpret_cast<Z4<T>*>(smem_raw) + (size_t)wid * PK;
    const T* lnchi = win + (size_t)row * (sp.nb + 1) * Np;
    T* prow = part + ((size_t)row * part_rows + rg.z) * PK;
    const Z4<T>* zwp = reinterpret_cast<const Z4<T>*>(pick<T>(sp.zw4d, sp.zw4f));
    const T* lnell = pick<T>(sp.lnell, sp.lnell_f);
    const T lkmin = pick_s<T>(sp.lnk_min, sp.lnk_min_f), lkmax = pick_s<T>(sp.lnk_max, sp.lnk_max_f);
    const T inv_dk = pick_s<T>(1.0 / sp.dlnk, sp.inv_dlnk_f);
    const Q zero(T(0), T(0));
    const std::integral_constant<int, 0> all_taps;
    const std::integral_constant<int, 3> last_tap;
    for (int l0 = 0; l0 < n_ell; l0 += 32) {
        const int l = l0 + lane;
        const bool act = l < n_ell;
        const T lne = lnell[act ? l : n_ell - 1];
        const T* gvp = gv_in + ((size_t)row * n_ell + (act ? l : n_ell - 1)) * Np;
        int jc = sp.zrp[lo], ik = -1;
        Z4<T> a[4];                            // by column tap
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q].a = a[q].b = zero;
        // add the register gradients of the lanes with f to their columns, from tap q0 on
        auto add_columns = [&](bool mine, auto q0) {
#pragma unroll
            for (int q = decltype(q0)::value; q < 4; ++q) {
                if (mine) {
                    Z4<T> s = acc[ik + q];
                    s.a = Q::add(s.a, a[q].a);
                    s.b = Q::add(s.b, a[q].b);
                    acc[ik + q] = s;
                }
                __syncwarp();
            }
        };
        auto flush = [&](bool f, auto q0) {
            const int before = __shfl_up_sync(ALL, f ? ik : -1 - lane, 1);
            if (sorted && !__any_sync(ALL, f && lane > 0 && before == ik)) {
                add_columns(f, q0);
                return;
            }
            const unsigned same = __match_any_sync(ALL, f ? ik : -1 - lane);
            const int turn = __popc(same & ((1u << lane) - 1u));
            for (int t = 0; __any_sync(ALL, f && turn >= t); ++t) add_columns(f && turn == t, q0);
        };
        // rows jc .. to - 1 are complete for this warp: write them out, move the rest up
        auto advance = [&](int to) {
            const int steps = to - jc;
            T* out = prow + (size_t)(jc - rg.w) * PK;
            for (int k = lane; k < PK; k += 32) {
                Z4<T> s = acc[k];
                for (int i = 0; i < steps; ++i) {
                    T* o = out + (size_t)i * PK + k;
                    *o = l0 ? *o + s.a.v.x : s.a.v.x;
                    s.a = Q(s.a.v.y, s.b.v.x);
                    s.b = Q(s.b.v.y, T(0));
                }
                acc[k] = s;
            }
            jc = to;
            __syncwarp();
        };
        for (int k = lane; k < PK; k += 32) acc[k].a = acc[k].b = zero;
        __syncwarp();
        // four nodes per load of g_v and ln chi (both padded to 4), requested one quad ahead
        Z4<T> g_n = *reinterpret_cast<const Z4<T>*>(gvp + (lo & ~3));
        Z4<T> lc_n = *reinterpret_cast<const Z4<T>*>(lnchi + (lo & ~3));
#pragma unroll 1
        for (int n4 = lo & ~3; n4 < hi; n4 += 4) {
            const Z4<T> g4 = g_n, lc4 = lc_n;
            if (n4 + 4 < hi) {
                g_n = *reinterpret_cast<const Z4<T>*>(gvp + n4 + 4);
                lc_n = *reinterpret_cast<const Z4<T>*>(lnchi + n4 + 4);
            }
            const T gn[4] = {g4.a.v.x, g4.a.v.y, g4.b.v.x, g4.b.v.y};
            const T ln[4] = {lc4.a.v.x, lc4.a.v.y, lc4.b.v.x, lc4.b.v.y};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (n4 + i < lo || n4 + i >= hi) continue;
                const int zr = sp.zrp[n4 + i];
                const Z4<T> wz = zwp[n4 + i];
                if (zr != jc) {
                    flush(ik >= 0, all_taps);
                    advance(zr);
                    ik = -1;
                }
                const T uk = (fmin(fmax(lne - ln[i], lkmin), lkmax) - lkmin) * inv_dk;
                const int ik_n = min((int)uk, n_k - 2);   // uk >= 0
                if (__any_sync(ALL, act && ik_n != ik)) {
                    const bool slide = act && ik_n == ik - 1;
                    if (__any_sync(ALL, slide)) {         // one column leaves, one enters
                        flush(slide, last_tap);
                        if (slide) {
                            ik = ik_n;
#pragma unroll
                            for (int q = 3; q > 0; --q) a[q] = a[q - 1];
                            a[0].a = a[0].b = zero;
                        }
                    }
                    const bool jump = act && ik_n != ik;
                    if (__any_sync(ALL, jump)) {
                        flush(jump && ik >= 0, all_taps);
                        if (jump) {
                            ik = ik_n;
#pragma unroll
                            for (int q = 0; q < 4; ++q) a[q].a = a[q].b = zero;
                        }
                    }
                }
                // doubled Catmull-Rom weights in ln k (the z-weights are doubled too)
                const T t = uk - (T)ik_n, t2 = t * t;
                const T wk[4] = {t * (t * (T(2) - t) - T(1)), T(2) + t2 * (T(3) * t - T(5)),
                                 t * (T(1) + t * (T(4) - T(3) * t)), t2 * (t - T(1))};
                const Q ga = Q::mul(Q(gn[i], gn[i]), wz.a), gb = Q::mul(Q(gn[i], gn[i]), wz.b);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const Q w(wk[q], wk[q]);
                    a[q].a = Q::fma(ga, w, a[q].a);
                    a[q].b = Q::fma(gb, w, a[q].b);
                }
            }
        }
        flush(ik >= 0, all_taps);
        advance(jc + 4);
    }
}

// ------------------------------------------------------------------ table gradient
// g_table of one row: partial row x of padded table row r, x in [ptr[r], ptr[r+1]),
// summed in warp order; ghost columns, then ghost rows folded back (the reverse
// of the linear extrapolation).  OUT: put(row, index, value).
template <typename T, typename OUT>
__global__ void __launch_bounds__(256)
k_table_adj(const T* __restrict__ part, int part_rows, const int* __restrict__ ptr, const int* __restrict__ idx, int n_z,
            int n_k, const OUT out, const int* __restrict__ nrows) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int* sp_ = reinterpret_cast<int*>(smem_raw);   // n_z + 3 offsets, then the partial rows in order
    int* si = sp_ + n_z + 3;
    const int PK = n_k + 2;
    for (int i = threadIdx.x; i < n_z + 3; i += blockDim.x) sp_[i] = ptr[i];
    for (int i = threadIdx.x; i < part_rows; i += blockDim.x) si[i] = idx[i] * PK;
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    __syncthreads();
    const T* p = part + (size_t)row * part_rows * PK;
    auto at = [&](int r, int c) {
        T s = T(0);
#pragma unroll 4
        for (int x = sp_[r]; x < sp_[r + 1]; ++x) s += p[si[x] + c];
        return s;
    };
    auto cols = [&](int r, int c) {
        T s = at(r, c);
        if (c <= 2) s += (c == 1 ? T(2) : T(-1)) * at(r, 0);
        if (c >= n_k - 1) s += (c == n_k ? T(2) : T(-1)) * at(r, n_k + 1);
        return s;
    };
    // rows r0 .. r1 - 1 of this block; ra .. rb - 1 of them take no ghost row, and their
    // partial rows, contiguous in the index, are loaded eight at a time (one row's two or
    // three at a time left a load's latency between any two rows: 188 us for 4096
    // evaluations of the 39-d problem, 153 us so); a block with one row has none to overlap
    const int per = (n_z + gridDim.y - 1) / gridDim.y;
    const int r0 = 1 + blockIdx.y * per, r1 = min(n_z + 1, r0 + per);
    const int ra = n_k >= 4 && per > 1 ? min(max(r0, 3), r1) : r1, rb = max(ra, min(r1, n_z - 1));
    for (int c = 1 + threadIdx.x; c <= n_k; c += blockDim.x) {
        auto put = [&](int r, T s) { out.put(row, (r - 1) * n_k + c - 1, n_z * n_k, s); };
        auto edge_row = [&](int r) {
            T s = cols(r, c);
            if (r <= 2) s += (r == 1 ? T(2) : T(-1)) * cols(0, c);
            if (r >= n_z - 1) s += (r == n_z ? T(2) : T(-1)) * cols(n_z + 1, c);
            put(r, s);
        };
        for (int r = r0; r < ra; ++r) edge_row(r);
        if (ra < rb) {
            const bool ghost = c <= 2 || c >= n_k - 1;
            const int cg = c <= 2 ? 0 : n_k + 1;
            const T f = (c == 1 || c == n_k) ? T(2) : T(-1);
            int r = ra, end = sp_[ra + 1];
            const int last = sp_[rb];
            T s = T(0);
            for (int x = sp_[ra]; x < last; x += 8) {
                T v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    v[i] = T(0);
                    if (x + i < last) {
                        v[i] = p[si[x + i] + c];
                        if (ghost) v[i] += f * p[si[x + i] + cg];
                    }
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (x + i >= last) break;
                    while (x + i >= end) {
                        put(r, s);
                        s = T(0);
                        end = sp_[++r + 1];
                    }
                    s += v[i];
                }
            }
            for (; r < rb; ++r) {
                put(r, s);
                s = T(0);
            }
        }
        for (int r = rb; r < r1; ++r) edge_row(r);
    }
}

// ------------------------------------------------------------------ windows and distances
// Exclusive prefix (or suffix) sums of NV arrays at once, x[v * pitch + i] over
// i in [0, n): thread t scans a contiguous chunk.  red: NV values per warp.
template <int NV, bool SUFFIX, typename T>
__device__ __forceinline__ void block_scan(T* x, int pitch, int n, T* red) {
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    const int chunk = (n + nt - 1) / nt;
    const int lo = min(n, tid * chunk), hi = min(n, lo + chunk);
    T s[NV], e[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) s[v] = T(0);
    for (int i = lo; i < hi; ++i)
#pragma unroll
        for (int v = 0; v < NV; ++v) s[v] += x[v * pitch + i];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        T y = s[v];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T z = SUFFIX ? __shfl_down_sync(0xffffffffu, y, o) : __shfl_up_sync(0xffffffffu, y, o);
            if (SUFFIX ? lane + o < 32 : lane >= o) y += z;
        }
        e[v] = y - s[v];
        if (lane == (SUFFIX ? 0 : 31)) red[wid * NV + v] = y;
    }
    __syncthreads();
    for (int w = SUFFIX ? wid + 1 : 0; w < (SUFFIX ? nw : wid); ++w)
#pragma unroll
        for (int v = 0; v < NV; ++v) e[v] += red[w * NV + v];
    for (int q = 0; q < hi - lo; ++q) {
        const int i = SUFFIX ? hi - 1 - q : lo + q;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const T y = x[v * pitch + i];
            x[v * pitch + i] = e[v];
            e[v] += y;
        }
    }
    __syncthreads();
}

enum { S_OM = 0, S_CHIH, S_W0, S_WA, S_GAMMA, S_PREF, S_AIA, S_ETA, S_COUNT };
// Threads per SM: one CTA while an SM holds one evaluation; from 153 evaluations on
// two CTAs share the SM (27 arrays of 1025 FP32 nodes are 111 KB) and run through one
// another's barriers (4096 evaluations: 769 -> 556 us).  A CTA's share is cut to the
// warps that keep the number of passes over the nodes (1025 nodes: 352 threads in
// 3 passes 519 us, 288 in 4 601, 256 in 5 550, 224 in 5 586).
template <typename T> constexpr int kWinAdjThreads = sizeof(T) == 4 ? 704 : 512;

// elements of the per-evaluation arrays of k_windows_adj
__host__ __device__ inline size_t windows_adj_elems(int N, int nb) { return (size_t)(7 + 4 * nb) * N; }

template <typename T, int NB>
__global__ void __launch_bounds__(kWinAdjThreads<T>)
k_windows_adj(const ShearParams sp, const double* __restrict__ theta_full, const T* __restrict__ gV,
              const T* __restrict__ glnc, T* __restrict__ scratch, double* __restrict__ gfull,
              const int* __restrict__ nrows) {
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = sp.N, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
    T* S = scratch ? scratch + (size_t)row * windows_adj_elems(N, NB) : reinterpret_cast<T*>(smem_raw);
    T *chi = S, *Ez = S + N, *omw = S + 2 * N, *fg = S + 3 * N;
    T *gomw = S + 4 * N, *gE = gomw;             // g_omw makes room for g_E node by node,
    T *Dg = S + 5 * N, *t1 = Dg;                 // ln D and D for g_S,
    T *gchi = S + 6 * N, *t2 = gchi;             // g_chi for its suffix sums (beside t1)
    T *raw = S + 7 * N, *nchi = raw + NB * N, *E0 = nchi + NB * N, *E1 = E0 + NB * N;
    constexpr int NS = S_COUNT + 3 * NB, NR = NS > 2 * NB ? NS : 2 * NB;
    __shared__ T red[(kWinAdjThreads<T> / 32) * NR];
    __shared__ T th[16];
    const T* a_ = pick<T>(sp.a, sp.a_f);
    const T* lna_ = pick<T>(sp.lna, sp.lna_f);
    const T* z_ = pick<T>(sp.z, sp.z_f);
    const T* wa_ = pick<T>(sp.wa, sp.wa_f);
    const T* nz_mu = pick<T>(sp.nz_mean, sp.nz_mean_f);
    const T* nz_sg = pick<T>(sp.nz_sigma, sp.nz_sigma_f);
    const T* ia_ = pick<T>(sp.ia, sp.ia_f);
    const Z4<T>* gl_ia = reinterpret_cast<const Z4<T>*>(pick<T>(sp.gl_ia, sp.gl_ia_f));   // four points per interval
    const Z4<T>* gl_ln = reinterpret_cast<const Z4<T>*>(pick<T>(sp.gl_ln, sp.gl_ln_f));
    const Z4<T>* gl_1ma = reinterpret_cast<const Z4<T>*>(pick<T>(sp.gl_1ma, sp.gl_1ma_f));
    const T lnpiv = pick_s<T>(sp.ln_pivot, sp.ln_pivot_f), c1rho = pick_s<T>(sp.c1rho, sp.c1rho_f);
    if (tid < 11 + NB) th[tid] = (T)theta_full[(size_t)row * sp.n_params + tid];
    __syncthreads();
    const T h = th[2];
    const T om = (th[0] + th[1]) / (h * h);
    const T w0 = th[5], wa = th[6];
    const T pde = T(3) * (T(1) + w0 + wa);
    const T chiH = T(kCover100) / h;
    const T gamma = T(0.55) + T(0.05) * (T(1) + w0 + T(0.5) * wa);
    const T pref = T(1.5) * om / (chiH * chiH);
    const T A_IA = th[9], eta = th[10], iom = T(1) / om, ichiH = T(1) / chiH;
    T sum[NS];                                  // scalars, then per bin: g_nchi nchi u / sigma, g_nchi nchi, d norm / d D_z
#pragma unroll
    for (int q = 0; q < NS; ++q) sum[q] = T(0);

    // ---- forward
    for (int n = tid; n < N; n += nt) {
        const T a = a_[n], ia = ia_[n];
        const T de = ex<T>(-pde * lna_[n] - T(3) * wa * (T(1) - a));
        Ez[n] = sqrt(om * (ia * ia * ia) + (T(1) - om) * de);
        T inc = T(0);
        if (n < N - 1) {
            const Z4<T> qi = gl_ia[n], ql = gl_ln[n], qa = gl_1ma[n];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const T ig = qi[g];
                const T e2 = om * ig * ig * ig + (T(1) - om) * ex<T>(-pde * ql[g] - T(3) * wa * qa[g]);
                inc += glw<T>(g) * ig * ig * rsq(e2);
            }
            inc *= chiH * T(0.5) * (a - a_[n + 1]);
        }
        chi[n] = inc;
    }
    __syncthreads();
    block_scan<1, false>(chi, N, N, red);
    T pn[NB], isg[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) { pn[i] = T(0); isg[i] = T(1) / nz_sg[i]; }
    for (int n = tid; n < N; n += nt) {
        const T ie = T(1) / Ez[n], ia = ia_[n], ia2 = wa_[n] * (ia * ia);
        const T oma = om * (ia * ia * ia) * (ie * ie);
        fg[n] = ex<T>(gamma * lg<T>(oma));
        omw[n] = ia2 * chiH * ie;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const T u = (z_[n] - th[11 + i] - nz_mu[i]) * isg[i];
            const T rw = ex<T>(T(-0.5) * u * u);
            raw[i * N + n] = rw;
            pn[i] += ia2 * rw;
            sum[S_COUNT + 2 * NB + i] += ia2 * rw * u * isg[i];
        }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const T s = warp_sum(pn[i]);
        if (lane == 0) red[wid * NB + i] = s;
    }
    __syncthreads();
    T inorm[NB];                                // 1 / (chiH norm)
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        T s = T(0);
        for (int w = 0; w < nt / 32; ++w) s += red[w * NB + i];
        inorm[i] = T(1) / (chiH * s);
    }
    __syncthreads();
    for (int n = tid; n < N; n += nt) {
        Dg[n] = (n < N - 1) ? T(0.5) * (fg[n] + fg[n + 1]) * (lna_[n] - lna_[n + 1]) : T(0);
        const T o = omw[n], e = Ez[n], ic = n >= 1 ? T(1) / chi[n] : T(0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const T nc = raw[i * N + n] * e * inorm[i];
            nchi[i * N + n] = nc;
            E0[i * N + n] = (n >= 1) ? o * nc : T(0);
            E1[i * N + n] = (n >= 1) ? o * nc * ic : T(0);
        }
    }
    __syncthreads();
    block_scan<1, false>(Dg, N, N, red);
    block_scan<2 * NB, true>(E0, N, N, red);

    // ---- windows: V = sqrt(omw)/chi * W, W = pc (E0 - chi E1) - amp nchi, amp = A_IA q c1rho Om / D
    for (int n = tid; n < N; n += nt) {
        const T D_n = ex<T>(-Dg[n]);
        if (n == 0) {                           // carries no window value
            for (int i = 0; i < NB; ++i) { raw[i * N] = T(0); E0[i * N] = T(0); E1[i * N] = T(0); }
            gchi[0] = T(0); gomw[0] = T(0); t1[0] = T(0);
            continue;
        }
        const T c = chi[n], ian = ia_[n], so = sqrt(omw[n]), ic = T(1) / c;
        const T lq = -lna_[n] - lnpiv;          // ln((1 + z) / pivot)
        const T ampc = ex<T>(eta * lq) * c1rho * om / D_n;   // amp = A_IA * ampc
        const T pc = pref * c * ian;
        T g_so = T(0), g_c = T(0), g_amp = T(0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const T e0 = E0[i * N + n], e1 = E1[i * N + n], nc = nchi[i * N + n];
            const T W = pc * (e0 - c * e1) - A_IA * ampc * nc;
            const T gVv = gV[((size_t)row * NB + i) * N + n];
            const T gW = gVv * so * ic;
            g_so += gVv * W * ic;
            g_c += -gVv * so * W * ic * ic;
            const T gpc = gW * (e0 - c * e1);
            sum[S_PREF] += gpc * c * ian;
            g_c += gpc * pref * ian - gW * pc * e1;
            E0[i * N + n] = gW * pc;            // the adjoints take the place of the suffix sums
            E1[i * N + n] = -gW * pc * c;
            g_amp += -gW * nc;
            raw[i * N + n] = -gW * A_IA * ampc; // g_nchi, direct term
        }
        gomw[n] = g_so * T(0.5) / so;
        gchi[n] = glnc[(size_t)row * N + n] * ic + g_c;
        sum[S_AIA] += g_amp * ampc;
        sum[S_ETA] += g_amp * A_IA * ampc * lq;
        sum[S_OM] += g_amp * A_IA * ampc * iom;
        t1[n] = g_amp * A_IA * ampc;            // g_S = -g_D D, g_D = -g_amp amp / D
    }
    __syncthreads();
    // E0_i(n) = sum_{m>n} omw_m nchi_m  ->  G0(m) = sum_{n<m} gE0(n)
    block_scan<2 * NB, false>(E0, N, N, red);
    for (int m = tid; m < N; m += nt) {
        const T ie = T(1) / Ez[m], o = omw[m], ic = m >= 1 ? T(1) / chi[m] : T(0);
        T go = gomw[m], gc = gchi[m], ge = T(0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            T gnc = raw[i * N + m];
            const T nc = nchi[i * N + m];
            if (m >= 1) {
                const T G1 = E1[i * N + m] * ic, G = E0[i * N + m] + G1;
                go += nc * G;
                gnc += o * G;
                gc += -o * nc * G1 * ic;
            }
            // nchi = raw E / (chiH norm); raw and norm depend on D_z through u
            const T u = (z_[m] - th[11 + i] - nz_mu[i]) * isg[i];
            const T gn = gnc * nc;
            ge += gn * ie;
            sum[S_COUNT + i] += gn * u * isg[i];
            sum[S_COUNT + NB + i] += gn;
        }
        // omw = wa chiH / (a^2 E)
        sum[S_CHIH] += go * o * ichiH;
        gE[m] = ge - go * o * ie;
        t2[m] = gc;
    }
    __syncthreads();
    // growth: D_n = exp(-S_n), S_n = sum_{m<n} seg_m -> g_seg_m = sum_{n>m} g_S_n;
    // distances: chi_n = sum_{m<n} dchi_m -> g_dchi_m = sum_{n>m} g_chi_n
    block_scan<2, true>(t1, N, N, red);
    for (int m = tid; m < N; m += nt) {
        const T a = a_[m], lna = lna_[m], ie = T(1) / Ez[m], ia = ia_[m];
        T gf = T(0);
        if (m < N - 1) gf += T(0.5) * t1[m] * (lna - lna_[m + 1]);
        if (m >= 1) gf += T(0.5) * t1[m - 1] * (lna_[m - 1] - lna);
        const T ia3 = ia * ia * ia;
        const T oma = om * ia3 * (ie * ie);
        const T gff = gf * fg[m];
        sum[S_GAMMA] += gff * lg<T>(oma);
        sum[S_OM] += gff * gamma * iom;
        // node E: E^2 = om a^-3 + (1 - om) de
        const T ge2 = (gE[m] - T(2) * gff * gamma * ie) * T(0.5) * ie;
        const T de = ex<T>(-pde * lna - T(3) * wa * (T(1) - a));
        sum[S_OM] += ge2 * (ia3 - de);
        sum[S_W0] += ge2 * (T(1) - om) * de * (T(-3) * lna);
        sum[S_WA] += ge2 * (T(1) - om) * de * (T(-3) * lna - T(3) * (T(1) - a));
        if (m < N - 1) {
            const T g = t2[m], half = T(0.5) * (a - a_[m + 1]);
            T inc = T(0);
            const Z4<T> qi = gl_ia[m], ql = gl_ln[m], qa = gl_1ma[m];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const T lgg = ql[q], ig = qi[q], oma_q = qa[q], i3 = ig * ig * ig;
                const T deg = ex<T>(-pde * lgg - T(3) * wa * oma_q);
                const T rs = rsq(om * i3 + (T(1) - om) * deg);
                const T F = ig * ig * rs;
                inc += glw<T>(q) * F;
                const T gE2 = g * chiH * half * glw<T>(q) * T(-0.5) * F * (rs * rs);
                sum[S_OM] += gE2 * (i3 - deg);
                sum[S_W0] += gE2 * (T(1) - om) * deg * (T(-3) * lgg);
                sum[S_WA] += gE2 * (T(1) - om) * deg * (T(-3) * lgg - T(3) * oma_q);
            }
            sum[S_CHIH] += g * half * inc;
        }
    }
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        const T s = warp_sum(sum[q]);
        if (lane == 0) red[wid * NS + q] = s;
    }
    __syncthreads();
    if (tid < NS) {
        T s = T(0);
        for (int w = 0; w < nt / 32; ++w) s += red[w * NS + tid];
        red[tid] = s;                           // warp 0's slot of value tid, read by this thread only
    }
    __syncthreads();
    if (tid == 0) {
        const T* gs = red;
        T chih = gs[S_CHIH];
        double* g = gfull + (size_t)row * sp.n_params;
        for (int i = 0; i < NB; ++i) {
            const T gn = gs[S_COUNT + NB + i];
            chih -= gn * ichiH;                 // nchi ~ 1 / chiH
            g[11 + i] += (double)(gs[S_COUNT + i] - gn * (inorm[i] * chiH) * gs[S_COUNT + 2 * NB + i]);
        }
        // pref = 1.5 om / chiH^2; gamma = 0.55 + 0.05 (1 + w0 + wa/2)
        const T g_om = gs[S_OM] + gs[S_PREF] * pref / om;
        const T g_chih = chih - T(2) * gs[S_PREF] * pref / chiH;
        // om = (wb + wc) / h^2; chiH = c / (100 h)
        g[0] += (double)(g_om / (h * h));
        g[1] += (double)(g_om / (h * h));
        g[2] += (double)(-T(2) * g_om * om / h - g_chih * chiH / h);
        g[5] += (double)(gs[S_W0] + T(0.05) * gs[S_GAMMA]);
        g[6] += (double)(gs[S_WA] + T(0.025) * gs[S_GAMMA]);
        g[9] += (double)gs[S_AIA];
        g[10] += (double)gs[S_ETA];
    }
}

struct OutT64 {
    double* p;
    __device__ __forceinline__ void put(int row, int i, int n, double v) const { p[(size_t)row * n + i] = v; }
};
// scaled and in bf16 planes: the operand of the emulator's backward GEMMs
template <int P>
struct OutPlaneT {
    __nv_bfloat16* p;
    long long stride;
    int pitch;
    float s;
    __device__ __forceinline__ void put(int row, int i, int, float v) const {
        tc::plane_store<P>(s * v, p + (size_t)row * pitch + i, stride);
    }
};
struct OutT32 {
    float* p;
    __device__ __forceinline__ void put(int row, int i, int n, float v) const { p[(size_t)row * n + i] = v; }
};

}  // namespace adj

// Node ranges of the W warps of an evaluation, the partial rows they write (row
// r of range w: padded table rows jlo .. jhi + 3) and, per padded table row, the
// partial rows that hold a share of it.
static void build_split(const std::vector<int>& zrp, int N, int n_z, int W, std::vector<int4>& ranges, int* rows,
                        std::vector<int>& ptr, std::vector<int>& idx) {
    std::vector<std::vector<int>> of(n_z + 2);
    int off = 0;
    for (int w = 0; w < W; ++w) {
        const int lo = 1 + (int)((long long)(N - 1) * w / W), hi = 1 + (int)((long long)(N - 1) * (w + 1) / W);
        int4 r = make_int4(lo, hi, off, 0);
        if (lo < hi) {
            r.w = zrp[lo];
            for (int j = zrp[lo]; j <= zrp[hi - 1] + 3; ++j) of[j].push_back(off++);
        }
        ranges.push_back(r);
    }
    *rows = off;
    for (int j = 0; j < n_z + 2; ++j) {
        ptr.push_back((int)idx.size());
        idx.insert(idx.end(), of[j].begin(), of[j].end());
    }
    ptr.push_back((int)idx.size());
}

// Warps per evaluation: with eight, 152 evaluations and more give every SM eight to
// its limit of 28 warps; fewer evaluations get shorter node ranges (64 evaluations of
// the 39-d problem: 32 warps, 14 per SM), at the price of four more partial rows a
// range.  k_limber_nodes splits an evaluation's nodes over 4, 2 or 1 CTAs by the
// same lines.
static int limber_adj_split(int rows) { return rows <= 76 ? 2 : rows <= 152 ? 1 : 0; }

int projection_adj_create(const ShearParams& sp, int elt, int cap, ProjectionAdj* a) {
    if (sp.n_ell > 64 || sp.n_params > 128) return NS_ENOTSUP;
    auto alloc = [&](size_t bytes, void** out) -> int {
        if (cudaMalloc(out, bytes) != cudaSuccess) return NS_ENOMEM;
        a->owned.push_back(*out);
        return NS_OK;
    };
    const size_t n = (size_t)elt * cap, Np = (sp.N + 3) & ~3;
    NS_TRY(alloc(n * (sp.nb + 1) * Np, &a->win));
    if (elt == 8) NS_TRY(alloc(n * window_node_values(sp.nb) * sp.N, &a->win_nodes));
    NS_TRY(alloc(n * sp.D, &a->resid));
    NS_TRY(alloc(n * sp.D, &a->C));
    NS_TRY(alloc(n * sp.D, &a->gC));
    NS_TRY(alloc(n * sp.nb * sp.N, &a->gV));
    NS_TRY(alloc(n * sp.N, &a->glnc));
    NS_TRY(alloc(n * sp.n_ell * Np, &a->gv));
    std::vector<double> lnell(sp.n_ell);
    NS_CUDA_TRY(cudaMemcpy(lnell.data(), sp.lnell, sizeof(double) * sp.n_ell, cudaMemcpyDeviceToHost));
    a->sorted = std::is_sorted(lnell.begin(), lnell.end());
    std::vector<int> zrp(sp.N);
    NS_CUDA_TRY(cudaMemcpy(zrp.data(), sp.zrp, sizeof(int) * sp.N, cudaMemcpyDeviceToHost));
    size_t part = 0;
    for (int k = 0; k < 3; ++k) {
        std::vector<int4> ranges;
        std::vector<int> ptr, idx;
        build_split(zrp, sp.N, sp.n_z, 8 << k, ranges, &a->part_rows[k], ptr, idx);
        const int most = k == 2 ? std::min(cap, 76) : k == 1 ? std::min(cap, 152) : cap;
        part = std::max(part, (size_t)a->part_rows[k] * most);
        void* v;
        NS_TRY(alloc(sizeof(int4) * ranges.size(), &v));
        a->ranges[k] = (int4*)v;
        NS_CUDA_TRY(cudaMemcpy(v, ranges.data(), sizeof(int4) * ranges.size(), cudaMemcpyHostToDevice));
        NS_TRY(alloc(sizeof(int) * ptr.size(), &v));
        a->ptr[k] = (int*)v;
        NS_CUDA_TRY(cudaMemcpy(v, ptr.data(), sizeof(int) * ptr.size(), cudaMemcpyHostToDevice));
        NS_TRY(alloc(sizeof(int) * idx.size(), &v));
        a->idx[k] = (int*)v;
        NS_CUDA_TRY(cudaMemcpy(v, idx.data(), sizeof(int) * idx.size(), cudaMemcpyHostToDevice));
    }
    NS_TRY(alloc((size_t)elt * part * (sp.n_k + 2), &a->part));
    const size_t elems = adj::windows_adj_elems(sp.N, sp.nb);
    a->win_smem = elems * elt;
    if (a->win_smem > kAdjSmemMax) {
        NS_TRY(alloc(n * elems, &a->scratch));
        a->win_smem = 0;
    }
    NS_CUDA_TRY(cudaStreamCreateWithFlags(&a->side, cudaStreamNonBlocking));
    NS_CUDA_TRY(cudaEventCreateWithFlags(&a->ev_fork, cudaEventDisableTiming));
    NS_CUDA_TRY(cudaEventCreateWithFlags(&a->ev_join, cudaEventDisableTiming));
    return NS_OK;
}

void projection_adj_free(ProjectionAdj* a) {
    for (void* q : a->owned) cudaFree(q);
    a->owned.clear();
    if (a->ev_fork) cudaEventDestroy(a->ev_fork);
    if (a->ev_join) cudaEventDestroy(a->ev_join);
    if (a->side) cudaStreamDestroy(a->side);
    a->ev_fork = a->ev_join = nullptr;
    a->side = nullptr;
}

template <typename T>
int launch_projection_adj_windows(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const int* nrows,
                                  int grid_rows, cudaStream_t st) {
    NS_CUDA_TRY(cudaEventRecord(a->ev_fork, st));
    NS_CUDA_TRY(cudaStreamWaitEvent(a->side, a->ev_fork, 0));
    NS_TRY((launch_windows<T, false>(sp, theta_full, (T*)a->win, nrows, grid_rows, a->side, (T*)a->win_nodes)));
    NS_CUDA_TRY(cudaEventRecord(a->ev_join, a->side));
    return NS_OK;
}

template <typename T, int RB>
static int launch_chi2_adj(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const T* LinvT,
                           const T* Linv, double c0, double* gfull, OutPtr logL, const int* nrows, int grid_rows,
                           cudaStream_t st) {
    const size_t smem = sizeof(T) * adj::chi2_adj_elems(sp.D, adj::kChiV<T>, sp.nb, sp.n_pairs, sp.n_tmpl, RB);
    static bool attr = false;
    if (!attr) {
        NS_CUDA_TRY(cudaFuncSetAttribute(adj::k_chi2_adj<T, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax));
        attr = true;
    }
    NS_CUDA_TRY(launch_pdl(adj::k_chi2_adj<T, RB>, dim3((grid_rows + RB - 1) / RB), dim3(adj::kChiThreads), smem, st, sp, theta_full,
                           (const T*)a->resid, (const T*)a->C, LinvT, Linv, c0, (T*)a->gC, gfull, logL, nrows));
    return NS_OK;
}

template <typename T, int NB>
static int launch_reverse(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const T* table,
                          const TableGrad& out, double* gfull, const int* nrows, int grid_rows, cudaStream_t st) {
    const int k = limber_adj_split(grid_rows), W = 8 << k, PK = sp.n_k + 2;
    // the padded table beside g_C in shared memory; very wide tables stay in global memory
    const size_t g_bytes = sizeof(adj::Z4<T>) * (size_t)((sp.n_ell + 1) / 2) * adj::kGQuads<T, NB> +
                           sizeof(adj::P2<T>) * (size_t)(((sp.n_ell + 1) / 2 + 1) & ~1);
    const size_t t_bytes = sizeof(T) * (size_t)(sp.n_z + 2) * PK;
    // a warp's columns of gradients; CTAs shrink to one warp where tables are very wide
    const size_t col = sizeof(adj::Z4<T>) * (size_t)PK;
    int nw = kAdjWarps;
    while (nw > 1 && nw * col > kAdjSmemMax) nw >>= 1;
    if (nw * col > kAdjSmemMax) return NS_ENOTSUP;
    static bool attr = false;
    if (!attr) {
        NS_CUDA_TRY(cudaFuncSetAttribute(adj::k_limber_nodes<T, NB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax));
        NS_CUDA_TRY(cudaFuncSetAttribute(adj::k_limber_adj<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax));
        NS_CUDA_TRY(cudaFuncSetAttribute(adj::k_windows_adj<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax));
        attr = true;
    }
    auto nodes = [&](auto kern, size_t smem) -> int {
        // few evaluations: the nodes of one over several CTAs
        NS_CUDA_TRY(launch_pdl(kern, dim3(grid_rows, 1 << k), dim3(adj::kNodeThreads), smem, st, sp, table,
                               (const T*)a->win, (const T*)a->gC, (T*)a->gv, (T*)a->gV, (T*)a->glnc, nrows));
        return NS_OK;
    };
    if (g_bytes + t_bytes <= kAdjSmemMax) NS_TRY(nodes(adj::k_limber_nodes<T, NB, true>, g_bytes + t_bytes));
    else NS_TRY(nodes(adj::k_limber_nodes<T, NB, false>, g_bytes));
    NS_CUDA_TRY(launch_pdl(adj::k_limber_adj<T>, dim3(grid_rows * (W / nw)), dim3(32 * nw), nw * col, st, sp,
                           (const T*)a->win, (const T*)a->gv, (const int4*)a->ranges[k], W, a->part_rows[k],
                           (T*)a->part, a->sorted, nrows));
    // a table row per block for few evaluations, the whole table from 1024 on (4096
    // evaluations: one block 153 us, three 161, six 173)
    const dim3 g(grid_rows, grid_rows < 256 ? sp.n_z : grid_rows < 1024 ? 3 : 1);
    const dim3 b(std::min(256, (sp.n_k + 31) & ~31));
    auto table_adj = [&](auto o) -> int {
        NS_CUDA_TRY(launch_pdl(adj::k_table_adj<T, decltype(o)>, g, b, sizeof(int) * (sp.n_z + 3 + a->part_rows[k]), st,
                               (const T*)a->part, a->part_rows[k],
                               (const int*)a->ptr[k], (const int*)a->idx[k], sp.n_z, sp.n_k, o, nrows));
        return NS_OK;
    };
    if constexpr (sizeof(T) == 8) {
        NS_TRY(table_adj(adj::OutT64{(double*)out.table}));
    } else {
        if (out.px == 3) NS_TRY(table_adj(adj::OutPlaneT<3>{out.planes, out.stride, out.pitch, out.scale}));
        else if (out.px == 2) NS_TRY(table_adj(adj::OutPlaneT<2>{out.planes, out.stride, out.pitch, out.scale}));
        else NS_TRY(table_adj(adj::OutT32{(float*)out.table}));
    }
    // two CTAs per SM where their arrays fit (FP64: 221 KB for 1025 nodes, one)
    const bool pairs = grid_rows > 152 && 2 * a->win_smem <= kAdjSmemMax;
    const int share = pairs ? adj::kWinAdjThreads<T> / 2 : adj::kWinAdjThreads<T>;
    const int passes = (sp.N + share - 1) / share, threads = ((sp.N + passes - 1) / passes + 31) & ~31;
    NS_CUDA_TRY(launch_pdl(adj::k_windows_adj<T, NB>, dim3(grid_rows), dim3(threads),
                           a->win_smem, st, sp,
                           theta_full, (const T*)a->gV, (const T*)a->glnc, (T*)a->scratch, gfull, nrows));
    return NS_OK;
}

template <typename T>
int launch_projection_adj(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const T* table,
                          const T* LinvT, const T* Linv, double c0, const TableGrad& out, double* gfull, OutPtr logL,
                          const int* nrows, int grid_rows, int* err, cudaStream_t st) {
    NS_CUDA_TRY(cudaStreamWaitEvent(st, a->ev_join, 0));
    NS_TRY((launch_limber<T, false>(sp, theta_full, table, (const T*)a->win, (T*)a->resid, nullptr, nrows, grid_rows,
                                    err, st, (T*)a->C)));
    // one row per block spreads few rows over the chip, eight share the reads of L^-1
    if (grid_rows < 1024 || sizeof(T) * adj::chi2_adj_elems(sp.D, adj::kChiV<T>, sp.nb, sp.n_pairs, sp.n_tmpl, 8) > kAdjSmemMax)
        NS_TRY((launch_chi2_adj<T, 1>(sp, a, theta_full, LinvT, Linv, c0, gfull, logL, nrows, grid_rows, st)));
    else
        NS_TRY((launch_chi2_adj<T, 8>(sp, a, theta_full, LinvT, Linv, c0, gfull, logL, nrows, grid_rows, st)));
    switch (sp.nb) {
        case 1: return launch_reverse<T, 1>(sp, a, theta_full, table, out, gfull, nrows, grid_rows, st);
        case 2: return launch_reverse<T, 2>(sp, a, theta_full, table, out, gfull, nrows, grid_rows, st);
        case 3: return launch_reverse<T, 3>(sp, a, theta_full, table, out, gfull, nrows, grid_rows, st);
        case 4: return launch_reverse<T, 4>(sp, a, theta_full, table, out, gfull, nrows, grid_rows, st);
        case 5: return launch_reverse<T, 5>(sp, a, theta_full, table, out, gfull, nrows, grid_rows, st);
        default: return NS_ENOTSUP;
    }
}

#define NS_INST(T)                                                                                                    \
    template int launch_projection_adj_windows<T>(const ShearParams&, ProjectionAdj*, const double*, const int*, int, \
                                                  cudaStream_t);                                                      \
    template int launch_projection_adj<T>(const ShearParams&, ProjectionAdj*, const double*, const T*, const T*,      \
                                          const T*, double, const TableGrad&, double*, OutPtr, const int*, int,      \
                                          int*, cudaStream_t);
NS_INST(double)
NS_INST(float)
#undef NS_INST

}  // namespace gpuns
