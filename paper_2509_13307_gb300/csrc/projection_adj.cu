// Adjoint of the shear projection (row A14): from the emulator table and theta
// to log L, d log L / d table and d log L / d theta (emulator inputs' share
// through the emulator excluded).  The forward stages are the likelihood's own
// kernels (projection.cu), with the Limber sums kept; the reverse stages are
//
//   k_chi2_adj     y = L^-1 r, log L, g_m = L^-T y; g_C = g_m (1+m_i)(1+m_j);
//                  gradients of the biases and the noise templates
//   k_limber_adj   per node and multipole: g_P = sum_p g_C V_i V_j;
//                  g_V_i += g_C V_j P; g_v = ln 10 P g_P spread over the 16 table
//                  taps; d v / d ln k (Catmull-Rom derivative) gives g_ln chi
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
// Bound: FP32 instruction issue.  The one-kernel form it replaced kept 250 KB
// of intermediates per evaluation in global memory and added 16 atomics per
// (node, multipole) to the table gradient.  Whole BF16 gradient calls of the
// 39-d problem: 4096 rows 9978 -> 6496 us, 64 rows 608 -> 413 us.
#include <algorithm>
#include <vector>

#include "likelihood.cuh"
#include "projection_adj.cuh"

namespace gpuns {
namespace adj {

// 4-point Gauss-Legendre nodes and weights as compile-time constants of the
// kernel's type (no double -> float conversions at run time).
template <typename T> __device__ __forceinline__ T glx(int g) {
    return g == 0 ? T(-0.86113631159405257522) : g == 1 ? T(-0.33998104358485626480)
         : g == 2 ? T(0.33998104358485626480) : T(0.86113631159405257522);
}
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
// 10^v and its FP32 form on exp2
__device__ __forceinline__ double p10(double v) { return exp(v * kLn10); }
__device__ __forceinline__ float p10(float v) { return exp2f(v * 3.32192809488736234787f); }

// ------------------------------------------------------------------ chi^2
// RB rows per block: each entry of L^-1 read serves RB rows, whose values lie
// beside one another in shared memory.
template <typename T, int RB>
__global__ void __launch_bounds__(256)
k_chi2_adj(const ShearParams sp, const double* __restrict__ theta_full, const T* __restrict__ resid,
           const T* __restrict__ C, const T* __restrict__ LinvT, const T* __restrict__ Linv, double c0,
           T* __restrict__ gC, double* __restrict__ gfull, double* __restrict__ logL, const int* __restrict__ nrows) {
    pdl_begin();
    const int M = *nrows, r0 = blockIdx.x * RB;
    if (r0 >= M) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int D = sp.D, P = sp.n_params, nb = sp.nb, n_ell = sp.n_ell, nt = sp.n_tmpl, np = sp.n_pairs;
    T* r = reinterpret_cast<T*>(smem_raw);     // D x RB, later g_m
    T* y = r + D * RB;                         // D x RB
    T* th = y + D * RB;                        // RB x nb: 1 + m_i
    T* S = th + RB * nb;                       // np x RB: sum_ell g_m C
    T* tp = S + np * RB;                       // 8 x RB x nt partial template sums
    __shared__ T red[32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < RB * D; i += 256) {
        const int j = i / D, a = i - j * D;
        r[a * RB + j] = r0 + j < M ? resid[(size_t)(r0 + j) * D + a] : T(0);
    }
    for (int i = tid; i < RB * nb; i += 256) {
        const int j = i / nb;
        th[i] = r0 + j < M ? T(1) + (T)theta_full[(size_t)(r0 + j) * P + 11 + nb + i % nb] : T(0);
    }
    __syncthreads();
    T sq[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) sq[j] = T(0);
    for (int a = tid; a < D; a += 256) {
        T acc[RB];
#pragma unroll
        for (int j = 0; j < RB; ++j) acc[j] = T(0);
#pragma unroll 4
        for (int b = 0; b <= a; ++b) {
            const T l = LinvT[(size_t)b * D + a];
#pragma unroll
            for (int j = 0; j < RB; ++j) acc[j] = fma(l, r[b * RB + j], acc[j]);
        }
#pragma unroll
        for (int j = 0; j < RB; ++j) {
            y[a * RB + j] = acc[j];
            sq[j] = fma(acc[j], acc[j], sq[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < RB; ++j) {
        const T s = block_sum(sq[j], red);     // also orders y before its reads
        if (tid == 0 && r0 + j < M) logL[r0 + j] = c0 - 0.5 * (double)s;
    }
    // g_m = L^-T y: (g_m)_a = sum_{b >= a} (L^-1)[b][a] y_b
    for (int a = tid; a < D; a += 256) {
        T acc[RB];
#pragma unroll
        for (int j = 0; j < RB; ++j) acc[j] = T(0);
#pragma unroll 4
        for (int b = a; b < D; ++b) {
            const T l = Linv[(size_t)b * D + a];
#pragma unroll
            for (int j = 0; j < RB; ++j) acc[j] = fma(l, y[b * RB + j], acc[j]);
        }
        const int p = a / n_ell, i = sp.pi[p], k = sp.pj[p];
#pragma unroll
        for (int j = 0; j < RB; ++j) {
            r[a * RB + j] = acc[j];
            if (r0 + j < M) gC[(size_t)(r0 + j) * D + a] = acc[j] * th[j * nb + i] * th[j * nb + k];
        }
    }
    __syncthreads();
    for (int q = tid; q < np * RB; q += 256) {
        const int p = q / RB, j = q % RB;
        T s = T(0);
        if (r0 + j < M)
            for (int e = 0; e < n_ell; ++e) s = fma(r[(p * n_ell + e) * RB + j], C[(size_t)(r0 + j) * D + p * n_ell + e], s);
        S[q] = s;
    }
    {   // templates: warp w sums the w-th eighth of the data vector, lanes over templates
        const T* tm = pick<T>(sp.tmpl, sp.tmpl_f);
        const int lo = D * wid / 8, hi = D * (wid + 1) / 8;
        for (int t = lane; t < nt; t += 32) {
            T acc[RB];
#pragma unroll
            for (int j = 0; j < RB; ++j) acc[j] = T(0);
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
    for (int q = tid; q < RB * P; q += 256) {
        const int j = q / P, i = q % P - (11 + nb);
        if (r0 + j >= M) continue;
        T v = T(0);
        if (i >= 0 && i < nb) {
            for (int p = 0; p < np; ++p) {
                if (sp.pi[p] == i) v = fma(S[p * RB + j], th[j * nb + sp.pj[p]], v);
                if (sp.pj[p] == i) v = fma(S[p * RB + j], th[j * nb + sp.pi[p]], v);
            }
        } else if (i >= nb) {
            for (int w = 0; w < 8; ++w) v += tp[(w * RB + j) * nt + i - nb];
        }
        gfull[(size_t)(r0 + j) * P + q % P] = (double)v;
    }
}

// ------------------------------------------------------------------ Limber
template <typename T> struct alignas(16) V4 { T x, y, z, w; };

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
    if (r == 0) return T(2) * padded_row(t, n_k, c) - padded_row(t + n_k, n_k, c);
    if (r == n_z + 1)
        return T(2) * padded_row(t + (size_t)(n_z - 1) * n_k, n_k, c) - padded_row(t + (size_t)(n_z - 2) * n_k, n_k, c);
    return padded_row(t + (size_t)(r - 1) * n_k, n_k, c);
}

// Sum of 8 values per lane over the warp: lane l gets the sum of value l & 7.
template <typename T>
__device__ __forceinline__ T warp_transpose_sum8(T (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 4; off >= 1; off >>= 1) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const T send = upper ? v[i] : v[i + off];
            const T keep = upper ? v[i + off] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    T s = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 8);
    return s + __shfl_xor_sync(0xffffffffu, s, 16);
}

// One warp walks a contiguous range of chi nodes, one multipole per lane.
// Neighbouring nodes fall into the same z cell, and at most distances into the
// same ln k cell (u moves by ~0.05 cells per node), so a lane keeps the 16 taps
// of its cell and their 16 gradients in registers and exchanges them only when
// its cell changes (about one lane per node): the gradients go to the warp's own
// columns in shared memory (four z-taps of a column side by side), and when the
// warp enters the next z cell the rows it has left go to the warp's partial
// rows in global memory.  No two lanes add to one column at a time: lanes with
// equal cells take turns.  Sums over multipoles (g_V, g_ln chi) are warp
// reductions of 8 values at once.
template <typename T, int NB>
__global__ void __launch_bounds__(32 * kAdjWarps, sizeof(T) == 4 ? 4 : 2)
k_limber_adj(const ShearParams sp, const T* __restrict__ table, const T* __restrict__ win, const T* __restrict__ gC,
             const int4* __restrict__ ranges, int W, int part_rows, T* __restrict__ part, T* __restrict__ gV,
             T* __restrict__ glnc, int stage, const int* __restrict__ nrows) {
    constexpr int NP = NB * (NB + 1) / 2;
    pdl_begin();
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per_row = W / nw, row = blockIdx.x / per_row;
    if (row >= *nrows) return;
    const int4 rg = ranges[(blockIdx.x % per_row) * nw + wid];
    const int lo = rg.x, hi = rg.y;
    if (lo >= hi) return;                      // warps work alone: no block barrier below
    const int N = sp.N, n_k = sp.n_k, n_z = sp.n_z, n_ell = sp.n_ell, D = sp.D, PK = n_k + 2, Np = (N + 3) & ~3;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V4<T>* acc = reinterpret_cast<V4<T>*>(smem_raw) + (size_t)wid * PK * (stage ? 2 : 1);
    V4<T>* tab = acc + PK;                     // when staged: the four table rows of the current z cell
    const T* src = table + (size_t)row * n_z * n_k;
    const T* lnchi = win + (size_t)row * (NB + 1) * Np;
    const T* V = lnchi + Np;
    T* prow = part + ((size_t)row * part_rows + rg.z) * PK;
    const T* zwp = pick<T>(sp.zw4d, sp.zw4f);
    const T* lnell = pick<T>(sp.lnell, sp.lnell_f);
    const T lkmin = pick_s<T>(sp.lnk_min, sp.lnk_min_f), lkmax = pick_s<T>(sp.lnk_max, sp.lnk_max_f);
    const T inv_dk = pick_s<T>(1.0 / sp.dlnk, sp.inv_dlnk_f);
    for (int l0 = 0; l0 < n_ell; l0 += 32) {
        const int l = l0 + lane;
        const bool act = l < n_ell;
        const T lne = lnell[act ? l : n_ell - 1];
        T G[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) G[p] = act ? gC[(size_t)row * D + p * n_ell + l] : T(0);
        int jc = sp.zrp[lo], ik = -1;
        T c[4][4], a[4][4];                    // [column tap][row tap]
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) { c[q][r] = T(0); a[q][r] = T(0); }
        auto load_rows = [&]() {
            if (stage)
                for (int k = lane; k < PK; k += 32)
                    tab[k] = V4<T>{padded(src, n_z, n_k, jc, k), padded(src, n_z, n_k, jc + 1, k),
                                   padded(src, n_z, n_k, jc + 2, k), padded(src, n_z, n_k, jc + 3, k)};
        };
        // add the register gradients of the lanes with f to their columns
        auto flush = [&](bool f) {
            const unsigned same = __match_any_sync(0xffffffffu, f ? ik : -1 - lane);
            const int turn = __popc(same & ((1u << lane) - 1u));
            for (int t = 0; __any_sync(0xffffffffu, f && turn >= t); ++t) {
                const bool mine = f && turn == t;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (mine) {
                        V4<T> s = acc[ik + q];
                        s.x += a[q][0]; s.y += a[q][1]; s.z += a[q][2]; s.w += a[q][3];
                        acc[ik + q] = s;
                    }
                    __syncwarp();
                }
            }
        };
        // rows jc .. to - 1 are complete for this warp: write them out, shift the rest
        auto advance = [&](int to) {
            const int n = to - jc;
            T* out = prow + (size_t)(jc - rg.w) * PK;
            for (int k = lane; k < PK; k += 32) {
                V4<T> s = acc[k];
                for (int i = 0; i < n; ++i) {
                    T* o = out + (size_t)i * PK + k;
                    *o = l0 ? *o + s.x : s.x;
                    s = V4<T>{s.y, s.z, s.w, T(0)};
                }
                acc[k] = s;
            }
            __syncwarp();
        };
        for (int k = lane; k < PK; k += 32) acc[k] = V4<T>{T(0), T(0), T(0), T(0)};
        load_rows();
        __syncwarp();
        // node constants one node ahead
        int zr_n = jc;
        T lc_n = lnchi[lo], w_n[4], v_n[NB];
#pragma unroll
        for (int r = 0; r < 4; ++r) w_n[r] = zwp[4 * lo + r];
#pragma unroll
        for (int i = 0; i < NB; ++i) v_n[i] = V[i * Np + lo];
#pragma unroll 1
        for (int n = lo; n < hi; ++n) {
            const int zr = zr_n;
            const T lc = lc_n;
            T wz[4], vv[NB];
#pragma unroll
            for (int r = 0; r < 4; ++r) wz[r] = w_n[r];
#pragma unroll
            for (int i = 0; i < NB; ++i) vv[i] = v_n[i];
            if (n + 1 < hi) {
                zr_n = sp.zrp[n + 1];
                lc_n = lnchi[n + 1];
#pragma unroll
                for (int r = 0; r < 4; ++r) w_n[r] = zwp[4 * (n + 1) + r];
#pragma unroll
                for (int i = 0; i < NB; ++i) v_n[i] = V[i * Np + n + 1];
            }
            if (zr != jc) {
                flush(ik >= 0);
                advance(zr);
                jc = zr;
                ik = -1;
                load_rows();
                __syncwarp();
            }
            const T s_raw = lne - lc;
            const bool clamped = (s_raw < lkmin) || (s_raw > lkmax);
            const T uk = (fmin(fmax(s_raw, lkmin), lkmax) - lkmin) * inv_dk;
            const int ik_n = min(max((int)floor(uk), 0), n_k - 2);
            const bool move = act && ik_n != ik;
            if (__any_sync(0xffffffffu, move)) {
                flush(move && ik >= 0);
                if (move) {
                    ik = ik_n;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        V4<T> s;
                        if (stage) s = tab[ik + q];
                        else s = V4<T>{padded(src, n_z, n_k, jc, ik + q), padded(src, n_z, n_k, jc + 1, ik + q),
                                       padded(src, n_z, n_k, jc + 2, ik + q), padded(src, n_z, n_k, jc + 3, ik + q)};
                        c[q][0] = s.x; c[q][1] = s.y; c[q][2] = s.z; c[q][3] = s.w;
                        a[q][0] = a[q][1] = a[q][2] = a[q][3] = T(0);
                    }
                }
                __syncwarp();
            }
            // doubled Catmull-Rom weights in ln k and their derivatives (the z-weights are doubled too)
            const T t = uk - (T)ik_n, t2 = t * t;
            const T wk[4] = {t * (t * (T(2) - t) - T(1)), T(2) + t2 * (T(3) * t - T(5)),
                             t * (T(1) + t * (T(4) - T(3) * t)), t2 * (t - T(1))};
            const T dk[4] = {T(-1) + t * (T(4) - T(3) * t), t * (T(9) * t - T(10)), T(1) + t * (T(8) - T(9) * t),
                             t * (T(3) * t - T(2))};
            T v = T(0), dv = T(0);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const T col = wz[0] * c[q][0] + wz[1] * c[q][1] + wz[2] * c[q][2] + wz[3] * c[q][3];
                v = fma(wk[q], col, v);
                dv = fma(dk[q], col, dv);
            }
            const T Pw = p10(T(0.25) * v);
            // h_i = sum_{j >= i} G_ij V_j; g_P = sum_i V_i h_i; g_V_i = P (h_i + sum_{j <= i} G_ji V_j)
            T red[8];
            T gP = T(0);
#pragma unroll
            for (int i = 0; i < 8; ++i) red[i] = T(0);
            {
                int p = 0;
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    T h = T(0);
#pragma unroll
                    for (int j = i; j < NB; ++j) {
                        h = fma(G[p], vv[j], h);
                        red[j] = fma(G[p], vv[i], red[j]);
                        ++p;
                    }
                    gP = fma(vv[i], h, gP);
                    red[i] += h;
                }
            }
#pragma unroll
            for (int i = 0; i < NB; ++i) red[i] *= Pw;
            const T gv = gP * Pw * (T)(kLn10 * 0.25);     // d log L / d (doubled-weight sum)
            red[NB] = clamped ? T(0) : -gv * dv * inv_dk; // s = ln(ell + 1/2) - ln chi
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const T g = gv * wz[r];
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q][r] = fma(g, wk[q], a[q][r]);
            }
            T sum = warp_transpose_sum8(red);
            if (lane <= NB) {
                T* o = lane < NB ? gV + ((size_t)row * NB + lane) * N + n : glnc + (size_t)row * N + n;
                *o = l0 ? *o + sum : sum;
            }
        }
        flush(ik >= 0);
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
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    const int PK = n_k + 2;
    const T* p = part + (size_t)row * part_rows * PK;
    auto at = [&](int r, int c) {
        T s = T(0);
        for (int x = ptr[r]; x < ptr[r + 1]; ++x) s += p[(size_t)idx[x] * PK + c];
        return s;
    };
    auto cols = [&](int r, int c) {
        T s = at(r, c);
        if (c <= 2) s += (c == 1 ? T(2) : T(-1)) * at(r, 0);
        if (c >= n_k - 1) s += (c == n_k ? T(2) : T(-1)) * at(r, n_k + 1);
        return s;
    };
    for (int i = blockIdx.y * 256 + threadIdx.x; i < n_z * n_k; i += gridDim.y * 256) {
        const int r = i / n_k + 1, c = i % n_k + 1;
        T s = cols(r, c);
        if (r <= 2) s += (r == 1 ? T(2) : T(-1)) * cols(0, c);
        if (r >= n_z - 1) s += (r == n_z ? T(2) : T(-1)) * cols(n_z + 1, c);
        out.put(row, i, n_z * n_k, s);
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
constexpr int kWinAdjThreads = 512;

// elements of the per-evaluation arrays of k_windows_adj
__host__ __device__ inline size_t windows_adj_elems(int N, int nb) { return (size_t)(10 + 4 * nb) * N; }

template <typename T, int NB>
__global__ void __launch_bounds__(kWinAdjThreads)
k_windows_adj(const ShearParams sp, const double* __restrict__ theta_full, const T* __restrict__ gV,
              const T* __restrict__ glnc, T* __restrict__ scratch, double* __restrict__ gfull,
              const int* __restrict__ nrows) {
    pdl_begin();
    const int row = blockIdx.x;
    if (row >= *nrows) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = sp.N, tid = threadIdx.x, nt = kWinAdjThreads, lane = tid & 31, wid = tid >> 5;
    T* S = scratch ? scratch + (size_t)row * windows_adj_elems(N, NB) : reinterpret_cast<T*>(smem_raw);
    T *chi = S, *Ez = S + N, *Dg = S + 2 * N, *omw = S + 3 * N, *fg = S + 4 * N;
    T *gchi = S + 5 * N, *gE = S + 6 * N, *gomw = S + 7 * N, *t1 = S + 8 * N, *t2 = S + 9 * N;
    T *raw = S + 10 * N, *nchi = raw + NB * N, *E0 = nchi + NB * N, *E1 = E0 + NB * N;
    constexpr int NS = S_COUNT + 3 * NB, NR = NS > 2 * NB ? NS : 2 * NB;
    __shared__ T red[(kWinAdjThreads / 32) * NR];
    __shared__ T th[16];
    const T* a_ = pick<T>(sp.a, sp.a_f);
    const T* lna_ = pick<T>(sp.lna, sp.lna_f);
    const T* z_ = pick<T>(sp.z, sp.z_f);
    const T* wa_ = pick<T>(sp.wa, sp.wa_f);
    const T* nz_mu = pick<T>(sp.nz_mean, sp.nz_mean_f);
    const T* nz_sg = pick<T>(sp.nz_sigma, sp.nz_sigma_f);
    const T ia_piv = pick_s<T>(sp.ia_pivot, sp.ia_pivot_f), c1rho = pick_s<T>(sp.c1rho, sp.c1rho_f);
    if (tid < 11 + NB) th[tid] = (T)theta_full[(size_t)row * sp.n_params + tid];
    __syncthreads();
    const T h = th[2];
    const T om = (th[0] + th[1]) / (h * h);
    const T w0 = th[5], wa = th[6];
    const T pde = T(3) * (T(1) + w0 + wa);
    const T chiH = T(kCover100) / h;
    const T gamma = T(0.55) + T(0.05) * (T(1) + w0 + T(0.5) * wa);
    const T pref = T(1.5) * om / (chiH * chiH);
    const T A_IA = th[9], eta = th[10];
    T sum[NS];                                  // scalars, then per bin: g_nchi nchi u / sigma, g_nchi nchi, d norm / d D_z
#pragma unroll
    for (int q = 0; q < NS; ++q) sum[q] = T(0);

    // ---- forward
    for (int n = tid; n < N; n += nt) {
        const T a = a_[n], lna = lna_[n];
        const T de = ex<T>(-pde * lna - T(3) * wa * (T(1) - a));
        Ez[n] = sqrt(om * ex<T>(T(-3) * lna) + (T(1) - om) * de);
        T inc = T(0);
        if (n < N - 1) {
            const T a1 = a_[n + 1];
            const T mid = T(0.5) * (a + a1), half = T(0.5) * (a - a1);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const T ag = mid + half * glx<T>(g);
                const T e2 = om / (ag * ag * ag) + (T(1) - om) * ex<T>(-pde * lg<T>(ag) - T(3) * wa * (T(1) - ag));
                inc += glw<T>(g) / (ag * ag * sqrt(e2));
            }
            inc *= chiH * half;
        }
        chi[n] = inc;
    }
    __syncthreads();
    block_scan<1, false>(chi, N, N, red);
    T pn[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) pn[i] = T(0);
    for (int n = tid; n < N; n += nt) {
        const T e = Ez[n], ia2 = wa_[n] / (a_[n] * a_[n]);
        const T oma = om * ex<T>(T(-3) * lna_[n]) / (e * e);
        fg[n] = ex<T>(gamma * lg<T>(oma));
        omw[n] = ia2 * chiH / e;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const T u = (z_[n] - th[11 + i] - nz_mu[i]) / nz_sg[i];
            const T rw = ex<T>(T(-0.5) * u * u);
            raw[i * N + n] = rw;
            pn[i] += ia2 * rw;
            sum[S_COUNT + 2 * NB + i] += ia2 * rw * u / nz_sg[i];
        }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const T s = warp_sum(pn[i]);
        if (lane == 0) red[wid * NB + i] = s;
    }
    __syncthreads();
    T norm[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        norm[i] = T(0);
        for (int w = 0; w < nt / 32; ++w) norm[i] += red[w * NB + i];
    }
    __syncthreads();
    for (int n = tid; n < N; n += nt) {
        Dg[n] = (n < N - 1) ? T(0.5) * (fg[n] + fg[n + 1]) * (lna_[n] - lna_[n + 1]) : T(0);
        const T o = omw[n], ic = n >= 1 ? T(1) / chi[n] : T(0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const T nc = raw[i * N + n] * Ez[n] / (chiH * norm[i]);
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
        Dg[n] = D_n;
        if (n == 0) {                           // carries no window value
            for (int i = 0; i < NB; ++i) { raw[i * N] = T(0); E0[i * N] = T(0); E1[i * N] = T(0); }
            gchi[0] = T(0); gomw[0] = T(0); t1[0] = T(0);
            continue;
        }
        const T c = chi[n], an = a_[n], so = sqrt(omw[n]), ic = T(1) / c;
        const T lq = lg<T>((T(1) + z_[n]) / ia_piv);
        const T ampc = ex<T>(eta * lq) * c1rho * om / D_n;   // amp = A_IA * ampc
        const T pc = pref * c / an;
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
            sum[S_PREF] += gpc * c / an;
            g_c += gpc * pref / an - gW * pc * e1;
            E0[i * N + n] = gW * pc;            // the adjoints take the place of the suffix sums
            E1[i * N + n] = -gW * pc * c;
            g_amp += -gW * nc;
            raw[i * N + n] = -gW * A_IA * ampc; // g_nchi, direct term
        }
        gomw[n] = g_so * T(0.5) / so;
        gchi[n] = glnc[(size_t)row * N + n] * ic + g_c;
        sum[S_AIA] += g_amp * ampc;
        sum[S_ETA] += g_amp * A_IA * ampc * lq;
        sum[S_OM] += g_amp * A_IA * ampc / om;
        t1[n] = g_amp * A_IA * ampc;            // g_S = -g_D D, g_D = -g_amp amp / D
    }
    __syncthreads();
    // E0_i(n) = sum_{m>n} omw_m nchi_m  ->  G0(m) = sum_{n<m} gE0(n)
    block_scan<2 * NB, false>(E0, N, N, red);
    for (int m = tid; m < N; m += nt) {
        const T e = Ez[m], o = omw[m];
        T go = gomw[m], gc = gchi[m], ge = T(0);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            T gnc = raw[i * N + m];
            const T nc = nchi[i * N + m];
            if (m >= 1) {
                const T ic = T(1) / chi[m];
                const T G0 = E0[i * N + m], G1 = E1[i * N + m] * ic, G = G0 + G1;
                go += nc * G;
                gnc += o * G;
                gc += -o * nc * G1 * ic;
            }
            // nchi = raw E / (chiH norm); raw and norm depend on D_z through u
            const T u = (z_[m] - th[11 + i] - nz_mu[i]) / nz_sg[i];
            const T gn = gnc * nc;
            ge += gn / e;
            sum[S_COUNT + i] += gn * u / nz_sg[i];
            sum[S_COUNT + NB + i] += gn;
        }
        // omw = wa chiH / (a^2 E)
        sum[S_CHIH] += go * o / chiH;
        gE[m] = ge - go * o / e;
        t2[m] = gc;
    }
    __syncthreads();
    // growth: D_n = exp(-S_n), S_n = sum_{m<n} seg_m -> g_seg_m = sum_{n>m} g_S_n;
    // distances: chi_n = sum_{m<n} dchi_m -> g_dchi_m = sum_{n>m} g_chi_n
    block_scan<2, true>(t1, N, N, red);
    for (int m = tid; m < N; m += nt) {
        const T a = a_[m], lna = lna_[m], e = Ez[m];
        T gf = T(0);
        if (m < N - 1) gf += T(0.5) * t1[m] * (lna - lna_[m + 1]);
        if (m >= 1) gf += T(0.5) * t1[m - 1] * (lna_[m - 1] - lna);
        const T ia3 = ex<T>(T(-3) * lna);
        const T oma = om * ia3 / (e * e);
        const T gff = gf * fg[m];
        sum[S_GAMMA] += gff * lg<T>(oma);
        sum[S_OM] += gff * gamma / om;
        // node E: E^2 = om a^-3 + (1 - om) de
        const T ge2 = (gE[m] - T(2) * gff * gamma / e) / (T(2) * e);
        const T de = ex<T>(-pde * lna - T(3) * wa * (T(1) - a));
        sum[S_OM] += ge2 * (ia3 - de);
        sum[S_W0] += ge2 * (T(1) - om) * de * (T(-3) * lna);
        sum[S_WA] += ge2 * (T(1) - om) * de * (T(-3) * lna - T(3) * (T(1) - a));
        if (m < N - 1) {
            const T g = t2[m], a1 = a_[m + 1];
            const T mid = T(0.5) * (a + a1), half = T(0.5) * (a - a1);
            T inc = T(0);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const T ag = mid + half * glx<T>(q);
                const T lgg = lg<T>(ag), i3 = T(1) / (ag * ag * ag);
                const T deg = ex<T>(-pde * lgg - T(3) * wa * (T(1) - ag));
                const T e2 = om * i3 + (T(1) - om) * deg;
                const T F = T(1) / (ag * ag * sqrt(e2));
                inc += glw<T>(q) * F;
                const T gE2 = g * chiH * half * glw<T>(q) * T(-0.5) * F / e2;
                sum[S_OM] += gE2 * (i3 - deg);
                sum[S_W0] += gE2 * (T(1) - om) * deg * (T(-3) * lgg);
                sum[S_WA] += gE2 * (T(1) - om) * deg * (T(-3) * lgg - T(3) * (T(1) - ag));
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
            chih -= gn / chiH;                  // nchi ~ 1 / chiH
            g[11 + i] += (double)(gs[S_COUNT + i] - gn / norm[i] * gs[S_COUNT + 2 * NB + i]);
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

// Warps per evaluation: eight keep the chip's 2432 resident warps busy from 304
// evaluations on; fewer evaluations get shorter node ranges (64 evaluations of
// the 39-d problem: 32 warps).
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
    NS_TRY(alloc(n * sp.D, &a->resid));
    NS_TRY(alloc(n * sp.D, &a->C));
    NS_TRY(alloc(n * sp.D, &a->gC));
    NS_TRY(alloc(n * sp.nb * sp.N, &a->gV));
    NS_TRY(alloc(n * sp.N, &a->glnc));
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
    NS_TRY((launch_windows<T, false>(sp, theta_full, (T*)a->win, nrows, grid_rows, a->side)));
    NS_CUDA_TRY(cudaEventRecord(a->ev_join, a->side));
    return NS_OK;
}

template <typename T, int RB>
static int launch_chi2_adj(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const T* LinvT,
                           const T* Linv, double c0, double* gfull, double* logL, const int* nrows, int grid_rows,
                           cudaStream_t st) {
    const size_t smem = sizeof(T) * RB * (2 * (size_t)sp.D + sp.nb + sp.n_pairs + 8 * (size_t)sp.n_tmpl);
    static bool attr = false;
    if (!attr) {
        NS_CUDA_TRY(cudaFuncSetAttribute(adj::k_chi2_adj<T, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax));
        attr = true;
    }
    NS_CUDA_TRY(launch_pdl(adj::k_chi2_adj<T, RB>, dim3((grid_rows + RB - 1) / RB), dim3(256), smem, st, sp, theta_full,
                           (const T*)a->resid, (const T*)a->C, LinvT, Linv, c0, (T*)a->gC, gfull, logL, nrows));
    return NS_OK;
}

template <typename T, int NB>
static int launch_reverse(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const T* table,
                          const TableGrad& out, double* gfull, const int* nrows, int grid_rows, cudaStream_t st) {
    const int k = limber_adj_split(grid_rows), W = 8 << k, PK = sp.n_k + 2;
    // a warp's columns of gradients and of the current table rows; the rows stay
    // in global memory, and CTAs shrink to one warp, where tables are very wide
    const size_t col = sizeof(adj::V4<T>) * (size_t)PK;
    const int stage = 2 * col <= kAdjSmemMax;
    int nw = kAdjWarps;
    while (nw > 1 && nw * col * (stage ? 2 : 1) > kAdjSmemMax) nw >>= 1;
    const size_t smem = nw * col * (stage ? 2 : 1);
    if (smem > kAdjSmemMax) return NS_ENOTSUP;
    static bool attr = false;
    if (!attr) {
        NS_CUDA_TRY(cudaFuncSetAttribute(adj::k_limber_adj<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax));
        NS_CUDA_TRY(cudaFuncSetAttribute(adj::k_windows_adj<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax));
        attr = true;
    }
    NS_CUDA_TRY(launch_pdl(adj::k_limber_adj<T, NB>, dim3(grid_rows * (W / nw)), dim3(32 * nw), smem, st, sp, table,
                           (const T*)a->win, (const T*)a->gC, (const int4*)a->ranges[k], W, a->part_rows[k],
                           (T*)a->part, (T*)a->gV, (T*)a->glnc, stage, nrows));
    const dim3 g(grid_rows, grid_rows < 256 ? 8 : 2);
    if constexpr (sizeof(T) == 8) {
        NS_CUDA_TRY(launch_pdl(adj::k_table_adj<T, adj::OutT64>, g, dim3(256), 0, st, (const T*)a->part, a->part_rows[k],
                               (const int*)a->ptr[k], (const int*)a->idx[k], sp.n_z, sp.n_k,
                               adj::OutT64{(double*)out.table}, nrows));
    } else {
        NS_CUDA_TRY(launch_pdl(adj::k_table_adj<T, adj::OutT32>, g, dim3(256), 0, st, (const T*)a->part, a->part_rows[k],
                               (const int*)a->ptr[k], (const int*)a->idx[k], sp.n_z, sp.n_k,
                               adj::OutT32{(float*)out.table}, nrows));
    }
    NS_CUDA_TRY(launch_pdl(adj::k_windows_adj<T, NB>, dim3(grid_rows), dim3(adj::kWinAdjThreads), a->win_smem, st, sp,
                           theta_full, (const T*)a->gV, (const T*)a->glnc, (T*)a->scratch, gfull, nrows));
    return NS_OK;
}

template <typename T>
int launch_projection_adj(const ShearParams& sp, ProjectionAdj* a, const double* theta_full, const T* table,
                          const T* LinvT, const T* Linv, double c0, const TableGrad& out, double* gfull, double* logL,
                          const int* nrows, int grid_rows, int* err, cudaStream_t st) {
    NS_CUDA_TRY(cudaStreamWaitEvent(st, a->ev_join, 0));
    NS_TRY((launch_limber<T, false>(sp, theta_full, table, (const T*)a->win, (T*)a->resid, nullptr, nrows, grid_rows,
                                    err, st, (T*)a->C)));
    // two rows per block spread few rows over the chip, eight share the reads of L^-1
    if (grid_rows < 1024)
        NS_TRY((launch_chi2_adj<T, 2>(sp, a, theta_full, LinvT, Linv, c0, gfull, logL, nrows, grid_rows, st)));
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
                                          const T*, double, const TableGrad&, double*, double*, const int*, int,      \
                                          int*, cudaStream_t);
NS_INST(double)
NS_INST(float)
#undef NS_INST

}  // namespace gpuns
