// Row transforms of the IIM solve: DST-I of lines of n = 2^4 .. 2^11 points,
// X_k = sum_{j=1}^{n-1} x_j sin(pi j k / n), through three complex FFTs of n/4 points.
//
// With m = n/2 and M = n/4, the line is folded into its parts odd and even about the middle,
//   w_j = x_j + x_{n-j}  (j = 0..m, x_0 = x_n = 0),     d_j = x_j - x_{n-j}  (j = 0..m-1):
//   X_{2k+1} is the DST-III of w -- as a DCT-III of w reversed, the inverse real FFT of length m of
//     V_j = e^{i pi j / n} (w_{m-j} - i w_j) / 2, evaluated as an M-point complex FFT (Makhoul, "A fast
//     cosine transform in one and two dimensions", 1980); with t = e^{i pi j / n}, p = w_{m-j} - i w_j
//     and q = e^{-i pi/4} (w_{M+j} + i w_{M-j}) its input is G_j = (t (p + q) + i t^5 (p - q)) / 2;
//   X_{2k} is the DST-I of d (m points), minus the imaginary part of the real FFT of d padded with
//     zeros to length 2m: the packed pairs c_t = d_{2t} + i d_{2t+1}, t < M, transformed as M points
//     give its even frequencies, and c_t e^{-2 pi i t / 2M} its odd ones.
// Every step is a rotation or a butterfly of size O(1), so the rounding error grows like log n.  The
// packing of the line into one n/2-point FFT (dst.cuh: sin(j pi/n) (x_j + x_{n-j}) + (x_j - x_{n-j}) / 2
// and a running sum of the odd outputs) costs as many points and loses a factor of about sqrt(n):
// relative error of a white FP32 line of 1024 points 1.3e-6 against 1.2e-7 here.  In the mixed solve
// that noise, differenced at weight 1/h^2, is what a refinement leaves of the residual.
//
// The threads of a group share its lines.  Per line: x in one buffer; the fold writes the three FFT
// inputs into the other; Stockham passes ping-pong between the buffers (radix 16 x 16 for n = 1024,
// 16 x 8 for 512, 8 x 8 x 8 for 2048, one butterfly of registers per thread and step; radix 8 / 4 / 2
// loops for the other sizes); the last step combines the frequencies 4k .. 4k + 3 in one thread, which
// hands them to the caller's output as one 16-byte (FP32) vector.  96 threads on two 1024-point lines:
// every pass is exactly one radix-16 butterfly per thread.
#pragma once

#include <type_traits>

#include "dst.cuh"
#include "iim_ops.cuh"

namespace iim {

// N: compile-time line length, 0 any size (one warp per line).  L: lines per block.  With many rows
// L is the largest that gives every thread one butterfly per pass (96 threads; four warps of one line
// each for N = 0); with few, blocks of one line spread them over the SMs: a band of 270 rows of 512
// points in FP64 is 68 blocks of four lines, and the FP64 pipes of the other SMs would idle.
template <int N, int L>
struct Sine {
    static constexpr int kThreads = N == 0 ? 32 : (N == 2048 || L > 1) ? 96 : 64;   // per group
    static constexpr int kLines = N ? L : 1;                                        // per group
    static constexpr int kGroups = N ? 1 : L;                                       // per block
    static constexpr int kBlock = kThreads * kGroups;
};
// Compile-time size a line length runs with, and the lines per block for a launch of `rows` lines: one
// per block below three full blocks per SM.
__host__ __device__ constexpr int sine_path(int n) { return n == 512 || n == 1024 || n == 2048 ? n : 0; }
inline int sine_lines(int n, long rows) {
    const int most = n == 1024 ? 2 : n == 2048 ? 1 : 4;
    return rows >= 3L * sm_count() * most ? most : 1;
}
// Calls go(N, L) with the size and lines per block as integral constants.
template <typename Go>
inline iim_status sine_dispatch(int n, int lines, Go&& go) {
    using std::integral_constant;
    const integral_constant<int, 1> one;
    if (n == 2048) return go(integral_constant<int, 2048>{}, one);
    if (n == 1024) return lines == 2 ? go(integral_constant<int, 1024>{}, integral_constant<int, 2>{})
                                     : go(integral_constant<int, 1024>{}, one);
    const integral_constant<int, 4> four;
    if (n == 512) return lines == 4 ? go(integral_constant<int, 512>{}, four) : go(integral_constant<int, 512>{}, one);
    return lines == 4 ? go(integral_constant<int, 0>{}, four) : go(integral_constant<int, 0>{}, one);
}

// Work arrays hold element i of an FFT at i + i / 16: with 8-byte (16-byte) elements the strided
// stores of a radix pass then fall into distinct banks.  Stride between FFTs in elements (even).
__host__ __device__ constexpr int sine_pad(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int sine_stride(int M) { return (M + M / 16 + 1) & ~1; }
// Elements of one of the two buffers per line.
__host__ __device__ constexpr int sine_buf(int n) { return 3 * sine_stride(n / 4); }
template <typename T>
inline size_t sine_smem(int n, int lines) {
    return (size_t)2 * lines * sine_buf(n) * sizeof(cpx<T>);
}

// Radix of each pass of an M-point FFT, `rem` factors of two left: 16 x 16 (M = 256), 16 x 8 (128),
// else 8 while three are left, then 4 or 2.
__host__ __device__ constexpr int sine_radix(int M, int rem) {
    return (M == 256 && (rem == 8 || rem == 4)) || (M == 128 && rem == 7) ? 16 : rem >= 3 ? 8 : rem == 2 ? 4 : 2;
}
__host__ __device__ constexpr int log2_radix(int R) { return R == 16 ? 4 : R == 8 ? 3 : R == 4 ? 2 : 1; }

// Table of a line length (complex entries; M = n / 4): [0, M) t_j / 2; [M, 2M) i t_j^5 / 2; [2M, 3M)
// e^{-2 pi i t / 2M}; [3M, 5M) (cos, sin)(2 pi k / n) / 2; then, for every pass after the first (Ns = the
// product of the radices before it), e^{-2 pi i k r / (Ns R)} at r Ns + k, r < R, k < Ns.
__host__ __device__ constexpr int sine_region(int n) { return 7 * (n / 4) + 64; }

// e^{-i pi t / n} from the 4096-entry table of e^{-i pi k / 4096}
template <typename T>
__device__ __forceinline__ cpx<T> sine_root(const cpx<T>* __restrict__ g_tw, int n, int shift, int t) {
    t &= 2 * n - 1;
    const cpx<T> w = g_tw[(t & (n - 1)) << shift];
    return t >= n ? cpx<T>{-w.x, -w.y} : w;
}

template <typename T>
__global__ void k_sine_region(const cpx<T>* __restrict__ g_tw, int n, int logn, cpx<T>* __restrict__ out) {
    pdl_wait();
    const int M = n / 4, shift = kTwLog - logn;
    const T hf = T(0.5);
    for (int e = threadIdx.x; e < 5 * M; e += blockDim.x) {
        cpx<T> v;
        if (e < M) {                      // t / 2, t = conj(root(j))
            v = sine_root(g_tw, n, shift, e);
            v = {hf * v.x, -hf * v.y};
        } else if (e < 2 * M) {           // i conj(root(5 j)) / 2
            v = sine_root(g_tw, n, shift, 5 * (e - M));
            v = {hf * v.y, hf * v.x};
        } else if (e < 3 * M) {
            v = sine_root(g_tw, n, shift, 4 * (e - 2 * M));
        } else {
            v = sine_root(g_tw, n, shift, 2 * (e - 3 * M));
            v = {hf * v.x, -hf * v.y};
        }
        out[e] = v;
    }
    int off = 5 * M, Ns = 1, rem = logn - 2;
    while (rem > 0) {
        const int R = sine_radix(M, rem);
        if (Ns > 1) {
            for (int e = threadIdx.x; e < R * Ns; e += blockDim.x) {
                const int r = e / Ns, k = e - r * Ns;
                out[off + e] = sine_root(g_tw, n, shift, (2 * n / (Ns * R)) * k * r);
            }
            off += R * Ns;
        }
        Ns *= R;
        rem -= log2_radix(R);
    }
}

template <int N>
__device__ __forceinline__ void sine_sync() {
    if constexpr (N == 0) __syncwarp();
    else __syncthreads();
}

// The three FFT inputs of every line of the group: x (natural, reals, line stride 2 BUF, slot 0 zero) in
// X, FFT f of line l at P + (l * 3 + f) * FS.
template <typename T, int N, int L>
__device__ __forceinline__ void sine_fold(const T* X, cpx<T>* P, const cpx<T>* __restrict__ tab, int n, int tid) {
    using S = Sine<N, L>;
    const int M = n >> 2, m = n >> 1, FS = sine_stride(M), BUF = 3 * FS;
    const T r2 = T(0.70710678118654752440);
    const int na = M / 2 + 1;
    for (int it = tid; it < S::kLines * na; it += S::kThreads) {
        const int l = S::kLines == 1 ? 0 : it / na, j = it - l * na;
        const T* x = X + (size_t)l * 2 * BUF;
        cpx<T>* A = P + (size_t)l * BUF;
        const T w0 = j ? x[j] + x[n - j] : T(0);
        const T w1 = x[m - j] + x[m + j];                   // w_{m - j}
        const T a = x[M + j] + x[n - M - j], b = x[M - j] + x[n - M + j];
        {
            const T qx = r2 * (a + b), qy = r2 * (b - a);
            const cpx<T> s = {w1 + qx, qy - w0}, d = {w1 - qx, -w0 - qy};
            const cpx<T> t1 = tab[j], t5 = tab[M + j];
            const cpx<T> g1 = cmul(t1, s), g5 = cmul(t5, d);
            A[sine_pad(j)] = {g1.x + g5.x, -(g1.y + g5.y)};
        }
        if (j && 2 * j != M) {                               // the partner M - j sees the same four w
            const T qx = r2 * (w1 + w0), qy = r2 * (w0 - w1);
            const cpx<T> s = {a + qx, qy - b}, d = {a - qx, -b - qy};
            const cpx<T> t1 = tab[M - j], t5 = tab[2 * M - j];
            const cpx<T> g1 = cmul(t1, s), g5 = cmul(t5, d);
            A[sine_pad(M - j)] = {g1.x + g5.x, -(g1.y + g5.y)};
        }
    }
    for (int it = tid; it < S::kLines * M; it += S::kThreads) {
        const int l = S::kLines == 1 ? 0 : it / M, t = it - l * M;
        const T* x = X + (size_t)l * 2 * BUF;
        cpx<T>* B = P + (size_t)l * BUF + FS;
        const vec2_t<T> v = *reinterpret_cast<const vec2_t<T>*>(x + 2 * t);
        const cpx<T> c = {t ? v.x - x[n - 2 * t] : T(0), v.y - x[n - 1 - 2 * t]};
        B[sine_pad(t)] = c;
        B[FS + sine_pad(t)] = cmul(c, tab[2 * M + t]);
    }
}

// One Stockham pass of radix R over the group's FFTs.
template <typename T, int N, int L, int R>
__device__ __forceinline__ void sine_pass(const cpx<T>* in, cpx<T>* out, const cpx<T>* __restrict__ tw, int M, int Ns,
                                          int tid) {
    using S = Sine<N, L>;
    const int J = M / R, FS = sine_stride(M), total = S::kLines * 3 * J;
    for (int b = tid; b < total; b += S::kThreads) {
        const int f = b / J, j = b - f * J;      // FFT f of the group, butterfly j
        const cpx<T>* src = in + (size_t)f * FS;
        cpx<T>* dst = out + (size_t)f * FS;
        cpx<T> v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = src[sine_pad(j + r * J)];
        const int k = j & (Ns - 1);
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[r * Ns + k]);
        }
        dft<T, R>(v);
        const int o = (j - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) dst[sine_pad(o + r * Ns)] = v[r];
    }
}

// Whether sine_transform's last step reads P (even number of passes); its output may then go to Q.
__host__ __device__ constexpr bool sine_ends_in_p(int n) { return !(n == 2048 || n <= 32); }

// DST-I of the group's lines: x in the reals of Q (line l at 2 l BUF, slots 0 .. n-1, slot 0 zero),
// both buffers kLines * BUF entries; every thread of the group has synchronised after writing x.
// emit(line, k, X) gets X_{4k} .. X_{4k+3} (X_0 = 0).
template <typename T, int N, int L, typename Emit>
__device__ __forceinline__ void sine_transform(cpx<T>* P, cpx<T>* Q, const cpx<T>* __restrict__ tab, int n_rt, int tid,
                                               Emit emit) {
    using S = Sine<N, L>;
    const int n = N ? N : n_rt, M = n >> 2, FS = sine_stride(M), BUF = 3 * FS;
    sine_fold<T, N, L>(reinterpret_cast<const T*>(Q), P, tab, n, tid);
    sine_sync<N>();
    const cpx<T>* tw = tab + 5 * M;
    const cpx<T>* F = P;
    if constexpr (N == 1024) {
        sine_pass<T, N, L, 16>(P, Q, tw, 256, 1, tid);
        sine_sync<N>();
        sine_pass<T, N, L, 16>(Q, P, tw, 256, 16, tid);
    } else if constexpr (N == 512) {
        sine_pass<T, N, L, 16>(P, Q, tw, 128, 1, tid);
        sine_sync<N>();
        sine_pass<T, N, L, 8>(Q, P, tw, 128, 16, tid);
    } else if constexpr (N == 2048) {
        sine_pass<T, N, L, 8>(P, Q, tw, 512, 1, tid);
        sine_sync<N>();
        sine_pass<T, N, L, 8>(Q, P, tw, 512, 8, tid);
        sine_sync<N>();
        sine_pass<T, N, L, 8>(P, Q, tw + 64, 512, 64, tid);
        F = Q;
    } else {
        int Ns = 1, rem = 31 - __clz(M);
        cpx<T>* in = P;
        cpx<T>* out = Q;
        while (rem > 0) {
            const int R = sine_radix(0, rem);
            if (R == 8) sine_pass<T, N, L, 8>(in, out, tw, M, Ns, tid);
            else if (R == 4) sine_pass<T, N, L, 4>(in, out, tw, M, Ns, tid);
            else sine_pass<T, N, L, 2>(in, out, tw, M, Ns, tid);
            sine_sync<N>();
            if (Ns > 1) tw += R * Ns;
            Ns *= R;
            rem -= log2_radix(R);
            cpx<T>* t = in; in = out; out = t;
        }
        F = in;
    }
    if constexpr (N != 0) sine_sync<N>();
#pragma unroll 2
    for (int it = tid; it < S::kLines * M; it += S::kThreads) {
        const int l = S::kLines == 1 ? 0 : it / M, k = it - l * M;
        const cpx<T>* A = F + (size_t)l * BUF;
        const cpx<T>* B = A + FS;
        const cpx<T>* C = B + FS;
        const T* u = reinterpret_cast<const T*>(A);
        T X[4];
        const cpx<T> h0 = tab[3 * M + 2 * k], h1 = tab[3 * M + 2 * k + 1];
        {
            const cpx<T> f = B[sine_pad(k)], g = B[sine_pad((M - k) & (M - 1))];
            X[0] = h0.x * (f.x - g.x) + (h0.y * (f.y + g.y) + T(0.5) * (g.y - f.y));
        }
        {
            const cpx<T> f = C[sine_pad(k)], g = C[sine_pad(M - 1 - k)];
            X[2] = h1.x * (f.x - g.x) + (h1.y * (f.y + g.y) + T(0.5) * (g.y - f.y));
        }
        // u_k (real part at even k, minus the imaginary part at odd k), and -u_{m-1-k}
        const int e = 2 * M - 1 - k;
        const T y1 = u[2 * sine_pad(k >> 1) + (k & 1)], y3 = u[2 * sine_pad(e >> 1) + (e & 1)];
        X[1] = (k & 1) ? -y1 : y1;
        X[3] = (k & 1) ? -y3 : y3;
        emit(l, k, X);
    }
}

// X as the aligned vectors of T's output rows
template <typename T>
__device__ __forceinline__ void store4(T* __restrict__ p, const T (&X)[4]) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(X[0], X[1], X[2], X[3]);
    } else {
        reinterpret_cast<double2*>(p)[0] = make_double2(X[0], X[1]);
        reinterpret_cast<double2*>(p)[1] = make_double2(X[2], X[3]);
    }
}

// Forward row transforms.  Row r (interior row index) of the input is
//   dense[r*dld + doff + i] (FP64, optional) + box terms / h^2 (optional ring)
//   + gsign * gamma at the affected points of the row (optional)
// and the transformed row is written to out (padded layout, slot 0 of a row zero).
template <typename T, int N, int L>
__device__ __forceinline__ void
sine_rows_fwd_body(int NX, int NY, int n_rt, int row0, int nrows, const double* __restrict__ dense, int dld, int doff,
                   const double* __restrict__ ring, double ih2, const int* __restrict__ aff_row_ptr,
                   const int* __restrict__ aff_node, VecArg gam, double gsign, const cpx<T>* __restrict__ tab,
                   T* __restrict__ out) {
    using S = Sine<N, L>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = N ? N : n_rt, BUF = sine_buf(n);
    const int grp = N ? 0 : threadIdx.x / S::kThreads, tid = N ? threadIdx.x : threadIdx.x % S::kThreads;
    cpx<T>* P = reinterpret_cast<cpx<T>*>(smem_raw) + (size_t)grp * 2 * S::kLines * BUF;
    cpx<T>* Q = P + (size_t)S::kLines * BUF;
    const int r0 = row0 + (blockIdx.x * S::kGroups + grp) * S::kLines, rend = min(row0 + nrows, NY);
    if (N == 0 && r0 >= rend) return;   // whole warp; a block of the other sizes always has a row
    constexpr int TPL = S::kThreads / S::kLines;   // threads per line while loading
    const int l = tid / TPL, t = tid - l * TPL, r = r0 + l;
    T* x = reinterpret_cast<T*>(Q) + (size_t)l * 2 * BUF;
    const bool live = r < rend;
    if (live && dense && !ring && dld == n && doff == 1) {
        // padded row: 16-byte loads, slot 0 is a zero pad
        const double2* src = reinterpret_cast<const double2*>(dense + (size_t)r * n);
        constexpr int B = N ? (N / 2 + TPL - 1) / TPL : 8;
        for (int q0 = t; q0 < n / 2; q0 += B * TPL) {
            double2 v[B];
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (q0 + b * TPL < n / 2) v[b] = src[q0 + b * TPL];
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (q0 + b * TPL < n / 2) {
                    vec2_t<T> w;
                    w.x = (T)v[b].x;
                    w.y = (T)v[b].y;
                    reinterpret_cast<vec2_t<T>*>(x)[q0 + b * TPL] = w;
                }
        }
        if (t == 0) x[0] = T(0);
    } else if (live && (dense || ring)) {
        // element i + 1 is thread i mod TPL's throughout
        constexpr int B = N ? (N + TPL - 1) / TPL : 8;
        const double* src = dense ? dense + (size_t)r * dld + doff : nullptr;
        for (int i0 = t; i0 < NX; i0 += B * TPL) {
            double v[B];
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (i0 + b * TPL < NX) v[b] = src ? src[i0 + b * TPL] : 0.0;
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (i0 + b * TPL < NX) x[i0 + b * TPL + 1] = (T)v[b];
        }
        if (t == 0) x[0] = T(0);
        if (ring) {   // bottom row (nx+1), top row (nx+1), left column (ny-1), right column (ny-1)
            const int nxp1 = NX + 2;
            if (t == 0) x[1] += (T)(ring[2 * nxp1 + r] * ih2);
            if (t == (NX - 1) % TPL) x[NX] += (T)(ring[2 * nxp1 + NY + r] * ih2);
            for (int edge = 0; edge < 2; ++edge) {
                if (r != (edge ? NY - 1 : 0)) continue;
                const double* g = ring + edge * nxp1 + 1;
#pragma unroll 8
                for (int i = t; i < NX; i += TPL) x[i + 1] += (T)(__ldg(g + i) * ih2);
            }
        }
    } else {
        for (int q = t; q < n / 2; q += TPL) reinterpret_cast<vec2_t<T>*>(x)[q] = vec2_t<T>{T(0), T(0)};
    }
    if (gam.base) {
        sine_sync<N>();
        if (live) {
            const double* gv = gam.get();
            const int a0 = aff_row_ptr[r], a1 = aff_row_ptr[r + 1];
            for (int a = a0 + t; a < a1; a += TPL) x[aff_node[a] - r * n] += (T)(gsign * gv[a]);
        }
    }
    sine_sync<N>();
    sine_transform<T, N, L>(P, Q, tab, n, tid, [&](int ln, int k, const T (&X)[4]) {
        if (r0 + ln < rend) store4<T>(out + (size_t)(r0 + ln) * n + 4 * k, X);
    });
}

// blockIdx.y selects one of several fields: dense input dfs and output ofs elements apart.  `stop`
// (optional): a set flag makes the launch a no-op.
template <typename T, int N, int L>
__global__ void __launch_bounds__((Sine<N, L>::kBlock))
k_sine_rows_fwd(int NX, int NY, int n, int row0, int nrows, const double* __restrict__ dense, int dld, int doff,
                const double* __restrict__ ring, double ih2, const int* __restrict__ aff_row_ptr,
                const int* __restrict__ aff_node, VecArg gam, double gsign, const cpx<T>* __restrict__ tab,
                T* __restrict__ out, const int* __restrict__ stop, long dfs, long ofs) {
    pdl_wait();
    if (stop && *stop) return;
    sine_rows_fwd_body<T, N, L>(NX, NY, n, row0, nrows, dense ? dense + (long)blockIdx.y * dfs : nullptr, dld, doff, ring,
                             ih2, aff_row_ptr, aff_node, gam, gsign, tab, out + (long)blockIdx.y * ofs);
}

// The body constants' step of a correction, psibar += x (circulation bodies), beside the recovery.
struct PsibarStep {
    int ncirc;
    const int* ids;
    const double* x;
    double* psibar;
    __device__ __forceinline__ void apply() const {
        for (int c = threadIdx.x; c < ncirc; c += blockDim.x) psibar[ids[c]] += x[c];
    }
};

// Inverse row transforms of rows [row0, row0 + nrows) of a padded buffer, modes as RowsInvMode (in and outT
// may be the same rows: a block reads its lines before it writes them).
template <typename T, int MODE, int N, int L>
__device__ __forceinline__ void
sine_rows_inv_body(int NX, int NY, int n_rt, int row0, int nrows, const T* in, T* outT,
                   double* __restrict__ out64, int old, int ooff, const uint8_t* __restrict__ cls,
                   const cpx<T>* __restrict__ tab) {
    using S = Sine<N, L>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = N ? N : n_rt, BUF = sine_buf(n);
    const int grp = N ? 0 : threadIdx.x / S::kThreads, tid = N ? threadIdx.x : threadIdx.x % S::kThreads;
    cpx<T>* P = reinterpret_cast<cpx<T>*>(smem_raw) + (size_t)grp * 2 * S::kLines * BUF;
    cpx<T>* Q = P + (size_t)S::kLines * BUF;
    const int r0 = row0 + (blockIdx.x * S::kGroups + grp) * S::kLines, rend = min(row0 + nrows, NY);
    if (N == 0 && r0 >= rend) return;
    constexpr int V = 16 / (int)sizeof(T);
    constexpr int TPL = S::kThreads / S::kLines, B = N ? (N / V + TPL - 1) / TPL : 8;
    const int l = tid / TPL, t = tid - l * TPL, r = r0 + l;
    {
        using VT = vec16_t<T>;
        VT* x = reinterpret_cast<VT*>(reinterpret_cast<T*>(Q) + (size_t)l * 2 * BUF);
        const bool live = r < rend;
        const VT* src = reinterpret_cast<const VT*>(in + (size_t)(live ? r : r0) * n);
        for (int q0 = t; q0 < n / V; q0 += B * TPL) {
            VT v[B];
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (q0 + b * TPL < n / V) v[b] = src[q0 + b * TPL];
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (q0 + b * TPL < n / V) x[q0 + b * TPL] = v[b];
        }
    }
    sine_sync<N>();
    sine_transform<T, N, L>(P, Q, tab, n, tid, [&](int ln, int k, const T (&X)[4]) {
        const int rr = r0 + ln;
        if (rr >= rend) return;
        if constexpr (MODE == INV_STORE_T) {
            store4<T>(outT + (size_t)rr * n + 4 * k, X);
        } else if constexpr (MODE == INV_STORE_F64) {
            double* dst = out64 + (size_t)rr * old + ooff + 4 * k - 1;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (k || e) dst[e] = (double)X[e];
        } else if constexpr (MODE == INV_ACCUM_T) {
            T* dst = outT + (size_t)rr * n + 4 * k;
            T Y[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) Y[e] = dst[e] + X[e];
            store4<T>(dst, Y);
        } else {
            // fluid nodes only: 16-byte FP64 read-modify-writes, one 4-byte class load
            const size_t base = (size_t)rr * n + 4 * k;
            const uchar4 c = *reinterpret_cast<const uchar4*>(cls + base);
            double2* o = reinterpret_cast<double2*>(out64 + base);
            double2 o0 = o[0], o1 = o[1];
            if (c.x <= CLS_PLUS && k) o0.x += (double)X[0];   // slot 0 of a row is a pad
            if (c.y <= CLS_PLUS) o0.y += (double)X[1];
            if (c.z <= CLS_PLUS) o1.x += (double)X[2];
            if (c.w <= CLS_PLUS) o1.y += (double)X[3];
            o[0] = o0;
            o[1] = o1;
        }
    });
}

template <typename T, int MODE, int N, int L>
__global__ void __launch_bounds__((Sine<N, L>::kBlock))
k_sine_rows_inv(int NX, int NY, int n, int row0, int nrows, const T* in, T* outT,
                double* __restrict__ out64, int old, int ooff, const uint8_t* __restrict__ cls,
                const cpx<T>* __restrict__ tab, const int* __restrict__ stop, long fstride, PsibarStep ps) {
    pdl_wait();
    if (stop && *stop) return;
    if (MODE == INV_ACCUM_FLUID && blockIdx.x == 0) ps.apply();
    sine_rows_inv_body<T, MODE, N, L>(NX, NY, n, row0, nrows, in + (long)blockIdx.y * fstride,
                                   outT ? outT + (long)blockIdx.y * fstride : nullptr, out64, old,
                                   ooff + (int)blockIdx.y * old, cls, tab);
}

// s / d of positive d well inside the FP32 range: the FP32 reciprocal and two Newton steps, to about an ulp (a
// division is correctly rounded; the box solve's error against 64 bits is 5e-16 at 64^2 either way, where
// the packed transforms left 1e-15, and 5e-16 at 2048 x 512, where they left 4e-14).
__device__ __forceinline__ double quotient(double s, double d) {
    double r = (double)__frcp_rn((float)d);
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    return s * r;
}

// Column pass of the box solve: DST-I of the columns, division by the eigenvalues
// lam_x + lam_y = (2 - 2 cos(pi p / nx) + 2 - 2 cos(pi q / n)) / h^2, DST-I back.  kLines adjacent padded
// columns per group; `scale` carries the normalisation and h^2; tw: the table of e^{-i pi k / 4096}.
// Each transform leaves its result in the buffer that its last step does not read.  Dynamic shared memory
// sine_smem<T>(n, L).  Bound by FP64 arithmetic; against the packed transforms (dst.cuh), whole box solve in
// FP64: 64^2 45 -> 28 us, 256^2 73 -> 48, 512^2 102 -> 88, 1024^2 303 -> 300, 2048^2 1465 -> 1093,
// 64 x 2048 257 -> 104.  Only at 1024 points is this pass the slower one (162 -> 168 us: 512 blocks of two
// columns leave a fifth of the FP64 pipes idle at the end).
template <typename T, int N, int L>
__global__ void __launch_bounds__((Sine<N, L>::kBlock))
k_sine_cols(int nx, int n_rt, T* __restrict__ buf, T scale, const cpx<T>* __restrict__ tab, const cpx<T>* __restrict__ tw) {
    pdl_wait();
    using S = Sine<N, L>;
    constexpr int KL = S::kLines;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = N ? N : n_rt, BUF = sine_buf(n);
    const int grp = N ? 0 : threadIdx.x / S::kThreads, tid = N ? threadIdx.x : threadIdx.x % S::kThreads;
    cpx<T>* P = reinterpret_cast<cpx<T>*>(smem_raw) + (size_t)grp * 2 * KL * BUF;
    cpx<T>* Q = P + (size_t)KL * BUF;
    const int c0 = (blockIdx.x * S::kGroups + grp) * KL;   // nx is a multiple of L
    T* x = reinterpret_cast<T*>(Q);   // line l at 2 l BUF
    constexpr int B = N ? (KL * N + S::kThreads - 1) / S::kThreads : 8;
    for (int e0 = tid; e0 < KL * n; e0 += B * S::kThreads) {
        T v[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int e = e0 + b * S::kThreads, j = e / KL, l = e % KL;
            v[b] = e < KL * n && j ? buf[(size_t)(j - 1) * nx + c0 + l] : T(0);
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int e = e0 + b * S::kThreads, j = e / KL, l = e % KL;
            if (e < KL * n) x[(size_t)l * 2 * BUF + j] = v[b];
        }
    }
    sine_sync<N>();
    cpx<T>* O = sine_ends_in_p(n) ? Q : P;
    cpx<T>* I = sine_ends_in_p(n) ? P : Q;
    x = reinterpret_cast<T*>(O);
    sine_transform<T, N, L>(P, Q, tab, n, tid, [&](int l, int k, const T (&X)[4]) {
        const T lx = T(2) - T(2) * tw[(c0 + l) * (kTwN / nx)].x;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const T ly = T(2) - T(2) * tw[(4 * k + e) * (kTwN / n)].x;
            x[(size_t)l * 2 * BUF + 4 * k + e] = (k || e) ? X[e] * quotient(scale, lx + ly) : T(0);   // slot 0 stays zero
        }
    });
    sine_sync<N>();
    x = reinterpret_cast<T*>(sine_ends_in_p(n) ? O : I);
    sine_transform<T, N, L>(I, O, tab, n, tid, [&](int l, int k, const T (&X)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) x[(size_t)l * 2 * BUF + 4 * k + e] = X[e];
    });
    sine_sync<N>();
#pragma unroll 4
    for (int e = tid; e < KL * (n - 1); e += S::kThreads) {
        const int j = e / KL, l = e % KL;
        buf[(size_t)j * nx + c0 + l] = x[(size_t)l * 2 * BUF + j + 1];
    }
}

}  // namespace iim
