// Krylov steps of the Schur system on one thread-block cluster per problem.
//
// The steps of a GMRES iteration on vectors of ns = 10^2..10^4 values are short and depend on one
// another: as separate launches each costs its launch and a pass over a few MB, and on one block the
// FP64 pipe of one SM (two lanes per clock) bounds the Gram-Schmidt passes.  A cluster of CL blocks
// owns ns / CL rows each; inner products are exchanged through distributed shared memory (every block
// writes its partial sums to all the others, then one cluster barrier, then every block adds them in
// the same order), so all blocks hold the same scalars bit for bit and take the same decisions.
//   * k_start: norm, tolerance and first basis vector of a correction or a restart.
//   * k_arnoldi: one Arnoldi step (two classical Gram-Schmidt passes, norm, Givens rotations, scaling).
//     1756 unknowns, restart 64 (plain FP64 512^2): six launches of 51 us per step before, 21.5 us here; 9486
//     unknowns, few columns: 50 us before, 17 us here (event times less their overhead).
//   * k_krylov: the whole correction solve with the dense operator (iim_opts.precond 3): start, all
//     iterations z_j = M v_j, v_{j+1} = S z_j, Arnoldi step, restarts, x = sum y_j z_j.  The matrices
//     come from L2 at the rate of CL SMs, so it is used up to kKrylovRows unknowns; basis and z_j stay in
//     shared memory (a global store before a cluster barrier would put its latency into it).  Beyond, the
//     products take the whole GPU (k_dense_matvec) between k_arnoldi launches.  Both forms do the same
//     arithmetic in the same order.
//     1450 unknowns: 38 us per iteration as launches, 23 us here.
#pragma once

#include <cooperative_groups.h>

#include <algorithm>

#include "iim_ops.cuh"

namespace iim {

constexpr int kKrylovThreads = 512;
constexpr int kKrylovRows = 2560;
static_assert(8 * 65 >= kKrylovThreads, "the update's partial sums fit a pass's products");

// Cluster size for ns unknowns (16 needs the non-portable size, which this GPU has), and whether the
// correction solve with the dense operator runs as one cluster.
inline int krylov_cluster(int ns) { return ns <= 512 ? 8 : 16; }
inline bool krylov_fits(int ns) { return ns <= kKrylovRows; }
// Problems of one lockstep group share both.
inline int krylov_class(int ns) { return ns <= 512 ? 0 : krylov_fits(ns) ? 1 : 2; }

// Leading dimension of the dense matrices M and S: rows start on 128-byte lines, columns ns .. ld - 1
// are zero.
__host__ __device__ inline long dense_ld(int ns) { return ((long)ns + 31) & ~31L; }

template <int CL>
struct Cluster {
    static __device__ __forceinline__ int rank() { return (int)cooperative_groups::this_cluster().block_rank(); }
    static __device__ __forceinline__ void sync() { cooperative_groups::this_cluster().sync(); }
    template <typename P>
    static __device__ __forceinline__ P* at(P* p, int r) { return cooperative_groups::this_cluster().map_shared_rank(p, r); }
};

// Shared scratch of the steps: partial sums of the two passes and of a norm, coefficients (entry j + 1 of
// the second pass: the squared norm before it), rotations.
template <int CL>
struct KrylovShared {
    double part[3][CL][65];  // part[0] also holds the updates' partial sums
    double h[65], hc[64], cs[64], sn[64];
    double sq, nrm, inv;     // the last squared norm, the norm and its reciprocal (0 for a zero norm)
    double resid;
};

// Squared norm, norm and reciprocal of w over the cluster (this block's rows w[0..nr)) into s, the same in
// every block; ends synchronised.  One warp does the scalar work: an FP64 instruction occupies the pipe
// for 16 cycles per warp, so a square root or division repeated by 16 warps would cost microseconds.
template <int CL>
__device__ __forceinline__ void norm_cluster(const double* w, int nr, KrylovShared<CL>& s) {
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        double acc = 0.0;
        for (int e = lane; e < nr; e += 32) acc += w[e] * w[e];
        acc = warp_sum(acc);
        if (lane < CL) *Cluster<CL>::at(&s.part[2][Cluster<CL>::rank()][0], lane) = acc;
    }
    Cluster<CL>::sync();
    if (threadIdx.x < 32) {
        const double t = warp_sum(lane < CL ? s.part[2][lane][0] : 0.0);
        const double n = sqrt(t);
        if (lane == 0) {
            s.sq = t;
            s.nrm = n;
            s.inv = n > 0.0 ? 1.0 / n : 0.0;
        }
    }
    __syncthreads();
}

// The absolute Krylov tolerance of a correction with right-hand side norm `beta`.
__device__ __forceinline__ double krylov_tolerance(const KTol& t, double beta, const double* small) {
    const double a = t.rel * beta;
    return t.kappa > 0.0 ? fmin(a, fmax(t.kappa * sqrt(small[SM_RES2]), t.last * small[SM_FNORM])) : a;
}

// Start of a correction (init_maxit >= 0: counters, ||b||^2, tolerance) or of a restart cycle from the
// residual r: V_0 = r / ||r||, gv = (||r||, 0, ...), the stop flag set when there is nothing to do.
template <int CL>
__device__ __forceinline__ void start_cluster_body(int ns, const double* __restrict__ r, double* __restrict__ v0,
                                                   KLayout L, double* __restrict__ K, int* __restrict__ di,
                                                   int init_maxit, KTol tol, double* __restrict__ small) {
    constexpr int NT = kKrylovThreads;
    __shared__ KrylovShared<CL> s;
    extern __shared__ double s_w[];
    const int tid = threadIdx.x, rank = Cluster<CL>::rank();
    const int R = (ns + CL - 1) / CL, r0 = min(rank * R, ns), nr = min(R, ns - r0);
    for (int e = tid; e < nr; e += NT) s_w[e] = r[r0 + e];
    Cluster<CL>::sync();
    norm_cluster<CL>(s_w, nr, s);
    const double b2 = s.sq, beta = s.nrm;
    for (int e = tid; e < nr; e += NT) v0[r0 + e] = s_w[e] * s.inv;
    if (rank == 0) {
        for (int i = tid; i <= L.m; i += NT) K[L.gv() + i] = i ? 0.0 : beta;
        if (tid == 0) {
            if (init_maxit >= 0) {
                small[SM_NORM] = b2;
                di[DI_IT] = 0;
                di[DI_MAXIT] = init_maxit;
                di[DI_CONV] = 0;
                di[DI_TMPJ] = 0;
                di[DI_LOOP] = 0;
                di[DI_LOOPERR] = 0;
                K[L.scal() + SC_TOL] = krylov_tolerance(tol, beta, small);
            }
            K[L.scal() + SC_BETA] = beta;
            K[L.scal() + SC_RESID] = beta;
            di[DI_J] = 0;
            int stop = di[DI_IT] >= di[DI_MAXIT] ? 1 : 0;
            if (!(beta > K[L.scal() + SC_TOL])) {
                di[DI_CONV] = 1;
                stop = 1;
            }
            di[DI_STOP] = stop;
        }
    }
}

// Two classical Gram-Schmidt passes of w (this block's rows w[0..nr)) against V_0..V_j (this block's rows,
// column i at V + i ldv) and the norm of the result (s.nrm, s.inv); s.hc[i] = the two passes'
// coefficients summed.  The norm comes with the second pass's products, ||w||^2 less the squares of its
// coefficients (V is orthonormal), which saves an exchange; where they are not small against ||w||^2 the
// norm is taken of the result itself.  Ends synchronised.
template <int CL, int NT>
__device__ __forceinline__ void orthogonalise(const double* V, long ldv, int j, int nr, double* w, KrylovShared<CL>& s) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = Cluster<CL>::rank();
    // many columns (plain GMRES): 1756 unknowns, 64 columns, a step 23.5 -> 21.5 us on average; with few the
    // extra barrier costs more than it saves (a 2048^2 solve of 14 iterations 3.13 -> 3.25 ms)
    const bool wide = j >= NW;
    for (int pass = 0; pass < 2; ++pass) {
        // one product per warp while there are warps enough, then four: their loads overlap, and halving
        // exchanges add them with 6 FP64 additions instead of 20
        for (int i = warp; !wide && i <= j + pass; i += NW) {
            const double* vi = i <= j ? V + (long)i * ldv : w;
            double acc = 0.0;
            for (int e = lane; e < nr; e += 32) acc += vi[e] * w[e];
            acc = warp_sum(acc);
            if (lane < CL) *Cluster<CL>::at(&s.part[pass][rank][i], lane) = acc;
        }
        for (int i0 = 4 * warp; wide && i0 <= j + pass; i0 += 4 * NW) {
            const double* vi[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) vi[u] = i0 + u <= j ? V + (long)(i0 + u) * ldv : w;
            double a[4] = {};
#pragma unroll 4
            for (int e = lane; e < nr; e += 32) {
                const double we = w[e];
#pragma unroll
                for (int u = 0; u < 4; ++u) a[u] = fma(vi[u][e], we, a[u]);
            }
#pragma unroll
            for (int half = 2, off = 16; half >= 1; half /= 2, off /= 2) {
                const bool up = lane & off;
#pragma unroll
                for (int u = 0; u < half; ++u) {
                    const double send = up ? a[u] : a[u + half], keep = up ? a[u + half] : a[u];
                    a[u] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                }
            }
#pragma unroll
            for (int off = 4; off >= 1; off /= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], off);
            const int i = i0 + (lane >> 3);   // this lane's product
            if (i <= j + pass)
                for (int c = lane & 7; c < CL; c += 8) *Cluster<CL>::at(&s.part[pass][rank][i], c) = a[0];
        }
        Cluster<CL>::sync();
        if (tid <= j + pass) {
            double a = 0.0;
#pragma unroll
            for (int c = 0; c < CL; ++c) a += s.part[pass][c][tid];
            s.h[tid] = a;
            if (tid <= j) s.hc[tid] = pass ? s.hc[tid] + a : a;
        }
        __syncthreads();
        if (pass && warp == NW - 1) {   // the scalars beside the update below
            double q = 0.0;
            for (int i = lane; i <= j; i += 32) q += s.h[i] * s.h[i];
            const double t = s.h[j + 1], n2 = t - warp_sum(q);
            if (lane == 0) {
                const double n = n2 > 0.0 ? sqrt(n2) : 0.0;
                s.sq = n2 > 0.5 * t ? 1.0 : 0.0;   // whether the difference may stand for the norm
                s.nrm = n;
                s.inv = n > 0.0 ? 1.0 / n : 0.0;
            }
        }
        // update: G groups of threads share the columns of a row (part[0] has been read; nothing writes it
        // from outside before the next cluster barrier)
        const int gw = (nr + 31) & ~31, G = wide && gw > 0 && 2 * gw <= NT ? NT / gw : 1;
        double* red = &s.part[0][0][0];
        if (G > 1) {
            const int g = tid / gw, e = tid - g * gw;
            double a = 0.0;
            if (g < G && e < nr) {
#pragma unroll 4
                for (int i = g; i <= j; i += G) a = fma(s.h[i], V[(long)i * ldv + e], a);
                red[tid] = a;
            }
            __syncthreads();
            if (tid < nr) {
                double t = 0.0;
                for (int q = 0; q < G; ++q) t += red[q * gw + tid];
                w[tid] -= t;
            }
        } else {
            for (int e = tid; e < nr; e += NT) {
                double a = 0.0;
#pragma unroll 4
                for (int i = 0; i <= j; ++i) a = fma(s.h[i], V[(long)i * ldv + e], a);
                w[e] -= a;
            }
        }
        __syncthreads();
    }
    if (s.sq == 0.0) norm_cluster<CL>(w, nr, s);   // the same in every block (NaN and zero vectors too)
}

// Givens rotations of Hessenberg column j (in s.hc, the subdiagonal nrm) with the rotations s.cs, s.sn
// of the columns before it, which the new one joins; col[0..j] is the rotated column; g0 = gv[j] on
// entry, *gj and *gj1 are gv[j] and gv[j + 1] after.  One thread.
template <int CL>
__device__ __forceinline__ void rotate_column(KrylovShared<CL>& s, int j, double nrm, double g0, double* gj, double* gj1) {
    double a = s.hc[0];
    for (int i = 0; i < j; ++i) {
        const double b = s.hc[i + 1];
        s.hc[i] = s.cs[i] * a + s.sn[i] * b;
        a = -s.sn[i] * a + s.cs[i] * b;
    }
    const double d = hypot(a, nrm);
    const double c = d > 0.0 ? a / d : 1.0, t = d > 0.0 ? nrm / d : 0.0;
    s.cs[j] = c;
    s.sn[j] = t;
    s.hc[j] = d;
    *gj1 = -t * g0;
    *gj = c * g0;
}

// One Arnoldi step on V_{j+1} (j = di[DI_J]); rows split over the cluster.
template <int CL>
__device__ __forceinline__ void arnoldi_cluster_body(int* __restrict__ di, double* __restrict__ V, int ns, KLayout L,
                                                     double* __restrict__ K) {
    constexpr int NT = kKrylovThreads;
    __shared__ KrylovShared<CL> s;
    extern __shared__ double s_w[];
    const int tid = threadIdx.x, rank = Cluster<CL>::rank();
    const int j = di[DI_J], off = di[DI_STOP];
    if (off) return;   // the same in every block: set by an earlier kernel
    const int R = (ns + CL - 1) / CL, r0 = min(rank * R, ns), nr = min(R, ns - r0);
    double* wg = V + (long)(j + 1) * ns + r0;
    for (int e = tid; e < nr; e += NT) s_w[e] = wg[e];
    if (rank == 0 && tid < j) {
        s.cs[tid] = K[L.cs() + tid];
        s.sn[tid] = K[L.sn() + tid];
    }
    Cluster<CL>::sync();   // every block runs before one writes to its shared memory
    orthogonalise<CL, NT>(V + r0, ns, j, nr, s_w, s);
    for (int e = tid; e < nr; e += NT) wg[e] = s_w[e] * s.inv;
    if (rank == 0) {
        if (tid == 0) {
            double gj, gj1;
            const double nrm = s.nrm;
            rotate_column<CL>(s, j, nrm, K[L.gv() + j], &gj, &gj1);
            K[L.cs() + j] = s.cs[j];
            K[L.sn() + j] = s.sn[j];
            K[L.gv() + j] = gj;
            K[L.gv() + j + 1] = gj1;
            const double resid = fabs(gj1);
            K[L.scal() + SC_INV] = s.inv;
            K[L.scal() + SC_RESID] = resid;
            const int jn = j + 1, it = di[DI_IT] + 1;
            di[DI_J] = jn;
            di[DI_IT] = it;
            const bool conv = !(resid > K[L.scal() + SC_TOL]);   // also stops on NaN
            if (conv) di[DI_CONV] = 1;
            if (conv || jn >= L.m || it >= di[DI_MAXIT] || nrm == 0.0) di[DI_STOP] = 1;
        }
        __syncthreads();
        double* col = K + L.H() + (long)j * (L.m + 1);
        if (tid <= j) col[tid] = s.hc[tid];
        if (tid == j + 1) col[tid] = 0.0;
    }
}

// s[k] = a[k] . v for NR rows of one warp; v in shared memory, nq float4s (zero padded to a row's leading
// dimension); the sums in every lane.  8 NR 16-byte loads in flight per lane.
template <int NR>
__device__ __forceinline__ void dot_rows(const float* const (&a)[NR], const float* v, int nq, int lane, float (&s)[NR]) {
    const float4* y = reinterpret_cast<const float4*>(v);
    float p[NR][4];
#pragma unroll
    for (int k = 0; k < NR; ++k)
#pragma unroll
        for (int b = 0; b < 4; ++b) p[k][b] = 0.f;
    for (int q = lane; q < nq; q += 8 * 32) {
        float4 u[NR][8];
#pragma unroll
        for (int b = 0; b < 8; ++b)
#pragma unroll
            for (int k = 0; k < NR; ++k)
                u[k][b] = q + 32 * b < nq ? __ldg(reinterpret_cast<const float4*>(a[k]) + q + 32 * b)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            if (q + 32 * b < nq) {
                const float4 t = y[q + 32 * b];
#pragma unroll
                for (int k = 0; k < NR; ++k)
                    p[k][b & 3] = fmaf(u[k][b].x, t.x, fmaf(u[k][b].y, t.y, fmaf(u[k][b].z, t.z, fmaf(u[k][b].w, t.w, p[k][b & 3]))));
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        s[k] = (p[k][0] + p[k][1]) + (p[k][2] + p[k][3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    }
}

// Dense product of the whole GPU: out = A v for A (n x n, leading dimension ld), v = column *jidx of a basis
// (vbase itself without jidx), out = column *jidx + 1 when ostride > 0.  v is staged once per block as FP32;
// the blocks walk the rows, two per warp at a time when there are more rows than warps.  Bound by the
// matrix: from L2 at 10^3 unknowns, from HBM beyond about 5000:
// 9486 unknowns 159 -> 67 us (5.4 TB/s), 1450 unknowns 4.4 -> 3 us.
constexpr int kDenseWarps = 8;
inline int dense_blocks(int n) { return std::min((n + kDenseWarps - 1) / kDenseWarps, 2 * sm_count()); }
inline size_t dense_smem(int n) { return sizeof(float) * (size_t)dense_ld(n); }
__device__ __forceinline__ void dense_matvec_body(int n, const float* __restrict__ A, long ld,
                                                  const double* __restrict__ vbase, const int* __restrict__ jidx,
                                                  long vstride, double* __restrict__ out, long ostride,
                                                  const int* __restrict__ stop) {
    if (stop && *stop) return;
    extern __shared__ __align__(16) float s_vec[];
    const double* v = jidx ? vbase + (long)(*jidx) * vstride : vbase;
    if (ostride) out += (long)(*jidx + 1) * ostride;
    for (int e = threadIdx.x; e < ld; e += kDenseWarps * 32) s_vec[e] = e < n ? (float)v[e] : 0.f;
    __syncthreads();
    const int lane = threadIdx.x & 31, nq = (int)(ld / 4), nw = gridDim.x * kDenseWarps;
    int row = blockIdx.x * kDenseWarps + (threadIdx.x >> 5);
    for (; row + nw < n; row += 2 * nw) {
        float s[2];
        dot_rows<2>({A + (long)row * ld, A + (long)(row + nw) * ld}, s_vec, nq, lane, s);
        if (lane == 0) {
            out[row] = (double)s[0];
            out[row + nw] = (double)s[1];
        }
    }
    if (row < n) {
        float s[1];
        dot_rows<1>({A + (long)row * ld}, s_vec, nq, lane, s);
        if (lane == 0) out[row] = (double)s[0];
    }
}

// Arguments of the whole correction solve.
struct KrylovArgs {
    int ns;
    long ld;                 // dense_ld(ns)
    const float *M, *S;
    const double* b;
    double* x;
    KLayout L;
    double* K;
    int* di;
    double* small;
    KTol tol;
    int max_iter, from_its;  // budget: max_iter, less di[DI_ITS] when from_its
    int cap;                 // most restart cycles
};

// Shared memory: v_j and z_j (all rows, FP32), the rotated columns, gv, y; this block's rows of w, of the
// basis (FP64) and of the z_j (FP32, as the product leaves them).
inline size_t krylov_smem(int ns, int m, int cl) {
    const size_t R = (ns + cl - 1) / cl;
    return 2 * dense_ld(ns) * sizeof(float) + ((size_t)(m + 1) * m + 2 * (m + 1)) * sizeof(double) +
           R * (m + 1) * sizeof(double) + R * m * sizeof(float);
}
inline size_t arnoldi_smem(int ns, int cl) { return (size_t)((ns + cl - 1) / cl) * sizeof(double); }

// Solves S x = b to the tolerance by flexible GMRES with restarts; di and the scalars of K are left as
// the separate kernels leave them.
template <int CL>
__device__ void krylov_body(const KrylovArgs& g) {
    constexpr int NT = kKrylovThreads, NW = NT / 32;
    __shared__ KrylovShared<CL> s;
    extern __shared__ __align__(16) float s_vec[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = Cluster<CL>::rank();
    const int ns = g.ns, m = g.L.m, nq = (int)(g.ld / 4);
    float* vf = s_vec;                                           // v_j, all rows
    float* zf = vf + g.ld;                                       // z_j
    double* H = reinterpret_cast<double*>(zf + g.ld);            // rotated columns, stride m + 1
    double* gv = H + (size_t)(m + 1) * m;
    double* y = gv + m + 1;
    const int R = (ns + CL - 1) / CL, r0 = min(rank * R, ns), nr = min(R, ns - r0);
    double* w = y + m + 1;                                       // this block's rows of the current vector,
    double* V = w + R;                                           // of the basis (column i at i R)
    float* Z = reinterpret_cast<float*>(V + (size_t)R * m);      // and of the z_i
    for (int e = tid; e < 2 * g.ld; e += NT) vf[e] = 0.f;        // the padding stays zero
    for (int e = tid; e < nr; e += NT) g.x[r0 + e] = 0.0;
    const int left = g.from_its ? g.max_iter - g.di[DI_ITS] : g.max_iter;
    const int maxit = max(left, 1);

    // the next basis vector: this block's rows kept, and into every block's FP32 copy
    auto share = [&](int col) {
        double* vc = V + (size_t)col * R;
        for (int e = tid; e < nr; e += NT) {
            vc[e] = w[e] * s.inv;
            vf[r0 + e] = (float)vc[e];
        }
        __syncthreads();
        for (int c = warp; c < CL; c += NW) {
            if (c == rank) continue;
            float* to = Cluster<CL>::at(vf + r0, c);
            for (int e = lane; e < nr; e += 32) to[e] = vf[r0 + e];
        }
    };
    // rows r0 .. of A times the shared vector; put(row, value) in every lane of the row's warp
    auto product = [&](const float* A, const float* v, auto put) {
        int q = warp;
        for (; q + NW < nr; q += 2 * NW) {
            float t[2];
            dot_rows<2>({A + (long)(r0 + q) * g.ld, A + (long)(r0 + q + NW) * g.ld}, v, nq, lane, t);
            put(q, t[0]);
            put(q + NW, t[1]);
        }
        if (q < nr) {
            float t[1];
            dot_rows<1>({A + (long)(r0 + q) * g.ld}, v, nq, lane, t);
            put(q, t[0]);
        }
    };
    Cluster<CL>::sync();   // every block's shared memory is initialised before a remote write
    for (int e = tid; e < nr; e += NT) w[e] = g.b[r0 + e];
    __syncthreads();
    norm_cluster<CL>(w, nr, s);
    const double b2 = s.sq;
    if (tid == 0) y[0] = krylov_tolerance(g.tol, s.nrm, g.small);
    __syncthreads();
    const double tol = y[0];
    double beta = s.nrm, resid = beta;
    int it = 0, cyc = 0, j = 0;
    bool conv = !(beta > tol), capped = false;
    while (!conv && it < maxit) {
        // a cycle from the residual in w, of norm beta
        if (tid == 0) gv[0] = beta;
        share(0);
        Cluster<CL>::sync();
        bool stop = false;
        for (j = 0; !stop;) {
            product(g.M, vf, [&](int q, float t) {
                if (lane < CL) *Cluster<CL>::at(zf + r0 + q, lane) = t;
                if (lane == 0) Z[(size_t)j * R + q] = t;
            });
            Cluster<CL>::sync();
            product(g.S, zf, [&](int q, float t) {
                if (lane == 0) w[q] = (double)t;
            });
            __syncthreads();
            orthogonalise<CL, NT>(V, R, j, nr, w, s);
            // the next basis vector goes out while one thread rotates the Hessenberg column
            const bool more = j + 1 < m && it + 1 < maxit;
            const double nrm = s.nrm;
            if (tid == NT - 32) {
                double gj, gj1;
                rotate_column<CL>(s, j, nrm, gv[j], &gj, &gj1);
                gv[j] = gj;
                gv[j + 1] = gj1;
                s.resid = fabs(gj1);
            }
            if (more) share(j + 1);
            Cluster<CL>::sync();
            if (tid <= j) H[(long)j * (m + 1) + tid] = s.hc[tid];
            resid = s.resid;
            ++j;
            ++it;
            conv = !(resid > tol);   // also stops on NaN
            stop = conv || !more || nrm == 0.0;
        }
        __syncthreads();
        // y = H^-1 gv, x += sum y_i z_i (as update_body)
        if (tid < j) {
            y[tid] = gv[tid];
            const double d = H[(long)tid * (m + 1) + tid];
            s.h[tid] = d != 0.0 ? 1.0 / d : 0.0;
        }
        __syncthreads();
        if (warp == 0) {
            for (int i = j - 1; i >= 0; --i) {
                const double yi = y[i] * s.h[i];
                __syncwarp();
                for (int l = lane; l < i; l += 32) y[l] -= H[(long)i * (m + 1) + l] * yi;
                if (lane == 0) y[i] = yi;
                __syncwarp();
            }
        }
        __syncthreads();
        for (int e = tid; e < nr; e += NT) {
            double a = 0.0;
            for (int i = 0; i < j; ++i) a += y[i] * (double)Z[(size_t)i * R + e];
            g.x[r0 + e] += a;
        }
        ++cyc;
        if (conv || it >= maxit) break;
        if (cyc >= g.cap) {
            capped = true;
            break;
        }
        // restart: w = b - S x
        __syncthreads();
        for (int c = warp; c < CL; c += NW) {
            float* to = Cluster<CL>::at(zf + r0, c);
            for (int e = lane; e < nr; e += 32) to[e] = (float)g.x[r0 + e];
        }
        Cluster<CL>::sync();
        product(g.S, zf, [&](int q, float t) {
            if (lane == 0) w[q] = g.b[r0 + q] - (double)t;
        });
        __syncthreads();
        norm_cluster<CL>(w, nr, s);
        beta = s.nrm;
        resid = beta;
        conv = !(beta > tol);
    }
    if (rank == 0 && tid == 0) {
        g.small[SM_NORM] = b2;
        g.K[g.L.scal() + SC_RESID] = resid;
        g.K[g.L.scal() + SC_TOL] = tol;
        g.di[DI_J] = j;
        g.di[DI_STOP] = 1;
        g.di[DI_IT] = it;
        g.di[DI_MAXIT] = maxit;
        g.di[DI_CONV] = conv ? 1 : 0;
        g.di[DI_TMPJ] = 0;
        g.di[DI_LOOP] = 0;
        g.di[DI_LOOPERR] = 0;
        if (g.from_its && capped) g.di[DI_CYCERR] = 1;
    }
    Cluster<CL>::sync();   // no block leaves while another may still write to its shared memory
}

template <int CL>
__global__ void __launch_bounds__(kKrylovThreads)
k_start(int ns, const double* __restrict__ r, double* __restrict__ v0, KLayout L, double* __restrict__ K,
        int* __restrict__ di, int init_maxit, KTol tol, double* __restrict__ small) {
    pdl_wait();
    start_cluster_body<CL>(ns, r, v0, L, K, di, init_maxit, tol, small);
}
template <int CL>
__global__ void __launch_bounds__(kKrylovThreads)
k_arnoldi(int* __restrict__ di, double* __restrict__ V, int ns, KLayout L, double* __restrict__ K) {
    pdl_wait();
    arnoldi_cluster_body<CL>(di, V, ns, L, K);
}
template <int CL>
__global__ void __launch_bounds__(kKrylovThreads) k_krylov(KrylovArgs g) {
    pdl_wait();
    krylov_body<CL>(g);
}

// End of a cycle of the separate kernels: y = H^-1 gv over the first k = di[DI_J] columns (every block for
// itself, from shared memory), then x += sum y_i B_i on the block's rows; B: column i at i ns (the basis
// V, or the z_i).
constexpr int kUpdateRows = 256;
__device__ __forceinline__ void update_body(const int* __restrict__ di, KLayout L, const double* __restrict__ K,
                                            const double* __restrict__ B, int ns, double* __restrict__ x) {
    __shared__ double y[64], inv[64];
    extern __shared__ double s_h[];   // k x k, column l at l k
    const int k = di[DI_J], tid = threadIdx.x;
    for (int e = tid; e < k * k; e += kUpdateRows) s_h[e] = K[L.H() + (long)(e / k) * (L.m + 1) + e % k];
    if (tid < k) {
        y[tid] = K[L.gv() + tid];
        const double d = K[L.H() + (long)tid * (L.m + 1) + tid];
        inv[tid] = d != 0.0 ? 1.0 / d : 0.0;
    }
    __syncthreads();
    if (tid < 32) {
        for (int i = k - 1; i >= 0; --i) {
            const double yi = y[i] * inv[i];
            __syncwarp();
            for (int l = tid; l < i; l += 32) y[l] -= s_h[i * k + l] * yi;
            if (tid == 0) y[i] = yi;
            __syncwarp();
        }
    }
    __syncthreads();
    const int e = blockIdx.x * kUpdateRows + tid;
    if (e >= ns) return;
    double a = 0.0;
#pragma unroll 4
    for (int i = 0; i < k; ++i) a += y[i] * B[(long)i * ns + e];
    x[e] += a;
}
inline size_t update_smem(int m) { return sizeof(double) * (size_t)m * m; }
// k<<<(cl, 1, nz), kKrylovThreads, smem, s>>> as clusters of cl blocks along x, with launch accounting.
template <typename... KArgs, typename... Args>
inline iim_status launch_cluster(const char* name, double bytes, void (*k)(KArgs...), int cl, int nz, size_t smem,
                                 cudaStream_t s, Args... args) {
    IIM_CHECK(allow_cluster((const void*)k, smem));
    KTrace t(name, s, bytes, 0.0);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl, 1, nz);
    cfg.blockDim = dim3(kKrylovThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chain_launch(s) ? 2 : 1;
    IIM_TRY(cudaLaunchKernelEx(&cfg, k, args...));
    return IIM_OK;
}

}  // namespace iim
