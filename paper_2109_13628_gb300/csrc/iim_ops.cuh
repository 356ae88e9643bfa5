// Device bodies of the IIM solve's kernels.  solve.cu wraps each in a kernel that works on
// one problem per launch; lockstep.cu wraps the same bodies in kernels that work on many
// problems of one size per launch (blockIdx.z selects the problem), so that both paths do
// identical arithmetic per problem.
#pragma once

#include <cmath>
#include <mutex>
#include <utility>
#include <vector>

#include "common.cuh"
#include "dst.cuh"
#include "tri.cuh"

namespace iim {

// ------------------------------------------------------------------------- transform plan
template <typename T>
struct Plan {
    int NX, NY, nx, ny, lognx, logny;
    const T* lam_x;
    const T* lam_y;
    const cpx<T>* tw;
    T norm;
    int cols_c = 4;   // columns per block of the column pass (tile width)
    int wide = 0;     // 64 threads per 1024-point line instead of one warp
    ScanTab<T> scan{};   // factors of the tridiagonal column pass (lim == nullptr: column transforms)
};

// Algorithmic flops of one DST-I of n - 1 points through an n/2-point complex FFT
// (2.5 n log2(2n): the half-length FFT plus the packing and split steps).
inline double dst_flops(int n) { return 2.5 * n * std::log2(2.0 * n); }

template <typename T>
constexpr int cols_per_block() { return 4; }
constexpr int kRowWarps = 4;

template <typename T>
inline size_t rows_smem(int n, bool wide = false) {
    const int fp = fft_path(n, wide);
    return twiddle_smem<T>(n, fp) + (size_t)kRowWarps * (2 * line_len(n, fp) + kLineScratch) * sizeof(T);
}
template <typename T>
inline size_t cols_smem(int n, int C = cols_per_block<T>(), bool wide = false) {
    const int pad = sizeof(T) == 4 ? 4 : 2;
    const int fp = fft_path(n, wide);
    return twiddle_smem<T>(n, fp) + (size_t)n * sizeof(T) +
           (size_t)C * (2 * line_len(n, fp) + pad + kLineScratch) * sizeof(T);
}

// Tile widths the column pass supports: FP32 4 or 8 columns, FP64 2 or 4 (16-byte row segments).
template <typename T>
inline int tile_width(int requested) {
    if (sizeof(T) == 4) return requested >= 8 ? 8 : 4;
    return requested <= 2 ? 2 : 4;
}

// Streaming multiprocessors of the current device (queried once per device).
inline int sm_count() {
    static std::mutex m;
    static int cached[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(m);
    if (dev >= 0 && dev < 64 && cached[dev] == 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 1;
        cached[dev] = v;
    }
    return dev >= 0 && dev < 64 ? cached[dev] : 1;
}

// Raises a kernel's dynamic shared memory limit once per (device, kernel, size).  A failed
// attribute call is reported (IIM_ERR_CUDA) and not recorded, so the next call tries again.
inline std::mutex g_attr_mutex;
inline std::vector<std::pair<std::pair<int, const void*>, size_t>> g_attr_done;

template <typename KernelT>
inline iim_status allow_smem(KernelT k, size_t bytes) {
    int dev = 0;
    IIM_TRY(cudaGetDevice(&dev));
    const void* key = (const void*)k;
    std::lock_guard<std::mutex> lock(g_attr_mutex);
    for (auto& e : g_attr_done)
        if (e.first.first == dev && e.first.second == key && e.second >= bytes) return IIM_OK;
    IIM_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    g_attr_done.push_back({{dev, key}, bytes});
    return IIM_OK;
}

// The same for a kernel launched as clusters of up to 16 blocks.
inline iim_status allow_cluster(const void* k, size_t bytes) {
    int dev = 0;
    IIM_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(g_attr_mutex);
    for (auto& e : g_attr_done)
        if (e.first.first == dev && e.first.second == k && e.second >= bytes) return IIM_OK;
    IIM_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    IIM_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    g_attr_done.push_back({{dev, k}, bytes});
    return IIM_OK;
}

// ------------------------------------------------------------------------- reductions
template <int BLOCK>
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[BLOCK / 32];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = (l < BLOCK / 32) ? red[l] : 0.0;
        for (int off = 16; off > 0; off >>= 1) r += __shfl_down_sync(0xffffffffu, r, off);
    }
    return r;   // valid in thread 0
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// small[] layout
enum { SM_RES2 = 0, SM_CIRC_ERR = 1, SM_CIRC = 8, SM_RC = 8 + 64, SM_REG = 8 + 128, SM_NORM = 2048, SM_SEED = 2049,
       SM_CAPC = 2112, SM_CAPP = 2176, SM_FNORM = 2240, SM_REL = 2241 };
// Blocks per region sum (small[] holds their partial sums).
__host__ __device__ constexpr int region_parts(int ncirc) { return ncirc <= 8 ? 64 : 16; }

// Device state (int): [0] j (column of the current cycle), [1] stop, [2] iterations of this
// call, [3] max iterations of this call, [4] converged, [5] scratch column index,
// [32, 96) circulation body ids
enum { DI_J = 0, DI_STOP = 1, DI_IT = 2, DI_MAXIT = 3, DI_CONV = 4, DI_TMPJ = 5, DI_LOOP = 6, DI_LOOPERR = 7,
       // device-driven whole solve: refinements, Krylov iterations (all / first correction),
       // cycles of the current correction, cap hits, non-finite residual, cycles and restarts
       DI_REF = 8, DI_ITS = 9, DI_FIRST = 10, DI_CYC = 11, DI_CYCERR = 12, DI_NONFIN = 13, DI_CYCS = 14,
       DI_RSS = 15, DI_TICKET = 18, DI_CIRC = 32 };

// Krylov small-storage layout inside g->H (m <= 64):
//   H (m+1) x m column-major | cs[m] | sn[m] | gv[m+1] | scal[8]
struct KLayout {
    int m;
    __host__ __device__ long H() const { return 0; }
    __host__ __device__ long cs() const { return (long)(m + 1) * m; }
    __host__ __device__ long sn() const { return cs() + m; }
    __host__ __device__ long gv() const { return sn() + m; }
    __host__ __device__ long scal() const { return gv() + m + 1; }
    __host__ __device__ long total() const { return scal() + 8; }
};
enum { SC_INV = 0, SC_RESID = 1, SC_BETA = 2, SC_TOL = 3 };

template <typename T, int BLOCK>
__device__ __forceinline__ void gather_body(int na, int nga, const int* __restrict__ ptr, const int* __restrict__ idx,
                                            const double* __restrict__ w, const T* __restrict__ psi,
                                            const int* __restrict__ cp_body, const int* __restrict__ body_circ,
                                            const int* __restrict__ aff_body, VecArg vin, int use_xc,
                                            double* __restrict__ outb, const int* __restrict__ jidx, long stride,
                                            const int* __restrict__ stop) {
    if (stop && *stop) return;
    const double* v = vin.base ? vin.get() : nullptr;
    double* out = jidx ? outb + (long)(*jidx + 1) * stride : outb;
    if ((int)blockIdx.x < nga) {
        // one warp per affected point, the lanes over its CSR entries
        const int a = blockIdx.x * (BLOCK / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (a >= na) return;
        const double* xc = (use_xc && v) ? v + na : nullptr;
        double acc = 0.0;
        for (int e = ptr[a] + lane; e < ptr[a + 1]; e += 32) {
            const int q = idx[e];
            if (q >= 0) {
                acc += w[e] * (double)psi[q];
            } else if (xc) {
                const int bc = body_circ[cp_body[-q - 1]];
                if (bc >= 0) acc -= w[e] * xc[bc];
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) out[a] = (v ? v[a] : 0.0) + acc;
    } else {
        if (!v) return;
        const int c = blockIdx.x - nga;
        double acc = 0.0;
        for (int a = threadIdx.x; a < na; a += BLOCK)
            if (body_circ[aff_body[a]] == c) acc += v[a];
        acc = block_sum<BLOCK>(acc);
        if (threadIdx.x == 0) out[na + c] = acc;
    }
}

__device__ __forceinline__ void ghost_body(int nm, const int* __restrict__ minus_node, const int* __restrict__ ptr,
                                           const int* __restrict__ idx, const double* __restrict__ w,
                                           const double* __restrict__ psi_b, const double* __restrict__ psibar,
                                           const int* __restrict__ cp_body, double* __restrict__ psi) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= nm) return;
    double acc = 0.0;
    for (int e = ptr[m]; e < ptr[m + 1]; ++e) {
        const int q = idx[e];
        if (q >= 0) acc += w[e] * psi[q];
        else {
            const int c = -q - 1;
            acc += w[e] * ((psi_b ? psi_b[c] : 0.0) + psibar[cp_body[c]]);
        }
    }
    psi[minus_node[m]] = acc;
}

template <int BLOCK>
__device__ __forceinline__ void residual_body(int NX, int NY, double ih2, const double* __restrict__ psi,
                                              const double* __restrict__ omega, const uint8_t* __restrict__ cls,
                                              const double* __restrict__ ring, double* __restrict__ res,
                                              double* __restrict__ partial) {
    const int nx = NX + 1;               // a power of two: row index by shift, column by mask
    const int sh = __ffs(nx) - 1;
    const int n = nx * NY;               // < 2^31 for the supported sizes
    double acc = 0.0;
    for (int k = blockIdx.x * BLOCK + threadIdx.x; k < n; k += gridDim.x * BLOCK) {
        const int j = k >> sh, i = (k & (nx - 1)) - 1;
        double r = 0.0;
        if (i >= 0 && cls[k] <= CLS_PLUS) {
            const double c = psi[k];
            const double wv = i > 0 ? psi[k - 1] : (ring ? ring[2 * (NX + 2) + j] : 0.0);
            const double ev = i < NX - 1 ? psi[k + 1] : (ring ? ring[2 * (NX + 2) + NY + j] : 0.0);
            const double sv = j > 0 ? psi[k - nx] : (ring ? ring[i + 1] : 0.0);
            const double nv = j < NY - 1 ? psi[k + nx] : (ring ? ring[(NX + 2) + i + 1] : 0.0);
            r = omega[(long)j * NX + i] - (4.0 * c - wv - ev - sv - nv) * ih2;
            acc += r * r;
        }
        res[k] = r;
    }
    acc = block_sum<BLOCK>(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// What follows the residual kernel: per circulation body the sum of the residual over R_k and the measured
// circulation -h sum_{dR}(grad_h psi).n (Eq. discretecircconstraint), then small[SM_RES2] = sum partial
// + sum rc^2 with rc_c = (Gamma_k - circ_k) / h^2, bcirc[c] = sum_{R_k} r - rc_c and max |Gamma_k - circ_k|.
struct FinishArgs {
    int nparts;
    const double* partial;
    int nx;
    const double *psi, *res;
    const iim_region* R;
    int* di;                 // circulation body ids, ticket
    int ncirc;
    const double* gamma;
    double ih2;
    double *small, *bcirc;
};
__host__ __device__ constexpr int finish_blocks(int ncirc) { return ncirc > 0 ? ncirc * (region_parts(ncirc) + 1) : 1; }

// One launch of finish_blocks(ncirc) blocks: region parts and circulations, and the block that ends last
// adds everything up in a fixed order.  True in that block's thread 0.
template <int BLOCK>
__device__ __forceinline__ bool finish_body(const FinishArgs& a, int blk) {
    const int P = region_parts(a.ncirc), nblk = finish_blocks(a.ncirc);
    const int* ids = a.di + DI_CIRC;
    if (a.ncirc > 0) {
        const int c = blk / (P + 1), part = blk - c * (P + 1);
        const iim_region r = a.R[ids[c]];
        double acc = 0.0;
        if (part < P) {
            const int w = r.rx - r.lx + 1;
            for (int j = r.ly + part; j <= r.ry; j += P)
                for (int i = threadIdx.x; i < w; i += BLOCK) acc += a.res[(long)(j - 1) * a.nx + r.lx + i];
            acc = block_sum<BLOCK>(acc);
            if (threadIdx.x == 0) a.small[SM_REG + c * P + part] = acc;
        } else {
            auto at = [&](int i, int j) { return a.psi[(long)(j - 1) * a.nx + i]; };
            for (int j = r.ly + threadIdx.x; j <= r.ry; j += BLOCK)
                acc += (at(r.rx + 1, j) - at(r.rx, j)) - (at(r.lx, j) - at(r.lx - 1, j));
            for (int i = r.lx + threadIdx.x; i <= r.rx; i += BLOCK)
                acc += (at(i, r.ry + 1) - at(i, r.ry)) - (at(i, r.ly) - at(i, r.ly - 1));
            acc = block_sum<BLOCK>(acc);
            if (threadIdx.x == 0) a.small[SM_CIRC + c] = -acc;
        }
        __shared__ int last;
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(a.di + DI_TICKET, 1) == nblk - 1;
            if (last) a.di[DI_TICKET] = 0;
        }
        __syncthreads();
        if (!last) return false;
        __threadfence();
    }
    __shared__ double reg[64];
    const int lane = threadIdx.x & 31;
    for (int c = threadIdx.x >> 5; c < a.ncirc; c += BLOCK / 32) {
        double v = 0.0;
        for (int p = lane; p < P; p += 32) v += __ldcg(a.small + SM_REG + c * P + p);
        v = warp_sum(v);
        if (lane == 0) reg[c] = v;
    }
    double s = 0.0;
    for (int b = threadIdx.x; b < a.nparts; b += BLOCK) s += a.partial[b];
    s = block_sum<BLOCK>(s);   // synchronises: reg is complete
    if (threadIdx.x != 0) return false;
    double cerr = 0.0;
    for (int c = 0; c < a.ncirc; ++c) {
        const double diff = (a.gamma ? a.gamma[ids[c]] : 0.0) - __ldcg(a.small + SM_CIRC + c);
        cerr = fmax(cerr, fabs(diff));
        const double rc = diff * a.ih2;
        a.small[SM_RC + c] = rc;
        s += rc * rc;
        if (a.bcirc) a.bcirc[c] = reg[c] - rc;
    }
    a.small[SM_RES2] = s;
    a.small[SM_CIRC_ERR] = cerr;
    return true;
}

__device__ __forceinline__ void init_psi_body(int NX, int NY, const double* __restrict__ guess,
                                              const uint8_t* __restrict__ cls, double* __restrict__ psi) {
    const int nx = NX + 1;               // a power of two
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nx * NY) return;
    const int j = k >> (__ffs(nx) - 1), i = (k & (nx - 1)) - 1;
    psi[k] = (guess && i >= 0 && cls[k] <= CLS_PLUS) ? guess[(long)j * NX + i] : 0.0;
}

__device__ __forceinline__ void init_psibar_body(int nb, const int* __restrict__ body_circ,
                                                 const double* __restrict__ in, int keep_circ,
                                                 double* __restrict__ out) {
    const int k = threadIdx.x;
    if (k >= nb) return;
    const double v = in ? in[k] : 0.0;
    out[k] = (body_circ[k] >= 0 && !keep_circ) ? 0.0 : v;
}

__device__ __forceinline__ void add_psibar_body(int ncirc, const int* __restrict__ circ_ids,
                                                const double* __restrict__ x, double* __restrict__ psibar) {
    const int c = threadIdx.x;
    if (c < ncirc) psibar[circ_ids[c]] += x[c];
}

__device__ __forceinline__ void cap_update_body(long npad, int ncirc, const double* __restrict__ resp,
                                                const double* __restrict__ coef, double* __restrict__ psi) {
    const long p = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npad) return;
    double acc = 0.0;
    for (int l = 0; l < ncirc; ++l) acc += coef[l] * resp[(long)l * npad + p];
    psi[p] += acc;
}

__device__ __forceinline__ void velocity_body(int NX, int NY, double inv2h, const double* __restrict__ psi,
                                              const uint8_t* __restrict__ cls, const double* __restrict__ ring,
                                              double* __restrict__ psi_out, double* __restrict__ ux,
                                              double* __restrict__ uy) {
    const int n = NX * NY;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int nx = NX + 1;
    const int j = k / NX, i = k - j * NX;
    const int p = j * nx + 1 + i;
    const bool fl = cls[p] <= CLS_PLUS;
    if (psi_out) psi_out[k] = fl ? psi[p] : 0.0;
    if (!ux && !uy) return;
    double vx = 0.0, vy = 0.0;
    if (fl) {
        const double wv = i > 0 ? psi[p - 1] : (ring ? ring[2 * (NX + 2) + j] : 0.0);
        const double ev = i < NX - 1 ? psi[p + 1] : (ring ? ring[2 * (NX + 2) + NY + j] : 0.0);
        const double sv = j > 0 ? psi[p - nx] : (ring ? ring[i + 1] : 0.0);
        const double nv = j < NY - 1 ? psi[p + nx] : (ring ? ring[(NX + 2) + i + 1] : 0.0);
        vx = (nv - sv) * inv2h;
        vy = -(ev - wv) * inv2h;
    }
    if (ux) ux[k] = vx;
    if (uy) uy[k] = vy;
}

// Krylov tolerance of a correction: rel ||b||, and with kappa > 0 at most max(kappa ||r||, last ||f||), r
// and f the un-reduced residual of the correction and of psi = 0.  The Schur residual b - S x is what
// the correction leaves at the affected nodes of the un-reduced residual, whose other rows keep FP32
// noise of about kappa ||r||; ||b|| itself is larger than ||r|| by the 1/h^2 of the extrapolation (by 20
// to 1000 on the grids here), so rel alone stops early: five bodies at 2048^2 then contract by 20 per
// correction instead of several hundred.  last ||f|| = a hundredth of the target, so that the last correction
// adds nothing to what the FP32 noise leaves.  A tenth saves one iteration of some solves (1024^2 with one
// body, precond 3: 596 instead of 616 us) but ends them nearer to the target: over 76 solves and batches at
// rtol 1e-12 the error against the exact solution is on average 0.25 of that of a tolerance of rel alone with
// a hundredth, 0.39 with a tenth; a thousandth changes nothing more.  Stronger corrections also mean fewer of
// them: 11 of the 76 end with a larger error than rel alone gave, one refinement earlier, below the target.
struct KTol {
    double rel, kappa, last;
};

// Capacitance coefficients coef = C^-1 (h^2 rc) and the body constants' step psibar += coef . Pb (one block).
__device__ __forceinline__ void cap_coef_body(int nc, const double* __restrict__ rc, const double* __restrict__ cinv,
                                              const double* __restrict__ pb, double h2, double* __restrict__ coef,
                                              const int* __restrict__ circ_ids, double* __restrict__ psibar) {
    __shared__ double c_sh[64];
    const int t = threadIdx.x;
    if (t < nc) {
        double a = 0.0;
        for (int k = 0; k < nc; ++k) a += cinv[t * nc + k] * (rc[k] * h2);
        c_sh[t] = a;
        coef[t] = a;
    }
    __syncthreads();
    if (t < nc) {
        double d = 0.0;
        for (int l = 0; l < nc; ++l) d += c_sh[l] * pb[l * nc + t];
        psibar[circ_ids[t]] += d;
    }
}

__device__ __forceinline__ void final_rel_body(int* __restrict__ di, double* __restrict__ small) {
    const double r2 = small[SM_RES2], fn = small[SM_FNORM];
    if (!isfinite(r2)) di[DI_NONFIN] = 1;
    small[SM_REL] = fn > 0.0 ? sqrt(r2) / fn : 0.0;
}

// ------------------------------------------------------------------------- graph capture
// Stream capture into an existing graph in pieces, so that conditional nodes can be placed
// between the pieces: `deps` is the frontier the next node depends on.
struct CapSeg {
    cudaStream_t s;
    cudaGraph_t graph;
    std::vector<cudaGraphNode_t> deps;
    cudaError_t begin() {
        return cudaStreamBeginCaptureToGraph(s, graph, deps.empty() ? nullptr : deps.data(), nullptr, deps.size(),
                                             cudaStreamCaptureModeThreadLocal);
    }
    cudaError_t end() {
        cudaStreamCaptureStatus cs;
        const cudaGraphNode_t* d = nullptr;
        size_t nd = 0;
        cudaError_t e = cudaStreamGetCaptureInfo(s, &cs, nullptr, nullptr, &d, nullptr, &nd);
        std::vector<cudaGraphNode_t> tail;
        if (e == cudaSuccess && d) tail.assign(d, d + nd);
        cudaGraph_t out = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(s, &out);
        if (e == cudaSuccess && e2 == cudaSuccess) deps = tail;
        return e != cudaSuccess ? e : e2;
    }
    // a conditional node after the frontier; *body receives its body graph
    cudaError_t cond(cudaGraphConditionalHandle h, cudaGraphConditionalNodeType type, cudaGraph_t* body) {
        cudaGraphNodeParams p = {};
        p.type = cudaGraphNodeTypeConditional;
        p.conditional.handle = h;
        p.conditional.type = type;
        p.conditional.size = 1;
        cudaGraphNode_t node = nullptr;
        cudaError_t e = cudaGraphAddNode(&node, graph, deps.empty() ? nullptr : deps.data(), nullptr, deps.size(), &p);
        if (e == cudaSuccess) {
            deps.assign(1, node);
            *body = p.conditional.phGraph_out[0];
        }
        return e;
    }
};

// Kernel nodes directly in a graph (not inside its conditional bodies).
inline long long kernel_nodes(cudaGraph_t graph) {
    size_t n = 0;
    if (cudaGraphGetNodes(graph, nullptr, &n) != cudaSuccess || n == 0) return 0;
    std::vector<cudaGraphNode_t> nodes(n);
    if (cudaGraphGetNodes(graph, nodes.data(), &n) != cudaSuccess) return 0;
    long long k = 0;
    for (cudaGraphNode_t nd : nodes) {
        cudaGraphNodeType t;
        if (cudaGraphNodeGetType(nd, &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) ++k;
    }
    return k;
}

}  // namespace iim
