// Free-space (unbounded) rectangular solve: the operator nabla_h^-2 with unbounded conditions
// on the edge of the box (Sec. 4.1: psi from the convolution of the source with a Green's
// function whose constant fixes the gauge; Sec. 4.2: the FFT solution operator with unbounded
// boundary conditions).
//
// On the grid, psi(x) = h^2 sum_y G(x - y) f(y) with G the lattice Green's function of the
// five-point Laplacian (-L G = delta on Z^2, L = sum of the four neighbours minus four times the
// centre, gauge G(0, 0) = 0).  It is evaluated by James's method, which needs only the
// Dirichlet-box solver of the library and one boundary sum:
//   1. psi_1 = box solve of f with zero box data.  Extended by zero outside the box, psi_1 has
//      -nabla_h^2 psi_1 = f + q with the screening charge q = -psi_1(neighbour) / h^2 on the
//      box ring (each non-corner ring node has one interior neighbour), and a compact function
//      is the lattice potential of its own charge: psi_1 = G * (f + q).
//   2. So G * f = psi_1 - G * q.  On the ring, psi_1 = 0 and
//      rho(x) = -(G * q)(x) = sum_{y on the ring} G(x - y) psi_1(neighbour of y).
//   3. Inside the box, -G * q is harmonic with boundary values rho: the box solve of a zero
//      source with box data rho.  psi = psi_1 + that solve, and psi = rho on the ring.
// This file holds the lattice Green's function table, the extraction of psi_1 next to the box
// and the ring sum; solve.cu strings them together with the box solves.
//
// Outflow plane (Sec. 5.2): the vorticity mirrored evenly across the vertical plane through
// the right box edge (node column nx).  The mirrored interior sources are a field harmonic
// inside the box whose values on the ring are those of the free-space field at the mirror
// points, so the ring kernel becomes K(x, y) = G(x - y) + G(x* - y), x* = (2 nx - i, j) (table
// columns up to 2 nx); sources on the plane column are their own images and are data: their
// potential h^2 sum_j G(x - (nx, j)) w_j enters the ring equations, and through them the
// correction of each refinement.
//
// The table G(m, n), 0 <= m <= nx, 0 <= n <= ny, depends on the lattice only (not on h), so it
// is built once per (device, nx, ny) and shared by every geometry of that size:
//   max(m, n) < 64: -G(m, n) = (1 / 2 pi) int_0^pi (1 - cos(m t) e^(-n a)) / sinh(a) dt,
//     cosh a = 2 - cos t (the Fourier representation with one integral done in closed form),
//     by 256 uniform panels of 16-point Gauss-Legendre in FP64;
//   otherwise the far-field expansion
//     G = -(1/2 pi)(log r + euler_gamma + (3/2) log 2) + cos(4 phi) / (24 pi r^2)
//         + (18 cos(4 phi) + 25 cos(8 phi)) / (480 pi r^4) + O(r^-6),
//     accurate to about 2e-12 at r = 64 and better beyond (checked against the quadrature).
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "iim_ops.cuh"

namespace iim {

constexpr int kLgfQuadRadius = 64;   // max(|m|, |n|) below which G is integrated
constexpr int kLgfPanels = 256;

struct GaussRule {
    double x[16], w[16];
};

// 16-point Gauss-Legendre rule on [-1, 1]: Newton iteration on the Legendre polynomial P_16 from
// the Chebyshev guesses; weights 2 / ((1 - x^2) P_16'(x)^2).
static GaussRule gauss16() {
    GaussRule g;
    const int n = 16;
    for (int i = 0; i < n; ++i) {
        double x = std::cos(M_PI * (i + 0.75) / (n + 0.5));
        double dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (x * p1 - p0) / (x * x - 1.0);
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) break;
        }
        g.x[i] = x;
        g.w[i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
    return g;
}

__device__ double lgf_quadrature(int m, int n, const GaussRule& R) {
    double acc = 0.0;
    const double hw = 0.5 * M_PI / kLgfPanels;
    for (int p = 0; p < kLgfPanels; ++p) {
        const double mid = (2 * p + 1) * hw;
        double pacc = 0.0;
#pragma unroll 4
        for (int q = 0; q < 16; ++q) {
            const double t = mid + hw * R.x[q];
            const double st = sin(0.5 * t);
            const double eps = 2.0 * st * st;                       // cosh a - 1 = 1 - cos t
            const double a = log1p(eps + sqrt(eps * (2.0 + eps)));   // acosh(1 + eps) without cancellation
            const double sm = sin(0.5 * m * t);
            const double num = 2.0 * sm * sm - cos(m * t) * expm1(-n * a);
            pacc += R.w[q] * num / sinh(a);
        }
        acc += pacc * hw;
    }
    return -acc / (2.0 * M_PI);
}

__device__ double lgf_far(int m, int n) {
    const double r2 = (double)m * m + (double)n * n;
    const double r = sqrt(r2);
    const double c4 = ((double)m * m * m * m - 6.0 * m * m * (double)n * n + (double)n * n * n * n) / (r2 * r2);
    const double c8 = 2.0 * c4 * c4 - 1.0;
    const double euler_gamma = 0.57721566490153286061;
    return -(log(r) + euler_gamma + 1.5 * log(2.0)) / (2.0 * M_PI) + c4 / (24.0 * M_PI * r2) +
           (18.0 * c4 + 25.0 * c8) / (480.0 * M_PI * r2 * r2);
}

// G[n * (M + 1) + m] for 0 <= m <= M, 0 <= n <= N, and the same values transposed behind it,
// GT[m * (N + 1) + n]: the ring sums read along whichever index their lanes run over.
__global__ void k_lgf_table(int M, int N, GaussRule R, double* __restrict__ G) {
    pdl_wait();
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long)(M + 1) * (N + 1)) return;
    const int m = (int)(k % (M + 1)), n = (int)(k / (M + 1));
    double v = 0.0;
    if (m == 0 && n == 0) v = 0.0;
    else if (m < kLgfQuadRadius && n < kLgfQuadRadius) v = lgf_quadrature(m, n, R);
    else v = lgf_far(m, n);
    G[k] = v;
    G[(long)(M + 1) * (N + 1) + (long)m * (N + 1) + n] = v;
}

static std::mutex g_lgf_mutex;
static std::map<std::tuple<int, int, int>, double*> g_lgf_tables;

// The table G(m, n), 0 <= m <= nx, 0 <= n <= ny (row stride nx + 1) and its transpose, on the current device
// (built on first use, kept until the process exits).  Synchronizes the device on first use.
iim_status lgf_table(int nx, int ny, const double** out) {
    int dev = 0;
    IIM_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(g_lgf_mutex);
    auto key = std::make_tuple(dev, nx, ny);
    auto it = g_lgf_tables.find(key);
    if (it != g_lgf_tables.end()) {
        *out = it->second;
        return IIM_OK;
    }
    double* G = nullptr;
    const long n = (long)(nx + 1) * (ny + 1);
    IIM_TRY(cudaMalloc(&G, sizeof(double) * 2 * n));
    const GaussRule R = gauss16();
    launch("lgf_table", 0.0, 0.0, k_lgf_table, (unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)0, nx, ny, R, G);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(G);
        record_cuda_error(e, "lgf_table", __FILE__, __LINE__);
        return IIM_ERR_CUDA;
    }
    g_lgf_tables[key] = G;
    *out = G;
    return IIM_OK;
}

// psi_1 next to the left and right box edges, from the column-processed buffer (row j holds the
// x-sine coefficients c_k of psi_1's row j, slots 1..NX of the padded row):
//   psi_1(first interior column, j) = sum_k c_k sin(pi k / nx),
//   psi_1(last interior column, j)  = sum_k c_k (-1)^(k+1) sin(pi k / nx).
// One warp per row, the sines (from the table of e^{-i pi k / 4096}) in shared memory; a lane's k keep
// their parity, so both sums come from one product.  512^2 in FP32:
// 39 -> 5 us (a sine evaluated per element in FP64 before).
constexpr int kBndRows = 4;
template <typename T>
__global__ void __launch_bounds__(32 * kBndRows)
k_bnd_cols(int NX, int NY, int nx, const cpx<double>* __restrict__ tw, const T* __restrict__ buf, double* __restrict__ vl,
           double* __restrict__ vr, const int* __restrict__ stop) {
    pdl_wait();
    if (stop && *stop) return;
    extern __shared__ double sine[];
    for (int k = threadIdx.x; k < NX; k += 32 * kBndRows) sine[k] = -tw[(k + 1) * (kTwN / nx)].y;
    __syncthreads();
    const int j = blockIdx.x * kBndRows + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (j >= NY) return;
    const T* row = buf + (size_t)j * nx + 1;
    double a = 0.0;
    for (int k0 = lane; k0 < NX; k0 += 8 * 32) {
        T c[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) c[u] = k0 + 32 * u < NX ? row[k0 + 32 * u] : T(0);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (k0 + 32 * u < NX) a = fma((double)c[u], sine[k0 + 32 * u], a);
    }
    const double b = warp_sum(lane & 1 ? -a : a);   // (-1)^(k+2) for mode k + 1
    a = warp_sum(a);
    if (lane == 0) {
        vl[j] = a;
        vr[j] = b;
    }
}

// Ring layout: bottom j = 0, i = 0..nx; top j = ny; left i = 0, j = 1..ny-1; right i = nx.
__device__ __forceinline__ void ring_node(int t, int nx, int ny, int& i, int& j) {
    if (t <= nx) { i = t; j = 0; }
    else if (t <= 2 * nx + 1) { i = t - (nx + 1); j = ny; }
    else if (t < 2 * (nx + 1) + (ny - 1)) { i = 0; j = t - 2 * (nx + 1) + 1; }
    else { i = nx; j = t - 2 * (nx + 1) - (ny - 1) + 1; }
}

// K(x, y) = G(x - y) (+ G(x* - y) with the outflow plane, sym).  Sources on the bottom and top run over i,
// those on the sides over j: the first read G, the second its transpose, so that lanes read neighbours.
struct RingKernel {
    const double* G;
    int ld, ldt, nx, sym;   // row strides of G and of its transpose
    __device__ __forceinline__ double operator()(int xi, int xj, int yi, int yj, bool side) const {
        const double* GT = G + (size_t)ld * ldt;
        const int di = abs(xi - yi), dj = abs(xj - yj);
        double k = side ? GT[(size_t)di * ldt + dj] : G[(size_t)dj * ld + di];
        if (sym) {
            const int dm = abs(2 * nx - xi - yi);
            k += side ? GT[(size_t)dm * ldt + dj] : G[(size_t)dj * ld + dm];
        }
        return k;
    }
};

// Ring sums are FP64-bound (a multiply-add per pair of ring nodes): a block takes kRingX consecutive ring
// nodes, a thread one source at a time for all of them, and the kRingX partial sums of a warp are added
// with halving exchanges (9 additions for 8 sums instead of 5 each).
constexpr int kRingX = 8, kRingBlock = 256;
__device__ __forceinline__ double ring_sums(double (&a)[kRingX]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int half = kRingX / 2, off = 16; half >= 1; half /= 2, off /= 2) {
        const bool up = lane & off;
#pragma unroll
        for (int u = 0; u < half; ++u) {
            const double send = up ? a[u] : a[u + half], keep = up ? a[u + half] : a[u];
            a[u] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    __shared__ double part[kRingBlock / 32][kRingX];
    if ((lane & 3) == 0) part[threadIdx.x >> 5][lane >> 2] = a[0];   // lane >> 2: the sum's index
    __syncthreads();
    double v = 0.0;
    if (threadIdx.x < kRingX)
        for (int w = 0; w < kRingBlock / 32; ++w) v += part[w][threadIdx.x];
    return v;   // of ring node blockIdx.x * kRingX + threadIdx.x
}

// rho(x) = sum over the non-corner ring nodes y of K(x, y) psi_1(neighbour of y), for every ring node x,
// minus sub(x) where given; ring (where given) moves by the result.  bnd: psi_1 on the first interior row
// (NX values) then on the last (NX values); vl, vr: psi_1 on the first and last interior columns (NY values
// each).  512^2: 17 -> 12 us with one block per ring node before, against 8.3 us of multiply-adds.
__global__ void __launch_bounds__(kRingBlock)
k_ring_conv(int nx, int ny, RingKernel K, const double* __restrict__ bnd, const double* __restrict__ vl,
            const double* __restrict__ vr, const double* __restrict__ sub, double* __restrict__ rho,
            double* __restrict__ ring, const int* __restrict__ stop) {
    pdl_wait();
    if (stop && *stop) return;
    const int t0 = blockIdx.x * kRingX, n = 2 * (nx + ny);   // n is a multiple of kRingX
    int xi[kRingX], xj[kRingX];
#pragma unroll
    for (int u = 0; u < kRingX; ++u) ring_node(t0 + u, nx, ny, xi[u], xj[u]);
    const int NX = nx - 1, NY = ny - 1, nsrc = 2 * NX + 2 * NY;
    double acc[kRingX] = {};
    for (int s = threadIdx.x; s < nsrc; s += kRingBlock) {
        int si, sj;
        double v;
        if (s < NX) { si = s + 1; sj = 0; v = bnd[s]; }
        else if (s < 2 * NX) { si = s - NX + 1; sj = ny; v = bnd[s]; }
        else if (s < 2 * NX + NY) { si = 0; sj = s - 2 * NX + 1; v = vl[sj - 1]; }
        else { si = nx; sj = s - 2 * NX - NY + 1; v = vr[sj - 1]; }
        const bool side = s >= 2 * NX;
#pragma unroll
        for (int u = 0; u < kRingX; ++u) acc[u] = fma(K(xi[u], xj[u], si, sj, side), v, acc[u]);
    }
    const double r = ring_sums(acc);
    const int t = t0 + threadIdx.x;
    if (threadIdx.x < kRingX && t < n) {
        const double v = sub ? r - sub[t] : r;
        rho[t] = v;
        if (ring) ring[t] += v;
    }
}

// Ring equations of the free-space system (the FP64 residual's ring rows).  For the free-space
// potential of sources inside the box, the discrete Green's second identity on the interior
// nodes, with G(x - .) harmonic there for x on the ring, gives
//   psi(x) = sum over the non-corner ring nodes z of G(x - z) psi(n(z)) - G(x - n(z)) psi(z),
// n(z) the interior neighbour of z; a field harmonic inside the box leaves exactly its ring
// values in  rres(x) = psi(x) - that sum,  so a ring error that the interior rows cannot see
// shows here.  With the outflow plane (sym) the kernel is K(x, y) = G(x - y) + G(x* - y) (the
// mirrored part is harmonic inside the box, and so is G(x* - .)), and the potential of the
// plane sources, h^2 sum_j G(x - (nx, j)) plane_j (harmonic inside), is the data of the row and
// is subtracted (plane null: no plane sources).  psi: padded interior field; ring: psi on the
// ring.  Blocks as k_ring_conv, two multiply-adds per pair.  512^2: 32 -> 22 us.
__global__ void __launch_bounds__(kRingBlock)
k_ring_residual(int nx, int ny, double h2, RingKernel K, const double* __restrict__ plane, const double* __restrict__ psi,
                const double* __restrict__ ring, double* __restrict__ rres) {
    pdl_wait();
    const int t0 = blockIdx.x * kRingX, n = 2 * (nx + ny);
    int xi[kRingX], xj[kRingX];
#pragma unroll
    for (int u = 0; u < kRingX; ++u) ring_node(t0 + u, nx, ny, xi[u], xj[u]);
    const int NX = nx - 1, NY = ny - 1, nsrc = 2 * NX + 2 * NY;
    double acc[kRingX] = {};
    for (int s = threadIdx.x; s < nsrc; s += kRingBlock) {
        int zi, zj, ai, aj, zr;   // ring node, its interior neighbour, its ring index
        if (s < NX) { zi = s + 1; zj = 0; ai = zi; aj = 1; zr = zi; }
        else if (s < 2 * NX) { zi = s - NX + 1; zj = ny; ai = zi; aj = ny - 1; zr = nx + 1 + zi; }
        else if (s < 2 * NX + NY) { zi = 0; zj = s - 2 * NX + 1; ai = 1; aj = zj; zr = 2 * (nx + 1) + zj - 1; }
        else { zi = nx; zj = s - 2 * NX - NY + 1; ai = nx - 1; aj = zj; zr = 2 * (nx + 1) + NY + zj - 1; }
        const double pa = psi[(size_t)(aj - 1) * nx + ai], pz = ring[zr];
        const bool side = s >= 2 * NX;
#pragma unroll
        for (int u = 0; u < kRingX; ++u)
            acc[u] = fma(-K(xi[u], xj[u], ai, aj, side), pz, fma(K(xi[u], xj[u], zi, zj, side), pa, acc[u]));
    }
    if (K.sym && plane) {
        const double* GT = K.G + (size_t)K.ld * K.ldt;
        for (int j = 1 + threadIdx.x; j <= NY; j += kRingBlock) {
            const double p = h2 * plane[j - 1];
#pragma unroll
            for (int u = 0; u < kRingX; ++u) acc[u] += GT[(size_t)abs(xi[u] - nx) * K.ldt + abs(xj[u] - j)] * p;
        }
    }
    const double r = ring_sums(acc);
    const int t = t0 + threadIdx.x;
    if (threadIdx.x < kRingX && t < n) rres[t] = ring[t] - r;
}

template <typename T>
iim_status launch_bnd_cols(int NX, int NY, int nx, const T* buf, double* vl, double* vr, const int* stop,
                           cudaStream_t s) {
    launch("free_bnd_cols", (double)NX * NY * sizeof(T), 4.0 * NX * NY, k_bnd_cols<T>, (NY + kBndRows - 1) / kBndRows,
           32 * kBndRows, sizeof(double) * NX, s, NX, NY, nx, twiddles64(), buf, vl, vr, stop);
    IIM_LAUNCHED();
    return IIM_OK;
}
template iim_status launch_bnd_cols<float>(int, int, int, const float*, double*, double*, const int*, cudaStream_t);
template iim_status launch_bnd_cols<double>(int, int, int, const double*, double*, double*, const int*, cudaStream_t);

iim_status launch_ring_conv(int nx, int ny, const double* G, int ld, int sym, const double* bnd, const double* vl,
                            const double* vr, const double* sub, double* rho, double* ring, const int* stop,
                            cudaStream_t s) {
    const double nsrc = 2.0 * (nx - 1) + 2.0 * (ny - 1);
    launch("free_ring_conv", 0.0, (sym ? 4.0 : 2.0) * nsrc * 2.0 * (nx + ny), k_ring_conv, 2 * (nx + ny) / kRingX,
           kRingBlock, 0, s, nx, ny, RingKernel{G, ld, ny + 1, nx, sym}, bnd, vl, vr, sub, rho, ring, stop);
    IIM_LAUNCHED();
    return IIM_OK;
}

iim_status launch_ring_residual(int nx, int ny, double h, const double* G, int ld, int sym, const double* plane,
                                const double* psi, const double* ring, double* rres, cudaStream_t s) {
    launch("free_ring_residual", 0.0, 0.0, k_ring_residual, 2 * (nx + ny) / kRingX, kRingBlock, 0, s, nx, ny, h * h,
           RingKernel{G, ld, ny + 1, nx, sym}, plane, psi, ring, rres);
    IIM_LAUNCHED();
    return IIM_OK;
}

}  // namespace iim
