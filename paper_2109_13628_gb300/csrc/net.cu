// Learned initial guess for the IIM Poisson iteration: a small fully convolutional network
// (3x3 convolutions with dilation, ReLU between layers, BF16 weights, FP32 accumulation),
// trained on solves that the method itself produces, with hand-written forward, backward and
// Adam kernels.  The paper has no learned component; the solver's own residual decides
// whether a guess is used (iim_poisson_solve falls back to zero when the guess raises it).
//
//   y[b,o,i,j] = bias[o] + sum_{c,ky,kx} W[o,c,ky,kx] x[b,c,i + d(ky-1), j + d(kx-1)]  (zero padding)
//   loss = sum(mask (pred - target)^2) / sum(mask)
//   input gradient  = convolution of the (ReLU-gated) output gradient with the flipped kernel
//   weight gradient = sum over pixels of output gradient x shifted input
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <initializer_list>
#include <random>
#include <vector>

#include "common.cuh"
#include "iim_ops.cuh"
#include "tcgen05.cuh"

// Buffers that grow with the sizes of the calls (grow() below).
struct NetBuffers {
    size_t n = 0;             // items they hold
    std::vector<void*> old;   // outgrown
};

struct iim_net_s {
    int device = 0;
    int cin = 0, hidden = 0, nl = 0;
    std::vector<int> dil, ci, co;        // per layer
    std::vector<long long> woff, boff;   // parameter offsets
    long long np = 0;
    float* p = nullptr;                  // FP32 master parameters
    float* gr = nullptr;                 // gradients
    float* m = nullptr;                  // Adam moments
    float* v = nullptr;
    __nv_bfloat16* wb = nullptr;         // BF16 weights used by the kernels
    __nv_bfloat16* wt = nullptr;         // flipped / transposed BF16 weights (input gradient)
    long long t = 0;                     // Adam step
    float* act = nullptr;                // layer outputs, nl x cap floats
    float* g0 = nullptr;                 // gradient ping-pong, 2 x cap floats
    float* red = nullptr;                // reductions
    NetBuffers acts;                     // act and g0; items: floats per layer (cap())
    size_t act_try = 0;                  // largest size inference has asked them for
    size_t cap() const { return acts.n; }
    float* h_red = nullptr;              // pinned
    int tc = 0;                          // tensor cores (k_conv_tc): 0 off, 1 the 32 -> 32 layers, 2 every layer
    __nv_bfloat16* wtc = nullptr;        // one layer's weights in the tensor-core operand layout
    float* wgp = nullptr;                // weight gradient: one buffer of sums per block
    int wg_blocks = 0;
    // inference on the tensor cores: every layer's weights in the operand layout, and two activation
    // buffers of BF16 channel units with a zero border.  Every call writes what it reads of them (a captured
    // call replays between others).
    __nv_bfloat16* wunit = nullptr;
    uint4* unit[2] = {nullptr, nullptr};
    NetBuffers units;                    // both; items: units of one
    int* tc_err = nullptr;               // set by k_conv_tc when its wait for the MMAs timed out
};

namespace iim {

constexpr int TX = 16, TY = 16;

// out = conv(x) (+bias) (+ReLU); input values gated by `gate > 0` when gate is given.
template <int CO_T>
__global__ void __launch_bounds__(TX * TY)
k_conv(const float* __restrict__ x, const float* __restrict__ gate, const __nv_bfloat16* __restrict__ w,
       const float* __restrict__ bias, float* __restrict__ y, int Ci, int Co, int H, int W, int d, int relu) {
    pdl_wait();
    extern __shared__ float sm[];
    const int tw = TX + 2 * d, th = TY + 2 * d;
    float* tile = sm;
    float* wsm = sm + tw * th;
    const int ncot = (Co + CO_T - 1) / CO_T;
    const int b = blockIdx.z / ncot, co0 = (blockIdx.z % ncot) * CO_T;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const size_t plane = (size_t)H * W;
    float acc[CO_T];
#pragma unroll
    for (int c = 0; c < CO_T; ++c) acc[c] = 0.f;
    for (int ci = 0; ci < Ci; ++ci) {
        const float* xc = x + ((size_t)b * Ci + ci) * plane;
        const float* gc = gate ? gate + ((size_t)b * Ci + ci) * plane : nullptr;
        for (int t = tid; t < tw * th; t += TX * TY) {
            const int ly = t / tw, lx = t - ly * tw;
            const int gy = y0 - d + ly, gx = x0 - d + lx;
            float v = 0.f;
            if (gy >= 0 && gy < H && gx >= 0 && gx < W) {
                v = xc[(size_t)gy * W + gx];
                if (gc && !(gc[(size_t)gy * W + gx] > 0.f)) v = 0.f;
            }
            tile[t] = v;
        }
        for (int t = tid; t < CO_T * 9; t += TX * TY) {
            const int c = co0 + t / 9;
            wsm[t] = c < Co ? __bfloat162float(w[((size_t)c * Ci + ci) * 9 + t % 9]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const float v = tile[(ty + d * (k / 3)) * tw + tx + d * (k % 3)];
#pragma unroll
            for (int c = 0; c < CO_T; ++c) acc[c] = fmaf(wsm[c * 9 + k], v, acc[c]);
        }
        __syncthreads();
    }
    const int gy = y0 + ty, gx = x0 + tx;
    if (gy < H && gx < W) {
#pragma unroll
        for (int c = 0; c < CO_T; ++c) {
            if (co0 + c >= Co) break;
            float v = acc[c] + (bias ? bias[co0 + c] : 0.f);
            if (relu) v = fmaxf(v, 0.f);
            y[((size_t)b * Co + co0 + c) * plane + (size_t)gy * W + gx] = v;
        }
    }
}

// Convolution of Ci <= 32 input to Co <= 32 output channels as an implicit GEMM on the tensor
// cores (tcgen05, BF16 operands, FP32 accumulation in tensor memory).  One CTA computes a run of
// TC_M = 128 pixels of one image row for NO output columns (16 or 32, the MMA's N; outputs
// o >= Co are zero columns): D (128 x NO) = sum over the 9 taps and the CG / 2 16-channel parts of
// the CG staged 8-channel groups (CG = 2 or 4; channels c >= Ci are zero) of
// A_tap (128 pixels x 16 channels) * B_tap^T (NO outputs x 16 channels), MMAs of M = 128, K = 16.
//
// Shared memory, in 16-byte units of 8 BF16 channels:
//   A: input rows row - d, row, row + d (r = 0, 1, 2), channel group g, pixel p = 0 .. NP - 1
//      standing for column x0 - d + p (NP = 128 + 2 d), unit (r * CG + g) * NP + p; zero outside
//      the image.  The operand of tap (ky, kx) starts at pixel kx * d of row ky: consecutive
//      pixels are 16 bytes apart (stride byte offset 128 per 8 rows), the second channel group of
//      an MMA is NP units further (leading byte offset).
//   B: tap t, channel group g, output o: unit (t * CG + g) * NO + o (packed by k_pack_w_tc).
// The input is rounded to BF16 on the way in (optionally gated by gate > 0, as k_conv); the
// epilogue adds the bias, applies the ReLU and writes FP32 in the NCHW layout of k_conv.
// A wait for the MMAs that runs past one second sets *err and skips the epilogue.
constexpr int TC_M = 128, TC_C = 32;

__host__ __device__ constexpr size_t conv_tc_smem(int d, int cg, int no) {
    return (size_t)16 * (3 * cg * (TC_M + 2 * d) + 9 * cg * no) + 16;
}

// wp[((t * CG + g) * NO + o) * 8 + e] = w[(o * Ci + 8 g + e) * 9 + t], zero for o >= Co or
// 8 g + e >= Ci
template <int CG, int NO>
__global__ void k_pack_w_tc(const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wp, int Ci, int Co) {
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 9 * CG * NO * 8) return;
    const int e = i & 7, o = (i >> 3) % NO, g = ((i >> 3) / NO) % CG, t = (i >> 3) / (NO * CG);
    const int c = 8 * g + e;
    wp[i] = (o < Co && c < Ci) ? w[(o * Ci + c) * 9 + t] : __float2bfloat16(0.f);
}

__device__ __forceinline__ uint32_t bf16x2_bits(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);   // a at the lower address
    return *reinterpret_cast<const uint32_t*>(&v);
}

template <int CG, int NO>
__global__ void __launch_bounds__(128)
k_conv_tc(const float* __restrict__ x, const float* __restrict__ gate, const __nv_bfloat16* __restrict__ wp,
          const float* __restrict__ bias, float* __restrict__ y, int Ci, int Co, int H, int W, int d, int relu,
          int* __restrict__ err) {
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int NP = TC_M + 2 * d;
    uint4* sA = reinterpret_cast<uint4*>(smem_raw);
    uint4* sB = sA + 3 * CG * NP;
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sB + 9 * CG * NO);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int x0 = blockIdx.x * TC_M, row = blockIdx.y, b = blockIdx.z;
    const size_t plane = (size_t)H * W;
    const float* xb = x + (size_t)b * Ci * plane;
    const float* gb = gate ? gate + (size_t)b * Ci * plane : nullptr;

    if (warp == 0) tc::tmem_alloc(tslot, 32);
    if (tid == 0) tc::mbar_init(mbar, 1);
    const uint4* wsrc = reinterpret_cast<const uint4*>(wp);
    for (int i = tid; i < 9 * CG * NO; i += 128) sB[i] = wsrc[i];
    // UB units per thread and round, all their loads issued before any conversion
    constexpr int UB = 2;
    const int units = 3 * CG * NP;
    for (int u0 = tid; u0 < units; u0 += UB * 128) {
        float v[UB][8];
        bool in[UB];
        size_t off[UB];
        int c0[UB];
#pragma unroll
        for (int q = 0; q < UB; ++q) {
            const int u = u0 + q * 128;
            const int rg = u / NP, p = u - rg * NP;
            const int r = rg / CG, g = rg - r * CG;
            const int gy = row + (r - 1) * d, gx = x0 - d + p;
            in[q] = u < units && gy >= 0 && gy < H && gx >= 0 && gx < W;
            c0[q] = 8 * g;
            off[q] = in[q] ? (size_t)(8 * g) * plane + (size_t)gy * W + gx : 0;
#pragma unroll
            for (int e = 0; e < 8; ++e) v[q][e] = (in[q] && c0[q] + e < Ci) ? xb[off[q] + (size_t)e * plane] : 0.f;
        }
        if (gb) {
#pragma unroll
            for (int q = 0; q < UB; ++q)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (in[q] && c0[q] + e < Ci && !(gb[off[q] + (size_t)e * plane] > 0.f)) v[q][e] = 0.f;
        }
#pragma unroll
        for (int q = 0; q < UB; ++q) {
            const int u = u0 + q * 128;
            if (u < units)
                sA[u] = make_uint4(bf16x2_bits(v[q][0], v[q][1]), bf16x2_bits(v[q][2], v[q][3]),
                                   bf16x2_bits(v[q][4], v[q][5]), bf16x2_bits(v[q][6], v[q][7]));
        }
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tslot;
    if (tid == 0) {
        const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
        constexpr uint32_t idesc = tc::idesc_bf16_f32(TC_M, NO);
#pragma unroll 1
        for (int t = 0; t < 9; ++t) {
            const int ky = t / 3, kx = t - 3 * ky;
#pragma unroll
            for (int s = 0; s < CG / 2; ++s) {
                const uint64_t ad =
                    tc::desc_kmajor(a0 + (uint32_t)(16 * ((ky * CG + 2 * s) * NP + kx * d)), (uint32_t)(16 * NP), 128u);
                const uint64_t bd = tc::desc_kmajor(b0 + (uint32_t)(16 * (t * CG + 2 * s) * NO), 16u * NO, 128u);
                tc::mma_bf16(tmem, ad, bd, idesc, (t | s) != 0);
            }
        }
        tc::commit(mbar);
    }
    __syncwarp();
    const bool ok = __all_sync(0xffffffffu, tc::mbar_wait_bounded(mbar, 0, 1000000000ull));
    tc::fence_after_sync();
    if (ok) {
        float acc[NO];
        if constexpr (NO == 32) tc::tmem_ld_32x32(tmem + ((uint32_t)(32 * warp) << 16), acc);
        else tc::tmem_ld_32x16(tmem + ((uint32_t)(32 * warp) << 16), acc);
        const int gx = x0 + 32 * warp + lane;
        if (gx < W) {
            float* yo = y + (size_t)b * Co * plane + (size_t)row * W + gx;
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                if (o >= Co) break;
                float v = acc[o] + (bias ? bias[o] : 0.f);
                if (relu) v = fmaxf(v, 0.f);
                yo[(size_t)o * plane] = v;
            }
        }
    } else if (lane == 0) {
        atomicExch(err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        if (!ok) (void)tc::mbar_wait_bounded(mbar, 0, 1000000000ull);
        tc::tmem_dealloc(tmem, 32);
    }
}

// ---- inference: the same convolutions (same operands, MMAs in the same order, the same bits) on
// activations that stay in the operand layout between layers.
//
// A layer's output is rounded to BF16 by its writer instead of by its readers and kept as units of 8
// channels of one pixel (16 bytes), one plane of units per 8-channel group, with a border of zeros wide
// enough for every dilation: 64 bytes per pixel instead of 128 + 128, and the operand of a run of pixels is a
// contiguous piece of memory, so one bulk copy per row and group brings it into shared memory with no
// thread touching it and no test at the image's edges.  A block computes runs of UN_M = 128 pixels on
// UN_R = 4 output rows d apart, which share their input rows (6 instead of 12), each row in accumulator
// columns of its own, side by side: an input row's operand (one shift kx, 16 channels) meets the weights
// of all three ky at once, one MMA of N = 96 onto the columns of the three output rows it belongs to,
// because an MMA of N = 32 is bound by reading its 128-row operand.  Every accumulator still gets its
// products in the order of the taps.  Blocks are persistent, keep the weights, and start the next tile's
// copies as soon as the MMAs have read this one's.  Two or three blocks per SM overlap copies, MMAs and
// epilogues.  1023^2, six layers: 0.84 ms (one row of
// FP32 planes converted by its block's threads per tile) -> 0.21 ms; the forward pass 0.86 -> 0.22 ms.
constexpr int UN_M = 128, UN_R = 4;

struct UnitLayout {
    int H, W, Hp, Wp, D;   // image, padded planes (units), border
    __host__ __device__ size_t at(int plane, int y, int x) const { return ((size_t)plane * Hp + y + D) * Wp + x + D; }
};
__host__ __device__ constexpr size_t conv_units_smem(int d, int cg, int no) {
    return (size_t)16 * ((UN_R + 2) * cg * (UN_M + 2 * d) + 9 * cg * no) + 32 * 4 + 32;
}
__host__ __device__ constexpr int mma_groups(int c) { return c <= 16 ? 2 : 4; }     // 8-channel groups of the MMA's K
__host__ __device__ constexpr int mma_cols(int c) { return c <= 16 ? 16 : 32; }     // its N

// Units of one layer's packed weights (the largest layer's).
constexpr int WUNIT = 9 * 4 * TC_C;
struct UnitLayers {
    int n, ci[16], co[16];
    long woff[16];
};
// k / w and k % w of a k < n, in 32 bits where n allows it.
__device__ __forceinline__ void split(long k, long n, int w, int& y, int& x) {
    if (n <= 0x7fffffffL) {
        y = (int)((unsigned)k / (unsigned)w);
        x = (int)((unsigned)k - (unsigned)y * (unsigned)w);
    } else {
        y = (int)(k / w);
        x = (int)(k - (long)y * w);
    }
}
// *p = v, without a store where it is so already: the weights, which every block of every layer reads, then
// stay where the last call left them in the L2 cache.  127^2: 44.3 us for the pass, 48.1 with the store.
__device__ __forceinline__ void settle(uint4* p, uint4 v) {
    const uint4 o = *p;
    if (((o.x ^ v.x) | (o.y ^ v.y) | (o.z ^ v.z) | (o.w ^ v.w)) != 0u) *p = v;
}
// What one forward pass needs before its first layer, in blocks of 256 items:
//   * nw blocks: the weights, unit l WUNIT + ((kx CG + g) * 3 + 2 - ky) * NO + o of wp =
//     w_l[o][8 g .. 8 g + 7][ky][kx], zero for o >= Co and channels >= Ci;
//   * nb blocks for each of P planes: the zero border of both buffers as far as a layer reads it, D columns
//     on either side, D rows above and one row below (k_conv_units takes it for every row beyond);
//   * nx blocks for each image and group: the FP32 planes x (B, C, H, W) as units (zero channels beyond C).
// Done by every call (see iim_net_s).  Bound by the bytes of the planes, units and borders.  Against a pass that
// keeps weights and borders of the call before it: 127^2 43.7 -> 44.3 us, 511^2 79.4 -> 80.6, 1023^2
// 221.5 -> 224.6.
__global__ void __launch_bounds__(256)
k_units_begin(const float* __restrict__ x, int C, UnitLayout u, uint4* __restrict__ buf0, uint4* __restrict__ buf1,
              const __nv_bfloat16* __restrict__ w, UnitLayers L, uint4* __restrict__ wp, int nw, int nb, int P, int nx) {
    pdl_wait();
    int blk = blockIdx.x;
    if (blk < nw) {
        const int i = blk * 256 + threadIdx.x, l = i / WUNIT, r = i - l * WUNIT;
        if (l >= L.n) return;
        const int ci = L.ci[l], co = L.co[l], CG = mma_groups(ci), NO = mma_cols(co);   // powers of two
        if (r >= 9 * CG * NO) return;
        const int o = r & (NO - 1), q = r >> (NO == 32 ? 5 : 4), ky = 2 - q % 3, g = q / 3 & (CG - 1);
        const int kx = q / 3 >> (CG == 4 ? 2 : 1);
        const unsigned short* src = reinterpret_cast<const unsigned short*>(w) + L.woff[l] + (o * ci + 8 * g) * 9 + 3 * ky + kx;
        unsigned v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = o < co && 8 * g + e < ci ? src[9 * e] : 0u;
        settle(wp + i, make_uint4(v[0] | v[1] << 16, v[2] | v[3] << 16, v[4] | v[5] << 16, v[6] | v[7] << 16));
        return;
    }
    blk -= nw;
    if (blk < nb * P) {
        const int D = u.D, wide = u.W + 2 * D;
        const long rows = (D + 1) * (long)wide, n = rows + 2L * D * u.H, t = (long)(blk % nb) * 256 + threadIdx.x;
        if (t >= n) return;
        int yy, xx;
        if (t < rows) {
            split(t, n, wide, yy, xx);
            yy = yy < D ? yy - D : u.H;
            xx -= D;
        } else {
            split(t - rows, n, 2 * D, yy, xx);
            xx = xx < D ? xx - D : u.W + xx - D;
        }
        const size_t q = u.at(blk / nb, yy, xx);
        buf0[q] = make_uint4(0u, 0u, 0u, 0u);
        buf1[q] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    blk -= nb * P;
    const int G = (C + 7) / 8, g = blk / nx % G, b = blk / nx / G;
    const long k = (long)(blk % nx) * 256 + threadIdx.x, plane = (long)u.H * u.W;
    if (k >= plane) return;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = 8 * g + e < C ? x[((long)b * C + 8 * g + e) * plane + k] : 0.f;
    int yy, xx;
    split(k, plane, u.W, yy, xx);
    buf0[u.at(b * G + g, yy, xx)] =
        make_uint4(bf16x2_bits(v[0], v[1]), bf16x2_bits(v[2], v[3]), bf16x2_bits(v[4], v[5]), bf16x2_bits(v[6], v[7]));
}

// One layer: units in (gin groups) -> units out (gout groups, ReLU), or with y the FP32 plane of output 0
// (no ReLU).  Tiles are (image, row block, run), runs fastest; row block r covers rows (r / d) UN_R d + r % d
// + k d, k < UN_R.
template <int CG, int NO>
__global__ void __launch_bounds__(128)
k_conv_units(const uint4* __restrict__ in, int gin, const __nv_bfloat16* __restrict__ wp,
             const float* __restrict__ bias, int Co, uint4* __restrict__ out, int gout, float* __restrict__ y,
             UnitLayout u, int d, int nx, int nr, int tiles, int* __restrict__ err) {
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int NP = UN_M + 2 * d;
    uint4* sA = reinterpret_cast<uint4*>(smem_raw);
    uint4* sB = sA + (UN_R + 2) * CG * NP;
    float* sbias = reinterpret_cast<float*>(sB + 9 * CG * NO);
    uint64_t* full = reinterpret_cast<uint64_t*>(sbias + 32);
    uint64_t* done = full + 1;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t COLS = UN_R * NO;
    if (warp == 0) tc::tmem_alloc(tslot, COLS);
    if (tid == 0) {
        tc::mbar_init(full, 1);
        tc::mbar_init(done, 1);
    }
    const uint4* wsrc = reinterpret_cast<const uint4*>(wp);
    for (int i = tid; i < 9 * CG * NO; i += 128) sB[i] = wsrc[i];
    if (tid < 32) sbias[tid] = tid < Co ? bias[tid] : 0.f;
    for (int i = tid; i < (UN_R + 2) * (CG - gin) * NP; i += 128) {   // groups without channels stay zero
        const int p = i % NP, q = i / NP, r = q / (CG - gin), g = gin + q - r * (CG - gin);
        sA[(r * CG + g) * NP + p] = make_uint4(0u, 0u, 0u, 0u);
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tslot;
    float2 bia[NO / 2];
#pragma unroll
    for (int o = 0; o < NO / 2; ++o) bia[o] = make_float2(sbias[2 * o], sbias[2 * o + 1]);
    auto row0 = [&](int t) { const int r = (t / nx) % nr; return (r / d) * UN_R * d + r % d; };
    auto load = [&](int t) {   // warp 0: one copy per lane (at most 6 rows x 4 groups)
        const int x0 = (t % nx) * UN_M, y0 = row0(t), b = t / (nx * nr);
        if (lane == 0) tc::mbar_expect(full, (uint32_t)(16 * (UN_R + 2) * gin * NP));
        __syncwarp();
        if (lane < (UN_R + 2) * gin) {
            const int i = lane / gin, g = lane - i * gin;
            const int yy = min(y0 + (i - 1) * d, u.H);   // rows below the image: its first border row
            tc::bulk_load(sA + (i * CG + g) * NP, in + u.at(b * gin + g, yy, x0 - d), (uint32_t)(16 * NP), full);
        }
    };
    // row blocks past the image's last row (when UN_R d does not divide the height) have no output
    auto next = [&](int t) {
        while (t < tiles && row0(t) >= u.H) t += gridDim.x;
        return t;
    };
    bool ok = true;
    uint32_t phase = 0;
    int t = next(blockIdx.x);
    if (t < tiles && warp == 0) load(t);
    while (t < tiles) {
        const int x0 = (t % nx) * UN_M, y0 = row0(t), b = t / (nx * nr);
        if (tid == 0) {
            if (tc::mbar_wait_bounded(full, phase, 1000000000ull)) {
                // operand addresses move by 16-byte units, the unit of the descriptors' address field
                const uint64_t ad = tc::desc_kmajor(tc::smem_u32(sA), (uint32_t)(16 * NP), 128u);
                const uint64_t bd = tc::desc_kmajor(tc::smem_u32(sB), 48u * NO, 128u);
                const int nk = min(UN_R, (u.H - y0 + d - 1) / d);   // output rows of the tile
#pragma unroll
                for (int i = 0; i < UN_R + 2; ++i) {
                    // input row i: output rows lo .. hi (ky = i - row); row i starts here
                    const int lo = i > 2 ? i - 2 : 0, hi = min(i, nk - 1);
                    if (hi < lo) break;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
#pragma unroll
                        for (int s = 0; s < CG / 2; ++s) {
                            const uint64_t a = ad + (uint32_t)((i * CG + 2 * s) * NP + kx * d);
                            const uint64_t w = bd + (uint32_t)(((kx * CG + 2 * s) * 3 + lo - i + 2) * NO);
                            const bool first = (kx | s) == 0 && hi == i;   // the first products of row i overwrite
                            const int n = hi - lo + 1 - (first ? 1 : 0);
                            if (n > 0) tc::mma_bf16(tmem + (uint32_t)(lo * NO), a, w, tc::idesc_bf16_f32(UN_M, n * NO), 1);
                            if (first) tc::mma_bf16(tmem + (uint32_t)(i * NO), a, w + (uint32_t)(n * NO), tc::idesc_bf16_f32(UN_M, NO), 0);
                        }
                    }
                }
                tc::commit(done);
            }
        }
        __syncwarp();
        ok = __all_sync(0xffffffffu, tc::mbar_wait_bounded(done, phase, 2000000000ull));
        // a copy or an MMA that gave no sign of completing: leave (every warp waits on the same barrier)
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        tc::fence_after_sync();
        const int tn = next(t + gridDim.x);
        if (tn < tiles && warp == 0) load(tn);   // the MMAs have read this tile's operands
        const int gx = x0 + tid;
#pragma unroll 1
        for (int k = 0; k < UN_R; ++k) {
            const int gy = y0 + k * d;
            if (gy >= u.H) break;
            float acc[NO];
            __syncwarp();   // the load below is a whole-warp instruction
            const uint32_t ta = tmem + (uint32_t)(k * NO) + ((uint32_t)(32 * warp) << 16);
            if constexpr (NO == 32) tc::tmem_ld_32x32(ta, acc);
            else tc::tmem_ld_32x16(ta, acc);
            if (gx >= u.W) continue;
            if (y) {
                y[(size_t)b * u.H * u.W + (size_t)gy * u.W + gx] = acc[0] + bia[0].x;
                continue;
            }
            // bias, rounding to BF16, ReLU (channels beyond Co: zero weights and bias)
            uint32_t v[NO / 2];
#pragma unroll
            for (int o = 0; o < NO / 2; ++o) {
                const __nv_bfloat162 r = __floats2bfloat162_rn(acc[2 * o] + bia[o].x, acc[2 * o + 1] + bia[o].y);
                const __nv_bfloat162 q = __hmax2(r, __floats2bfloat162_rn(0.f, 0.f));
                v[o] = *reinterpret_cast<const uint32_t*>(&q);
            }
#pragma unroll
            for (int g = 0; g < NO / 8; ++g)
                if (g < gout) out[u.at(b * gout + g, gy, gx)] = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
        }
        tc::fence_before_sync();
        __syncthreads();   // the accumulators have been read
        tc::fence_after_sync();
        t = tn;
        phase ^= 1;
    }
    if (!ok) {
        if (tid == 0) {
            atomicExch(err, 1);
            (void)tc::mbar_wait_bounded(full, phase, 1000000000ull);   // no copy may land after the block has left
        }
        __syncthreads();
    }
    if (warp == 0) tc::tmem_dealloc(tmem, COLS);
}

// Weight gradient dW[o,c,k] = sum_{b,p} g[b,o,p] x[b,c,p + d off(k)], db[o] = sum g (g gated by
// gate > 0), FP32 throughout, as nine 32 x 32 products with the pixels as the reduction.
//
// One warp per tap; a lane holds an 8 x 4 (output x input channel) tile in registers, so a pixel
// costs 32 FMAs for three 16-byte shared-memory loads: bound by the FP32 pipe.  A block takes strips
// of WG_PX pixels of one image row: the strip's g and the three x rows it meets, staged
// [pixel][channel] (four channels per 16-byte store; a row of 32 channels padded to 36 floats, so
// neither the stores nor the loads conflict).  With fewer channels the lanes without a channel tile
// of their own split the pixels instead (layer 3 -> 32: eight ways, 32 -> 1: four ways).  Blocks walk
// contiguous ranges of strips and leave their sums in a buffer of their own; k_wgrad_sum adds the
// buffers in a fixed order (no atomics: the gradient is reproducible).  The sums run over a strip
// first, then over strips, then over blocks.  8 x 127^2, 32 channels (backward's six launches):
// 17.96 ms for one thread per (output, tap) with two shared loads per FMA; now
// 0.59 ms (8.1 TMAC/s, about a quarter of the FP32 rate, the staging of the strips between the
// products; a training step 18.6 -> 1.13 ms).
constexpr int WG_PX = 64, WG_THREADS = 288, WG_PART = 32 * 32 * 9 + 32;

__host__ __device__ constexpr int wg_groups(int ch, int per) {   // tiles of `per` channels, a power of two
    return ch <= per ? 1 : ch <= 2 * per ? 2 : ch <= 4 * per ? 4 : 8;
}
__host__ __device__ constexpr int wg_stride(int ch) { return ch == 32 ? 36 : ch; }
inline size_t wgrad_smem(int nog, int ncg, int d) {
    return sizeof(float) * ((size_t)WG_PX * wg_stride(8 * nog) + (size_t)3 * (WG_PX + 2 * d) * wg_stride(4 * ncg));
}

__global__ void __launch_bounds__(WG_THREADS, 2)
k_conv_wgrad(const float* __restrict__ x, const float* __restrict__ g, const float* __restrict__ gate,
             float* __restrict__ part, int Ci, int Co, int H, int W, int d, int strips) {
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int nog = wg_groups(Co, 8), ncg = wg_groups(Ci, 4);
    const int GP = wg_stride(8 * nog), XP = wg_stride(4 * ncg);
    float* gs = reinterpret_cast<float*>(smem_raw);
    float* xs = gs + WG_PX * GP;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ky = warp / 3, kx = warp - 3 * ky;
    const int og = lane >> 3, cg = lane & 7;
    const int o0 = 8 * (og & (nog - 1)), c0 = 4 * (cg & (ncg - 1));
    const int S = (4 / nog) * (8 / ncg), sub = og / nog + (4 / nog) * (cg / ncg);
    const size_t plane = (size_t)H * W;
    const int NX = WG_PX + 2 * d, spr = (W + WG_PX - 1) / WG_PX;
    float acc[8][4], bacc[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        bacc[a] = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = 0.f;
    }
    const int s_end = (int)((long)strips * (blockIdx.x + 1) / gridDim.x);
    for (int st = (int)((long)strips * blockIdx.x / gridDim.x); st < s_end; ++st) {
        const int row = st / spr, px0 = (st - row * spr) * WG_PX, b = row / H, y = row - b * H;
        __syncthreads();   // the previous strip has been consumed
        for (int u = tid; u < WG_PX * 2 * nog; u += WG_THREADS) {
            const int p = u % WG_PX, q = u / WG_PX, gx = px0 + p;
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int o = 4 * q + e;
                v[e] = 0.f;
                if (o < Co && gx < W) {
                    const size_t idx = ((size_t)b * Co + o) * plane + (size_t)y * W + gx;
                    v[e] = g[idx];
                    if (gate && !(gate[idx] > 0.f)) v[e] = 0.f;
                }
            }
            *reinterpret_cast<float4*>(gs + p * GP + 4 * q) = make_float4(v[0], v[1], v[2], v[3]);
        }
        for (int u = tid; u < 3 * ncg * NX; u += WG_THREADS) {
            const int rq = u / NX, p = u - rq * NX, r = rq / ncg, q = rq - r * ncg;
            const int gy = y + (r - 1) * d, gx = px0 - d + p;
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = 4 * q + e;
                v[e] = (c < Ci && gy >= 0 && gy < H && gx >= 0 && gx < W)
                           ? x[((size_t)b * Ci + c) * plane + (size_t)gy * W + gx] : 0.f;
            }
            *reinterpret_cast<float4*>(xs + (r * NX + p) * XP + 4 * q) = make_float4(v[0], v[1], v[2], v[3]);
        }
        __syncthreads();
        const float* gp = gs + sub * GP + o0;
        const float* xp = xs + (ky * NX + kx * d + sub) * XP + c0;
        float s[8][4];
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) s[a][c] = 0.f;
        float sb[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
        for (int p = sub; p < WG_PX; p += S) {
            const float4 g0 = *reinterpret_cast<const float4*>(gp), g1 = *reinterpret_cast<const float4*>(gp + 4);
            const float4 xv = *reinterpret_cast<const float4*>(xp);
            gp += S * GP;
            xp += S * XP;
            const float ga[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                s[a][0] = fmaf(ga[a], xv.x, s[a][0]);
                s[a][1] = fmaf(ga[a], xv.y, s[a][1]);
                s[a][2] = fmaf(ga[a], xv.z, s[a][2]);
                s[a][3] = fmaf(ga[a], xv.w, s[a][3]);
            }
            if (warp == 4) {
#pragma unroll
                for (int a = 0; a < 8; ++a) sb[a] += ga[a];
            }
        }
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            bacc[a] += sb[a];
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][c] += s[a][c];
        }
    }
    // lanes that split the pixels of one tile: add across them (their bits of the lane index)
    float* out = part + (size_t)blockIdx.x * WG_PART;
#pragma unroll
    for (int bit = 1; bit < 32; bit <<= 1) {
        if (bit < 8 ? bit >= ncg : (bit >> 3) >= nog) {
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                bacc[a] += __shfl_xor_sync(0xffffffffu, bacc[a], bit);
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[a][c] += __shfl_xor_sync(0xffffffffu, acc[a][c], bit);
            }
        }
    }
    if (sub == 0) {
#pragma unroll
        for (int a = 0; a < 8; ++a) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (o0 + a < Co && c0 + c < Ci) out[((o0 + a) * Ci + c0 + c) * 9 + warp] = acc[a][c];
            if (warp == 4 && c0 == 0 && o0 + a < Co) out[Co * Ci * 9 + o0 + a] = bacc[a];
        }
    }
}

// dst[e] = sum over the blocks' buffers of entry e (n entries): 32 entries x 8 slices of the
// buffers per block.
__global__ void __launch_bounds__(256)
k_wgrad_sum(int nblk, int n, const float* __restrict__ part, float* __restrict__ dst) {
    pdl_wait();
    __shared__ float red[8][33];
    const int e = blockIdx.x * 32 + (threadIdx.x & 31), sl = threadIdx.x >> 5;
    float s = 0.f;
    if (e < n)
        for (int b = sl; b < nblk; b += 8) s += part[(size_t)b * WG_PART + e];
    red[sl][threadIdx.x & 31] = s;
    __syncthreads();
    if (sl == 0 && e < n) {
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
        dst[e] = t;
    }
}

// diff = (pred - target) mask; partial sums of diff^2 and mask
__global__ void k_mse_partial(long n, const float* __restrict__ pred, const float* __restrict__ target,
                              const float* __restrict__ mask, float* __restrict__ diff, float* __restrict__ part) {
    pdl_wait();
    float s2 = 0.f, sm_ = 0.f;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float m = mask ? mask[i] : 1.f;
        const float dd = (pred[i] - target[i]) * m;
        diff[i] = dd;
        s2 += dd * dd;
        sm_ += m;
    }
    for (int off = 16; off > 0; off >>= 1) {
        s2 += __shfl_down_sync(0xffffffffu, s2, off);
        sm_ += __shfl_down_sync(0xffffffffu, sm_, off);
    }
    __shared__ float a[32], c[32];
    if ((threadIdx.x & 31) == 0) { a[threadIdx.x >> 5] = s2; c[threadIdx.x >> 5] = sm_; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float x2 = 0.f, xm = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { x2 += a[w]; xm += c[w]; }
        part[2 * blockIdx.x] = x2;
        part[2 * blockIdx.x + 1] = xm;
    }
}

__global__ void k_mse_finish(int nb, float* __restrict__ part, float* __restrict__ out) {
    pdl_wait();
    if (threadIdx.x != 0) return;
    float x2 = 0.f, xm = 0.f;
    for (int b = 0; b < nb; ++b) { x2 += part[2 * b]; xm += part[2 * b + 1]; }
    out[0] = xm > 0.f ? x2 / xm : 0.f;
    out[1] = xm > 0.f ? 2.f / xm : 0.f;
}

__global__ void k_scale_vec(long n, float* __restrict__ v, const float* __restrict__ s) {
    pdl_wait();
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) v[i] *= *s;
}

__global__ void k_adam(long n, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       float lr, float b1, float b2, float eps, float c1, float c2) {
    pdl_wait();
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void k_to_bf16(long n, const float* __restrict__ p, __nv_bfloat16* __restrict__ out) {
    pdl_wait();
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = __float2bfloat16(p[i]);
}

// wt[c][o][k] = W[o][c][8 - k]
__global__ void k_flip(int Ci, int Co, const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wt) {
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= Ci * Co * 9) return;
    const int k = t % 9, o = (t / 9) % Co, c = t / (9 * Co);
    wt[t] = w[((size_t)o * Ci + c) * 9 + (8 - k)];
}

// x[b] = (omega s0, phi s1, ub s2) on the interior grid, channel planes of NX x NY
__global__ void k_net_input(int NX, int NY, const double* __restrict__ omega, const double* __restrict__ phi,
                            const double* __restrict__ ub, float s0, float s1, float s2, float* __restrict__ x) {
    pdl_wait();
    const long n = (long)NX * NY;
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int i = (int)(k % NX), j = (int)(k / NX);
    const double ph = phi[(long)(j + 1) * (NX + 2) + (i + 1)];
    x[k] = (float)(ph >= 0.0 ? omega[k] * s0 : 0.0);
    x[n + k] = (float)(ph * s1);
    x[2 * n + k] = (float)(ub[k] * s2);
}

// psi = ub + y / s
__global__ void k_net_guess(long n, const double* __restrict__ ub, const float* __restrict__ y, float inv_s,
                            double* __restrict__ psi) {
    pdl_wait();
    const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) psi[k] = ub[k] + (double)(y[k] * inv_s);
}

static size_t conv_smem(int d, int co_t) { return sizeof(float) * ((size_t)(TX + 2 * d) * (TY + 2 * d) + 9 * co_t); }

static iim_status conv(iim_net_s* net, const float* x, const float* gate, const __nv_bfloat16* w, const float* bias,
                       float* y, int B, int Ci, int Co, int H, int W, int d, int relu, cudaStream_t s) {
    const dim3 blk(TX, TY);
    // tensor cores: mode 1 the 32 -> 32 layers, mode 2 every layer (K and N padded to 16 / 32)
    if ((net->tc == 1 && Ci == TC_C && Co == TC_C) || (net->tc == 2 && Ci <= TC_C && Co <= TC_C)) {
        auto go = [&](auto pack, auto kern, int cg, int no) -> iim_status {
            launch_next("net_pack_w_tc", 0.0, 0.0, pack, (9 * cg * no * 8 + 255) / 256, 256, 0, s, w, net->wtc, Ci, Co);
            IIM_LAUNCHED();
            const size_t sm = conv_tc_smem(d, cg, no);
            IIM_CHECK(allow_smem(kern, sm));
            launch_next("net_conv_tc", 4.0 * (double)B * H * W * (Ci * (gate ? 2 : 1) + Co),
                   18.0 * (double)B * H * W * Ci * Co, kern, dim3((W + TC_M - 1) / TC_M, H, B), 128, sm, s, x, gate,
                   (const __nv_bfloat16*)net->wtc, bias, y, Ci, Co, H, W, d, relu, net->tc_err);
            IIM_LAUNCHED();
            return IIM_OK;
        };
        if (Ci <= 16 && Co <= 16) return go(k_pack_w_tc<2, 16>, k_conv_tc<2, 16>, 2, 16);
        if (Ci <= 16) return go(k_pack_w_tc<2, 32>, k_conv_tc<2, 32>, 2, 32);
        if (Co <= 16) return go(k_pack_w_tc<4, 16>, k_conv_tc<4, 16>, 4, 16);
        return go(k_pack_w_tc<4, 32>, k_conv_tc<4, 32>, 4, 32);
    }
    if (Co > 1) {
        const int ncot = (Co + 31) / 32;
        const size_t sm = conv_smem(d, 32);
        IIM_CHECK(allow_smem(k_conv<32>, sm));
        launch_next("net_conv", 4.0 * (double)B * H * W * (Ci + Co), 18.0 * (double)B * H * W * Ci * Co, k_conv<32>,
               dim3((W + TX - 1) / TX, (H + TY - 1) / TY, B * ncot), blk, sm, s, x, gate, w, bias, y, Ci, Co, H, W, d, relu);
    } else {
        const size_t sm = conv_smem(d, 1);
        launch_next("net_conv", 4.0 * (double)B * H * W * (Ci + Co), 18.0 * (double)B * H * W * Ci * Co, k_conv<1>,
               dim3((W + TX - 1) / TX, (H + TY - 1) / TY, B), blk, sm, s, x, gate, w, bias, y, Ci, Co, H, W, d, relu);
    }
    IIM_LAUNCHED();
    return IIM_OK;
}

static int max_dilation(const iim_net_s* net) { return *std::max_element(net->dil.begin(), net->dil.end()); }

// The buffers at `parts` (bytes per item each) grown to hold `need` items.  Outgrown ones are kept until the
// net is destroyed, since a caller's graph may hold them; they grow by doubling, so that those add up to
// less than the last.  Only where the device has no room beside them are they given up (`optional`: left as
// they are, with an error).
struct NetPart {
    void** p;
    size_t bytes;
};
static iim_status grow(NetBuffers& b, size_t need, std::initializer_list<NetPart> parts, bool optional = false) {
    if (need <= b.n) return IIM_OK;
    std::vector<void*> got;
    auto alloc = [&](size_t n) {
        for (const NetPart& part : parts) {
            void* q = nullptr;
            const cudaError_t e = cudaMalloc(&q, n * part.bytes);
            if (e != cudaSuccess) {
                cudaGetLastError();
                for (void* r : got) cudaFree(r);
                got.clear();
                return e;
            }
            got.push_back(q);
        }
        return cudaSuccess;
    };
    size_t n = std::max(need, 2 * b.n);
    cudaError_t e = alloc(n);
    if (e == cudaErrorMemoryAllocation && !optional) {
        for (void* q : b.old) cudaFree(q);
        b.old.clear();
        for (const NetPart& part : parts) {
            cudaFree(*part.p);
            *part.p = nullptr;
        }
        b.n = 0;
        n = need;
        e = alloc(n);
    }
    if (e != cudaSuccess) {
        if (!optional) record_cuda_error(e, "cudaMalloc", __FILE__, __LINE__);
        return IIM_ERR_CUDA;
    }
    size_t k = 0;
    for (const NetPart& part : parts) {
        if (*part.p) b.old.push_back(*part.p);
        *part.p = got[k++];
    }
    b.n = n;
    return IIM_OK;
}
// Activations and gradients of training (and of inference off the tensor cores) for B images.
static size_t act_floats(const iim_net_s* net, int B, int H, int W) {
    return (size_t)B * H * W * std::max(net->hidden, 1);
}
static iim_status ensure_acts(iim_net_s* net, size_t need, bool optional = false) {
    return grow(net->acts, need, {{(void**)&net->act, sizeof(float) * net->nl}, {(void**)&net->g0, sizeof(float) * 2}},
                optional);
}

// The whole network on the tensor cores for inference (every layer; net->tc == 2): y (batch, 1, h, w).
static iim_status forward_units(iim_net_s* net, int B, int H, int W, const float* x, float* y, cudaStream_t s) {
    const int D = max_dilation(net);
    const UnitLayout u{H, W, H + 2 * D, (W + UN_M - 1) / UN_M * UN_M + 2 * D, D};
    int planes = (net->cin + 7) / 8;
    if (net->nl > 1) planes = std::max(planes, (net->hidden + 7) / 8);
    const size_t need = (size_t)B * planes * u.Hp * u.Wp;
    IIM_CHECK(grow(net->units, need, {{(void**)&net->unit[0], sizeof(uint4)}, {(void**)&net->unit[1], sizeof(uint4)}}));
    if (!net->wunit) IIM_TRY(cudaMalloc(&net->wunit, sizeof(uint4) * WUNIT * net->nl));
    UnitLayers L{net->nl};
    for (int l = 0; l < net->nl; ++l) {
        L.ci[l] = net->ci[l];
        L.co[l] = net->co[l];
        L.woff[l] = net->woff[l];
    }
    const long plane = (long)H * W, border = (long)(D + 1) * (W + 2 * D) + 2L * D * H;
    const int nw = (WUNIT * net->nl + 255) / 256, nb = (int)((border + 255) / 256), P = B * planes;
    const int nx0 = (int)((plane + 255) / 256);
    launch_next("net_to_units", 4.0 * plane * B * net->cin, 0.0, k_units_begin,
           nw + nb * P + nx0 * ((net->cin + 7) / 8) * B, 256, 0, s, x, net->cin, u, net->unit[0], net->unit[1],
           (const __nv_bfloat16*)net->wb, L, reinterpret_cast<uint4*>(net->wunit), nw, nb, P, nx0);
    IIM_LAUNCHED();
    for (int l = 0; l < net->nl; ++l) {
        const int ci = net->ci[l], co = net->co[l], d = net->dil[l], gin = (ci + 7) / 8;
        const bool last = l == net->nl - 1;
        const int nx = (W + UN_M - 1) / UN_M, nr = (H + UN_R * d - 1) / (UN_R * d) * d, tiles = nx * nr * B;
        auto go = [&](auto kern, int cg, int no) -> iim_status {
            const size_t sm = conv_units_smem(d, cg, no);
            IIM_CHECK(allow_smem(kern, sm));
            const int per_sm = std::max(1, (int)(227 * 1024 / (sm + 1024)));   // resident blocks (also 512 TMEM columns / 128)
            const int blocks = std::min(tiles, std::min(per_sm, 4) * sm_count());
            launch_next("net_conv_tc", 2.0 * plane * B * (8.0 * gin + (last ? 2.0 : 8.0 * ((co + 7) / 8))),
                   18.0 * (double)B * plane * ci * co, kern, blocks, 128, sm, s, (const uint4*)net->unit[l & 1], gin,
                   (const __nv_bfloat16*)(net->wunit + (size_t)WUNIT * 8 * l), (const float*)(net->p + net->boff[l]), co,
                   net->unit[(l + 1) & 1], (co + 7) / 8, last ? y : (float*)nullptr, u, d, nx, nr, tiles, net->tc_err);
            IIM_LAUNCHED();
            return IIM_OK;
        };
        const int cg = mma_groups(ci), no = mma_cols(co);
        IIM_CHECK(cg == 2 ? (no == 16 ? go(k_conv_units<2, 16>, 2, 16) : go(k_conv_units<2, 32>, 2, 32))
                          : (no == 16 ? go(k_conv_units<4, 16>, 4, 16) : go(k_conv_units<4, 32>, 4, 32)));
    }
    return IIM_OK;
}

static iim_status forward(iim_net_s* net, int B, int H, int W, const float* x, cudaStream_t s) {
    IIM_CHECK(ensure_acts(net, act_floats(net, B, H, W)));
    const float* in = x;
    for (int l = 0; l < net->nl; ++l) {
        float* out = net->act + (size_t)l * net->cap();
        IIM_CHECK(conv(net, in, nullptr, net->wb + net->woff[l], net->p + net->boff[l], out, B, net->ci[l], net->co[l], H, W,
                       net->dil[l], l < net->nl - 1, s));
        in = out;
    }
    return IIM_OK;
}

// gradients of sum(dy * pred) w.r.t. the parameters (into net->gr); dy is overwritten
static iim_status backward(iim_net_s* net, int B, int H, int W, const float* x, float* dy, cudaStream_t s) {
    float* g = dy;
    for (int l = net->nl - 1; l >= 0; --l) {
        const float* xin = l == 0 ? x : net->act + (size_t)(l - 1) * net->cap();
        const float* gate = l == net->nl - 1 ? nullptr : net->act + (size_t)l * net->cap();
        const int d = net->dil[l];
        const size_t sm = wgrad_smem(wg_groups(net->co[l], 8), wg_groups(net->ci[l], 4), d);
        const int strips = B * H * ((W + WG_PX - 1) / WG_PX), nblk = std::min(strips, net->wg_blocks);
        const int nw = net->ci[l] * net->co[l] * 9 + net->co[l];   // the layer's weights, then its biases
        IIM_CHECK(allow_smem(k_conv_wgrad, sm));
        launch_next("net_wgrad", 4.0 * (double)B * H * W * (net->ci[l] + net->co[l]), 2.0 * B * H * W * 9.0 * net->ci[l] * net->co[l],
               k_conv_wgrad, nblk, WG_THREADS, sm, s, xin, (const float*)g, gate, net->wgp, net->ci[l], net->co[l], H, W, d,
               strips);
        launch_next("net_wgrad_sum", 4.0 * nblk * (double)nw, 0.0, k_wgrad_sum, (nw + 31) / 32, 256, 0, s, nblk, nw,
               (const float*)net->wgp, net->gr + net->woff[l]);
        IIM_LAUNCHED();
        if (l > 0) {
            const int n = net->ci[l] * net->co[l] * 9;
            launch_next("net_flip", 0.0, 0.0, k_flip, (n + 255) / 256, 256, 0, s, net->ci[l], net->co[l],
                   (const __nv_bfloat16*)(net->wb + net->woff[l]), net->wt);
            float* gprev = net->g0 + (size_t)((net->nl - 1 - l) & 1) * net->cap();
            IIM_CHECK(conv(net, g, gate, net->wt, nullptr, gprev, B, net->co[l], net->ci[l], H, W, d, 0, s));
            g = gprev;
        }
    }
    return IIM_OK;
}

static iim_status sync_bf16(iim_net_s* net, cudaStream_t s) {
    launch_next("net_bf16", 0.0, 0.0, k_to_bf16, (unsigned)((net->np + 255) / 256), 256, 0, s, (long)net->np,
           (const float*)net->p, net->wb);
    IIM_LAUNCHED();
    return IIM_OK;
}

}  // namespace iim

using namespace iim;

extern "C" iim_status iim_net_create(int in_channels, int hidden, int n_layers, const int* dilations,
                                     unsigned long long seed, iim_net* out) {
    if (!out) return IIM_ERR_INVALID_ARG;
    *out = nullptr;
    if (in_channels < 1 || in_channels > 32 || hidden < 1 || hidden > 32 || n_layers < 1 || n_layers > 16 || !dilations)
        return IIM_ERR_INVALID_ARG;
    for (int l = 0; l < n_layers; ++l)
        if (dilations[l] < 1 || dilations[l] > 32) return IIM_ERR_INVALID_ARG;
    iim_net_s* net = new iim_net_s();
    cudaGetDevice(&net->device);
    net->cin = in_channels;
    net->hidden = hidden;
    net->nl = n_layers;
    long long off = 0;
    for (int l = 0; l < n_layers; ++l) {
        net->dil.push_back(dilations[l]);
        net->ci.push_back(l == 0 ? in_channels : hidden);
        net->co.push_back(l == n_layers - 1 ? 1 : hidden);
        net->woff.push_back(off);
        off += (long long)net->ci[l] * net->co[l] * 9;
        net->boff.push_back(off);
        off += net->co[l];
    }
    net->np = off;
    std::vector<float> h(off, 0.f);
    std::mt19937_64 rng(seed);
    for (int l = 0; l < n_layers; ++l) {
        // He-uniform initialisation, zero biases
        const float a = std::sqrt(6.f / (9.f * net->ci[l]));
        std::uniform_real_distribution<float> U(-a, a);
        for (long long k = 0; k < (long long)net->ci[l] * net->co[l] * 9; ++k) h[net->woff[l] + k] = U(rng);
    }
    auto fail = [&](cudaError_t e) {
        record_cuda_error(e, "iim_net_create", __FILE__, __LINE__);
        cudaFree(net->p); cudaFree(net->gr); cudaFree(net->m); cudaFree(net->v); cudaFree(net->wb); cudaFree(net->wt);
        cudaFree(net->red); cudaFree(net->wtc); cudaFree(net->tc_err); cudaFree(net->wgp);
        delete net;
        return IIM_ERR_CUDA;
    };
    cudaError_t e;
    if ((e = cudaMalloc(&net->p, sizeof(float) * off)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->gr, sizeof(float) * off)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->m, sizeof(float) * off)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->v, sizeof(float) * off)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->wb, sizeof(__nv_bfloat16) * off)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->wt, sizeof(__nv_bfloat16) * 32 * 32 * 9)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->red, sizeof(float) * 4096)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->wtc, sizeof(__nv_bfloat16) * 9 * 4 * TC_C * 8)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc(&net->tc_err, sizeof(int))) != cudaSuccess) return fail(e);
    net->wg_blocks = 2 * sm_count();   // two resident blocks per SM
    if ((e = cudaMalloc(&net->wgp, sizeof(float) * (size_t)net->wg_blocks * WG_PART)) != cudaSuccess) return fail(e);
    cudaMemset(net->tc_err, 0, sizeof(int));
    net->tc = 2;
    if ((e = cudaMemcpy(net->p, h.data(), sizeof(float) * off, cudaMemcpyHostToDevice)) != cudaSuccess) return fail(e);
    cudaMemset(net->m, 0, sizeof(float) * off);
    cudaMemset(net->v, 0, sizeof(float) * off);
    if (cudaMallocHost(&net->h_red, 4 * sizeof(float)) != cudaSuccess) return fail(cudaErrorMemoryAllocation);
    if (sync_bf16(net, nullptr) != IIM_OK) return fail(cudaGetLastError());
    cudaDeviceSynchronize();
    *out = net;
    return IIM_OK;
}

extern "C" long long iim_net_num_params(iim_net net) { return net ? net->np : 0; }

extern "C" iim_status iim_net_get_params(iim_net net, float* host, long long n) {
    if (!net || !host || n != net->np) return IIM_ERR_INVALID_ARG;
    IIM_TRY(cudaMemcpy(host, net->p, sizeof(float) * n, cudaMemcpyDeviceToHost));
    return IIM_OK;
}

extern "C" iim_status iim_net_set_params(iim_net net, const float* host, long long n) {
    if (!net || !host || n != net->np) return IIM_ERR_INVALID_ARG;
    IIM_TRY(cudaMemcpy(net->p, host, sizeof(float) * n, cudaMemcpyHostToDevice));
    IIM_TRY(cudaMemset(net->m, 0, sizeof(float) * n));
    IIM_TRY(cudaMemset(net->v, 0, sizeof(float) * n));
    net->t = 0;
    IIM_CHECK(sync_bf16(net, nullptr));
    IIM_TRY(cudaDeviceSynchronize());
    return IIM_OK;
}

extern "C" iim_status iim_net_forward(iim_net net, int batch, int height, int width, const float* x, float* y,
                                      iim_stream stream) {
    if (!net || !x || !y || batch < 1 || height < 1 || width < 1) return IIM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    // one image's planes and the tiles are counted in 32 bits
    if (net->tc == 2 && (long long)batch * ((height + 127) / 4 + 1) * (width / UN_M + 1) < (1LL << 30) && batch <= 65535) {
        // the buffers of a training step of this size, which a stream capture could not allocate after this
        // call; inference itself does without them
        const size_t need = act_floats(net, batch, height, width);
        if (need > net->act_try) {
            cudaStreamCaptureStatus st = cudaStreamCaptureStatusActive;
            if (cudaStreamIsCapturing(s, &st) != cudaSuccess) cudaGetLastError();
            if (st == cudaStreamCaptureStatusNone) {
                net->act_try = need;
                (void)ensure_acts(net, need, true);
            }
        }
        return forward_units(net, batch, height, width, x, y, s);
    }
    IIM_CHECK(forward(net, batch, height, width, x, s));
    IIM_TRY(cudaMemcpyAsync(y, net->act + (size_t)(net->nl - 1) * net->cap(), sizeof(float) * (size_t)batch * height * width,
                            cudaMemcpyDeviceToDevice, s));
    return IIM_OK;
}

extern "C" iim_status iim_net_backward(iim_net net, int batch, int height, int width, const float* x, const float* dy,
                                       float* grad_host, iim_stream stream) {
    if (!net || !x || !dy || batch < 1 || height < 1 || width < 1) return IIM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    IIM_CHECK(forward(net, batch, height, width, x, s));
    const size_t n = (size_t)batch * height * width;
    float* g = net->g0 + net->cap();   // scratch copy of dy (the backward pass overwrites its input)
    IIM_TRY(cudaMemcpyAsync(g, dy, sizeof(float) * n, cudaMemcpyDeviceToDevice, s));
    IIM_CHECK(backward(net, batch, height, width, x, g, s));
    if (grad_host) {
        IIM_TRY(cudaMemcpyAsync(grad_host, net->gr, sizeof(float) * (size_t)net->np, cudaMemcpyDeviceToHost, s));
        IIM_TRY(cudaStreamSynchronize(s));
    }
    return IIM_OK;
}

extern "C" iim_status iim_net_train_step(iim_net net, int batch, int height, int width, const float* x,
                                         const float* target, const float* mask, float lr, float* loss,
                                         iim_stream stream) {
    if (!net || !x || !target || batch < 1 || height < 1 || width < 1 || !(lr >= 0.f)) return IIM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    IIM_CHECK(forward(net, batch, height, width, x, s));
    const long n = (long)batch * height * width;
    const float* pred = net->act + (size_t)(net->nl - 1) * net->cap();
    float* diff = net->g0 + net->cap();
    const int nb = 256;
    launch_next("net_mse", 12.0 * n, 0.0, k_mse_partial, nb, 256, 0, s, n, pred, target, mask, diff, net->red);
    launch_next("net_mse_finish", 0.0, 0.0, k_mse_finish, 1, 32, 0, s, nb, net->red, net->red + 1024);
    launch_next("net_scale", 0.0, 0.0, k_scale_vec, (unsigned)((n + 255) / 256), 256, 0, s, n, diff, (const float*)(net->red + 1025));
    IIM_LAUNCHED();
    IIM_CHECK(backward(net, batch, height, width, x, diff, s));
    net->t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)net->t), c2 = 1.f - std::pow(b2, (float)net->t);
    launch_next("net_adam", 0.0, 0.0, k_adam, (unsigned)((net->np + 255) / 256), 256, 0, s, (long)net->np, net->p,
           (const float*)net->gr, net->m, net->v, lr, b1, b2, 1e-8f, c1, c2);
    IIM_LAUNCHED();
    IIM_CHECK(sync_bf16(net, s));
    if (loss) {
        IIM_TRY(cudaMemcpyAsync(net->h_red, net->red + 1024, sizeof(float), cudaMemcpyDeviceToHost, s));
        IIM_TRY(cudaStreamSynchronize(s));
        *loss = net->h_red[0];
    }
    return IIM_OK;
}

extern "C" iim_status iim_net_prepare_input(int nx, int ny, const double* omega, const double* phi_nodes,
                                            const double* u_box, float s_omega, float s_phi, float s_box, float* x,
                                            iim_stream stream) {
    if (nx < 3 || ny < 3 || !omega || !phi_nodes || !u_box || !x) return IIM_ERR_INVALID_ARG;
    const long n = (long)(nx - 1) * (ny - 1);
    launch_next("net_input", 0.0, 0.0, k_net_input, (unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream, nx - 1, ny - 1,
           omega, phi_nodes, u_box, s_omega, s_phi, s_box, x);
    IIM_LAUNCHED();
    return IIM_OK;
}

extern "C" iim_status iim_net_compose_guess(long long n, const double* u_box, const float* y, float s_out,
                                            double* psi_guess, iim_stream stream) {
    if (n < 0 || !u_box || !y || !psi_guess || !(s_out != 0.f)) return IIM_ERR_INVALID_ARG;
    launch_next("net_guess", 0.0, 0.0, k_net_guess, (unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream, (long)n, u_box, y,
           1.f / s_out, psi_guess);
    IIM_LAUNCHED();
    return IIM_OK;
}

extern "C" iim_status iim_net_set_tensor_cores(iim_net net, int on) {
    if (!net || on < 0 || on > 2) return IIM_ERR_INVALID_ARG;
    net->tc = on;
    return IIM_OK;
}

extern "C" iim_status iim_net_tensor_core_status(iim_net net, int* on, int* timed_out) {
    if (!net || !on || !timed_out) return IIM_ERR_INVALID_ARG;
    *on = net->tc;
    IIM_TRY(cudaDeviceSynchronize());
    IIM_TRY(cudaMemcpy(timed_out, net->tc_err, sizeof(int), cudaMemcpyDeviceToHost));
    return IIM_OK;
}

extern "C" void iim_net_destroy(iim_net net) {
    if (!net) return;
    cudaFree(net->p); cudaFree(net->gr); cudaFree(net->m); cudaFree(net->v); cudaFree(net->wb); cudaFree(net->wt);
    cudaFree(net->act); cudaFree(net->g0); cudaFree(net->red); cudaFree(net->wgp);
    for (const NetBuffers* b : {&net->acts, &net->units})
        for (void* p : b->old) cudaFree(p);
    cudaFree(net->wunit); cudaFree(net->unit[0]); cudaFree(net->unit[1]); cudaFree(net->wtc); cudaFree(net->tc_err);
    if (net->h_red) cudaFreeHost(net->h_red);
    delete net;
}
