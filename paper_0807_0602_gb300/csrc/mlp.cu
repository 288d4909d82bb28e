// Surrogate network of include/mlp.h: 6 -> 128 -> 128 -> 128 -> 3 with the
// exact GELU, bfloat16 GEMM operands and FP32 accumulation on the tensor
// cores (mma.sync.m16n8k16), FP32 biases, activations and Adam state.
//
// What bounds these kernels is latency, not a rate: a call has a few hundred
// to a few thousand rows, 34 kFLOP each, and a chain of four layers.  So
//   - a CTA of 16 warps takes 16 (or 64) rows through the whole chain in
//     shared memory, each warp one 8-column slice of every hidden layer;
//   - the weights are kept in global memory in the order in which the lanes
//     of an mma fragment hold them (one 16-byte load covers two k steps), in
//     the forward and in the transposed order; the warps load them straight
//     into registers, all layers at once, so no load waits for a layer;
//   - the forward and the backward pass of a training step are one kernel
//     (the GELU derivatives stay in registers between them);
//   - the gradients sum over the rows in order, in chunks of 512 rows that
//     the kernel of the Adam update adds in order (it also refreshes the
//     packed weights): deterministic, no atomics;
//   - the three kernels of a step are launched with programmatic dependent
//     launch, which hides the launch gaps.
// tcgen05 tiles are 128 rows: at these batches they would occupy 4 to 32 of
// the 152 SMs and add TMEM set-up to each link of the chain.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "mlp.h"

namespace {

constexpr int NL = 4;
// valid fan-in / fan-out per layer, and both padded to the mma tile (16, 8)
__host__ __device__ constexpr int IN(int l) { return l == 0 ? 6 : 128; }
__host__ __device__ constexpr int OUT(int l) { return l == 3 ? 3 : 128; }
__host__ __device__ constexpr int KP(int l) { return l == 0 ? 16 : 128; }
__host__ __device__ constexpr int NP(int l) { return l == 3 ? 8 : 128; }
// first parameter of layer l's weights and biases in the flat vector
constexpr int kHidden0 = 6 * 128 + 128, kHidden = 128 * 128 + 128;
__host__ __device__ constexpr int WOFF(int l) { return l == 0 ? 0 : kHidden0 + (l - 1) * kHidden; }
__host__ __device__ constexpr int BOFF(int l) { return WOFF(l) + IN(l) * OUT(l); }
static_assert(BOFF(3) + OUT(3) == MLP_N_PARAMS, "layer offsets");

constexpr int NBIAS = 3 * 128 + 3;          // bias gradients of all layers, layer order
constexpr int NPART = MLP_N_PARAMS + 5;     // row of the chunk partials (weights, biases; padded)
constexpr int kChunkRows = 512;            // rows per chunk of the gradient sums
constexpr int kDzf = 388;                   // row of the FP32 dL/dz of all layers (biases, padded)
constexpr int kWgradThreads = 256;

struct Dev {
    float* theta;            // FP32 master parameters, flat layer order
    float* m;                // Adam first moment
    float* v;                // Adam second moment
    // packed bfloat16 weights in mma B-fragment order: layer l as the k x n
    // operand of the forward pass (wf), and transposed for the backward (wb)
    __nv_bfloat16* wf[NL];
    __nv_bfloat16* wb[NL];
    // activation scratch for max_batch rows
    __nv_bfloat16* A[NL];    // layer inputs [rows][KP]
    __nv_bfloat16* DZ[NL];   // dL/dz per layer [rows][NP]
    float* DZF;              // the same in FP32, all layers side by side [rows][kDzf]: bias gradients
    float* lpart;            // sums of squared errors per tile
    float* part;             // [chunks][NPART] partial gradients
    float* lchunk;           // partial losses per chunk
};

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p))
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p))
                 : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(smem_addr(p))
                 : "memory");
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Fragment layout of m16n8k16: lane = 4 g + q; A holds rows g, g + 8 and
// columns 2q, 2q + 1, 2q + 8, 2q + 9; B holds rows 2q, 2q + 1 (register 0),
// 2q + 8, 2q + 9 (register 1) of column g; C holds (g, 2q), (g, 2q + 1),
// (g + 8, 2q), (g + 8, 2q + 1).
//
// Packed position (in bfloat16 units) of element (k, c) of a B operand with
// K = 128 (two k steps per 16-byte lane word) or K = 16 (8-byte lane words).
__device__ __forceinline__ int frag_pos(bool k128, int k, int c) {
    const int nt = c >> 3, g = c & 7, ks = k >> 4, kk = k & 15;
    const int lane = g * 4 + ((kk & 7) >> 1), reg = kk >> 3;
    if (k128) return ((((nt * 4 + (ks >> 1)) * 32 + lane) * 4) + (ks & 1) * 2 + reg) * 2 + (kk & 1);
    return (((nt * 32 + lane) * 2) + reg) * 2 + (kk & 1);
}

// Writes weight (k, c) of layer l into both packed copies.
__device__ __forceinline__ void pack_weight(const Dev& d, int l, int k, int c, float w) {
    const __nv_bfloat16 b = __float2bfloat16_rn(w);
    d.wf[l][frag_pos(l != 0, k, c)] = b;
    if (l > 0) d.wb[l][frag_pos(l != 3, c, k)] = b;
}

// Layer and element of weight parameter i (false for a bias).
__device__ __forceinline__ bool weight_of(int i, int& l, int& k, int& c) {
    l = i < WOFF(1) ? 0 : (i < WOFF(2) ? 1 : (i < WOFF(3) ? 2 : 3));
    const int base = l == 0 ? WOFF(0) : (l == 1 ? WOFF(1) : (l == 2 ? WOFF(2) : WOFF(3)));
    const int j = i - base, out = OUT(l);
    if (j >= IN(l) * out) return false;
    k = l == 3 ? j / 3 : j >> 7;
    c = j - k * out;
    return true;
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

constexpr int kThreads = 512;   // 16 warps: one 8-column slice of a hidden layer each
constexpr int kLd = 128 + 8;    // row stride of the activation tiles (conflict-free ldmatrix)

// B fragments of one 8-column slice of a K = 128 operand.
struct Frag128 {
    uint4 w[4];
    __device__ __forceinline__ void load(const __nv_bfloat16* p, int nt, int lane) {
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = reinterpret_cast<const uint4*>(p)[(nt * 4 + j) * 32 + lane];
    }
};
// c += A[16 x 128] B over ascending k; a: the lane's ldmatrix row of the tile
__device__ __forceinline__ void mma128(float (&c)[4], const __nv_bfloat16* a, const Frag128& f) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t x[4], y[4];
        ldsm4(x, a + 32 * j);
        ldsm4(y, a + 32 * j + 16);
        mma16816(c, x, f.w[j].x, f.w[j].y);
        mma16816(c, y, f.w[j].z, f.w[j].w);
    }
}

__device__ __forceinline__ void store2(__nv_bfloat16* p, float lo, float hi) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(lo, hi);
}

// Forward pass of tiles of 16 MT rows; a CTA keeps its weights in registers
// over all the tiles it takes.  Bound by the latency of the chain of layers
// (1201 rows: 2.9 us; with fragments assembled element by element from global
// memory by 4 warps it was 23.9 us), from about 30 000 rows on by erff (65536
// rows: 38 us, before 109 us).
template <int MT>
__global__ void __launch_bounds__(kThreads) k_fwd(Dev d, const float* __restrict__ X, int n, float* __restrict__ Y) {
    __shared__ __align__(16) __nv_bfloat16 act[2][16 * MT][kLd];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
    pdl_launch();
    pdl_wait();
    const int arow = lane & 15, acol = (lane >> 4) * 8;   // ldmatrix row and column of this lane
    const int col = warp * 8 + 2 * q;
    const uint2 w0 = reinterpret_cast<const uint2*>(d.wf[0])[warp * 32 + lane];
    Frag128 w[2], w3;
    w[0].load(d.wf[1], warp, lane);
    w[1].load(d.wf[2], warp, lane);
    if (warp < MT) w3.load(d.wf[3], 0, lane);
    float bias[3][2];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        bias[l][0] = d.theta[BOFF(l) + col];
        bias[l][1] = d.theta[BOFF(l) + col + 1];
    }
    const float b3[2] = {2 * q < 3 ? d.theta[BOFF(3) + 2 * q] : 0.f, 2 * q + 1 < 3 ? d.theta[BOFF(3) + 2 * q + 1] : 0.f};
    const int ntiles = (n + 16 * MT - 1) / (16 * MT);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int row0 = tile * 16 * MT;
        for (int i = tid; i < 16 * MT * 16; i += kThreads) {
            const int r = i >> 4, c = i & 15;
            const float v = (row0 + r < n && c < 6) ? X[(long long)(row0 + r) * 6 + c] : 0.0f;
            act[0][r][c] = __float2bfloat16_rn(v);
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const int cur = l & 1, nxt = cur ^ 1;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                float c[4] = {0.f, 0.f, 0.f, 0.f};
                const __nv_bfloat16* a = &act[cur][16 * mt + arow][acol];
                if (l == 0) {
                    uint32_t x[4];
                    ldsm4(x, a);
                    mma16816(c, x, w0.x, w0.y);
                } else {
                    mma128(c, a, w[l - 1]);
                }
                __nv_bfloat16* o = &act[nxt][16 * mt + g][col];
                store2(o, gelu(c[0] + bias[l][0]), gelu(c[1] + bias[l][1]));
                store2(o + 8 * kLd, gelu(c[2] + bias[l][0]), gelu(c[3] + bias[l][1]));
            }
            __syncthreads();
        }
        if (warp < MT) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            mma128(c, &act[1][16 * warp + arow][acol], w3);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int r = row0 + 16 * warp + g + (e >> 1) * 8, cc = 2 * q + (e & 1);
                if (cc < 3 && r < n) Y[(long long)r * 3 + cc] = c[e] + b3[e & 1];
            }
        }
    }
}

// Forward and backward pass of 16 MT rows: layer inputs and dL/dz of every
// layer in bfloat16 (the operands of the weight gradients), dL/dz in FP32
// (the bias gradients) and the squared error per 16 rows.  idx: the batch is
// the rows idx[0 .. n) of X and T (nullptr: the first n rows); gathering them
// here costs a load in front of the chain instead of two kernels per batch.
template <int MT>
__global__ void __launch_bounds__(kThreads) k_train(Dev d, const float* __restrict__ X, const float* __restrict__ T,
                                                    const long long* __restrict__ idx, long long nrows, int n) {
    __shared__ __align__(16) __nv_bfloat16 act[2][16 * MT][kLd];
    __shared__ float sq[MT][48];   // squared errors of each 16 rows, row by row
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
    pdl_launch();
    pdl_wait();
    const int row0 = blockIdx.x * 16 * MT;
    const int arow = lane & 15, acol = (lane >> 4) * 8;
    const int col = warp * 8 + 2 * q;
    const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
    // element e of mma tile mt of this lane: row row0 + row(mt, e / 2)
    auto row = [&](int mt, int e) { return 16 * mt + g + 8 * e; };
    auto live = [&](int mt, int e) { return row0 + row(mt, e) < n; };
    auto source = [&](int r) -> long long {   // row of X and T (row 0 for a number out of range)
        if (!idx) return r;
        const long long i = idx[r];
        return i >= 0 && i < nrows ? i : 0;
    };
    float xv = 0.0f;
    const int xr = tid >> 4, xc = tid & 15;
    if (xr < 16 * MT && row0 + xr < n && xc < 6) xv = X[source(row0 + xr) * 6 + xc];
    const uint2 w0 = reinterpret_cast<const uint2*>(d.wf[0])[warp * 32 + lane];
    Frag128 w[2], w3;
    w[0].load(d.wf[1], warp, lane);
    w[1].load(d.wf[2], warp, lane);
    float t3[4] = {0.f, 0.f, 0.f, 0.f}, b3[2] = {0.f, 0.f};
    if (warp < MT) {
        w3.load(d.wf[3], 0, lane);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int cc = 2 * q + (e & 1);
            if (cc < 3 && live(warp, e >> 1)) t3[e] = T[source(row0 + row(warp, e >> 1)) * 3 + cc];
            if (cc < 3) b3[e & 1] = d.theta[BOFF(3) + cc];
        }
    }
    float bias[3][2];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        bias[l][0] = d.theta[BOFF(l) + col];
        bias[l][1] = d.theta[BOFF(l) + col + 1];
    }
    if (xr < 16 * MT) {
        const __nv_bfloat16 b = __float2bfloat16_rn(xv);
        act[0][xr][xc] = b;
        d.A[0][(long long)(row0 + xr) * 16 + xc] = b;
    }
    __syncthreads();
    float dg[3][MT][4];   // GELU derivatives of this lane's elements
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const int cur = l & 1, nxt = cur ^ 1;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            const __nv_bfloat16* a = &act[cur][16 * mt + arow][acol];
            if (l == 0) {
                uint32_t x[4];
                ldsm4(x, a);
                mma16816(c, x, w0.x, w0.y);
            } else {
                mma128(c, a, w[l - 1]);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float za = c[2 * e] + bias[l][0], zb = c[2 * e + 1] + bias[l][1];
                const __nv_bfloat162 h = __floats2bfloat162_rn(gelu(za), gelu(zb));
                dg[l][mt][2 * e] = gelu_grad(za);
                dg[l][mt][2 * e + 1] = gelu_grad(zb);
                *reinterpret_cast<__nv_bfloat162*>(&act[nxt][row(mt, e)][col]) = h;
                // rows beyond the batch enter the weight gradients as zeros
                *reinterpret_cast<__nv_bfloat162*>(d.A[l + 1] + (long long)(row0 + row(mt, e)) * 128 + col) =
                    live(mt, e) ? h : zero;
            }
        }
        __syncthreads();
    }
    const uint2 v3 = reinterpret_cast<const uint2*>(d.wb[3])[warp * 32 + lane];
    Frag128 v[2];
    v[1].load(d.wb[2], warp, lane);
    v[0].load(d.wb[1], warp, lane);
    // output layer (one warp per 16 rows): y, dL/dy = 2 (y - t) / (3 n), the squared error
    if (warp < MT) {
        const float scale = 2.0f / (float)(n * 3);
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma128(c, &act[1][16 * warp + arow][acol], w3);
        float dz[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int cc = 2 * q + (e & 1);
            const float err = (cc < 3 && live(warp, e >> 1)) ? c[e] + b3[e & 1] - t3[e] : 0.0f;
            dz[e] = scale * err;
            if (cc < 3) {
                sq[warp][(g + 8 * (e >> 1)) * 3 + cc] = err * err;
                d.DZF[(long long)(row0 + row(warp, e >> 1)) * kDzf + 384 + cc] = dz[e];
            }
        }
        // act[0] becomes the dL/dz tile; columns 8 .. 15 pad its K of 16
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(dz[2 * e], dz[2 * e + 1]);
            *reinterpret_cast<__nv_bfloat162*>(&act[0][row(warp, e)][2 * q]) = b;
            *reinterpret_cast<__nv_bfloat162*>(&act[0][row(warp, e)][8 + 2 * q]) = zero;
            *reinterpret_cast<__nv_bfloat162*>(d.DZ[3] + (long long)(row0 + row(warp, e)) * 8 + 2 * q) = b;
        }
    }
    __syncthreads();
#pragma unroll
    for (int l = 3; l >= 1; --l) {
        // dL/dz_{l-1} = (dL/dz_l W_l^T) gelu'(z_{l-1})
        const int cur = (3 - l) & 1, nxt = cur ^ 1;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            const __nv_bfloat16* a = &act[cur][16 * mt + arow][acol];
            if (l == 3) {
                uint32_t x[4];
                ldsm4(x, a);
                mma16816(c, x, v3.x, v3.y);
            } else {
                mma128(c, a, v[l - 1]);
            }
            float dz[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) dz[e] = live(mt, e >> 1) ? c[e] * dg[l - 1][mt][e] : 0.0f;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(dz[2 * e], dz[2 * e + 1]);
                if (l > 1) *reinterpret_cast<__nv_bfloat162*>(&act[nxt][row(mt, e)][col]) = h;
                *reinterpret_cast<__nv_bfloat162*>(d.DZ[l - 1] + (long long)(row0 + row(mt, e)) * 128 + col) = h;
                *reinterpret_cast<float2*>(d.DZF + (long long)(row0 + row(mt, e)) * kDzf + (l - 1) * 128 + col) =
                    make_float2(dz[2 * e], dz[2 * e + 1]);
            }
        }
        if (l > 1) __syncthreads();
    }
    if (tid < MT) {   // the squared errors of the tile, in order
        float t = 0.0f;
#pragma unroll
        for (int i = 0; i < 48; ++i) t += sq[tid][i];
        d.lpart[blockIdx.x * MT + tid] = t;
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Weight gradient of one block of layer l over the rows [r0, r1) (r1 - r0 a
// multiple of 16): gW = A_l^T DZ_l, WM x WN warps with one 16 x 8 mma tile each,
// the rows in ascending order in one accumulator.  The rows stream through S
// shared stages of 64; both operands are row-major in the rows (the mma's K),
// so the fragments come from transposing ldmatrix.
template <int WM, int WN, int S>
struct WgradTile {
    static constexpr int BI = WM * 16, BO = WN * 8;              // block: inputs x outputs
    static constexpr int LI = BI + 8, LO = BO + (BO == 8 ? 16 : 8);   // padded rows: no bank conflicts
    static constexpr int KB = 64;
    static constexpr int STAGE = KB * (LI + LO), ELEMS = S * STAGE;
    static_assert(WM * WN == kWgradThreads / 32, "one tile per warp");

    static __device__ __forceinline__ void run(__nv_bfloat16* sm, const __nv_bfloat16* A, int lda,
                                               const __nv_bfloat16* Z, int ldz, int r0, int r1, float* out, int ldo,
                                               int vi, int vo) {
        const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
        const int wm = warp / WN, wn = warp % WN;
        const int nst = (r1 - r0 + KB - 1) / KB;
        auto load = [&](int st) {   // stage st (nothing beyond the last one); always commits a group
            if (st < nst) {
                __nv_bfloat16* sa = sm + st % S * STAGE;
                __nv_bfloat16* sz = sa + KB * LI;
                const int r = r0 + st * KB, rows = min(KB, r1 - r);
                for (int i = tid; i < rows * (BI / 8); i += kWgradThreads) {
                    const int rr = i / (BI / 8), cc = i % (BI / 8) * 8;
                    cp_async16(sa + rr * LI + cc, A + (long long)(r + rr) * lda + cc);
                }
                for (int i = tid; i < rows * (BO / 8); i += kWgradThreads) {
                    const int rr = i / (BO / 8), cc = i % (BO / 8) * 8;
                    cp_async16(sz + rr * LO + cc, Z + (long long)(r + rr) * ldz + cc);
                }
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int st = 0; st < S - 1; ++st) load(st);
        for (int st = 0; st < nst; ++st) {
            asm volatile("cp.async.wait_group %0;\n" ::"n"(S - 2) : "memory");
            __syncthreads();   // stage st has landed, and every warp is done with stage st - 1
            load(st + S - 1);
            const __nv_bfloat16* sa = sm + st % S * STAGE;
            const __nv_bfloat16* sz = sa + KB * LI;
            const int ks = min(KB, r1 - r0 - st * KB) / 16;
            auto frags = [&](int k, uint32_t (&fa)[4], uint32_t (&fb)[2]) {
                ldsm4t(fa, sa + (k * 16 + (lane & 7) + (lane >> 4) * 8) * LI + wm * 16 + ((lane >> 3) & 1) * 8);
                ldsm2t(fb, sz + (k * 16 + (lane & 15)) * LO + wn * 8);
            };
            uint32_t fa[KB / 16][4], fb[KB / 16][2];
            if (ks == KB / 16) {   // a whole stage: every fragment load ahead of the chain of mma
#pragma unroll
                for (int k = 0; k < KB / 16; ++k) frags(k, fa[k], fb[k]);
#pragma unroll
                for (int k = 0; k < KB / 16; ++k) mma16816(c, fa[k], fb[k][0], fb[k][1]);
            } else {
                for (int k = 0; k < ks; ++k) {
                    frags(k, fa[0], fb[0]);
                    mma16816(c, fa[0], fb[0][0], fb[0][1]);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int m = wm * 16 + g + (e >> 1) * 8, o = wn * 8 + 2 * q + (e & 1);
            if (m < vi && o < vo) out[m * ldo + o] = c[e];
        }
    }
};

// Bias gradients of 32 columns j0 .. of the flat order (layer 3: columns
// 384 .. 386): the rows [r0, r1) stream through four shared stages of 64, and
// one thread per column adds them in order.
__device__ __forceinline__ void bias_sums(float* sm, const float* DZF, int j0, int r0, int r1, float* part) {
    constexpr int KB = 64, S = 4, NC = 32;
    const int tid = threadIdx.x, quads = min(NC, kDzf - j0) / 4, nst = (r1 - r0 + KB - 1) / KB;
    auto load = [&](int st) {
        if (st < nst) {
            const int r = r0 + st * KB, rows = min(KB, r1 - r);
            for (int i = tid; i < rows * 8; i += kWgradThreads)
                if ((i & 7) < quads)
                    cp_async16(sm + (st % S * KB + (i >> 3)) * NC + (i & 7) * 4,
                               DZF + (long long)(r + (i >> 3)) * kDzf + j0 + (i & 7) * 4);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    for (int st = 0; st < S - 1; ++st) load(st);
    float s = 0.0f;
    for (int st = 0; st < nst; ++st) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(S - 2) : "memory");
        __syncthreads();
        load(st + S - 1);
        if (tid < NC) {
            const float* z = sm + st % S * KB * NC + tid;
            const int rows = min(KB, r1 - r0 - st * KB);   // a multiple of 16
            for (int k = 0; k < rows; k += 16)
#pragma unroll
                for (int e = 0; e < 16; ++e) s += z[(k + e) * NC];
        }
    }
    const int j = j0 + tid;
    if (tid < NC && j < NBIAS) {
        const int l = j >> 7;
        part[(l == 0 ? BOFF(0) : (l == 1 ? BOFF(1) : (l == 2 ? BOFF(2) : BOFF(3)))) + j - 128 * l] = s;
    }
}

// blockIdx.x: 0-15 the 32 x 32 blocks of layer 1, 16-31 of layer 2, 32-33 the
// 16 x 64 blocks of layer 0, 34 layer 3, 35-47 the bias gradients and the
// loss; blockIdx.y: chunk of kChunkRows rows.  Within a chunk every sum runs
// over the rows in order (one accumulator), so the gradient of a batch of up
// to 512 rows does not depend on how it is split.  Bound by that chain (32
// steps of mma, 512 additions) and by the latency of the loads.  The three
// kernels of a gradient take 13.3 us at 512 rows and 22.3 at 4096; with one
// warp per 16 x 8 block and one thread per bias walking the whole batch in
// global memory they took 85 and 275.
constexpr int kWgradBlocks = 35 + (NBIAS + 31) / 32;
__global__ void __launch_bounds__(kWgradThreads) k_wgrad(Dev d, int n16) {
    using Big = WgradTile<2, 4, 4>;
    using L0 = WgradTile<1, 8, 3>;
    using L3 = WgradTile<8, 1, 2>;
    static_assert(Big::BI == 32 && Big::BO == 32 && L0::BO == 64 && L3::BI == 128, "block map below");
    static_assert(L3::ELEMS >= Big::ELEMS && L3::ELEMS >= L0::ELEMS, "shared stages");
    __shared__ __align__(16) __nv_bfloat16 sm[L3::ELEMS];
    pdl_launch();
    pdl_wait();
    const int b = blockIdx.x, r0 = blockIdx.y * kChunkRows, r1 = min(n16, r0 + kChunkRows);
    float* part = d.part + (long long)blockIdx.y * NPART;
    if (b < 32) {
        const int l = 1 + (b >> 4), m0 = ((b >> 2) & 3) * 32, o0 = (b & 3) * 32;
        Big::run(sm, d.A[l] + m0, 128, d.DZ[l] + o0, 128, r0, r1, part + WOFF(l) + m0 * 128 + o0, 128, 32, 32);
    } else if (b < 34) {
        const int o0 = (b - 32) * 64;
        L0::run(sm, d.A[0], 16, d.DZ[0] + o0, 128, r0, r1, part + WOFF(0) + o0, 128, 6, 64);
    } else if (b == 34) {
        L3::run(sm, d.A[3], 128, d.DZ[3], 8, r0, r1, part + WOFF(3), 3, 128, 3);
    } else {
        const int bb = b - 35;
        bias_sums(reinterpret_cast<float*>(sm), d.DZF, bb * 32, r0, r1, part);
        if (bb == 0 && threadIdx.x == 32) {   // a thread of another warp: the loss
            float s = 0.0f;
#pragma unroll 16
            for (int t = r0 / 16; t < r1 / 16; ++t) s += d.lpart[t];
            d.lchunk[blockIdx.y] = s;
        }
    }
}

// Sums the chunk partials in order; ADAM: updates the parameters and both
// packed copies, otherwise writes the gradient.
template <bool ADAM>
__global__ void __launch_bounds__(128) k_update(Dev d, int chunks, int n, float* __restrict__ grad,
                                                float* __restrict__ loss, float lr, float c1, float c2) {
    pdl_launch();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && loss) {
        float s = 0.0f;
        for (int c = 0; c < chunks; ++c) s += d.lchunk[c];
        *loss = s / (float)(n * 3);
    }
    if (i >= MLP_N_PARAMS) return;
    float gi = 0.0f;
#pragma unroll 8
    for (int c = 0; c < chunks; ++c) gi += d.part[(long long)c * NPART + i];
    if (!ADAM) {
        grad[i] = gi;
        return;
    }
    const float m = 0.9f * d.m[i] + 0.1f * gi;
    const float v = 0.999f * d.v[i] + 0.001f * gi * gi;
    d.m[i] = m;
    d.v[i] = v;
    const float th = d.theta[i] - lr * (m * c1) / (sqrtf(v * c2) + 1e-8f);
    d.theta[i] = th;
    int l, k, c;
    if (weight_of(i, l, k, c)) pack_weight(d, l, k, c, th);
}

// Refreshes the packed bfloat16 weights from the FP32 master copy (their
// padding is zero from creation on).
__global__ void k_pack(Dev d) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int l, k, c;
    if (i < MLP_N_PARAMS && weight_of(i, l, k, c)) pack_weight(d, l, k, c, d.theta[i]);
}

}  // namespace

struct mlp_s {
    Dev d;
    int max_batch = 0;
    int64_t steps = 0;
    cudaStream_t stream = nullptr;
    std::vector<void*> allocs;
    int sms = 1;   // streaming multiprocessors of the device
};

namespace {

int fail(cudaError_t e) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? MLP_ENOMEM : MLP_ECUDA;
}

template <typename T>
T* mal(mlp_t* h, size_t count) {
    void* p = nullptr;
    if (cudaMalloc(&p, count * sizeof(T) + 16) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    h->allocs.push_back(p);
    return static_cast<T*>(p);
}

// Launches `fn` so that its launch overlaps the end of the kernel before it on
// the stream (every kernel above waits for that kernel before it touches memory).
template <typename... P, typename... Q>
cudaError_t launch_pdl(void (*fn)(P...), dim3 grid, int threads, cudaStream_t s, Q... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

// Rows per CTA: 16 keeps the chain of layers shortest while each tile has an
// SM of its own; beyond that 32 (up to two tiles per SM) and 64 rows pass the
// weight registers on to more mma rows.  GB300, us with 16 / 32 / 64 rows per
// CTA: 2.9 / 4.2 / 6.4 at 1201 rows, 4.7 / 4.3 / 6.5 at 4096, 8.2 / 7.3 / 6.6
// at 8192, 47.8 / 42.9 / 37.8 at 65536.  Two CTAs per SM (64 registers) gave
// no more: 41.2 / 40.4 / 38.3 at 65536.
int forward_impl(mlp_t* h, const float* x, int n, float* y) {
    const int t16 = (n + 15) / 16;
    auto grid = [&](int mt) { return dim3(std::min((n + 16 * mt - 1) / (16 * mt), h->sms)); };
    cudaError_t e;
    if (t16 <= h->sms) e = launch_pdl(k_fwd<1>, grid(1), kThreads, h->stream, h->d, x, n, y);
    else if (t16 <= 2 * h->sms) e = launch_pdl(k_fwd<2>, grid(2), kThreads, h->stream, h->d, x, n, y);
    else e = launch_pdl(k_fwd<4>, grid(4), kThreads, h->stream, h->d, x, n, y);
    return e == cudaSuccess ? MLP_OK : fail(e);
}

// Forward, backward and the chunk partials of every gradient.
int grad_impl(mlp_t* h, const float* x, const float* t, int n, int* chunks, const long long* idx = nullptr,
              long long nrows = 0) {
    const int tiles = (n + 15) / 16, n16 = tiles * 16;
    *chunks = (n16 + kChunkRows - 1) / kChunkRows;
    // 16 rows per CTA while every tile has an SM of its own, then 32 (4096 rows: the
    // whole gradient 18.7 us against 24.5 with 16, measured with split sums)
    cudaError_t e = tiles <= h->sms
                        ? launch_pdl(k_train<1>, dim3(tiles), kThreads, h->stream, h->d, x, t, idx, nrows, n)
                        : launch_pdl(k_train<2>, dim3((tiles + 1) / 2), kThreads, h->stream, h->d, x, t, idx, nrows, n);
    if (e == cudaSuccess)
        e = launch_pdl(k_wgrad, dim3(kWgradBlocks, *chunks), kWgradThreads, h->stream, h->d, n16);
    return e == cudaSuccess ? MLP_OK : fail(e);
}

constexpr int kUpdateGrid = (MLP_N_PARAMS + 127) / 128;

// One training step on the first n rows, or on the rows idx[0 .. n).
int train_impl(mlp_t* h, const float* x, const float* t, int n, float lr, float* loss, const long long* idx = nullptr,
               long long nrows = 0) {
    int chunks = 0;
    const int rc = grad_impl(h, x, t, n, &chunks, idx, nrows);
    if (rc) return rc;
    h->steps += 1;
    const double c1 = 1.0 / (1.0 - std::pow(0.9, (double)h->steps));
    const double c2 = 1.0 / (1.0 - std::pow(0.999, (double)h->steps));
    const cudaError_t e = launch_pdl(k_update<true>, dim3(kUpdateGrid), 128, h->stream, h->d, chunks, n,
                                     (float*)nullptr, loss, lr, (float)c1, (float)c2);
    return e == cudaSuccess ? MLP_OK : fail(e);
}

}  // namespace

extern "C" {

int mlp_create(int max_batch, const float* params, void* stream, mlp_t** out) {
    if (!out || max_batch < 1 || max_batch > (1 << 24)) return MLP_EINVAL;
    *out = nullptr;
    mlp_t* h = new mlp_s();
    h->max_batch = max_batch;
    h->stream = static_cast<cudaStream_t>(stream);
    Dev& d = h->d;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();   // without a device the allocations below fail
        h->sms = 1;
    }
    const size_t rows = (size_t)(max_batch + 31) / 32 * 32;   // whole tiles of k_train
    const size_t chunks = (rows + kChunkRows - 1) / kChunkRows;
    bool ok = true;
    auto get = [&](auto*& p, size_t count) {
        p = mal<std::remove_reference_t<decltype(*p)>>(h, count);
        ok = ok && p;
    };
    get(d.theta, MLP_N_PARAMS);
    get(d.m, MLP_N_PARAMS);
    get(d.v, MLP_N_PARAMS);
    for (int l = 0; l < NL; ++l) {
        // both copies are padded to the mma tile: K to 16, N to 8 (transposed: the fan-out to 16)
        const size_t nf = (size_t)KP(l) * NP(l), nb = (size_t)KP(l) * std::max(16, NP(l));
        get(d.wf[l], nf);
        get(d.wb[l], nb);
        if (ok && (cudaMemset(d.wf[l], 0, nf * 2) != cudaSuccess || cudaMemset(d.wb[l], 0, nb * 2) != cudaSuccess)) {
            mlp_destroy(h);
            return MLP_ECUDA;
        }
        get(d.A[l], rows * KP(l));
        get(d.DZ[l], rows * NP(l));
    }
    get(d.DZF, rows * kDzf);
    get(d.lpart, rows / 16);
    get(d.part, chunks * NPART);
    get(d.lchunk, chunks);
    if (!ok) {
        mlp_destroy(h);
        return MLP_ENOMEM;
    }
    std::vector<float> init(MLP_N_PARAMS, 0.0f);
    if (params) memcpy(init.data(), params, sizeof(float) * MLP_N_PARAMS);
    int rc = mlp_set_params(h, init.data());
    if (rc) {
        mlp_destroy(h);
        return rc;
    }
    *out = h;
    return MLP_OK;
}

int mlp_set_params(mlp_t* h, const float* params) {
    if (!h || !params) return MLP_EINVAL;
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e == cudaSuccess) e = cudaMemcpy(h->d.theta, params, sizeof(float) * MLP_N_PARAMS, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(h->d.m, 0, sizeof(float) * MLP_N_PARAMS);
    if (e == cudaSuccess) e = cudaMemset(h->d.v, 0, sizeof(float) * MLP_N_PARAMS);
    if (e != cudaSuccess) return fail(e);
    k_pack<<<kUpdateGrid, 128, 0, h->stream>>>(h->d);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return fail(e);
    h->steps = 0;
    return MLP_OK;
}

int mlp_get_params(mlp_t* h, float* params) {
    if (!h || !params) return MLP_EINVAL;
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e == cudaSuccess) e = cudaMemcpy(params, h->d.theta, sizeof(float) * MLP_N_PARAMS, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? MLP_OK : fail(e);
}

int mlp_forward(mlp_t* h, const float* x, int n, float* y) {
    if (!h || !x || !y || n < 1 || n > h->max_batch) return MLP_EINVAL;
    return forward_impl(h, x, n, y);
}

int mlp_gradients(mlp_t* h, const float* x, const float* t, int n, float* grad, float* loss) {
    if (!h || !x || !t || !grad || n < 1 || n > h->max_batch) return MLP_EINVAL;
    int chunks = 0;
    int rc = grad_impl(h, x, t, n, &chunks);
    if (rc) return rc;
    cudaError_t e = launch_pdl(k_update<false>, dim3(kUpdateGrid), 128, h->stream, h->d, chunks, n, grad, loss, 0.0f,
                               0.0f, 0.0f);
    return e == cudaSuccess ? MLP_OK : fail(e);
}

int mlp_train_step(mlp_t* h, const float* x, const float* t, int n, float lr, float* loss) {
    if (!h || !x || !t || n < 1 || n > h->max_batch || !std::isfinite(lr)) return MLP_EINVAL;
    return train_impl(h, x, t, n, lr, loss);
}

int mlp_train_steps(mlp_t* h, const float* x, const float* t, int64_t rows, const int64_t* idx, int n, int steps,
                    float lr, float* loss) {
    if (!h || !x || !t || !idx || rows < 1 || n < 1 || n > h->max_batch || steps < 0 || !std::isfinite(lr))
        return MLP_EINVAL;
    for (int s = 0; s < steps; ++s) {
        const int rc = train_impl(h, x, t, n, lr, loss ? loss + s : nullptr,
                                  reinterpret_cast<const long long*>(idx) + (size_t)s * n, rows);
        if (rc) return rc;
    }
    return MLP_OK;
}

int64_t mlp_step_count(const mlp_t* h) { return h ? h->steps : -1; }

void mlp_destroy(mlp_t* h) {
    if (!h) return;
    cudaStreamSynchronize(h->stream);
    for (void* p : h->allocs)
        if (p) cudaFree(p);
    cudaGetLastError();
    delete h;
}

}  // extern "C"
