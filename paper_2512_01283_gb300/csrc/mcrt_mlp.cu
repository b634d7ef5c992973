// mcrt_mlp.cu -- learned surrogate of the grain optics (the paper's Sec. 2.2 allows
// the Mueller matrix to come from analytic forms, tables or neural networks; Sec. 4
// motivates networks for multi-dimensional grain optics).
//
// The network maps (n_i, n_s, s) -- incident and scattered directions in the grain
// frame and the position s in [-1, 1] of ln x between the first and last tabulated
// size parameter -- to 20 numbers: ln M11 of the 4x4 scattering matrix in the
// scattering-plane basis and its other 15 entries relative to M11 (the rotations into
// and out of the plane stay exact geometry in the kernels that use the network), the
// extinction elements alpha1..3 at the incident polar angle, and ln N(s), N(s) = max
// P11.  Architecture 16 (7 inputs, zero padded) -> 128 -> 128 ->
// 128 -> 128 -> 24 (20 used), SiLU; BF16 weights and activations, FP32 accumulation on
// the tensor cores (mma.sync m16n8k16), FP32 master weights and Adam.
//
// Training labels are generated on the GPU from the method's own tables, a fresh
// Philox-drawn batch every step.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "mcrt.h"
#include "mcrt_device.cuh"
#include "mcrt_internal.h"
#include "mcrt_mlp_infer.cuh"
#include "mcrt_mlp_tc.cuh"

namespace mcrt {
namespace {

typedef __nv_bfloat16 bf16;

using mlp::kHid;
using mlp::kIn;
using mlp::kInPad;
using mlp::kLayers;
using mlp::kOut;
using mlp::kOutPad;
__host__ __device__ constexpr int layer_in(int l) { return l == 0 ? kInPad : kHid; }
__host__ __device__ constexpr int layer_out(int l) { return l == kLayers - 1 ? kOutPad : kHid; }
// parameter layout: per layer W [out][in] then b [out], layers in order
__host__ __device__ constexpr int layer_offset(int l) {
    int off = 0;
    for (int i = 0; i < l; ++i) off += layer_out(i) * layer_in(i) + layer_out(i);
    return off;
}
constexpr int kParams = layer_offset(kLayers);
__host__ __device__ constexpr int wbf_offset(int l) {
    int off = 0;
    for (int i = 0; i < l; ++i) off += layer_out(i) * layer_in(i);
    return off;
}
constexpr int kWeights = wbf_offset(kLayers);

// ---------------------------------------------------------------------------------
// training labels from the tables
// ---------------------------------------------------------------------------------
struct LabelTables {
    const float4* bins;  // [n_bins][n_theta][2] (P11,P12,P22,P33),(P34,P44,0,0)
    const float4* kext;  // [n_ktheta]
    int n_bins, n_theta, n_ktheta;
};

__device__ void interp_row(const LabelTables& T, int k, int j, float f, float w, float P[6]) {
    const float4 a0 = T.bins[((size_t)k * T.n_theta + j) * 2], a1 = T.bins[((size_t)k * T.n_theta + j) * 2 + 1];
    const float4 b0 = T.bins[((size_t)k * T.n_theta + j + 1) * 2], b1 = T.bins[((size_t)k * T.n_theta + j + 1) * 2 + 1];
    const float g = 1.f - f;
    P[0] += w * (g * a0.x + f * b0.x);
    P[1] += w * (g * a0.y + f * b0.y);
    P[2] += w * (g * a0.z + f * b0.z);
    P[3] += w * (g * a0.w + f * b0.w);
    P[4] += w * (g * a1.x + f * b1.x);
    P[5] += w * (g * a1.y + f * b1.y);
}

// 20 targets for (n_i, n_s, s): tables interpolated linearly in the scattering angle
// and in ln x between bins; the scattering-plane matrix M as ln M11 and M_rc / M11;
// alpha1..3; ln of the maximum interpolated P11.
__device__ void surrogate_label(const LabelTables& T, const V3<float>& ni, const V3<float>& ns, float s,
                                float out[kOut]) {
    // bins k and k1 = k + 1 around s (one bin: k = k1 = 0)
    int k = 0, k1 = 0;
    float fb = 0.f;
    if (T.n_bins > 1) {
        const float b = (fminf(fmaxf(s, -1.f), 1.f) + 1.f) * 0.5f * (float)(T.n_bins - 1);
        k = (int)floorf(b);
        k = k > T.n_bins - 2 ? T.n_bins - 2 : (k < 0 ? 0 : k);
        k1 = k + 1;
        fb = b - (float)k;
    }
    float N = 0.f;
    for (int j = 0; j < T.n_theta; ++j) {
        const float v = (1.f - fb) * T.bins[((size_t)k * T.n_theta + j) * 2].x +
                        fb * T.bins[((size_t)k1 * T.n_theta + j) * 2].x;
        N = fmaxf(N, v);
    }
    const float mu = fminf(fmaxf(dot<kFree>(ni, ns), -1.f), 1.f);
    const float x = acosf(mu) * 0.31830988618379067f * (float)(T.n_theta - 1);
    int j = (int)floorf(x);
    j = j > T.n_theta - 2 ? T.n_theta - 2 : (j < 0 ? 0 : j);
    const float ft = x - (float)j;
    float P[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    interp_row(T, k, j, ft, 1.f - fb, P);
    interp_row(T, k1, j, ft, fb, P);
    // scattering-plane matrix [[P11,P12,0,0],[P12,P22,0,0],[0,0,P33,P34],[0,0,-P34,P44]]
    // as ln M11 and the entries relative to M11 (equal relative accuracy over the
    // decades that P11 spans)
    const float inv = 1.f / P[0];
    const float Z[16] = {P[0], P[1], 0.f, 0.f, P[1], P[2], 0.f, 0.f, 0.f, 0.f, P[3], P[4], 0.f, 0.f, -P[4], P[5]};
    out[0] = logf(P[0]);
    for (int k = 1; k < 16; ++k) out[k] = Z[k] * inv;
    const float xk = acosf(fminf(fmaxf(ni.z, -1.f), 1.f)) * 0.31830988618379067f * (float)(T.n_ktheta - 1);
    int jk = (int)floorf(xk);
    jk = jk > T.n_ktheta - 2 ? T.n_ktheta - 2 : (jk < 0 ? 0 : jk);
    const float fk = xk - (float)jk;
    const float4 ka = T.kext[jk], kb = T.kext[jk + 1];
    out[16] = (1.f - fk) * ka.x + fk * kb.x;
    out[17] = (1.f - fk) * ka.y + fk * kb.y;
    out[18] = (1.f - fk) * ka.z + fk * kb.z;
    out[19] = logf(N);
}

__device__ V3<float> iso_unit(float ua, float ub) {
    const float ct = 2.f * ua - 1.f;
    float st = (1.f - ct) * (1.f + ct);
    st = st > 0.f ? sqrtf(st) : 0.f;
    float sp, cp;
    sincospif(2.f * ub, &sp, &cp);
    return V3<float>{st * cp, st * sp, ct};
}

// Training batch of step step0 + *iter: inputs and targets.
__global__ void k_gen_batch(LabelTables T, unsigned seed, unsigned step0, const unsigned* __restrict__ iter, int B,
                            float* __restrict__ X, float* __restrict__ Y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B) return;
    const unsigned step = step0 + *iter;
    const Draw4<float> u0 = draw4<float>(i, step, 0x51u, seed, 0x5A17u);
    const Draw4<float> u1 = draw4<float>(i, step, 0x52u, seed, 0x5A17u);
    const V3<float> ni = iso_unit(u0.a, u0.b), ns = iso_unit(u0.c, u0.d);
    const float s = 2.f * u1.a - 1.f;
    const float in[kIn] = {ni.x, ni.y, ni.z, ns.x, ns.y, ns.z, s};
    for (int c = 0; c < kIn; ++c) X[(size_t)i * kIn + c] = in[c];
    float out[kOut];
    surrogate_label(T, ni, ns, s, out);
    for (int c = 0; c < kOut; ++c) Y[(size_t)i * kOut + c] = out[c];
}

// Labels of given inputs [n][7] (diagnostics and the error map).
__global__ void k_labels(LabelTables T, int n, const float* __restrict__ in, float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float* u = in + (size_t)i * kIn;
    float o[kOut];
    surrogate_label(T, V3<float>{u[0], u[1], u[2]}, V3<float>{u[3], u[4], u[5]}, u[6], o);
    for (int c = 0; c < kOut; ++c) out[(size_t)i * kOut + c] = o[c];
}

// ---------------------------------------------------------------------------------
// Forward pass, loss and backward pass of a batch in one kernel.  BF16 operands, FP32
// accumulation (mma.sync m16n8k16); activations, the output gradient and every hidden layer's
// gradient are rounded to BF16, pre-activations stay in FP32.
//
// A block takes tiles of 16 MT rows through all layers: weights (119 kB) and activations in
// shared memory, the pre-activations in the registers of the warp that owns their 16 columns,
// which also owns them on the way back.  A layer's gradient overwrites its activations.  The
// weight gradients of a tile are added with FP32 reductions of two columns to one of n_parts
// partial gradients, which the blocks share by index; folded() sums these in FP64.
//
// What bounds it: at a tile per SM the chain of ten small products (22 us for 2048 rows), at many
// tiles the shared-memory reads of the operands (216 us for 65536 rows).  A gradient call, host
// arrays to host arrays, against one launch per product and epilogue with every operand through
// memory (25 dependent launches): 2048 rows 82 us (395), 8192 102 us (545), 2^20 3.9 ms (54.1);
// a training step of 1024 rows 45 us (278), of 8192 66 us (436).
// ---------------------------------------------------------------------------------
__device__ __forceinline__ float silu_f(float z) { return mlp::silu(z); }
__device__ __forceinline__ float silu_grad_f(float z) { return mlp::silu_grad(z); }

constexpr int kPassThreads = 256, kPassWarps = kPassThreads / 32;
constexpr int kLdX = mlp::kLd0, kLdH = mlp::kLdH, kLdY = 40;  // row strides (elements), free of bank conflicts
constexpr int kOutMma = 32;                                  // output columns as a K of the products
// weights in shared memory: element offset and row stride of layer l (layer 4 has 32 rows, 8 of zeros)
__host__ __device__ constexpr int pass_w(int l) { return l == 0 ? 0 : kHid * kLdX + (l - 1) * kHid * kLdH; }
__host__ __device__ constexpr int pass_ld(int l) { return l == 0 ? kLdX : kLdH; }
constexpr int kPassW = pass_w(kLayers - 1) + kOutMma * kLdH;
constexpr size_t pass_smem(int mt) {
    return sizeof(bf16) * (size_t)(kPassW + 16 * mt * (kLdX + 4 * kLdH + kLdY)) + kPassWarps * sizeof(double);
}
static_assert(kHid == 16 * kPassWarps, "a warp owns 16 columns of a hidden layer");

struct LossWeights {
    float w[kOut];
};

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(unsigned a, unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(a)
                 : "memory");
}

template <int MT>
__global__ void __launch_bounds__(kPassThreads, 1)
    k_pass(int B, const float* __restrict__ in, const float* __restrict__ target, const LossWeights lw,
           const bf16* __restrict__ wbf, const float* __restrict__ params, float* __restrict__ parts, int n_parts,
           double* __restrict__ loss, const unsigned* __restrict__ iter) {
    constexpr int R = 16 * MT;
    extern __shared__ __align__(16) unsigned char pass_sm[];
    bf16* const ws = reinterpret_cast<bf16*>(pass_sm);
    bf16* const xs = ws + kPassW;
    bf16* const hs = xs + R * kLdX;
    bf16* const ys = hs + 4 * R * kLdH;
    double* const part = reinterpret_cast<double*>(ys + R * kLdY);
    float* const grads = parts + (size_t)((int)blockIdx.x % n_parts) * kParams;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gr = lane >> 2, tc = lane & 3;
    // ldmatrix rows and columns of this lane.  A operand with k contiguous, or its transpose from
    // rows of k; B operand with k contiguous (16 columns), or from rows of k
    const int a_row = lane & 15, a_col = (lane >> 4) * 8;
    const int at_row = (lane & 7) + (lane >> 4) * 8, at_col = ((lane >> 3) & 1) * 8;
    const int b_row = (lane & 7) + (lane >> 4) * 8, b_col = ((lane >> 3) & 1) * 8;
    const int bt_row = (lane & 7) + ((lane >> 3) & 1) * 8, bt_col = (lane >> 4) * 8;
    const unsigned ws_a = mlp::smem_addr(ws), xs_a = mlp::smem_addr(xs), hs_a = mlp::smem_addr(hs),
                   ys_a = mlp::smem_addr(ys);
    // weights: one group of copies per layer, waited for when the layer is reached
#pragma unroll
    for (int l = 0; l < kLayers; ++l) {
        const int per_row = layer_in(l) / 8, n = layer_out(l) * per_row;
        for (int i = tid; i < n; i += kPassThreads)
            cp_async16(ws_a + (unsigned)(pass_w(l) + i / per_row * pass_ld(l) + i % per_row * 8) * 2,
                       wbf + wbf_offset(l) + i * 8);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const bf16 zero = __float2bfloat16(0.f);
    for (int i = tid; i < (kOutMma - kOutPad) * kLdH; i += kPassThreads)
        ws[pass_w(kLayers - 1) + kOutPad * kLdH + i] = zero;
    for (int i = tid; i < R * kLdY; i += kPassThreads) ys[i] = zero;
    const float scale = 2.f / ((float)B * (float)kOut);
    double lsum = 0.0;
    const int n_tiles = (B + R - 1) / R;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int row0 = tile * R;
        __syncthreads();  // the tile before is done with the input rows
        for (int i = tid; i < R; i += kPassThreads) {
            float u[kIn];
            for (int c = 0; c < kIn; ++c) u[c] = row0 + i < B ? in[(size_t)(row0 + i) * kIn + c] : 0.f;
            mlp::store_input_row(xs + i * kLdX, u);
        }
        // ---- forward: z = h W^T + b, h = SiLU(z)
        float z[4][MT][2][4];
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            if (l == 0) cp_async_wait<4>();
            if (l == 1) cp_async_wait<3>();
            if (l == 2) cp_async_wait<2>();
            if (l == 3) cp_async_wait<1>();
            __syncthreads();
            float acc[MT][2][4] = {};
            const unsigned src = l == 0 ? xs_a : hs_a + (unsigned)((l - 1) * R * kLdH * 2);
            const int ld = l == 0 ? kLdX : kLdH;
#pragma unroll
            for (int ks = 0; ks < layer_in(l); ks += 16) {
                unsigned b[4];
                mlp::ldsm_x4_fenced(ws_a + (unsigned)(pass_w(l) + (warp * 16 + b_row) * pass_ld(l) + ks + b_col) * 2, b[0],
                                    b[1], b[2], b[3]);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    unsigned a[4];
                    mlp::ldsm_x4_fenced(src + (unsigned)((mt * 16 + a_row) * ld + ks + a_col) * 2, a[0], a[1], a[2], a[3]);
                    mlp::mma16816(acc[mt][0], a, b[0], b[1]);
                    mlp::mma16816(acc[mt][1], a, b[2], b[3]);
                }
            }
            const float* const bias = params + layer_offset(l) + kHid * layer_in(l);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                const int n = warp * 16 + nt * 8 + tc * 2;
                const float b0 = __ldg(bias + n), b1 = __ldg(bias + n + 1);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float z0 = acc[mt][nt][h * 2] + b0, z1 = acc[mt][nt][h * 2 + 1] + b1;
                        z[l][mt][nt][h * 2] = z0;
                        z[l][mt][nt][h * 2 + 1] = z1;
                        *reinterpret_cast<unsigned*>(hs + (l * R + mt * 16 + gr + h * 8) * kLdH + n) =
                            mlp::pack_bf16(silu_f(z0), silu_f(z1));
                    }
            }
        }
        cp_async_wait<0>();
        __syncthreads();
        // ---- output, loss and dY = 2 w (Y - T) / (B * 20): one 16 x 8 tile per warp
        if (warp < 3 * MT) {
            const int mt = warp / 3, nt = warp % 3;
            float acc[4] = {};
#pragma unroll
            for (int ks = 0; ks < kHid; ks += 16) {
                unsigned a[4], b0, b1;
                mlp::ldsm_x4_fenced(hs_a + (unsigned)((3 * R + mt * 16 + a_row) * kLdH + ks + a_col) * 2, a[0], a[1], a[2],
                                    a[3]);
                mlp::ldsm_x2(ws_a + (unsigned)(pass_w(4) + (nt * 8 + (lane & 7)) * kLdH + ks + b_col) * 2, b0, b1);
                mlp::mma16816(acc, a, b0, b1);
            }
            const float* const bias = params + layer_offset(4) + kOutPad * kHid;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = mt * 16 + gr + h * 8, o = nt * 8 + tc * 2;
                float d[2] = {0.f, 0.f};
                if (row0 + r < B && o < kOut) {
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float y = acc[h * 2 + e] + __ldg(bias + o + e);
                        const float res = y - target[(size_t)(row0 + r) * kOut + o + e];
                        lsum += (double)(lw.w[o + e] * res * res);
                        d[e] = scale * lw.w[o + e] * res;
                    }
                }
                *reinterpret_cast<unsigned*>(ys + r * kLdY + o) = mlp::pack_bf16(d[0], d[1]);
            }
        }
        __syncthreads();
        // ---- backward
#pragma unroll
        for (int l = kLayers - 1; l >= 0; --l) {
            constexpr int kLast = kLayers - 1;
            const int no = layer_out(l), ni = layer_in(l);
            const bf16* const dz = l == kLast ? ys : hs + l * R * kLdH;
            const unsigned dz_a = l == kLast ? ys_a : hs_a + (unsigned)(l * R * kLdH * 2);
            const int dz_ld = l == kLast ? kLdY : kLdH;
            const unsigned in_a = l == 0 ? xs_a : hs_a + (unsigned)((l - 1) * R * kLdH * 2);
            const int in_ld = l == 0 ? kLdX : kLdH;
            float* const gW = grads + layer_offset(l);
            // dW = dZ^T H: 16 x 16 tiles, a row of them per warp (layer 4: a column of two)
            const int tiles = l == kLast ? 2 : ni / 16;
            for (int t = 0; t < tiles; ++t) {
                const int m0 = (l == kLast ? t : warp) * 16, n0 = (l == kLast ? warp : t) * 16;
                float acc[2][4] = {};
#pragma unroll
                for (int ks = 0; ks < R; ks += 16) {
                    unsigned a[4], b[4];
                    ldsm_x4_t(dz_a + (unsigned)((ks + at_row) * dz_ld + m0 + at_col) * 2, a[0], a[1], a[2], a[3]);
                    ldsm_x4_t(in_a + (unsigned)((ks + bt_row) * in_ld + n0 + bt_col) * 2, b[0], b[1], b[2], b[3]);
                    mlp::mma16816(acc[0], a, b[0], b[1]);
                    mlp::mma16816(acc[1], a, b[2], b[3]);
                }
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int m = m0 + gr + h * 8, n = n0 + nt * 8 + tc * 2;
                        if (l == 0) {
                            // a master weight feeds the column of the high parts and that of the low parts
                            for (int e = 0; e < 2; ++e)
                                if (n + e < 2 * kIn)
                                    atomicAdd(gW + m * kInPad + (n + e < kIn ? n + e : n + e - kIn), acc[nt][h * 2 + e]);
                        } else if (m < no) {
                            atomicAdd(reinterpret_cast<float2*>(gW + m * ni + n),
                                      make_float2(acc[nt][h * 2], acc[nt][h * 2 + 1]));
                        }
                    }
            }
            // db = column sums of dZ
            if (tid < no) {
                float sum = 0.f;
#pragma unroll 8
                for (int r = 0; r < R; ++r) sum += __bfloat162float(dz[r * dz_ld + tid]);
                atomicAdd(gW + no * ni + tid, sum);
            }
            if (l == 0) break;
            // dZ of the layer below = (dZ W) SiLU'(z)
            float acc[MT][2][4] = {};
#pragma unroll
            for (int ks = 0; ks < (l == kLast ? kOutMma : kHid); ks += 16) {
                unsigned b[4];
                ldsm_x4_t(ws_a + (unsigned)(pass_w(l) + (ks + bt_row) * kLdH + warp * 16 + bt_col) * 2, b[0], b[1], b[2],
                          b[3]);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    unsigned a[4];
                    mlp::ldsm_x4_fenced(dz_a + (unsigned)((mt * 16 + a_row) * dz_ld + ks + a_col) * 2, a[0], a[1], a[2],
                                        a[3]);
                    mlp::mma16816(acc[mt][0], a, b[0], b[1]);
                    mlp::mma16816(acc[mt][1], a, b[2], b[3]);
                }
            }
            __syncthreads();  // the activations of the layer below have been read
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int r = mt * 16 + gr + h * 8, n = warp * 16 + nt * 8 + tc * 2;
                        const bool live = row0 + r < B;
                        const float d0 = acc[mt][nt][h * 2] * silu_grad_f(z[l - 1][mt][nt][h * 2]);
                        const float d1 = acc[mt][nt][h * 2 + 1] * silu_grad_f(z[l - 1][mt][nt][h * 2 + 1]);
                        *reinterpret_cast<unsigned*>(hs + ((l - 1) * R + r) * kLdH + n) =
                            live ? mlp::pack_bf16(d0, d1) : 0u;
                    }
            __syncthreads();
        }
    }
    for (int off = 16; off > 0; off >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, off);
    if (lane == 0) part[warp] = lsum;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kPassWarps; ++w) lsum += part[w];
        atomicAdd(loss + (iter ? *iter : 0u), lsum / ((double)B * kOut));
    }
}

// Gradient of parameter i from the partial ones.
__device__ __forceinline__ float folded(const float* __restrict__ parts, int n_parts, int i) {
    double sum = 0.0;
#pragma unroll 4
    for (int k = 0; k < n_parts; ++k) sum += parts[(size_t)k * kParams + i];
    return (float)sum;
}

__global__ void k_fold(const float* __restrict__ parts, int n_parts, float* __restrict__ grads) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kParams) grads[i] = folded(parts, n_parts, i);
}

// ---------------------------------------------------------------------------------
// FP32 mode of the training passes, for gradient checks at FP32 accuracy: the same
// layers and fused epilogues with FP32 operands and activations on the FP32 pipe (no
// BF16 rounding anywhere), C[m][n] = sum_k A(m,k) B(k,n),
//   A(m,k) = a_t ? A[k*lda + m] : A[m*lda + k],  B(k,n) = b_kn ? B[k*ldb + n] : B[n*ldb + k].
// Block tile 64x64x16, 256 threads of 4x4 outputs each.
// ---------------------------------------------------------------------------------
enum { EPI_HIDDEN = 0, EPI_OUT = 1, EPI_DX = 2, EPI_DW = 3 };

struct GemmArgs32 {
    int M, N, K;
    const float* A;
    int lda, a_t;
    const float* B;
    int ldb, b_kn;
    const float* bias;
    float* Zout;
    int ldz;
    float* Hout;
    int ldh;
    const float* Zprev;
};

constexpr int kT32 = 64, kK32 = 16;

template <int EPI> __global__ void __launch_bounds__(256) k_gemm32(const GemmArgs32 g) {
    __shared__ float As[kK32][kT32 + 4];  // [k][m]
    __shared__ float Bs[kK32][kT32 + 4];  // [k][n]
    const int m0 = blockIdx.y * kT32, n0 = blockIdx.x * kT32;
    const int tid = threadIdx.x, tm = (tid / 16) * 4, tn = (tid % 16) * 4;
    float acc[4][4];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    int kb = 0, ke = g.K;
    if (EPI == EPI_DW && gridDim.z > 1) {
        const int per = ((g.K + gridDim.z - 1) / gridDim.z + kK32 - 1) / kK32 * kK32;
        kb = blockIdx.z * per;
        ke = kb + per < g.K ? kb + per : g.K;
    }
    for (int k0 = kb; k0 < ke; k0 += kK32) {
        for (int i = tid; i < kT32 * kK32; i += blockDim.x) {
            const int r = i / kK32, kk = i % kK32, k = k0 + kk;
            const int m = m0 + r, n = n0 + r;
            float a = 0.f, b = 0.f;
            if (m < g.M && k < ke) a = g.a_t ? g.A[(size_t)k * g.lda + m] : g.A[(size_t)m * g.lda + k];
            if (n < g.N && k < ke) b = g.b_kn ? g.B[(size_t)k * g.ldb + n] : g.B[(size_t)n * g.ldb + k];
            As[kk][r] = a;
            Bs[kk][r] = b;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kK32; ++kk) {
            float a[4], b[4];
            for (int i = 0; i < 4; ++i) a[i] = As[kk][tm + i];
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tn + j];
            for (int i = 0; i < 4; ++i)
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) {
            const int m = m0 + tm + i, n = n0 + tn + j;
            if (m >= g.M || n >= g.N) continue;
            const float v = acc[i][j];
            if (EPI == EPI_HIDDEN) {
                const float z = v + g.bias[n];
                g.Zout[(size_t)m * g.ldz + n] = z;
                g.Hout[(size_t)m * g.ldh + n] = silu_f(z);
            } else if (EPI == EPI_OUT) {
                g.Zout[(size_t)m * g.ldz + n] = v + g.bias[n];
            } else if (EPI == EPI_DX) {
                g.Hout[(size_t)m * g.ldh + n] = v * silu_grad_f(g.Zprev[(size_t)m * g.ldz + n]);
            } else {
                if (gridDim.z > 1)
                    atomicAdd(&g.Zout[(size_t)m * g.ldz + n], v);
                else
                    g.Zout[(size_t)m * g.ldz + n] = v;
            }
        }
}

template <int EPI> cudaError_t gemm32(const GemmArgs32& g, cudaStream_t s) {
    (void)cudaGetLastError();
    dim3 grid((g.N + kT32 - 1) / kT32, (g.M + kT32 - 1) / kT32);
    if (EPI == EPI_DW) {
        int z = 256 / (int)(grid.x * grid.y);
        const int kmax = (g.K + 4 * kK32 - 1) / (4 * kK32);
        z = z < kmax ? z : kmax;
        grid.z = z > 1 ? z : 1;
    }
    k_gemm32<EPI><<<grid, 256, 0, s>>>(g);
    return cudaGetLastError();
}

// FP32 inputs [n][7] as the first 7 of 16 columns (the rest zero): in FP32 the input
// needs no high and low parts.
__global__ void k_pack_inputs32(int n, const float* __restrict__ in, float* __restrict__ X) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int c = 0; c < kInPad; ++c) X[(size_t)i * kInPad + c] = c < kIn ? in[(size_t)i * kIn + c] : 0.f;
}

// dY = 2 w (Y - T) / (B * 20) in FP32 and the loss sum.
__global__ void k_loss_grad32(int B, const float* __restrict__ Y, const float* __restrict__ T,
                              const float* __restrict__ w, float* __restrict__ dY, double* __restrict__ loss) {
    __shared__ double part[256];
    double acc = 0.0;
    const float scale = 2.f / ((float)B * (float)kOut);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B * kOutPad; i += gridDim.x * blockDim.x) {
        const int b = i / kOutPad, o = i % kOutPad;
        float d = 0.f;
        if (o < kOut) {
            const float r = Y[(size_t)b * kOutPad + o] - T[(size_t)b * kOut + o];
            acc += (double)(w[o] * r * r);
            d = scale * w[o] * r;
        }
        dY[i] = d;
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) part[threadIdx.x] += part[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, part[0] / ((double)B * kOut));
}

// db[n] = sum over rows of dZ[b][n] (FP32 input).
__global__ void k_colsum32(int B, int N, const float* __restrict__ dZ, float* __restrict__ db) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    float s = 0.f;
    for (int b = blockIdx.y; b < B; b += gridDim.y) s += dZ[(size_t)b * N + n];
    atomicAdd(&db[n], s);
}

// Adam on the FP32 master parameters, from k_pass's partial gradients; the learning rate and the
// two bias corrections of the iteration are sched[3 * *iter + 0..2].
__global__ void k_adam(int P, float* __restrict__ p, const float* __restrict__ parts, int n_parts,
                       float* __restrict__ m, float* __restrict__ v, const float* __restrict__ sched,
                       const unsigned* __restrict__ iter, float b1, float b2, float eps) {
    const float* sc = sched + 3 * (size_t)*iter;
    const float lr = sc[0], c1 = sc[1], c2 = sc[2];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
        const float g = folded(parts, n_parts, i);
        const float mi = b1 * m[i] + (1.f - b1) * g;
        const float vi = b2 * v[i] + (1.f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// BF16 copies of the weights for the training GEMMs.  Layer 0 columns 7-13 repeat
// columns 0-6 (they multiply the low parts of the split inputs).  As the last kernel
// of a training step it also advances the step's iteration counter (iter_inc).
__global__ void k_pack_weights(const float* __restrict__ p, bf16* __restrict__ wbf, unsigned* __restrict__ iter_inc) {
    if (iter_inc && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(iter_inc, 1u);
    for (int l = 0; l < kLayers; ++l) {
        const int n = layer_out(l) * layer_in(l);
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
            int src = i;
            float v;
            if (l == 0) {
                const int o = i / kInPad, c = i % kInPad;
                src = o * kInPad + (c < kIn ? c : c - kIn);
                v = c < 2 * kIn ? p[layer_offset(0) + src] : 0.f;
            } else {
                v = p[layer_offset(l) + src];
            }
            wbf[wbf_offset(l) + i] = __float2bfloat16(v);
        }
    }
}

// Inference image (layout in mcrt_mlp_infer.cuh) from the FP32 parameters.
__global__ void k_pack_image(const float* __restrict__ p, unsigned char* __restrict__ img) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (int l = 0; l < kLayers; ++l) {
        const int ld = l == 0 ? mlp::kLd0 : mlp::kLdH;
        bf16* w = reinterpret_cast<bf16*>(img + mlp::img_w(l));
        const int rows = layer_out(l), n = rows * ld;
        for (int i = tid; i < n; i += nth) {
            const int o = i / ld, c = i % ld;
            float v = 0.f;
            if (l == 0) {
                if (c < 2 * kIn) v = p[layer_offset(0) + o * kInPad + (c < kIn ? c : c - kIn)];
            } else if (c < layer_in(l)) {
                v = p[layer_offset(l) + o * layer_in(l) + c];
            }
            w[i] = __float2bfloat16(v);
        }
        float* b = reinterpret_cast<float*>(img + mlp::kImgBias) + mlp::bias_off(l);
        for (int i = tid; i < rows; i += nth) b[i] = p[layer_offset(l) + rows * layer_in(l) + i];
    }
}

// Weights N(0, 1/fan_in) (Box-Muller on Philox draws), biases zero.
__global__ void k_init_params(float* __restrict__ p, unsigned seed) {
    for (int l = 0; l < kLayers; ++l) {
        const int nw = layer_out(l) * layer_in(l), nb = layer_out(l);
        const float sd = rsqrtf((float)(l == 0 ? kIn : layer_in(l)));
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nw + nb; i += gridDim.x * blockDim.x) {
            float v = 0.f;
            if (i < nw) {
                const int col = i % layer_in(l);
                if (l == 0 && col >= kIn) {
                    v = 0.f;
                } else {
                    const Draw4<float> u = draw4<float>(i, (unsigned)l, 0x1A17u, seed, 0x5A17u);
                    v = sd * sqrtf(-2.f * logf(u.a)) * cospif(2.f * u.b);
                }
            }
            p[layer_offset(l) + i] = v;
        }
    }
}

// Inference image for the tcgen05 engine (mcrt_mlp_tc.cuh layout) from the FP32
// parameters: weights in 8x16-byte core matrices, layer 0 columns 7-13 repeating
// columns 0-6, output rows 24-31 zero; biases, output ones padded with zeros.  The
// hidden layers hold W / 2 and b / 2 (exact), so their epilogue gets z / 2 directly.
__global__ void k_pack_image_tc(const float* __restrict__ p, unsigned char* __restrict__ img) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    for (int l = 0; l < kLayers; ++l) {
        const int K = l == 0 ? 16 : 128, N = l == kLayers - 1 ? tc::kN4 : 128;
        __nv_bfloat16* w = reinterpret_cast<__nv_bfloat16*>(img + tc::w_off(l));
        for (int i = tid; i < N * K; i += nth) {
            const int r = i / K, k = i % K;
            float v = 0.f;
            if (l == 0) {
                if (k < 2 * kIn) v = p[layer_offset(0) + r * kInPad + (k < kIn ? k : k - kIn)];
            } else if (r < layer_out(l)) {
                v = p[layer_offset(l) + r * layer_in(l) + k];
            }
            const float half = l < kLayers - 1 ? 0.5f : 1.f;
            w[tc::core_off(r, k, K) / 2] = __float2bfloat16(v * half);
        }
        float* b = reinterpret_cast<float*>(img + tc::kBias) + 128 * l;
        const float half = l < kLayers - 1 ? 0.5f : 1.f;
        for (int i = tid; i < N; i += nth)
            b[i] = i < layer_out(l) ? half * p[layer_offset(l) + layer_out(l) * layer_in(l) + i] : 0.f;
    }
}

// outputs [n][20] of inputs [n][7] on the tcgen05 engine: 128 rows per tile, kTcGroups
// tiles in flight per CTA
constexpr int kTcGroups = 3;
__global__ void __launch_bounds__(tc::kRows * kTcGroups, 1)
    k_infer_tc(const unsigned char* __restrict__ img, long long n, const float* __restrict__ in,
               float* __restrict__ out, unsigned* __restrict__ error) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) unsigned long long mbar[kTcGroups];
    __shared__ unsigned tmem_slot;
    const tc::Group g = tc::setup(kTcGroups, sm, img, mbar, &tmem_slot);
    unsigned phase = 0;
    bool failed = false;
    const long long ntile = (n + tc::kRows - 1) / tc::kRows;
    const int gi = threadIdx.x / tc::kRows;
    for (long long tile = (long long)blockIdx.x * kTcGroups + gi; tile < ntile; tile += (long long)gridDim.x * kTcGroups) {
        const long long row = tile * tc::kRows + g.t;
        float u[kIn];
        for (int c = 0; c < kIn; ++c) u[c] = row < n ? in[row * kIn + c] : 0.f;
        tc::store_input(g, u);
        float y[24];
        if (!tc::forward(g, y, phase, 2000000000ull)) {
            failed = true;
            if (g.t == 0) atomicOr(error, 1u);
            break;
        }
        if (row < n)
            for (int o = 0; o < kOut; ++o) out[row * kOut + o] = y[o];
        tc::group_sync(g);  // every row has read its outputs before the next tile's layer 0
    }
    tc::teardown(kTcGroups, g, failed, phase, 2000000000ull);
}

// ---------------------------------------------------------------------------------
// fused inference (mcrt_mlp_infer.cuh): evaluation, error map, extinction table
// ---------------------------------------------------------------------------------
constexpr int kInferBlock = 256;
struct WarpTile {
    bf16 in[16 * mlp::kLd0];
    float out[16 * mlp::kOutLd];
};
static_assert(sizeof(WarpTile) % 16 == 0, "tiles stay 16-byte aligned");
constexpr size_t kInferSmem = mlp::kImgBytes + (kInferBlock / 32) * sizeof(WarpTile);

__device__ __forceinline__ WarpTile& warp_tile(unsigned char* sm) {
    return reinterpret_cast<WarpTile*>(sm + mlp::kImgBytes)[threadIdx.x >> 5];
}

// outputs [n][20] of inputs [n][7]
__global__ void __launch_bounds__(kInferBlock) k_infer(const unsigned char* __restrict__ img, long long n,
                                                       const float* __restrict__ in, float* __restrict__ out) {
    extern __shared__ __align__(128) unsigned char sm[];
    mlp::load_image(sm, img);
    __syncthreads();
    WarpTile& wt = warp_tile(sm);
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const long long ntile = (n + 15) / 16;
    for (long long tile = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); tile < ntile; tile += (long long)gridDim.x * wpb) {
        const long long row = tile * 16 + lane;
        if (lane < 16) {
            float u[kIn];
            for (int c = 0; c < kIn; ++c) u[c] = row < n ? in[row * kIn + c] : 0.f;
            mlp::store_input_row(wt.in + lane * mlp::kLd0, u);
        }
        __syncwarp();
        mlp::warp_mlp16(sm, wt.in, wt.out, lane);
        __syncwarp();
        if (lane < 16 && row < n)
            for (int o = 0; o < kOut; ++o) out[row * kOut + o] = wt.out[lane * mlp::kOutLd + o];
        __syncwarp();
    }
}

// Error map: for n samples (uniform directions, uniform s) the largest error of the
// network's scattering matrix against the tables relative to the true M11, per cell
// of (cos theta_i, cos theta_s, delta phi, s).  map: 4096 floats, zeroed by the
// caller (non-negative floats compare like their bit patterns).
__global__ void __launch_bounds__(kInferBlock) k_errmap(const unsigned char* __restrict__ img, LabelTables T,
                                                        long long n, unsigned seed, float* __restrict__ map) {
    extern __shared__ __align__(128) unsigned char sm[];
    mlp::load_image(sm, img);
    __syncthreads();
    WarpTile& wt = warp_tile(sm);
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const long long ntile = (n + 15) / 16;
    for (long long tile = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); tile < ntile; tile += (long long)gridDim.x * wpb) {
        const long long i = tile * 16 + lane;
        float lab[kOut];
        V3<float> ni{0.f, 0.f, 1.f}, ns{0.f, 0.f, 1.f};
        float s = 0.f;
        if (lane < 16) {
            const Draw4<float> u0 = draw4<float>(i, 0u, 0x61u, seed, 0xE77u);
            const Draw4<float> u1 = draw4<float>(i, 0u, 0x62u, seed, 0xE77u);
            ni = iso_unit(u0.a, u0.b);
            ns = iso_unit(u0.c, u0.d);
            s = 2.f * u1.a - 1.f;
            surrogate_label(T, ni, ns, s, lab);
            const float u[kIn] = {ni.x, ni.y, ni.z, ns.x, ns.y, ns.z, s};
            mlp::store_input_row(wt.in + lane * mlp::kLd0, u);
        }
        __syncwarp();
        mlp::warp_mlp16(sm, wt.in, wt.out, lane);
        __syncwarp();
        if (lane < 16 && i < n) {
            const float* y = wt.out + lane * mlp::kOutLd;
            const float r = __expf(y[0] - lab[0]);  // M11 of the network / true M11
            float e = fabsf(r - 1.f);
            for (int o = 1; o < 16; ++o) e = fmaxf(e, fabsf(r * y[o] - lab[o]));
            if (!(e <= 3.0e38f)) e = 3.0e38f;  // NaN or inf: always falls back
            const int idx = mlp::errmap_index(ni.z, ns.z, atan2f(ns.y, ns.x) - atan2f(ni.y, ni.x), s);
            atomicMax(reinterpret_cast<int*>(map) + idx, __float_as_int(e));
        }
        __syncwarp();
    }
}

// Extinction elements alpha1..3 of the network on the grid theta'_j = pi j / (n_k - 1):
// the mean over 16 scattered directions and sizes of outputs 16..18 at
// n_i = (sin theta', 0, cos theta').  Rows that are not realizable (alpha1 <= 0 or
// |alpha2| >= alpha1) keep the table's row and are counted.
__global__ void __launch_bounds__(kInferBlock) k_distill_kext(const unsigned char* __restrict__ img, int n_k,
                                                              const float4* __restrict__ table,
                                                              float4* __restrict__ out, unsigned* __restrict__ n_fixed) {
    extern __shared__ __align__(128) unsigned char sm[];
    mlp::load_image(sm, img);
    __syncthreads();
    WarpTile& wt = warp_tile(sm);
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    for (int j = blockIdx.x * wpb + (threadIdx.x >> 5); j < n_k; j += gridDim.x * wpb) {
        if (lane < 16) {
            float st, ct, sp, cp;
            sincospif((float)j / (float)(n_k - 1), &st, &ct);
            const float z = 1.f - (2.f * lane + 1.f) / 16.f, rho = sqrtf(fmaxf(0.f, 1.f - z * z));
            sincosf(2.39996323f * (float)lane, &sp, &cp);
            const float u[kIn] = {st, 0.f, ct, rho * cp, rho * sp, z, -1.f + (2.f * lane + 1.f) / 16.f};
            mlp::store_input_row(wt.in + lane * mlp::kLd0, u);
        }
        __syncwarp();
        mlp::warp_mlp16(sm, wt.in, wt.out, lane);
        __syncwarp();
        if (lane == 0) {
            float a[3] = {0.f, 0.f, 0.f};
            for (int r = 0; r < 16; ++r)
                for (int e = 0; e < 3; ++e) a[e] += wt.out[r * mlp::kOutLd + 16 + e] * (1.f / 16.f);
            const bool ok = a[0] > 0.f && fabsf(a[1]) < a[0] && fabsf(a[2]) < 3.0e38f;
            if (ok) {
                out[j] = make_float4(a[0], a[1], a[2], 0.f);
            } else {
                out[j] = table[j];
                atomicAdd(n_fixed, 1u);
            }
        }
        __syncwarp();
    }
}

}  // namespace

// ---------------------------------------------------------------------------------
// host side: the surrogate object
// ---------------------------------------------------------------------------------
}  // namespace mcrt

using namespace mcrt;

struct mcrt_surrogate {
    cudaStream_t stream = nullptr;
    float4* d_bins = nullptr;
    float4* d_kext = nullptr;
    int n_bins = 0, n_theta = 0, n_ktheta = 0;
    float* d_params = nullptr;
    float* d_grads = nullptr;
    float* d_m = nullptr;
    float* d_v = nullptr;
    float* d_w = nullptr;  // loss weights [20]
    bf16* d_wbf = nullptr;
    double* d_loss = nullptr;
    float* d_in = nullptr;  // inputs of a user or of a training step
    size_t in_cap = 0;
    float* d_t = nullptr;  // targets
    size_t t_cap = 0;
    float* d_parts = nullptr;  // partial gradients
    size_t parts_cap = 0;
    unsigned seed = 0;
    long long step = 0;
    unsigned char* d_image = nullptr;  // inference image of the current parameters
    float* d_map = nullptr;            // error map [4096]
    bool map_valid = false;
    int n_sm = 0;
};

namespace {

#define SK(call)                                                                                        \
    do {                                                                                                \
        cudaError_t e_ = (call);                                                                        \
        if (e_ != cudaSuccess) {                                                                        \
            (void)cudaGetLastError();                                                                   \
            return mcrt_fail_noctx(MCRT_E_CUDA, "surrogate: %s: %s", #call, cudaGetErrorString(e_));    \
        }                                                                                               \
    } while (0)

// Room for n rows of inputs, and of targets.
mcrt_status ensure(float*& d, size_t& cap, size_t bytes) {
    if (cap >= bytes) return MCRT_OK;
    cudaFree(d);
    d = nullptr;
    cap = 0;
    SK(cudaMalloc(&d, bytes));
    cap = bytes;
    return MCRT_OK;
}

LabelTables tables_of(const mcrt_surrogate* s) {
    return LabelTables{s->d_bins, s->d_kext, s->n_bins, s->n_theta, s->n_ktheta};
}

// How a batch of B rows runs.  Tiles of 16 rows while there is an SM for each (a training step of
// 1024 rows 45 us, 47 with 32), else of 32, which add the weight gradients half as often (2^16
// rows: 0.31 ms, 0.45 with 16).  Partial gradients: as many as keep the FP32 sum over the tiles as
// close to the rows' exact sum as split products did that took in 64 tiles of 128 rows and more.
// Error of the sum in norm, split products, one sum and these: 512 rows 2.9e-8, 2.6e-8, 1.3e-8; 2048
// 4.2e-8, 5.5e-8, 1.8e-8; 8192 6.2e-8, 1.6e-7, 3.8e-8; 2^16 2.8e-7, 9.3e-7, 3.8e-8.  More (32) cost 7 us
// at 8193 rows; up to 8 tiles one is enough, and the call saves 10 us of k_fold.
struct PassShape {
    int rows, grid, n_parts;
    float* parts;
};
PassShape pass_shape(const mcrt_surrogate* s, int B) {
    const int rows = B <= 16 * s->n_sm ? 16 : 32, tiles = (B + rows - 1) / rows;
    const int n_parts = tiles <= 8 ? 1 : (tiles <= 256 ? 4 : 16);
    return PassShape{rows, tiles < s->n_sm ? tiles : s->n_sm, n_parts, n_parts == 1 ? s->d_grads : s->d_parts};
}

// Room for the inputs, the targets and the partial gradients of B rows.
mcrt_status pass_buffers(mcrt_surrogate* s, int B) {
    mcrt_status st = ensure(s->d_in, s->in_cap, (size_t)B * kIn * sizeof(float));
    if (st == MCRT_OK) st = ensure(s->d_t, s->t_cap, (size_t)B * kOut * sizeof(float));
    const int n_parts = pass_shape(s, B).n_parts;
    if (st == MCRT_OK && n_parts > 1) st = ensure(s->d_parts, s->parts_cap, sizeof(float) * kParams * n_parts);
    return st;
}

// Loss and gradients of the B rows in d_in and d_t: gradients of all parameters into the partial
// ones (d_grads itself if there is but one), the loss added to loss[*iter] (loss[0] without an iteration counter).
mcrt_status pass(mcrt_surrogate* s, int B, const LossWeights& w, double* loss, const unsigned* iter) {
    const PassShape h = pass_shape(s, B);
    SK(cudaMemsetAsync(h.parts, 0, sizeof(float) * kParams * h.n_parts, s->stream));
    (void)cudaGetLastError();
    if (h.rows == 16) {
        SK(cudaFuncSetAttribute(k_pass<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pass_smem(1)));
        k_pass<1><<<h.grid, kPassThreads, pass_smem(1), s->stream>>>(B, s->d_in, s->d_t, w, s->d_wbf, s->d_params,
                                                                     h.parts, h.n_parts, loss, iter);
    } else {
        SK(cudaFuncSetAttribute(k_pass<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pass_smem(2)));
        k_pass<2><<<h.grid, kPassThreads, pass_smem(2), s->stream>>>(B, s->d_in, s->d_t, w, s->d_wbf, s->d_params,
                                                                     h.parts, h.n_parts, loss, iter);
    }
    SK(cudaGetLastError());
    return MCRT_OK;
}

mcrt_status stage_inputs(mcrt_surrogate* s, const float* in, long long n) {
    const size_t bytes = (size_t)n * kIn * sizeof(float);
    const mcrt_status st = ensure(s->d_in, s->in_cap, bytes);
    if (st != MCRT_OK) return st;
    SK(cudaMemcpyAsync(s->d_in, in, bytes, cudaMemcpyDefault, s->stream));
    return MCRT_OK;
}

// Inference image of the current parameters (on the surrogate's stream).
mcrt_status pack_image(mcrt_surrogate* s) {
    (void)cudaGetLastError();
    k_pack_image<<<64, 256, 0, s->stream>>>(s->d_params, s->d_image);
    SK(cudaGetLastError());
    return MCRT_OK;
}

template <typename K> mcrt_status infer_attr(K kernel) {
    SK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kInferSmem));
    return MCRT_OK;
}

int infer_grid(const mcrt_surrogate* s, long long tiles) {
    const long long per_block = kInferBlock / 32;
    long long g = (tiles + per_block - 1) / per_block;
    const long long cap = (long long)(s->n_sm > 0 ? s->n_sm : 1) * 1;
    return (int)(g < cap ? (g > 0 ? g : 1) : cap);
}

mcrt_status compute_error_map(mcrt_surrogate* s, long long n_samples) {
    mcrt_status st = pack_image(s);
    if (st != MCRT_OK) return st;
    st = infer_attr(k_errmap);
    if (st != MCRT_OK) return st;
    SK(cudaMemsetAsync(s->d_map, 0, sizeof(float) * kErrMapCells, s->stream));
    k_errmap<<<infer_grid(s, (n_samples + 15) / 16), kInferBlock, kInferSmem, s->stream>>>(
        s->d_image, tables_of(s), n_samples, s->seed ^ 0x9E3779B9u, s->d_map);
    SK(cudaGetLastError());
    SK(cudaStreamSynchronize(s->stream));
    s->map_valid = true;
    return MCRT_OK;
}

}  // namespace

// Inference data of the surrogate for a model's transport: the inference image, the
// error map (computed with 2^22 samples if not yet done) and the distilled extinction
// table on n_ktheta angles (rows that are not realizable come from `table`).
mcrt_status mcrt_surrogate_export(mcrt_surrogate* s, int n_ktheta, const float4* table, unsigned char* d_image,
                                  unsigned char* d_image_tc, float* d_map, float4* d_kext, int* n_fixed) {
    if (!s->map_valid) {
        mcrt_status st = compute_error_map(s, 1ll << 22);
        if (st != MCRT_OK) return st;
    }
    mcrt_status st = pack_image(s);
    if (st != MCRT_OK) return st;
    st = infer_attr(k_distill_kext);
    if (st != MCRT_OK) return st;
    unsigned* d_fixed = nullptr;
    SK(cudaMalloc(&d_fixed, sizeof(unsigned)));
    cudaError_t e = cudaMemsetAsync(d_fixed, 0, sizeof(unsigned), s->stream);
    if (e == cudaSuccess) {
        (void)cudaGetLastError();
        k_distill_kext<<<infer_grid(s, n_ktheta), kInferBlock, kInferSmem, s->stream>>>(s->d_image, n_ktheta, table,
                                                                                      d_kext, d_fixed);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_image, s->d_image, mlp::kImgBytes, cudaMemcpyDeviceToDevice, s->stream);
    if (e == cudaSuccess) {
        k_pack_image_tc<<<64, 256, 0, s->stream>>>(s->d_params, d_image_tc);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_map, s->d_map, sizeof(float) * kErrMapCells, cudaMemcpyDeviceToDevice, s->stream);
    unsigned fixed = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&fixed, d_fixed, sizeof(unsigned), cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    cudaFree(d_fixed);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return mcrt_fail_noctx(MCRT_E_CUDA, "surrogate export: %s", cudaGetErrorString(e));
    }
    if (n_fixed) *n_fixed = (int)fixed;
    return MCRT_OK;
}

extern "C" {

mcrt_status mcrt_surrogate_create(mcrt_surrogate** out, const mcrt_ctx* optics, uint32_t seed) {
    if (!out) return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_create: out is NULL");
    *out = nullptr;
    TablesDev t{};
    if (mcrt_ctx_tables(optics, &t) != MCRT_OK || t.model != MCRT_SCAT_TABLE)
        return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_create: the model needs tabulated optics");
    mcrt_surrogate* s = new (std::nothrow) mcrt_surrogate();
    if (!s) return mcrt_fail_noctx(MCRT_E_NOMEM, "mcrt_surrogate_create: host allocation");
    s->n_bins = t.n_bins;
    s->n_theta = t.n_theta;
    s->n_ktheta = t.n_ktheta;
    s->seed = seed;
    cudaError_t e = cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking);
    const size_t nbins = (size_t)t.n_bins * t.n_theta * 2;
    if (e == cudaSuccess) e = cudaMalloc(&s->d_bins, nbins * sizeof(float4));
    if (e == cudaSuccess) e = cudaMalloc(&s->d_kext, (size_t)t.n_ktheta * sizeof(float4));
    if (e == cudaSuccess) e = cudaMalloc(&s->d_params, sizeof(float) * kParams);
    if (e == cudaSuccess) e = cudaMalloc(&s->d_grads, sizeof(float) * kParams);
    if (e == cudaSuccess) e = cudaMalloc(&s->d_m, sizeof(float) * kParams);
    if (e == cudaSuccess) e = cudaMalloc(&s->d_v, sizeof(float) * kParams);
    if (e == cudaSuccess) e = cudaMalloc(&s->d_w, sizeof(float) * kOut);
    if (e == cudaSuccess) e = cudaMalloc(&s->d_wbf, sizeof(bf16) * kWeights);
    if (e == cudaSuccess) e = cudaMalloc(&s->d_loss, sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&s->d_image, mlp::kImgBytes);
    if (e == cudaSuccess) e = cudaMalloc(&s->d_map, sizeof(float) * kErrMapCells);
    if (e == cudaSuccess) {
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&s->n_sm, cudaDevAttrMultiProcessorCount, dev);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(s->d_bins, t.bins, nbins * sizeof(float4), cudaMemcpyDeviceToDevice, s->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(s->d_kext, t.kext, (size_t)t.n_ktheta * sizeof(float4), cudaMemcpyDeviceToDevice, s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->d_m, 0, sizeof(float) * kParams, s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->d_v, 0, sizeof(float) * kParams, s->stream);
    if (e == cudaSuccess) {
        std::vector<float> w(kOut, 1.f);
        e = cudaMemcpyAsync(s->d_w, w.data(), sizeof(float) * kOut, cudaMemcpyHostToDevice, s->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    }
    if (e == cudaSuccess) {
        (void)cudaGetLastError();
        k_init_params<<<64, 256, 0, s->stream>>>(s->d_params, seed);
        k_pack_weights<<<64, 256, 0, s->stream>>>(s->d_params, s->d_wbf, nullptr);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) {
        mcrt_surrogate_destroy(s);
        return mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_create: %s", cudaGetErrorString(e));
    }
    *out = s;
    return MCRT_OK;
}

mcrt_status mcrt_surrogate_train(mcrt_surrogate* s, int64_t n_steps, int32_t batch, double lr, double* loss_history) {
    if (!s || n_steps < 0 || batch < 64 || batch > (1 << 20) || n_steps > (1ll << 31))
        return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_train: bad arguments");
    {
        const mcrt_status st = pass_buffers(s, batch);
        if (st != MCRT_OK) return st;
    }
    s->map_valid = false;
    if (n_steps == 0) return MCRT_OK;
    const LabelTables T = tables_of(s);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    // schedule of every step: cosine decay of the learning rate over the call's steps
    // and Adam's bias corrections of the global step
    std::vector<float> sched((size_t)n_steps * 3);
    for (long long it = 0; it < n_steps; ++it) {
        const unsigned step = (unsigned)(s->step + it);
        const double frac = n_steps > 1 ? (double)it / (double)(n_steps - 1) : 0.0;
        sched[3 * it] = (float)(lr * (0.05 + 0.95 * 0.5 * (1.0 + std::cos(3.141592653589793 * frac))));
        sched[3 * it + 1] = 1.f - std::pow(b1, (float)(step + 1));
        sched[3 * it + 2] = 1.f - std::pow(b2, (float)(step + 1));
    }
    // one allocation: loss per step (FP64), schedule, iteration counter
    const size_t hist_bytes = (size_t)n_steps * sizeof(double), sched_bytes = sched.size() * sizeof(float);
    unsigned char* work = nullptr;
    SK(cudaMalloc(&work, hist_bytes + sched_bytes + 16));
    double* d_hist = reinterpret_cast<double*>(work);
    float* d_sched = reinterpret_cast<float*>(work + hist_bytes);
    unsigned* d_iter = reinterpret_cast<unsigned*>(work + hist_bytes + sched_bytes);
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    auto done = [&](mcrt_status st) {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        cudaStreamSynchronize(s->stream);
        cudaFree(work);
        return st;
    };
    cudaError_t e = cudaMemcpyAsync(d_sched, sched.data(), sched_bytes, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_hist, 0, hist_bytes, s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_iter, 0, sizeof(unsigned), s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);  // the schedule left the host buffer
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return done(mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_train: %s", cudaGetErrorString(e)));
    }
    // one training step, captured once and replayed: every launch of the step reads its
    // iteration from d_iter, which the step's last kernel advances
    (void)cudaGetLastError();
    e = cudaStreamBeginCapture(s->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return done(mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_train: %s", cudaGetErrorString(e)));
    mcrt_status st = MCRT_OK;
    k_gen_batch<<<(batch + 127) / 128, 128, 0, s->stream>>>(T, s->seed, (unsigned)s->step, d_iter, batch, s->d_in,
                                                            s->d_t);
    if (cudaGetLastError() != cudaSuccess) st = MCRT_E_CUDA;
    if (st == MCRT_OK) {
        LossWeights w;
        for (float& v : w.w) v = 1.f;
        st = pass(s, batch, w, d_hist, d_iter);
    }
    if (st == MCRT_OK) {
        const PassShape h = pass_shape(s, batch);
        k_adam<<<128, 256, 0, s->stream>>>(kParams, s->d_params, h.parts, h.n_parts, s->d_m, s->d_v, d_sched, d_iter, b1,
                                           b2, eps);
        k_pack_weights<<<64, 256, 0, s->stream>>>(s->d_params, s->d_wbf, d_iter);
        if (cudaGetLastError() != cudaSuccess) st = MCRT_E_CUDA;
    }
    e = cudaStreamEndCapture(s->stream, &graph);
    if (st != MCRT_OK) return done(mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_train: capture of the step failed"));
    if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
    for (long long it = 0; it < n_steps && e == cudaSuccess; ++it) e = cudaGraphLaunch(exec, s->stream);
    if (e == cudaSuccess && loss_history)
        e = cudaMemcpyAsync(loss_history, d_hist, hist_bytes, cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return done(mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_train: %s", cudaGetErrorString(e)));
    }
    s->step += n_steps;
    return done(MCRT_OK);
}

mcrt_status mcrt_surrogate_eval(mcrt_surrogate* s, int64_t n, const float* inputs, float* outputs) {
    if (!s || n < 0 || (n > 0 && (!inputs || !outputs))) return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_eval: bad arguments");
    if (n == 0) return MCRT_OK;
    mcrt_status st = stage_inputs(s, inputs, n);
    if (st != MCRT_OK) return st;
    st = pack_image(s);
    if (st != MCRT_OK) return st;
    st = infer_attr(k_infer);
    if (st != MCRT_OK) return st;
    float* d_out = nullptr;
    SK(cudaMalloc(&d_out, (size_t)n * kOut * sizeof(float)));
    (void)cudaGetLastError();
    k_infer<<<infer_grid(s, (n + 15) / 16), kInferBlock, kInferSmem, s->stream>>>(s->d_image, n, s->d_in, d_out);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(outputs, d_out, (size_t)n * kOut * sizeof(float), cudaMemcpyDefault, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    cudaFree(d_out);
    if (e != cudaSuccess) return mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_eval: %s", cudaGetErrorString(e));
    return MCRT_OK;
}

mcrt_status mcrt_surrogate_eval_engine(mcrt_surrogate* s, int32_t engine, int64_t n, const float* inputs,
                                       float* outputs) {
    if (engine == MCRT_ENGINE_MMA_SYNC) return mcrt_surrogate_eval(s, n, inputs, outputs);
    if (!s || engine != MCRT_ENGINE_TCGEN05 || n < 0 || (n > 0 && (!inputs || !outputs)))
        return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_eval_engine: bad arguments");
    if (n == 0) return MCRT_OK;
    mcrt_status st = stage_inputs(s, inputs, n);
    if (st != MCRT_OK) return st;
    unsigned char* d_img = nullptr;
    float* d_out = nullptr;
    unsigned* d_err = nullptr;
    unsigned err = 0;
    cudaError_t e = cudaMalloc(&d_img, tc::kImgBytes);
    if (e == cudaSuccess) e = cudaMalloc(&d_out, (size_t)n * kOut * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&d_err, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemsetAsync(d_err, 0, sizeof(unsigned), s->stream);
    if (e == cudaSuccess) {
        (void)cudaGetLastError();
        k_pack_image_tc<<<64, 256, 0, s->stream>>>(s->d_params, d_img);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_infer_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::smem_bytes(kTcGroups));
    if (e == cudaSuccess) {
        const long long tiles = (n + tc::kRows * kTcGroups - 1) / (tc::kRows * kTcGroups);
        const int grid = (int)(tiles < s->n_sm ? tiles : s->n_sm);
        k_infer_tc<<<grid, tc::kRows * kTcGroups, tc::smem_bytes(kTcGroups), s->stream>>>(d_img, n, s->d_in, d_out, d_err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(outputs, d_out, (size_t)n * kOut * sizeof(float), cudaMemcpyDefault, s->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, d_err, sizeof(unsigned), cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    cudaFree(d_img);
    cudaFree(d_out);
    cudaFree(d_err);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_eval_engine: %s", cudaGetErrorString(e));
    }
    if (err) return mcrt_fail_noctx(MCRT_E_TIMEOUT, "mcrt_surrogate_eval_engine: a tensor-core wait timed out");
    return MCRT_OK;
}

mcrt_status mcrt_surrogate_error_map(mcrt_surrogate* s, int64_t n_samples, float* map) {
    if (!s || n_samples < 16 || n_samples > (1ll << 34))
        return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_error_map: bad arguments");
    mcrt_status st = compute_error_map(s, n_samples);
    if (st != MCRT_OK) return st;
    if (map) {
        SK(cudaMemcpyAsync(map, s->d_map, sizeof(float) * kErrMapCells, cudaMemcpyDefault, s->stream));
        SK(cudaStreamSynchronize(s->stream));
    }
    return MCRT_OK;
}

mcrt_status mcrt_surrogate_labels(mcrt_surrogate* s, int64_t n, const float* inputs, float* labels) {
    if (!s || n < 0 || (n > 0 && (!inputs || !labels))) return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_labels: bad arguments");
    if (n == 0) return MCRT_OK;
    mcrt_status st = stage_inputs(s, inputs, n);
    if (st != MCRT_OK) return st;
    float* d_out = nullptr;
    SK(cudaMalloc(&d_out, (size_t)n * kOut * sizeof(float)));
    (void)cudaGetLastError();
    k_labels<<<(unsigned)((n + 127) / 128), 128, 0, s->stream>>>(tables_of(s), (int)n, s->d_in, d_out);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(labels, d_out, (size_t)n * kOut * sizeof(float), cudaMemcpyDefault, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    cudaFree(d_out);
    if (e != cudaSuccess) return mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_labels: %s", cudaGetErrorString(e));
    return MCRT_OK;
}

mcrt_status mcrt_surrogate_grad(mcrt_surrogate* s, int64_t n, const float* inputs, const float* targets,
                                const float* loss_weights, float* grads, double* loss) {
    if (!s || n < 1 || n > (1 << 20) || !inputs || !targets || !grads)
        return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_grad: bad arguments");
    mcrt_status st = pass_buffers(s, (int)n);
    if (st == MCRT_OK) st = stage_inputs(s, inputs, n);
    if (st != MCRT_OK) return st;
    SK(cudaMemcpyAsync(s->d_t, targets, (size_t)n * kOut * sizeof(float), cudaMemcpyDefault, s->stream));
    LossWeights w;
    for (int o = 0; o < kOut; ++o) w.w[o] = loss_weights ? loss_weights[o] : 1.f;
    SK(cudaMemsetAsync(s->d_loss, 0, sizeof(double), s->stream));
    st = pass(s, (int)n, w, s->d_loss, nullptr);
    if (st != MCRT_OK) return st;
    const PassShape h = pass_shape(s, (int)n);
    if (h.n_parts > 1) k_fold<<<(kParams + 127) / 128, 128, 0, s->stream>>>(h.parts, h.n_parts, s->d_grads);
    SK(cudaGetLastError());
    SK(cudaMemcpyAsync(grads, s->d_grads, sizeof(float) * kParams, cudaMemcpyDefault, s->stream));
    double l = 0.0;
    SK(cudaMemcpyAsync(&l, s->d_loss, sizeof(double), cudaMemcpyDeviceToHost, s->stream));
    SK(cudaStreamSynchronize(s->stream));
    if (loss) *loss = l;
    return MCRT_OK;
}

// The FP32 mode of mcrt_surrogate_grad: forward, loss gradient and backward with FP32
// operands, activations and gradients (k_gemm32), the FP32 master weights as they
// are.  Its buffers live for the call only.
mcrt_status mcrt_surrogate_grad_fp32(mcrt_surrogate* s, int64_t n, const float* inputs, const float* targets,
                                     const float* loss_weights, float* grads, double* loss) {
    if (!s || n < 1 || n > (1 << 20) || !inputs || !targets || !grads)
        return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_grad_fp32: bad arguments");
    mcrt_status st = stage_inputs(s, inputs, n);
    if (st != MCRT_OK) return st;
    const int B = (int)n;
    // x [B][16], z and h [4][B][128], y [B][24], t [B][20], dy [B][24], dz [2][B][128]
    const size_t nx = (size_t)B * kInPad, nh = (size_t)B * kHid, ny = (size_t)B * kOutPad;
    const size_t total = nx + 8 * nh + ny + (size_t)B * kOut + ny + 2 * nh;
    float* base = nullptr;
    SK(cudaMalloc(&base, total * sizeof(float)));
    float* x = base;
    float* z[4];
    float* h[4];
    for (int i = 0; i < 4; ++i) {
        z[i] = x + nx + (size_t)(2 * i) * nh;
        h[i] = z[i] + nh;
    }
    float* y = x + nx + 8 * nh;
    float* t = y + ny;
    float* dy = t + (size_t)B * kOut;
    float* dzb[2] = {dy + ny, dy + ny + nh};
    cudaError_t e = cudaSuccess;
    auto ck = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
    };
    k_pack_inputs32<<<(unsigned)((n + 127) / 128), 128, 0, s->stream>>>(B, s->d_in, x);
    ck(cudaGetLastError());
    ck(cudaMemcpyAsync(t, targets, (size_t)n * kOut * sizeof(float), cudaMemcpyDefault, s->stream));
    std::vector<float> w(kOut, 1.f);
    if (loss_weights) std::memcpy(w.data(), loss_weights, sizeof(float) * kOut);
    ck(cudaMemcpyAsync(s->d_w, w.data(), sizeof(float) * kOut, cudaMemcpyHostToDevice, s->stream));
    for (int l = 0; l < kLayers && e == cudaSuccess; ++l) {
        GemmArgs32 g{};
        g.M = B;
        g.N = layer_out(l);
        g.K = layer_in(l);
        g.A = l == 0 ? x : h[l - 1];
        g.lda = layer_in(l);
        g.B = s->d_params + layer_offset(l);
        g.ldb = layer_in(l);
        g.bias = s->d_params + layer_offset(l) + layer_out(l) * layer_in(l);
        if (l < kLayers - 1) {
            g.Zout = z[l];
            g.ldz = kHid;
            g.Hout = h[l];
            g.ldh = kHid;
            ck(gemm32<EPI_HIDDEN>(g, s->stream));
        } else {
            g.Zout = y;
            g.ldz = kOutPad;
            ck(gemm32<EPI_OUT>(g, s->stream));
        }
    }
    ck(cudaMemsetAsync(s->d_loss, 0, sizeof(double), s->stream));
    if (e == cudaSuccess) {
        k_loss_grad32<<<256, 256, 0, s->stream>>>(B, y, t, s->d_w, dy, s->d_loss);
        ck(cudaGetLastError());
    }
    ck(cudaMemsetAsync(s->d_grads, 0, sizeof(float) * kParams, s->stream));
    const float* dZ = dy;
    int cur = 0;
    for (int l = kLayers - 1; l >= 0 && e == cudaSuccess; --l) {
        const int no = layer_out(l), ni = layer_in(l);
        GemmArgs32 gw{};
        gw.M = no;
        gw.N = ni;
        gw.K = B;
        gw.A = dZ;
        gw.lda = no;
        gw.a_t = 1;
        gw.B = l == 0 ? x : h[l - 1];
        gw.ldb = ni;
        gw.b_kn = 1;
        gw.Zout = s->d_grads + layer_offset(l);
        gw.ldz = ni;
        ck(gemm32<EPI_DW>(gw, s->stream));
        k_colsum32<<<dim3((no + 127) / 128, 64), 128, 0, s->stream>>>(B, no, dZ,
                                                                      s->d_grads + layer_offset(l) + no * ni);
        ck(cudaGetLastError());
        if (l == 0) break;
        GemmArgs32 gx{};
        gx.M = B;
        gx.N = ni;
        gx.K = no;
        gx.A = dZ;
        gx.lda = no;
        gx.B = s->d_params + layer_offset(l);
        gx.ldb = ni;
        gx.b_kn = 1;
        gx.Zprev = z[l - 1];
        gx.ldz = kHid;
        gx.Hout = dzb[cur];
        gx.ldh = kHid;
        ck(gemm32<EPI_DX>(gx, s->stream));
        dZ = dzb[cur];
        cur ^= 1;
    }
    double lv = 0.0;
    ck(cudaMemcpyAsync(grads, s->d_grads, sizeof(float) * kParams, cudaMemcpyDefault, s->stream));
    ck(cudaMemcpyAsync(&lv, s->d_loss, sizeof(double), cudaMemcpyDeviceToHost, s->stream));
    std::vector<float> ones(kOut, 1.f);
    ck(cudaMemcpyAsync(s->d_w, ones.data(), sizeof(float) * kOut, cudaMemcpyHostToDevice, s->stream));
    ck(cudaStreamSynchronize(s->stream));
    cudaFree(base);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return mcrt_fail_noctx(MCRT_E_CUDA, "mcrt_surrogate_grad_fp32: %s", cudaGetErrorString(e));
    }
    if (loss) *loss = lv;
    return MCRT_OK;
}

mcrt_status mcrt_surrogate_params(mcrt_surrogate* s, float* params, int32_t set) {
    if (!s || !params) return mcrt_fail_noctx(MCRT_E_INVAL, "mcrt_surrogate_params: bad arguments");
    if (set) {
        s->map_valid = false;
        SK(cudaMemcpyAsync(s->d_params, params, sizeof(float) * kParams, cudaMemcpyDefault, s->stream));
        (void)cudaGetLastError();
        k_pack_weights<<<64, 256, 0, s->stream>>>(s->d_params, s->d_wbf, nullptr);
        SK(cudaGetLastError());
    } else {
        SK(cudaMemcpyAsync(params, s->d_params, sizeof(float) * kParams, cudaMemcpyDefault, s->stream));
    }
    SK(cudaStreamSynchronize(s->stream));
    return MCRT_OK;
}

int64_t mcrt_surrogate_param_count(void) { return kParams; }

mcrt_status mcrt_surrogate_destroy(mcrt_surrogate* s) {
    if (!s) return MCRT_OK;
    if (s->stream) cudaStreamSynchronize(s->stream);
    cudaFree(s->d_t);
    cudaFree(s->d_parts);
    cudaFree(s->d_bins);
    cudaFree(s->d_kext);
    cudaFree(s->d_params);
    cudaFree(s->d_grads);
    cudaFree(s->d_m);
    cudaFree(s->d_v);
    cudaFree(s->d_w);
    cudaFree(s->d_wbf);
    cudaFree(s->d_loss);
    cudaFree(s->d_in);
    cudaFree(s->d_image);
    cudaFree(s->d_map);
    if (s->stream) cudaStreamDestroy(s->stream);
    delete s;
    return MCRT_OK;
}

}  // extern "C"
