// Features (per triangle, stored order; lengths over sqrt(S_j), ratios as logarithms):
// angles opposite the three edges, log(|e_q|/sqrt S), log(d_q/sqrt S) (4 on a boundary edge),
// log(S_neighbour/S) (0 on a boundary edge).
//
// Learned spectral radius: features, the 12-64-64-1 MLP (forward on BF16 tensor cores with
// FP32 accumulation, or an FP32 debug path), its backward pass on the argmax rows, Adam, the
// per-mesh max aggregation, and the certified bracket used to accept a prediction.
//
// The paper fixes dt by the highest mode, dt < 2/omega_max (eq. 20), found by the "complex
// time" power iteration (Section 2).  The network predicts a correction z_j per triangle from
// scale-free geometry on top of base_j = log sqrt(K_jj) (K = -L_E L_B): rho_hat =
// max_j exp(z_j + base_j).  A prediction is used only inside the bracket
// [1.05 rho_lo, rho_hi]: rho_lo from max_j K_jj and a Rayleigh quotient of K^5 delta_j* near
// the argmax triangle, rho_hi from Gershgorin on S^{1/2} K S^{-1/2} (K = -L_E L_B).
//
// Parameter layout (floats): W1 [64x12] row-major, b1 [64], W2 [64x64] row-major, b2 [64],
// w3 [64], b3 [1]  (5,057 values).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "device.cuh"

namespace ue {

namespace {

constexpr int kH = 64, kD = 12;
constexpr int kOffW1 = 0, kOffB1 = kH * kD, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH;
constexpr int kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH, kNParams = kOffB3 + 1;
static_assert(kNParams == 5057, "parameter count");

// ---------------------------------------------------------------------------------------
// features (FP32, from FP64 geometry) and the per-triangle bracket terms
// ---------------------------------------------------------------------------------------
// Rounding slack of the FP32 bracket terms.  K_jj and the Gershgorin row bound are sums and
// products of positive values, formed from FP64 inputs by conversions and correctly rounded
// adds and multiplies (<= 2^-24 relative each), __frcp_rn (<= 2^-24) and the 2-ulp
// __fdividef and rsqrtf (<= 2^-22 each).  Along any path the errors add up to at most
// 20 * 2^-24 (11 for K_jj, 20 for the Gershgorin bound, first order), so the computed values lie
// within a factor 1 +- 20 * 2^-24 of the exact ones; scaling by 1 -+ 2^-16 keeps the bounds
// certified with 12x room.  Outside the normal FP32 range the terms give no bound (K_jj -> 0,
// Gershgorin -> +inf).
constexpr double kBracketSlack = 1.0 / 65536.0;

// One triangle's features, FP32.  The edge vectors are differences taken in FP64 (small
// triangles far from the origin lose nothing), then rounded; lengths and areas enter as logs
// of ratios near 1 (fast logs: every feature is rounded to BF16 before the first layer).
// The angle opposite edge q lies at vertex q+2, between E_{q+2} and -E_{q+1}; the third angle
// is pi minus the other two.  f[12] = base = log sqrt(K_jj).  kdiag = K_jj and gersh = the
// Gershgorin row bound of S^{1/2} K S^{-1/2}, both before the slack above.  The gathers are
// issued in two dependent rounds (row j's tables, then what they point to).
__device__ __forceinline__ void triangle_features(const double* __restrict__ xy,
                                                  const int32_t* __restrict__ tn,
                                                  const int32_t* __restrict__ code,
                                                  const int32_t* __restrict__ tnb,
                                                  const double* __restrict__ elen,
                                                  const double* __restrict__ d,
                                                  const double* __restrict__ S, int64_t j,
                                                  int64_t n_ei, float* f, float& kdiag,
                                                  float& gersh) {
    int vtx[3], nb[3];
    int64_t k[3];
    for (int q = 0; q < 3; ++q) {
        vtx[q] = tn[3 * j + q];
        k[q] = code[3 * j + q] >> 1;
        nb[q] = tnb[3 * j + q];
    }
    const double Sjd = S[j];
    double px[3], py[3], el[3], dd[3], sn[3];
    for (int q = 0; q < 3; ++q) {
        px[q] = xy[2 * vtx[q]];
        py[q] = xy[2 * vtx[q] + 1];
        const bool in = k[q] < n_ei;
        el[q] = in ? elen[k[q]] : 0.0;
        dd[q] = in ? d[k[q]] : 1.0;
        sn[q] = in ? S[nb[q]] : 1.0;
    }
    float ex[3], ey[3];
    for (int q = 0; q < 3; ++q) {
        const int b = q == 2 ? 0 : q + 1;
        ex[q] = (float)(px[b] - px[q]);
        ey[q] = (float)(py[b] - py[q]);
    }
    const float Sj = (float)Sjd;
    const float invS = __frcp_rn(Sj);
    const float rs = rsqrtf(Sj);
    for (int q = 0; q < 2; ++q) {
        const int u = q + 2 > 2 ? q - 1 : q + 2, v = q + 1;
        f[q] = atan2f(fabsf(ex[u] * ey[v] - ey[u] * ex[v]), -(ex[u] * ex[v] + ey[u] * ey[v]));
    }
    f[2] = 3.14159265358979f - f[0] - f[1];
    float kd = 0.f, off = 0.f;
    bool normal = Sj >= 1e-30f;
    for (int q = 0; q < 3; ++q) {
        f[3 + q] = 0.5f * __logf((ex[q] * ex[q] + ey[q] * ey[q]) * invS);
        if (k[q] < n_ei) {
            const float dk = (float)dd[q], Sn = (float)sn[q];
            const float w = __fdividef((float)el[q], dk);
            f[6 + q] = __logf(dk * rs);
            f[9 + q] = __logf(Sn * invS);
            kd = __fadd_rn(kd, w);
            off = __fadd_rn(off, __fmul_rn(__fmul_rn(w, rs), rsqrtf(Sn)));
            normal = normal && Sn >= 1e-30f && dk >= 1e-30f;
        } else {
            f[6 + q] = 4.f;    // boundary: a dual so long the edge adds nothing to K
            f[9 + q] = 0.f;
        }
    }
    kdiag = __fmul_rn(kd, invS);
    gersh = __fadd_rn(kdiag, off);
    f[12] = kd > 0.f ? 0.5f * __logf(kdiag) : -1e30f;
    if (!normal || !(kdiag <= 1e37f) || !(gersh <= 1e37f)) {
        kdiag = 0.f;
        gersh = INFINITY;
    }
}

__global__ void k_features(const double* __restrict__ xy, const int32_t* __restrict__ tn,
                           const int32_t* __restrict__ code, const int32_t* __restrict__ tnb,
                           const double* __restrict__ elen, const double* __restrict__ d,
                           const double* __restrict__ S, int64_t n_t, int64_t n_ei,
                           float* __restrict__ X, float* __restrict__ base) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_t) return;
    float f[kD + 1], kd, ge;
    triangle_features(xy, tn, code, tnb, elen, d, S, j, n_ei, f, kd, ge);
    for (int i = 0; i < kD; ++i) X[j * kD + i] = f[i];
    base[j] = f[kD];
}

// ---------------------------------------------------------------------------------------
// forward, BF16 tensor cores: one warp per 16 rows, mma.sync m16n8k16 (row.col), FP32 accum.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

constexpr int kW1S = 16 + 8;     // smem row stride (bf16) of W1 padded to K = 16
constexpr int kW2S = 64 + 8;     // smem row stride (bf16) of W2

// The network as the tensor-core layers read it: BF16 weights at the padded row strides (rows
// 16-byte aligned and 8 rows of an ldmatrix on distinct banks), FP32 biases.
struct PackedNet {
    __nv_bfloat16 w1[kH * kW1S];
    __nv_bfloat16 w2[kH * kW2S];
    float b1[kH], b2[kH], w3[kH];
    float b3[4];
};
static_assert(sizeof(PackedNet) % 16 == 0, "bulk copies move multiples of 16 bytes");

// N from the parameter vector: weights to BF16 (round to nearest even), zeros in the padding.
__device__ void pack_net(PackedNet& N, const float* __restrict__ P, int tid, int nth) {
    for (int i = tid; i < kH * kW1S; i += nth) {
        const int r = i / kW1S, c = i % kW1S;
        N.w1[i] = __float2bfloat16_rn(c < kD ? P[kOffW1 + r * kD + c] : 0.f);
    }
    for (int i = tid; i < kH * kW2S; i += nth) {
        const int r = i / kW2S, c = i % kW2S;
        N.w2[i] = __float2bfloat16_rn(c < kH ? P[kOffW2 + r * kH + c] : 0.f);
    }
    for (int i = tid; i < kH; i += nth) {
        N.b1[i] = P[kOffB1 + i];
        N.b2[i] = P[kOffB2 + i];
        N.w3[i] = P[kOffW3 + i];
    }
    if (tid < 4) N.b3[tid] = tid == 0 ? P[kOffB3] : 0.f;
}

// four 8x8 BF16 matrices from shared memory; lane l supplies row (l & 7) of matrix (l >> 3)
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void* row) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(row)));
}

// One 16-row tile through the network on the tensor cores.  a0..a3: the A fragments of the
// BF16 inputs (rows g and g+8, k 2t.. and 2t+8..).  The accumulators start at the biases; the
// B fragments of two n-tiles come with one ldmatrix.x4.  Returns w3 . relu(h2) for rows g (s0)
// and g+8 (s1), without b3, on all four lanes of each quad.
__device__ __forceinline__ void mlp16(const PackedNet& N, uint32_t a0, uint32_t a1, uint32_t a2,
                                      uint32_t a3, float& s0, float& s1) {
    const int lane = threadIdx.x & 31, t = lane & 3, mrow = lane & 7, mi = lane >> 3;
    float h1[8][4];
#pragma unroll
    for (int np = 0; np < 4; ++np) {
        uint32_t b[4];
        ldsm_x4(b, N.w1 + ((2 * np + (mi >> 1)) * 8 + mrow) * kW1S + (mi & 1) * 8);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int nt = 2 * np + h;
            const float2 bb = *reinterpret_cast<const float2*>(N.b1 + nt * 8 + 2 * t);
            h1[nt][0] = bb.x;
            h1[nt][1] = bb.y;
            h1[nt][2] = bb.x;
            h1[nt][3] = bb.y;
            mma_bf16(h1[nt], a0, a1, a2, a3, b[2 * h], b[2 * h + 1]);
        }
    }
    // relu, then BF16: the C fragments of layer 1 (n-tiles 2kt, 2kt+1) are the A fragments of
    // layer 2's k-tile kt
    uint32_t c[4][4];
#pragma unroll
    for (int kt = 0; kt < 4; ++kt) {
        c[kt][0] = pack_bf16(fmaxf(h1[2 * kt][0], 0.f), fmaxf(h1[2 * kt][1], 0.f));
        c[kt][1] = pack_bf16(fmaxf(h1[2 * kt][2], 0.f), fmaxf(h1[2 * kt][3], 0.f));
        c[kt][2] = pack_bf16(fmaxf(h1[2 * kt + 1][0], 0.f), fmaxf(h1[2 * kt + 1][1], 0.f));
        c[kt][3] = pack_bf16(fmaxf(h1[2 * kt + 1][2], 0.f), fmaxf(h1[2 * kt + 1][3], 0.f));
    }
    float h2[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const float2 bb = *reinterpret_cast<const float2*>(N.b2 + nt * 8 + 2 * t);
        h2[nt][0] = bb.x;
        h2[nt][1] = bb.y;
        h2[nt][2] = bb.x;
        h2[nt][3] = bb.y;
    }
#pragma unroll
    for (int kt = 0; kt < 4; ++kt) {
#pragma unroll
        for (int np = 0; np < 4; ++np) {
            uint32_t b[4];
            ldsm_x4(b, N.w2 + ((2 * np + (mi >> 1)) * 8 + mrow) * kW2S + kt * 16 + (mi & 1) * 8);
            mma_bf16(h2[2 * np], c[kt][0], c[kt][1], c[kt][2], c[kt][3], b[0], b[1]);
            mma_bf16(h2[2 * np + 1], c[kt][0], c[kt][1], c[kt][2], c[kt][3], b[2], b[3]);
        }
    }
    float x0 = 0.f, x1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const float2 w = *reinterpret_cast<const float2*>(N.w3 + nt * 8 + 2 * t);
        x0 += w.x * fmaxf(h2[nt][0], 0.f) + w.y * fmaxf(h2[nt][1], 0.f);
        x1 += w.x * fmaxf(h2[nt][2], 0.f) + w.y * fmaxf(h2[nt][3], 0.f);
    }
    x0 += __shfl_xor_sync(0xffffffffu, x0, 1);
    x0 += __shfl_xor_sync(0xffffffffu, x0, 2);
    x1 += __shfl_xor_sync(0xffffffffu, x1, 1);
    x1 += __shfl_xor_sync(0xffffffffu, x1, 2);
    s0 = x0;
    s1 = x1;
}

// Forward on few rows: one warp per 16, the network packed in the block's shared memory.  A warp takes
// a tile or two, and filling the registers of k_mlp_fwd_bf16 with the whole network took longer than
// reading what a tile needs.
__global__ void __launch_bounds__(128) k_mlp_fwd_few(const float* __restrict__ P, const float* __restrict__ X, int64_t n,
                                                     float* __restrict__ z) {
    __shared__ __align__(16) PackedNet net;
    pack_net(net, P, threadIdx.x, blockDim.x);
    __syncthreads();
    const float b3 = net.b3[0];
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t tile = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); tile * 16 < n; tile += warps) {
        const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
        auto xv = [&](int64_t r, int c) { return (r < n && c < kD) ? __ldg(X + r * kD + c) : 0.f; };
        const uint32_t a0 = pack_bf16(xv(r0, 2 * t), xv(r0, 2 * t + 1));
        const uint32_t a1 = pack_bf16(xv(r1, 2 * t), xv(r1, 2 * t + 1));
        const uint32_t a2 = pack_bf16(xv(r0, 2 * t + 8), xv(r0, 2 * t + 9));
        const uint32_t a3 = pack_bf16(xv(r1, 2 * t + 8), xv(r1, 2 * t + 9));
        float s0, s1;
        mlp16(net, a0, a1, a2, a3, s0, s1);
        if (t == 0) {
            if (r0 < n) z[r0] = s0 + b3;
            if (r1 < n) z[r1] = s1 + b3;
        }
    }
}

// Forward on BF16 tensor cores (mma.sync m16n8k16, FP32 accumulation): one warp per 16 rows.  The
// whole network sits in a warp's registers as B fragments (16 for layer 1, 64 for layer 2), so a
// tile is its loads, its products and its ReLUs; the next tile's inputs are loaded a tile ahead.
// Bound by the warp-level tensor pipe: 40 products per 16 rows, about 15 cycles each on every SM
// quarter, which is why the gain over fragments read from shared memory at every tile (460
// instructions per tile, scalar input loads) is small.  5.07M rows: 192 -> 177 us at 384 threads per
// SM (197 at 256, 195 at 512, where registers spill); 100k rows: 17 -> 13 us at 256 (15 at 384).  Only
// inputs off 16-byte alignment, of 50,000 rows or more, come here.
template <int NT>
__global__ void __launch_bounds__(NT, 1) k_mlp_fwd_bf16(const float* __restrict__ P,
                                                        const float* __restrict__ X, int64_t n,
                                                        float* __restrict__ z) {
    __shared__ __align__(16) float bias[3 * kH];   // b1, b2, w3
    for (int i = threadIdx.x; i < kH; i += NT) {
        bias[i] = P[kOffB1 + i];
        bias[kH + i] = P[kOffB2 + i];
        bias[2 * kH + i] = P[kOffW3 + i];
    }
    const float b3 = __ldg(P + kOffB3);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // B fragments: column n = 8 nt + g, rows 2t, 2t + 1 and 2t + 8, 2t + 9 of each k-tile
    uint32_t w1[8][2], w2[4][8][2];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const float* r1 = P + kOffW1 + (8 * nt + g) * kD;
        const float* r2 = P + kOffW2 + (8 * nt + g) * kH;
        w1[nt][0] = pack_bf16(__ldg(r1 + 2 * t), __ldg(r1 + 2 * t + 1));
        w1[nt][1] = t < 2 ? pack_bf16(__ldg(r1 + 2 * t + 8), __ldg(r1 + 2 * t + 9)) : 0u;
#pragma unroll
        for (int kt = 0; kt < 4; ++kt) {
            w2[kt][nt][0] = pack_bf16(__ldg(r2 + 16 * kt + 2 * t), __ldg(r2 + 16 * kt + 2 * t + 1));
            w2[kt][nt][1] = pack_bf16(__ldg(r2 + 16 * kt + 2 * t + 8), __ldg(r2 + 16 * kt + 2 * t + 9));
        }
    }
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * (NT / 32);
    const bool pair = ((uintptr_t)X & 7u) == 0;   // rows are 48 bytes: pairs of floats together
    auto load2 = [&](int64_t r, int c) {
        float2 v = make_float2(0.f, 0.f);
        if (r < n) {
            const float* x = X + r * kD + c;
            if (pair) v = __ldg(reinterpret_cast<const float2*>(x));
            else v = make_float2(__ldg(x), __ldg(x + 1));
        }
        return v;
    };
    auto load = [&](int64_t tile, float2 (&x)[4]) {
        const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
        x[0] = load2(r0, 2 * t);
        x[1] = load2(r1, 2 * t);
        x[2] = t < 2 ? load2(r0, 2 * t + 8) : make_float2(0.f, 0.f);
        x[3] = t < 2 ? load2(r1, 2 * t + 8) : make_float2(0.f, 0.f);
    };
    int64_t tile = (int64_t)blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
    float2 x[4];
    if (tile * 16 < n) load(tile, x);
    for (; tile * 16 < n; tile += stride) {
        const uint32_t a0 = pack_bf16(x[0].x, x[0].y), a1 = pack_bf16(x[1].x, x[1].y);
        const uint32_t a2 = pack_bf16(x[2].x, x[2].y), a3 = pack_bf16(x[3].x, x[3].y);
        if ((tile + stride) * 16 < n) load(tile + stride, x);
        // relu, then BF16: the C fragments of layer 1 (n-tiles 2kt, 2kt + 1) are the A fragments
        // of layer 2's k-tile kt
        uint32_t c[4][4];
#pragma unroll
        for (int kt = 0; kt < 4; ++kt) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int nt = 2 * kt + h;
                const float2 bb = *reinterpret_cast<const float2*>(bias + nt * 8 + 2 * t);
                float h1[4] = {bb.x, bb.y, bb.x, bb.y};
                mma_bf16(h1, a0, a1, a2, a3, w1[nt][0], w1[nt][1]);
                c[kt][2 * h] = pack_bf16(fmaxf(h1[0], 0.f), fmaxf(h1[1], 0.f));
                c[kt][2 * h + 1] = pack_bf16(fmaxf(h1[2], 0.f), fmaxf(h1[3], 0.f));
            }
        }
        float x0 = 0.f, x1 = 0.f;
#pragma unroll
        for (int half = 0; half < 2; ++half) {   // four n-tiles at a time: 16 accumulators, not 32
            float h2[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 bb = *reinterpret_cast<const float2*>(bias + kH + (4 * half + i) * 8 + 2 * t);
                h2[i][0] = bb.x;
                h2[i][1] = bb.y;
                h2[i][2] = bb.x;
                h2[i][3] = bb.y;
            }
#pragma unroll
            for (int kt = 0; kt < 4; ++kt)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    mma_bf16(h2[i], c[kt][0], c[kt][1], c[kt][2], c[kt][3], w2[kt][4 * half + i][0], w2[kt][4 * half + i][1]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 w = *reinterpret_cast<const float2*>(bias + 2 * kH + (4 * half + i) * 8 + 2 * t);
                x0 += w.x * fmaxf(h2[i][0], 0.f) + w.y * fmaxf(h2[i][1], 0.f);
                x1 += w.x * fmaxf(h2[i][2], 0.f) + w.y * fmaxf(h2[i][3], 0.f);
            }
        }
        x0 += __shfl_xor_sync(0xffffffffu, x0, 1);
        x0 += __shfl_xor_sync(0xffffffffu, x0, 2);
        x1 += __shfl_xor_sync(0xffffffffu, x1, 1);
        x1 += __shfl_xor_sync(0xffffffffu, x1, 2);
        if (t == 0) {
            const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
            if (r0 < n) z[r0] = x0 + b3;
            if (r1 < n) z[r1] = x1 + b3;
        }
    }
}

// The same forward with layer 2 on tcgen05 (kind::f16, FP32 accumulators in tensor memory), for large
// sets of rows.  kTcGroups warp groups of 128 threads per SM each take 128 rows at a time:
// - the rows arrive by bulk copies, kTcStages tiles ahead;
// - layer 1 stays on mma.sync: its sums, which are rounded to BF16, keep their bits.  A C fragment,
//   ReLU'd and rounded, has the layout of tcgen05.st.16x128b: it goes straight to tensor memory as
//   layer 2's A operand;
// - one thread issues b2 as a product of its own (three BF16 parts that add up to it, times ones) and the
//   four K = 16 steps of 128 x 64 x 64 into the group's 64 accumulator columns;
// - every thread reads its row's 64 sums back, relu and w3.
// While one group waits for its products the others compute.  (With h1 through shared memory its
// stores, the operand's reads and the other accesses kept the shared memory 55% busy: 132 us, 113 with
// eight groups.)  5.07M rows: 107 us; the copy time of their 264 MB is 39.  k_mlp_fwd_bf16, whose 40
// mma.sync per 16 rows bound it, 177 us.  Three or five groups, and layer 1 of the next tile computed
// while the products run, change nothing (112, 113, 107): neither latency nor issue slots (44%) but
// the pipes that the 16 mma.sync per 32 rows, ReLU and rounding share (ALU 50%, tensor 37%) are what is left.
// Waits are bounded: when one runs out the group leaves its remaining scores NaN and sets *err (host
// memory; NULL: none).
constexpr int kTcGroups = 4, kTcStages = 3, kTcRows = 128;
constexpr uint32_t kTcTile = kTcRows * kD * 4;   // bytes of a full input tile
static_assert(kTcTile % 16 == 0);
// D = FP32, A = B = BF16, B K-major, N = 64, M = 128
constexpr uint32_t kTcInstr = (1u << 4) | (1u << 7) | (1u << 10) | ((64u / 8) << 17) | ((128u / 16) << 24);

struct TcSmem {
    unsigned char w2[kH * 128];              // [n][k], swizzled
    unsigned char bias[kH * 128];            // [n][3 parts of b2, 0 ...], swizzled (16 columns are read)
    float x[kTcGroups][kTcStages][kTcRows * kD];
    float b1[kH], w3[kH];
    uint64_t full[kTcGroups][kTcStages], done[kTcGroups];
    uint32_t tmem;
};

// K-major operand, 128-byte swizzle, groups of 8 rows 1024 bytes apart
__device__ __forceinline__ uint64_t tc_desc(const void* p) {
    return (uint64_t)((smem_addr(p) & 0x3FFFFu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t acc) {
    asm volatile("{.reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;}" ::"r"(d),
                 "r"(a), "l"(b), "r"(kTcInstr), "r"(acc)
                 : "memory");
}
// 16 rows x 64 BF16 as pairs: c[2 j] = row lane / 4, columns 8 j + 2 (lane % 4) and the next, c[2 j + 1] the
// same of row lane / 4 + 8
__device__ __forceinline__ void tc_store_frag(uint32_t t, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(t),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// 16 of a row's sums; the wait in the same statement, so that the registers are not read before it
__device__ __forceinline__ void tc_load16(uint32_t t, float (&v)[16]) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(t)
        : "memory");
}
// two products at once: acc += a * b on both halves
__device__ __forceinline__ void fma2(unsigned long long& acc, float a0, float a1, unsigned long long b) {
    asm("{.reg .b64 a; mov.b64 a, {%1, %2}; fma.rn.f32x2 %0, a, %3, %0;}" : "+l"(acc) : "f"(a0), "f"(a1), "l"(b));
}
// relu of two BF16 values (of a pair with a NaN, 0 for it, as fmaxf)
__device__ __forceinline__ uint32_t relu2(uint32_t v) {
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0u));
    return r;
}
// element (row, k) of a swizzled operand of 64 columns
__device__ __forceinline__ __nv_bfloat16* tc_at(unsigned char* p, int row, int k) {
    return reinterpret_cast<__nv_bfloat16*>(p + row * 128 + ((((k >> 3) ^ row) & 7) << 4) + 2 * (k & 7));
}

__global__ void __launch_bounds__(128 * kTcGroups, 1) k_mlp_fwd_tc(const float* __restrict__ P, const float* __restrict__ X,
                                                                  int64_t n, float* __restrict__ z,
                                                                  volatile unsigned* err, int test) {
    constexpr int G = kTcGroups, ST = kTcStages, NT = 128 * G;
    // tensor memory columns: the accumulators, h1 (two values per column) and the ones
    constexpr uint32_t kAcc = 0, kH1 = 64 * G, kOnes = 96 * G, kCols = 512;
    static_assert(kOnes + 8 <= kCols);
    extern __shared__ unsigned char tc_raw[];
    TcSmem& S = *reinterpret_cast<TcSmem*>(tc_raw + ((1024u - (smem_addr(tc_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, wg = tid >> 7, wt = tid & 127, warp = wt >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int64_t tiles = (n + kTcRows - 1) / kTcRows, stride = (int64_t)gridDim.x * G;
    const int64_t tile0 = (int64_t)blockIdx.x * G + wg;
    auto fetch = [&](int64_t tile, int st) {   // one thread
        const uint32_t rows = (uint32_t)min((int64_t)kTcRows, n - tile * kTcRows);
        bulk_g2s(S.x[wg][st], X + tile * kTcRows * kD, rows * kD * 4, &S.full[wg][st]);
    };
    if (wt == 0) {
        for (int i = 0; i < ST; ++i) mbar_init(&S.full[wg][i], 1);
        mbar_init(&S.done[wg], 1);
        fence_mbar_init();
        // tests only: one group also waits for bytes that no copy brings
        if (test && tid == 0 && blockIdx.x == 0) asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], 16;" ::"r"(smem_addr(&S.full[0][0])) : "memory");
        for (int i = 0; i < ST; ++i)
            if (tile0 + i * stride < tiles) fetch(tile0 + i * stride, i);
    }
    __syncwarp();
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&S.tmem)), "r"(kCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < kH * kH; i += NT) *tc_at(S.w2, i >> 6, i & 63) = __float2bfloat16_rn(__ldg(P + kOffW2 + i));
    for (int i = tid; i < kH * 16; i += NT) {
        const int c = i >> 4, k = i & 15;
        const float b = __ldg(P + kOffB2 + c);
        const __nv_bfloat16 hi = __float2bfloat16_rz(b);
        __nv_bfloat16 v = k == 0 ? hi : __float2bfloat16_rn(0.f);
        if (k == 1 || k == 2) {
            const float r = isfinite(b) ? b - __bfloat162float(hi) : 0.f;
            const __nv_bfloat16 mid = __float2bfloat16_rz(r);
            v = k == 1 ? mid : __float2bfloat16_rn(r - __bfloat162float(mid));
        }
        *tc_at(S.bias, c, k) = v;
    }
    if (tid < kH) {
        S.b1[tid] = __ldg(P + kOffB1 + tid);
        S.w3[tid] = __ldg(P + kOffW3 + tid);
    }
    const float b3 = __ldg(P + kOffB3);
    // B fragments of layer 1, as in k_mlp_fwd_bf16
    uint32_t w1[8][2];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const float* r1 = P + kOffW1 + (8 * nt + g) * kD;
        w1[nt][0] = pack_bf16(__ldg(r1 + 2 * t), __ldg(r1 + 2 * t + 1));
        w1[nt][1] = t < 2 ? pack_bf16(__ldg(r1 + 2 * t + 8), __ldg(r1 + 2 * t + 9)) : 0u;
    }
    fence_proxy_async();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = *(volatile uint32_t*)&S.tmem, lanes = (uint32_t)(32 * warp) << 16;
    if (wg == 0) {   // rows {1, 1, 1, 0 ...}
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %3, %3, %3, %3, %3};" ::"r"(tm + lanes + kOnes),
                     "r"(0x3F803F80u), "r"(0x00003F80u), "r"(0u)
                     : "memory");
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t acc_t = tm + kAcc + 64u * (uint32_t)wg, h1_t = tm + kH1 + 32u * (uint32_t)wg;
    const uint64_t db = tc_desc(S.w2), dbias = tc_desc(S.bias);
    bool ok = true;
    uint32_t phase = 0, par = 0;
    int st = 0;
    int64_t tile = tile0;
    for (; tile < tiles; tile += stride) {
        uint32_t c[2][16];
        if (!mbar_wait(&S.full[wg][st], par)) ok = false;
        const float* xs = S.x[wg][st] + (32 * warp + g) * kD + 2 * t;
        if (++st == ST) {
            st = 0;
            par ^= 1u;
        }
        uint32_t a[2][4];
#pragma unroll
        for (int sub = 0; sub < 2; ++sub) {
            auto two = [&](int off) {
                const float2 v = *reinterpret_cast<const float2*>(xs + 16 * sub * kD + off);
                return pack_bf16(v.x, v.y);
            };
            a[sub][0] = two(0);
            a[sub][1] = two(8 * kD);
            a[sub][2] = t < 2 ? two(8) : 0u;
            a[sub][3] = t < 2 ? two(8 * kD + 8) : 0u;
        }
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const float2 bb = *reinterpret_cast<const float2*>(S.b1 + nt * 8 + 2 * t);
#pragma unroll
            for (int sub = 0; sub < 2; ++sub) {
                float v[4] = {bb.x, bb.y, bb.x, bb.y};
                mma_bf16(v, a[sub][0], a[sub][1], a[sub][2], a[sub][3], w1[nt][0], w1[nt][1]);
                c[sub][2 * nt] = relu2(pack_bf16(v[0], v[1]));
                c[sub][2 * nt + 1] = relu2(pack_bf16(v[2], v[3]));
            }
        }
        __syncwarp();
        tc_store_frag(h1_t + lanes, c[0]);
        tc_store_frag(h1_t + lanes + (16u << 16), c[1]);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        // the group's threads have read the inputs and the sums of the tile before, and written h1
        uint32_t all;
        asm volatile("{.reg .pred p, q; setp.ne.b32 p, %1, 0; bar.red.and.pred q, %2, 128, p; selp.u32 %0, 1, 0, q;}"
                     : "=r"(all)
                     : "r"(ok ? 1u : 0u), "r"(wg + 1)
                     : "memory");
        if (!all) {
            ok = false;
            break;
        }
        if (wt == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            tc_mma(acc_t, tm + kOnes, dbias, 0u);
#pragma unroll
            for (int k = 0; k < 4; ++k) tc_mma(acc_t, h1_t + 8u * k, db + 2u * k, 1u);   // 16 columns of B: 32 bytes
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(&S.done[wg])) : "memory");
            if (tile + ST * stride < tiles) fetch(tile + ST * stride, st == 0 ? ST - 1 : st - 1);
        }
        __syncwarp();
        if (!mbar_wait(&S.done[wg], phase)) ok = false;
        phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncwarp();
        unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int quart = 0; quart < 4; ++quart) {
            float v[16];
            tc_load16(acc_t + lanes + 16u * quart, v);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(S.w3 + 16 * quart + 4 * i);
                fma2(acc[(2 * i) & 3], fmaxf(v[4 * i], 0.f), fmaxf(v[4 * i + 1], 0.f), w.x);
                fma2(acc[(2 * i + 1) & 3], fmaxf(v[4 * i + 2], 0.f), fmaxf(v[4 * i + 3], 0.f), w.y);
            }
        }
        auto sum = [](unsigned long long q) { return __uint_as_float((uint32_t)q) + __uint_as_float((uint32_t)(q >> 32)); };
        const float s = (sum(acc[0]) + sum(acc[1])) + (sum(acc[2]) + sum(acc[3]));
        const int64_t row = tile * kTcRows + wt;
        if (row < n) z[row] = ok ? s + b3 : __int_as_float(0x7fffffff);
    }
    if (!ok) {   // a wait ran out: no scores, and the copies in flight end before their memory is given up
        for (int64_t k = tile; k < tiles; k += stride)
            if (k * kTcRows + wt < n) z[k * kTcRows + wt] = __int_as_float(0x7fffffff);
        if (wt == 0) {
            for (int i = 0; i < ST; ++i) {
                mbar_wait(&S.full[wg][i], 0);
                mbar_wait(&S.full[wg][i], 1);
            }
            if (err) {
                *err = 1u;
                __threadfence_system();
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(kCols) : "memory");
}

// Fused inference for one mesh, one launch: features -> BF16 MLP -> score z_j + base_j, the
// per-block maxima of the score (with its row), of K_jj and of the Gershgorin row bound; the
// last block to finish (counter in the work space) reduces the block partials and computes the
// Rayleigh quotient lower bound near the argmax triangle.  Each warp takes 32 triangles at a
// time: every lane builds one triangle's features in shared memory, then the warp runs the
// tensor-core layers of k_mlp_fwd_bf16 on the two 16-row halves.  No feature array is written.
constexpr int kInferWarps = 4, kInferThreads = 32 * kInferWarps;
constexpr int kRing = 6, kLoc = 256;

struct InferSmem {
    PackedNet net;
    float feat[kInferWarps][32][kD + 1];
};
static_assert(offsetof(InferSmem, feat) == sizeof(PackedNet), "packed net leads the block's smem");
constexpr int kHash = 1024;      // open-addressing table of the neighbourhood, > 4 kLoc slots
struct RqSmem {
    int32_t ids[kLoc];          // triangles of rings 0..6 around the argmax, ring by ring
    int32_t hkey[kHash];        // triangle id, -1 empty
    int32_t hval[kHash];        // local index of the member holding the key
    int32_t nbq[kLoc][3];       // triangle across each edge (-1 boundary); later its local
                                // index (-1 outside the set)
    int32_t kq[kLoc][3];        // interior edge index of each edge (>= n_ei: boundary)
    float a[kLoc][3];           // |e| / (d S_i) of each interior edge (K's off-diagonal weight)
    float sv[kLoc], v[kLoc], kv[kLoc];
};
union RhoSmem {
    InferSmem a;
    RqSmem b;
};

struct RhoPart {
    float best;
    int32_t arg;
    float kmax, gmax;
};

// max of the score, ties to the smaller row (rows < 0 are empty)
__device__ __forceinline__ void better(float& b, int32_t& a, float ob, int32_t oa) {
    if (oa >= 0 && (a < 0 || ob > b || (ob == b && oa < a))) {
        b = ob;
        a = oa;
    }
}

__device__ __forceinline__ uint32_t hash_slot(int32_t key) {
    return ((uint32_t)key * 2654435761u) >> 22;   // 10 bits: kHash = 1024
}

// slot holding key (inserted if absent), -1 when the table is full
__device__ __forceinline__ int hash_insert(RqSmem& R, int32_t key) {
    uint32_t h = hash_slot(key);
    for (int p = 0; p < kHash; ++p, h = (h + 1) & (kHash - 1)) {
        const int32_t prev = atomicCAS(&R.hkey[h], -1, key);
        if (prev == -1 || prev == key) return (int)h;
    }
    return -1;
}

__device__ __forceinline__ int hash_find(const RqSmem& R, int32_t key) {
    uint32_t h = hash_slot(key);
    for (int p = 0; p < kHash; ++p, h = (h + 1) & (kHash - 1)) {
        const int32_t k = R.hkey[h];
        if (k == key) return (int)h;
        if (k == -1) return -1;
    }
    return -1;
}

// Slack of the local Rayleigh quotient.  Any vector's quotient lower-bounds lambda_max(K), so
// the rounding of the five FP32 power steps costs only accuracy; what must be bounded is the
// rounding of <v, K v>_S and <v, v>_S for the computed v.  Three FMAs per entry of K v and
// sums of at most kLoc terms in a tree of depth <= 11 give a relative error below
// 30 * 2^-24 * G / RQ, where G >= lambda_max is the Gershgorin bound.  Scaling by 1 - 2^-12
// covers that while G / RQ <= 100; beyond, the quotient is dropped.
constexpr double kRqSlack = 1.0 / 4096.0;
constexpr double kRqMaxRatio = 100.0;

// <v, K v>_S / <v, v>_S of v = K^5 delta_j0, on the rings 0..6 around j0 (exact there: K
// couples edge neighbours only, so K^5 delta_j0 lives on rings 0..5).  Returns 0 when the
// neighbourhood exceeds kLoc triangles.
// Warp 0 walks the rings breadth first, without block barriers.  The candidates of a ring are
// the table rows of its members; their own rows are loaded as soon as they are named, so the
// deduplication (__match_any_sync keeps the first lane of equal candidates, the shared hash
// drops members already in the set) runs under the load latency.  The local order (first
// naming in candidate order, hence the rounding of the sums) does not depend on timing.  Then
// all threads form K's weights and apply the scaled operator c K (c = 1/K_j0j0, so that FP32
// does not overflow over five powers) six times.  Returns the value on every thread.
__device__ float local_rayleigh(RqSmem& R, const int32_t* __restrict__ code,
                                const int32_t* __restrict__ tnb, const double* __restrict__ elen,
                                const double* __restrict__ d, const double* __restrict__ S,
                                int64_t n_ei, int32_t j0, float* red) {
    __shared__ int s_n;
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31;
    for (int i = tid; i < kHash; i += nth) R.hkey[i] = -1;
    __syncthreads();
    if (tid < 32) {
        if (lane == 0) {
            R.hval[hash_insert(R, j0)] = 0;
            R.ids[0] = j0;
            for (int q = 0; q < 3; ++q) {
                R.nbq[0][q] = tnb[3 * (int64_t)j0 + q];
                R.kq[0][q] = code[3 * (int64_t)j0 + q] >> 1;
            }
            R.sv[0] = (float)S[j0];
        }
        __syncwarp();
        int n = 1, start = 0, end = 1;
        bool over = false;
        for (int r = 1; r <= kRing && !over; ++r) {
            const int cnt = 3 * (end - start);
            for (int c0 = 0; c0 < cnt; c0 += 32) {
                const int c = c0 + lane;
                const int32_t o = c < cnt ? R.nbq[start + c / 3][c % 3] : -1;
                int32_t t[3] = {-1, -1, -1}, kk[3] = {0, 0, 0};
                double so = 0.0;
                if (o >= 0) {   // the candidate's rows, in flight during the deduplication
                    for (int q = 0; q < 3; ++q) {
                        t[q] = tnb[3 * (int64_t)o + q];
                        kk[q] = code[3 * (int64_t)o + q];
                    }
                    so = S[o];
                }
                const unsigned same = __match_any_sync(0xffffffffu, o);
                const bool keep = o >= 0 && lane == __ffs(same) - 1 && hash_find(R, o) < 0;
                const unsigned m = __ballot_sync(0xffffffffu, keep);
                const int pos = n + __popc(m & ((1u << lane) - 1u));
                if (keep) {
                    const int h = pos < kLoc ? hash_insert(R, o) : -1;
                    if (h < 0) {
                        over = true;
                    } else {
                        R.hval[h] = pos;
                        R.ids[pos] = o;
                        for (int q = 0; q < 3; ++q) {
                            R.nbq[pos][q] = t[q];
                            R.kq[pos][q] = kk[q] >> 1;
                        }
                        R.sv[pos] = (float)so;
                    }
                }
                n += __popc(m);
                over = __any_sync(0xffffffffu, over);
                __syncwarp();
            }
            if (n >= kLoc) over = true;
            start = end;
            end = n;
        }
        if (lane == 0) s_n = over ? -1 : n;
    }
    __syncthreads();
    const int n = s_n;
    if (n < 0) return 0.f;
    // local neighbour indices and weights
    for (int e = tid; e < 3 * n; e += nth) {
        const int i = e / 3, q = e % 3;
        const int64_t k = R.kq[i][q];
        int loc = -1;
        float w = 0.f;
        if (k < n_ei) {
            const int h = hash_find(R, R.nbq[i][q]);
            if (h >= 0) loc = R.hval[h];
            w = __fdividef((float)elen[k], (float)d[k] * R.sv[i]);
        }
        R.nbq[i][q] = loc;
        R.a[i][q] = w;
    }
    for (int i = tid; i < n; i += nth) R.v[i] = i == 0 ? 1.f : 0.f;
    __syncthreads();
    const float kjj = R.a[0][0] + R.a[0][1] + R.a[0][2];
    if (!(kjj > 0.f)) return 0.f;
    const float c = 1.f / kjj;
    // (c K v)_i = c sum_q a_iq (v_i - v_nbr), a neighbour outside the set holding 0; six
    // products, ping-ponging between v and kv, leave (cK)^5 delta in kv and (cK)^6 delta in v
    float* va = R.v;
    float* vb = R.kv;
    for (int it = 0; it < 6; ++it) {
        for (int i = tid; i < n; i += nth) {
            const float vi = va[i];
            float acc = 0.f;
            for (int q = 0; q < 3; ++q) {
                const int nb = R.nbq[i][q];
                acc = fmaf(R.a[i][q], vi - (nb >= 0 ? va[nb] : 0.f), acc);
            }
            vb[i] = acc * c;
        }
        __syncthreads();
        float* t = va;
        va = vb;
        vb = t;
    }
    float num = 0.f, den = 0.f;
    for (int i = tid; i < n; i += nth) {
        num += R.sv[i] * R.kv[i] * R.v[i];
        den += R.sv[i] * R.kv[i] * R.kv[i];
    }
    for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if (lane == 0) {
        red[2 * (tid >> 5)] = num;
        red[2 * (tid >> 5) + 1] = den;
    }
    __syncthreads();
    num = den = 0.f;
    for (int w = 0; w < (nth >> 5); ++w) {
        num += red[2 * w];
        den += red[2 * w + 1];
    }
    return den > 0.f ? num / (den * c) : 0.f;
}

// Resident state of the fused inference (no allocation per call): the parameters, their packed
// form, the block partials and the completion counter (zero between launches; the last block
// resets it).
constexpr int kInferMaxBlocks = 152 * 6;
__device__ float g_rho_params[kNParams];
__device__ __align__(128) PackedNet g_rho_packed;
__device__ RhoPart g_rho_parts[kInferMaxBlocks];
__device__ unsigned int g_rho_counter;

// out = {log rho_hat, row, max K_jj (rounded down), max Gershgorin (rounded up), Rayleigh
// quotient}; host-mapped memory in the library's use, any device-visible buffer works.
__global__ void __launch_bounds__(kInferThreads, 6) k_rho_infer(
    const double* __restrict__ xy, const int32_t* __restrict__ tn,
    const int32_t* __restrict__ code, const int32_t* __restrict__ tnb, const double* __restrict__ elen,
    const double* __restrict__ d, const double* __restrict__ S, int64_t n, int64_t n_ei,
    double* __restrict__ out, unsigned long long seq) {
    __shared__ __align__(128) RhoSmem sm;
    __shared__ __align__(8) uint64_t net_bar;
    __shared__ RhoPart red[kInferWarps];
    __shared__ float dred[2 * kInferWarps];
    __shared__ int s_last;
    InferSmem& A = sm.a;
    unsigned int* counter = &g_rho_counter;
    RhoPart* part = g_rho_parts;
    // the packed network arrives by one bulk copy while the first features are gathered
    if (threadIdx.x == 0) {
        mbar_init(&net_bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) bulk_g2s(&A.net, &g_rho_packed, (uint32_t)sizeof(PackedNet), &net_bar);
    bool net_ready = false;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    float (*F)[kD + 1] = A.feat[warp];
    float best = -INFINITY, kmax = 0.f, gmax = 0.f;
    int32_t arg = -1;
    const int64_t warps = (int64_t)gridDim.x * kInferWarps;
    for (int64_t tile = (int64_t)blockIdx.x * kInferWarps + warp; tile * 32 < n; tile += warps) {
        const int64_t j = tile * 32 + lane;
        if (j < n) {
            float kd, ge;
            triangle_features(xy, tn, code, tnb, elen, d, S, j, n_ei, F[lane], kd, ge);
            kmax = fmaxf(kmax, kd);
            gmax = fmaxf(gmax, ge);
        } else {
            for (int i = 0; i < kD; ++i) F[lane][i] = 0.f;
            F[lane][kD] = -1e30f;
        }
        __syncwarp();
        if (!net_ready) net_ready = mbar_wait(&net_bar, 0);
        const float b3 = A.net.b3[0];
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            const float* x0 = F[16 * half + g];
            const float* x1 = F[16 * half + g + 8];
            auto xv = [&](const float* x, int c) { return c < kD ? x[c] : 0.f; };
            const uint32_t a0 = pack_bf16(xv(x0, 2 * t), xv(x0, 2 * t + 1));
            const uint32_t a1 = pack_bf16(xv(x1, 2 * t), xv(x1, 2 * t + 1));
            const uint32_t a2 = pack_bf16(xv(x0, 2 * t + 8), xv(x0, 2 * t + 9));
            const uint32_t a3 = pack_bf16(xv(x1, 2 * t + 8), xv(x1, 2 * t + 9));
            float s0, s1;
            mlp16(A.net, a0, a1, a2, a3, s0, s1);
            if (t == 0) {
                const int64_t r0 = tile * 32 + 16 * half + g, r1 = r0 + 8;
                if (r0 < n) better(best, arg, s0 + b3 + x0[kD], (int32_t)r0);
                if (r1 < n) better(best, arg, s1 + b3 + x1[kD], (int32_t)r1);
            }
        }
        __syncwarp();
    }
    // no thread leaves (and no smem is reused) while the copy may still be writing
    if (!net_ready) net_ready = mbar_wait(&net_bar, 0);
    if (!net_ready) best = NAN;   // the wait ran out: poison the prediction (power iteration)
    for (int o = 16; o > 0; o >>= 1) {
        better(best, arg, __shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, arg, o));
        kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
        gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    }
    if (lane == 0) red[warp] = RhoPart{best, arg, kmax, gmax};
    __syncthreads();
    if (threadIdx.x == 0) {
        RhoPart r = red[0];
        for (int w = 1; w < kInferWarps; ++w) {
            better(r.best, r.arg, red[w].best, red[w].arg);
            r.kmax = fmaxf(r.kmax, red[w].kmax);
            r.gmax = fmaxf(r.gmax, red[w].gmax);
        }
        part[blockIdx.x] = r;
        __threadfence();
        s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    // last block: every other block's partial is visible (fence before its counter update)
    __threadfence();
    best = -INFINITY;
    arg = -1;
    kmax = gmax = 0.f;
    // all of a thread's partials in flight at once (at most kInferMaxBlocks / kInferThreads)
    constexpr int kPer = (kInferMaxBlocks + kInferThreads - 1) / kInferThreads;
    float4 q[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = threadIdx.x + u * kInferThreads;
        q[u] = i < (int)gridDim.x ? __ldcg(reinterpret_cast<const float4*>(part + i))
                                  : make_float4(-INFINITY, __int_as_float(-1), 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        better(best, arg, q[u].x, __float_as_int(q[u].y));
        kmax = fmaxf(kmax, q[u].z);
        gmax = fmaxf(gmax, q[u].w);
    }
    for (int o = 16; o > 0; o >>= 1) {
        better(best, arg, __shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, arg, o));
        kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
        gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
    }
    __syncthreads();
    if (lane == 0) red[warp] = RhoPart{best, arg, kmax, gmax};
    __syncthreads();
    RhoPart r = red[0];
    for (int w = 1; w < kInferWarps; ++w) {
        better(r.best, r.arg, red[w].best, red[w].arg);
        r.kmax = fmaxf(r.kmax, red[w].kmax);
        r.gmax = fmaxf(r.gmax, red[w].gmax);
    }
    double rq = r.arg >= 0 ? (double)local_rayleigh(sm.b, code, tnb, elen, d, S, n_ei, r.arg, dred) : 0.0;
    rq = rq > 0.0 && (double)r.gmax <= kRqMaxRatio * rq ? rq * (1.0 - kRqSlack) : 0.0;
    if (threadIdx.x == 0) {
        *counter = 0u;
        out[0] = (double)r.best;
        out[1] = (double)r.arg;
        out[2] = (double)r.kmax * (1.0 - kBracketSlack);
        out[3] = (double)r.gmax * (1.0 + kBracketSlack);
        out[4] = rq;
        // completion word last: the host may read out[0..4] once it sees seq
        __threadfence_system();
        reinterpret_cast<volatile unsigned long long*>(out)[5] = seq;
    }
}

// FP32 debug forward: one thread per row, CUDA cores.
__global__ void k_mlp_fwd_f32(const float* __restrict__ P, const float* __restrict__ X, int64_t n,
                              float* __restrict__ z) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    float x[kD], h1[kH];
    for (int i = 0; i < kD; ++i) x[i] = X[r * kD + i];
    for (int o = 0; o < kH; ++o) {
        float a = P[kOffB1 + o];
        for (int i = 0; i < kD; ++i) a = fmaf(P[kOffW1 + o * kD + i], x[i], a);
        h1[o] = fmaxf(a, 0.f);
    }
    float s = P[kOffB3];
    for (int o = 0; o < kH; ++o) {
        float a = P[kOffB2 + o];
        for (int i = 0; i < kH; ++i) a = fmaf(P[kOffW2 + o * kH + i], h1[i], a);
        s = fmaf(P[kOffW3 + o], fmaxf(a, 0.f), s);
    }
    z[r] = s;
}

// ---------------------------------------------------------------------------------------
// backward for selected rows, summed over the rows in an order that does not change.
// bf16 = 1 repeats the forward's BF16 rounding of x, W1, W2 and h1.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float rb(float x, int bf16) {
    return bf16 ? __bfloat162float(__float2bfloat16_rn(x)) : x;
}

// A block keeps the network in shared memory and its share of the gradient in registers (16 + 3
// weights per thread and its unit's biases) over its rows, four rows at a time: 64 threads, one per
// hidden unit, take a row forward and back, then all 256 add the four outer products.  One sum per
// block is written; with one gradient row per mesh row (20 KB) the sum over them read it all
// again, one thread per parameter in a row: 37 us together on 400 rows, milliseconds on 20,000, against
// 13 here on 400 rows (bound by the latency of the weights and of a row's chain of sums).  Up to four rows
// are one block, which writes the gradient itself: 8.2 us for a row, 14.4 with the sum over blocks and the
// weights loaded as they were stored.
constexpr int kBwdRows = 4, kBwdThreads = kH * kBwdRows, kW2P = kH + 1;   // padded row: no bank conflicts
__global__ void __launch_bounds__(kBwdThreads) k_mlp_bwd(const float* __restrict__ P, const float* __restrict__ X,
                                                         const int64_t* __restrict__ rows, const float* __restrict__ dz,
                                                         int64_t m, int bf16, float* __restrict__ part) {
    __shared__ float w1[kH * (kD + 1)], w2[kH * kW2P], b1[kH], b2[kH], w3[kH];
    __shared__ float x[kBwdRows][kD], h1[kBwdRows][kH], h2[kBwdRows][kH], d1[kBwdRows][kH], d2[kBwdRows][kH], dzr[kBwdRows];
    const int tid = threadIdx.x, o = tid & (kH - 1), p = tid / kH;   // hidden unit, row of the group
    // all of a thread's weights in flight at once: a call on few rows is this latency and a row's
    float v1[kH * kD / kBwdThreads], v2[kH * kH / kBwdThreads];
#pragma unroll
    for (int u = 0; u < kH * kD / kBwdThreads; ++u) v1[u] = __ldg(P + kOffW1 + tid + u * kBwdThreads);
#pragma unroll
    for (int u = 0; u < kH * kH / kBwdThreads; ++u) v2[u] = __ldg(P + kOffW2 + tid + u * kBwdThreads);
#pragma unroll
    for (int u = 0; u < kH * kD / kBwdThreads; ++u) {
        const int i = tid + u * kBwdThreads;
        w1[(i / kD) * (kD + 1) + i % kD] = rb(v1[u], bf16);
    }
#pragma unroll
    for (int u = 0; u < kH * kH / kBwdThreads; ++u) {
        const int i = tid + u * kBwdThreads;
        w2[(i / kH) * kW2P + i % kH] = rb(v2[u], bf16);
    }
    if (tid < kH) {
        b1[tid] = P[kOffB1 + tid];
        b2[tid] = P[kOffB2 + tid];
        w3[tid] = P[kOffW3 + tid];
    }
    float gw2[kH / kBwdRows] = {}, gw1[kD / kBwdRows] = {}, gb1 = 0.f, gb2 = 0.f, gw3 = 0.f, gb3 = 0.f;
    for (int64_t i0 = (int64_t)blockIdx.x * kBwdRows; i0 < m; i0 += (int64_t)gridDim.x * kBwdRows) {
        const int64_t i = i0 + p;
        const int64_t r = i < m ? rows[i] : -1;   // -1: an empty segment's row adds nothing
        __syncthreads();
        if (o < kD) x[p][o] = r >= 0 ? rb(X[r * kD + o], bf16) : 0.f;
        if (o == 0) dzr[p] = r >= 0 ? dz[i] : 0.f;
        __syncthreads();
        float a1 = b1[o];
        for (int k = 0; k < kD; ++k) a1 += w1[o * (kD + 1) + k] * x[p][k];
        h1[p][o] = rb(fmaxf(a1, 0.f), bf16);
        __syncthreads();
        float a2 = b2[o];
#pragma unroll 16
        for (int k = 0; k < kH; ++k) a2 += w2[o * kW2P + k] * h1[p][k];
        const float g = dzr[p];
        h2[p][o] = g * fmaxf(a2, 0.f);
        d2[p][o] = a2 > 0.f ? g * w3[o] : 0.f;
        __syncthreads();
        float s = 0.f;
#pragma unroll 16
        for (int k = 0; k < kH; ++k) s += d2[p][k] * w2[k * kW2P + o];
        d1[p][o] = a1 > 0.f ? s : 0.f;
        __syncthreads();
        for (int q = 0; q < kBwdRows; ++q) {
            const float e2 = d2[q][o], e1 = d1[q][o];
#pragma unroll
            for (int k = 0; k < kH / kBwdRows; ++k) gw2[k] += e2 * h1[q][p * (kH / kBwdRows) + k];
#pragma unroll
            for (int k = 0; k < kD / kBwdRows; ++k) gw1[k] += e1 * x[q][p * (kD / kBwdRows) + k];
            if (p == 0) {
                gb1 += e1;
                gb2 += e2;
                gw3 += h2[q][o];
                if (o == 0) gb3 += dzr[q];
            }
        }
    }
    float* G = part + (int64_t)blockIdx.x * kNParams;
#pragma unroll
    for (int k = 0; k < kH / kBwdRows; ++k) G[kOffW2 + o * kH + p * (kH / kBwdRows) + k] = gw2[k];
#pragma unroll
    for (int k = 0; k < kD / kBwdRows; ++k) G[kOffW1 + o * kD + p * (kD / kBwdRows) + k] = gw1[k];
    if (p == 0) {
        G[kOffB1 + o] = gb1;
        G[kOffB2 + o] = gb2;
        G[kOffW3 + o] = gw3;
        if (o == 0) G[kOffB3] = gb3;
    }
}

// grad[p] = sum of the blocks' shares: 64 parameters and 16 slices of the blocks per block
constexpr int kSumParams = 64, kSumSlices = 16;
__global__ void __launch_bounds__(kSumParams * kSumSlices) k_colsum(const float* __restrict__ G, int nb,
                                                                    float* __restrict__ g) {
    __shared__ float red[kSumSlices][kSumParams];
    const int c = threadIdx.x & (kSumParams - 1), q = threadIdx.x / kSumParams;
    const int p = blockIdx.x * kSumParams + c;
    float s = 0.f;
    if (p < kNParams) {
#pragma unroll 4
        for (int i = q; i < nb; i += kSumSlices) s += G[(int64_t)i * kNParams + p];
    }
    red[q][c] = s;
    __syncthreads();
    if (q == 0 && p < kNParams) {
        for (int i = 1; i < kSumSlices; ++i) s += red[i][c];
        g[p] = s;
    }
}

// Adam (Kingma & Ba 2015) with bias correction.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float mi = b1 * m[i] + (1.f - b1) * g[i];
    const float vi = b2 * v[i] + (1.f - b2) * g[i] * g[i];
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Per segment (mesh): best = max_j (z_j + base_j) and its row (first on ties).  NT threads per segment,
// eight rows per thread in flight (one at a time in blocks of 256, 400 segments of up to 50k rows took twice
// as long).  Blocks hold 256 threads at least, several segments when NT is less.
constexpr int kArgRows = 8;
template <int NT>
__global__ void __launch_bounds__(NT < 256 ? 256 : NT) k_seg_argmax(const float* __restrict__ z, const float* __restrict__ base,
                                                                    const int64_t* __restrict__ off, int n_seg,
                                                                    float* __restrict__ best, int64_t* __restrict__ arg) {
    constexpr int PER = NT < 256 ? 256 / NT : 1, W = NT / 32;   // segments per block, warps per segment
    const int s = blockIdx.x * PER + threadIdx.x / NT, tid = threadIdx.x % NT;
    __shared__ float bv[PER][W];
    __shared__ int64_t bi[PER][W];
    float v = -INFINITY;
    int64_t a = -1;
    const int64_t end = s < n_seg ? off[s + 1] : 0;
    for (int64_t j0 = s < n_seg ? off[s] + tid : 0; j0 < end; j0 += NT * kArgRows) {
        float x[kArgRows], b[kArgRows];
#pragma unroll
        for (int u = 0; u < kArgRows; ++u) {
            const int64_t j = j0 + u * NT;
            x[u] = j < end ? __ldg(z + j) : 0.f;
            b[u] = j < end ? __ldg(base + j) : -INFINITY;
        }
#pragma unroll
        for (int u = 0; u < kArgRows; ++u) {
            const float t = x[u] + b[u];
            if (t > v) {
                v = t;
                a = j0 + u * NT;
            }
        }
    }
    auto take = [&](float w, int64_t wi) {
        if (w > v || (w == v && wi >= 0 && (a < 0 || wi < a))) {
            v = w;
            a = wi;
        }
    };
    auto lanes = [&](int n) {
        for (int o = n / 2; o > 0; o >>= 1) {
            const float w = __shfl_xor_sync(0xffffffffu, v, o);
            const int64_t wi = __shfl_xor_sync(0xffffffffu, (long long)a, o);
            take(w, wi);
        }
    };
    lanes(32);
    if constexpr (W > 1) {
        if ((tid & 31) == 0) {
            bv[threadIdx.x / NT][tid >> 5] = v;
            bi[threadIdx.x / NT][tid >> 5] = a;
        }
        __syncthreads();
        if (tid < 32) {   // W values in every group of W lanes
            v = bv[threadIdx.x / NT][tid % W];
            a = bi[threadIdx.x / NT][tid % W];
            lanes(W);
        }
    }
    if (tid == 0 && s < n_seg) {
        best[s] = v;
        arg[s] = a;
    }
}

// Loss per mesh (best - target)^2 and dL/dz of its argmax row: 2 (best - target).
__global__ void k_rho_loss(const float* __restrict__ best, const float* __restrict__ target,
                           int n_seg, float* __restrict__ dz, float* __restrict__ loss) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_seg) return;
    const float r = best[s] - target[s];
    dz[s] = 2.f * r;
    loss[s] = r * r;
}

}  // namespace

int mlp_n_params() { return kNParams; }

cudaError_t launch_features(const double* xy, const int32_t* tri_nodes, const int32_t* tri_code,
                            const int32_t* tri_nb, const double* elen, const double* d, const double* S,
                            int64_t n_t, int64_t n_ei, float* X, float* base, cudaStream_t s) {
    if (n_t <= 0) return cudaSuccess;
    k_features<<<(unsigned)((n_t + 255) / 256), 256, 0, s>>>(xy, tri_nodes, tri_code, tri_nb, elen, d, S,
                                                             n_t, n_ei, X, base);
    return cudaGetLastError();
}

// Whether the forward on n rows takes the kernel with bounded waits.
bool mlp_forward_waits(const float* X, int64_t n, int bf16) { return bf16 && n >= 32768 && ((uintptr_t)X & 15u) == 0; }

cudaError_t launch_mlp_forward(const float* P, const float* X, int64_t n, int bf16, float* z, unsigned* err,
                               bool test, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (bf16) {
        const int64_t tiles = (n + 15) / 16;
        auto grid = [&](int nt) { return (unsigned)std::min<int64_t>((tiles + nt / 32 - 1) / (nt / 32), 152); };
        // From 32,768 rows of 16-byte aligned inputs layer 2 goes to tcgen05: 20k rows 9.9 us either way,
        // 40k 10.1 (10.9), 100k 10.5 (13.2), 1M 27 (45).  Inputs off that alignment keep the network in
        // registers from 50,000 rows, one block per SM: 8 warps, whose start is shorter, while a warp has
        // few tiles, else 12.  Rows in a train of calls, in shared memory against registers: 16 rows
        // 6.4 us (8.2), 20k 8.2 (10.2), 32k 8.3 (10.3), 50k 10.3 (10.3), 100k 16.4 (12.3).
        if (mlp_forward_waits(X, n, bf16)) {
            const size_t smem = sizeof(TcSmem) + 1024;   // aligned to 1024 inside
            const cudaError_t e = cudaFuncSetAttribute(k_mlp_fwd_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            const int64_t blocks = (n + kTcRows * kTcGroups - 1) / (kTcRows * kTcGroups);
            k_mlp_fwd_tc<<<(unsigned)std::min<int64_t>(blocks, 152), 128 * kTcGroups, smem, s>>>(P, X, n, z, err, test ? 1 : 0);
            return cudaGetLastError();
        }
        if (n < 50000) {
            const unsigned blocks = (unsigned)((tiles + 3) / 4);
            k_mlp_fwd_few<<<blocks, 128, 0, s>>>(P, X, n, z);
            return cudaGetLastError();
        }
        if (tiles < 152 * 8 * 32) k_mlp_fwd_bf16<256><<<grid(256), 256, 0, s>>>(P, X, n, z);
        else k_mlp_fwd_bf16<384><<<grid(384), 384, 0, s>>>(P, X, n, z);
    } else {
        k_mlp_fwd_f32<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(P, X, n, z);
    }
    return cudaGetLastError();
}

cudaError_t launch_mlp_backward(const float* P, const float* X, const int64_t* rows, const float* dz,
                                int64_t m, int bf16, float* work, float* grad, cudaStream_t s) {
    if (m <= 0) return cudaMemsetAsync(grad, 0, sizeof(float) * kNParams, s);
    // at most two blocks per SM; no more shares than the m gradient rows `work` holds
    const int64_t groups = (m + kBwdRows - 1) / kBwdRows;
    const int blocks = (int)(groups < 304 ? groups : 304);
    k_mlp_bwd<<<blocks, kBwdThreads, 0, s>>>(P, X, rows, dz, m, bf16, blocks > 1 ? work : grad);
    if (blocks > 1) k_colsum<<<(kNParams + kSumParams - 1) / kSumParams, kSumParams * kSumSlices, 0, s>>>(work, blocks, grad);
    return cudaGetLastError();
}

cudaError_t launch_adam(float* p, const float* g, float* m, float* v, int n, float lr, float b1,
                        float b2, float eps, int t, cudaStream_t s) {
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    k_adam<<<(n + 255) / 256, 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

cudaError_t launch_seg_argmax(const float* z, const float* base, const int64_t* off, int n_seg,
                              float* best, int64_t* arg, cudaStream_t s) {
    if (n_seg <= 0) return cudaSuccess;
    // As many threads per segment as let all segments run at once on 152 SMs, down to a warp: their
    // lengths are on the device only.  In a train of calls: 400 segments of 1,000 to 50,000 rows 12 us, 400
    // of 100 rows 4.2 us (6.2 with 512 threads each), 2,000 of 1,000 6.2 (16.4), 20,000 of 10 8.3 (117).
    auto run = [&](auto kern, int nt) {
        const int per = nt < 256 ? 256 / nt : 1;
        kern<<<(n_seg + per - 1) / per, nt < 256 ? 256 : nt, 0, s>>>(z, base, off, n_seg, best, arg);
    };
    if (n_seg <= 152 * 2) run(k_seg_argmax<512>, 512);
    else if (n_seg <= 152 * 4) run(k_seg_argmax<256>, 256);
    else if (n_seg <= 152 * 16) run(k_seg_argmax<128>, 128);
    else run(k_seg_argmax<32>, 32);
    return cudaGetLastError();
}

cudaError_t launch_rho_loss(const float* best, const float* target, int n_seg, float* dz,
                            float* loss, cudaStream_t s) {
    if (n_seg <= 0) return cudaSuccess;
    k_rho_loss<<<(n_seg + 255) / 256, 256, 0, s>>>(best, target, n_seg, dz, loss);
    return cudaGetLastError();
}

// g_rho_packed from g_rho_params: weights to BF16 (round to nearest even) at the padded smem
// strides, zeros in the padding.
__global__ void k_pack_net() { pack_net(g_rho_packed, g_rho_params, threadIdx.x, blockDim.x); }

// Blocks of the fused inference: enough for every warp to take one 32-triangle tile, at most
// 6 resident blocks on each of the 152 SMs.
static int rho_infer_grid(int64_t n_t) {
    const int64_t need = (n_t + kInferThreads - 1) / kInferThreads;
    return (int)(need < 1 ? 1 : need > kInferMaxBlocks ? kInferMaxBlocks : need);
}

cudaError_t rho_infer_upload(const float* P_host, cudaStream_t s) {
    cudaError_t e = cudaMemcpyToSymbolAsync(g_rho_params, P_host, sizeof(float) * kNParams, 0,
                                            cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    k_pack_net<<<1, 256, 0, s>>>();
    return cudaGetLastError();
}

cudaError_t launch_rho_infer(const double* xy, const int32_t* tri_nodes, const int32_t* tri_code,
                             const int32_t* tri_nb, const double* elen, const double* d, const double* S,
                             int64_t n_t, int64_t n_ei, double* out, unsigned long long seq,
                             cudaStream_t s) {
    k_rho_infer<<<rho_infer_grid(n_t), kInferThreads, 0, s>>>(xy, tri_nodes, tri_code, tri_nb, elen, d,
                                                             S, n_t, n_ei, out, seq);
    return cudaGetLastError();
}

}  // namespace ue
