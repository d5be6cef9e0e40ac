// The highest eigenmodes of the semi-discrete system by the "complex time" method with
// deflation (Section 2).
//
// With t -> i t the modes grow like exp(omega t), so repeated application of K = -L_E L_B to
// a vector, normalised each time, converges to the top mode; the paper finds the next modes
// the same way while keeping the ones already found from growing back.  Here the m columns of
// a block are advanced together: V <- K V, then the block is made S-orthonormal again
// (Cholesky QR: G = W^T S W = R^T R, V = W R^{-1}).  Column i is thereby kept clear of the
// directions of columns 0..i-1, which is the deflation applied to all columns at once.  Cholesky
// QR only changes the basis of the columns' span, so K V may be taken several times before it: as
// many as keep the block well conditioned (modes_run).  A final Rayleigh-Ritz step on the block (eigenvectors of V^T S K V) gives the modes.
// Everything is FP64.  Blocks of vectors are row-major [n_t][m]: a triangle's m values are
// contiguous, so each gather reads one contiguous row.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "device.cuh"

namespace ue {

namespace {

constexpr int kMdThreads = 256;

// SplitMix64 (Steele, Lea, Flood 2014), published constants.
__device__ __forceinline__ uint64_t md_splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

unsigned md_blocks(int64_t n) { return (unsigned)((n + kMdThreads - 1) / kMdThreads); }

// Records of K's rows, made once per call: the triangles across the three edges (the triangle
// itself on the boundary, with weight 0) and the weights c_q / S_j, c = |e| / d.
__global__ void k_md_prep(const int4* __restrict__ tri, const int2* __restrict__ rl,
                          const double* __restrict__ elen, const double* __restrict__ d,
                          const double* __restrict__ S, int4* __restrict__ nb, double2* __restrict__ w,
                          int64_t n_ei, int64_t n_t) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_t) return;
    const int4 t = tri[j];
    const int code[3] = {t.x, t.y, t.z};
    int o[3];
    double x[3];
    const double inv = 1.0 / S[j];
    for (int q = 0; q < 3; ++q) {
        const int64_t k = code[q] >> 1;
        o[q] = (int)j;
        x[q] = 0.0;
        if (k < n_ei) {
            const int2 r = rl[k];
            o[q] = (code[q] & 1) ? r.x : r.y;
            x[q] = elen[k] / d[k] * inv;
        }
    }
    nb[j] = make_int4(o[0], o[1], o[2], 0);
    w[2 * j] = make_double2(x[0], x[1]);
    w[2 * j + 1] = make_double2(x[2], x[0] + x[1] + x[2]);
}

// V[j][col] uniform in [-1, 1), keyed by the caller id of triangle j and the column
__global__ void k_md_init(double* __restrict__ V, const int64_t* __restrict__ perm, uint32_t seed,
                          int64_t n_t, int m) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_t * m) return;
    const int64_t j = i / m;
    const int col = (int)(i - j * m);
    const uint64_t z = md_splitmix64(((uint64_t)seed << 32) + (uint64_t)perm[j] * (uint64_t)m + (uint64_t)col);
    V[i] = (double)(z >> 11) * 0x1.0p-53 * 2.0 - 1.0;
}

// W = K V in one pass: each triangle reads its own row and its three neighbours' (a signed sum of
// edge differences c (V_R - V_L) is a sum of c (V_j - V_neighbour): both signs turn together).
// Written as two passes over edges and triangles, each product moved the block's edge values,
// 1.5 rows per triangle, out and in again: 11 + 18 us against 10 us here on 90k triangles and 16
// columns (L2-resident; FP64 issue is the bound).  threadIdx.x: pair of columns, y: row.
// CHEB: one step of the Chebyshev recurrence with it, Y1 = a (K Y - c Y) + b Y0 (Y0 may be NULL),
// the product in difference form, which keeps the small values of smooth fields; without it
// K_jj V_j - sum w V (four operations per value; FP64 is scarce), for the top of the spectrum.
template <bool CHEB>
__global__ void __launch_bounds__(kMdThreads) k_md_K(const int4* __restrict__ nb, const double2* __restrict__ w,
                                                     const double2* __restrict__ Y, const double2* __restrict__ Y0,
                                                     double2* __restrict__ out, double a, double c, double b,
                                                     int64_t n_t, int m2) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
    if (j >= n_t) return;
    const int col = threadIdx.x;
    const int4 o = __ldg(nb + j);
    const double2 w01 = __ldg(w + 2 * j), w2k = __ldg(w + 2 * j + 1);
    const double2 v = __ldg(Y + j * m2 + col);
    const double2 p = __ldg(Y + (int64_t)o.x * m2 + col), q = __ldg(Y + (int64_t)o.y * m2 + col),
                  r = __ldg(Y + (int64_t)o.z * m2 + col);
    double2 y;
    if constexpr (CHEB) {
        y.x = fma(w2k.x, v.x - r.x, fma(w01.y, v.x - q.x, w01.x * (v.x - p.x)));
        y.y = fma(w2k.x, v.y - r.y, fma(w01.y, v.y - q.y, w01.x * (v.y - p.y)));
        y.x = a * (y.x - c * v.x);
        y.y = a * (y.y - c * v.y);
        if (Y0) {
            const double2 u = __ldg(Y0 + j * m2 + col);
            y.x = fma(b, u.x, y.x);
            y.y = fma(b, u.y, y.y);
        }
    } else {
        y.x = fma(-w2k.x, r.x, fma(-w01.y, q.x, fma(-w01.x, p.x, w2k.y * v.x)));
        y.y = fma(-w2k.x, r.y, fma(-w01.y, q.y, fma(-w01.x, p.y, w2k.y * v.y)));
    }
    out[j * m2 + col] = y;
}

// Block partials of the upper triangle of G[a][b] = sum_j S_j X[j][a] Y[j][b] (a <= b; G is
// symmetric for X = Y, and for Y = K X up to rounding): rows in tiles of kMdRows staged in
// shared memory, each thread owning the pairs tid, tid + 256, ... (m <= 32: at most 3 pairs of
// the 528).  Pair p enumerates (a, b) row by row.  Narrow blocks (at most 128 pairs) split each
// tile's rows among 256 / pairs groups of threads, summed at the end in group order.
constexpr int kMdRows = 32, kMdMaxM = 32;
__global__ void __launch_bounds__(kMdThreads) k_md_gram(const double* __restrict__ S,
                                                        const double* __restrict__ X,
                                                        const double* __restrict__ Y, int64_t n_t,
                                                        int m, double* __restrict__ part) {
    __shared__ double xs[kMdRows][kMdMaxM + 1], ys[kMdRows][kMdMaxM + 1];
    const int tid = threadIdx.x, npair = m * (m + 1) / 2;
    const int groups = npair <= kMdThreads / 2 ? kMdThreads / npair : 1;
    const int grp = groups > 1 ? tid / npair : 0, first = groups > 1 ? tid - grp * npair : tid;
    int pa[3], pb[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
        int p = first + u * kMdThreads, a = 0;
        while (a < m && p >= m - a) {
            p -= m - a;
            ++a;
        }
        pa[u] = a;
        pb[u] = a + p;
    }
    double acc[3] = {0.0, 0.0, 0.0};
    for (int64_t r0 = (int64_t)blockIdx.x * kMdRows; r0 < n_t; r0 += (int64_t)gridDim.x * kMdRows) {
        const int rows = (int)(n_t - r0 < kMdRows ? n_t - r0 : kMdRows);
        __syncthreads();
        for (int e = tid; e < kMdRows * m; e += kMdThreads) {
            const int r = e / m, col = e - r * m;
            double x = 0.0, y = 0.0;
            if (r < rows) {
                const int64_t j = r0 + r;
                x = S[j] * X[j * m + col];
                y = Y[j * m + col];
            }
            xs[r][col] = x;
            ys[r][col] = y;
        }
        __syncthreads();
        if (groups > 1) {
            if (grp < groups) {
                double s = acc[0];
                for (int r = grp; r < kMdRows; r += groups) s = fma(xs[r][pa[0]], ys[r][pb[0]], s);
                acc[0] = s;
            }
        } else {
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                if (tid + u * kMdThreads < npair) {
                    const int a = pa[u], b = pb[u];
                    double s = acc[u];
                    for (int r = 0; r < kMdRows; ++r) s = fma(xs[r][a], ys[r][b], s);
                    acc[u] = s;
                }
            }
        }
    }
    if (groups > 1) {
        __syncthreads();
        double* red = &xs[0][0];   // kMdRows * (kMdMaxM + 1) >= kMdThreads values
        red[tid] = acc[0];
        __syncthreads();
        if (tid < npair) {
            double s = 0.0;
            for (int g = 0; g < groups; ++g) s += red[tid + g * npair];
            part[(int64_t)blockIdx.x * npair + tid] = s;
        }
        return;
    }
#pragma unroll
    for (int u = 0; u < 3; ++u) {
        const int p = tid + u * kMdThreads;
        if (p < npair) part[(int64_t)blockIdx.x * npair + p] = acc[u];
    }
}

// G[p] = sum over blocks of part[b][p], one warp per pair, in an order that does not change (one
// thread per pair summed 608 partials in a row: 50 us against 5)
__global__ void k_md_sum(const double* __restrict__ part, int nb, int npair, double* __restrict__ G) {
    const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (p >= npair) return;
    double s = 0.0;
#pragma unroll 4
    for (int b = lane; b < nb; b += 32) s += part[(int64_t)b * npair + p];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) G[p] = s;
}

// V[j][col] = sum_a W[j][a] T[a][col] (T is m x m, row-major; upper: T[a][col] = 0 for
// a > col).  One thread per row: the row sits in registers, T (zero-padded to MW x MW) in
// shared memory is read by every thread of a warp at the same address, and the sums are
// unrolled at compile time, so the triangle below the diagonal costs nothing.
template <int MW, bool UPPER>
__global__ void __launch_bounds__(kMdThreads) k_md_apply(const double* __restrict__ W,
                                                         const double* __restrict__ T,
                                                         double* __restrict__ V, int64_t n_t, int m) {
    __shared__ double ts[MW * MW];
    for (int e = threadIdx.x; e < MW * MW; e += blockDim.x) {
        const int r = e / MW, c = e - r * MW;
        ts[e] = (r < m && c < m) ? T[r * m + c] : 0.0;
    }
    __syncthreads();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_t) return;
    const double2* w = reinterpret_cast<const double2*>(W + j * m);   // m is even
    double x[MW];
#pragma unroll
    for (int a = 0; a < MW; a += 2) {
        const double2 v = a < m ? __ldg(w + a / 2) : make_double2(0.0, 0.0);
        x[a] = v.x;
        x[a + 1] = v.y;
    }
    double2* v = reinterpret_cast<double2*>(V + j * m);
#pragma unroll
    for (int col = 0; col < MW; col += 2) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int a = 0; a < (UPPER ? col + 1 : MW); ++a) s0 = fma(x[a], ts[a * MW + col], s0);
#pragma unroll
        for (int a = 0; a < (UPPER ? col + 2 : MW); ++a) s1 = fma(x[a], ts[a * MW + col + 1], s1);
        if (col < m) v[col / 2] = make_double2(s0, s1);
    }
}

template <bool UPPER>
void md_apply(const double* W, const double* T, double* V, int64_t n_t, int m, cudaStream_t s) {
    const unsigned g = md_blocks(n_t);
    if (m <= 8) k_md_apply<8, UPPER><<<g, kMdThreads, 0, s>>>(W, T, V, n_t, m);
    else if (m <= 16) k_md_apply<16, UPPER><<<g, kMdThreads, 0, s>>>(W, T, V, n_t, m);
    else if (m <= 24) k_md_apply<24, UPPER><<<g, kMdThreads, 0, s>>>(W, T, V, n_t, m);
    else k_md_apply<32, UPPER><<<g, kMdThreads, 0, s>>>(W, T, V, n_t, m);
}

// out[col * n_t + perm[j]] = V[j][col] for col < n_out (caller triangle order)
__global__ void k_md_scatter(const double* __restrict__ V, const int64_t* __restrict__ perm,
                             double* __restrict__ out, int64_t n_t, int m, int n_out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_t * n_out) return;
    const int col = (int)(i / n_t);
    const int64_t j = i - (int64_t)col * n_t;
    out[(int64_t)col * n_t + perm[j]] = V[j * m + col];
}

// Gershgorin bound of S^(1/2) K S^(-1/2) (the S-symmetric form of K, same eigenvalues): row j
// has K_jj = sum_q c_q / S_j and off-diagonal c_q / sqrt(S_j S_k), c = |e| / d, for the triangle k
// across interior edge q; the largest row sum bounds lambda_max from above.  Positive doubles order
// like their bit patterns, so the maximum is an integer atomic.
__global__ void k_md_gersh(const int4* __restrict__ tri, const int2* __restrict__ rl,
                           const double* __restrict__ elen, const double* __restrict__ d,
                           const double* __restrict__ S, int64_t n_t, int64_t n_ei,
                           unsigned long long* __restrict__ out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_t) return;
    const int4 q = tri[j];
    const int code[3] = {q.x, q.y, q.z};
    const double sj = S[j];
    double row = 0.0;
    for (int k = 0; k < 3; ++k) {
        const int64_t e = code[k] >> 1;
        if (e >= n_ei) continue;
        const int2 t = rl[e];
        const int64_t o = t.x == j ? t.y : t.x;
        const double c = elen[e] / d[e];
        row += c / sj + c / sqrt(sj * S[o]);
    }
    atomicMax(out, (unsigned long long)__double_as_longlong(row));
}

// ---- host: small dense algebra on m x m matrices (m <= 32) --------------------------------

// upper-triangular R with G = R^T R; false if G is not positive definite
bool cholesky_upper(const std::vector<double>& G, int m, std::vector<double>& R) {
    R.assign((size_t)m * m, 0.0);
    for (int i = 0; i < m; ++i) {
        double s = G[(size_t)i * m + i];
        for (int k = 0; k < i; ++k) s -= R[(size_t)k * m + i] * R[(size_t)k * m + i];
        if (!(s > 0.0)) return false;
        const double rii = std::sqrt(s);
        R[(size_t)i * m + i] = rii;
        for (int j = i + 1; j < m; ++j) {
            double t = 0.5 * (G[(size_t)i * m + j] + G[(size_t)j * m + i]);
            for (int k = 0; k < i; ++k) t -= R[(size_t)k * m + i] * R[(size_t)k * m + j];
            R[(size_t)i * m + j] = t / rii;
        }
    }
    return true;
}

// inverse of an upper-triangular matrix (back substitution, column by column)
void upper_inverse(const std::vector<double>& R, int m, std::vector<double>& T) {
    T.assign((size_t)m * m, 0.0);
    for (int c = 0; c < m; ++c) {
        for (int i = c; i >= 0; --i) {
            double s = i == c ? 1.0 : 0.0;
            for (int k = i + 1; k <= c; ++k) s -= R[(size_t)i * m + k] * T[(size_t)k * m + c];
            T[(size_t)i * m + c] = s / R[(size_t)i * m + i];
        }
    }
}

// eigenpairs of a symmetric matrix by cyclic Jacobi rotations: values in lam, vectors as the
// columns of Q (row-major), sorted by decreasing eigenvalue
void jacobi_eigen(std::vector<double> A, int m, std::vector<double>& lam, std::vector<double>& Q) {
    Q.assign((size_t)m * m, 0.0);
    for (int i = 0; i < m; ++i) Q[(size_t)i * m + i] = 1.0;
    for (int sweep = 0; sweep < 100; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int i = 0; i < m; ++i)
            for (int j = 0; j < m; ++j) {
                const double v = A[(size_t)i * m + j] * A[(size_t)i * m + j];
                tot += v;
                if (i != j) off += v;
            }
        if (off <= 1e-30 * tot) break;
        for (int p = 0; p < m - 1; ++p)
            for (int q = p + 1; q < m; ++q) {
                const double apq = A[(size_t)p * m + q];
                if (apq == 0.0) continue;
                const double app = A[(size_t)p * m + p], aqq = A[(size_t)q * m + q];
                const double theta = 0.5 * (aqq - app) / apq;
                const double t = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
                const double cs = 1.0 / std::sqrt(t * t + 1.0), sn = t * cs;
                for (int k = 0; k < m; ++k) {   // A <- A J (columns p, q)
                    const double akp = A[(size_t)k * m + p], akq = A[(size_t)k * m + q];
                    A[(size_t)k * m + p] = cs * akp - sn * akq;
                    A[(size_t)k * m + q] = sn * akp + cs * akq;
                }
                for (int k = 0; k < m; ++k) {   // A <- J^T A (rows p, q)
                    const double apk = A[(size_t)p * m + k], aqk = A[(size_t)q * m + k];
                    A[(size_t)p * m + k] = cs * apk - sn * aqk;
                    A[(size_t)q * m + k] = sn * apk + cs * aqk;
                }
                for (int k = 0; k < m; ++k) {   // Q <- Q J
                    const double qkp = Q[(size_t)k * m + p], qkq = Q[(size_t)k * m + q];
                    Q[(size_t)k * m + p] = cs * qkp - sn * qkq;
                    Q[(size_t)k * m + q] = sn * qkp + cs * qkq;
                }
            }
    }
    std::vector<int> ord(m);
    for (int i = 0; i < m; ++i) ord[i] = i;
    std::sort(ord.begin(), ord.end(), [&](int a, int b) { return A[(size_t)a * m + a] > A[(size_t)b * m + b]; });
    std::vector<double> Qs((size_t)m * m);
    lam.resize(m);
    for (int c = 0; c < m; ++c) {
        lam[c] = A[(size_t)ord[c] * m + ord[c]];
        for (int k = 0; k < m; ++k) Qs[(size_t)k * m + c] = Q[(size_t)k * m + ord[c]];
    }
    Q = Qs;
}

}  // namespace

namespace {

// What both iterations share: K's records, the small dense matrices and the block operations.
struct Block {
    int64_t n_t;
    int m, npair, nup, nb;
    const double* S;
    int4* onb;
    double2* w;
    double *part, *G, *T;
    cudaStream_t s;
    std::vector<double> Gu, Gh, R, Th;
    bool lost = false;

    // the work space after `bufs` blocks of n_t * m values
    Block(int64_t n_t_, int m_, const double* S_, double* work, int bufs, cudaStream_t s_)
        : n_t(n_t_), m(m_), npair(m_ * m_), nup(m_ * (m_ + 1) / 2),
          nb((int)std::min<int64_t>(152 * 4, (n_t_ + kMdRows - 1) / kMdRows)), S(S_), s(s_), Gu(nup), Gh(npair) {
        double* p = work + (int64_t)bufs * n_t * m;
        onb = reinterpret_cast<int4*>(p);
        w = reinterpret_cast<double2*>(p + 2 * n_t);
        part = p + 6 * n_t;
        G = part + (int64_t)nb * nup;
        T = G + npair;
    }
    static size_t doubles(int64_t n_t, int m, int bufs) {
        const int64_t nb = std::min<int64_t>(152 * 4, (n_t + kMdRows - 1) / kMdRows);
        return (size_t)(bufs * n_t * m + 6 * n_t + nb * (int64_t)m * (m + 1) / 2 + 2 * m * m + 8);
    }
    void prep(const int4* tri, const int2* rl, const double* elen, const double* d, int64_t n_ei) {
        k_md_prep<<<md_blocks(n_t), kMdThreads, 0, s>>>(tri, rl, elen, d, S, onb, w, n_ei, n_t);
    }
    template <bool CHEB>
    void K(const double* Y, const double* Y0, double* out, double a, double c, double b) {
        const int m2 = m / 2, rows = kMdThreads / m2;
        k_md_K<CHEB><<<(unsigned)((n_t + rows - 1) / rows), dim3(m2, rows), 0, s>>>(
            onb, w, (const double2*)Y, (const double2*)Y0, (double2*)out, a, c, b, n_t, m2);
    }
    void product(const double* X, double* Y) { K<false>(X, nullptr, Y, 0.0, 0.0, 0.0); }
    cudaError_t gram(const double* X, const double* Y) {   // Gh = X^T S Y
        k_md_gram<<<nb, kMdThreads, 0, s>>>(S, X, Y, n_t, m, part);
        k_md_sum<<<(nup + 7) / 8, 256, 0, s>>>(part, nb, nup, G);
        cudaError_t e = cudaMemcpyAsync(Gu.data(), G, sizeof(double) * nup, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
        for (int a = 0, p = 0; a < m; ++a)
            for (int b = a; b < m; ++b, ++p) Gh[(size_t)a * m + b] = Gh[(size_t)b * m + a] = Gu[p];
        return cudaSuccess;
    }
    template <bool UPPER>
    cudaError_t rotate(const double* X, const std::vector<double>& M, double* Y) {   // Y = X M
        const cudaError_t e = cudaMemcpyAsync(T, M.data(), sizeof(double) * npair, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return e;
        md_apply<UPPER>(X, T, Y, n_t, m, s);
        return cudaGetLastError();
    }
    // Y = X R^{-1}, X^T S X = R^T R; sets lost (and leaves Y) when X has lost rank
    cudaError_t orthonormalize(const double* X, double* Y) {
        const cudaError_t e = gram(X, X);
        if (e != cudaSuccess) return e;
        lost = !cholesky_upper(Gh, m, R);
        if (lost) return cudaSuccess;
        upper_inverse(R, m, Th);
        return rotate<true>(X, Th, Y);
    }
};

}  // namespace

int modes_block_size(int n_modes) { return std::min(kMdMaxM, 2 * n_modes); }

size_t modes_work_doubles(int64_t n_t, int m) { return Block::doubles(n_t, m, 3); }

// How many products K V to take before the next Cholesky QR.  It only has to come before the
// columns' norms and angles drift so far apart that forming W^T S W loses digits; the diagonal of
// R, over the `p` products that led to it, tells the drift per product.  Products until it
// reaches 100 (an error of the basis, not of its span, of 1e-12, gone at the next QR), at most 16,
// and none that could overflow the Gram matrix.  One QR per product took 150 of the 180 us of an
// iteration on 90k triangles with 16 columns; with up to 8 products an iteration takes 31 us, with up to
// 16 25 us (12 of them the product).
static int products_until_qr(const std::vector<double>& R, int m, int p) {
    constexpr double kMost = 16.0;
    double lo = R[0], hi = R[0];
    for (int i = 1; i < m; ++i) {
        lo = std::min(lo, R[(size_t)i * m + i]);
        hi = std::max(hi, R[(size_t)i * m + i]);
    }
    const double drift = std::log10(hi / lo) / p, size = std::fabs(std::log10(hi)) / p;
    const double most = std::min(drift > 0 ? 2.0 / drift : kMost, size > 0 ? 140.0 / size : kMost);
    return (int)std::max(1.0, std::min(kMost, most));
}

cudaError_t modes_run(const int2* rl, const int4* tri, const double* elen, const double* d,
                      const double* S, const int64_t* perm, int64_t n_t, int64_t n_ei, int n_modes,
                      int iters, uint32_t seed, double* work, double* omega, double* B_dev,
                      bool* lost_rank, cudaStream_t s) {
    const int m = modes_block_size(n_modes);
    Block k(n_t, m, S, work, 3, s);
    double *V = work, *W = V + n_t * m, *W2 = W + n_t * m;
    *lost_rank = false;
    cudaError_t e;
    k.prep(tri, rl, elen, d, n_ei);
    k_md_init<<<md_blocks(n_t * m), kMdThreads, 0, s>>>(V, perm, seed, n_t, m);
    // start: the random block made S-orthonormal
    if ((e = k.orthonormalize(V, W)) != cudaSuccess || (*lost_rank = k.lost)) return e;
    std::swap(V, W);
    int p = 1, last = 1;
    for (int it = 0; it < iters;) {
        p = std::min(p, iters - it);
        const double* X = V;   // V stays: a block that lost rank over p products is taken again one by one
        for (int i = 0; i < p; ++i) {
            double* Y = X == W ? W2 : W;
            k.product(X, Y);
            X = Y;
        }
        double* Y = X == W ? W2 : W;
        if ((e = k.orthonormalize(X, Y)) != cudaSuccess) return e;
        if (k.lost) {
            if (p == 1) {
                *lost_rank = true;
                return cudaSuccess;
            }
            p = 1;
            continue;
        }
        it += p;
        last = p;
        std::swap(V, Y == W ? W : W2);
        p = products_until_qr(k.R, m, p);
    }
    // After several products once more, now near identity: columns S-orthonormal to rounding for
    // Rayleigh-Ritz, as they are after one (on 2k triangles this is 20 of the 150 us of a single iteration)
    if (last > 1) {
        if ((e = k.orthonormalize(V, W)) != cudaSuccess || (*lost_rank = k.lost)) return e;
        std::swap(V, W);
    }
    // Rayleigh-Ritz: H = V^T S K V, its eigenvectors rotate V into the modes
    k.product(V, W);
    if ((e = k.gram(V, W)) != cudaSuccess) return e;
    std::vector<double> lam, Q;
    jacobi_eigen(k.Gh, m, lam, Q);
    for (int i = 0; i < n_modes; ++i) omega[i] = std::sqrt(std::max(lam[i], 0.0));
    if (B_dev) {
        if ((e = k.rotate<false>(V, Q, W)) != cudaSuccess) return e;
        k_md_scatter<<<md_blocks(n_t * n_modes), kMdThreads, 0, s>>>(W, perm, B_dev, n_t, m, n_modes);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

size_t modes_low_work_doubles(int64_t n_t, int m) { return Block::doubles(n_t, m, 4) + 8; }

// The lowest n_modes eigenpairs of K by Chebyshev-filtered subspace iteration: each outer
// iteration applies to the block the degree-`degree` Chebyshev polynomial that stays within
// [-1, 1] on [lo, hi] (hi a certified Gershgorin bound of lambda_max, lo the block's largest
// Ritz value) and grows fast below lo, then makes the block S-orthonormal (Cholesky QR) and
// rotates it by Rayleigh-Ritz.  The columns beyond n_modes guard the convergence.  Omegas
// ascending; B_dev as in modes_run.
cudaError_t modes_low_run(const int2* rl, const int4* tri, const double* elen, const double* d,
                          const double* S, const int64_t* perm, int64_t n_t, int64_t n_ei, int n_modes,
                          int iters, int degree, uint32_t seed, double* work, double* omega,
                          double* B_dev, bool* lost_rank, cudaStream_t s) {
    const int m = modes_block_size(n_modes);
    Block k(n_t, m, S, work, 4, s);
    double* buf[4];
    for (int i = 0; i < 4; ++i) buf[i] = work + (int64_t)i * n_t * m;
    unsigned long long* gmax = reinterpret_cast<unsigned long long*>(work + Block::doubles(n_t, m, 4));
    *lost_rank = false;
    cudaError_t e;
    if ((e = cudaMemsetAsync(gmax, 0, 8, s)) != cudaSuccess) return e;
    k.prep(tri, rl, elen, d, n_ei);
    k_md_gersh<<<md_blocks(n_t), kMdThreads, 0, s>>>(tri, rl, elen, d, S, n_t, n_ei, gmax);
    k_md_init<<<md_blocks(n_t * m), kMdThreads, 0, s>>>(buf[0], perm, seed, n_t, m);
    unsigned long long hb = 0;
    if ((e = cudaMemcpyAsync(&hb, gmax, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    double hi;
    std::memcpy(&hi, &hb, 8);
    hi *= 1.0 + 1e-12;
    std::vector<double> lam, Q;
    // The block is buf[v]; the recurrence and the basis changes move it among the four buffers.
    int v = 0;
    auto orthonormal = [&]() -> cudaError_t {
        const cudaError_t e2 = k.orthonormalize(buf[v], buf[(v + 1) & 3]);
        v = (v + 1) & 3;
        return e2;
    };
    // the block -> its Ritz vectors (V^T S K V diagonal), lam ascending
    auto rayleigh_ritz = [&]() -> cudaError_t {
        double* W = buf[(v + 1) & 3];
        k.K<true>(buf[v], nullptr, W, 1.0, 0.0, 0.0);   // K V, in difference form
        cudaError_t e2 = k.gram(buf[v], W);
        if (e2 != cudaSuccess) return e2;
        jacobi_eigen(k.Gh, m, lam, Q);
        std::reverse(lam.begin(), lam.end());
        for (int r = 0; r < m; ++r) std::reverse(Q.begin() + (size_t)r * m, Q.begin() + (size_t)(r + 1) * m);
        e2 = k.rotate<false>(buf[v], Q, W);
        v = (v + 1) & 3;
        return e2;
    };
    if ((e = orthonormal()) != cudaSuccess || (*lost_rank = k.lost)) return e;
    if ((e = rayleigh_ritz()) != cudaSuccess) return e;
    std::vector<double> prev(n_modes, -1.0);
    for (int it = 0; it < iters; ++it) {
        // the interval to damp: [lo, hi], lo the block's largest Ritz value (at least a small
        // fraction of hi, so that the first filters, on a random block, damp only the top)
        const double lo = std::max(lam[m - 1], 1e-3 * hi);
        const double cc = 0.5 * (hi + lo), ee = 0.5 * (hi - lo);
        // scaled three-term recurrence: T_k((x - cc)/ee) / T_k((0 - cc)/ee) (Zhou and Saad)
        const double sig1 = ee / (0.0 - cc);
        double sig = sig1;
        int yp = v, yc = (v + 1) & 3, yn = (v + 2) & 3;   // T_{k-1}, T_k, T_{k+1}
        k.K<true>(buf[yp], nullptr, buf[yc], sig1 / ee, cc, 0.0);
        for (int q = 2; q <= degree; ++q) {
            const double sn = 1.0 / (2.0 / sig1 - sig);
            k.K<true>(buf[yc], buf[yp], buf[yn], 2.0 * sn / ee, cc, -sig * sn);
            sig = sn;
            const int t = yp;
            yp = yc;
            yc = yn;
            yn = t;
        }
        v = yc;
        if ((e = orthonormal()) != cudaSuccess || (*lost_rank = k.lost)) return e;
        if ((e = rayleigh_ritz()) != cudaSuccess) return e;
        bool done = true;
        for (int i = 0; i < n_modes; ++i) {
            if (std::fabs(lam[i] - prev[i]) > 1e-15 * hi) done = false;
            prev[i] = lam[i];
        }
        if (done && it > 0) break;
    }
    for (int i = 0; i < n_modes; ++i) omega[i] = std::sqrt(std::max(lam[i], 0.0));
    if (B_dev) k_md_scatter<<<md_blocks(n_t * n_modes), kMdThreads, 0, s>>>(buf[v], perm, B_dev, n_t, m, n_modes);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

}  // namespace ue
