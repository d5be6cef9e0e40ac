// Mesh optimisation by the jello model with flip refinement (Section 3, "Mesh generation").
//
// Nodes joined by springs along the triangle edges and along the heights relax, strongly
// damped (first order, Euler), towards near-equilateral triangles of a given size; the nodes of
// the input geometry (the boundary) stay.  Every few steps the triangulation is refreshed by
// Lawson flips, because deformed triangles stop the relaxation around them.
// Model: unit springs, so the force is -grad E with
//   E = sum_edges (|ab| - L0)^2 / 2 + sum_heights (|v - m| - H0)^2 / 2,
// a height spring joining vertex v to the midpoint m of its opposite edge; L0 = (h_a + h_b)/2,
// H0 = sqrt(3)/2 times the mean L0 of the triangle's edges.  One step: x += tau F, the
// displacement clamped to 0.1 of the node's shortest rest edge and to 0.15 of the smallest
// height h of its triangles: moves of at most d per vertex change twice a triangle's area by at
// most 3 d L + 4 d^2 <= 0.54 h L (L its longest edge), less than the h L it has, so no triangle
// turns over.
// GPU, FP64, positions double-buffered: per step one thread per triangle evaluates its three
// height springs, its cap and the edge springs it owns once each, then one thread per node gathers
// its edges' and its triangles' shares.  The lists are made on the device after every round of
// flips, which also marks the edges that may not be Delaunay; the flips themselves, whose order
// decides the result's rows, are made on the host from those marks.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <type_traits>
#include <unordered_set>
#include <utility>
#include <vector>

#include "device.cuh"

namespace ue {

namespace {

constexpr int kRxThreads = 256;
// The two step kernels use small blocks: 40k triangles are 636 blocks for 152 SMs, where 159 of 256
// threads gave seven SMs twice the work of the others.
constexpr int kRxStepThreads = 64;

// Device arrays of one relaxation.  A corner or an edge is a code s = 3 i + q of triangle i: the
// corner q, the edge from it to the next corner.
struct RxDev {
    double *x0, *x1;      // positions, before and after a step
    double* h;            // size per node
    double* H0;           // rest height per triangle
    double* cap;          // displacement cap per node
    double* tri_out;      // per triangle: {F_0, F_1, F_2 (x, y each), cap, 0}
    double* edge_out;     // per owned edge s: its pull on its first node
    int32_t *t, *nb;      // corners; the triangle across edge s, -1 none
    int32_t *off, *cnt;   // node v: its corners at code[off[v] .. off[v] + cnt[v]), ascending
    int32_t* code;
    int32_t* e_cnt;       // node v: its edges at e_ref[2 off[v] ..], by the other node's number
    uint32_t* e_ref;      // 2 s + (1: v is the edge's second node) of the slot s that owns the edge
    uint8_t *own, *fixed; // slot s owns its edge; boundary nodes and anchors
    uint8_t* anchor;
    uint8_t* marks;       // per slot, for the flips: kSeed, kSeed | kLook
    int32_t* ctl;         // {list cursor, a node has too many triangles, an edge is not shared by two}
    size_t cleared;       // bytes from cnt on that a rebuild starts at zero
};

// Corners per node that one thread sorts (about 6 in a triangulation of any quality); a mesh with a
// node of more is listed on the host.
constexpr int kRxValence = 32;
constexpr uint8_t kSeed = 1, kLook = 2;
constexpr int64_t kRxMarked = 384;

// 1/|w| and |w| of w^2 = n2: one Heron step on n2 rsqrt(n2) gives the root to about half an ulp, so
// springs and caps keep the precision of a square root and a division at the cost of one rsqrt.
__device__ __forceinline__ double root(double n2, double* r) {
    *r = rsqrt(n2);
    const double y = n2 * *r;
    return fma(fma(-y, y, n2), 0.5 * *r, y);
}

// Per triangle, once per step: the three height springs' pulls on its vertices and the cap
// 0.15 * (2 area / longest edge).  Spring q (apex q over the edge (q+1, q+2)) with
// g_q = ((|w| - H0) / |w|) w, w = x_q - (x_{q+1} + x_{q+2}) / 2, pulls the apex by -g_q and each
// end of its edge by g_q / 2, so vertex j takes -g_j + (g_{j+1} + g_{j+2}) / 2.  The springs along
// the edges that it owns: the pull on the second node is the negative.
// Bound by the FP64 pipe (two lanes per SM and clock): every edge and height is evaluated once,
// with one rsqrt for its root and its division.  40k triangles: 17 us, the FP64 pipe busy for 78% of
// the active cycles (23 us with an edge length per triangle and a root and a division per spring).
__global__ void __launch_bounds__(kRxStepThreads) k_rx_tri(const __grid_constant__ RxDev a, const double* __restrict__ x,
                                                           int64_t n_tris) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tris) return;
    double px[3], py[3], h[3];
    uint8_t own[3];
    for (int q = 0; q < 3; ++q) {
        const int32_t n = a.t[3 * t + q];
        const double2 p = reinterpret_cast<const double2*>(x)[n];
        px[q] = p.x;
        py[q] = p.y;
        h[q] = a.h[n];
        own[q] = a.own[3 * t + q];
    }
    const double h0 = a.H0[t];
    const double a2 = fabs((px[1] - px[0]) * (py[2] - py[0]) - (py[1] - py[0]) * (px[2] - px[0]));
    double l2[3];
    double2* eo = reinterpret_cast<double2*>(a.edge_out) + 3 * t;
    for (int q = 0; q < 3; ++q) {
        const int p = q == 2 ? 0 : q + 1;
        const double ex = px[p] - px[q], ey = py[p] - py[q];
        l2[q] = ex * ex + ey * ey;
        if (own[q]) {
            double r;
            const double s = (root(l2[q], &r) - 0.5 * (h[q] + h[p])) * r;
            eo[q] = make_double2(s * ex, s * ey);
        }
    }
    double gx[3], gy[3];
    for (int q = 0; q < 3; ++q) {
        const int p = q == 2 ? 0 : q + 1, r = q == 0 ? 2 : q - 1;
        const double wx = px[q] - 0.5 * (px[p] + px[r]), wy = py[q] - 0.5 * (py[p] + py[r]);
        double rm;
        const double hm = root(wx * wx + wy * wy, &rm);
        const double sc = (hm - h0) * rm;
        gx[q] = sc * wx;
        gy[q] = sc * wy;
    }
    double f[6];
    for (int j = 0; j < 3; ++j) {
        const int p = j == 2 ? 0 : j + 1, r = j == 0 ? 2 : j - 1;
        f[2 * j] = 0.5 * (gx[p] + gx[r]) - gx[j];
        f[2 * j + 1] = 0.5 * (gy[p] + gy[r]) - gy[j];
    }
    double rl;
    const double lm = root(fmax(fmax(l2[0], l2[1]), l2[2]), &rl);
    double ht = a2 * rl;
    ht = fma(fma(-lm, ht, a2), rl, ht);
    double2* o = reinterpret_cast<double2*>(a.tri_out) + 4 * t;
    o[0] = make_double2(f[0], f[1]);
    o[1] = make_double2(f[2], f[3]);
    o[2] = make_double2(f[4], f[5]);
    o[3] = make_double2(0.15 * ht, 0.0);
}

// Per node: its edge springs, its shares of its triangles' height springs, the smallest cap;
// then the capped Euler step (fixed nodes copy through).  Bound by the latency of its gathers: the
// first kRxHeld entries of both lists are read together, and what they name is then loaded at once.
// (As a programmatic dependent of the triangles' kernel, the lists read before its end, a step took
// 35 us instead of 29: waiting blocks held the registers of those to come.)  20k nodes: 12 us (30 us with every edge's spring evaluated here,
// at both of its ends).
constexpr int kRxHeld = 8;
__global__ void __launch_bounds__(kRxStepThreads) k_rx_node(const __grid_constant__ RxDev a, const double* __restrict__ x,
                                                            double* __restrict__ xn, double tau, int64_t n_nodes) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n_nodes) return;
    const double2 p = reinterpret_cast<const double2*>(x)[v];
    if (a.fixed[v]) {
        reinterpret_cast<double2*>(xn)[v] = p;
        return;
    }
    const int32_t off = a.off[v], ne = a.e_cnt[v], nt = a.cnt[v];
    double c = a.cap[v];
    const uint32_t* er = a.e_ref + 2 * (int64_t)off;
    const int32_t* cd = a.code + off;
    uint32_t r[kRxHeld];
    int32_t s[kRxHeld];
#pragma unroll
    for (int i = 0; i < kRxHeld; ++i) {
        r[i] = i < ne ? er[i] : 0u;
        s[i] = i < nt ? cd[i] : 0;
    }
    auto edge = [&](uint32_t ref) { return reinterpret_cast<const double2*>(a.edge_out)[ref >> 1]; };
    auto share = [&](int32_t code, double* cap) {
        const int32_t t = code / 3;
        const double2* o = reinterpret_cast<const double2*>(a.tri_out) + 4 * (int64_t)t;
        *cap = reinterpret_cast<const double*>(o + 3)[0];
        return o[code - 3 * t];
    };
    double2 ev[kRxHeld], tv[kRxHeld];
    double cv[kRxHeld];
#pragma unroll
    for (int i = 0; i < kRxHeld; ++i) {
        if (i < ne) ev[i] = edge(r[i]);
        if (i < nt) tv[i] = share(s[i], &cv[i]);
    }
    double fx = 0.0, fy = 0.0;
    auto pull = [&](uint32_t ref, double2 e) {   // edge springs
        fx += ref & 1 ? -e.x : e.x;
        fy += ref & 1 ? -e.y : e.y;
    };
    auto height = [&](double2 f, double cap) {   // its triangles' height springs
        fx += f.x;
        fy += f.y;
        c = fmin(c, cap);
    };
#pragma unroll
    for (int i = 0; i < kRxHeld; ++i)
        if (i < ne) pull(r[i], ev[i]);
    for (int32_t i = kRxHeld; i < ne; ++i) pull(er[i], edge(er[i]));
#pragma unroll
    for (int i = 0; i < kRxHeld; ++i)
        if (i < nt) height(tv[i], cv[i]);
    for (int32_t i = kRxHeld; i < nt; ++i) {
        double cap;
        const double2 f = share(cd[i], &cap);
        height(f, cap);
    }
    double dx = tau * fx, dy = tau * fy;
    const double n2 = dx * dx + dy * dy;
    if (!(n2 < c * c * (1.0 - 1e-15))) {   // else the root is below c too
        const double n = sqrt(n2);
        if (n > c) {
            const double k = c / n;
            dx *= k;
            dy *= k;
        }
    }
    reinterpret_cast<double2*>(xn)[v] = make_double2(p.x + dx, p.y + dy);
}

// --- the lists: corners counted, offsets handed out block by block (any order serves), corners
// filled in and sorted per node.  Five launches, 55 us together for 40k triangles; on the host the lists,
// their upload and the flips' matching of edges took 6 ms per round of flips.

__global__ void k_rx_count(const __grid_constant__ RxDev a, int64_t n_tris) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tris) return;
    double s = 0.0;
    for (int q = 0; q < 3; ++q) {
        const int32_t n = a.t[3 * t + q], m = a.t[3 * t + (q == 2 ? 0 : q + 1)];
        atomicAdd(a.cnt + n, 1);
        s += 0.5 * (a.h[n] + a.h[m]);
    }
    a.H0[t] = sqrt(3.0) / 2.0 * s / 3.0;
}

__global__ void __launch_bounds__(kRxThreads) k_rx_offsets(const __grid_constant__ RxDev a, int64_t n_nodes) {
    __shared__ int32_t w[kRxThreads / 32];
    __shared__ int32_t base;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int32_t n = v < n_nodes ? a.cnt[v] : 0;
    if (n > kRxValence) a.ctl[1] = 1;
    int32_t inc = n;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) w[threadIdx.x >> 5] = inc;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t sum = 0;
        for (int i = 0; i < kRxThreads / 32; ++i) {
            const int32_t u = w[i];
            w[i] = sum;
            sum += u;
        }
        base = atomicAdd(a.ctl, sum);
    }
    __syncthreads();
    if (v < n_nodes) a.off[v] = base + w[threadIdx.x >> 5] + inc - n;
}

__global__ void k_rx_fill(const __grid_constant__ RxDev a, int64_t n_slots) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_slots) return;
    const int32_t n = a.t[s];
    a.code[a.off[n] + atomicAdd(a.e_cnt + n, 1)] = (int32_t)s;   // e_cnt: a cursor until k_rx_lists
}

// Node v's corners in ascending order, its edges by the other node's number (each owned by the lowest
// slot that names it, as at its other end), its cap; an edge named once is on the boundary, its
// ends fixed.
__global__ void __launch_bounds__(kRxStepThreads) k_rx_lists(const __grid_constant__ RxDev a, int64_t n_nodes) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n_nodes) return;
    const int32_t n = a.cnt[v];
    if (n > kRxValence) return;
    int32_t* cd = a.code + a.off[v];
    unsigned long long key[2 * kRxValence];
    key[0] = 0;
    int m = 0;
    auto put = [&](int32_t b, int32_t s, uint32_t second) {
        const unsigned long long k = (unsigned long long)b << 32 | ((unsigned)s << 1 | second);
        int i = m++;
        for (; i > 0 && key[i - 1] > k; --i) key[i] = key[i - 1];
        key[i] = k;
    };
    for (int32_t k = 0; k < n; ++k) {
        const int32_t s = cd[k];
        int32_t i = k;
        for (; i > 0 && cd[i - 1] > s; --i) cd[i] = cd[i - 1];
        cd[i] = s;
        const int32_t t = s / 3, q = s - 3 * t, p = q == 2 ? 0 : q + 1, r = q == 0 ? 2 : q - 1;
        put(a.t[3 * (int64_t)t + p], s, 0);
        put(a.t[3 * (int64_t)t + r], 3 * t + r, 1);
    }
    uint32_t* er = a.e_ref + 2 * (int64_t)a.off[v];
    int32_t ne = 0;
    double cap = INFINITY;
    for (int k = 0; k < m;) {
        int r = k + 1;
        while (r < m && key[r] >> 32 == key[k] >> 32) ++r;
        const int32_t b = (int32_t)(key[k] >> 32);
        const uint32_t ref = (uint32_t)key[k];
        if (r - k == 1) a.fixed[v] = a.fixed[b] = 1;
        a.own[ref >> 1] = 1;
        er[ne++] = ref;
        cap = fmin(cap, 0.1 * (0.5 * (a.h[v] + a.h[b])));
        k = r;
    }
    a.e_cnt[v] = ne;
    a.cap[v] = cap;
    if (a.anchor[v]) a.fixed[v] = 1;
}

// The triangle across each edge, from the corners of its second node.  Edges of more than two
// triangles, or of two on one side, are reported: the host's order of matching then decides.
__global__ void k_rx_nb(const __grid_constant__ RxDev a, int64_t n_slots) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_slots || a.ctl[1] != 0) return;
    const int64_t i = s / 3;
    const int q = (int)(s - 3 * i);
    const int32_t n0 = a.t[s], n1 = a.t[3 * i + (q == 2 ? 0 : q + 1)];
    int32_t nb = -1;
    int twins = 0, same = 0;
    for (int32_t k = a.off[n1], e = k + a.cnt[n1]; k < e; ++k) {
        const int32_t c = a.code[k], j = c / 3, r = c - 3 * j;
        if (j == (int32_t)i) continue;
        if (a.t[3 * (int64_t)j + (r == 2 ? 0 : r + 1)] == n0) {
            nb = j;
            ++twins;
        }
        if (a.t[3 * (int64_t)j + (r == 0 ? 2 : r - 1)] == n0) ++same;
    }
    if (twins > 1 || same > 0) a.ctl[2] = 1;
    a.nb[s] = nb;
}

// Marks for the flips: every edge once (the slot of its lower triangle), and whether the in-circle
// test of in_circle() below could hold at these positions: the threshold is lowered by a
// thousandth, far above the test's rounding (about 1e-14 of s^2), and what is not a number, or so
// small that products underflow, is marked.
__global__ void k_rx_marks(const __grid_constant__ RxDev m, const double* __restrict__ x, int64_t n_slots) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_slots) return;
    const int64_t i = s / 3, j = m.nb[s];
    uint8_t mark = 0;
    if (j > i) {
        const int q = (int)(s - 3 * i);
        const int32_t a = m.t[s], b = m.t[3 * i + (q == 2 ? 0 : q + 1)], c = m.t[3 * i + (q == 0 ? 2 : q - 1)];
        int32_t d = m.t[3 * j];
        for (int r = 1; r < 3; ++r)
            if (d == a || d == b) d = m.t[3 * j + r];
        const double2* p = reinterpret_cast<const double2*>(x);
        const double2 pa = p[a], pb = p[b], pc = p[c], pd = p[d];
        const double ax = pa.x - pd.x, ay = pa.y - pd.y, bx = pb.x - pd.x, by = pb.y - pd.y, cx = pc.x - pd.x,
                     cy = pc.y - pd.y;
        const double a2 = ax * ax + ay * ay, b2 = bx * bx + by * by, c2 = cx * cx + cy * cy;
        const double det = a2 * (bx * cy - by * cx) - b2 * (ax * cy - ay * cx) + c2 * (ax * by - ay * bx);
        const double l = fmax(a2, fmax(b2, c2));
        mark = kSeed;
        if (!(det <= 0.999e-10 * l * l) || !(l * l > 1e-280) || !(l * l < 1e280)) mark |= kLook;
    }
    m.marks[s] = mark;
}

double orient2d(const std::vector<double>& x, int a, int b, int c) {
    return (x[2 * b] - x[2 * a]) * (x[2 * c + 1] - x[2 * a + 1]) -
           (x[2 * b + 1] - x[2 * a + 1]) * (x[2 * c] - x[2 * a]);
}

// d strictly inside the circumcircle of the CCW triangle abc, beyond a relative 1e-10 margin
bool in_circle(const std::vector<double>& x, int a, int b, int c, int d) {
    const double ax = x[2 * a] - x[2 * d], ay = x[2 * a + 1] - x[2 * d + 1];
    const double bx = x[2 * b] - x[2 * d], by = x[2 * b + 1] - x[2 * d + 1];
    const double cx = x[2 * c] - x[2 * d], cy = x[2 * c + 1] - x[2 * d + 1];
    const double a2 = ax * ax + ay * ay, b2 = bx * bx + by * by, c2 = cx * cx + cy * cy;
    const double det = a2 * (bx * cy - by * cx) - b2 * (ax * cy - ay * cx) + c2 * (ax * by - ay * bx);
    const double s = std::max(a2, std::max(b2, c2));
    return det > 1e-10 * s * s;
}

uint64_t edge_key(int32_t a, int32_t b) {
    return ((uint64_t)(uint32_t)std::min(a, b) << 32) | (uint32_t)std::max(a, b);
}

// node -> corners 3 i + q (CSR by counting), ascending
void node_corners(int64_t nn, const std::vector<int32_t>& t, std::vector<int32_t>& off, std::vector<int32_t>& code) {
    off.assign(nn + 1, 0);
    for (int32_t n : t) ++off[n + 1];
    for (int64_t v = 0; v < nn; ++v) off[v + 1] += off[v];
    code.assign(off[nn], 0);
    std::vector<int32_t> p(off.begin(), off.end() - 1);
    for (size_t s = 0; s < t.size(); ++s) code[p[t[s]]++] = (int32_t)s;
}

// nb[3 i + q]: the triangle across edge q = (t[q], t[q+1]) of triangle i (-1 on the boundary); marks
// of all edges.
void host_neighbours(int64_t nn, const std::vector<int32_t>& t, std::vector<int32_t>& nb, std::vector<uint8_t>& marks) {
    const int64_t nt = (int64_t)t.size() / 3;
    nb.assign(3 * nt, -1);
    // the twin of a -> b in triangle i is b -> a in one of b's other triangles
    std::vector<int32_t> off, code;
    node_corners(nn, t, off, code);
    for (int64_t i = 0; i < nt; ++i)
        for (int q = 0; q < 3; ++q) {
            if (nb[3 * i + q] >= 0) continue;   // found from the other side
            const int32_t a = t[3 * i + q], b = t[3 * i + (q + 1) % 3];
            for (int32_t k = off[b]; k < off[b + 1] && nb[3 * i + q] < 0; ++k) {
                const int32_t j = code[k] / 3;
                if (j == i) continue;
                for (int r = 0; r < 3; ++r)
                    if (t[3 * j + r] == b && t[3 * j + (r + 1) % 3] == a) {
                        nb[3 * i + q] = j;
                        nb[3 * j + r] = (int32_t)i;
                        break;
                    }
            }
        }
    marks.assign(3 * nt, 0);
    for (int64_t s = 0; s < 3 * nt; ++s)
        if (nb[s] > s / 3) marks[s] = kSeed | kLook;
}

// Lawson flips until every interior edge is locally Delaunay; returns the number of flips.
// nb: as host_neighbours; it follows the flips.
// Edges are taken in the order of their slots, those that flips bring up before the next: a
// stack holds (triangle, a, b) for a directed CCW edge a->b; an entry whose triangle no longer
// holds that edge is stale and skipped: every flip pushes its four outer edges with their current
// triangles, so no live edge is lost.  An edge marked kSeed alone is Delaunay and passed by unless a
// flip has changed one of its two triangles since.
// keep: edges (edge_key) that are never flipped (the input geometry's).
int64_t lawson(const std::vector<double>& x, std::vector<int32_t>& t, std::vector<int32_t>& nb,
               std::vector<uint8_t>& marks, const std::unordered_set<uint64_t>& keep) {
    const int64_t n_slots = (int64_t)t.size();
    const std::vector<int32_t> t0 = t;   // the seeds' edges
    struct Item { int32_t tri, a, b; };
    std::vector<Item> stack;
    auto slot_of = [&](int64_t i, int32_t a, int32_t b) -> int {
        for (int q = 0; q < 3; ++q)
            if (t[3 * i + q] == a && t[3 * i + (q + 1) % 3] == b) return q;
        return -1;
    };
    auto look = [&](int64_t i) {
        if (i >= 0)
            for (int q = 0; q < 3; ++q) marks[3 * i + q] |= kLook;
    };
    int64_t flips = 0;
    for (int64_t seed = 0; seed < n_slots; ++seed) {
        uint64_t eight;
        if (seed + 8 <= n_slots && (std::memcpy(&eight, &marks[seed], 8), (eight & (0x0101010101010101ull * kLook)) == 0)) {
            seed += 7;
            continue;
        }
        if (marks[seed] != (kSeed | kLook)) continue;
        const int32_t si = (int32_t)(seed / 3);
        stack.push_back({si, t0[seed], t0[3 * (int64_t)si + (seed % 3 + 1) % 3]});
        while (!stack.empty()) {
            const Item it = stack.back();
            stack.pop_back();
            const int64_t i = it.tri;
            const int qi = slot_of(i, it.a, it.b);
            if (qi < 0) continue;                       // stale: the edge left this triangle
            const int64_t j = nb[3 * i + qi];
            if (j < 0) continue;
            const int32_t a = it.a, b = it.b, c = t[3 * i + (qi + 2) % 3];
            if (!keep.empty() && keep.count(edge_key(a, b))) continue;
            const int qj = slot_of(j, b, a);
            const int32_t d = t[3 * j + (qj + 2) % 3];
            if (!in_circle(x, a, b, c, d)) continue;
            if (orient2d(x, a, d, c) <= 0 || orient2d(x, d, b, c) <= 0) continue;   // not convex
            const int32_t X_bc = nb[3 * i + (qi + 1) % 3], X_ca = nb[3 * i + (qi + 2) % 3];
            const int32_t X_ad = nb[3 * j + (qj + 1) % 3], X_db = nb[3 * j + (qj + 2) % 3];
            // new i = (a, d, c), new j = (d, b, c)
            t[3 * i] = a; t[3 * i + 1] = d; t[3 * i + 2] = c;
            t[3 * j] = d; t[3 * j + 1] = b; t[3 * j + 2] = c;
            nb[3 * i] = X_ad; nb[3 * i + 1] = (int32_t)j; nb[3 * i + 2] = X_ca;
            nb[3 * j] = X_db; nb[3 * j + 1] = X_bc; nb[3 * j + 2] = (int32_t)i;
            auto repoint = [&](int64_t X, int64_t from, int64_t to) {
                if (X < 0) return;
                for (int q = 0; q < 3; ++q)
                    if (nb[3 * X + q] == from) { nb[3 * X + q] = (int32_t)to; return; }
            };
            repoint(X_ad, j, i);
            repoint(X_bc, i, j);
            for (int64_t X : {i, j, (int64_t)X_ad, (int64_t)X_db, (int64_t)X_bc, (int64_t)X_ca}) look(X);
            ++flips;
            stack.push_back({(int32_t)i, a, d});
            stack.push_back({(int32_t)j, d, b});
            stack.push_back({(int32_t)j, b, c});
            stack.push_back({(int32_t)i, c, a});
        }
    }
    return flips;
}

// The lists of k_rx_offsets, k_rx_fill and k_rx_lists on the host, for meshes with a node of more
// than kRxValence triangles: sorted in n log n.
struct RxLists {
    std::vector<int32_t> off, cnt, code, e_cnt;
    std::vector<uint32_t> e_ref;
    std::vector<uint8_t> own, fixed;
    std::vector<double> cap;
};

void build_lists(int64_t nn, const std::vector<int32_t>& t, const std::vector<double>& h, const std::vector<uint8_t>& anchor,
                 RxLists& L) {
    node_corners(nn, t, L.off, L.code);
    L.cnt.resize(nn);
    L.e_cnt.assign(nn, 0);
    L.e_ref.assign(2 * L.code.size(), 0);
    L.own.assign(t.size(), 0);
    L.fixed = anchor;
    L.cap.assign(nn, INFINITY);
    std::vector<uint64_t> key;
    for (int64_t v = 0; v < nn; ++v) {
        key.clear();
        L.cnt[v] = L.off[v + 1] - L.off[v];
        for (int32_t k = L.off[v]; k < L.off[v + 1]; ++k) {
            const int32_t s = L.code[k], q = s % 3, p = s - q + (q + 1) % 3, r = s - q + (q + 2) % 3;
            key.push_back((uint64_t)t[p] << 32 | (uint32_t)s << 1);
            key.push_back((uint64_t)t[r] << 32 | (uint32_t)r << 1 | 1);
        }
        std::sort(key.begin(), key.end());
        uint32_t* er = L.e_ref.data() + 2 * (size_t)L.off[v];
        for (size_t k = 0; k < key.size();) {
            size_t r = k + 1;
            while (r < key.size() && key[r] >> 32 == key[k] >> 32) ++r;
            const int32_t b = (int32_t)(key[k] >> 32);
            if (r - k == 1) L.fixed[v] = L.fixed[b] = 1;
            L.own[(uint32_t)key[k] >> 1] = 1;
            er[L.e_cnt[v]++] = (uint32_t)key[k];
            L.cap[v] = std::min(L.cap[v], 0.1 * (0.5 * (h[v] + h[b])));
            k = r;
        }
    }
}

}  // namespace

namespace {

// Orients the triangles CCW in t (a copy of tris); accumulates the area.
int orient_input(const std::vector<double>& x, int64_t nn, std::vector<int32_t>& t, double* area,
                 std::string& err) {
    const int64_t nt = (int64_t)t.size() / 3;
    for (int64_t i = 0; i < nt; ++i) {
        int32_t* r = &t[3 * i];
        for (int q = 0; q < 3; ++q)
            if (r[q] < 0 || r[q] >= nn) {
                err = "triangle node index out of range";
                return UE_ERR_ARG;
            }
        double o = orient2d(x, r[0], r[1], r[2]);
        if (o < 0) {
            std::swap(r[1], r[2]);
            o = -o;
        }
        if (!(o > 0)) {
            err = "degenerate triangle " + std::to_string(i);
            return UE_ERR_DEGENERATE;
        }
        *area += 0.5 * o;
    }
    return UE_OK;
}

int keep_set(const int32_t* segs, int64_t n_segs, int64_t nn, std::unordered_set<uint64_t>& keep,
             std::string& err) {
    for (int64_t k = 0; k < n_segs; ++k) {
        const int32_t a = segs[2 * k], b = segs[2 * k + 1];
        if (a < 0 || b < 0 || a >= nn || b >= nn || a == b) {
            err = "kept edge " + std::to_string(k) + " has a bad node id";
            return UE_ERR_ARG;
        }
        keep.insert(edge_key(a, b));
    }
    return UE_OK;
}

}  // namespace

// See include/ue.h (ue_mesh_flip): the remesh step alone, on the host.
int mesh_flip(const double* xy, int64_t nn, const int32_t* tris, int64_t nt, const int32_t* segs,
              int64_t n_segs, int32_t* tris_out, int64_t* n_flips, std::string& err) {
    std::vector<double> x(xy, xy + 2 * nn);
    std::vector<int32_t> t(tris, tris + 3 * nt);
    double area = 0.0;
    std::unordered_set<uint64_t> keep;
    int rc = orient_input(x, nn, t, &area, err);
    if (rc == UE_OK) rc = keep_set(segs, n_segs, nn, keep, err);
    if (rc != UE_OK) return rc;
    std::vector<int32_t> nb;
    std::vector<uint8_t> marks;
    host_neighbours(nn, t, nb, marks);
    const int64_t k = lawson(x, t, nb, marks, keep);
    std::copy(t.begin(), t.end(), tris_out);
    if (n_flips) *n_flips = k;
    return UE_OK;
}

int mesh_relax(const double* xy, int64_t nn, const int32_t* tris, int64_t nt, const double* h_nodes,
               int32_t iters, int32_t flip_every, double tau, const int32_t* anchors, int64_t n_anchors,
               const int32_t* segs, int64_t n_segs, double* xy_out, int32_t* tris_out, int64_t* n_flips,
               cudaStream_t s, std::string& err) {
    std::vector<double> x(xy, xy + 2 * nn);
    std::vector<int32_t> t(tris, tris + 3 * nt);
    double area = 0.0;
    std::unordered_set<uint64_t> keep;
    {
        int rc = orient_input(x, nn, t, &area, err);
        if (rc == UE_OK) rc = keep_set(segs, n_segs, nn, keep, err);
        if (rc != UE_OK) return rc;
        for (int64_t k = 0; k < n_anchors; ++k)
            if (anchors[k] < 0 || anchors[k] >= nn) {
                err = "anchor " + std::to_string(k) + " is not a node id";
                return UE_ERR_ARG;
            }
    }
    std::vector<double> h(nn);
    if (h_nodes) {
        for (int64_t v = 0; v < nn; ++v) {
            if (!(h_nodes[v] > 0)) {
                err = "sizes must be positive";
                return UE_ERR_ARG;
            }
            h[v] = h_nodes[v];
        }
    } else {
        std::fill(h.begin(), h.end(), std::sqrt(4.0 * area / (std::sqrt(3.0) * (double)nt)));
    }
    std::vector<uint8_t> anchor(nn, 0);
    for (int64_t k = 0; k < n_anchors; ++k) anchor[anchors[k]] = 1;

    // one device block for the call, a one-off preprocessing step outside any mesh
    RxDev a = {};
    size_t bytes = 0;
    char* block = nullptr;
    auto lay = [&]() {   // twice: the size, then the pointers
        bytes = 0;
        auto cut = [&](auto*& p, size_t n) {
            p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(block + bytes);
            bytes += (n * sizeof(*p) + 255) / 256 * 256;
        };
        cut(a.x0, 2 * nn);
        cut(a.x1, 2 * nn);
        cut(a.h, nn);
        cut(a.H0, nt);
        cut(a.cap, nn);
        cut(a.tri_out, 8 * nt);
        cut(a.edge_out, 6 * nt);
        cut(a.t, 3 * nt);
        cut(a.nb, 3 * nt);
        cut(a.off, nn);
        cut(a.code, 3 * nt);
        cut(a.e_ref, 6 * nt);
        cut(a.anchor, nn);
        cut(a.marks, 3 * nt);
        const size_t z = bytes;
        cut(a.cnt, nn);
        cut(a.e_cnt, nn);
        cut(a.own, 3 * nt);
        cut(a.fixed, nn);
        cut(a.ctl, 4);
        a.cleared = bytes - z;
    };
    lay();
    cudaError_t e = cudaMalloc(&block, bytes);
    lay();
    auto ck = [&](cudaError_t r) {
        if (e == cudaSuccess && r != cudaSuccess) e = r;
    };
    const int64_t n_slots = 3 * nt;
    // Marks and neighbours of few triangles are sooner found on the host (about 0.1 us a triangle) than
    // launched, copied and waited for (25 us)
    const bool marked = flip_every > 0 && nt >= kRxMarked;
    auto blocks = [](int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); };
    int32_t ctl[4] = {};
    // after a change of t: the lists of every node and, where flips follow, the neighbours
    auto relist = [&]() {
        ck(cudaMemcpyAsync(a.t, t.data(), 4 * n_slots, cudaMemcpyHostToDevice, s));
        ck(cudaMemsetAsync(a.cnt, 0, a.cleared, s));
        if (e != cudaSuccess) return;
        k_rx_count<<<blocks(nt, kRxThreads), kRxThreads, 0, s>>>(a, nt);
        k_rx_offsets<<<blocks(nn, kRxThreads), kRxThreads, 0, s>>>(a, nn);
        k_rx_fill<<<blocks(n_slots, kRxThreads), kRxThreads, 0, s>>>(a, n_slots);
        k_rx_lists<<<blocks(nn, kRxStepThreads), kRxStepThreads, 0, s>>>(a, nn);
        if (marked) k_rx_nb<<<blocks(n_slots, kRxThreads), kRxThreads, 0, s>>>(a, n_slots);
        ck(cudaGetLastError());
        ck(cudaMemcpyAsync(ctl, a.ctl, sizeof(ctl), cudaMemcpyDeviceToHost, s));
        ck(cudaStreamSynchronize(s));   // t may change after this
        if (e != cudaSuccess || ctl[1] == 0) return;
        RxLists L;
        build_lists(nn, t, h, anchor, L);
        ck(cudaMemcpyAsync(a.off, L.off.data(), 4 * nn, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.cnt, L.cnt.data(), 4 * nn, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.code, L.code.data(), 4 * n_slots, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.e_cnt, L.e_cnt.data(), 4 * nn, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.e_ref, L.e_ref.data(), 8 * n_slots, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.own, L.own.data(), n_slots, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.fixed, L.fixed.data(), nn, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.cap, L.cap.data(), 8 * nn, cudaMemcpyHostToDevice, s));
        ck(cudaStreamSynchronize(s));
    };
    if (e == cudaSuccess) {
        ck(cudaMemcpyAsync(a.x0, x.data(), 16 * nn, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.h, h.data(), 8 * nn, cudaMemcpyHostToDevice, s));
        ck(cudaMemcpyAsync(a.anchor, anchor.data(), nn, cudaMemcpyHostToDevice, s));
        relist();
    }
    int64_t flips = 0;
    std::vector<int32_t> nb;
    std::vector<uint8_t> marks;
    bool nb_fresh = false;   // nb follows t
    for (int32_t it = 0; it < iters && e == cudaSuccess; ++it) {
        k_rx_tri<<<blocks(nt, kRxStepThreads), kRxStepThreads, 0, s>>>(a, a.x0, nt);
        k_rx_node<<<blocks(nn, kRxStepThreads), kRxStepThreads, 0, s>>>(a, a.x0, a.x1, tau, nn);
        ck(cudaGetLastError());
        std::swap(a.x0, a.x1);
        if (flip_every > 0 && (it + 1) % flip_every == 0 && e == cudaSuccess) {
            const bool listed = marked && ctl[1] == 0 && ctl[2] == 0;
            ck(cudaMemcpyAsync(x.data(), a.x0, 16 * nn, cudaMemcpyDeviceToHost, s));
            if (listed) {
                k_rx_marks<<<blocks(n_slots, kRxThreads), kRxThreads, 0, s>>>(a, a.x0, n_slots);
                ck(cudaGetLastError());
                nb.resize(n_slots);
                marks.resize(n_slots);
                ck(cudaMemcpyAsync(marks.data(), a.marks, n_slots, cudaMemcpyDeviceToHost, s));
                if (!nb_fresh) ck(cudaMemcpyAsync(nb.data(), a.nb, 4 * n_slots, cudaMemcpyDeviceToHost, s));
            }
            ck(cudaStreamSynchronize(s));
            if (e != cudaSuccess) break;
            if (!listed) host_neighbours(nn, t, nb, marks);
            nb_fresh = true;
            const int64_t k = lawson(x, t, nb, marks, keep);
            flips += k;
            if (k > 0) {
                relist();
                nb_fresh = false;
            }
        }
    }
    if (e == cudaSuccess) {
        ck(cudaMemcpyAsync(x.data(), a.x0, 16 * nn, cudaMemcpyDeviceToHost, s));
        ck(cudaStreamSynchronize(s));
    }
    if (block) cudaFree(block);
    if (e != cudaSuccess) {
        err = std::string("mesh relaxation: ") + cudaGetErrorString(e);
        return UE_ERR_CUDA;
    }
    for (int64_t i = 0; i < nt; ++i)
        if (!(orient2d(x, t[3 * i], t[3 * i + 1], t[3 * i + 2]) > 0)) {
            err = "relaxation inverted triangle " + std::to_string(i) + ": lower tau";
            return UE_ERR_DEGENERATE;
        }
    std::copy(x.begin(), x.end(), xy_out);
    std::copy(t.begin(), t.end(), tris_out);
    if (n_flips) *n_flips = flips;
    return UE_OK;
}

}  // namespace ue
