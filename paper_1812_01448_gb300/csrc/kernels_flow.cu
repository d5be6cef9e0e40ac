// Resident leap-frog: a mesh that fits the chip's registers and shared memory is advanced by
// many steps in one cooperative launch (eqs. 14-15 with eqs. 3-6, and the PML frame's cells).
//
// The plain step is two launches per step, each reading its tables again: on a mesh of a few
// hundred thousand triangles a launch is latency, not bandwidth.  Here every CTA keeps a run of
// consecutive stored triangles (and of frame cells) for the whole call: one thread holds a
// triangle's B and its three edges' circulations, coefficients in registers or shared memory, and
// only B crosses between CTAs.
//
// Edges as their triangles see them: with s_q the orientation sign of eq. 4, V_q = s_q U_q.  The
// triangle is R of the edge exactly when s_q = +1, so eq. 3 reads
//   V_q = fma(dt|e|/d, rn(b - b_neighbour), V_q)
// on both sides, rounding as U += (dt|e|/d) rn(B_R - B_L) does (round-to-nearest is odd), and
// eq. 4 is b = fma(-dt/S, rn(rn(V_0 + V_1) + V_2), b) as it stands.  The current (V and J change
// sign together) and the source likewise.  Both triangles of an edge compute the same value.
//
// Exchange: no grid barrier.  A triangle with a neighbour in another CTA publishes its B as one
// 64-bit word {value, tag} (FP64: two words), the tag counting steps; readers poll the word until
// it carries the step they need.  Two words per triangle, alternating: a triangle writes step
// s + 1 only after its neighbours' step s has arrived, hence after they have read its step s - 1,
// which the word held.  Per step a CTA polls its remote neighbours once into shared memory, one
// barrier, then every triangle reads its neighbours there.  All CTAs are resident (cooperative
// launch) and every wait is bounded: one that runs out sets the error word and ends the launch.
//
// What bounds it: a step is at least one exchange through L2 (store, poll, barrier: 1.2 us here)
// up to about 1,000 triangles per SM, then the SM's issue slots.  Measured per step on GB300 with
// a line source, against graph replays of the two plain kernels: 90k triangles 1.23 us (6.2 us),
// 305k 1.89; one CTA alone 0.35 us on 1,040 triangles (2.9 us).  Against k_tbp (8 steps per launch,
// ring-ordered tiles) on 480k to 500k triangles 2.4 us (5.0 us), with a plasma current 4.4
// (k_tb 4.7), with a 16-cell PML frame 4.3 (10.0, the frame's tiles stepping by plain launches).
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "exchange.cuh"
#include "frame.cuh"

namespace ue {

namespace {

// Per triangle slot, two words: byte offsets of the three neighbours' B in the CTA's buffer (16
// bits each), then flags.
constexpr unsigned kSrc = 1u << 16;        // 3 bits: the edge has a source
constexpr unsigned kPublish = 1u << 19;    // a neighbour is in another CTA
constexpr unsigned kIface = 1u << 20;      // 3 bits: the edge borders a frame cell
constexpr unsigned kWall = 1u << 23;       // 3 bits: a conductor's edge (its offset is the triangle's own)
constexpr unsigned kFar = 1u << 26;        // 3 bits: neighbour polled by this thread (the CTA's list is full)
constexpr int kCellFar = 1 << 30;          // the same for a frame cell's neighbour
constexpr int kNoEntry = 0xFFFF;

template <typename T>
struct FlowArgs {
    const int4* tri;
    const int2* rl;
    const T* cU;
    const double* cB64;
    T* U;
    T* B;
    const T* pb;
    T* J;
    T pa, mdt;
    const int2* hash;
    unsigned bits;
    const T* src_c;
    const int32_t* src_grp;
    const double* gtab;
    int gstride;
    int gbase;              // this launch's first entry in the g table
    int has_src, n_grp;
    int n_t, n_ei, n_ei_pad;
    int per;                // triangles per CTA
    int hcap, scap;         // capacities of the CTA's lists: remote neighbours, source edges
    unsigned long long* slots[2];
    unsigned* ctl;          // {tag of the next launch, CTAs done, error word}
    long long* step;
    int n_steps;
    int skip;               // tests only (-1 otherwise): this CTA returns at once
    FrameDev f;
    T* Uif;                 // circulations of the frame's interface edges
    int fper;               // frame cells per CTA
};

template <typename T>
struct Vec4 {
    T x, y, z, w;
};
template <>
struct __align__(16) Vec4<float> {
    float x, y, z, w;
};

// A triangle with source edges: s_q dt |e| a of each edge (0 without a source), and its group's
// offset in the g table.
template <typename T>
struct SrcEntry {
    T c[3];
    int g;
};

// the source index of stored edge k (k_edge_half's table), or -1
template <typename T>
__device__ __forceinline__ int src_index(const FlowArgs<T>& a, int k) {
    const unsigned size = 1u << a.bits;
    unsigned h = ((unsigned)k * 2654435761u) >> (32 - a.bits);
    int2 e = __ldg(a.hash + h);
    for (unsigned p = 1; e.x != k && p < size; ++p) {
        h = (h + 1) & (size - 1);
        e = __ldg(a.hash + h);
    }
    return e.x == k ? e.y : -1;
}

// Rare paths of a step, out of line so that they cost the common one no registers: the source
// term of edge k looked up again (the CTA's source list is full), and a neighbour's B polled by
// the thread that needs it (the CTA's list of remote neighbours is full).
template <typename T>
__device__ __noinline__ T source_again(const FlowArgs<T>* a, int code, int at, T v) {
    const int x = src_index(*a, code >> 1);
    if (x < 0) return v;
    const T sc = __ldg(a->src_c + x);
    const T g = (T)__ldg(a->gtab + (size_t)__ldg(a->src_grp + x) * a->gstride + at);
    return rn_fma((code & 1) ? -sc : sc, g, v);
}
template <typename T>
__device__ __noinline__ T poll_one(const unsigned long long* slots, int o, unsigned tag, bool* ok) {
    Word<T> w;
    w.load(slots, o);
    if (!word_wait(w, slots, o, tag)) *ok = false;
    return w.value();
}

__device__ __forceinline__ bool neg_bit(float c) { return __float_as_uint(c) >> 31; }
__device__ __forceinline__ bool neg_bit(double c) { return (unsigned long long)__double_as_longlong(c) >> 63; }

// Coefficients sit in registers while they fit beside the state, else in shared memory.
template <typename T, int TS>
constexpr bool kCoefRegs = sizeof(T) * TS <= 8;

// Shared memory of a CTA of cap triangle slots and `cells` frame cells.
template <typename T, bool PLASMA>
__host__ __device__ constexpr size_t flow_smem(bool coef_regs, int cap, int hcap, int scap, int cells) {
    return (coef_regs ? 0 : sizeof(Vec4<T>) * (size_t)cap * (PLASMA ? 2 : 1)) + sizeof(SrcEntry<T>) * (size_t)scap +
           2 * sizeof(T) * ((size_t)cap + hcap) + sizeof(T) * (size_t)kFlowSteps + 4 * (size_t)hcap + 2 * (size_t)cap +
           3 * sizeof(Vec4<T>) * (size_t)cells;
}

// NT: threads of a CTA (at most, for TS = 1); a thread holds local triangles tid + i * NT, i < TS.
// SOLO: one CTA holds the whole mesh, nothing is published.
template <typename T, int NT, int TS, bool PLASMA, bool FRAME, bool SOLO>
__global__ void __launch_bounds__(NT, 1) k_flow(const __grid_constant__ FlowArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_hcnt, s_scnt;
    const int tid = threadIdx.x, nth = TS > 1 ? NT : (int)blockDim.x, cap = TS * nth;
    Vec4<T>* C = reinterpret_cast<Vec4<T>*>(smraw);                  // dt|e|/d of the three edges, dt/S
    constexpr bool CR = kCoefRegs<T, TS>;
    Vec4<T>* P = C + (CR ? 0 : cap);                                 // pb of the three edges
    Vec4<T>* Fc = P + (CR || !PLASMA ? 0 : cap);                     // a frame cell's a, b of its sides and itself
    SrcEntry<T>* S = reinterpret_cast<SrcEntry<T>*>(Fc + (FRAME ? 3 * a.fper : 0));
    const int bcap = cap + a.hcap;
    T* Bb = reinterpret_cast<T*>(S + a.scap);                        // two buffers: own, then remote B
    T* gs = Bb + 2 * bcap;                                           // g of the launch's steps (one group)
    int* hlist = reinterpret_cast<int*>(gs + kFlowSteps);            // the remote neighbours
    unsigned short* spos = reinterpret_cast<unsigned short*>(hlist + a.hcap);   // source entry of a triangle
    const int j0 = blockIdx.x * a.per;
    const int nloc = max(0, min(a.per, a.n_t - j0));
    if (tid == 0) s_hcnt = s_scnt = 0;
    const unsigned tag0 = SOLO ? 0u : *(volatile unsigned*)a.ctl;
    __syncthreads();
    bool ok = true;
    if (SOLO || (int)blockIdx.x != a.skip) {
        T V[TS][3], J[TS][3], b[TS];
        Vec4<T> Cr[CR ? TS : 1], Pr[CR && PLASMA ? TS : 1];
        unsigned n01[TS], n2f[TS];
        // the list entry of a neighbour in another CTA, or -1 when the list is full
        auto remote = [&](int o) {
            const int pos = atomicAdd(&s_hcnt, 1);
            if (pos >= a.hcap) return -1;
            hlist[pos] = o;
            return cap + pos;
        };
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = tid + i * nth;
            n01[i] = n2f[i] = 0;
            b[i] = T(0);
            if (l >= nloc) continue;
            const int j = j0 + l;
            const int4 t = __ldg(a.tri + j);
            const int code[3] = {t.x, t.y, t.z};
            T c[3], pb[3];
            int src[3] = {-1, -1, -1};
            unsigned f = 0, off[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int k = code[q] >> 1;
                const bool neg = code[q] & 1;
                c[q] = pb[q] = T(0);
                V[i][q] = T(0);
                if constexpr (PLASMA) J[i][q] = T(0);
                int n = -1;
                if (k < a.n_ei) {
                    const int2 r = __ldg(a.rl + k);
                    const int o = neg ? r.x : r.y;
                    const T cu = __ldg(a.cU + k), u = a.U[k];
                    c[q] = fabs(cu);
                    V[i][q] = neg ? -u : u;
                    if constexpr (PLASMA) {
                        const T jj = a.J[k];
                        J[i][q] = neg ? -jj : jj;
                        pb[q] = __ldg(a.pb + k);
                    }
                    if (SOLO || (o >= j0 && o < j0 + nloc)) n = o - j0;
                    else {
                        n = remote(o);
                        f |= kPublish | (n < 0 ? kFar << q : 0u);
                    }
                    if (a.has_src && neg_bit(cu)) src[q] = src_index(a, k);
                } else if (FRAME && k >= a.n_ei_pad) {
                    const int e = k - a.n_ei_pad;
                    const T u = a.Uif[e];
                    c[q] = ((const T*)a.f.icU)[e];
                    V[i][q] = neg ? -u : u;
                    n = remote(a.n_t + a.f.icell[e]);
                    f |= kPublish | (kIface << q) | (n < 0 ? kFar << q : 0u);
                } else {
                    f |= kWall << q;
                }
                off[q] = (unsigned)(n < 0 ? l : n) * (unsigned)sizeof(T);
            }
            T cb;
            if constexpr (sizeof(T) == 4) cb = __int_as_float(t.w);
            else cb = __ldg(a.cB64 + j);
            const Vec4<T> cv{c[0], c[1], c[2], cb}, pv{pb[0], pb[1], pb[2], T(0)};
            if constexpr (CR) Cr[i] = cv;
            else C[l] = cv;
            if constexpr (CR && PLASMA) Pr[i] = pv;
            else if constexpr (PLASMA) P[l] = pv;
            if (src[0] >= 0 || src[1] >= 0 || src[2] >= 0) {
                const int e = atomicAdd(&s_scnt, 1);
                spos[l] = (unsigned short)(e < a.scap ? e : kNoEntry);   // the list is full: looked up at every step
                SrcEntry<T> se{{T(0), T(0), T(0)}, 0};
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if (src[q] < 0) continue;
                    const T sc = __ldg(a.src_c + src[q]);
                    se.c[q] = (code[q] & 1) ? -sc : sc;
                    se.g = (int)__ldg(a.src_grp + src[q]) * a.gstride;
                    f |= kSrc << q;
                }
                if (e < a.scap) S[e] = se;
            }
            n01[i] = off[0] | (off[1] << 16);
            n2f[i] = off[2] | f;
            b[i] = a.B[j];
            Bb[l] = b[i];
        }
        // a frame cell: sides X in bottom, top, left, right order, each with the cell's own
        // counter-clockwise sign, so that every one advances by (own B - neighbour's B)
        unsigned ifm = 0;   // sides that are interface edges: no decay, one fused multiply-add
        T X[4], Bx = T(0), By = T(0);
        int cn[4];
        const int cell = FRAME ? (int)blockIdx.x * a.fper + tid : 0;
        const bool has_cell = FRAME && tid < a.fper && cell < (int)a.f.n_fc;
        if constexpr (FRAME) {
            if (has_cell) {
                const FrameDev& f = a.f;
                const Tab<T> tb = tabs<T>(f);
                T ca[4], cd[4];
                int I, Jc;
                frame_ij(f, cell, I, Jc);
                const bool in_x = I >= f.W && I < f.W + f.nx, in_y = Jc >= f.W && Jc < f.W + f.ny;
                const int di[4] = {0, 0, -1, 1}, dj[4] = {-1, 1, 0, 0};
                // interface edge on that side, or -1
                const int kif[4] = {in_x && Jc == f.W + f.ny ? f.nx + (I - f.W) : -1, in_x && Jc == f.W - 1 ? I - f.W : -1,
                                    in_y && I == f.W + f.nx ? 2 * f.nx + f.ny + (Jc - f.W) : -1,
                                    in_y && I == f.W - 1 ? 2 * f.nx + (Jc - f.W) : -1};
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    X[d] = ca[d] = cd[d] = T(0);
                    cn[d] = -1;
                    if (frame_is_cell(f, I + di[d], Jc + dj[d])) {
                        if (d < 2) {
                            const int at = Jc + d;
                            const T u = ((const T*)f.H)[(int64_t)at * f.NX + I];
                            X[d] = d == 0 ? u : -u;
                            ca[d] = tb.aH[at];
                            cd[d] = tb.bH[at];
                        } else {
                            const int at = I + (d - 2);
                            const T u = ((const T*)f.V)[(int64_t)Jc * (f.NX + 1) + at];
                            X[d] = d == 2 ? -u : u;
                            ca[d] = tb.aV[at];
                            cd[d] = tb.bV[at];
                        }
                        const int o = a.n_t + (int)frame_cell(f, I + di[d], Jc + dj[d]), n = remote(o);
                        cn[d] = n < 0 ? o | kCellFar : n;
                    } else if (kif[d] >= 0) {
                        const int code = f.itri[kif[d]];
                        const T u = a.Uif[kif[d]];
                        X[d] = code >= 0 ? -u : u;
                        ifm |= 1u << d;
                        cd[d] = ((const T*)f.icU)[kif[d]];
                        const int o = code >= 0 ? code : ~code, n = remote(o);
                        cn[d] = n < 0 ? o | kCellFar : n;
                    }
                }
                Bx = ((const T*)f.Bx)[cell];
                By = ((const T*)f.By)[cell];
                Fc[3 * tid] = Vec4<T>{ca[0], ca[1], ca[2], ca[3]};
                Fc[3 * tid + 1] = Vec4<T>{cd[0], cd[1], cd[2], cd[3]};
                Fc[3 * tid + 2] = Vec4<T>{tb.axc[I], tb.bxc[I], tb.ayc[Jc], tb.byc[Jc]};
            }
        }
        if constexpr (!SOLO) {
            // published only after this thread's reads of U, J and the frame are done: their
            // owners write them back after later steps
            __threadfence();
#pragma unroll
            for (int i = 0; i < TS; ++i)
                if (n2f[i] & kPublish) slot_put(a.slots[0], j0 + tid + i * nth, tag0, b[i]);
            if (has_cell) slot_put(a.slots[0], a.n_t + cell, tag0, rn_add(Bx, By));
        }
        const bool one_g = a.has_src && a.n_grp == 1;
        if (one_g)
            for (int e = tid; e < a.n_steps; e += nth) gs[e] = (T)__ldg(a.gtab + a.gbase + e);
        __syncthreads();
        const int hn = SOLO ? 0 : min(s_hcnt, a.hcap);
        auto poll = [&](int p, unsigned tag, int o) -> T {
            bool fine = true;
            const T v = poll_one<T>(p ? a.slots[1] : a.slots[0], o, tag, &fine);
            if (!fine) ok = false;
            return v;
        };
#pragma unroll 1
        for (int s = 1; s <= a.n_steps; ++s) {
            const int p = (s - 1) & 1;
            const unsigned tag = tag0 + (unsigned)(s - 1);
            T* Bp = Bb + (p ? bcap : 0);
            T* Bn = Bb + (p ? 0 : bcap);
            const uint32_t ba = smem_addr(Bp);
            if constexpr (SOLO) {
                if (s > 1) __syncthreads();
            } else {
                // the remote neighbours' B of the last step, a few polls in flight per thread
                constexpr int kPoll = 4;
                for (int e0 = tid; e0 < hn; e0 += kPoll * nth) {
                    Word<T> w[kPoll];
#pragma unroll
                    for (int u = 0; u < kPoll; ++u)
                        if (e0 + u * nth < hn) w[u].load(p ? a.slots[1] : a.slots[0], hlist[e0 + u * nth]);
#pragma unroll
                    for (int u = 0; u < kPoll; ++u) {
                        const int e = e0 + u * nth;
                        if (e < hn) {
                            if (!word_wait(w[u], p ? a.slots[1] : a.slots[0], hlist[e], tag)) ok = false;
                            Bp[cap + e] = w[u].value();
                        }
                    }
                }
                ok = __syncthreads_and(ok ? 1 : 0) != 0;
                if (!ok) break;
            }
            const T g1 = one_g ? gs[s - 1] : T(0);
#pragma unroll
            for (int i = 0; i < TS; ++i) {
                const int l = tid + i * nth;
                if (l >= nloc) break;
                Vec4<T> c, pv;
                if constexpr (CR) c = Cr[i];
                else c = C[l];
                if constexpr (CR && PLASMA) pv = Pr[i];
                else if constexpr (PLASMA) pv = P[l];
                T nv[3] = {lds_val<T>(ba + (n01[i] & 0xFFFFu)), lds_val<T>(ba + (n01[i] >> 16)),
                           lds_val<T>(ba + (n2f[i] & 0xFFFFu))};
                const T cq[3] = {c.x, c.y, c.z};
                const T pq[3] = {PLASMA ? pv.x : T(0), PLASMA ? pv.y : T(0), PLASMA ? pv.z : T(0)};
                if (!SOLO && (n2f[i] & (7u * kFar))) {
                    const int4 t = __ldg(a.tri + j0 + l);
                    const int code[3] = {t.x, t.y, t.z};
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (!(n2f[i] & (kFar << q))) continue;
                        const int k = code[q] >> 1;
                        int o;
                        if (k < a.n_ei) {
                            const int2 r = __ldg(a.rl + k);
                            o = (code[q] & 1) ? r.x : r.y;
                        } else {
                            o = a.n_t + a.f.icell[k - a.n_ei_pad];
                        }
                        nv[q] = poll(p, tag, o);
                    }
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const T uo = V[i][q];
                    T un = rn_fma(cq[q], rn_sub(b[i], nv[q]), uo);
                    if constexpr (PLASMA) {
                        // an interface edge carries no current
                        const T x = FRAME && (n2f[i] & (kIface << q)) ? T(0) : rn_mul(pq[q], uo);
                        const T jn = rn_fma(a.pa, J[i][q], x);
                        un = rn_fma(a.mdt, jn, un);
                        J[i][q] = jn;
                    }
                    V[i][q] = un;
                }
                if (n2f[i] & (7u * kWall)) {   // a conductor's edge stays 0, whatever the fields
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (!(n2f[i] & (kWall << q))) continue;
                        V[i][q] = T(0);
                        if constexpr (PLASMA) J[i][q] = T(0);
                    }
                }
                if (n2f[i] & (7u * kSrc)) {
                    const int e = spos[l];
                    if (e != kNoEntry) {
                        const SrcEntry<T> se = S[e];
                        const T g = one_g ? g1 : (T)__ldg(a.gtab + se.g + a.gbase + s - 1);
#pragma unroll
                        for (int q = 0; q < 3; ++q)
                            if (n2f[i] & (kSrc << q)) V[i][q] = rn_fma(se.c[q], g, V[i][q]);
                    } else {
                        const int4 t = __ldg(a.tri + j0 + l);
                        const int code[3] = {t.x, t.y, t.z};
#pragma unroll
                        for (int q = 0; q < 3; ++q)
                            if (n2f[i] & (kSrc << q)) V[i][q] = source_again<T>(&a, code[q], a.gbase + s - 1, V[i][q]);
                    }
                }
                b[i] = rn_fma(-c.w, rn_add(rn_add(V[i][0], V[i][1]), V[i][2]), b[i]);
                Bn[l] = b[i];
                if constexpr (!SOLO) {
                    if ((n2f[i] & kPublish) && s < a.n_steps) slot_put(p ? a.slots[0] : a.slots[1], j0 + l, tag + 1u, b[i]);
                }
            }
            if constexpr (FRAME) {
                if (has_cell) {
                    const T F = rn_add(Bx, By);
                    const Vec4<T> va = Fc[3 * tid], vd = Fc[3 * tid + 1], vc = Fc[3 * tid + 2];
                    const T ca[4] = {va.x, va.y, va.z, va.w}, cd[4] = {vd.x, vd.y, vd.z, vd.w};
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        if (cn[d] < 0) continue;
                        const T df = rn_sub(F, cn[d] >= kCellFar ? poll(p, tag, cn[d] & ~kCellFar) : Bp[cn[d]]);
                        X[d] = (ifm >> d) & 1u ? rn_fma(cd[d], df, X[d]) : rn_fma(ca[d], X[d], rn_mul(cd[d], df));
                    }
                    Bx = rn_sub(rn_mul(vc.x, Bx), rn_mul(vc.y, rn_add(X[3], X[2])));
                    By = rn_sub(rn_mul(vc.z, By), rn_mul(vc.w, rn_add(X[0], X[1])));
                    if (s < a.n_steps) slot_put(p ? a.slots[0] : a.slots[1], a.n_t + cell, tag + 1u, rn_add(Bx, By));
                }
            }
        }
        if (!SOLO) ok = __syncthreads_and(ok ? 1 : 0) != 0;
        if (ok) {
            if (!SOLO) __threadfence();
            // each edge by its R triangle, each interface edge by its triangle, each frame side
            // by the cell above or to its right
#pragma unroll
            for (int i = 0; i < TS; ++i) {
                const int l = tid + i * nth;
                if (l >= nloc) break;
                const int4 t = __ldg(a.tri + j0 + l);
                const int code[3] = {t.x, t.y, t.z};
                a.B[j0 + l] = b[i];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int k = code[q] >> 1;
                    const bool neg = code[q] & 1;
                    if (k < a.n_ei) {
                        if (neg) continue;
                        a.U[k] = V[i][q];
                        if constexpr (PLASMA) a.J[k] = J[i][q];
                    } else if (FRAME && k >= a.n_ei_pad) {
                        a.Uif[k - a.n_ei_pad] = neg ? -V[i][q] : V[i][q];
                    }
                }
            }
            if constexpr (FRAME) {
                if (has_cell) {
                    int I, Jc;
                    frame_ij(a.f, cell, I, Jc);
                    ((T*)a.f.Bx)[cell] = Bx;
                    ((T*)a.f.By)[cell] = By;
                    if (frame_is_cell(a.f, I, Jc - 1)) ((T*)a.f.H)[(int64_t)Jc * a.f.NX + I] = X[0];
                    if (frame_is_cell(a.f, I - 1, Jc)) ((T*)a.f.V)[(int64_t)Jc * (a.f.NX + 1) + I] = -X[2];
                }
            }
        }
    }
    if (tid == 0) {
        if (!ok) atomicOr(a.ctl + 2, 1u);
        if (blockIdx.x == 0) *a.step += a.n_steps;
        if constexpr (!SOLO) {
            // the last CTA moves the tags on: every CTA has read this launch's by then
            __threadfence();
            if (atomicAdd(a.ctl + 1, 1u) == gridDim.x - 1) {
                a.ctl[1] = 0u;
                a.ctl[0] = tag0 + (unsigned)a.n_steps + 1u;
                __threadfence();
            }
        }
    }
}

__global__ void k_flow_init(unsigned* ctl) {
    if (threadIdx.x == 0) {
        ctl[0] = 1u;   // words start with tag 0
        ctl[1] = ctl[2] = 0u;
    }
}

// Launch shapes, the first that fits.  One slot per thread keeps everything in registers (64 at
// 1,024 threads); eight at 512 threads (128 registers) keep the state in registers and read the
// coefficients from shared memory: 2.4 us per step on 500k triangles, the same as four slots at
// 1,024 threads, and 2.0 against 2.4 without a source.
struct FlowShape {
    int nt, ts;        // most threads, slots per thread
};
constexpr FlowShape kShapes[3] = {{1024, 1}, {1024, 2}, {512, 8}};

template <typename T, bool PLASMA, bool FRAME, bool SOLO, int SH>
cudaError_t launch_shape(const FlowArgs<T>& a, int grid, int threads, cudaStream_t s) {
    auto kern = k_flow<T, kShapes[SH].nt, kShapes[SH].ts, PLASMA, FRAME, SOLO>;
    const size_t smem = flow_smem<T, PLASMA>(kCoefRegs<T, kShapes[SH].ts>, kShapes[SH].ts * threads, a.hcap, a.scap, FRAME ? a.fper : 0);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = SOLO ? 0 : 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template <typename T, bool PLASMA, bool FRAME>
cudaError_t launch_flow_pf(const FlowArgs<T>& a, const FlowDev& fl, cudaStream_t s) {
    if (fl.grid == 1) {
        if constexpr (FRAME) return cudaErrorInvalidValue;
        else {
            if (fl.shape == 0) return launch_shape<T, PLASMA, false, true, 0>(a, 1, fl.threads, s);
            return launch_shape<T, PLASMA, false, true, 1>(a, 1, fl.threads, s);
        }
    }
    if (fl.shape == 0) return launch_shape<T, PLASMA, FRAME, false, 0>(a, fl.grid, fl.threads, s);
    if (fl.shape == 1) return launch_shape<T, PLASMA, FRAME, false, 1>(a, fl.grid, fl.threads, s);
    if constexpr (sizeof(T) == 4) return launch_shape<T, PLASMA, FRAME, false, 2>(a, fl.grid, fl.threads, s);
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_flow_t(const FlowDev& fl, const DevMesh& m, void* Uif, int n_steps, int gbase, cudaStream_t s) {
    FlowArgs<T> a;
    a.tri = m.tri;
    a.rl = m.rl;
    a.cU = (const T*)m.cU;
    a.cB64 = (const double*)m.cB;
    a.U = (T*)m.U;
    a.B = (T*)m.B;
    a.pb = (const T*)m.pb;
    a.J = (T*)m.J;
    a.pa = (T)m.pa;
    a.mdt = (T)(-m.dt);
    a.hash = m.src_hash;
    a.bits = (unsigned)m.src_bits;
    a.src_c = (const T*)m.src_c;
    a.src_grp = m.src_grp;
    a.gtab = m.gtab;
    a.gstride = m.gtab_size;
    a.gbase = gbase;
    a.has_src = m.n_src > 0;
    a.n_grp = m.n_grp;
    a.n_t = (int)m.n_t;
    a.n_ei = (int)m.n_ei;
    a.n_ei_pad = (int)m.n_ei_pad;
    a.per = fl.per;
    a.hcap = fl.hcap;
    a.scap = fl.scap;
    a.slots[0] = fl.slots;
    a.slots[1] = fl.slots + fl.slot_words;
    a.ctl = fl.ctl;
    a.step = m.step;
    a.n_steps = n_steps;
    a.skip = fl.skip;
    if (m.frame) a.f = *m.frame;
    a.Uif = (T*)Uif;
    a.fper = fl.fper;
    if (m.frame) return m.plasma ? launch_flow_pf<T, true, true>(a, fl, s) : launch_flow_pf<T, false, true>(a, fl, s);
    return m.plasma ? launch_flow_pf<T, true, false>(a, fl, s) : launch_flow_pf<T, false, false>(a, fl, s);
}

constexpr size_t kFlowSmem = 226 * 1024;

}  // namespace

bool flow_plan(int64_t n_t, int64_t n_fc, bool f64, int sms, FlowDev& fl) {
    fl = FlowDev();
    if (n_t < 1 || sms < 1 || n_t + n_fc >= kCellFar / 2) return false;
    const int esz = f64 ? 8 : 4;
    // one CTA holds up to 2,048 triangles: without an exchange its step takes 0.35-0.5 us, less
    // than the 1.2 us of one
    if (n_fc == 0 && n_t <= 2048) {
        fl.grid = 1;
        fl.shape = n_t <= 1024 ? 0 : 1;
        fl.per = (int)n_t;
    } else {
        const int64_t per = (n_t + sms - 1) / sms, fper = (n_fc + sms - 1) / sms;
        fl.shape = -1;
        for (int i = 0; i < (f64 ? 2 : 3) && fl.shape < 0; ++i)
            if (per <= (int64_t)kShapes[i].nt * kShapes[i].ts && fper <= kShapes[i].nt) fl.shape = i;
        if (fl.shape < 0) return false;
        fl.per = (int)((per + 31) / 32 * 32);
        fl.per = std::min(fl.per, kShapes[fl.shape].nt * kShapes[fl.shape].ts);
        fl.grid = std::max((int)((n_t + fl.per - 1) / fl.per), 2);
        if (n_fc > 0) fl.grid = std::max<int>(fl.grid, (int)std::min<int64_t>(sms, (n_fc + 63) / 64));
        fl.fper = (int)((n_fc + fl.grid - 1) / fl.grid);
        if (fl.fper > kShapes[fl.shape].nt) return false;
    }
    const int ts = kShapes[fl.shape].ts;
    fl.threads = ts > 1 ? kShapes[fl.shape].nt : std::min((std::max(fl.per, fl.fper) + 31) / 32 * 32, kShapes[fl.shape].nt);
    const int cap = ts * fl.threads;
    // what shared memory the coefficients (with a current's, which may come later) and the own
    // B values leave goes to the lists: source edges, then remote neighbours
    const bool cr = (f64 ? 8 : 4) * ts <= 8;   // kCoefRegs
    const size_t fixed = f64 ? flow_smem<double, true>(cr, cap, 0, 0, fl.fper) : flow_smem<float, true>(cr, cap, 0, 0, fl.fper);
    if (fixed + 8192 > kFlowSmem) return false;
    const size_t left = kFlowSmem - fixed;
    fl.scap = (int)std::min<size_t>(std::min(cap, 0x8000), left / 3 / (f64 ? 32 : 16)) & ~1;
    if (fl.grid > 1)
        fl.hcap = (int)std::min(std::min<size_t>((size_t)3 * cap + 4 * (size_t)fl.fper,
                                                 (left - (size_t)fl.scap * (f64 ? 32 : 16)) / (2 * esz + 4)),
                                (size_t)(65536 / esz - cap)) & ~3;   // 16-bit byte offsets
    fl.slot_words = fl.grid > 1 ? (n_t + n_fc) * (f64 ? 2 : 1) : 0;
    return true;
}

cudaError_t launch_flow_init(const FlowDev& fl, cudaStream_t s) {
    k_flow_init<<<1, 32, 0, s>>>(fl.ctl);
    return cudaGetLastError();
}

cudaError_t launch_flow(const FlowDev& fl, const DevMesh& m, void* Uif, int n_steps, int gbase, cudaStream_t s) {
    if (n_steps < 1) return cudaErrorInvalidValue;
    return m.precision == UE_PREC_FP64 ? launch_flow_t<double>(fl, m, Uif, n_steps, gbase, s)
                                       : launch_flow_t<float>(fl, m, Uif, n_steps, gbase, s);
}

}  // namespace ue
