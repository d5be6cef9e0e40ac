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
// barrier, then every triangle reads its neighbours there; with one triangle per thread, where a step
// is all latency, each thread polls its own (90k triangles: 0.97 us per step with the list, now 0.84;
// with several slots a thread's polls hold up its others).  All CTAs are resident (cooperative
// launch) and every wait is bounded: one that runs out sets the error word and ends the launch.
//
// A plan made once (k_flow_plan, after the source is set) orders each CTA's triangles into slots:
// those that publish first, so that their values travel while the rest is computed, then those
// with a source or a conductor's edge, so that few warps take that branch, then the others in
// stored order; and it turns each triangle's neighbours into shared-memory addresses.
//
// What bounds it: one exchange through L2 (store, poll, barrier: about 0.8 us) up to some 1,000
// triangles per SM, then that exchange and the latency of a slot's chain of shared gathers and arithmetic
// at 16 warps per SM (500k triangles: issue slots 32% busy, the shared-memory path 42%; an instruction
// waits 11.5 cycles, 3.7 of them for the words of other CTAs and 1.4 at the barrier; about 25 instructions
// per triangle, everything a slot needs at a compile-time offset from one register).  Measured per step on GB300, with a line
// source, against graph replays of the two plain kernels: 90k triangles 0.84 us (6.2), 305k 1.20,
// 1.2M 3.06 (9.3); one CTA alone 0.41 us on 1,040 triangles, 0.30 without a source (2.9).  Against
// k_tbp (8 steps per launch, ring-ordered tiles) on 500k triangles 1.38 us (5.0), with a plasma
// current 1.70 (k_tb 4.7), with a 16-cell PML frame 1.75 (10.0: the frame's tiles step by plain
// launches).  With slots in stored order, neighbours found at each launch and unpacked addresses
// hoisted into (then spilled) registers the same steps took 1.23, 1.89, -, 0.52, 2.44, 4.4 and 4.3.
// 1,024 threads leave 64 registers each.  What still spills, in bytes of stores and loads per thread: two
// slots with a current 44 and 56, with a frame 76 and 96, with both 196 and 216; the 16-slot shape, on
// 512 threads, 152 and 172; FP64 with a frame, where a thread
// computes its triangle's three edges, 380 to 1,032 and 464 to 1,168 (146k triangles with a 16-cell
// frame: 8.1 us per step with a current, the launches 12.1).
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "exchange.cuh"
#include "frame.cuh"

namespace ue {

namespace {

// Launch shapes, the first that fits: threads of a CTA, triangle slots per thread, and remote
// neighbours a CTA lists (FP32, FP64).  Up to two slots (one in FP64) the coefficients sit in
// registers too, else in shared memory.  The last shape is for vacuum media without a frame: 6 words
// of state per slot leave room for 16 of them, a current's 9 do not.
struct FlowShape {
    int nt, ts, halo32, halo64;
};
constexpr FlowShape kShapes[4] = {{1024, 1, 3072, 3072}, {1024, 2, 6144, 3072}, {512, 8, 3456, 0}, {512, 16, 2560, 0}};
constexpr int kVacuumShape = 3;
template <typename T, int SH>
constexpr int kHalo = sizeof(T) == 4 ? kShapes[SH].halo32 : kShapes[SH].halo64;
template <typename T, int SH>
constexpr int kBuffer = kShapes[SH].nt * kShapes[SH].ts + kHalo<T, SH>;   // B values per buffer

// Slot record {triangle, n01, n2f, 0}: byte offsets of the three neighbours' B in a buffer, 16 bits
// each (own slots, then the CTA's remote neighbours), and flags above the third.
constexpr unsigned kSrc = 1u << 16;     // 3 bits: the edge has a source
constexpr unsigned kWall = 1u << 19;    // 3 bits: a conductor's edge (the offset is the slot's own)
constexpr unsigned kIface = 1u << 22;   // 3 bits: the edge borders a frame cell

template <typename T>
struct Vec4 {
    T x, y, z, w;
};
template <>
struct __align__(16) Vec4<float> {
    float x, y, z, w;
};

// A source triangle's s_q dt |e| a of its edges (0 without a source) and its group's offset in the g
// table; indexed like the slot records.
template <typename T>
struct SrcEntry {
    T c[3];
    int g;
};
template <>
struct __align__(16) SrcEntry<float> {
    float c[3];
    int g;
};
template <>
struct __align__(16) SrcEntry<double> {
    double c[3];
    int g;
};

template <typename T>
struct FlowArgs {
    const int4* tri;
    const T* cU;
    const double* cB64;
    T* U;
    T* B;
    const T* pb;
    T* J;
    T pa, mdt;
    const int4* rec;        // cap per CTA
    const SrcEntry<T>* sent;
    const int* hlist;       // halo per CTA: places (CTA * cap + slot, then the frame cells)
    const int2* cnt;        // per CTA: publishing triangles, remote neighbours
    const int4* crec;       // fper per CTA: offsets of a frame cell's neighbours, -1 none
    const int2* erec;       // FP64 without a frame: edge records and {inner, all} edges per CTA
    const int2* ecnt;
    const double* gtab;
    int one_grp;            // one source group: its g is staged in shared memory
    int n_t, n_ei, n_ei_pad;
    int per;                // triangles per CTA
    unsigned long long* slots[2];
    unsigned* ctl;          // {tag of the next launch, CTAs done, error word, plan overflow}
    long long* step;
    int n_steps;
    int skip;               // tests only (-1 otherwise): this CTA returns at once
    FrameDev f;
    T* Uif;                 // circulations of the frame's interface edges
    int fper;               // frame cells per CTA
    FlowChecks chk;
    double* epart;
    unsigned* ecount;       // kFlowChecks counters
};

__device__ __forceinline__ bool neg_bit(float c) { return __float_as_uint(c) >> 31; }
__device__ __forceinline__ bool neg_bit(double c) { return (unsigned long long)__double_as_longlong(c) >> 63; }

struct PlanArgs {
    const int4* tri;
    const int2* rl;
    const void* cU;
    const int2* hash;
    unsigned bits;
    const void* src_c;
    const int32_t* src_grp;
    int gstride, has_src;
    int n_t, n_ei, n_ei_pad, per, cap, halo;
    int* place;             // [n_t]
    int4* rec;
    void* sent;
    int* hlist;
    int2* cnt;
    int4* crec;
    int2 *erec, *ecnt;
    int* eslot;
    int edges;              // edge records of a CTA
    unsigned* ctl;
    FrameDev f;
    int fper;
};

// the source index of stored edge k (k_edge_half's table), or -1
__device__ __forceinline__ int src_index(const PlanArgs& a, int k) {
    const unsigned size = 1u << a.bits;
    unsigned h = ((unsigned)k * 2654435761u) >> (32 - a.bits);
    int2 e = __ldg(a.hash + h);
    for (unsigned p = 1; e.x != k && p < size; ++p) {
        h = (h + 1) & (size - 1);
        e = __ldg(a.hash + h);
    }
    return e.x == k ? e.y : -1;
}

// The plan, one block per CTA of the resident launch.  First each triangle's place (CTA * cap +
// slot) and how many publish; then the records, and the CTA's remote neighbours as places.  A CTA
// with more of these than its list holds sets ctl[3]: the mesh then keeps its launches.
template <typename T>
__global__ void __launch_bounds__(1024) k_flow_order(const __grid_constant__ PlanArgs a) {
    __shared__ int wsum[3][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = blockIdx.x * a.per, nloc = max(0, min(a.per, a.n_t - j0));
    const T* cU = (const T*)a.cU;
    // class 0: a neighbour in another CTA (or a frame cell), 1: a source or a conductor, 2: others
    auto classify = [&](int l) {
        const int4 t = __ldg(a.tri + j0 + l);
        const int code[3] = {t.x, t.y, t.z};
        int cls = 2;
        for (int q = 0; q < 3; ++q) {
            const int k = code[q] >> 1;
            if (k < a.n_ei) {
                const int2 r = __ldg(a.rl + k);
                const int o = (code[q] & 1) ? r.x : r.y;
                if (o < j0 || o >= j0 + nloc) return 0;
                if (a.has_src && neg_bit(__ldg(cU + k))) cls = 1;
            } else if (k >= a.n_ei_pad && a.fper > 0) {
                return 0;
            } else {
                cls = 1;
            }
        }
        return cls;
    };
    int cls[8];   // of local triangles tid + 1024 i (cap <= 8192)
    int total[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (1024 * i >= a.per) break;
        const int l = tid + 1024 * i;
        cls[i] = l < nloc ? classify(l) : -1;
        for (int k = 0; k < 3; ++k) total[k] += __syncthreads_count(cls[i] == k);
    }
    int base[3] = {0, total[0], total[0] + total[1]};
#pragma unroll
    for (int i = 0; i < 8; ++i) {   // stable: rank in class, in stored order
        if (1024 * i >= a.per) break;
        const int l = tid + 1024 * i;
        unsigned m[3];
        for (int k = 0; k < 3; ++k) {
            m[k] = __ballot_sync(0xffffffffu, cls[i] == k);
            if (lane == 0) wsum[k][warp] = __popc(m[k]);
        }
        __syncthreads();
        for (int k = 0; k < 3; ++k) {
            int before = 0, all = 0;
            for (int w = 0; w < 32; ++w) {
                before += w < warp ? wsum[k][w] : 0;
                all += wsum[k][w];
            }
            if (cls[i] == k)
                a.place[j0 + l] = (int)blockIdx.x * a.cap + base[k] + before + __popc(m[k] & ((1u << lane) - 1u));
            base[k] += all;
        }
        __syncthreads();
    }
    if (tid == 0) a.cnt[blockIdx.x].x = total[0];
}

template <typename T>
__global__ void __launch_bounds__(1024) k_flow_plan(const __grid_constant__ PlanArgs a) {
    __shared__ int s_halo;
    const int tid = threadIdx.x;
    const int j0 = blockIdx.x * a.per, nloc = max(0, min(a.per, a.n_t - j0)), p0 = (int)blockIdx.x * a.cap;
    const int cell0 = (int)gridDim.x * a.cap;   // place of frame cell 0
    const T* cU = (const T*)a.cU;
    if (tid == 0) s_halo = 0;
    __syncthreads();
    int* hl = a.hlist + (size_t)blockIdx.x * a.halo;
    auto remote = [&](int place) -> unsigned {   // its offset; the first of the list when that is full
        const int h = atomicAdd(&s_halo, 1);
        if (h >= a.halo) return (unsigned)a.cap * (unsigned)sizeof(T);
        hl[h] = place;
        return (unsigned)(a.cap + h) * (unsigned)sizeof(T);
    };
    for (int l = tid; l < nloc; l += 1024) {
        const int slot = a.place[j0 + l] - p0;
        const int4 t = __ldg(a.tri + j0 + l);
        const int code[3] = {t.x, t.y, t.z};
        unsigned off[3], f = 0;
        SrcEntry<T> se{{T(0), T(0), T(0)}, 0};
        for (int q = 0; q < 3; ++q) {
            const int k = code[q] >> 1;
            off[q] = (unsigned)slot * (unsigned)sizeof(T);
            if (k < a.n_ei) {
                const int2 r = __ldg(a.rl + k);
                const int o = (code[q] & 1) ? r.x : r.y, place = a.place[o];
                if (o >= j0 && o < j0 + nloc) off[q] = (unsigned)(place - p0) * (unsigned)sizeof(T);
                else off[q] = remote(place);
                const int x = a.has_src && neg_bit(__ldg(cU + k)) ? src_index(a, k) : -1;
                if (x >= 0) {
                    const T sc = __ldg((const T*)a.src_c + x);
                    se.c[q] = (code[q] & 1) ? -sc : sc;
                    se.g = (int)__ldg(a.src_grp + x) * a.gstride;
                    f |= kSrc << q;
                }
            } else if (k >= a.n_ei_pad && a.fper > 0) {
                off[q] = remote(cell0 + a.f.icell[k - a.n_ei_pad]);
                f |= kIface << q;
            } else {
                f |= kWall << q;
            }
        }
        a.rec[p0 + slot] = make_int4(j0 + l, (int)(off[0] | (off[1] << 16)), (int)(off[2] | f), 0);
        if (f & (7u * kSrc)) ((SrcEntry<T>*)a.sent)[p0 + slot] = se;
    }
    for (int t = tid; t < a.fper; t += 1024) {
        const int cell = (int)blockIdx.x * a.fper + t;
        if (cell >= (int)a.f.n_fc) break;
        const FrameDev& f = a.f;
        int I, J;
        frame_ij(f, cell, I, J);
        const bool in_x = I >= f.W && I < f.W + f.nx, in_y = J >= f.W && J < f.W + f.ny;
        const int di[4] = {0, 0, -1, 1}, dj[4] = {-1, 1, 0, 0};   // bottom, top, left, right
        const int kif[4] = {in_x && J == f.W + f.ny ? f.nx + (I - f.W) : -1, in_x && J == f.W - 1 ? I - f.W : -1,
                            in_y && I == f.W + f.nx ? 2 * f.nx + f.ny + (J - f.W) : -1,
                            in_y && I == f.W - 1 ? 2 * f.nx + (J - f.W) : -1};
        int cn[4];
        for (int d = 0; d < 4; ++d) {
            cn[d] = -1;
            if (frame_is_cell(f, I + di[d], J + dj[d])) {
                cn[d] = (int)remote(cell0 + (int)frame_cell(f, I + di[d], J + dj[d]));
            } else if (kif[d] >= 0) {
                const int code = f.itri[kif[d]];
                cn[d] = (int)remote(a.place[code >= 0 ? code : ~code]);
            }
        }
        a.crec[cell] = make_int4(cn[0], cn[1], cn[2], cn[3]);
    }
    __syncthreads();
    if (tid == 0) {
        a.cnt[blockIdx.x].y = min(s_halo, a.halo);
        if (s_halo > a.halo) atomicOr(a.ctl + 3, 1u);
    }
}

template <typename T, int TS>
constexpr bool kCoefRegs = sizeof(T) * TS <= 8;

// Shared memory of a CTA: two buffers of B, the coefficients (with a current's), g, the remote
// neighbours, the frame cells' coefficients.
template <typename T, bool PLASMA, int SH>
constexpr size_t flow_smem(int cells) {
    const size_t cap = (size_t)kShapes[SH].nt * kShapes[SH].ts;
    return 2 * sizeof(T) * (size_t)kBuffer<T, SH> +
           (kCoefRegs<T, kShapes[SH].ts> ? 0 : sizeof(T) * cap * (PLASMA ? 7 : 4)) + sizeof(T) * (size_t)kFlowSteps +
           4 * (size_t)kHalo<T, SH> + 3 * sizeof(Vec4<T>) * (size_t)cells;
}

// Shared accesses at an address plus a compile-time offset.  A step's loads read the buffer that
// its stores do not touch, so they may move among the stores.
template <int OFF>
__device__ __forceinline__ float lds_at(uint32_t addr, float) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(addr), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ double lds_at(uint32_t addr, double) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1+%2];" : "=d"(v) : "r"(addr), "n"(OFF));
    return v;
}
// The same at the address in the low (HI = false) or high half of a word; one volatile statement, as
// the unpacked addresses of all slots, hoisted out of the step loop, would not fit the registers.
template <int OFF, bool HI>
__device__ __forceinline__ float lds_half(unsigned w, float) {
    float v;
    if constexpr (HI) asm volatile("{.reg .b32 t; shr.u32 t, %1, 16; ld.shared.f32 %0, [t+%2];}" : "=f"(v) : "r"(w), "n"(OFF));
    else asm volatile("{.reg .b32 t; and.b32 t, %1, 65535; ld.shared.f32 %0, [t+%2];}" : "=f"(v) : "r"(w), "n"(OFF));
    return v;
}
template <int OFF, bool HI>
__device__ __forceinline__ double lds_half(unsigned w, double) {
    double v;
    if constexpr (HI) asm volatile("{.reg .b32 t; shr.u32 t, %1, 16; ld.shared.f64 %0, [t+%2];}" : "=d"(v) : "r"(w), "n"(OFF));
    else asm volatile("{.reg .b32 t; and.b32 t, %1, 65535; ld.shared.f64 %0, [t+%2];}" : "=d"(v) : "r"(w), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ Vec4<float> lds4_at(uint32_t addr, float) {
    Vec4<float> v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4+%5];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ Vec4<double> lds4_at(uint32_t addr, double) {
    Vec4<double> v;
    asm volatile("ld.shared.v2.f64 {%0,%1}, [%2+%3];" : "=d"(v.x), "=d"(v.y) : "r"(addr), "n"(OFF));
    asm volatile("ld.shared.v2.f64 {%0,%1}, [%2+%3];" : "=d"(v.z), "=d"(v.w) : "r"(addr), "n"(OFF + 16));
    return v;
}
template <int OFF>
__device__ __forceinline__ void sts_at(uint32_t addr, float v) {
    asm volatile("st.shared.f32 [%0+%1], %2;" ::"r"(addr), "n"(OFF), "f"(v));
}
template <int OFF>
__device__ __forceinline__ void sts_at(uint32_t addr, double v) {
    asm volatile("st.shared.f64 [%0+%1], %2;" ::"r"(addr), "n"(OFF), "d"(v));
}

// slot_put at a pointer plus a compile-time number of values, and a source entry likewise: one
// pointer per thread serves all its slots.
template <int N>
__device__ __forceinline__ void slot_put_at(unsigned long long* s, unsigned tag, float v) {
    const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0+%1], %2;" ::"l"(s), "n"(8 * N), "l"(w) : "memory");
}
template <int N>
__device__ __forceinline__ void slot_put_at(unsigned long long* s, unsigned tag, double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0+%1], {%2, %3};" ::"l"(s), "n"(16 * N), "l"(t | (b & 0xFFFFFFFFull)),
                 "l"(t | (b >> 32))
                 : "memory");
}
template <int N>
__device__ __forceinline__ SrcEntry<float> entry_at(const SrcEntry<float>* e) {
    SrcEntry<float> v;
    asm volatile("ld.global.nc.v4.b32 {%0,%1,%2,%3}, [%4+%5];"
                 : "=f"(v.c[0]), "=f"(v.c[1]), "=f"(v.c[2]), "=r"(v.g)
                 : "l"(e), "n"((int)sizeof(v) * N));
    return v;
}
template <int N>
__device__ __forceinline__ SrcEntry<double> entry_at(const SrcEntry<double>* e) {
    SrcEntry<double> v;
    asm volatile("ld.global.nc.v2.f64 {%0,%1}, [%2+%3];" : "=d"(v.c[0]), "=d"(v.c[1]) : "l"(e), "n"((int)sizeof(v) * N));
    asm volatile("ld.global.nc.f64 %0, [%1+%2];" : "=d"(v.c[2]) : "l"(e), "n"((int)sizeof(v) * N + 16));
    asm volatile("ld.global.nc.b32 %0, [%1+%2];" : "=r"(v.g) : "l"(e), "n"((int)sizeof(v) * N + 24));
    return v;
}

// A thread holds slots tid + i * NT, i < TS.  SOLO: one CTA holds the whole mesh, nothing is
// published.
template <typename T, int SH, bool PLASMA, bool FRAME, bool SOLO>
struct Flow {
    static constexpr int NT = kShapes[SH].nt, TS = kShapes[SH].ts, CAP = NT * TS;
    static constexpr int STRIDE = kBuffer<T, SH> * (int)sizeof(T);   // bytes between the two buffers
    static constexpr bool CR = kCoefRegs<T, TS>;
    static constexpr bool OWN = TS == 1 && !FRAME && !SOLO;   // threads poll for themselves
    static_assert(STRIDE + 2048 < 65536, "16-bit shared addresses");

    T V[TS][3], J[PLASMA ? TS : 1][3], b[TS];
    Vec4<T> Cr[CR ? TS : 1];
    T Pr[CR && PLASMA ? TS : 1][3];
    unsigned n01[TS], n2f[TS];
    int at[OWN ? 3 : 1];    // places of the remote neighbours, -1: the neighbour is in this CTA
    // frame cell: sides X in bottom, top, left, right order, each with the cell's own
    // counter-clockwise sign, so that every one advances by (own B - neighbour's B)
    T X[FRAME ? 4 : 1], Bx, By;
    int cn[FRAME ? 4 : 1];
    unsigned ifm;           // sides that are interface edges: no decay, one fused multiply-add
    bool has_cell, ok;
    int nloc, npub, hn;
    uint32_t bufs, own;     // shared addresses: the buffers, this thread's first slot
    Vec4<T>* C;
    T* P;
    Vec4<T>* Fc;
    T* gs;
    int* hl;
    unsigned tag0;
    unsigned long long* put[2];   // this thread's first slot's exchange words
    const SrcEntry<T>* sent;      // its first source entry

    __device__ __forceinline__ void setup(const FlowArgs<T>& a, unsigned char* sm) {
        const int tid = threadIdx.x;
        bufs = smem_addr(sm);
        own = bufs + (uint32_t)tid * (uint32_t)sizeof(T);
        C = reinterpret_cast<Vec4<T>*>(sm + 2 * STRIDE);
        P = reinterpret_cast<T*>(C + (CR ? 0 : CAP));
        Fc = reinterpret_cast<Vec4<T>*>(P + (CR || !PLASMA ? 0 : 3 * CAP));
        gs = reinterpret_cast<T*>(Fc + (FRAME ? 3 * a.fper : 0));
        hl = reinterpret_cast<int*>(gs + kFlowSteps);
        const int j0 = blockIdx.x * a.per;
        nloc = max(0, min(a.per, a.n_t - j0));
        const int2 cn2 = __ldg(a.cnt + blockIdx.x);
        npub = SOLO ? 0 : cn2.x;
        hn = SOLO || OWN ? 0 : cn2.y;
        tag0 = SOLO ? 0u : *(volatile unsigned*)a.ctl;
        ok = true;
        const size_t first = (size_t)blockIdx.x * CAP + tid;
        for (int p = 0; p < 2; ++p) put[p] = a.slots[p] + first * (sizeof(T) / 4);
        sent = a.sent + first;
        const int4* rec = a.rec + (size_t)blockIdx.x * CAP;
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = tid + i * NT;
            n01[i] = n2f[i] = 0;
            b[i] = T(0);
            if (l >= nloc) continue;
            const int4 r = __ldg(rec + l);
            n01[i] = (unsigned)r.y + (bufs | (bufs << 16));
            n2f[i] = (unsigned)r.z + bufs;
            if constexpr (OWN) {
                const unsigned off[3] = {(unsigned)r.y & 0xFFFFu, (unsigned)r.y >> 16, (unsigned)r.z & 0xFFFFu};
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int h = (int)(off[q] / (unsigned)sizeof(T)) - CAP;
                    at[q] = h < 0 ? -1 : __ldg(a.hlist + (size_t)blockIdx.x * kHalo<T, SH> + h);
                }
            }
            const int4 t = __ldg(a.tri + r.x);
            const int code[3] = {t.x, t.y, t.z};
            T c[3], pb[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int k = code[q] >> 1;
                const bool neg = code[q] & 1;
                c[q] = pb[q] = V[i][q] = T(0);
                if constexpr (PLASMA) J[i][q] = T(0);
                if (k < a.n_ei) {
                    const T u = a.U[k];
                    c[q] = fabs(__ldg(a.cU + k));
                    V[i][q] = neg ? -u : u;
                    if constexpr (PLASMA) {
                        const T jj = a.J[k];
                        J[i][q] = neg ? -jj : jj;
                        pb[q] = __ldg(a.pb + k);
                    }
                } else if (FRAME && k >= a.n_ei_pad) {
                    const T u = a.Uif[k - a.n_ei_pad];
                    c[q] = ((const T*)a.f.icU)[k - a.n_ei_pad];
                    V[i][q] = neg ? -u : u;
                }
            }
            T cb;
            if constexpr (sizeof(T) == 4) cb = __int_as_float(t.w);
            else cb = __ldg(a.cB64 + r.x);
            const Vec4<T> cv{c[0], c[1], c[2], cb};
            if constexpr (CR) Cr[i] = cv;
            else C[l] = cv;
            if constexpr (PLASMA) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if constexpr (CR) Pr[i][q] = pb[q];
                    else P[q * CAP + l] = pb[q];
                }
            }
            b[i] = a.B[r.x];
            reinterpret_cast<T*>(sm)[l] = b[i];
        }
        has_cell = false;
        if constexpr (FRAME) {
            const int cell = (int)blockIdx.x * a.fper + tid;
            has_cell = tid < a.fper && cell < (int)a.f.n_fc;
            ifm = 0;
            Bx = By = T(0);
            if (has_cell) {
                const FrameDev& f = a.f;
                const Tab<T> tb = tabs<T>(f);
                T ca[4], cd[4];
                int I, Jc;
                frame_ij(f, cell, I, Jc);
                const int4 cr = __ldg(a.crec + cell);
                const int off[4] = {cr.x, cr.y, cr.z, cr.w};
                const int di[4] = {0, 0, -1, 1}, dj[4] = {-1, 1, 0, 0};
                const int kif[4] = {f.nx + (I - f.W), I - f.W, 2 * f.nx + f.ny + (Jc - f.W), 2 * f.nx + (Jc - f.W)};
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    X[d] = ca[d] = cd[d] = T(0);
                    cn[d] = off[d] < 0 ? -1 : (int)bufs + off[d];
                    if (off[d] < 0) continue;
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
                    } else {   // interface edge kif[d]
                        const T u = a.Uif[kif[d]];
                        X[d] = f.itri[kif[d]] >= 0 ? -u : u;
                        ifm |= 1u << d;
                        cd[d] = ((const T*)f.icU)[kif[d]];
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
            for (int e = tid; e < hn; e += NT) hl[e] = __ldg(a.hlist + (size_t)blockIdx.x * kHalo<T, SH> + e);
            // published only after this thread's reads of U, J and the frame are done: their
            // owners write them back after later steps
            __threadfence();
#pragma unroll
            for (int i = 0; i < TS; ++i)
                if (tid + i * NT < npub) slot_put(a.slots[0], (int)blockIdx.x * CAP + tid + i * NT, tag0, b[i]);
            if (FRAME && has_cell) slot_put(a.slots[0], ((int)gridDim.x * CAP) + (int)blockIdx.x * a.fper + tid, tag0, rn_add(Bx, By));
        }
        if (a.one_grp)
            for (int e = tid; e < a.n_steps; e += NT) gs[e] = (T)__ldg(a.gtab + e);
        __syncthreads();
    }

    // Step s + 1 from the B of step s in buffer PB = s & 1.
    template <int PB>
    __device__ __forceinline__ bool step(const FlowArgs<T>& a, int s) {
        constexpr int RD = PB * STRIDE;
        const int tid = threadIdx.x;
        const unsigned tag = tag0 + (unsigned)s;
        if constexpr (SOLO) {
            if (s > 0) __syncthreads();
        } else if constexpr (!OWN) {
            // the remote neighbours' B, a few polls in flight per thread
            constexpr int kPoll = 4;
            const unsigned long long* sl = a.slots[PB];
            for (int e0 = tid; e0 < hn; e0 += kPoll * NT) {
                Word<T> w[kPoll];
#pragma unroll
                for (int u = 0; u < kPoll; ++u)
                    if (e0 + u * NT < hn) w[u].load(sl, hl[e0 + u * NT]);
#pragma unroll
                for (int u = 0; u < kPoll; ++u) {
                    const int e = e0 + u * NT;
                    if (e < hn) {
                        if (!word_wait(w[u], sl, hl[e], tag)) ok = false;
                        sts_at<RD>(bufs + (uint32_t)(CAP + e) * (uint32_t)sizeof(T), w[u].value());
                    }
                }
            }
            ok = __syncthreads_and(ok ? 1 : 0) != 0;
            if (!ok) return false;
        }
        if constexpr (FRAME) {
            if (has_cell) {
                const T F = rn_add(Bx, By);
                const Vec4<T> va = Fc[3 * tid], vd = Fc[3 * tid + 1], vc = Fc[3 * tid + 2];
                const T ca[4] = {va.x, va.y, va.z, va.w}, cd[4] = {vd.x, vd.y, vd.z, vd.w};
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    if (cn[d] < 0) continue;
                    const T df = rn_sub(F, lds_at<RD>((uint32_t)cn[d], T(0)));
                    X[d] = (ifm >> d) & 1u ? rn_fma(cd[d], df, X[d]) : rn_fma(ca[d], X[d], rn_mul(cd[d], df));
                }
                Bx = rn_sub(rn_mul(vc.x, Bx), rn_mul(vc.y, rn_add(X[3], X[2])));
                By = rn_sub(rn_mul(vc.z, By), rn_mul(vc.w, rn_add(X[0], X[1])));
                slot_put(a.slots[PB ^ 1], (int)gridDim.x * CAP + (int)blockIdx.x * a.fper + tid, tag + 1u, rn_add(Bx, By));
            }
        }
        slots_from<PB, 0>(a, s, tag);
        if constexpr (OWN) ok = __syncthreads_and(ok ? 1 : 0) != 0;
        return ok;
    }

    template <int PB, int I>
    __device__ __forceinline__ void slots_from(const FlowArgs<T>& a, int s, unsigned tag) {
        if constexpr (I < TS) {
            constexpr int RD = PB * STRIDE, WR = (PB ^ 1) * STRIDE;
            // pb of the slot's edges, after the buffers and the coefficients
            constexpr int PS = CAP * (int)sizeof(T), PO = 2 * STRIDE + CAP * (int)sizeof(Vec4<T>) + I * NT * (int)sizeof(T);
            const int l = threadIdx.x + I * NT;
            if (l < nloc) {
                Vec4<T> c;
                if constexpr (CR) c = Cr[I];
                else c = lds4_at<2 * STRIDE + I * NT * (int)sizeof(Vec4<T>)>(bufs + threadIdx.x * (uint32_t)sizeof(Vec4<T>), T(0));
                const T cq[3] = {c.x, c.y, c.z};
                T nv[3];
                if (OWN && l < npub) {
                    Word<T> w[3];
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        if (at[q] >= 0) w[q].load(a.slots[PB], at[q]);
                    if (at[0] < 0) nv[0] = lds_half<RD, false>(n01[I], T(0));
                    if (at[1] < 0) nv[1] = lds_half<RD, true>(n01[I], T(0));
                    if (at[2] < 0) nv[2] = lds_half<RD, false>(n2f[I], T(0));
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        if (at[q] >= 0) {
                            if (!word_wait(w[q], a.slots[PB], at[q], tag)) ok = false;
                            nv[q] = w[q].value();
                        }
                } else {
                    nv[0] = lds_half<RD, false>(n01[I], T(0));
                    nv[1] = lds_half<RD, true>(n01[I], T(0));
                    nv[2] = lds_half<RD, false>(n2f[I], T(0));
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const T uo = V[I][q];
                    T un = rn_fma(cq[q], rn_sub(b[I], nv[q]), uo);
                    if constexpr (PLASMA) {
                        T pq;
                        if constexpr (CR) pq = Pr[I][q];
                        else pq = q == 0 ? lds_at<PO>(own, T(0)) : q == 1 ? lds_at<PO + PS>(own, T(0)) : lds_at<PO + 2 * PS>(own, T(0));
                        // an interface edge carries no current
                        const T x = FRAME && (n2f[I] & (kIface << q)) ? T(0) : rn_mul(pq, uo);
                        const T jn = rn_fma(a.pa, J[I][q], x);
                        un = rn_fma(a.mdt, jn, un);
                        J[I][q] = jn;
                    }
                    V[I][q] = un;
                }
                if (n2f[I] & (7u * (kSrc | kWall))) special<I>(a, s);
                b[I] = rn_fma(-c.w, rn_add(rn_add(V[I][0], V[I][1]), V[I][2]), b[I]);
                sts_at<WR + I * NT * (int)sizeof(T)>(own, b[I]);
                if (!SOLO && l < npub) slot_put_at<I * NT>(put[PB ^ 1], tag + 1u, b[I]);
            }
            slots_from<PB, I + 1>(a, s, tag);
        }
    }

    // Source terms, and conductors' edges, which stay 0 whatever the fields.
    template <int I>
    __device__ __forceinline__ void special(const FlowArgs<T>& a, int s) {
        if (n2f[I] & (7u * kSrc)) {
            const SrcEntry<T> se = entry_at<I * NT>(sent);
            const T g = a.one_grp ? gs[s] : (T)__ldg(a.gtab + se.g + s);
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (n2f[I] & (kSrc << q)) V[I][q] = rn_fma(se.c[q], g, V[I][q]);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (!(n2f[I] & (kWall << q))) continue;
            V[I][q] = T(0);
            if constexpr (PLASMA) J[I][q] = T(0);
        }
    }

    // This thread's share of the energy of eq. 8: its triangles' own terms and those of the edges that
    // they are R of.
    __device__ __forceinline__ double energy(const FlowArgs<T>& a) const {
        double x = 0.0;
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = threadIdx.x + i * NT;
            if (l >= nloc) break;
            const int j = __ldg(&a.rec[(size_t)blockIdx.x * CAP + l].x);
            const int4 t = __ldg(a.tri + j);
            const int code[3] = {t.x, t.y, t.z};
            x += __ldg(a.chk.S + j) * (double)b[i] * (double)b[i];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int k = code[q] >> 1;
                if (k < a.n_ei && !(code[q] & 1)) x += __ldg(a.chk.we + k) * (double)V[i][q] * (double)V[i][q];
            }
        }
        return x;
    }

    // Each edge by its R triangle, each interface edge by its triangle, each frame side by the
    // cell above or to its right.
    __device__ __forceinline__ void write_back(const FlowArgs<T>& a) {
        const int tid = threadIdx.x;
        if (!SOLO) __threadfence();
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = tid + i * NT;
            if (l >= nloc) break;
            const int j = __ldg(&a.rec[(size_t)blockIdx.x * CAP + l].x);
            const int4 t = __ldg(a.tri + j);
            const int code[3] = {t.x, t.y, t.z};
            a.B[j] = b[i];
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
                const int cell = (int)blockIdx.x * a.fper + tid;
                int I, Jc;
                frame_ij(a.f, cell, I, Jc);
                ((T*)a.f.Bx)[cell] = Bx;
                ((T*)a.f.By)[cell] = By;
                if (frame_is_cell(a.f, I, Jc - 1)) ((T*)a.f.H)[(int64_t)Jc * a.f.NX + I] = X[0];
                if (frame_is_cell(a.f, I - 1, Jc)) ((T*)a.f.V)[(int64_t)Jc * (a.f.NX + 1) + I] = -X[2];
            }
        }
    }
};

// An energy check (check c of the launch) from the threads' shares, without leaving the launch: the
// last CTA to arrive sums the CTAs' shares in order and updates the watchdog.  Checks are handled
// in turn: the last arrival at one has arrived, and finished, at those before.  It is bound by the
// latency of its loads (three deep); ending the launch at every check instead and summing in two
// kernels cost 19 us more per check at 92k triangles (256 steps, a check every 32: 606 us, now 454 us).
template <bool SOLO, typename T>
__device__ __forceinline__ void energy_check(const FlowArgs<T>& a, int c, double x) {
    __shared__ double red[32];
    __shared__ bool last;
    const int tid = threadIdx.x;
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((tid & 31) == 0) red[tid >> 5] = x;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < (int)blockDim.x / 32; ++w) x += red[w];
        a.epart[(size_t)c * gridDim.x + blockIdx.x] = x;
        __threadfence();
        last = SOLO || atomicAdd(a.ecount + c, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last && tid < 32) {
        __threadfence();
        double w = 0.0;
        for (int i = tid; i < (int)gridDim.x; i += 32) w += __ldcg(a.epart + (size_t)c * gridDim.x + i);
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        if (tid == 0) {
            watchdog_update(a.chk.wd, w);
            __threadfence();
        }
    }
    __syncthreads();
}

// A launch of n_steps steps by F, with its checks.
template <typename F, bool SOLO, typename T>
__device__ __forceinline__ void flow_body(const FlowArgs<T>& a, unsigned char* sm) {
    const unsigned tag0 = SOLO ? 0u : *(volatile unsigned*)a.ctl;
    bool ok = true;
    if (SOLO || (int)blockIdx.x != a.skip) {
        F f;
        f.setup(a, sm);
        int c = 0, next = a.chk.first > 0 ? a.chk.first : a.n_steps + 1;
        bool go = true;
#pragma unroll 1
        for (int s = 0; s < a.n_steps && go;) {
            const int end = min(next, a.n_steps);
#pragma unroll 1
            for (;;) {
                if (!(s & 1)) {
                    if (!(go = f.template step<0>(a, s)) || ++s == end) break;
                }
                if (!(go = f.template step<1>(a, s)) || ++s == end) break;
            }
            if (go && (s == next || (s == a.n_steps && a.chk.end))) {
                energy_check<SOLO>(a, c++, f.energy(a));
                next += a.chk.period;
            }
        }
        ok = SOLO || __syncthreads_and(f.ok ? 1 : 0) != 0;
        if (ok) f.write_back(a);
    }
    if (threadIdx.x == 0) {
        if (!ok) atomicOr(a.ctl + 2, 1u);
        if (blockIdx.x == 0) *a.step += a.n_steps;
        if constexpr (!SOLO) {
            // the last CTA moves the tags on: every CTA has read this launch's by then
            __threadfence();
            if (atomicAdd(a.ctl + 1, 1u) == gridDim.x - 1) {
                if (a.chk.first > 0 || a.chk.end)
                    for (int i = 0; i < kFlowChecks; ++i) a.ecount[i] = 0u;
                a.ctl[1] = 0u;
                a.ctl[0] = tag0 + (unsigned)a.n_steps + 1u;
                __threadfence();
            }
        }
    }
}

template <typename T, int SH, bool PLASMA, bool FRAME, bool SOLO>
__global__ void __launch_bounds__(kShapes[SH].nt, 1) k_flow(const __grid_constant__ FlowArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    flow_body<Flow<T, SH, PLASMA, FRAME, SOLO>, SOLO>(a, smraw);
}

// --- FP64 without a frame -------------------------------------------------------------------
// GB300's FP64 pipe takes two lanes per SM and clock, so what counts is FP64 instructions, and a
// triangle's thread that computes its three edges computes every edge twice.  Here a thread holds
// edges (J and their addresses in registers, U and the coefficients in shared memory) and triangles (B):
// each step updates the edges once, U passing through shared memory, and sums the triangles:
// 10.5 FP64 instructions per triangle with a current instead of 18, plus one side of the edges whose
// other triangle is in another CTA.  Those come last in a CTA's edge list; the thread that holds one
// polls the other triangle's word itself, after the inner edges have been computed.  The larger shape
// spills: 84 bytes of stores and 212 of loads per thread, with a current 220 and 452.  On 241k
// triangles with a current a step takes 6.7 us, in vacuum 3.9 (9.9 with a triangle's edges in its thread,
// 11.9 as two launches).
struct EdgeShape {
    int ts, es, edges;   // triangle and edge slots per thread, edges of a CTA
};
constexpr EdgeShape kEdgeShapes[2] = {{1, 3, 3072}, {2, 5, 4608}};
// a CTA with all its triangles and a full list of remote neighbours has this many edges at most
static_assert(2 * kEdgeShapes[0].edges >= 3 * 1024 + kShapes[0].halo64 && 2 * kEdgeShapes[1].edges >= 3 * 2048 + kShapes[1].halo64);
constexpr unsigned kEdgeMask = (1u << 28) - 1, kEdgeSrc = 1u << 28, kEdgeOwn = 1u << 29;

// Accesses from packed words, each one volatile statement: hoisted out of the step loop, the
// unpacked addresses and signs would not fit the registers.
// the word of the place in an edge's w
__device__ __forceinline__ void word_at(Word<double>& x, const unsigned long long* sl, unsigned w) {
    asm volatile("{.reg .b32 i; .reg .b64 p; shr.u32 i, %3, 12; mad.wide.u32 p, i, 16, %2; ld.relaxed.gpu.global.v2.u64 {%0, %1}, [p];}"
                 : "=l"(x.a), "=l"(x.b)
                 : "l"(sl), "r"(w)
                 : "memory");
}
// word_wait of it
__device__ __forceinline__ bool word_wait_at(Word<double>& x, const unsigned long long* sl, unsigned w, unsigned tag) {
    if (x.ready(tag)) return true;
    const long long t0 = clock64();
    for (unsigned n = 1;; ++n) {
        word_at(x, sl, w);
        if (x.ready(tag)) return true;
        if ((n & 255u) == 0 && clock64() - t0 > (2LL << 30)) return false;
    }
}
// B of the slot in an edge's w
__device__ __forceinline__ double lds_slot(uint32_t bufs, unsigned w) {
    double v;
    asm volatile("{.reg .b32 t; and.b32 t, %1, 0xFFE; shl.b32 t, t, 2; add.u32 t, t, %2; ld.shared.f64 %0, [t];}"
                 : "=d"(v)
                 : "r"(w), "r"(bufs));
    return v;
}
// U at the address in a half of w, negated when bit 16 + Q of signs is set
template <bool HI, int Q>
__device__ __forceinline__ double lds_signed(unsigned w, unsigned signs) {
    double v;
    if constexpr (HI)
        asm volatile("{.reg .b32 t, s, l, h; shr.u32 t, %1, 16; shl.b32 s, %2, %3; and.b32 s, s, 0x80000000; ld.shared.v2.b32 {l, h}, [t]; xor.b32 h, h, s; mov.b64 %0, {l, h};}"
                     : "=d"(v)
                     : "r"(w), "r"(signs), "n"(15 - Q));
    else
        asm volatile("{.reg .b32 t, s, l, h; and.b32 t, %1, 65535; shl.b32 s, %2, %3; and.b32 s, s, 0x80000000; ld.shared.v2.b32 {l, h}, [t]; xor.b32 h, h, s; mov.b64 %0, {l, h};}"
                     : "=d"(v)
                     : "r"(w), "r"(signs), "n"(15 - Q));
    return v;
}

struct __align__(16) EdgeSrc {
    double c;
    long long g;
};
template <int N>
__device__ __forceinline__ EdgeSrc entry_at(const EdgeSrc* e) {
    EdgeSrc v;
    asm volatile("ld.global.nc.v2.b64 {%0,%1}, [%2+%3];" : "=d"(v.c), "=l"(v.g) : "l"(e), "n"((int)sizeof(v) * N));
    return v;
}

template <int SH, bool PLASMA>
struct EdgeFlow {
    static constexpr int NT = 1024, TS = kEdgeShapes[SH].ts, ES = kEdgeShapes[SH].es, NE = kEdgeShapes[SH].edges;
    static constexpr int CAP = NT * TS, VO = 8 * CAP, CO = VO + 8 * (NE + 2), PO = CO + 8 * NE, GO = PO + (PLASMA ? 8 * NE : 0);
    static constexpr size_t SMEM = GO + 8 * (size_t)kFlowSteps;
    static_assert(CO + 4096 < 65536, "16-bit shared addresses");
};

template <int SH, bool PLASMA, bool SOLO>
struct Flow64 : EdgeFlow<SH, PLASMA> {
    using L = EdgeFlow<SH, PLASMA>;
    static constexpr int NT = L::NT, TS = L::TS, ES = L::ES, NE = L::NE, CAP = L::CAP, VO = L::VO, CO = L::CO, PO = L::PO;

    double J[PLASMA ? ES : 1], b[TS], cB[TS];
    unsigned w[ES];         // inner: shared addresses of B_R, B_L; cut: place << 12 | slot << 1 | here is R
    unsigned n01[TS], n2s[TS];   // shared addresses of the three U, signs (1: negative) from bit 16
    unsigned src;           // bit i: edge slot i has a source
    int ni, ne, nloc, npub;
    uint32_t bufs, own;
    double* gs;
    unsigned tag0;
    bool ok;
    unsigned long long* put[2];
    const EdgeSrc* sent;

    __device__ __forceinline__ void setup(const FlowArgs<double>& a, unsigned char* sm) {
        const int tid = threadIdx.x;
        bufs = smem_addr(sm);
        own = bufs + 8u * (uint32_t)tid;
        gs = reinterpret_cast<double*>(sm + L::GO);
        nloc = max(0, min(a.per, a.n_t - (int)blockIdx.x * a.per));
        npub = SOLO ? 0 : __ldg(&a.cnt[blockIdx.x].x);
        const int2 en = __ldg(a.ecnt + blockIdx.x);
        ni = en.x;
        ne = en.y;
        tag0 = SOLO ? 0u : *(volatile unsigned*)a.ctl;
        ok = true;
        const size_t first = (size_t)blockIdx.x * CAP + tid;
        for (int p = 0; p < 2; ++p) put[p] = a.slots[p] + 2 * first;
        const size_t e0 = (size_t)blockIdx.x * NE + tid;
        sent = reinterpret_cast<const EdgeSrc*>(a.sent) + e0;
        src = 0;
#pragma unroll
        for (int i = 0; i < ES; ++i) {
            const int e = tid + i * NT;
            w[i] = 0;
            if constexpr (PLASMA) J[i] = 0.0;
            if (e >= ne) continue;
            const int2 r = __ldg(a.erec + e0 + i * NT);
            const int k = r.x & kEdgeMask;
            if (r.x & kEdgeSrc) src |= 1u << i;
            w[i] = (unsigned)r.y + (e < ni ? bufs | (bufs << 16) : 0u);
            *reinterpret_cast<double*>(sm + VO + 8 * e) = a.U[k];
            *reinterpret_cast<double*>(sm + CO + 8 * e) = fabs(__ldg(a.cU + k));
            if constexpr (PLASMA) {
                J[i] = a.J[k];
                *reinterpret_cast<double*>(sm + PO + 8 * e) = __ldg(a.pb + k);
            }
        }
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = tid + i * NT;
            n01[i] = n2s[i] = 0;
            b[i] = cB[i] = 0.0;
            if (l >= nloc) continue;
            const int4 r = __ldg(a.rec + first + i * NT);
            n01[i] = (unsigned)r.y + (bufs | (bufs << 16));
            n2s[i] = (unsigned)r.z + bufs;
            b[i] = a.B[r.x];
            cB[i] = __ldg(a.cB64 + r.x);
            reinterpret_cast<double*>(sm)[l] = b[i];
        }
        if (tid < 2) *reinterpret_cast<double*>(sm + VO + 8 * (NE + tid)) = 0.0;   // the walls' U
        if (a.one_grp)
            for (int e = tid; e < a.n_steps; e += NT) gs[e] = __ldg(a.gtab + e);
        // published only after this CTA's reads of U and J are done: their owners write them back
        // after later steps
        if (!SOLO) __threadfence();
        __syncthreads();
        if constexpr (!SOLO) {
            __threadfence();
#pragma unroll
            for (int i = 0; i < TS; ++i)
                if (tid + i * NT < npub) slot_put(a.slots[0], (int)blockIdx.x * CAP + tid + i * NT, tag0, b[i]);
        }
    }

    // Step s + 1 from the B of step s; remote B in the words of parity PB = s & 1.
    template <int PB>
    __device__ __forceinline__ bool step(const FlowArgs<double>& a, int s) {
        const unsigned tag = tag0 + (unsigned)s;
        inner<0>(a, s);
        if constexpr (SOLO) {
            __syncthreads();
        } else {
            cut<0>(a, a.slots[PB], tag, s);
            ok = __syncthreads_and(ok ? 1 : 0) != 0;
            if (!ok) return false;
        }
        sums<PB, 0>(tag);
        __syncthreads();
        return true;
    }

    template <int I>
    __device__ __forceinline__ void update(const FlowArgs<double>& a, int s, double bR, double bL) {
        const double uo = lds_at<VO + 8 * I * NT>(own, 0.0);
        double un = rn_fma(lds_at<CO + 8 * I * NT>(own, 0.0), rn_sub(bR, bL), uo);
        if constexpr (PLASMA) {
            const double jn = rn_fma(a.pa, J[I], rn_mul(lds_at<PO + 8 * I * NT>(own, 0.0), uo));
            un = rn_fma(a.mdt, jn, un);
            J[I] = jn;
        }
        if ((src >> I) & 1u) {
            const EdgeSrc se = entry_at<I * NT>(sent);
            un = rn_fma(se.c, a.one_grp ? gs[s] : __ldg(a.gtab + se.g + s), un);
        }
        sts_at<VO + 8 * I * NT>(own, un);
    }

    template <int I>
    __device__ __forceinline__ void inner(const FlowArgs<double>& a, int s) {
        if constexpr (I < ES) {
            if ((int)threadIdx.x + I * NT < ni) update<I>(a, s, lds_half<0, false>(w[I], 0.0), lds_half<0, true>(w[I], 0.0));
            inner<I + 1>(a, s);
        }
    }

    // Edges to other CTAs, two slots' polls in flight.
    template <int I>
    __device__ __forceinline__ bool is_cut() const {
        const int e = (int)threadIdx.x + I * NT;
        return e >= ni && e < ne;
    }
    template <int I>
    __device__ __forceinline__ void arrive(const FlowArgs<double>& a, const unsigned long long* sl, unsigned tag, int s, Word<double>& x) {
        if (!word_wait_at(x, sl, w[I], tag)) ok = false;
        const double r = x.value(), h = lds_slot(bufs, w[I]);
        update<I>(a, s, w[I] & 1u ? h : r, w[I] & 1u ? r : h);
    }
    template <int I>
    __device__ __forceinline__ void cut(const FlowArgs<double>& a, const unsigned long long* sl, unsigned tag, int s) {
        if constexpr (I < ES) {
            Word<double> x, y;
            if (is_cut<I>()) word_at(x, sl, w[I]);
            if constexpr (I + 1 < ES) {
                if (is_cut<I + 1>()) word_at(y, sl, w[I + 1]);
            }
            if (is_cut<I>()) arrive<I>(a, sl, tag, s, x);
            if constexpr (I + 1 < ES) {
                if (is_cut<I + 1>()) arrive<I + 1>(a, sl, tag, s, y);
            }
            cut<I + 2>(a, sl, tag, s);
        }
    }

    template <int PB, int I>
    __device__ __forceinline__ void sums(unsigned tag) {
        if constexpr (I < TS) {
            const int l = (int)threadIdx.x + I * NT;
            if (l < nloc) {
                const double v0 = lds_signed<false, 0>(n01[I], n2s[I]), v1 = lds_signed<true, 1>(n01[I], n2s[I]),
                             v2 = lds_signed<false, 2>(n2s[I], n2s[I]);
                b[I] = rn_fma(-cB[I], rn_add(rn_add(v0, v1), v2), b[I]);
                sts_at<8 * I * NT>(own, b[I]);
                if (!SOLO && l < npub) slot_put_at<I * NT>(put[PB ^ 1], tag + 1u, b[I]);
            }
            sums<PB, I + 1>(tag);
        }
    }

    __device__ __forceinline__ double energy(const FlowArgs<double>& a) const {
        double x = 0.0;
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = (int)threadIdx.x + i * NT;
            if (l < nloc) x += __ldg(a.chk.S + __ldg(&a.rec[(size_t)blockIdx.x * CAP + l].x)) * b[i] * b[i];
        }
#pragma unroll
        for (int i = 0; i < ES; ++i) {
            const int e = (int)threadIdx.x + i * NT;
            if (e >= ne) continue;
            const unsigned k = (unsigned)__ldg(&a.erec[(size_t)blockIdx.x * NE + e].x);
            const double u = lds_val<double>(own + VO + 8 * i * NT);
            if (k & kEdgeOwn) x += __ldg(a.chk.we + (k & kEdgeMask)) * u * u;
        }
        return x;
    }

    __device__ __forceinline__ void write_back(const FlowArgs<double>& a) {
        if (!SOLO) __threadfence();
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = (int)threadIdx.x + i * NT;
            if (l < nloc) a.B[__ldg(&a.rec[(size_t)blockIdx.x * CAP + l].x)] = b[i];
        }
#pragma unroll
        for (int i = 0; i < ES; ++i) {
            const int e = (int)threadIdx.x + i * NT;
            if (e >= ne) continue;
            const unsigned k = (unsigned)__ldg(&a.erec[(size_t)blockIdx.x * NE + e].x);
            if (!(k & kEdgeOwn)) continue;
            a.U[k & kEdgeMask] = lds_val<double>(own + VO + 8 * i * NT);
            if constexpr (PLASMA) a.J[k & kEdgeMask] = J[i];
        }
    }
};

template <int SH, bool PLASMA, bool SOLO>
__global__ void __launch_bounds__(1024, 1) k_flow64(const __grid_constant__ FlowArgs<double> a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    flow_body<Flow64<SH, PLASMA, SOLO>, SOLO>(a, smraw);
}

// Its plan, after k_flow_order: a CTA's inner edges by their R triangle, then the cut ones, both in
// stored order (fixed, so that energies repeat), and where each triangle finds its edges.
__global__ void __launch_bounds__(1024) k_flow_edges(const __grid_constant__ PlanArgs a) {
    __shared__ int wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = blockIdx.x * a.per, nloc = max(0, min(a.per, a.n_t - j0)), p0 = (int)blockIdx.x * a.cap;
    const double* cU = (const double*)a.cU;
    int at[2], base = 0;   // edges before triangles tid and tid + 1024: inner | cut << 16
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int l = tid + 1024 * i;
        int n = 0;
        if (l < nloc) {
            const int4 t = __ldg(a.tri + j0 + l);
            const int code[3] = {t.x, t.y, t.z};
            for (int q = 0; q < 3; ++q) {
                const int k = code[q] >> 1;
                if (k >= a.n_ei) continue;
                const int2 r = __ldg(a.rl + k);
                const int o = (code[q] & 1) ? r.x : r.y;
                if (o < j0 || o >= j0 + nloc) n += 1 << 16;
                else if (!(code[q] & 1)) ++n;
            }
        }
        int inc = n;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        int before = base;
        for (int k = 0; k < 32; ++k) {
            before += k < warp ? wsum[k] : 0;
            base += wsum[k];
        }
        at[i] = before + inc - n;
        __syncthreads();
    }
    const int ni = base & 0xFFFF, nc = base >> 16;
    if (tid == 0) a.ecnt[blockIdx.x] = make_int2(ni, ni + nc);
    if (nc > a.halo || ni + nc > a.edges) {
        if (tid == 0) atomicOr(a.ctl + 3, 1u);
        return;
    }
    int2* erec = a.erec + (size_t)blockIdx.x * a.edges;
    EdgeSrc* sent = (EdgeSrc*)a.sent + (size_t)blockIdx.x * a.edges;
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int l = tid + 1024 * i;
            if (l >= nloc) continue;
            const int slot = a.place[j0 + l] - p0;
            const int4 t = __ldg(a.tri + j0 + l);
            const int code[3] = {t.x, t.y, t.z};
            int in = at[i] & 0xFFFF, out = ni + (at[i] >> 16);
            unsigned v[3], signs = 0;
            for (int q = 0; q < 3; ++q) {
                const int k = code[q] >> 1;
                const bool neg = code[q] & 1;
                int e = a.edges;   // a wall's: the slot that stays 0
                if (k < a.n_ei) {
                    const int2 r = __ldg(a.rl + k);
                    const int o = neg ? r.x : r.y;
                    const bool remote = o < j0 || o >= j0 + nloc;
                    e = remote ? out++ : !neg ? in++ : pass == 1 ? a.eslot[k] : 0;
                    if (neg) signs |= 1u << (16 + q);
                    if (pass == 0 && (remote || !neg)) {
                        int2 x = make_int2(k | (neg ? 0 : (int)kEdgeOwn), 0);
                        if (remote) x.y = a.place[o] << 12 | slot << 1 | (neg ? 0 : 1);
                        else x.y = 8 * slot | (8 * (a.place[o] - p0)) << 16;
                        const int h = a.has_src && neg_bit(__ldg(cU + k)) ? src_index(a, k) : -1;
                        if (h >= 0) {
                            x.x |= (int)kEdgeSrc;
                            sent[e] = EdgeSrc{__ldg((const double*)a.src_c + h), (long long)__ldg(a.src_grp + h) * a.gstride};
                        }
                        erec[e] = x;
                        if (!remote) a.eslot[k] = e;
                    }
                }
                v[q] = 8u * (unsigned)(a.cap + e);
            }
            if (pass == 1) a.rec[p0 + slot] = make_int4(j0 + l, (int)(v[0] | v[1] << 16), (int)(v[2] | signs), 0);
        }
        __syncthreads();
    }
}

__global__ void k_flow_init(unsigned* ctl) {
    if (threadIdx.x == 0) {
        ctl[0] = 1u;   // words start with tag 0
        ctl[1] = ctl[2] = ctl[3] = 0u;
    }
}

// no steps: looks only whether the launch fits (flow_ready)
template <typename T>
cudaError_t launch_resident(void (*kern)(FlowArgs<T>), const FlowArgs<T>& a, int grid, int threads, size_t smem, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (a.n_steps == 0) {
        int dev = 0, sms = 0, per = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem)) != cudaSuccess) return e;
        return per * sms >= grid ? cudaSuccess : cudaErrorCooperativeLaunchTooLarge;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = grid > 1 ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template <typename T, bool PLASMA, bool FRAME, bool SOLO, int SH>
cudaError_t launch_shape(const FlowArgs<T>& a, int grid, cudaStream_t s) {
    if constexpr (sizeof(T) == 8 && !FRAME)
        return launch_resident<T>(k_flow64<SH, PLASMA, SOLO>, a, grid, 1024, EdgeFlow<SH, PLASMA>::SMEM, s);
    else
        return launch_resident<T>(k_flow<T, SH, PLASMA, FRAME, SOLO>, a, grid, kShapes[SH].nt,
                                  flow_smem<T, PLASMA, SH>(FRAME ? a.fper : 0), s);
}

template <typename T, bool PLASMA, bool FRAME>
cudaError_t launch_flow_pf(const FlowArgs<T>& a, const FlowDev& fl, cudaStream_t s) {
    if (fl.grid == 1) {
        if constexpr (FRAME) return cudaErrorInvalidValue;
        else {
            if (fl.shape == 0) return launch_shape<T, PLASMA, false, true, 0>(a, 1, s);
            if constexpr (sizeof(T) == 4) return launch_shape<T, PLASMA, false, true, 1>(a, 1, s);
            return cudaErrorInvalidValue;
        }
    }
    if (fl.shape == 0) return launch_shape<T, PLASMA, FRAME, false, 0>(a, fl.grid, s);
    if (fl.shape == 1) return launch_shape<T, PLASMA, FRAME, false, 1>(a, fl.grid, s);
    if constexpr (sizeof(T) == 4) {
        if (fl.shape == 2) return launch_shape<T, PLASMA, FRAME, false, 2>(a, fl.grid, s);
        if constexpr (!PLASMA && !FRAME) return launch_shape<T, false, false, false, kVacuumShape>(a, fl.grid, s);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_flow_t(const FlowDev& fl, const DevMesh& m, void* Uif, int n_steps, const FlowChecks& chk, cudaStream_t s) {
    FlowArgs<T> a;
    a.tri = m.tri;
    a.cU = (const T*)m.cU;
    a.cB64 = (const double*)m.cB;
    a.U = (T*)m.U;
    a.B = (T*)m.B;
    a.pb = (const T*)m.pb;
    a.J = (T*)m.J;
    a.pa = (T)m.pa;
    a.mdt = (T)(-m.dt);
    a.rec = fl.rec;
    a.sent = (const SrcEntry<T>*)fl.sent;
    a.hlist = fl.hlist;
    a.cnt = fl.cnt;
    a.crec = fl.crec;
    a.erec = fl.erec;
    a.ecnt = fl.ecnt;
    a.gtab = m.gtab;
    a.one_grp = m.n_src > 0 && m.n_grp == 1;
    a.n_t = (int)m.n_t;
    a.n_ei = (int)m.n_ei;
    a.n_ei_pad = (int)m.n_ei_pad;
    a.per = fl.per;
    a.slots[0] = fl.slots;
    a.slots[1] = fl.slots + fl.slot_words;
    a.ctl = fl.ctl;
    a.step = m.step;
    a.n_steps = n_steps;
    a.skip = fl.skip;
    if (m.frame) a.f = *m.frame;
    a.Uif = (T*)Uif;
    a.fper = fl.fper;
    a.chk = chk;
    a.epart = fl.epart;
    a.ecount = fl.epart ? reinterpret_cast<unsigned*>(fl.epart + (size_t)kFlowChecks * fl.grid) : nullptr;
    if (m.frame) return m.plasma ? launch_flow_pf<T, true, true>(a, fl, s) : launch_flow_pf<T, false, true>(a, fl, s);
    return m.plasma ? launch_flow_pf<T, true, false>(a, fl, s) : launch_flow_pf<T, false, false>(a, fl, s);
}

// Most shared memory of a CTA, a current's coefficients counted in (it may be set later).
size_t smem_of(bool f64, int sh, int cells) {
    if (f64 && cells == 0) return sh == 0 ? EdgeFlow<0, true>::SMEM : EdgeFlow<1, true>::SMEM;
    if (f64) return sh == 0 ? flow_smem<double, true, 0>(cells) : flow_smem<double, true, 1>(cells);
    return sh == 0   ? flow_smem<float, true, 0>(cells)
           : sh == 1 ? flow_smem<float, true, 1>(cells)
           : sh == 2 ? flow_smem<float, true, 2>(cells)
                     : flow_smem<float, false, kVacuumShape>(cells);
}

}  // namespace

bool flow_shape(int64_t n_t, int64_t n_fc, bool f64, int sms, FlowDev& fl) {
    fl = FlowDev();
    if (n_t < 1 || sms < 1 || n_t + n_fc >= INT32_MAX / 2) return false;
    // one CTA holds up to 2,048 triangles: without an exchange its step takes 0.3 to 0.6 us, less
    // than the 0.9 us of one.  In FP64 one SM's pipe takes 2 to 3.3 us for 1,000 triangles, an exchange
    // 1.2 to 1.4
    if (n_fc == 0 && n_t <= (f64 ? 512 : 2048)) {
        fl.grid = 1;
        fl.shape = n_t <= 1024 ? 0 : 1;
        fl.per = (int)n_t;
    } else {
        const int64_t per = (n_t + sms - 1) / sms, fper = (n_fc + sms - 1) / sms;
        fl.shape = -1;
        for (int i = 0; i < (f64 ? 2 : n_fc > 0 ? kVacuumShape : 4) && fl.shape < 0; ++i)
            if (per <= (int64_t)kShapes[i].nt * kShapes[i].ts && fper <= kShapes[i].nt) fl.shape = i;
        if (fl.shape < 0) return false;
        fl.per = std::min((int)((per + 31) / 32 * 32), kShapes[fl.shape].nt * kShapes[fl.shape].ts);
        fl.grid = std::max((int)((n_t + fl.per - 1) / fl.per), 2);
        if (n_fc > 0) fl.grid = std::max<int>(fl.grid, (int)std::min<int64_t>(sms, (n_fc + 63) / 64));
        fl.fper = (int)((n_fc + fl.grid - 1) / fl.grid);
        if (fl.fper > kShapes[fl.shape].nt) return false;
    }
    if (smem_of(f64, fl.shape, fl.fper) > (size_t)226 * 1024) return false;
    fl.cap = kShapes[fl.shape].nt * kShapes[fl.shape].ts;
    fl.halo = f64 ? kShapes[fl.shape].halo64 : kShapes[fl.shape].halo32;
    fl.slot_words = fl.grid > 1 ? ((int64_t)fl.grid * fl.cap + n_fc) * (f64 ? 2 : 1) : 0;
    fl.sent_bytes = (size_t)fl.grid * fl.cap * (f64 ? sizeof(SrcEntry<double>) : sizeof(SrcEntry<float>));
    if (f64 && n_fc == 0) {
        if ((int64_t)fl.grid * fl.cap > 1 << 20) return false;   // places in an edge record
        fl.edges = kEdgeShapes[fl.shape].edges;
        fl.sent_bytes = (size_t)fl.grid * fl.edges * sizeof(EdgeSrc);
    }
    return true;
}

int64_t flow_capacity(bool f64, int sms) {
    FlowDev fl;
    int64_t lo = 0, hi = (int64_t)sms * 512 * 16 + 1;   // fits (none does), does not
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) / 2;
        (flow_shape(mid, 0, f64, sms, fl) ? lo : hi) = mid;
    }
    return lo;
}

bool flow_takes(const FlowDev& fl, const DevMesh& m) { return fl.grid > 0 && (fl.shape != kVacuumShape || !m.plasma); }

cudaError_t launch_flow_init(const FlowDev& fl, cudaStream_t s) {
    k_flow_init<<<1, 32, 0, s>>>(fl.ctl);
    return cudaGetLastError();
}

cudaError_t launch_flow_plan(const FlowDev& fl, const DevMesh& m, cudaStream_t s) {
    PlanArgs a;
    a.tri = m.tri;
    a.rl = m.rl;
    a.cU = m.cU;
    a.hash = m.src_hash;
    a.bits = (unsigned)m.src_bits;
    a.src_c = m.src_c;
    a.src_grp = m.src_grp;
    a.gstride = m.gtab_size;
    a.has_src = m.n_src > 0;
    a.n_t = (int)m.n_t;
    a.n_ei = (int)m.n_ei;
    a.n_ei_pad = (int)m.n_ei_pad;
    a.per = fl.per;
    a.cap = fl.cap;
    a.halo = fl.halo;
    a.rec = fl.rec;
    a.sent = fl.sent;
    a.hlist = fl.hlist;
    a.cnt = fl.cnt;
    a.crec = fl.crec;
    a.ctl = fl.ctl;
    if (m.frame) a.f = *m.frame;
    a.fper = fl.fper;
    a.place = fl.place;
    a.erec = fl.erec;
    a.ecnt = fl.ecnt;
    a.eslot = fl.eslot;
    a.edges = fl.edges;
    if (m.precision == UE_PREC_FP64) {
        k_flow_order<double><<<fl.grid, 1024, 0, s>>>(a);
        if (fl.edges > 0) k_flow_edges<<<fl.grid, 1024, 0, s>>>(a);
        else k_flow_plan<double><<<fl.grid, 1024, 0, s>>>(a);
    } else {
        k_flow_order<float><<<fl.grid, 1024, 0, s>>>(a);
        k_flow_plan<float><<<fl.grid, 1024, 0, s>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_flow(const FlowDev& fl, const DevMesh& m, void* Uif, int n_steps, const FlowChecks& chk, cudaStream_t s) {
    if (n_steps < 1 || n_steps > kFlowSteps) return cudaErrorInvalidValue;
    if ((chk.first > 0 || chk.end) && (!fl.epart || !chk.we || !chk.S || !chk.wd)) return cudaErrorInvalidValue;
    return m.precision == UE_PREC_FP64 ? launch_flow_t<double>(fl, m, Uif, n_steps, chk, s)
                                       : launch_flow_t<float>(fl, m, Uif, n_steps, chk, s);
}

cudaError_t flow_ready(const FlowDev& fl, const DevMesh& m) {
    return m.precision == UE_PREC_FP64 ? launch_flow_t<double>(fl, m, nullptr, 0, FlowChecks(), nullptr)
                                       : launch_flow_t<float>(fl, m, nullptr, 0, FlowChecks(), nullptr);
}

}  // namespace ue
