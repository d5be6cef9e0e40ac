// Power iteration for rho(M) (Section 2, the "complex time" method) on a mesh without a PML frame:
// v <- K v, K = -L_E L_B, from a SplitMix64 vector, and the Rayleigh quotient of the last iterate in
// the S metric.  FP64.
//
// (K v)_j = sum_q w_q (v_j - v_q), w_q = |e_q| / (d_q S_j) over the triangles q across j's edges, so
// an iteration is one pass over triangles: K_jj v_j - sum_q w_q v_q, four FP64 operations per
// triangle (GB300 issues about two per SM and cycle) on a 48-byte record.  The iterate is not
// normalised every time: K is scaled by the power of two below 1 / (2 max K_jj), a bound of its
// norm and at most four times lambda_max, so that an iterate shrinks by at most a quarter per
// product, and it is scaled up, by a power of two, every kSeg products.  Scaling by powers of two
// rounds nothing.  Sums are taken only at those points and for the final quotient.
//
// Meshes that fit the chip iterate resident, kSeg products per cooperative launch, the iterate in
// shared memory, values between CTAs through tagged words (exchange.cuh); larger ones launch once per
// product.  Measured for 200 products (was: two launches per product through edge values, each
// normalised by a reduction in the last block):
//   10k triangles 2.70 ms -> 0.27, 234k 5.38 ms -> 0.62 (3.1 us per product), 1.9M 23.5 ms -> 9.6.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "device.cuh"
#include "exchange.cuh"

namespace ue {

namespace {

constexpr int kThreads = 256;
constexpr int kSeg = 100;   // products between rescalings: the squares of the quotient's sums shrink
                            // by at most 2^-400 over them

unsigned blocks_for(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

// SplitMix64 (Steele, Lea, Flood 2014), published constants.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// ctl words: [0] max K_jj (bits of a positive double, which order like integers), [1] <v, K v>_S,
// [2] <v, v>_S of the last segment, [3] CTA counter, [4] error
struct PowerCtl {
    unsigned long long kmax;
    double num, den;
    unsigned done, err;
};

// Records, the start vector and the largest K_jj.
__global__ void __launch_bounds__(kThreads) k_pw_prep(const int4* __restrict__ tri, const int2* __restrict__ rl,
                                                      const double* __restrict__ elen, const double* __restrict__ d,
                                                      const double* __restrict__ S, const int64_t* __restrict__ perm,
                                                      uint32_t seed, int4* __restrict__ nb, double2* __restrict__ w,
                                                      double* __restrict__ v, int64_t n_ei, int64_t n_t,
                                                      PowerCtl* __restrict__ ctl) {
    const int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    double kjj = 0.0;
    if (j < n_t) {
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
        kjj = x[0] + x[1] + x[2];
        nb[j] = make_int4(o[0], o[1], o[2], 0);
        w[2 * j] = make_double2(x[0], x[1]);
        w[2 * j + 1] = make_double2(x[2], kjj);
        const uint64_t z = splitmix64(((uint64_t)seed << 32) + (uint64_t)perm[j]);
        v[j] = (double)(z >> 11) * 0x1.0p-53 * 2.0 - 1.0;
    }
    for (int o = 16; o > 0; o >>= 1) kjj = fmax(kjj, __shfl_xor_sync(0xffffffffu, kjj, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&ctl->kmax, (unsigned long long)__double_as_longlong(kjj));
}

// 2^-e with 2^(e-1) <= 2 max K_jj < 2^e
__device__ __forceinline__ double power_scale(const PowerCtl* ctl) {
    int e;
    frexp(2.0 * __longlong_as_double((long long)ctl->kmax), &e);
    return ldexp(1.0, -e);
}
// the power of two that brings an iterate of S-norm sqrt(den) near 1
__device__ __forceinline__ double lift(double den) {
    int e = 0;
    if (den > 0.0 && isfinite(den)) frexp(den, &e);
    return ldexp(1.0, -(e / 2));
}

// Sums (x, y) over the grid into ctl->num, ctl->den: block sums to part, added in block order by
// the last block to finish.  All threads of the block call it.
template <int NT>
__device__ void power_sums(double x, double y, double2* part, PowerCtl* ctl) {
    __shared__ double2 red[NT / 32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = (blockDim.x + 31) >> 5;
    auto warp_sum = [&](double& a, double& b) {
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
    };
    auto block_sum = [&](double& a, double& b) {   // on warp 0
        warp_sum(a, b);
        __syncthreads();
        if (lane == 0) red[warp] = make_double2(a, b);
        __syncthreads();
        if (warp == 0) {
            a = lane < warps ? red[lane].x : 0.0;
            b = lane < warps ? red[lane].y : 0.0;
            warp_sum(a, b);
        }
    };
    block_sum(x, y);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = make_double2(x, y);
        __threadfence();
        last = atomicAdd(&ctl->done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    x = y = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        const double2 p = __ldcg(part + i);
        x += p.x;
        y += p.y;
    }
    block_sum(x, y);
    if (threadIdx.x == 0) {
        ctl->num = x;
        ctl->den = y;
        ctl->done = 0u;
    }
}

// One product per launch.  LIFT: the first of a segment, the iterate scaled up on the way; SUMS: the
// last of one.  Bound by HBM on large meshes: 48 bytes of record, 8 + 8 of iterate per triangle.
template <bool LIFT, bool SUMS>
__global__ void __launch_bounds__(kThreads) k_pw_step(const int4* __restrict__ nb, const double2* __restrict__ w,
                                                      const double* __restrict__ S, const double* __restrict__ v,
                                                      double* __restrict__ vn, int64_t n_t, double2* part,
                                                      PowerCtl* ctl) {
    const int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    int4 o = make_int4(0, 0, 0, 0);
    double2 a = make_double2(0.0, 0.0), b = a;
    if (j < n_t) {   // records: not written by the launch before, so read ahead of its end
        o = __ldg(nb + j);
        a = __ldg(w + 2 * j);
        b = __ldg(w + 2 * j + 1);
    }
    grid_dependency_wait();
    grid_dependents_launch();
    double x = 0.0, u = 0.0;
    if (j < n_t) {
        const double sc = power_scale(ctl) * (LIFT ? lift(ctl->den) : 1.0);
        u = v[j];
        x = sc * fma(-b.x, v[o.z], fma(-a.y, v[o.y], fma(-a.x, v[o.x], b.y * u)));
        vn[j] = x;
        if (LIFT) u *= sc / power_scale(ctl);
    }
    if constexpr (SUMS) {
        const double t = j < n_t ? S[j] * u : 0.0;
        power_sums<kThreads>(t * x, t * u, part, ctl);
    }
}

// kSeg products (or the rest) in one cooperative launch.  CTA c keeps triangles [c per, (c+1) per);
// a thread holds slots tid + i * NT; the iterate and, with several slots, the records' weights sit
// in shared memory.  Exchange as in kernels_flow.cu: with several slots the CTA polls its remote
// neighbours into shared memory and a barrier follows; with one, whose product is all latency, each
// thread polls those of its triangle itself, a store, a poll and four FMAs (10k triangles: 1.94 us
// per product with the list and its barrier, now 1.33; with two slots a thread's polls hold up its other
// slot: 234k triangles 3.1 us, 3.5 that way, and the same with the triangles that publish in front).
struct PowerArgs {
    const int4* nb;
    const double2* w;
    const double* S;
    double* v;
    unsigned long long* slots[2];
    double2* part;
    PowerCtl* ctl;
    int n_t, per, hcap, n_it;
    unsigned tag0;
    int first, last;   // segment: the first takes the start vector as it is, the last leaves none
};

constexpr unsigned kPwPublish = 1u << 16;
constexpr unsigned kPwFar = 1u << 17;   // 3 bits: a remote neighbour that the list had no room for
__device__ __forceinline__ int far_of(const int4* nb, int j, int q) {
    const int4 r = __ldg(nb + j);
    return q == 0 ? r.x : q == 1 ? r.y : r.z;
}

template <int TS>
__host__ __device__ constexpr size_t power_smem(int cap, int hcap) {
    return (TS > 1 ? 32 * (size_t)cap : 0) + 16 * ((size_t)cap + (TS > 1 ? hcap : 0)) + 4 * (size_t)hcap;
}

template <int NT, int TS, bool SOLO>
__global__ void __launch_bounds__(NT, 1) k_pw_res(const __grid_constant__ PowerArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    constexpr bool OWN = TS == 1;   // threads poll for themselves
    __shared__ int s_hcnt;
    const int tid = threadIdx.x, nth = TS > 1 ? NT : (int)blockDim.x, cap = TS * nth, bcap = cap + (OWN ? 0 : a.hcap);
    double2* W = reinterpret_cast<double2*>(smraw);
    double* Vb = reinterpret_cast<double*>(W + (TS > 1 ? 2 * cap : 0));
    int* hlist = reinterpret_cast<int*>(Vb + 2 * bcap);
    const int j0 = blockIdx.x * a.per, nloc = max(0, min(a.per, a.n_t - j0));
    if (tid == 0) s_hcnt = 0;
    __syncthreads();
    const double sc = power_scale(a.ctl), up = a.first ? 1.0 : lift(a.ctl->den);
    double v[TS], old[TS];
    double2 wa[TS > 1 ? 1 : TS], wb[TS > 1 ? 1 : TS];
    unsigned n01[TS], n2f[TS];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < TS; ++i) {
        const int l = tid + i * nth;
        v[i] = old[i] = 0.0;
        n01[i] = n2f[i] = 0;
        if (l >= nloc) continue;
        const int j = j0 + l;
        const int4 r = __ldg(a.nb + j);
        const int o[3] = {r.x, r.y, r.z};
        unsigned off[3], f = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            int n = o[q] - j0;
            if (!SOLO && (n < 0 || n >= nloc)) {
                const int pos = atomicAdd(&s_hcnt, 1);
                n = l;
                f |= kPwPublish;
                if (pos < a.hcap) {
                    hlist[pos] = o[q];
                    n = cap + pos;   // beyond the slots: the list's entry
                } else {
                    f |= kPwFar << q;
                }
            }
            off[q] = (unsigned)n * 8u;
        }
        n01[i] = off[0] | (off[1] << 16);
        n2f[i] = off[2] | f;
        const double2 x = __ldg(a.w + 2 * (int64_t)j), y = __ldg(a.w + 2 * (int64_t)j + 1);
        const double2 xs = make_double2(sc * x.x, sc * x.y), ys = make_double2(sc * y.x, sc * y.y);
        if constexpr (TS > 1) {
            W[2 * l] = xs;
            W[2 * l + 1] = ys;
        } else {
            wa[0] = xs;
            wb[0] = ys;
        }
        v[i] = up * a.v[j];
        Vb[l] = v[i];
        if (!SOLO && (f & kPwPublish)) slot_put(a.slots[0], j, a.tag0, v[i]);
    }
    __syncthreads();
    const int hn = SOLO ? 0 : min(s_hcnt, a.hcap);
#pragma unroll 1
    for (int s = 0; s < a.n_it; ++s) {
        const int p = s & 1;
        const unsigned tag = a.tag0 + (unsigned)s;
        const unsigned long long* sl = p ? a.slots[1] : a.slots[0];
        double* Vp = Vb + (p ? bcap : 0);
        double* Vn = Vb + (p ? 0 : bcap);
        const uint32_t va = smem_addr(Vp);
        if constexpr (!SOLO && !OWN) {
            constexpr int kPoll = 2;
            for (int e0 = tid; e0 < hn; e0 += kPoll * nth) {
                Word<double> x[kPoll];
#pragma unroll
                for (int u = 0; u < kPoll; ++u)
                    if (e0 + u * nth < hn) x[u].load(sl, hlist[e0 + u * nth]);
#pragma unroll
                for (int u = 0; u < kPoll; ++u) {
                    const int e = e0 + u * nth;
                    if (e < hn) {
                        if (!word_wait(x[u], sl, hlist[e], tag)) ok = false;
                        Vp[cap + e] = x[u].value();
                    }
                }
            }
            ok = __syncthreads_and(ok ? 1 : 0) != 0;
            if (!ok) break;
        }
#pragma unroll
        for (int i = 0; i < TS; ++i) {
            const int l = tid + i * nth;
            if (l >= nloc) break;
            double2 x, y;
            if constexpr (TS > 1) {
                x = W[2 * l];
                y = W[2 * l + 1];
            } else {
                x = wa[0];
                y = wb[0];
            }
            double n[3];
            if (OWN && !SOLO && (n2f[i] & kPwPublish)) {
                const unsigned off[3] = {n01[i] & 0xFFFFu, n01[i] >> 16, n2f[i] & 0xFFFFu};
                Word<double> t[3];
                int at[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    at[q] = -1;
                    if (off[q] >= 8u * (unsigned)cap) at[q] = hlist[(off[q] >> 3) - cap];
                    else if (n2f[i] & (kPwFar << q)) at[q] = far_of(a.nb, j0 + l, q);
                    if (at[q] >= 0) t[q].load(sl, at[q]);
                    else n[q] = lds_val<double>(va + off[q]);
                }
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (at[q] >= 0) {
                        if (!word_wait(t[q], sl, at[q], tag)) ok = false;
                        n[q] = t[q].value();
                    }
            } else {
                n[0] = lds_val<double>(va + (n01[i] & 0xFFFFu));
                n[1] = lds_val<double>(va + (n01[i] >> 16));
                n[2] = lds_val<double>(va + (n2f[i] & 0xFFFFu));
                if (!OWN && !SOLO && (n2f[i] & (7u * kPwFar))) {
                    for (int q = 0; q < 3; ++q) {
                        if (!(n2f[i] & (kPwFar << q))) continue;
                        const int o = far_of(a.nb, j0 + l, q);
                        Word<double> t;
                        t.load(sl, o);
                        if (!word_wait(t, sl, o, tag)) ok = false;
                        n[q] = t.value();
                    }
                }
            }
            old[i] = v[i];
            v[i] = fma(-y.x, n[2], fma(-x.y, n[1], fma(-x.x, n[0], y.y * v[i])));
            if (!SOLO && (n2f[i] & kPwPublish) && s + 1 < a.n_it) slot_put(p ? a.slots[0] : a.slots[1], j0 + l, tag + 1u, v[i]);
            Vn[l] = v[i];
        }
        if constexpr (SOLO) {
            __syncthreads();
        } else if constexpr (OWN) {
            ok = __syncthreads_and(ok ? 1 : 0) != 0;
            if (!ok) break;
        }
    }
    if constexpr (!SOLO && !OWN) ok = __syncthreads_and(ok ? 1 : 0) != 0;
    if (!ok && tid == 0) atomicOr(&a.ctl->err, 1u);
    double num = 0.0, den = 0.0;
#pragma unroll
    for (int i = 0; i < TS; ++i) {
        const int l = tid + i * nth;
        if (l >= nloc) break;
        const int j = j0 + l;
        const double t = a.S[j] * old[i];
        num += t * v[i];
        den += t * old[i];
        if (!a.last) a.v[j] = v[i];
    }
    __syncthreads();
    power_sums<NT>(num, den, a.part, a.ctl);
}

struct PowerShape {
    int nt, ts;
};
constexpr PowerShape kShapes[3] = {{1024, 1}, {1024, 2}, {512, 8}};
constexpr size_t kSmem = 225 * 1024;

struct PowerPlan {
    int grid = 0, threads = 0, shape = 0, per = 0, hcap = 0;
};

// The resident launch for n_t triangles; grid 0 when they do not fit.
PowerPlan power_plan(int64_t n_t, int sms) {
    PowerPlan pl;
    if (n_t > (int64_t)sms * kShapes[2].nt * kShapes[2].ts) return pl;
    if (n_t <= 2048) {
        pl.grid = 1;
        pl.shape = n_t <= 1024 ? 0 : 1;
        pl.per = (int)n_t;
    } else {
        const int64_t per = (n_t + sms - 1) / sms;
        while (per > kShapes[pl.shape].nt * kShapes[pl.shape].ts) ++pl.shape;
        pl.per = std::min((int)((per + 31) / 32 * 32), kShapes[pl.shape].nt * kShapes[pl.shape].ts);
        pl.grid = std::max((int)((n_t + pl.per - 1) / pl.per), 2);
    }
    const int ts = kShapes[pl.shape].ts;
    pl.threads = ts > 1 ? kShapes[pl.shape].nt : (pl.per + 31) / 32 * 32;
    const int cap = ts * pl.threads;
    if (pl.grid > 1) {
        const size_t fixed = ts > 1 ? power_smem<2>(cap, 0) : power_smem<1>(cap, 0);
        pl.hcap = (int)std::min(std::min<size_t>(3 * (size_t)cap, (kSmem - fixed) / (ts > 1 ? 20 : 4)), (size_t)(8192 - cap)) & ~3;
    }
    return pl;
}

template <int SH, bool SOLO>
cudaError_t launch_res(const PowerArgs& a, const PowerPlan& pl, cudaStream_t s) {
    auto kern = k_pw_res<kShapes[SH].nt, kShapes[SH].ts, SOLO>;
    const size_t smem = power_smem<kShapes[SH].ts>(kShapes[SH].ts * pl.threads, pl.hcap);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)pl.grid);
    cfg.blockDim = dim3((unsigned)pl.threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = SOLO ? 0 : 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// dep: a programmatic dependent of the launch before, which must be another product (the records a
// step reads ahead of its wait were written before that one)
template <bool LIFT, bool SUMS, typename... A>
cudaError_t launch_step(int64_t n_t, bool dep, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks_for(n_t));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dep ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_pw_step<LIFT, SUMS>, args...);
}

int64_t part_count(int64_t n_t) { return std::max<int64_t>((n_t + kThreads - 1) / kThreads, 1024); }

}  // namespace

// records 6 n_t doubles, two iterates, exchange words 4 n_t, partials, control
size_t power_work_doubles(int64_t n_t) { return (size_t)(12 * n_t + 2 * part_count(n_t) + 16); }

cudaError_t power_iteration_mesh(const int2* rl, const int4* tri, const double* elen, const double* d,
                                 const double* S, const int64_t* perm, int64_t n_t, int64_t n_ei, int iters,
                                 uint32_t seed, double* work, double* rho, cudaStream_t s) {
    int4* nb = reinterpret_cast<int4*>(work);
    double2* w = reinterpret_cast<double2*>(work + 2 * n_t);
    unsigned long long* slots = reinterpret_cast<unsigned long long*>(work + 6 * n_t);
    double2* part = reinterpret_cast<double2*>(work + 10 * n_t);
    double* v[2] = {work + 10 * n_t + 2 * part_count(n_t), work + 11 * n_t + 2 * part_count(n_t)};
    PowerCtl* ctl = reinterpret_cast<PowerCtl*>(work + 12 * n_t + 2 * part_count(n_t));
    int dev = 0, sms = 0, coop = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ctl, 0, sizeof(PowerCtl), s)) != cudaSuccess) return e;
    k_pw_prep<<<blocks_for(n_t), kThreads, 0, s>>>(tri, rl, elen, d, S, perm, seed, nb, w, v[0], n_ei, n_t, ctl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    PowerPlan pl;
    if (coop) pl = power_plan(n_t, sms);
    if (pl.grid > 1 && (e = cudaMemsetAsync(slots, 0, 32 * n_t, s)) != cudaSuccess) return e;
    int done = 0;
    if (pl.grid > 0) {
        PowerArgs a;
        a.nb = nb;
        a.w = w;
        a.S = S;
        a.v = v[0];
        a.slots[0] = slots;
        a.slots[1] = slots + 2 * n_t;
        a.part = part;
        a.ctl = ctl;
        a.n_t = (int)n_t;
        a.per = pl.per;
        a.hcap = pl.hcap;
        for (int seg = 0; done < iters; ++seg) {
            a.n_it = std::min(kSeg, iters - done);
            a.tag0 = 1u + (unsigned)seg * (unsigned)(kSeg + 1);
            a.first = seg == 0;
            a.last = done + a.n_it == iters;
            if (pl.grid == 1) e = pl.shape == 0 ? launch_res<0, true>(a, pl, s) : launch_res<1, true>(a, pl, s);
            else if (pl.shape == 0) e = launch_res<0, false>(a, pl, s);
            else if (pl.shape == 1) e = launch_res<1, false>(a, pl, s);
            else e = launch_res<2, false>(a, pl, s);
            if (e == cudaErrorCooperativeLaunchTooLarge && seg == 0) {   // launched one by one instead
                cudaGetLastError();
                break;
            }
            if (e != cudaSuccess) return e;
            done += a.n_it;
        }
    }
    for (int it = done; it < iters; ++it) {   // done: 0, or all
        const bool up = it > 0 && it % kSeg == 0, sum = it % kSeg == kSeg - 1 || it == iters - 1;
        const int c = it & 1;
        const int4* nbc = nb;
        const double2* wc = w;
        const double* vc = v[c];
        if (up && sum) e = launch_step<true, true>(n_t, it > done, s, nbc, wc, S, vc, v[c ^ 1], n_t, part, ctl);
        else if (up) e = launch_step<true, false>(n_t, it > done, s, nbc, wc, S, vc, v[c ^ 1], n_t, part, ctl);
        else if (sum) e = launch_step<false, true>(n_t, it > done, s, nbc, wc, S, vc, v[c ^ 1], n_t, part, ctl);
        else e = launch_step<false, false>(n_t, it > done, s, nbc, wc, S, vc, v[c ^ 1], n_t, part, ctl);
        if (e != cudaSuccess) return e;
    }
    PowerCtl h;
    if ((e = cudaMemcpyAsync(&h, ctl, sizeof(h), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    if (h.err) return cudaErrorLaunchTimeout;   // a bounded wait between the CTAs ran out
    double kmax;
    static_assert(sizeof(kmax) == sizeof(h.kmax), "bits of a double");
    memcpy(&kmax, &h.kmax, 8);
    int ex;
    frexp(2.0 * kmax, &ex);
    const double lam = h.den > 0.0 ? ldexp(h.num / h.den, ex) : 0.0;
    *rho = sqrt(lam > 0.0 ? lam : 0.0);
    return cudaSuccess;
}

}  // namespace ue
