// Values exchanged between the CTAs of one cooperative launch without a grid barrier: each value
// travels with a 32-bit tag in the same 64-bit word, so a reader that sees the tag has the value.
// Used by the resident step and the resident power iteration (kernels_flow.cu, kernels_power.cu).
#pragma once

#include "device.cuh"

namespace ue {

// One published value: {32 bits, tag} words.  64-bit accesses are single-copy atomic.
__device__ __forceinline__ void slot_put(unsigned long long* s, int i, unsigned tag, float v) {
    const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(s + i), "l"(w) : "memory");
}
__device__ __forceinline__ void slot_put(unsigned long long* s, int i, unsigned tag, double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(s + 2 * (size_t)i), "l"(t | (b & 0xFFFFFFFFull)),
                 "l"(t | (b >> 32))
                 : "memory");
}
template <typename T>
struct Word;
template <>
struct Word<float> {
    unsigned long long w;
    __device__ __forceinline__ void load(const unsigned long long* s, int i) {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(s + i) : "memory");
    }
    __device__ __forceinline__ bool ready(unsigned tag) const { return (unsigned)(w >> 32) == tag; }
    __device__ __forceinline__ float value() const { return __uint_as_float((unsigned)w); }
};
template <>
struct Word<double> {
    unsigned long long a, b;
    __device__ __forceinline__ void load(const unsigned long long* s, int i) {
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(s + 2 * (size_t)i) : "memory");
    }
    __device__ __forceinline__ bool ready(unsigned tag) const {
        return (unsigned)(a >> 32) == tag && (unsigned)(b >> 32) == tag;
    }
    __device__ __forceinline__ double value() const {
        return __longlong_as_double((long long)((a & 0xFFFFFFFFull) | (b << 32)));
    }
};

// Poll a word until it carries the tag; bounded (about a second of SM clock): false when the
// wait runs out.
template <typename T>
__device__ __forceinline__ bool word_wait(Word<T>& w, const unsigned long long* s, int i, unsigned tag) {
    if (w.ready(tag)) return true;
    const long long t0 = clock64();
    for (unsigned n = 1;; ++n) {
        w.load(s, i);
        if (w.ready(tag)) return true;
        if ((n & 255u) == 0 && clock64() - t0 > (2LL << 30)) return false;
    }
}

// Shared load at a 32-bit shared address: a step's loads read the buffer that its stores do not
// touch, so they may move among the stores.
template <typename T>
__device__ __forceinline__ T lds_val(uint32_t addr);
template <>
__device__ __forceinline__ float lds_val<float>(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
template <>
__device__ __forceinline__ double lds_val<double>(uint32_t addr) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(addr));
    return v;
}

}  // namespace ue
