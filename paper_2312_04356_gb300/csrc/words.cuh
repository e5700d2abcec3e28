// Vector access to limb words and the reductions of 128-bit sums, shared by the kernel files.
#pragma once
#include "launch.cuh"

constexpr int EW_THREADS = 256;

// grid of the one-thread-per-V-words kernels
inline dim3 ewv_grid(int n, int nlimbs, int v) {
    int x = n / (EW_THREADS * v);
    if (x < 1) x = 1;
    return dim3(x, nlimbs);
}
inline bool al16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// A thread's V words of a limb (V = 2 or 4: 16-byte loads and stores, used when every pointer of the
// launch is 16-byte aligned): pairs j, j + 1 and, for V = 4, EW_THREADS pairs further on, so that
// every access of a warp covers 512 consecutive bytes (with four consecutive words per thread each
// access used half of the 128-byte lines it touched: 12.3 against 8.3 us to read and write 62 limbs).
// All operands are loaded before any store, so in-place calls (o == a) are safe.
template <int V>
__device__ __forceinline__ void ldv(const u64* p, u64 (&r)[V]) {
    if constexpr (V == 1) {
        r[0] = p[0];
    } else {
#pragma unroll
        for (int k = 0; k < V; k += 2) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p + k * EW_THREADS);
            r[k] = t.x;
            r[k + 1] = t.y;
        }
    }
}
// streaming load (evict-first in L1 and L2): for data read once, so that it does not push
// reused data out of L2
template <int V>
__device__ __forceinline__ void ldv_cs(const u64* p, u64 (&r)[V]) {
    if constexpr (V == 1) {
        r[0] = __ldcs(p);
    } else {
#pragma unroll
        for (int k = 0; k < V; k += 2) {
            const ulonglong2 t = __ldcs(reinterpret_cast<const ulonglong2*>(p + k * EW_THREADS));
            r[k] = t.x;
            r[k + 1] = t.y;
        }
    }
}
template <int V>
__device__ __forceinline__ void stv(u64* p, const u64 (&r)[V]) {
    if constexpr (V == 1) {
        p[0] = r[0];
    } else {
#pragma unroll
        for (int k = 0; k < V; k += 2)
            *reinterpret_cast<ulonglong2*>(p + k * EW_THREADS) = make_ulonglong2(r[k], r[k + 1]);
    }
}
// first word of the thread: the CTA's V EW_THREADS words start at blockIdx.x V EW_THREADS
template <int V>
__device__ __forceinline__ int ewv_first(int block) {
    return block * (V * EW_THREADS) + (V == 1 ? 1 : 2) * (int)threadIdx.x;
}
#define EWV_BEGIN(n)                          \
    const int j = ewv_first<V>(blockIdx.x);   \
    if (j >= (n)) return;

// Reduction of a 128-bit sum of products of residues to its canonical residue: folded where every
// modulus of the context qualifies (fold.cuh), else by Shoup products.
template <bool FOLD>
struct Reducer;
template <>
struct Reducer<true> {
    u64 q;
    FoldMod f;
    __device__ __forceinline__ explicit Reducer(const DevPrime& P) : q(P.m.q), f(P.f) {}
    __device__ __forceinline__ u64 operator()(u64 hi, u64 lo) const { return fold_128(hi, lo, q, f); }
    __device__ __forceinline__ u64 mul(u64 a, u64 b) const {
        u64 lo = 0, hi = 0;
        mac128(lo, hi, a, b);
        return fold_128(hi, lo, q, f);
    }
};
template <>
struct Reducer<false> {
    const DevPrime P;
    u64 q;
    __device__ __forceinline__ explicit Reducer(const DevPrime& p) : P(p), q(p.m.q) {}
    __device__ __forceinline__ u64 operator()(u64 hi, u64 lo) const { return reduce128_lazy(hi, lo, P); }
    __device__ __forceinline__ u64 mul(u64 a, u64 b) const { return mul_mod(a, b, P.m); }
};
