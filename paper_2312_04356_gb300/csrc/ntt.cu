// Negacyclic number-theoretic transforms.
//
// Layout: limb r of polynomial p is the row p * pstride + r N (or loff[r] N) of the data and uses
// the prime with global id ids[r]; one CTA row of the grid (blockIdx.y) is one limb, so the modulus
// is uniform inside a CTA.
//
// Every kernel is written once over an arithmetic: ArFold for contexts whose primes all lie next
// to a power of two (fold.cuh; every chain of the named parameter sets), ArShoup for any other
// primes below 2^61.  Both return the same canonical residues.  The twiddle tables hold the pairs
// of hostmath::ntt_pair for the context's arithmetic.
#include "launch.cuh"

#include <cooperative_groups.h>
namespace cg = cooperative_groups;

namespace {

// ---- Harvey's lazy butterflies on Shoup products: forward values stay below 8q (the upper input
// is reduced on odd stages only; an uncorrected stage maps [0, b q) to [0, (b + 2) q), a corrected
// one, valid for b <= 8, to [0, 6q)), inverse values below 2q.
struct ArShoup {
    static constexpr bool LAZY = false;   // in k_ntt_pass
    u64 q, q2;
    __device__ __forceinline__ explicit ArShoup(const DevPrime* P) : q(P->m.q), q2(2 * P->m.q) {}
    __device__ __forceinline__ bool folds() const { return false; }
    __device__ __forceinline__ u64 open(u64 v) const { return v; }
    template <int U>
    __device__ __forceinline__ void fwd(u64& x, u64& y, ulonglong2 w) const {
        if ((U & 1) && x >= 2 * q2) x -= 2 * q2;
        const u64 t = y * w.x - __umul64hi(y, w.y) * q;   // [0, 2q)
        y = x - t + q2;
        x = x + t;
    }
    __device__ __forceinline__ u64 canon(u64 v) const {
        if (v >= 2 * q2) v -= 2 * q2;
        if (v >= q2) v -= q2;
        return v >= q ? v - q : v;
    }
    __device__ __forceinline__ void inv(u64& x, u64& y, ulonglong2 w) const {
        u64 s = x + y;
        if (s >= q2) s -= q2;
        const u64 d = x - y + q2;
        y = d * w.x - __umul64hi(d, w.y) * q;             // [0, 2q)
        x = s;
    }
    __device__ __forceinline__ u64 sum_out(u64 v) const { return v; }
    __device__ __forceinline__ u64 sum(u64 x, u64 y) const { return x + y; }          // below 4 q
    __device__ __forceinline__ u64 diff(u64 x, u64 y) const { return x - y + q2; }
    __device__ __forceinline__ u64 scale(u64 v, ulonglong2 w) const { return mul_shoup(v, w.x, w.y, q); }
};

// ---- butterflies on folded products (fold.cuh): r = y w within R, values signed.
// Forward: x + r, x - r, so a stage widens the range by R.  42- and 48-bit primes run all sixteen
// stages within 17 R < 2^62; 60-bit primes are folded when a group of four stages opens (1.1 2^60,
// then at most 1.02 2^60 more per stage).
// Inverse: a sum doubles per stage, so a group of four stages ends with its sums folded (16 R < 2^62),
// and 60-bit primes fold them after two stages as well (4.2 2^60 at most).
struct ArFold {
    static constexpr bool LAZY = true;
    u64 q;
    FoldMod f;
    __device__ __forceinline__ explicit ArFold(const DevPrime* P) : q(P->m.q), f(P->f) {}
    __device__ __forceinline__ bool folds() const { return f.big != 0; }
    __device__ __forceinline__ u64 open(u64 v) const { return (u64)fold_word((int64_t)v, f); }
    template <int U>
    __device__ __forceinline__ void fwd(u64& x, u64& y, ulonglong2 w) const {
        const u64 s = x + (u64)fold_mul((int64_t)y, w.x, w.y, f);
        y = 2 * x - s;       // x - r; in this form both results land in place, without register moves
        x = s;
    }
    __device__ __forceinline__ u64 canon(u64 v) const { return fold_canon((int64_t)v, q, f); }
    __device__ __forceinline__ void inv(u64& x, u64& y, ulonglong2 w) const {
        const u64 d = x - y;
        x = x + y;
        y = (u64)fold_mul((int64_t)d, w.x, w.y, f);
    }
    __device__ __forceinline__ u64 sum_out(u64 v) const { return (u64)fold_word((int64_t)v, f); }
    __device__ __forceinline__ u64 sum(u64 x, u64 y) const { return x + y; }
    __device__ __forceinline__ u64 diff(u64 x, u64 y) const { return x - y; }
    __device__ __forceinline__ u64 scale(u64 v, ulonglong2 w) const {
        return fold_canon(fold_mul((int64_t)v, w.x, w.y, f), q, f);
    }
};

// the inverse transform's final factor f and f times the last stage's twiddle
struct OutFactor {
    ulonglong2 f, fw;
};

// S stages on 16 register values, stage s pairing i with i + 2^(S-1-s); widx(s, i) is the twiddle
// index of the pair's lower element i
template <int S, class AR, class F>
__device__ __forceinline__ void fwd_stages(u64 (&x)[16], const AR& ar, const ulonglong2* __restrict__ tw, F widx) {
    if (ar.folds()) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = ar.open(x[i]);
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int is = 1 << (S - 1 - s);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (i & is) continue;
            const ulonglong2 w = __ldg(tw + widx(s, i));
            if (s & 1)
                ar.template fwd<1>(x[i], x[i + is], w);
            else
                ar.template fwd<0>(x[i], x[i + is], w);
        }
    }
}

// the S stages in reverse order.  LAST: the transform's last stage (one twiddle) carries the output
// factor: sums are scaled by out.f, differences by out.fw = f w, and the results are canonical.
template <bool LAST, int S, class AR, class F>
__device__ __forceinline__ void inv_stages(u64 (&x)[16], const AR& ar, const ulonglong2* __restrict__ itw, F widx,
                                           const OutFactor& out = OutFactor{}) {
#pragma unroll
    for (int j = 0; j < S; ++j) {
        const int is = 1 << j;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (i & is) continue;
            if (LAST && j == S - 1) {
                const u64 s = ar.sum(x[i], x[i + is]), d = ar.diff(x[i], x[i + is]);
                x[i] = ar.scale(s, out.f);
                x[i + is] = ar.scale(d, out.fw);
            } else {
                ar.inv(x[i], x[i + is], __ldg(itw + widx(S - 1 - j, i)));
            }
        }
        if (j == S - 1 ? !LAST : j == 1 && ar.folds()) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (!(i & is)) x[i] = ar.sum_out(x[i]);
        }
    }
}

// What a transform reads or writes besides the data array (X kernels).
// Inverse, first pass: row k reads src + (k / lpp) * src_pstride + (k % lpp) N and the result goes to the
// data array, so the input is left as it is (no copy before an out-of-place transform); scaled
// replaces the final factor N^{-1} by w (w2: times the last twiddle), e.g. k N^{-1} to multiply the
// result by the integer k.
// Forward, first pass: every row of polynomial p is the centred lift of the one row
// src + p * src_pstride with modulus lift_q (a signed word is what the lazy butterflies take; one
// fold brings a wider source prime's word into range); lift_q 0: row k reads src + (k / lpp) src_pstride +
// (k % lpp) N as it is.
// Inverse, last pass: dst not null takes row k at dst + k N instead of the data array.
struct NttSrc {
    const u64* src;
    size_t src_pstride;
    bool scaled;
    ulonglong2 w, w2;
    u64 lift_q;
    u64* dst;
};
// Forward, last pass: row k receives (a - x) s, or a ks - x s when has_k, instead of the transform x; row k
// of a at a + (k / lpp) a_pstride + (k % lpp) N, s and ks as ntt_pair pairs per row k % lpp.
// Against a lift kernel before and a tail kernel after the transform (each a pass over every limb):
// block 8.94 -> 8.51 ms, 8 ciphertexts in lockstep 62.0 -> 58.6 ms, composite ReLU 6.83 -> 6.14 ms.
// a's 16 words have to be loaded before the first store: left between the stores they were 16
// dependent round trips, and the fused pass was slower than the two kernels (9.50 ms).
struct NttTailArgs {
    const u64* a;
    size_t a_pstride;
    const ulonglong2* s;
    int has_k;
    int per_out;           // 0: in place, else polynomials per entry of outs
    u64* outs[kern::NttTail::MAX_OUTS];
    ulonglong2 ks[ScalarVec::MAX];
    // row r (of lpp) of polynomial p
    __device__ __forceinline__ u64* row(u64* data_row, int p, int r, int lpp, int logn) const {
        return per_out ? outs[p / per_out] + (((size_t)(p % per_out) * lpp + r) << logn) : data_row;
    }
};
template <bool TAIL>
struct NttArgs {
    typedef NttSrc type;
};
template <>
struct NttArgs<true> {
    typedef NttTailArgs type;
};
// the centred residue of v mod lq as a signed word, folded
__device__ __forceinline__ u64 lift_word(u64 v, u64 lq, const FoldMod& f) {
    return (u64)fold_word((int64_t)(v > (lq >> 1) ? v - lq : v), f);
}
// the tail of one word; x lazy
__device__ __forceinline__ u64 tail_word(u64 a, u64 x, const NttTailArgs& tl, ulonglong2 s, int r, u64 q,
                                         const FoldMod& f) {
    if (tl.has_k) {
        const ulonglong2 ks = tl.ks[r];
        return fold_canon(fold_mul((int64_t)a, ks.x, ks.y, f) - fold_mul((int64_t)x, s.x, s.y, f), q, f);
    }
    return fold_canon(fold_mul((int64_t)(a - x), s.x, s.y, f), q, f);
}
// the inverse transform's final factor of row r (osc: [rows][f, f w])
__device__ __forceinline__ OutFactor out_factor(const DevPrime* P, const u64* osc, int r, const NttSrc& io) {
    if (io.scaled) return OutFactor{io.w, io.w2};
    if (!osc) return OutFactor{P->n_inv, P->n_inv_w};
    const ulonglong2* o = reinterpret_cast<const ulonglong2*>(osc) + 2 * r;
    return OutFactor{o[0], o[1]};
}

// ---- any ring: c consecutive stages from s0 in shared memory, one barrier per stage.  Only index
// bits log2(T1)..log2(T0) move (T0 = N >> (s0+1), T1 = N >> (s0+c)), so the limb splits into
// independent sub-problems of 2^c elements j = hi*2T0 + k*T1 + lo; a CTA stages 2^logsub of them.
// ArShoup keeps canonical values throughout.  ArFold's are lazy, with the folds of ArFold's ranges:
// a product made canonical in every butterfly costs more than a Shoup product (N = 2^15, 200 limbs,
// forward: 238 us, 210 with Shoup products, 198 lazy; N = 2^13, rescale at level 5: 90, 87, 82).
// A transform of more than sixteen stages (N = 2^17) is folded between its passes.
constexpr int NTT_THREADS = 256;

template <class AR, bool INV>
__global__ void __launch_bounds__(NTT_THREADS)
    k_ntt_pass(u64* __restrict__ data, const DevPrime* __restrict__ primes, const int* __restrict__ ids, int lpp,
               size_t pstride, const int* __restrict__ loff, int logn, int s0, int c, int logsub, int scale_out,
               const u64* __restrict__ osc) {
    griddep_entry();
    extern __shared__ u64 sm[];
    const int limb = blockIdx.y;
    const DevPrime* P = primes + ids[limb % lpp];
    const AR ar(P);
    const u64 q = ar.q;
    u64* a = data + (size_t)(limb / lpp) * pstride + ((size_t)(loff ? loff[limb % lpp] : limb % lpp) << logn);
    const int span = 1 << c;
    const int SUB = 1 << logsub;
    const int stride = SUB > 1 ? SUB + 1 : 1;
    const int logT1 = logn - s0 - c;
    const int T1 = 1 << logT1;
    const int log2T0 = logn - s0;
    const int sid0 = blockIdx.x * SUB;
    const int total = SUB << c;

    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        int s, k;
        if (T1 == 1) {
            s = e >> c;
            k = e & (span - 1);
        } else {
            k = e >> logsub;
            s = e & (SUB - 1);
        }
        int sid = sid0 + s;
        size_t j = ((size_t)(sid >> logT1) << log2T0) + ((size_t)k << logT1) + (sid & (T1 - 1));
        sm[k * stride + s] = a[j];
    }
    __syncthreads();

    const int nbf = total >> 1;
    for (int u = 0; u < c; ++u) {
        const int uu = INV ? (c - 1 - u) : u;
        const int sg = s0 + uu;               // global stage
        const int lt = c - 1 - uu;            // log2 of the local stride
        const int tk = 1 << lt;
        for (int e = threadIdx.x; e < nbf; e += blockDim.x) {
            const int s = e & (SUB - 1);
            const int b = e >> logsub;
            const int k = ((b >> lt) << (lt + 1)) | (b & (tk - 1));
            const int sid = sid0 + s;
            const size_t j = ((size_t)(sid >> logT1) << log2T0) + ((size_t)k << logT1) + (sid & (T1 - 1));
            const int widx = (1 << sg) + (int)(j >> (logn - sg));
            u64* px = sm + k * stride + s;
            u64* py = sm + (k + tk) * stride + s;
            u64 x = *px, y = *py;
            const ulonglong2 w = (INV ? P->itw : P->tw)[widx];
            if constexpr (!AR::LAZY) {
                if (!INV) {
                    const u64 v = ar.scale(y, w);
                    *px = add_mod(x, v, q);
                    *py = sub_mod(x, v, q);
                } else {
                    *px = add_mod(x, y, q);
                    *py = ar.scale(sub_mod(x, y, q), w);
                }
            } else if (!INV) {
                if (u % 4 == 0 && (ar.folds() || (u == 0 && s0 + c > 16))) {
                    x = ar.open(x);
                    y = ar.open(y);
                }
                ar.template fwd<0>(x, y, w);
                *px = x;
                *py = y;
            } else {
                ar.inv(x, y, w);
                if (u % 4 == 3 || u == c - 1 || (ar.folds() && u % 2)) x = ar.sum_out(x);
                *px = x;
                *py = y;
            }
        }
        __syncthreads();
    }

    // the inverse transform's final factor: N^{-1}, or per row a caller-given pair
    const ulonglong2 ni = out_factor(P, osc, limb % lpp, NttSrc{}).f;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        int s, k;
        if (T1 == 1) {
            s = e >> c;
            k = e & (span - 1);
        } else {
            k = e >> logsub;
            s = e & (SUB - 1);
        }
        int sid = sid0 + s;
        size_t j = ((size_t)(sid >> logT1) << log2T0) + ((size_t)k << logT1) + (sid & (T1 - 1));
        u64 v = sm[k * stride + s];
        if (scale_out) v = ar.scale(v, ni);
        if (AR::LAZY && !INV && T1 == 1) v = ar.canon(v);
        a[j] = v;
    }
}

// ---- N = 2^8 .. 2^12: a whole limb in one CTA of N / 16 threads, 16 values per thread, register
// rounds of four stages (the last of LOGN mod 4, on 16 consecutive elements) with one shared-memory
// exchange between them.  In the round whose register bits start at bit p the thread holds
// k(i) = (t >> p) 2^(p+4) + i 2^p + t mod 2^p.
template <int LOGN>
__device__ __forceinline__ int sk(int t, int i, int p) {
    return ((t >> p) << (p + 4)) | (i << p) | (t & ((1 << p) - 1));
}
__device__ __forceinline__ int spad(int k) { return k + (k >> 4); }

template <class AR, bool INV, int LOGN, bool TAIL = false>
__global__ void __launch_bounds__(1 << (LOGN - 4))
    k_ntt_one(u64* __restrict__ data, const DevPrime* __restrict__ primes, const int* __restrict__ ids, int lpp,
              size_t pstride, const int* __restrict__ loff, const u64* __restrict__ osc,
              const __grid_constant__ NttSrc io, const __grid_constant__ typename NttArgs<TAIL>::type tl) {
    griddep_entry();
    constexpr int N = 1 << LOGN, NR = (LOGN + 3) / 4, LAST = LOGN - 4 * (NR - 1);   // rounds, stages of the last
    __shared__ u64 sm[N + N / 16];
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const DevPrime* P = primes + ids[r];
    const AR ar(P);
    u64* a = data + (size_t)(limb / lpp) * pstride + ((size_t)(loff ? loff[r] : r) << LOGN);
    const int t = threadIdx.x;
    u64 x[16];
    if (!INV) {
        if (io.lift_q) {
            const u64* src = io.src + (size_t)(limb / lpp) * io.src_pstride;
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = lift_word(src[sk<LOGN>(t, i, LOGN - 4)], io.lift_q, ar.f);
        } else {
            const u64* src = io.src ? io.src + (size_t)(limb / lpp) * io.src_pstride + ((size_t)r << LOGN) : a;
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = src[sk<LOGN>(t, i, LOGN - 4)];
        }
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
            const int p = rr < NR - 1 ? LOGN - 4 - 4 * rr : 0, s0 = 4 * rr;
            if (rr > 0) {
                const int pp = LOGN - 4 * rr;           // register bits of the previous round
                if (rr > 1) __syncthreads();
#pragma unroll
                for (int i = 0; i < 16; ++i) sm[spad(sk<LOGN>(t, i, pp))] = x[i];
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 16; ++i) x[i] = sm[spad(sk<LOGN>(t, i, p))];
            }
            auto widx = [&](int s, int i) { return (1 << (s0 + s)) + (sk<LOGN>(t, i, p) >> (LOGN - s0 - s)); };
            if (rr < NR - 1) fwd_stages<4>(x, ar, P->tw, widx);
            else fwd_stages<LAST>(x, ar, P->tw, widx);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[spad(16 * t + i)] = TAIL ? x[i] : ar.canon(x[i]);
        if constexpr (TAIL) {
            const u64* A = tl.a + (size_t)(limb / lpp) * tl.a_pstride + ((size_t)r << LOGN);
            const ulonglong2 s = tl.s[r];
            u64* o = tl.row(a, limb / lpp, r, lpp, LOGN);
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = __ldg(A + i * (N / 16) + t);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int j = i * (N / 16) + t;
                o[j] = tail_word(x[i], sm[spad(j)], tl, s, r, ar.q, ar.f);
            }
        } else {
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 16; ++i) a[i * (N / 16) + t] = sm[spad(i * (N / 16) + t)];
        }
    } else {
        const u64* src = io.src ? io.src + (size_t)(limb / lpp) * io.src_pstride + ((size_t)r << LOGN) : a;
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[spad(i * (N / 16) + t)] = src[i * (N / 16) + t];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[spad(16 * t + i)];
#pragma unroll
        for (int rr = NR - 1; rr >= 0; --rr) {
            const int p = rr < NR - 1 ? LOGN - 4 - 4 * rr : 0, s0 = 4 * rr;
            auto widx = [&](int s, int i) { return (1 << (s0 + s)) + (sk<LOGN>(t, i, p) >> (LOGN - s0 - s)); };
            if (rr == 0) inv_stages<true, 4>(x, ar, P->itw, widx, out_factor(P, osc, r, io));
            else if (rr < NR - 1) inv_stages<false, 4>(x, ar, P->itw, widx);
            else inv_stages<false, LAST>(x, ar, P->itw, widx);
            if (rr > 0) {
                const int pn = LOGN - 4 * rr;           // register bits of the next round
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 16; ++i) sm[spad(sk<LOGN>(t, i, p))] = x[i];
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 16; ++i) x[i] = sm[spad(sk<LOGN>(t, i, pn))];
            }
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) a[sk<LOGN>(t, i, LOGN - 4)] = x[i];
    }
}

// ---- N = 2^16: two passes of 8 stages, each as two radix-16 rounds.
// A pass works on 256-element sub-problems (k = 0..255), 16 threads per sub-problem,
// 16 values per thread in registers.  Round A covers local stages u = 0..3 on the
// elements k = t + 16 i, round B covers u = 4..7 on k = 16 t + i; one shared-memory
// exchange separates them.  Twiddle of local stage u for element k of sub-problem hi:
// index 2^(s0+u) + hi 2^u + (k >> (8 - u)).  Values between the passes are lazy.
// Shared words per sub-problem: 256 + 16 pad + the offset that puts the sub-problems a half-warp
// works on in different banks (COL with SUBS columns: 16 / SUBS threads t of each column).
template <int SUBS>
constexpr int f_stride = 272 + 16 / (SUBS < 16 ? SUBS : 16);
template <int SUBS>
__device__ __forceinline__ int f_slot(int sp, int k) { return sp * f_stride<SUBS> + k + (k >> 4); }
// The twiddles of round B are stored so that the threads of a sub-problem read consecutive ones
// (hostmath::ntt_tw_pos): the 2^u twiddles j = t 2^(u-4) + jj of local stage u at jj 16 + t.

template <bool ROUND_B, class AR>
__device__ __forceinline__ void fwd_round(u64 (&x)[16], int t, int hi, int s0, const ulonglong2* __restrict__ tw,
                                          const AR& ar) {
    fwd_stages<4>(x, ar, tw, [&](int s, int i) {
        const int u = (ROUND_B ? 4 : 0) + s;
        const int base = (1 << (s0 + u)) + (hi << u);
        return ROUND_B ? base + t + 16 * (i >> (4 - s)) : base + (i >> (4 - s));
    });
}
template <bool ROUND_B, bool LAST, class AR>
__device__ __forceinline__ void inv_round(u64 (&x)[16], int t, int hi, int s0, const ulonglong2* __restrict__ itw,
                                          const AR& ar, const OutFactor& out = OutFactor{}) {
    inv_stages<LAST, 4>(x, ar, itw, [&](int s, int i) {
        const int u = (ROUND_B ? 4 : 0) + s;
        const int base = (1 << (s0 + u)) + (hi << u);
        return ROUND_B ? base + t + 16 * (i >> (4 - s)) : base + (i >> (4 - s));
    }, out);
}

// COL: sub-problems are columns (s0 = 0, T1 = 256, element j = k*256 + lo), threads with
//      consecutive tid take consecutive columns.  ROW: sub-problems are contiguous rows
//      (s0 = 8, T1 = 1, j = hi*256 + k), consecutive tid take consecutive k.
template <class AR, bool COL, bool INV, int SUBS, int MINB, bool X = false>
__global__ void __launch_bounds__(16 * SUBS, MINB) k_ntt16(u64* __restrict__ data, const DevPrime* __restrict__ primes,
                                                    const int* __restrict__ ids, int lpp, size_t pstride,
                                                    const int* __restrict__ loff, const u64* __restrict__ osc,
                                                    const __grid_constant__ typename NttArgs<X && !INV && !COL>::type io) {
    static_assert(!X || !(INV && COL), "the inverse's last pass has no X form");
    griddep_entry();
    __shared__ u64 sm[SUBS * f_stride<SUBS>];
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const DevPrime* P = primes + ids[r];
    const AR ar(P);
    u64* a = data + (size_t)(limb / lpp) * pstride + ((size_t)(loff ? loff[r] : r) << 16);
    const int tid = threadIdx.x;
    const int sp = COL ? (tid % SUBS) : (tid >> 4);
    const int t = COL ? (tid / SUBS) : (tid & 15);
    const int sub = blockIdx.x * SUBS + sp;            // global sub-problem: column lo or row hi
    const int s0 = COL ? 0 : 8;
    const int hi = COL ? 0 : sub;
    u64 x[16];
    auto gidx = [&](int k) -> size_t { return COL ? ((size_t)k << 8) + sub : ((size_t)sub << 8) + k; };

    if (!INV) {
        if constexpr (X && !INV && COL) {
            const u64* src = io.src + (size_t)(limb / lpp) * io.src_pstride;
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = lift_word(src[gidx(t + 16 * i)], io.lift_q, ar.f);
        } else {
            const u64* sr = a;
            if constexpr (COL && !INV) sr = io.src ? io.src + (size_t)(limb / lpp) * io.src_pstride + ((size_t)r << 16) : a;
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = sr[gidx(t + 16 * i)];
        }
        fwd_round<false>(x, t, hi, s0, P->tw, ar);
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<SUBS>(sp, t + 16 * i)] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<SUBS>(sp, 16 * t + i)];
        fwd_round<true>(x, t, hi, s0, P->tw, ar);
        if (COL) {
#pragma unroll
            for (int i = 0; i < 16; ++i) a[gidx(16 * t + i)] = x[i];     // lazy
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (!X) x[i] = ar.canon(x[i]);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 16; ++i) sm[f_slot<SUBS>(sp, 16 * t + i)] = x[i];
            if constexpr (X && !INV && !COL) {
                // all of a's words in flight at once (loads cannot pass the stores below)
                const u64* A = io.a + (size_t)(limb / lpp) * io.a_pstride + ((size_t)r << 16);
                const ulonglong2 s = io.s[r];
                u64* o = io.row(a, limb / lpp, r, lpp, 16);
#pragma unroll
                for (int i = 0; i < 16; ++i) x[i] = __ldg(A + gidx(t + 16 * i));
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    o[gidx(t + 16 * i)] = tail_word(x[i], sm[f_slot<SUBS>(sp, t + 16 * i)], io, s, r, ar.q, ar.f);
            } else {
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 16; ++i) a[gidx(t + 16 * i)] = sm[f_slot<SUBS>(sp, t + 16 * i)];
            }
        }
    } else {
        if (COL) {
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = a[gidx(16 * t + i)];
        } else {
            const u64* sr = a;
            if constexpr (X && INV) sr = io.src + (size_t)(limb / lpp) * io.src_pstride + ((size_t)r << 16);
#pragma unroll
            for (int i = 0; i < 16; ++i) sm[f_slot<SUBS>(sp, t + 16 * i)] = sr[gidx(t + 16 * i)];
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<SUBS>(sp, 16 * t + i)];
            __syncthreads();
        }
        inv_round<true, false>(x, t, hi, s0, P->itw, ar);
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<SUBS>(sp, 16 * t + i)] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<SUBS>(sp, t + 16 * i)];
        if constexpr (COL && INV) inv_round<false, true>(x, t, hi, s0, P->itw, ar, out_factor(P, osc, r, io));
        else inv_round<false, false>(x, t, hi, s0, P->itw, ar);
        if constexpr (COL && INV) {
            if (io.dst) a = io.dst + ((size_t)limb << 16);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) a[gidx(t + 16 * i)] = x[i];     // canonical (COL), lazy (ROW)
    }
}

// ---- the same pass with 4 values per thread: four radix-4 register rounds (local stages
// 2r, 2r+1), three shared-memory exchanges, 64 threads per sub-problem and 4 sub-problems
// per 256-thread CTA: four times the threads of k_ntt16, for launches over few limbs.
// In round r thread t holds k0 + {0, e, d, d + e} (d = 128 >> 2r, e = d / 2), k0 = t with
// zero bits inserted at the positions of d and e.
__device__ __forceinline__ int ins0(int t, int p) { return ((t >> p) << (p + 1)) | (t & ((1 << p) - 1)); }

// where twiddle j of local stage u lies (see f_slot)
__device__ __forceinline__ int tw_pos(int u, int j) {
    return u <= 4 ? j : ((j & ((1 << (u - 4)) - 1)) << 4) | (j >> (u - 4));
}

template <class AR, bool COL, bool INV, bool SRC = false>
__global__ void __launch_bounds__(256) k_ntt16s(u64* __restrict__ data, const DevPrime* __restrict__ primes,
                                                const int* __restrict__ ids, int lpp, size_t pstride,
                                                const int* __restrict__ loff, const u64* __restrict__ osc,
                                                NttSrc io) {
    static_assert(!SRC || (INV && !COL), "only the inverse transform's first pass reads a separate source");
    griddep_entry();
    __shared__ u64 sm[4 * f_stride<4>];
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const DevPrime* P = primes + ids[r];
    const AR ar(P);
    u64* a = data + (size_t)(limb / lpp) * pstride + ((size_t)(loff ? loff[r] : r) << 16);
    const int tid = threadIdx.x;
    const int sp = COL ? (tid & 3) : (tid >> 6);
    const int t = COL ? (tid >> 2) : (tid & 63);
    const int sub = blockIdx.x * 4 + sp;
    const int s0 = COL ? 0 : 8;
    const int hi = COL ? 0 : sub;
    auto gidx = [&](int k) -> size_t { return COL ? ((size_t)k << 8) + sub : ((size_t)sub << 8) + k; };
    u64 x[4];
    int k0 = 0;
    if (!INV) {
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
            const int u = 2 * rr, d = 128 >> u, e = d >> 1;
            k0 = ins0(ins0(t, 6 - u), 7 - u);
            const int ks[4] = {k0, k0 + e, k0 + d, k0 + d + e};
            if (rr == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = a[gidx(ks[i])];
            } else {
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = sm[f_slot<4>(sp, ks[i])];
            }
            if (!(rr & 1) && ar.folds()) {
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = ar.open(x[i]);
            }
            // stage u: pairs (0, 2), (1, 3), one twiddle
            {
                const ulonglong2 w = __ldg(P->tw + (1 << (s0 + u)) + (hi << u) + tw_pos(u, k0 >> (8 - u)));
                ar.template fwd<0>(x[0], x[2], w);
                ar.template fwd<0>(x[1], x[3], w);
            }
            // stage u + 1: pairs (0, 1), (2, 3)
            {
                const int base = (1 << (s0 + u + 1)) + (hi << (u + 1));
                const ulonglong2 w0 = __ldg(P->tw + base + tw_pos(u + 1, k0 >> (7 - u)));
                const ulonglong2 w1 = __ldg(P->tw + base + tw_pos(u + 1, (k0 + d) >> (7 - u)));
                ar.template fwd<1>(x[0], x[1], w0);
                ar.template fwd<1>(x[2], x[3], w1);
            }
            if (rr < 3) {
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 4; ++i) sm[f_slot<4>(sp, ks[i])] = x[i];
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) a[gidx(ks[i])] = COL ? x[i] : ar.canon(x[i]);
            }
        }
    } else {
#pragma unroll
        for (int rr = 3; rr >= 0; --rr) {
            const int u = 2 * rr, d = 128 >> u, e = d >> 1;
            k0 = ins0(ins0(t, 6 - u), 7 - u);
            const int ks[4] = {k0, k0 + e, k0 + d, k0 + d + e};
            if (rr == 3) {
                const u64* sr = SRC ? io.src + (size_t)(limb / lpp) * io.src_pstride + ((size_t)r << 16) : a;
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = sr[gidx(ks[i])];
            } else {
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 4; ++i) x[i] = sm[f_slot<4>(sp, ks[i])];
            }
            // stage u + 1 first: pairs (0, 1), (2, 3)
            {
                const int base = (1 << (s0 + u + 1)) + (hi << (u + 1));
                const ulonglong2 w0 = __ldg(P->itw + base + tw_pos(u + 1, k0 >> (7 - u)));
                const ulonglong2 w1 = __ldg(P->itw + base + tw_pos(u + 1, (k0 + d) >> (7 - u)));
                ar.inv(x[0], x[1], w0);
                ar.inv(x[2], x[3], w1);
            }
            // stage u: pairs (0, 2), (1, 3); the transform's last carries the output factor
            if (rr == 0 && COL) {
                const OutFactor out = out_factor(P, osc, r, io);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const u64 s = ar.sum(x[i], x[i + 2]), d = ar.diff(x[i], x[i + 2]);
                    x[i] = ar.scale(s, out.f);
                    x[i + 2] = ar.scale(d, out.fw);
                }
            } else {
                const ulonglong2 w = __ldg(P->itw + (1 << (s0 + u)) + (hi << u) + tw_pos(u, k0 >> (8 - u)));
                ar.inv(x[0], x[2], w);
                ar.inv(x[1], x[3], w);
                x[0] = ar.sum_out(x[0]);
                x[1] = ar.sum_out(x[1]);
            }
            if (rr > 0) {
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 4; ++i) sm[f_slot<4>(sp, ks[i])] = x[i];
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) a[gidx(ks[i])] = x[i];     // canonical (COL), lazy (ROW)
            }
        }
    }
}

// ---- the whole N = 2^16 transform in one launch: a cluster of 8 CTAs per limb (512 threads
// each, 16 values per thread).  Forward: CTA r runs stages 0-7 on columns 32r .. 32r+31 (the
// COL pass of k_ntt16 with 32 sub-problems), writes them to its shared memory as [row][32],
// and after a cluster barrier reads rows 32r .. 32r+31 from all eight CTAs through
// distributed shared memory for stages 8-15 (the ROW pass).  Inverse: the same in reverse
// order.  The data makes one trip through HBM instead of two.  Every thread of every CTA
// reaches both cluster barriers (no early exit), and the second barrier keeps each CTA's
// shared memory alive until the other CTAs have read it.
constexpr int CL_SUBS = 32, CL_THREADS = 512, CL_SMEM_WORDS = CL_SUBS * f_stride<CL_SUBS>;

template <class AR, bool INV>
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(CL_THREADS, 2)
    k_ntt_cl(u64* __restrict__ data, const DevPrime* __restrict__ primes, const int* __restrict__ ids, int lpp,
             size_t pstride, const int* __restrict__ loff, const u64* __restrict__ osc, NttSrc io) {
    griddep_entry();
    extern __shared__ u64 sm[];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const DevPrime* P = primes + ids[r];
    const AR ar(P);
    u64* a = data + (size_t)(limb / lpp) * pstride + ((size_t)(loff ? loff[r] : r) << 16);
    const int tid = threadIdx.x;
    // COL mapping: column 32 rank + spc, elements (rows) t + 16 i / 16 t + i
    const int spc = tid % CL_SUBS, tc = tid / CL_SUBS, col = CL_SUBS * rank + spc;
    // ROW mapping: row 32 rank + spr, elements (columns) t + 16 i / 16 t + i
    const int spr = tid >> 4, tr = tid & 15, row = CL_SUBS * rank + spr;
    u64 x[16];
    if (!INV) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = a[((size_t)(tc + 16 * i) << 8) + col];
        fwd_round<false>(x, tc, 0, 0, P->tw, ar);
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<CL_SUBS>(spc, tc + 16 * i)] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<CL_SUBS>(spc, 16 * tc + i)];
        fwd_round<true>(x, tc, 0, 0, P->tw, ar);                 // column col, rows 16 tc + i
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[(16 * tc + i) * CL_SUBS + spc] = x[i];
        cl.sync();
#pragma unroll
        for (int i = 0; i < 16; ++i) {                               // column tr + 16 i of row `row`
            const u64* src = cl.map_shared_rank(sm, i >> 1);
            x[i] = src[row * CL_SUBS + tr + 16 * (i & 1)];
        }
        cl.sync();
        fwd_round<false>(x, tr, row, 8, P->tw, ar);
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<CL_SUBS>(spr, tr + 16 * i)] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<CL_SUBS>(spr, 16 * tr + i)];
        fwd_round<true>(x, tr, row, 8, P->tw, ar);
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = ar.canon(x[i]);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<CL_SUBS>(spr, 16 * tr + i)] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) a[((size_t)row << 8) + tr + 16 * i] = sm[f_slot<CL_SUBS>(spr, tr + 16 * i)];
    } else {
        const u64* sr = io.src ? io.src + (size_t)(limb / lpp) * io.src_pstride + ((size_t)r << 16) : a;
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<CL_SUBS>(spr, tr + 16 * i)] = sr[((size_t)row << 8) + tr + 16 * i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<CL_SUBS>(spr, 16 * tr + i)];
        __syncthreads();
        inv_round<true, false>(x, tr, row, 8, P->itw, ar);
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<CL_SUBS>(spr, 16 * tr + i)] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<CL_SUBS>(spr, tr + 16 * i)];
        inv_round<false, false>(x, tr, row, 8, P->itw, ar);            // row `row`, columns tr + 16 i
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[spr * 256 + tr + 16 * i] = x[i];
        cl.sync();
        {
            const u64* src = cl.map_shared_rank(sm, tc >> 1);          // rows 16 tc + i live there
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = src[(16 * (tc & 1) + i) * 256 + col];
        }
        cl.sync();
        inv_round<true, false>(x, tc, 0, 0, P->itw, ar);
#pragma unroll
        for (int i = 0; i < 16; ++i) sm[f_slot<CL_SUBS>(spc, 16 * tc + i)] = x[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = sm[f_slot<CL_SUBS>(spc, tc + 16 * i)];
        inv_round<false, true>(x, tc, 0, 0, P->itw, ar, out_factor(P, osc, r, io));
#pragma unroll
        for (int i = 0; i < 16; ++i) a[((size_t)(tc + 16 * i) << 8) + col] = x[i];
    }
}

// Launch shapes (identical results).  NTT_MIX, the default of fold contexts at every size, takes the best
// shape of each pass: 8 columns per COL CTA (64-byte runs; 4 columns leave half of every 64-byte access
// unused, 14.3 against 10.3 us just to read and write 62 limbs in that pattern) and 2 or 4 rows
// per ROW CTA (rows are contiguous, and CTAs of one or two warps fill the last wave best).  us per
// pass with the CTA's sub-problems x least resident CTAs, 62 / 368 limbs: forward COL 8x6 22.7 / 98,
// 16x3 23.9 / 104; forward ROW 2x20 25.0 / 115, 4x8 25.8 / 120; inverse ROW 4x12 22.8 / 105, 4x8
// 23.3 / 113; inverse COL 8x5 26.2 / 119, 8x4 26.8 / 123, 16x3 28.7 / 137; below 16 limbs they agree
// within 1 us of 8 to 12.  (Each figure holds about 4 us of the two events around the launch.)
// The 80-register shapes spill, inverse ROW 4x12 most: 32 bytes a thread; 4x8 has none and is the slower one.
// What is left between these and the butterflies alone (31 cycles per warp and SM quarter: 75 us for
// 368 limbs) are the loads of data and twiddles that other warps do not cover.  ckks_autotune times
// every shape per limb-count class.  Contexts on Shoup products have 16 sub-problems at two register budgets
// in the places of NTT_V16 and NTT_MIX; their default is NTT_V4 (64 / 200 limbs forward, events included:
// 62 / 161 us, NTT_V16 65 / 172; inverse 65 / 173 and 66 / 180; a block 9.82 ms, NTT_V16 from 16 limbs on 10.04).
enum NttVariant {
    NTT_V16 = 0, NTT_MIX = 1, NTT_V16_R64 = 1, NTT_V4 = 2, NTT_V4_R80 = 3, NTT_X4 = 4, NTT_CL = 5, NTT_NVARIANTS = 6
};

template <class AR, bool COL, bool INV, bool X>
void launch_ntt16_ar(const ckks_ctx* cx, int v, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride,
                     const int* loff, const u64* osc, const typename NttArgs<X && !INV && !COL>::type& io) {
    constexpr bool FOLD = AR::LAZY;
#define NTT16(SUBS, MINB)                                                                          \
    klaunch(cx, k_ntt16<AR, COL, INV, SUBS, MINB, X>, dim3(256 / SUBS, nlimbs), 16 * SUBS, 0,      \
            data, cx->d_primes, ids, lpp, pstride, loff, osc, io)
    switch (v) {
        case NTT_V16: NTT16(16, 3); break;
        case NTT_MIX:
            if constexpr (!FOLD) NTT16(16, 4);
            else if constexpr (COL) NTT16(8, INV ? 5 : 6);
            else if constexpr (INV) NTT16(4, 12);
            else NTT16(2, 20);
            break;
        case NTT_V4: NTT16(4, 8); break;
        case NTT_V4_R80: NTT16(4, 12); break;
        default:
            if constexpr (!X || INV)
                klaunch(cx, k_ntt16s<AR, COL, INV, X>, dim3(256 / 4, nlimbs), 256, 0,
                        data, cx->d_primes, ids, lpp, pstride, loff, osc, io);
            break;
    }
#undef NTT16
}

template <bool COL, bool INV, bool X = false>
void launch_ntt16_variant(const ckks_ctx* cx, int v, u64* data, int nlimbs, const int* ids, int lpp,
                          size_t pstride, const int* loff, const u64* osc,
                          const typename NttArgs<X && !INV && !COL>::type& io) {
    if constexpr (!X || INV) {      // lifts and tails are built into the folded passes only
        if (!cx->fold) return launch_ntt16_ar<ArShoup, COL, INV, X>(cx, v, data, nlimbs, ids, lpp, pstride, loff, osc, io);
    }
    launch_ntt16_ar<ArFold, COL, INV, X>(cx, v, data, nlimbs, ids, lpp, pstride, loff, osc, io);
}

inline int ntt_class(int nlimbs) {
    int c = 0;
    while (c < 7 && (2 << c) <= nlimbs) ++c;   // classes: 1, 2-3, 4-7, 8-15, 16-31, 32-63, 64-127, >=128
    return c;
}

template <class AR, bool INV>
void launch_ntt_cl(const ckks_ctx* cx, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride,
                   const int* loff, const u64* osc, const NttSrc& io) {
    static std::atomic<unsigned> done{0};
    allow_dynamic_smem((const void*)k_ntt_cl<AR, INV>, CL_SMEM_WORDS * (int)sizeof(u64), done);
    klaunch(cx, k_ntt_cl<AR, INV>, dim3(8, nlimbs), CL_THREADS, CL_SMEM_WORDS * sizeof(u64),
            data, cx->d_primes, ids, lpp, pstride, loff, osc, io);
}

// One whole N = 2^16 transform with variant v: the cluster kernel, or the two passes (forward:
// COL then ROW; inverse: ROW then COL).  Algorithmic bytes: one read and one write of the
// limbs per transform, split evenly over the two passes.
// (io: a separate source of the first pass, a separate destination of the inverse's last and an output
// factor, as NttSrc describes; vcol: another variant for the COL pass)
template <bool INV>
void launch_ntt_variant(const ckks_ctx* cx, int v, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride,
                        const int* loff, const u64* osc = nullptr, const NttSrc& io = NttSrc{}, int vcol = -1) {
    const char* nm = INV ? "ntt_inv" : "ntt_fwd";
    const double bytes = 2.0 * nlimbs * cx->n * 8.0;
    const int vc = vcol >= 0 ? vcol : v;
    if (v == NTT_CL) {
        KTimer kt_(cx, nm, bytes);
        (cx->fold ? launch_ntt_cl<ArFold, INV> : launch_ntt_cl<ArShoup, INV>)(cx, data, nlimbs, ids, lpp, pstride, loff, osc, io);
        return;
    }
    {
        KTimer kt_(cx, nm, bytes / 2);
        if (INV && io.src)     // the inverse's first pass is the ROW pass
            launch_ntt16_variant<false, true, true>(cx, v, data, nlimbs, ids, lpp, pstride, loff, osc, io);
        else
            launch_ntt16_variant<!INV, INV>(cx, INV ? v : vc, data, nlimbs, ids, lpp, pstride, loff, osc, io);
    }
    {
        KTimer kt_(cx, nm, bytes / 2);
        launch_ntt16_variant<INV, INV>(cx, INV ? vc : v, data, nlimbs, ids, lpp, pstride, loff, osc, io);
    }
}

// the variant that transforms of nlimbs limbs use: the tuned one of their size class, else the default
inline int ntt_pick(const ckks_ctx* cx, int nlimbs) {
    const int v = cx->ntt_choice[ntt_class(nlimbs)];
    return v >= 0 ? v : cx->fold ? NTT_MIX : NTT_V4;
}

template <bool INV>
void launch_ntt_transform(const ckks_ctx* cx, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride,
                          const int* loff = nullptr, const u64* osc = nullptr, const NttSrc& io = NttSrc{}) {
    launch_ntt_variant<INV>(cx, ntt_pick(cx, nlimbs), data, nlimbs, ids, lpp, pstride, loff, osc, io);
}

// N = 2^8 .. 2^12 of a fold context: the whole limb in one CTA
inline bool ntt_one_cta(const ckks_ctx* cx) { return cx->fold && cx->logn >= 8 && cx->logn <= 12; }

template <bool INV, bool TAIL = false>
void launch_ntt_one(const ckks_ctx* cx, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride,
                    const u64* osc = nullptr, const NttSrc& io = NttSrc{},
                    const typename NttArgs<TAIL>::type& tl = typename NttArgs<TAIL>::type{},
                    const int* loff = nullptr) {
    KTimer kt_(cx, INV ? "ntt_inv" : "ntt_fwd", 2.0 * nlimbs * cx->n * 8.0);
#define ONE(LOGN)                                                                                                   \
    klaunch(cx, k_ntt_one<ArFold, INV, LOGN, TAIL>, dim3(1, nlimbs), 1 << (LOGN - 4), 0, data, cx->d_primes, ids,   \
            lpp, pstride, loff, osc, io, tl)
    switch (cx->logn) {
        case 8: ONE(8); break;
        case 9: ONE(9); break;
        case 10: ONE(10); break;
        case 11: ONE(11); break;
        default: ONE(12); break;
    }
#undef ONE
}

struct PassPlan {
    int s0, c;
};

inline std::vector<PassPlan> ntt_passes(int logn) {
    if (logn <= 12) return {{0, logn}};
    return {{0, logn - 8}, {logn - 8, 8}};
}

template <bool INV>
void launch_pass(const ckks_ctx* cx, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride, PassPlan p,
                 int scale_out, const u64* osc = nullptr, const int* loff = nullptr) {
    const int logn = cx->logn;
    int logsub = 12 - p.c;
    if (logsub < 0) logsub = 0;
    if (logsub > logn - p.c) logsub = logn - p.c;
    const int SUB = 1 << logsub;
    const int tiles = (1 << (logn - p.c)) / SUB;
    const int stride = SUB > 1 ? SUB + 1 : 1;
    const size_t smem = (size_t)stride * (1 << p.c) * sizeof(u64);
    dim3 grid(tiles, nlimbs);
    KTimer kt_(cx, INV ? "ntt_inv" : "ntt_fwd", 2.0 * nlimbs * cx->n * 8.0 * p.c / logn);
    if (cx->fold)
        klaunch(cx, k_ntt_pass<ArFold, INV>, grid, NTT_THREADS, smem, data, cx->d_primes, ids, lpp, pstride, loff, logn,
                p.s0, p.c, logsub, scale_out, osc);
    else
        klaunch(cx, k_ntt_pass<ArShoup, INV>, grid, NTT_THREADS, smem, data, cx->d_primes, ids, lpp, pstride, loff, logn,
                p.s0, p.c, logsub, scale_out, osc);
}

}  // namespace

namespace kern {

#define LAUNCH_CHECK() CUDA_CHECK(cudaGetLastError())

void ntt_forward(const ckks_ctx* c, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride) {
    if (nlimbs <= 0) return;
    if (pstride == 0) pstride = (size_t)lpp * c->n;
    if (c->logn == 16) {
        launch_ntt_transform<false>(c, data, nlimbs, ids, lpp, pstride);
        LAUNCH_CHECK();
        return;
    }
    if (ntt_one_cta(c)) {
        launch_ntt_one<false>(c, data, nlimbs, ids, lpp, pstride);
        LAUNCH_CHECK();
        return;
    }
    for (const PassPlan& p : ntt_passes(c->logn)) launch_pass<false>(c, data, nlimbs, ids, lpp, pstride, p, 0);
    LAUNCH_CHECK();
}

// out = the transform of `in` through the tail (NttLift, NttTail).  Where the transform's passes
// have the lift and the tail built in (a fold context whose variant is made of k_ntt16 passes, or
// the one-CTA rings) that is all; elsewhere the lift, the transform in place and the tail run one
// after another.
void ntt_forward_fused(const ckks_ctx* c, u64* out, int nlimbs, const int* ids, int lpp, const NttLift* lift,
                       const NttTail* tail) {
    if (nlimbs <= 0) return;
    CK_CHECK(lpp >= 1 && nlimbs % lpp == 0, CKKS_EINVAL, "whole polynomials only");
    const size_t n = c->n, ps = (size_t)lpp * n;
    const int v = c->logn == 16 ? ntt_pick(c, nlimbs) : -1;
    const bool one = ntt_one_cta(c);
    if (!c->fold || lpp > ScalarVec::MAX || (!one && (c->logn != 16 || v > NTT_V4_R80))) {
        if (lift) lift_centred(c, lift->src, lift->src_id, out, nlimbs, ids, lpp, lift->src_pstride);
        ntt_forward(c, out, nlimbs, ids, lpp);
        if (!tail) return;
        const int per = tail->outs ? tail->per_out : nlimbs / lpp;        // polynomials per output array
        for (int p0 = 0; p0 < nlimbs / lpp; p0 += per) {
            const u64* A = tail->a + p0 * tail->a_pstride;
            u64 *x = out + p0 * ps, *o = tail->outs ? tail->outs[p0 / per] : x;
            if (tail->ks)
                sub_mul2_scalar(c, A, x, *tail->ks, tail->s.w, tail->s.wp, o, per * lpp, ids, lpp, tail->a_pstride);
            else
                sub_mul_scalar(c, A, x, tail->s.w, tail->s.wp, o, per * lpp, ids, lpp, tail->a_pstride);
        }
        return;
    }
    NttSrc io{};
    if (lift) {
        io.src = lift->src;
        io.src_pstride = lift->src_pstride;
        io.lift_q = c->mod_of[lift->src_id];
    }
    NttTailArgs tl;
    if (tail) {
        tl.a = tail->a;
        tl.a_pstride = tail->a_pstride;
        tl.s = tail->s.pair;
        tl.has_k = tail->ks != nullptr;
        tl.per_out = tail->outs ? tail->per_out : 0;
        CK_CHECK(!tail->outs || (tail->per_out >= 1 && nlimbs <= NttTail::MAX_OUTS * tail->per_out * lpp), CKKS_EINVAL,
                 "too many outputs for one tail");
        if (tail->outs)
            for (int i = 0; i * tail->per_out * lpp < nlimbs; ++i) tl.outs[i] = tail->outs[i];
        if (tail->ks)
            for (int i = 0; i < lpp; ++i) {
                u64 w[2];
                hostmath::ntt_pair(tail->ks->v[i], c->q[i], true, w);
                tl.ks[i] = make_ulonglong2(w[0], w[1]);
            }
    }
    if (one) {
        if (tail) launch_ntt_one<false, true>(c, out, nlimbs, ids, lpp, ps, nullptr, io, tl);
        else launch_ntt_one<false>(c, out, nlimbs, ids, lpp, ps, nullptr, io);
        LAUNCH_CHECK();
        return;
    }
    const double bytes = (double)nlimbs * n * 8.0;
    {
        KTimer kt_(c, "ntt_fwd", bytes);
        if (lift) launch_ntt16_variant<true, false, true>(c, v, out, nlimbs, ids, lpp, ps, nullptr, nullptr, io);
        else launch_ntt16_variant<true, false>(c, v, out, nlimbs, ids, lpp, ps, nullptr, nullptr, io);
    }
    {
        KTimer kt_(c, "ntt_fwd", bytes);
        if (tail) launch_ntt16_variant<false, false, true>(c, v, out, nlimbs, ids, lpp, ps, nullptr, nullptr, tl);
        else launch_ntt16_variant<false, false>(c, v, out, nlimbs, ids, lpp, ps, nullptr, nullptr, io);
    }
    LAUNCH_CHECK();
}

// Time every NTT variant (forward + inverse) on scratch limbs of each size class and keep the
// fastest per class in ctx->ntt_choice.  Results are identical for every variant.
void autotune_ntt(ckks_ctx* c, int reps) {
    if (c->logn != 16) return;
    const int sizes[8] = {1, 2, 7, 14, 24, 48, 96, 192};
    DevBuf buf((size_t)192 << 16, c->stream);
    CUDA_CHECK(cudaMemsetAsync(buf.ptr, 0, ((size_t)192 << 16) * 8, c->stream));
    std::vector<int> ids(192);
    for (int i = 0; i < 192; ++i) ids[i] = i % c->nall;
    DevBuf dids(96, c->stream);
    CUDA_CHECK(cudaMemcpyAsync(dids.ptr, ids.data(), 192 * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    for (int k = 0; k < 8; ++k) {
        const int nl = sizes[k];
        float best = 1e30f;
        int bestv = -1;
        for (int v = 0; v < NTT_NVARIANTS; ++v) {
            for (int w = 0; w < 2; ++w) {   // warm up, then time
                cudaEventRecord(e0, c->stream);
                for (int r = 0; r < reps; ++r) {
                    const int* d = (const int*)dids.ptr;
                    launch_ntt_variant<false>(c, v, buf.ptr, nl, d, nl, (size_t)nl << 16, nullptr);
                    launch_ntt_variant<true>(c, v, buf.ptr, nl, d, nl, (size_t)nl << 16, nullptr);
                }
                cudaEventRecord(e1, c->stream);
                CUDA_CHECK(cudaEventSynchronize(e1));
            }
            float ms = 0;
            cudaEventElapsedTime(&ms, e0, e1);
            if (ms < best) {
                best = ms;
                bestv = v;
            }
        }
        c->ntt_choice[k] = bestv;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    LAUNCH_CHECK();
}

void ntt_forward_list(const ckks_ctx* c, u64* data, int nlimbs, const int* off, const int* ids, int nb,
                      size_t bstride) {
    if (nlimbs <= 0 || nb <= 0) return;
    if (c->logn == 16) {
        launch_ntt_transform<false>(c, data, nlimbs * nb, ids, nlimbs, bstride, off);
    } else if (ntt_one_cta(c)) {
        launch_ntt_one<false>(c, data, nlimbs * nb, ids, nlimbs, bstride, nullptr, NttSrc{}, NttArgs<false>::type{}, off);
    } else {
        for (const PassPlan& p : ntt_passes(c->logn))
            launch_pass<false>(c, data, nlimbs * nb, ids, nlimbs, bstride, p, 0, nullptr, off);
    }
    LAUNCH_CHECK();
}

void ntt_inverse(const ckks_ctx* c, u64* data, int nlimbs, const int* ids, int lpp, size_t pstride, const u64* osc) {
    if (nlimbs <= 0) return;
    if (pstride == 0) pstride = (size_t)lpp * c->n;
    if (c->logn == 16) {
        launch_ntt_transform<true>(c, data, nlimbs, ids, lpp, pstride, nullptr, osc);
        LAUNCH_CHECK();
        return;
    }
    if (ntt_one_cta(c)) {
        launch_ntt_one<true>(c, data, nlimbs, ids, lpp, pstride, osc);
        LAUNCH_CHECK();
        return;
    }
    std::vector<PassPlan> ps = ntt_passes(c->logn);
    for (int i = (int)ps.size() - 1; i >= 0; --i)
        launch_pass<true>(c, data, nlimbs, ids, lpp, pstride, ps[i], ps[i].s0 == 0 ? 1 : 0,
                          ps[i].s0 == 0 ? osc : nullptr);
    LAUNCH_CHECK();
}

void ntt_inverse_from(const ckks_ctx* c, const u64* src, size_t src_pstride, u64* data, int nlimbs, const int* ids,
                      int lpp, size_t pstride, const u64* osc, u64 kres, int k_id) {
    if (nlimbs <= 0) return;
    if (pstride == 0) pstride = (size_t)lpp * c->n;
    const bool scaled = k_id >= 0 && kres != 1;
    CK_CHECK(nlimbs % lpp == 0, CKKS_EINVAL, "whole polynomials only");
    CK_CHECK(!scaled || (lpp == 1 && osc == nullptr && pstride == c->n), CKKS_EINVAL,
             "an integer factor needs one contiguous row per polynomial and no output scale table");
    if (c->logn == 16 || ntt_one_cta(c)) {
        NttSrc io{src, src_pstride, scaled, {}, {}, 0, nullptr};
        if (scaled) {
            const u64 q = c->mod_of[k_id];
            u64 w[4];
            hostmath::ntt_out_factor(hostmath::mulmod(kres, hostmath::invmod((u64)c->n % q, q), q), c->ipsi_half[k_id], q,
                                     c->fold, w);
            io.w = make_ulonglong2(w[0], w[1]);
            io.w2 = make_ulonglong2(w[2], w[3]);
        }
        if (c->logn == 16) launch_ntt_transform<true>(c, data, nlimbs, ids, lpp, pstride, nullptr, osc, io);
        else launch_ntt_one<true>(c, data, nlimbs, ids, lpp, pstride, osc, io);
        LAUNCH_CHECK();
        return;
    }
    // the other rings: copy (and scale), then transform in place
    if (scaled) {
        ScalarVec sv;
        sv.v[0] = kres;
        sv.vp[0] = hostmath::shoup(kres, c->mod_of[k_id]);
        mul_scalar_v(c, src, sv, data, nlimbs, ids, 1, src_pstride);
    } else {
        CUDA_CHECK(cudaMemcpy2DAsync(data, pstride * 8, src, src_pstride * 8, (size_t)lpp * c->n * 8, nlimbs / lpp,
                                     cudaMemcpyDeviceToDevice, c->stream));
    }
    ntt_inverse(c, data, nlimbs, ids, lpp, pstride, osc);
}

bool ntt_host_io(const ckks_ctx* c, int nlimbs) {
    return ntt_one_cta(c) || (c->logn == 16 && ntt_pick(c, nlimbs) <= NTT_V4_R80);
}

// Columns of a COL CTA that touches host memory: the link moves 128-byte runs (16 columns) of a large
// transfer best (30 limbs out, whole export: 132 us with 64-byte runs, 122 with 128-byte ones, of which
// the link alone takes about 90); small ones want the CTAs.  8 and 16 columns agree at 4 limbs.  The 4
// columns of Shoup contexts make 32-byte runs, which the link moves worst: they take 16 at every size (4 limbs
// out: 38 -> 35 us).
static int host_columns(const ckks_ctx* c, int nlimbs) { return nlimbs >= 16 || !c->fold ? (int)NTT_V16 : -1; }

void ntt_forward_from_host(const ckks_ctx* c, const u64* host, u64* data, int nlimbs, const int* ids, int lpp) {
    const size_t ps = (size_t)lpp * c->n;
    const NttSrc io{host, ps, false, {}, {}, 0, nullptr};
    if (c->logn == 16)
        launch_ntt_variant<false>(c, ntt_pick(c, nlimbs), data, nlimbs, ids, lpp, ps, nullptr, nullptr, io,
                                  host_columns(c, nlimbs));
    else
        launch_ntt_one<false>(c, data, nlimbs, ids, lpp, ps, nullptr, io);
    LAUNCH_CHECK();
}

void ntt_inverse_to_host(const ckks_ctx* c, const u64* src, size_t src_pstride, u64* work, u64* host, int nlimbs,
                         const int* ids, int lpp) {
    const size_t ps = (size_t)lpp * c->n;
    const NttSrc io{src, src_pstride, false, {}, {}, 0, host};
    if (c->logn == 16)
        launch_ntt_variant<true>(c, ntt_pick(c, nlimbs), work, nlimbs, ids, lpp, ps, nullptr, nullptr, io,
                                 host_columns(c, nlimbs));
    else
        launch_ntt_one<true>(c, host, nlimbs, ids, lpp, ps, nullptr, io);
    LAUNCH_CHECK();
}

}  // namespace kern
