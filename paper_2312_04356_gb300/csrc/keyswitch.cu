// The products of key switching: a rotation's or relinearisation's inner product with its key, the
// inner sums of a BSGS map, and both in one pass (the hoisted rotations of a BSGS map are never
// stored).  Each output word is one 128-bit sum of products, reduced once (words.cuh).
//
// A product added to a 128-bit sum costs about 20 cycles of the integer-multiply pipe per warp and SM
// quarter; the reduction cost 72 with two Shoup products (90 in all) and costs 16 folded, which
// was half the work of a baby with three digits.  The c0 term rides in the same sum.  At N = 2^16,
// level 23: the seven maps of a bootstrapped block 2.19 -> 1.85 ms (6.5 TB/s by algorithmic
// bytes, the keys and diagonals read once: HBM), eight ciphertexts in lockstep 15.0 -> 12.5 ms
// (bound by the products), the key switches of a block 1.14 -> 1.07 ms.
// Contexts on Shoup products take one word a thread: two in 16-byte accesses measured slower (N = 2^16,
// level 23: a map of 64 stored babies 2.56 -> 2.64 ms, a rotation 257 -> 261 us).
#include "words.cuh"

#include <atomic>

namespace {

// row e of digit d of ciphertext t (the CTA's e is fixed, so this is uniform)
__device__ __forceinline__ const u64* digit_row(const kern::Digits& D, int d, int e, int t, int next, size_t dstr,
                                                int logn) {
    if (e < D.nl && e / D.alpha == d) return D.own + t * D.own_str + ((size_t)e << logn);
    return D.D + t * dstr + (((size_t)d * next + e) << logn);
}

// ------------------------------------------------- BSGS inner products ----
// o[g][poly][limb] = sum_b a_b[poly][limb] * p_{g,b}[limb] for NG giant steps at once: each
// baby value is loaded once and multiplied into every giant step's sum; the products are
// summed exactly in 128 bits (each < 2^122, at most 32 terms) and reduced once.
// blockIdx.y = row * nbt + t: ciphertext t of a batch (babies at T.a[b] + t astr, outputs at
// T.o[g] + t ostr; the diagonals are shared and read by neighbouring CTAs)
template <bool FOLD, int V, int NG>
__global__ void k_bsgs_inner_giants(kern::BsgsGiants T, const DevPrime* __restrict__ primes, int nl,
                                    const int* __restrict__ ids, int logn, int nbt, size_t astr, size_t ostr) {
    griddep_entry();
    const int t = blockIdx.y % nbt;
    const int limb = blockIdx.y / nbt;     // 0 .. 2 nl - 1, polynomial-major
    const int r = limb % nl;
    const Reducer<FOLD> red(primes[ids[r]]);
    const size_t offa = t * astr + ((size_t)limb << logn), offo = t * ostr + ((size_t)limb << logn);
    const size_t offp = (size_t)r << logn;
    EWV_BEGIN(1 << logn)
    u64 lo[NG][V], hi[NG][V];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int v = 0; v < V; ++v) lo[g][v] = hi[g][v] = 0;
    for (int b = 0; b < T.nb; ++b) {
        u64 x[V];
        ldv<V>(T.a[b] + offa + j, x);
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const u64* pg = T.p[g][b];
            if (!pg) continue;
            u64 y[V];
            ldv<V>(pg + offp + j, y);
#pragma unroll
            for (int v = 0; v < V; ++v) mac128(lo[g][v], hi[g][v], x[v], y[v]);
        }
    }
#pragma unroll
    for (int g = 0; g < NG; ++g) {
        u64 res[V];
#pragma unroll
        for (int v = 0; v < V; ++v) res[v] = red(hi[g][v], lo[g][v]);
        if ((T.acc >> g) & 1u) {
            u64 prev[V];
            ldv<V>(T.o[g] + offo + j, prev);
#pragma unroll
            for (int v = 0; v < V; ++v) res[v] = add_mod(res[v], prev[v], red.q);
        }
        stv<V>(T.o[g] + offo + j, res);
    }
}

// Baby rotations fused with the giant-step inner sums (see kern::bsgs_fused): per baby the
// key-switch product and the automorphed c0 term are summed in 128 bits and reduced, and the
// reduced baby multiplied into every giant step's 128-bit sum; the babies stay in registers.
// Same residues as k_ks_inner_d followed by k_bsgs_inner_giants.
// The next baby's operands (key words, gathered digit words, c0, diagonal words) are copied
// into shared memory by per-thread asynchronous copies while the current baby is computed:
// two stages of NS words per thread, so the memory latency of a baby overlaps the arithmetic
// of the previous one without holding the words in registers (a version loading them into
// registers ran 1.7x slower on a top-level CtoS level, latency bound at 36% warp occupancy).
__device__ __forceinline__ void cp_async8(u64* dst_smem, const u64* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// NC ciphertexts of a batch per thread: the key, diagonal and automorphism index of an element serve
// all of them, so NC = 2 moves 18 words per baby and element for two ciphertexts (3 digits, 4 giant
// steps) where NC = 1 moves 28.  Eight ciphertexts at the
// top level, six sums of a block: 12.59 -> 11.84 ms.
template <bool FOLD, int NDIG, int NG, int NC>
__global__ void __launch_bounds__(256, NC == 1 ? 3 : 2)
    k_bsgs_fused_async(const __grid_constant__ kern::BsgsFused T, const __grid_constant__ kern::Digits D,
                       const u64* __restrict__ c0, const u64* __restrict__ c1, int nl, int next,
                       const int* __restrict__ ext_ids, const u64* __restrict__ s0,
                       const DevPrime* __restrict__ P, int logn, size_t kstride, kern::KsBatch bt) {
    griddep_entry();
    // words of a stage: kb, ka per digit, diagonals; then per ciphertext D per digit, c0 (gathered or row), c1 row
    constexpr int OWN = 2 * NDIG + NG, NS = OWN + NC * (NDIG + 2);
    extern __shared__ u64 sbuf[];               // [2][NS][256]
    const int e = blockIdx.y;
    const int id = ext_ids[e];
    const Reducer<FOLD> red(P[id]);
    const u64 q = red.q;
    const size_t n = (size_t)1 << logn;
    const bool qrow = e < nl;
    const u64 w = qrow ? s0[e] : 0;
    const int tid = threadIdx.x;
    // ciphertexts t .. t + NC - 1 of a batch (fastest varying, so that the CTAs reading the same key and
    // diagonal words run side by side and share them through L2): D + t dstr, c0 / c1 + t xstr, outputs
    // + t ostr
    const int groups = bt.nb / NC, t = blockIdx.x % groups * NC;
    const int j = (blockIdx.x / groups) * 256 + tid;
    if (j >= (int)n) return;
    const u64* Dr[NC][NDIG];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int d = 0; d < NDIG; ++d) Dr[c][d] = digit_row(D, d, e, t + c, next, bt.dstr, logn);
    c0 += t * bt.xstr;
    c1 += t * bt.xstr;
    auto slot = [&](int st, int k) -> u64* { return sbuf + ((size_t)(st * NS + k) << 8) + tid; };
    auto own = [&](int st, int c, int k) -> u64* { return slot(st, OWN + c * (NDIG + 2) + k); };
    auto issue = [&](int b, int st) {
        if (!T.kb[b]) {
            if (qrow) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    cp_async8(own(st, c, NDIG), c0 + c * bt.xstr + (size_t)e * n + j);
                    cp_async8(own(st, c, NDIG + 1), c1 + c * bt.xstr + (size_t)e * n + j);
                }
            }
        } else {
            const unsigned src = galois_src(j, T.gal[b], logn);
#pragma unroll
            for (int d = 0; d < NDIG; ++d) {
                const size_t kk = d * kstride + (size_t)id * n + j;
                cp_async8(slot(st, d), T.kb[b] + kk);
                cp_async8(slot(st, NDIG + d), T.ka[b] + kk);
#pragma unroll
                for (int c = 0; c < NC; ++c) cp_async8(own(st, c, d), Dr[c][d] + src);
            }
            if (qrow) {
#pragma unroll
                for (int c = 0; c < NC; ++c) cp_async8(own(st, c, NDIG), c0 + c * bt.xstr + (size_t)e * n + src);
            }
        }
#pragma unroll
        for (int g = 0; g < NG; ++g)
            if (T.p[g][b]) cp_async8(slot(st, 2 * NDIG + g), T.p[g][b] + (size_t)e * n + j);
        cp_async_commit();
    };
    u64 lob[NC][NG], hib[NC][NG], loa[NC][NG], hia[NC][NG];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int g = 0; g < NG; ++g) lob[c][g] = hib[c][g] = loa[c][g] = hia[c][g] = 0;
    issue(0, 0);
    if (T.nb > 1) issue(1, 1);
    else cp_async_commit();
    for (int b = 0; b < T.nb; ++b) {
        const int st = b & 1;
        cp_async_wait<1>();                          // the group of baby b has landed
        // the baby: sum of the digits' products with the key and w c0 (w = P mod q), reduced once
        u64 rb[NC], ra[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            u64 bl = 0, bh = 0, al = 0, ah = 0;
            if (!T.kb[b]) {
                if (qrow) {
                    mac128(bl, bh, *own(st, c, NDIG), w);
                    mac128(al, ah, *own(st, c, NDIG + 1), w);
                }
            } else {
#pragma unroll
                for (int d = 0; d < NDIG; ++d) {
                    const u64 x = *own(st, c, d), yb = *slot(st, d), ya = *slot(st, NDIG + d);
                    mac128(bl, bh, x, yb);
                    mac128(al, ah, x, ya);
                }
                if (qrow) mac128(bl, bh, *own(st, c, NDIG), w);
            }
            rb[c] = red(bh, bl);
            ra[c] = red(ah, al);
        }
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            if (!T.p[g][b]) continue;
            const u64 y = *slot(st, 2 * NDIG + g);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                mac128(lob[c][g], hib[c][g], rb[c], y);
                mac128(loa[c][g], hia[c][g], ra[c], y);
            }
        }
        if (b + 2 < T.nb) issue(b + 2, st);          // this stage has been read
        else cp_async_commit();                      // keep one group per iteration
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            u64 vb = red(hib[c][g], lob[c][g]), va = red(hia[c][g], loa[c][g]);
            u64* ob = T.o[g] + (t + c) * bt.ostr + (size_t)e * n + j;
            u64* oa = T.o[g] + (t + c) * bt.ostr + ((size_t)next + e) * n + j;
            if ((T.acc >> g) & 1u) {
                vb = add_mod(vb, *ob, q);
                va = add_mod(va, *oa, q);
            }
            *ob = vb;
            *oa = va;
        }
}

// ---------------------------------------------------- key-switch product ----
// Key-switch inner product over NDIG digits: every digit's key words and gathered input are
// loaded before any arithmetic, the products are summed exactly in 128 bits (each < 2^122) and
// reduced once per output word.
// A batch of bt.nb key switches with the same key: ciphertext t's digits at D + t dstr, its
// outputs at ob / oa + t ostr, its x0 / x1 at + t xstr.  The ciphertext index is the fastest
// varying part of blockIdx.x, so the CTAs that read the same key words run side by side and
// all but the first find them in L2: the key streams from HBM about once per batch.
// Several rotations of one polynomial (blockIdx.z, outputs at ob / oa + z rstr) share a launch.
// NC of its ciphertexts share a thread and with it the key words and the automorphism.  Eight ciphertexts,
// the 49 of a block: 5.86 -> 5.71 ms (4.7 TB/s of algorithmic bytes).
template <bool FOLD, int V, int NDIG, int NC>
__global__ void k_ks_inner_d(const __grid_constant__ kern::Digits D, int next, const int* __restrict__ ext_ids,
                             const __grid_constant__ kern::KsRotations R, u64* __restrict__ ob, u64* __restrict__ oa,
                             size_t rstr, const DevPrime* __restrict__ P, int logn, size_t kstride,
                             const u64* __restrict__ x0, const u64* __restrict__ x1, int x0rows,
                             const u64* __restrict__ s0, kern::KsBatch bt) {
    griddep_entry();
    const int e = blockIdx.y;
    const int id = ext_ids[e];
    const Reducer<FOLD> red(P[id]);
    const size_t n = (size_t)1 << logn;
    const int groups = bt.nb / NC, t = blockIdx.x % groups * NC;
    const int j = V * ((blockIdx.x / groups) * blockDim.x + threadIdx.x);
    if (j >= (int)n) return;
    const u64 *kb = R.kb[blockIdx.z], *ka = R.ka[blockIdx.z], g = R.g[blockIdx.z];
    ob += blockIdx.z * rstr + t * bt.ostr + (size_t)e * n + j;
    oa += blockIdx.z * rstr + t * bt.ostr + (size_t)e * n + j;
    if (x0) x0 += t * bt.xstr + (size_t)e * n;
    if (x1) x1 += t * bt.xstr + (size_t)e * n;
    unsigned src[V];
#pragma unroll
    for (int v = 0; v < V; ++v) src[v] = g == 1 ? (unsigned)(j + v) : galois_src(j + v, g, logn);
    u64 x[NC][NDIG][V], yb[NDIG][V], ya[NDIG][V];
#pragma unroll
    for (int d = 0; d < NDIG; ++d) {
        const size_t kk = d * kstride + (size_t)id * n + j;
        if (bt.nb == 1) {
            ldv_cs<V>(kb + kk, yb[d]);   // each key word is read once per key switch: keep the
            ldv_cs<V>(ka + kk, ya[d]);   // raised digits, which every rotation re-reads, in L2
        } else {
            ldv<V>(kb + kk, yb[d]);      // the other ciphertexts of the batch read them next
            ldv<V>(ka + kk, ya[d]);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const u64* Dd = digit_row(D, d, e, t + c, next, bt.dstr, logn);
#pragma unroll
            for (int v = 0; v < V; ++v) x[c][d][v] = Dd[src[v]];
        }
    }
    // the sums: digits times key and w x0, w x1 (w = s0's row, or 1)
    u64 bl[NC][V], bh[NC][V], al[NC][V], ah[NC][V];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int v = 0; v < V; ++v) bl[c][v] = bh[c][v] = al[c][v] = ah[c][v] = 0;
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int v = 0; v < V; ++v) {
#pragma unroll
            for (int d = 0; d < NDIG; ++d) {
                mac128(bl[c][v], bh[c][v], x[c][d][v], yb[d][v]);
                mac128(al[c][v], ah[c][v], x[c][d][v], ya[d][v]);
            }
        }
    if (x0 && e < x0rows) {
        const u64 w = s0 ? s0[e] : 1;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
#pragma unroll
            for (int v = 0; v < V; ++v) mac128(bl[c][v], bh[c][v], x0[c * bt.xstr + src[v]], w);
            if (x1) {
#pragma unroll
                for (int v = 0; v < V; ++v) mac128(al[c][v], ah[c][v], x1[c * bt.xstr + src[v]], w);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        u64 rb[V], ra[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            rb[v] = red(bh[c][v], bl[c][v]);
            ra[v] = red(ah[c][v], al[c][v]);
        }
        stv<V>(ob + c * bt.ostr, rb);
        stv<V>(oa + c * bt.ostr, ra);
    }
}

// The key switches of several rotations (each with its own key, automorphism and raised polynomial: the
// rotated giant steps of an HMatmul) summed into one output: rotation k of ciphertext t has the digits
// of polynomial k nb + t of D and adds x0(sigma_k) of x0 + (k nb + t) xstr on every row.  One 128-bit
// sum and one reduction for all of them; a launch per rotation read and wrote the output each time.
// Bound by HBM like k_ks_inner_d: block 8.13 -> 7.98 ms, eight ciphertexts 54.2 -> 53.5 ms, conv at level 1
// 250 -> 241 us, downsampling layer 12.07 -> 11.81 ms.
template <bool FOLD, int V, int NDIG, int NC>
__global__ void k_ks_rotations(const __grid_constant__ kern::KsRotations R, const __grid_constant__ kern::Digits D,
                               int next, const int* __restrict__ ext_ids, const u64* __restrict__ x0,
                               u64* __restrict__ ob, u64* __restrict__ oa, const DevPrime* __restrict__ P, int logn,
                               size_t kstride, bool accumulate, int t0, int groups, kern::KsBatch bt) {
    griddep_entry();
    const int e = blockIdx.y;
    const int id = ext_ids[e];
    const Reducer<FOLD> red(P[id]);
    const size_t n = (size_t)1 << logn;
    const int t = t0 + blockIdx.x % groups * NC;
    const int j = V * ((blockIdx.x / groups) * blockDim.x + threadIdx.x);
    if (j >= (int)n) return;
    ob += t * bt.ostr + (size_t)e * n + j;
    oa += t * bt.ostr + (size_t)e * n + j;
    u64 bl[NC][V], bh[NC][V], al[NC][V], ah[NC][V];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int v = 0; v < V; ++v) bl[c][v] = bh[c][v] = al[c][v] = ah[c][v] = 0;
        if (accumulate) {
            ldv<V>(ob + c * bt.ostr, bl[c]);
            ldv<V>(oa + c * bt.ostr, al[c]);
        }
    }
    for (int k = 0; k < R.nr; ++k) {
        unsigned src[V];
#pragma unroll
        for (int v = 0; v < V; ++v) src[v] = galois_src(j + v, R.g[k], logn);
        u64 x[NC][NDIG][V], z[NC][V], yb[NDIG][V], ya[NDIG][V];
#pragma unroll
        for (int d = 0; d < NDIG; ++d) {
            const size_t kk = d * kstride + (size_t)id * n + j;
            if (bt.nb == 1) {
                ldv_cs<V>(R.kb[k] + kk, yb[d]);
                ldv_cs<V>(R.ka[k] + kk, ya[d]);
            } else {
                ldv<V>(R.kb[k] + kk, yb[d]);
                ldv<V>(R.ka[k] + kk, ya[d]);
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int poly = k * bt.nb + t + c;
            const u64* xr = x0 + poly * bt.xstr + (size_t)e * n;
#pragma unroll
            for (int v = 0; v < V; ++v) z[c][v] = xr[src[v]];
#pragma unroll
            for (int d = 0; d < NDIG; ++d) {
                const u64* Dd = digit_row(D, d, e, poly, next, bt.dstr, logn);
#pragma unroll
                for (int v = 0; v < V; ++v) x[c][d][v] = Dd[src[v]];
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                bl[c][v] += z[c][v];
                bh[c][v] += bl[c][v] < z[c][v];
#pragma unroll
                for (int d = 0; d < NDIG; ++d) {
                    mac128(bl[c][v], bh[c][v], x[c][d][v], yb[d][v]);
                    mac128(al[c][v], ah[c][v], x[c][d][v], ya[d][v]);
                }
            }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        u64 rb[V], ra[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            rb[v] = red(bh[c][v], bl[c][v]);
            ra[v] = red(ah[c][v], al[c][v]);
        }
        stv<V>(ob + c * bt.ostr, rb);
        stv<V>(oa + c * bt.ostr, ra);
    }
}

}  // namespace

namespace kern {

#define LAUNCH_CHECK() CUDA_CHECK(cudaGetLastError())

template <bool FOLD, int V>
static void launch_bsgs_giants(const ckks_ctx* c, const BsgsGiants& t, int nl, const int* ids, const KsBatch& bt) {
    const dim3 grid = ewv_grid(c->n, 2 * nl * bt.nb, V);
#define GIANTS_CASE(NG)                                                                                         \
    klaunch(c, k_bsgs_inner_giants<FOLD, V, NG>, grid, EW_THREADS, 0, t, c->d_primes, nl, ids, c->logn, bt.nb, bt.dstr, \
            bt.ostr)
    switch (t.ng) {
        case 1: GIANTS_CASE(1); break;
        case 2: GIANTS_CASE(2); break;
        case 3: GIANTS_CASE(3); break;
        case 4: GIANTS_CASE(4); break;
        case 5: GIANTS_CASE(5); break;
        case 6: GIANTS_CASE(6); break;
        case 7: GIANTS_CASE(7); break;
        default: GIANTS_CASE(8); break;
    }
#undef GIANTS_CASE
}

void bsgs_inner_giants(const ckks_ctx* c, const BsgsGiants& t, int nl, const int* ids, const KsBatch& bt) {
    CK_CHECK(t.nb >= 1 && t.nb <= BsgsGiants::MAXB && t.ng >= 1 && t.ng <= BsgsGiants::MAXG, CKKS_EINVAL,
             "1..32 baby steps and 1..8 giant steps per inner-sum launch");
    int terms = 0;
    bool vec = true;
    for (int b = 0; b < t.nb; ++b) vec = vec && al16(t.a[b]);
    for (int g = 0; g < t.ng; ++g) {
        vec = vec && al16(t.o[g]);
        for (int b = 0; b < t.nb; ++b)
            if (t.p[g][b]) {
                ++terms;
                vec = vec && al16(t.p[g][b]);
            }
    }
    {
        // algorithmic bytes: every baby (2 polynomials) once, every diagonal once, each giant's
        // output written (and read when accumulating)
        int accs = 0;
        for (int g = 0; g < t.ng; ++g) accs += (t.acc >> g) & 1u;
        KTimer kt_(c, "bsgs_inner", (bt.nb * (2.0 * t.nb + 2.0 * t.ng + 2.0 * accs) + terms) * nl * c->n * 8.0);
        if (c->fold && vec)
            launch_bsgs_giants<true, 2>(c, t, nl, ids, bt);
        else if (c->fold)
            launch_bsgs_giants<true, 1>(c, t, nl, ids, bt);
        else
            launch_bsgs_giants<false, 1>(c, t, nl, ids, bt);
    }
    LAUNCH_CHECK();
}

// the digits from ciphertext k of a batch on
static Digits digits_from(Digits D, size_t k, size_t dstr) {
    D.D += k * dstr;
    D.own += k * D.own_str;
    return D;
}

template <bool FOLD, int NDIG, int NG, int NC>
static void launch_bsgs_async_nc(const ckks_ctx* c, const BsgsFused& t, const Digits& D, const u64* c0,
                                 const u64* c1, int nl, int next, const int* ext, const u64* s, const KsBatch& bt) {
    constexpr int NS = 2 * NDIG + NG + NC * (NDIG + 2);
    const size_t smem = 2 * (size_t)NS * 256 * sizeof(u64);
    static std::atomic<unsigned> done{0};
    allow_dynamic_smem((const void*)k_bsgs_fused_async<FOLD, NDIG, NG, NC>, (int)smem, done);
    const dim3 grid((c->n + 255) / 256 * (bt.nb / NC), next);
    klaunch(c, k_bsgs_fused_async<FOLD, NDIG, NG, NC>, grid, 256, smem, t, D, c0, c1, nl, next, ext, s, c->d_primes,
            c->logn, (size_t)c->nall << c->logn, bt);
}

// the ciphertexts of a batch in pairs, the last of an odd number by itself
template <bool FOLD, int NDIG, int NG>
static void launch_bsgs_async_one(const ckks_ctx* c, const BsgsFused& t, const Digits& D, const u64* c0,
                                  const u64* c1, int nl, int next, const int* ext, const u64* s,
                                  const KsBatch& bt) {
    const int pairs = bt.nb / 2;
    if (pairs) {
        KsBatch b2 = bt;
        b2.nb = 2 * pairs;
        launch_bsgs_async_nc<FOLD, NDIG, NG, 2>(c, t, D, c0, c1, nl, next, ext, s, b2);
    }
    if (bt.nb & 1) {
        const size_t k = bt.nb - 1;
        BsgsFused t1 = t;
        for (int g = 0; g < t.ng; ++g) t1.o[g] += k * bt.ostr;
        KsBatch b1 = bt;
        b1.nb = 1;
        launch_bsgs_async_nc<FOLD, NDIG, NG, 1>(c, t1, digits_from(D, k, bt.dstr), c0 + k * bt.xstr, c1 + k * bt.xstr, nl, next, ext, s, b1);
    }
}

template <bool FOLD, int NDIG>
static void launch_bsgs_async_g(const ckks_ctx* c, const BsgsFused& t, const Digits& D, const u64* c0, const u64* c1,
                                int nl, int next, const int* ext, const u64* s, const KsBatch& bt) {
    switch (t.ng) {
        case 1: launch_bsgs_async_one<FOLD, NDIG, 1>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
        case 2: launch_bsgs_async_one<FOLD, NDIG, 2>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
        case 3: launch_bsgs_async_one<FOLD, NDIG, 3>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
        default: launch_bsgs_async_one<FOLD, NDIG, 4>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
    }
}

template <bool FOLD>
static void launch_bsgs_async(const ckks_ctx* c, const BsgsFused& t, const Digits& D, const u64* c0, const u64* c1,
                              int nl, int next, const int* ext, const u64* s, const KsBatch& bt) {
    switch (t.ndig) {
        case 1: launch_bsgs_async_g<FOLD, 1>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
        case 2: launch_bsgs_async_g<FOLD, 2>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
        case 3: launch_bsgs_async_g<FOLD, 3>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
        default: launch_bsgs_async_g<FOLD, 4>(c, t, D, c0, c1, nl, next, ext, s, bt); break;
    }
}

void bsgs_fused(const ckks_ctx* c, const BsgsFused& t, const Digits& D, const u64* c0, const u64* c1, int nl,
                int next, const int* ext_ids, const u64* s, const KsBatch& bt) {
    CK_CHECK(t.nb >= 1 && t.nb <= BsgsFused::MAXB && t.ng >= 1 && t.ng <= BsgsFused::MAXG && t.ndig >= 1 &&
                 t.ndig <= 4, CKKS_EINVAL, "fused BSGS: 1..32 babies, 1..4 giant steps, 1..4 digits");
    int terms = 0, rots = 0;
    for (int b = 0; b < t.nb; ++b) {
        if (t.kb[b]) ++rots;
        for (int g = 0; g < t.ng; ++g)
            if (t.p[g][b]) ++terms;
    }
    int accs = 0;
    for (int g = 0; g < t.ng; ++g) accs += (t.acc >> g) & 1u;
    {
        // algorithmic bytes: per rotation the digits, both key halves and c0 on the Q rows; the
        // identity's c0 and c1; every diagonal once; each giant's output (read when accumulating)
        // (a batch reads the keys and diagonals once, and its ciphertexts' own words each)
        const double shared = (double)rots * 2.0 * t.ndig + terms;
        const double own = (double)rots * (t.ndig * next + nl) / next + (t.nb - rots) * 2.0 * nl / next +
                           2.0 * t.ng + 2.0 * accs;
        KTimer kt_(c, "bsgs_fused", (shared + bt.nb * own) * next * c->n * 8.0);
        if (c->fold)
            launch_bsgs_async<true>(c, t, D, c0, c1, nl, next, ext_ids, s, bt);
        else
            launch_bsgs_async<false>(c, t, D, c0, c1, nl, next, ext_ids, s, bt);
    }
    LAUNCH_CHECK();
}

template <bool FOLD, int V, int NC>
static void launch_ks_inner_nc(const ckks_ctx* c, const Digits& D, int ndig, int next, const int* ext_ids,
                               const KsRotations& R, u64* ob, u64* oa, size_t rstr, const u64* x0, const u64* x1,
                               int x0rows, const u64* s0, const KsBatch& bt) {
    dim3 grid = ewv_grid(c->n, next, V);
    grid.x *= bt.nb / NC;
    grid.z = R.nr;
    const size_t ks = (size_t)c->nall << c->logn;
#define KS_CASE(NDIG)                                                                                                   \
    klaunch(c, k_ks_inner_d<FOLD, V, NDIG, NC>, grid, EW_THREADS, 0, D, next, ext_ids, R, ob, oa, rstr, c->d_primes,    \
            c->logn, ks, x0, x1, x0rows, s0, bt)
    switch (ndig) {
        case 1: KS_CASE(1); break;
        case 2: KS_CASE(2); break;
        case 3: KS_CASE(3); break;
        default: KS_CASE(4); break;
    }
#undef KS_CASE
}

// the ciphertexts of a batch in pairs, the last of an odd number by itself
template <bool FOLD, int V>
static void launch_ks_inner(const ckks_ctx* c, const Digits& D, int ndig, int next, const int* ext_ids,
                            const KsRotations& R, u64* ob, u64* oa, size_t rstr, const u64* x0, const u64* x1, int x0rows,
                            const u64* s0, const KsBatch& bt) {
    KsBatch part = bt;
    part.nb = bt.nb & ~1;
    if (part.nb) launch_ks_inner_nc<FOLD, V, 2>(c, D, ndig, next, ext_ids, R, ob, oa, rstr, x0, x1, x0rows, s0, part);
    if (bt.nb & 1) {
        const size_t k = part.nb;
        part.nb = 1;
        launch_ks_inner_nc<FOLD, V, 1>(c, digits_from(D, k, bt.dstr), ndig, next, ext_ids, R, ob + k * bt.ostr,
                                       oa + k * bt.ostr, rstr, x0 ? x0 + k * bt.xstr : x0, x1 ? x1 + k * bt.xstr : x1,
                                       x0rows, s0, part);
    }
}

static bool al16_keys(const KsRotations& R) {
    bool vec = true;
    for (int k = 0; k < R.nr; ++k) vec = vec && al16(R.kb[k]) && al16(R.ka[k]);
    return vec;
}

void ks_inner(const ckks_ctx* c, const Digits& D, int ndig, int next, const int* ext_ids, const KsRotations& R, u64* ob,
              u64* oa, size_t rstr, const u64* x0, int x0rows, const u64* s, const u64* x1, const KsBatch& bt) {
    CK_CHECK(bt.nb >= 1 && ndig >= 1 && ndig <= 4 && R.nr >= 1 && R.nr <= KsRotations::MAXR, CKKS_EINVAL,
             "key switching takes 1..4 digits");
    const bool vec = al16_keys(R) && al16(ob) && al16(oa) && rstr % 2 == 0;
    {
        // algorithmic bytes: the keys once for the whole batch, per ciphertext its digits, outputs
        // and the x0 / x1 rows
        const double extra = x0 ? (double)x0rows * (x1 ? 2.0 : 1.0) / next : 0.0;
        KTimer kt_(c, "ks_inner", R.nr * (2.0 * ndig + bt.nb * (ndig + 2.0 + extra)) * next * c->n * 8.0);
#define KS(FOLD, V) launch_ks_inner<FOLD, V>(c, D, ndig, next, ext_ids, R, ob, oa, rstr, x0, x1, x0rows, s, bt)
        if (c->fold && vec) KS(true, 2);
        else if (c->fold) KS(true, 1);
        else KS(false, 1);
#undef KS
    }
    LAUNCH_CHECK();
}

template <bool FOLD, int V>
static void launch_ks_rotations(const ckks_ctx* c, const Digits& D, int ndig, int next, const int* ext_ids,
                                const KsRotations& R, const u64* x0, u64* ob, u64* oa, bool accumulate,
                                const KsBatch& bt) {
    const dim3 tiles = ewv_grid(c->n, next, V);
    const size_t ks = (size_t)c->nall << c->logn;
    // ciphertexts in pairs, the last of an odd number by itself
#define KSR_CASE(NDIG, NC, T0, GROUPS)                                                                                 \
    klaunch(c, k_ks_rotations<FOLD, V, NDIG, NC>, dim3(tiles.x * (GROUPS), tiles.y), EW_THREADS, 0, R, D, next, ext_ids, \
            x0, ob, oa, c->d_primes, c->logn, ks, accumulate, T0, GROUPS, bt)
#define KSR_NDIG(NDIG)                                                \
    do {                                                              \
        if (bt.nb >= 2) KSR_CASE(NDIG, 2, 0, bt.nb / 2);              \
        if (bt.nb & 1) KSR_CASE(NDIG, 1, bt.nb - 1, 1);               \
    } while (0)
    switch (ndig) {
        case 1: KSR_NDIG(1); break;
        case 2: KSR_NDIG(2); break;
        case 3: KSR_NDIG(3); break;
        default: KSR_NDIG(4); break;
    }
#undef KSR_NDIG
#undef KSR_CASE
}

void ks_rotations(const ckks_ctx* c, const Digits& D, int ndig, int next, const int* ext_ids, const KsRotations& R,
                  const u64* x0, u64* ob, u64* oa, bool accumulate, const KsBatch& bt) {
    CK_CHECK(bt.nb >= 1 && ndig >= 1 && ndig <= 4 && R.nr >= 1 && R.nr <= KsRotations::fits(ndig), CKKS_EINVAL,
             "key switching takes 1..4 digits and as many rotations as one sum holds");
    const bool vec = al16_keys(R) && al16(ob) && al16(oa);
    {
        // algorithmic bytes: the keys once for the whole batch, per ciphertext its digits and x0 rows, and
        // the outputs (read too when accumulating)
        KTimer kt_(c, "ks_inner",
                   (R.nr * 2.0 * ndig + bt.nb * (R.nr * (ndig + 1.0) + (accumulate ? 4.0 : 2.0))) * next * c->n * 8.0);
        if (c->fold && vec) launch_ks_rotations<true, 2>(c, D, ndig, next, ext_ids, R, x0, ob, oa, accumulate, bt);
        else if (c->fold) launch_ks_rotations<true, 1>(c, D, ndig, next, ext_ids, R, x0, ob, oa, accumulate, bt);
        else launch_ks_rotations<false, 1>(c, D, ndig, next, ext_ids, R, x0, ob, oa, accumulate, bt);
    }
    LAUNCH_CHECK();
}

}  // namespace kern
