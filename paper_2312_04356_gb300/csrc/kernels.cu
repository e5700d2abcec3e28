// Device kernels of the RNS-CKKS hot path (all but the transforms, ntt.cu, the key-switch
// products, keyswitch.cu, and the tensor-core base conversion, convert_tc.cu) and their launchers.
//
// Layout: a polynomial is [limb][N] uint64, limb k of an array of several
// polynomials uses the prime with global id ids[k % lpp].  One CTA row of the
// grid (blockIdx.y) is one limb, so the modulus is uniform inside a CTA.
#include "words.cuh"

#include <atomic>

// ------------------------------------------------------------ DevBuf -------
thread_local const DevAlloc* tl_alloc = nullptr;

DevBuf::DevBuf(size_t w, cudaStream_t s) : words(w), stream(s) {
    if (w && tl_alloc && tl_alloc->alloc) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        CUDA_CHECK(cudaStreamIsCapturing(s, &cs));
        if (cs == cudaStreamCaptureStatusNone) {
            void* p = tl_alloc->alloc(tl_alloc->user, w * sizeof(u64), (void*)s);
            CK_CHECK(p != nullptr, CKKS_ENOMEM, "the caller's device allocator returned NULL");
            CK_CHECK(((uintptr_t)p & 15) == 0, CKKS_EINVAL, "the caller's device allocator returned a pointer "
                                                            "that is not 16-byte aligned");
            ptr = (u64*)p;
            al = *tl_alloc;
            return;
        }
    }
    if (w) {
        cudaError_t e = cudaMallocAsync((void**)&ptr, w * sizeof(u64), s);
        if (e != cudaSuccess) {
            ptr = nullptr;
            CK_THROW(CKKS_ENOMEM, std::string("device allocation failed: ") + cudaGetErrorString(e));
        }
    }
}
DevBuf::~DevBuf() { reset(); }
DevBuf& DevBuf::operator=(DevBuf&& o) noexcept {
    if (this != &o) {
        reset();
        ptr = o.ptr;
        words = o.words;
        stream = o.stream;
        al = o.al;
        o.ptr = nullptr;
        o.words = 0;
        o.al = DevAlloc();
    }
    return *this;
}
void DevBuf::reset() {
    if (ptr) {
        if (al.free)
            al.free(al.user, ptr, words * sizeof(u64), (void*)stream);
        else if (!al.alloc)
            cudaFreeAsync(ptr, stream);
    }
    ptr = nullptr;
    words = 0;
    al = DevAlloc();
}

static cudaEvent_t take_event(const ckks_ctx* c) {
    if (!c->event_pool.empty()) {
        cudaEvent_t e = c->event_pool.back();
        c->event_pool.pop_back();
        return e;
    }
    cudaEvent_t e;
    cudaEventCreate(&e);
    return e;
}

KTimer::KTimer(const ckks_ctx* ctx, const char* nm, double algo_bytes) : c(ctx), name(nm), bytes(algo_bytes) {
    ++c->launches;
    if (c->timing) {
        a = take_event(c);
        b = take_event(c);
        cudaEventRecord(a, c->stream);
    }
}

KTimer::~KTimer() {
    if (a) {
        cudaEventRecord(b, c->stream);
        c->pending.push_back({name, a, b, bytes});
        if (c->pending.size() > 4096) c->collect_timing();
    }
}

void ckks_ctx::collect_timing() const {
    if (pending.empty()) return;
    cudaEventSynchronize(pending.back().b);
    for (const Pending& p : pending) {
        float ms = 0;
        cudaEventElapsedTime(&ms, p.a, p.b);
        KStat& st = kstats[p.name];
        st.launches += 1;
        st.ms += ms;
        st.bytes += p.bytes;
        event_pool.push_back(p.a);
        event_pool.push_back(p.b);
    }
    pending.clear();
}

namespace {

inline dim3 ew_grid(int n, int nlimbs) {
    int x = n / (EW_THREADS * 4);
    if (x < 1) x = 1;
    return dim3(x, nlimbs);
}

#define EW_LOOP(n) for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < (n); j += gridDim.x * blockDim.x)

// words per thread of the elementwise kernels when every pointer is 16-byte aligned and a CTA's
// words lie in one limb
constexpr int EWV_VEC = 4;
#define EWV_LAUNCH(K, vec, nl, ...)                                                          \
    do {                                                                                     \
        if ((vec) && c->n >= EWV_VEC * EW_THREADS)                                           \
            klaunch(c, K<EWV_VEC>, ewv_grid(c->n, (nl), EWV_VEC), EW_THREADS, 0, __VA_ARGS__); \
        else                                                                                 \
            klaunch(c, K<1>, ewv_grid(c->n, (nl), 1), EW_THREADS, 0, __VA_ARGS__);        \
    } while (0)
// the same for kernels that reduce products
#define EWV_LAUNCH_RED(K, V, vec, zdim, nl, ...)                                             \
    do {                                                                                     \
        const bool vec_ = (vec) && c->n >= (V) * EW_THREADS;                                 \
        dim3 grid_ = ewv_grid(c->n, (nl), vec_ ? (V) : 1);                                   \
        grid_.z = (zdim);                                                                    \
        if (vec_ && c->fold) klaunch(c, K<V, true>, grid_, EW_THREADS, 0, __VA_ARGS__);      \
        else if (vec_) klaunch(c, K<V, false>, grid_, EW_THREADS, 0, __VA_ARGS__);           \
        else if (c->fold) klaunch(c, K<1, true>, grid_, EW_THREADS, 0, __VA_ARGS__);         \
        else klaunch(c, K<1, false>, grid_, EW_THREADS, 0, __VA_ARGS__);                     \
    } while (0)

// ----------------------------------------------------------- elementwise ----
template <int V>
__global__ void k_add(const u64* a, const u64* b, u64* o, const DevPrime* P, const int* ids, int lpp, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const u64 q = P[ids[limb % lpp]].m.q;
    const size_t off = (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V], y[V];
    ldv<V>(a + off + j, x);
    ldv<V>(b + off + j, y);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = add_mod(x[v], y[v], q);
    stv<V>(o + off + j, x);
}
template <int V>
__global__ void k_sub(const u64* a, const u64* b, u64* o, const DevPrime* P, const int* ids, int lpp, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const u64 q = P[ids[limb % lpp]].m.q;
    const size_t off = (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V], y[V];
    ldv<V>(a + off + j, x);
    ldv<V>(b + off + j, y);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = sub_mod(x[v], y[v], q);
    stv<V>(o + off + j, x);
}
template <int V>
__global__ void k_neg(const u64* a, u64* o, const DevPrime* P, const int* ids, int lpp, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const u64 q = P[ids[limb % lpp]].m.q;
    const size_t off = (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V];
    ldv<V>(a + off + j, x);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = neg_mod(x[v], q);
    stv<V>(o + off + j, x);
}
// bmod > 0: b is broadcast, row limb % bmod of b multiplies row limb of a (one plaintext times
// every polynomial of a batch of ciphertexts)
template <int V, bool FOLD>
__global__ void k_mul(const u64* a, const u64* b, u64* o, const DevPrime* P, const int* ids, int lpp, int logn,
                      int bmod) {
    griddep_entry();
    const int limb = blockIdx.y;
    const Reducer<FOLD> red(P[ids[limb % lpp]]);
    const size_t off = (size_t)limb << logn;
    const size_t boff = (size_t)(bmod ? limb % bmod : limb) << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V], y[V];
    ldv<V>(a + off + j, x);
    ldv<V>(b + boff + j, y);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = red.mul(x[v], y[v]);
    stv<V>(o + off + j, x);
}
// tensor product of two ciphertexts: d0 = a0 b0, d1 = a0 b1 + a1 b0 (d [2][nl][N]), d2 = a1 b1
// (e [nl][N]); a, b [2][nl][N]; one pass over the nl limbs
// blockIdx.z: ciphertext t of a batch, its operands at a + t abs, b + t abs, d + t dbs, e + t ebs
template <int V, bool FOLD>
__global__ void k_tensor(const u64* a, const u64* b, u64* d, u64* e, const DevPrime* P, const int* ids, int nl,
                         int logn, size_t abs, size_t dbs, size_t ebs) {
    griddep_entry();
    const int limb = blockIdx.y;
    const Reducer<FOLD> red(P[ids[limb]]);
    const size_t off = (size_t)limb << logn, ps = (size_t)nl << logn;
    a += blockIdx.z * abs;
    b += blockIdx.z * abs;
    d += blockIdx.z * dbs;
    e += blockIdx.z * ebs;
    EWV_BEGIN(1 << logn)
    u64 a0[V], a1[V], b0[V], b1[V], d0[V], d1[V], d2[V];
    ldv<V>(a + off + j, a0);
    ldv<V>(a + ps + off + j, a1);
    ldv<V>(b + off + j, b0);
    ldv<V>(b + ps + off + j, b1);
#pragma unroll
    for (int v = 0; v < V; ++v) {
        d0[v] = red.mul(a0[v], b0[v]);
        u64 lo = 0, hi = 0;
        mac128(lo, hi, a0[v], b1[v]);
        mac128(lo, hi, a1[v], b0[v]);
        d1[v] = red(hi, lo);
        d2[v] = red.mul(a1[v], b1[v]);
    }
    stv<V>(d + off + j, d0);
    stv<V>(d + ps + off + j, d1);
    stv<V>(e + off + j, d2);
}
template <int V, bool FOLD>
__global__ void k_mul_acc(const u64* a, const u64* b, u64* o, const DevPrime* P, const int* ids, int lpp, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const Reducer<FOLD> red(P[ids[limb % lpp]]);
    const size_t off = (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V], y[V], z[V];
    ldv<V>(a + off + j, x);
    ldv<V>(b + off + j, y);
    ldv<V>(o + off + j, z);
#pragma unroll
    for (int v = 0; v < V; ++v) z[v] = add_mod(z[v], red.mul(x[v], y[v]), red.q);
    stv<V>(o + off + j, z);
}
template <int V>
__global__ void k_mul_scalar(const u64* a, const u64* s, const u64* sp, u64* o, const DevPrime* P, const int* ids,
                             int lpp, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const u64 q = P[ids[r]].m.q;
    const u64 w = s[r], wp = sp[r];
    const size_t off = (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V];
    ldv<V>(a + off + j, x);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = mul_shoup(x[v], w, wp, q);
    stv<V>(o + off + j, x);
}
// per-limb scalars passed by value (no host-to-device copy, so the launch can be captured)
template <int V>
__global__ void k_mul_scalar_v(const u64* a, ScalarVec sv, u64* o, const DevPrime* P, const int* ids, int lpp,
                               size_t a_pstride, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const u64 q = P[ids[r]].m.q;
    const u64 w = sv.v[r], wp = sv.vp[r];
    const size_t off = (size_t)limb << logn;
    const size_t offa = a_pstride ? (size_t)(limb / lpp) * a_pstride + ((size_t)r << logn) : off;
    EWV_BEGIN(1 << logn)
    u64 x[V];
    ldv<V>(a + offa + j, x);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = mul_shoup(x[v], w, wp, q);
    stv<V>(o + off + j, x);
}
template <int V>
__global__ void k_lincomb(const __grid_constant__ kern::LinComb T, u64* __restrict__ o,
                          const DevPrime* __restrict__ P, const int* __restrict__ ids, int lpp, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const u64 q = P[ids[r]].m.q;
    const size_t off = (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = 0;
    for (int t = 0; t < T.n; ++t) {
        const u64 w = T.w[t][r], wp = T.wp[t][r];
        u64 x[V];
        ldv<V>(T.a[t] + off + j, x);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = add_mod(acc[v], mul_shoup(x[v], w, wp, q), q);
    }
    stv<V>(o + off + j, acc);
}
// ps > 0: row limb of a at (limb / lpp) ps + (limb % lpp) N (e.g. c0 of every ciphertext of a batch)
template <int V>
__global__ void k_add_scalar_v(u64* a, ScalarVec sv, const DevPrime* P, const int* ids, int lpp, int logn,
                               size_t ps) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const u64 q = P[ids[r]].m.q;
    const u64 c = sv.v[r];
    const size_t off = ps ? (size_t)(limb / lpp) * ps + ((size_t)r << logn) : (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V];
    ldv<V>(a + off + j, x);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = add_mod(x[v], c, q);
    stv<V>(a + off + j, x);
}
template <int V>
__global__ void k_add_scalar(u64* a, const u64* vals, const DevPrime* P, const int* ids, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const u64 q = P[ids[limb]].m.q;
    const u64 c = vals[limb];
    const size_t off = (size_t)limb << logn;
    EWV_BEGIN(1 << logn)
    u64 x[V];
    ldv<V>(a + off + j, x);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = add_mod(x[v], c, q);
    stv<V>(a + off + j, x);
}
__global__ void k_small_to_rns(const int64_t* v, u64* o, const DevPrime* P, const int* ids, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const DevMod m = P[ids[limb]].m;
    const size_t off = (size_t)limb << logn;
    EW_LOOP(1 << logn) {
        const int64_t x = v[j];
        if (x >= 0) {
            o[off + j] = reduce64((u64)x, m);
        } else {
            const u64 r = reduce64((u64)(-(x + 1)) + 1ull, m);
            o[off + j] = r ? m.q - r : 0;
        }
    }
}
__global__ void k_automorph(const u64* a, u64* o, u64 g, int logn) {
    griddep_entry();
    const size_t off = (size_t)blockIdx.y << logn;
    EW_LOOP(1 << logn) o[off + j] = a[off + galois_src(j, g, logn)];
}
__global__ void k_imult(const u64* a, u64* o, const DevPrime* P, const int* ids, int lpp, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const DevPrime* pr = P + ids[limb % lpp];
    const u64 q = pr->m.q;
    // X^{N/2} at psi^(2r+1): psi^{N/2} when r is even, -psi^{N/2} when r is odd;
    // psi^{N/2} is the prime's im
    const u64 w = pr->im, wp = pr->im_p;
    const size_t off = (size_t)limb << logn;
    EW_LOOP(1 << logn) {
        u64 v = mul_shoup(a[off + j], w, wp, q);
        unsigned r = brev_bits(j, logn);
        o[off + j] = (r & 1) ? neg_mod(v, q) : v;
    }
}
template <int V>
__global__ void k_lift_centred(const u64* src, u64 qs, u64* o, const DevPrime* P, const int* ids, int lpp,
                               size_t src_pstride, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const DevMod t = P[ids[limb % lpp]].m;
    const size_t off = (size_t)limb << logn;
    const u64* sr = src + (size_t)(limb / lpp) * src_pstride;
    EWV_BEGIN(1 << logn)
    u64 x[V];
    ldv<V>(sr + j, x);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = centred_to(x[v], qs, t);
    stv<V>(o + off + j, x);
}
template <int V>
__global__ void k_sub_mul2_scalar(const u64* a, const u64* b, ScalarVec s1, const u64* s2, const u64* s2p, u64* o,
                                  const DevPrime* P, const int* ids, int lpp, size_t a_pstride, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const u64 q = P[ids[r]].m.q;
    const u64 w1 = s1.v[r], w1p = s1.vp[r], w2 = s2[r], w2p = s2p[r];
    const size_t off = (size_t)limb << logn;
    const size_t offa = a_pstride ? (size_t)(limb / lpp) * a_pstride + ((size_t)r << logn) : off;
    EWV_BEGIN(1 << logn)
    u64 x[V], y[V];
    ldv<V>(a + offa + j, x);
    ldv<V>(b + off + j, y);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = sub_mod(mul_shoup(x[v], w1, w1p, q), mul_shoup(y[v], w2, w2p, q), q);
    stv<V>(o + off + j, x);
}
template <int V>
__global__ void k_sub_mul_scalar(const u64* a, const u64* b, const u64* s, const u64* sp, u64* o,
                                 const DevPrime* P, const int* ids, int lpp, size_t a_pstride, int logn) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const u64 q = P[ids[r]].m.q;
    const u64 w = s[r], wp = sp[r];
    const size_t off = (size_t)limb << logn;
    const size_t offa = a_pstride ? (size_t)(limb / lpp) * a_pstride + ((size_t)r << logn) : off;
    EWV_BEGIN(1 << logn)
    u64 x[V], y[V];
    ldv<V>(a + offa + j, x);
    ldv<V>(b + off + j, y);
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = mul_shoup(sub_mod(x[v], y[v], q), w, wp, q);
    stv<V>(o + off + j, x);
}

// ------------------------------------------------------- base conversion ----
// y_m = sum_i [x_i * qhat_i^{-1}]_{q_i} * (qhat_i mod p_m)  (no correction term), or, for an
// exact table, minus v (Q mod p_m) with v = round(sum_i xhat_i / q_i) (Halevi, Polyakov,
// Shoup 2019), evaluated in 58-bit fixed point (conv_round_term): y then represents the
// centred remainder of x mod Q, up to a rounding error that matters only within 2^-53 of a
// half-integer.
// One thread per coefficient; grid.z walks over (job, group of MC <= CONV_OUT outputs), so
// the digits of one ModUp (or the two halves of one ModDown) share a launch.  The products
// are summed exactly in 128 bits (each < 2^122, at most 16 terms) and reduced once:
// (H 2^64 + L) mod p = H (2^64 mod p) + L mod p.  The output loop is unrolled so that the
// MC independent accumulations interleave.
constexpr int MAX_CONV_IN = 16;
constexpr int CONV_OUT = 8;
// MAXIN: compile-time bound on the jobs' input counts (4, 8 or 16), so that the unrolled
// input loops carry no predicated-off iterations for the common 7- and 8-limb conversions.
// SPLIT (every modulus below 2^60, MAXIN <= 8): x = xu 2^30 + xl, c = cu 2^30 + cl; the four
// partial products (each < 2^60) go into three 64-bit sums by one 32x32->64 multiply-add
// each (at most 16 terms per sum: no overflow); the 128-bit total ll + m 2^30 + hh 2^60 is
// then reduced as in the general path.
// MC: outputs per CTA group (4..8), chosen per launch to leave the fewest idle output slots.
template <int MAXIN, bool SPLIT, int MC>
__global__ void __launch_bounds__(256, (MC <= 6 ? 4 : 3)) k_base_convert(kern::ConvJobs J, const DevPrime* __restrict__ P, int logn) {
    griddep_entry();
    __shared__ u64 s_qi[MAX_CONV_IN], s_qinv[MAX_CONV_IN], s_qinvp[MAX_CONV_IN];
    __shared__ u64 s_c[CONV_OUT][MAX_CONV_IN];
    __shared__ DevPrime s_pm[CONV_OUT];
    __shared__ int s_row[CONV_OUT];
    __shared__ u64 s_invm[MAX_CONV_IN];
    __shared__ int s_invs[MAX_CONV_IN];
    __shared__ u64 s_corr[CONV_OUT];
    __shared__ uint2 s_c2[CONV_OUT][MAXIN];     // SPLIT: (c mod 2^30, c >> 30)
    // which job and output group this CTA serves
    int z = blockIdx.z, jb = 0;
    while (jb < J.n - 1 && z >= J.job[jb].ngroups) {
        z -= J.job[jb].ngroups;
        ++jb;
    }
    const kern::ConvJob& job = J.job[jb];
    const int nin = job.nin, nout = job.nout;
    const int m0 = z * MC;
    const int mcount = min(MC, nout - m0);
    const int tid = threadIdx.x;
    const bool exact = job.inv_q != nullptr;
    if (tid < nin) {
        s_qi[tid] = P[job.in_ids[tid]].m.q;
        s_qinv[tid] = job.qinv[tid];
        s_qinvp[tid] = job.qinv[nin + tid];
        s_invm[tid] = exact ? job.inv_q[tid] : 0;
        s_invs[tid] = exact ? (int)job.inv_q[nin + tid] : 64;
    }
    if (tid < CONV_OUT * MAX_CONV_IN) {
        const int m = tid / MAX_CONV_IN, i = tid % MAX_CONV_IN;
        const u64 c = (m < mcount && i < nin) ? job.qmod[(size_t)(m0 + m) * nin + i] : 0;
        s_c[m][i] = c;
        if (SPLIT && i < MAXIN) s_c2[m][i] = make_uint2((unsigned)(c & ((1ull << 30) - 1)), (unsigned)(c >> 30));
    }
    if (tid < mcount) {
        s_pm[tid] = P[job.out_ids[m0 + tid]];
        s_row[tid] = job.out_rows[m0 + tid];
        s_corr[tid] = exact ? job.corr[m0 + tid] : 0;
    }
    __syncthreads();
    const u64* in = job.in + blockIdx.y * job.in_pstride;
    u64* out = job.out + blockIdx.y * job.out_pstride;
    const int j = blockIdx.x * blockDim.x + tid;
    if (j >= (1 << logn)) return;
    const size_t n = (size_t)1 << logn;
    u64 xh[MAXIN];
#pragma unroll
    for (int i = 0; i < MAXIN; ++i)
        if (i < nin) xh[i] = job.prescaled ? in[i * n + j] : mul_shoup(in[i * n + j], s_qinv[i], s_qinvp[i], s_qi[i]);
    u64 lo[MC], hi[MC];
    if (SPLIT) {
        constexpr u64 M30 = (1ull << 30) - 1;
        u64 ll[MC], mm[MC], hh[MC];
#pragma unroll
        for (int m = 0; m < MC; ++m) ll[m] = mm[m] = hh[m] = 0;
#pragma unroll
        for (int i = 0; i < MAXIN; ++i) {
            if (i < nin) {
                const unsigned xl = (unsigned)(xh[i] & M30), xu = (unsigned)(xh[i] >> 30);
#pragma unroll
                for (int m = 0; m < MC; ++m) {
                    const uint2 cc = s_c2[m][i];
                    ll[m] += (u64)xl * cc.x;
                    mm[m] += (u64)xl * cc.y;
                    mm[m] += (u64)xu * cc.x;
                    hh[m] += (u64)xu * cc.y;
                }
            }
        }
#pragma unroll
        for (int m = 0; m < MC; ++m) {
            u64 l = ll[m], h = (mm[m] >> 34) + (hh[m] >> 4);
            const u64 t1 = mm[m] << 30;
            l += t1;
            h += l < t1 ? 1ull : 0ull;
            const u64 t2 = hh[m] << 60;
            l += t2;
            h += l < t2 ? 1ull : 0ull;
            lo[m] = l;
            hi[m] = h;
        }
    } else {
#pragma unroll
        for (int m = 0; m < MC; ++m) lo[m] = hi[m] = 0;
#pragma unroll
        for (int i = 0; i < MAXIN; ++i) {
            if (i < nin) {
#pragma unroll
                for (int m = 0; m < MC; ++m) {
                    const u64 c = s_c[m][i];
                    const u64 pl = xh[i] * c, ph = __umul64hi(xh[i], c);
                    lo[m] += pl;
                    hi[m] += ph + (lo[m] < pl ? 1ull : 0ull);
                }
            }
        }
    }
    if (exact) {
        u64 f = 0;
#pragma unroll
        for (int i = 0; i < MAXIN; ++i)
            if (i < nin) f += conv_round_term(xh[i], s_invm[i], s_invs[i]);
        const u64 v = conv_round_finish(f);
#pragma unroll
        for (int m = 0; m < MC; ++m) {
            const u64 pl = v * s_corr[m], ph = __umul64hi(v, s_corr[m]);
            lo[m] += pl;
            hi[m] += ph + (lo[m] < pl ? 1ull : 0ull);
        }
    }
#pragma unroll
    for (int m = 0; m < MC; ++m)
        if (m < mcount) out[(size_t)s_row[m] * n + j] = reduce128_lazy(hi[m], lo[m], s_pm[m]);
}

// o += a * s[limb % lpp] (Shoup pairs s, sp)
template <int V>
// o_ps > 0: row limb of o at (limb / lpp) o_ps + (limb % lpp) N (a contiguous)
__global__ void k_mul_scalar_acc(const u64* a, const u64* s, const u64* sp, u64* o, const DevPrime* P, const int* ids,
                                 int lpp, int logn, size_t o_ps) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int r = limb % lpp;
    const u64 q = P[ids[r]].m.q;
    const u64 w = s[r], wp = sp[r];
    const size_t off = (size_t)limb << logn;
    const size_t ooff = o_ps ? (size_t)(limb / lpp) * o_ps + ((size_t)r << logn) : off;
    EWV_BEGIN(1 << logn)
    u64 x[V], z[V];
    ldv<V>(a + off + j, x);
    ldv<V>(o + ooff + j, z);
#pragma unroll
    for (int v = 0; v < V; ++v) z[v] = add_mod(z[v], mul_shoup(x[v], w, wp, q), q);
    stv<V>(o + ooff + j, z);
}

// ------------------------------------------------------------- decoding ----
// Column j of the limbs: mixed-radix digits v_i = (r_i - sum_{t<i} v_t prod_{k<t} q_k)
// (prod_{k<i} q_k)^{-1} mod q_i, written over the residues; (Q - 1) / 2 has the digits (q_i - 1) / 2, so the
// first digit from the top that differs decides the sign, and Q - x has the digits q_i - 1 - v_i
// plus one.  tab[i][t] = prod_{k<t} q_k mod q_i (t < i),
// tab[i][i] the inverse.  A host loop over 65536 coefficients of 6 limbs took 27 ms; this
// kernel and the copy of N doubles take under 0.1 ms.
__global__ void k_garner(u64* __restrict__ limbs, double* __restrict__ out, const DevPrime* __restrict__ P,
                         const ulonglong2* __restrict__ tab, int nl, int nq, int logn) {
    griddep_entry();
    const size_t n = (size_t)1 << logn;
    EW_LOOP(1 << logn) {
        u64* col = limbs + j;
        for (int i = 0; i < nl; ++i) {
            const u64 q = P[i].m.q;
            u64 acc = 0;
            for (int t = 0; t < i; ++t) {
                const ulonglong2 w = tab[(size_t)i * nq + t];
                acc = add_mod(acc, mul_shoup(col[t * n], w.x, w.y, q), q);
            }
            const ulonglong2 w = tab[(size_t)i * nq + i];
            col[i * n] = mul_shoup(sub_mod(col[i * n], acc, q), w.x, w.y, q);
        }
        bool neg = false;
        for (int i = nl - 1; i >= 0; --i) {
            const u64 v = col[i * n], h = (P[i].m.q - 1) / 2;
            if (v != h) {
                neg = v > h;
                break;
            }
        }
        if (neg) {
            u64 carry = 1;
            for (int i = 0; i < nl; ++i) {
                const u64 q = P[i].m.q;
                u64 v = q - 1 - col[i * n] + carry;
                carry = v == q;
                col[i * n] = carry ? 0 : v;
            }
        }
        double x = 0.0;
        for (int i = nl - 1; i >= 0; --i) x = fma(x, (double)P[i].m.q, (double)col[i * n]);
        out[j] = neg ? -x : x;
    }
}

// ------------------------------------------------------------ sampling ----
__device__ __forceinline__ u64 d_mix(u64 z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
__device__ __forceinline__ u64 d_word(u64 key, u64 i) { return d_mix(key + (i + 1) * 0x9E3779B97F4A7C15ULL); }

__global__ void k_sample_uniform(u64* o, const DevPrime* P, const int* ids, int logn, u64 key) {
    griddep_entry();
    const int limb = blockIdx.y;
    const int id = ids[limb];
    const DevMod m = P[id].m;
    const u64 two64 = barrett_reduce128(1, 0, m);   // 2^64 mod q
    const size_t off = (size_t)limb << logn;
    EW_LOOP(1 << logn) {
        const u64 k = ((u64)id << logn) + (u64)j;
        const u64 w1 = d_word(key, 2 * k), w2 = d_word(key, 2 * k + 1);
        o[off + j] = add_mod(mul_mod(reduce64(w1, m), two64, m), reduce64(w2, m), m.q);
    }
}
__global__ void k_sample_small(int64_t* o, int logn, u64 key, int kind, const u64* gauss) {
    griddep_entry();
    EW_LOOP(1 << logn) {
        const u64 w = d_word(key, (u64)j);
        if (kind == 0) {
            o[j] = (int64_t)(w % 3ull) - 1;
        } else {
            const u64 u = w >> 1;
            int k = 0;
            while (k < 38 && u >= gauss[k]) ++k;
            o[j] = (int64_t)k - 19;
        }
    }
}

}  // namespace

// ------------------------------------------------------------- launchers ---
namespace kern {

#define LAUNCH_CHECK() CUDA_CHECK(cudaGetLastError())

void add(const ckks_ctx* c, const u64* a, const u64* b, u64* o, int nl, const int* ids, int lpp) {
    if (nl <= 0) return;
    { KTimer kt_(c, "add", 3.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_add, al16(a) && al16(b) && al16(o), nl, a, b, o, c->d_primes, ids, lpp, c->logn);
    }
    LAUNCH_CHECK();
}
void sub(const ckks_ctx* c, const u64* a, const u64* b, u64* o, int nl, const int* ids, int lpp) {
    if (nl <= 0) return;
    { KTimer kt_(c, "sub", 3.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_sub, al16(a) && al16(b) && al16(o), nl, a, b, o, c->d_primes, ids, lpp, c->logn);
    }
    LAUNCH_CHECK();
}
void neg(const ckks_ctx* c, const u64* a, u64* o, int nl, const int* ids, int lpp) {
    if (nl <= 0) return;
    { KTimer kt_(c, "neg", 2.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_neg, al16(a) && al16(o), nl, a, o, c->d_primes, ids, lpp, c->logn);
    }
    LAUNCH_CHECK();
}
void mul(const ckks_ctx* c, const u64* a, const u64* b, u64* o, int nl, const int* ids, int lpp, int bmod) {
    if (nl <= 0) return;
    { KTimer kt_(c, "mul", (bmod ? 2.0 + (double)bmod / nl : 3.0) * (double)nl * c->n * 8.0);
    EWV_LAUNCH_RED(k_mul, EWV_VEC, al16(a) && al16(b) && al16(o), 1, nl, a, b, o, c->d_primes, ids, lpp, c->logn, bmod);
    }
    LAUNCH_CHECK();
}
void tensor(const ckks_ctx* c, const u64* a, const u64* b, u64* d, u64* e, int nl, const int* ids, int nb,
            size_t ab_bstride, size_t d_bstride, size_t e_bstride) {
    if (nl <= 0 || nb <= 0) return;
    { KTimer kt_(c, "tensor", 7.0 * (double)nl * nb * c->n * 8.0);
    EWV_LAUNCH_RED(k_tensor, 2, al16(a) && al16(b) && al16(d) && al16(e), nb, nl, a, b, d, e, c->d_primes, ids, nl,
                   c->logn, ab_bstride, d_bstride, e_bstride);
    }
    LAUNCH_CHECK();
}
void mul_acc(const ckks_ctx* c, const u64* a, const u64* b, u64* o, int nl, const int* ids, int lpp) {
    if (nl <= 0) return;
    { KTimer kt_(c, "mul_acc", 4.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH_RED(k_mul_acc, EWV_VEC, al16(a) && al16(b) && al16(o), 1, nl, a, b, o, c->d_primes, ids, lpp, c->logn);
    }
    LAUNCH_CHECK();
}
void mul_scalar(const ckks_ctx* c, const u64* a, const u64* s, const u64* sp, u64* o, int nl, const int* ids,
                int lpp) {
    if (nl <= 0) return;
    { KTimer kt_(c, "mul_scalar", 2.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_mul_scalar, al16(a) && al16(o), nl, a, s, sp, o, c->d_primes, ids, lpp, c->logn);
    }
    LAUNCH_CHECK();
}
void mul_scalar_v(const ckks_ctx* c, const u64* a, const ScalarVec& sv, u64* o, int nl, const int* ids, int lpp,
                  size_t a_pstride) {
    if (nl <= 0) return;
    CK_CHECK(lpp <= ScalarVec::MAX, CKKS_EINVAL, "too many limbs for a by-value scalar vector");
    { KTimer kt_(c, "mul_scalar", 2.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_mul_scalar_v, al16(a) && al16(o) && a_pstride % 2 == 0, nl, a, sv, o, c->d_primes, ids, lpp,
               a_pstride, c->logn);
    }
    LAUNCH_CHECK();
}
void sub_mul2_scalar(const ckks_ctx* c, const u64* a, const u64* b, const ScalarVec& s1, const u64* s2,
                     const u64* s2p, u64* o, int nl, const int* ids, int lpp, size_t a_pstride) {
    if (nl <= 0) return;
    CK_CHECK(lpp <= ScalarVec::MAX, CKKS_EINVAL, "too many limbs for a by-value scalar vector");
    { KTimer kt_(c, "sub_mul_scalar", 3.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_sub_mul2_scalar, al16(a) && al16(b) && al16(o) && a_pstride % 2 == 0, nl, a, b, s1, s2, s2p, o,
               c->d_primes, ids, lpp, a_pstride, c->logn);
    }
    LAUNCH_CHECK();
}
void lincomb(const ckks_ctx* c, const LinComb& t, u64* o, int nl, const int* ids, int lpp) {
    if (nl <= 0) return;
    CK_CHECK(t.n >= 1 && t.n <= LinComb::MAX && lpp <= LinComb::MAXL, CKKS_EINVAL,
             "1..16 terms over at most 40 limbs per linear combination");
    bool vec = al16(o);
    for (int i = 0; i < t.n; ++i) vec = vec && al16(t.a[i]);
    { KTimer kt_(c, "lincomb", (t.n + 1.0) * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_lincomb, vec, nl, t, o, c->d_primes, ids, lpp, c->logn);
    }
    LAUNCH_CHECK();
}
void add_scalar_v(const ckks_ctx* c, u64* a, const ScalarVec& sv, int nl, const int* ids, int lpp,
                  size_t a_pstride) {
    if (nl <= 0) return;
    CK_CHECK(lpp <= ScalarVec::MAX, CKKS_EINVAL, "too many limbs for a by-value scalar vector");
    { KTimer kt_(c, "add_scalar", 2.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_add_scalar_v, al16(a) && a_pstride % 2 == 0, nl, a, sv, c->d_primes, ids, lpp, c->logn, a_pstride);
    }
    LAUNCH_CHECK();
}
void add_const_term(const ckks_ctx* c, u64* a, const u64* v, int nl, const int* ids) {
    if (nl <= 0) return;
    { KTimer kt_(c, "add_scalar", 2.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_add_scalar, al16(a), nl, a, v, c->d_primes, ids, c->logn);
    }
    LAUNCH_CHECK();
}
void small_to_rns(const ckks_ctx* c, const int64_t* v, u64* o, int nl, const int* ids) {
    if (nl <= 0) return;
    { KTimer kt_(c, "small_to_rns", (nl + 1.0) * c->n * 8.0);
    klaunch(c, k_small_to_rns, ew_grid(c->n, nl), EW_THREADS, 0, v, o, c->d_primes, ids, c->logn);
    }
    LAUNCH_CHECK();
}
void automorph(const ckks_ctx* c, const u64* a, u64* o, int nl, u64 g) {
    if (nl <= 0) return;
    { KTimer kt_(c, "automorph", 2.0 * (double)nl * c->n * 8.0);
    klaunch(c, k_automorph, ew_grid(c->n, nl), EW_THREADS, 0, a, o, g, c->logn);
    }
    LAUNCH_CHECK();
}
void imult(const ckks_ctx* c, const u64* a, u64* o, int nl, const int* ids, int lpp) {
    if (nl <= 0) return;
    { KTimer kt_(c, "imult", 2.0 * (double)nl * c->n * 8.0);
    klaunch(c, k_imult, ew_grid(c->n, nl), EW_THREADS, 0, a, o, c->d_primes, ids, lpp, c->logn);
    }
    LAUNCH_CHECK();
}
void lift_centred(const ckks_ctx* c, const u64* src, int src_id, u64* o, int nl, const int* ids, int lpp,
                  size_t src_pstride) {
    if (nl <= 0) return;
    if (lpp <= 0) lpp = nl;
    { KTimer kt_(c, "lift_centred", (nl + 1.0) * c->n * 8.0);
    EWV_LAUNCH(k_lift_centred, al16(src) && al16(o) && src_pstride % 2 == 0, nl, src, c->mod_of[src_id], o,
               c->d_primes, ids, lpp, src_pstride, c->logn);
    }
    LAUNCH_CHECK();
}
void sub_mul_scalar(const ckks_ctx* c, const u64* a, const u64* b, const u64* s, const u64* sp, u64* o, int nl,
                    const int* ids, int lpp, size_t a_pstride) {
    if (nl <= 0) return;
    { KTimer kt_(c, "sub_mul_scalar", 3.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_sub_mul_scalar, al16(a) && al16(b) && al16(o) && a_pstride % 2 == 0, nl, a, b, s, sp, o, c->d_primes,
               ids, lpp, a_pstride, c->logn);
    }
    LAUNCH_CHECK();
}
void base_convert(const ckks_ctx* c, const ConvTab& t, const u64* in, size_t in_stride, u64* out,
                  size_t out_stride, int npoly, size_t in_pstride, size_t out_pstride, bool prescaled) {
    CK_CHECK(in_stride == (size_t)c->n && out_stride == (size_t)c->n, CKKS_EINVAL, "limbs must be contiguous");
    ConvJobs J;
    J.n = 0;
    add_conv_job(J, t, in, out, in_pstride, out_pstride, prescaled);
    base_convert_jobs(c, J, npoly);
}

void add_conv_job(ConvJobs& J, const ConvTab& t, const u64* in, u64* out, size_t in_pstride, size_t out_pstride,
                  bool prescaled) {
    CK_CHECK(J.n < ConvJobs::MAX, CKKS_EINVAL, "too many base-conversion jobs");
    CK_CHECK(t.nin <= MAX_CONV_IN, CKKS_EINVAL, "base conversion with more than 16 input limbs");
    ConvJob& j = J.job[J.n++];
    j.in = in;
    j.out = out;
    j.in_ids = t.d_in_ids;
    j.out_ids = t.d_out_ids;
    j.out_rows = t.d_out_ids + t.nout;
    j.qinv = t.d_qhat_inv;
    j.qmod = t.d_qhat_mod;
    j.inv_q = t.d_inv_q;
    j.outs = t.d_outs;
    j.corr = t.d_corr;
    j.nin = t.nin;
    j.nout = t.nout;
    j.ngroups = (t.nout + CONV_OUT - 1) / CONV_OUT;
    j.in_pstride = in_pstride;
    j.out_pstride = out_pstride;
    j.prescaled = prescaled;
    j.tcb = t.d_tcb;
    j.tcr = t.d_tcr;
    j.tc_nin2 = t.tc_nin2;
    j.tc_S = t.tc_S;
}

template <int MAXIN, bool SPLIT>
static void launch_base_convert(const ckks_ctx* c, const ConvJobs& J, dim3 grid, int mc) {
    switch (mc) {
        case 4: klaunch(c, k_base_convert<MAXIN, SPLIT, 4>, grid, 256, 0, J, c->d_primes, c->logn); break;
        case 5: klaunch(c, k_base_convert<MAXIN, SPLIT, 5>, grid, 256, 0, J, c->d_primes, c->logn); break;
        case 6: klaunch(c, k_base_convert<MAXIN, SPLIT, 6>, grid, 256, 0, J, c->d_primes, c->logn); break;
        case 7: klaunch(c, k_base_convert<MAXIN, SPLIT, 7>, grid, 256, 0, J, c->d_primes, c->logn); break;
        default: klaunch(c, k_base_convert<MAXIN, SPLIT, 8>, grid, 256, 0, J, c->d_primes, c->logn); break;
    }
}

// Outputs per group MC in 4..8: the one with the fewest idle output slots over the launch's
// jobs (sum of ceil(nout / MC) MC - nout); on ties 6, 5, 4 (4 resident CTAs per SM) before
// 8, 7 (3 per SM).
void base_convert_jobs(const ckks_ctx* c, const ConvJobs& J0, int npoly) {
    if (conv_tc_eligible(c, J0)) {
        base_convert_tc_jobs(c, J0, npoly);
        LAUNCH_CHECK();
        return;
    }
    int best_mc = CONV_OUT, best_slots = -1;
    for (int mc : {6, 5, 4, 8, 7}) {
        int slots = 0;
        for (int i = 0; i < J0.n; ++i) slots += (J0.job[i].nout + mc - 1) / mc * mc;
        if (best_slots < 0 || slots < best_slots) {
            best_slots = slots;
            best_mc = mc;
        }
    }
    ConvJobs J = J0;
    int groups = 0;
    double bytes = 0;
    for (int i = 0; i < J.n; ++i) {
        J.job[i].ngroups = (J.job[i].nout + best_mc - 1) / best_mc;
        groups += J.job[i].ngroups;
        bytes += (double)npoly * (J.job[i].nin + J.job[i].nout) * c->n * 8.0;
    }
    if (groups == 0) return;
    int maxin = 0;
    for (int i = 0; i < J.n; ++i) maxin = std::max(maxin, J.job[i].nin);
    dim3 grid((c->n + 255) / 256, npoly, groups);
    { KTimer kt_(c, "base_convert", bytes);
    if (maxin <= 4)
        launch_base_convert<4, false>(c, J, grid, best_mc);
    else if (maxin <= 8 && c->mods_below_2_60)
        launch_base_convert<8, true>(c, J, grid, best_mc);
    else if (maxin <= 8)
        launch_base_convert<8, false>(c, J, grid, best_mc);
    else
        launch_base_convert<MAX_CONV_IN, false>(c, J, grid, best_mc);
    }
    LAUNCH_CHECK();
}

void mul_scalar_acc(const ckks_ctx* c, const u64* a, const u64* s, const u64* sp, u64* o, int nl, const int* ids,
                    int lpp, size_t o_pstride) {
    if (nl <= 0) return;
    { KTimer kt_(c, "mul_scalar_acc", 3.0 * (double)nl * c->n * 8.0);
    EWV_LAUNCH(k_mul_scalar_acc, al16(a) && al16(o) && o_pstride % 2 == 0, nl, a, s, sp, o, c->d_primes, ids, lpp,
               c->logn, o_pstride);
    }
    LAUNCH_CHECK();
}
void garner(const ckks_ctx* c, u64* limbs, double* out, int nl) {
    { KTimer kt_(c, "garner", (nl + 1.0) * c->n * 8.0);
    klaunch(c, k_garner, dim3((c->n + 127) / 128), 128, 0, limbs, out, c->d_primes, (const ulonglong2*)c->d_garner, nl,
            c->nq, c->logn);
    }
    LAUNCH_CHECK();
}
void sample_uniform(const ckks_ctx* c, u64* o, int nl, const int* ids, u64 key) {
    if (nl <= 0) return;
    { KTimer kt_(c, "sample_uniform", (double)nl * c->n * 8.0);
    klaunch(c, k_sample_uniform, ew_grid(c->n, nl), EW_THREADS, 0, o, c->d_primes, ids, c->logn, key);
    }
    LAUNCH_CHECK();
}
void sample_small(const ckks_ctx* c, int64_t* o, u64 key, int kind) {
    { KTimer kt_(c, "sample_small", c->n * 8.0);
    klaunch(c, k_sample_small, ew_grid(c->n, 1), EW_THREADS, 0, o, c->logn, key, kind, c->d_gauss);
    }
    LAUNCH_CHECK();
}

}  // namespace kern
