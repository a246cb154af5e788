// Device helpers: window evaluation, bulk async copies with bounded mbarrier
// waits, and the shared-memory mixed-radix FFT used for the oversampled grids.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "internal.cuh"

namespace agft {

// ---------------------------------------------------------- grid elements --

// Storage type of an FP32-computing plan's grids: complex FP32 (float2) or a
// pair of 16-bit floats (FP16 or BF16); values are widened to FP32 on load and
// rounded to nearest on store, every sum stays in FP32.
template <typename G>
struct GridEl;
template <>
struct GridEl<float2> {
    static __device__ __forceinline__ float2 load(float2 v) { return v; }
    static __device__ __forceinline__ float2 store(float a, float b) { return make_float2(a, b); }
};
template <>
struct GridEl<__half2> {
    static __device__ __forceinline__ float2 load(__half2 v) { return __half22float2(v); }
    static __device__ __forceinline__ __half2 store(float a, float b) { return __floats2half2_rn(a, b); }
};
template <>
struct GridEl<__nv_bfloat162> {
    static __device__ __forceinline__ float2 load(__nv_bfloat162 v) { return __bfloat1622float2(v); }
    static __device__ __forceinline__ __nv_bfloat162 store(float a, float b) { return __floats2bfloat162_rn(a, b); }
};

// ------------------------------------------------------------ cosine terms --
//
// A term of the half-period cosine system (Sec. 5) runs on the exponential
// grids: prod_t cos(pi k_t x_t) = 2^{-s} sum over sign patterns eps of
// exp(2 pi i <eps k, x / 2>), so with the nodes halved (plan time) its block
// coefficient fhat_k, k in {1..N/2-1}^s (N the term's doubled bandwidth),
// stands for 2^{-s/2} fhat_k at each of the 2^s exponential frequencies eps k,
// and the adjoint's coefficient is 2^{-s/2} times the sum over those
// frequencies.  cos_decode: block position q -> k (row-major, last axis
// fastest); cos_mirror: grid position of sign pattern sg (bit t negates axis
// t; negative frequencies at k + n) and the product of its deconvolution
// factors (column table on the last axis, row table on the others).
__device__ __forceinline__ void cos_decode(long long q, int s, int N, int (&k)[3]) {
    const int nc = N / 2 - 1;
    for (int t = s - 1; t >= 0; --t) {
        k[t] = (int)(q % nc) + 1;
        q /= nc;
    }
}

template <typename R>
__device__ __forceinline__ int cos_mirror(const int (&k)[3], int s, int sg, int N, int n, const R *deconv, int dc_off,
                                          int dr_off, R &D) {
    int pos = 0, mul = 1;
    for (int t = s - 1; t >= 0; --t) {
        const int kt = (sg >> t) & 1 ? -k[t] : k[t];
        const int it = kt < 0 ? kt + N / 2 : kt + N / 2 - 1;   // index in I_N minus {0}
        pos += (kt < 0 ? kt + n : kt) * mul;
        mul *= n;
        D *= (t == s - 1) ? deconv[dc_off + it] : deconv[dr_off + it];
    }
    return pos;
}

// 2^{-s/2}
__host__ __device__ __forceinline__ double cos_amp(int s) {
    return s == 1 ? 0.70710678118654752440 : s == 2 ? 0.5 : 0.35355339059327376220;
}

// ---- packed FP32 pairs ----
//
// sm_100-class GPUs execute two FP32 fused multiply-adds of one lane in one
// instruction (fma.rn.f32x2 on a 64-bit register pair) at the same FMA rate,
// which halves the issue slots of independent pairs of operations; each half
// rounds exactly as the scalar fmaf does.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(f32x2 r, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// ---------------------------------------------------------------- windows --

// ---- TF32 tensor-core products with FP32-level accuracy ----
//
// The fragment layouts of mma.m16n8k8 with TF32 operands (PTX ISA), lane =
// 4 g + t: A (16 x 8) a0 = A[g][t], a1 = A[g + 8][t], a2 = A[g][t + 4],
// a3 = A[g + 8][t + 4]; B (8 x 8) b0 = B[t][g], b1 = B[t + 4][g]; C, D
// (16 x 8) d0 = D[g][2t], d1 = D[g][2t + 1], d2 = D[g + 8][2t],
// d3 = D[g + 8][2t + 1].  A product a b of FP32 values is taken as
// ah bh + ah bl + al bh with x = xh + xl split below.

// x = hi + lo for two finite values at once, in three packed operations: c = fl(x + 2^13 x) =
// fl(8193 x), hi = c - 2^13 x (exact: one fma), lo = x - hi (exact: the
// rounding error of c).  ulp(c) >= 2^13 ulp(x), so hi is a multiple of
// 2^13 ulp(x) no larger than 2 |x| in magnitude: at most 11 significant
// bits, exact in TF32.  |lo| <= ulp(c) / 2 <= 2^-10 |x| (2^-11 |x| unless the
// mantissa of x is within 2^-13 of 2), and the tensor core's truncation of lo
// errs by less than 2^-20 |x|.  Finite |x| below 2^114 (c must not overflow).
// Written with fma rather than as Veltkamp's c - (c - x): in a probe of the
// packed subtraction form the compiled code returned hi = x.
__device__ __forceinline__ void split_tf32_x2(f32x2 x, unsigned &h0, unsigned &l0, unsigned &h1, unsigned &l1) {
    const f32x2 c = fma2(x, pk2(8192.0f, 8192.0f), x);
    const f32x2 hi = fma2(x, pk2(-8192.0f, -8192.0f), c);
    const f32x2 lo = sub2(x, hi);
    float a, b;
    upk2(hi, a, b);
    h0 = __float_as_uint(a);
    h1 = __float_as_uint(b);
    upk2(lo, a, b);
    l0 = __float_as_uint(a);
    l1 = __float_as_uint(b);
}

// d += a b on the tensor core (mma.m16n8k8, TF32 operands, FP32 sums)
__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Horner evaluation of a degree-7 polynomial held in registers.
__device__ __forceinline__ float horner8(const float c[NCOEF], float v) {
    float s = c[NCOEF - 1];
#pragma unroll
    for (int i = NCOEF - 2; i >= 0; --i) s = fmaf(s, v, c[i]);
    return s;
}

// Direct evaluation of the normalised Kaiser--Bessel window at distance d
// (grid units), for the FP64 plans' tables.
__device__ __forceinline__ double kb_direct_d(double d, int m, double b, double inv_psi0) {
    double s2 = fma(-d, d, (double)(m * m));
    if (s2 <= 0.0) return s2 == 0.0 ? b / 3.141592653589793238 * inv_psi0 : 0.0;
    double s = sqrt(s2);
    return sinh(b * s) / (3.141592653589793238 * s) * inv_psi0;
}

// Grid position of a coordinate x in [-1/2, 1/2): t = (x + 1/2) n wrapped to
// [0, n).  Returns floor(t) and writes tau = t - floor(t).
__device__ __forceinline__ int grid_pos(float x, int n, float &tau) {
    float t = (x + 0.5f) * (float)n;
    float fl = floorf(t);
    tau = t - fl;
    int i = (int)fl;
    if (i >= n) i -= n;   // x rounded up to 1/2
    if (i < 0) i += n;
    return i;
}

__device__ __forceinline__ int grid_pos_d(double x, int n, double &tau) {
    double t = (x + 0.5) * (double)n;
    double fl = floor(t);
    tau = t - fl;
    int i = (int)fl;
    if (i >= n) i -= n;
    if (i < 0) i += n;
    return i;
}

__device__ __forceinline__ int wrap(int i, int n) {
    i = i < 0 ? i + n : i;
    return i >= n ? i - n : i;
}

// ------------------------------------------------------- async bulk copies --

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// ---- cp.async (Ampere-style asynchronous copies to shared memory) ----
// 16 bytes through L2 only (no L1 line is allocated)
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
// wait until at most N of this thread's most recent groups are pending
template <int N>
__device__ __forceinline__ void cp_async_wait_n() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// L2 prefetch of bytes (a multiple of 16) at a 16-byte aligned global address
__device__ __forceinline__ void prefetch_l2_bulk(const void *src, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// global -> shared bulk copy (16-byte aligned, size multiple of 16), completion
// counted on the mbarrier.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Bounded wait for the mbarrier phase with parity `parity`.  Gives up after
// `limit` polls, records `code` in *err and returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, int *err, int code,
                                          long long limit = (1LL << 22)) {
    uint32_t a = smem_addr(bar);
    for (long long it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    if (err) atomicCAS(err, 0, code);
    return false;
}

// ----------------------------------------------------------- shared FFT ---

// Division of x < 2^16 by a fixed d < 2^16 with one high multiplication:
// m = ceil(2^32 / d), and the error x (m d - 2^32) / 2^32 < x d / 2^32 < 1 / d
// never carries the quotient over an integer.
struct FastDiv {
    unsigned d, m;
    __device__ __forceinline__ explicit FastDiv(int d_) : d((unsigned)d_), m(0xffffffffu / (unsigned)d_ + 1u) {}
    __device__ __forceinline__ int div(int x) const { return d == 1 ? x : (int)__umulhi((unsigned)x, m); }
    __device__ __forceinline__ int div(int x, int &rem) const {
        const int q = div(x);
        rem = x - q * (int)d;
        return q;
    }
};

template <typename C, typename R>
struct CplxOps;

template <>
struct CplxOps<float2, float> {
    static __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
    static __device__ __forceinline__ void sincospi_(float x, float *s, float *c) { sincospif(x, s, c); }
};
template <>
struct CplxOps<double2, double> {
    static __device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
    static __device__ __forceinline__ void sincospi_(double x, double *s, double *c) { sincospi(x, s, c); }
};

template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
    C r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}

// Discrete Fourier transform of RADIX values in registers,
// v[q] <- sum_r v[r] exp(sign 2 pi i r q / RADIX), sign = +-1 in sg.
template <int RADIX, typename C, typename R>
__device__ __forceinline__ void dft_regs(C (&v)[RADIX], R sg) {
    using O = CplxOps<C, R>;
    auto add = [](C a, C b) { return O::mk(a.x + b.x, a.y + b.y); };
    auto sub = [](C a, C b) { return O::mk(a.x - b.x, a.y - b.y); };
    auto imul = [sg](C a) { return O::mk(-sg * a.y, sg * a.x); };   // sign i a
    if constexpr (RADIX == 2) {
        const C a = v[0];
        v[0] = add(a, v[1]);
        v[1] = sub(a, v[1]);
    } else if constexpr (RADIX == 3) {
        const R c = (R)-0.5, s = (R)0.86602540378443864676;   // cos, sin of 2 pi / 3
        const C t = add(v[1], v[2]), d = sub(v[1], v[2]);
        const C m = O::mk(fma(c, t.x, v[0].x), fma(c, t.y, v[0].y));
        const C n = imul(O::mk(s * d.x, s * d.y));
        v[0] = add(v[0], t);
        v[1] = add(m, n);
        v[2] = sub(m, n);
    } else if constexpr (RADIX == 4) {
        const C s0 = add(v[0], v[2]), d0 = sub(v[0], v[2]), s1 = add(v[1], v[3]), d1 = imul(sub(v[1], v[3]));
        v[0] = add(s0, s1);
        v[1] = add(d0, d1);
        v[2] = sub(s0, s1);
        v[3] = sub(d0, d1);
    } else if constexpr (RADIX == 5) {
        // cos and sin of 2 pi / 5 and 4 pi / 5
        const R c1 = (R)0.30901699437494742410, c2 = (R)-0.80901699437494742410;
        const R s1 = (R)0.95105651629515357212, s2 = (R)0.58778525229247312917;
        const C t1 = add(v[1], v[4]), t2 = add(v[2], v[3]), t3 = sub(v[1], v[4]), t4 = sub(v[2], v[3]);
        const C m1 = O::mk(fma(c1, t1.x, fma(c2, t2.x, v[0].x)), fma(c1, t1.y, fma(c2, t2.y, v[0].y)));
        const C m2 = O::mk(fma(c2, t1.x, fma(c1, t2.x, v[0].x)), fma(c2, t1.y, fma(c1, t2.y, v[0].y)));
        const C n1 = imul(O::mk(fma(s1, t3.x, s2 * t4.x), fma(s1, t3.y, s2 * t4.y)));
        const C n2 = imul(O::mk(fma(s2, t3.x, -s1 * t4.x), fma(s2, t3.y, -s1 * t4.y)));
        v[0] = add(v[0], add(t1, t2));
        v[1] = add(m1, n1);
        v[2] = add(m2, n2);
        v[3] = sub(m2, n2);
        v[4] = sub(m1, n1);
    } else {
        static_assert(RADIX == 8, "radices 2, 3, 4, 5, 8");
        const R h = (R)0.70710678118654752440;   // exp(sign i pi / 4) = h (1 + sign i)
        C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft_regs<4, C, R>(e, sg);
        dft_regs<4, C, R>(o, sg);
        const C o1 = imul(o[1]), o3 = imul(o[3]);
        const C w1 = O::mk(h * (o[1].x + o1.x), h * (o[1].y + o1.y));
        const C w2 = imul(o[2]);
        const C w3 = O::mk(h * (o3.x - o[3].x), h * (o3.y - o[3].y));
        v[0] = add(e[0], o[0]);
        v[4] = sub(e[0], o[0]);
        v[1] = add(e[1], w1);
        v[5] = sub(e[1], w1);
        v[2] = add(e[2], w2);
        v[6] = sub(e[2], w2);
        v[3] = add(e[3], w3);
        v[7] = sub(e[3], w3);
    }
}

// Entries of the twiddle table exp(sign 2 pi i k / n), k < n, kept in shared
// memory behind the two FFT arrays; longer axes evaluate each factor.
template <typename C>
__host__ __device__ constexpr int fft_table_max() {
    return 16384 / (int)sizeof(C);
}
// shared memory of a block that transforms arrays of at most fft_elems values
// with axes of at most max_n; the adjoint also stages a stored grid of at most
// stage_elems values behind the first array
template <typename C>
inline size_t fft_smem_bytes(int fft_elems, int max_n, int stage_elems = 0) {
    const int tw = max_n < fft_table_max<C>() ? max_n : fft_table_max<C>();
    return ((size_t)fft_elems + (fft_elems + tw > stage_elems ? fft_elems + tw : stage_elems)) * sizeof(C);
}
constexpr int FFT_THREADS = 512;
constexpr int FFT_MAX_SMEM = 220 * 1024;   // two 100 KB arrays, the table, and room for static shared memory

// One Stockham stage over every line of one axis: element i of the line at
// base = (outer, inner position) lies at base + i * inner.  Consecutive
// threads take neighbouring lines of a strided axis (contiguous addresses) and
// neighbouring elements of the last axis.
template <int RADIX, typename C, typename R>
__device__ __forceinline__ void fft_stage(const C *src, C *dst, int fe, int n, int inner, int Ns, R sg, const C *tw) {
    const int nb = n / RADIX, step = nb / Ns;
    const FastDiv by_inner(inner), by_nb(nb), by_Ns(Ns);
    for (int w = threadIdx.x; w < fe / RADIX; w += blockDim.x) {
        int li, j, jm;
        const int rest = by_inner.div(w, li);
        const int lo = by_nb.div(rest, j);
        by_Ns.div(j, jm);
        const int base = lo * inner * n + li;
        const C *in = src + base + j * inner;
        C v[RADIX];
#pragma unroll
        for (int r = 0; r < RADIX; ++r) v[r] = in[r * nb * inner];
        if (jm) {
            const int k = jm * step;   // r k < n
#pragma unroll
            for (int r = 1; r < RADIX; ++r) {
                C t;
                if (tw) {
                    t = tw[r * k];
                } else {
                    CplxOps<C, R>::sincospi_(sg * (R)(2 * r * k) / (R)n, &t.y, &t.x);
                }
                v[r] = cmul(v[r], t);
            }
        }
        dft_regs<RADIX, C, R>(v, sg);
        C *out = dst + base + ((j - jm) * RADIX + jm) * inner;
#pragma unroll
        for (int r = 0; r < RADIX; ++r) out[r * Ns * inner] = v[r];
    }
}

// Unnormalised FFT with sign `sign` along every axis of an n^s array held in
// shared memory (a; b is scratch of the same size, followed by the twiddle
// table), s = 1..3, radices 8, 4, 2, 3, 5.  All threads of the block call it
// after filling a (it synchronises first); returns the buffer that holds the
// result.  What bounds it is the latency of a block's few stages: the former
// stages, with per-butterfly sincospi, run-time radix loops over arrays in
// local memory and hardware divisions, took 52 us for the 211 terms of the
// d = 20 workload (n = 64) and 147 us for 120 three-dimensional terms (n = 20).
template <typename C, typename R>
__device__ C *grid_fft(C *a, C *b, int n, int s, int sign) {
    int fe = n;
    for (int j = 1; j < s; ++j) fe *= n;
    C *tw = nullptr;
    if (n <= fft_table_max<C>()) {
        tw = b + fe;
        for (int k = threadIdx.x; k < n; k += blockDim.x)
            CplxOps<C, R>::sincospi_((R)(2 * sign * k) / (R)n, &tw[k].y, &tw[k].x);
    }
    __syncthreads();
    const R sg = (R)sign;
    C *src = a, *dst = b;
    int inner = 1;
    for (int ax = 0; ax < s; ++ax) {
        int left = n, Ns = 1;
        while (left > 1) {
            const int radix = left % 8 == 0 ? 8 : left % 4 == 0 ? 4 : left % 2 == 0 ? 2 : left % 3 == 0 ? 3 : 5;
            switch (radix) {
                case 8: fft_stage<8, C, R>(src, dst, fe, n, inner, Ns, sg, tw); break;
                case 4: fft_stage<4, C, R>(src, dst, fe, n, inner, Ns, sg, tw); break;
                case 2: fft_stage<2, C, R>(src, dst, fe, n, inner, Ns, sg, tw); break;
                case 3: fft_stage<3, C, R>(src, dst, fe, n, inner, Ns, sg, tw); break;
                default: fft_stage<5, C, R>(src, dst, fe, n, inner, Ns, sg, tw); break;
            }
            __syncthreads();
            C *t = src;
            src = dst;
            dst = t;
            Ns *= radix;
            left /= radix;
        }
        inner *= n;
    }
    return src;
}

// Block-wide FP64 sum in a fixed order, valid in thread 0 (sh: 32 doubles;
// blockDim a multiple of 32).
__device__ __forceinline__ double block_sum_fixed(double v, double *sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;
}

// Position of coefficient q of an exponential block on the term's FFT array
// (k mod n per axis, last axis fastest) and the product of its deconvolution
// factors (column table on the last axis, row table on the others).
template <typename R>
__device__ __forceinline__ int exp_position(int q, int s, int N, int n, const FastDiv &by_Nm, const R *deconv,
                                            int dc_off, int dr_off, R &D) {
    int pos = 0, mul = 1;
    D = (R)1;
    for (int t = s - 1; t >= 0; --t) {
        int it;
        q = by_Nm.div(q, it);
        const int k = it < N / 2 ? it - N / 2 : it - N / 2 + 1;
        pos += (k < 0 ? k + n : k) * mul;
        mul *= n;
        D *= deconv[(t == s - 1 ? dc_off : dr_off) + it];
    }
    return pos;
}

// Periodic grid of a term into a (n^s values) from its stored grid with halos:
// entries of the stored grid that repeat a periodic one are added.  `load2`
// returns the stored values 2 i, 2 i + 1 (rows are even in length); they pass
// through `stage` (halo_stage_elems), so that global memory is read once, 16
// bytes or more at a time.  All threads of the block call it.
__host__ __device__ inline int halo_cols(const Term &T) { return (T.n + 2 * T.hc + 2) & ~1; }   // even row length
__host__ __device__ inline int halo_stage_elems(const Term &T) { return T.order > 2 ? 0 : T.erows * halo_cols(T); }

template <typename C, typename Load2>
__device__ __forceinline__ void fold_halo(const Term &T, C *a, C *stage, int fe, Load2 load2) {
    const int n = T.n, cols = T.order > 2 ? n : halo_cols(T), rows = T.erows, half = cols >> 1;
    C *dst = T.order > 2 ? a : stage;
    {
        const FastDiv by_half(half);
        for (int i = threadIdx.x; i < rows * half; i += blockDim.x) {
            int c2;
            const int r = by_half.div(i, c2);
            C v0, v1;
            load2((r * T.stride >> 1) + c2, v0, v1);
            dst[r * cols + 2 * c2] = v0;
            dst[r * cols + 2 * c2 + 1] = v1;
        }
    }
    if (T.order > 2) return;
    __syncthreads();
    const int ecw = n + 2 * T.hc + 1;
    const FastDiv by_n(n);
    for (int e = threadIdx.x; e < fe; e += blockDim.x) {
        int qc;
        const int qr = by_n.div(e, qc);
        C v;
        v.x = v.y = 0;
        for (int er = T.order == 2 ? (qr + T.hr >= n ? qr + T.hr - n : qr + T.hr) : 0; er < rows; er += n)
            for (int ec = qc + T.hc >= n ? qc + T.hc - n : qc + T.hc; ec < ecw; ec += n) {
                const C u = stage[er * cols + ec];
                v.x += u.x;
                v.y += u.y;
            }
        a[e] = v;
    }
}

}  // namespace agft
