// Direct summation of plans whose terms all have small bandwidths (the paper's own
// experiments: N = 26 / 6 / 4, and 82 / 10 for the cosine system).
//
// f_j = sum_u sum_k fhat_k exp(2 pi i <k, x_j>) term by term (Definition "grouped
// Fourier transform" and the stacked adjoint, Sec. 3; cosine functions of Sec. 5
// likewise), axis by axis: a third-order term of bandwidth 4 has 27 coefficients
// where the window has 512 points, so the sum itself costs less than the NFFT's
// gather or spread, has no window error, and needs neither grids nor sorted nodes.
// One kernel per direction.  What bounds them: FP32 multiply-adds (two per
// coefficient on the innermost axis, where k and -k share their products) at the
// solvers' sizes, launch latency at the smallest.
//
// Frequencies of the innermost axis are handled in pairs +-k, k < K = N / 2, and
// -K alone; cosine axes have the functions sqrt(2) cos(2 pi k x), k = 1 .. N / 2 - 1,
// at the plan's halved nodes.  z_t = exp(2 pi i x_t) is kept per node and coordinate,
// and its powers come from multiplications: at most 4 in a row (cosine axes 8), on
// order-1 axes 7 from a power that is evaluated from the node itself.
#include <algorithm>
#include <atomic>
#include <cstring>

#include "device.cuh"
#include "internal.cuh"

namespace agft {

constexpr int DT_THREADS = 256, DA_THREADS = 128;
constexpr int DIRECT_MAX_COEF = 80;       // float4 of staged coefficients per warp (at most 25 rows of 3)
constexpr int ORD1_GROUP = 8;             // frequencies per order-1 unit and item
constexpr float SQRT2 = 1.41421356237309504880f;

// exp(2 pi i k x) from the fraction of k x, which fma makes exact
__device__ __forceinline__ float2 unit_power(float x, int k) {
    const float fk = (float)k, p = fk * x, e = fmaf(fk, x, -p);
    float2 w;
    sincospif(2.f * ((p - rintf(p)) + e), &w.y, &w.x);
    return w;
}

// z = exp(2 pi i x) for every coordinate and node
__global__ void k_unit_table(const float *__restrict__ x, float2 *z, long long total) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
        z[i] = unit_power(x[i], 1);
}

// frequencies of an axis: exponential K = N / 2 (pairs +-k, the last one alone),
// cosine the N / 2 - 1 functions (N doubled)
static int axis_count(const Term &T) { return T.basis == ANOVA_BASIS_COS ? T.N / 2 - 1 : T.N / 2; }
template <bool COS>
__host__ __device__ constexpr int axis_coefs(int K) {
    return COS ? K : 2 * K - 1;
}
// rows of the outer axes that one adjoint item takes: all, of the larger
// third-order terms those of one index of the first axis
template <bool COS>
__host__ __device__ constexpr int group_rows(int order, int K) {
    const int n = axis_coefs<COS>(K);
    return order == 1 ? 1 : (order == 3 && !COS && K <= 2 ? n * n : n);
}
template <bool COS>
__host__ __device__ constexpr int adjoint_groups(int order, int K) {
    const int n = axis_coefs<COS>(K);
    return order == 1 ? (K + ORD1_GROUP - 1) / ORD1_GROUP
                      : (order == 3 ? n * n / group_rows<COS>(order, K) : 1);
}
static int groups_of(const Term &T) {
    return T.basis == ANOVA_BASIS_COS ? adjoint_groups<true>(T.order, axis_count(T))
                                      : adjoint_groups<false>(T.order, axis_count(T));
}
// second-order terms with more than 64 partial sums per adjoint item: a kernel of their
// own, with more registers and fewer blocks per SM
static bool is_big(const Term &T) {
    const int K = axis_count(T);
    return T.order > 1 && (T.basis == ANOVA_BASIS_COS ? K > 5 : K > 3);
}

// ------------------------------------------------------------ forward ----

// the value a node's table keeps per power: exp(2 pi i k x), cosine sqrt(2) cos(2 pi k x)
template <bool COS>
struct Power {
    using T = float2;
    static __device__ __forceinline__ T of(float2 w) { return w; }
};
template <>
struct Power<true> {
    using T = float;
    static __device__ __forceinline__ T of(float2 w) { return SQRT2 * w.x; }
};

// sum over the innermost axis of row `c` (float4 per pair: coefficient sums and
// differences; cosine: float2 per function) at NPL nodes
template <int K, int NPL, bool COS>
__device__ __forceinline__ void row_inner(const float4 *c, const typename Power<COS>::T (&e)[K][NPL], float2 (&r)[NPL]) {
#pragma unroll
    for (int u = 0; u < NPL; ++u) r[u] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if constexpr (COS) {
            const float2 v = ((const float2 *)c)[k];
#pragma unroll
            for (int u = 0; u < NPL; ++u) {
                r[u].x = fmaf(v.x, e[k][u], r[u].x);
                r[u].y = fmaf(v.y, e[k][u], r[u].y);
            }
        } else {
            const float4 v = c[k];   // s = c_k + c_-k, d = c_k - c_-k: (s.x, s.y, d.x, d.y)
#pragma unroll
            for (int u = 0; u < NPL; ++u) {
                r[u].x = fmaf(v.x, e[k][u].x, fmaf(-v.w, e[k][u].y, r[u].x));
                r[u].y = fmaf(v.y, e[k][u].x, fmaf(v.z, e[k][u].y, r[u].y));
            }
        }
    }
}

// s += w r, w a row function's value (cosine: real)
__device__ __forceinline__ void add_scaled(float2 &s, float w, float2 r) {
    s.x = fmaf(w, r.x, s.x);
    s.y = fmaf(w, r.y, s.y);
}
__device__ __forceinline__ void add_scaled(float2 &s, float2 w, float2 r) {
    s.x = fmaf(w.x, r.x, fmaf(-w.y, r.y, s.x));
    s.y = fmaf(w.x, r.y, fmaf(w.y, r.x, s.y));
}

// a term of order 2 or 3 at NPL nodes of this lane; tab: powers [coordinate][k][node]
template <int K, int NPL, bool COS>
__device__ __forceinline__ void term_rows(const DirectTerm &T, const float4 *st, const typename Power<COS>::T *tab, int KT,
                                          float2 (&acc)[NPL]) {
    constexpr int NB = 32 * NPL, W = COS ? (K + 1) / 2 : K;   // float4 per row
    using E = typename Power<COS>::T;
    constexpr int n = COS ? K : 2 * K - 1;
    const int lane = threadIdx.x & 31;
    E e[K][NPL];
    const E *tc = tab + T.col * KT * NB + lane;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int u = 0; u < NPL; ++u) e[k][u] = tc[k * NB + 32 * u];
    const E *tr = tab + (T.order == 3 ? T.row1 : T.row0) * KT * NB + lane;
    E er[K][NPL];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int u = 0; u < NPL; ++u) er[k][u] = tr[k * NB + 32 * u];
    // value at coefficient position it of an axis: k = -K .. -1, 1 .. K - 1 (cosine 1 .. K)
    auto power = [](const E (&w)[K][NPL], int it, int u) {
        if constexpr (COS) {
            return w[it][u];
        } else {
            float2 v = w[it < K ? K - 1 - it : it - K][u];
            if (it < K) v.y = -v.y;
            return v;
        }
    };
    // the rows of one block of the first axis (order 2: the term)
    auto block = [&](float2 (&s)[NPL]) {
#pragma unroll
        for (int b = 0; b < n; ++b) {
            float2 r[NPL];
            row_inner<K, NPL, COS>(st + b * W, e, r);
#pragma unroll
            for (int u = 0; u < NPL; ++u) add_scaled(s[u], power(er, b, u), r[u]);
        }
        st += n * W;
    };
    if (T.order == 2) {
        block(acc);
        return;
    }
    if constexpr (K <= (COS ? 4 : 3)) {
        const E *ta = tab + T.row0 * KT * NB + lane;
        for (int a = 0; a < n; ++a) {
            float2 s[NPL];
#pragma unroll
            for (int u = 0; u < NPL; ++u) s[u] = make_float2(0.f, 0.f);
            block(s);
            const int k = COS ? a : (a < K ? K - 1 - a : a - K);   // |k| - 1
#pragma unroll
            for (int u = 0; u < NPL; ++u) {
                E w = ta[k * NB + 32 * u];
                if constexpr (!COS) w.y = a < K ? -w.y : w.y;
                add_scaled(acc[u], w, s[u]);
            }
        }
    }
}

// Units that a warp adds in one FP32 chain (up to 9 rows each) before their sum goes to
// its total, kept in shared memory (in registers it spilled): the error of a chain grows
// with the root of its length, and one over the 58 units of a warp at d = 30, N = 16/8
// left 2.8e-7 at M = 3e4 where the NFFT has 2.1e-7.  Plans whose warps have no more units
// than that run kernels without totals (CHAINS false): d = 3, N = 16/8/4, M = 2e5 24.5 ->
// 23.6 us, d = 1, N = 16, M = 1e7 599 -> 533.
constexpr int DT_CHAIN = 8;

// A CTA takes 32 NPL nodes and every gridDim.y-th set of work units (active term,
// frequency group of order 1), its warps one unit each in turn; the warps' sums are
// added in order, and so are the CTAs' of a node block by the last one to finish
// (bitwise reproducible).
template <int NPL, bool COS, bool CHAINS>
__global__ void __launch_bounds__(DT_THREADS, NPL == 4 ? 2 : 3)
direct_trafo(DevPlan P, const float2 *__restrict__ fhat, float2 *__restrict__ f, int KT,
             const DirectTerm *__restrict__ units, int n_units, float2 *fpart, int *count) {
    using E = typename Power<COS>::T;
    __shared__ int s_last;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NB = 32 * NPL, NW = DT_THREADS / 32;
    if (P.skip && *P.skip) return;
    float2 *red = (float2 *)smem;                                          // [NW][NB]
    float4 *stage = (float4 *)(red + NW * NB);                             // [NW][DIRECT_MAX_COEF]
    E *tab = (E *)(stage + NW * DIRECT_MAX_COEF);                          // [d][KT][NB]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long M = P.M, j0 = (long long)blockIdx.x * NB;
    for (int i = tid; i < P.d * NB && KT > 0; i += DT_THREADS) {
        const int t = i / NB, u = i % NB;
        const float2 z = __ldg(P.z + (long long)t * M + min(j0 + u, M - 1));
        float2 w = z;
        for (int k = 0; k < KT; ++k) {
            tab[(t * KT + k) * NB + u] = Power<COS>::of(w);
            w = cmul(w, z);
        }
    }
    __syncthreads();
    float4 *st = stage + warp * DIRECT_MAX_COEF;
    const int first = blockIdx.y * NW + warp, step = NW * gridDim.y;
    float2 acc[NPL];
    float2 *sum = red + warp * NB + lane;   // this lane's sums of the chains before
#pragma unroll
    for (int u = 0; u < NPL; ++u) acc[u] = make_float2(0.f, 0.f);
    int chain_end = first + DT_CHAIN * step;
    auto end_chain = [&]() {
        const bool later = CHAINS && chain_end != first + DT_CHAIN * step;   // not the first chain
#pragma unroll
        for (int u = 0; u < NPL; ++u) {
            sum[32 * u] = later ? make_float2(sum[32 * u].x + acc[u].x, sum[32 * u].y + acc[u].y) : acc[u];
            acc[u] = make_float2(0.f, 0.f);
        }
    };
    // A unit's coefficients are loaded while the unit before it is summed, and its
    // record before that: a lane holds up to three pairs (c_k, c_-k) of a term of
    // order >= 2 (cosine: three coefficients), an order-1 group all its coefficients.
    constexpr int PF = 3;
    float2 cp[PF], cm[PF];
    auto prefetch = [&](const DirectTerm &T) {
        const float2 *c = fhat + T.coef_off;
        const int n = axis_coefs<COS>(T.K), rows = T.order == 3 ? n * n : n, len = T.order == 1 ? 0 : rows * T.K;
        const FastDiv by_K(T.K);
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int q = lane + 32 * i;
            cp[i] = cm[i] = make_float2(0.f, 0.f);
            if (q >= len) continue;
            int k;
            const int r = by_K.div(q, k);   // pair k + 1 of row r
            if (COS) {
                cp[i] = __ldg(c + q);
            } else {
                cm[i] = __ldg(c + r * n + T.K - 1 - k);
                if (k + 1 < T.K) cp[i] = __ldg(c + r * n + T.K + k);
            }
        }
    };
    DirectTerm next, after;
    if (first < n_units) next = units[first];
    if (first + step < n_units) after = units[first + step];
    if (first < n_units) prefetch(next);
    for (int s = first; s < n_units; s += step) {
        if (CHAINS && s == chain_end) {
            end_chain();
            chain_end += DT_CHAIN * step;
        }
        const DirectTerm T = next;
        if (T.order == 1) {
            next = after;
            if (s + step < n_units) prefetch(next);
            if (s + 2 * step < n_units) after = units[s + 2 * step];
            const float2 *c = fhat + T.coef_off;
            const int K = T.K, k0 = 1 + ORD1_GROUP * T.group;
            float2 vp[ORD1_GROUP], vm[ORD1_GROUP];   // the group's coefficients: all loads in flight
#pragma unroll
            for (int i = 0; i < ORD1_GROUP; ++i) {
                const int k = k0 + i;
                vp[i] = vm[i] = make_float2(0.f, 0.f);
                if (COS) {
                    if (k <= K) vp[i] = __ldg(c + k - 1);
                } else {
                    if (k <= K) vm[i] = __ldg(c + K - k);
                    if (k < K) vp[i] = __ldg(c + K - 1 + k);
                }
            }
            float2 z[NPL], w[NPL];
#pragma unroll
            for (int u = 0; u < NPL; ++u) {
                const long long j = min(j0 + lane + 32 * u, M - 1);
                w[u] = unit_power(__ldg(P.x + (long long)T.col * M + j), k0);
                z[u] = __ldg(P.z + (long long)T.col * M + j);
            }
#pragma unroll
            for (int i = 0; i < ORD1_GROUP; ++i) {
                const float sx = vp[i].x + vm[i].x, sy = vp[i].y + vm[i].y, dx = vp[i].x - vm[i].x, dy = vp[i].y - vm[i].y;
#pragma unroll
                for (int u = 0; u < NPL; ++u) {
                    if (COS) {
                        add_scaled(acc[u], SQRT2 * w[u].x, vp[i]);
                    } else {
                        acc[u].x = fmaf(sx, w[u].x, fmaf(-dy, w[u].y, acc[u].x));
                        acc[u].y = fmaf(sy, w[u].x, fmaf(dx, w[u].y, acc[u].y));
                    }
                    w[u] = cmul(w[u], z[u]);
                }
            }
            continue;
        }
        // the term's coefficients by rows of the innermost axis
        const int n = axis_coefs<COS>(T.K), len = (T.order == 3 ? n * n : n) * T.K;
        __syncwarp();   // the previous term's rows are read
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int q = lane + 32 * i;
            if (q >= len) break;
            if (COS) {
                const int r = q / T.K, k = q - r * T.K;
                ((float2 *)st)[r * (2 * ((T.K + 1) / 2)) + k] = cp[i];
            } else {
                st[q] = make_float4(cp[i].x + cm[i].x, cp[i].y + cm[i].y, cp[i].x - cm[i].x, cp[i].y - cm[i].y);
            }
        }
        __syncwarp();
        next = after;
        if (s + step < n_units) prefetch(next);
        if (s + 2 * step < n_units) after = units[s + 2 * step];
        switch (T.K) {
            case 1: term_rows<1, NPL, COS>(T, st, tab, KT, acc); break;
            case 2: term_rows<2, NPL, COS>(T, st, tab, KT, acc); break;
            case 3: term_rows<3, NPL, COS>(T, st, tab, KT, acc); break;
            case 4: term_rows<4, NPL, COS>(T, st, tab, KT, acc); break;
            case 5: term_rows<5, NPL, COS>(T, st, tab, KT, acc); break;
            default:
                if constexpr (COS) switch (T.K) {
                    case 6: term_rows<6, NPL, COS>(T, st, tab, KT, acc); break;
                    case 7: term_rows<7, NPL, COS>(T, st, tab, KT, acc); break;
                    case 8: term_rows<8, NPL, COS>(T, st, tab, KT, acc); break;
                    default: term_rows<9, NPL, COS>(T, st, tab, KT, acc); break;
                }
        }
    }
    end_chain();
    __syncthreads();
    const int S = gridDim.y;
    auto write = [&](int u, float2 v) {
        for (int e = 0; e < P.n_empty; ++e) {
            const float2 c = fhat[P.empty_off[e]];
            v.x += c.x;
            v.y += c.y;
        }
        f[j0 + u] = v;
    };
    for (int u = tid; u < NB; u += DT_THREADS) {
        if (j0 + u >= M) break;
        float2 v = make_float2(0.f, 0.f);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            v.x += red[w * NB + u].x;
            v.y += red[w * NB + u].y;
        }
        if (S == 1)
            write(u, v);
        else
            fpart[blockIdx.y * M + j0 + u] = v;
    }
    if (S == 1) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(count + blockIdx.x, 1) == S - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) count[blockIdx.x] = 0;
    for (int u = tid; u < NB; u += DT_THREADS) {
        if (j0 + u >= M) break;
        float2 v = make_float2(0.f, 0.f);
        for (int s = 0; s < S; ++s) {
            const float2 w = __ldcg(fpart + s * M + j0 + u);
            v.x += w.x;
            v.y += w.y;
        }
        write(u, v);
    }
}

// ------------------------------------------------------------ adjoint ----

// A thread adds at most DA_CHAIN nodes in FP32; the block's sums over such runs are added
// in FP64.  An FP32 chain's error grows with the root of its length: at d = 6, N = 16/8,
// M = 1e6 one chain of 601 nodes left 4.8e-7, where the NFFT has 2.8e-7.  One exchange of
// the block's sums per run is 2 % of its products at most.  Items of more than a run have
// kernels of their own (RUNS): the loop over runs cost 13 registers and 1.5 % at the
// solvers' sizes, which have one.
constexpr int DA_CHAIN = 128, DA_RUN = DA_CHAIN * DA_THREADS;

// Block sums of R values per thread (R padded to a multiple of 32 with zeros in v):
// each warp halves the values it keeps per exchange.  The sums of all calls from the
// `first` to the `last` go to out[0, R); tot: [R], the sums so far.
template <int R>
__device__ __forceinline__ void block_sums(float (&v)[R], float *out, float *sh, double *tot, bool first, bool last) {
    static_assert(R % 32 == 0, "padded");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int b = 0; b < R; b += 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < o; ++i) {
                const float keep = up ? v[b + i + o] : v[b + i], send = up ? v[b + i] : v[b + i + o];
                v[b + i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        sh[warp * R + b + lane] = v[b];   // value b + lane
    }
    __syncthreads();
    for (int i = threadIdx.x; i < R; i += blockDim.x) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < DA_THREADS / 32; ++w) s += sh[w * R + i];
        if (first && last) {
            out[i] = s;
        } else {
            const double t = first ? (double)s : tot[i] + s;   // the thread's own value
            if (last)
                out[i] = (float)t;
            else
                tot[i] = t;
        }
    }
    if (!last) __syncthreads();   // sh is read before the next run's sums
}

// ROWS rows of a term of order ORD over nodes [a, b): all of them, or those of index
// `ia` of a third-order term's first axis.  Per row and innermost
// pair the sums of u.x c, u.y s, u.y c, u.x s (u = y times the conjugate outer powers,
// (c, s) the innermost power); cosine: u.x c, u.y c per function.
template <int K, bool COS, int ORD, bool RUNS>
__device__ __forceinline__ void adjoint_rows(const DevPlan &P, const DirectTerm &T, const float2 *__restrict__ y,
                                             long long a, long long b, float *out, float *sh, double *tot) {
    constexpr int ROWS = group_rows<COS>(ORD, K), PER = COS ? 2 : 4, R = (ROWS * K * PER + 31) / 32 * 32;
    constexpr int N = axis_coefs<COS>(K);
    constexpr bool ALL = ORD == 3 && ROWS == N * N;
    static_assert(R <= DA_MAX_ACC, "partial sums of an item");
    const int ia = T.group;
    float acc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = 0.f;
    const long long M = P.M;
    const float2 *zc = P.z + (long long)T.col * M, *zr = P.z + (long long)(ORD == 3 ? T.row1 : T.row0) * M,
                 *za = P.z + (long long)T.row0 * M;
    // exp(-2 pi i k x) by coefficient position k = -K .. -1, 1 .. K - 1 (one past the
    // end: K, unused); cosine: the functions' values in x
    auto conj_powers = [](float2 z, float2 (&pw)[2 * K]) {
        float2 w = z;
#pragma unroll
        for (int k = 1; k <= K; ++k) {
            if (COS) {
                pw[k - 1] = make_float2(SQRT2 * w.x, 0.f);
            } else {
                pw[K - k] = w;
                pw[K - 1 + k] = make_float2(w.x, -w.y);
            }
            w = cmul(w, z);
        }
    };
    // the next node's values are loaded while this one's are used
    long long j = a + threadIdx.x;
    float2 ny, nz, nr, na = make_float2(1.f, 0.f);
    auto load = [&](long long i) {
        i = min(i, M - 1);
        ny = __ldg(y + i);
        nz = __ldg(zc + i);
        nr = __ldg(zr + i);
        if (ORD == 3) na = __ldg(za + i);
    };
    load(j);
    for (long long r1 = RUNS ? min(b, a + DA_RUN) : b;; r1 = min(b, r1 + DA_RUN)) {
        for (; j < r1; j += DA_THREADS) {
            const float2 yv = ny, z = nz, zrow = nr, zfirst = na;
            load(j + DA_THREADS);
            float2 e[K], pw[2 * K], pa[2 * K], ya = yv;
            e[0] = z;
#pragma unroll
            for (int k = 1; k < K; ++k) e[k] = cmul(e[k - 1], z);
            conj_powers(zrow, pw);
            if (ORD == 3) {
                conj_powers(zfirst, pa);
                if (!ALL) {   // the one index of the first axis
                    float2 w = pa[0];
#pragma unroll
                    for (int k = 1; k < N; ++k)
                        if (k == ia) w = pa[k];
                    ya = COS ? make_float2(yv.x * w.x, yv.y * w.x) : cmul(yv, w);
                }
            }
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const float2 w = pw[ALL ? r % N : r];
                if (ALL && r % N == 0) ya = COS ? make_float2(yv.x * pa[r / N].x, yv.y * pa[r / N].x) : cmul(yv, pa[r / N]);
                const float2 u = COS ? make_float2(ya.x * w.x, ya.y * w.x) : cmul(ya, w);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    float *v = acc + (r * K + k) * PER;
                    if (COS) {
                        v[0] = fmaf(u.x, e[k].x, v[0]);
                        v[1] = fmaf(u.y, e[k].x, v[1]);
                    } else {
                        v[0] = fmaf(u.x, e[k].x, v[0]);
                        v[1] = fmaf(u.y, e[k].y, v[1]);
                        v[2] = fmaf(u.y, e[k].x, v[2]);
                        v[3] = fmaf(u.x, e[k].y, v[3]);
                    }
                }
            }
        }
        block_sums<R>(acc, out, sh, tot, !RUNS || r1 - DA_RUN <= a, !RUNS || r1 == b);
        if (!RUNS || r1 == b) break;
#pragma unroll
        for (int i = 0; i < R; ++i) acc[i] = 0.f;
    }
}

// frequencies 1 + ORD1_GROUP group .. of an order-1 term
template <bool COS, bool RUNS>
__device__ __forceinline__ void adjoint_order1(const DevPlan &P, const DirectTerm &T, const float2 *__restrict__ y,
                                               long long a, long long b, float *out, float *sh, double *tot) {
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
    const float *x = P.x + (long long)T.col * P.M;
    const float2 *zc = P.z + (long long)T.col * P.M;
    long long j = a + threadIdx.x;
    for (long long r1 = RUNS ? min(b, a + DA_RUN) : b;; r1 = min(b, r1 + DA_RUN)) {
        for (; j < r1; j += DA_THREADS) {
            const float2 u = __ldg(y + j), z = __ldg(zc + j);
            float2 w = unit_power(__ldg(x + j), 1 + ORD1_GROUP * T.group);
#pragma unroll
            for (int k = 0; k < ORD1_GROUP; ++k) {
                float *v = acc + 4 * k;
                v[0] = fmaf(u.x, w.x, v[0]);
                v[2] = fmaf(u.y, w.x, v[2]);
                if (!COS) {
                    v[1] = fmaf(u.y, w.y, v[1]);
                    v[3] = fmaf(u.x, w.y, v[3]);
                }
                w = cmul(w, z);
            }
        }
        block_sums<32>(acc, out, sh, tot, !RUNS || r1 - DA_RUN <= a, !RUNS || r1 == b);
        if (!RUNS || r1 == b) break;
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = 0.f;
    }
}

// Work item (active term or -1 for the empty set, row group, node chunk, chunks; its
// term): partial sums into part[item]; the last block of a term to finish adds them
// over the chunks in order and writes the coefficients.  BIG: plans that have
// a second-order term with more than 64 sums per item.  RUNS: items of more than DA_RUN nodes.
template <bool COS, bool BIG, bool RUNS>
__global__ void __launch_bounds__(DA_THREADS, BIG ? DIRECT_RESIDENT_BIG : DIRECT_RESIDENT)
direct_adjoint(DevPlan P, const DirectItem *__restrict__ items, const float2 *__restrict__ y, float2 *__restrict__ fhat,
               float *part, int *count) {
    __shared__ float sh[DA_MAX_ACC * (DA_THREADS / 32)];
    __shared__ double shd[32], tot[RUNS ? DA_MAX_ACC : 1];
    __shared__ int s_last;
    if (P.skip && *P.skip) return;
    const DirectItem itm = items[blockIdx.x];
    const DirectTerm &T = itm.term;
    const int C = itm.chunks;
    const long long M = P.M, a = M * itm.chunk / C, b = M * (itm.chunk + 1) / C;
    float *out = part + (long long)blockIdx.x * DA_MAX_ACC;
    int blocks = C, *cnt = count;
    if (itm.act < 0) {
        double sx = 0.0, sy = 0.0;
        for (long long j = a + threadIdx.x; j < b; j += DA_THREADS) {
            const float2 v = __ldg(y + j);
            sx += v.x;
            sy += v.y;
        }
        sx = block_sum_fixed(sx, shd);
        sy = block_sum_fixed(sy, shd);
        if (threadIdx.x == 0) *(double2 *)out = make_double2(sx, sy);
    } else {
        blocks *= adjoint_groups<COS>(T.order, T.K);
        cnt = count + 1 + itm.act;
        if (T.order == 1) {
            adjoint_order1<COS, RUNS>(P, T, y, a, b, out, sh, tot);
        } else if constexpr (COS) {
            if (T.order == 3) switch (T.K) {
                case 1: adjoint_rows<1, true, 3, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 2: adjoint_rows<2, true, 3, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 3: adjoint_rows<3, true, 3, RUNS>(P, T, y, a, b, out, sh, tot); break;
                default: adjoint_rows<4, true, 3, RUNS>(P, T, y, a, b, out, sh, tot); break;
            } else if (!BIG || T.K <= 5) switch (T.K) {
                case 1: adjoint_rows<1, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 2: adjoint_rows<2, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 3: adjoint_rows<3, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 4: adjoint_rows<4, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                default: adjoint_rows<5, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
            } else if constexpr (BIG) switch (T.K) {
                case 6: adjoint_rows<6, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 7: adjoint_rows<7, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 8: adjoint_rows<8, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                default: adjoint_rows<9, true, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
            }
        } else {
            if (T.order == 3) switch (T.K) {
                case 1: adjoint_rows<1, false, 3, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 2: adjoint_rows<2, false, 3, RUNS>(P, T, y, a, b, out, sh, tot); break;
                default: adjoint_rows<3, false, 3, RUNS>(P, T, y, a, b, out, sh, tot); break;
            } else if (!BIG || T.K <= 3) switch (T.K) {
                case 1: adjoint_rows<1, false, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                case 2: adjoint_rows<2, false, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
                default: adjoint_rows<3, false, 2, RUNS>(P, T, y, a, b, out, sh, tot); break;
            } else if constexpr (BIG) {
                if (T.K == 4) adjoint_rows<4, false, 2, RUNS>(P, T, y, a, b, out, sh, tot);
                else adjoint_rows<5, false, 2, RUNS>(P, T, y, a, b, out, sh, tot);
            }
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(cnt, 1) == blocks - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) *cnt = 0;
    const float *first = part + (long long)((int)blockIdx.x - (itm.act < 0 ? itm.chunk : T.group * C + itm.chunk)) * DA_MAX_ACC;
    if (itm.act < 0) {
        if (threadIdx.x == 0) {
            double sx = 0.0, sy = 0.0;
            for (int c = 0; c < C; ++c) {
                const double2 v = __ldcg((const double2 *)(first + (long long)c * DA_MAX_ACC));
                sx += v.x;
                sy += v.y;
            }
            for (int e = 0; e < P.n_empty; ++e) fhat[P.empty_off[e]] = make_float2((float)sx, (float)sy);
        }
        return;
    }
    const int K = T.K, n = axis_coefs<COS>(K), per = group_rows<COS>(T.order, K);
    const int len = T.order == 1 ? n : (T.order == 2 ? n * n : n * n * n);
    const FastDiv by_n(n);
    for (int q = threadIdx.x; q < len; q += DA_THREADS) {
        int it, row = 0, group, at;   // partial sums at `at` of the group's items
        if (T.order == 1)
            it = q;
        else
            row = by_n.div(q, it);
        const int k = COS ? it : (it < K ? K - 1 - it : it - K);   // |k| - 1
        if (T.order == 1) {
            group = k / ORD1_GROUP;
            at = (k % ORD1_GROUP) * 4;
        } else {
            group = row / per;
            at = ((row - group * per) * K + k) * (COS ? 2 : 4);
        }
        const float *src = first + (long long)group * C * DA_MAX_ACC + at;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        auto add = [&](float (&r)[4], int c0, int c1) {
            for (int c = c0; c < c1; ++c) {
                const float *s = src + (long long)c * DA_MAX_ACC;
                if (COS && T.order > 1) {
                    r[0] += __ldcg(s);
                    r[2] += __ldcg(s + 1);
                } else {
                    const float4 w = __ldcg((const float4 *)s);
                    r[0] += w.x;
                    r[1] += w.y;
                    r[2] += w.z;
                    r[3] += w.w;
                }
            }
        };
        if (C <= DIRECT_MAX_CHUNKS) {
            add(v, 0, C);
        } else {   // in runs, which keeps the FP32 chains as short as those of fewer chunks
            for (int c = 0; c < C; c += DIRECT_MAX_CHUNKS) {
                float r[4] = {0.f, 0.f, 0.f, 0.f};
                add(r, c, min(C, c + DIRECT_MAX_CHUNKS));
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] += r[i];
            }
        }
        float2 g;
        if (COS)   // the innermost function's amplitude
            g = make_float2(SQRT2 * v[0], SQRT2 * v[2]);
        else   // u conj(w) for k > 0, u w for k < 0
            g = it >= K ? make_float2(v[0] + v[1], v[2] - v[3]) : make_float2(v[0] - v[1], v[2] + v[3]);
        fhat[T.coef_off + q] = g;
    }
}

// --------------------------------------------------------------- host ----

// Whether the kernels take a term.
bool direct_term(const Term &T) {
    const int K = axis_count(T);
    if (T.order == 1) return K <= 128;
    if (T.basis == ANOVA_BASIS_COS) return T.order == 2 ? K <= 9 : K <= 4;
    return T.order == 2 ? K <= 5 : K <= 3;
}

// Whether a plan of such terms is faster summed directly: both ways' times per transform
// (the mean of the two directions) in nanoseconds.  The constants of a term are
// least-squares fits to both ways measured at 66 shapes: d = 5 .. 20, |u| <= 1, 2, 3, both
// systems, 500 to 300 000 nodes; the faster way is taken at each of them but one, where
// they differ by 2 %.  Direct: order 1 per frequency, the others per multiply-add.  NFFT:
// per tile of 16 nodes (half a tile more per cell for the ragged last one) and per cell.
//   d  |u|    N            M        direct us         NFFT us    (forward / adjoint)
//   9   3  26/6/4      10 000       23 / 15           93 / 107
//   6   2   16/8       300 000      62 / 62           78 / 101
//   8   2   32/10      100 000      54 / 56           60 / 73
//   8   2   32/10      300 000     136 / 143         117 / 142
//  20   1     64       100 000      60 / 43           44 / 40
//  12   2  82/10 cos   100 000     136 / 195         102 / 122
// Beyond these, from 20 shapes at 100 000 to 10 million nodes (d = 1 .. 30):
// * every node costs both ways the same whatever the terms (blocks of few units, the
//   accumulators' pass): what plans of one or two coordinates take at a million nodes;
// * beyond 40 MB of powers and values, a third of L2, the adjoint's items wait for their
//   reads, those of the larger second-order terms, with two blocks to an SM, longer than
//   the others, with four;
// * the tiles' accumulators, 16 bytes a node, outgrow L2 and are added to from memory by
//   all terms but a few;
// * up to three third-order terms, of at most 64 items each, leave SMs idle.
//   1   1     16     1 000 000      49 / 39           66 / 56
//   4   2   16/8     1 000 000     121 / 96          128 / 124
//   4   2   16/8     3 000 000     415 / 494         317 / 307
//   6   2   16/8     1 000 000     202 / 338         199 / 220
//   6   2   16/4     3 000 000     490 / 492         520 / 564
//   6   2   16/8    10 000 000    2128 / 3334       4732 / 1846
// The slower way is taken at three of these 97 measurements, by 9, 10 and 16 %.
bool direct_faster(const Term *terms, int n_terms, int d, long long M) {
    double t_direct = DIRECT_FIXED_NS + 0.023 * M, t_nfft = NFFT_FIXED_NS + 0.020 * M, read = 0.0;
    int n3 = 0;
    bool big = false;
    for (int s = 0; s < n_terms; ++s) {
        const Term &T = terms[s];
        const int K = axis_count(T);
        if (T.order == 1) {
            t_direct += 7.5e-4 * K * (double)M;
        } else {
            const bool c = T.basis == ANOVA_BASIS_COS;
            const int n = c ? axis_coefs<true>(K) : axis_coefs<false>(K);
            const double ops = (T.order == 2 ? n : n * n) * (c ? 2.0 * K + 2.0 : 4.0 * K + 8.0);
            t_direct += (1.84e-3 + 4.4e-5 * ops) * (double)M;
        }
        read += (double)groups_of(T) * (T.order == 1 ? 20 : 8 + 8 * T.order);
        big = big || is_big(T);
        n3 += T.order == 3;
        double cells = T.n;
        for (int j = 1; j < T.order; ++j) cells *= T.n;
        cells = std::min(cells, (double)M);
        const double tiles = M / 16.0 + 0.5 * cells;
        t_nfft += T.order == 3 ? 0.46 * tiles + 1.54 * cells : 0.131 * tiles + 0.041 * cells;
    }
    if (8.0 * (d + 1) * M > 40e6) t_direct += 0.5 * read * (big ? 3.0e-4 : 1.05e-4) * M;   // one of two directions
    if (16.0 * M > 80e6) t_nfft += 0.007 * std::max(0, n_terms - 3) * (double)M;
    if (n3 > 0) t_nfft += 0.46 * M / 16.0 * std::max(0.0, 3.4 - n3);
    return t_direct < t_nfft;
}

int direct_groups(const Term &T) { return groups_of(T); }
int direct_axis(const Term &T) { return axis_count(T); }
bool direct_big(const Term &T) { return is_big(T); }
size_t direct_smem(int d, int kt, int npl, bool cosine) {
    return (size_t)(DT_THREADS / 32) * (32 * npl * sizeof(float2) + DIRECT_MAX_COEF * sizeof(float4)) +
           (size_t)d * kt * 32 * npl * (cosine ? sizeof(float) : sizeof(float2));
}

static DirectTerm term_record(const Term &T, int group) {
    DirectTerm r;
    r.order = T.order;
    r.K = axis_count(T);
    r.col = T.col;
    r.row0 = T.row0;
    r.row1 = T.row1;
    r.coef_off = (int)T.coef_off;
    r.group = group;
    r.pad = 0;
    return r;
}

// adjoint items of the active terms (and the empty set): C chunks each
int direct_items(const Plan &p, DirectItem *out) {
    long long groups = p.n_empty > 0 ? 1 : 0;
    for (int s = 0; s < p.n_act; ++s) groups += groups_of(p.h_terms[p.h_act[s]]);
    if (groups == 0) return 0;
    // rounds of resident blocks times a block's nodes, a block's own cost being that
    // of about 2000 nodes
    const long long R = (long long)p.sm_count * (p.direct_big ? DIRECT_RESIDENT_BIG : DIRECT_RESIDENT);
    int C = 1;
    double best = 0.0;
    for (int c = 1; c <= direct_max_chunks(p.M, p.direct_kt == 0); ++c) {
        if (c > 1 && groups * c > DIRECT_MAX_BLOCKS) break;
        const double t = (double)((groups * c + R - 1) / R) * ((double)p.M / c + 2000.0);
        if (c == 1 || t < 0.98 * best) {
            best = t;
            C = c;
        }
    }
    int n = 0;
    DirectItem it;
    std::memset(&it, 0, sizeof(it));
    it.chunks = C;
    for (int s = 0; s < p.n_act; ++s) {
        const Term &T = p.h_terms[p.h_act[s]];
        it.act = s;
        for (int g = 0; g < groups_of(T); ++g) {
            it.term = term_record(T, g);
            for (it.chunk = 0; it.chunk < C; ++it.chunk) out[n++] = it;
        }
    }
    it.act = -1;
    if (p.n_empty > 0)
        for (it.chunk = 0; it.chunk < C; ++it.chunk) out[n++] = it;
    return n;
}

// forward units of the active terms, order 1 by frequency groups
int direct_unit_list(const Plan &p, DirectTerm *out) {
    int n = 0;
    for (int s = 0; s < p.n_act; ++s) {
        const Term &T = p.h_terms[p.h_act[s]];
        for (int g = 0; g < (T.order == 1 ? groups_of(T) : 1); ++g) out[n++] = term_record(T, g);
    }
    return n;
}

int build_unit_table(Plan &p) {
    const long long total = (long long)p.d * p.M;
    if (total == 0) return ANOVA_OK;
    k_unit_table<<<(int)std::min<long long>(4096, (total + 255) / 256), 256, 0, p.stream>>>((const float *)p.x, p.z, total);
    return cuda_status(cudaGetLastError());
}

// nodes per lane: each coefficient read serves them all (300 000 nodes, d = 12, cosine
// system: 351 us at four, 398 us at two)
int direct_npl(int d, int kt, long long M, bool cosine) {
    int npl = M >= 20000 ? 4 : M >= 2000 ? 2 : 1;
    while (npl > 1 && direct_smem(d, kt, npl, cosine) > DIRECT_MAX_SMEM) npl /= 2;
    return npl;
}
int direct_splits(long long n_units, long long M, int npl, int sm_count) {
    // rounds of resident CTAs times a warp's units, a CTA's own cost (its table and
    // reduction) being that of about three
    const long long blocks = (M + 32 * npl - 1) / (32 * npl), R = 3LL * sm_count, NW = DT_THREADS / 32;
    int best = 1;
    double cost = 0.0;
    for (int S = 1; S <= DIRECT_MAX_SPLITS; ++S) {
        const double t = (double)((blocks * S + R - 1) / R) * ((double)((n_units + NW * S - 1) / (NW * S)) + 3.0);
        if (S == 1 || t < 0.98 * cost) {
            best = S;
            cost = t;
        }
    }
    return best;
}

template <int NPL, bool COS>
static void launch_trafo(Plan &p, const DevPlan &v, const float2 *fhat, float2 *f) {
    static std::atomic<unsigned long long> attr_seen{0};
    once_per_device(attr_seen, [] {
        cudaFuncSetAttribute(direct_trafo<NPL, COS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, DIRECT_MAX_SMEM);
        cudaFuncSetAttribute(direct_trafo<NPL, COS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, DIRECT_MAX_SMEM);
    });
    const int NB = 32 * NPL;
    const dim3 grid((unsigned)((p.M + NB - 1) / NB), p.direct_split);
    const bool chains = p.n_direct_units > DT_CHAIN * (DT_THREADS / 32) * p.direct_split;
    auto k = chains ? direct_trafo<NPL, COS, true> : direct_trafo<NPL, COS, false>;
    k<<<grid, DT_THREADS, direct_smem(p.d, p.direct_kt, NPL, COS), p.stream>>>(
        v, fhat, f, p.direct_kt, p.direct_units, p.n_direct_units, p.direct_fpart, p.direct_fcount);
}

int launch_direct_trafo(Plan &p, const float2 *fhat, float2 *f) {
    const DevPlan v = dev_view(p);
    stage_begin(p, ST_GATHER);
    if (p.basis == ANOVA_BASIS_COS)
        p.direct_npl == 4   ? launch_trafo<4, true>(p, v, fhat, f)
        : p.direct_npl == 2 ? launch_trafo<2, true>(p, v, fhat, f)
                            : launch_trafo<1, true>(p, v, fhat, f);
    else
        p.direct_npl == 4   ? launch_trafo<4, false>(p, v, fhat, f)
        : p.direct_npl == 2 ? launch_trafo<2, false>(p, v, fhat, f)
                            : launch_trafo<1, false>(p, v, fhat, f);
    stage_end(p, ST_GATHER);
    return cuda_status(cudaGetLastError());
}

int launch_direct_adjoint(Plan &p, const float2 *y, float2 *fhat) {
    const DevPlan v = dev_view(p);
    if (p.M == 0) {
        cudaMemsetAsync(fhat, 0, sizeof(float2) * p.n_coeffs, p.stream);
        return cuda_status(cudaGetLastError());
    }
    if (p.n_items == 0) return ANOVA_OK;
    stage_begin(p, ST_SPREAD);
    auto of = [&](auto runs) {
        constexpr bool R = decltype(runs)::value;
        return p.basis == ANOVA_BASIS_COS ? (p.direct_big ? direct_adjoint<true, true, R> : direct_adjoint<true, false, R>)
                                          : (p.direct_big ? direct_adjoint<false, true, R> : direct_adjoint<false, false, R>);
    };
    const int C = p.h_ditems[0].chunks;   // the same for every item
    auto k = (p.M + C - 1) / C > DA_RUN ? of(std::true_type()) : of(std::false_type());
    k<<<p.n_items, DA_THREADS, 0, p.stream>>>(v, p.direct_items, y, fhat, p.direct_part, p.direct_count);
    stage_end(p, ST_SPREAD);
    return cuda_status(cudaGetLastError());
}

}  // namespace agft
