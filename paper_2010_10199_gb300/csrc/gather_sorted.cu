// Forward gather over the cell-sorted node records (every term with records:
// all terms of an FP32 plan that keeps them), the window interpolation step
// of the NFFT behind eq. (somafm), Sec. 3, FP32.
//
// Work items are the adjoint's (active term, node chunk) pairs.  A CTA copies
// the term's stored grid into shared memory.  gather_sorted_f32 gives each
// thread two consecutive records: the thread evaluates each node's 8 column
// and 2 m_row row window weights from the per-tap polynomials (coefficients
// broadcast from shared memory, 16 bytes at a time), reads the 6 x 8 grid
// values around the cell (the nodes of a warp mostly share a cell, so the
// reads are broadcasts, and one read serves both nodes when the pair shares a
// cell) and adds sum_i w_row[i] sum_t w_col[t] g[i][t] into node j's
// accumulator.  Plans with node tiles form the same sums on the tensor cores
// (gather_tiles.cu).  The accumulators are 64-bit integers holding the values in
// fixed point, v * 2^e with 2^e chosen from ||fhat||_1 (a bound on every
// partial sum), so the additions are exact and their order, which the
// hardware does not fix, cannot change the result: the forward is bitwise
// reproducible.  A last pass writes f, the empty set's coefficient plus
// acc * 2^-e, and zeroes the accumulators for the next call.
#include <algorithm>
#include <cstring>

#include "device.cuh"
#include "internal.cuh"

namespace agft {

constexpr int GS_THREADS = 256;

__device__ __forceinline__ void red_add_u64(unsigned long long *addr, long long v) {
    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ const DevPlan &plan_of(const DevPlan &single, const BatchArgs &B, int prob) {
    return B.plans ? B.plans[prob] : single;
}

constexpr int FIN_UNROLL = 4;

// per problem (blockIdx.y): f[j] = empty-set coefficient + acc[j] * 2^-e; leaves
// the accumulators and the launch's item counter at zero for the next call
__global__ void k_fixed_point_finish(DevPlan single, BatchArgs B, const float2 *__restrict__ fhat_base,
                                     float2 *f_base, int *counter) {
    const DevPlan &P = plan_of(single, B, blockIdx.y);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 2) counter[threadIdx.x] = 0;
    if (P.skip && *P.skip) return;
    const float2 *fhat = fhat_base + P.vec_coef_off;
    float2 c0 = make_float2(0.f, 0.f);
    for (int e = 0; e < P.n_empty; ++e) {
        const float2 c = fhat[P.empty_off[e]];
        c0.x += c.x;
        c0.y += c.y;
    }
    // a coefficient that is not finite reaches every node (the accumulators hold no such value)
    const double sc = P.fexp[2] ? __longlong_as_double(0x7ff8000000000000LL) : ldexp(1.0, -*P.fexp);
    float2 *__restrict__ f = f_base + P.vec_node_off;
    longlong2 *__restrict__ acc = (longlong2 *)P.facc;
    const long long M = P.M, step = (long long)gridDim.x * blockDim.x;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < M; j += FIN_UNROLL * step) {
        longlong2 a[FIN_UNROLL];   // independent loads in flight
#pragma unroll
        for (int u = 0; u < FIN_UNROLL; ++u) a[u] = j + u * step < M ? acc[j + u * step] : make_longlong2(0, 0);
#pragma unroll
        for (int u = 0; u < FIN_UNROLL; ++u) {
            if (j + u * step >= M) break;
            acc[j + u * step] = make_longlong2(0, 0);
            f[j + u * step] = make_float2(c0.x + (float)((double)a[u].x * sc), c0.y + (float)((double)a[u].y * sc));
        }
    }
}

// polynomial of tap t from the shared coefficient table (two float4 per tap),
// at two arguments; the same operations as horner8
__device__ __forceinline__ void horner_pair(const float4 *c, float v0, float v1, float &w0, float &w1) {
    const float4 lo = c[0], hi = c[1];
    float a = hi.w, b = hi.w;
    a = fmaf(a, v0, hi.z);
    b = fmaf(b, v1, hi.z);
    a = fmaf(a, v0, hi.y);
    b = fmaf(b, v1, hi.y);
    a = fmaf(a, v0, hi.x);
    b = fmaf(b, v1, hi.x);
    a = fmaf(a, v0, lo.w);
    b = fmaf(b, v1, lo.w);
    a = fmaf(a, v0, lo.z);
    b = fmaf(b, v1, lo.z);
    a = fmaf(a, v0, lo.y);
    b = fmaf(b, v1, lo.y);
    w0 = fmaf(a, v0, lo.x);
    w1 = fmaf(b, v1, lo.x);
}

template <int MR>
__global__ void __launch_bounds__(GS_THREADS, 3)
gather_sorted_f32(DevPlan single, BatchArgs B, const int4 *__restrict__ items, int item_end, int *counter,
                  long long max_grid_bytes) {
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *S = (float2 *)smem;
    float4 *coef = (float4 *)(smem + max_grid_bytes);   // [8 column taps + 8 row taps][2]
    int &s_item = *(int *)(coef + 32);
    const int tid = threadIdx.x;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= item_end) break;
        const int4 itm = items[item];
        const DevPlan &P = plan_of(single, B, itm.x);
        if (P.skip && *P.skip) continue;
        const long long M = P.M;
        unsigned long long *__restrict__ acc = P.facc;
        const float sc = __int_as_float((127 + *P.fexp) << 23);   // 2^e, exact scaling
        const Term &T = P.terms[P.act[itm.y]];
        if (T.sort_slot < 0) continue;   // no records: the point-major gather has the term
        const long long j0 = M * itm.z / itm.w, j1 = M * (itm.z + 1) / itm.w;
        // the term's grid and window coefficients into shared memory
        {
            const float4 *g = (const float4 *)(P.grids + T.grid_off);
            float4 *S4 = (float4 *)S;
            const long long n4 = T.grid_bytes / 16;
            for (long long e = tid; e < n4; e += GS_THREADS) S4[e] = __ldg(g + e);
            if (tid < 32) {
                const int tap = tid >> 1, h = tid & 1;
                const float *src = tap < 8 ? P.windows[T.wc].c[tap] : P.windows[T.wr].c[min(tap - 8, 2 * MR - 1)];
                coef[tid] = make_float4(__ldg(src + 4 * h), __ldg(src + 4 * h + 1), __ldg(src + 4 * h + 2),
                                        __ldg(src + 4 * h + 3));
            }
        }
        __syncthreads();
        const float4 *rec = P.frec + (long long)T.sort_slot * M;
        const int stride = T.stride;
        const bool two = T.order == 2;
        if (T.order == 3) {
            // one node per thread: two records (window arguments and index; the
            // cell's grid indices), 2 MR x 2 MR rows of 8 taps, indices modulo n
            const int n = T.n;
            for (long long p = j0 + tid; p < j1; p += GS_THREADS) {
                const float4 q = __ldg(rec + 2 * p), qc = __ldg(rec + 2 * p + 1);
                const int fa = __float_as_int(qc.x), fb = __float_as_int(qc.y), fc = __float_as_int(qc.z);
                float wc[8], wb[2 * MR], dummy;
                int col[8], rb[2 * MR];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    horner_pair(coef + 2 * t, q.z, q.z, wc[t], dummy);
                    col[t] = wrap(fc - T.mc + 1 + t, n);
                }
#pragma unroll
                for (int i = 0; i < 2 * MR; ++i) {
                    horner_pair(coef + 16 + 2 * i, q.y, q.y, wb[i], dummy);
                    rb[i] = wrap(fb - MR + 1 + i, n);
                }
                float sx = 0.f, sy = 0.f;
#pragma unroll 1
                for (int ia = 0; ia < 2 * MR; ++ia) {
                    float wa;
                    horner_pair(coef + 16 + 2 * ia, q.x, q.x, wa, dummy);
                    const int ra = wrap(fa - MR + 1 + ia, n) * n;
                    float ux = 0.f, uy = 0.f;
#pragma unroll
                    for (int ib = 0; ib < 2 * MR; ++ib) {
                        const float2 *row = S + (ra + rb[ib]) * stride;
                        float tx = 0.f, ty = 0.f;
#pragma unroll
                        for (int t = 0; t < 8; ++t) {
                            const float2 g = row[col[t]];
                            tx = fmaf(wc[t], g.x, tx);
                            ty = fmaf(wc[t], g.y, ty);
                        }
                        ux = fmaf(wb[ib], tx, ux);
                        uy = fmaf(wb[ib], ty, uy);
                    }
                    sx = fmaf(wa, ux, sx);
                    sy = fmaf(wa, uy, sy);
                }
                unsigned long long *a0 = acc + 2 * (long long)__float_as_int(q.w);
                red_add_u64(a0, __float2ll_rn(sx * sc));
                red_add_u64(a0 + 1, __float2ll_rn(sy * sc));
            }
            __syncthreads();
            continue;
        }
        // a thread takes two consecutive records (mostly of one cell: then
        // every grid value read serves both); the warp iterates as a whole
        const int lane = tid & 31;
        for (long long wb = j0 + 2 * (tid - lane); wb < j1; wb += 2 * GS_THREADS) {
            const long long p = wb + 2 * lane;
            const bool ok0 = p < j1, ok1 = p + 1 < j1;
            const float4 q0 = __ldg(rec + (ok0 ? p : j1 - 1)), q1 = __ldg(rec + (ok1 ? p + 1 : j1 - 1));
            float wc0[8], wc1[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) horner_pair(coef + 2 * t, q0.y, q1.y, wc0[t], wc1[t]);
            const int off0 = __float_as_int(q0.z), off1 = __float_as_int(q1.z);
            const bool same = __all_sync(0xffffffffu, off0 == off1);
            float sx0 = 0.f, sy0 = 0.f, sx1 = 0.f, sy1 = 0.f;
            if (two) {
#pragma unroll
                for (int i = 0; i < 2 * MR; ++i) {
                    float wr0, wr1;
                    horner_pair(coef + 16 + 2 * i, q0.x, q1.x, wr0, wr1);
                    const float2 *r0 = S + off0 + i * stride, *r1 = S + off1 + i * stride;
                    float tx0 = 0.f, ty0 = 0.f, tx1 = 0.f, ty1 = 0.f;
                    if (same) {
#pragma unroll
                        for (int t = 0; t < 8; ++t) {
                            const float2 a = r0[t];
                            tx0 = fmaf(wc0[t], a.x, tx0);
                            ty0 = fmaf(wc0[t], a.y, ty0);
                            tx1 = fmaf(wc1[t], a.x, tx1);
                            ty1 = fmaf(wc1[t], a.y, ty1);
                        }
                    } else {
#pragma unroll
                        for (int t = 0; t < 8; ++t) {
                            const float2 a = r0[t], c = r1[t];
                            tx0 = fmaf(wc0[t], a.x, tx0);
                            ty0 = fmaf(wc0[t], a.y, ty0);
                            tx1 = fmaf(wc1[t], c.x, tx1);
                            ty1 = fmaf(wc1[t], c.y, ty1);
                        }
                    }
                    sx0 = fmaf(wr0, tx0, sx0);
                    sy0 = fmaf(wr0, ty0, sy0);
                    sx1 = fmaf(wr1, tx1, sx1);
                    sy1 = fmaf(wr1, ty1, sy1);
                }
            } else {
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const float2 a = S[off0 + t], c = same ? a : S[off1 + t];
                    sx0 = fmaf(wc0[t], a.x, sx0);
                    sy0 = fmaf(wc0[t], a.y, sy0);
                    sx1 = fmaf(wc1[t], c.x, sx1);
                    sy1 = fmaf(wc1[t], c.y, sy1);
                }
            }
            if (ok0) {
                unsigned long long *a0 = acc + 2 * (long long)__float_as_int(q0.w);
                red_add_u64(a0, __float2ll_rn(sx0 * sc));
                red_add_u64(a0 + 1, __float2ll_rn(sy0 * sc));
            }
            if (ok1) {
                unsigned long long *a1 = acc + 2 * (long long)__float_as_int(q1.w);
                red_add_u64(a1, __float2ll_rn(sx1 * sc));
                red_add_u64(a1 + 1, __float2ll_rn(sy1 * sc));
            }
        }
        __syncthreads();   // the grid is read by every thread before the next item replaces it
    }
}

int gather_sorted_launch(cudaStream_t st, const DevPlan &v, const BatchArgs &B, int P, const float2 *fhat,
                         float2 *f, const int4 *items, int n_items3, int n_items, int *counter,
                         long long max_grid_bytes, long long max_M, int sm_count, int mr, bool tc) {
    static std::atomic<unsigned long long> attr_seen{0};
    once_per_device(attr_seen, [] {
        cudaFuncSetAttribute(gather_sorted_f32<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
        cudaFuncSetAttribute(gather_sorted_f32<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
    });
    if (tc) {
        gather_tiles_launch(st, v, B, items, n_items, n_items3 > 0, counter, max_grid_bytes, sm_count, mr);
    } else if (n_items > 0) {
        const size_t smem = (size_t)max_grid_bytes + 32 * sizeof(float4) + 16;
        const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(3, (size_t)(MAX_SMEM + 1024) / (smem + 1024)));
        const int ctas = std::max(1, std::min(n_items, per_sm * sm_count));
        if (mr <= 3)
            gather_sorted_f32<3><<<ctas, GS_THREADS, smem, st>>>(v, B, items, n_items, counter, max_grid_bytes);
        else
            gather_sorted_f32<4><<<ctas, GS_THREADS, smem, st>>>(v, B, items, n_items, counter, max_grid_bytes);
    }
    // two rounds of four nodes per thread for the largest problem, at least one
    // round filling the chip; a batch's smaller problems leave their blocks idle
    const int nb = (int)std::max<long long>(1, (max_M + 256 * 2 * FIN_UNROLL - 1) / (256 * 2 * FIN_UNROLL));
    k_fixed_point_finish<<<dim3(nb, P), 256, 0, st>>>(v, B, fhat, f, counter);
    return cuda_status(cudaGetLastError());
}

// single plan: every term has records (third-order ones without records were
// handled by the point-major gather, which then wrote f; see trafo.cu)
int launch_gather_sorted_f32(Plan &p, const float2 *fhat, float2 *f) {
    DevPlan v = dev_view(p);
    BatchArgs B;
    std::memset(&B, 0, sizeof(B));
    int mr = 3;
    for (int s = 0; s < p.n_terms; ++s)
        if (p.h_terms[s].mr > 0) mr = p.h_terms[s].mr;
    return gather_sorted_launch(p.stream, v, B, 1, fhat, f, p.items, p.n_items3, p.n_items, p.counter,
                                p.max_grid_bytes, p.M, p.sm_count, mr, p.cell_tc && !p.frec);
}

}  // namespace agft
