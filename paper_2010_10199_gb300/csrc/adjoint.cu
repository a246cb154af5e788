// Adjoint grouped transform fhat = F^H y (stacked adjoint after the error
// remark, Sec. 3), FP32.
//
//   1. spread: work items (term, node chunk) from a global queue.  An item
//      accumulates y_j times the window into a shared-memory copy of the
//      term's stored grid (halos included), then writes it to partial grid z
//      of the term (z = chunk index).  With cell-sorted node records the sums
//      of one grid cell's nodes are formed first -- on the tensor cores
//      (spread_tiles.cu) or in registers on the CUDA cores (spread_f32 sorted
//      items, spread3_f32) -- and added to the shared grid
//      once per cell; without records every node's window is added with
//      shared-memory atomics.
//   2. adjoint_post: per term, sum the partial grids in a fixed order
//      (reduce_partials before it where there are many), fold the halos back
//      onto the periodic grid, FFT with sign -, multiply by the deconvolution
//      factors and crop the block (I_N minus {0})^{|u|}.
//   3. empty-set terms: sum_j y_j, partial sums first, added by adjoint_post.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "device.cuh"
#include "internal.cuh"

namespace agft {

// shared-memory float reduction without a returned value
__device__ __forceinline__ void red_add(float *addr, float v) {
    asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(smem_addr(addr)), "f"(v) : "memory");
}

constexpr int POST_MAX_CHUNKS = 16;   // chunks per term summed inside adjoint_post_f32
constexpr int SUM_Y_BLOCKS = 608;     // partial sums of y (at most this many per problem)

constexpr int SP_CH = 512;   // nodes staged per block of a work item (order 1/2: SP_CH or SP_CH / 2)

__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// staging area after the grid: the larger of the unsorted layout
// (float4 [2][SP]) and the sorted one (float4 [3][SP] node records, float2
// [2][SP] values of y), SP nodes per block
__host__ __device__ constexpr size_t sp_stage_bytes(int sp) { return (size_t)sp * (3 * 16 + 2 * 8); }
// third-order items (spread3_f32): 8 warp runs of 32 nodes, two records each
constexpr size_t SP3_STAGE_BYTES = 3 * 256 * 32 + 2 * 256 * 8;


// shared memory of spread_f32 (o3 = false, sp nodes per block) or spread3_f32:
// grid, node blocks, item slot
size_t spread_smem_bytes(long long max_grid_bytes, bool o3, int sp) {
    return (size_t)max_grid_bytes + (o3 ? SP3_STAGE_BYTES : sp_stage_bytes(sp)) + 16;
}

// CTAs per SM that shared memory allows for spread_f32 with sp-node blocks
static size_t smem_ctas(long long max_grid_bytes, int sp) {
    const size_t per = spread_smem_bytes(max_grid_bytes, false, sp) + 1024;   // + the per-CTA reserve
    return (size_t)(MAX_SMEM + 1024) / per;
}

// CTAs per SM of spread_f32 with sp-node blocks: at most 4 (64 registers) for
// SP_CH / 2, 3 (80 registers) for SP_CH
static int ctas_for(long long max_grid_bytes, int sp) {
    const size_t cap = sp == SP_CH ? 3 : SPREAD_MAX_CTAS_PER_SM;
    return (int)std::max<size_t>(1, std::min(cap, smem_ctas(max_grid_bytes, sp)));
}

// nodes per staging block.  The larger block runs best where registers, not
// shared memory, hold it at 3 CTAs per SM (small grids); where the grids fill
// shared memory, the smaller block gains a fourth CTA per SM (measured on the
// d = 20 workloads: bandwidths 64/32 gain, 32/16 lose with the smaller block).
int spread_block_nodes(long long max_grid_bytes) {
    const bool smem_bound = smem_ctas(max_grid_bytes, SP_CH) < (size_t)SPREAD_MAX_CTAS_PER_SM;
    return smem_bound && ctas_for(max_grid_bytes, SP_CH / 2) > ctas_for(max_grid_bytes, SP_CH) ? SP_CH / 2 : SP_CH;
}

int spread_ctas_per_sm(long long max_grid_bytes) { return ctas_for(max_grid_bytes, spread_block_nodes(max_grid_bytes)); }

// Nanoseconds a CTA takes per node of an order-1/2 and of a third-order term, and
// per work item (grid copies, first cells): measured at d = 20, M = 1e6 and d = 10,
// M = 5e5.  Only their ratios matter here.
constexpr double NS_NODE = 3.0, NS_NODE3 = 16.0, NS_ITEM = 4000.0;

// Time of n3 items of d3 followed by n items of d <= d3 on R CTAs that take the next
// item when they are free.
static double queue_time(long long n3, double d3, long long n, double d, long long R) {
    const long long base = n3 / R, rem = n3 % R;
    const double early = base * d3, late = (base + (rem > 0)) * d3;
    if (n == 0) return late;
    for (long long k = n / R;; ++k) {   // an early CTA takes k more items
        const double t = early + k * d;
        const long long l = t > early + d3 ? (long long)((t - early - d3) / d + 1e-9) : 0;
        if ((R - rem) * k + rem * l >= n) return std::max(late, t);
    }
}

int spread_chunks_for(long long M, int n_terms, int n_terms3, int kmax, long long max_grid_bytes,
                      long long grid_elems, int sm_count, bool tc) {
    // the chunk count whose items fill the CTAs of the spread and of the gather
    // best: at d = 20, M = 1e6 the former rule's 5 chunks per term (three items per
    // CTA) left the gather's third round of 456 CTAs a third full, 1.76 ms
    const bool order3 = n_terms3 > 0;
    const long long Rs = (long long)sm_count * (tc ? spread_tiles_ctas_per_sm(max_grid_bytes, order3)
                                                   : spread_ctas_per_sm(max_grid_bytes));
    const long long Rg = (long long)sm_count * (tc ? gather_tiles_ctas_per_sm(max_grid_bytes, order3) : 3);
    const int n = n_terms - n_terms3;
    int best = 1;
    double cost = 0.0;
    for (int K = 1; K <= kmax; ++K) {
        const double d3 = NS_NODE3 * M / K + NS_ITEM, d = NS_NODE * M / K + NS_ITEM;
        const double c = queue_time((long long)n_terms3 * K, d3, (long long)n * K, d, Rs) +
                         queue_time((long long)n_terms3 * K, d3, (long long)n * K, d, Rg) +
                         K * grid_elems * 8 / 2500.0;   // partial grids written and read at 5 bytes per ps
        if (K == 1 || c < 0.995 * cost) {
            best = K;
            cost = c;
        }
    }
    return best;
}

// chunks of problem p of a batch: items of about equal cost, ten per CTA
int batch_chunks_for(long long M, double total_ns, int kmax, long long ctas) {
    const double item = std::max(total_ns / (10.0 * ctas), NS_ITEM);
    return (int)std::max<long long>(1, std::min<long long>(kmax, (long long)std::ceil(NS_NODE * M / item)));
}

double batch_cost_ns(long long M, int n_terms, int n_terms3) {
    return M * (NS_NODE * (n_terms - n_terms3) + NS_NODE3 * n_terms3);
}

int append_spread_items(const Plan &p, int prob, int K, int4 *out, int sel) {
    int n = 0;
    for (int order = sel == 3 ? 3 : 2; order >= (sel == 3 ? 3 : 1); --order)
        for (int s = 0; s < p.n_act; ++s) {
            if (p.h_terms[p.h_act[s]].order != order) continue;
            for (int z = 0; z < K; ++z) out[n++] = make_int4(prob, s, z, K);
        }
    return n;
}

// Window weights of one node for a half-warp, lane (r, k): lanes r = 0
// evaluate the column tap k, lanes r = 1 the row tap k (clamped to the
// window), each from its own coefficients wcf; shuffles hand every lane the
// column weight of its tap and the row weights of rows r, r + 2, ...
template <int MR>
__device__ __forceinline__ void node_weights(const float wcf[NCOEF], float vrow, float vcol, int half, int r, int k,
                                             float &cw, float w[MR]) {
    const float wt = horner8(wcf, r ? vrow : vcol);
    cw = __shfl_sync(0xffffffffu, wt, (half << 4) | k);
#pragma unroll
    for (int j = 0; j < MR; ++j) w[j] = __shfl_sync(0xffffffffu, wt, (half << 4) | 8 | (r + 2 * j));
}

// Sorted item: the item's nodes in cell order of its term, as records
// (window arguments, first-tap grid offset, original index).  The item's node
// range is cut into 16 contiguous runs, one per half-warp; block c of the
// staging holds records c*RUN .. c*RUN+RUN-1 of every run.  Records pass
// through shared memory by cp.async two blocks ahead, the values y[index] one
// block ahead (their addresses come from the staged records).  A half-warp
// sums the contributions of a cell in registers (lane (r, k): column tap k,
// rows r, r + 2, ..), two nodes per step, and adds the sums to the shared
// grid when the cell changes and at the end of its run.  Order 1: the lane
// groups r = 0, 1 take alternate nodes of the run.
template <int MR, int SP>
__device__ __forceinline__ void spread_sorted_item(const DevPlan &P, const Term &T, const float2 *__restrict__ y,
                                                   long long j0, long long j1, float2 *S, unsigned char *stg_raw,
                                                   const float wcf[NCOEF]) {
    constexpr int RUN = SP / 16;
    const int tid = threadIdx.x;
    const int lane = tid & 31, half = lane >> 4, sub = lane & 15;
    const int r = sub >> 3, k = sub & 7;
    const int hw = (tid >> 5) * 2 + half;
    const int stride = T.stride;
    const float4 *src = P.srec + (long long)T.sort_slot * P.M + j0;
    float4 *rbuf = (float4 *)stg_raw;            // [3][SP]
    float2 *ybuf = (float2 *)(rbuf + 3 * SP); // [2][SP]
    const long long len = j1 - j0;
    const long long L = (len + 15) / 16;           // run length
    const long long nblk = (L + RUN - 1) / RUN;
    // records of run h: [h L, min((h+1) L, len))
    auto run_len = [&](int h) { return max(0LL, min(L, len - (long long)h * L)); };
    auto stage_a = [&](long long c) {
        const int b = (int)(c % 3) * SP;
        for (int e = tid; e < SP; e += SPREAD_THREADS) {
            const int h = e / RUN, t = e % RUN;
            const long long q = c * RUN + t;
            if (q < run_len(h)) cp_async16(&rbuf[b + e], src + (long long)h * L + q);
        }
    };
    // reads records this thread staged itself (same e), so its own wait suffices
    auto stage_b = [&](long long c) {
        const int b = (int)(c % 3) * SP, yb = (int)(c & 1) * SP;
        for (int e = tid; e < SP; e += SPREAD_THREADS) {
            const int h = e / RUN, t = e % RUN;
            if (c * RUN + t < run_len(h)) cp_async8(&ybuf[yb + e], y + __float_as_int(rbuf[b + e].w));
        }
    };
    const long long my_len = run_len(hw);
    int cur = -1;   // grid offset of the cell being summed
    float ax[MR], ay[MR];
#pragma unroll
    for (int j = 0; j < MR; ++j) ax[j] = ay[j] = 0.f;
    auto flush2 = [&]() {
        float *base = (float *)(S + cur + r * stride + k);
#pragma unroll
        for (int j = 0; j < MR; ++j) {
            red_add(base + 4 * j * stride, ax[j]);
            red_add(base + 4 * j * stride + 1, ay[j]);
            ax[j] = ay[j] = 0.f;
        }
    };
    auto flush1 = [&]() {
        float *base = (float *)(S + cur + k);
        red_add(base, ax[0]);
        red_add(base + 1, ay[0]);
        ax[0] = ay[0] = 0.f;
    };
    const int col_src = (half << 4) | k, row_src = (half << 4) | 8 | r;
    if (nblk > 0) stage_a(0);
    cp_async_commit();
    if (nblk > 1) stage_a(1);
    cp_async_commit();
    cp_async_wait1();
    if (nblk > 0) stage_b(0);
    cp_async_commit();
    for (long long c = 0; c < nblk; ++c) {
        cp_async_wait0();
        __syncthreads();
        if (c + 1 < nblk) stage_b(c + 1);
        cp_async_commit();
        if (c + 2 < nblk) stage_a(c + 2);
        cp_async_commit();
        const float4 *rb = rbuf + (int)(c % 3) * SP + hw * RUN;
        const float2 *yb = ybuf + (int)(c & 1) * SP + hw * RUN;
        const long long left = my_len - c * RUN;   // records of this run still to come
        if (T.order == 2) {
            // both half-warps of a warp run all steps (shuffles); a node past
            // the run's end computes on record 0, adds zero and keeps the cell
            for (int t = 0; t < RUN; t += 2) {
                const bool ok0 = t < left, ok1 = t + 1 < left;
                const float4 q0 = rb[ok0 ? t : 0], q1 = rb[ok1 ? t + 1 : 0];
                const float wt0 = horner8(wcf, r ? q0.x : q0.y);
                const float wt1 = horner8(wcf, r ? q1.x : q1.y);
                const float cw0 = __shfl_sync(0xffffffffu, wt0, col_src);
                const float cw1 = __shfl_sync(0xffffffffu, wt1, col_src);
                float w0[MR], w1[MR];
#pragma unroll
                for (int j = 0; j < MR; ++j) {
                    w0[j] = __shfl_sync(0xffffffffu, wt0, row_src + 2 * j);
                    w1[j] = __shfl_sync(0xffffffffu, wt1, row_src + 2 * j);
                }
                const float2 y0 = ok0 ? yb[t] : make_float2(0.f, 0.f);
                const float2 y1 = ok1 ? yb[t + 1] : make_float2(0.f, 0.f);
                const int off0 = ok0 ? __float_as_int(q0.z) : cur;
                const int off1 = ok1 ? __float_as_int(q1.z) : off0;
                if (off0 != cur) {
                    if (cur >= 0) flush2();
                    cur = off0;
                }
                const float y0x = y0.x * cw0, y0y = y0.y * cw0;
#pragma unroll
                for (int j = 0; j < MR; ++j) {
                    ax[j] = fmaf(y0x, w0[j], ax[j]);
                    ay[j] = fmaf(y0y, w0[j], ay[j]);
                }
                if (off1 != cur) {
                    flush2();
                    cur = off1;
                }
                const float y1x = y1.x * cw1, y1y = y1.y * cw1;
#pragma unroll
                for (int j = 0; j < MR; ++j) {
                    ax[j] = fmaf(y1x, w1[j], ax[j]);
                    ay[j] = fmaf(y1y, w1[j], ay[j]);
                }
            }
        } else {
            for (int t = r; t < RUN; t += 2) {
                if (t >= left) break;
                const float4 q = rb[t];
                const int off = __float_as_int(q.z);
                if (off != cur) {
                    if (cur >= 0) flush1();
                    cur = off;
                }
                const float cw = horner8(wcf, q.y);
                const float2 yv = yb[t];
                ax[0] = fmaf(yv.x, cw, ax[0]);
                ay[0] = fmaf(yv.y, cw, ay[0]);
            }
        }
        __syncthreads();
    }
    cp_async_wait0();
    if (cur >= 0) {
        if (T.order == 2)
            flush2();
        else
            flush1();
    }
}

// Sorted third-order item: two records per node (window arguments and
// original index; the cell's grid indices).  The item's nodes are cut into 8
// runs, one per warp; blocks of 32 nodes per run are staged like the order-2
// path (records two blocks ahead, y one block ahead).  A warp takes one node
// at a time: lane (g, k), g = lane / 8, owns column tap k and the row pairs
// (ia, ib) with ib in {g, g + 4}, keeps their sums for the current cell in
// registers and adds them to the shared grid (indices modulo n) when the cell
// changes and at the end of its run.  Lanes 0..7 evaluate the first row
// coordinate's taps, lanes 8..15 the second's; shuffles hand them round.
constexpr int SP3_RUN = 32;                     // nodes per warp and block
constexpr int SP3_BLK = SP3_RUN * (SPREAD_THREADS / 32);
static_assert(3 * SP3_BLK * 32 + 2 * SP3_BLK * 8 <= SP3_STAGE_BYTES, "third-order staging");

template <int MR>
__device__ __forceinline__ void spread_sorted_item3(const DevPlan &P, const Term &T, const float2 *__restrict__ y,
                                                    long long j0, long long j1, float2 *S, unsigned char *stg_raw,
                                                    const float cc[NCOEF]) {
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 3, k = lane & 7;
    const int n = T.n, stride = T.stride, mc = T.mc;
    const float4 *src = P.srec + (long long)T.sort_slot * P.M + 2 * j0;
    float4 *rbuf = (float4 *)stg_raw;                   // [3][SP3_BLK][2]
    float2 *ybuf = (float2 *)(rbuf + 3 * 2 * SP3_BLK);  // [2][SP3_BLK]
    float rcf[NCOEF];
    {
        const float *c = P.windows[T.wr].c[min(k, 2 * MR - 1)];
#pragma unroll
        for (int q = 0; q < NCOEF; ++q) rcf[q] = __ldg(c + q);
    }
    const long long len = j1 - j0;
    const long long L = (len + 7) / 8;   // run length
    const long long nblk = (L + SP3_RUN - 1) / SP3_RUN;
    auto run_len = [&](int h) { return max(0LL, min(L, len - (long long)h * L)); };
    // thread tid stages node t_s of run h_s in every block
    const int h_s = tid / SP3_RUN, t_s = tid % SP3_RUN;
    const long long len_s = run_len(h_s);
    auto stage_a = [&](long long c) {
        const long long q = c * SP3_RUN + t_s;
        if (q < len_s) {
            float4 *d = rbuf + ((int)(c % 3) * SP3_BLK + tid) * 2;
            const float4 *gsrc = src + 2 * ((long long)h_s * L + q);
            cp_async16(d, gsrc);
            cp_async16(d + 1, gsrc + 1);
        }
    };
    auto stage_b = [&](long long c) {   // reads this thread's own staged record
        if (c * SP3_RUN + t_s < len_s)
            cp_async8(&ybuf[(int)(c & 1) * SP3_BLK + tid],
                      y + __float_as_int(rbuf[((int)(c % 3) * SP3_BLK + tid) * 2].w));
    };
    const long long my_len = run_len(warp);
    const bool ib1_ok = g + 4 < 2 * MR;
    int cfa = -1, cfb = 0, cfc = 0;
    float ax[2 * MR][2], ay[2 * MR][2];
#pragma unroll
    for (int a = 0; a < 2 * MR; ++a) ax[a][0] = ax[a][1] = ay[a][0] = ay[a][1] = 0.f;
    auto flush = [&]() {
        const int col = wrap(cfc - mc + 1 + k, n);
        const int rb0 = wrap(cfb - MR + 1 + g, n), rb1 = wrap(cfb - MR + 1 + g + 4, n);
#pragma unroll
        for (int a = 0; a < 2 * MR; ++a) {
            const int ra = wrap(cfa - MR + 1 + a, n) * n;
            if (g < 2 * MR) {
                float *cp = (float *)(S + (ra + rb0) * stride + col);
                red_add(cp, ax[a][0]);
                red_add(cp + 1, ay[a][0]);
            }
            if (ib1_ok) {
                float *cp = (float *)(S + (ra + rb1) * stride + col);
                red_add(cp, ax[a][1]);
                red_add(cp + 1, ay[a][1]);
            }
            ax[a][0] = ax[a][1] = ay[a][0] = ay[a][1] = 0.f;
        }
    };
    if (nblk > 0) stage_a(0);
    cp_async_commit();
    if (nblk > 1) stage_a(1);
    cp_async_commit();
    cp_async_wait1();
    if (nblk > 0) stage_b(0);
    cp_async_commit();
    for (long long c = 0; c < nblk; ++c) {
        cp_async_wait0();
        __syncthreads();
        if (c + 1 < nblk) stage_b(c + 1);
        cp_async_commit();
        if (c + 2 < nblk) stage_a(c + 2);
        cp_async_commit();
        const float4 *rb = rbuf + ((int)(c % 3) * SP3_BLK + warp * SP3_RUN) * 2;
        const float2 *yb = ybuf + (int)(c & 1) * SP3_BLK + warp * SP3_RUN;
        const long long left = my_len - c * SP3_RUN;
        for (int t = 0; t < SP3_RUN; ++t) {
            if (t >= left) break;   // warp-uniform
            const float4 q = rb[2 * t], qc = rb[2 * t + 1];
            const float cw = horner8(cc, q.z);
            const float wt = horner8(rcf, g == 0 ? q.x : q.y);   // lanes 0..7: first row, 8..15: second
            float wa[2 * MR];
#pragma unroll
            for (int a = 0; a < 2 * MR; ++a) wa[a] = __shfl_sync(0xffffffffu, wt, a);
            const float wb0 = __shfl_sync(0xffffffffu, wt, 8 + min(g, 2 * MR - 1));
            const float wb1 = __shfl_sync(0xffffffffu, wt, 8 + min(g + 4, 2 * MR - 1));
            const int fa = __float_as_int(qc.x), fb = __float_as_int(qc.y), fc = __float_as_int(qc.z);
            if (fa != cfa || fb != cfb || fc != cfc) {
                if (cfa >= 0) flush();
                cfa = fa;
                cfb = fb;
                cfc = fc;
            }
            const float2 yv = yb[t];
            const float yx = yv.x * cw, yy = yv.y * cw;
            const float u0x = yx * wb0, u0y = yy * wb0, u1x = yx * wb1, u1y = yy * wb1;
#pragma unroll
            for (int a = 0; a < 2 * MR; ++a) {
                ax[a][0] = fmaf(u0x, wa[a], ax[a][0]);
                ay[a][0] = fmaf(u0y, wa[a], ay[a][0]);
                ax[a][1] = fmaf(u1x, wa[a], ax[a][1]);
                ay[a][1] = fmaf(u1y, wa[a], ay[a][1]);
            }
        }
        __syncthreads();
    }
    cp_async_wait0();
    if (cfa >= 0) flush();
}

// Unsorted item (order 3, or a plan without sorted copies): the item's nodes
// in their original order, staged as float4 (first-row coordinate, last
// coordinate, y) one block ahead; every node adds its window to the shared
// grid with shared-memory atomics.
template <int MR, bool O3, int SP>
__device__ __forceinline__ void spread_unsorted_item(const DevPlan &P, const Term &T, const float2 *__restrict__ y,
                                                     long long j0, long long j1, float2 *S, unsigned char *stg_raw,
                                                     const float wcf[NCOEF]) {
    const int tid = threadIdx.x;
    const int lane = tid & 31, half = lane >> 4, sub = lane & 15;
    const int r = sub >> 3, k = sub & 7;
    const int warp = tid >> 5;
    constexpr int NW = SPREAD_THREADS / 32;
    const int order = T.order, n = T.n, stride = T.stride;
    const long long M = P.M;
    float4 *stage = (float4 *)stg_raw;   // [2][SP]
    const float *__restrict__ X = P.x;
    const float *xr = X + (long long)(order >= 2 ? T.row0 : T.col) * M;
    const float *xc = X + (long long)T.col * M;
    const float *xr1 = order == 3 ? X + (long long)T.row1 * M : nullptr;
    const long long nblk = (j1 - j0 + SP - 1) / SP;
    auto stage_block = [&](long long c, int buf) {
        const long long a = j0 + c * SP;
        const int cnt = (int)min((long long)SP, j1 - a);
        float4 *dst = stage + buf * SP;
        for (int e = tid; e < cnt; e += SPREAD_THREADS) {
            const long long j = a + e;
            cp_async4(&dst[e].x, xr + j);
            cp_async4(&dst[e].y, xc + j);
            cp_async8(&dst[e].z, y + j);
        }
    };
    if (nblk > 0) stage_block(0, 0);
    cp_async_commit();
    for (long long c = 0; c < nblk; ++c) {
        if (c + 1 < nblk) stage_block(c + 1, (int)((c + 1) & 1));
        cp_async_commit();
        cp_async_wait1();
        __syncthreads();
        const float4 *stg = stage + (int)(c & 1) * SP;
        const long long a = j0 + c * SP;
        const int cnt = (int)min((long long)SP, j1 - a);
        if (order == 2) {
            for (int i0 = 2 * warp; i0 < cnt; i0 += 2 * NW) {
                const int i = i0 + half;
                const bool ok = i < cnt;
                const float4 q = stg[ok ? i : i0];
                float ta, tb;
                const int fa = grid_pos(q.x, n, ta);
                const int fb = grid_pos(q.y, n, tb);
                float cw, w[MR];
                node_weights<MR>(wcf, 2.f * ta - 1.f, 2.f * tb - 1.f, half, r, k, cw, w);
                const float yx = q.z * cw, yy = q.w * cw;
                float *base = (float *)(S + (fa + r) * stride + fb + k);
                if (ok) {
#pragma unroll
                    for (int j = 0; j < MR; ++j) {
                        red_add(base + 4 * j * stride, yx * w[j]);
                        red_add(base + 4 * j * stride + 1, yy * w[j]);
                    }
                }
            }
        } else if (order == 1) {
            const int g = tid >> 3;
            for (int i = g; i < cnt; i += SPREAD_THREADS / 8) {
                const float4 q = stg[i];
                float tb;
                const int fb = grid_pos(q.y, n, tb);
                const float cw = horner8(wcf, 2.f * tb - 1.f);
                float *base = (float *)(S + fb + k);
                red_add(base, q.z * cw);
                red_add(base + 1, q.w * cw);
            }
        } else if constexpr (O3) {
            // order 3: rows wrap modulo n; row weights from the per-tap
            // polynomials, lane (0, k) the first row coordinate's tap k, lane
            // (1, k) the second's, handed round by shuffles (the whole warp
            // iterates together; a half-warp past the end adds nothing)
            float rcf[NCOEF];
            {
                const float *src = P.windows[T.wr].c[min(k, 2 * MR - 1)];
#pragma unroll
                for (int q = 0; q < NCOEF; ++q) rcf[q] = __ldg(src + q);
            }
            const int mc = T.mc;
            for (int i0 = 2 * warp; i0 < cnt; i0 += 2 * NW) {
                const int i = i0 + half;
                const bool ok = i < cnt;
                const int ii = ok ? i : i0;
                const float4 q = stg[ii];
                float ta, tb, tc;
                const int fa = grid_pos(q.x, n, ta);
                const int fb = grid_pos(__ldg(xr1 + a + ii), n, tb);
                const int fc = grid_pos(q.y, n, tc);
                const float cw = horner8(wcf, 2.f * tc - 1.f);
                const float wrow = horner8(rcf, r ? 2.f * tb - 1.f : 2.f * ta - 1.f);
                float wa[2 * MR], wb[MR];
#pragma unroll
                for (int t = 0; t < 2 * MR; ++t) wa[t] = __shfl_sync(0xffffffffu, wrow, (half << 4) | t);
#pragma unroll
                for (int j = 0; j < MR; ++j) wb[j] = __shfl_sync(0xffffffffu, wrow, (half << 4) | 8 | (r + 2 * j));
                if (!ok) continue;
                const int cidx = wrap(fc - mc + 1 + k, n);
                const float yx = q.z * cw, yy = q.w * cw;
#pragma unroll
                for (int ia = 0; ia < 2 * MR; ++ia) {
                    const int row = wrap(fa - MR + 1 + ia, n) * n;
                    const float ax = yx * wa[ia], ay = yy * wa[ia];
#pragma unroll
                    for (int j = 0; j < MR; ++j) {
                        const int rbj = wrap(fb - MR + 1 + r + 2 * j, n);
                        float *cp = (float *)(S + (row + rbj) * stride + cidx);
                        red_add(cp, ax * wb[j]);
                        red_add(cp + 1, ay * wb[j]);
                    }
                }
            }
        }
        __syncthreads();
    }
    cp_async_wait0();
}

// One work item (x = problem, y = active term, z = node chunk, w = chunks per
// term) spreads nodes [M z / w, M (z+1) / w) of one term (in the term's cell
// order if the plan keeps sorted copies and the term has order <= 2, else in
// the original order) into a shared-memory copy of the term's stored grid
// (halos included) and writes it to partial grid z of its problem.  CTAs take
// items from a global counter.  O3: third-order items.
template <int MR, typename G, bool O3, int SP>
__device__ __forceinline__ void spread_items(const DevPlan &single, const BatchArgs &B,
                                             const float2 *__restrict__ y_base, int item_begin, int item_end,
                                             int *counter, long long max_grid_bytes) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2 *S = (float2 *)smem_raw;
    unsigned char *stg_raw = smem_raw + max_grid_bytes;
    constexpr int NT = SPREAD_THREADS;
    int &s_item = *(int *)(stg_raw + (O3 ? SP3_STAGE_BYTES : sp_stage_bytes(SP)));
    const int tid = threadIdx.x;
    const int k = tid & 7;
    for (;;) {
        if (tid == 0) s_item = item_begin + atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= item_end) break;
        const int4 itm = B.items[item];
        const DevPlan &P = B.plans ? B.plans[itm.x] : single;
        if (P.skip && *P.skip) continue;
        const Term &T = P.terms[P.act[itm.y]];
        const long long M = P.M;
        const long long j0 = M * itm.z / itm.w, j1 = M * (itm.z + 1) / itm.w;
        const long long elems = T.grid_bytes / (long long)sizeof(G);   // shared copy is FP32 complex
        float4 *S4 = (float4 *)S;
        for (long long e = tid; e < elems / 2; e += NT) S4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        const float2 *y = y_base + P.vec_node_off;
        // window coefficients of this lane: row tap k for lanes r = 1 of an
        // order-2 term (see node_weights), column tap k otherwise
        float wcf[NCOEF];
        {
            const bool row = T.order == 2 && (tid & 8);
            const float *wsrc = row ? P.windows[T.wr].c[min(k, 2 * MR - 1)] : P.windows[T.wc].c[k];
#pragma unroll
            for (int i = 0; i < NCOEF; ++i) wcf[i] = __ldg(wsrc + i);
        }
        // in a batch whose problems differ in form, a problem may hold node tiles, which
        // only the tensor-core kernels read
        const bool sorted = T.sort_slot >= 0 && P.srec && !P.tile_cell;
        __syncthreads();   // grid zeroed before any addition
        if constexpr (O3) {
            if (sorted)
                spread_sorted_item3<MR>(P, T, y, j0, j1, S, stg_raw, wcf);
            else
                spread_unsorted_item<MR, true, SP>(P, T, y, j0, j1, S, stg_raw, wcf);
        } else {
            if (sorted)
                spread_sorted_item<MR, SP>(P, T, y, j0, j1, S, stg_raw, wcf);
            else
                spread_unsorted_item<MR, false, SP>(P, T, y, j0, j1, S, stg_raw, wcf);
        }
        __syncthreads();
        if constexpr (std::is_same<G, float2>::value) {
            float4 *dst = (float4 *)(P.partials + (long long)itm.z * P.grid_elems + T.grid_off);
            for (long long e = tid; e < elems / 2; e += NT) dst[e] = S4[e];
        } else {
            G *dst = (G *)P.partials + (long long)itm.z * P.grid_elems + T.grid_off;
            for (long long e = tid; e < elems; e += NT) dst[e] = GridEl<G>::store(S[e].x, S[e].y);
        }
        __syncthreads();
    }
}

// the order-1/2 items (3 CTAs per SM) and the third-order items (more
// registers for the 2 x 2 m_row row-pair sums, 2 CTAs per SM)
template <int MR, typename G, int SP>
__global__ void __launch_bounds__(SPREAD_THREADS, SP == SP_CH ? 3 : SPREAD_MAX_CTAS_PER_SM)
spread_f32(DevPlan single, BatchArgs B, const float2 *__restrict__ y_base, int item_begin, int item_end,
           int *counter, long long max_grid_bytes) {
    spread_items<MR, G, false, SP>(single, B, y_base, item_begin, item_end, counter, max_grid_bytes);
}

template <int MR, typename G>
__global__ void __launch_bounds__(SPREAD_THREADS, 2)
spread3_f32(DevPlan single, BatchArgs B, const float2 *__restrict__ y_base, int item_begin, int item_end,
            int *counter, long long max_grid_bytes) {
    spread_items<MR, G, true, SP_CH / 2>(single, B, y_base, item_begin, item_end, counter, max_grid_bytes);
}

template <typename G>
__global__ void reduce_partials_f32(DevPlan single, BatchArgs B) {
    const DevPlan &P = B.plans ? B.plans[blockIdx.y] : single;
    if (P.skip && *P.skip) return;
    const int nparts = P.spread_chunks;
    if constexpr (std::is_same<G, float2>::value) {
        const float4 *__restrict__ partials = (const float4 *)P.partials;
        float4 *__restrict__ out = (float4 *)P.grids;
        const long long n4 = P.grid_elems / 2, pstride4 = n4;
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4;
             i += (long long)gridDim.x * blockDim.x) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int c = 0; c < nparts; ++c) {
                float4 v = __ldg(partials + (long long)c * pstride4 + i);
                a.x += v.x;
                a.y += v.y;
                a.z += v.z;
                a.w += v.w;
            }
            out[i] = a;
        }
    } else {
        // 16-bit partials and grid: widen, sum in FP32, round once
        const G *__restrict__ partials = (const G *)P.partials;
        G *__restrict__ out = (G *)P.grids;
        const long long ne = P.grid_elems;
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < ne;
             i += (long long)gridDim.x * blockDim.x) {
            float ax = 0.f, ay = 0.f;
            for (int c = 0; c < nparts; ++c) {
                const float2 v = GridEl<G>::load(partials[(long long)c * ne + i]);
                ax += v.x;
                ay += v.y;
            }
            out[i] = GridEl<G>::store(ax, ay);
        }
    }
}

// the empty-set coefficients from the partial sums of y (one block)
__device__ __forceinline__ void sum_y_finish(const DevPlan &P, const double2 *part, int nparts, float2 *fhat_base) {
    __shared__ double sh[32];
    if (P.n_empty == 0 || (P.skip && *P.skip)) return;
    double sx = 0, sy = 0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) {
        sx += part[i].x;
        sy += part[i].y;
    }
    sx = block_sum_fixed(sx, sh);
    sy = block_sum_fixed(sy, sh);
    if (threadIdx.x != 0) return;
    float2 *fhat = fhat_base + P.vec_coef_off;
    for (int e = 0; e < P.n_empty; ++e) fhat[P.empty_off[e]] = make_float2((float)sx, (float)sy);
}

// One block per active term, and behind them one block per problem that adds
// the empty-set coefficient's partial sums and, in block 0, returns the work
// counters to zero.  With nparts > 0 the FP32 partial grids are summed (in
// chunk order) while the halos are folded, which saves the reduction's launch
// and its pass over the grid; many chunks per term read faster spread over the
// whole chip (reduce_partials_f32, then nparts = 0).
template <typename G>
__global__ void __launch_bounds__(FFT_THREADS)
adjoint_post_f32(DevPlan single, BatchArgs B, float2 *__restrict__ fhat_base, int n_blocks, int *counter,
                 bool fuse_reduce, const double2 *y_part, int n_ypart) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    if (blockIdx.x == 0 && threadIdx.x < 2) counter[threadIdx.x] = 0;
    if ((int)blockIdx.x >= n_blocks) {
        const int p = (int)blockIdx.x - n_blocks;
        sum_y_finish(B.plans ? B.plans[p] : single, y_part + (long long)p * n_ypart, n_ypart, fhat_base);
        return;
    }
    const int pb = B.plans ? B.blk_prob[blockIdx.x] : 0;
    const DevPlan &P = B.plans ? B.plans[pb] : single;
    const int sblk = B.plans ? (int)blockIdx.x - B.blk0[pb] : (int)blockIdx.x;
    if (P.skip && *P.skip) return;
    if (sblk == 0 && threadIdx.x == 0) P.err[ERR_YMAX] = 0;
    float2 *__restrict__ fhat = fhat_base + P.vec_coef_off;
    const Term T = P.terms[P.act[sblk]];
    const int n = T.n, s = T.order, N = T.N;
    int fe = n;
    for (int j = 1; j < s; ++j) fe *= n;
    float2 *a = (float2 *)smem_raw;
    float2 *b = a + fe;
    // fold the stored (halo) grid onto the periodic grid
    if (fuse_reduce) {
        const float4 *g = (const float4 *)(P.partials + T.grid_off);
        const int K = P.spread_chunks;
        const long long pstride = P.grid_elems / 2;
        fold_halo(T, a, b, fe, [&](int i, float2 &v0, float2 &v1) {
            v0 = v1 = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int c = 0; c < K; ++c) {
                const float4 u = __ldg(g + c * pstride + i);
                v0.x += u.x;
                v0.y += u.y;
                v1.x += u.z;
                v1.y += u.w;
            }
        });
    } else {
        const G *g = (const G *)P.grids + T.grid_off;
        fold_halo(T, a, b, fe, [&](int i, float2 &v0, float2 &v1) {
            v0 = GridEl<G>::load(g[2 * i]);
            v1 = GridEl<G>::load(g[2 * i + 1]);
        });
    }
    // FFT along every axis, sign -
    const float2 *cur = grid_fft<float2, float>(a, b, n, s, -1);
    // crop and deconvolve
    const int len = (int)T.coef_len;
    if (T.basis == ANOVA_BASIS_COS) {
        // cosine term: 2^{-s/2} times the sum over its 2^s mirrored frequencies
        for (int q = threadIdx.x; q < len; q += blockDim.x) {
            int k[3];
            cos_decode(q, s, N, k);
            float sx = 0.f, sy = 0.f;
            for (int sg = 0; sg < (1 << s); ++sg) {
                float D = (float)cos_amp(s);
                const float2 v = cur[cos_mirror(k, s, sg, N, n, P.deconv, T.dc_off, T.dr_off, D)];
                sx = fmaf(v.x, D, sx);
                sy = fmaf(v.y, D, sy);
            }
            fhat[T.coef_off + q] = make_float2(sx, sy);
        }
        return;
    }
    const FastDiv by_Nm(N - 1);
    for (int q = threadIdx.x; q < len; q += blockDim.x) {
        float D;
        const float2 v = cur[exp_position(q, s, N, n, by_Nm, P.deconv, T.dc_off, T.dr_off, D)];
        fhat[T.coef_off + q] = make_float2(v.x * D, v.y * D);
    }
}

// partial sums of y for the empty-set coefficients, one per block (of the
// problem blockIdx.y), which adjoint_post_f32 adds; with find_max also the
// largest |Re|, |Im| of y as float bits (NaN above all), for the scale of the
// third-order terms' FP16 operands
__global__ void sum_y_partial(DevPlan single, BatchArgs B, const float2 *__restrict__ y_base, double2 *part_base,
                              bool find_max) {
    __shared__ double sh[32];
    const DevPlan &P = B.plans ? B.plans[blockIdx.y] : single;
    if (P.skip && *P.skip) return;
    const float2 *__restrict__ y = y_base + P.vec_node_off;
    double sx = 0, sy = 0;
    unsigned m = 0u;
    const long long M = P.M, step = (long long)gridDim.x * blockDim.x;
#pragma unroll 4
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < M; i += step) {
        const float2 v = __ldg(y + i);
        sx += v.x;
        sy += v.y;
        m = max(m, max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu));
    }
    if (find_max) {
        m = __reduce_max_sync(0xffffffffu, m);
        if ((threadIdx.x & 31) == 0 && m) atomicMax((unsigned *)P.err + ERR_YMAX, m);
    }
    if (P.n_empty == 0) return;
    sx = block_sum_fixed(sx, sh);
    sy = block_sum_fixed(sy, sh);
    if (threadIdx.x == 0) part_base[(long long)blockIdx.y * gridDim.x + blockIdx.x] = make_double2(sx, sy);
}

template <typename G>
static void adjoint_attrs() {
    static std::atomic<unsigned long long> attr_seen{0};
    once_per_device(attr_seen, [] {
        cudaFuncSetAttribute(adjoint_post_f32<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, FFT_MAX_SMEM);
        cudaFuncSetAttribute(spread_f32<3, G, SP_CH>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
        cudaFuncSetAttribute(spread_f32<4, G, SP_CH>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
        cudaFuncSetAttribute(spread_f32<3, G, SP_CH / 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
        cudaFuncSetAttribute(spread_f32<4, G, SP_CH / 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
        cudaFuncSetAttribute(spread3_f32<3, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
        cudaFuncSetAttribute(spread3_f32<4, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM);
    });
}

// spread + reduce + post for grids stored as G; sgrid = bytes of the largest
// grid in FP32 (the spread's shared-memory copy).  n_ypart > 0: partial sums of
// y for the empty set wait in y_part.
template <typename G>
static void adjoint_kernels(Plan *prof, cudaStream_t st, const DevPlan &v, const BatchArgs &B, int P,
                            const float2 *y, float2 *fhat, int n_items, int n_items3, int *counter, int n_blocks,
                            int mr, long long sgrid, int max_fft_elems, int max_n, int max_stage, int sm_count,
                            long long max_grid_elems, int max_chunks, const double2 *y_part, int n_ypart, int prec,
                            bool tc) {
    adjoint_attrs<G>();
    if (n_blocks > 0) {
        if (prof) stage_begin(*prof, ST_SPREAD);
        const int sp = spread_block_nodes(sgrid), per_sm = spread_ctas_per_sm(sgrid);
        if (tc) {
            spread_tiles_launch(st, v, B, y, n_items, n_items3 > 0, counter, sgrid, sm_count, mr, prec);
        } else if (n_items3 > 0) {
            const int c3 = std::max(1, std::min(n_items3, std::min(per_sm, 2) * sm_count));
            auto k = mr <= 3 ? spread3_f32<3, G> : spread3_f32<4, G>;
            k<<<c3, SPREAD_THREADS, spread_smem_bytes(sgrid, true, sp), st>>>(v, B, y, 0, n_items3, counter, sgrid);
        }
        if (!tc && n_items > n_items3) {
            const int c = std::max(1, std::min(n_items - n_items3, per_sm * sm_count));
            auto k = mr <= 3 ? (sp == SP_CH ? spread_f32<3, G, SP_CH> : spread_f32<3, G, SP_CH / 2>)
                             : (sp == SP_CH ? spread_f32<4, G, SP_CH> : spread_f32<4, G, SP_CH / 2>);
            k<<<c, SPREAD_THREADS, spread_smem_bytes(sgrid, false, sp), st>>>(v, B, y, n_items3, n_items, counter + 1,
                                                                             sgrid);
        }
        if (prof) stage_end(*prof, ST_SPREAD);
    }
    const bool fuse = std::is_same<G, float2>::value && max_chunks <= POST_MAX_CHUNKS;
    if (n_blocks > 0 && !fuse) {
        const long long n4 = max_grid_elems / 2;
        const int rb =
            (int)std::max<long long>(1, std::min<long long>(sm_count * 8LL / std::max(1, P) + 1, (n4 + 255) / 256));
        if (prof) stage_begin(*prof, ST_REDUCE);
        reduce_partials_f32<G><<<dim3(rb, P), 256, 0, st>>>(v, B);
        if (prof) stage_end(*prof, ST_REDUCE);
    }
    const int blocks = n_blocks + (n_ypart > 0 ? P : 0);
    if (blocks == 0) return;
    if (prof) stage_begin(*prof, ST_POST);
    adjoint_post_f32<G><<<blocks, FFT_THREADS, fft_smem_bytes<float2>(max_fft_elems, max_n, max_stage), st>>>(
        v, B, fhat, n_blocks, counter, fuse, y_part, n_ypart);
    if (prof) stage_end(*prof, ST_POST);
}

// The adjoint kernels for one problem (B.plans == null) or a batch of P problems.
int adjoint_launch(Plan *prof, cudaStream_t st, const DevPlan &v, const BatchArgs &B, int P, const float2 *y,
                   float2 *fhat, int n_items, int n_items3, int *counter, int n_blocks, int mr,
                   long long max_grid_bytes, int max_fft_elems, int max_n, int max_stage, int sm_count, long long max_grid_elems,
                   int max_chunks, bool any_empty, double2 *scratch, int prec, bool tc) {
    const bool find_max = tc && n_items3 > 0;
    // enough blocks to fill the chip, shared among the problems
    const int ny = std::max(32, SUM_Y_BLOCKS / P), n_ypart = any_empty ? ny : 0;
    if (any_empty || find_max) {
        if (prof) stage_begin(*prof, ST_SUMY);
        sum_y_partial<<<dim3(ny, P), 256, 0, st>>>(v, B, y, scratch, find_max);
        if (prof) stage_end(*prof, ST_SUMY);
    }
    auto run = prec == ANOVA_PREC_F16    ? adjoint_kernels<__half2>
               : prec == ANOVA_PREC_BF16 ? adjoint_kernels<__nv_bfloat162>
                                         : adjoint_kernels<float2>;
    const long long sgrid = prec == ANOVA_PREC_F32 ? max_grid_bytes : 2 * max_grid_bytes;
    run(prof, st, v, B, P, y, fhat, n_items, n_items3, counter, n_blocks, mr, sgrid, max_fft_elems, max_n, max_stage,
        sm_count, max_grid_elems, max_chunks, scratch, n_ypart, prec, tc);
    return cuda_status(cudaGetLastError());
}

int launch_adjoint_f32(Plan &p, const float2 *y, float2 *fhat) {
    if (p.direct) return launch_direct_adjoint(p, y, fhat);
    DevPlan v = dev_view(p);
    BatchArgs B;
    std::memset(&B, 0, sizeof(B));
    B.items = p.items;
    if (p.M == 0) {
        cudaMemsetAsync(fhat, 0, sizeof(float2) * p.n_coeffs, p.stream);
        return cuda_status(cudaGetLastError());
    }
    int mr = 3;
    for (int s = 0; s < p.n_terms; ++s) mr = p.h_terms[s].mr > 0 ? p.h_terms[s].mr : mr;
    return adjoint_launch(&p, p.stream, v, B, 1, y, fhat, p.n_items, p.n_items3, p.counter, p.n_act, mr,
                          p.max_grid_bytes, p.max_fft_elems, p.max_n, p.max_stage, p.sm_count, p.grid_elems, p.spread_K, p.n_empty > 0,
                          (double2 *)p.scratch, p.precision, p.srec && p.cell_tc);
}

}  // namespace agft
