// Nodes sorted by grid cell, per term of order <= 2 (built once per plan).
//
// The adjoint spreads y_j psi(n x_j - l) onto the oversampled grid of every
// term (stacked adjoint after the error remark, Sec. 3).  Nodes whose grid
// position has the same integer part (the same cell) touch the same window
// footprint, so with the nodes of a term in cell order the spread sums a
// cell's contributions in registers and adds them to the grid once per cell.
// This file builds that order: a counting sort of the node indices by cell,
// one term per blockIdx.y, and per sorted node a 16-byte record with the
// window arguments, the grid offset of its cell and its original index.
// The order inside a cell is left to the atomics of the scatter; it changes
// only the rounding order of the sums.  FP64 plans sort by the bases of their
// window tables (records carry only the cell offset and the node index).
#include <algorithm>

#include "device.cuh"
#include "internal.cuh"
#include "tiles.cuh"

namespace agft {

__device__ __forceinline__ int cell_bins(const Term &T) {
    return T.order == 3 ? T.n * T.n * T.n : (T.order == 2 ? T.n * T.n : T.n);
}

// cell of a node: (i_row0 * n + i_row1) * n + i_col over the term's coordinates
__device__ __forceinline__ int cell_of(const Term &T, float xr, float xr1, float xc) {
    float t;
    const int fc = grid_pos(xc, T.n, t);
    if (T.order == 1) return fc;
    const int fr = grid_pos(xr, T.n, t);
    if (T.order == 2) return fr * T.n + fc;
    const int fr1 = grid_pos(xr1, T.n, t);
    return (fr * T.n + fr1) * T.n + fc;
}

// counts[slot][cell] += nodes of the block's range in that cell
__global__ void k_cell_count(const Term *terms, const float *x, long long M, int *counts, int max_bins) {
    extern __shared__ int hist[];
    const Term &T = terms[blockIdx.y];
    if (T.sort_slot < 0) return;
    const int nb = cell_bins(T);
    for (int b = threadIdx.x; b < nb; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    const float *xr = x + (long long)(T.order >= 2 ? T.row0 : T.col) * M;
    const float *xr1 = x + (long long)(T.order == 3 ? T.row1 : T.col) * M;
    const float *xc = x + (long long)T.col * M;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < M; j += (long long)gridDim.x * blockDim.x)
        atomicAdd(&hist[cell_of(T, xr[j], xr1[j], xc[j])], 1);
    __syncthreads();
    int *cnt = counts + (long long)T.sort_slot * max_bins;
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        if (hist[b]) atomicAdd(&cnt[b], hist[b]);
}

// exclusive prefix sum of counts[slot][0..bins) in place, one block per term
__global__ void k_cell_scan(const Term *terms, int *counts, int max_bins) {
    __shared__ int wsum[32];
    const Term &T = terms[blockIdx.x];
    if (T.sort_slot < 0) return;
    const int nb = cell_bins(T);
    int *c = counts + (long long)T.sort_slot * max_bins;
    const int per = (nb + blockDim.x - 1) / blockDim.x;
    const int b0 = min(nb, (int)threadIdx.x * per), b1 = min(nb, b0 + per);
    int local = 0;
    for (int b = b0; b < b1; ++b) local += c[b];
    // inclusive scan of the per-thread sums across the block
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int v = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) wsum[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    int run = v - local + (wid > 0 ? wsum[wid - 1] : 0);   // exclusive prefix of this thread's range
    for (int b = b0; b < b1; ++b) {
        const int t = c[b];
        c[b] = run;
        run += t;
    }
}

// scatter: every node goes to the next free place of its cell, as a record.
// Order <= 2: (2 tau_row - 1, 2 tau_col - 1, first-tap grid offset, original
// index).  Order 3, two records: (2 tau_row0 - 1, 2 tau_row1 - 1, 2 tau_col - 1,
// original index) and the cell's grid indices and cell number (i_row0, i_row1,
// i_col, (i_row0 n + i_row1) n + i_col).
__global__ void k_cell_scatter(const Term *terms, const float *x, long long M, int *cursor, int max_bins,
                               float4 *srec) {
    const Term &T = terms[blockIdx.y];
    if (T.sort_slot < 0) return;
    const float *xr = x + (long long)(T.order >= 2 ? T.row0 : T.col) * M;
    const float *xr1 = x + (long long)(T.order == 3 ? T.row1 : T.col) * M;
    const float *xc = x + (long long)T.col * M;
    int *cur = cursor + (long long)T.sort_slot * max_bins;
    float4 *dst = srec + (long long)T.sort_slot * M;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < M;
         j += (long long)gridDim.x * blockDim.x) {
        float tc, tr = 0.f, tr1 = 0.f;
        const int fc = grid_pos(xc[j], T.n, tc);
        int fr = 0, fr1 = 0;
        if (T.order >= 2) fr = grid_pos(xr[j], T.n, tr);
        if (T.order == 3) fr1 = grid_pos(xr1[j], T.n, tr1);
        if (T.order == 3) {
            const int pos = atomicAdd(&cur[(fr * T.n + fr1) * T.n + fc], 1);
            dst[2 * pos] = make_float4(2.f * tr - 1.f, 2.f * tr1 - 1.f, 2.f * tc - 1.f, __int_as_float((int)j));
            dst[2 * pos + 1] = make_float4(__int_as_float(fr), __int_as_float(fr1), __int_as_float(fc),
                                           __int_as_float((fr * T.n + fr1) * T.n + fc));
        } else {
            const int pos = atomicAdd(&cur[fr * (T.order == 2 ? T.n : 0) + fc], 1);
            const int off = fr * T.stride + fc;
            dst[pos] = make_float4(T.order == 2 ? 2.f * tr - 1.f : 0.f, 2.f * tc - 1.f, __int_as_float(off),
                                   __int_as_float((int)j));
        }
    }
}

// FP64 plans: the cell of a node is that of its window-table bases (the
// spread adds at exactly those bases); records (0, 0, offset, index)
__device__ __forceinline__ int cell_of64(const Term &T, const int *wb, long long M, long long j, int &off) {
    const int fc = wb[(long long)T.slot_c * M + j];
    if (T.order != 2) {
        off = fc;
        return fc;
    }
    const int fr = wb[(long long)T.slot_r0 * M + j];
    off = fr * T.stride + fc;
    return fr * T.n + fc;
}

__global__ void k_cell_count64(const Term *terms, const int *wb, long long M, int *counts, int max_bins) {
    extern __shared__ int hist[];
    const Term &T = terms[blockIdx.y];
    if (T.sort_slot < 0) return;
    const int nb = cell_bins(T);
    for (int b = threadIdx.x; b < nb; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < M; j += (long long)gridDim.x * blockDim.x) {
        int off;
        atomicAdd(&hist[cell_of64(T, wb, M, j, off)], 1);
    }
    __syncthreads();
    int *cnt = counts + (long long)T.sort_slot * max_bins;
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        if (hist[b]) atomicAdd(&cnt[b], hist[b]);
}

__global__ void k_cell_scatter64(const Term *terms, const int *wb, long long M, int *cursor, int max_bins,
                                 float4 *srec) {
    const Term &T = terms[blockIdx.y];
    if (T.sort_slot < 0) return;
    int *cur = cursor + (long long)T.sort_slot * max_bins;
    float4 *dst = srec + (long long)T.sort_slot * M;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < M;
         j += (long long)gridDim.x * blockDim.x) {
        int off;
        const int pos = atomicAdd(&cur[cell_of64(T, wb, M, j, off)], 1);
        dst[pos] = make_float4(0.f, 0.f, __int_as_float(off), __int_as_float((int)j));
    }
}

// ---- node tiles (tiles.cuh) ----
//
// A counting sort per term with the node range cut into S slices, one block
// each.  The blocks' histograms are kept, and the scan turns them into every
// block's first place in every cell, so that the scatter counts in shared memory
// only.  Scattered writes are what bounds it: they run at DRAM speed in partial
// sectors once the terms in work outgrow L2.  So for order <= 2 a block first sorts
// its slice's node numbers in shared memory and writes them by cells, runs of 15 at
// d = 20, M = 1e6, where a write per node took 4.8 ms instead of 1.4; only the
// 4-byte indices are written, and a second pass, in tile order, reads the coordinates
// through L2 and writes whole lines.
constexpr int SORT_THREADS = 512;

__device__ __forceinline__ int tile_bin(const Term &T, int fr, int fr1, int fc) {
    return T.order == 3 ? (fr1 * T.n + fc) * T.n + fr : (T.order == 2 ? fr * T.n + fc : fc);
}

// hist[(term S + slice) max_bins + cell] = nodes of the slice in the cell
__global__ void __launch_bounds__(SORT_THREADS)
k_tile_count(const Term *terms, const float *x, long long M, int *hist, int max_bins) {
    extern __shared__ int bins[];
    const Term &T = terms[blockIdx.y];
    const int nb = cell_bins(T), S = gridDim.x, n = T.n, order = T.order;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) bins[b] = 0;
    __syncthreads();
    const float *xr = x + (long long)(order >= 2 ? T.row0 : T.col) * M;
    const float *xr1 = x + (long long)(order == 3 ? T.row1 : T.col) * M;
    const float *xc = x + (long long)T.col * M;
    const long long j1 = M * (blockIdx.x + 1) / S;
    for (long long j = M * blockIdx.x / S + threadIdx.x; j < j1; j += blockDim.x) {
        float t;
        const int fc = grid_pos(xc[j], n, t);
        const int fr = order >= 2 ? grid_pos(xr[j], n, t) : 0, fr1 = order == 3 ? grid_pos(xr1[j], n, t) : 0;
        atomicAdd(&bins[tile_bin(T, fr, fr1, fc)], 1);
    }
    __syncthreads();
    int *out = hist + ((long long)blockIdx.y * S + blockIdx.x) * max_bins;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) out[b] = bins[b];
}

constexpr int SORT_MAX_SLICES = 16;

// One block per term: first places of every slice in every cell (in place of the
// histograms), (first tile, nodes) of every cell and the number of tiles.
__global__ void __launch_bounds__(1024) k_tile_scan(const Term *terms, int *hist, int S, int max_bins, int2 *cell_info,
                                                    int *tile_count) {
    __shared__ int wsum[32];
    const Term &T = terms[blockIdx.x];
    const int nb = cell_bins(T);
    int *h = hist + (long long)blockIdx.x * S * max_bins;
    int2 *info = cell_info + (long long)blockIdx.x * max_bins;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int carry = 0;
    for (int b0 = 0; b0 < nb; b0 += blockDim.x) {
        const int b = b0 + threadIdx.x;
        int k[SORT_MAX_SLICES], count = 0;
#pragma unroll
        for (int s = 0; s < SORT_MAX_SLICES; ++s) k[s] = s < S && b < nb ? h[(long long)s * max_bins + b] : 0;
#pragma unroll
        for (int s = 0; s < SORT_MAX_SLICES; ++s) count += k[s];
        const int tiles = (count + TILE - 1) / TILE;
        int v = tiles;   // inclusive scan across the block
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) wsum[wid] = v;
        __syncthreads();
        if (wid == 0) {
            int w = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += u;
            }
            wsum[lane] = w;
        }
        __syncthreads();
        const int tile0 = carry + v - tiles + (wid > 0 ? wsum[wid - 1] : 0);
        carry += wsum[31];
        __syncthreads();   // wsum is read before the next round
        if (b >= nb) continue;
        info[b] = make_int2(tile0, count);
        int place = tile0 * TILE;
#pragma unroll
        for (int s = 0; s < SORT_MAX_SLICES; ++s) {
            if (s < S) h[(long long)s * max_bins + b] = place;
            place += k[s];
        }
    }
    if (threadIdx.x == 0) tile_count[blockIdx.x] = carry;
}

// the tiles' cells and the padding of the block's share of a term's cells
template <typename Pad>
__device__ __forceinline__ void tile_cells(const Term &T, int nb, const int2 *info, int *cells, Pad pad) {
    const int n = T.n, S = gridDim.x, b1 = (int)((long long)nb * (blockIdx.x + 1) / S);
    for (int b = (int)((long long)nb * blockIdx.x / S) + threadIdx.x; b < b1; b += blockDim.x) {
        const int2 c = info[b];   // first tile, nodes
        int cell = b;
        if (T.order == 2) cell = b / n * T.stride + b % n;
        if (T.order == 3) cell = b % n | b / (n * n) << 8 | b / n % n << 16;   // a, b, c
        for (int i = 0; i * TILE < c.y; ++i) cells[c.x + i] = cell | (c.y - i * TILE <= TILE / 2 ? TILE_HALF : 0);
        for (int k = c.y; k % TILE; ++k) pad(c.x * TILE + k);
    }
}

// order 3: the slice's nodes to their places
__global__ void __launch_bounds__(SORT_THREADS)
k_tile_scatter(const Term *terms, const float *x, long long M, const int *hist, const int2 *cell_info, int max_bins,
               float4 *srec, int *tile_cell) {
    extern __shared__ int bins[];
    const Term &T = terms[blockIdx.y];
    if (T.order != 3) return;
    const int nb = cell_bins(T), S = gridDim.x, n = T.n;
    const int *in = hist + ((long long)blockIdx.y * S + blockIdx.x) * max_bins;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) bins[b] = in[b];
    __syncthreads();
    const float *xr = x + (long long)T.row0 * M, *xr1 = x + (long long)T.row1 * M, *xc = x + (long long)T.col * M;
    float4 *rec = srec + T.rec_off;
    const long long j1 = M * (blockIdx.x + 1) / S;
    for (long long j = M * blockIdx.x / S + threadIdx.x; j < j1; j += blockDim.x) {
        float tc, tr, tr1;
        const int fc = grid_pos(xc[j], n, tc), fr = grid_pos(xr[j], n, tr), fr1 = grid_pos(xr1[j], n, tr1);
        const int pos = atomicAdd(&bins[tile_bin(T, fr, fr1, fc)], 1);
        rec[pos] = make_float4(2.f * tr - 1.f, 2.f * tr1 - 1.f, 2.f * tc - 1.f, __int_as_float((int)j));
    }
    tile_cells(T, nb, cell_info + (long long)blockIdx.y * max_bins, tile_cell + T.tile_off,
               [&](int pos) { rec[pos] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1)); });
}

// order <= 2: the slice's node numbers to their places, in parts of at most `cap`
// nodes (16-bit numbers) that are sorted by cell in shared memory: [cells] ends of the
// part's runs, [cells] next places, [cap] numbers.  A slice of one part takes its counts
// from the histograms.
constexpr int PLACE_THREADS = 1024, PLACE_MAX = 65536;
__global__ void __launch_bounds__(PLACE_THREADS)
k_tile_place(const Term *terms, const float *x, long long M, const int *hist, const int2 *cell_info, int max_bins,
             int place_bins, int cap, float4 *srec, int *tile_cell) {
    extern __shared__ int sm[];
    __shared__ int wsum[32];
    const Term &T = terms[blockIdx.y];
    if (T.order == 3) return;
    const int nb = cell_bins(T), S = gridDim.x, n = T.n, order = T.order, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int *ends = sm, *place = sm + place_bins;
    unsigned short *list = (unsigned short *)(place + place_bins);
    const int *in = hist + ((long long)blockIdx.y * S + blockIdx.x) * max_bins;
    const int2 *info = cell_info + (long long)blockIdx.y * max_bins;
    const float *xr = x + (long long)(order >= 2 ? T.row0 : T.col) * M, *xc = x + (long long)T.col * M;
    int *out = (int *)(srec + T.rec_off + 8);   // indices of tile 0
    auto put = [&](int pos, int id) { out[(long long)(pos >> 4) * (tile_f4(2) * 4) + (pos & 7) * 2 + ((pos >> 3) & 1)] = id; };
    const long long j0 = M * blockIdx.x / S, len = M * (blockIdx.x + 1) / S - j0;
    const int parts = (int)((len + cap - 1) / cap);
    for (int b = tid; b < nb; b += PLACE_THREADS) place[b] = in[b];
    for (int c = 0; c < parts; ++c) {
        const long long a = j0 + len * c / parts;
        const int m = (int)(j0 + len * (c + 1) / parts - a);
        auto bin = [&](int i) {
            float t;
            const int fc = grid_pos(xc[a + i], n, t), fr = order >= 2 ? grid_pos(xr[a + i], n, t) : 0;
            return tile_bin(T, fr, 0, fc);
        };
        if (parts == 1) {
            for (int b = tid; b < nb; b += PLACE_THREADS)
                ends[b] = ((int)blockIdx.x + 1 < S ? in[max_bins + b] : info[b].x * TILE + info[b].y) - in[b];
        } else {
            for (int b = tid; b < nb; b += PLACE_THREADS) {
                if (c > 0) place[b] += ends[b] - (b > 0 ? ends[b - 1] : 0);
            }
            __syncthreads();
            for (int b = tid; b < nb; b += PLACE_THREADS) ends[b] = 0;
            __syncthreads();
            for (int i = tid; i < m; i += PLACE_THREADS) atomicAdd(&ends[bin(i)], 1);
        }
        __syncthreads();
        {   // counts to first numbers: a thread's consecutive cells, then the threads
            const int per = (nb + PLACE_THREADS - 1) / PLACE_THREADS, b0 = min(nb, tid * per), b1 = min(nb, b0 + per);
            int sum = 0;
            for (int b = b0; b < b1; ++b) sum += ends[b];
            int v = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            if (lane == 31) wsum[wid] = v;
            __syncthreads();
            if (wid == 0) {
                int w = wsum[lane];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, w, o);
                    if (lane >= o) w += u;
                }
                wsum[lane] = w;
            }
            __syncthreads();
            int at = v - sum + (wid > 0 ? wsum[wid - 1] : 0);
            for (int b = b0; b < b1; ++b) {
                const int k = ends[b];
                ends[b] = at;
                at += k;
            }
        }
        __syncthreads();
        for (int i = tid; i < m; i += PLACE_THREADS) list[atomicAdd(&ends[bin(i)], 1)] = (unsigned short)i;
        __syncthreads();
        // 16 lanes per cell's run
        for (int b = tid >> 4; b < nb; b += PLACE_THREADS / 16) {
            const int first = b > 0 ? ends[b - 1] : 0, k = ends[b] - first, at = place[b];
            for (int i = tid & 15; i < k; i += 16) put(at + i, (int)a + list[first + i]);
        }
        __syncthreads();
    }
    tile_cells(T, nb, info, tile_cell + T.tile_off, [&](int pos) { put(pos, -1); });
}

// order <= 2: the window arguments of the tiles' nodes, a lane per node and two
// tiles per warp; lane p < 8 of a tile writes the pair (p, p + 8)
__global__ void __launch_bounds__(256) k_tile_fill(const Term *terms, const float *__restrict__ x, long long M,
                                                   float4 *srec, const int *tile_count) {
    const Term &T = terms[blockIdx.y];
    if (T.order == 3) return;
    const int nt = tile_count[blockIdx.y], n = T.n, lane = threadIdx.x & 31, p = lane & 15;
    const bool two = T.order == 2;
    const float *xr = x + (long long)(two ? T.row0 : T.col) * M, *xc = x + (long long)T.col * M;
    float4 *rec = srec + T.rec_off;
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int i0 = 2 * (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); i0 < nt; i0 += 2 * warps) {
        const int i = i0 + (lane >> 4);
        float4 *tile = rec + (long long)i * tile_f4(2);
        const int j = i < nt ? ((const int *)(tile + 8))[(p & 7) * 2 + (p >> 3)] : -1;
        float vr = 0.f, vc = 0.f;
        if (j >= 0) {
            float t;
            grid_pos(xc[j], n, t);
            vc = 2.f * t - 1.f;
            if (two) {
                grid_pos(xr[j], n, t);
                vr = 2.f * t - 1.f;
            }
        }
        const float vr8 = __shfl_down_sync(0xffffffffu, vr, 8), vc8 = __shfl_down_sync(0xffffffffu, vc, 8);
        if (p < 8 && i < nt) tile[p] = make_float4(vr, vr8, vc, vc8);
    }
}

static int sort_tiles(Plan &p) {
    int max_bins = 1, place_bins = 0, n3 = 0;   // place_bins: of the terms of order <= 2
    for (int s = 0; s < p.n_terms; ++s) {
        const Term &T = p.h_terms[s];
        max_bins = std::max(max_bins, T.order == 3 ? T.n * T.n * T.n : (T.order == 2 ? T.n * T.n : T.n));
        if (T.order == 3)
            ++n3;
        else
            place_bins = std::max(place_bins, T.order == 2 ? T.n * T.n : T.n);
    }
    // slices of at least 16384 nodes (a block also moves a histogram)
    int S = (int)std::max<long long>(1, std::min<long long>(SORT_MAX_SLICES, p.M / 16384));
    const size_t n_bins = (size_t)p.n_terms * max_bins;
    // (first tile, nodes) per cell, then the slices' histograms: in the partial
    // grids, which hold nothing yet, where they fit
    int2 *info = nullptr, *own = nullptr;
    const size_t room = (size_t)p.spread_kmax * (size_t)p.grid_elems * (p.precision == ANOVA_PREC_F32 ? 8 : 4);
    cudaError_t e = cudaSuccess;
    auto need = [&]() { return sizeof(int2) * n_bins + sizeof(int) * n_bins * S; };
    if (need() > room && (e = plan_malloc(&own, need())) != cudaSuccess && S > 1) {
        cudaGetLastError();   // one slice takes up to six times less
        S = 1;
        e = need() > room ? plan_malloc(&own, need()) : cudaSuccess;
    }
    if (e != cudaSuccess) return cuda_status(e);
    info = own ? own : (int2 *)p.partials;
    const size_t bytes = sizeof(int) * (size_t)max_bins;
    static std::atomic<unsigned long long> attr_seen{0};
    once_per_device(attr_seen, [] {
        cudaFuncSetAttribute(k_tile_count, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(k_tile_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(k_tile_place, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
    });
    // a part's numbers beside the cells' ends and places (at most 100 KB: 12800 cells)
    const size_t cells = 2 * sizeof(int) * (size_t)place_bins;
    const int cap = (int)std::min<long long>({(long long)PLACE_MAX, (long long)((TILES_MAX_SMEM - cells) / 2), (p.M + S - 1) / S});
    const size_t place_bytes = cells + sizeof(unsigned short) * (size_t)cap;
    {
        const dim3 grid(S, p.n_terms);
        const float *x = (const float *)p.x;
        int *hist = (int *)(info + n_bins);
        k_tile_count<<<grid, SORT_THREADS, bytes, p.stream>>>(p.terms, x, p.M, hist, max_bins);
        k_tile_scan<<<p.n_terms, 1024, 0, p.stream>>>(p.terms, hist, S, max_bins, info, p.tile_count);
        if (n3 > 0)
            k_tile_scatter<<<grid, SORT_THREADS, bytes, p.stream>>>(p.terms, x, p.M, hist, info, max_bins, p.srec,
                                                                    p.tile_cell);
        if (n3 < p.n_terms) {
            k_tile_place<<<grid, PLACE_THREADS, place_bytes, p.stream>>>(p.terms, x, p.M, hist, info, max_bins,
                                                                         place_bins, cap, p.srec, p.tile_cell);
            // about 16 steps per warp
            const int fb = (int)std::max<long long>(1, std::min<long long>(256, p.M / 4096));
            k_tile_fill<<<dim3(fb, p.n_terms), 256, 0, p.stream>>>(p.terms, x, p.M, p.srec, p.tile_count);
        }
        e = cudaGetLastError();
    }
    if (own) {
        if (e == cudaSuccess) e = cudaStreamSynchronize(p.stream);
        cudaFree(own);
    }
    return cuda_status(e);
}

// records of every term with sort_slot >= 0, n_slots slots of M
static int sort_records(Plan &p, float4 *srec, int n_slots) {
    int max_bins = 1;
    for (int s = 0; s < p.n_terms; ++s) {
        const Term &T = p.h_terms[s];
        if (T.sort_slot >= 0)
            max_bins = std::max(max_bins, T.order == 3 ? T.n * T.n * T.n : (T.order == 2 ? T.n * T.n : T.n));
    }
    int *counts = nullptr, *own = nullptr;
    const size_t need = sizeof(int) * (size_t)n_slots * max_bins;
    cudaError_t e = cudaSuccess;
    // beside tiles in the partial grids, which hold nothing yet, where they fit
    if (p.frec && need <= (size_t)p.spread_kmax * (size_t)p.grid_elems * 8) {
        counts = (int *)p.partials;
    } else {
        e = plan_malloc(&own, need);
        if (e != cudaSuccess) return cuda_status(e);
        counts = own;
    }
    const size_t hist_bytes = sizeof(int) * (size_t)max_bins;
    const bool f64 = p.precision == ANOVA_PREC_F64;
    if (hist_bytes > 48 * 1024)
        e = cudaFuncSetAttribute(f64 ? (const void *)k_cell_count64 : (const void *)k_cell_count,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hist_bytes);
    const int bx = (int)std::max<long long>(1, std::min<long long>(64, (p.M + 4095) / 4096));
    const dim3 grid(bx, p.n_terms);
    if (e == cudaSuccess) e = cudaMemsetAsync(counts, 0, need, p.stream);
    if (e == cudaSuccess) {
        if (f64)
            k_cell_count64<<<grid, 256, hist_bytes, p.stream>>>(p.terms, p.wb64, p.M, counts, max_bins);
        else
            k_cell_count<<<grid, 256, hist_bytes, p.stream>>>(p.terms, (const float *)p.x, p.M, counts, max_bins);
        k_cell_scan<<<p.n_terms, 1024, 0, p.stream>>>(p.terms, counts, max_bins);
        if (f64)
            k_cell_scatter64<<<grid, 256, 0, p.stream>>>(p.terms, p.wb64, p.M, counts, max_bins, srec);
        else
            k_cell_scatter<<<grid, 256, 0, p.stream>>>(p.terms, (const float *)p.x, p.M, counts, max_bins, srec);
        e = cudaGetLastError();
    }
    if (own) {
        if (e == cudaSuccess) e = cudaStreamSynchronize(p.stream);
        cudaFree(own);
    }
    return cuda_status(e);
}

int sort_nodes_by_cell(Plan &p) {
    if (!p.srec || p.n_sorted == 0 || p.M == 0) return ANOVA_OK;
    if (!p.cell_tc) return sort_records(p, p.srec, p.n_sorted);
    int rc = sort_tiles(p);
    if (rc || !p.frec) return rc;
    rc = sort_records(p, p.frec, p.n_frec);
    if (rc == ANOVA_ERR_NOMEM) {   // the forward runs over the tiles then
        cudaGetLastError();
        p.frec = nullptr;
        p.n_frec = 0;
        rc = ANOVA_OK;
    }
    return rc;
}

}  // namespace agft
