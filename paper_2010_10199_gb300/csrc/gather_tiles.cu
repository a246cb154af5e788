// Forward gather over the cell-aligned node tiles on the tensor cores, the
// window interpolation step of the NFFT behind eq. (somafm), Sec. 3, FP32.
//
// Work items are the adjoint's (active term, node chunk) pairs, a chunk being a
// range of the term's tiles.  A CTA copies the term's stored grid into shared
// memory; each warp takes a contiguous run of the chunk's tiles.
//
// Every tap weight is a degree-7 polynomial in the node's cell offset v, kept in
// the product basis (tiles.cuh): psi_k = sum_i C[k][i] Phi_i.  For the nodes j of
// one cell with grid window G (m_row x 8, complex)
//     f_j = sum_{r,k} G[r][k] psi_row,r(j) psi_col,k(j)
//         = sum_{l,i} Phi_l(v_row,j) H[l][i] Phi_i(v_col,j),   H = C_row^T G C_col,
// so a cell change costs two small products that turn G into H (8 x 8, complex),
// and a tile of 16 nodes takes P = Phi_col H^T (16 x 16: 8 rows of H, real and
// imaginary) in two mma.m16n8k8 of three TF32 products each and f_j = sum_l
// Phi_l(v_row,j) P[j][l].  The contraction index is permuted (2t, 2t + 1 -> t, t +
// 4), so that lane (g, t) needs Phi_2t and Phi_2t+1 of the column coordinate of nodes
// g and g + 8; the 16 columns are ordered so that the lane's four accumulators of
// a node belong to one part (t / 2: real or imaginary) and rows l = 4 (t mod 2) + 0
// .. 3: it needs these four functions of the row coordinate, sums them itself and
// adds its neighbour's half.  Each lane evaluates just these functions, 15 packed
// operations per tile, from the tile's records in its registers: nothing
// passes through shared memory but the grid window of a new cell.
//
// The sums go to 64-bit fixed-point accumulators (gather_sorted.cu), one (node,
// real or imaginary part) per lane.
#include <algorithm>
#include <cstring>

#include "tiles.cuh"

namespace agft {

constexpr int GT_THREADS = 256;
constexpr int GT_CTAS_PER_SM = 3;     // plans without third-order terms (80 registers)
constexpr int GT3_CTAS_PER_SM = 2;    // with them (128 registers)
constexpr int GT_PREFETCH = 12;       // tiles between the L2 prefetch and the loads
// third order, per warp: the tile's first-row weights, 8 taps of 16 nodes, twice
constexpr size_t GT3_WARP_BYTES = 16 * 8 * 2 * sizeof(float);

__device__ __forceinline__ void red_add_i64(unsigned long long *addr, long long v) {
    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(addr), "l"(v) : "memory");
}

// 2^31 a to the nearest integer for |a| < 2^31, in two halves of 31 bits (both
// exact): the one-instruction conversion to 64 bits runs on the FP64 unit, 16
// cycles of an SM per warp, a third of that unit's time at M = 3e5.
__device__ __forceinline__ long long to_fixed(float a) {
    const int h = __float2int_rz(a);
    const int l = __float2int_rn((a - (float)h) * 2147483648.f);
    return ((long long)h << 31) + l;
}

// H = C_row^T G C_col of the 2 MR x 8 window whose lane (g, t) holds grid values
// g0 = G[g][t], g1 = G[g][t + 4] (zero where no row g exists).  Stage 1: D1_x[i][r]
// = sum_k C_col[k][i] G_x[r][k] (A = C_col^T, rows 8..15 zero; B[k][r] =
// G_x[r][k]); stage 2: H_x[l][i] = sum_r C_row[r][l] D1_x[i][r] (A[m][k] =
// C_row[r(k)][l(m)], B[k][i] = D1_x[i][r(k)], r(t) = 2t, r(t + 4) = 2t + 1).  c0, c1 =
// C_col[t][g], C_col[t + 4][g]; r0[], r1[] = C_row[2t][l], C_row[2t + 1][l] for l =
// l_of(g), l_of(g) + 2.  Returns, for the part x = g / 4 (real, imaginary), H_x[l][2t],
// H_x[l][2t + 1] for these two l: the B fragments of the tile's two products.
__device__ __forceinline__ int l_of(int g) { return 4 * ((g >> 1) & 1) + (g & 1); }
__device__ __forceinline__ void window_to_basis(float2 g0, float2 g1, float c0, float c1, const float (&r0)[2],
                                                const float (&r1)[2], float (&h)[4]) {
    const int g = (threadIdx.x & 31) >> 2;
    unsigned c1h[4], c1l[4], c2h[4], c2l[4];
    split_tf32_x2(pk2(c0, c1), c1h[0], c1l[0], c1h[2], c1l[2]);
    split_tf32_x2(pk2(r0[0], r1[0]), c2h[0], c2l[0], c2h[2], c2l[2]);
    split_tf32_x2(pk2(r0[1], r1[1]), c2h[1], c2l[1], c2h[3], c2l[3]);
    c1h[1] = c1h[3] = c1l[1] = c1l[3] = 0u;
    unsigned gh[4], gl[4];   // B of stage 1: (re k = t, re k = t + 4, im t, im t + 4)
    split_tf32_x2(pk2(g0.x, g1.x), gh[0], gl[0], gh[1], gl[1]);
    split_tf32_x2(pk2(g0.y, g1.y), gh[2], gl[2], gh[3], gl[3]);
    float ur[4], ui[4];
    mma3_tf32_0(ur, c1h, c1l, gh[0], gh[1], gl[0], gl[1]);
    mma3_tf32_0(ui, c1h, c1l, gh[2], gh[3], gl[2], gl[3]);
    // ur = (D1_re[i = g][r = 2t], D1_re[g][2t + 1], 0, 0): the B fragment of stage 2
    unsigned uh[4], ul[4];
    split_tf32_x2(pk2(ur[0], ur[1]), uh[0], ul[0], uh[1], ul[1]);
    split_tf32_x2(pk2(ui[0], ui[1]), uh[2], ul[2], uh[3], ul[3]);
    float hr[4], hi[4];
    mma3_tf32_0(hr, c2h, c2l, uh[0], uh[1], ul[0], ul[1]);
    mma3_tf32_0(hi, c2h, c2l, uh[2], uh[3], ul[2], ul[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = g < 4 ? hr[q] : hi[q];
}

// f = sum over the lane's four functions x of the row coordinate (of nodes g, g +
// 8) times its accumulators, plus the neighbour's half: lane t ends with part t /
// 2 of node g (t even) or g + 8 (t odd).  p0, p1: (l = 0, 1), (2, 3) of node g; q0,
// q1: of node g + 8.
__device__ __forceinline__ float row_sum(const f32x2 (&x)[4], f32x2 p0, f32x2 p1, f32x2 q0, f32x2 q1, bool odd) {
    float a[4], b[4], u[4], w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) upk2(x[k], a[k], b[k]);
    upk2(p0, u[0], u[1]);
    upk2(p1, u[2], u[3]);
    upk2(q0, w[0], w[1]);
    upk2(q1, w[2], w[3]);
    const float s = fmaf(a[3], u[3], fmaf(a[2], u[2], fmaf(a[1], u[1], a[0] * u[0])));
    const float r = fmaf(b[3], w[3], fmaf(b[2], w[2], fmaf(b[1], w[1], b[0] * w[0])));
    return (odd ? r : s) + __shfl_xor_sync(0xffffffffu, odd ? s : r, 1);
}

// Tiles [0, nt) of an order-1/2 term for one warp.  Order 1: C_row = e_0 e_0^T and
// only grid row 0 exists.  sc: the fixed-point scale times 2^-31.
template <int MR>
__device__ __forceinline__ void gather_run12(const float4 *__restrict__ rec, const int *__restrict__ cells, int nt,
                                             const float2 *S, int stride, bool ord2, const float *__restrict__ pbr,
                                             const float *__restrict__ pbc, unsigned long long *__restrict__ acc,
                                             float sc) {
    constexpr int F4 = tile_f4(2);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const BasisFactors F = basis_factors(2 * t);
    const f32x2 rc = dup2(t & 1 ? 8.f : 0.f);
    int cur = -1;            // cell whose H is in bh, bl
    unsigned bh[4], bl[4];   // B fragments of the two products, times sc
    auto load_h = [&](int off) {
        float2 g0 = make_float2(0.f, 0.f), g1 = g0;
        if (ord2 ? g < 2 * MR : g == 0) {   // grid row g of the window exists
            g0 = S[off + g * stride + t];
            g1 = S[off + g * stride + t + 4];
        }
        const int l = l_of(g);
        float r0[2] = {l == 0 && t == 0 ? 1.f : 0.f, 0.f}, r1[2] = {0.f, 0.f};
        if (ord2) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                r0[k] = __ldg(pbr + 2 * t * NCOEF + l + 2 * k);
                r1[k] = __ldg(pbr + (2 * t + 1) * NCOEF + l + 2 * k);
            }
        }
        float h[4];
        window_to_basis(g0, g1, __ldg(pbc + t * NCOEF + g), __ldg(pbc + (t + 4) * NCOEF + g), r0, r1, h);
#pragma unroll
        for (int k = 0; k < 4; ++k) h[k] = uncut(h[k] * sc, ord2 ? 3.f : 2.f);
        split_tf32_x2(pk2(h[0], h[1]), bh[0], bl[0], bh[1], bl[1]);
        split_tf32_x2(pk2(h[2], h[3]), bh[2], bl[2], bh[3], bl[3]);
    };
    struct Tile {
        float4 q;   // (vr_g, vr_g+8, vc_g, vc_g+8)
        int id;     // of node g (t even) or g + 8 (t odd)
        int cell;
    };
    // tile 0 .. 3 from rec, cells on; loads run up to 3 tiles past the run's end,
    // inside the buffers
    const int *ids = (const int *)(rec + 8) + 2 * g + (t & 1);
    rec += g;
    auto load = [&](int k) {
        Tile T;
        T.q = __ldg(rec + k * F4);
        T.id = __ldg(ids + k * F4 * 4);
        T.cell = __ldg(cells + k) & ~TILE_HALF;
        return T;
    };
    acc += t >> 1;   // this lane's part (real or imaginary)
    auto tile = [&](const Tile &T, bool valid) {
        f32x2 ce, co, x[4];
        basis_even_odd(pk2(T.q.z, T.q.w), F, ce, co);   // Phi_2t, Phi_2t+1 of the column coordinate, nodes (g, g + 8)
        basis_four(pk2(T.q.x, T.q.y), rc, x);
        // A: a0 = Phi_2t(v_col) of node g, a1 = of node g + 8, a2 = Phi_2t+1(v_col) of g, a3 = of g + 8
        unsigned ah[4], al[4];
        split_tf32_x2(ce, ah[0], al[0], ah[1], al[1]);
        split_tf32_x2(co, ah[2], al[2], ah[3], al[3]);
        float d0[4], d1[4];
        mma3_tf32_0(d0, ah, al, bh[0], bh[1], bl[0], bl[1]);
        mma3_tf32_0(d1, ah, al, bh[2], bh[3], bl[2], bl[3]);
        const float v = row_sum(x, pk2(d0[0], d0[1]), pk2(d1[0], d1[1]), pk2(d0[2], d0[3]), pk2(d1[2], d1[3]), t & 1);
        if (valid && T.id >= 0) red_add_i64(acc + 2 * (long long)T.id, to_fixed(v));
    };
    auto pair = [&](const Tile &c0, const Tile &c1, bool two) {
        if (c0.cell == cur && c1.cell == cur) {   // two independent chains without a branch between them
            tile(c0, true);
            tile(c1, two);
            return;
        }
        if (c0.cell != cur) load_h(cur = c0.cell);
        tile(c0, true);
        if (two) {
            if (c1.cell != cur) load_h(cur = c1.cell);
            tile(c1, true);
        }
    };
    Tile a0 = load(0), a1 = load(1);
    for (int left = nt; left > 0; left -= 4) {
        // the tiles GT_PREFETCH ahead into L2 (whole tiles of the run only)
        if (lane == 0 && left >= GT_PREFETCH + 4) prefetch_l2_bulk(rec + GT_PREFETCH * F4, 4 * F4 * 16);
        const Tile b0 = load(2), b1 = load(3);
        pair(a0, a1, left > 1);
        if (left <= 2) break;
        rec += 4 * F4;
        ids += 4 * F4 * 4;
        cells += 4;
        if (left > 4) {
            a0 = load(0);
            a1 = load(1);
        }
        pair(b0, b1, left > 3);
    }
}

// Tiles [0, nt) of a third-order term (a, b, c) for one warp:
//     f_j = sum_ia psi_a,ia(j) sum_{l,i} Phi_l(v_b,j) T_ia[l][i] Phi_i(v_c,j),
// T_ia = C_b^T G_ia C_c for the 2 MR grid planes ia the window touches.  The
// planes' T stay in registers as B fragments (FP16 high and low parts); since
// cells run along a, a new cell usually drops one plane and transforms one.  A
// tile takes per plane P_ia = Phi_c T_ia^T on the tensor core and adds psi_a,ia
// times it in registers; the sum over l follows once, as in the order-2 tile.
// What bounds it: the warp instructions (four products and four packed FMAs per
// plane beside the tile's bases and the planes' transforms); FP16 with k = 16
// holds Phi's high and low parts in one product, half the TF32 form's time.
template <int MR>
__device__ __forceinline__ void gather_run3(const float4 *__restrict__ rec, const int *__restrict__ cells, int nt,
                                            const float2 *S, const Term &T, const Window *__restrict__ wr,
                                            const Window *__restrict__ wc, float gscale,
                                            unsigned long long *__restrict__ acc, float sc, float4 *psi) {
    constexpr int NP = 2 * MR;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int n = T.n, stride = T.stride, mc = T.mc;
    const BasisFactors F = basis_factors(2 * t);
    const f32x2 rc = dup2(t & 1 ? 8.f : 0.f);
    // first-row weights: this lane evaluates taps 2t, 2t + 1 of nodes g, g + 8
    f32x2 pc[NCOEF];
#pragma unroll
    for (int k = 0; k < NCOEF; ++k)
        pc[k] = 2 * t < NP ? pk2(__ldg(&wr->c[2 * t][k]), __ldg(&wr->c[2 * t + 1][k])) : pk2(0.f, 0.f);
    uint4 pl[NP];   // plane fragments: (product 0 high, low, product 1 high, low), times gscale
    auto load_plane = [&](int ip, int fb, int fc) {
        float2 g0 = make_float2(0.f, 0.f), g1 = g0;
        if (g < NP) {
            const float2 *row = S + (ip * n + wrap(fb - MR + 1 + g, n)) * stride;
            g0 = row[wrap(fc - mc + 1 + t, n)];
            g1 = row[wrap(fc - mc + 5 + t, n)];
        }
        const int l = l_of(g);
        const float r0[2] = {__ldg(&wr->pb[2 * t][l]), __ldg(&wr->pb[2 * t][l + 2])};
        const float r1[2] = {__ldg(&wr->pb[2 * t + 1][l]), __ldg(&wr->pb[2 * t + 1][l + 2])};
        float h[4];
        window_to_basis(g0, g1, __ldg(&wc->pb[t][g]), __ldg(&wc->pb[t + 4][g]), r0, r1, h);
        uint4 r;
#pragma unroll
        for (int k = 0; k < 4; ++k) h[k] = uncut(h[k] * gscale, 3.f);
        split_f16(h[0], h[1], r.x, r.y);
        split_f16(h[2], h[3], r.z, r.w);
        return r;
    };
    int cur = -1;   // cell whose planes are held
    auto new_cell = [&](int cell) {
        const int fa = cell & 255, fb = (cell >> 8) & 255, fc = cell >> 16;
        int step = NP;
        if (cur >= 0 && (cur >> 8) == (cell >> 8)) step = min(NP, fa - (cur & 255));   // cells ascend
        if (step <= 0) step = NP;
#pragma unroll 1
        for (int k = step; k > 0; --k) {
            // drop plane 0, append the plane of tap NP - 1 of first cell fa - k + 1
            uint4 next = pl[0];   // an axis as long as the window: the planes rotate
            if (n != NP || step == NP) next = load_plane(wrap(wrap(fa - k + 1 + MR, n), n), fb, fc);
#pragma unroll
            for (int a = 0; a + 1 < NP; ++a) pl[a] = pl[a + 1];
            pl[NP - 1] = next;
        }
        cur = cell;
    };
    acc += t >> 1;
    const int idw = t & 1;
    float4 n0 = __ldg(rec + g), n1 = __ldg(rec + 8 + g);   // (va, vb, vc, index) of nodes g, g + 8
    int ncell = __ldg(cells) & ~TILE_HALF;
    for (int i = 0; i < nt; ++i) {
        const float4 q0 = n0, q1 = n1;
        const int cell = ncell;
        if (lane == 0 && i + GT_PREFETCH < nt) prefetch_l2_bulk(rec + GT_PREFETCH * TILE, TILE * 16);
        // the next tile's records (one tile past the run's end, inside the buffers)
        rec += TILE;
        n0 = __ldg(rec + g);
        n1 = __ldg(rec + 8 + g);
        ncell = __ldg(cells + i + 1) & ~TILE_HALF;
        if (cell != cur) new_cell(cell);
        // first-row weights of the tile, handed round through shared memory, each
        // twice for the packed sums: psi[16 s + 8 h + p] = tap 2s + h of nodes p, p, p + 8, p + 8
        {
            f32x2 w0 = pc[NCOEF - 1], w1 = w0;
            const f32x2 v0 = dup2(q0.x), v1 = dup2(q1.x);
#pragma unroll
            for (int k = NCOEF - 2; k >= 0; --k) {
                w0 = fma2(w0, v0, pc[k]);
                w1 = fma2(w1, v1, pc[k]);
            }
            float a0, a1, b0, b1;   // taps 2t, 2t + 1 of node g; of node g + 8
            upk2(w0, a0, a1);
            upk2(w1, b0, b1);
            __syncwarp();   // the previous tile's weights are read
            psi[16 * t + g] = make_float4(a0, a0, b0, b0);
            psi[16 * t + 8 + g] = make_float4(a1, a1, b1, b1);
        }
        unsigned A[4];   // (Phi_2t, Phi_2t+1) of the column coordinate, nodes g, g + 8: high parts, low parts
        {
            f32x2 ce, co;
            basis_even_odd(pk2(q0.z, q1.z), F, ce, co);
            float e0, e1, o0, o1;
            upk2(ce, e0, e1);
            upk2(co, o0, o1);
            split_f16(e0, o0, A[0], A[2]);
            split_f16(e1, o1, A[1], A[3]);
        }
        __syncwarp();
        // sums over planes of psi_a times the lane's accumulators: nodes g and g + 8
        f32x2 p0 = 0ull, p1 = 0ull, r0 = 0ull, r1 = 0ull;
#pragma unroll
        for (int a = 0; a < NP; ++a) {
            const uint4 f = pl[a];
            float d0[4], d1[4];
            mma_f16_k8_0(d0, A[0], A[1], f.y);
            mma_f16_k8_0(d1, A[0], A[1], f.w);
            mma_f16_k16(d0, A, f.x, f.x);
            mma_f16_k16(d1, A, f.z, f.z);
            const ulonglong2 w = *(const ulonglong2 *)&psi[8 * a + g];
            p0 = fma2(w.x, pk2(d0[0], d0[1]), p0);
            p1 = fma2(w.x, pk2(d1[0], d1[1]), p1);
            r0 = fma2(w.y, pk2(d0[2], d0[3]), r0);
            r1 = fma2(w.y, pk2(d1[2], d1[3]), r1);
        }
        f32x2 x[4];
        basis_four(pk2(q0.y, q1.y), rc, x);
        const float v = row_sum(x, p0, p1, r0, r1, idw) * sc;
        const int j = __float_as_int(idw ? q1.w : q0.w);
        if (j >= 0) red_add_i64(acc + 2 * (long long)j, to_fixed(v));
    }
}

// O3: the plan (or batch) has third-order terms
template <int MR, bool O3>
__global__ void __launch_bounds__(GT_THREADS, O3 ? GT3_CTAS_PER_SM : GT_CTAS_PER_SM)
gather_tiles(DevPlan single, BatchArgs B, const int4 *__restrict__ items, int n_items, int *counter,
             long long max_grid_bytes) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_item;
    __shared__ unsigned s_max;
    constexpr int NW = GT_THREADS / 32;
    float2 *S = (float2 *)smem;
    const int tid = threadIdx.x, warp = tid >> 5;
    for (;;) {
        if (tid == 0) {
            s_item = atomicAdd(counter, 1);
            s_max = 0u;
        }
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= n_items) break;
        const int4 itm = items[item];
        const DevPlan &P = B.plans ? B.plans[itm.x] : single;
        if (P.skip && *P.skip) continue;
        const int term = P.act[itm.y];
        const Term &T = P.terms[term];
        const int nt = P.tile_count[term];
        const int t0 = (int)((long long)nt * itm.z / itm.w), t1 = (int)((long long)nt * (itm.z + 1) / itm.w);
        if (t0 >= t1) continue;
        {
            const float4 *gsrc = (const float4 *)(P.grids + T.grid_off);
            float4 *S4 = (float4 *)S;
            const int n4 = (int)(T.grid_bytes / 16);
            unsigned m = 0u;
            for (int e = tid; e < n4; e += GT_THREADS) {
                const float4 v = __ldg(gsrc + e);
                S4[e] = v;
                if (O3)   // largest magnitude, as the bits of a non-negative float (NaN above all)
                    m = max(max(max(m, __float_as_uint(v.x) & 0x7fffffffu), __float_as_uint(v.y) & 0x7fffffffu),
                            max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu));
            }
            if (O3 && T.order == 3) {
                m = __reduce_max_sync(0xffffffffu, m);
                if ((tid & 31) == 0) atomicMax(&s_max, m);
            }
        }
        __syncthreads();
        const float sc = ldexpf(1.f, P.fexp[0] - 31);   // 2^(e - 31), exact scaling
        // warp w takes a contiguous run of the chunk's tiles
        const int per = (t1 - t0 + NW - 1) / NW;
        const int a = t0 + warp * per, b = min(t1, a + per);
        if (a < b) {
            const float4 *rec = P.srec + T.rec_off + (long long)a * tile_f4(T.order);
            const int *cells = P.tile_cell + T.tile_off + a;
            const Window *wr = P.windows + T.wr, *wc = P.windows + T.wc;
            if (O3 && T.order == 3) {
                // |T| <= (sum of |C_b| column) (sum of |C_c| column) max |G| < 2^4 max |G|
                const float gs = scale_to(s_max, 10);
                const float inv = __int_as_float((254 - (__float_as_int(gs) >> 23)) << 23);
                gather_run3<MR>(rec, cells, b - a, S, T, wr, wc, gs, P.facc, sc * inv,
                                (float4 *)(smem + max_grid_bytes + warp * GT3_WARP_BYTES));
            } else {
                gather_run12<MR>(rec, cells, b - a, S, T.stride, T.order == 2, &wr->pb[0][0], &wc->pb[0][0], P.facc,
                                 sc);
            }
        }
        __syncthreads();   // the grid is read by every warp before the next item replaces it
    }
}

static size_t gather_tiles_smem(long long max_grid_bytes, bool order3) {
    return (size_t)max_grid_bytes + (order3 ? GT3_WARP_BYTES * (GT_THREADS / 32) : 0);
}

int gather_tiles_ctas_per_sm(long long max_grid_bytes, bool order3) {
    const size_t per = gather_tiles_smem(max_grid_bytes, order3) + 1024 + 16;   // + the per-CTA reserve and the static words
    return (int)std::max<size_t>(1, std::min<size_t>(order3 ? GT3_CTAS_PER_SM : GT_CTAS_PER_SM,
                                                     (size_t)(MAX_SMEM + 1024) / per));
}

// the gather of items [0, n_items) of one problem (B.plans == null) or a batch
void gather_tiles_launch(cudaStream_t st, const DevPlan &v, const BatchArgs &B, const int4 *items, int n_items,
                         bool order3, int *counter, long long max_grid_bytes, int sm_count, int mr) {
    static std::atomic<unsigned long long> attr_seen{0};
    once_per_device(attr_seen, [] {
        cudaFuncSetAttribute(gather_tiles<3, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(gather_tiles<4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(gather_tiles<3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(gather_tiles<4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
    });
    if (n_items <= 0) return;
    const size_t smem = gather_tiles_smem(max_grid_bytes, order3);
    const int ctas = std::max(1, std::min(n_items, gather_tiles_ctas_per_sm(max_grid_bytes, order3) * sm_count));
    auto k = mr <= 3 ? (order3 ? gather_tiles<3, true> : gather_tiles<3, false>)
                     : (order3 ? gather_tiles<4, true> : gather_tiles<4, false>);
    k<<<ctas, GT_THREADS, smem, st>>>(v, B, items, n_items, counter, max_grid_bytes);
}

}  // namespace agft
