// Adjoint spread over the cell-aligned node tiles on the tensor cores (stacked
// adjoint after the error remark, Sec. 3), FP32 sums, grids stored as FP32 or
// as 16-bit pairs.
//
// Work items are (active term, node chunk) pairs, a chunk being a range of the
// term's tiles.  A CTA adds the chunk's window sums into a shared-memory copy of
// the term's stored grid and writes it to the chunk's partial grid; each warp
// takes a contiguous run of the chunk's tiles and adds to the shared grid once
// per cell.
#include <algorithm>
#include <cstring>

#include "tiles.cuh"

namespace agft {

// without third-order terms 12 warps per CTA, 2 CTAs per SM (80 registers); with
// them 8 warps per CTA, 2 CTAs per SM (128 registers)
constexpr int ST_THREADS = 384, ST_CTAS_PER_SM = 2, ST3_THREADS = 256, ST3_CTAS_PER_SM = 2;

__device__ __forceinline__ void red_add_f32(float *addr, float v) {
    asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(smem_addr(addr)), "f"(v) : "memory");
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Adds a lane's (g, t) window taps G (moments_to_window) to the elements c0 and c1 of
// the shared grid.  Lanes whose grid rows fall into the same banks (rows g of a pitch
// that is 8 mod 16: g of one parity) start at different words: one bank per lane
// instead of four lanes per bank, a quarter of the additions' shared-memory wavefronts
// (2.6e7 -> 6.6e6 at d = 20, M = 3e5; third order, d = 10, M = 5e5: 3.36 -> 3.16 ms).
__device__ __forceinline__ void add_taps(float2 *c0, float2 *c1, const float (&G)[4], int g) {
    float v[4] = {G[0], G[2], G[1], G[3]}, u[4], w[4];
    const int s = g >> 1;
#pragma unroll
    for (int q = 0; q < 4; ++q) u[q] = s & 1 ? v[(q + 1) & 3] : v[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = s & 2 ? u[(q + 2) & 3] : u[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) red_add_f32((float *)((q + s) & 2 ? c1 : c0) + ((q + s) & 1), w[q]);
}

// Window block of a cell from its moments: G = C_col Mo C_row^T, with lane (g, t)
// holding d = Mo (re i = g, l = 2t), (re g, 2t + 1), (im g, 2t), (im g, 2t + 1) and
// the coefficients cr0, cr1 = C_row[g][2t], C_row[g][2t + 1] (zero where no row g
// exists) and cc0, cc1 = C_col[g][2t], C_col[g][2t + 1].  Two products with the
// contraction index permuted (2t, 2t + 1 -> t, t + 4), so that each D fragment is
// the next product's operand as it stands.  Returns G = (re, row tap g, column
// tap 2t), (re, g, 2t + 1), (im, g, 2t), (im, g, 2t + 1).
__device__ __forceinline__ void moments_to_window(const float (&d)[4], float cr0, float cr1, float cc0, float cc1,
                                                  float (&G)[4]) {
    unsigned ah[4], al[4], ch0, cl0, ch1, cl1;
    split_tf32_x2(pk2(cr0, cr1), ah[0], al[0], ah[2], al[2]);
    ah[1] = ah[3] = al[1] = al[3] = 0u;
    split_tf32_x2(pk2(cc0, cc1), ch0, cl0, ch1, cl1);
    // Q_x[j][i] = sum_l C_row[j][l] Mo_x[i][l]: A = C_row (rows 8..15 zero),
    // B[k][i] = Mo_x[i][l(k)] with l(t) = 2t, l(t + 4) = 2t + 1
    unsigned mh[4], ml[4];
    split_tf32_x2(pk2(d[0], d[1]), mh[0], ml[0], mh[1], ml[1]);
    split_tf32_x2(pk2(d[2], d[3]), mh[2], ml[2], mh[3], ml[3]);
    float qr[4], qi[4];
    mma3_tf32_0(qr, ah, al, mh[0], mh[1], ml[0], ml[1]);
    mma3_tf32_0(qi, ah, al, mh[2], mh[3], ml[2], ml[3]);
    // q = Q_x[j = g][i = 2t], Q_x[g][2t + 1] (entries 2, 3: zero rows).
    // G_x^T[j][k] = sum_i Q_x[j][i] C_col[k][i]: A[(x, j)][k'] = Q_x[j][i(k')],
    // B[k'][k] = C_col[k][i(k')]
    unsigned qh[4], ql[4];
    split_tf32_x2(pk2(qr[0], qi[0]), qh[0], ql[0], qh[1], ql[1]);
    split_tf32_x2(pk2(qr[1], qi[1]), qh[2], ql[2], qh[3], ql[3]);
    mma3_tf32_0(G, qh, ql, ch0, ch1, cl0, cl1);
}

// ---- order 1 and 2 ----
//
// The nodes of a cell build the moment matrix Mo[(re/im, i)][l] = sum_j y_j
// X_i(v_col,j) X_l(v_row,j) in the Chebyshev basis (Window::ch), a product A B
// with A[(re/im, i)][j] = y_j X_i(v_col,j) (16 x n) and B[j][l] = X_l(v_row,j)
// (n x 8): per group of 8 nodes one mma.m16n8k8, each operand split x = hi + lo
// into TF32 parts, three products.  Two tiles make a step of 32 nodes, one per
// lane.  The recurrence is linear, so starting it at y instead of 1 gives the
// lane y_j X_i(v_col,j), real and imaginary part at once, for the cost of the
// basis alone; the values pass through shared memory to the lanes that hold them
// as fragments (lane (g, t): index g of nodes 2t, 2t + 1 of a group, 16 bytes of A
// and 8 of B per read, rows padded to keep the reads free of bank conflicts).
// The records, y[index] and the tiles' cells are loaded to registers two steps, one step
// and one step ahead (the cells when needed: d = 20, M = 1e6 2.25 ms instead of 2.01; the
// values two steps ahead: 2.12); a bulk prefetch brings the records into L2 before that.  Each tile gets a fresh
// tensor-core sum, added to the cell's in FP32 with rounding to nearest: the
// tensor core's own accumulation is not rounded to nearest, and its bias would
// grow with the cell's node count.  Order 1: B = e_0 (the single grid row).
// Row 0 of B, X_0 = 1, is one row for all warps; a warp's buffer is a multiple of 128
// bytes, so that the row keeps its place in the banks' order for each of them.
constexpr int ST_AROW = 40, ST_BROW = 40;   // row strides: float2 (320 bytes) and float (160 bytes)
constexpr size_t ST_A_BYTES = NCOEF * ST_AROW * sizeof(float2);
constexpr size_t ST_B_BYTES = (NCOEF - 1) * ST_BROW * sizeof(float);
constexpr size_t ST_ONE_BYTES = ST_BROW * sizeof(float);
constexpr size_t ST_WARP_BYTES = (ST_A_BYTES + ST_B_BYTES + 127) / 128 * 128;
static_assert(ST_A_BYTES % 128 == 0, "B starts on a bank's first word");

template <int MR, bool ORD2>
__device__ __forceinline__ void spread_run12(const float4 *__restrict__ rec, const int *__restrict__ cells, int nt,
                                             const float2 *__restrict__ y, float2 *S, int stride,
                                             const float *__restrict__ chr, const float *__restrict__ chc,
                                             unsigned char *buf, const float *ones) {
    constexpr int F4 = tile_f4(2), PF = 14;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    float2 *as = (float2 *)buf;
    float *bs = (float *)(buf + ST_A_BYTES) - ST_BROW;   // rows 1 .. 7
    int cur = -1;   // grid offset of the cell being summed
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    auto flush = [&]() {
        float cr0 = ORD2 ? 0.f : (g == 0 && t == 0 ? 1.f : 0.f), cr1 = 0.f;
        if (ORD2 && g < 2 * MR) {
            cr0 = __ldg(chr + g * NCOEF + 2 * t);
            cr1 = __ldg(chr + g * NCOEF + 2 * t + 1);
        }
        float G[4];
        moments_to_window(d, cr0, cr1, __ldg(chc + g * NCOEF + 2 * t), __ldg(chc + g * NCOEF + 2 * t + 1), G);
        if (ORD2 ? g < 2 * MR : g == 0) {
            float2 *c = S + cur + g * stride + 2 * t;
            add_taps(c, c + 1, G, g);
        }
        d[0] = d[1] = d[2] = d[3] = 0.f;
    };
    // this lane's node: number lane % 16 of tile 2 s + lane / 16 of step s
    const int p = lane & 15, half = lane >> 4, ns = (nt + 1) / 2;
    const float *rv = (const float *)(rec + half * F4) + (p & 7) * 4 + (p >> 3);
    const int *ri = (const int *)(rec + half * F4 + 8) + (p & 7) * 2 + (p >> 3);
    struct Rec {
        float vr, vc;
        int id;
    };
    // past an odd run's end: a padding node
    auto load = [&](int s) {
        const bool ok = 2 * s + half < nt;
        Rec r;
        r.vr = ORD2 && ok ? __ldg(rv + s * (F4 * 8)) : 0.f;
        r.vc = ok ? __ldg(rv + s * (F4 * 8) + 2) : 0.f;
        r.id = ok ? __ldg(ri + s * (F4 * 8)) : -1;
        return r;
    };
    auto load_y = [&](int id) { return id >= 0 ? __ldcg(y + id) : make_float2(0.f, 0.f); };
    Rec r0 = load(0), r1 = load(min(1, ns - 1));
    float2 y0 = load_y(r0.id);
    int n0 = __ldg(cells), n1 = __ldg(cells + 1);
    for (int s = 0; s < ns; ++s) {
        const int c0 = n0, c1 = 2 * s + 1 < nt ? n1 : (c0 & ~TILE_HALF);
        n0 = __ldg(cells + 2 * s + 2);   // the next step's (inside the buffer past the run's end)
        n1 = __ldg(cells + 2 * s + 3);
        if (lane == 0 && 2 * s + PF + 2 <= nt) prefetch_l2_bulk(rec + (long long)(2 * s + PF) * F4, 2 * F4 * 16);
        const float2 yv = y0;
        const float vr = r0.vr, vc = r0.vc;
        r0 = r1;
        y0 = load_y(s + 1 < ns ? r1.id : -1);
        if (s + 2 < ns) r1 = load(s + 2);
        __syncwarp();   // the previous step's values are read
        {
            // X_{k+1} = X_{k-1} + (-1)^k 2 v X_k: the column coordinate's times y, and the row's
            f32x2 zm = pk2(yv.x, yv.y);
            const f32x2 vv = pk2(vc, vc), up = mul2(vv, pk2(2.f, 2.f)), um = mul2(vv, pk2(-2.f, -2.f));
            f32x2 z = mul2(vv, zm);
            float xm = 1.f, x = vr;
            const float ru = 2.f * vr, rm = -2.f * vr;
            f32x2 *aw = (f32x2 *)as + lane;
            float *bw = bs + lane;
            aw[0] = zm;
            aw[ST_AROW] = z;
            if (ORD2) bw[ST_BROW] = x;
#pragma unroll
            for (int k = 2; k < NCOEF; ++k) {
                const f32x2 zn = fma2((k & 1) ? up : um, z, zm);
                zm = z;
                z = zn;
                aw[k * ST_AROW] = z;
                if (ORD2) {
                    const float xn = fmaf((k & 1) ? ru : rm, x, xm);
                    xm = x;
                    x = xn;
                    bw[k * ST_BROW] = x;
                }
            }
        }
        __syncwarp();
        const float4 *ar = (const float4 *)(as + g * ST_AROW) + t;   // + 4 per group: nodes 2t, 2t + 1
        const float2 *br = (const float2 *)(g == 0 ? ones : bs + g * ST_BROW) + t;
        auto group = [&](float (&e)[4], int h, bool first) {
            const float4 z = ar[4 * h];
            unsigned ah[4], al[4];
            split_tf32_x2(pk2(z.x, z.y), ah[0], al[0], ah[1], al[1]);
            split_tf32_x2(pk2(z.z, z.w), ah[2], al[2], ah[3], al[3]);
            if (ORD2) {
                const float2 x = br[4 * h];
                unsigned bh0, bl0, bh1, bl1;
                split_tf32_x2(pk2(x.x, x.y), bh0, bl0, bh1, bl1);
                if (first)
                    mma3_tf32_0(e, ah, al, bh0, bh1, bl0, bl1);
                else
                    mma3_tf32(e, ah, al, bh0, bh1, bl0, bl1);
            } else {
                const unsigned one = g == 0 ? 0x3f800000u : 0u;
                if (first)
                    mma_tf32_0(e, al, one, one);
                else
                    mma_tf32(e, al, one, one);
                mma_tf32(e, ah, one, one);
            }
        };
        float e0[4], e1[4];
        if (((c0 | c1) & TILE_HALF) == 0) {
            group(e0, 0, true);
            group(e1, 2, true);
            group(e0, 1, false);
            group(e1, 3, false);
        } else {   // the second halves that are all padding are left out
            group(e0, 0, true);
            group(e1, 2, true);
            if (!(c0 & TILE_HALF)) group(e0, 1, false);
            if (!(c1 & TILE_HALF)) group(e1, 3, false);
        }
        const int k0 = c0 & ~TILE_HALF, k1 = c1 & ~TILE_HALF;
        if (k0 != cur) {
            if (cur >= 0) flush();
            cur = k0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] += e0[q];
        if (k1 != cur) {
            flush();
            cur = k1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] += e1[q];
    }
    if (cur >= 0) flush();
}

// ---- order 3 ----
//
// For a term (a, b, c) the window sums of a cell are, per grid plane ia,
//     Mo_ia[(re/im, i)][l] = sum_j y_j Phi_i(v_c,j) psi_a,ia(j) Phi_l(v_b,j)
// in the product basis along b and c: per tile and plane one product A B_ia, A
// (16 x 16 nodes) shared by the planes, in FP16 with both operands split into
// high and low parts (three mma.m16n8k16; y scaled to FP16's range by a power of
// two).  Cells run along a, so the 2 m_row planes' moments stay in registers: a
// new cell drops one plane, turns its moments into window taps and adds them to
// the shared grid, where the sums of every cell's planes used to go on each new
// cell (32 additions per lane instead of 4).
// Lane (g, t) evaluates function g of both coordinates of nodes 2t, 2t + 1, 2t + 8,
// 2t + 9 itself; the first-row weights are evaluated once per node and read
// through shared memory.
constexpr int ST3_RING = 4;   // tiles in a warp's record ring
constexpr size_t ST3_WARP_BYTES = (size_t)ST3_RING * TILE * 16 + 16 * 8 * sizeof(float);   // ring, weights
static_assert(ST3_WARP_BYTES <= ST_WARP_BYTES, "one buffer per warp serves every order");

template <int MR>
__device__ __forceinline__ void spread_run3(const float4 *__restrict__ rec, const int *__restrict__ cells, int nt,
                                            const float2 *__restrict__ y, float2 *S, const Term &T,
                                            const Window *__restrict__ wr, const Window *__restrict__ wc, float ys,
                                            float inv_ys, unsigned char *buf) {
    constexpr int NP = 2 * MR, PF = 12;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int n = T.n, stride = T.stride, mc = T.mc;
    float4 *ring = (float4 *)buf;
    float4 *psi = ring + ST3_RING * TILE;
    const BasisFactors F = basis_factors(g);
    f32x2 pc[NCOEF];   // first-row taps 2t, 2t + 1
#pragma unroll
    for (int k = 0; k < NCOEF; ++k)
        pc[k] = 2 * t < NP ? pk2(__ldg(&wr->c[2 * t][k]), __ldg(&wr->c[2 * t + 1][k])) : pk2(0.f, 0.f);
    f32x2 d[NP][2];   // moments of the planes: (re i = g, l = 2t, 2t + 1), (im ..)
#pragma unroll
    for (int a = 0; a < NP; ++a) d[a][0] = d[a][1] = 0ull;
    // plane tap 0 of cell (fa, fb, fc) to the shared grid
    auto flush_plane = [&](int fa, int fb, int fc) {
        float m[4], G[4];
        upk2(d[0][0], m[0], m[1]);
        upk2(d[0][1], m[2], m[3]);
        float cr0 = 0.f, cr1 = 0.f;
        if (g < NP) {
            cr0 = __ldg(&wr->pb[g][2 * t]);
            cr1 = __ldg(&wr->pb[g][2 * t + 1]);
        }
        moments_to_window(m, cr0, cr1, __ldg(&wc->pb[g][2 * t]), __ldg(&wc->pb[g][2 * t + 1]), G);
        if (g < NP) {
            float2 *row = S + (wrap(wrap(fa - MR + 1, n), n) * n + wrap(fb - MR + 1 + g, n)) * stride;
#pragma unroll
            for (int q = 0; q < 4; ++q) G[q] *= inv_ys;
            add_taps(row + wrap(fc - mc + 1 + 2 * t, n), row + wrap(fc - mc + 2 + 2 * t, n), G, g);
        }
    };
    int cur = -1;
    // drops the planes that a window at first index fa + step no longer touches
    auto advance = [&](int step) {
        const int fa = cur & 255, fb = (cur >> 8) & 255, fc = cur >> 16;
        for (int k = 0; k < step; ++k) {
            flush_plane(fa + k >= n ? fa + k - n : fa + k, fb, fc);
#pragma unroll
            for (int a = 0; a + 1 < NP; ++a) {
                d[a][0] = d[a + 1][0];
                d[a][1] = d[a + 1][1];
            }
            d[NP - 1][0] = d[NP - 1][1] = 0ull;
        }
    };
    // ring slot i % ST3_RING: tile i
    auto fetch = [&](int i) {
        if (i < nt && lane < TILE) cp_async16(ring + (i % ST3_RING) * TILE + lane, rec + (long long)i * TILE + lane);
        cp_async_commit();
    };
    float2 yn[4];   // values of nodes 2t, 2t + 8, 2t + 1, 2t + 9 of the next tile
    auto load_y = [&](int i) {
        const float4 *X = ring + (i % ST3_RING) * TILE + 2 * t;
        const int id[4] = {__float_as_int(X[0].w), __float_as_int(X[8].w), __float_as_int(X[1].w), __float_as_int(X[9].w)};
#pragma unroll
        for (int q = 0; q < 4; ++q) yn[q] = id[q] >= 0 ? __ldcg(y + id[q]) : make_float2(0.f, 0.f);
    };
    __syncwarp();   // an earlier run's reads of the ring are done
    fetch(0);
    fetch(1);
    fetch(2);
    cp_async_wait_n<2>();
    __syncwarp();
    load_y(0);
    int ncell = __ldg(cells);
    for (int i = 0; i < nt; ++i) {
        const int cell = ncell & ~TILE_HALF;
        ncell = __ldg(cells + i + 1);   // the next tile's (inside the buffer past the run's end)
        if (lane == 0 && i + PF < nt) prefetch_l2_bulk(rec + (long long)(i + PF) * TILE, TILE * 16);
        float2 yv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) yv[q] = yn[q];
        cp_async_wait_n<1>();   // tile i + 1 has landed (tiles i + 1, i + 2 were in flight)
        __syncwarp();           // and is visible; the previous tile's slot and weights are read
        fetch(i + 3);
        if (i + 1 < nt) load_y(i + 1);
        const float4 *X = ring + (i % ST3_RING) * TILE;
        {   // psi[8 s + p] = taps 2s, 2s + 1 of nodes p, p + 8
            f32x2 w0 = pc[NCOEF - 1], w1 = w0;
            const f32x2 v0 = dup2(X[g].x), v1 = dup2(X[g + 8].x);
#pragma unroll
            for (int k = NCOEF - 2; k >= 0; --k) {
                w0 = fma2(w0, v0, pc[k]);
                w1 = fma2(w1, v1, pc[k]);
            }
            float4 w;
            upk2(w0, w.x, w.z);
            upk2(w1, w.y, w.w);
            psi[8 * t + g] = w;
        }
        // functions g of nodes (2t, 2t + 8) and (2t + 1, 2t + 9)
        const float4 q0 = X[2 * t], q1 = X[2 * t + 1], q8 = X[2 * t + 8], q9 = X[2 * t + 9];
        const f32x2 xb0 = basis_one(pk2(q0.y, q8.y), F), xb1 = basis_one(pk2(q1.y, q9.y), F);
        unsigned ah[4], al[4];
        {
            const f32x2 s = pk2(ys, ys);
            float c0, c8, c1, c9;
            upk2(mul2(basis_one(pk2(q0.z, q8.z), F), s), c0, c8);
            upk2(mul2(basis_one(pk2(q1.z, q9.z), F), s), c1, c9);
            split_f16(yv[0].x * c0, yv[2].x * c1, ah[0], al[0]);
            split_f16(yv[0].y * c0, yv[2].y * c1, ah[1], al[1]);
            split_f16(yv[1].x * c8, yv[3].x * c9, ah[2], al[2]);
            split_f16(yv[1].y * c8, yv[3].y * c9, ah[3], al[3]);
        }
        if (cell != cur) {
            if (cur >= 0) {
                const int step = (cur >> 8) == (cell >> 8) ? (cell & 255) - (cur & 255) : NP;   // cells ascend
                advance(step > 0 && step < NP ? step : NP);
            }
            cur = cell;
        }
        __syncwarp();   // the weights are visible
#pragma unroll
        for (int s = 0; s < MR; ++s) {
            const float4 w0 = psi[8 * s + 2 * t], w1 = psi[8 * s + 2 * t + 1];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float p0, p8, p1, p9;
                upk2(mul2(h ? pk2(w0.z, w0.w) : pk2(w0.x, w0.y), xb0), p0, p8);
                upk2(mul2(h ? pk2(w1.z, w1.w) : pk2(w1.x, w1.y), xb1), p1, p9);
                unsigned bh0, bl0, bh1, bl1;
                split_f16(p0, p1, bh0, bl0);
                split_f16(p8, p9, bh1, bl1);
                float e[4];
                mma_f16_k16_0(e, al, bh0, bh1);
                mma_f16_k16(e, ah, bl0, bl1);
                mma_f16_k16(e, ah, bh0, bh1);
                d[2 * s + h][0] = add2(d[2 * s + h][0], pk2(e[0], e[1]));
                d[2 * s + h][1] = add2(d[2 * s + h][1], pk2(e[2], e[3]));
            }
        }
    }
    cp_async_wait0();
    if (cur >= 0) advance(NP);
}

// O3: the plan (or batch) has third-order terms
template <int MR, typename G, bool O3>
__global__ void __launch_bounds__(O3 ? ST3_THREADS : ST_THREADS, O3 ? ST3_CTAS_PER_SM : ST_CTAS_PER_SM)
spread_tiles(DevPlan single, BatchArgs B, const float2 *__restrict__ y_base, int n_items, int *counter,
             long long max_grid_bytes) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_item;
    constexpr int NT = O3 ? ST3_THREADS : ST_THREADS, NW = NT / 32;
    float2 *S = (float2 *)smem;
    const int tid = threadIdx.x, warp = tid >> 5;
    float *ones = (float *)(smem + max_grid_bytes);
    unsigned char *buf = smem + max_grid_bytes + ST_ONE_BYTES + warp * ST_WARP_BYTES;
    if (tid < 32) ones[tid] = 1.f;   // visible after the first item's barriers
    for (;;) {
        if (tid == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= n_items) break;
        const int4 itm = B.items[item];
        const DevPlan &P = B.plans ? B.plans[itm.x] : single;
        if (P.skip && *P.skip) continue;
        const int term = P.act[itm.y];
        const Term &T = P.terms[term];
        const int elems = (int)(T.grid_bytes / (long long)sizeof(G));   // the shared copy is FP32 complex
        float4 *S4 = (float4 *)S;
        for (int e = tid; e < elems / 2; e += NT) S4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        const float2 *y = y_base + P.vec_node_off;
        const int nt = P.tile_count[term];
        const int t0 = (int)((long long)nt * itm.z / itm.w), t1 = (int)((long long)nt * (itm.z + 1) / itm.w);
        const int per = (t1 - t0 + NW - 1) / NW;
        const int a = t0 + warp * per, b = min(t1, a + per);
        __syncthreads();   // grid zeroed before any addition
        if (a < b) {
            const float4 *rec = P.srec + T.rec_off + (long long)a * tile_f4(T.order);
            const int *cells = P.tile_cell + T.tile_off + a;
            const Window *wr = P.windows + T.wr, *wc = P.windows + T.wc;
            if (O3 && T.order == 3) {
                const float ys = scale_to((unsigned)P.err[ERR_YMAX], 14);
                const float inv = __int_as_float((254 - (__float_as_int(ys) >> 23)) << 23);
                spread_run3<MR>(rec, cells, b - a, y, S, T, wr, wc, ys, inv, buf);
            } else if (T.order == 2) {
                spread_run12<MR, true>(rec, cells, b - a, y, S, T.stride, &wr->ch[0][0], &wc->ch[0][0],
                                                    buf, ones);
            } else {
                spread_run12<MR, false>(rec, cells, b - a, y, S, T.stride, nullptr, &wc->ch[0][0], buf,
                                                     ones);
            }
        }
        __syncthreads();
        if constexpr (std::is_same<G, float2>::value) {
            float4 *dst = (float4 *)(P.partials + (long long)itm.z * P.grid_elems + T.grid_off);
            for (int e = tid; e < elems / 2; e += NT) dst[e] = S4[e];
        } else {
            G *dst = (G *)P.partials + (long long)itm.z * P.grid_elems + T.grid_off;
            for (int e = tid; e < elems; e += NT) dst[e] = GridEl<G>::store(S[e].x, S[e].y);
        }
        __syncthreads();
    }
}

static size_t spread_tiles_smem(long long sgrid, bool order3) {
    return (size_t)sgrid + ST_ONE_BYTES + ST_WARP_BYTES * ((order3 ? ST3_THREADS : ST_THREADS) / 32);
}

int spread_tiles_ctas_per_sm(long long sgrid, bool order3) {
    const size_t per = spread_tiles_smem(sgrid, order3) + 1024 + 16;   // + the per-CTA reserve and the static words
    return (int)std::max<size_t>(1, std::min<size_t>(order3 ? ST3_CTAS_PER_SM : ST_CTAS_PER_SM, (size_t)(MAX_SMEM + 1024) / per));
}

template <typename G>
static void launch(cudaStream_t st, const DevPlan &v, const BatchArgs &B, const float2 *y, int n_items, bool order3,
                   int *counter, long long sgrid, int sm_count, int mr) {
    static std::atomic<unsigned long long> attr_seen{0};
    once_per_device(attr_seen, [] {
        cudaFuncSetAttribute(spread_tiles<3, G, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(spread_tiles<4, G, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(spread_tiles<3, G, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
        cudaFuncSetAttribute(spread_tiles<4, G, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_MAX_SMEM);
    });
    if (n_items <= 0) return;
    const int c = std::max(1, std::min(n_items, spread_tiles_ctas_per_sm(sgrid, order3) * sm_count));
    auto k = mr <= 3 ? (order3 ? spread_tiles<3, G, true> : spread_tiles<3, G, false>)
                     : (order3 ? spread_tiles<4, G, true> : spread_tiles<4, G, false>);
    k<<<c, order3 ? ST3_THREADS : ST_THREADS, spread_tiles_smem(sgrid, order3), st>>>(v, B, y, n_items, counter, sgrid);
}

// the spread of items [0, n_items) of one problem (B.plans == null) or a batch;
// sgrid: bytes of the largest grid in FP32
void spread_tiles_launch(cudaStream_t st, const DevPlan &v, const BatchArgs &B, const float2 *y, int n_items,
                         bool order3, int *counter, long long sgrid, int sm_count, int mr, int prec) {
    auto run = prec == ANOVA_PREC_F16 ? launch<__half2> : prec == ANOVA_PREC_BF16 ? launch<__nv_bfloat162> : launch<float2>;
    run(st, v, B, y, n_items, order3, counter, sgrid, sm_count, mr);
}

}  // namespace agft
