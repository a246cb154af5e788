// Cell-aligned node tiles: the sorted node records of the tensor-core kernels.
//
// The nodes of a term are sorted by grid cell and every cell's nodes fill whole
// tiles of 16, the last one padded, so that a tile lies in one cell and the
// kernels test for a new cell once per tile instead of masking groups that
// straddle two.  Padding costs 6 % of the tiles at 122 nodes per cell and a
// third at 24, where the straddling groups of an unpadded order cost more (they
// run once per cell they touch).
//
// A tile stores what one lane of a warp needs side by side, position p < 8 pairing
// nodes p and p + 8:
//   order <= 2 (192 bytes): float4 (vr_p, vr_p+8, vc_p, vc_p+8) for p < 8, then
//     the 16 original indices as int2 (index_p, index_p+8);
//   order 3 (256 bytes): float4 (va, vb, vc, index bits) per node;
// v = 2 tau - 1 is the window argument along a row axis or the column axis (vr = 0
// for order 1); padding has index -1 and arguments 0.  Built in sort.cu by the same
// FP32 operations the unsorted kernels apply.  (Order 2 with one float4 per node:
// gather 1.86 instead of 1.71 ms at d = 20, M = 1e6; with (vr, vc) pairs and indices
// apart 1.88; through a cp.async ring in shared memory 2.03.)
//
// One int per tile names its cell: order <= 2 the stored-grid offset of the
// first tap, order 3 a | b << 8 | c << 16 (grid indices of the two row axes and
// the column; n <= 23); TILE_HALF is set when nodes 8..15 are all padding.
// Third-order cells run with the first row axis fastest, so that neighbouring
// cells share all but one of the grid planes their windows touch.
#pragma once

#include "device.cuh"

namespace agft {

constexpr int TILE = 16;
constexpr int TILES_MAX_SMEM = MAX_SMEM - 1024;   // dynamic shared memory beside a few static words
constexpr int TILE_HALF = 1 << 30;
__host__ __device__ constexpr int tile_f4(int order) { return order == 3 ? 16 : 12; }   // float4 per tile
// most tiles that M nodes in `cells` cells can fill
inline long long tile_capacity(long long M, long long cells) { return M / TILE + (M < cells ? M : cells) + 1; }
constexpr int TILE_SLACK = 4;   // tiles allocated behind the last term's: the kernels' loads run ahead of a run's end

// ---- the product basis ----
//
// Phi_i(v) = v^{i0} T_2(v)^{i1} T_4(v)^{i2}, i = i0 + 2 i1 + 4 i2 < 8, spans the
// polynomials of degree 7 as the Chebyshev polynomials do, its functions are
// bounded by 1 on [-1, 1], and unlike the three-term recurrence one function
// costs a lane three factors, whichever one it holds (Window::pb).
//
// With s = v^2: T_2 = 2 s - 1 and T_4 = s (8 s - 8) + 1; a factor that a function
// lacks is 1, so every lane runs the same operations with its own constants.
struct BasisFactors {   // of the lane's function i: v or 1 = a0 v + b0; T_2 or 1 = a1 s + b1; T_4 or 1 = s (c s - c) + 1
    f32x2 a0, b0, a1, b1, c;
};
__device__ __forceinline__ f32x2 dup2(float a) { return pk2(a, a); }
__device__ __forceinline__ BasisFactors basis_factors(int i) {
    BasisFactors F;
    F.a0 = dup2(i & 1 ? 1.f : 0.f);
    F.b0 = dup2(i & 1 ? 0.f : 1.f);
    F.a1 = dup2(i & 2 ? 2.f : 0.f);
    F.b1 = dup2(i & 2 ? -1.f : 1.f);
    F.c = dup2(i & 4 ? 8.f : 0.f);
    return F;
}
__device__ __forceinline__ f32x2 t4_factor(f32x2 s, f32x2 c) {
    return fma2(mul2(c, s), sub2(s, dup2(1.f)), dup2(1.f));
}
// Phi_i of two arguments
__device__ __forceinline__ f32x2 basis_one(f32x2 v, const BasisFactors &F) {
    const f32x2 s = mul2(v, v);
    return mul2(mul2(fma2(F.a0, v, F.b0), fma2(F.a1, s, F.b1)), t4_factor(s, F.c));
}
// Phi_i and Phi_i+1 = v Phi_i of two arguments, i even
__device__ __forceinline__ void basis_even_odd(f32x2 v, const BasisFactors &F, f32x2 &even, f32x2 &odd) {
    const f32x2 s = mul2(v, v);
    even = mul2(fma2(F.a1, s, F.b1), t4_factor(s, F.c));
    odd = mul2(v, even);
}
// Phi_i .. Phi_i+3 of two arguments, i = 0 or 4 (c = 0 or 8)
__device__ __forceinline__ void basis_four(f32x2 v, f32x2 c, f32x2 (&x)[4]) {
    const f32x2 s = mul2(v, v), T2 = fma2(dup2(2.f), s, dup2(-1.f));
    x[0] = t4_factor(s, c);
    x[1] = mul2(v, x[0]);
    x[2] = mul2(T2, x[0]);
    x[3] = mul2(v, x[2]);
}

// d = a b (the zero accumulator is no register)
__device__ __forceinline__ void mma_tf32_0(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// d += a b and d = a b with both operands in high and low parts
__device__ __forceinline__ void mma3_tf32(float (&d)[4], const unsigned (&ah)[4], const unsigned (&al)[4],
                                          unsigned bh0, unsigned bh1, unsigned bl0, unsigned bl1) {
    mma_tf32(d, al, bh0, bh1);
    mma_tf32(d, ah, bl0, bl1);
    mma_tf32(d, ah, bh0, bh1);
}
__device__ __forceinline__ void mma3_tf32_0(float (&d)[4], const unsigned (&ah)[4], const unsigned (&al)[4],
                                            unsigned bh0, unsigned bh1, unsigned bl0, unsigned bl1) {
    mma_tf32_0(d, al, bh0, bh1);
    mma_tf32(d, ah, bl0, bl1);
    mma_tf32(d, ah, bh0, bh1);
}

// The tensor core cuts its sums off at 24 bits where FP32 rounds them.  A stage of the
// split products leaves its value short by 2^-24 of it on average: half a unit of the last
// place, 0.72 x 2^-24 of a value with an evenly spread mantissa, and what smaller addends
// lose where they are aligned to it.  The gather's stages (two window products, the basis
// sum; order 1 has one window product) so left f short by 3 and 1.9 x 2^-24 (measured
// against FP64 plans on the same window, N = 4 .. 64), the larger part of its error beside
// the CUDA cores'.  The window values take it back in between, once per cell: error of f
// against 64-bit sums at order 2, N = 32 2.47e-7 -> 1.65e-7 (CUDA cores 1.48), orders 1 to 3,
// N = 36/32/4 2.63 -> 1.95 (1.79); d = 20, M = 1e6 1.660 -> 1.662 ms, 0.7 % at three nodes per cell.
__device__ __forceinline__ float uncut(float h, float stages) { return fmaf(h, stages * 0x1p-24f, h); }

// ---- FP16 tensor-core products of scaled operands ----
//
// x = h + l with h the nearest FP16 value and l the remainder rounded to FP16: for |x|
// in [2^-3, 2^15] the two hold 22 bits of x, and below that the error is at most 2^-25
// in absolute size.  Operands bounded by 1 are used as they are; others are scaled by a
// power of two to a maximum near 2^14, so what is lost is below 2^-22 of the value or
// 2^-39 of the largest one.  Products are h h + l h + h l as in the TF32 form, at twice
// its rate (m16n8k16).  h is rounded, not cut off: remainders of one sign left out a
// product l l of the result's own sign, 1.2e-7 of the adjoint (d = 10, M = 5e5 adjoint
// 3.11 -> 3.14 ms, forward 2.94 -> 2.95; rounding by the TF32 form's packed split: 3.56).
// Fragments (PTX ISA), lane = 4 g + t: A (16 x 16) a0 = A[g][2t, 2t+1], a1 =
// A[g + 8][2t, 2t+1], a2 = A[g][2t + 8, 2t + 9], a3 = A[g + 8][2t + 8, 2t + 9]; B
// (16 x 8) b0 = B[2t, 2t+1][g], b1 = B[2t + 8, 2t + 9][g]; the k8 form has a0, a1
// and b0 only; D as in the TF32 form.
__device__ __forceinline__ unsigned pack_f16(float lo, float hi) {
    unsigned r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// (x0, x1) in high parts and remainders
__device__ __forceinline__ void split_f16(float x0, float x1, unsigned &h, unsigned &l) {
    const __half2 hh = __floats2half2_rn(x0, x1);
    const float2 hf = __half22float2(hh);
    h = *(const unsigned *)&hh;
    l = pack_f16(x0 - hf.x, x1 - hf.y);
}
__device__ __forceinline__ void mma_f16_k16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_k16_0(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_f16_k8_0(float (&d)[4], unsigned a0, unsigned a1, unsigned b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%7, %7, %7, %7};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0), "f"(0.f));
}

// power of two that takes values of magnitude at most m (bits of a non-negative
// float) to at most 2^top; 1 for zero, infinite and NaN m
__device__ __forceinline__ float scale_to(unsigned mbits, int top) {
    const int e = (int)(mbits >> 23);   // m < 2^(e - 126)
    if (mbits == 0u || e == 255) return 1.f;
    return __int_as_float(min(253, max(1, 127 + top - (e - 126))) << 23);
}

}  // namespace agft
