// Forward grouped transform f = F fhat (Definition "grouped Fourier transform"
// and eq. (somafm), Sec. 3), FP32.
//
//   1. trafo_pre: per term, zero-extend the block fhat(u) to ghat(u) on the
//      n^{|u|} grid (the extension before eq. (somafm)), multiply by the
//      deconvolution factors, run the oversampled FFT (sign +) in shared
//      memory and store the grid with its halos.
//   2. gather: all terms fused, point-major.  A CTA owns a tile of 128 nodes;
//      each half-warp owns 8 nodes and evaluates them one at a time with its
//      16 lanes = 2 rows x 8 columns of the window, reading the term's grid from
//      shared memory (double-buffered bulk async copies from L2).  Lanes keep
//      per-node partial sums over all terms in registers; one transposed
//      reduce-scatter per tile leaves node i's value in lane i.
#include <cstdio>
#include <cstring>

#include "device.cuh"
#include "internal.cuh"

namespace agft {

// ------------------------------------------------------------ pre-pass ----

// One block per active term.  grids stored as G (FP32 complex, or a pair of
// 16-bit floats rounded from the FP32 FFT).  With fixed-point accumulators
// (P.fexp) the block also sums |Re| + |Im| of its block of fhat into
// part[blockIdx.x], and the last block of a problem to finish turns the sums
// (added in a fixed order) into the accumulators' exponent, which saves two
// launches on the smallest problems' critical path.
template <typename G>
__device__ __forceinline__ void trafo_pre_body(const DevPlan &single, const BatchArgs &B,
                                               const float2 *__restrict__ fhat_base, double *part) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double sh[32];
    __shared__ int s_last;
    const int pb = B.plans ? B.blk_prob[blockIdx.x] : 0;
    const DevPlan &P = B.plans ? B.plans[pb] : single;
    const int blk0 = B.plans ? B.blk0[pb] : 0;
    const int sblk = (int)blockIdx.x - blk0;
    if (P.skip && *P.skip) return;
    const float2 *fhat = fhat_base + P.vec_coef_off;
    G *grids = (G *)P.grids;
    const Term T = P.terms[P.act[sblk]];
    const int n = T.n, s = T.order, N = T.N;
    int fe = n;
    for (int j = 1; j < s; ++j) fe *= n;
    float2 *a = (float2 *)smem_raw;
    float2 *b = a + fe;
    for (int i = threadIdx.x; i < fe; i += blockDim.x) a[i] = make_float2(0.f, 0.f);
    __syncthreads();
    // zero-extended, deconvolved coefficients at k mod n
    double l1 = 0.0;
    const int len = (int)T.coef_len;
    if (T.basis == ANOVA_BASIS_COS) {
        // cosine term: the coefficient at its 2^s mirrored frequencies
        for (int q = threadIdx.x; q < len; q += blockDim.x) {
            int k[3];
            cos_decode(q, s, N, k);
            const float2 c = fhat[T.coef_off + q];
            l1 += fabs((double)c.x) + fabs((double)c.y);
            for (int sg = 0; sg < (1 << s); ++sg) {
                float D = (float)cos_amp(s);
                const int pos = cos_mirror(k, s, sg, N, n, P.deconv, T.dc_off, T.dr_off, D);
                a[pos] = make_float2(c.x * D, c.y * D);
            }
        }
    } else {
        const FastDiv by_Nm(N - 1);
        for (int q = threadIdx.x; q < len; q += blockDim.x) {
            float D;
            const int pos = exp_position(q, s, N, n, by_Nm, P.deconv, T.dc_off, T.dr_off, D);
            const float2 c = fhat[T.coef_off + q];
            l1 += fabs((double)c.x) + fabs((double)c.y);
            a[pos] = make_float2(c.x * D, c.y * D);
        }
    }
    // FFT along every axis (sign +): g_q = sum_k ghat_k exp(+2 pi i k q / n)
    const float2 *cur = grid_fft<float2, float>(a, b, n, s, +1);
    // store with halos
    G *g = grids + T.grid_off;
    const FastDiv by_cols(T.stride);
    const int total = T.erows * T.stride;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        int ec;
        const int er = by_cols.div(e, ec);
        float2 v = make_float2(0.f, 0.f);
        if (s <= 2) {
            if (ec < n + 2 * T.hc + 1) {
                const int qc = wrap(ec - T.hc, n);
                const int qr = s == 2 ? wrap(er - T.hr, n) : 0;
                v = cur[qr * n + qc];
            }
        } else {
            if (ec < n) v = cur[er * n + ec];
        }
        g[e] = GridEl<G>::store(v.x, v.y);
    }
    if (!P.fexp) return;
    // fixed-point exponent e for the accumulators: 2^e * 2 sum |fhat| <= 2^62
    // (every partial sum of a node's terms is bounded by sum_k |fhat_k| of the
    // active blocks up to the window error), clamped so that 2^e stays a normal
    // float.  The sums are added in a fixed order, so e never depends on timing.
    if (sblk == 0 && threadIdx.x == 0)
        for (int i = 0; i < P.n_empty; ++i) {
            const float2 c = fhat[P.empty_off[i]];
            l1 += fabs((double)c.x) + fabs((double)c.y);
        }
    l1 = block_sum_fixed(l1, sh);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = l1;
        __threadfence();
        s_last = atomicAdd(P.fexp + 1, 1) == P.n_act - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double sum = 0.0;
    for (int i = threadIdx.x; i < P.n_act; i += blockDim.x) sum += __ldcg(part + blk0 + i);
    sum = block_sum_fixed(sum, sh);
    if (threadIdx.x == 0) {
        int e = 100;
        // a cosine coefficient stands for 2^s exponential ones of 2^{-s/2} its size
        // (s <= 3): their absolute sum is at most 2^{3/2} = 2.83 times larger
        const bool finite = sum <= 1.7976931348623157e308;
        if (sum > 0 && finite) e = 61 - (int)ceil(log2(sum)) - (P.basis == ANOVA_BASIS_COS ? 2 : 0);
        P.fexp[0] = max(-100, min(100, e));
        P.fexp[1] = 0;
        P.fexp[2] = !finite;   // fixed point holds no infinity: the finish writes NaN
    }
}

__global__ void __launch_bounds__(FFT_THREADS)
trafo_pre_f32(DevPlan single, BatchArgs B, const float2 *__restrict__ fhat_base, double *part) {
    trafo_pre_body<float2>(single, B, fhat_base, part);
}
__global__ void __launch_bounds__(FFT_THREADS)
trafo_pre_f16(DevPlan single, BatchArgs B, const float2 *__restrict__ fhat_base, double *part) {
    trafo_pre_body<__half2>(single, B, fhat_base, part);
}
__global__ void __launch_bounds__(FFT_THREADS)
trafo_pre_bf16(DevPlan single, BatchArgs B, const float2 *__restrict__ fhat_base, double *part) {
    trafo_pre_body<__nv_bfloat162>(single, B, fhat_base, part);
}

// ------------------------------------------------------- empty plan case --

__global__ void fill_const_f32(float2 *f, long long M, const float2 *__restrict__ fhat, const long long *eoff,
                               int n_empty, const int *skip) {
    if (skip && *skip) return;
    float2 c0 = make_float2(0.f, 0.f);
    for (int e = 0; e < n_empty; ++e) {
        float2 c = fhat[eoff[e]];
        c0.x += c.x;
        c0.y += c.y;
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < M; i += (long long)gridDim.x * blockDim.x)
        f[i] = c0;
}

int launch_trafo_f32(Plan &p, const float2 *fhat, float2 *f) {
    DevPlan v = dev_view(p);
    if (p.n_act == 0) {
        int blocks = (int)std::min<long long>(1024, (p.M + 255) / 256);
        fill_const_f32<<<blocks, 256, 0, p.stream>>>(f, p.M, fhat, p.empty_off, p.n_empty, p.skip);
        return cuda_status(cudaGetLastError());
    }
    if (p.direct) return launch_direct_trafo(p, fhat, f);
    const size_t pre_smem = fft_smem_bytes<float2>(p.max_fft_elems, p.max_n);
    static std::atomic<unsigned long long> attr_seen{0};
    once_per_device(attr_seen, [] {
        cudaFuncSetAttribute(trafo_pre_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, FFT_MAX_SMEM);
        cudaFuncSetAttribute(trafo_pre_f16, cudaFuncAttributeMaxDynamicSharedMemorySize, FFT_MAX_SMEM);
        cudaFuncSetAttribute(trafo_pre_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize, FFT_MAX_SMEM);
    });
    stage_begin(p, ST_PRE);
    BatchArgs B;
    std::memset(&B, 0, sizeof(B));
    auto pre = p.precision == ANOVA_PREC_F16 ? trafo_pre_f16 : p.precision == ANOVA_PREC_BF16 ? trafo_pre_bf16 : trafo_pre_f32;
    pre<<<p.n_act, FFT_THREADS, pre_smem, p.stream>>>(v, B, fhat, (double *)p.scratch);
    stage_end(p, ST_PRE);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e);
    stage_begin(p, ST_GATHER);
    int rc;
    if (p.srec && p.facc && p.precision == ANOVA_PREC_F32 && p.n_act3 == 0)
        rc = launch_gather_sorted_f32(p, fhat, f);   // every term over its cell-sorted records
    else
        rc = launch_gather_f32(p, fhat, f);
    stage_end(p, ST_GATHER);
    return rc;
}

}  // namespace agft
