// Internal definitions shared by the CUDA translation units of the library.
//
// Method: grouped Fourier transform of Sec. 3 (Definition "grouped Fourier
// transform", identity eq. (somafm), stacked adjoint), evaluated per ANOVA term
// with an NFFT: deconvolution by the window's Fourier coefficients, an
// oversampled FFT, and a Kaiser--Bessel window gather (forward) or spread
// (adjoint).  The window is
//     psi(d) = sinh(b sqrt(m^2 - d^2)) / (pi sqrt(m^2 - d^2)),  |d| <= m,
// in grid units d = n x - q, with b = pi (2 - 1/sigma), sigma = n/N, and
// Fourier transform (1/n) I_0(m sqrt(b^2 - (2 pi k / n)^2)) of psi(n x).
#pragma once

#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>
#include <cstddef>
#include <new>

#include "anova_gft.h"

namespace agft {

constexpr int MAX_ORDER = 3;
constexpr int MAXM = 8;          // largest window half-width
constexpr int NCOEF = 8;         // coefficients of the per-tap polynomial (degree 7)
constexpr int GATHER_TILE = 128;   // nodes per gather tile (gather.cu)
constexpr int SPREAD_THREADS = 256;
constexpr int SPREAD_MAX_CTAS_PER_SM = 4;
constexpr int SPREAD_MAX_K = 64;     // largest number of node chunks (partial grids) per term
constexpr int MAX_SMEM = 227 * 1024;

// One window shape (half-width m, oversampling sigma).  Tap j of a node with
// grid position t = n x sits at grid index floor(t) - m + 1 + j and has weight
// psi(tau + m - 1 - j) / psi(0), tau = t - floor(t); the weight is stored as a
// degree-7 polynomial in v = 2 tau - 1 (Chebyshev interpolation, monomial form).
// The same polynomial in the Chebyshev basis: tap j = sum_i ch[j][i] X_i(v) with
// X_i = s_i T_i, signs s = (+, +, -, -, +, +, -, -), which turn the three-term
// recurrence into X_{i+1} = X_{i-1} + (-1)^i 2 v X_i (one fma per step).
struct Window {
    float c[2 * MAXM][NCOEF];
    float ch[2 * MAXM][NCOEF];
    float pb[2 * MAXM][NCOEF];   // the same polynomials in the product basis (tiles.cuh)
    int m;
    float b;          // shape parameter pi (2 - 1/sigma)
    float inv_psi0;   // 1 / psi(0)
    double bd, inv_psi0d;
};

// A term in kernel schedule order.  Grid layout: erows x stride (complex
// elements), the last coordinate of the term along a row.  Orders 1 and 2
// store halos so that a window never wraps: periodic column q sits at stored
// column q + hc (hc = m_col - 1) and the stored columns q + hc +- n repeat it;
// order-2 rows likewise with hr = m_row - 1.  Order-3 grids have no halo: the
// row index is i_first * n + i_second and all indices wrap modulo n.  The row
// stride is = 8 (mod 16) complex elements, so two consecutive rows of eight
// columns fall in complementary shared-memory bank halves.
struct Term {
    int order;          // 1..3 (the empty set is handled separately)
    int col;            // coordinate along the row
    int row0, row1;     // other coordinates (-1 if absent)
    int N, n, stride;
    int rows;           // n^(order-1)
    int wc, wr;         // window ids: column axis, row axes
    int mc, mr;         // their half-widths
    int new_rowgroup;   // 1 if the row weights cached by the gather must be recomputed
    int hr, hc;         // halo widths (rows, columns): stored index = periodic index + halo
    int erows;          // stored rows (order 2: n + 2 hr + 1; order 1: 1; order 3: n^2, no halo)
    int sort_slot;      // slot of this term's cell-sorted node copy (-1: none)
    long long rec_off;  // node tiles: first record (float4 units) and first tile
    long long tile_off;
    long long grid_off;   // element offset in the grid buffer
    long long grid_bytes; // bytes (multiple of 16)
    long long coef_off;   // offset in the coefficient vector
    long long coef_len;
    int dc_off, dr_off;   // offsets of the column / row deconvolution factors
    int user_index;
    int slot_c;           // FP64 plans: window-table slots of the column and row coordinates
    int slot_r0, slot_r1;
    int basis;            // ANOVA_BASIS_EXP, or ANOVA_BASIS_COS (N above is then the doubled bandwidth)
};

// What the forward gather needs of an active term, in one 48-byte record
// (prefetched by every warp one term ahead).
struct ActRec {
    int order, newgroup;   // newgroup: 1 if the row weights must be recomputed
    int wc, wr;            // window ids (column axis, row axes)
    int col, row0, n, stride;
    long long grid_off;
    int grid_bytes, term;  // term: index into the term table
};

inline ActRec make_act_rec(const Term &T, int term, int newgroup) {
    ActRec a;
    a.order = T.order;
    a.newgroup = newgroup;
    a.wc = T.wc;
    a.wr = T.wr;
    a.col = T.col;
    a.row0 = T.row0;
    a.n = T.n;
    a.stride = T.stride;
    a.grid_off = T.grid_off;
    a.grid_bytes = (int)T.grid_bytes;
    a.term = term;
    return a;
}

// A node in the cell order of one term, plans whose cell products run on the
// CUDA cores and FP64 plans (16 bytes, stored as float4; the tensor-core kernels'
// tiles: tiles.cuh):
//   x: 2 tau_row - 1 (order 2; 0 for order 1), y: 2 tau_col - 1, the window
//   polynomial arguments of the node's fractional grid positions;
//   z (int bits): stored-grid offset of the first tap, i_row * stride + i_col
//   (order 1: i_col), which identifies the cell;
//   w (int bits): the node's original index.
// Built in sort.cu by the same FP32 operations the unsorted kernels apply.

// Direct summation (direct.cu): a term as its kernels need it, and an adjoint item.
struct DirectTerm {
    int order, K;            // K: frequencies per axis
    int col, row0, row1;
    int coef_off;
    int group, pad;          // frequency or row group of the unit
};
struct DirectItem {
    int act, chunk, chunks, pad;   // active term (-1: the empty set), node chunk of chunks
    DirectTerm term;
};
constexpr int DA_MAX_ACC = 192;                // partial sums of an adjoint item

// Device-visible view of a plan (passed by value to kernels).
struct DevPlan {
    int d;
    long long M;
    int n_terms;              // scheduled (non-empty) terms
    int n_empty;              // empty-set terms
    const float *x;           // [d][M] FP32 nodes (or null)
    const double *xd;         // [d][M] FP64 nodes (or null)
    const float2 *z;          // [d][M] exp(2 pi i x), plans summed directly (or null)
    const Term *terms;
    const Window *windows;
    const float *deconv;      // deconvolution factors
    const double *deconvd;
    const long long *empty_off;  // coefficient offsets of the empty terms
    long long grid_elems;     // total grid elements (complex)
    long long max_grid_bytes;
    int *err;                 // device error word (bounded waits)
    const int *act;           // active schedule: indices into terms, n_act entries
    const ActRec *act_rec;    // per active entry: the gather's view of the term
    int n_act;
    const int *skip;          // if non-null and nonzero, kernels return at once
    const float2 *grids;      // stored grids of this problem
    float2 *partials;         // adjoint partial grids [spread_chunks][grid_elems]
    int spread_chunks;        // node chunks of the adjoint (one partial grid each)
    const float4 *srec;       // nodes sorted by grid cell: [slot][M] records, or node tiles if tile_cell is set
    const float4 *frec;       // records of the forward on the CUDA cores (srec, or a copy beside tiles; null: tiles only)
    const int *tile_cell;     // cell of every tile (null: srec holds records)
    const int *tile_count;    // tiles per scheduled term
    unsigned long long *facc; // sorted forward: fixed-point accumulators [M][2] (or null), zero between calls
    int *fexp;                // their exponent, a block counter (zero between launches), 1 if a coefficient is not finite
    long long n_coeffs;
    long long vec_node_off;   // offset of this problem's nodes in batched node vectors
    long long vec_coef_off;   // offset of this problem's coefficients in batched coefficient vectors
    int basis;                // ANOVA_BASIS_EXP or ANOVA_BASIS_COS
};

// Work lists of a launch over several problems (a batch).  With plans == null
// the launch covers the single problem given by the DevPlan parameter and
// every table below is unused.
struct BatchArgs {
    const DevPlan *plans;     // device array [P]
    int P;
    const int *tile_prob;     // gather: problem of each tile of 128 nodes
    const int *tile0;         // first tile of each problem
    const int4 *items;        // spread work items (problem, active term, node chunk, chunks)
    const int *blk_prob;      // pre/post: problem of each (problem, active term) block
    const int *blk0;          // first block of each problem
};

// words of DevPlan::err: the error code of bounded waits; 1 if a node coordinate is not
// finite; the largest |Re|, |Im| of the adjoint's input (float bits, zero between calls)
enum { ERR_CODE = 0, ERR_NODE = 1, ERR_YMAX = 2 };

constexpr int N_STAGES = 7;
// How a plan keeps its nodes, and so which kernels read them.
enum NodeForm {
    FORM_NONE = 0,      // no sorted copy: point-major gather, spread with per-node atomics
    FORM_RECORDS = 1,   // cell-sorted records: CUDA cores
    FORM_TILES = 2,     // node tiles: tensor cores
    FORM_DIRECT = 3     // no grid either: direct sums
};
// The form in which a batch's kernels can read all its problems' nodes: tiles and
// records are laid out differently, and a kernel reads one of them, so a batch that
// holds both runs over the nodes in their own order.
int batch_form(const int *forms, int n);

struct Profiler;   // per-stage CUDA-event timing (profile.cu)

struct Plan {
    Profiler *prof;
    int device;
    cudaStream_t stream;
    int precision;
    int basis;              // ANOVA_BASIS_EXP or ANOVA_BASIS_COS
    double eps;             // target relative error of the transforms
    int d;
    long long M;
    int n_user_terms;
    long long n_coeffs;
    // host copies
    Term *h_terms;
    int n_terms;
    int n_empty;
    long long *h_user_off;  // per user term: coefficient offset
    long long *h_user_len;
    int *h_user_n, *h_user_mc, *h_user_mr, *h_user_order;
    // device memory: parts of arena, the sorted copies and accumulators of arena_opt
    void *arena, *arena_opt;
    void *x;                // FP32 or FP64 nodes [d][M]
    Term *terms;
    Window *windows;
    int n_windows;
    float *deconv;
    double *deconvd;
    long long *empty_off;
    void *grids;            // complex grid buffer (precision dependent)
    long long grid_elems;
    long long max_grid_bytes;
    int max_fft_elems;      // largest n^order
    int max_n;              // largest n
    int max_stage;          // largest staged halo grid of the adjoint's fold (elements)
    int pitch2;             // row pitch shared by all order-2 grids
    // active term list (all scheduled terms unless a group mask restricts it)
    int *act;
    ActRec *act_rec;
    ActRec *act_rec3;       // active third-order terms without sorted records (point-major gather)
    int n_act3;
    int n_act;
    int *h_act;
    const int *skip;        // device flag read by every transform kernel (or null)
    void *partials;         // adjoint partial grids [spread_kmax][grid_elems]
    int spread_kmax;        // partial grids allocated (largest chunk count per term)
    int spread_K;           // node chunks per term for the current active list
    int4 *items;            // spread work items (device, n_terms * spread_kmax slots)
    int4 *h_items;
    int n_items;
    int n_items3;           // the first n_items3 items are those of third-order terms
    int *counter;           // work-queue counters (2), zero between calls
    float4 *srec;           // cell-sorted node records (null: none), n_sorted slots of M
    bool cell_tc;           // srec holds node tiles: cell products on the tensor cores
    float4 *frec;           // records beside tiles, for the forward (n_frec slots of M; null: none)
    int n_frec;
    int *tile_cell;         // tiles: their cells, and the tiles per scheduled term
    int *tile_count;
    int n_sorted;
    unsigned long long *facc;   // sorted forward: fixed-point accumulators [M][2]
    int *fexp;              // and their exponent
    // plans of small bandwidths, summed directly (direct.cu)
    bool direct;
    float2 *z;              // [d][M] exp(2 pi i x)
    float *direct_part;     // partial sums of the adjoint's items
    int *direct_count;      // finished blocks per active term and of the empty set, zero between calls
    int direct_kt;          // powers per coordinate of the forward's table
    int direct_npl, direct_split;   // forward: nodes per lane, sets of terms per node block
    float2 *direct_fpart;   // their sums [direct_split][M] (one set: null), finished CTAs per node block
    int *direct_fcount;
    bool direct_big;        // adjoint: the kernel for many sums per item
    DirectTerm *direct_units, *h_units;    // forward work units of the active terms
    DirectItem *direct_items, *h_ditems;   // adjoint work items (n_items of them)
    int n_direct_units;
    // FP64 plans: window weights per (window, coordinate) slot and node, the
    // precomputed form of psi (taps 0..2m-1, zero padded to 8), and the first
    // tap's grid index floor(n x + n/2) in [0, n)
    double *wt64;           // [n_slots][M][8]
    int *wb64;              // [n_slots][M]
    int4 *slots64;          // per slot: (window id, coordinate, n, m)
    int n_slots64;
    int gather_ctas;
    int *err;
    void *scratch;          // reduction scratch
    size_t scratch_bytes;
    int sm_count;
    void *solver;           // solver workspaces (solvers.cu), created on first use
    void (*solver_free)(void *);
};

DevPlan dev_view(const Plan &p);
inline int node_form(const Plan &p) {
    return p.direct ? FORM_DIRECT : !p.srec ? FORM_NONE : p.cell_tc ? FORM_TILES : FORM_RECORDS;
}
int set_active_terms(Plan &p, const unsigned char *user_mask);
inline cudaError_t cuda_err_of(int status) {
    return status == ANOVA_OK ? cudaSuccess : status == ANOVA_ERR_NOMEM ? cudaErrorMemoryAllocation : cudaErrorUnknown;
}

// Allocations of plan construction and of the solver workspaces go through
// these two, so that a test can make the k-th of them fail the way an
// exhausted device or host would (anova_debug_fail_allocation).
bool alloc_fault();
cudaError_t plan_malloc_raw(void **ptr, size_t bytes);
template <typename T>
inline cudaError_t plan_malloc(T **ptr, size_t bytes) {
    return plan_malloc_raw((void **)ptr, bytes);
}
template <typename T>
inline T *plan_new(size_t n) {
    return alloc_fault() ? nullptr : new (std::nothrow) T[n];
}

// host-side table builders shared with plan construction (plan.cu)
double deconv_factor(int k, int n, int m, double b);
void window_polys(Window &w, int m, double b);
int fft_size(int N, double sigma);
int row_stride(int n);
// out = in * scale wrapped into [-1/2, 1/2) (scale 1/2 for cosine plans: x in [0, 1] -> x / 2);
// *bad = 1 for a coordinate that is not finite (bad: may be null)
__global__ void wrap_nodes_f32(const float *in, float *out, long long total, float scale, int *bad);

// stage timing: call stage_begin before and stage_end after a kernel launch
void stage_begin(Plan &p, int stage);
void stage_end(Plan &p, int stage);
void profiler_free(Plan &p);
enum { ST_PRE = 0, ST_GATHER = 1, ST_SPREAD = 2, ST_REDUCE = 3, ST_POST = 4, ST_SUMY = 5, ST_SOLVER = 6 };

// kernels launched by the entry points (trafo.cu / adjoint.cu)
int launch_trafo_f32(Plan &p, const float2 *fhat, float2 *f);
int launch_gather_f32(Plan &p, const float2 *fhat, float2 *f);
bool gather_fits(long long max_grid_bytes, int dmax);   // its shared memory
// Sorted forward (gather_sorted.cu), every term over its cell-sorted records:
// f = empty-set coefficient + all terms.
int launch_gather_sorted_f32(Plan &p, const float2 *fhat, float2 *f);
// The same for one problem (B.plans == null) or a batch of P problems, every one
// with records and accumulators: the gather of items [0, n_items), the first
// n_items3 of them third-order ones, and the fixed-point pass after it.  tc: the
// plans hold node tiles, the gather runs on the tensor cores.
int gather_sorted_launch(cudaStream_t st, const DevPlan &v, const BatchArgs &B, int P, const float2 *fhat,
                         float2 *f, const int4 *items, int n_items3, int n_items, int *counter,
                         long long max_grid_bytes, long long max_M, int sm_count, int mr, bool tc);
int launch_adjoint_f32(Plan &p, const float2 *y, float2 *fhat);
int adjoint_launch(Plan *prof, cudaStream_t st, const DevPlan &v, const BatchArgs &B, int P, const float2 *y,
                   float2 *fhat, int n_items, int n_items3, int *counter, int n_blocks, int mr,
                   long long max_grid_bytes, int max_fft_elems, int max_n, int max_stage, int sm_count,
                   long long max_grid_elems, int max_chunks, bool any_empty, double2 *scratch, int prec, bool tc);
size_t spread_smem_bytes(long long max_grid_bytes, bool o3, int sp);
int spread_block_nodes(long long max_grid_bytes);
// Sorts the nodes by grid cell for every term with sort_slot >= 0 (sort.cu).
int sort_nodes_by_cell(Plan &p);
// Direct summation (direct.cu).
constexpr int DIRECT_MAX_SMEM = 100 * 1024;   // forward: two CTAs per SM
constexpr int DIRECT_MAX_CHUNKS = 64, DIRECT_MAX_BLOCKS = 8192;   // adjoint
constexpr int DIRECT_RESIDENT = 4, DIRECT_RESIDENT_BIG = 2;       // its blocks per SM
constexpr int DIRECT_MAX_SPLITS = 16;         // forward: sets of terms per node block
constexpr double DIRECT_FIXED_NS = 8400.0, NFFT_FIXED_NS = 33000.0;   // launches and latencies of a transform
bool direct_term(const Term &T);
bool direct_faster(const Term *terms, int n_terms, int d, long long M);
size_t direct_smem(int d, int kt, int npl, bool cosine);
int direct_npl(int d, int kt, long long M, bool cosine);
int direct_splits(long long n_units, long long M, int npl, int sm_count);
// Node chunks of an adjoint item, at most: of 256 nodes up to 64 chunks.  Plans of order-1
// terms alone, whose items cost the same, then take chunks of 16384 nodes, one FP32 chain
// per thread: one coordinate's plan had 128 blocks at any size (d = 1, N = 16, M = 1e7
// 755 -> 183 us, 2e6 72 -> 53).
inline long long direct_max_chunks(long long M, bool order1) {
    const long long c = std::min<long long>(DIRECT_MAX_CHUNKS, std::max<long long>(1, M / 256));
    return order1 ? std::max(c, (M + 16383) / 16384) : c;
}
int direct_unit_list(const Plan &p, DirectTerm *out);
bool direct_big(const Term &T);
int direct_axis(const Term &T);
int direct_groups(const Term &T);
int direct_items(const Plan &p, DirectItem *out);
int build_unit_table(Plan &p);
int launch_direct_trafo(Plan &p, const float2 *fhat, float2 *f);
int launch_direct_adjoint(Plan &p, const float2 *y, float2 *fhat);
// anova_plan_create.  direct: the plan may be summed directly (a batch's plans and the
// tuner's reference are not); records: beside its tiles, for the forward, 1 yes, 0 no,
// -1 by few_nodes3 of its own terms (a batch's plans: of the batch's).
struct PlanUse {
    bool direct;
    int records;
};
int plan_create(anova_plan_t *out, int d, int64_t M, const void *x_dev, int n_terms, const int32_t *term_dims,
                const int32_t *bandwidth, const anova_plan_options *opts, void *stream, PlanUse use);
// Nodes and grid cells of the third-order terms of a valid or invalid term list (terms
// that a plan refuses are left out), and whether the forward of such a node density is
// faster over records (plan.cu).
struct Cells3 {
    double nodes = 0.0, cells = 0.0;
};
void add_cells3(Cells3 &c, int64_t M, int n_terms, const int32_t *term_dims, const int32_t *bandwidth,
                const anova_plan_options &o);
bool few_nodes3(const Cells3 &c);
// FP64 path (f64.cu): window tables, forward and adjoint transforms.
int build_window_tables_f64(Plan &p);
int launch_trafo_f64(Plan &p, const double2 *fhat, double2 *f);
int launch_adjoint_f64(Plan &p, const double2 *y, double2 *fhat);
// Node tiles (gather_tiles.cu, spread_tiles.cu, sort.cu).
void gather_tiles_launch(cudaStream_t st, const DevPlan &v, const BatchArgs &B, const int4 *items, int n_items,
                         bool order3, int *counter, long long max_grid_bytes, int sm_count, int mr);
void spread_tiles_launch(cudaStream_t st, const DevPlan &v, const BatchArgs &B, const float2 *y, int n_items,
                         bool order3, int *counter, long long sgrid, int sm_count, int mr, int prec);
int spread_tiles_ctas_per_sm(long long sgrid, bool order3);
int gather_tiles_ctas_per_sm(long long max_grid_bytes, bool order3);
// CTAs per SM of the order-1/2 spread kernel on the CUDA cores
int spread_ctas_per_sm(long long max_grid_bytes);
// Node chunks per term for a problem of n_terms active terms, n_terms3 of them
// third-order, at most kmax.
int spread_chunks_for(long long M, int n_terms, int n_terms3, int kmax, long long max_grid_bytes,
                      long long grid_elems, int sm_count, bool tc);
// The same for one problem of a batch whose problems cost total_ns (the sum of
// batch_cost_ns) on ctas CTAs.
double batch_cost_ns(long long M, int n_terms, int n_terms3);
int batch_chunks_for(long long M, double total_ns, int kmax, long long ctas);
// Appends the spread work items of one problem, K chunks per active term:
// those of the third-order terms (sel = 3) or of the others, order 2 before
// order 1 (sel = 0).  Returns the count.
int append_spread_items(const Plan &p, int prob, int K, int4 *out, int sel);
int lipschitz_estimate(Plan &p, double *L);
int fista_impl(Plan &p, const float2 *y, const double *w, const double *lambdas, int n_lambda, int max_it,
               double tol, int step_mode, double L0, double eta, const uint8_t *mask, const float2 *f0,
               float2 *path, anova_solve_info *info, double *L_out);

// Runs `set` (kernel attribute calls) unless it already ran on the current
// device: attributes such as the dynamic shared-memory limit belong to a
// device, so each device needs its own call.  One bit per device id < 64 in
// `seen`; larger ids run `set` every time.  Concurrent first calls may both
// run `set`, which is harmless.
template <typename F>
inline void once_per_device(std::atomic<unsigned long long> &seen, F &&set) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
    const unsigned long long bit = dev >= 0 && dev < 64 ? 1ULL << dev : 0ULL;
    if (bit && (seen.load(std::memory_order_acquire) & bit)) return;
    set();
    if (bit) seen.fetch_or(bit, std::memory_order_release);
}

// status from a CUDA error
inline int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return ANOVA_OK;
    if (e == cudaErrorMemoryAllocation) return ANOVA_ERR_NOMEM;
    return ANOVA_ERR_CUDA;
}

}  // namespace agft

struct anova_plan_s {
    agft::Plan p;
};
