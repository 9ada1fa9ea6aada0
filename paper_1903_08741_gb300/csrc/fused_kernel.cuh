// Device side of the persistent fused solver (kernel templates), shared by
// the translation units that instantiate them.
//
// Each CTA takes samples from an atomic queue and runs, for its sample, the
// complete method of arXiv 1903.08741 Sec. 4: backward-Euler time loop,
// modified Picard iteration on the mixed form (Eq. Mixed_based_3), and for
// every Picard step the cell-centred multigrid solve (five-point harmonic-mean
// stencil, Eq. five_stencil; red-black Gauss-Seidel; 1/4-sum restriction and
// piecewise-constant prolongation, Eq. transfer; coarse operators by
// rediscretisation with arithmetic means of face coefficients, Fig.
// diffUpscale; exact coarsest solve).  All control flow is per sample and uniform
// over its threads (decisions come from reductions over the CTA, or over the
// cluster of CTAs that shares a sample: gmax, gdot), so a sample never waits for
// another and there is no host round trip inside a solve.
//
// Memory: every CTA, or cluster of them, owns one scratch slot holding its
// sample's hierarchy; the slots of the resident CTAs are largely L2 (small grids:
// L1) resident.  Scratch arrays are read with plain loads: they are rewritten
// inside the kernel, and __syncthreads orders the accesses of one CTA.  What one
// CTA of a cluster writes another reads only behind the cluster's barrier
// (GClu::sync, or gmax and gdot, which hold one).
//
// Precision and instruction budget.  GB300 issues 2 FP64 FMAs per SM and
// clock (1/64 of its FP32 rate), so the FP64 V-cycle is written to minimise
// FP64 instructions:
//   * every level stores the Jacobi-scaled coefficients w = T/D of its four
//     faces and the scaled right-hand side f/D, so a Gauss-Seidel update is
//     dp_P = f_P/D_P + sum w dp_nb (4 FMAs instead of 6 operations);
//   * after a black half-sweep the black residuals are zero up to rounding
//     (each black value was just solved from its red neighbours), so the
//     restriction after pre-smoothing and the stopping norm after
//     post-smoothing evaluate red cells only (exactly the same quantities in
//     exact arithmetic; full evaluation when nu = 0);
//   * divisions by dt are multiplications by 1/dt.
// TM = double is the FP64 path (the oracle's algorithm and stopping tests);
// TM = float runs FP32 V-cycles (unscaled coefficients: FP32 operations are
// cheap, bytes are not) inside an FP64 defect-correction loop that performs
// a tunable number of V-cycles per FP64 defect (FP64 Picard residual, FP64
// outer residual, FP64 correction and stopping norm).

#pragma once
#include "rich_internal.cuh"
#include "fixed.cuh"
#include <cooperative_groups.h>
#include <math.h>
#include <type_traits>

// launch parameters and slot layout, shared across translation units
namespace rich_fused {

constexpr unsigned long long ABS_MASK = 0x7FFFFFFFFFFFFFFFull;
constexpr unsigned long long INF_BITS = 0x7FF0000000000000ull;
constexpr int MAXL = RICH_MAX_LEVELS;
constexpr int MIXED_INNER_DEFAULT = 2;   // FP32 V-cycles per FP64 defect evaluation
constexpr int ADJ_M = 12;                // GMRES restart length of the adjoint's J^T solves

// FP64 unscaled operator (all levels): faces, mass term, diagonal, Dirichlet faces
enum { A_TX, A_TZ, A_CDT, A_D, A_TBT, A_TBB, N64 };
// multigrid arrays in the cycle precision, colour-split on every level but
// the coarsest.  FP64: wE wW wN wS q=1/D fh dp D.  FP32: Tx Tz - D 1/D f dp -.
enum { B_0, B_1, B_2, B_3, B_4, B_5, B_6, B_7, NMG };

struct FParams {
    int S, nlev, mixed;
    int nx[MAXL], nz[MAXL];
    unsigned mnx[MAXL], mhx[MAXL];          // magic reciprocals of nx and nx/2
    long long o64[MAXL][N64];               // byte offsets in the slot (-1: absent)
    long long omg[MAXL][NMG];
    long long osm[MAXL];                    // level's dp in dynamic shared memory at this
                                            // byte offset (-1: in the slot)
    long long osm_alt;                      // likewise the finest level's second red half
    int lw;                                 // first level run by warp 0 alone (nlev: none)
    int lx;                                 // a cluster's sample: levels below lx run on all its CTAs
    long long s64[MAXL][N64];               // levels below the finest of at most 256 cells: every
    long long smg[MAXL][NMG];               // array of the cycles in dynamic shared memory at these
                                            // byte offsets (-1: not there)
    long long smem_bytes;                   // dynamic shared memory of a CTA
    long long o_f64, o_dp64, o_p, o_thold, o_Ks, o_a, o_K, o_th;
    long long slot_bytes;
    char* scratch;
    const double* lnKs;
    const double* alpha;
    double alpha_scale;
    double* qoi;
    double* p_final;
    int32_t* status;
    int64_t* pic_total;
    int64_t* mg_total;
    int64_t* t_ns;                          // per-sample solve time on its CTA (ns; may be null)
    int32_t* maxpic;
    int* queue;
    int nsteps, picard_maxit, mg_maxit, nu1, nu2, gamma;
    double inv_dt, tr, ts, p_top, p_bot, p_init, picard_tol, mg_tol, h, two_over_h2;
    // adjoint (k_adjoint only)
    int mixed_inner;            // FP32 V-cycles per FP64 defect (mixed path)
    int ckpt_every, keep_states, adj_maxit, adj_inner;
    double adj_tol;
    double* states;             // keep_states: every step's p, [slot][nsteps][cells]
    long long o_ckpt, o_seg, o_lam, o_rhs, o_r, o_dE, o_dW, o_dN, o_dS, o_dg, o_g;
    int adj_method;             // J^T solver: 0 defect correction, 1 BiCGStab, 2 GMRES(ADJ_M)
    long long o_rh, o_pk, o_v, o_t, o_ph, o_sh;   // BiCGStab vectors
    long long o_kry;                              // GMRES: ADJ_M + 1 Krylov and ADJ_M preconditioned vectors
    double* g_out;
    // closure 1 (van Genuchten-Mualem): per-cell n, theta_s, theta_r inputs
    // (theta arrays may be null: the problem's constants), continuation
    // shifts, and the slot arrays n, m = 1 - 1/n, theta_r, theta_s
    int closure;
    double alpha_shift, n_shift, init_decay;
    const double* n_in;
    const double* ts_in;
    const double* tr_in;
    long long o_n, o_m, o_trc, o_tsc;
};

// allow a kernel `bytes` of dynamic shared memory above the 48 KB default; the
// attribute is set once per (kernel, device, larger size)
inline int allow_dyn_smem(const void* kernel, size_t bytes) {
    if (bytes <= 32 * 1024) return 0;        // with the kernel's static arrays within the 48 KB default
    struct Grant { const void* k; int dev; size_t bytes; };
    static Grant grants[128];
    static int ngrants = 0;
    int dev = 0;
    RICH_CUDA(cudaGetDevice(&dev));
    int i = 0;
    while (i < ngrants && !(grants[i].k == kernel && grants[i].dev == dev)) ++i;
    if (i < ngrants && grants[i].bytes >= bytes) return 0;
    RICH_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    if (i == ngrants && ngrants < 128) ++ngrants;
    if (i < 128) grants[i] = Grant{kernel, dev, bytes};
    return 0;
}

// Occupancy query and launch of the fused kernel's instantiations, one
// translation unit per (cycle precision, closure) so that they compile in
// parallel: fused_g64.cu (FP64, Gardner), fused_g32.cu (mixed, Gardner),
// fused_vg64.cu, fused_vg32.cu (van Genuchten-Mualem).
int rich_occ_g64(const FParams& P, size_t smem, int nt, int* occ);
int rich_occ_g32(const FParams& P, size_t smem, int nt, int* occ);
int rich_occ_vg64(const FParams& P, size_t smem, int nt, int* occ);
int rich_occ_vg32(const FParams& P, size_t smem, int nt, int* occ);
void rich_launch_g64(const FParams& P, int grid, size_t smem, int nt, cudaStream_t st);
void rich_launch_g32(const FParams& P, int grid, size_t smem, int nt, cudaStream_t st);
void rich_launch_vg64(const FParams& P, int grid, size_t smem, int nt, cudaStream_t st);
void rich_launch_vg32(const FParams& P, int grid, size_t smem, int nt, cudaStream_t st);
int rich_cluster_g64(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit);
int rich_cluster_g32(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit);
int rich_cluster_vg64(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit);
int rich_cluster_vg32(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit);
// the adjoint kernel's instantiations (fused_adj64.cu, fused_adj32.cu): the
// kernel's address (occupancy queries) and its launch with 512 threads
const void* rich_adjoint_kernel64(bool wcycle);
const void* rich_adjoint_kernel32(bool wcycle);
int rich_adjoint_cluster64(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit);
int rich_adjoint_cluster32(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit);
void rich_adjoint_launch64(const FParams& P, int grid, size_t smem, cudaStream_t st);
void rich_adjoint_launch32(const FParams& P, int grid, size_t smem, cudaStream_t st);

}  // namespace rich_fused

namespace {
using namespace rich_fused;

// c / d for c * d < 2^32 (m = floor(2^32 / d) + 1), d = 1 handled apart
__device__ __forceinline__ int fdiv(int c, int d, unsigned m) {
    return d == 1 ? c : (int)__umulhi((unsigned)c, m);
}

// the GPU's global nanosecond timer (per-sample solve times)
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & ABS_MASK;
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    return v;
}

// block-wide sum of v in a fixed order (warp trees, then the warp partials in
// warp order), returned to every thread
__device__ __forceinline__ double block_sum(double v, double* red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < nw ? red[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[32] = v;
    }
    __syncthreads();
    const double r = red[32];
    __syncthreads();
    return r;
}

// block-wide max of v, returned to every thread
__device__ __forceinline__ unsigned long long block_max(unsigned long long v, unsigned long long* red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_max_u64(v);
    if (lane == 0) red[wid] = v;
    __syncthreads();
    // every warp reduces the partials itself: one barrier less than a
    // broadcast of warp 0's result
    v = warp_max_u64(lane < nw ? red[lane] : 0ull);
    __syncthreads();
    return v;
}

struct Lv64 {
    int nx, nz, nc;
    unsigned mnx;
    double *Tx, *Tz, *Cdt, *D, *Tbt, *Tbb;
};

// multigrid level in cycle precision T.  FP64 (scaled): c = {wE, wW, wN, wS},
// q = 1/D (below the finest level 1/(4 D), see restrict_cells), f = f/D (the
// coarsest level keeps f unscaled for the direct solve).
// FP32 (unscaled): c = {Tx, Tz, -, -}, q = 1/D, f = f.
// Layout: every level that is smoothed stores its cells colour-split, the red
// cells ((i + j) even) first and then the black ones, each half row-major with
// hx = nx/2 cells per row: cell (i, j) sits at ((i + j) & 1) H + j hx + i/2
// (H = hx nz).  A half-sweep then reads its own cells, and the neighbours of
// the other colour, at unit stride (no shared-memory bank conflicts, full
// sectors from L2).  The coarsest level (direct solve; its sides may be odd)
// keeps the natural row-major order (H = 0).  The two halves of dp have a
// pointer each, both to be indexed like the other arrays: dp (red cells; all of
// them on the coarsest level) and db (black cells: H before their first one).
// They point at one array, except on the finest FP64 level, whose second red
// half, alt, swaps with dp.
template <typename T>
struct Lv {
    int nx, nz, hx, nc, H;
    unsigned mnx, mhx;
    T *c0, *c1, *c2, *c3, *D, *q, *f, *dp, *db, *alt;
};

// storage index of cell (i, j) on a level
template <typename T>
__device__ __forceinline__ int sidx(const Lv<T>& L, int i, int j) {
    return L.H ? ((i + j) & 1) * L.H + j * L.hx + (i >> 1) : j * L.nx + i;
}

// the correction at cell (i, j)
template <typename T>
__device__ __forceinline__ T dp_at(const Lv<T>& L, int i, int j) {
    return (((i + j) & 1) && L.H ? L.db : L.dp)[sidx(L, i, j)];
}

// storage indices of a cell of a colour-split level (col 0 red, 1 black; c its
// place in its colour's half, i its column) and of its east, west, north and
// south neighbours (valid where the neighbour exists)
struct Nb { int own, e, w, n, s; };
__device__ __forceinline__ Nb nb_half(int col, int c, int i, int hx, int H) {
    const int oth = (1 - col) * H + c;
    return Nb{col * H + c, oth + (i & 1), oth - 1 + (i & 1), oth + hx, oth - hx};
}

template <typename T> struct Scaled { static constexpr bool value = sizeof(T) == 8; };

// Thread groups that run a level's loops: the whole CTA (barrier
// __syncthreads), warp 0 alone (barrier __syncwarp) on the smallest coarse
// levels, whose cells do not pay for CTA-wide barriers and which keep every
// array in shared memory, or a cluster of CTAs.  Each level function ends with
// its group synchronised.
struct GCta {
    static __device__ __forceinline__ int rank() { return threadIdx.x; }
    static __device__ __forceinline__ int size() { return blockDim.x; }
    static __device__ __forceinline__ void sync() { __syncthreads(); }
};
struct GWarp {
    static __device__ __forceinline__ int rank() { return threadIdx.x & 31; }
    static __device__ __forceinline__ int size() { return 32; }
    static __device__ __forceinline__ void sync() { __syncwarp(); }
};
// all CTAs of a thread-block cluster (one sample): the barrier orders their
// global and shared accesses
constexpr int CLUSTER_THREADS = 512;
struct GClu {
    static __device__ __forceinline__ cooperative_groups::cluster_group c() { return cooperative_groups::this_cluster(); }
    static __device__ __forceinline__ int rank() { return (int)(c().block_rank() * blockDim.x + threadIdx.x); }
    static __device__ __forceinline__ int size() { return (int)(c().num_blocks() * blockDim.x); }
    static __device__ __forceinline__ void sync() { c().sync(); }
};

// Gauss-Seidel value of a cell (storage indices b) from its current
// neighbours, in the half `o` of dp, with the level's arrays passed as
// restrict-qualified pointers: every caller reads dp only at cells that it does
// not write in the same pass (see rbgs_cells), so the compiler may keep several
// cells' loads in flight ahead of the stores.
//   FP64 (scaled): c0..c3 = wE, wW, wN, wS; value f + sum w dp_nb.
//   FP32 (unscaled): c0 = Tx (east face), c1 = Tz (north face); the west and
//   south faces are the neighbours'; value (f + sum T dp_nb) / D.
template <typename T>
__device__ __forceinline__ T gs_at(const Nb& b, bool hE, bool hW, bool hN, bool hS, const T* __restrict__ f,
                                   const T* __restrict__ c0, const T* __restrict__ c1,
                                   const T* __restrict__ c2, const T* __restrict__ c3,
                                   const T* __restrict__ q, const T* __restrict__ o) {
    if constexpr (Scaled<T>::value) {
        T v = f[b.own];
        if (hE) v += c0[b.own] * o[b.e];
        if (hW) v += c1[b.own] * o[b.w];
        if (hN) v += c2[b.own] * o[b.n];
        if (hS) v += c3[b.own] * o[b.s];
        return v;
    } else {
        T t = T(0);
        if (hE) t += c0[b.own] * o[b.e];
        if (hW) t += c0[b.w] * o[b.w];
        if (hN) t += c1[b.own] * o[b.n];
        if (hS) t += c1[b.s] * o[b.s];
        return (f[b.own] + t) * q[b.own];
    }
}

// residual f - A dp (unscaled) of a cell whose correction is d: FP64
// D (value - d), FP32 f - (D d - sum T dp_nb)
template <typename T>
__device__ __forceinline__ T resid_at(const Nb& b, bool hE, bool hW, bool hN, bool hS,
                                      const T* __restrict__ f, const T* __restrict__ c0,
                                      const T* __restrict__ c1, const T* __restrict__ c2,
                                      const T* __restrict__ c3, const T* __restrict__ q,
                                      const T* __restrict__ D, const T* __restrict__ o, T d) {
    if constexpr (Scaled<T>::value) {
        return D[b.own] * (gs_at<T>(b, hE, hW, hN, hS, f, c0, c1, c2, c3, q, o) - d);
    } else {
        T t = T(0);
        if (hE) t += c0[b.own] * o[b.e];
        if (hW) t += c0[b.w] * o[b.w];
        if (hN) t += c1[b.own] * o[b.n];
        if (hS) t += c1[b.s] * o[b.s];
        return f[b.own] - (D[b.own] * d - t);
    }
}

// a + b, not contracted with the product that gave a or b: the one-cell and the
// two-cell loops of a level give the same bits
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

// 16-byte accesses: two FP64 or four FP32 neighbours of one colour
__device__ __forceinline__ void ld_vec(const double* p, double (&v)[2]) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x; v[1] = t.y;
}
__device__ __forceinline__ void ld_vec(const float* p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void st_vec(double* p, const double (&v)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
}
__device__ __forceinline__ void st_vec(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <typename T> struct Vec { static constexpr int W = 16 / sizeof(T); };

// Gauss-Seidel values of W = 2 (FP64) or 4 (FP32) cells c, c + 1, ... of one
// colour in row j (c a multiple of W, hx too: 16-byte aligned), bit for bit
// those of gs_at.  The half-sweeps are bound by the latency of their loads and
// by the FP64 pipe (a warp's DFMA holds its quarter of the SM for 64 cycles),
// so a thread's loads are 16 bytes wide and all issued before the arithmetic:
// 9 (FP64) or 11 (FP32) loads instead of 18 or 40.  A 128^2 batch of 608
// samples, two steps, 512 threads: FP32 cycles 399 -> 310 ms, FP64 650 -> 590 ms
// (with the first red half-sweep taken from the norm and the black-only
// prolongation).  Missing neighbours count as zero; their face coefficient is
// zero too.
template <typename T>
__device__ __forceinline__ void gs_vec(int c, int j, int nz, int hx, int H, int colour, const T* __restrict__ f,
                                       const T* __restrict__ c0, const T* __restrict__ c1,
                                       const T* __restrict__ c2, const T* __restrict__ c3,
                                       const T* __restrict__ q, const T* __restrict__ o, T (&v)[Vec<T>::W]) {
    constexpr int W = Vec<T>::W;
    const int k = c - j * hx, s = (j + colour) & 1, own = colour * H + c, oth = (1 - colour) * H + c;
    const bool hN = j < nz - 1, hS = j > 0, hX = s ? k + W < hx : k > 0;
    const int x = s ? oth + W : oth - 1;              // the neighbour beside the W in the own row
    T a0[W], a1[W], a2[W], a3[W], qq[W], m[W], n[W] = {}, u[W] = {}, side = T(0), wside = T(0), cw[W], cs[W] = {};
    ld_vec(f + own, v);
    ld_vec(c0 + own, a0);
    ld_vec(c1 + own, a1);
    if constexpr (Scaled<T>::value) {
        ld_vec(c2 + own, a2);
        ld_vec(c3 + own, a3);
    } else {
        ld_vec(q + own, qq);
        ld_vec(c0 + oth, cw);
        if (hS) ld_vec(c1 + oth - hx, cs);
        if (!s && hX) wside = c0[x];
    }
    ld_vec(o + oth, m);
    if (hN) ld_vec(o + oth + hx, n);
    if (hS) ld_vec(o + oth - hx, u);
    if (hX) side = o[x];
#pragma unroll
    for (int t = 0; t < W; ++t) {
        const T e = !s ? m[t] : t + 1 < W ? m[t + 1 < W ? t + 1 : 0] : side;
        const T w = s ? m[t] : t > 0 ? m[t > 0 ? t - 1 : 0] : side;
        if constexpr (Scaled<T>::value) {
            v[t] = fma(a0[t], e, v[t]);
            v[t] = fma(a1[t], w, v[t]);
            v[t] = fma(a2[t], n[t], v[t]);
            v[t] = fma(a3[t], u[t], v[t]);
        } else {
            const T tw = s ? cw[t] : t > 0 ? cw[t > 0 ? t - 1 : 0] : wside;
            T z = T(0);
            z += a0[t] * e;
            z += tw * w;
            z += a1[t] * n[t];
            z += cs[t] * u[t];
            v[t] = (v[t] + z) * qq[t];
        }
    }
}

// whether a level's loops take W cells of a colour at a time: aligned rows, and
// still a cell for every thread of the group (a level with fewer cells is
// faster spread over more warps, one cell a thread)
template <typename T, typename G>
__device__ __forceinline__ bool wide(int hx, int H) {
    return hx % Vec<T>::W == 0 && H >= Vec<T>::W * G::size();
}

// one colour of red-black Gauss-Seidel over a colour-split level (red:
// i + j even).  The corrections are read through one restrict-qualified view
// (the other colour's half) and written through another (its own).
template <typename T, typename G>
__device__ __forceinline__ void rbgs_cells(int nx, int nz, int hx, int H, unsigned mhx, int colour,
                                           const T* __restrict__ f, const T* __restrict__ c0,
                                           const T* __restrict__ c1, const T* __restrict__ c2,
                                           const T* __restrict__ c3, const T* __restrict__ q,
                                           const T* __restrict__ o, T* __restrict__ own) {
    if (wide<T, G>(hx, H)) {
        for (int c = Vec<T>::W * G::rank(); c < H; c += Vec<T>::W * G::size()) {
            T v[Vec<T>::W];
            gs_vec<T>(c, fdiv(c, hx, mhx), nz, hx, H, colour, f, c0, c1, c2, c3, q, o, v);
            st_vec(own + colour * H + c, v);
        }
    } else {
#pragma unroll 1
        for (int c = G::rank(); c < H; c += G::size()) {
            const int j = fdiv(c, hx, mhx);
            const int i = 2 * (c - j * hx) + ((j + colour) & 1);
            const Nb b = nb_half(colour, c, i, hx, H);
            own[b.own] = gs_at<T>(b, i < nx - 1, i > 0, j < nz - 1, j > 0, f, c0, c1, c2, c3, q, o);
        }
    }
    G::sync();
}

template <typename T, typename G>
__device__ __forceinline__ void rbgs(const Lv<T>& L, int colour) {
    rbgs_cells<T, G>(L.nx, L.nz, L.hx, L.H, L.mhx, colour, L.f, L.c0, L.c1, L.c2, L.c3, L.q,
                     colour ? L.dp : L.db, colour ? L.db : L.dp);
}

template <typename T, typename G>
__device__ __forceinline__ void prolong(const Lv<T>& F, const Lv<T>& C, bool black_only);

// nu red-black sweeps; with seeded true the first red half-sweep is skipped
// because the restriction already stored its result (see restrict_cells)
template <typename T, typename G>
__device__ __forceinline__ void smooth(const Lv<T>& L, int nu, bool seeded = false) {
    for (int it = 0; it < nu; ++it) {
        if (!(seeded && it == 0)) rbgs<T, G>(L, 0);
        rbgs<T, G>(L, 1);
    }
}

// prolongation and post-smoothing of level l from level l+1
template <typename T, typename G>
__device__ __forceinline__ void prolong_smooth(const Lv<T>& F, const Lv<T>& C, int nu2) {
    prolong<T, G>(F, C, nu2 > 0);
    smooth<T, G>(F, nu2);
}

// restricted residual (Eq. transfer, R = 1/4 sum of the children); after a
// black half-sweep only the two red children carry a residual.  Reads the
// fine level, writes the coarse one (distinct arrays: restrict views).  The
// fine level is colour-split: the children of coarse cell (I, J) are the red
// cells r0 = 2J hx + I and r0 + hx and the black cells H + r0, H + r0 + hx.
// FP64: the coarse level's cq is 1/(4 D), so that one multiplication takes the
// mean and scales the right-hand side.
// The coarse correction starts at zero; when the coarse level is smoothed
// next (seed), its red cells get at once the value the first red half-sweep
// would compute from all-zero neighbours, f q (FP64: the scaled f), so that
// half-sweep is skipped; its black cells are overwritten before they are read.
template <typename T, typename G>
__device__ __forceinline__ void restrict_cells(const Lv<T>& F, const Lv<T>& C, bool red_only, bool coarsest, bool seed,
                                               const T* __restrict__ f, const T* __restrict__ c0,
                                               const T* __restrict__ c1, const T* __restrict__ c2,
                                               const T* __restrict__ c3, const T* __restrict__ q,
                                               const T* __restrict__ D, const T* __restrict__ dr,
                                               const T* __restrict__ db, const T* __restrict__ cq,
                                               T* __restrict__ cf, T* __restrict__ cdp) {
    const int nx = F.nx, nz = F.nz, hx = F.hx, H = F.H;
    if constexpr (Scaled<T>::value) {
        // two coarse cells a thread, 16-byte loads (see gs_vec); the black rows
        // j and j + 1 serve both red rows
        if (red_only && !coarsest && wide<T, G>(hx, C.nc)) {
            for (int c = 2 * G::rank(); c < C.nc; c += 2 * G::size()) {
                const int J = fdiv(c, C.nx, C.mnx), I = c - J * C.nx, j = 2 * J, r0 = j * hx + I, r1 = r0 + hx;
                double bs[2] = {}, b0[2], b1[2], bn[2] = {}, lo = 0.0, hi = 0.0, v0[2], v1[2], a[2], d[2];
                ld_vec(db + H + r0, b0);
                ld_vec(db + H + r1, b1);
                if (j > 0) ld_vec(db + H + r0 - hx, bs);
                if (j + 2 < nz) ld_vec(db + H + r1 + hx, bn);
                if (I > 0) lo = db[H + r0 - 1];
                if (I + 2 < hx) hi = db[H + r1 + 2];
                ld_vec(f + r0, v0);
                ld_vec(f + r1, v1);
                const double e0[2] = {b0[0], b0[1]}, w0[2] = {lo, b0[0]}, e1[2] = {b1[1], hi}, w1[2] = {b1[0], b1[1]};
                auto face = [&](const double* w, const double (&x0)[2], const double (&x1)[2]) {
                    ld_vec(w + r0, a);
                    v0[0] = fma(a[0], x0[0], v0[0]); v0[1] = fma(a[1], x0[1], v0[1]);
                    ld_vec(w + r1, a);
                    v1[0] = fma(a[0], x1[0], v1[0]); v1[1] = fma(a[1], x1[1], v1[1]);
                };
                face(c0, e0, e1);
                face(c1, w0, w1);
                face(c2, b1, bn);
                face(c3, bs, b0);
                ld_vec(dr + r0, d); v0[0] -= d[0]; v0[1] -= d[1];
                ld_vec(dr + r1, d); v1[0] -= d[0]; v1[1] -= d[1];
                ld_vec(D + r1, d); v1[0] *= d[0]; v1[1] *= d[1];
                ld_vec(D + r0, d);
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int cs = sidx(C, I + t, J);
                    const double fc = cq[cs] * add_rn(__dmul_rn(d[t], v0[t]), v1[t]);
                    cf[cs] = fc;
                    if (!seed) cdp[cs] = 0.0;
                    else if (!((I + t + J) & 1)) cdp[cs] = fc;
                }
            }
            G::sync();
            return;
        }
    }
#pragma unroll(Scaled<T>::value ? 1 : 2)
    for (int c = G::rank(); c < C.nc; c += G::size()) {
        const int J = fdiv(c, C.nx, C.mnx), I = c - J * C.nx;
        const int i = 2 * I, j = 2 * J, r0 = j * hx + I, r1 = r0 + hx;
        // red (i, j): neighbours black; red (i+1, j+1) likewise
        const T r11 = resid_at<T>(nb_half(0, r1, i + 1, hx, H), i + 1 < nx - 1, true, j + 1 < nz - 1, true, f, c0,
                                  c1, c2, c3, q, D, db, dr[r1]);
        const T r00 = resid_at<T>(nb_half(0, r0, i, hx, H), true, i > 0, true, j > 0, f, c0, c1, c2, c3, q, D, db,
                                  dr[r0]);
        T sum;
        if (red_only) {
            sum = add_rn(r00, r11);
        } else {
            const T r10 = resid_at<T>(nb_half(1, r0, i + 1, hx, H), i + 1 < nx - 1, true, true, j > 0, f, c0, c1, c2,
                                      c3, q, D, dr, db[H + r0]);
            const T r01 = resid_at<T>(nb_half(1, r1, i, hx, H), true, i > 0, j + 1 < nz - 1, true, f, c0, c1, c2, c3,
                                      q, D, dr, db[H + r1]);
            sum = r00 + r10 + r01 + r11;
        }
        const int cs = sidx(C, I, J);
        const T fc = Scaled<T>::value && !coarsest ? sum * cq[cs] : T(0.25) * sum;
        cf[cs] = fc;
        if (!coarsest) {                              // (the coarsest solve writes its own)
            if (!seed) cdp[cs] = T(0);
            else if (!((I + J) & 1)) cdp[cs] = Scaled<T>::value ? fc : fc * cq[cs];
        }
    }
    G::sync();
}

template <typename T, typename G>
__device__ __forceinline__ void resid_restrict(const Lv<T>& F, const Lv<T>& C, bool red_only, bool coarsest,
                                               bool seed = false) {
    restrict_cells<T, G>(F, C, red_only, coarsest, seed, F.f, F.c0, F.c1, F.c2, F.c3, F.q, F.D, F.dp, F.db,
                         C.q, C.f, C.dp);
}

// piecewise-constant prolongation and correction: each coarse cell adds its
// value to its own four children, so no two iterations touch one element.  When
// a red half-sweep follows (black_only) the red children are left alone: that
// half-sweep replaces them without reading them.
template <typename T, typename G>
__device__ __forceinline__ void prolong(const Lv<T>& F, const Lv<T>& C, bool black_only) {
    const T* __restrict__ e = C.dp;                   // (a coarse level's halves are one array)
    T* __restrict__ dr = F.dp;
    T* __restrict__ db = F.db;
    const int hx = F.hx, H = F.H;
    if constexpr (Scaled<T>::value) {
        if (black_only && wide<T, G>(hx, C.nc)) {     // two coarse cells a thread, 16-byte accesses
            for (int c = 2 * G::rank(); c < C.nc; c += 2 * G::size()) {
                const int J = fdiv(c, C.nx, C.mnx), I = c - J * C.nx, r0 = H + 2 * J * hx + I;
                const double v0 = e[sidx(C, I, J)], v1 = e[sidx(C, I + 1, J)];
                double a[2], b[2];
                ld_vec(db + r0, a);
                ld_vec(db + r0 + hx, b);
                a[0] += v0; a[1] += v1; b[0] += v0; b[1] += v1;
                st_vec(db + r0, a);
                st_vec(db + r0 + hx, b);
            }
            G::sync();
            return;
        }
    }
#pragma unroll 2
    for (int c = G::rank(); c < C.nc; c += G::size()) {
        const int J = fdiv(c, C.nx, C.mnx), I = c - J * C.nx;
        const T v = e[sidx(C, I, J)];
        const int r0 = 2 * J * hx + I;
        db[H + r0] += v; db[H + r0 + hx] += v;
        if (!black_only) { dr[r0] += v; dr[r0 + hx] += v; }
    }
    G::sync();
}

// Exact coarsest solve: Gaussian elimination of the assembled five-point
// matrix (symmetric positive definite, diagonally dominant: no pivoting) in
// shared memory.  The matrix is factored once per Picard iteration -- the upper
// triangle, the row multipliers below it and the reciprocals of the pivots in
// the extra column -- and a cycle's visit substitutes its right-hand side with
// the same operations in the same order.  A visit then has no division: n
// dependent FP64 divisions of about 560 cycles each for the pivots and as many
// for the multipliers made it 5000 cycles on a 2^2 coarsest level; it is about
// 1600 without them.  Run by warp 0.
template <typename T>
__device__ void coarse_factor_warp(int nx, int nz, const T* Tx, const T* Tz, const T* D, T* A) {
    const int nn = nx * nz, ld = nn + 1, lane = threadIdx.x & 31;
    for (int r = lane; r < nn; r += 32) {
        for (int c = 0; c < nn; ++c) A[r * ld + c] = T(0);
        int j = r / nx, i = r - j * nx;
        A[r * ld + r] = D[r];
        if (i < nx - 1) A[r * ld + r + 1] = -Tx[r];
        if (i > 0)      A[r * ld + r - 1] = -Tx[r - 1];
        if (j < nz - 1) A[r * ld + r + nx] = -Tz[r];
        if (j > 0)      A[r * ld + r - nx] = -Tz[r - nx];
    }
    __syncwarp();
    for (int k = 0; k < nn; ++k) {
        for (int r = k + 1 + lane; r < nn; r += 32) {
            const T m = A[r * ld + k] / A[k * ld + k];
            A[r * ld + k] = m;
            for (int c = k + 1; c < nn; ++c) A[r * ld + c] = fma(-m, A[k * ld + c], A[r * ld + c]);
        }
        __syncwarp();
    }
    for (int r = lane; r < nn; r += 32) A[r * ld + nn] = T(1) / A[r * ld + r];
    __syncwarp();
}

// s / u given r = 1/u rounded to nearest: the quotient s r corrected by its
// exact remainder is the correctly rounded s / u, but for quotients within about
// 2^-52 units of a midpoint (after Markstein, IBM J. Res. Dev. 34, 1990; tiny and
// huge operands, where the remainder may not be exact, and a zero or non-finite
// pivot take the division)
__device__ __forceinline__ double div_by(double s, double u, double r) {
    const double q = s * r;
    const int eq = (__double2hiint(q) >> 20 & 0x7FF) - 1023, eu = (__double2hiint(u) >> 20 & 0x7FF) - 1023;
    if (abs(eq) < 600 && abs(eu) < 300) return fma(fma(-q, u, s), r, q);
    return s / u;
}
__device__ __forceinline__ float div_by(float s, float u, float) { return s / u; }

template <typename T>
__device__ __forceinline__ void coarse_solve_warp(int nn, const T* f, T* dp, const T* A) {
    const int ld = nn + 1, lane = threadIdx.x & 31;
    // forward: lane r mod 32 owns row r (dp holds the eliminated right-hand side)
    for (int r = lane; r < nn; r += 32) dp[r] = f[r];
    __syncwarp();
    if (nn <= 8) {                                    // a handful of rows: one lane, no exchanges
        if (lane == 0) {
            for (int k = 0; k < nn; ++k)
                for (int r = k + 1; r < nn; ++r) dp[r] = fma(-A[r * ld + k], dp[k], dp[r]);
        }
    } else {
        for (int k = 0; k < nn; ++k) {
            for (int r = k + 1 + lane; r < nn; r += 32) dp[r] = fma(-A[r * ld + k], dp[k], dp[r]);
            __syncwarp();
        }
    }
    if (lane == 0) {
        for (int k = nn - 1; k >= 0; --k) {
            T sum = dp[k];
            for (int c = k + 1; c < nn; ++c) sum = fma(-A[k * ld + c], dp[c], sum);
            dp[k] = div_by(sum, A[k * ld + k], A[k * ld + nn]);
        }
    }
    __syncwarp();
}

// exact solve on the coarsest level c (f0 is the unscaled right-hand side when
// c is the finest level), by warp 0; the CTA group waits for it at a barrier
template <typename T, typename G>
__device__ __forceinline__ void coarsest(const Lv<T>* L, int c, const T* A, const T* f0) {
    if (threadIdx.x < 32) coarse_solve_warp<T>(L[c].nc, Scaled<T>::value && c == 0 ? f0 : L[c].f, L[c].dp, A);
    if constexpr (std::is_same<G, GCta>::value) __syncthreads();
}

// One multigrid cycle rooted at level `root`: V-cycle for gamma = 1, else the
// cycle of index gamma (W-cycle for gamma = 2, the paper's cycle, Sec. 4.2):
// every visit of level l < nlev-2 runs gamma cycles on level l+1, the visit
// of nlev-2 one exact coarsest solve.  The recursion is unrolled into a
// depth-first walk whose per-level visit counts sit in 4-bit fields of one
// register (no device stack).  Run by the CTA, each visit of level lw (the
// first small level) is handed to warp 0 as a complete cycle rooted at lw.
// A level entered right after the restriction into it (fresh) skips its
// first red half-sweep, which the restriction seeded; a level cycled again
// (gamma > 1) starts from its previous correction and smooths in full.
template <typename T, typename G>
__device__ __forceinline__ void gwalk(const Lv<T>* L, int root, int nlev, int lw, int nu1, int nu2,
                                      int gamma, T* A, const T* f0, bool root_fresh) {
    static_assert(RICH_MAX_LEVELS * 4 <= 64, "visit counters must fit one 64-bit word");
    unsigned long long cnt = 0;
    int l = root;
    bool fresh = root_fresh;
    const bool seed = nu1 > 0;
    for (;;) {
        for (; l < nlev - 1 && l != lw; ++l) {            // enter l: pre-smooth, restrict
            smooth<T, G>(L[l], nu1, fresh && seed);
            resid_restrict<T, G>(L[l], L[l + 1], nu1 > 0, l + 1 == nlev - 1, seed);
            cnt &= ~(15ull << (4 * l));
            fresh = true;
        }
        if constexpr (std::is_same<G, GCta>::value) {
            if (l == lw && lw < nlev - 1) {
                if (threadIdx.x < 32)
                    gwalk<T, GWarp>(L, lw, nlev, nlev, nu1, nu2, gamma, A, f0, fresh && seed);
                __syncthreads();
            } else {
                coarsest<T, G>(L, nlev - 1, A, f0);
            }
        } else {
            coarsest<T, G>(L, nlev - 1, A, f0);
        }
        for (;;) {                                        // leave l+1, back on l
            if (--l < root) return;
            cnt += 1ull << (4 * l);
            const int reps = (l + 1 == nlev - 1) ? 1 : gamma;
            if ((int)((cnt >> (4 * l)) & 15) < reps) { ++l; fresh = false; break; }   // cycle l+1 again
            prolong_smooth<T, G>(L[l], L[l + 1], nu2);
        }
    }
}

// V-cycle with the levels from lw down handed to warp 0 (lw = nlev: none);
// every level below the finest is fresh (seeded by its restriction), the
// finest when `fresh`.  A cluster (G = GClu) runs the levels below lx on all its
// CTAs; the first CTA runs the others while the rest wait.
template <typename T, typename G>
__device__ __forceinline__ void vcycle(const Lv<T>* L, int nlev, int lx, int lw, int nu1, int nu2, T* A, const T* f0,
                                       bool fresh) {
    constexpr bool CLU = std::is_same<G, GClu>::value;
    const bool seed = nu1 > 0;
    const int top = min(lw, nlev - 1);       // levels 0 .. top-1 run on the whole CTA
    if constexpr (CLU) {
        for (int l = 0; l < lx; ++l) {
            smooth<T, GClu>(L[l], nu1, (l > 0 || fresh) && seed);
            resid_restrict<T, GClu>(L[l], L[l + 1], nu1 > 0, l + 1 == nlev - 1, seed);
        }
    }
    const int l0 = CLU ? lx : 0;
    if (!CLU || GClu::c().block_rank() == 0) {
        for (int l = l0; l < top; ++l) {
            smooth<T, GCta>(L[l], nu1, (l > 0 || fresh) && seed);
            resid_restrict<T, GCta>(L[l], L[l + 1], nu1 > 0, l + 1 == nlev - 1, seed);
        }
        if (lw < nlev - 1) {
            if (threadIdx.x < 32) {
                for (int l = lw; l < nlev - 1; ++l) {
                    smooth<T, GWarp>(L[l], nu1, seed);
                    resid_restrict<T, GWarp>(L[l], L[l + 1], nu1 > 0, l + 1 == nlev - 1, seed);
                }
                coarsest<T, GWarp>(L, nlev - 1, A, f0);
                for (int l = nlev - 2; l >= lw; --l) prolong_smooth<T, GWarp>(L[l], L[l + 1], nu2);
            }
            __syncthreads();
        } else {
            coarsest<T, GCta>(L, nlev - 1, A, f0);
        }
        for (int l = top - 1; l >= l0; --l) prolong_smooth<T, GCta>(L[l], L[l + 1], nu2);
    }
    if constexpr (CLU) {
        GClu::sync();
        for (int l = lx - 1; l >= 0; --l) prolong_smooth<T, GClu>(L[l], L[l + 1], nu2);
    }
}

// ||f - A dp||_inf on the finest (FP64) level after a cycle ending with a black
// half-sweep (red cells only) or, with red_only false, over every cell.  The
// red cells' scaled residual is g - dp with g the value that the next red
// half-sweep would store: with `next` given, g is kept there, and the next
// cycle starts from that half (see Cta::mg_solve) instead of sweeping.
// Returns the thread's part of the maximum.
template <typename T, typename G>
__device__ __forceinline__ unsigned long long resid_norm(const Lv<T>& L, bool red_only, T* __restrict__ next) {
    static_assert(Scaled<T>::value, "the mixed path's norm is its FP64 defect's");
    unsigned long long m = 0;
    const int nx = L.nx, nz = L.nz, hx = L.hx, H = L.H;
    if (H) {
        for (int col = 0; col < (red_only ? 1 : 2); ++col) {
            const T* __restrict__ own = col ? L.db : L.dp;
            const T* __restrict__ oth = col ? L.dp : L.db;
            const T* __restrict__ D = L.D;
            if (wide<T, G>(hx, H)) {
                for (int c = 2 * G::rank(); c < H; c += 2 * G::size()) {
                    T g[2], d[2], x[2];
                    gs_vec<T>(c, fdiv(c, hx, L.mhx), nz, hx, H, col, L.f, L.c0, L.c1, L.c2, L.c3, L.q, oth, g);
                    ld_vec(D + col * H + c, d);
                    ld_vec(own + col * H + c, x);
                    if (next) st_vec(next + c, g);
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const unsigned long long b = abs_bits(d[t] * (g[t] - x[t]));
                        m = b > m ? b : m;
                    }
                }
                continue;
            }
#pragma unroll 1
            for (int c = G::rank(); c < H; c += G::size()) {
                const int j = fdiv(c, hx, L.mhx);
                const int i = 2 * (c - j * hx) + ((j + col) & 1);
                const Nb s = nb_half(col, c, i, hx, H);
                const T g = gs_at<T>(s, i < nx - 1, i > 0, j < nz - 1, j > 0, L.f, L.c0, L.c1, L.c2, L.c3, L.q, oth);
                if (next) next[c] = g;
                const unsigned long long b = abs_bits(D[s.own] * (g - own[s.own]));
                m = b > m ? b : m;
            }
        }
    } else {                                          // one level only: natural order
        for (int c = G::rank(); c < L.nc; c += G::size()) {
            const int j = fdiv(c, nx, L.mnx), i = c - j * nx;
            T v = L.f[c];
            if (i < nx - 1) v += L.c0[c] * L.dp[c + 1];
            if (i > 0) v += L.c1[c] * L.dp[c - 1];
            if (j < nz - 1) v += L.c2[c] * L.dp[c + nx];
            if (j > 0) v += L.c3[c] * L.dp[c - nx];
            const unsigned long long b = abs_bits(L.D[c] * (v - L.dp[c]));
            m = b > m ? b : m;
        }
    }
    return m;
}

// van Genuchten-Mualem closure at p < 0 (Eqs. Sw, sc_van, Krw) with
// m = 1 - 1/n and an = (a|p|)^n: S = (1 + an)^-m, K_rw = S^(1/2) (1 - (an /
// (1 + an))^m)^2 (1 - S^(1/m) = an/(1 + an) exactly) and dS/dp = m n S an /
// ((1 + an) |p|), the Eq. sc_van capacity divided by theta_s - theta_r.  In
// logarithms: an = exp(n log(a|p|)), S = exp(-m log1p(an)), and since
// m n = n - 1, (an / (1 + an))^m = an^m S = (an / (a|p|)) S: one exp fewer
// than exp(m (n log(a|p|) - log1p(an))), and in FP64 no cancellation between the
// two logarithms in the dry limit.
// The fixed-point evaluation (fixed.cuh) takes every soil of practice; what
// leaves its ranges takes the FP64 functions.  It does subtract the logarithms,
// whose errors are absolute and below an FP64 rounding of one: 1 - exp is then off
// by no more than the rounding of the exp.
__device__ __forceinline__ double vg_sat(double a, double n, double m, double p) {
    const double ap = -a * p;
    rich_fx::VgLog o;
    if (rich_fx::vg_log(ap, n, m, o)) return rich_fx::vg_s(o);
    return exp(-m * log1p(exp(n * log(ap))));
}

__device__ __forceinline__ void vg_eval(double a, double n, double m, double p, double& S, double& krw,
                                        double& dS) {
    const double ap = -a * p;
    rich_fx::VgLog o;
    if (rich_fx::vg_log(ap, n, m, o)) {
        S = rich_fx::vg_s(o);
        rich_fx::vg_k(o, krw, dS);
        dS *= m * n * a;
        return;
    }
    const double an = exp(n * log(ap));
    const double l1 = log1p(an);
    S = exp(-m * l1);
    const double b = 1.0 - S * (an / ap);
    krw = sqrt(S) * b * b;
    dS = m * n * S * an / ((1.0 + an) * (-p));
}

// Cooperative building blocks of one sample's solve on its CTA (G0 = GCta) or its
// cluster of CTAs (GClu).  Every method is called by all threads of the group
// and ends with the group synchronised; tid and nt count over the group.
template <typename TM, bool WC = false, int CL = 0, typename G0 = GCta>
struct Cta {
    static constexpr bool CLU = std::is_same<G0, GClu>::value;   // the sample's group is a cluster
    static constexpr bool SC = Scaled<TM>::value;
    const FParams& P;
    Lv64* L64;
    Lv<TM>* LM;
    TM* Amat;
    unsigned long long* red;
    // cluster: the CTAs' maxima, or the warps' sums (gdot); two sets used in turn
    unsigned long long (*cred)[CLUSTER_THREADS / 32] = nullptr;
    int cpar = 0;
    double *f64, *dp64, *p, *thold, *Ks, *aa, *K, *th;
    double *nn, *mm, *trc, *tsc;          // closure 1: per-cell n, m, theta_r, theta_s
    int nx, nz, nc, nlev, tid, nt;
    double h, t2h, idt, tr, ts;

    __device__ Cta(const FParams& P_, char* slot, Lv64* l64, Lv<TM>* lm, TM* A, unsigned long long* r)
        : P(P_), L64(l64), LM(lm), Amat(A), red(r) {
        f64 = (double*)(slot + P.o_f64);
        dp64 = SC ? nullptr : (double*)(slot + P.o_dp64);
        p = (double*)(slot + P.o_p);
        thold = (double*)(slot + P.o_thold);
        Ks = (double*)(slot + P.o_Ks);
        aa = (double*)(slot + P.o_a);
        K = (double*)(slot + P.o_K);
        th = (double*)(slot + P.o_th);
        if constexpr (CL == 1) {
            nn = (double*)(slot + P.o_n); mm = (double*)(slot + P.o_m);
            trc = (double*)(slot + P.o_trc); tsc = (double*)(slot + P.o_tsc);
        } else {
            nn = mm = trc = tsc = nullptr;
        }
        nx = L64[0].nx; nz = L64[0].nz; nc = L64[0].nc; nlev = P.nlev;
        tid = G0::rank(); nt = G0::size();
        h = P.h; t2h = P.two_over_h2; idt = P.inv_dt; tr = P.tr; ts = P.ts;
    }

    // maximum over the group, returned to every thread
    __device__ __forceinline__ unsigned long long gmax(unsigned long long v) {
        v = block_max(v, red);
        if constexpr (CLU) {
            auto c = GClu::c();
            const int n = (int)c.num_blocks();
            if ((int)threadIdx.x < n) *c.map_shared_rank(&cred[cpar][c.block_rank()], threadIdx.x) = v;
            c.sync();
            for (int k = 0; k < n; ++k) v = cred[cpar][k] > v ? cred[cpar][k] : v;
            cpar ^= 1;                                 // the next but one write waits for the next barrier
        }
        return v;
    }
    // sum of a b over the cells, returned to every thread: one CTA's 512 chains
    // (cell q in chain q mod 512), its warps' trees and the tree over the warps, on
    // any group, so that a sample's sums do not depend on how many CTAs, and with
    // them how many other samples, the call gives it.  A cluster deals the 16
    // warps' chains out to its CTAs; a and b are complete (a barrier lies behind).
    __device__ __forceinline__ double gdot(const double* a, const double* b) {
        double s = 0.0;
        if constexpr (CLU) {
            constexpr int NW = CLUSTER_THREADS / 32;
            auto c = GClu::c();
            const int n = (int)c.num_blocks(), lane = threadIdx.x & 31;
            const int w = (int)(threadIdx.x >> 5) * n + (int)c.block_rank();
            if (w < NW) {
#pragma unroll 8
                for (int q = 32 * w + lane; q < nc; q += CLUSTER_THREADS) s = fma(a[q], b[q], s);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane < n)
                    *c.map_shared_rank(&cred[cpar][w], lane) = (unsigned long long)__double_as_longlong(s);
            }
            c.sync();
            s = lane < NW ? __longlong_as_double((long long)cred[cpar][lane]) : 0.0;
            cpar ^= 1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            return s;
        } else {
            for (int q = tid; q < nc; q += nt) s = fma(a[q], b[q], s);
            return block_sum(s, reinterpret_cast<double*>(red));
        }
    }
    // a level's threads in the set-up loops: a cluster's levels beyond lx belong
    // to its first CTA (their arrays may be in its shared memory)
    __device__ __forceinline__ bool mine(int l) const { return !CLU || l <= P.lx || tid < (int)blockDim.x; }
    __device__ __forceinline__ int rank_on(int l) const { return CLU && l > P.lx ? (int)threadIdx.x : tid; }
    __device__ __forceinline__ int size_on(int l) const { return CLU && l > P.lx ? (int)blockDim.x : nt; }
    __device__ __forceinline__ void sync_on(int l) const {
        if (!CLU || l <= P.lx) G0::sync();
        else if (tid < (int)blockDim.x) __syncthreads();
    }

    // the assembly's quotients (the same bits either way): with the van Genuchten
    // closure the integer pipes are the busier ones and the FP64 division is faster
    // (the cost map, 4096 samples of 32^2: 172 -> 168 ms), with Gardner's it is not (fixed.cuh)
    static __device__ __forceinline__ double quot(double a, double b) {
        if constexpr (CL == 0) return rich_fx::fx_div(a, b);
        else return a / b;
    }

    // conductivity of cell q's soil at head pp (Dirichlet faces, QoI)
    __device__ __forceinline__ double k_at(int q, double pp) const {
        if constexpr (CL == 0) {
            return pp < 0.0 ? Ks[q] * exp(aa[q] * pp) : Ks[q];
        } else {
            if (!(pp < 0.0)) return Ks[q];
            double S, krw, dS;
            vg_eval(aa[q], nn[q], mm[q], pp, S, krw, dS);
            return Ks[q] * krw;
        }
    }

    // Ks, alpha * scale + shift, (closure 1: n + shift, m, theta_r, theta_s),
    // initial head (uniform, or p_init (1 - exp(-init_decay z)) at the cell
    // centres, Eq. travellingwave), Dirichlet faces (fixed for the solve)
    __device__ void setup(int s) {
        const Lv64& F = L64[0];
        const size_t o = (size_t)s * nc;
        const double* lk = P.lnKs + o;
        const double* al = P.alpha + o;
        for (int q = tid; q < nc; q += nt) {
            Ks[q] = exp(lk[q]);
            aa[q] = al[q] * P.alpha_scale + P.alpha_shift;
            if (P.init_decay > 0.0) {
                const int j = fdiv(q, nx, F.mnx);
                p[q] = P.p_init * (1.0 - exp(-P.init_decay * (j + 0.5) * h));
            } else {
                p[q] = P.p_init;
            }
            if constexpr (CL == 1) {
                const double n = P.n_in[o + q] + P.n_shift;
                nn[q] = n;
                mm[q] = 1.0 - 1.0 / n;
                trc[q] = P.tr_in ? P.tr_in[o + q] : tr;
                tsc[q] = P.ts_in ? P.ts_in[o + q] : ts;
            }
        }
        G0::sync();
        for (int i = tid; i < nx; i += nt) {
            int T = (nz - 1) * nx + i, B = i;
            F.Tbt[i] = t2h * k_at(T, P.p_top);
            F.Tbb[i] = t2h * k_at(B, P.p_bot);
        }
        G0::sync();
        for (int l = 1; l < nlev; ++l) {
            if (mine(l)) {
                for (int I = rank_on(l); I < L64[l].nx; I += size_on(l)) {
                    L64[l].Tbt[I] = 0.25 * (0.5 * (L64[l - 1].Tbt[2 * I] + L64[l - 1].Tbt[2 * I + 1]));
                    L64[l].Tbb[I] = 0.25 * (0.5 * (L64[l - 1].Tbb[2 * I] + L64[l - 1].Tbb[2 * I + 1]));
                }
            }
            sync_on(l);
        }
    }

    // theta^n of the step's old head
    __device__ void theta_old() {
        for (int q = tid; q < nc; q += nt) {
            double pp = p[q];
            if constexpr (CL == 0) {
                thold[q] = pp < 0.0 ? tr + (ts - tr) * rich_fx::fx_exp(aa[q] * pp) : ts;
            } else {
                const double r = trc[q], t = tsc[q];
                thold[q] = pp < 0.0 ? r + (t - r) * vg_sat(aa[q], nn[q], mm[q], pp) : t;
            }
        }
        G0::sync();
    }

    // a cell's correction at the start of a solve on the finest level: zero, or
    // (nu1 > 0) in red cells the value v = f/D that the first red half-sweep
    // would give them, which the first cycle then skips
    __device__ __forceinline__ void start_cell(const Lv<TM>& M0, int i, int j, TM v) const {
        const bool black = (i + j) & 1;
        (black && M0.H ? M0.db : M0.dp)[sidx(M0, i, j)] = black || !M0.H || P.nu1 == 0 ? TM(0) : v;
    }

    // Picard system at p (Gardner closure, harmonic faces, f = -R), all levels;
    // returns ||f||_inf as a bit pattern
    __device__ unsigned long long assemble() {
        const Lv64& F = L64[0];
        const Lv<TM>& M0 = LM[0];
        for (int q = tid; q < nc; q += nt) {
            double pp = p[q], ks = Ks[q];
            if constexpr (CL == 0) {
                if (pp < 0.0) {
                    double a = aa[q];
                    double E = rich_fx::fx_exp(a * pp);
                    K[q] = ks * E;
                    th[q] = tr + (ts - tr) * E;
                    F.Cdt[q] = ((ts - tr) * a * E) * idt;
                } else {
                    K[q] = ks; th[q] = ts; F.Cdt[q] = 0.0;
                }
            } else {
                const double r = trc[q], t = tsc[q];
                if (pp < 0.0) {
                    double S, krw, dS;
                    vg_eval(aa[q], nn[q], mm[q], pp, S, krw, dS);
                    K[q] = ks * krw;
                    th[q] = r + (t - r) * S;
                    F.Cdt[q] = ((t - r) * dS) * idt;
                } else {
                    K[q] = ks; th[q] = t; F.Cdt[q] = 0.0;
                }
            }
        }
        G0::sync();
        for (int q = tid; q < nc; q += nt) {
            int j = fdiv(q, nx, F.mnx), i = q - j * nx;
            double kp = K[q];
            if (i < nx - 1) { double ke = K[q + 1]; F.Tx[q] = quot(t2h * kp * ke, kp + ke); }
            else F.Tx[q] = 0.0;
            if (j < nz - 1) { double kn = K[q + nx]; F.Tz[q] = quot(t2h * kp * kn, kp + kn); }
            else F.Tz[q] = 0.0;
        }
        G0::sync();
        unsigned long long m = 0;
        for (int q = tid; q < nc; q += nt) {
            int j = fdiv(q, nx, F.mnx), i = q - j * nx;
            double pp = p[q];
            double R = (th[q] - thold[q]) * idt;
            double d = F.Cdt[q];
            double te = 0.0, tw = 0.0, tn = 0.0, tsf = 0.0;
            if (i < nx - 1) { te = F.Tx[q];     R += -te * (p[q + 1] - pp); d += te; }
            if (i > 0)      { tw = F.Tx[q - 1]; R += -tw * (p[q - 1] - pp); d += tw; }
            if (j < nz - 1) { tn = F.Tz[q];     R += -tn * (p[q + nx] - pp) - tn * h; d += tn; }
            else { double t = F.Tbt[i]; R += -t * (P.p_top - pp) - t * h / 2.0; d += t; }
            if (j > 0)      { tsf = F.Tz[q - nx]; R += -tsf * (p[q - nx] - pp) + tsf * h; d += tsf; }
            else { double t = F.Tbb[i]; R += t * (pp - P.p_bot) + t * h / 2.0; d += t; }
            if (!SC || nlev == 1) F.D[q] = d;     // read by the defect, or the only level's factorisation
            f64[q] = -R;
            const int sq = sidx(M0, i, j);
            if constexpr (SC) {
                double inv = quot(1.0, d);
                M0.q[sq] = inv; M0.D[sq] = d;
                M0.c0[sq] = te * inv; M0.c1[sq] = tw * inv; M0.c2[sq] = tn * inv; M0.c3[sq] = tsf * inv;
                M0.f[sq] = -R * inv;
                start_cell(M0, i, j, -R * inv);
            } else {
                const float qf = 1.0f / (float)d;
                M0.c0[sq] = (TM)te; M0.c1[sq] = (TM)tn; M0.D[sq] = (TM)d;
                M0.q[sq] = (TM)qf;
                M0.f[sq] = (TM)(-R);
                dp64[q] = 0.0;
                start_cell(M0, i, j, (TM)(-R) * (TM)qf);
            }
            unsigned long long b = abs_bits(R);
            m = b > m ? b : m;
        }
        const unsigned long long fb = gmax(m);
        // coarse operators (Fig. diffUpscale)
        for (int l = 1; l < nlev; ++l) {
            const Lv64& Fl = L64[l - 1];
            const Lv64& Cl = L64[l];
            const Lv<TM>& Ml = LM[l];
            const int fx = Fl.nx;
            for (int c = mine(l) ? rank_on(l) : Cl.nc; c < Cl.nc; c += size_on(l)) {
                int J = fdiv(c, Cl.nx, Cl.mnx), I = c - J * Cl.nx;
                int f00 = (2 * J) * fx + 2 * I, f01 = f00 + fx;
                double cd = 0.25 * (Fl.Cdt[f00] + Fl.Cdt[f00 + 1] + Fl.Cdt[f01] + Fl.Cdt[f01 + 1]);
                double d = cd, te = 0.0, tw = 0.0, tn = 0.0, tsf = 0.0;
                if (I < Cl.nx - 1) { te = 0.25 * (0.5 * (Fl.Tx[f00 + 1] + Fl.Tx[f01 + 1])); d += te; }
                if (I > 0)         { tw = 0.25 * (0.5 * (Fl.Tx[f00 - 1] + Fl.Tx[f01 - 1])); d += tw; }
                if (J < Cl.nz - 1) { tn = 0.25 * (0.5 * (Fl.Tz[f01] + Fl.Tz[f01 + 1])); d += tn; }
                else d += Cl.Tbt[I];
                if (J > 0)         { tsf = 0.25 * (0.5 * (Fl.Tz[f00 - fx] + Fl.Tz[f00 - fx + 1])); d += tsf; }
                else d += Cl.Tbb[I];
                Cl.Tx[c] = te; Cl.Tz[c] = tn; Cl.Cdt[c] = cd;
                if (SC && l == nlev - 1) Cl.D[c] = d;
                const int sc = sidx(Ml, I, J);
                if constexpr (SC) {
                    double inv = quot(1.0, d);
                    Ml.q[sc] = 0.25 * inv; Ml.D[sc] = d;
                    Ml.c0[sc] = te * inv; Ml.c1[sc] = tw * inv; Ml.c2[sc] = tn * inv; Ml.c3[sc] = tsf * inv;
                } else {
                    Ml.c0[sc] = (TM)te; Ml.c1[sc] = (TM)tn; Ml.D[sc] = (TM)d;
                    Ml.q[sc] = (TM)(1.0f / (float)d);
                }
            }
            sync_on(l);
        }
        if (tid < 32) {
            const Lv64& Z = L64[nlev - 1];
            const Lv<TM>& Mz = LM[nlev - 1];
            if constexpr (SC) coarse_factor_warp<TM>(Z.nx, Z.nz, Z.Tx, Z.Tz, Z.D, Amat);
            else coarse_factor_warp<TM>(Z.nx, Z.nz, Mz.c0, Mz.c1, Mz.D, Amat);
        }
        G0::sync();
        return fb;
    }

    // one multigrid cycle: the V-cycle, or (WC, a separate kernel
    // instantiation so the V kernels keep their register allocation) the
    // cycle of index P.gamma
    // (fresh: the red cells already hold their first half-sweep's values)
    __device__ void mgcycle(const TM* f0, bool fresh) {
        if constexpr (WC) gwalk<TM, GCta>(LM, 0, nlev, P.lw, P.nu1, P.nu2, P.gamma, Amat, f0, fresh);
        else vcycle<TM, G0>(LM, nlev, P.lx, P.lw, P.nu1, P.nu2, Amat, f0, fresh);
    }

    // x += e (FP64, natural order += FP32 finest-level correction), then the
    // CTA synchronises
    __device__ __forceinline__ void add_correction(double* __restrict__ x, const TM* __restrict__ e) const {
        // (the mixed path's halves of dp never swap: e is one array)
        const Lv<TM>& M0 = LM[0];
        const unsigned mnx = L64[0].mnx;
#pragma unroll 4
        for (int q = tid; q < nc; q += nt) {
            const int j = fdiv(q, nx, mnx), i = q - j * nx;
            x[q] += (double)e[sidx(M0, i, j)];
        }
        G0::sync();
    }

    // FP64 defect r = f - A x of the finest operator, stored as the next FP32
    // right-hand side rf (with the FP32 correction ef at its start values, see
    // start_cell); returns this thread's max |r| as a bit pattern (distinct
    // arrays: restrict views)
    __device__ __forceinline__ unsigned long long defect(const double* __restrict__ f, const double* __restrict__ x,
                                                         const double* __restrict__ Tx,
                                                         const double* __restrict__ Tz,
                                                         const double* __restrict__ D,
                                                         const TM* __restrict__ qf, TM* __restrict__ rf,
                                                         TM* __restrict__ ef) const {
        const unsigned mnx = L64[0].mnx;
        const bool seed = P.nu1 > 0 && nlev > 1;
        unsigned long long mm = 0;
#pragma unroll 2
        for (int q = tid; q < nc; q += nt) {
            const int j = fdiv(q, nx, mnx), i = q - j * nx;
            double sn = 0.0;
            if (i < nx - 1) sn += Tx[q] * x[q + 1];
            if (i > 0)      sn += Tx[q - 1] * x[q - 1];
            if (j < nz - 1) sn += Tz[q] * x[q + nx];
            if (j > 0)      sn += Tz[q - nx] * x[q - nx];
            const double r = f[q] - (D[q] * x[q] - sn);
            const int sq = sidx(LM[0], i, j);
            rf[sq] = (TM)r;
            ef[sq] = seed && !((i + j) & 1) ? (TM)r * qf[sq] : TM(0);
            const unsigned long long b = abs_bits(r);
            mm = b > mm ? b : mm;
        }
        return mm;
    }

    // multigrid solve of A dp = f from dp = 0 (set up by assemble()); stops
    // when ||f - A dp||_inf < mg_tol max(1, ||f||_inf).  Returns false when a
    // norm is not finite.
    __device__ bool mg_solve(unsigned long long fb, long long& mg_tot, int& status) {
        const Lv<TM>& M0 = LM[0];
        const double fn = __longlong_as_double((long long)fb);
        const double target = P.mg_tol * (fn > 1.0 ? fn : 1.0);
        double rn = fn;
        int cyc = 0;
        // FP64: the stopping norm evaluates the next red half-sweep's values
        // anyway; it stores them in the second red half, and a cycle that
        // follows starts from that half (2 of about 30 FP64 instructions per
        // cell and cycle).  The accepted correction keeps the old half.
        const bool keep = SC && P.nu1 > 0 && P.nu2 > 0 && nlev > 1;
        bool fresh = true;                            // assemble() seeded the red cells
        while (rn >= target && cyc < P.mg_maxit) {
            unsigned long long rb;
            if constexpr (SC) {
                if (cyc > 0) {
                    if (keep) {
                        if (threadIdx.x == 0) { TM* t = LM[0].dp; LM[0].dp = LM[0].alt; LM[0].alt = t; }
                        __syncthreads();
                    }
                    fresh = keep;
                }
                mgcycle((const TM*)f64, fresh);
                ++cyc;
                rb = gmax(resid_norm<TM, G0>(M0, P.nu2 > 0 && nlev > 1, keep ? M0.alt : nullptr));
            } else {
                for (int in = 0; in < P.mixed_inner && cyc < P.mg_maxit; ++in) {
                    mgcycle(nullptr, in == 0);
                    ++cyc;
                }
                // dp += e in FP64, then the FP64 defect: stopping norm and the
                // next FP32 right-hand side
                add_correction(dp64, M0.dp);
                rb = gmax(defect(f64, dp64, L64[0].Tx, L64[0].Tz, L64[0].D, M0.q, M0.f, M0.dp));
            }
            if (rb > INF_BITS - 1) { mg_tot += cyc; return false; }
            rn = __longlong_as_double((long long)rb);
        }
        if constexpr (SC) {
            if (cyc == 0) {                           // nothing to solve: the correction is zero, not its seed
                for (int c = tid; c < M0.H; c += nt) M0.dp[c] = TM(0);
                G0::sync();
            }
        }
        mg_tot += cyc;
        if (!(rn < target)) status = max(status, (int)RICH_MG_MAXIT);
        return true;
    }

    // one implicit-Euler step by modified Picard (Sec. 4.1); returns false if
    // the sample failed.  A failure (PICARD_MAXIT, NONFINITE) replaces any
    // earlier MG_MAXIT flag: the sample's QoI is undefined, whatever happened
    // in its multigrid solves before
    __device__ bool time_step(long long& pic_tot, long long& mg_tot, int& maxpic, int& status) {
        theta_old();
        int k = 0;
        bool alive = true;
        for (;;) {
            const unsigned long long fb = assemble();
            if (fb > INF_BITS - 1) { status = RICH_NONFINITE; alive = false; break; }
            if (!mg_solve(fb, mg_tot, status)) { status = RICH_NONFINITE; alive = false; break; }
            unsigned long long dm = 0;
            for (int q = tid; q < nc; q += nt) {
                double d;
                if constexpr (SC) {
                    const int j = fdiv(q, nx, L64[0].mnx);
                    d = dp_at(LM[0], q - j * nx, j);
                } else {
                    d = dp64[q];
                }
                p[q] += d;
                unsigned long long b = abs_bits(d);
                dm = b > dm ? b : dm;
            }
            const unsigned long long db = gmax(dm);
            ++k;
            ++pic_tot;
            if (db > INF_BITS - 1) { status = RICH_NONFINITE; alive = false; break; }
            if (__longlong_as_double((long long)db) < P.picard_tol) break;
            if (k >= P.picard_maxit) { status = RICH_PICARD_MAXIT; alive = false; break; }
        }
        maxpic = max(maxpic, k);
        return alive;
    }

    // mean outward Darcy flux through the bottom faces (valid in warp 0)
    __device__ double qoi_warp0() const {
        double acc = 0.0;
        for (int i = tid; i < nx; i += 32) {
            double kb = k_at(i, P.p_bot);
            acc += kb * (2.0 * (p[i] - P.p_bot) / h + 1.0);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        return acc / nx;
    }

    // ------------------------------------------------------------ adjoint
    // Jacobian pieces at the assembled state p = p^n: for every cell c and each
    // interior face f (E, W, N, S) D_fc = T_f - g_cf dT_f/dp_c with
    // g_cf = p_nb - p_c + s h (s = +1 north, -1 south), and the diagonal
    // C_c/dt + Dirichlet T_b; so (J^T lam)_c = dg_c lam_c + sum_f D_fc (lam_c - lam_nb).
    __device__ void adj_prepare(double* dE, double* dW, double* dN, double* dS, double* dg) {
        const Lv64& F = L64[0];
        for (int q = tid; q < nc; q += nt) {
            int j = fdiv(q, nx, F.mnx), i = q - j * nx;
            const double pc = p[q], kc = K[q];
            const double dk = pc < 0.0 ? aa[q] * kc : 0.0;      // dK_c/dp_c
            double e = 0.0, w = 0.0, n = 0.0, s = 0.0, d = F.Cdt[q];
            if (i < nx - 1) { double kn = K[q + 1], den = kc + kn;
                e = F.Tx[q] - (p[q + 1] - pc) * (t2h * kn * kn / (den * den)) * dk; }
            if (i > 0)      { double kn = K[q - 1], den = kc + kn;
                w = F.Tx[q - 1] - (p[q - 1] - pc) * (t2h * kn * kn / (den * den)) * dk; }
            if (j < nz - 1) { double kn = K[q + nx], den = kc + kn;
                n = F.Tz[q] - (p[q + nx] - pc + h) * (t2h * kn * kn / (den * den)) * dk; }
            else d += F.Tbt[i];
            if (j > 0)      { double kn = K[q - nx], den = kc + kn;
                s = F.Tz[q - nx] - (p[q - nx] - pc - h) * (t2h * kn * kn / (den * den)) * dk; }
            else d += F.Tbb[i];
            dE[q] = e; dW[q] = w; dN[q] = n; dS[q] = s; dg[q] = d;
        }
        G0::sync();
    }

    __device__ __forceinline__ double jt_apply(const double* dE, const double* dW, const double* dN,
                                               const double* dS, const double* dg, const double* lam,
                                               int q) const {
        int j = fdiv(q, nx, L64[0].mnx), i = q - j * nx;
        const double l = lam[q];
        double v = dg[q] * l;
        if (i < nx - 1) v += dE[q] * (l - lam[q + 1]);
        if (i > 0)      v += dW[q] * (l - lam[q - 1]);
        if (j < nz - 1) v += dN[q] * (l - lam[q + nx]);
        if (j > 0)      v += dS[q] * (l - lam[q - nx]);
        return v;
    }

    // approximate e = A^{-1} r by ninner V-cycles from e = 0 (A: the Picard
    // operator assembled at the same state); e is returned in the finest
    // level's dp
    __device__ void mg_apply(const double* r, int ninner) {
        const Lv<TM>& M0 = LM[0];
        for (int q = tid; q < nc; q += nt) {
            const int j = fdiv(q, nx, L64[0].mnx), sq = sidx(M0, q - j * nx, j);
            const TM v = (TM)r[q] * M0.q[sq];
            M0.f[sq] = SC ? v : (TM)r[q];
            start_cell(M0, q - j * nx, j, v);
        }
        G0::sync();
        for (int k = 0; k < ninner; ++k) {
            if constexpr (SC) mgcycle(r, k == 0);
            else mgcycle(nullptr, k == 0);
        }
    }

    // J^T lam = rhs by defect correction preconditioned with CCMG on A:
    // lam += A^{-1}(rhs - J^T lam) until ||rhs - J^T lam|| <= adj_tol ||rhs||.
    // Returns the number of outer iterations (adj_maxit + 1 when not converged).
    __device__ int adj_solve(const double* dE, const double* dW, const double* dN, const double* dS,
                             const double* dg, const double* rhs, double* lam, double* r) {
        const Lv<TM>& M0 = LM[0];
        unsigned long long m = 0;
        for (int q = tid; q < nc; q += nt) {
            lam[q] = 0.0;
            r[q] = rhs[q];
            unsigned long long b = abs_bits(rhs[q]);
            m = b > m ? b : m;
        }
        const unsigned long long b0 = gmax(m);
        const double target = P.adj_tol * __longlong_as_double((long long)b0);
        if (b0 == 0) return 0;
        for (int it = 1; it <= P.adj_maxit; ++it) {
            mg_apply(r, P.adj_inner);
            for (int q = tid; q < nc; q += nt) {
                const int j = fdiv(q, nx, L64[0].mnx);
                lam[q] += (double)dp_at(M0, q - j * nx, j);
            }
            G0::sync();
            unsigned long long mm = 0;
            for (int q = tid; q < nc; q += nt) {
                double v = rhs[q] - jt_apply(dE, dW, dN, dS, dg, lam, q);
                r[q] = v;
                unsigned long long b = abs_bits(v);
                mm = b > mm ? b : mm;
            }
            const unsigned long long rb = gmax(mm);
            if (rb > INF_BITS - 1) return P.adj_maxit + 1;
            if (__longlong_as_double((long long)rb) <= target) return it;
        }
        return P.adj_maxit + 1;
    }

    // e = M^{-1} r: ninner cycles of the Picard operator A from zero (a fixed
    // linear operator: the same cycles on the same matrix), copied to out
    __device__ void precond(const double* r, double* out) {
        mg_apply(r, P.adj_inner);
        for (int q = tid; q < nc; q += nt) {
            const int j = fdiv(q, nx, L64[0].mnx);
            out[q] = (double)dp_at(LM[0], q - j * nx, j);
        }
        G0::sync();
    }

    // y = J^T x over all cells, then the CTA synchronises
    __device__ void jt_vec(const double* dE, const double* dW, const double* dN, const double* dS,
                           const double* dg, const double* x, double* y) {
        for (int q = tid; q < nc; q += nt) y[q] = jt_apply(dE, dW, dN, dS, dg, x, q);
        G0::sync();
    }

    // J^T lam = rhs by BiCGStab (van der Vorst 1992) right-preconditioned with
    // the CCMG cycles of A: converged when the TRUE residual ||rhs - J^T lam||
    // <= adj_tol ||rhs|| (checked explicitly whenever the recursive residual
    // says so; a mismatch restarts the recurrence from the true residual).
    // Returns the number of preconditioner applications (adj_maxit + 1 when
    // not converged); w holds the vectors r (also s), r^, p, v, t, p^, s^.
    __device__ int adj_solve_bicgstab(const double* dE, const double* dW, const double* dN, const double* dS,
                                      const double* dg, const double* rhs, double* lam, double* r, double* rh,
                                      double* pk, double* v, double* t, double* ph, double* sh) {
        unsigned long long m = 0;
        for (int q = tid; q < nc; q += nt) {
            lam[q] = 0.0;
            unsigned long long b = abs_bits(rhs[q]);
            m = b > m ? b : m;
        }
        const unsigned long long b0 = gmax(m);
        if (b0 == 0) return 0;
        const double target = P.adj_tol * __longlong_as_double((long long)b0);
        int apps = 0;
        bool restart = true;
        double rho = 1.0, alpha = 1.0, omega = 1.0;
        while (apps < P.adj_maxit) {
            if (restart) {                          // r = r^ = rhs - J^T lam, p = v = 0
                unsigned long long rm = 0;
                for (int q = tid; q < nc; q += nt) {
                    const double rv = rhs[q] - jt_apply(dE, dW, dN, dS, dg, lam, q);
                    r[q] = rv; rh[q] = rv; pk[q] = 0.0; v[q] = 0.0;
                    unsigned long long b = abs_bits(rv);
                    rm = b > rm ? b : rm;
                }
                const unsigned long long rb = gmax(rm);
                if (rb > INF_BITS - 1) break;
                if (__longlong_as_double((long long)rb) <= target) return apps;
                rho = alpha = omega = 1.0;
                restart = false;
                if (apps > 0) ++apps;               // a restart counts as one application
            }
            const double rho_new = gdot(rh, r);
            if (!(fabs(rho_new) > 0.0) || !isfinite(rho_new)) { restart = true; if (!isfinite(rho_new)) break; continue; }
            const double beta = (rho_new / rho) * (alpha / omega);
            for (int q = tid; q < nc; q += nt) pk[q] = r[q] + beta * (pk[q] - omega * v[q]);
            G0::sync();
            precond(pk, ph); ++apps;
            jt_vec(dE, dW, dN, dS, dg, ph, v);
            const double den = gdot(rh, v);
            if (!(fabs(den) > 0.0) || !isfinite(den)) { restart = true; if (!isfinite(den)) break; continue; }
            alpha = rho_new / den;
            unsigned long long sm = 0;
            for (int q = tid; q < nc; q += nt) {
                const double sv = r[q] - alpha * v[q];
                r[q] = sv;                                  // r now holds s
                unsigned long long b = abs_bits(sv);
                sm = b > sm ? b : sm;
            }
            const unsigned long long sb = gmax(sm);
            if (sb > INF_BITS - 1) break;
            if (__longlong_as_double((long long)sb) <= target) {
                for (int q = tid; q < nc; q += nt) lam[q] += alpha * ph[q];
                G0::sync();
                if (true_resid_ok(dE, dW, dN, dS, dg, rhs, lam, target)) return apps;
                restart = true;
                continue;
            }
            precond(r, sh); ++apps;
            jt_vec(dE, dW, dN, dS, dg, sh, t);
            const double ts = gdot(t, r);
            const double tt = gdot(t, t);
            omega = tt > 0.0 ? ts / tt : 0.0;
            unsigned long long rm = 0;
            for (int q = tid; q < nc; q += nt) {
                lam[q] += alpha * ph[q] + omega * sh[q];
                const double rv = r[q] - omega * t[q];
                r[q] = rv;
                unsigned long long b = abs_bits(rv);
                rm = b > rm ? b : rm;
            }
            const unsigned long long rb = gmax(rm);
            if (rb > INF_BITS - 1) break;
            if (__longlong_as_double((long long)rb) <= target) {
                if (true_resid_ok(dE, dW, dN, dS, dg, rhs, lam, target)) return apps;
                restart = true;
                continue;
            }
            if (!(omega != 0.0)) restart = true;
            rho = rho_new;
        }
        return P.adj_maxit + 1;
    }

    // J^T lam = rhs by restarted GMRES(ADJ_M) (Saad & Schultz 1986), right-
    // preconditioned with the CCMG cycles of A, modified Gram-Schmidt, Givens
    // rotations; each cycle ends with the update lam += Z y and the TRUE
    // residual ||rhs - J^T lam||_inf <= adj_tol ||rhs||_inf decides.  The
    // Hessenberg matrix and rotations are computed by every thread from the
    // same block sums (uniform control flow).  One CTA only (not a cluster).  Returns the number of
    // preconditioner applications (adj_maxit + 1 when not converged).
    __device__ int adj_solve_gmres(const double* dE, const double* dW, const double* dN, const double* dS,
                                   const double* dg, const double* rhs, double* lam, double* kry) {
        // Hessenberg matrix, rotations, right-hand side and solution of the
        // small least-squares problem: one copy per CTA, updated by thread 0
        __shared__ double sH[ADJ_M + 1][ADJ_M], scs[ADJ_M], ssn[ADJ_M], sg[ADJ_M + 1], sy[ADJ_M];
        double* redd = reinterpret_cast<double*>(red);
        double* V = kry;                                  // [ADJ_M + 1][nc]
        double* Z = kry + (size_t)(ADJ_M + 1) * nc;       // [ADJ_M][nc]
        unsigned long long m = 0;
        for (int q = tid; q < nc; q += nt) {
            lam[q] = 0.0;
            unsigned long long b = abs_bits(rhs[q]);
            m = b > m ? b : m;
        }
        const unsigned long long b0 = block_max(m, red);
        if (b0 == 0) return 0;
        const double target = P.adj_tol * __longlong_as_double((long long)b0);
        int apps = 0;
        while (apps < P.adj_maxit) {
            // r = rhs - J^T lam (the true residual), its inf-norm and 2-norm
            unsigned long long rm = 0;
            double s2 = 0.0;
            for (int q = tid; q < nc; q += nt) {
                const double rv = rhs[q] - jt_apply(dE, dW, dN, dS, dg, lam, q);
                V[q] = rv;
                s2 += rv * rv;
                unsigned long long b = abs_bits(rv);
                rm = b > rm ? b : rm;
            }
            const unsigned long long rb = block_max(rm, red);
            const double beta = sqrt(block_sum(s2, redd));
            if (rb > INF_BITS - 1 || !(beta > 0.0)) break;
            if (__longlong_as_double((long long)rb) <= target) return apps;
            const double ib = 1.0 / beta;
            for (int q = tid; q < nc; q += nt) V[q] *= ib;
            if (tid == 0) {
                for (int i = 0; i <= ADJ_M; ++i) sg[i] = 0.0;
                sg[0] = beta;
            }
            __syncthreads();
            int k = 0;
            for (; k < ADJ_M && apps < P.adj_maxit; ++k) {
                double* vk = V + (size_t)k * nc;
                double* zk = Z + (size_t)k * nc;
                double* w = V + (size_t)(k + 1) * nc;
                precond(vk, zk); ++apps;
                jt_vec(dE, dW, dN, dS, dg, zk, w);
                for (int i = 0; i <= k; ++i) {                  // modified Gram-Schmidt
                    const double* vi = V + (size_t)i * nc;
                    double d = 0.0;
                    for (int q = tid; q < nc; q += nt) d += w[q] * vi[q];
                    const double h = block_sum(d, redd);
                    if (tid == 0) sH[i][k] = h;
                    for (int q = tid; q < nc; q += nt) w[q] -= h * vi[q];
                    __syncthreads();
                }
                double d = 0.0;
                for (int q = tid; q < nc; q += nt) d += w[q] * w[q];
                const double hn = sqrt(block_sum(d, redd));
                if (hn > 0.0) {
                    const double ih = 1.0 / hn;
                    for (int q = tid; q < nc; q += nt) w[q] *= ih;
                }
                if (tid == 0) {                                  // rotations on column k
                    sH[k + 1][k] = hn;
                    for (int i = 0; i < k; ++i) {
                        const double a = sH[i][k], b = sH[i + 1][k];
                        sH[i][k] = scs[i] * a + ssn[i] * b;
                        sH[i + 1][k] = -ssn[i] * a + scs[i] * b;
                    }
                    const double a = sH[k][k], b = sH[k + 1][k];
                    const double rr = sqrt(a * a + b * b);
                    scs[k] = rr > 0.0 ? a / rr : 1.0;
                    ssn[k] = rr > 0.0 ? b / rr : 0.0;
                    sH[k][k] = rr; sH[k + 1][k] = 0.0;
                    sg[k + 1] = -ssn[k] * sg[k];
                    sg[k] = scs[k] * sg[k];
                }
                __syncthreads();
                const double gk = sg[k + 1];
                // the 2-norm estimate bounds the inf-norm: the cycle may stop early
                if (!(hn > 0.0) || !isfinite(gk) || fabs(gk) <= target) { ++k; break; }
            }
            if (tid == 0) {                                      // y = H^{-1} g, k x k upper triangular
                for (int i = k - 1; i >= 0; --i) {
                    double t = sg[i];
                    for (int j = i + 1; j < k; ++j) t -= sH[i][j] * sy[j];
                    sy[i] = sH[i][i] != 0.0 ? t / sH[i][i] : 0.0;
                }
            }
            __syncthreads();
            for (int q = tid; q < nc; q += nt) {
                double acc = lam[q];
                for (int j = 0; j < k; ++j) acc += sy[j] * Z[(size_t)j * nc + q];
                lam[q] = acc;
            }
            __syncthreads();
        }
        return true_resid_ok(dE, dW, dN, dS, dg, rhs, lam, target) ? apps : P.adj_maxit + 1;
    }

    // ||rhs - J^T lam||_inf <= target (the true residual)
    __device__ bool true_resid_ok(const double* dE, const double* dW, const double* dN, const double* dS,
                                  const double* dg, const double* rhs, const double* lam, double target) {
        unsigned long long m = 0;
        for (int q = tid; q < nc; q += nt) {
            unsigned long long b = abs_bits(rhs[q] - jt_apply(dE, dW, dN, dS, dg, lam, q));
            m = b > m ? b : m;
        }
        const unsigned long long rb = gmax(m);
        return rb <= INF_BITS - 1 && __longlong_as_double((long long)rb) <= target;
    }

    // g -= (dR/dm)^T lam at the assembled state (m = ln Ks): interior faces
    // contribute -g_cf (lam_c - lam_nb) dT_f/dm_c with dT_f/dm_c =
    // (2/h^2) K_nb^2 K_c / (K_c + K_nb)^2; Dirichlet faces -g_b T_b lam_c
    __device__ void adj_grad_update(const double* lam, double* g) {
        const Lv64& F = L64[0];
        for (int q = tid; q < nc; q += nt) {
            int j = fdiv(q, nx, F.mnx), i = q - j * nx;
            const double pc = p[q], kc = K[q], lc = lam[q];
            double v = 0.0;
            if (i < nx - 1) { double kn = K[q + 1], den = kc + kn;
                v -= (p[q + 1] - pc) * (lc - lam[q + 1]) * (t2h * kn * kn * kc / (den * den)); }
            if (i > 0)      { double kn = K[q - 1], den = kc + kn;
                v -= (p[q - 1] - pc) * (lc - lam[q - 1]) * (t2h * kn * kn * kc / (den * den)); }
            if (j < nz - 1) { double kn = K[q + nx], den = kc + kn;
                v -= (p[q + nx] - pc + h) * (lc - lam[q + nx]) * (t2h * kn * kn * kc / (den * den)); }
            else v -= (P.p_top - pc + h / 2.0) * F.Tbt[i] * lc;
            if (j > 0)      { double kn = K[q - nx], den = kc + kn;
                v -= (p[q - nx] - pc - h) * (lc - lam[q - nx]) * (t2h * kn * kn * kc / (den * den)); }
            else v -= (P.p_bot - pc - h / 2.0) * F.Tbb[i] * lc;
            g[q] -= v;
        }
        G0::sync();
    }
};

template <typename TM>
__device__ __forceinline__ void init_levels(const FParams& P, char* slot, unsigned char* sm, Lv64* L64,
                                            Lv<TM>* LM) {
    constexpr bool SC = Scaled<TM>::value;
    const int nlev = P.nlev;
    if ((int)threadIdx.x < nlev) {
        const int l = threadIdx.x;
        Lv64& a = L64[l];
        a.nx = P.nx[l]; a.nz = P.nz[l]; a.nc = a.nx * a.nz; a.mnx = P.mnx[l];
        double** pp[N64] = {&a.Tx, &a.Tz, &a.Cdt, &a.D, &a.Tbt, &a.Tbb};
        for (int k = 0; k < N64; ++k)
            *pp[k] = P.s64[l][k] >= 0 ? (double*)(sm + P.s64[l][k]) : (double*)(slot + P.o64[l][k]);
        Lv<TM>& b = LM[l];
        b.nx = a.nx; b.nz = a.nz; b.hx = a.nx >> 1; b.nc = a.nc; b.mnx = P.mnx[l]; b.mhx = P.mhx[l];
        b.H = l < nlev - 1 ? b.hx * b.nz : 0;             // colour-split unless coarsest
        TM** qq[NMG] = {&b.c0, &b.c1, &b.c2, &b.c3, &b.q, &b.f, &b.dp, &b.D};
        for (int k = 0; k < NMG; ++k)
            *qq[k] = P.smg[l][k] >= 0 ? (TM*)(sm + P.smg[l][k])
                   : P.omg[l][k] >= 0 ? (TM*)(slot + P.omg[l][k]) : nullptr;
        if (P.osm[l] >= 0) b.dp = (TM*)(sm + P.osm[l]);   // corrections of small levels on chip
        // the second red half: on chip beside dp, else the natural-order diagonal's
        // place in the slot (the FP64 cycles read their own copy of it)
        b.alt = l > 0 || !SC ? nullptr : P.osm_alt >= 0 ? (TM*)(sm + P.osm_alt) : (TM*)a.D;
        b.db = b.dp;
        if constexpr (!SC) { b.D = b.c3; b.c3 = nullptr; }   // FP32: D in the c3 slot
    }
    __syncthreads();
}

// one sample on its group, results to the caller's arrays; a group holds `sms`
// CTAs (the time it is charged)
template <typename C_t>
__device__ __forceinline__ void solve_sample(C_t& C, const FParams& P, int s, int sms) {
    const int nc = C.nc, tid = C.tid, nt = C.nt;
    const unsigned long long t0 = globaltimer_ns();
    C.setup(s);
    int status = RICH_OK, maxpic = 0;
    bool alive = true;
    long long pic_tot = 0, mg_tot = 0;
    for (int step = 0; step < P.nsteps && alive; ++step)
        alive = C.time_step(pic_tot, mg_tot, maxpic, status);
    if (tid < 32) {
        const double q = C.qoi_warp0();
        if (tid == 0) {
            P.qoi[s] = alive ? q : __longlong_as_double(0x7FF8000000000000ll);
            if (P.status) P.status[s] = status;
            if (P.pic_total) P.pic_total[s] = pic_tot;
            if (P.mg_total) P.mg_total[s] = mg_tot;
            if (P.maxpic) P.maxpic[s] = maxpic;
            if (P.t_ns) P.t_ns[s] = (int64_t)(globaltimer_ns() - t0) * sms;
        }
    }
    if (P.p_final)
        for (int q = tid; q < nc; q += nt) P.p_final[(size_t)s * nc + q] = C.p[q];
}

template <typename TM, int NT, bool WC, int CL>
__global__ void __launch_bounds__(NT, NT == 32 ? 32 : NT <= 128 ? 8 : NT <= 256 ? 4 : NT == 512 ? 2 : 1)
k_fused(const FParams P) {
    extern __shared__ unsigned char smraw[];
    __shared__ unsigned long long red[33];
    __shared__ int s_sample;
    __shared__ Lv64 L64[MAXL];
    __shared__ Lv<TM> LM[MAXL];
    char* slot = P.scratch + (size_t)blockIdx.x * P.slot_bytes;
    init_levels<TM>(P, slot, smraw, L64, LM);
    Cta<TM, WC, CL> C(P, slot, L64, LM, reinterpret_cast<TM*>(smraw), red);
    const int tid = C.tid;
    for (;;) {
        if (tid == 0) s_sample = atomicAdd(P.queue, 1);
        __syncthreads();
        const int s = s_sample;
        __syncthreads();
        if (s >= P.S) break;
        solve_sample(C, P, s, 1);
        __syncthreads();
    }
}

// The same with a cluster of CTAs, each on an SM of its own, per sample: a batch
// with fewer samples than half the SMs leaves the others idle, and a large grid's
// half-sweeps are long enough to pay for a cluster barrier (about a microsecond
// with the reads that follow it) after each.  Fine levels run on all CTAs, their
// arrays in the slot; the first CTA runs the rest (vcycle).  256^2 x 24 samples,
// mixed: 247 -> 86 ms; one 64^2 sample, FP64: 146 -> 104 ms.
template <typename TM, int CL>
__global__ void __launch_bounds__(CLUSTER_THREADS, 1)
k_fused_cluster(const FParams P) {
    extern __shared__ unsigned char smraw[];
    __shared__ unsigned long long red[33];
    __shared__ unsigned long long cred[2][CLUSTER_THREADS / 32];
    __shared__ int s_sample;
    __shared__ Lv64 L64[MAXL];
    __shared__ Lv<TM> LM[MAXL];
    auto c = GClu::c();
    const int n = (int)c.num_blocks();
    char* slot = P.scratch + (size_t)(blockIdx.x / n) * P.slot_bytes;
    init_levels<TM>(P, slot, smraw, L64, LM);
    Cta<TM, false, CL, GClu> C(P, slot, L64, LM, reinterpret_cast<TM*>(smraw), red);
    C.cred = cred;
    c.sync();                                         // every CTA runs before its memory is written to
    for (;;) {
        if (C.tid == 0) {
            const int s = atomicAdd(P.queue, 1);
            for (int k = 0; k < n; ++k) *c.map_shared_rank(&s_sample, k) = s;
        }
        c.sync();
        const int s = s_sample;
        if (s >= P.S) break;
        solve_sample(C, P, s, n);
        c.sync();
    }
}

}  // namespace

namespace {
// launch shapes of one (cycle precision, closure) pair: 128, 256, 512 or 1024
// threads, each with the V-cycle and the gamma >= 2 cycle instantiation
template <typename TM, int NT, bool WC, int CL>
int occ_one(const FParams& P, size_t smem, int* occ) {
    if (int e = allow_dyn_smem((const void*)k_fused<TM, NT, WC, CL>, smem)) return e;
    RICH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k_fused<TM, NT, WC, CL>, NT, smem));
    if (*occ < 1) *occ = 1;
    return 0;
}

template <typename TM, int CL>
int occ_shapes(const FParams& P, size_t smem, int nt, int* occ) {
    const bool wc = P.gamma > 1;
    if (nt == 1024) return wc ? occ_one<TM, 1024, true, CL>(P, smem, occ) : occ_one<TM, 1024, false, CL>(P, smem, occ);
    if (nt == 256) return wc ? occ_one<TM, 256, true, CL>(P, smem, occ) : occ_one<TM, 256, false, CL>(P, smem, occ);
    if (nt == 128) return wc ? occ_one<TM, 128, true, CL>(P, smem, occ) : occ_one<TM, 128, false, CL>(P, smem, occ);
    if (nt == 32) return wc ? occ_one<TM, 32, true, CL>(P, smem, occ) : occ_one<TM, 32, false, CL>(P, smem, occ);
    return wc ? occ_one<TM, 512, true, CL>(P, smem, occ) : occ_one<TM, 512, false, CL>(P, smem, occ);
}

template <typename TM, int CL>
void launch_shapes(const FParams& P, int grid, size_t smem, int nt, cudaStream_t st) {
    const bool wc = P.gamma > 1;
    if (nt == 1024) {
        if (wc) k_fused<TM, 1024, true, CL><<<grid, 1024, smem, st>>>(P);
        else k_fused<TM, 1024, false, CL><<<grid, 1024, smem, st>>>(P);
    } else if (nt == 256) {
        if (wc) k_fused<TM, 256, true, CL><<<grid, 256, smem, st>>>(P);
        else k_fused<TM, 256, false, CL><<<grid, 256, smem, st>>>(P);
    } else if (nt == 128) {
        if (wc) k_fused<TM, 128, true, CL><<<grid, 128, smem, st>>>(P);
        else k_fused<TM, 128, false, CL><<<grid, 128, smem, st>>>(P);
    } else if (nt == 32) {
        if (wc) k_fused<TM, 32, true, CL><<<grid, 32, smem, st>>>(P);
        else k_fused<TM, 32, false, CL><<<grid, 32, smem, st>>>(P);
    } else {
        if (wc) k_fused<TM, 512, true, CL><<<grid, 512, smem, st>>>(P);
        else k_fused<TM, 512, false, CL><<<grid, 512, smem, st>>>(P);
    }
}

// clusters of n CTAs: fit != null asks how many the GPU holds at a time, else
// `clusters` of them are launched
inline int cluster_call(void (*kernel)(FParams), const FParams& P, size_t smem, int n, int clusters, cudaStream_t st,
                        int* fit) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n; at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(clusters * n)); cfg.blockDim = dim3(CLUSTER_THREADS);
    cfg.dynamicSmemBytes = smem; cfg.stream = st; cfg.attrs = at; cfg.numAttrs = 1;
    if (fit) {
        if (int e = allow_dyn_smem((const void*)kernel, smem)) return e;
        RICH_CUDA(cudaOccupancyMaxActiveClusters(fit, kernel, &cfg));
        return 0;
    }
    RICH_CUDA(cudaLaunchKernelEx(&cfg, kernel, P));
    return 0;
}
}  // namespace
