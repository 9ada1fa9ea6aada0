// Persistent fused solver: one kernel launch solves a whole batch (host
// side: slot layout, launch shapes, entry points; the kernels are in
// fused_kernel.cuh).
#include "fused_kernel.cuh"
#include <algorithm>
#include <mutex>

namespace {

unsigned magic(int d) { return d <= 1 ? 0u : (unsigned)((0x100000000ull / (unsigned)d) + 1); }
size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// Dynamic shared memory of a CTA (no device work): the coarsest level's
// factored matrix; then the arrays that the cycles read on the small coarse levels
// (levels l >= 1 with at most WARP_CELLS cells: the
// multigrid arrays, and for FP64 the coarsest level's faces and diagonal,
// from which the matrix is assembled); then the corrections dp of as many of the other levels
// (coarsest first) as fit the budget of the launch shape (one 1024-thread CTA
// per SM may use ~220 KB, two 512-thread CTAs ~104 KB each, four 256-thread
// CTAs ~50 KB each, eight 128-thread CTAs ~24 KB each), so that the
// Gauss-Seidel neighbour reads of those levels
// stay on chip; levels that do not fit keep dp in the slot.  Results do not
// depend on where an array lives.
constexpr int WARP_CELLS = 256;
// Warp 0 alone runs the on-chip levels, in FP64 only those of at most 64 cells: it
// reaches a quarter of the SM's FP64 pipe, where a half-sweep of a 16^2 level takes
// 1024 clocks against 256 on four warps, more than the barrier it saves (ms with
// 256 / 64 / 16 cells: 32^2 x 64 117 / 104 / 104, 64^2 x 1 103 / 96 / 97, 32^2 x 608
// 82 / 71 / 75, 64^2 x 48 adjoint 146 / 137 / 138, cost map 188 / 184 / 188, a
// 16^2...64^2 MLMC estimate 707 / 666 / 686; full batches of large grids alike).
constexpr int WARP_CELLS64 = 64;

// A cluster (cells > 0) runs its levels of at least `cells` cells on all its CTAs
// (lx of them): their corrections, and the next level's, stay in the slot.
static void plan_smem(FParams& P, int nt, long long cells = 0) {
    const size_t w = P.mixed ? 4 : 8;
    const int c = P.nlev - 1;
    const size_t nnc = (size_t)P.nx[c] * P.nz[c];
    auto al16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    size_t off = al16(nnc * (nnc + 1) * w);
    const size_t budget = nt == 1024 ? 220 * 1024 : nt == 512 ? 104 * 1024 : nt == 256 ? 50 * 1024
                        : nt == 128 ? 24 * 1024 : 3 * 1024;
    for (int l = 0; l < MAXL; ++l) {
        P.osm[l] = -1;
        for (int k = 0; k < N64; ++k) P.s64[l][k] = -1;
        for (int k = 0; k < NMG; ++k) P.smg[l][k] = -1;
    }
    // small levels below the finest run on warp 0 with their arrays on chip;
    // a one-warp CTA (32 threads, 32 CTAs per SM) runs every level itself and
    // keeps them in its slot: on-chip copies would cost it its occupancy
    int ls = P.nlev;                          // first level with its arrays on chip
    for (int l = 1; l < P.nlev && nt > 32; ++l)
        if ((size_t)P.nx[l] * P.nz[l] <= (size_t)WARP_CELLS) { ls = l; break; }
    P.lw = ls;
    while (!P.mixed && P.lw < P.nlev && P.nx[P.lw] * P.nz[P.lw] > WARP_CELLS64) ++P.lw;
    P.lx = 0;
    while (cells > 0 && P.lx < std::min(ls, P.nlev - 1) - 1 && (long long)P.nx[P.lx] * P.nz[P.lx] >= cells) ++P.lx;
    for (int l = ls; l < P.nlev; ++l) {
        const size_t nc = (size_t)P.nx[l] * P.nz[l];
        if (!P.mixed) {
            for (int k = 0; k < N64; ++k) {
                if (!(l == c && (k == A_TX || k == A_TZ || k == A_D))) continue;
                P.s64[l][k] = (long long)off;
                off = al16(off + nc * 8);
            }
        }
        for (int k = 0; k < NMG; ++k) {
            if (P.omg[l][k] < 0) continue;
            P.smg[l][k] = (long long)off;
            off = al16(off + nc * w);
        }
    }
    for (int l = ls - 1; l >= (P.lx > 0 ? P.lx + 1 : 0); --l) {
        const size_t bytes = al16((size_t)P.nx[l] * P.nz[l] * w);
        if (off + bytes > budget) break;
        P.osm[l] = (long long)off;
        off += bytes;
    }
    // the finest FP64 level's second red half goes with its dp
    P.osm_alt = -1;
    const size_t half = al16((size_t)P.nx[0] * P.nz[0] / 2 * w);
    if (!P.mixed && P.osm[0] >= 0 && off + half <= budget) { P.osm_alt = (long long)off; off += half; }
    P.smem_bytes = (long long)off;
}

static int fused_setup(const rich_problem_t* pb, int S, FParams& P, int ckpt_every = 0, bool keep_states = false) {
    P = FParams{};
    const int nlev = rich_count_levels(pb->nx, pb->nz);
    if (nlev < 1) return RICH_ERR_INVALID;
    const bool mixed = pb->precision == RICH_MIXED;
    // index arithmetic uses 32-bit magic division: cell index * row length < 2^32
    if ((unsigned long long)pb->nx * pb->nz * pb->nx >= (1ull << 32)) return RICH_ERR_INVALID;
    P.S = S; P.nlev = nlev; P.mixed = mixed;
    size_t off = 0;
    int lx = pb->nx, lz = pb->nz;
    const size_t w = mixed ? 4 : 8;
    for (int l = 0; l < nlev; ++l) {
        P.nx[l] = lx; P.nz[l] = lz; P.mnx[l] = magic(lx); P.mhx[l] = magic(lx / 2);
        const size_t nc = (size_t)lx * lz;
        for (int k = 0; k < N64; ++k) {
            size_t bytes = (k == A_TBT || k == A_TBB) ? (size_t)lx * 8 : nc * 8;
            P.o64[l][k] = (long long)off; off = al256(off + bytes);
        }
        for (int k = 0; k < NMG; ++k) {
            // FP64: wE wW wN wS q f dp D ; FP32: Tx Tz - D q f dp - (slots B_2, B_7 unused)
            if (mixed && (k == B_2 || k == B_7)) { P.omg[l][k] = -1; continue; }
            P.omg[l][k] = (long long)off; off = al256(off + nc * w);
        }
        lx /= 2; lz /= 2;
    }
    const size_t nc8 = (size_t)pb->nx * pb->nz * 8;
    P.o_f64 = off; off = al256(off + nc8);
    if (mixed) { P.o_dp64 = off; off = al256(off + nc8); } else P.o_dp64 = -1;
    P.o_p = off; off = al256(off + nc8);
    P.o_thold = off; off = al256(off + nc8);
    P.o_Ks = off; off = al256(off + nc8);
    P.o_a = off; off = al256(off + nc8);
    P.o_K = off; off = al256(off + nc8);
    P.o_th = off; off = al256(off + nc8);
    P.closure = pb->closure;
    if (pb->closure == RICH_VAN_GENUCHTEN) {
        long long* cl[] = {&P.o_n, &P.o_m, &P.o_trc, &P.o_tsc};
        for (long long* o : cl) { *o = (long long)off; off = al256(off + nc8); }
    } else {
        P.o_n = P.o_m = P.o_trc = P.o_tsc = -1;
    }
    if (ckpt_every > 0) {
        const int nck = (pb->nsteps + ckpt_every - 1) / ckpt_every;
        P.ckpt_every = ckpt_every;
        P.keep_states = keep_states;
        P.o_ckpt = off; off = al256(off + (keep_states ? 0 : nc8 * std::max(nck, 1)));
        P.o_seg = off; off = al256(off + (keep_states ? 0 : nc8 * ckpt_every));
        long long* adj[] = {&P.o_lam, &P.o_rhs, &P.o_r, &P.o_dE, &P.o_dW, &P.o_dN, &P.o_dS, &P.o_dg, &P.o_g,
                            &P.o_rh, &P.o_pk, &P.o_v, &P.o_t, &P.o_ph, &P.o_sh};
        for (long long* o : adj) { *o = (long long)off; off = al256(off + nc8); }
        P.o_kry = (long long)off; off = al256(off + nc8 * (2 * ADJ_M + 1));
    }
    P.slot_bytes = (long long)off;
    P.nsteps = pb->nsteps; P.picard_maxit = pb->picard_maxit; P.mg_maxit = pb->mg_maxit;
    P.nu1 = pb->nu1; P.nu2 = pb->nu2; P.gamma = pb->cycle < 1 ? 1 : pb->cycle;
    P.inv_dt = 1.0 / pb->dt; P.tr = pb->theta_r; P.ts = pb->theta_s; P.p_top = pb->p_top;
    P.p_bot = pb->p_bottom; P.p_init = pb->p_init; P.picard_tol = pb->picard_tol; P.mg_tol = pb->mg_tol;
    P.h = 1.0 / pb->nz; P.two_over_h2 = 2.0 / (P.h * P.h);
    P.init_decay = pb->init_decay;
    return 0;
}

static size_t fused_smem(const FParams& P) { return (size_t)P.smem_bytes; }

// the fused kernel's instantiations live in one translation unit per (cycle
// precision, closure): fused_g64.cu, fused_g32.cu, fused_vg64.cu, fused_vg32.cu
static int fused_occupancy(const FParams& P, size_t smem, int nt, int* occ) {
    if (P.closure == RICH_VAN_GENUCHTEN)
        return P.mixed ? rich_occ_vg32(P, smem, nt, occ) : rich_occ_vg64(P, smem, nt, occ);
    return P.mixed ? rich_occ_g32(P, smem, nt, occ) : rich_occ_g64(P, smem, nt, occ);
}

static int fused_cluster(const FParams& P, size_t smem, int n, int clusters, cudaStream_t st, int* fit) {
    if (P.closure == RICH_VAN_GENUCHTEN)
        return P.mixed ? rich_cluster_vg32(P, smem, n, clusters, st, fit) : rich_cluster_vg64(P, smem, n, clusters, st, fit);
    return P.mixed ? rich_cluster_g32(P, smem, n, clusters, st, fit) : rich_cluster_g64(P, smem, n, clusters, st, fit);
}

static int fused_launch(const FParams& P, int grid, size_t smem, int nt, cudaStream_t st, int cluster = 0) {
    RICH_CUDA(cudaMemsetAsync(P.queue, 0, sizeof(int), st));
    rich_count_launch();
    if (cluster > 1) return fused_cluster(P, smem, cluster, grid, st, nullptr);
    if (P.closure == RICH_VAN_GENUCHTEN) {
        if (P.mixed) rich_launch_vg32(P, grid, smem, nt, st);
        else rich_launch_vg64(P, grid, smem, nt, st);
    } else if (P.mixed) {
        rich_launch_g32(P, grid, smem, nt, st);
    } else {
        rich_launch_g64(P, grid, smem, nt, st);
    }
    RICH_CUDA(cudaGetLastError());
    return 0;
}

// Threads per CTA when the caller has not chosen them (rich_set_tuning 0).  A
// CTA runs one sample: too many threads leave a small grid's levels with idle
// warps at every barrier and too few samples on an SM; too few leave a large
// grid's loads exposed.  Where the lines lie (ms of a batch on GB300, FP64
// Gardner unless stated, 32 / 128 / 256 / 512 / 1024 threads):
//   8^2   x 8192:  18 / 24 / 37 / 72 / 150       16^2 x 1216: 18 / 13 / 16 / 24 / 43
//   16^2  x 8192:  60 / 64 / 81 / 135 / 264      32^2 x 1:    28 / 11 / 9.3 / 9.3 / 9.7
//   32^2  x 4864:  193 / 141 / 151 / 211 / 345   32^2 x 608:  68 / 33 / 31 / 36 / 53
//   48x40 x 2048:  281 / 185 / 179 / 237 / 365   48x40 x 152: 201 / 93 / 77 / 74 / 74
//   64^2  x 1216:  - / 268 / 203 / 190 / 257     64^2 x 1:    - / 33 / 23 / 22 / 23
//   128^2 x 608:   - / 457 / 304 / 296 / 325     128^2 x 304: - / 293 / 193 / 166 / 144
//   256^2 x 152:   - / - / 610 / 409 / 350
// Mixed precision and the van Genuchten closure rank the shapes alike.
static int default_threads(long long nc, int S, int sms) {
    const long long per_sm = (S + sms - 1) / std::max(sms, 1);
    if (nc <= 64) return per_sm > 16 ? 32 : 128;
    if (nc <= 256) return 128;
    if (nc <= 1024) return per_sm > 16 ? 128 : 256;
    if (nc <= 2048) return per_sm > 8 ? 256 : 512;
    if (nc <= 8192) return 512;
    // one 1024-thread CTA per SM keeps more of a large grid in L2 and on chip;
    // two 512-thread CTAs overlap better once the batch fills the GPU twice
    return nc > 32768 || per_sm <= 2 ? 1024 : 512;
}

// Smallest level that a cluster runs on all its CTAs, and the smallest grid that
// takes a cluster.  ms without / with (CTAs a sample), levels from 64^2 or 128^2:
//   FP64:  64^2 x 1 146 / 104 (8), 64^2 x 48 314 / 265 (3), 128^2 x 24 220 / 102 (6;
//          110 from 128^2), 128^2 x 76 181 / 118 (2; 121)
//   mixed: 128^2 x 24 116 / 69 (6; 75 from 64^2), 128^2 x 76 100 / 71 (2; 80),
//          256^2 x 24 247 / 86 (6; 90)
// (how many clusters fit at a time depends on which SMs a GPU has in use: 48 samples took
// two CTAs each and 24 took five on another)
// An FP64 half-sweep of a 32^2 level is 1024 clocks of one SM's FP64 pipe, about
// what the barrier costs; FP32 cells are cheaper, so their line lies higher.  No
// finest grid between 32^2 and 64^2 (FP64) or 64^2 and 128^2 (mixed) was measured:
// such a grid takes no cluster.
constexpr long long CLUSTER_CELLS64 = 4096, CLUSTER_CELLS32 = 16384;

// CTAs of a sample's cluster (0: one CTA per sample), with the plan of shared
// memory made for it.  Only where the launch shape is free (rich_set_tuning 0),
// for V-cycles, and when clusters for all samples are resident together.
using cluster_fn = int (*)(const FParams&, size_t smem, int n, int clusters, cudaStream_t, int* fit);
static int pick_cluster(const rich_ctx* ctx, const rich_problem_t* pb, int S, FParams& P, cluster_fn call, int* cluster) {
    *cluster = 0;
    const long long cells = P.mixed ? CLUSTER_CELLS32 : CLUSTER_CELLS64;
    if (S < 1 || ctx->tune_threads || P.gamma > 1 || (long long)pb->nx * pb->nz < cells || 2ll * S > ctx->sm_count) return 0;
    plan_smem(P, 512, cells);
    if (P.lx == 0) return 0;
    for (int n = std::min(8, ctx->sm_count / S); n >= 2; --n) {
        int fit = 0;
        if (int e = call(P, fused_smem(P), n, S, nullptr, &fit)) return e;
        if (fit >= S) { *cluster = n; return 0; }
    }
    return 0;
}

// a device buffer of at least `bytes` (what it held is lost when it grows)
static int grow(void** buf, size_t* have, size_t bytes) {
    if (*have >= bytes) return 0;
    if (*buf) cudaFree(*buf);
    *buf = nullptr; *have = 0;
    if (cudaMalloc(buf, bytes) != cudaSuccess) { cudaGetLastError(); *buf = nullptr; return RICH_ERR_OOM; }
    *have = bytes;
    return 0;
}

// Fused persistent solve of S samples; stats arrays live in ctx->ws, the
// per-CTA slots and the queue counter in ctx->fused_scratch.
int rich_solve_fused(rich_ctx* ctx, const rich_problem_t* pb, int S, const double* lnKs,
                     const double* alpha, double alpha_scale, double* qoi, double* p_final,
                     int32_t* status, cudaStream_t st, const rich_soil_in* soil) {
    rich_samplebuf& w = ctx->sb;
    FParams P;
    if (pb->closure == RICH_VAN_GENUCHTEN && (!soil || !soil->n)) return RICH_ERR_INVALID;
    const int nt = (ctx->tune_threads == 1024 || ctx->tune_threads == 256 || ctx->tune_threads == 128 ||
                    ctx->tune_threads == 32 || ctx->tune_threads == 512)
                       ? ctx->tune_threads : default_threads((long long)pb->nx * pb->nz, S, ctx->sm_count);
    if (int e = fused_setup(pb, S, P)) return e;
    // a cluster of CTAs per sample where they all fit at once (grid: the clusters)
    int occ = 1, cluster = 0, grid = S;
    if (int e = pick_cluster(ctx, pb, S, P, fused_cluster, &cluster)) return e;
    if (cluster == 0) plan_smem(P, nt);
    if (soil) {
        P.n_in = soil->n; P.ts_in = soil->theta_s; P.tr_in = soil->theta_r;
        P.alpha_shift = soil->alpha_shift; P.n_shift = soil->n_shift;
    }
    const size_t off = (size_t)P.slot_bytes;
    const size_t smem = fused_smem(P);
    P.mixed_inner = ctx->tune_mixed_inner > 0 ? ctx->tune_mixed_inner : MIXED_INNER_DEFAULT;
    if (cluster == 0) {
        if (int e = fused_occupancy(P, smem, nt, &occ)) return e;
        grid = std::max(1, std::min(S, ctx->sm_count * occ));
    }
    // a slot for every CTA that the GPU holds at a time, fewer where memory is short:
    // the samples come from a queue, so fewer CTAs only take longer
    while (int e = grow(&ctx->fused_scratch, &ctx->fused_bytes, (size_t)grid * off + 256)) {
        if (cluster || grid <= ctx->sm_count) return e;
        grid = std::max(ctx->sm_count, grid / 2);
    }
    P.scratch = (char*)ctx->fused_scratch + 256;
    P.queue = (int*)ctx->fused_scratch;
    P.lnKs = lnKs; P.alpha = alpha; P.alpha_scale = alpha_scale;
    P.qoi = qoi; P.p_final = p_final; P.status = w.status;
    P.pic_total = w.pic_total; P.mg_total = w.mg_total; P.maxpic = w.maxpic; P.t_ns = w.t_ns;
    // CTAs that share an SM during the solve: a grid smaller than the GPU's
    // resident capacity is spread over the SMs first
    w.last_occ = std::max(1, std::min(occ, (grid + ctx->sm_count - 1) / std::max(ctx->sm_count, 1)));
    rich_prof_begin(ctx, st);
    if (int e = fused_launch(P, grid, smem, nt, st, cluster)) return e;
    rich_prof_end(ctx, st, 0.0, 0.0);
    w.last = S;
    if (status)
        RICH_CUDA(cudaMemcpyAsync(status, w.status, sizeof(int32_t) * S, cudaMemcpyDeviceToDevice, st));
    return 0;
}

// Discrete adjoint of S samples: QoI and dQ/d ln Ks [S][nz][nx] (g_out).
int rich_adjoint_fused(rich_ctx* ctx, const rich_problem_t* pb, int S, const double* lnKs,
                       const double* alpha, double alpha_scale, int ckpt_every, double adj_tol,
                       int adj_maxit, int adj_method, double* qoi, double* g_out, cudaStream_t st) {
    rich_samplebuf& w = ctx->sb;
    FParams P;
    if (ckpt_every < 1 || pb->closure != RICH_GARDNER) return RICH_ERR_INVALID;
    size_t smem = 0;
    int grid = 0, cluster = 0;
    // the states of all steps where the context's limit and the device's memory
    // allow them, else the checkpointed layout
    for (bool keep : {true, false}) {
        if (int e = fused_setup(pb, S, P, ckpt_every, keep)) return e;
        // (the GMRES option keeps its small system in one CTA)
        cluster = 0;
        if (adj_method != 2)
            if (int e = pick_cluster(ctx, pb, S, P, P.mixed ? rich_adjoint_cluster32 : rich_adjoint_cluster64, &cluster))
                return e;
        if (cluster == 0) plan_smem(P, 512);
        smem = fused_smem(P);
        int occ = 0;
        const void* kern = P.mixed ? rich_adjoint_kernel32(P.gamma > 1) : rich_adjoint_kernel64(P.gamma > 1);
        if (int e = allow_dyn_smem(kern, smem)) return e;
        RICH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 512, smem));
        occ = std::max(occ, 1);
        grid = cluster ? S : std::max(1, std::min(S, ctx->sm_count * occ));
        const size_t states = keep ? (size_t)grid * std::max(pb->nsteps, 1) * pb->nx * pb->nz * 8 : 0;
        if (states > ctx->adj_memory) continue;
        const int e1 = grow(&ctx->fused_scratch, &ctx->fused_bytes, (size_t)grid * (size_t)P.slot_bytes + 256);
        const int e2 = e1 ? e1 : grow(&ctx->adj_states, &ctx->adj_states_bytes, states);
        if (e2 == 0) break;
        if (!keep) return e2;
    }
    P.states = (double*)ctx->adj_states;
    P.adj_tol = adj_tol; P.adj_maxit = adj_maxit; P.adj_inner = pb->precision == RICH_MIXED ? 2 : 1;
    P.adj_method = adj_method;
    P.mixed_inner = ctx->tune_mixed_inner > 0 ? ctx->tune_mixed_inner : MIXED_INNER_DEFAULT;
    P.scratch = (char*)ctx->fused_scratch + 256;
    P.queue = (int*)ctx->fused_scratch;
    P.lnKs = lnKs; P.alpha = alpha; P.alpha_scale = alpha_scale;
    P.qoi = qoi; P.p_final = nullptr; P.status = w.status; P.g_out = g_out;
    P.pic_total = w.pic_total; P.mg_total = w.mg_total; P.maxpic = w.maxpic;
    RICH_CUDA(cudaMemsetAsync(P.queue, 0, sizeof(int), st));
    rich_count_launch();
    rich_prof_begin(ctx, st);
    if (cluster) {
        const auto call = P.mixed ? rich_adjoint_cluster32 : rich_adjoint_cluster64;
        if (int e = call(P, smem, cluster, grid, st, nullptr)) return e;
    } else if (P.mixed) rich_adjoint_launch32(P, grid, smem, st);
    else rich_adjoint_launch64(P, grid, smem, st);
    rich_prof_end(ctx, st, 0.0, 0.0);
    RICH_CUDA(cudaGetLastError());
    return 0;
}

// ---------------------------------------------------------------------------
// Allocation-free variant.  Its scratch (queue counter + per-CTA slots) is a
// file-scope device array of RICH_NOALLOC_SCRATCH_BYTES, created when the
// library is loaded and held by every GPU that loads it until the process
// exits.  Host code may not use the array's name as a device address (on the
// host it names a shadow object), so the address is looked up once per device
// with cudaGetSymbolAddress and cached; the look-up runs under a mutex, so
// first calls from several host threads resolve it once.  The cached address
// belongs to the device's primary context: after cudaDeviceReset on that
// device the array is gone and this entry point must not be called again in
// the process.
// ---------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_noalloc_scratch[RICH_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr int NOALLOC_MAX_DEVICES = 64;
void* g_noalloc_addr[NOALLOC_MAX_DEVICES];
int g_noalloc_sms[NOALLOC_MAX_DEVICES];
std::mutex g_noalloc_mu;
}

extern "C" int rich_solve_batch_noalloc(const rich_problem_t* pb, int32_t nsamples,
                                        const double* lnKs, const double* alpha, double alpha_scale,
                                        double* qoi, int32_t* status, void* stream) {
    if (rich_check_problem(pb) || nsamples < 0) {
        rich_set_error("invalid problem or sample count", __FILE__, __LINE__);
        return RICH_ERR_INVALID;
    }
    if (pb->closure != RICH_GARDNER) {
        rich_set_error("the allocation-free entry point takes the Gardner closure only", __FILE__, __LINE__);
        return RICH_ERR_INVALID;
    }
    if (nsamples == 0) return 0;
    if (!lnKs || !alpha || !qoi) {
        rich_set_error("lnKs, alpha and qoi are required", __FILE__, __LINE__);
        return RICH_ERR_INVALID;
    }
    int dev = -1;
    RICH_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
        rich_set_error("device index beyond the allocation-free table", __FILE__, __LINE__);
        return RICH_ERR_INVALID;
    }
    char* base = nullptr;
    int dev_sms = 0;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {      // first call on this device: resolve the symbol
            void* ptr = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
            if (e != cudaSuccess || !ptr) {
                cudaGetLastError();
                rich_set_error(e != cudaSuccess ? cudaGetErrorString(e) : "null symbol address", __FILE__,
                               __LINE__);
                return RICH_ERR_CUDA;
            }
            int sms = 0;
            RICH_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
            g_noalloc_sms[dev] = sms;
            g_noalloc_addr[dev] = ptr;
        }
        base = (char*)g_noalloc_addr[dev];
        dev_sms = g_noalloc_sms[dev];
    }
    FParams P;
    if (int e = fused_setup(pb, nsamples, P)) {
        rich_set_error("unsupported grid", __FILE__, __LINE__);
        return e;
    }
    plan_smem(P, 512);
    const size_t slot = (size_t)P.slot_bytes;
    const size_t slots = (RICH_NOALLOC_SCRATCH_BYTES - 256) / slot;
    if (slots < 1) {
        rich_set_error("grid needs more scratch per CTA than the allocation-free entry point holds "
                       "(RICH_NOALLOC_SCRATCH_BYTES)", __FILE__, __LINE__);
        return RICH_ERR_INVALID;
    }
    const size_t smem = fused_smem(P);
    P.mixed_inner = MIXED_INNER_DEFAULT;
    int occ = 0;
    if (int e = fused_occupancy(P, smem, 512, &occ)) return e;
    const int grid = (int)std::min<long long>({(long long)nsamples, (long long)dev_sms * occ, (long long)slots});
    P.queue = (int*)base;                 // cleared by fused_launch before the kernel
    P.scratch = base + 256;
    P.lnKs = lnKs; P.alpha = alpha; P.alpha_scale = alpha_scale;
    P.qoi = qoi; P.p_final = nullptr; P.status = status;
    P.pic_total = nullptr; P.mg_total = nullptr; P.maxpic = nullptr;
    return fused_launch(P, grid, smem, 512, (cudaStream_t)stream);
}
