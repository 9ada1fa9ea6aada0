// Device side of the discrete adjoint (kernel template), shared by the
// translation units that instantiate it; the Cta methods it calls (Jacobian
// pieces, J^T products and solvers, gradient update) live with the forward
// solver in fused_kernel.cuh.
#pragma once
#include "fused_kernel.cuh"

namespace {

// Discrete adjoint of the converged time-stepped solve (one sample per CTA):
// forward with a checkpoint of p every ckpt_every steps, then per segment
// (last first) recompute its states from the checkpoint and step backwards.
// With keep_states the forward sweep keeps every step's p instead (one segment, in
// a buffer of its own) and nothing is recomputed: the second forward solve was
// nearly half of the call (64^2 x 48 samples x 6 steps: 281 -> 147 ms).  Same bits.
//   J_N^T lam_N = dQ/dp^N,  J_n^T lam_n = diag(C(p^n)/dt) lam_{n+1},
//   dQ/dm = dQ/dm|explicit - sum_n (dR_n/dm)^T lam_n     (m = ln Ks).
// one sample's forward and reverse sweep on its group of threads, in slot k
template <typename Gr, typename C_t>
__device__ __forceinline__ void adjoint_sample(C_t& C, const FParams& P, int k, int s) {
    char* slot = P.scratch + (size_t)k * P.slot_bytes;
    const int nc = C.nc, nx = C.nx, tid = C.tid, nt = C.nt;
    const bool keep = P.keep_states != 0;
    const int CK = keep ? max(P.nsteps, 1) : P.ckpt_every;
    double* ckpt = (double*)(slot + P.o_ckpt);      // [nck][nc]
    double* seg = keep ? P.states + (size_t)k * CK * nc : (double*)(slot + P.o_seg);      // [CK][nc]
    double* lam = (double*)(slot + P.o_lam);
    double* rhs = (double*)(slot + P.o_rhs);
    double* r = (double*)(slot + P.o_r);
    double* dE = (double*)(slot + P.o_dE);
    double* dW = (double*)(slot + P.o_dW);
    double* dN = (double*)(slot + P.o_dN);
    double* dS = (double*)(slot + P.o_dS);
    double* dg = (double*)(slot + P.o_dg);
    double* g = (double*)(slot + P.o_g);
    const double NaN = __longlong_as_double(0x7FF8000000000000ll);
    C.setup(s);
    int status = RICH_OK, maxpic = 0;
    bool alive = true;
    long long pic_tot = 0, mg_tot = 0, adj_its = 0;
    // ---- forward with checkpoints p^0, p^CK, p^2CK, ...
    for (int n = 1; n <= P.nsteps && alive; ++n) {
        if (!keep && (n - 1) % CK == 0) {
            double* dst = ckpt + (size_t)((n - 1) / CK) * nc;
            for (int q = tid; q < nc; q += nt) dst[q] = C.p[q];
            Gr::sync();
        }
        alive = C.time_step(pic_tot, mg_tot, maxpic, status);
        if (keep) {
            double* dst = seg + (size_t)(n - 1) * nc;
            for (int q = tid; q < nc; q += nt) dst[q] = C.p[q];
            Gr::sync();
        }
    }
    double qv = 0.0;
    if (tid < 32) qv = C.qoi_warp0();
    if (alive) {
        // ---- dQ/dp^N (rhs) and the explicit dQ/dm (g), bottom cells
        for (int q = tid; q < nc; q += nt) {
            double gv = 0.0, rv = 0.0;
            if (q < nx) {
                double kb = P.p_bot < 0.0 ? C.Ks[q] * exp(C.aa[q] * P.p_bot) : C.Ks[q];
                rv = kb * (2.0 / C.h) / nx;
                gv = kb * (2.0 * (C.p[q] - P.p_bot) / C.h + 1.0) / nx;
            }
            rhs[q] = rv;
            g[q] = gv;
        }
        Gr::sync();
        const int nck = (P.nsteps + CK - 1) / CK;
        for (int sg = nck - 1; sg >= 0 && alive; --sg) {
            const int n0 = sg * CK, n1 = min(n0 + CK, P.nsteps);
            // recompute p^{n0+1..n1} from the checkpoint
            if (!keep) {
                for (int q = tid; q < nc; q += nt) C.p[q] = ckpt[(size_t)sg * nc + q];
                Gr::sync();
            }
            long long dpic = 0, dmg = 0;
            int dmax = 0, dst = RICH_OK;
            for (int n = n0 + 1; n <= n1 && alive && !keep; ++n) {
                alive = C.time_step(dpic, dmg, dmax, dst);
                double* dstp = seg + (size_t)(n - n0 - 1) * nc;
                for (int q = tid; q < nc; q += nt) dstp[q] = C.p[q];
                Gr::sync();
            }
            if (!alive) { status = dst; break; }
            for (int n = n1; n > n0; --n) {
                // state p^n, operator and Jacobian at p^n
                const double* pn = seg + (size_t)(n - n0 - 1) * nc;
                for (int q = tid; q < nc; q += nt) C.p[q] = pn[q];
                Gr::sync();
                C.assemble();
                if (n < P.nsteps) {       // rhs = diag(C(p^n)/dt) lam_{n+1}
                    for (int q = tid; q < nc; q += nt) rhs[q] = C.L64[0].Cdt[q] * lam[q];
                    Gr::sync();
                }
                C.adj_prepare(dE, dW, dN, dS, dg);
                int its;
                if (P.adj_method == 1)
                    its = C.adj_solve_bicgstab(dE, dW, dN, dS, dg, rhs, lam, r, (double*)(slot + P.o_rh),
                                               (double*)(slot + P.o_pk), (double*)(slot + P.o_v),
                                               (double*)(slot + P.o_t), (double*)(slot + P.o_ph),
                                               (double*)(slot + P.o_sh));
                else if (C_t::CLU || P.adj_method == 0)
                    its = C.adj_solve(dE, dW, dN, dS, dg, rhs, lam, r);
                else if constexpr (!C_t::CLU)
                    its = C.adj_solve_gmres(dE, dW, dN, dS, dg, rhs, lam, (double*)(slot + P.o_kry));
                adj_its += its;
                // status is OK or MG_MAXIT here (the sample is alive);
                // a J^T solve stopped at its cap outranks both
                if (its > P.adj_maxit) status = RICH_ADJ_MAXIT;
                C.adj_grad_update(lam, g);
            }
        }
    }
    if (tid == 0) {
        P.qoi[s] = alive ? qv : NaN;
        if (P.status) P.status[s] = status;
        if (P.pic_total) P.pic_total[s] = pic_tot;
        if (P.mg_total) P.mg_total[s] = adj_its;
        if (P.maxpic) P.maxpic[s] = maxpic;
    }
    for (int q = tid; q < nc; q += nt) P.g_out[(size_t)s * nc + q] = alive ? g[q] : NaN;
}

template <typename TM, bool WC>
__global__ void __maxnreg__(128)
k_adjoint(const FParams P) {
    extern __shared__ unsigned char smraw[];
    __shared__ unsigned long long red[33];
    __shared__ int s_sample;
    __shared__ Lv64 L64[MAXL];
    __shared__ Lv<TM> LM[MAXL];
    char* slot = P.scratch + (size_t)blockIdx.x * P.slot_bytes;
    init_levels<TM>(P, slot, smraw, L64, LM);
    Cta<TM, WC> C(P, slot, L64, LM, reinterpret_cast<TM*>(smraw), red);
    for (;;) {
        if (threadIdx.x == 0) s_sample = atomicAdd(P.queue, 1);
        __syncthreads();
        const int s = s_sample;
        __syncthreads();
        if (s >= P.S) break;
        adjoint_sample<GCta>(C, P, blockIdx.x, s);
        __syncthreads();
    }
}

// the same with a cluster of CTAs per sample (see k_fused_cluster): 48 samples of
// 64^2 on three SMs each, 6 steps, 124 -> 111 ms
template <typename TM>
__global__ void __launch_bounds__(CLUSTER_THREADS, 1)
k_adjoint_cluster(const FParams P) {
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
    Cta<TM, false, 0, GClu> C(P, slot, L64, LM, reinterpret_cast<TM*>(smraw), red);
    C.cred = cred;
    c.sync();
    for (;;) {
        if (C.tid == 0) {
            const int s = atomicAdd(P.queue, 1);
            for (int k = 0; k < n; ++k) *c.map_shared_rank(&s_sample, k) = s;
        }
        c.sync();
        const int s = s_sample;
        if (s >= P.S) break;
        adjoint_sample<GClu>(C, P, blockIdx.x / n, s);
        c.sync();
    }
}

}  // namespace
