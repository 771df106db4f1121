// P_tilde of Eq. (AppPrec) in storage precisions SP (Theta_tilde's GMRES basis
// and the S_tilde recurrence) and SI (Rana's sweep, V-cycles, coarse stencils).
// Arithmetic is double when SP is double, else float.
//
// apply(r):   z_V = Theta_tilde^{-1} r_V, all nt time blocks batched (inner
//             GMRES, right-preconditioned by P_int);
//             g_{n+1} = r_{v,n+1} + tau sum_i b_i z_{V,n,i}; w = M^{-1} g (FD: w = g);
//             z_{v,0} = w_0, z_{v,n+1} = w_{n+1} + z_{v,n} - tau (b^T (x) I)
//             Theta_tilde^{-1} (e (x) K z_{v,n})    (forward substitution, Eq. AppSchur).
// apply_T(r): u_nt = r_{v,nt}, u_n = r_{v,n} + u_{n+1} - tau (e^T (x) K)
//             Theta_tilde^{-T} (b (x) u_{n+1}); z_v = M^{-1} u;
//             z_V = Theta_tilde^{-T} (r_V + tau (b (x) M) z_{v,n+1}).
#pragma once

#include <algorithm>
#include <cstring>
#include <memory>
#include <type_traits>

#include "arnoldi.cuh"
#include "cluster_mg.cuh"
#include "handle.cuh"
#include "mg.cuh"

namespace aao {

template <class SP, class SI>
class Precond : public PrecondBase {
    using A = typename PT<SP>::A;
    static_assert(std::is_same<typename PT<SP>::A, typename PT<SI>::A>::value,
                  "P and P_int arithmetic must agree");

    struct Level {
        Geo g;
        // per-stage stored stencils (levels >= 1)
        SI* sten[kMaxS] = {};
        float* sten_sc[kMaxS] = {};
        // scratch, Bmax items of nx each
        Vec<SI> T0, T1, Rr, Bb, X;
    };

    Handle* h;
    Arena ar;
    int Bmax = 0;
    int L = 0;
    Level lev[kMaxLevels];
    A* Dinv[kMaxS] = {};           // dense coarsest inverse per stage
    A* jacw[kClMaxLevels][kMaxS] = {};   // 2D: Jacobi weights omega / a_PP of the distributed levels
    Faces<A> facesA;
    SpaceOp<A> sopA;                 // fine-grid K (and M for Q1) for the stage kernels
    A* cheb[3] = {};                 // Q1: Chebyshev x, r, d ((nt+1)*nx each)
    int kin = 0;                   // inner maxit
    double itol = 0.0;
    // inner GMRES state
    Vec<SP> V0;                    // (kin+1) bases, stride vstride elements
    long long vstride = 0;
    Vec<SI> Z0;                    // kin bases, stride zstride
    long long zstride = 0;
    A* wv = nullptr;               // Bmax * s*nx
    Vec<SI> mgb;                   // Rana rhs, Bmax * nx
    double *Hh = nullptr, *csh = nullptr, *snh = nullptr, *gh = nullptr, *yh = nullptr, *betah = nullptr;
    int *activeh = nullptr, *itsh = nullptr, *nonfin = nullptr, *brk = nullptr;
    long long* itcount = nullptr;  // running total of inner iterations (device)
    double* gramh = nullptr;       // products of the basis vectors, kin*kin per item
    double* ar_part = nullptr;     // partial sums of the Arnoldi kernels
    unsigned int* ar_count = nullptr;   // their arrival counters, Bmax, zero between launches
    // Schur state
    A* wbuf = nullptr;             // (nt+1)*nx
    A* tbuf = nullptr;             // s*nx
    A* qbuf = nullptr;             // s*nx
    A* tV = nullptr;               // nt*s*nx (transposed apply)
    double* tmp64 = nullptr;       // Bmax*s*nx staging for component entry points
    cudaEvent_t e0, e1, e2;
    int nact = 0;                  // active items of the current batch (exact only while profiling)
    // Fused on-chip tail: two variants, for single-item V-cycles (the Schur
    // sweep, where a smaller tail plus fused level kernels is faster) and for
    // batched V-cycles (every item's tail on its own SM).
    struct Tail {
        int lc = 0;                // first level handled by the tail kernel
        size_t smem = 0;
        TailCtx<SI> ctx[kMaxS];
    };
    Tail tails[2];                 // [0]: B == 1, [1]: B > 1
    int tail_threads = 1024;
    // Cluster-resident shifted solves for single 2D items (the Schur sweep).
    int cl_C = 0;                  // CTAs per cluster of the single-item plan; 0: no cluster plan
    struct ClPlan {
        int C = 0;                 // CTAs per cluster; 0: none
        int resident = 0;          // clusters on the device at once
        size_t smem = 0;
        void (*kernel)(const ClCtx<SI>, const int*, Vec<SI>, Vec<SI>) = nullptr;
        ClCtx<SI> ctx[kMaxS];      // one context per stage, passed by value
    };
    static constexpr int kClPlans = 4;
    ClPlan clp[kClPlans];          // [0] single items (16 or 8 CTAs), then batches: 8, 4 and 2 CTAs
    int* hact = nullptr;           // pinned mirror of activeh (profiling)

    cudaStream_t cur_stream = nullptr;     // stream of the next launch (capture stream while capturing)
    cudaStream_t cap_stream = nullptr;
    // one captured graph per step kind [transpose][kind]: 0 one time step, 1 a batched MGRIT
    // relaxation step, 2 the batched C-point residual step, 3 a batched relaxation step that also
    // relaxes the shorter final interval (mg_r > 0)
    cudaGraphExec_t gexec[2][4] = {};
    long long graph_nodes[2][4] = {};
    StepPtrs* stepp = nullptr;
    // two-level MGRIT for S_tilde's recurrence (mg_m = 0: forward substitution): the coarse
    // propagator is the substitution step of a second preconditioner built for step size
    // mg_m tau and mg_nc = nt / mg_m (rounded down) steps; C-points are the multiples of mg_m, and
    // the mg_r = nt - mg_nc mg_m steps after the last one form a shorter final interval
    int mg_m = 0, mg_nc = 0, mg_r = 0;
    std::unique_ptr<Handle> hc;
    Precond* coarse = nullptr;
    double* ebuf = nullptr;        // (nc+1)*nx: coarse error recurrence
    double* rbufT = nullptr;       // (nc+1)*nx: transposed C-point residuals (the coarse source)
    // The intervals' recurrences run as single-item steps on worker preconditioners (same
    // operators, one stream each, their own Krylov and reduction workspace; they read this
    // preconditioner's w), ordered by events: the dataflow of one two-level MGRIT iteration.
    static constexpr int kMaxWorkers = 16;
    int nwork = 0;
    std::unique_ptr<Handle> hw[kMaxWorkers];
    Precond* work[kMaxWorkers] = {};
    cudaStream_t wst[kMaxWorkers] = {};
    cudaEvent_t ev_start = nullptr, ev_join[kMaxWorkers] = {};
    std::vector<cudaEvent_t> ev_f1, ev_c;    // per interval: first relaxation done, C-point corrected
    const A* wsrc = nullptr;       // a worker's source w (the owner's wbuf); nullptr: its own

    cudaStream_t st() const { return cur_stream; }

    // While a launch profile is open, read back how many batch items are still
    // active so the byte hints count only the work that is done.
    void refresh_nact(int B) {
        nact = B;
        if (!g_prof_on || !hact) return;
        cudaMemcpyAsync(hact, activeh, sizeof(int) * B, cudaMemcpyDeviceToHost, st());
        cudaStreamSynchronize(st());
        int c = 0;
        for (int b = 0; b < B; ++b) c += hact[b] != 0;
        nact = c;
    }

    template <class S> aao_status alloc_vec(Vec<S>& v, long long items, long long item_len, int n0) {
        AAO_TRY(ar.alloc(&v.d, (size_t)(items * item_len)));
        v.bs = item_len;
        v.sc = nullptr;
        if (PT<S>::scaled) AAO_TRY(ar.alloc(&v.sc, (size_t)(items * item_len / n0)));
        return AAO_OK;
    }

  public:
    explicit Precond(Handle* hh) : h(hh), cur_stream(hh->stream) {}
    ~Precond() override { release(); }

    void release() override {
        if (coarse) delete coarse;
        coarse = nullptr;
        hc.reset();
        for (int w = 0; w < kMaxWorkers; ++w) {
            if (work[w]) delete work[w];
            work[w] = nullptr;
            hw[w].reset();
            if (wst[w]) cudaStreamDestroy(wst[w]);
            wst[w] = nullptr;
            if (ev_join[w]) cudaEventDestroy(ev_join[w]);
            ev_join[w] = nullptr;
        }
        nwork = 0;
        for (cudaEvent_t e : ev_f1) cudaEventDestroy(e);
        for (cudaEvent_t e : ev_c) cudaEventDestroy(e);
        ev_f1.clear();
        ev_c.clear();
        if (ev_start) cudaEventDestroy(ev_start);
        ev_start = nullptr;
        for (int i = 0; i < 2; ++i)
            for (int k = 0; k < 4; ++k) {
                if (gexec[i][k]) cudaGraphExecDestroy(gexec[i][k]);
                gexec[i][k] = nullptr;
            }
        if (cap_stream) cudaStreamDestroy(cap_stream);
        cap_stream = nullptr;
        ar.release();
        if (hact) cudaFreeHost(hact);
        hact = nullptr;
    }

    aao_status setup() override {
        const Geo& g0 = h->g;
        const int s = h->s;
        if (PT<SI>::scaled || PT<SP>::scaled) {
            if (g0.n0 > kMaxRowLen) {
                set_error("16-bit storage needs n[0] <= 512");
                return AAO_ERR_ARG;
            }
        }
        Bmax = h->nt;
        kin = h->opt.inner_maxit;
        itol = h->opt.inner_tol;
        // ---- levels
        L = 0;
        Geo g = g0;
        while (true) {
            lev[L].g = g;
            ++L;
            bool more = g.nx > kCoarsestTarget && g.n0 / 2 >= 2 && g.n1 / 2 >= 2 && (g.d == 2 || g.n2 / 2 >= 2);
            if (!more || L == kMaxLevels) break;
            Geo c = g;
            c.n0 = g.n0 / 2;
            c.n1 = g.n1 / 2;
            c.n2 = g.d == 3 ? g.n2 / 2 : 1;
            c.nx = (long long)c.n0 * c.n1 * c.n2;
            c.R = c.n1 * c.n2;
            g = c;
        }
        if (lev[L - 1].g.nx > kMaxCoarsest) {
            set_error("coarsest multigrid level too large (anisotropic grid?)");
            return AAO_ERR_ARG;
        }
        // ---- faces in arithmetic precision
        if (h->has_kappa) {
            long long nfx = (long long)(g0.n0 + 1) * g0.R;
            long long nfy = (long long)g0.n0 * (g0.n1 + 1) * g0.n2;
            long long nfz = g0.d == 3 ? (long long)g0.nx / g0.n2 * (g0.n2 + 1) : 0;
            A *fx, *fy, *fz = nullptr;
            AAO_TRY(ar.alloc(&fx, nfx));
            AAO_TRY(ar.alloc(&fy, nfy));
            if (nfz) AAO_TRY(ar.alloc(&fz, nfz));
            launch(k_convert<double, A>, (unsigned)((nfx + 255) / 256), 256, 0, st(), h->faces64.fx, fx, nfx);
            launch(k_convert<double, A>, (unsigned)((nfy + 255) / 256), 256, 0, st(), h->faces64.fy, fy, nfy);
            if (nfz) launch(k_convert<double, A>, (unsigned)((nfz + 255) / 256), 256, 0, st(), h->faces64.fz, fz, nfz);
            AAO_LAUNCH_CHECK();
            facesA.fx = fx;
            facesA.fy = fy;
            facesA.fz = fz;
        }
        sopA.faces = facesA;
        sopA.q1 = h->q1;
        if (h->q1) {
            for (int a = 0; a < 3; ++a)
                for (int e = 0; e < 3; ++e) {
                    sopA.q.m[a][e] = (A)h->q1d.m[a][e];
                    sopA.q.k[a][e] = (A)h->q1d.k[a][e];
                }
        }
        // ---- Galerkin hierarchy per stage shift c_i = tau d_i
        const int ncoef = g0.d == 3 ? 27 : 9;
        double* sten0 = nullptr;             // Q1: stored fine-level stencil of M + c K (FP64)
        if (h->q1) AAO_TRY(ar.alloc(&sten0, (size_t)(ncoef * g0.nx)));
        double* sten64[kMaxLevels] = {};
        for (int l = 1; l < L; ++l) AAO_TRY(ar.alloc(&sten64[l], (size_t)(ncoef * lev[l].g.nx)));
        const Geo& gcst = lev[L - 1].g;
        const int ncst = (int)gcst.nx;
        double *dense, *dinv64;
        int* fail;
        const long long nn = (long long)ncst * ncst;
        AAO_TRY(ar.alloc(&dense, (size_t)(s * nn)));
        AAO_TRY(ar.alloc(&dinv64, (size_t)(s * nn)));
        AAO_TRY(ar.alloc(&fail, 1));
        AAO_CUDA_TRY(cudaMemsetAsync(fail, 0, sizeof(int), st()));
        for (int i = 0; i < s; ++i) {
            FineDesc fd;
            fd.g = g0;
            fd.fine = 1;
            fd.sigma = 1.0;
            fd.c = h->tau * h->D[i];
            fd.faces = h->faces64;
            fd.sten = nullptr;
            if (h->q1) {
                launch(k_q1_stencil, (unsigned)((g0.nx + 127) / 128), 128, 0, st(), g0, h->q1d, h->tau * h->D[i],
                       sten0);
                AAO_LAUNCH_CHECK();
                AAO_TRY(store_stencil(0, i, sten0, ncoef));
                fd.fine = 0;
                fd.sigma = 0.0;
                fd.c = 0.0;
                fd.sten = sten0;
            }
            for (int l = 1; l < L; ++l) {
                launch(k_galerkin, (unsigned)((lev[l].g.nx + 127) / 128), 128, 0, st(), fd, lev[l].g, sten64[l]);
                AAO_LAUNCH_CHECK();
                AAO_TRY(store_stencil(l, i, sten64[l], ncoef));
                FineDesc nd;
                nd.g = lev[l].g;
                nd.fine = 0;
                nd.sigma = 0;
                nd.c = 0;
                nd.sten = sten64[l];
                fd = nd;   // level l+1 is the Galerkin product of this level
            }
            // coarsest dense inverse from the FP64 description of level L-1
            FineDesc cd;
            if (L == 1) {
                cd.g = g0;
                cd.fine = h->q1 ? 0 : 1;
                cd.sigma = h->q1 ? 0.0 : 1.0;
                cd.c = h->q1 ? 0.0 : h->tau * h->D[i];
                cd.faces = h->faces64;
                cd.sten = h->q1 ? sten0 : nullptr;
            } else {
                cd.g = gcst;
                cd.fine = 0;
                cd.sigma = 0;
                cd.c = 0;
                cd.sten = sten64[L - 1];
            }
            launch(k_dense_level, (unsigned)((ncst + 127) / 128), 128, 0, st(), cd, dense + i * nn);
            AAO_LAUNCH_CHECK();
        }
        // the stages' coarsest inverses in one launch, a cluster each
        AAO_TRY(launch_gauss_jordan(dense, dinv64, ncst, s, fail, st()));
        for (int i = 0; i < s; ++i) {
            AAO_TRY(ar.alloc(&Dinv[i], (size_t)nn));
            launch(k_convert_dense<A>, (unsigned)((nn + 255) / 256), 256, 0, st(), (const double*)(dinv64 + i * nn),
                   Dinv[i], nn);
            AAO_LAUNCH_CHECK();
        }
        int hfail = 0;
        AAO_CUDA_TRY(cudaMemcpyAsync(&hfail, fail, sizeof(int), cudaMemcpyDeviceToHost, st()));
        AAO_CUDA_TRY(cudaStreamSynchronize(st()));
        if (hfail) {
            set_error("coarsest multigrid operator is not positive definite");
            return AAO_ERR_BREAKDOWN;
        }
        // ---- fused tails: the coarsest levels that fit on one SM
        int optin = 0;
        {
            int dev = 0;
            AAO_CUDA_TRY(cudaGetDevice(&dev));
            AAO_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        }
        for (int v = 0; v < 2; ++v) AAO_TRY(build_tail(tails[v], v == 0 ? kTailMaxPointsSingle : kTailMaxPoints, optin));
        // the attribute is per kernel for the whole process: always set the device's
        // opt-in maximum so that handles with larger tails keep working
        AAO_CUDA_TRY(cudaFuncSetAttribute(k_vcycle_tail<SI>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
        AAO_CUDA_TRY(cudaFuncSetAttribute(k_vcycle_tail_2d<SI>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
        AAO_TRY(build_cluster(optin));
        // ---- level scratch
        for (int l = 0; l < L; ++l) {
            const Geo& gl = lev[l].g;
            AAO_TRY(alloc_vec(lev[l].T0, Bmax, gl.nx, gl.n0));
            AAO_TRY(alloc_vec(lev[l].T1, Bmax, gl.nx, gl.n0));
            AAO_TRY(alloc_vec(lev[l].Rr, Bmax, gl.nx, gl.n0));
            if (l > 0) {
                AAO_TRY(alloc_vec(lev[l].Bb, Bmax, gl.nx, gl.n0));
                AAO_TRY(alloc_vec(lev[l].X, Bmax, gl.nx, gl.n0));
            }
        }
        // ---- inner GMRES state
        const long long item = (long long)s * g0.nx;
        vstride = (long long)Bmax * item;
        zstride = vstride;
        AAO_TRY(alloc_vec(V0, (long long)(kin + 1) * Bmax, item, g0.n0));
        V0.bs = item;
        AAO_TRY(alloc_vec(Z0, (long long)kin * Bmax, item, g0.n0));
        Z0.bs = item;
        AAO_TRY(ar.alloc(&wv, (size_t)(Bmax * item)));
        AAO_TRY(alloc_vec(mgb, Bmax, g0.nx, g0.n0));
        AAO_TRY(ar.alloc(&Hh, (size_t)Bmax * (kin + 1) * kin));
        AAO_TRY(ar.alloc(&csh, (size_t)Bmax * kin));
        AAO_TRY(ar.alloc(&snh, (size_t)Bmax * kin));
        AAO_TRY(ar.alloc(&gh, (size_t)Bmax * (kin + 1)));
        AAO_TRY(ar.alloc(&yh, (size_t)Bmax * kin));
        AAO_TRY(ar.alloc(&betah, (size_t)Bmax));
        AAO_TRY(ar.alloc(&gramh, (size_t)Bmax * kin * kin));
        AAO_TRY(ar.alloc(&ar_part, (size_t)(kArBlocks + Bmax) * (2 * (kin <= kArSmallK ? kArSmallK : kMaxInner) - 1)));
        AAO_TRY(ar.alloc(&ar_count, (size_t)Bmax));
        AAO_CUDA_TRY(cudaMemsetAsync(ar_count, 0, sizeof(unsigned int) * Bmax, st()));
        AAO_TRY(ar.alloc(&activeh, (size_t)Bmax));
        AAO_TRY(ar.alloc(&itsh, (size_t)Bmax));
        AAO_TRY(ar.alloc(&nonfin, 2));
        brk = nonfin + 1;
        AAO_TRY(ar.alloc(&itcount, 1));
        AAO_CUDA_TRY(cudaMemsetAsync(nonfin, 0, 2 * sizeof(int), st()));
        AAO_CUDA_TRY(cudaMemsetAsync(itcount, 0, sizeof(long long), st()));
        // ---- Schur state
        if (h->opt.mgrit_m > 0) {
            mg_m = h->opt.mgrit_m;
            mg_nc = h->nt / mg_m;
            mg_r = h->nt - mg_nc * mg_m;
        }
        const long long steps_b = std::max(mg_nc + (mg_r > 0 ? 1 : 0), 1);     // items of a batched step
        AAO_TRY(ar.alloc(&wbuf, (size_t)((h->nt + 1) * g0.nx)));
        AAO_TRY(ar.alloc(&tbuf, (size_t)(steps_b * item)));
        AAO_TRY(ar.alloc(&qbuf, (size_t)(steps_b * item)));
        AAO_TRY(ar.alloc(&tV, (size_t)(h->nt * item)));
        AAO_TRY(ar.alloc(&tmp64, (size_t)(Bmax * item)));
        AAO_TRY(ar.alloc(&stepp, 1));
        if (h->q1)
            for (int i = 0; i < 3; ++i) AAO_TRY(ar.alloc(&cheb[i], (size_t)((h->nt + 1) * g0.nx)));
        AAO_CUDA_TRY(cudaEventCreate(&e0));
        AAO_CUDA_TRY(cudaEventCreate(&e1));
        AAO_CUDA_TRY(cudaEventCreate(&e2));
        AAO_CUDA_TRY(cudaMallocHost((void**)&hact, sizeof(int) * Bmax));
        if (mg_m > 0) {
            // the coarse level of MGRIT: the same operators with step mg_m tau over mg_nc steps
            hc.reset(new Handle(*h));
            hc->arena = Arena();
            hc->P = nullptr;
            hc->nt = mg_nc;
            hc->tau = mg_m * h->tau;
            hc->nv = (long long)(mg_nc + 1) * g0.nx;
            hc->nst = hc->nv + (long long)mg_nc * s * g0.nx;
            hc->opt.mgrit_m = 0;
            coarse = new Precond(hc.get());
            AAO_TRY(coarse->setup());
            AAO_TRY(ar.alloc(&ebuf, (size_t)((mg_nc + 1) * g0.nx)));
            AAO_TRY(ar.alloc(&rbufT, (size_t)((mg_nc + 1) * g0.nx)));
            // the dataflow schedule needs no clusters: with a cluster plan the lock-step schedule runs
            nwork = cl_C > 0 ? 0 : std::min(mg_nc, (int)kMaxWorkers);
            for (int w = 0; w < nwork; ++w) {
                AAO_CUDA_TRY(cudaStreamCreateWithFlags(&wst[w], cudaStreamNonBlocking));
                AAO_CUDA_TRY(cudaEventCreateWithFlags(&ev_join[w], cudaEventDisableTiming));
                hw[w].reset(new Handle(*h));
                Handle* q = hw[w].get();
                q->arena = Arena();
                q->P = nullptr;
                q->nt = 1;
                q->nv = 2 * g0.nx;
                q->nst = q->nv + (long long)s * g0.nx;
                q->opt.mgrit_m = 0;
                q->stream = wst[w];
                q->red = Red{};        // (a worker's own reductions have its preconditioner's scratch)
                work[w] = new Precond(q);
                AAO_TRY(work[w]->setup());
                work[w]->wsrc = wbuf;
            }
            ev_f1.assign(mg_nc, nullptr);
            ev_c.assign(mg_nc + 1, nullptr);
            for (auto& e : ev_f1) AAO_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
            for (auto& e : ev_c) AAO_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
            AAO_CUDA_TRY(cudaEventCreateWithFlags(&ev_start, cudaEventDisableTiming));
        }
        AAO_CUDA_TRY(cudaStreamSynchronize(st()));
        return AAO_OK;
    }

    // Choose the tail's top level (at most max_points points, shared memory within the
    // device limit) and fill its per-stage contexts.
    aao_status build_tail(Tail& T, long long max_points, int optin) {
        const Geo& g0 = h->g;
        const int s = h->s;
        const size_t cap = 200 * 1024;
        const int ncf = g0.d == 3 ? 27 : 9;
        int lc = L - 1;
        size_t acc = 0;
        for (int l = L - 1; l >= 0; --l) {
            acc += 3 * (size_t)lev[l].g.nx * sizeof(A);
            if (lev[l].g.nx > max_points || lev[l].g.nx > (long long)kTailPmax * tail_threads || acc > cap) break;
            lc = l;
        }
        size_t vec_bytes = 0;
        for (int l = lc; l < L; ++l) vec_bytes += 3 * (size_t)lev[l].g.nx * sizeof(A);
        vec_bytes = (vec_bytes + 15) / 16 * 16;
        // stage as many of the coarsest stencils as fit next to the vectors
        int stage_from = L;
        size_t sb = 0;
        for (int l = L - 1; l >= (lc > 1 ? lc : 1); --l) {
            size_t add = ((size_t)ncf * lev[l].g.nx * sizeof(SI) + 15) / 16 * 16;
            if (vec_bytes + sb + add > cap) break;
            sb += add;
            stage_from = l;
        }
        T.lc = lc;
        T.smem = vec_bytes + sb;
        if ((long long)T.smem > optin) {
            set_error("fused multigrid tail does not fit in shared memory");
            return AAO_ERR_ARG;
        }
        for (int i = 0; i < s; ++i) {
            TailCtx<SI>& t = T.ctx[i];
            t.lc = lc;
            t.L = L;
            int o = 0;
            for (int l = lc; l < L; ++l) {
                t.op[l] = level_op(l, i);
                t.off[l] = o;
                o += 3 * (int)lev[l].g.nx;
            }
            t.vec_bytes = (int)vec_bytes;
            t.stage_from = stage_from;
            size_t so = vec_bytes;
            for (int l = 0; l < kMaxLevels; ++l) t.sten_off[l] = 0;
            for (int l = stage_from; l < L; ++l) {
                t.sten_off[l] = (int)so;
                so += ((size_t)ncf * lev[l].g.nx * sizeof(SI) + 15) / 16 * 16;
            }
            t.Dinv = Dinv[i];
            t.omega = (A)h->opt.mg_omega;
            t.nu1 = h->opt.mg_pre;
            t.nu2 = h->opt.mg_post;
        }
        return AAO_OK;
    }

    // Plan the cluster-resident shifted solve: 2D, at least one level above the coarsest, every
    // CTA owning rows of every distributed level, its share within shared memory, and the cluster
    // co-resident on the device.  Up to four plans: one for single items (16 CTAs where a layout
    // fits, else 8) and others for batches (8, 4 and 2 CTAs, so that more items run at once: 7 clusters of 16 are
    // resident, 15 of 8, 36 of 4, 76 of 2).  deep: ghost rows for whole smoothing phases (1: on
    // the coarse levels, 2: on the finest too), else one ghost row.  lean: what is read from global
    // memory (L2) instead of being staged: 1: the rows of A_c^{-1}, 2: the first coarse stencil, 3: every
    // coarse stencil.  All give the same values.
    using ClKernel = void (*)(const ClCtx<SI>, const int*, Vec<SI>, Vec<SI>);
    // The instance with the code a plan needs: faces of a kappa field, stencils in global memory (less
    // code is fetched without them).
    static ClKernel cluster_kernel(const ClCtx<SI>& t) {
        bool global = false;
        for (int l = 0; l < t.T; ++l) global = global || t.sten_global[l];
        if (t.has_faces) return global ? (ClKernel)k_cluster_mg<SI, true, true> : (ClKernel)k_cluster_mg<SI, true, false>;
        return global ? (ClKernel)k_cluster_mg<SI, false, true> : (ClKernel)k_cluster_mg<SI, false, false>;
    }

    bool plan_cluster(int C, int deep, int lean, long long dyn_max, ClCtx<SI>& t, long long& bytes, int& resident) {
        if (L > kClMaxLevels) return false;
        ClSpec spec{};
        spec.C = C;
        spec.deep = deep;
        spec.lean = lean;
        spec.L = L;
        for (int l = 0; l < L; ++l) {
            spec.n0[l] = lev[l].g.n0;
            spec.n1[l] = lev[l].g.n1;
        }
        spec.fine0 = h->q1 ? 0 : 1;
        spec.faces = spec.fine0 && h->has_kappa ? 1 : 0;
        spec.fuse0 = spec.fine0 && !spec.faces && !PT<SI>::scaled ? 1 : 0;
        spec.cycles = h->opt.mg_cycles;
        spec.nu1 = h->opt.mg_pre;
        spec.nu2 = h->opt.mg_post;
        spec.vn = ClVec<A>::n;
        spec.size = (int)sizeof(A);
        t = ClCtx<SI>{};
        bytes = cl_layout(t, spec);
        if (bytes < 0 || bytes > dyn_max) return false;
        t.sigma = A(1);
        t.fx = facesA.fx;
        t.fy = facesA.fy;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = (size_t)bytes;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(&nclusters, cluster_kernel(t), &cfg) != cudaSuccess || nclusters < 1) {
            cudaGetLastError();
            return false;
        }
        resident = nclusters;
        return true;
    }

    aao_status store_cluster_plan(ClPlan& pl, const ClCtx<SI>& plan, long long bytes, int resident) {
        ClCtx<SI> t = plan;
        const std::vector<ClOp> prog = cl_program(t);
        ClOp* dprog;
        AAO_TRY(ar.alloc(&dprog, prog.size()));
        // on the stream of the images' kernel, which reads it (a copy on the legacy stream from pageable memory may
        // end after the call, unordered with a non-blocking stream)
        AAO_CUDA_TRY(cudaMemcpyAsync(dprog, prog.data(), sizeof(ClOp) * prog.size(), cudaMemcpyHostToDevice, st()));
        for (int i = 0; i < h->s; ++i) {
            ClCtx<SI>& q = pl.ctx[i];
            q = t;
            const double c = h->tau * h->D[i], hx2 = h->g.hx2, hy2 = h->g.hy2;
            q.c = (A)c;
            // omega / a_PP by the staged weights' operations
            const A kd = A(2) * (A)hx2 + A(2) * (A)hy2;
            q.w0 = (A)h->opt.mg_omega / std::fma((A)c, kd, A(1));
            q.hx2 = (A)hx2;
            q.hy2 = (A)hy2;
            q.ex = (A)(c * hx2);
            q.ey = (A)(c * hy2);
            for (int l = 0; l < L; ++l) {
                q.sten[l] = lev[l].sten[i];
                q.sten_sc[l] = lev[l].sten_sc[i];
                q.W[l] = jacw[l][i];
            }
            q.Dinv = Dinv[i];
            const int ncst = (int)lev[L - 1].g.nx;
            A* dpad = nullptr;
            if (t.dinv_global && t.ncp != ncst) {
                AAO_TRY(ar.alloc(&dpad, (size_t)ncst * t.ncp));
                AAO_CUDA_TRY(cudaMemsetAsync(dpad, 0, sizeof(A) * (size_t)ncst * t.ncp, st()));
                AAO_CUDA_TRY(cudaMemcpy2DAsync(dpad, sizeof(A) * t.ncp, Dinv[i], sizeof(A) * ncst, sizeof(A) * ncst, ncst,
                                               cudaMemcpyDeviceToDevice, st()));
            }
            A* img;
            AAO_TRY(ar.alloc(&img, (size_t)t.img_len * t.C));
            AAO_CUDA_TRY(cudaMemsetAsync(img, 0, sizeof(A) * (size_t)t.img_len * t.C, st()));
            launch(k_cluster_image<SI>, (unsigned)t.C, kBlock, 0, st(), q, img, (const ClOp*)dprog, (int)prog.size());
            AAO_LAUNCH_CHECK();
            q.img = img;
            if (dpad) q.Dinv = dpad;
        }
        AAO_CUDA_TRY(cudaStreamSynchronize(st()));       // prog is read until here
        pl.C = t.C;
        pl.smem = (size_t)bytes;
        pl.kernel = cluster_kernel(t);
        pl.resident = resident;
        return AAO_OK;
    }

    aao_status build_cluster(int optin) {
        cl_C = 0;
        for (ClPlan& pl : clp) pl.C = 0;
        const Geo& g0 = h->g;
        if (g0.d != 2 || L < 2) return AAO_OK;
        long long dyn_max = optin;
        for (ClKernel k : {(ClKernel)k_cluster_mg<SI, false, false>, (ClKernel)k_cluster_mg<SI, false, true>,
                           (ClKernel)k_cluster_mg<SI, true, false>, (ClKernel)k_cluster_mg<SI, true, true>}) {
            cudaFuncAttributes fa;
            AAO_CUDA_TRY(cudaFuncGetAttributes(&fa, (const void*)k));
            dyn_max = std::min(dyn_max, (long long)optin - (long long)fa.sharedSizeBytes);
            if (dyn_max <= 0) return AAO_OK;
            AAO_CUDA_TRY(cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              optin - (int)fa.sharedSizeBytes));
            AAO_CUDA_TRY(cudaFuncSetAttribute((const void*)k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        }
        ClCtx<SI> t;
        long long bytes = 0;
        int resident = 0;
        // FP64 arithmetic is too slow for redundant rows; else the deepest ghost regions that fit, before
        // staging less
        const int deepest = std::is_same<A, double>::value ? 0 : 2;
        auto find = [&](int C) {
            for (int lo = 0; lo <= 2; lo += 2)          // lean 0 and 1 for every depth, then 2 and 3
                for (int deep = deepest; deep >= 0; --deep)
                    for (int lean = lo; lean <= lo + 1; ++lean)
                        if (plan_cluster(C, deep, lean, dyn_max, t, bytes, resident)) return true;
            return false;
        };
        if (!find(16) && !find(8)) return AAO_OK;
        for (int l = 0; l < L - 1; ++l) {
            if (l == 0 && !h->q1 && !h->has_kappa) continue;     // the scalar weight
            for (int i = 0; i < h->s; ++i) {
                AAO_TRY(ar.alloc(&jacw[l][i], (size_t)lev[l].g.nx));
                launch(k_jacobi_weights<SI>, (unsigned)((lev[l].g.nx + kBlock - 1) / kBlock), kBlock, 0, st(),
                       level_op(l, i), (A)h->opt.mg_omega, jacw[l][i]);
            }
        }
        AAO_LAUNCH_CHECK();
        AAO_TRY(store_cluster_plan(clp[0], t, bytes, resident));
        if (clp[0].C == 8) clp[1] = clp[0];
        else if (find(8)) AAO_TRY(store_cluster_plan(clp[1], t, bytes, resident));
        // 16-bit storage keeps to its two plans: its larger batches round intermediates as the level kernels do
        if constexpr (!PT<SI>::scaled) {
            if (find(4)) AAO_TRY(store_cluster_plan(clp[2], t, bytes, resident));
            if (find(2)) AAO_TRY(store_cluster_plan(clp[3], t, bytes, resident));
        }
        cl_C = clp[0].C;
        return AAO_OK;
    }

    // Keep the FP64 stencil of level l (shift `stage`) in the P_int storage type.
    aao_status store_stencil(int l, int i, const double* s64, int ncoef) {
        const long long n = (long long)ncoef * lev[l].g.nx;
        if constexpr (std::is_same<SI, double>::value) {
            SI* keep;
            AAO_TRY(ar.alloc(&keep, (size_t)n));
            AAO_CUDA_TRY(cudaMemcpyAsync(keep, s64, sizeof(double) * n, cudaMemcpyDeviceToDevice, st()));
            lev[l].sten[i] = keep;
        } else {
            float* sc;
            AAO_TRY(ar.alloc(&sc, ncoef));
            if (PT<SI>::scaled) {
                launch(k_stencil_absmax, ncoef, kBlock, 0, st(), s64, lev[l].g.nx, sc);
            } else {
                AAO_CUDA_TRY(cudaMemsetAsync(sc, 0, sizeof(float) * ncoef, st()));
            }
            SI* out;
            AAO_TRY(ar.alloc(&out, (size_t)n));
            launch(k_stencil_convert<SI>, (unsigned)((n + 255) / 256), 256, 0, st(), s64, lev[l].g.nx, ncoef,
                   (const float*)sc, out);
            AAO_LAUNCH_CHECK();
            lev[l].sten[i] = out;
            lev[l].sten_sc[i] = sc;
        }
        return AAO_OK;
    }

    // Q1: buf <- M^{-1} buf for B blocks of n_x by `cheb_steps` Chebyshev steps
    // with Jacobi splitting on the spectrum bounds [2^-d, (3/2)^d] of D^{-1}M.
    aao_status mass_inverse(A* buf, int B) {
        const Geo& g = h->g;
        const long long n = (long long)B * g.nx;
        const double lo = std::pow(0.5, g.d), hi = std::pow(1.5, g.d);
        const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
        double dinv = 1.0;
        for (int a = 0; a < g.d; ++a) dinv /= h->q1d.m[a][1];
        double rho = 1.0 / sigma;
        const unsigned nb = (unsigned)((n + 255) / 256);
        const PtMap pm = ptmap(g.n0);
        launch(k_cheb_init<A>, nb, 256, 0, st(), n, (const A*)buf, (A)(dinv / theta), cheb[0], cheb[1], cheb[2]);
        for (int it = 0; it < h->opt.cheb_steps; ++it) {
            launch(k_cheb_a<A>, pt_grid(pm, g.R, B), pt_block(pm), 0, st(), g, pm, B, sopA.q,
                   (const A*)cheb[2], cheb[0], cheb[1]);
            const double rn = 1.0 / (2.0 * sigma - rho);
            launch(k_cheb_b<A>, nb, 256, 0, st(), n, (A)(rn * rho), (A)(2.0 * rn / delta * dinv), (const A*)cheb[1],
                   cheb[2]);
            rho = rn;
        }
        AAO_CUDA_TRY(cudaMemcpyAsync(buf, cheb[0], sizeof(A) * n, cudaMemcpyDeviceToDevice, st()));
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    // ---------------------------------------------------------------- MG
    LevelOp<SI> level_op(int l, int stage) const {
        LevelOp<SI> op;
        op.g = lev[l].g;
        op.ncoef = op.g.d == 3 ? 27 : 9;
        if (l == 0 && !h->q1) {
            op.fine = 1;
            op.sigma = A(1);
            op.c = (A)(h->tau * h->D[stage]);
            op.faces = facesA;
        } else {
            op.fine = 0;
            op.sten = lev[l].sten[stage];
            op.sten_sc = lev[l].sten_sc[stage];
        }
        return op;
    }

    template <class S> static Vec<S> shift_vec(Vec<S> v, long long elems, int n0) {
        v.d += elems;
        if (PT<S>::scaled) v.sc += elems / n0;
        return v;
    }

    // Smoother and residual launches specialised by level kind (2D matrix-free, 2D stored; 3D generic).
    // Large batches of the 2D matrix-free level (kappa = 1) take the streaming strip kernel.
    void launch_smooth(int kind, dim3 grid, dim3 block, const LevelOp<SI>& op, const PtMap& pm, int B, const int* act,
                       Vec<SI> x, Vec<SI> b, Vec<SI> out, A om) {
        if constexpr (PT<SI>::scaled) {
            if (vec16_ok(op)) {
                const int gs = vec16_group(op.g.n0);
                if (x.d) launch(k_vec16<SI, 0>, vec16_grid(op, B), kVecThreads, 0, st(), op, gs, B, act, x, b, out, om);
                else launch(k_vec16<SI, 1>, vec16_grid(op, B), kVecThreads, 0, st(), op, gs, B, act, x, b, out, om);
                return;
            }
        }
        if constexpr (!PT<SI>::scaled) {
            if (kind == 4 && grid.y >= 16 && strip_ok(op)) {
                if (x.d) launch(k_strip2d<SI, 0>, strip_grid(op, B), kStripThreads, 0, st(), op, B, act, x, b, out, om);
                else launch(k_strip2d<SI, 1>, strip_grid(op, B), kStripThreads, 0, st(), op, B, act, x, b, out, om);
                return;
            }
            if (kind == 2 && grid.y >= 16 && strip_st_ok(op)) {
                const int rs = strip_st_rows(op, B);
                if (x.d) launch(k_strip2d_st<SI, 0>, strip_st_grid(op, B, rs), kStripThreads, 0, st(), op, B, act, x, b, out, om, rs);
                else launch(k_strip2d_st<SI, 1>, strip_st_grid(op, B, rs), kStripThreads, 0, st(), op, B, act, x, b, out, om, rs);
                return;
            }
        }
        if constexpr (std::is_same<A, float>::value) {
            if (st27_ok(op, B)) {
                const int gs = row_group(op.g.n0, 4);
                const dim3 gr = row_group_grid<SI>(op.g, 4, B);
                if (x.d) launch(k_st27<SI, 0>, gr, kVecThreads, 0, st(), op, gs, act, x, b, out, om);
                else launch(k_st27<SI, 1>, gr, kVecThreads, 0, st(), op, gs, act, x, b, out, om);
                return;
            }
        }
        launch_smooth_rows(kind, grid, block, op, pm, B, act, x, b, out, om);
    }
    // Large 2D batches take four rows per thread, a column each (grid.y = items), where a block spans the row; wider
    // rows (more than kPtMaxThreads columns) take the kernels that walk over their columns.
    static bool rows_ok(dim3 grid, dim3 block, const Geo& g) { return grid.y >= 16 && (int)block.x >= g.n0; }
    template <class... Args> void launch_smooth_rows(int kind, dim3 grid, dim3 block, const LevelOp<SI>& op,
                                                          Args... args) {
        if constexpr (!PT<SI>::scaled) {
            constexpr int kRows = 4;
            if ((kind == 4 || kind == 2) && rows_ok(grid, block, op.g)) {
                dim3 gr((grid.x + kRows - 1) / kRows, grid.y);
                if (kind == 4) launch(k_smooth_rows<SI, 4, kRows>, gr, block, 0, st(), op, args...);
                else launch(k_smooth_rows<SI, 2, kRows>, gr, block, 0, st(), op, args...);
                return;
            }
        }
        if (kind == 4) launch(k_smooth<SI, 4>, grid, block, 0, st(), op, args...);
        else if (kind == 2) launch(k_smooth<SI, 2>, grid, block, 0, st(), op, args...);
        else if (kind == 3) launch(k_smooth<SI, 3>, grid, block, 0, st(), op, args...);
        else launch(k_smooth<SI, 0>, grid, block, 0, st(), op, args...);
    }
    void launch_residual(int kind, dim3 grid, dim3 block, const LevelOp<SI>& op, const PtMap& pm, int B,
                         const int* act, Vec<SI> x, Vec<SI> b, Vec<SI> out) {
        if constexpr (PT<SI>::scaled) {
            if (vec16_ok(op) && x.d) {
                launch(k_vec16<SI, 2>, vec16_grid(op, B), kVecThreads, 0, st(), op, vec16_group(op.g.n0), B, act, x,
                       b, out, A(0));
                return;
            }
        }
        if constexpr (!PT<SI>::scaled) {
            if (kind == 4 && grid.y >= 16 && strip_ok(op) && x.d) {
                launch(k_strip2d<SI, 2>, strip_grid(op, B), kStripThreads, 0, st(), op, B, act, x, b, out, A(0));
                return;
            }
            if (kind == 2 && grid.y >= 16 && strip_st_ok(op) && x.d) {
                const int rs = strip_st_rows(op, B);
                launch(k_strip2d_st<SI, 2>, strip_st_grid(op, B, rs), kStripThreads, 0, st(), op, B, act, x, b, out, A(0), rs);
                return;
            }
        }
        if constexpr (std::is_same<A, float>::value) {
            if (st27_ok(op, B) && x.d) {
                launch(k_st27<SI, 2>, row_group_grid<SI>(op.g, 4, B), kVecThreads, 0, st(), op, row_group(op.g.n0, 4), act, x,
                       b, out, A(0));
                return;
            }
        }
        launch_residual_rows(kind, grid, block, op, pm, B, act, x, b, out);
    }
    void launch_restrict(const Geo& gf, const Geo& gc, int B, const int* act, Vec<SI> r, Vec<SI> bc) {
        if constexpr (PT<SI>::scaled) {
            if (transfer16_ok<SI>(gf)) {
                launch(k_restrict16<SI>, row_group_grid<SI>(gc, 4, B), kVecThreads, 0, st(), gf, gc, row_group(gc.n0, 4), act,
                       r, bc);
                return;
            }
        }
        if constexpr (!PT<SI>::scaled) {
            if (transfer2d_ok<SI>(gf, B)) {
                const long long pos = (long long)(gf.n0 / (16 / (int)sizeof(SI))) * gc.n1;
                launch(k_restrict2d<SI>, dim3((unsigned)((pos + kVecThreads - 1) / kVecThreads), (unsigned)B), kVecThreads, 0,
                       st(), gf, gc, act, r, bc);
                return;
            }
        }
        const PtMap pmc = ptmap(gc.n0);
        launch(k_restrict<SI>, pt_grid(pmc, gc.R, B), pt_block(pmc), 0, st(), gf, gc, pmc, B, act, r, bc);
    }
    void launch_prolong(const Geo& gf, const Geo& gc, int B, const int* act, Vec<SI> xc, Vec<SI> x, Vec<SI> out) {
        const PtMap pm = ptmap(gf.n0);
        const dim3 pbl = pt_grid(pm, gf.R, B), pth = pt_block(pm);
        if constexpr (PT<SI>::scaled) {
            if (transfer16_ok<SI>(gf)) {
                launch(k_prolong16<SI>, row_group_grid<SI>(gf, 8, B), kVecThreads, 0, st(), gf, gc, row_group(gf.n0, 8), act,
                       xc, x, out);
                return;
            }
        } else if (transfer2d_ok<SI>(gf, B)) {
            const long long pos = (long long)(gf.n0 / (16 / (int)sizeof(SI))) * ((gf.n1 + 1) / 2);
            launch(k_prolong2d<SI>, dim3((unsigned)((pos + kVecThreads - 1) / kVecThreads), (unsigned)B), kVecThreads, 0, st(),
                   gf, gc, act, xc, x, out);
            return;
        } else if (gf.d == 2 && rows_ok(pbl, pth, gf)) {
            launch(k_prolong_add_rows<SI, 4>, dim3((pbl.x + 3) / 4, pbl.y), pth, 0, st(), gf, gc, pm, B, act, xc, x, out);
            return;
        }
        launch(k_prolong_add<SI>, pbl, pth, 0, st(), gf, gc, pm, B, act, xc, x, out);
    }
    template <class... Args> void launch_residual_rows(int kind, dim3 grid, dim3 block, const LevelOp<SI>& op,
                                                            Args... args) {
        if constexpr (!PT<SI>::scaled) {
            constexpr int kRows = 4;
            if ((kind == 4 || kind == 2) && rows_ok(grid, block, op.g)) {
                dim3 gr((grid.x + kRows - 1) / kRows, grid.y);
                if (kind == 4) launch(k_residual_rows<SI, 4, kRows>, gr, block, 0, st(), op, args...);
                else launch(k_residual_rows<SI, 2, kRows>, gr, block, 0, st(), op, args...);
                return;
            }
        }
        if (kind == 4) launch(k_residual<SI, 4>, grid, block, 0, st(), op, args...);
        else if (kind == 2) launch(k_residual<SI, 2>, grid, block, 0, st(), op, args...);
        else if (kind == 3) launch(k_residual<SI, 3>, grid, block, 0, st(), op, args...);
        else launch(k_residual<SI, 0>, grid, block, 0, st(), op, args...);
    }

    // x_out = V-cycle(l) applied to (x_in, b); x_in.d == nullptr: zero guess.
    aao_status vcycle(int l, int stage, int B, const int* act, Vec<SI> xin, Vec<SI> b, Vec<SI> xout) {
        const Geo& g = lev[l].g;
        const PtMap pm = ptmap(g.n0);
        const dim3 pbl = pt_grid(pm, g.R, B), pth = pt_block(pm);
        const Tail& T = tails[B > 1 ? 1 : 0];
        // (a tail that is the coarsest level alone: its rows on as many SMs instead of one)
        if (l == T.lc && l < L - 1) {
            bytes_hint((xin.d ? 3.0 : 2.0) * nact * g.nx * sizeof(SI));
            if (g.d == 2)
                launch(k_vcycle_tail_2d<SI>, (unsigned)B, dim3(32, 32), T.smem, st(), T.ctx[stage], B, act, b, xin,
                       xout);
            else
                launch(k_vcycle_tail<SI>, (unsigned)B, tail_threads, T.smem, st(), T.ctx[stage], B, act, b, xin, xout);
            AAO_LAUNCH_CHECK();
            return AAO_OK;
        }
        if (l == L - 1) {
            bytes_hint(2.0 * nact * g.nx * sizeof(SI));
            launch(k_coarse_solve<SI>, dim3((unsigned)g.R, (unsigned)B), kCoarseThreads, 0, st(), g, B, act,
                   (const A*)Dinv[stage], b, xout);
            AAO_LAUNCH_CHECK();
            return AAO_OK;
        }
        LevelOp<SI> op = level_op(l, stage);
        const Geo& gc = lev[l + 1].g;
        const PtMap pmc = ptmap(gc.n0);
        const dim3 cbl = pt_grid(pmc, gc.R, B), cth = pt_block(pmc);
        const A om = (A)h->opt.mg_omega;
        const int nu1 = h->opt.mg_pre, nu2 = h->opt.mg_post;
        // Fused kernels trade recomputation for launches: they pay off where the
        // V-cycle is latency bound (small batches: the Schur sweep), not in the
        // bandwidth- or FP64-bound batched phase.  Only on 2D levels and on the
        // matrix-free fine level (a 27-point stored stencil makes the neighbour
        // recomputation too costly).
        // (a finest level that streams through k_vec16 is not fused: its separate sweeps are cheaper
        // than the fused kernels' recomputation)
        const bool fuse = (long long)B * g.nx <= kFuseMaxPoints && (g.d == 2 || op.fine) && !vec16_ok(op);
        const bool f2 = fuse && nu1 >= 2, fps = fuse && nu2 >= 1;
        const bool tiles = t3_ok(op) && B <= 65535;
        const int pre_l = f2 ? nu1 - 1 : nu1;
        const int post_l = fps ? nu2 : nu2 + 1;
        const int nops = pre_l + post_l;
        Vec<SI> cur = xin;
        int opi = 0;
        auto dest = [&](void) -> Vec<SI> {
            ++opi;
            if (opi == nops) return xout;
            return (cur.d == lev[l].T0.d) ? lev[l].T1 : lev[l].T0;
        };
        int q = 0;
        if (f2) {
            Vec<SI> d = dest();
            bytes_hint((cur.d ? 3.0 : 2.0) * nact * g.nx * sizeof(SI));
            if (tiles)
                launch(k_smooth2_tile<SI>, t3_grid(g.n1, g.n2, kT3, B), kT3Threads, t3_smem_smooth2(g.n0, sizeof(A)), st(),
                       op, inv_h2<A>(g), act, cur, b, d, om);
            else launch(k_smooth2<SI>, pbl, pth, 0, st(), op, pm, B, act, cur, b, d, om);
            cur = d;
            q = 2;
        }
        for (; q < nu1; ++q) {
            Vec<SI> d = dest();
            bytes_hint((cur.d ? 3.0 : 2.0) * nact * g.nx * sizeof(SI));
            launch_smooth(level_kind(op.fine, g.d, g.nx), pbl, pth, op, pm, B, act, cur, b, d, om);
            cur = d;
        }
        // residual and restriction
        if (fuse) {
            bytes_hint(((cur.d ? 2.0 : 1.0) * g.nx + gc.nx) * nact * sizeof(SI));
            if (tiles)
                launch(k_resid_restrict_tile<SI>, t3_grid(gc.n1, gc.n2, kT3 / 2, B), kT3Threads,
                       t3_smem_restrict(g.n0, sizeof(A)), st(), op, inv_h2<A>(g), gc, act, cur, b, lev[l + 1].Bb);
            else launch(k_resid_restrict<SI>, cbl, cth, 0, st(), op, gc, pmc, B, act, cur, b, lev[l + 1].Bb);
        } else if (cur.d == nullptr) {
            bytes_hint(1.0 * nact * (g.nx + gc.nx) * sizeof(SI));
            launch_restrict(g, gc, B, act, b, lev[l + 1].Bb);
        } else {
            bytes_hint(3.0 * nact * g.nx * sizeof(SI));
            launch_residual(level_kind(op.fine, g.d, g.nx), pbl, pth, op, pm, B, act, cur, b, lev[l].Rr);
            bytes_hint(1.0 * nact * (g.nx + gc.nx) * sizeof(SI));
            launch_restrict(g, gc, B, act, lev[l].Rr, lev[l + 1].Bb);
        }
        AAO_LAUNCH_CHECK();
        Vec<SI> zero{};
        AAO_TRY(vcycle(l + 1, stage, B, act, zero, lev[l + 1].Bb, lev[l + 1].X));
        q = 0;
        if (fps) {
            Vec<SI> d = dest();
            bytes_hint(1.0 * nact * (gc.nx + (cur.d ? 3.0 : 2.0) * g.nx) * sizeof(SI));
            if (tiles)
                launch(k_prolong_smooth_tile<SI>, t3_grid(g.n1, g.n2, kT3, B), kT3Threads, t3_smem_prolong(g.n0, sizeof(A)),
                       st(), op, inv_h2<A>(g), gc, act, lev[l + 1].X, cur, b, d, om);
            else launch(k_prolong_smooth<SI>, pbl, pth, 0, st(), op, gc, pm, B, act, lev[l + 1].X, cur, b, d, om);
            cur = d;
            q = 1;
        } else {
            Vec<SI> d = dest();
            bytes_hint(1.0 * nact * (gc.nx + (cur.d ? 2.0 : 1.0) * g.nx) * sizeof(SI));
            launch_prolong(g, gc, B, act, lev[l + 1].X, cur, d);
            cur = d;
        }
        for (; q < nu2; ++q) {
            Vec<SI> d = dest();
            bytes_hint(3.0 * nact * g.nx * sizeof(SI));
            launch_smooth(level_kind(op.fine, g.d, g.nx), pbl, pth, op, pm, B, act, cur, b, d, om);
            cur = d;
        }
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    // us of three cycles of B items on the clusters of a plan: waves of resident clusters times a launch, whose
    // steps cost 14 us per distributed level and 5.5 us per 1000 points of a CTA beyond 2500, 15% more where every sweep on
    // the finest level is followed by an exchange (FP64: 22 and 55 per 1000 points); per sweep, relative to V(2,2)-cycles.
    double cluster_cost(const ClPlan& pl, int B) const {
        const double per = (double)h->g.nx / pl.C, sweeps = h->opt.mg_pre + h->opt.mg_post;
        const double launch = std::is_same<A, double>::value
                                  ? (22.0 * (L - 1) + 55e-3 * per) * (0.42 + 0.145 * sweeps)
                                  : (14.0 * (L - 1) + 5.5e-3 * std::max(0.0, per - 2500.0)) * (0.66 + 0.085 * sweeps) *
                                        (pl.ctx[0].H[0] > 1 ? 1.0 : 1.15);
        return launch * ((B + pl.resident - 1) / pl.resident);
    }
    // The same on the level kernels: the tail, an SM per item, and each level above it by its points, less where whole batches
    // stream (kFuseMaxPoints), least on the finest level with kappa = 1 and rows of whole vectors.
    double levels_cost(int B) const {
        const bool f64 = std::is_same<A, double>::value;
        const int lc = tails[B > 1 ? 1 : 0].lc, sweeps = h->opt.mg_pre + h->opt.mg_post;
        const double tail = (f64 ? 93.0 + 121e-3 * lev[lc].g.nx : 113.0 + 17.5e-3 * lev[lc].g.nx) * ((B + 151) / 152);
        double above = 0.0;
        for (int l = 0; l < lc; ++l) {
            const long long points = (long long)B * lev[l].g.nx;
            const bool vectors = lev[l].g.n0 % kVN == 0 && (l > 0 || (!h->q1 && !h->has_kappa));
            const double us = points <= kFuseMaxPoints ? (f64 ? 1.7e-3 : 0.36e-3)
                              : vectors                ? (f64 ? 0.45e-3 : 0.061e-3)
                                                       : (f64 ? 0.68e-3 : 0.12e-3);
            above += us * (double)points;
        }
        return (tail + above) * (f64 ? 0.28 + 0.18 * sweeps : 0.56 + 0.11 * sweeps);
    }
    // The cluster plan of a batch, or null: the level kernels.  16-bit storage: 8 CTAs per item from kClBatch8
    // items on, up to kClMaxBatch items.  Else the plan of the least cost if that is below 0.8 of the level kernels'.  The
    // costs are fitted to inner solves of one step (two shifted solves; us, level kernels / 16 / 8 / 4 / 2 CTAs per item):
    //   FP32 64^2, B = 64: 455 / 674 / 372 / 202 / 157; 127 x 95, B = 24: 583 / 451 / 285 / 204 / 228;
    //   256^2, B = 64: 1873 / 1549 / 1119 / - / -, B = 128: 1726 / 2876 / 1969 / - / -
    //   FP64 64^2, B = 40: 1271 / 803 / 524 / 504 / 433; 127 x 95, B = 40: 2667 / 1441 / 1030 / 1070 / -;
    //   128^2, B = 256: 5618 / 9094 / 6599 / 5200 / -; 256^2, B = 40: 5842 / 4099 / - / - / -,
    //   B = 128: 9936 / 12708 / - / - / -
    // with about 70 us of Krylov kernels in each.  Over kappa, Q1, 1 and 3 cycles, one to six sweeps, 32^2 to 256^2 and 1 to 256
    // items the choice costs 17% more than the best one at most, 0.6% on average.
    const ClPlan* pick_cluster(int B) const {
        if (cl_C == 0) return nullptr;
        if constexpr (PT<SI>::scaled) {
            if (B > kClMaxBatch) return nullptr;
            return B >= kClBatch8 && clp[1].C > 0 ? &clp[1] : &clp[0];
        }
        const ClPlan* best = nullptr;
        // (a batch of one wave of the largest clusters: the level kernels are launch-bound there)
        double cost = B <= clp[0].resident ? 1e300 : 0.8 * levels_cost(B);
        for (const ClPlan& pl : clp) {
            if (pl.C == 0) continue;
            const double c = cluster_cost(pl, B);
            if (c < cost) {
                cost = c;
                best = &pl;
            }
        }
        return best;
    }

    aao_status mg_solve(int stage, int B, const int* act, Vec<SI> b, Vec<SI> out) {
        if (const ClPlan* plan = pick_cluster(B)) {
            // one cluster per item: small batches (single time steps, MGRIT's batched steps)
            const ClPlan& pl = *plan;
            bytes_hint(2.0 * nact * h->g.nx * sizeof(SI));
            launch_cluster(pl.kernel, dim3((unsigned)(pl.C * B)), dim3(kClThreads), pl.smem, st(), pl.C,
                           pl.ctx[stage], act, b, out);
            AAO_LAUNCH_CHECK();
            return AAO_OK;
        }
        Vec<SI> zero{};
        for (int cyc = 0; cyc < h->opt.mg_cycles; ++cyc) AAO_TRY(vcycle(0, stage, B, act, cyc == 0 ? zero : out, b, out));
        return AAO_OK;
    }

    // Z = P_int^{-1} V (items of s*nx), forward or backward stage sweep.
    aao_status rana(int B, const int* act, Vec<SP> V, Vec<SI> Z, int transpose) {
        const Geo& g = h->g;
        const int s = h->s;
        const PtMap pm0 = ptmap(g.n0);
        for (int t = 0; t < s; ++t) {
            int i = transpose ? s - 1 - t : t;
            const double* coef = (transpose ? h->d_LDb : h->d_LDf) + i * s;
            Vec<SI> Zi = shift_vec(Z, (long long)i * g.nx, g.n0);
            if constexpr (std::is_same<SP, SI>::value && !PT<SI>::scaled) {
                // the sweep's first stage has no coupling (L is unit lower triangular): its right-hand
                // side is V_i itself, which the shifted solve reads in place (the copy into mgb would
                // store the same values)
                if (t == 0) {
                    AAO_TRY(mg_solve(i, B, act, shift_vec(V, (long long)i * g.nx, g.n0), Zi));
                    continue;
                }
            }
            bytes_hint(1.0 * nact * g.nx * (sizeof(SP) + (transpose ? s - 1 - i : i) * sizeof(SI) + sizeof(SI)));
            if constexpr (!PT<SI>::scaled) {
                if (!h->q1) {
                    launch_rana_vec(B, act, V, i, Z, transpose);
                    AAO_TRY(mg_solve(i, B, act, mgb, Zi));
                    continue;
                }
            }
            if constexpr (PT<SI>::scaled) {
                if (!h->q1) {
                    launch(k_rana_pt<SP, SI>, pt_grid(pm0, g.R, B), pt_block(pm0), 0, st(), g, inv_h2<A>(g), pm0, B, act, V,
                           (long long)s * g.R, i, Z, stage_coef(i, transpose), facesA, mgb);
                    AAO_LAUNCH_CHECK();
                    AAO_TRY(mg_solve(i, B, act, mgb, Zi));
                    continue;
                }
            }
            launch(k_rana_rhs<SP, SI>, pt_grid(pm0, g.R, B), pt_block(pm0), 0, st(), g, pm0, B, act, V, i, Z, s,
                   coef, (A)h->tau, sopA, mgb);
            AAO_LAUNCH_CHECK();
            AAO_TRY(mg_solve(i, B, act, mgb, Zi));
        }
        return AAO_OK;
    }

    // ------------------------------------------------------- inner GMRES
    static constexpr int kVN = (int)(16 / sizeof(A));    // points per thread where rows are whole vectors
    bool rows_vec() const { return h->g.n0 % kVN == 0 && !h->q1; }
    template <class F> static void with_int(bool big, F&& f) {     // f(std::true_type) or f(std::false_type)
        if (big) f(std::true_type{});
        else f(std::false_type{});
    }
    static bool aligned16(const void* p) { return (reinterpret_cast<unsigned long long>(p) & 15ULL) == 0; }

    // Blocks per item of the Arnoldi kernels: one position per thread while that gives fewer than kArBlocks
    // blocks (48 per SM) over the batch, else the blocks stride over the item.
    ArRed ar_red(int B, long long positions) const {
        const long long full = (positions + kArThreads - 1) / kArThreads, cap = (kArBlocks + B - 1) / B;
        ArRed r;
        r.part = ar_part;
        r.count = ar_count;
        r.nchunk = (int)std::max<long long>(1, std::min(full, cap));
        return r;
    }
    ArItems ar_items() const {
        ArItems it;
        it.kin = kin;
        it.H = Hh;
        it.cs = csh;
        it.sn = snh;
        it.g = gh;
        it.beta = betah;
        it.y = yh;
        it.gram = gramh;
        it.active = activeh;
        it.its = itsh;
        it.nonfinite = nonfin;
        it.breakdown = brk;
        it.count = itcount;
        it.tol = itol;
        return it;
    }
    template <class S> Basis<S> basis_of(const Vec<S>& v, long long stride) const {
        return Basis<S>{v, stride, (long long)h->s * h->g.R, stride / h->g.n0};
    }

    // v = src / denom per item of s*n_x values (rep: src is one stage of n_x, used for every stage).
    template <class SR>
    void scale_basis(int B, const SR* src, long long sbs, const double* denom, long long dstride, Vec<SP> v, int rep,
                     StepPtrs* sp) {
        const Geo& g = h->g;
        const long long item = (long long)h->s * g.nx;
        if constexpr (PT<SP>::scaled) {
            const PtMap pm = ptmap(g.n0);
            const int rows = h->s * g.R;
            launch(k_scale_store<SP, SR>, pt_grid(pm, rows, B), pt_block(pm), 0, st(), pm, rows, B,
                   (const int*)activeh, src, sbs, denom, dstride, v, rep ? g.R : 0, sp);
        } else {
            constexpr int U = 2;
            const bool vec = g.n0 % kVN == 0 && (sizeof(SR) != sizeof(SP) || aligned16(src));
            with_int(vec, [&](auto big) {
                constexpr int N = decltype(big)::value ? kVN : 1;
                const long long per = (long long)U * kArThreads * N, n = rep ? g.nx : item;
                launch(k_scale_vec<SP, SR, N, U>, dim3((unsigned)((n + per - 1) / per), (unsigned)B), kArThreads, 0,
                       st(), item, g.nx, rep ? h->s : 0, (const int*)activeh, src, sbs, denom, dstride, v, sp);
            });
        }
    }

    StageCoef<A> stage_coef(int i, int transpose) const {
        const int s = h->s;
        StageCoef<A> cf{};
        cf.j0 = transpose ? i + 1 : 0;
        cf.j1 = transpose ? s : i;
        for (int j = cf.j0; j < cf.j1; ++j)
            cf.c[j] = (A)h->tau * (A)(transpose ? h->L[j * s + i] * h->D[i] : h->L[i * s + j] * h->D[j]);
        return cf;
    }

    void launch_rana_vec(int B, const int* act, Vec<SP> V, int i, Vec<SI> Z, int transpose) {
        const Geo& g = h->g;
        const int s = h->s;
        const StageCoef<A> cf = stage_coef(i, transpose);
        with_int(rows_vec(), [&](auto big) {
            constexpr int N = decltype(big)::value ? kVN : 1;
            const long long pos = (long long)(g.n0 / N) * g.R;
            const dim3 grid((unsigned)((pos + kArThreads - 1) / kArThreads), (unsigned)B);
            with_int(s > 3, [&](auto many) {
                constexpr int TS = decltype(many)::value ? kMaxS : 3;
                launch(k_rana_vec<SP, SI, N, TS>, grid, kArThreads, 0, st(), g, inv_h2<A>(g), act, V, i, Z, cf, facesA,
                       mgb);
            });
        });
    }

    // The Krylov steps of B items whose v_0 is in place (ar_init has run): on exit Z0 / yh / itsh hold
    // every item's solution.
    aao_status arnoldi(int B, int transpose) {
        const Geo& g = h->g;
        const int s = h->s;
        const long long item = (long long)s * g.nx;
        const unsigned rows = (unsigned)s * (unsigned)g.R;
        const Basis<SP> V = basis_of(V0, vstride);
        const ArItems it = ar_items();
        refresh_nact(B);
        for (int k = 0; k < kin; ++k) {
            Vec<SP> Vk = shift_vec(V0, k * vstride, g.n0);
            Vec<SI> Zk = shift_vec(Z0, k * zstride, g.n0);
            AAO_TRY(rana(B, activeh, Vk, Zk, transpose));
            with_int(rows_vec(), [&](auto big) {
                constexpr int N = decltype(big)::value ? kVN : 1;
                const long long pos = (long long)(g.n0 / N) * g.R;
                const ArRed rt = ar_red(B, pos), ru = ar_red(B, s * pos);
                with_int(kin > kArSmallK, [&](auto deep) {
                    constexpr int MK = decltype(deep)::value ? kMaxInner : kArSmallK;
                    with_int(s > 3, [&](auto many) {
                        constexpr int TS = decltype(many)::value ? kMaxS : 3;
                        bytes_hint(1.0 * nact * item * (sizeof(SI) + sizeof(A) + (k + 1) * sizeof(SP)));
                        launch(k_theta_dots<SI, SP, A, N, TS, MK>, dim3((unsigned)rt.nchunk, (unsigned)B), kArThreads,
                               0, st(), g, inv_h2<A>(g), (const int*)activeh, Zk, (long long)rows, wv, item, s,
                               (const double*)(transpose ? h->d_AT : h->d_A), (A)h->tau, sopA, V, k, rt, it);
                    });
                    bytes_hint(1.0 * nact * item * (2 * sizeof(A) + (k + 1) * sizeof(SP)));
                    launch(k_arnoldi_upd<SP, A, N, MK>, dim3((unsigned)ru.nchunk, (unsigned)B), kArThreads, 0, st(),
                           g.n0, rows, (const int*)activeh, wv, item, V, k, ru, it);
                });
            });
            AAO_LAUNCH_CHECK();
            refresh_nact(B);
            if (k + 1 < kin)
                scale_basis<A>(B, wv, item, Hh + (k + 1) * kin + k, (long long)(kin + 1) * kin,
                               shift_vec(V0, (k + 1) * vstride, g.n0), 0, nullptr);
            AAO_LAUNCH_CHECK();
        }
        return AAO_OK;
    }

    // out_b = sum_k y_k Z_k of every item.
    template <class SO> void combine(int B, SO* out, long long obs) {
        const Geo& g = h->g;
        const unsigned rows = (unsigned)h->s * (unsigned)g.R;
        with_int(g.n0 % kVN == 0 && (!std::is_same<SO, double>::value || std::is_same<A, float>::value || aligned16(out)),
                 [&](auto big) {
            constexpr int N = decltype(big)::value ? kVN : 1;
            const long long pos = (long long)(g.n0 / N) * rows;
            launch(k_combine_vec<SI, SO, N>, dim3((unsigned)((pos + kArThreads - 1) / kArThreads), (unsigned)B),
                   kArThreads, 0, st(), g.n0, rows, basis_of(Z0, zstride), (const double*)yh, kin, (const int*)itsh, out,
                   obs);
        });
    }

    // Batched GMRES(kin) on Theta_hat (or Theta_hat^T) for B items of s*nx;
    // rhs item b at src + b*sbs (type SR, unscaled).  On exit Z0/yh/itsh hold the
    // Krylov solution of every item; out (if given) receives sum_k y_k Z_k.
    template <class SR>
    aao_status inner(int B, const SR* src, long long sbs, double* out, long long obs, int transpose) {
        const long long item = (long long)h->s * h->g.nx;
        const ArRed red = ar_red(B, item / 16 + 1);
        launch(k_ar_start<SR>, dim3((unsigned)red.nchunk, (unsigned)B), kArThreads, 0, st(), item, src, sbs, red,
               ar_items());
        scale_basis<SR>(B, src, sbs, (const double*)betah, 1LL, V0, 0, nullptr);
        AAO_LAUNCH_CHECK();
        AAO_TRY(arnoldi(B, transpose));
        if (out) combine<double>(B, out, obs);
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    // One forward step of S_tilde's recurrence for B items, time index sp->n + b * stride (advanced by
    // one): t = K z_n, Theta_tilde^{-1} (e (x) t), and z_{n+1} or its C-point residual.
    aao_status forward_step(int B, int stride, const A* w, A* res) {
        const Geo& g = h->g;
        const int s = h->s;
        const ArRed red = ar_red(B, g.nx / 4 + 1);        // four points per thread: the reduction is the larger part
        with_int(h->q1 != 0, [&](auto q1) {
            launch(k_schur_start<A, decltype(q1)::value>, dim3((unsigned)red.nchunk, (unsigned)B), kArThreads, 0, st(), g, s,
                   (const StepPtrs*)stepp, stride, tbuf, sopA, red, ar_items());
        });
        scale_basis<A>(B, tbuf, g.nx, (const double*)betah, 1LL, V0, 1, stepp);
        AAO_LAUNCH_CHECK();
        AAO_TRY(arnoldi(B, 0));
        with_int(g.n0 % kVN == 0, [&](auto big) {
            constexpr int N = decltype(big)::value ? kVN : 1;
            const long long pos = (long long)(g.n0 / N) * g.R;
            launch(k_schur_finish<SI, A, N>, dim3((unsigned)((pos + kArThreads - 1) / kArThreads), (unsigned)B),
                   kArThreads, 0, st(), g, s, w, (const StepPtrs*)stepp, stride, basis_of(Z0, zstride), (const double*)yh,
                   kin, (const int*)itsh, (const double*)h->d_b, h->tau, res);
        });
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    // ------------------------------------------------------------- P_tilde
    // One step of the Schur substitution (forward: z_{v,n} -> z_{v,n+1};
    // transposed: u_{n+1} -> u_n), with n, z and r read from device memory.
    aao_status schur_step(int transpose) {
        const Geo& g = h->g;
        const int s = h->s;
        const long long item = (long long)s * g.nx;
        const unsigned nbr = blocks_for_rows(g.R);
        if (!transpose) {
            AAO_TRY(forward_step(1, 0, wsrc ? wsrc : (const A*)wbuf, nullptr));
        } else {
            launch(k_schurT_rhs<A>, (unsigned)((item + 255) / 256), 256, 0, st(), g.nx, s, (const StepPtrs*)stepp,
                   (const double*)h->d_b, tbuf);
            AAO_TRY(inner<A>(1, tbuf, item, nullptr, 0, 1));
            combine<A>(1, qbuf, item);
            launch(k_schurT_update<A>, nbr, kBlock, 0, st(), g, s, (const StepPtrs*)stepp, (const A*)qbuf, h->tau,
                   sopA);
            launch(k_step_add, 1, 1, 0, st(), stepp, -1);
        }
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    // A batched step of the recurrence over B of MGRIT's intervals (items b = 0..B-1 at time
    // indices sp->n +- b mg_m), or with `residual` the C-point residuals into the coarse source.
    aao_status schur_step_b(int transpose, int residual, int B) {
        const Geo& g = h->g;
        const int s = h->s;
        const int stride = mg_m;
        const long long item = (long long)s * g.nx;
        const unsigned nbr = blocks_for_rows(g.R);
        if (!transpose) {
            AAO_TRY(forward_step(B, stride, wbuf, residual ? coarse->wbuf : (A*)nullptr));
        } else {
            launch(k_schurT_rhs_b<A>, dim3((unsigned)((item + 255) / 256), (unsigned)B), 256, 0, st(), g.nx, s,
                   (const StepPtrs*)stepp, stride, (const double*)h->d_b, tbuf);
            AAO_TRY(inner<A>(B, tbuf, item, nullptr, 0, 1));
            combine<A>(B, qbuf, item);
            launch(k_schurT_update_b<A>, dim3(nbr, (unsigned)B), kBlock, 0, st(), g, s, (const StepPtrs*)stepp, stride,
                   (const A*)qbuf, h->tau, sopA, residual ? rbufT : (double*)nullptr, B);
            launch(k_step_add, 1, 1, 0, st(), stepp, -1);
        }
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    aao_status step_of_kind(int transpose, int kind) {
        if (kind == 0) return schur_step(transpose);
        return schur_step_b(transpose, kind == 2, kind == 3 ? mg_nc + 1 : mg_nc);
    }

    // Capture one step of a kind into a CUDA graph (on a private stream) the first time
    // it is needed; replays then issue the whole step with one launch.
    aao_status ensure_graph(int transpose, int kind) {
        if (gexec[transpose][kind]) return AAO_OK;
        if (!cap_stream) AAO_CUDA_TRY(cudaStreamCreateWithFlags(&cap_stream, cudaStreamNonBlocking));
        cudaStream_t keep = cur_stream;
        cur_stream = cap_stream;
        const long long before = g_thread_launches;
        AAO_CUDA_TRY(cudaStreamBeginCapture(cap_stream, cudaStreamCaptureModeThreadLocal));
        aao_status st_ = step_of_kind(transpose, kind);
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(cap_stream, &graph);
        cur_stream = keep;
        // captured launches run only when the graph is replayed: count them there
        g_launches -= g_thread_launches - before;
        g_thread_launches = before;
        if (st_ != AAO_OK) {
            if (graph) cudaGraphDestroy(graph);
            return st_;
        }
        if (e != cudaSuccess) {
            set_error(std::string("graph capture failed: ") + cudaGetErrorString(e));
            return AAO_ERR_CUDA;
        }
        size_t nodes = 0;
        cudaGraphGetNodes(graph, nullptr, &nodes);
        graph_nodes[transpose][kind] = (long long)nodes;
        e = cudaGraphInstantiate(&gexec[transpose][kind], graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            gexec[transpose][kind] = nullptr;
            set_error(std::string("graph instantiation failed: ") + cudaGetErrorString(e));
            return AAO_ERR_CUDA;
        }
        return AAO_OK;
    }

    // `count` steps of a kind, each a graph replay (eager launches while a launch profile is open,
    // which needs one event pair per kernel).
    aao_status run_steps(int transpose, int kind, int count) {
        const bool use_graph = !g_prof_on;
        if (use_graph) AAO_TRY(ensure_graph(transpose, kind));
        for (int q = 0; q < count; ++q) {
            if (use_graph) {
                AAO_CUDA_TRY(cudaGraphLaunch(gexec[transpose][kind], st()));
                g_launches += graph_nodes[transpose][kind];
            } else {
                AAO_TRY(step_of_kind(transpose, kind));
            }
        }
        return AAO_OK;
    }

    aao_status schur_sweep(int transpose) { return run_steps(transpose, 0, h->nt); }

    // S_tilde's recurrence z_0 = w_0, z_{n+1} = Phi(z_n) + w_{n+1} by one two-level MGRIT
    // iteration with C-points n = c m (F-relaxation; initial guess z_0 = w_0, zero C-points):
    //   1. interval c relaxes from its C-point to the next one; z_{cm+1} = Phi(0) + w_{cm+1} =
    //      w_{cm+1} for c > 0, and the interval's last step yields the next C-point's residual
    //      r_{c+1} = w_{(c+1)m} + Phi(z_{(c+1)m-1}) - 0 in place of that (zero) C-point;
    //   2. the coarse recurrence e_c = Phi_c(e_{c-1}) + r_c (the substitution step with step m tau),
    //      and the corrected C-point z_{cm} = 0 + e_c;
    //   3. a final F-relaxation of every interval from its corrected C-point.
    // The intervals run on the workers' streams; event c orders interval c's first relaxation before
    // coarse step c+1, and coarse step c before interval c's final relaxation, so the coarse chain
    // overlaps the intervals' work.  Used when the shifted solves run as level kernels (no cluster
    // plan): concurrent single-item steps then fill the GPU.  w is in wbuf; z_0 is set by the caller.
    aao_status mgrit_dataflow_forward(double* z) {
        const long long nx = h->g.nx;
        const int m = mg_m, nc = mg_nc, K = nwork;
        const unsigned nb = (unsigned)((nx + 255) / 256);
        AAO_CUDA_TRY(cudaEventRecord(ev_start, st()));
        for (int w = 0; w < K; ++w) AAO_CUDA_TRY(cudaStreamWaitEvent(wst[w], ev_start, 0));
        for (int c = 0; c < nc; ++c) {
            Precond* W = work[c % K];
            if (c == 0) {
                launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, (const double*)nullptr, 0);
                AAO_TRY(W->run_steps(0, 0, m));
            } else {
                launch(k_convert<A, double>, nb, 256, 0, W->st(), (const A*)(wbuf + (long long)(c * m + 1) * nx),
                       z + (long long)(c * m + 1) * nx, nx);
                launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, (const double*)nullptr, c * m + 1);
                AAO_TRY(W->run_steps(0, 0, m - 1));
            }
            AAO_CUDA_TRY(cudaEventRecord(ev_f1[c], W->st()));
        }
        AAO_CUDA_TRY(cudaMemsetAsync(coarse->wbuf, 0, sizeof(A) * nx, st()));
        AAO_CUDA_TRY(cudaMemsetAsync(ebuf, 0, sizeof(double) * nx, st()));
        launch(k_step_set, 1, 1, 0, st(), coarse->stepp, ebuf, (const double*)nullptr, 0);
        for (int c = 1; c <= nc; ++c) {
            AAO_CUDA_TRY(cudaStreamWaitEvent(st(), ev_f1[c - 1], 0));
            launch(k_convert<double, A>, nb, 256, 0, st(), (const double*)(z + (long long)c * m * nx),
                   coarse->wbuf + (long long)c * nx, nx);
            AAO_TRY(coarse->run_steps(0, 0, 1));
            AAO_CUDA_TRY(cudaMemcpyAsync(z + (long long)c * m * nx, ebuf + (long long)c * nx, sizeof(double) * nx,
                                         cudaMemcpyDeviceToDevice, st()));
            AAO_CUDA_TRY(cudaEventRecord(ev_c[c], st()));
        }
        for (int c = 0; c < nc; ++c) {
            Precond* W = work[c % K];
            if (c > 0) AAO_CUDA_TRY(cudaStreamWaitEvent(W->st(), ev_c[c], 0));
            launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, (const double*)nullptr, c * m);
            AAO_TRY(W->run_steps(0, 0, m - 1));
        }
        if (mg_r > 0) {           // the shorter final interval, from the last C-point
            Precond* W = work[nc % K];
            AAO_CUDA_TRY(cudaStreamWaitEvent(W->st(), ev_c[nc], 0));
            launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, (const double*)nullptr, nc * m);
            AAO_TRY(W->run_steps(0, 0, mg_r));
        }
        for (int w = 0; w < K; ++w) {
            AAO_CUDA_TRY(cudaEventRecord(ev_join[w], wst[w]));
            AAO_CUDA_TRY(cudaStreamWaitEvent(st(), ev_join[w], 0));
        }
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    // The same for S_tilde^T's backward recurrence u_nt = r_{v,nt}, u_n = Phi^T(u_{n+1}) + r_{v,n},
    // run forward in reversed time (C-points n = nt - c m).  u_nt is set by the caller.
    aao_status mgrit_dataflow_transpose(double* z, const double* r) {
        const long long nx = h->g.nx;
        const int m = mg_m, nc = mg_nc, K = nwork, nt = h->nt;
        AAO_CUDA_TRY(cudaEventRecord(ev_start, st()));
        for (int w = 0; w < K; ++w) AAO_CUDA_TRY(cudaStreamWaitEvent(wst[w], ev_start, 0));
        for (int c = 0; c < nc; ++c) {
            Precond* W = work[c % K];
            if (c == 0) {
                launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, r, nt - 1);
                AAO_TRY(W->run_steps(1, 0, m));
            } else {
                const long long n1 = nt - c * m - 1;
                AAO_CUDA_TRY(cudaMemcpyAsync(z + n1 * nx, r + n1 * nx, sizeof(double) * nx, cudaMemcpyDeviceToDevice,
                                             W->st()));
                launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, r, (int)n1 - 1);
                AAO_TRY(W->run_steps(1, 0, m - 1));
            }
            AAO_CUDA_TRY(cudaEventRecord(ev_f1[c], W->st()));
        }
        AAO_CUDA_TRY(cudaMemsetAsync(rbufT + (long long)nc * nx, 0, sizeof(double) * nx, st()));
        AAO_CUDA_TRY(cudaMemsetAsync(ebuf + (long long)nc * nx, 0, sizeof(double) * nx, st()));
        launch(k_step_set, 1, 1, 0, st(), coarse->stepp, ebuf, (const double*)rbufT, nc - 1);
        for (int c = 1; c <= nc; ++c) {
            AAO_CUDA_TRY(cudaStreamWaitEvent(st(), ev_f1[c - 1], 0));
            const long long zc = (long long)(nt - c * m) * nx, ec = (long long)(nc - c) * nx;
            AAO_CUDA_TRY(cudaMemcpyAsync(rbufT + ec, z + zc, sizeof(double) * nx, cudaMemcpyDeviceToDevice, st()));
            AAO_TRY(coarse->run_steps(1, 0, 1));
            AAO_CUDA_TRY(cudaMemcpyAsync(z + zc, ebuf + ec, sizeof(double) * nx, cudaMemcpyDeviceToDevice, st()));
            AAO_CUDA_TRY(cudaEventRecord(ev_c[c], st()));
        }
        for (int c = 0; c < nc; ++c) {
            Precond* W = work[c % K];
            if (c > 0) AAO_CUDA_TRY(cudaStreamWaitEvent(W->st(), ev_c[c], 0));
            launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, r, nt - c * m - 1);
            AAO_TRY(W->run_steps(1, 0, m - 1));
        }
        if (mg_r > 0) {           // the shorter final interval (the first steps in time)
            Precond* W = work[nc % K];
            AAO_CUDA_TRY(cudaStreamWaitEvent(W->st(), ev_c[nc], 0));
            launch(k_step_set, 1, 1, 0, W->st(), W->stepp, z, r, nt - nc * m - 1);
            AAO_TRY(W->run_steps(1, 0, mg_r));
        }
        for (int w = 0; w < K; ++w) {
            AAO_CUDA_TRY(cudaEventRecord(ev_join[w], wst[w]));
            AAO_CUDA_TRY(cudaStreamWaitEvent(st(), ev_join[w], 0));
        }
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    // Lock-step schedule of the same MGRIT iteration (used when a shifted solve runs on one
    // thread-block cluster: one launch then holds every interval's clusters): F-relaxation as
    // batched steps over the mg_nc intervals from z_0 = w_0 and zero C-points, the C-point
    // residuals, the coarse error recurrence e_c = Phi_c(e_{c-1}) + r_c by substitution with step
    // m tau, the C-point correction z_{cm} += e_c and a final F-relaxation (which also relaxes the
    // shorter last interval when m does not divide nt).  w is in wbuf; z_0 is set by the caller.
    aao_status mgrit_batched_forward(double* z) {
        const long long nx = h->g.nx;
        const int m = mg_m, nc = mg_nc;
        const unsigned nb = (unsigned)(((long long)nc * nx + 255) / 256);
        launch(k_mgrit_cpoints, nb, 256, 0, st(), z, (const double*)nullptr, nx, nc, m, 0, 1, 0, 1);
        launch(k_step_set, 1, 1, 0, st(), stepp, z, (const double*)nullptr, 0);
        AAO_LAUNCH_CHECK();
        AAO_TRY(run_steps(0, 1, m - 1));
        launch(k_step_set, 1, 1, 0, st(), stepp, z, (const double*)nullptr, m - 1);
        AAO_TRY(run_steps(0, 2, 1));
        AAO_CUDA_TRY(cudaMemsetAsync(coarse->wbuf, 0, sizeof(A) * nx, st()));
        AAO_CUDA_TRY(cudaMemsetAsync(ebuf, 0, sizeof(double) * nx, st()));
        launch(k_step_set, 1, 1, 0, st(), coarse->stepp, ebuf, (const double*)nullptr, 0);
        AAO_LAUNCH_CHECK();
        AAO_TRY(coarse->run_steps(0, 0, nc));
        launch(k_mgrit_cpoints, nb, 256, 0, st(), z, (const double*)ebuf, nx, nc, m, 0, 1, 0, 1);
        launch(k_step_set, 1, 1, 0, st(), stepp, z, (const double*)nullptr, 0);
        AAO_LAUNCH_CHECK();
        // the final F-relaxation; its first mg_r steps also relax the shorter final interval from
        // the last C-point
        if (mg_r > 0) AAO_TRY(run_steps(0, 3, mg_r));
        return run_steps(0, 1, m - 1 - mg_r);
    }

    // The same for S_tilde^T's backward recurrence u_nt = r_{v,nt}, u_n = Phi^T(u_{n+1}) + r_{v,n},
    // run forward in reversed time (C-points n = nt - c m).  u_nt is set by the caller.
    aao_status mgrit_batched_transpose(double* z, const double* r) {
        const long long nx = h->g.nx;
        const int m = mg_m, nc = mg_nc, nt = h->nt;
        const unsigned nb = (unsigned)(((long long)nc * nx + 255) / 256);
        launch(k_mgrit_cpoints, nb, 256, 0, st(), z, (const double*)nullptr, nx, nc, m, nt, -1, 0, 1);
        launch(k_step_set, 1, 1, 0, st(), stepp, z, r, nt - 1);
        AAO_LAUNCH_CHECK();
        AAO_TRY(run_steps(1, 1, m - 1));
        launch(k_step_set, 1, 1, 0, st(), stepp, z, r, nt - m);
        AAO_TRY(run_steps(1, 2, 1));
        AAO_CUDA_TRY(cudaMemsetAsync(rbufT + (long long)nc * nx, 0, sizeof(double) * nx, st()));
        AAO_CUDA_TRY(cudaMemsetAsync(ebuf + (long long)nc * nx, 0, sizeof(double) * nx, st()));
        launch(k_step_set, 1, 1, 0, st(), coarse->stepp, ebuf, (const double*)rbufT, nc - 1);
        AAO_LAUNCH_CHECK();
        AAO_TRY(coarse->run_steps(1, 0, nc));
        launch(k_mgrit_cpoints, nb, 256, 0, st(), z, (const double*)ebuf, nx, nc, m, nt, -1, nc, -1);
        launch(k_step_set, 1, 1, 0, st(), stepp, z, r, nt - 1);
        AAO_LAUNCH_CHECK();
        if (mg_r > 0) AAO_TRY(run_steps(1, 3, mg_r));
        return run_steps(1, 1, m - 1 - mg_r);
    }

    aao_status mgrit_forward(double* z) { return nwork ? mgrit_dataflow_forward(z) : mgrit_batched_forward(z); }
    aao_status mgrit_transpose(double* z, const double* r) {
        return nwork ? mgrit_dataflow_transpose(z, r) : mgrit_batched_transpose(z, r);
    }

    aao_status apply(const double* r, double* z, int transpose) override {
        const Geo& g = h->g;
        const int s = h->s, nt = h->nt;
        const long long nx = g.nx, nv = h->nv, item = (long long)s * nx;
        cudaEventRecord(e0, st());
        if (!transpose) {
            {
                NvtxRange range_("aao.precond.theta_phase");
                AAO_TRY(inner<double>(nt, r + nv, item, z + nv, item, 0));
            }
            cudaEventRecord(e1, st());
            long long tot = (nt + 1) * nx;
            if (h->q1) {
                // g = r_v - Psi_1 z_V with M, then w = M^{-1} g, z_{v,0} = w_0
                const PtMap pm = ptmap(g.n0);
                launch(k_schur_g_q1<A>, pt_grid(pm, g.R, nt + 1), pt_block(pm), 0, st(), g, pm, nt,
                       s, r, (const double*)(z + nv), (const double*)h->d_b, h->tau, sopA.q, wbuf);
                AAO_TRY(mass_inverse(wbuf, nt + 1));
                launch(k_convert<A, double>, (unsigned)((nx + 255) / 256), 256, 0, st(), (const A*)wbuf, z, nx);
            } else {
                launch(k_schur_g<A>, (unsigned)((tot + 255) / 256), 256, 0, st(), nx, nt, s, r,
                       (const double*)(z + nv), (const double*)h->d_b, h->tau, wbuf, z);
            }
            launch(k_step_set, 1, 1, 0, st(), stepp, z, r, 0);
            AAO_LAUNCH_CHECK();
            {
                NvtxRange range_("aao.precond.schur_sweep");
                AAO_TRY(mg_m > 0 ? mgrit_forward(z) : schur_sweep(0));
            }
            cudaEventRecord(e2, st());
        } else {
            // S_tilde^T: backward substitution, u stored in z's v-part (M = I: z_v = u)
            AAO_CUDA_TRY(cudaMemcpyAsync(z + nt * nx, r + nt * nx, sizeof(double) * nx, cudaMemcpyDeviceToDevice,
                                         st()));
            launch(k_step_set, 1, 1, 0, st(), stepp, z, r, nt - 1);
            AAO_LAUNCH_CHECK();
            {
                NvtxRange range_("aao.precond.schur_sweep_transposed");
                AAO_TRY(mg_m > 0 ? mgrit_transpose(z, r) : schur_sweep(1));
            }
            cudaEventRecord(e1, st());
            long long tot = (long long)nt * item;
            if (h->q1) {
                // z_v = M^{-1} u (Chebyshev in the recurrence precision), then the stage rhs with M
                const long long nvx = (long long)(nt + 1) * nx;
                launch(k_convert<double, A>, (unsigned)((nvx + 255) / 256), 256, 0, st(), (const double*)z, wbuf, nvx);
                AAO_TRY(mass_inverse(wbuf, nt + 1));
                launch(k_convert<A, double>, (unsigned)((nvx + 255) / 256), 256, 0, st(), (const A*)wbuf, z, nvx);
                const PtMap pm = ptmap(g.n0);
                launch(k_schurT_vrhs_q1<A>, pt_grid(pm, g.R, nt), pt_block(pm), 0, st(), g, pm, nt, s,
                       r + nv, (const double*)z, (const double*)h->d_b, h->tau, sopA.q, tV);
            } else {
                launch(k_schurT_vrhs<A>, (unsigned)((tot + 255) / 256), 256, 0, st(), nx, nt, s, r + nv,
                       (const double*)z, (const double*)h->d_b, h->tau, tV);
            }
            AAO_LAUNCH_CHECK();
            {
                NvtxRange range_("aao.precond.theta_phase_transposed");
                AAO_TRY(inner<A>(nt, tV, item, z + nv, item, 1));
            }
            cudaEventRecord(e2, st());
        }
        return AAO_OK;
    }

    void accumulate_times() override {
        float a = 0.f, b = 0.f;
        if (cudaEventElapsedTime(&a, e0, e1) == cudaSuccess && cudaEventElapsedTime(&b, e1, e2) == cudaSuccess) {
            t_theta_ms += a;
            t_schur_ms += b;
        }
        cudaGetLastError();
    }

    // ------------------------------------------------- component entry points
    aao_status shifted_solve(int stage, const double* b, double* x) override {
        const Geo& g = h->g;
        nact = 1;
        launch(k_scale_store<SI, double>, pt_grid(ptmap(g.n0), g.R, 1), pt_block(ptmap(g.n0)), 0, st(), ptmap(g.n0), g.R, 1,
               (const int*)nullptr, b, g.nx,
                                                                             nullptr, 0, mgb, 0,
               (StepPtrs*)nullptr);
        AAO_LAUNCH_CHECK();
        Vec<SI> out = Z0;   // item 0, stage 0 of the first Z basis
        AAO_TRY(mg_solve(stage, 1, nullptr, mgb, out));
        launch(k_load<SI, double>, pt_grid(ptmap(g.n0), g.R, 1), pt_block(ptmap(g.n0)), 0, st(), ptmap(g.n0), g.R, 1, out, x,
               g.nx);
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    aao_status pint_apply(const double* r, double* y, int transpose) override {
        const Geo& g = h->g;
        nact = 1;
        const long long rows = (long long)h->s * g.R;
        launch(k_scale_store<SP, double>, pt_grid(ptmap(g.n0), rows, 1), pt_block(ptmap(g.n0)), 0, st(), ptmap(g.n0),
               (int)rows, 1, (const int*)nullptr, r,
                                                                              (long long)h->s * g.nx, nullptr, 0, V0, 0, (StepPtrs*)nullptr);
        AAO_LAUNCH_CHECK();
        AAO_TRY(rana(1, nullptr, V0, Z0, transpose));
        launch(k_load<SI, double>, pt_grid(ptmap(g.n0), rows, 1), pt_block(ptmap(g.n0)), 0, st(), ptmap(g.n0), (int)rows, 1,
               Z0, y, (long long)h->s * g.nx);
        AAO_LAUNCH_CHECK();
        return AAO_OK;
    }

    aao_status inner_solve(int nblocks, const double* r, double* z, int* its_host) override {
        if (nblocks < 1 || nblocks > Bmax) {
            set_error("inner_solve: nblocks must be in 1..nt");
            return AAO_ERR_ARG;
        }
        const long long item = (long long)h->s * h->g.nx;
        AAO_TRY(inner<double>(nblocks, r, item, z, item, 0));
        if (its_host) {
            AAO_CUDA_TRY(cudaMemcpyAsync(its_host, itsh, sizeof(int) * nblocks, cudaMemcpyDeviceToHost, st()));
            AAO_CUDA_TRY(cudaStreamSynchronize(st()));
        }
        return AAO_OK;
    }

    long long inner_its() override {
        long long v = 0;
        cudaMemcpyAsync(&v, itcount, sizeof(long long), cudaMemcpyDeviceToHost, st());
        cudaStreamSynchronize(st());
        for (int w = 0; w < nwork; ++w) v += work[w]->inner_its();
        return v + (coarse ? coarse->inner_its() : 0);
    }
    void reset_inner_its() override {
        cudaMemsetAsync(itcount, 0, sizeof(long long), st());
        if (coarse) coarse->reset_inner_its();
        for (int w = 0; w < nwork; ++w) work[w]->reset_inner_its();
    }

    int nonfinite_flag() override {
        int v[2] = {0, 0};
        cudaMemcpyAsync(v, nonfin, 2 * sizeof(int), cudaMemcpyDeviceToHost, st());
        cudaStreamSynchronize(st());
        int wf = 0;
        for (int w = 0; w < nwork; ++w) wf |= work[w]->nonfinite_flag();
        return v[0] | v[1] | wf | (coarse ? coarse->nonfinite_flag() : 0);
    }
};

}  // namespace aao
