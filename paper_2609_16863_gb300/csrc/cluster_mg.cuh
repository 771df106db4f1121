// Cluster-resident multigrid for 2D items (the Schur sweep's shifted solves (M + c_i K) x = b, Sec. 5:
// three V-cycles per stage solve).
//
// The V-cycles of one shifted solve are a chain of about 30 dependent grid-wide steps per cycle.  One
// thread-block cluster per item (16 CTAs for single items, 8, 4 or 2 for batches) runs the chain on chip:
//   * every level above the coarsest is split by grid rows over the CTAs; a CTA keeps its rows of x (two
//     ping-pong buffers), b, the stored stencil and the Jacobi weights in shared memory, with H ghost
//     rows on each side and zero columns beside the grid (the Dirichlet boundary);
//   * the level-l partition follows the finest one: coarse row J belongs to the CTA owning fine row
//     2J+1, so restriction and interpolation touch at most one row beyond what they produce for;
//   * the coarsest level (at most a few hundred unknowns) is held whole by every CTA: each CTA
//     restricts its rows into every CTA's copy of b, applies its slice of rows of the dense inverse and
//     stores the results into every CTA's copy of x.
//
// What bounds it is latency and instruction supply.  Measured on 16 CTAs of 512 threads (2.07 GHz): a
// block barrier costs 45 cycles, a cluster barrier 137 without and 521 with its release fence, an exchange
// of edge rows (remote stores, barrier) 790 cycles; a step's own work was 850 cycles even for two
// rows, most of it call and index overhead and instruction fetches.  So:
//   * a step's result is computed on as many ghost rows as its inputs reach (`ext`), and rows are
//     exchanged only when a step has none left: with H = 3 (4 on the finest level, whose iterate
//     enters a cycle nonzero) a level needs two exchanges per cycle, of b after the restriction and of x
//     after the last sweep, instead of five; the redundant rows fit the threads that a step leaves
//     idle.  H = 1 exchanges after every sweep; levels fall back to it where shared memory is short and
//     everywhere in FP64, whose rate (two operations per cycle and SM) makes redundant rows dearer;
//   * the cycle is a program of 8-byte operations laid out by the host (cl_program), run by one loop
//     in which every kind of step is instantiated once: sweeps, zero-guess sweeps and residuals are the
//     same instructions with other coefficients;
//   * what does not change between launches (stencils, weights, faces, the slice of the coarsest
//     inverse) is laid out once per handle as each CTA's shared-memory image, padded rows included, and
//     copied linearly;
//   * a thread keeps one 16-byte vector of columns and walks down consecutive rows with the rows around
//     it in registers; on the finest level (FD, kappa = 1) the modes' constants are folded.  Rows are padded
//     to whole vectors with zeros, so odd widths take the same path.
//
// One launch of three V(2,2)-cycles, one item on 16 CTAs (event-timed; with one ghost row and an exchange after every step ->
// now): FP32 256^2 77.3 -> 69.2 us, 128^2 52.8 -> 46.7, 127 x 95 56.9 -> 46.7, 64^2 38.5 -> 32.9, Q1 80 x 72 51.9 -> 48.7;
// FP64 256^2 331 -> 308 (FP64-bound), 128^2 129 -> 118, 64^2 67.2 -> 62.1, 32^2 44.6 -> 37.5; eight to fifteen items of 256^2
// on 8 CTAs each 97 -> 93.  Deep ghost regions against single ghost rows on this kernel: 256^2 68 against 82, 64^2 FP64
// 60.1 against 60.3.
#pragma once

#include <type_traits>

#include "cluster_plan.h"
#include "mg.cuh"

namespace aao {

// Columns per thread: one 16-byte vector in FP32.  FP64 takes single columns: a step's chain of FP64 operations
// is long, and twice the warps hide twice as much of it.
template <class A> struct ClVec;
template <> struct ClVec<float> {
    using T = float4;
    static constexpr int n = 4;
};
template <> struct ClVec<double> {
    using T = double;
    static constexpr int n = 1;
};

// Plan of one shift (a kernel parameter: every field is read through the constant bank).
template <class SI> struct ClCtx : ClShape {
    using A = typename PT<SI>::A;
    A sigma, c;                           // level 0 (FD): sigma I + c K
    A hx2, hy2;
    A w0, ex, ey;                         // FD, kappa = 1: omega / a_PP; c / hx^2, c / hy^2
    const A* img;                         // C images
    const A* fx;
    const A* fy;
    const SI* sten[kClMaxLevels];
    const float* sten_sc[kClMaxLevels];
    const A* W[kClMaxLevels];             // omega / a_PP of every point (null: w0)
    const A* Dinv;                        // rows of ncp values (dinv_global and the image's source: nc)
};

// One distributed level as a step sees it (shared memory, built once per launch).  Positions are indices
// into the dynamic shared memory: accesses stay in the shared address space with 32-bit arithmetic (as
// pointers held in memory they would be generic, with 64-bit arithmetic and longer latency).
template <class A> struct alignas(16) ClL {
    int nr, a, rest, n0;                  // own rows, the first one, rows from it to the grid's end; columns
    int nvp, per;                         // vectors per row; rows per thread, of the own and ghost rows
    unsigned magicv;
    int H;                                // ghost rows
    int X, xs, ld, kind;                  // (own row 0, column 0) of buffer 0, buffer stride, row stride;
                                          // 0: stored stencil, 1: FD with kappa = 1, 2: FD with faces
    int W, ix, in, cs;                    // weights at (own row 0, column 0) with row stride nvp * VN; x inbox, rows
                                          // per side; stencil's component stride
    int S, fx, fy, far;                   // stencil at (own row 0, column 0), row stride nvp * VN; faces likewise (rows
                                          // of ld | of nvp * VN); 1: ghost rows reach beyond the next CTA
    int prev[kClReach], next[kClReach];   // rows of the CTAs before and after, nearest first (0: none)
    A cf[3][4];                           // kind 1, per mode (cl_fd)
    A mP[3];                              // kind 1, per mode: factor of P
    A sigma, c, hx2, hy2;                 // kind 2 (and kind 1 in 16-bit storage): sigma I + c K
    const void* Sg;                       // stencil in global memory at (own row 0, column 0), component stride cs,
    const float* Ssc;                     // row stride n0 (16-bit: times Ssc[k])
};

__device__ __forceinline__ unsigned cl_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Index of this CTA's cluster in the grid: the batch item the cluster solves.
__device__ __forceinline__ int cl_item() {
    unsigned r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return (int)r;
}

__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Barrier after a step: the cluster's where rows were stored into other CTAs, else the block's.
__device__ __forceinline__ void cl_step_sync(bool remote) {
    if (remote) cl_sync();
    else __syncthreads();
}

template <class A> __device__ __forceinline__ A* cl_sm() {
    extern __shared__ __align__(16) unsigned char cl_smem[];
    return reinterpret_cast<A*>(cl_smem);
}

// Stores into CTA `rank` of the cluster at index p of its dynamic shared memory: one value, one vector.
template <class A> __device__ __forceinline__ unsigned cl_remote(int p, int rank) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(cl_sm<A>() + p);
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(d), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_rstore(int p, int rank, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cl_remote<float>(p, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_rstore(int p, int rank, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cl_remote<double>(p, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_rvstore(int p, int rank, const float* v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(cl_remote<float>(p, rank)), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
}
__device__ __forceinline__ void cl_rvstore(int p, int rank, const double* v) {
    cl_rstore(p, rank, v[0]);
}

// p / d for magic = ceil(2^32 / d), d >= 2
__device__ __forceinline__ int cl_div(int p, unsigned magic) { return (int)__umulhi((unsigned)p, magic); }

template <class A>
__device__ __forceinline__ void cl_vload(const A* p, A* out) {
    using VT = typename ClVec<A>::T;
    const VT v = *reinterpret_cast<const VT*>(p);
    const A* q = reinterpret_cast<const A*>(&v);
#pragma unroll
    for (int t = 0; t < ClVec<A>::n; ++t) out[t] = q[t];
}

template <class A>
__device__ __forceinline__ void cl_vstore(A* p, const A* in) {
    using VT = typename ClVec<A>::T;
    VT v;
    A* q = reinterpret_cast<A*>(&v);
#pragma unroll
    for (int t = 0; t < ClVec<A>::n; ++t) q[t] = in[t];
    *reinterpret_cast<VT*>(p) = v;
}

// Store the vector at (own row lr, column c) into the ghost rows (depth rows) of the CTAs that need it:
// into buffer k, or (inbox) into their x inbox.
template <class A>
__device__ __forceinline__ void cl_push(const ClL<A>& v, int rank, int k, int lr, int c, const A* out, int depth,
                                        bool inbox) {
    const int at = (inbox ? v.in + v.ix * v.ld : v.X + k * v.xs) + lr * v.ld + c, ld = v.ld;
    if (lr < depth && v.prev[0] > 0) {
        // beyond the end of the CTA before
        cl_rvstore(at + (inbox ? 0 : v.prev[0] * ld), rank - 1, out);
        if (v.far) {
            int between = v.prev[0];
#pragma unroll
            for (int q = 1; q < kClReach; ++q) {
                if (lr >= depth - between || v.prev[q] == 0) break;
                cl_rvstore(at + (inbox ? between : between + v.prev[q]) * ld, rank - 1 - q, out);
                between += v.prev[q];
            }
        }
    }
    if (lr >= v.nr - depth && v.next[0] > 0) {
        // before the first row of the CTA after
        cl_rvstore(at - v.nr * ld, rank + 1, out);
        if (v.far) {
            int between = v.next[0];
#pragma unroll
            for (int q = 1; q < kClReach; ++q) {
                if (lr < v.nr - depth + between || v.next[q] == 0) break;
                cl_rvstore(at - (v.nr + between) * ld, rank + 1 + q, out);
                between += v.next[q];
            }
        }
    }
}

// This thread's column vector of the level and its consecutive rows of [lo, hi): own and ghost rows are dealt
// out once per level, per rows to a thread.
struct ClRows {
    int c, r0, r1;
};
template <class A>
__device__ __forceinline__ ClRows cl_rows(const ClL<A>& v, int lo, int hi) {
    const int tid = threadIdx.x;
    const int g = cl_div(tid, v.magicv), r = g * v.per - v.H;
    ClRows q;
    q.c = (tid - g * v.nvp) * ClVec<A>::n;
    q.r0 = max(r, lo);
    q.r1 = min(r + v.per, hi);
    return q;
}

// One point of a step with the FD operator, kappa = 1 (P, its neighbours and b).
// FP64: kw (b - (P + ex (2 P - W - E) + ey (2 P - S - N))) + (P or 0).  (Folding the constants further, into
// k0 P + kx (W + E) + ky (S + N) + w b, takes six operations, but makes the residual of a smooth x
// five to thirteen times and a sweep's result up to three times less accurate; subtracting the terms from b one by
// one shortens the chain, but rounds three times at b's size.)
// FP32 takes the differences P - W, ..., which are exact for smooth fields, so the residual's
// cancellation costs no digits: kw (b - (kP P + ex (...) + ey (...))) + mP P.  16-bit storage takes
// the level kernels' formula operation by operation: its results are rounded to the storage format, and the
// roundings are pinned.
template <bool SCALED>
__device__ __forceinline__ double cl_fd(const ClL<double>&, const double* cf, double, int mode, double b, double P, double W,
                                        double E, double S, double N) {
    const double dx = 2.0 * P - W - E, dy = 2.0 * P - S - N;
    double s = P;                         // sigma = 1
    s += cf[2] * dx;
    s += cf[3] * dy;
    return cf[0] * (b - s) + (mode == 0 ? P : 0.0);
}
template <bool SCALED>
__device__ __forceinline__ float cl_fd(const ClL<float>& v, const float* cf, float mP, int mode, float b, float P, float W,
                                       float E, float S, float N) {
    if constexpr (SCALED) {
        if (mode == 1) return cf[0] * b;
        const float K = v.hx2 * (2.f * P - W - E) + v.hy2 * (2.f * P - S - N);
        const float res = b - (v.sigma * P + v.c * K);
        return mode == 2 ? res : P + cf[0] * res;
    } else {
        float s = cf[1] * P;
        s += cf[2] * ((P - W) + (P - E));
        s += cf[3] * ((P - S) + (P - N));
        return cf[0] * (b - s) + mP * P;
    }
}

// One step of a level on own rows and ext ghost rows per side, from buffer kin (x) and b into buffer
// kout.  mode 0: damped Jacobi x + w (b - A x); 1: the same from x = 0 (w b); 2: the residual b - A x; 3 (FD,
// kappa = 1, kin = 2): two sweeps from x = 0, whose first is w0 b.  The modes are coefficients of one formula
// (mode 1 reads no x: zeros take its place).  depth > 0: also store the own edge rows into the other CTAs.
template <class SI, bool FACES, bool GLOBAL, class A>
__device__ __forceinline__ void cl_step(const ClL<A>& v, int rank, int mode, int kin, int kout, int ext, int depth,
                                        bool inbox) {
    constexpr int VN = ClVec<A>::n;
    A* const sm = cl_sm<A>();
    const ClRows q = cl_rows(v, max(-ext, -v.a), min(v.nr + ext, v.rest));
    if (q.r0 >= q.r1) return;
    const int ld = v.ld, c = q.c;
    const int nvalid = v.n0 - c;                  // columns from here on (below VN in a ragged last vector)
    const int at = v.X + q.r0 * ld + c;
    const A* xm = sm + at + kin * v.xs;
    const A* bm = sm + at + 2 * v.xs;
    A* om = sm + at + kout * v.xs;
    A S[VN], P[VN], N[VN];
#pragma unroll
    for (int i = 0; i < VN; ++i) S[i] = P[i] = N[i] = A(0);
    const bool ax = mode != 1;
    if (ax) {
        cl_vload(xm - ld, S);
        cl_vload(xm, P);
    }
    auto finish = [&](int lr, A* out) {
        if (VN > 1 && nvalid < VN) {
#pragma unroll
            for (int i = 0; i < VN; ++i)
                if (i >= nvalid) out[i] = A(0);
        }
        cl_vstore(om, out);
        if (depth > 0 && lr >= 0 && lr < v.nr) cl_push(v, rank, kout, lr, c, out, depth, inbox);
        om += ld;
        xm += ld;
        bm += ld;
#pragma unroll
        for (int i = 0; i < VN; ++i) {
            S[i] = P[i];
            P[i] = N[i];
        }
    };
    if (v.kind == 1) {
        A cf[4];
        const int m = mode == 3 ? 0 : mode;
#pragma unroll
        for (int i = 0; i < 4; ++i) cf[i] = v.cf[m][i];
        const A mP = v.mP[m];
        // mode 3: a sweep from w0 b, rounded as the first of the two sweeps would store it (a loop of its own: products
        // that the other modes skip would still take their turns of the FP64 pipe)
        auto rows = [&](auto from_b) {
            constexpr bool kFromB = decltype(from_b)::value;
            auto times = [&](A* x) {
#pragma unroll
                for (int i = 0; i < VN; ++i) x[i] *= cf[0];
            };
            if constexpr (kFromB) {
                times(S);
                times(P);
            }
#pragma unroll 1
            for (int r = q.r0; r < q.r1; ++r) {
                A b[VN], out[VN], l = A(0), e = A(0);
                cl_vload(bm, b);
                if (ax) {
                    cl_vload(xm + ld, N);
                    l = xm[-1];
                    e = xm[VN];
                    if constexpr (kFromB) {
                        times(N);
                        l *= cf[0];
                        e *= cf[0];
                    }
                }
#pragma unroll
                for (int i = 0; i < VN; ++i) {
                    const A W = i == 0 ? l : P[i - 1], E = i == VN - 1 ? e : P[i + 1];
                    out[i] = cl_fd<PT<SI>::scaled>(v, cf, mP, m, b[i], P[i], W, E, S[i], N[i]);
                }
                finish(r, out);
            }
        };
        if constexpr (!PT<SI>::scaled) {              // (16-bit storage's programs have no mode 3)
            if (mode == 3) {
                rows(std::true_type{});
                return;
            }
        }
        rows(std::false_type{});
        return;
    }
    const int wrow = v.nvp * VN;
    const A* wm = sm + v.W + q.r0 * wrow + c;
    const bool addx = mode == 0;
    if (FACES && v.kind == 2) {
        const A sigma = v.sigma, cK = v.c;
        const A* fx = sm + v.fx + q.r0 * ld + c;
        const A* fy = sm + v.fy + q.r0 * wrow + c;
#pragma unroll 1
        for (int r = q.r0; r < q.r1; ++r) {
            A b[VN], w[VN], out[VN];
            cl_vload(bm, b);
            cl_vload(wm, w);
            if (ax) {
                A f0[VN], s0[VN], s1[VN];
                cl_vload(xm + ld, N);
                cl_vload(fx, f0);
                const A f4 = fx[VN];
                cl_vload(fy, s0);
                cl_vload(fy + wrow, s1);
                const A l = xm[-1], e = xm[VN];
#pragma unroll
                for (int i = 0; i < VN; ++i) {
                    const A W = i == 0 ? l : P[i - 1], E = i == VN - 1 ? e : P[i + 1];
                    const A fE = i == VN - 1 ? f4 : f0[i + 1];
                    const A K = f0[i] * (P[i] - W) + fE * (P[i] - E) + s0[i] * (P[i] - S[i]) + s1[i] * (P[i] - N[i]);
                    b[i] -= sigma * P[i] + cK * K;
                }
            }
#pragma unroll
            for (int i = 0; i < VN; ++i) out[i] = (mode == 2 ? A(1) : w[i]) * b[i] + (addx ? P[i] : A(0));
            fx += ld;
            fy += wrow;
            wm += wrow;
            finish(r, out);
        }
        return;
    }
    // stored 9-point stencil: components (dx + 1) + 3 (dy + 1)
    A sl = A(0), sr = A(0), pl = A(0), pr = A(0), nl = A(0), nr = A(0);
    if (ax) {
        sl = xm[-ld - 1];
        sr = xm[-ld + VN];
        pl = xm[-1];
        pr = xm[VN];
    }
    const int cs = v.cs;
    const A* Sm = sm + v.S + q.r0 * wrow + c;
    const SI* Gm = reinterpret_cast<const SI*>(v.Sg) + q.r0 * v.n0 + c;
    const bool global = GLOBAL && v.Sg != nullptr;
#pragma unroll 1
    for (int r = q.r0; r < q.r1; ++r) {
        A b[VN], w[VN], out[VN];
        cl_vload(bm, b);
        cl_vload(wm, w);
        if (ax) {
            A K[9][VN];
            cl_vload(xm + ld, N);
            nl = xm[ld - 1];
            nr = xm[ld + VN];
            if (global) {
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    if constexpr (std::is_same<SI, A>::value) {
                        cl_vload(Gm + (long long)k * cs, K[k]);
                    } else {
                        // 16-bit storage: VN values (8 bytes) per component, times its scale
                        const uint2 raw = *reinterpret_cast<const uint2*>(Gm + (long long)k * cs);
                        const SI* e = reinterpret_cast<const SI*>(&raw);
#pragma unroll
                        for (int i = 0; i < VN; ++i) K[k][i] = PT<SI>::ld(e[i]) * v.Ssc[k];
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < 9; ++k) cl_vload(Sm + k * cs, K[k]);
            }
#pragma unroll
            for (int i = 0; i < VN; ++i) {
                // in the level kernels' order: a smooth x cancels late in the sum, where three chains, one per row, would
                // round larger partial sums (residual off by a third more) and take three operations more
                A acc = A(0);
                acc += K[0][i] * (i == 0 ? sl : S[i - 1]);
                acc += K[1][i] * S[i];
                acc += K[2][i] * (i == VN - 1 ? sr : S[i + 1]);
                acc += K[3][i] * (i == 0 ? pl : P[i - 1]);
                acc += K[4][i] * P[i];
                acc += K[5][i] * (i == VN - 1 ? pr : P[i + 1]);
                acc += K[6][i] * (i == 0 ? nl : N[i - 1]);
                acc += K[7][i] * N[i];
                acc += K[8][i] * (i == VN - 1 ? nr : N[i + 1]);
                b[i] -= acc;
            }
        }
        Gm += v.n0;
        Sm += wrow;
#pragma unroll
        for (int i = 0; i < VN; ++i) out[i] = (mode == 2 ? A(1) : w[i]) * b[i] + (addx ? P[i] : A(0));
        wm += wrow;
        finish(r, out);
        sl = pl;
        sr = pr;
        pl = nl;
        pr = nr;
    }
}

// b_c = P^T r (buffer kr of the fine level f) on the own rows of the distributed coarse level v, and
// (kx >= 0) its first sweep w b_c into buffer kx; both stored into the other CTAs' ghost rows too.
template <bool SCALED, class A>
__device__ __forceinline__ void cl_restrict(const ClL<A>& f, const ClL<A>& v, int rank, int kr, int kx) {
    constexpr int VN = ClVec<A>::n;
    A* const sm = cl_sm<A>();
    const ClRows q = cl_rows(v, 0, v.nr);
    const int nvalid = v.n0 - q.c, ld = f.ld;
    const A* row = sm + f.X + kr * f.xs + (2 * (v.a + q.r0) - f.a) * ld + 2 * q.c;    // fine row 2J (0-based) of three
    const int om = v.X + q.r0 * v.ld + q.c;
    const A* wm = sm + v.W + q.r0 * v.nvp * VN + q.c;
    int step = 0;
#pragma unroll 1
    for (int r = q.r0; r < q.r1; ++r) {
        A x[3][2 * VN + 1], out[VN];
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
            if constexpr (VN > 1) {
                cl_vload(row + dy * ld, x[dy]);
                cl_vload(row + dy * ld + VN, x[dy] + VN);
            } else {
                x[dy][0] = row[dy * ld];
                x[dy][1] = row[dy * ld + 1];
            }
            x[dy][2 * VN] = row[dy * ld + 2 * VN];
        }
        if constexpr (SCALED) {
#pragma unroll
            for (int i = 0; i < VN; ++i) out[i] = A(0);
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const A wy = dy == 1 ? A(1) : A(0.5);
#pragma unroll
                for (int i = 0; i < VN; ++i) {
                    out[i] += A(0.5) * wy * x[dy][2 * i];
                    out[i] += wy * x[dy][2 * i + 1];
                    out[i] += A(0.5) * wy * x[dy][2 * i + 2];
                }
            }
        } else {
            // weights 1/4, 1/2, 1/4 of the outer rows, twice that of the middle one
            A s[2 * VN + 1];
#pragma unroll
            for (int i = 0; i <= 2 * VN; ++i) s[i] = x[1][i] + A(0.5) * (x[0][i] + x[2][i]);
#pragma unroll
            for (int i = 0; i < VN; ++i) out[i] = s[2 * i + 1] + A(0.5) * (s[2 * i] + s[2 * i + 2]);
        }
        if (VN > 1 && nvalid < VN) {
#pragma unroll
            for (int i = 0; i < VN; ++i)
                if (i >= nvalid) out[i] = A(0);
        }
        cl_vstore(sm + om + 2 * v.xs + step * v.ld, out);
        cl_push(v, rank, 2, r, q.c, out, v.H, false);
        if (kx >= 0) {
            A w[VN];
            cl_vload(wm + step * v.nvp * VN, w);
#pragma unroll
            for (int i = 0; i < VN; ++i) out[i] *= w[i];
            cl_vstore(sm + om + kx * v.xs + step * v.ld, out);
            cl_push(v, rank, kx, r, q.c, out, v.H, false);
        }
        row += 2 * ld;
        ++step;
    }
}

// 1D interpolation of fine index F: injection from coarse j0, or the average of j0 and j1
// (index -1 or nc: the zero ghost row / column at the boundary).
__device__ __forceinline__ void cl_interp(int F, int& j0, int& j1, bool& inj) {
    const int g = F + 1;                 // 1-based; coarse j sits at fine 2(j+1)
    inj = (g & 1) == 0;
    if (inj) {
        j0 = g / 2 - 1;
        j1 = j0;
    } else {
        j0 = (g - 1) / 2 - 1;
        j1 = (g + 1) / 2 - 1;
    }
}

// x_f (buffer kx) += P x_c (buffer kc of the coarse level, its inbox beyond the own rows) on own rows and ext
// ghost rows, in place.  A vector starts at an even column c: its points average coarse columns
// c/2 - 1, c/2 and take c/2 in turn.  depth > 0: the last step of the level, stored into the inboxes.
template <bool SCALED, class A>
__device__ __forceinline__ void cl_prolong(const ClL<A>& f, const ClL<A>& v, int rank, int kx, int kc, int ext, int depth) {
    constexpr int VN = ClVec<A>::n;
    A* const sm = cl_sm<A>();
    const ClRows q = cl_rows(f, max(-ext, -f.a), min(f.nr + ext, f.rest));
    const int nvalid = f.n0 - q.c, ldc = v.ld;
    // row y of x_c: own rows in buffer kc, the others in the inbox (the coarsest level: all in the buffer)
    const int xc = v.X + kc * v.xs + (q.c >> 1), in = v.in + (q.c >> 1) + v.ix * ldc, ac = v.a, nc = v.nr, ix = v.ix;
    auto at = [&](int y) {
        const int lr = y - ac;
        if (ix == 0 || (lr >= 0 && lr < nc)) return xc + lr * ldc;
        return in + (lr < 0 ? lr : lr - nc) * ldc;
    };
    A* x = sm + f.X + kx * f.xs + q.r0 * f.ld + q.c;
#pragma unroll 1
    for (int r = q.r0; r < q.r1; ++r) {
        int y0, y1;
        bool yi;
        cl_interp(f.a + r, y0, y1, yi);
        const A* p0 = sm + at(y0);
        const A* p1 = sm + at(y1);
        A out[VN], m[VN / 2 + 2];
        cl_vload(x, out);
        if constexpr (VN == 1) {
            // column c averages coarse columns c/2 - 1 and c/2, or (c odd) takes c/2
            const int o = (q.c & 1) - 1;
            const A s0 = p0[o] + p1[o], s1 = p0[0] + p1[0];
            out[0] += A(0.25) * (s0 + s1);
        } else if constexpr (SCALED) {
            const A wy = yi ? A(1) : A(0.5);
#pragma unroll
            for (int i = 0; i < VN; ++i) {
                const bool xi = i & 1;
                const int x0 = xi ? i / 2 : i / 2 - 1, x1 = i / 2;
                const A wx = xi ? A(1) : A(0.5);
                const A w00 = wy * wx, w01 = xi ? A(0) : w00, w10 = yi ? A(0) : w00, w11 = (xi || yi) ? A(0) : w00;
                out[i] += w00 * p0[x0];
                out[i] += w01 * p0[x1];
                out[i] += w10 * p1[x0];
                out[i] += w11 * p1[x1];
            }
        } else {
            // the coarse row of this fine row: injected (y0 = y1) or the average of two
#pragma unroll
            for (int i = 0; i <= VN / 2; ++i) m[i] = A(0.5) * (p0[i - 1] + p1[i - 1]);
#pragma unroll
            for (int i = 0; i < VN / 2; ++i) {
                out[2 * i] += A(0.5) * (m[i] + m[i + 1]);
                out[2 * i + 1] += m[i + 1];
            }
        }
        if (VN > 1 && nvalid < VN) {
#pragma unroll
            for (int i = 0; i < VN; ++i)
                if (i >= nvalid) out[i] = A(0);
        }
        cl_vstore(x, out);
        if (depth > 0 && r >= 0 && r < f.nr) cl_push(f, rank, kx, r, q.c, out, depth, true);
        x += f.ld;
    }
}

// Asynchronous copies global -> shared of one value and of 16 bytes (aligned).
template <class A> __device__ __forceinline__ void cp_async1(A* smem_dst, const A* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    if constexpr (sizeof(A) == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem_src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}

// The staged constants of CTA blockIdx.x (a plan's images are laid out once per handle): stencils, weights
// and faces on own and ghost rows, padded to whole vectors with zeros, and the CTA's rows of the coarsest
// inverse, and the program (nprog operations).
template <class SI>
__global__ void __launch_bounds__(kBlock) k_cluster_image(const __grid_constant__ ClCtx<SI> t, typename PT<SI>::A* imgs,
                                                          const ClOp* prog, int nprog) {
    pdl_prologue();
    using A = typename PT<SI>::A;
    constexpr int VN = ClVec<A>::n;
    const int rank = blockIdx.x, tid = threadIdx.x;
    A* img = imgs + (long long)rank * t.img_len - t.img_off;      // indexed by shared-memory offsets
    for (int p = tid; p < nprog; p += kBlock)
        reinterpret_cast<ClOp*>(reinterpret_cast<char*>(img) + t.prog_off)[p] = prog[p];
    // rows [a - E, a + nr + E) of src(row, col) inside the grid, n columns, at dst (row -E first), stride ss
    auto rows = [&](A* dst, int ss, int l, int E, int extra, int n, auto&& src) {
        const int a = t.rlo[l][rank], nr = t.rlo[l][rank + 1] - a + extra, n1 = t.n1[l] + extra;
        for (int p = tid; p < (nr + 2 * E) * ss; p += kBlock) {
            const int r = p / ss, c = p - r * ss, row = a + r - E;
            dst[p] = c < n && row >= 0 && row < n1 ? src(row, c) : A(0);
        }
    };
    for (int l = 0; l < t.T; ++l) {
        const int np = t.nvp[l] * VN, n0 = t.n0[l], H = t.H[l];
        if (t.woff[l] >= 0)
            rows(img + t.woff[l], np, l, H, 0, n0, [&](int r, int c) { return t.W[l][(long long)r * n0 + c]; });
        if (t.soff[l] >= 0)
            for (int k = 0; k < 9; ++k)
                rows(img + t.soff[l] + k * (t.maxr[l] + 2 * (H - 1)) * np, np, l, H - 1, 0, n0, [&](int r, int c) {
                    A v = PT<SI>::ld(t.sten[l][(long long)k * n0 * t.n1[l] + (long long)r * n0 + c]);
                    if constexpr (PT<SI>::scaled) v *= t.sten_sc[l][k];
                    return v;
                });
    }
    if (t.has_faces) {
        const int n0 = t.n0[0], np = t.nvp[0] * VN, E = t.H[0] - 1;
        rows(img + t.fxoff, np + 2 * kClPad, 0, E, 0, n0 + 1, [&](int r, int c) { return t.fx[(long long)r * (n0 + 1) + c]; });
        rows(img + t.fyoff, np, 0, E, 1, n0, [&](int r, int c) { return t.fy[(long long)r * n0 + c]; });
    }
    if (!t.dinv_global) {
        const int nc = t.n0[t.T] * t.n1[t.T], m = (t.cs[rank + 1] - t.cs[rank]) * t.ncp;
        for (int p = tid; p < m; p += kBlock) {
            const int r = p / t.ncp, c = p - r * t.ncp;
            img[t.dinv_off + p] = c < nc ? t.Dinv[(long long)(t.cs[rank] + r) * nc + c] : A(0);
        }
    }
}

// All mg_cycles V-cycles of (M + c K) x = b, b and x in global memory: cluster k of the grid solves
// batch item k (grid = C x items CTAs; clusters never wait on one another).
template <class SI, bool FACES, bool GLOBAL>
__global__ void __launch_bounds__(kClThreads, 1) k_cluster_mg(const __grid_constant__ ClCtx<SI> t, const int* active,
                                                              Vec<SI> bv, Vec<SI> xout) {
    pdl_prologue();
    using A = typename PT<SI>::A;
    constexpr int VN = ClVec<A>::n;
    constexpr bool kSame = std::is_same<SI, A>::value;
    __shared__ ClL<A> lev[kClMaxLevels];
    A* const sm = cl_sm<A>();
    const int item = cl_item();               // one cluster per batch item
    if (active && !active[item]) return;      // the same decision in every CTA of the cluster
    const int tid = threadIdx.x, nthr = kClThreads;
    const int rank = (int)cl_rank();
    const int C = t.C, L = t.L, T = t.T;
    // ---- the constants' image
    {
        const A* src = t.img + (long long)rank * t.img_len;
        constexpr int N16 = 16 / (int)sizeof(A);
        for (int p = tid * N16; p < t.img_len; p += nthr * N16) cp_async16(sm + t.img_off + p, src + p);
    }
    // ---- b on own and ghost rows (rows beyond the grid and padding columns are zero)
    {
        const int a = t.rlo[0][rank], nr = t.rlo[0][rank + 1] - a, H = t.H[0], n0 = t.n0[0], n1 = t.n1[0];
        const int nvp = t.nvp[0], ld = nvp * VN + 2 * kClPad;
        A* B = sm + t.off[0] + 2 * (t.maxr[0] + 2 * H) * ld + kClPad;
        const A* src = reinterpret_cast<const A*>(bv.d) + (long long)item * bv.bs;
        View<SI> bs = view_of(bv, item, 0, n0);
        const bool vec = kSame && sizeof(A) == 4 && n0 % VN == 0 && (reinterpret_cast<unsigned long long>(src) & 15ULL) == 0;
        for (int i = tid; i < (nr + 2 * H) * nvp; i += nthr) {
            const int r = cl_div(i, t.magicv[0]), c = (i - r * nvp) * VN, row = a + r - H;
            A* d = B + r * ld + c;
            const bool in = row >= 0 && row < n1;
            if (in && vec && c < n0) {      // (rows of n0 = VN columns are padded to two vectors)
                cp_async16(d, src + (long long)row * n0 + c);
                continue;
            }
#pragma unroll
            for (int q = 0; q < VN; ++q) {
                if (!in || c + q >= n0) {
                    d[q] = A(0);
                } else if constexpr (kSame) {
                    cp_async1(d + q, src + (long long)row * n0 + c + q);
                } else {
                    d[q] = bs.at(row, c + q);
                }
            }
        }
        for (int i = tid; i < 2 * (t.maxr[0] + 2 * H); i += nthr)      // columns -1 and beside the last vector
            B[(i >> 1) * ld + ((i & 1) ? nvp * VN : -1)] = A(0);
    }
    // ---- zero x of every level, b of the others, the inboxes (the boundary's ghost rows and columns)
    {
        const A z[VN] = {};
        for (int l = 0; l < L; ++l) {
            const int xs = (t.maxr[l] + 2 * t.H[l]) * (t.nvp[l] * VN + 2 * kClPad);
            for (int p = tid * VN; p < (l == 0 ? 2 : 3) * xs; p += nthr * VN) cl_vstore(sm + t.off[l] + p, z);
            const int in = 2 * t.ix[l] * (t.nvp[l] * VN + 2 * kClPad);
            for (int p = tid * VN; p < in; p += nthr * VN) cl_vstore(sm + t.ioff[l] + p, z);
        }
        for (int p = tid; p < t.ncp; p += nthr) sm[t.boff + p] = A(0);      // the padding stays zero
    }
    // ---- the levels of this CTA
    if (tid < L) {
        const int l = tid;
        ClL<A>& v = lev[l];
        const int np = t.nvp[l] * VN, H = t.H[l];
        v.n0 = t.n0[l];
        v.nvp = t.nvp[l];
        v.ld = np + 2 * kClPad;
        v.H = H;
        v.ix = t.ix[l];
        v.xs = (t.maxr[l] + 2 * H) * v.ld;
        v.magicv = t.magicv[l];
        v.a = l < T ? t.rlo[l][rank] : 0;
        v.nr = l < T ? t.rlo[l][rank + 1] - v.a : t.n1[l];
        v.rest = t.n1[l] - v.a;
        v.per = t.per[l];
        v.X = t.off[l] + H * v.ld + kClPad;
        v.in = t.ioff[l] + kClPad;
        v.W = t.woff[l] + H * np;
        v.kind = l == 0 && t.fine0 ? (t.has_faces ? 2 : 1) : 0;
        v.fx = t.fxoff + (H - 1) * v.ld;
        v.fy = t.fyoff + (H - 1) * np;
        v.S = t.soff[l] + (H - 1) * np;
        v.cs = (t.maxr[l] + 2 * (H - 1)) * np;
        v.Sg = nullptr;
        v.Ssc = nullptr;
        if (l < T && t.sten_global[l]) {
            v.cs = v.n0 * t.n1[l];
            v.Sg = t.sten[l] + (long long)v.a * v.n0;
            v.Ssc = t.sten_sc[l];
        }
        for (int q = 0; q < 3; ++q) {
            v.cf[q][0] = q == 2 ? A(1) : t.w0;
            v.cf[q][1] = q == 1 ? A(0) : t.sigma;
            v.cf[q][2] = q == 1 ? A(0) : t.ex;
            v.cf[q][3] = q == 1 ? A(0) : t.ey;
            v.mP[q] = q == 0 ? A(1) : A(0);
        }
        v.hx2 = t.hx2;
        v.hy2 = t.hy2;
        v.sigma = t.sigma;
        v.c = t.c;
        auto rows = [&](int r) { return l < T && r >= 0 && r < C ? t.rlo[l][r + 1] - t.rlo[l][r] : 0; };
        const int reach = max(H, t.ix[l]);
        for (int q = 0; q < kClReach; ++q) {
            v.prev[q] = rows(rank - 1 - q);
            v.next[q] = rows(rank + 1 + q);
        }
        v.far = (v.prev[0] > 0 && v.prev[0] < reach) || (v.next[0] > 0 && v.next[0] < reach);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    cl_sync();     // every CTA of the cluster is resident and staged before any remote access
    const int nc = t.n0[T] * t.n1[T];
    const ClOp* prog = reinterpret_cast<const ClOp*>(cl_sm<unsigned char>() + t.prog_off);
#pragma unroll 1
    for (int cyc = 0; cyc < t.cycles; ++cyc) {
        const int part = cyc == 0 ? 0 : 2 - (cyc & 1);
        const int end = t.pc[part + 1];
        ClOp next = prog[t.pc[part]];
#pragma unroll 1
        for (int pc = t.pc[part]; pc < end; ++pc) {
            ClOp op = next;
            next = prog[pc + 1];                      // (the program ends with a spare operation)
            const ClL<A>& f = lev[op.lev];
            // the last operation's rows go to no further cycle
            if (pc == end - 1 && cyc == t.cycles - 1) op.depth = op.flags = 0;
            if (op.kind == kClStep) {
                cl_step<SI, FACES, GLOBAL>(f, rank, op.mode, op.kin, op.kc, op.ext, op.depth, (op.flags & 1) != 0);
            } else if (op.kind == kClProlong) {
                cl_prolong<PT<SI>::scaled>(f, lev[op.lev + 1], rank, op.kin, op.kc, op.ext, op.depth);
            } else if (op.kind == kClRestrict) {
                cl_restrict<PT<SI>::scaled>(f, lev[op.lev + 1], rank, op.kin, op.mode ? op.kc : -1);
            } else if (op.kind == kClRestrictLast) {
                // into every CTA's copy of the coarsest b: one value and one destination per thread
                const int n0c = t.n0[T], ja = t.rlo[T][rank], nv = (t.rlo[T][rank + 1] - ja) * n0c;
                for (int i = tid; i < nv * C; i += nthr) {
                    const int p = i / C, dst = i - p * C;
                    const int jr = cl_div(p, t.magic[T]), I = p - jr * n0c, J = ja + jr;
                    const A* row = sm + f.X + op.kin * f.xs + (2 * J - f.a) * f.ld + 2 * I;
                    A acc = A(0);
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        const A wy = dy == 1 ? A(1) : A(0.5);
                        acc += A(0.5) * wy * row[dy * f.ld];
                        acc += wy * row[dy * f.ld + 1];
                        acc += A(0.5) * wy * row[dy * f.ld + 2];
                    }
                    cl_rstore(t.boff + J * n0c + I, dst, acc);
                }
            } else if (op.kind == kClSolve) {
                // this CTA's rows of A_c^{-1} b, eight lanes per row (fewer sums across lanes than a warp per
                // row), stored into every CTA's x
                const A* b = sm + t.boff;
                const int lo = t.cs[rank], hi = t.cs[rank + 1], j = tid & 7, ncp = t.ncp;
                for (int p0 = lo; p0 < hi; p0 += nthr / 8) {
                    const int p = p0 + (tid >> 3);
                    A acc[4] = {A(0), A(0), A(0), A(0)};
                    if (p < hi) {
                        const A* row = t.dinv_global ? t.Dinv + (long long)p * ncp : sm + t.dinv_off + (p - lo) * ncp;
                        if constexpr (VN > 1) {
#pragma unroll 4
                            for (int q = j * VN; q < ncp; q += 8 * VN) {
                                A d[VN], u[VN];
                                cl_vload(row + q, d);
                                cl_vload(b + q, u);
#pragma unroll
                                for (int i = 0; i < VN; ++i) acc[i] += d[i] * u[i];
                            }
                        } else {
                            int q = j;
                            for (; q + 24 < ncp; q += 32)
#pragma unroll
                                for (int i = 0; i < 4; ++i) acc[i] += row[q + 8 * i] * b[q + 8 * i];
                            for (; q < ncp; q += 8) acc[0] += row[q] * b[q];
                        }
                    }
                    A s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    if (p < hi) {
                        const int lr = cl_div(p, t.magic[T]), at = f.X + lr * f.ld + p - lr * f.n0;
                        for (int d = j; d < C; d += 8) cl_rstore(at, d, s);
                    }
                }
            } else if (op.kind == kClInbox) {
                // the previous cycle's x: its ghost rows arrived in the inbox
                const int H = f.H;
                for (int i = tid; i < 2 * H * f.nvp; i += nthr) {
                    const int r = cl_div(i, f.magicv), c = (i - r * f.nvp) * VN;
                    A x[VN];
                    cl_vload(sm + f.in + r * f.ld + c, x);
                    cl_vstore(sm + f.X + op.kin * f.xs + (r < H ? r - H : f.nr + r - H) * f.ld + c, x);
                }
            } else {
                // no sweep on a zero guess: clear x for the interpolation later
                const A z[VN] = {};
                for (int i = tid; i < (f.nr + 2 * f.H) * f.nvp; i += nthr) {
                    const int r = cl_div(i, f.magicv), c = (i - r * f.nvp) * VN;
                    cl_vstore(sm + f.X + op.kin * f.xs + (r - f.H) * f.ld + c, z);
                }
            }
            cl_step_sync((op.flags & 2) != 0);
        }
    }
    // ---- write this CTA's rows of x_0
    {
        const ClL<A>& v = lev[0];
        const int k = t.kfin;
        if constexpr (PT<SI>::scaled) {
            const int w = tid >> 5, lane = tid & 31, nw = nthr >> 5;
            for (int lr = w; lr < v.nr; lr += nw) {
                SI* o;
                float* osc;
                row_store_ptrs(xout, item, 0, v.a + lr, v.n0, o, osc);
                const A* X = sm + v.X + k * v.xs + lr * v.ld;
                row_store<SI>(o, osc, v.n0, lane, [&](int c) -> A { return X[c]; });
            }
        } else {
            SI* o = xout.d + (long long)item * xout.bs + (long long)v.a * v.n0;
            const bool vec = v.n0 % VN == 0;
            for (int i = tid; i < v.nr * v.nvp; i += nthr) {
                const int r = cl_div(i, v.magicv), c = (i - r * v.nvp) * VN;
                if (c >= v.n0) continue;              // a vector of padding columns
                const A* x = sm + v.X + k * v.xs + r * v.ld + c;
                A* d = reinterpret_cast<A*>(o) + r * v.n0 + c;
                if (vec) {
                    A u[VN];
                    cl_vload(x, u);
                    cl_vstore(d, u);
                } else {
#pragma unroll
                    for (int q = 0; q < VN; ++q)
                        if (c + q < v.n0) d[q] = x[q];
                }
            }
        }
    }
}

// omega / a_PP of every point of a level, from its stored stencil or the FD diagonal.
template <class SI>
__global__ void __launch_bounds__(kBlock) k_jacobi_weights(LevelOp<SI> op, typename PT<SI>::A omega,
                                                           typename PT<SI>::A* out) {
    pdl_prologue();
    const long long p = (long long)blockIdx.x * kBlock + threadIdx.x;
    if (p >= op.g.nx) return;
    const int row = (int)(p / op.g.n0), c = (int)(p - (long long)row * op.g.n0);
    out[p] = omega / level_diag(op, row, row, 0, c);
}

}  // namespace aao
