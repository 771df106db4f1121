// Geometric Galerkin multigrid for the shifted operators M + c K (Sec. 5:
// "(M + cK)^{-1} by 3 V-cycles"; the paper's closed AMG is replaced by a
// geometric V-cycle with a fixed definition):
//   coarse points = even fine indices (1-based), N_c = N / 2 per axis;
//   1D interpolation: injection at coarse points, average of the two
//   neighbours at odd points (a Dirichlet neighbour counts 0); P = tensor
//   product, R = P^T, A_c = P^T A P stored as a 3^d-point stencil per point;
//   damped-Jacobi smoothing; dense exact solve at the coarsest level.
// All kernels are row kernels: one warp per (batch item, grid row), lanes
// along x, so a row's per-row scale (16-bit storage) is one warp reduction.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace aao {

// Operator of one level as the kernels see it, arithmetic type A.
template <class S> struct LevelOp {
    using A = typename PT<S>::A;
    Geo g;
    int fine = 1;            // 1: matrix-free sigma*u + c*K u; 0: stored stencil
    A sigma = A(1), c = A(0);
    Faces<A> faces;          // fine level, variable kappa (nullptr = kappa 1)
    const S* sten = nullptr; // coarse: ncoef*nx, component-major
    const float* sten_sc = nullptr;  // coarse, scaled types: one scale per component
    int ncoef = 9;
};

template <class S>
__device__ __forceinline__ typename PT<S>::A sten_coef(const LevelOp<S>& op, int q, long long p) {
    typename PT<S>::A v = PT<S>::ld(op.sten[(long long)q * op.g.nx + p]);
    if constexpr (PT<S>::scaled) v *= op.sten_sc[q];
    return v;
}

// (A u)_P and the diagonal a_PP at column c of row (j,k).
template <class S, class SU>
__device__ __forceinline__ void level_apply(const LevelOp<S>& op, const View<SU>& u, long long row, int j,
                                            int k, int c, typename PT<S>::A& Au,
                                            typename PT<S>::A& diag) {
    using A = typename PT<S>::A;
    const Geo& g = op.g;
    if (op.fine) {
        Au = op.sigma * A(u.at(row, c)) + op.c * A(fd_K(u, g, op.faces, row, j, k, c));
        diag = op.sigma + op.c * fd_K_diag<A>(g, op.faces, row, j, k, c);
        return;
    }
    const long long p = row * g.n0 + c;
    A acc = A(0);
    const int zlo = g.d == 3 ? -1 : 0, zhi = g.d == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz) {
        int kk = k + dz;
        if (kk < 0 || kk >= g.n2) continue;
        for (int dy = -1; dy <= 1; ++dy) {
            int jj = j + dy;
            if (jj < 0 || jj >= g.n1) continue;
            long long rr = row + dy + (long long)dz * g.n1;
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                int cc = c + dx;
                if (cc < 0 || cc >= g.n0) continue;
                int q = (dx + 1) + 3 * (dy + 1) + (g.d == 3 ? 9 * (dz + 1) : 0);
                acc += sten_coef(op, q, p) * A(u.at(rr, cc));
            }
        }
    }
    Au = acc;
    diag = sten_coef(op, g.d == 3 ? 13 : 4, p);
}

// (A u)_P and a_PP for a level whose values come from a getter u(row, col)
// (used by the fused kernels, where u is itself computed on the fly).
template <class S, class G>
__device__ __forceinline__ void level_apply_g(const LevelOp<S>& op, G&& u, long long row, int j, int k, int c,
                                              typename PT<S>::A& Au, typename PT<S>::A& diag) {
    using A = typename PT<S>::A;
    const Geo& g = op.g;
    if (op.fine) {
        A uP = u(row, c);
        A uW = c > 0 ? u(row, c - 1) : A(0);
        A uE = c + 1 < g.n0 ? u(row, c + 1) : A(0);
        A uS = j > 0 ? u(row - 1, c) : A(0);
        A uN = j + 1 < g.n1 ? u(row + 1, c) : A(0);
        A uD = A(0), uU = A(0);
        if (g.d == 3) {
            uD = k > 0 ? u(row - g.n1, c) : A(0);
            uU = k + 1 < g.n2 ? u(row + g.n1, c) : A(0);
        }
        A Ku;
        const Faces<A>& f = op.faces;
        if (f.fx == nullptr) {
            Ku = A(g.hx2) * (A(2) * uP - uW - uE) + A(g.hy2) * (A(2) * uP - uS - uN);
            if (g.d == 3) Ku += A(g.hz2) * (A(2) * uP - uD - uU);
        } else {
            const long long fxi = row * (g.n0 + 1) + c;
            const long long fyi = ((long long)k * (g.n1 + 1) + j) * g.n0 + c;
            Ku = A(f.fx[fxi]) * (uP - uW) + A(f.fx[fxi + 1]) * (uP - uE) + A(f.fy[fyi]) * (uP - uS) +
                 A(f.fy[fyi + g.n0]) * (uP - uN);
            if (g.d == 3) {
                const long long fzi = ((long long)k * g.n1 + j) * g.n0 + c;
                Ku += A(f.fz[fzi]) * (uP - uD) + A(f.fz[fzi + (long long)g.n1 * g.n0]) * (uP - uU);
            }
        }
        Au = op.sigma * uP + op.c * Ku;
        diag = op.sigma + op.c * fd_K_diag<A>(g, op.faces, row, j, k, c);
        return;
    }
    const long long p = row * g.n0 + c;
    A acc = A(0);
    const int zlo = g.d == 3 ? -1 : 0, zhi = g.d == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz) {
        int kk = k + dz;
        if (kk < 0 || kk >= g.n2) continue;
        for (int dy = -1; dy <= 1; ++dy) {
            int jj = j + dy;
            if (jj < 0 || jj >= g.n1) continue;
            long long rr = row + dy + (long long)dz * g.n1;
            for (int dx = -1; dx <= 1; ++dx) {
                int cc = c + dx;
                if (cc < 0 || cc >= g.n0) continue;
                int q = (dx + 1) + 3 * (dy + 1) + (g.d == 3 ? 9 * (dz + 1) : 0);
                acc += sten_coef(op, q, p) * u(rr, cc);
            }
        }
    }
    Au = acc;
    diag = sten_coef(op, g.d == 3 ? 13 : 4, p);
}

template <class S>
__device__ __forceinline__ typename PT<S>::A level_diag(const LevelOp<S>& op, long long row, int j, int k, int c) {
    using A = typename PT<S>::A;
    if (op.fine) return op.sigma + op.c * fd_K_diag<A>(op.g, op.faces, row, j, k, c);
    return sten_coef(op, op.g.d == 3 ? 13 : 4, row * op.g.n0 + c);
}

// Two damped-Jacobi sweeps in one pass: the first sweep is recomputed at the
// point and at its stencil neighbours (x_in.d == nullptr: zero initial guess).
template <class S>
__global__ void __launch_bounds__(kPtMaxThreads) k_smooth2(LevelOp<S> op, PtMap pm, int B, const int* active,
                                                           Vec<S> xin, Vec<S> bv, Vec<S> xout,
                                                           typename PT<S>::A omega) {
    pdl_prologue();
    using A = typename PT<S>::A;
    const Geo g = op.g;
    PtPos q = pt_pos(pm, B, g.R, active);
    if constexpr (!PT<S>::scaled) {
        if (!q.valid) return;
    }
    const long long row = q.row;
    int j, k;
    row_jk(g, row, j, k);
    View<S> bb = view_of(bv, q.b, 0, g.n0);
    const bool has = xin.d != nullptr;
    View<S> xx = has ? view_of(xin, q.b, 0, g.n0) : View<S>{nullptr, nullptr, g.n0};
    auto x1 = [&](long long rr, int cc) -> A {
        int jj, kk;
    row_jk(g, rr, jj, kk);
        if (!has) return omega * bb.at(rr, cc) / level_diag(op, rr, jj, kk, cc);
        A Au, dg;
        level_apply(op, xx, rr, jj, kk, cc, Au, dg);
        return xx.at(rr, cc) + omega * (bb.at(rr, cc) - Au) / dg;
    };
    S* out; float* osc;
    row_store_ptrs(xout, q.b, 0, row, g.n0, out, osc);
    pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int c) -> A {
        A Au, dg;
        level_apply_g(op, x1, row, j, k, c, Au, dg);
        return x1(row, c) + omega * (bb.at(row, c) - Au) / dg;
    });
}

// bc = P^T (b - A x) with the fine residual computed on the fly (coarse rows;
// x.d == nullptr: x = 0, residual = b).
template <class S>
__global__ void __launch_bounds__(kPtMaxThreads) k_resid_restrict(LevelOp<S> op, Geo gc, PtMap pm, int B,
                                                                  const int* active, Vec<S> xv, Vec<S> bv,
                                                                  Vec<S> bcv) {
    pdl_prologue();
    using A = typename PT<S>::A;
    const Geo gf = op.g;
    PtPos q = pt_pos(pm, B, gc.R, active);
    if constexpr (!PT<S>::scaled) {
        if (!q.valid) return;
    }
    const long long row = q.row;
    int J, Kc;
    row_jk(gc, row, J, Kc);
    View<S> bb = view_of(bv, q.b, 0, gf.n0);
    const bool has = xv.d != nullptr;
    View<S> xx = has ? view_of(xv, q.b, 0, gf.n0) : View<S>{nullptr, nullptr, gf.n0};
    S* out; float* osc;
    row_store_ptrs(bcv, q.b, 0, row, gc.n0, out, osc);
    pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int I) -> A {
        A acc = A(0);
        const int zlo = gf.d == 3 ? -1 : 0, zhi = gf.d == 3 ? 1 : 0;
        for (int dz = zlo; dz <= zhi; ++dz) {
            int fk = gf.d == 3 ? 2 * Kc + 1 + dz : 0;
            if (fk < 0 || fk >= gf.n2) continue;
            A wz = dz == 0 ? A(1) : A(0.5);
            for (int dy = -1; dy <= 1; ++dy) {
                int fj = 2 * J + 1 + dy;
                if (fj < 0 || fj >= gf.n1) continue;
                A wy = dy == 0 ? A(1) : A(0.5);
                long long frow = fj + (long long)gf.n1 * fk;
                for (int dx = -1; dx <= 1; ++dx) {
                    int fi = 2 * I + 1 + dx;
                    if (fi < 0 || fi >= gf.n0) continue;
                    A wx = dx == 0 ? A(1) : A(0.5);
                    A r = bb.at(frow, fi);
                    if (has) {
                        A Au, dg;
                        level_apply(op, xx, frow, fj, fk, fi, Au, dg);
                        r -= Au;
                    }
                    acc += wx * wy * wz * r;
                }
            }
        }
        return acc;
    });
}

// Whether offsets into a 3D level's 27 stencil components fit 32 bits (they pass 2^31 from 79.6 million points on).  The kernels
// that load every component of a point at once take such levels only: 64-bit offsets cost the 96^3 BF16 solve 2.9% and
// the 47 x 39 x 43 FP16 one 3.1%.  Larger levels take the kernels whose offsets are 64-bit.
constexpr bool sten32_ok(long long nx) { return 27 * nx <= 2147483647LL; }

// Level kinds known at compile time (fewer registers than the run-time dispatch of level_apply):
// 0 any, 1 matrix-free FD level, 2 stored 9-point (2D), 3 stored 27-point (3D),
// 4: matrix-free FD level in 2D.
inline int level_kind(int fine, int d, long long nx) {
    return fine ? (d == 2 ? 4 : 1) : (d == 2 ? 2 : (sten32_ok(nx) ? 3 : 0));
}

template <int KIND, class S, class SU>
__device__ __forceinline__ void level_apply_k(const LevelOp<S>& op, const View<SU>& u, long long row, int j, int k,
                                              int c, typename PT<S>::A& Au, typename PT<S>::A& diag) {
    using A = typename PT<S>::A;
    const Geo& g = op.g;
    if constexpr (KIND == 1) {
        Au = op.sigma * A(u.at(row, c)) + op.c * A(fd_K(u, g, op.faces, row, j, k, c));
        diag = op.sigma + op.c * fd_K_diag<A>(g, op.faces, row, j, k, c);
    } else if constexpr (KIND == 4) {
        // fd_K / fd_K_diag for d = 2 (same arithmetic, 32-bit indexing within the item)
        const int r = (int)row, n0 = g.n0;
        const A uP = A(u.at(r, c));
        const A uW = c > 0 ? A(u.at(r, c - 1)) : A(0);
        const A uE = c + 1 < n0 ? A(u.at(r, c + 1)) : A(0);
        const A uS = j > 0 ? A(u.at(r - 1, c)) : A(0);
        const A uN = j + 1 < g.n1 ? A(u.at(r + 1, c)) : A(0);
        A K, kd;
        if (op.faces.fx == nullptr) {
            K = A(g.hx2) * (A(2) * uP - uW - uE) + A(g.hy2) * (A(2) * uP - uS - uN);
            kd = A(2) * A(g.hx2) + A(2) * A(g.hy2);
        } else {
            const int fxi = r * (n0 + 1) + c, fyi = j * n0 + c;
            const A fx0 = A(op.faces.fx[fxi]), fx1 = A(op.faces.fx[fxi + 1]);
            const A fy0 = A(op.faces.fy[fyi]), fy1 = A(op.faces.fy[fyi + n0]);
            K = fx0 * (uP - uW) + fx1 * (uP - uE) + fy0 * (uP - uS) + fy1 * (uP - uN);
            kd = fx0 + fx1 + fy0 + fy1;
        }
        Au = op.sigma * uP + op.c * K;
        diag = op.sigma + op.c * kd;
    } else if constexpr (KIND == 2) {
        const long long p = row * g.n0 + c;
        A acc = A(0);
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            const int jj = j + dy;
            if (jj < 0 || jj >= g.n1) continue;
            const long long rr = row + dy;
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const int cc = c + dx;
                if (cc < 0 || cc >= g.n0) continue;
                acc += sten_coef(op, (dx + 1) + 3 * (dy + 1), p) * A(u.at(rr, cc));
            }
        }
        Au = acc;
        diag = sten_coef(op, 4, p);
    } else if constexpr (KIND == 3) {
        // stored 27-point stencil, 32-bit offsets (sten32_ok): every load is issued before the sum (a point outside the
        // grid adds an exact zero where level_apply skips it)
        const unsigned nx = (unsigned)g.nx, p = (unsigned)row * g.n0 + c;
        const bool xm = c > 0, xp = c + 1 < g.n0;
        A v[27];
#pragma unroll
        for (int r = 0; r < 9; ++r) {
            const int dy = r % 3 - 1, dz = r / 3 - 1;
            const bool in = j + dy >= 0 && j + dy < g.n1 && k + dz >= 0 && k + dz < g.n2;
            const int rr = (int)row + dy + dz * g.n1;
            v[3 * r] = in && xm ? A(u.at(rr, c - 1)) : A(0);
            v[3 * r + 1] = in ? A(u.at(rr, c)) : A(0);
            v[3 * r + 2] = in && xp ? A(u.at(rr, c + 1)) : A(0);
        }
        A s[27];
#pragma unroll
        for (int q = 0; q < 27; ++q) {
            s[q] = PT<S>::ld(op.sten[q * nx + p]);
            if constexpr (PT<S>::scaled) s[q] *= op.sten_sc[q];
        }
        A acc = A(0);
#pragma unroll
        for (int q = 0; q < 27; ++q) acc += s[q] * v[q];
        Au = acc;
        diag = s[13];
    } else {
        level_apply(op, u, row, j, k, c, Au, diag);
    }
}

template <int KIND, class S>
__device__ __forceinline__ typename PT<S>::A level_diag_k(const LevelOp<S>& op, long long row, int j, int k, int c) {
    using A = typename PT<S>::A;
    if constexpr (KIND == 1 || KIND == 4) return op.sigma + op.c * fd_K_diag<A>(op.g, op.faces, row, j, k, c);
    else if constexpr (KIND == 2) return sten_coef(op, 4, row * op.g.n0 + c);
    else if constexpr (KIND == 3) return sten_coef(op, 13, row * op.g.n0 + c);
    else return level_diag(op, row, j, k, c);
}

// x_out = x_in + omega D^{-1} (b - A x_in); x_in.d == nullptr means x_in = 0.
template <class S, int KIND = 0>
__global__ void __launch_bounds__(kPtMaxThreads) k_smooth(LevelOp<S> op, PtMap pm, int B, const int* active, Vec<S> xin,
                                                 Vec<S> bv, Vec<S> xout, typename PT<S>::A omega) {
    pdl_prologue();
    using A = typename PT<S>::A;
    const Geo g = op.g;
    PtPos q = pt_pos(pm, B, g.R, active);
    if constexpr (!PT<S>::scaled) {
        if (!q.valid) return;
    }
    const long long row = q.row;
    int j, k;
    row_jk(g, row, j, k);
    View<S> bb = view_of(bv, q.b, 0, g.n0);
    S* out; float* osc;
    row_store_ptrs(xout, q.b, 0, row, g.n0, out, osc);
    if (xin.d == nullptr) {
        pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int c) -> A {
            const A dg = level_diag_k<KIND>(op, row, j, k, c);
            return omega * bb.at(row, c) / dg;
        });
    } else {
        View<S> xx = view_of(xin, q.b, 0, g.n0);
        pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int c) -> A {
            A Au, dg;
            level_apply_k<KIND>(op, xx, row, j, k, c, Au, dg);
            return xx.at(row, c) + omega * (bb.at(row, c) - Au) / dg;
        });
    }
}

// k_smooth for unscaled storage with RPT rows per thread (rows r0, r0 + rpc, ...): all rows'
// values are computed before any store, so their loads are in flight together; fewer, longer CTAs
// for large batches.  One column per thread (n0 <= n0p).
template <class S, int KIND, int RPT>
__global__ void __launch_bounds__(kPtMaxThreads) k_smooth_rows(LevelOp<S> op, PtMap pm, int B, const int* active,
                                                               Vec<S> xin, Vec<S> bv, Vec<S> xout,
                                                               typename PT<S>::A omega) {
    pdl_prologue();
    using A = typename PT<S>::A;
    static_assert(!PT<S>::scaled, "unscaled storage only");
    const Geo g = op.g;
    const int b = blockIdx.y;
    if (b >= B || (active && !active[b])) return;
    const int c = threadIdx.x;
    if (c >= g.n0) return;
    const int r0 = blockIdx.x * pm.rpc * RPT + threadIdx.y;
    View<S> bb = view_of(bv, b, 0, g.n0);
    S* out = xout.d + (long long)b * xout.bs;
    A v[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = r0 + i * pm.rpc;
        v[i] = A(0);
        if (row < g.R) {
            if (xin.d == nullptr) {
                v[i] = omega * bb.at(row, c) / level_diag_k<KIND>(op, row, row, 0, c);
            } else {
                View<S> xx = view_of(xin, b, 0, g.n0);
                A Au, dg;
                level_apply_k<KIND>(op, xx, row, row, 0, c, Au, dg);
                v[i] = xx.at(row, c) + omega * (bb.at(row, c) - Au) / dg;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = r0 + i * pm.rpc;
        if (row < g.R) out[(long long)row * g.n0 + c] = PT<S>::st(v[i]);
    }
}

// ---------------------------------------------------------------------------
// Batched 2D matrix-free level (sigma I + c K, kappa = 1), unscaled storage, streaming form:
// a thread owns V consecutive columns (one 16-byte vector) of a strip of RS rows and keeps the
// rows j-1, j, j+1 of x in registers while it walks down the strip, so each point costs one
// vector load of x, one of b and one store (plus two scalar halo loads per row and two halo
// rows per strip); the next row's loads are issued before the current row is computed.
// MODE 0: damped Jacobi x + (omega / a_PP) (b - A x); MODE 1: the same from x = 0
// ((omega / a_PP) b, x is not read); MODE 2: the residual b - A x.  A x as level_apply_k<4>;
// the Jacobi weight omega / a_PP as the cluster V-cycle.  Block: 256 threads = (n0 / V)
// threads per row x strips; grid (ceil(n1 / (strips RS)), items).
// ---------------------------------------------------------------------------
template <class S> struct Vec16;
template <> struct Vec16<float> {
    using T = float4;
    static constexpr int n = 4;
};
template <> struct Vec16<double> {
    using T = double2;
    static constexpr int n = 2;
};
constexpr int kStripThreads = 256;
constexpr int kStripRows = 8;

template <class S, int MODE>
__global__ void __launch_bounds__(kStripThreads) k_strip2d(LevelOp<S> op, int B, const int* active, Vec<S> xin,
                                                           Vec<S> bv, Vec<S> out, S omega) {
    pdl_prologue();
    static_assert(!PT<S>::scaled, "unscaled storage only");
    using VT = typename Vec16<S>::T;
    constexpr int V = Vec16<S>::n;
    const Geo g = op.g;
    const int b = blockIdx.y;
    if (b >= B || (active && !active[b])) return;
    const int n0 = g.n0, n1 = g.n1;
    const int tpr = n0 / V;
    const int tx = threadIdx.x % tpr, ty = threadIdx.x / tpr;
    const int strips = blockDim.x / tpr;
    if (ty >= strips) return;
    const int j0 = (blockIdx.x * strips + ty) * kStripRows;
    if (j0 >= n1) return;
    const int j1 = j0 + kStripRows < n1 ? j0 + kStripRows : n1;
    const int c0 = tx * V;
    const S* X = MODE == 1 ? nullptr : xin.d + (long long)b * xin.bs;
    const S* Bp = bv.d + (long long)b * bv.bs;
    S* O = out.d + (long long)b * out.bs;
    const S hx2 = S(g.hx2), hy2 = S(g.hy2);
    const S kd = S(2) * hx2 + S(2) * hy2;
    const S wgt = omega / (op.sigma + op.c * kd);      // omega / a_PP, as the cluster V-cycle
    auto load_row = [&](int j, S* dst) {
        if (j >= 0 && j < n1) {
            VT v = *reinterpret_cast<const VT*>(X + (long long)j * n0 + c0);
            const S* q = reinterpret_cast<const S*>(&v);
#pragma unroll
            for (int t = 0; t < V; ++t) dst[t] = q[t];
        } else {
#pragma unroll
            for (int t = 0; t < V; ++t) dst[t] = S(0);
        }
    };
    auto load_b = [&](int j, S* dst) {
        VT v = *reinterpret_cast<const VT*>(Bp + (long long)j * n0 + c0);
        const S* q = reinterpret_cast<const S*>(&v);
#pragma unroll
        for (int t = 0; t < V; ++t) dst[t] = q[t];
    };
    // the loads of row j + 1 are issued before row j is computed (two rows in flight per thread)
    S sr[V], pr[V], nr[V], bq[V], nn[V], bn[V];
    S w = S(0), e = S(0), wn = S(0), en = S(0);
    load_b(j0, bq);
    if (MODE != 1) {
        load_row(j0 - 1, sr);
        load_row(j0, pr);
        load_row(j0 + 1, nr);
        w = c0 > 0 ? X[(long long)j0 * n0 + c0 - 1] : S(0);
        e = c0 + V < n0 ? X[(long long)j0 * n0 + c0 + V] : S(0);
    }
    for (int j = j0; j < j1; ++j) {
        const bool more = j + 1 < j1;
        if (more) {
            load_b(j + 1, bn);
            if (MODE != 1) {
                load_row(j + 2, nn);
                wn = c0 > 0 ? X[(long long)(j + 1) * n0 + c0 - 1] : S(0);
                en = c0 + V < n0 ? X[(long long)(j + 1) * n0 + c0 + V] : S(0);
            }
        }
        S res[V];
        if (MODE == 1) {
#pragma unroll
            for (int t = 0; t < V; ++t) res[t] = wgt * bq[t];
        } else {
#pragma unroll
            for (int t = 0; t < V; ++t) {
                const S uP = pr[t], uW = t == 0 ? w : pr[t - 1], uE = t == V - 1 ? e : pr[t + 1];
                const S K = hx2 * (S(2) * uP - uW - uE) + hy2 * (S(2) * uP - sr[t] - nr[t]);
                const S Au = op.sigma * uP + op.c * K;
                res[t] = MODE == 0 ? uP + wgt * (bq[t] - Au) : bq[t] - Au;
            }
        }
        VT ov;
        S* oq = reinterpret_cast<S*>(&ov);
#pragma unroll
        for (int t = 0; t < V; ++t) oq[t] = res[t];
        *reinterpret_cast<VT*>(O + (long long)j * n0 + c0) = ov;
        if (more) {
#pragma unroll
            for (int t = 0; t < V; ++t) {
                bq[t] = bn[t];
                if (MODE != 1) {
                    sr[t] = pr[t];
                    pr[t] = nr[t];
                    nr[t] = nn[t];
                }
            }
            w = wn;
            e = en;
        }
    }
}

// The same streaming form for a 2D level with a stored 9-point stencil (a coarse Galerkin level;
// unscaled storage): the stencil's 9 component rows are read as 16-byte vectors beside x (the
// stencil is shared by all items, so it stays in L1/L2), the corner and side neighbours of the
// vector come from the three rows in registers plus two scalars per row.  Per point the operations
// of level_apply_k<2> in its order (neighbours beyond the grid read as zero instead of being
// skipped: the same value) and of k_smooth / k_residual: x + omega (b - A x) / a_PP.
template <class S, int MODE>
__global__ void __launch_bounds__(kStripThreads) k_strip2d_st(LevelOp<S> op, int B, const int* active, Vec<S> xin,
                                                              Vec<S> bv, Vec<S> out, S omega, int rs) {
    pdl_prologue();
    static_assert(!PT<S>::scaled, "unscaled storage only");
    using VT = typename Vec16<S>::T;
    constexpr int V = Vec16<S>::n;
    const Geo g = op.g;
    const int b = blockIdx.y;
    if (b >= B || (active && !active[b])) return;
    const int n0 = g.n0, n1 = g.n1;
    const int tpr = n0 / V;
    const int tx = threadIdx.x % tpr, ty = threadIdx.x / tpr;
    const int strips = blockDim.x / tpr;
    if (ty >= strips) return;
    const int j0 = (blockIdx.x * strips + ty) * rs;     // rs rows per strip (strip_st_rows)
    if (j0 >= n1) return;
    const int j1 = j0 + rs < n1 ? j0 + rs : n1;
    const int c0 = tx * V;
    const long long nx = g.nx;
    const S* X = MODE == 1 ? nullptr : xin.d + (long long)b * xin.bs;
    const S* Bp = bv.d + (long long)b * bv.bs;
    S* O = out.d + (long long)b * out.bs;
    auto vld = [&](const S* p, S* dst) {
        VT v = *reinterpret_cast<const VT*>(p);
        const S* q = reinterpret_cast<const S*>(&v);
#pragma unroll
        for (int t = 0; t < V; ++t) dst[t] = q[t];
    };
    // row j of x as V values plus the points left and right of the vector (zeros beyond the grid)
    auto load_row = [&](int j, S* dst, S& l, S& r) {
        if (j >= 0 && j < n1) {
            vld(X + (long long)j * n0 + c0, dst);
            l = c0 > 0 ? X[(long long)j * n0 + c0 - 1] : S(0);
            r = c0 + V < n0 ? X[(long long)j * n0 + c0 + V] : S(0);
        } else {
#pragma unroll
            for (int t = 0; t < V; ++t) dst[t] = S(0);
            l = r = S(0);
        }
    };
    S sr[V], pr[V], nr[V], sl = S(0), srr = S(0), pl = S(0), prr = S(0), nl = S(0), nrr = S(0);
    if (MODE != 1) {
        load_row(j0 - 1, sr, sl, srr);
        load_row(j0, pr, pl, prr);
    }
    for (int j = j0; j < j1; ++j) {
        if (MODE != 1) load_row(j + 1, nr, nl, nrr);
        const long long p = (long long)j * n0 + c0;
        S bq[V], ctr[V], res[V];
        vld(Bp + p, bq);
        vld(op.sten + 4 * nx + p, ctr);
        if (MODE == 1) {
#pragma unroll
            for (int t = 0; t < V; ++t) res[t] = omega * bq[t] / ctr[t];
        } else {
            S st[9][V];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                if (k == 4) {
#pragma unroll
                    for (int t = 0; t < V; ++t) st[4][t] = ctr[t];
                } else {
                    vld(op.sten + (long long)k * nx + p, st[k]);
                }
            }
#pragma unroll
            for (int t = 0; t < V; ++t) {
                const S s0 = t == 0 ? sl : sr[t - 1], s2 = t == V - 1 ? srr : sr[t + 1];
                const S p0 = t == 0 ? pl : pr[t - 1], p2 = t == V - 1 ? prr : pr[t + 1];
                const S n0v = t == 0 ? nl : nr[t - 1], n2 = t == V - 1 ? nrr : nr[t + 1];
                S acc = S(0);
                acc += st[0][t] * s0;
                acc += st[1][t] * sr[t];
                acc += st[2][t] * s2;
                acc += st[3][t] * p0;
                acc += st[4][t] * pr[t];
                acc += st[5][t] * p2;
                acc += st[6][t] * n0v;
                acc += st[7][t] * nr[t];
                acc += st[8][t] * n2;
                res[t] = MODE == 0 ? pr[t] + omega * (bq[t] - acc) / ctr[t] : bq[t] - acc;
            }
        }
        VT ov;
        S* oq = reinterpret_cast<S*>(&ov);
#pragma unroll
        for (int t = 0; t < V; ++t) oq[t] = res[t];
        *reinterpret_cast<VT*>(O + p) = ov;
        if (MODE != 1) {
#pragma unroll
            for (int t = 0; t < V; ++t) {
                sr[t] = pr[t];
                pr[t] = nr[t];
            }
            sl = pl;
            srr = prr;
            pl = nl;
            prr = nrr;
        }
    }
}

// Whether a level takes k_strip2d: 2D matrix-free with kappa = 1, unscaled storage, rows of whole
// 16-byte vectors that tile a 256-thread block, and 16-byte aligned rows.
template <class S>
inline bool strip_ok(const LevelOp<S>& op) {
    if constexpr (PT<S>::scaled) {
        return false;
    } else {
        constexpr int V = Vec16<S>::n;
        const int n0 = op.g.n0;
        return op.fine && op.g.d == 2 && op.faces.fx == nullptr && n0 % V == 0 && n0 / V <= kStripThreads &&
               kStripThreads % (n0 / V) == 0;
    }
}
// Whether a level takes k_strip2d_st: a 2D stored 9-point stencil, unscaled storage, rows of whole
// 16-byte vectors that tile a 256-thread block.
template <class S>
inline bool strip_st_ok(const LevelOp<S>& op) {
    if constexpr (PT<S>::scaled) {
        return false;
    } else {
        constexpr int V = Vec16<S>::n;
        const int n0 = op.g.n0;
        return !op.fine && op.g.d == 2 && op.ncoef == 9 && op.sten != nullptr && n0 % V == 0 &&
               n0 / V <= kStripThreads && kStripThreads % (n0 / V) == 0;
    }
}

// Rows per strip of k_strip2d_st: 8, halved (down to 2) while the batch gives fewer than 1024 blocks,
// so that a coarse level (few rows per item) still spreads over every SM; the shorter strips re-read
// more halo rows, from L1/L2.
template <class S>
inline int strip_st_rows(const LevelOp<S>& op, int B) {
    const int strips = kStripThreads / (op.g.n0 / Vec16<S>::n);
    int rs = kStripRows;
    while (rs > 2 && (long long)B * ((op.g.n1 + strips * rs - 1) / (strips * rs)) < 1024) rs /= 2;
    return rs;
}
template <class S>
inline dim3 strip_st_grid(const LevelOp<S>& op, int B, int rs) {
    const int strips = kStripThreads / (op.g.n0 / Vec16<S>::n);
    return dim3((unsigned)((op.g.n1 + strips * rs - 1) / (strips * rs)), (unsigned)B, 1);
}

template <class S>
inline dim3 strip_grid(const LevelOp<S>& op, int B) {
    const int tpr = op.g.n0 / Vec16<S>::n;
    const int rows_per_block = (kStripThreads / tpr) * kStripRows;
    return dim3((unsigned)((op.g.n1 + rows_per_block - 1) / rows_per_block), (unsigned)B, 1);
}

// ---------------------------------------------------------------------------
// Finest matrix-free level (sigma I + c K, kappa = 1, 2D or 3D) in 16-bit storage with per-row
// scales: a thread owns 8 consecutive columns of a row (one 16-byte vector), the threads of a row
// form a group of gs lanes within one warp (gs = the power of two >= n0 / 8), so the row's scale
// is a shuffle reduction over the group and no block barrier is needed.  MODE 0: damped Jacobi
// x + omega (b - A x) / a_PP; MODE 1: from x = 0; MODE 2: residual b - A x.  Same arithmetic as
// level_apply_k and the same scale rule as pt_store.  Block 256 threads (256 / gs rows); grid
// (ceil(R / rows per block), items).
// ---------------------------------------------------------------------------
constexpr int kVecThreads = 256;

template <class S>
__device__ __forceinline__ void vec8_load(const S* p, float sc, float* out) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const S* q = reinterpret_cast<const S*>(&v);
#pragma unroll
    for (int t = 0; t < 8; ++t) out[t] = PT<S>::ld(q[t]) * sc;
}

template <class S, int MODE>
__global__ void __launch_bounds__(kVecThreads) k_vec16(LevelOp<S> op, int gs, int B, const int* active, Vec<S> xin,
                                                       Vec<S> bv, Vec<S> out, float omega) {
    pdl_prologue();
    static_assert(PT<S>::scaled, "16-bit storage only");
    const Geo g = op.g;
    const int b = blockIdx.y;
    if (b >= B || (active && !active[b])) return;
    const int n0 = g.n0, tpr = n0 / 8;
    const int lane = threadIdx.x & 31, grp = lane / gs, gl = lane - grp * gs;
    const int rows_per_warp = 32 / gs;
    const long long row = ((long long)blockIdx.x * (kVecThreads / 32) + (threadIdx.x >> 5)) * rows_per_warp + grp;
    const bool valid = row < g.R && gl < tpr;       // every lane of a row's group takes part in its reduction
    int j = 0, k = 0;
    if (row < g.R) row_jk(g, row, j, k);
    const int c0 = gl * 8;
    const long long base = (long long)b * bv.bs;    // the same item stride for x, b and out
    const S* X = MODE == 1 ? nullptr : xin.d + (long long)b * xin.bs;
    const float* XS = MODE == 1 ? nullptr : xin.sc + (long long)b * xin.bs / n0;
    const S* Bd = bv.d + base;
    const float* BS = bv.sc + base / n0;
    float res[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) res[t] = 0.f;
    if (valid) {
        const float hx2 = float(g.hx2), hy2 = float(g.hy2), hz2 = float(g.hz2);
        float kd = 2.f * hx2 + 2.f * hy2;
        if (g.d == 3) kd += 2.f * hz2;
        const float dg = float(op.sigma) + float(op.c) * kd;
        float bq[8];
        vec8_load(Bd + row * n0 + c0, BS[row], bq);
        if (MODE == 1) {
#pragma unroll
            for (int t = 0; t < 8; ++t) res[t] = omega * bq[t] / dg;
        } else {
            float P[8], Sv[8], Nv[8], Dv[8], Uv[8];
            vec8_load(X + row * n0 + c0, XS[row], P);
            if (j > 0) vec8_load(X + (row - 1) * n0 + c0, XS[row - 1], Sv);
            else for (int t = 0; t < 8; ++t) Sv[t] = 0.f;
            if (j + 1 < g.n1) vec8_load(X + (row + 1) * n0 + c0, XS[row + 1], Nv);
            else for (int t = 0; t < 8; ++t) Nv[t] = 0.f;
            if (g.d == 3) {
                if (k > 0) vec8_load(X + (row - g.n1) * n0 + c0, XS[row - g.n1], Dv);
                else for (int t = 0; t < 8; ++t) Dv[t] = 0.f;
                if (k + 1 < g.n2) vec8_load(X + (row + g.n1) * n0 + c0, XS[row + g.n1], Uv);
                else for (int t = 0; t < 8; ++t) Uv[t] = 0.f;
            }
            const float w = c0 > 0 ? PT<S>::ld(X[row * n0 + c0 - 1]) * XS[row] : 0.f;
            const float e = c0 + 8 < n0 ? PT<S>::ld(X[row * n0 + c0 + 8]) * XS[row] : 0.f;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float uP = P[t], uW = t == 0 ? w : P[t - 1], uE = t == 7 ? e : P[t + 1];
                float K = hx2 * (2.f * uP - uW - uE) + hy2 * (2.f * uP - Sv[t] - Nv[t]);
                if (g.d == 3) K += hz2 * (2.f * uP - Dv[t] - Uv[t]);
                const float Au = float(op.sigma) * uP + float(op.c) * K;
                res[t] = MODE == 0 ? uP + omega * (bq[t] - Au) / dg : bq[t] - Au;
            }
        }
    }
    // the row's power-of-two scale: maximum over the row's group of lanes
    float m = 0.f;
#pragma unroll
    for (int t = 0; t < 8; ++t) m = fmaxf(m, fabsf(res[t]));
    for (int o = gs >> 1; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    int ex = 0;
    float sc = 1.f, inv = 1.f;
    if (m > 0.f && m <= 3.0e38f) {
        frexpf(m, &ex);
        sc = ldexpf(1.f, ex - 14);
        inv = ldexpf(1.f, 14 - ex);
    }
    if (valid) {
        uint4 ov;
        S* oq = reinterpret_cast<S*>(&ov);
#pragma unroll
        for (int t = 0; t < 8; ++t) oq[t] = PT<S>::st(res[t] * inv);
        *reinterpret_cast<uint4*>(out.d + (long long)b * out.bs + row * n0 + c0) = ov;
        if (gl == 0) out.sc[(long long)b * out.bs / n0 + row] = sc;
    }
}

// Whether a level takes k_vec16: the matrix-free finest level with kappa = 1, 16-bit storage,
// rows of whole 16-byte vectors with at most 32 vectors per row.
template <class S>
inline bool vec16_ok(const LevelOp<S>& op) {
    if constexpr (!PT<S>::scaled) {
        return false;
    } else {
        const int n0 = op.g.n0;
        return op.fine && op.faces.fx == nullptr && n0 % 8 == 0 && n0 / 8 <= 32;
    }
}
inline int vec16_group(int n0) {
    int gs = 1;
    while (gs < n0 / 8) gs <<= 1;
    return gs;
}
template <class S>
inline dim3 vec16_grid(const LevelOp<S>& op, int B) {
    const int rows_per_block = (kVecThreads / 32) * (32 / vec16_group(op.g.n0));
    return dim3((unsigned)((op.g.R + rows_per_block - 1) / rows_per_block), (unsigned)B, 1);
}

// 1D interpolation stencil of fine 0-based index F: up to two coarse indices.
__device__ __forceinline__ int interp_1d(int F, int nc, int* J, float* wt) {
    int g = F + 1;  // 1-based
    if ((g & 1) == 0) {
        J[0] = g / 2 - 1;
        wt[0] = 1.f;
        return 1;
    }
    int m = 0;
    int j1 = (g - 1) / 2 - 1, j2 = (g + 1) / 2 - 1;
    if (j1 >= 0 && j1 < nc) { J[m] = j1; wt[m] = 0.5f; ++m; }
    if (j2 >= 0 && j2 < nc) { J[m] = j2; wt[m] = 0.5f; ++m; }
    return m;
}

// The power-of-two scale of a 16-bit row whose values res[0..N) are held by a group of gs lanes of a warp
// (pt_store's rule); returns its reciprocal.
template <int N> __device__ __forceinline__ float group_scale(const float* res, int gs, float& sc) {
    float m = 0.f;
#pragma unroll
    for (int t = 0; t < N; ++t) m = fmaxf(m, fabsf(res[t]));
    for (int o = gs >> 1; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    int ex = 0;
    sc = 1.f;
    float inv = 1.f;
    if (m > 0.f && m <= 3.0e38f) {
        frexpf(m, &ex);
        sc = ldexpf(1.f, ex - 14);
        inv = ldexpf(1.f, 14 - ex);
    }
    return inv;
}
// Lanes of a row's group: the power of two that holds n0 / N vectors.
inline int row_group(int n0, int N) {
    int gs = 1;
    while (gs < n0 / N) gs <<= 1;
    return gs;
}
template <class S> inline dim3 row_group_grid(const Geo& g, int N, int B) {
    const int rows = (kVecThreads / kWarp) * (kWarp / row_group(g.n0, N));
    return dim3((unsigned)((g.R + rows - 1) / rows), (unsigned)B, 1);
}

// A 3D level with a stored 27-point stencil, FP32 arithmetic: a thread owns 4 consecutive columns of a row, so
// a row of x costs one vector load and two scalars for 12 products and a stencil component one vector load
// for 4; the lanes of a row form a group within a warp for the storage scale.  MODE 0: damped Jacobi; 1: from x =
// 0; 2: residual.  The operations of level_apply_k<3> per point in its order.  Bound by instructions: one
// point per thread spent about 300 per point on addresses, conversions and predicates.
template <class S, int MODE>
__global__ void __launch_bounds__(kVecThreads) k_st27(LevelOp<S> op, int gs, const int* active, Vec<S> xin, Vec<S> bv,
                                                      Vec<S> out, float omega) {
    pdl_prologue();
    constexpr int N = 4;
    constexpr bool SC = PT<S>::scaled;
    using RT = typename std::conditional<sizeof(S) == 2, uint2, uint4>::type;
    __shared__ float ssc[27];
    if (SC) {
        if (threadIdx.x < 27) ssc[threadIdx.x] = op.sten_sc[threadIdx.x];
        __syncthreads();
    }
    const Geo& g = op.g;
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    const int n0 = g.n0, tpr = n0 / N, nx = (int)g.nx;
    const int lane = threadIdx.x & 31, grp = lane / gs, gl = lane - grp * gs;
    const int row = (blockIdx.x * (kVecThreads / 32) + (threadIdx.x >> 5)) * (32 / gs) + grp;
    const bool valid = row < g.R && gl < tpr;
    const int c = gl * N;
    float res[N] = {0.f, 0.f, 0.f, 0.f};
    auto ld4 = [](const S* p, float* v) {
        const RT r = *reinterpret_cast<const RT*>(p);
        const S* e = reinterpret_cast<const S*>(&r);
#pragma unroll
        for (int t = 0; t < N; ++t) v[t] = PT<S>::ld(e[t]);
    };
    if (valid) {
        int j, k;
        row_jk(g, row, j, k);
        const int p = row * n0 + c;
        const S* X = MODE == 1 ? nullptr : xin.d + (long long)b * xin.bs;
        const float* XS = SC && MODE != 1 ? xin.sc + (long long)b * xin.bs / n0 : nullptr;
        float bq[N], ctr[N], P[N];
        ld4(bv.d + (long long)b * bv.bs + p, bq);
        if (SC) {
            const float f = bv.sc[(long long)b * bv.bs / n0 + row];
#pragma unroll
            for (int t = 0; t < N; ++t) bq[t] *= f;
        }
        if (MODE == 1) {
            ld4(op.sten + 13 * nx + p, ctr);
#pragma unroll
            for (int t = 0; t < N; ++t) res[t] = omega * bq[t] / (SC ? ctr[t] * ssc[13] : ctr[t]);
        } else {
            float acc[N] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int r = 0; r < 9; ++r) {
                const int dy = r % 3 - 1, dz = r / 3 - 1;
                if (j + dy < 0 || j + dy >= g.n1 || k + dz < 0 || k + dz >= g.n2) continue;
                const int rr = row + dy + dz * g.n1;
                const S* xr = X + rr * n0 + c;
                float x[N + 2];
                ld4(xr, x + 1);
                x[0] = c > 0 ? PT<S>::ld(xr[-1]) : 0.f;
                x[N + 1] = c + N < n0 ? PT<S>::ld(xr[N]) : 0.f;
                if (SC) {
                    const float f = XS[rr];
#pragma unroll
                    for (int t = 0; t < N + 2; ++t) x[t] *= f;
                }
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    float s[N];
                    ld4(op.sten + (3 * r + d) * nx + p, s);
                    if (SC) {
                        const float f = ssc[3 * r + d];
#pragma unroll
                        for (int t = 0; t < N; ++t) s[t] *= f;
                    }
#pragma unroll
                    for (int t = 0; t < N; ++t) acc[t] += s[t] * x[t + d];
                    if (3 * r + d == 13) {
#pragma unroll
                        for (int t = 0; t < N; ++t) {
                            ctr[t] = s[t];
                            P[t] = x[t + 1];
                        }
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < N; ++t) res[t] = MODE == 0 ? P[t] + omega * (bq[t] - acc[t]) / ctr[t] : bq[t] - acc[t];
        }
    }
    S* o = out.d + (long long)b * out.bs + (long long)row * n0 + c;
    if constexpr (SC) {
        float sc;
        const float inv = group_scale<N>(res, gs, sc);
        if (valid) {
            RT ov;
            S* oq = reinterpret_cast<S*>(&ov);
#pragma unroll
            for (int t = 0; t < N; ++t) oq[t] = PT<S>::st(res[t] * inv);
            *reinterpret_cast<RT*>(o) = ov;
            if (gl == 0) out.sc[(long long)b * out.bs / n0 + row] = sc;
        }
    } else if (valid) {
        *reinterpret_cast<float4*>(o) = make_float4(res[0], res[1], res[2], res[3]);
    }
}
// Whether a level takes k_st27: FP32 arithmetic, 32-bit offsets, rows of whole 4-column vectors with at most 32 of them, and
// enough points to fill the GPU with a quarter of the threads (one sweep in us, k_st27 / point per thread: 48^3 6.7 /
// 9.3, eight items 13 / 34; 24^3 6.5 / 5.0, eight items 6.3 / 7.2; 12^3 6.6 / 4.8).
template <class S> inline bool st27_ok(const LevelOp<S>& op, int B) {
    return (long long)B * op.g.nx >= 1 << 16 && std::is_same<typename PT<S>::A, float>::value && !op.fine && op.g.d == 3 &&
           op.g.n0 % 4 == 0 && op.g.n0 <= 128 && sten32_ok(op.g.nx);
}

// x_out = x_in + P xc (x_in.d == nullptr: 0) for 16-bit storage: a thread owns 8 fine columns; each of the (one,
// two or four) coarse rows behind its row costs one vector load of 4 and two scalars.  Per point the sum of
// k_prolong_add in its order.  (That kernel formed indices, weights and predicates per point and coarse value:
// 17 us for a 96^3 item, 114 us for eight.)
template <class S>
__global__ void __launch_bounds__(kVecThreads) k_prolong16(Geo gf, Geo gc, int gs, const int* active, Vec<S> xcv,
                                                           Vec<S> xin, Vec<S> xout) {
    pdl_prologue();
    static_assert(PT<S>::scaled, "16-bit storage only");
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    const int n0 = gf.n0, tpr = n0 / 8;
    const int lane = threadIdx.x & 31, grp = lane / gs, gl = lane - grp * gs;
    const int row = (blockIdx.x * (kVecThreads / 32) + (threadIdx.x >> 5)) * (32 / gs) + grp;
    const bool valid = row < gf.R && gl < tpr;
    const int c0 = gl * 8, cc = gl * 4;
    float res[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) res[t] = 0.f;
    if (valid) {
        int j, k;
        row_jk(gf, row, j, k);
        int Jy[2] = {0, 0}, Jz[2] = {0, 0};
        float wy[2], wz[2] = {1.f, 0.f};
        const int my = interp_1d(j, gc.n1, Jy, wy), mz = gf.d == 3 ? interp_1d(k, gc.n2, Jz, wz) : 1;
        if (xin.d) vec8_load(xin.d + (long long)b * xin.bs + row * n0 + c0, xin.sc[(long long)b * xin.bs / n0 + row], res);
        const S* C = xcv.d + (long long)b * xcv.bs;
        const float* CS = xcv.sc + (long long)b * xcv.bs / gc.n0;
        for (int a = 0; a < mz; ++a)
            for (int q = 0; q < my; ++q) {
                const int cr = Jy[q] + gc.n1 * Jz[a];
                const float f = CS[cr], w = wy[q] * wz[a], h = w * 0.5f;
                const S* p = C + cr * gc.n0 + cc;
                const uint2 raw = *reinterpret_cast<const uint2*>(p);
                const S* e = reinterpret_cast<const S*>(&raw);
                float v[6];
                v[0] = cc > 0 ? PT<S>::ld(p[-1]) * f : 0.f;
#pragma unroll
                for (int t = 0; t < 4; ++t) v[t + 1] = PT<S>::ld(e[t]) * f;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    res[2 * t] += h * v[t];
                    res[2 * t] += h * v[t + 1];
                    res[2 * t + 1] += w * v[t + 1];
                }
            }
    }
    float sc;
    const float inv = group_scale<8>(res, gs, sc);
    if (valid) {
        uint4 ov;
        S* oq = reinterpret_cast<S*>(&ov);
#pragma unroll
        for (int t = 0; t < 8; ++t) oq[t] = PT<S>::st(res[t] * inv);
        *reinterpret_cast<uint4*>(xout.d + (long long)b * xout.bs + (long long)row * n0 + c0) = ov;
        if (gl == 0) xout.sc[(long long)b * xout.bs / n0 + row] = sc;
    }
}

// bc = P^T r for 16-bit storage: a thread owns 4 coarse columns, 8 fine columns (one vector) and the one after
// of each of its 9 (3 in 2D) fine rows; per point the sum of k_restrict in its order.
template <class S>
__global__ void __launch_bounds__(kVecThreads) k_restrict16(Geo gf, Geo gc, int gs, const int* active, Vec<S> rv,
                                                            Vec<S> bcv) {
    pdl_prologue();
    static_assert(PT<S>::scaled, "16-bit storage only");
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    const int n0 = gc.n0, tpr = n0 / 4;
    const int lane = threadIdx.x & 31, grp = lane / gs, gl = lane - grp * gs;
    const int row = (blockIdx.x * (kVecThreads / 32) + (threadIdx.x >> 5)) * (32 / gs) + grp;
    const bool valid = row < gc.R && gl < tpr;
    const int I0 = gl * 4, f0 = gl * 8;
    float res[4] = {0.f, 0.f, 0.f, 0.f};
    if (valid) {
        int J, K;
        row_jk(gc, row, J, K);
        const S* R = rv.d + (long long)b * rv.bs;
        const float* RS = rv.sc + (long long)b * rv.bs / gf.n0;
        const int nz = gf.d == 3 ? 3 : 1;
#pragma unroll 1
        for (int z = 0; z < nz; ++z) {
            const int fk = gf.d == 3 ? 2 * K + z : 0;
            if (fk >= gf.n2) continue;
            const float wz = nz == 1 || z == 1 ? 1.f : 0.5f;
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                const int fj = 2 * J + y;
                if (fj >= gf.n1) continue;
                const int fr = fj + gf.n1 * fk;
                const float w = (y == 1 ? 1.f : 0.5f) * wz, h = 0.5f * w, f = RS[fr];
                const S* p = R + fr * gf.n0 + f0;
                float v[9];
                vec8_load(p, f, v);
                v[8] = f0 + 8 < gf.n0 ? PT<S>::ld(p[8]) * f : 0.f;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    res[t] += h * v[2 * t];
                    res[t] += w * v[2 * t + 1];
                    res[t] += h * v[2 * t + 2];
                }
            }
        }
    }
    float sc;
    const float inv = group_scale<4>(res, gs, sc);
    if (valid) {
        uint2 ov;
        S* oq = reinterpret_cast<S*>(&ov);
#pragma unroll
        for (int t = 0; t < 4; ++t) oq[t] = PT<S>::st(res[t] * inv);
        *reinterpret_cast<uint2*>(bcv.d + (long long)b * bcv.bs + (long long)row * n0 + I0) = ov;
        if (gl == 0) bcv.sc[(long long)b * bcv.bs / n0 + row] = sc;
    }
}
// Whether two levels' transfers take the 16-bit vector kernels: fine rows of whole 16-byte vectors, at most 32.
template <class S> inline bool transfer16_ok(const Geo& gf) { return PT<S>::scaled && gf.n0 % 8 == 0 && gf.n0 <= 256; }

// r = b - A x for unscaled storage, RPT rows per thread (as k_smooth_rows).
template <class S, int KIND, int RPT>
__global__ void __launch_bounds__(kPtMaxThreads) k_residual_rows(LevelOp<S> op, PtMap pm, int B, const int* active,
                                                                 Vec<S> xv, Vec<S> bv, Vec<S> rv) {
    pdl_prologue();
    using A = typename PT<S>::A;
    static_assert(!PT<S>::scaled, "unscaled storage only");
    const Geo g = op.g;
    const int b = blockIdx.y;
    if (b >= B || (active && !active[b])) return;
    const int c = threadIdx.x;
    if (c >= g.n0) return;
    const int r0 = blockIdx.x * pm.rpc * RPT + threadIdx.y;
    View<S> xx = view_of(xv, b, 0, g.n0);
    View<S> bb = view_of(bv, b, 0, g.n0);
    S* out = rv.d + (long long)b * rv.bs;
    A v[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = r0 + i * pm.rpc;
        v[i] = A(0);
        if (row < g.R) {
            A Au, dg;
            level_apply_k<KIND>(op, xx, row, row, 0, c, Au, dg);
            v[i] = bb.at(row, c) - Au;
        }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = r0 + i * pm.rpc;
        if (row < g.R) out[(long long)row * g.n0 + c] = PT<S>::st(v[i]);
    }
}

// r = b - A x
template <class S, int KIND = 0>
__global__ void __launch_bounds__(kPtMaxThreads) k_residual(LevelOp<S> op, PtMap pm, int B, const int* active, Vec<S> xv,
                                                   Vec<S> bv, Vec<S> rv) {
    pdl_prologue();
    using A = typename PT<S>::A;
    const Geo g = op.g;
    PtPos q = pt_pos(pm, B, g.R, active);
    if constexpr (!PT<S>::scaled) {
        if (!q.valid) return;
    }
    const long long row = q.row;
    int j, k;
    row_jk(g, row, j, k);
    View<S> xx = view_of(xv, q.b, 0, g.n0);
    View<S> bb = view_of(bv, q.b, 0, g.n0);
    S* out; float* osc;
    row_store_ptrs(rv, q.b, 0, row, g.n0, out, osc);
    pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int c) -> A {
        A Au, dg;
        level_apply_k<KIND>(op, xx, row, j, k, c, Au, dg);
        return bb.at(row, c) - Au;
    });
}

// bc = P^T r  (coarse row kernel; pm maps the coarse rows)
template <class S>
__global__ void __launch_bounds__(kPtMaxThreads) k_restrict(Geo gf, Geo gc, PtMap pm, int B, const int* active, Vec<S> rv,
                                                   Vec<S> bcv) {
    pdl_prologue();
    using A = typename PT<S>::A;
    PtPos q = pt_pos(pm, B, gc.R, active);
    if constexpr (!PT<S>::scaled) {
        if (!q.valid) return;
    }
    const long long row = q.row;
    int J, Kc;
    row_jk(gc, row, J, Kc);
    View<S> rr = view_of(rv, q.b, 0, gf.n0);
    S* out; float* osc;
    row_store_ptrs(bcv, q.b, 0, row, gc.n0, out, osc);
    if (gf.d == 3) {
        // every load before the sum (rows and columns beyond the grid add exact zeros)
        pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int I) -> A {
            const bool xp = 2 * I + 2 < gf.n0;
            A v[27];
#pragma unroll
            for (int r = 0; r < 9; ++r) {
                const int fj = 2 * J + r % 3, fk = 2 * Kc + r / 3;
                const bool in = fj < gf.n1 && fk < gf.n2;
                const int frow = fj + gf.n1 * fk;
                v[3 * r] = in ? rr.at(frow, 2 * I) : A(0);
                v[3 * r + 1] = in ? rr.at(frow, 2 * I + 1) : A(0);
                v[3 * r + 2] = in && xp ? rr.at(frow, 2 * I + 2) : A(0);
            }
            A acc = A(0);
#pragma unroll
            for (int e = 0; e < 27; ++e) {
                const A wx = e % 3 == 1 ? A(1) : A(0.5), wy = e / 3 % 3 == 1 ? A(1) : A(0.5),
                        wz = e / 9 == 1 ? A(1) : A(0.5);
                acc += wx * wy * wz * v[e];
            }
            return acc;
        });
        return;
    }
    pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int I) -> A {
        A acc = A(0);
        const int zlo = gf.d == 3 ? -1 : 0, zhi = gf.d == 3 ? 1 : 0;
        for (int dz = zlo; dz <= zhi; ++dz) {
            int fk = gf.d == 3 ? 2 * Kc + 1 + dz : 0;
            if (fk < 0 || fk >= gf.n2) continue;
            A wz = dz == 0 ? A(1) : A(0.5);
            for (int dy = -1; dy <= 1; ++dy) {
                int fj = 2 * J + 1 + dy;
                if (fj < 0 || fj >= gf.n1) continue;
                A wy = dy == 0 ? A(1) : A(0.5);
                long long frow = fj + (long long)gf.n1 * fk;
#pragma unroll
                for (int dx = -1; dx <= 1; ++dx) {
                    int fi = 2 * I + 1 + dx;
                    if (fi < 0 || fi >= gf.n0) continue;
                    A wx = dx == 0 ? A(1) : A(0.5);
                    acc += wx * wy * wz * rr.at(frow, fi);
                }
            }
        }
        return acc;
    });
}

// x_out = x_in + P xc  (fine row kernel); x_in.d == nullptr means 0.
template <class S>
__global__ void __launch_bounds__(kPtMaxThreads) k_prolong_add(Geo gf, Geo gc, PtMap pm, int B, const int* active,
                                                      Vec<S> xcv, Vec<S> xin, Vec<S> xout) {
    pdl_prologue();
    using A = typename PT<S>::A;
    PtPos q = pt_pos(pm, B, gf.R, active);
    if constexpr (!PT<S>::scaled) {
        if (!q.valid) return;
    }
    const long long row = q.row;
    int j, k;
    row_jk(gf, row, j, k);
    View<S> xc = view_of(xcv, q.b, 0, gc.n0);
    const bool has_in = xin.d != nullptr;
    View<S> xi = has_in ? view_of(xin, q.b, 0, gf.n0) : View<S>{nullptr, nullptr, gf.n0};
    int Jy[2], Jz[2] = {0, 0};
    float wy[2], wz[2] = {1.f, 0.f};
    int my = interp_1d(j, gc.n1, Jy, wy);
    int mz = gf.d == 3 ? interp_1d(k, gc.n2, Jz, wz) : 1;
    S* out; float* osc;
    row_store_ptrs(xout, q.b, 0, row, gf.n0, out, osc);
    if (gf.d == 3) {
        // up to eight coarse points, every load before the sum (a missing one adds an exact zero)
        pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int c) -> A {
            int Jx[2] = {0, 0};
            float wx[2] = {0.f, 0.f};
            const int mx = interp_1d(c, gc.n0, Jx, wx);
            const A base = has_in ? xi.at(row, c) : A(0);
            A v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int x = e & 1, y = e >> 1 & 1, z = e >> 2;
                const bool in = x < mx && y < my && z < mz;
                v[e] = in ? xc.at(Jy[y] + gc.n1 * Jz[z], Jx[x]) : A(0);
            }
            A acc = base;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int x = e & 1, y = e >> 1 & 1, z = e >> 2;
                const bool in = x < mx && y < my && z < mz;
                const A w = in ? A(wy[y]) * A(wz[z]) * A(wx[x]) : A(0);
                acc += w * v[e];
            }
            return acc;
        });
        return;
    }
    pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int c) -> A {
        int Jx[2];
        float wx[2];
        int mx = interp_1d(c, gc.n0, Jx, wx);
        A acc = has_in ? xi.at(row, c) : A(0);
        for (int a = 0; a < mz; ++a)
            for (int bq = 0; bq < my; ++bq) {
                long long crow = Jy[bq] + (long long)gc.n1 * Jz[a];
                A wyz = A(wy[bq]) * A(wz[a]);
                for (int e = 0; e < mx; ++e) acc += wyz * A(wx[e]) * xc.at(crow, Jx[e]);
            }
        return acc;
    });
}

// k_prolong_add in 2D for unscaled storage, RPT rows per thread (as k_smooth_rows).
template <class S, int RPT>
__global__ void __launch_bounds__(kPtMaxThreads) k_prolong_add_rows(Geo gf, Geo gc, PtMap pm, int B, const int* active,
                                                                    Vec<S> xcv, Vec<S> xin, Vec<S> xout) {
    pdl_prologue();
    using A = typename PT<S>::A;
    static_assert(!PT<S>::scaled, "unscaled storage only");
    const int b = blockIdx.y;
    if (b >= B || (active && !active[b])) return;
    const int c = threadIdx.x;
    if (c >= gf.n0) return;
    const int r0 = blockIdx.x * pm.rpc * RPT + threadIdx.y;
    View<S> xc = view_of(xcv, b, 0, gc.n0);
    const bool has_in = xin.d != nullptr;
    View<S> xi = has_in ? view_of(xin, b, 0, gf.n0) : View<S>{nullptr, nullptr, gf.n0};
    S* out = xout.d + (long long)b * xout.bs;
    int Jx[2];
    float wx[2];
    const int mx = interp_1d(c, gc.n0, Jx, wx);
    A v[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = r0 + i * pm.rpc;
        v[i] = A(0);
        if (row < gf.R) {
            int Jy[2];
            float wy[2];
            const int my = interp_1d(row, gc.n1, Jy, wy);
            A acc = has_in ? xi.at(row, c) : A(0);
            for (int bq = 0; bq < my; ++bq) {
                const A wyz = A(wy[bq]) * A(1.f);
                for (int e = 0; e < mx; ++e) acc += wyz * A(wx[e]) * xc.at(Jy[bq], Jx[e]);
            }
            v[i] = acc;
        }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = r0 + i * pm.rpc;
        if (row < gf.R) out[(long long)row * gf.n0 + c] = PT<S>::st(v[i]);
    }
}

// Transfers of batched 2D levels in unscaled storage, a 16-byte vector of columns per thread; per point the sums of
// k_prolong_add and k_restrict in their order.  Bound by memory; a point per
// thread and row spent its time on indices and weights (33 us for the interpolation to 128 items of 256^2, where
// its traffic takes about 12; now 13 us on average over that level and the next, and 10 us for the restriction, both with
// the events' overhead).  With both, the FP32 solve on 256^2 with 128 items went from 288.8 to 280.4 ms.
// Interpolation: the fine rows 2J and 2J + 1 share their coarse rows J - 1 and J.
template <class S>
__global__ void __launch_bounds__(kVecThreads) k_prolong2d(Geo gf, Geo gc, const int* active, Vec<S> xcv, Vec<S> xin,
                                                           Vec<S> xout) {
    pdl_prologue();
    static_assert(!PT<S>::scaled, "unscaled storage only");
    using VT = typename Vec16<S>::T;
    constexpr int V = Vec16<S>::n, C = V / 2;
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    const int n0 = gf.n0, tpr = n0 / V;
    const int q = blockIdx.x * kVecThreads + threadIdx.x;
    const int J = q / tpr, c0 = (q - J * tpr) * V, cc = c0 / 2;
    if (2 * J >= gf.n1) return;
    const S* Xc = xcv.d + (long long)b * xcv.bs;
    S lo[C + 2], hi[C + 2];                       // coarse rows J - 1 and J, columns cc - 1 .. cc + C
#pragma unroll
    for (int t = 0; t < C + 2; ++t) {
        const int I = cc - 1 + t;
        const bool in = I >= 0 && I < gc.n0;
        lo[t] = in && J > 0 ? Xc[(J - 1) * gc.n0 + I] : S(0);
        hi[t] = in && J < gc.n1 ? Xc[J * gc.n0 + I] : S(0);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int row = 2 * J + r;
        if (row >= gf.n1) continue;
        S x[V];
        if (xin.d) {
            const VT v = *reinterpret_cast<const VT*>(xin.d + (long long)b * xin.bs + row * n0 + c0);
            const S* e = reinterpret_cast<const S*>(&v);
#pragma unroll
            for (int t = 0; t < V; ++t) x[t] = e[t];
        } else {
#pragma unroll
            for (int t = 0; t < V; ++t) x[t] = S(0);
        }
        const S w = r == 0 ? S(0.5) : S(1), h = S(0.5) * w;
#pragma unroll
        for (int t = 0; t < C; ++t) {
            if (r == 0) {
                x[2 * t] += h * lo[t];
                x[2 * t] += h * lo[t + 1];
                x[2 * t + 1] += w * lo[t + 1];
            }
            x[2 * t] += h * hi[t];
            x[2 * t] += h * hi[t + 1];
            x[2 * t + 1] += w * hi[t + 1];
        }
        VT o;
        S* e = reinterpret_cast<S*>(&o);
#pragma unroll
        for (int t = 0; t < V; ++t) e[t] = x[t];
        *reinterpret_cast<VT*>(xout.d + (long long)b * xout.bs + row * n0 + c0) = o;
    }
}

// Restriction: V / 2 coarse columns per thread (one vector and the column after it of three fine rows).
template <class S>
__global__ void __launch_bounds__(kVecThreads) k_restrict2d(Geo gf, Geo gc, const int* active, Vec<S> rv, Vec<S> bcv) {
    pdl_prologue();
    static_assert(!PT<S>::scaled, "unscaled storage only");
    using VT = typename Vec16<S>::T;
    constexpr int V = Vec16<S>::n, C = V / 2;
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    const int n0 = gf.n0, tpr = n0 / V;
    const int q = blockIdx.x * kVecThreads + threadIdx.x;
    const int J = q / tpr, f0 = (q - J * tpr) * V;
    if (J >= gc.n1) return;
    const S* R = rv.d + (long long)b * rv.bs;
    S v[3][V + 1];
#pragma unroll
    for (int y = 0; y < 3; ++y) {
        const int row = 2 * J + y;
        const bool in = row < gf.n1;
        if (in) {
            const VT u = *reinterpret_cast<const VT*>(R + row * n0 + f0);
            const S* e = reinterpret_cast<const S*>(&u);
#pragma unroll
            for (int t = 0; t < V; ++t) v[y][t] = e[t];
        } else {
#pragma unroll
            for (int t = 0; t < V; ++t) v[y][t] = S(0);
        }
        v[y][V] = in && f0 + V < n0 ? R[row * n0 + f0 + V] : S(0);
    }
#pragma unroll
    for (int t = 0; t < C; ++t) {
        S acc = S(0);
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const S w = y == 1 ? S(1) : S(0.5), h = S(0.5) * w;
            acc += h * v[y][2 * t];
            acc += w * v[y][2 * t + 1];
            acc += h * v[y][2 * t + 2];
        }
        bcv.d[(long long)b * bcv.bs + J * gc.n0 + f0 / 2 + t] = acc;
    }
}
// Whether batched 2D transfers take the vector kernels: rows of whole 16-byte vectors (their items then start on
// 16-byte boundaries too), and items enough to fill the chip with vectors instead of points.
template <class S> inline bool transfer2d_ok(const Geo& gf, int B) {
    return !PT<S>::scaled && gf.d == 2 && B >= 16 && gf.n0 % (16 / (int)sizeof(S)) == 0;
}

// x_out = xp + omega D^{-1} (b - A xp) with xp = x_in + P xc computed on the fly at
// the point and its stencil neighbours (prolongation fused with one sweep).
template <class S>
__global__ void __launch_bounds__(kPtMaxThreads) k_prolong_smooth(LevelOp<S> op, Geo gc, PtMap pm, int B,
                                                                  const int* active, Vec<S> xcv, Vec<S> xin,
                                                                  Vec<S> bv, Vec<S> xout, typename PT<S>::A omega) {
    pdl_prologue();
    using A = typename PT<S>::A;
    const Geo gf = op.g;
    PtPos q = pt_pos(pm, B, gf.R, active);
    if constexpr (!PT<S>::scaled) {
        if (!q.valid) return;
    }
    const long long row = q.row;
    int j, k;
    row_jk(gf, row, j, k);
    View<S> xc = view_of(xcv, q.b, 0, gc.n0);
    View<S> bb = view_of(bv, q.b, 0, gf.n0);
    const bool has = xin.d != nullptr;
    View<S> xi = has ? view_of(xin, q.b, 0, gf.n0) : View<S>{nullptr, nullptr, gf.n0};
    auto xp = [&](long long rr, int cc) -> A {
        int jj, kk;
    row_jk(gf, rr, jj, kk);
        int Jx[2], Jy[2], Jz[2] = {0, 0};
        float wx[2], wy[2], wz[2] = {1.f, 0.f};
        int mx = interp_1d(cc, gc.n0, Jx, wx);
        int my = interp_1d(jj, gc.n1, Jy, wy);
        int mz = gf.d == 3 ? interp_1d(kk, gc.n2, Jz, wz) : 1;
        A acc = has ? xi.at(rr, cc) : A(0);
        for (int a = 0; a < mz; ++a)
            for (int bq = 0; bq < my; ++bq) {
                long long crow = Jy[bq] + (long long)gc.n1 * Jz[a];
                A wyz = A(wy[bq]) * A(wz[a]);
                for (int e = 0; e < mx; ++e) acc += wyz * A(wx[e]) * xc.at(crow, Jx[e]);
            }
        return acc;
    };
    S* out; float* osc;
    row_store_ptrs(xout, q.b, 0, row, gf.n0, out, osc);
    pt_store<S>(out, osc, pm, q.c0, q.valid, [&](int c) -> A {
        A Au, dg;
        level_apply_g(op, xp, row, j, k, c, Au, dg);
        return xp(row, c) + omega * (bb.at(row, c) - Au) / dg;
    });
}

// ---------------------------------------------------------------------------
// The finest 3D level's fused steps (two sweeps; residual and restriction; interpolation and sweep), a tile of
// whole grid rows per CTA: the inner step's values are formed once in shared memory instead of being
// recomputed at every neighbour (seven times the arithmetic and 49 loads per point).  Same operations per
// point as k_smooth2, k_resid_restrict and k_prolong_smooth.  Tiles of 4 x 4 rows (2 x 2 coarse rows): a
// 47 x 39 x 43 grid gives 110 CTAs; a warp per row, so a row's storage scale is a warp reduction.
// ---------------------------------------------------------------------------
constexpr int kT3Threads = 256;
constexpr int kT3Warps = kT3Threads / kWarp;
constexpr int kT3 = 4;                       // output rows per axis
inline size_t t3_smem_smooth2(int n0, size_t a) { return (size_t)((kT3 + 4) * (kT3 + 4) + (kT3 + 2) * (kT3 + 2)) * n0 * a; }
inline size_t t3_smem_restrict(int n0, size_t a) { return (size_t)((kT3 + 3) * (kT3 + 3) + (kT3 + 1) * (kT3 + 1)) * n0 * a; }
inline size_t t3_smem_prolong(int n0, size_t a) { return (size_t)(kT3 + 2) * (kT3 + 2) * n0 * a; }
inline dim3 t3_grid(int n1, int n2, int tile, int B) {
    return dim3((unsigned)((n1 + tile - 1) / tile), (unsigned)((n2 + tile - 1) / tile), (unsigned)B);
}

// Rows of a tile region in shared memory: w rows per axis, the first one (j0, k0), n0 columns.
template <class A> struct T3Rows {
    const A* d;
    int w, j0, k0, n0;
    __device__ __forceinline__ A operator()(int j, int k, int c) const { return d[((k - k0) * w + j - j0) * n0 + c]; }
};

// (A u)_P and a_PP of the matrix-free 3D level from u(j, k, c) in shared memory.  (1 / h^2 comes beside the level: as fields
// of LevelOp its values would change the register allocation of every kernel that takes one: 96 instead of 118 for
// k_smooth2<double>, 10% slower.)
template <class S, class A>
__device__ __forceinline__ void t3_apply(const LevelOp<S>& op, const InvH2<A>& h, const T3Rows<A>& u, int j, int k, int c, A& Au, A& diag) {
    const Geo& g = op.g;
    const A uP = u(j, k, c);
    const A uW = c > 0 ? u(j, k, c - 1) : A(0), uE = c + 1 < g.n0 ? u(j, k, c + 1) : A(0);
    const A uS = j > 0 ? u(j - 1, k, c) : A(0), uN = j + 1 < g.n1 ? u(j + 1, k, c) : A(0);
    const A uD = k > 0 ? u(j, k - 1, c) : A(0), uU = k + 1 < g.n2 ? u(j, k + 1, c) : A(0);
    const Faces<A>& f = op.faces;
    A Ku, kd;
    if (f.fx == nullptr) {
        Ku = h.x * (A(2) * uP - uW - uE) + h.y * (A(2) * uP - uS - uN);
        Ku += h.z * (A(2) * uP - uD - uU);
        kd = A(2) * h.x + A(2) * h.y;
        kd += A(2) * h.z;
    } else {
        const int row = j + g.n1 * k, fxi = row * (g.n0 + 1) + c, fyi = (k * (g.n1 + 1) + j) * g.n0 + c;
        const int fzi = row * g.n0 + c, pl = g.n1 * g.n0;
        const A x0 = f.fx[fxi], x1 = f.fx[fxi + 1], y0 = f.fy[fyi], y1 = f.fy[fyi + g.n0], z0 = f.fz[fzi], z1 = f.fz[fzi + pl];
        Ku = x0 * (uP - uW) + x1 * (uP - uE) + y0 * (uP - uS) + y1 * (uP - uN);
        Ku += z0 * (uP - uD) + z1 * (uP - uU);
        kd = x0 + x1 + y0 + y1;
        kd += z0 + z1;
    }
    Au = op.sigma * uP + op.c * Ku;
    diag = op.sigma + op.c * kd;
}

// Load the rows [j0, j0 + w) x [k0, k0 + w) of v that lie inside the grid.
template <class S, class A>
__device__ __forceinline__ void t3_load(const Geo& g, const View<S>& v, int w, int j0, int k0, A* dst) {
    const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = wp; r < w * w; r += kT3Warps) {
        const int j = j0 + r % w, k = k0 + r / w;
        if (j < 0 || j >= g.n1 || k < 0 || k >= g.n2) continue;
#pragma unroll 2
        for (int c = lane; c < g.n0; c += kWarp) dst[r * g.n0 + c] = v.at(j + g.n1 * k, c);
    }
}

template <class S>
__global__ void __launch_bounds__(kT3Threads) k_smooth2_tile(LevelOp<S> op, InvH2<typename PT<S>::A> h, const int* active,
                                                             Vec<S> xin, Vec<S> bv, Vec<S> xout, typename PT<S>::A omega) {
    pdl_prologue();
    using A = typename PT<S>::A;
    extern __shared__ __align__(16) unsigned char t3_smem[];
    const Geo& g = op.g;
    const int b = blockIdx.z;
    if (active && !active[b]) return;
    const int j0 = blockIdx.x * kT3, k0 = blockIdx.y * kT3, n0 = g.n0;
    constexpr int W0 = kT3 + 4, W1 = kT3 + 2;
    A* x0 = reinterpret_cast<A*>(t3_smem);
    A* x1 = x0 + W0 * W0 * n0;
    View<S> bb = view_of(bv, b, 0, n0);
    const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool has = xin.d != nullptr;
    if (has) t3_load(g, view_of(xin, b, 0, n0), W0, j0 - 2, k0 - 2, x0);
    __syncthreads();
    const T3Rows<A> u0{x0, W0, j0 - 2, k0 - 2, n0};
    for (int r = wp; r < W1 * W1; r += kT3Warps) {
        const int j = j0 - 1 + r % W1, k = k0 - 1 + r / W1;
        if (j < 0 || j >= g.n1 || k < 0 || k >= g.n2) continue;
        for (int c = lane; c < n0; c += kWarp) {
            const A bp = bb.at(j + g.n1 * k, c);
            if (has) {
                A Au, dg;
                t3_apply(op, h, u0, j, k, c, Au, dg);
                x1[r * n0 + c] = u0(j, k, c) + omega * (bp - Au) / dg;
            } else {
                x1[r * n0 + c] = omega * bp / level_diag(op, j + g.n1 * k, j, k, c);
            }
        }
    }
    __syncthreads();
    const T3Rows<A> u1{x1, W1, j0 - 1, k0 - 1, n0};
    for (int r = wp; r < kT3 * kT3; r += kT3Warps) {
        const int j = j0 + r % kT3, k = k0 + r / kT3;
        if (j >= g.n1 || k >= g.n2) continue;
        A* x2 = x0 + r * n0;                      // x_in is not read again
        for (int c = lane; c < n0; c += kWarp) {
            A Au, dg;
            t3_apply(op, h, u1, j, k, c, Au, dg);
            x2[c] = u1(j, k, c) + omega * (bb.at(j + g.n1 * k, c) - Au) / dg;
        }
        S* out; float* osc;
        row_store_ptrs(xout, b, 0, j + g.n1 * k, n0, out, osc);
        row_store<S>(out, osc, n0, lane, [&](int c) -> A { return x2[c]; });
    }
}

template <class S>
__global__ void __launch_bounds__(kT3Threads) k_resid_restrict_tile(LevelOp<S> op, InvH2<typename PT<S>::A> h, Geo gc,
                                                                    const int* active, Vec<S> xv, Vec<S> bv, Vec<S> bcv) {
    pdl_prologue();
    using A = typename PT<S>::A;
    extern __shared__ __align__(16) unsigned char t3_smem[];
    const Geo& g = op.g;
    const int b = blockIdx.z;
    if (active && !active[b]) return;
    constexpr int CT = kT3 / 2, WR = kT3 + 1, WX = kT3 + 3;     // coarse rows; fine rows 2J .. 2J + 2; one more around
    const int J0 = blockIdx.x * CT, K0 = blockIdx.y * CT, j0 = 2 * J0, k0 = 2 * K0, n0 = g.n0;
    A* x0 = reinterpret_cast<A*>(t3_smem);
    A* rs = x0 + WX * WX * n0;
    View<S> bb = view_of(bv, b, 0, n0);
    const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool has = xv.d != nullptr;
    if (has) t3_load(g, view_of(xv, b, 0, n0), WX, j0 - 1, k0 - 1, x0);
    __syncthreads();
    const T3Rows<A> u{x0, WX, j0 - 1, k0 - 1, n0};
    for (int r = wp; r < WR * WR; r += kT3Warps) {
        const int j = j0 + r % WR, k = k0 + r / WR;
        const bool in = j < g.n1 && k < g.n2;
        for (int c = lane; c < n0; c += kWarp) {
            A res = A(0);
            if (in) {
                res = bb.at(j + g.n1 * k, c);
                if (has) {
                    A Au, dg;
                    t3_apply(op, h, u, j, k, c, Au, dg);
                    res -= Au;
                }
            }
            rs[r * n0 + c] = res;
        }
    }
    __syncthreads();
    for (int r = wp; r < CT * CT; r += kT3Warps) {
        const int J = J0 + r % CT, K = K0 + r / CT;
        if (J >= gc.n1 || K >= gc.n2) continue;
        const A* base = rs + ((2 * (r / CT)) * WR + 2 * (r % CT)) * n0;
        A* bc = x0 + r * n0;
        for (int I = lane; I < gc.n0; I += kWarp) {
            const bool xp = 2 * I + 2 < n0;
            A acc = A(0);
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                const A wy = e % 3 == 1 ? A(1) : A(0.5), wz = e / 3 == 1 ? A(1) : A(0.5);
                const A* row = base + ((e / 3) * WR + e % 3) * n0 + 2 * I;
                acc += A(0.5) * wy * wz * row[0];
                acc += wy * wz * row[1];
                acc += A(0.5) * wy * wz * (xp ? row[2] : A(0));
            }
            bc[I] = acc;
        }
        S* out; float* osc;
        row_store_ptrs(bcv, b, 0, J + gc.n1 * K, gc.n0, out, osc);
        row_store<S>(out, osc, gc.n0, lane, [&](int c) -> A { return bc[c]; });
    }
}

template <class S>
__global__ void __launch_bounds__(kT3Threads) k_prolong_smooth_tile(LevelOp<S> op, InvH2<typename PT<S>::A> h, Geo gc,
                                                                    const int* active, Vec<S> xcv, Vec<S> xin, Vec<S> bv,
                                                                    Vec<S> xout, typename PT<S>::A omega) {
    pdl_prologue();
    using A = typename PT<S>::A;
    extern __shared__ __align__(16) unsigned char t3_smem[];
    const Geo& g = op.g;
    const int b = blockIdx.z;
    if (active && !active[b]) return;
    const int j0 = blockIdx.x * kT3, k0 = blockIdx.y * kT3, n0 = g.n0;
    constexpr int W1 = kT3 + 2;
    A* xp = reinterpret_cast<A*>(t3_smem);
    View<S> bb = view_of(bv, b, 0, n0), xc = view_of(xcv, b, 0, gc.n0);
    const bool has = xin.d != nullptr;
    View<S> xi = has ? view_of(xin, b, 0, n0) : View<S>{nullptr, nullptr, n0};
    const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = wp; r < W1 * W1; r += kT3Warps) {
        const int j = j0 - 1 + r % W1, k = k0 - 1 + r / W1;
        if (j < 0 || j >= g.n1 || k < 0 || k >= g.n2) continue;
        int Jy[2] = {0, 0}, Jz[2] = {0, 0};
        float wy[2] = {0.f, 0.f}, wz[2] = {0.f, 0.f};
        const int my = interp_1d(j, gc.n1, Jy, wy), mz = interp_1d(k, gc.n2, Jz, wz);
        for (int c = lane; c < n0; c += kWarp) {
            int Jx[2] = {0, 0};
            float wx[2] = {0.f, 0.f};
            const int mx = interp_1d(c, gc.n0, Jx, wx);
            A acc = has ? xi.at(j + g.n1 * k, c) : A(0);
            A v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int x = e & 1, y = e >> 1 & 1, z = e >> 2;
                v[e] = x < mx && y < my && z < mz ? xc.at(Jy[y] + gc.n1 * Jz[z], Jx[x]) : A(0);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int x = e & 1, y = e >> 1 & 1, z = e >> 2;
                const A w = x < mx && y < my && z < mz ? A(wy[y]) * A(wz[z]) * A(wx[x]) : A(0);
                acc += w * v[e];
            }
            xp[r * n0 + c] = acc;
        }
    }
    __syncthreads();
    const T3Rows<A> u{xp, W1, j0 - 1, k0 - 1, n0};
    A val[4];
    for (int r = wp; r < kT3 * kT3; r += kT3Warps) {
        const int j = j0 + r % kT3, k = k0 + r / kT3;
        const bool in = j < g.n1 && k < g.n2;
        // columns lane, lane + 32, ... (at most four: t3_ok)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = lane + kWarp * q;
            val[q] = A(0);
            if (in && c < n0) {
                A Au, dg;
                t3_apply(op, h, u, j, k, c, Au, dg);
                val[q] = u(j, k, c) + omega * (bb.at(j + g.n1 * k, c) - Au) / dg;
            }
        }
        if (!in) continue;
        S* out; float* osc;
        row_store_ptrs(xout, b, 0, j + g.n1 * k, n0, out, osc);
        row_store<S>(out, osc, n0, lane, [&](int c) -> A {
            const int q = c / kWarp;
            return q == 0 ? val[0] : (q == 1 ? val[1] : (q == 2 ? val[2] : val[3]));
        });
    }
}

// Whether the finest level's fused steps take the tiles: 3D matrix-free, rows of at most 128 points whose tiles
// fit the default 48 KB of shared memory.
template <class S> inline bool t3_ok(const LevelOp<S>& op) {
    return op.fine && op.g.d == 3 && op.g.n0 <= 128 &&
           t3_smem_smooth2(op.g.n0, sizeof(typename PT<S>::A)) <= 48 * 1024;
}

// x = Dinv b at the coarsest level (Dinv dense, nc x nc, row-major, arithmetic type): a block per grid
// row, a warp per point of it, b in shared memory.  (One thread per point read its row of Dinv alone:
// nc dependent uncoalesced loads.)
constexpr int kCoarseThreads = 256;
template <class S>
__global__ void __launch_bounds__(kCoarseThreads) k_coarse_solve(Geo g, int B, const int* active,
                                                                 const typename PT<S>::A* Dinv, Vec<S> bv, Vec<S> xv) {
    pdl_prologue();
    using A = typename PT<S>::A;
    __shared__ A bs[kMaxCoarsest], xs[kMaxCoarsest];
    const int b = blockIdx.y, row = blockIdx.x, nc = (int)g.nx;
    if (b >= B || (active && !active[b])) return;
    View<S> bb = view_of(bv, b, 0, g.n0);
    for (int q = threadIdx.x; q < nc; q += kCoarseThreads) bs[q] = bb.at(q / g.n0, q % g.n0);
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = w; c < g.n0; c += kCoarseThreads / kWarp) {
        const A* D = Dinv + (long long)(row * g.n0 + c) * nc;
        A acc = A(0);
#pragma unroll 8
        for (int q = lane; q < nc; q += kWarp) acc += D[q] * bs[q];
        acc = warp_sum(acc);
        if (lane == 0) xs[c] = acc;
    }
    __syncthreads();
    if (w != 0) return;
    S* out; float* osc;
    row_store_ptrs(xv, b, 0, row, g.n0, out, osc);
    row_store<S>(out, osc, g.n0, lane, [&](int c) -> A { return xs[c]; });
}

// ---------------------------------------------------------------------------
// Set-up (FP64): Galerkin coarse stencil A_c = P^T A P, one thread per coarse
// point.  The fine operator is either matrix-free FD (sigma I + c K) or a
// stored FP64 3^d stencil.
// ---------------------------------------------------------------------------
struct FineDesc {
    Geo g;
    int fine;
    double sigma, c;
    Faces<double> faces;
    const double* sten;
};

__device__ __forceinline__ int fine_row_entries(const FineDesc& fd, int fi, int fj, int fk, int* gi, int* gj,
                                                int* gk, double* val) {
    const Geo& g = fd.g;
    long long row = fj + (long long)g.n1 * fk;
    int m = 0;
    if (fd.fine) {
        // diagonal and the 2d face neighbours
        double dg;
        if (fd.faces.fx == nullptr) {
            dg = 2 * g.hx2 + 2 * g.hy2 + (g.d == 3 ? 2 * g.hz2 : 0.0);
        } else {
            long long fxi = row * (g.n0 + 1) + fi;
            long long fyi = ((long long)fk * (g.n1 + 1) + fj) * g.n0 + fi;
            dg = fd.faces.fx[fxi] + fd.faces.fx[fxi + 1] + fd.faces.fy[fyi] + fd.faces.fy[fyi + g.n0];
            if (g.d == 3) {
                long long fzi = ((long long)fk * g.n1 + fj) * g.n0 + fi;
                dg += fd.faces.fz[fzi] + fd.faces.fz[fzi + (long long)g.n1 * g.n0];
            }
        }
        gi[m] = fi; gj[m] = fj; gk[m] = fk; val[m] = fd.sigma + fd.c * dg; ++m;
        for (int a = 0; a < g.d; ++a)
            for (int sg = -1; sg <= 1; sg += 2) {
                int ii = fi + (a == 0 ? sg : 0), jj = fj + (a == 1 ? sg : 0), kk = fk + (a == 2 ? sg : 0);
                if (ii < 0 || ii >= g.n0 || jj < 0 || jj >= g.n1 || kk < 0 || kk >= g.n2) continue;
                double face;
                if (fd.faces.fx == nullptr) {
                    face = a == 0 ? g.hx2 : (a == 1 ? g.hy2 : g.hz2);
                } else if (a == 0) {
                    face = fd.faces.fx[row * (g.n0 + 1) + fi + (sg > 0 ? 1 : 0)];
                } else if (a == 1) {
                    face = fd.faces.fy[((long long)fk * (g.n1 + 1) + fj + (sg > 0 ? 1 : 0)) * g.n0 + fi];
                } else {
                    face = fd.faces.fz[((long long)(fk + (sg > 0 ? 1 : 0)) * g.n1 + fj) * g.n0 + fi];
                }
                gi[m] = ii; gj[m] = jj; gk[m] = kk; val[m] = -fd.c * face; ++m;
            }
        return m;
    }
    long long p = row * g.n0 + fi;
    const int zlo = g.d == 3 ? -1 : 0, zhi = g.d == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                int ii = fi + dx, jj = fj + dy, kk = fk + dz;
                if (ii < 0 || ii >= g.n0 || jj < 0 || jj >= g.n1 || kk < 0 || kk >= g.n2) continue;
                int q = (dx + 1) + 3 * (dy + 1) + (g.d == 3 ? 9 * (dz + 1) : 0);
                double v = fd.sten[(long long)q * g.nx + p];
                if (v == 0.0) continue;
                gi[m] = ii; gj[m] = jj; gk[m] = kk; val[m] = v; ++m;
            }
    return m;
}

static __global__ void k_galerkin(FineDesc fd, Geo gc, double* out) {
    pdl_prologue();
    long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= gc.nx) return;
    const Geo& gf = fd.g;
    const int ncoef = gc.d == 3 ? 27 : 9;
    int I = (int)(p % gc.n0), J = (int)((p / gc.n0) % gc.n1), Kc = (int)(p / ((long long)gc.n0 * gc.n1));
    double acc[27];
    for (int q = 0; q < 27; ++q) acc[q] = 0.0;
    const int zlo = gf.d == 3 ? -1 : 0, zhi = gf.d == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz) {
        int fk = gf.d == 3 ? 2 * Kc + 1 + dz : 0;
        if (fk < 0 || fk >= gf.n2) continue;
        double wz = dz == 0 ? 1.0 : 0.5;
        for (int dy = -1; dy <= 1; ++dy) {
            int fj = 2 * J + 1 + dy;
            if (fj < 0 || fj >= gf.n1) continue;
            double wy = dy == 0 ? 1.0 : 0.5;
            for (int dx = -1; dx <= 1; ++dx) {
                int fi = 2 * I + 1 + dx;
                if (fi < 0 || fi >= gf.n0) continue;
                double wf = (dx == 0 ? 1.0 : 0.5) * wy * wz;   // P[f, I]
                int gi[27], gj[27], gk[27];
                double val[27];
                int m = fine_row_entries(fd, fi, fj, fk, gi, gj, gk, val);
                for (int e = 0; e < m; ++e) {
                    int Jx[2], Jy[2], Jz[2] = {0, 0};
                    float wx[2], wy2[2], wz2[2] = {1.f, 0.f};
                    int mx = interp_1d(gi[e], gc.n0, Jx, wx);
                    int my = interp_1d(gj[e], gc.n1, Jy, wy2);
                    int mz = gc.d == 3 ? interp_1d(gk[e], gc.n2, Jz, wz2) : 1;
                    for (int a = 0; a < mz; ++a)
                        for (int bq = 0; bq < my; ++bq)
                            for (int cq = 0; cq < mx; ++cq) {
                                int ox = Jx[cq] - I, oy = Jy[bq] - J, oz = gc.d == 3 ? Jz[a] - Kc : 0;
                                int q = (ox + 1) + 3 * (oy + 1) + (gc.d == 3 ? 9 * (oz + 1) : 0);
                                acc[q] += wf * val[e] * (double)wx[cq] * (double)wy2[bq] * (double)wz2[a];
                            }
                }
            }
        }
    }
    for (int q = 0; q < ncoef; ++q) out[(long long)q * gc.nx + p] = acc[q];
}

// Q1: the fine-level operator M + c K as a stored FP64 3^d-point stencil.
static __global__ void k_q1_stencil(Geo g, Q1<double> q, double c, double* out) {
    pdl_prologue();
    long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.nx) return;
    const int zlo = g.d == 3 ? -1 : 0, zhi = g.d == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const double mx = q.m[0][dx + 1], my = q.m[1][dy + 1], mz = g.d == 3 ? q.m[2][dz + 1] : 1.0;
                const double kx = q.k[0][dx + 1], ky = q.k[1][dy + 1], kz = g.d == 3 ? q.k[2][dz + 1] : 0.0;
                double kc = kx * my * mz + mx * ky * mz;
                if (g.d == 3) kc += mx * my * kz;
                int qi = (dx + 1) + 3 * (dy + 1) + (g.d == 3 ? 9 * (dz + 1) : 0);
                out[(long long)qi * g.nx + p] = mx * my * mz + c * kc;
            }
}

// Dense matrix of the coarsest level from its FP64 description (fine or stencil).
static __global__ void k_dense_level(FineDesc fd, double* Adense) {
    pdl_prologue();
    long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const Geo& g = fd.g;
    if (p >= g.nx) return;
    int fi = (int)(p % g.n0), fj = (int)((p / g.n0) % g.n1), fk = (int)(p / ((long long)g.n0 * g.n1));
    int gi[27], gj[27], gk[27];
    double val[27];
    int m = fine_row_entries(fd, fi, fj, fk, gi, gj, gk, val);
    for (long long q = 0; q < g.nx; ++q) Adense[p * g.nx + q] = 0.0;
    for (int e = 0; e < m; ++e) {
        long long q = gi[e] + (long long)g.n0 * (gj[e] + (long long)g.n1 * gk[e]);
        Adense[p * g.nx + q] += val[e];
    }
}

// Gauss--Jordan inverses (SPD input, no pivoting needed) of the coarsest level's matrices, one cluster
// of up to kGjCtas CTAs per matrix.  Bound by FP64 arithmetic: n^3 multiply-adds at about two per cycle and
// SM, so one CTA needs 9.0 ms for n = 256 while the rest of the chip idles (16 CTAs: 1.2 ms, three matrices at once).
// Here CTA r keeps rows r, r + ctas, ... in shared memory (in place: column k of the inverse replaces column k of A,
// half the arithmetic of an augmented matrix); the owner of pivot row k + 1 updates and scales that row
// first and stores it into every CTA's buffer, then all CTAs eliminate their rows with pivot row k,
// so one cluster barrier per pivot is left.  The same pivots and products as elimination of [A | I].
// Where no such cluster fits (a device shared out in small parts), smaller ones take its place, at last one CTA
// whose rows are in the result's memory.
constexpr int kGjCtas = 16;
constexpr int kGjThreads = 512;

// Shared memory: two pivot rows and (staged) a CTA's rows.
inline size_t gj_smem(int n, int ctas, bool staged) {
    return ((staged ? (size_t)((n + ctas - 1) / ctas) * n : 0) + 2 * (size_t)n) * sizeof(double);
}
// CTAs per cluster: the most whose cluster fits, 0 for one CTA without staged rows.
template <class Fits> inline int gj_ctas(Fits&& fits) {
    for (int c = kGjCtas; c >= 1; c /= 2)
        if (fits(c)) return c;
    return 0;
}

static __global__ void __launch_bounds__(kGjThreads) k_gauss_jordan(const double* Ain, double* Inv, int n, int ctas,
                                                                    int staged, int* fail) {
    pdl_prologue();
    extern __shared__ __align__(16) double gj_sm[];
    unsigned rank, mat;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(mat));
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = kGjThreads / 32;
    const int nr = n > (int)rank ? (n - (int)rank + ctas - 1) / ctas : 0;   // own rows
    const double* A = Ain + (long long)mat * n * n;
    double* O = Inv + (long long)mat * n * n;
    double* prow = gj_sm;                       // two pivot rows, scaled by 1 / pivot
    double* R = staged ? gj_sm + 2 * n : O;     // (not staged: one CTA, which owns every row)
    for (int i = w; i < nr; i += nw)
        for (int j = lane; j < n; j += 32) R[i * n + j] = A[(long long)(rank + i * ctas) * n + j];
    __syncthreads();
    // row i minus its column k times pivot row k; the pivot's own entry becomes 1 / pivot there, so
    // column k of every other row becomes -f / pivot
    auto eliminate = [&](double* row, const double* pr, int k) {
        const double f = row[k];
        __syncwarp();
        for (int j = lane; j < n; j += 32) row[j] = j == k ? -f * pr[j] : row[j] - f * pr[j];
    };
    auto publish = [&](int k) {                 // the owner: scale row k, store it into every CTA
        double* row = R + (k / ctas) * n;
        const double piv = row[k];
        if (tid == 0 && !(piv > 0.0)) *fail = 1;
        const double pinv = 1.0 / piv;
        __syncthreads();
        for (int j = tid; j < n; j += kGjThreads) {
            const double v = j == k ? pinv : row[j] * pinv;
            row[j] = v;
            double* dst = prow + (k & 1) * n + j;
            for (int c = 0; c < ctas; ++c) {
                unsigned long long q;
                asm volatile("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(dst), "r"(c));
                *reinterpret_cast<double*>(q) = v;
            }
        }
        __syncthreads();
    };
    auto cluster_barrier = [] {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    cluster_barrier();                          // every CTA has started before the first remote store
    if (rank == 0) publish(0);
    cluster_barrier();
    for (int k = 0; k < n; ++k) {
        const double* pr = prow + (k & 1) * n;
        const bool ahead = k + 1 < n && (k + 1) % ctas == (int)rank;
        const int ia = (k + 1) / ctas;
        if (ahead) {
            if (w == 0) eliminate(R + ia * n, pr, k);
            __syncthreads();
            publish(k + 1);                     // buffer (k + 1) & 1: last read before the previous barrier
        }
        for (int i = w; i < nr; i += nw) {
            if ((int)rank + i * ctas == k || (ahead && i == ia)) continue;
            eliminate(R + i * n, pr, k);
        }
        cluster_barrier();
    }
    if (!staged) return;
    for (int i = w; i < nr; i += nw)
        for (int j = lane; j < n; j += 32) O[(long long)(rank + i * ctas) * n + j] = R[i * n + j];
}

// Invert nmat consecutive n x n matrices; *fail is set when a pivot is not positive.
inline aao_status launch_gauss_jordan(const double* A, double* Inv, int n, int nmat, int* fail, cudaStream_t st) {
    int dev = 0, optin = 0;
    AAO_CUDA_TRY(cudaGetDevice(&dev));
    AAO_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    AAO_CUDA_TRY(cudaFuncSetAttribute(k_gauss_jordan, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    AAO_CUDA_TRY(cudaFuncSetAttribute(k_gauss_jordan, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    const int c = gj_ctas([&](int ctas) {
        if (gj_smem(n, ctas, true) > (size_t)optin) return false;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3(kGjThreads);
        cfg.dynamicSmemBytes = gj_smem(n, ctas, true);
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)ctas;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, k_gauss_jordan, &cfg) == cudaSuccess && fit > 0) return true;
        cudaGetLastError();
        return false;
    });
    const int ctas = c > 0 ? c : 1;
    launch_cluster(k_gauss_jordan, dim3((unsigned)(ctas * nmat)), dim3(kGjThreads), gj_smem(n, ctas, c > 0), st, ctas, A, Inv,
                   n, ctas, c > 0 ? 1 : 0, fail);
    AAO_LAUNCH_CHECK();
    return AAO_OK;
}

// Per-component max |coef| (one block per component) and conversion to S.
static __global__ void k_stencil_absmax(const double* sten, long long nx, float* cmax) {
    pdl_prologue();
    int q = blockIdx.x;
    double m = 0.0;
    for (long long p = threadIdx.x; p < nx; p += blockDim.x) m = fmax(m, fabs(sten[(long long)q * nx + p]));
    __shared__ double sh[kBlock];
    sh[threadIdx.x] = m;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double mm = sh[0];
        float sc = 1.f;
        if (mm > 0.0) {
            int e;
            frexp(mm, &e);
            sc = ldexpf(1.f, e - 14);
        }
        cmax[q] = sc;
    }
}

template <class S>
__global__ void k_stencil_convert(const double* sten, long long nx, int ncoef, const float* sc, S* out) {
    pdl_prologue();
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nx * ncoef) return;
    int q = (int)(i / nx);
    double v = sten[i];
    if constexpr (PT<S>::scaled) v /= (double)sc[q];
    out[i] = PT<S>::st((typename PT<S>::A)v);
}

template <class A>
__global__ void k_convert_dense(const double* in, A* out, long long n) {
    pdl_prologue();
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (A)in[i];
}

}  // namespace aao

namespace aao {

// ---------------------------------------------------------------------------
// Fused V-cycle tail: levels lc..L-1 of one batch item in one CTA, every level
// held on chip (x and b per level, arithmetic type A), Jacobi sweeps staged in
// registers, residual recomputed inside the restriction.  One launch replaces
// the ~7 launches per level of the level-by-level path.  Vectors that stay on
// chip are not rounded to the 16-bit storage format (that format is for data
// that travels through HBM).
// ---------------------------------------------------------------------------
constexpr int kTailPmax = 4;    // points per thread at level lc (kTailMaxPoints / 1024)
constexpr int kTailMaxPoints = 4096;         // batched V-cycles
constexpr int kTailMaxPointsSingle = 1024;   // single-item V-cycles (the Schur sweep)
constexpr long long kFuseMaxPoints = 1 << 20;   // fuse sweeps below this many points per launch

template <class SI> struct TailCtx {
    using A = typename PT<SI>::A;
    int lc, L;
    LevelOp<SI> op[kMaxLevels];
    int off[kMaxLevels];        // smem offset (A elements) of X_l; B_l and R_l follow
    int vec_bytes;              // bytes of all X_l, B_l
    int stage_from;             // levels >= stage_from (and >= 1) read their stencil from smem
    int sten_off[kMaxLevels];   // byte offset of a staged stencil (after the vectors)
    const A* Dinv;
    A omega;
    int nu1, nu2;
};

// The operator of tail level l, reading a staged stencil from shared memory.
template <class SI>
__device__ __forceinline__ LevelOp<SI> tail_op(const TailCtx<SI>& t, int l, const unsigned char* smem) {
    LevelOp<SI> op = t.op[l];
    if (l >= 1 && l >= t.stage_from) op.sten = reinterpret_cast<const SI*>(smem + t.sten_off[l]);
    return op;
}

// Damped-Jacobi sweeps of tail level l, ping-ponging between its two on-chip x
// buffers (one barrier per sweep); cur selects the buffer holding x.
template <class SI>
__device__ __forceinline__ void tail_smooth(const TailCtx<SI>& t, int l, typename PT<SI>::A* sm, int sweeps,
                                            bool zero_first, unsigned& curbits) {
    int cur = (curbits >> l) & 1u;
    using A = typename PT<SI>::A;
    const LevelOp<SI> op = tail_op(t, l, reinterpret_cast<const unsigned char*>(sm));
    const Geo& g = op.g;
    A* X0 = sm + t.off[l];
    const A* Bv = X0 + 2 * g.nx;
    const int nt = blockDim.x;
    for (int sw = 0; sw < sweeps; ++sw) {
        const bool zero = zero_first && sw == 0;
        const A* Xc = X0 + (long long)cur * g.nx;
        A* Xn = X0 + (long long)(1 - cur) * g.nx;
        View<A> xv{Xc, nullptr, g.n0};
        for (int p = threadIdx.x; p < g.nx; p += nt) {
            int c = p % g.n0;
            long long row = p / g.n0;
            int j, k;
    row_jk(g, row, j, k);
            if (zero) {
                Xn[p] = t.omega * Bv[p] / level_diag(op, row, j, k, c);
            } else {
                A Au, dg;
                if (op.fine) level_apply(op, xv, row, j, k, c, Au, dg);
                else level_apply_k<3>(op, xv, row, j, k, c, Au, dg);
                Xn[p] = Xc[p] + t.omega * (Bv[p] - Au) / dg;
            }
        }
        cur = 1 - cur;
        __syncthreads();
    }
    curbits = (curbits & ~(1u << l)) | ((unsigned)cur << l);
}

template <class SI>
__global__ void __launch_bounds__(1024) k_vcycle_tail(TailCtx<SI> t, int B, const int* active, Vec<SI> bv,
                                                      Vec<SI> xin, Vec<SI> xout) {
    pdl_prologue();
    using A = typename PT<SI>::A;
    extern __shared__ __align__(16) unsigned char tail_smem[];
    A* sm = reinterpret_cast<A*>(tail_smem);
    const int b = blockIdx.x;
    if (b >= B || (active && !active[b])) return;
    const int nt = blockDim.x, tid = threadIdx.x;
    const int lc = t.lc, L = t.L;
    // per level: X0, X1 (x ping-pong; the free one holds the residual), B
    unsigned cur = 0u;      // bit l: which of level l's two x buffers holds the iterate
    // copy the coarse stencils of levels >= stage_from into shared memory, 16 bytes at a time
    for (int l = t.stage_from; l < L; ++l) {
        if (l < 1) continue;
        const int n = t.op[l].ncoef * (int)t.op[l].g.nx, n16 = n * (int)sizeof(SI) / 16, per = 16 / (int)sizeof(SI);
        SI* dst = reinterpret_cast<SI*>(tail_smem + t.sten_off[l]);
        const SI* src = t.op[l].sten;
        for (int i = tid; i < n16; i += nt) reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(src)[i];
        for (int i = n16 * per + tid; i < n; i += nt) dst[i] = src[i];
    }
    {
        const Geo& g = t.op[lc].g;
        A* X = sm + t.off[lc];
        A* Bv = X + 2 * g.nx;
        View<SI> bs = view_of(bv, b, 0, g.n0);
        const bool has = xin.d != nullptr;
        View<SI> xs = has ? view_of(xin, b, 0, g.n0) : View<SI>{nullptr, nullptr, g.n0};
        for (int p = tid; p < g.nx; p += nt) {
            int c = p % g.n0, row = p / g.n0;
            Bv[p] = bs.at(row, c);
            X[p] = has ? xs.at(row, c) : A(0);
        }
    }
    __syncthreads();
    bool xzero = xin.d == nullptr;
    for (int l = lc; l < L - 1; ++l) {
        const LevelOp<SI> op = tail_op(t, l, tail_smem);
        const Geo& gf = op.g;
        const Geo& gc = t.op[l + 1].g;
        if (t.nu1 > 0) {
            tail_smooth(t, l, sm, t.nu1, xzero, cur);
            xzero = false;
        }
        A* X0 = sm + t.off[l];
        const A* Xf = X0 + (long long)((cur >> (l)) & 1u) * gf.nx;
        A* Rf = X0 + (long long)(1 - ((cur >> (l)) & 1u)) * gf.nx;   // the free x buffer holds the residual
        const A* Bv = X0 + 2 * gf.nx;
        A* Xc = sm + t.off[l + 1];
        A* Bc = Xc + 2 * gc.nx;
        if (xzero) {
            for (int p = tid; p < gf.nx; p += nt) Rf[p] = Bv[p];
        } else {
            View<A> xv{Xf, nullptr, gf.n0};
            for (int p = tid; p < gf.nx; p += nt) {
                int c = p % gf.n0;
                long long row = p / gf.n0;
                int j, k;
    row_jk(gf, row, j, k);
                A Au, dg;
                if (op.fine) level_apply(op, xv, row, j, k, c, Au, dg);
                else level_apply_k<3>(op, xv, row, j, k, c, Au, dg);
                Rf[p] = Bv[p] - Au;
            }
        }
        __syncthreads();
        for (int P = tid; P < gc.nx; P += nt) {
            int I = P % gc.n0;
            long long crow = P / gc.n0;
            int J, Kc;
    row_jk(gc, crow, J, Kc);
            A acc = A(0);
            const int zlo = gf.d == 3 ? -1 : 0, zhi = gf.d == 3 ? 1 : 0;
            for (int dz = zlo; dz <= zhi; ++dz) {
                int fk = gf.d == 3 ? 2 * Kc + 1 + dz : 0;
                if (fk < 0 || fk >= gf.n2) continue;
                A wz = dz == 0 ? A(1) : A(0.5);
                for (int dy = -1; dy <= 1; ++dy) {
                    int fj = 2 * J + 1 + dy;
                    if (fj < 0 || fj >= gf.n1) continue;
                    A wy = dy == 0 ? A(1) : A(0.5);
                    long long frow = fj + (long long)gf.n1 * fk;
                    for (int dx = -1; dx <= 1; ++dx) {
                        int fi = 2 * I + 1 + dx;
                        if (fi < 0 || fi >= gf.n0) continue;
                        A wx = dx == 0 ? A(1) : A(0.5);
                        acc += wx * wy * wz * Rf[frow * gf.n0 + fi];
                    }
                }
            }
            Bc[P] = acc;
            Xc[P] = A(0);      // coarse levels start from zero (buffer 0)
        }
        __syncthreads();
        xzero = true;
    }
    {
        const Geo& g = t.op[L - 1].g;
        A* X = sm + t.off[L - 1] + (long long)((cur >> (L - 1)) & 1u) * g.nx;
        const A* Bv = sm + t.off[L - 1] + 2 * g.nx;
        const int nc = (int)g.nx, w = tid >> 5, lane = tid & 31, nw = nt >> 5;
        for (int p = w; p < nc; p += nw) {         // a warp per row of the inverse
            const A* D = t.Dinv + (long long)p * nc;
            A acc = A(0);
#pragma unroll 4
            for (int q = lane; q < nc; q += kWarp) acc += D[q] * Bv[q];
            acc = warp_sum(acc);
            if (lane == 0) X[p] = acc;
        }
    }
    __syncthreads();
    for (int l = L - 2; l >= lc; --l) {
        const Geo& gf = t.op[l].g;
        const Geo& gc = t.op[l + 1].g;
        A* X = sm + t.off[l] + (long long)((cur >> (l)) & 1u) * gf.nx;
        const A* Xc = sm + t.off[l + 1] + (long long)((cur >> (l + 1)) & 1u) * gc.nx;
        for (int p = tid; p < gf.nx; p += nt) {
            int c = p % gf.n0;
            long long row = p / gf.n0;
            int j, k;
    row_jk(gf, row, j, k);
            int Jx[2], Jy[2], Jz[2] = {0, 0};
            float wx[2], wy[2], wz[2] = {1.f, 0.f};
            int mx = interp_1d(c, gc.n0, Jx, wx);
            int my = interp_1d(j, gc.n1, Jy, wy);
            int mz = gf.d == 3 ? interp_1d(k, gc.n2, Jz, wz) : 1;
            A acc = X[p];
            for (int a = 0; a < mz; ++a)
                for (int q = 0; q < my; ++q)
                    for (int e = 0; e < mx; ++e)
                        acc += A(wz[a]) * A(wy[q]) * A(wx[e]) * Xc[(Jz[a] * (long long)gc.n1 + Jy[q]) * gc.n0 + Jx[e]];
            X[p] = acc;
        }
        __syncthreads();
        if (t.nu2 > 0) tail_smooth(t, l, sm, t.nu2, false, cur);
    }
    // write level lc
    {
        const Geo& g = t.op[lc].g;
        const A* X = sm + t.off[lc] + (long long)((cur >> (lc)) & 1u) * g.nx;
        const int w = tid >> 5, lane = tid & 31, nw = nt >> 5;
        for (long long row = w; row < g.R; row += nw) {
            SI* o;
            float* osc;
            row_store_ptrs(xout, b, 0, row, g.n0, o, osc);
            row_store<SI>(o, osc, g.n0, lane, [&](int c) -> A { return X[row * g.n0 + c]; });
        }
    }
}

// ---------------------------------------------------------------------------
// 2D specialisation of the fused tail: a 32 x 32 thread block maps (column,
// row) directly, stencils are the unrolled 9-point (stored) or 5-point
// (matrix-free fine level) forms.  Same levels, buffers and arithmetic as
// k_vcycle_tail; only the indexing work per point is smaller.
// ---------------------------------------------------------------------------
template <class SI>
__device__ __forceinline__ typename PT<SI>::A tail2d_apply(const LevelOp<SI>& op, const typename PT<SI>::A* X, int c,
                                                           int j, typename PT<SI>::A& diag) {
    using A = typename PT<SI>::A;
    const Geo& g = op.g;
    const int n0 = g.n0, n1 = g.n1;
    if (op.fine) {
        A Au, dg;
        View<A> xv{X, nullptr, n0};
        level_apply(op, xv, j, j, 0, c, Au, dg);
        diag = dg;
        return Au;
    }
    const long long p = (long long)j * n0 + c;
    A acc = A(0);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
        const int jj = j + dy;
        if (jj < 0 || jj >= n1) continue;
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
            const int cc = c + dx;
            if (cc < 0 || cc >= n0) continue;
            acc += sten_coef(op, (dx + 1) + 3 * (dy + 1), p) * X[jj * n0 + cc];
        }
    }
    diag = sten_coef(op, 4, p);
    return acc;
}

template <class SI>
__device__ __forceinline__ void tail2d_smooth(const TailCtx<SI>& t, int l, typename PT<SI>::A* sm, int sweeps,
                                              bool zero_first, unsigned& curbits) {
    int cur = (curbits >> l) & 1u;
    using A = typename PT<SI>::A;
    const LevelOp<SI> op = tail_op(t, l, reinterpret_cast<const unsigned char*>(sm));
    const Geo& g = op.g;
    A* X0 = sm + t.off[l];
    const A* Bv = X0 + 2 * g.nx;
    for (int sw = 0; sw < sweeps; ++sw) {
        const bool zero = zero_first && sw == 0;
        const A* Xc = X0 + (long long)cur * g.nx;
        A* Xn = X0 + (long long)(1 - cur) * g.nx;
        for (int j = threadIdx.y; j < g.n1; j += blockDim.y)
            for (int c = threadIdx.x; c < g.n0; c += blockDim.x) {
                const int p = j * g.n0 + c;
                if (zero) {
                    Xn[p] = t.omega * Bv[p] / level_diag(op, j, j, 0, c);
                } else {
                    A dg;
                    const A Au = tail2d_apply(op, Xc, c, j, dg);
                    Xn[p] = Xc[p] + t.omega * (Bv[p] - Au) / dg;
                }
            }
        cur = 1 - cur;
        __syncthreads();
    }
    curbits = (curbits & ~(1u << l)) | ((unsigned)cur << l);
}

template <class SI>
__global__ void __launch_bounds__(1024) k_vcycle_tail_2d(TailCtx<SI> t, int B, const int* active, Vec<SI> bv,
                                                         Vec<SI> xin, Vec<SI> xout) {
    pdl_prologue();
    using A = typename PT<SI>::A;
    extern __shared__ __align__(16) unsigned char tail_smem[];
    A* sm = reinterpret_cast<A*>(tail_smem);
    const int b = blockIdx.x;
    if (b >= B || (active && !active[b])) return;
    const int tx = threadIdx.x, ty = threadIdx.y, bx = blockDim.x, by = blockDim.y;
    const int tid = ty * bx + tx, nt = bx * by;
    const int lc = t.lc, L = t.L;
    unsigned cur = 0u;      // bit l: which of level l's two x buffers holds the iterate
    for (int l = t.stage_from; l < L; ++l) {
        if (l < 1) continue;
        const int n = t.op[l].ncoef * (int)t.op[l].g.nx;
        SI* dst = reinterpret_cast<SI*>(tail_smem + t.sten_off[l]);
        for (int i = tid; i < n; i += nt) dst[i] = t.op[l].sten[i];
    }
    {
        const Geo& g = t.op[lc].g;
        A* X = sm + t.off[lc];
        A* Bv = X + 2 * g.nx;
        View<SI> bs = view_of(bv, b, 0, g.n0);
        const bool has = xin.d != nullptr;
        View<SI> xs = has ? view_of(xin, b, 0, g.n0) : View<SI>{nullptr, nullptr, g.n0};
        for (int j = ty; j < g.n1; j += by)
            for (int c = tx; c < g.n0; c += bx) {
                const int p = j * g.n0 + c;
                Bv[p] = bs.at(j, c);
                X[p] = has ? xs.at(j, c) : A(0);
            }
    }
    __syncthreads();
    bool xzero = xin.d == nullptr;
    for (int l = lc; l < L - 1; ++l) {
        const LevelOp<SI> op = tail_op(t, l, tail_smem);
        const Geo& gf = op.g;
        const Geo& gc = t.op[l + 1].g;
        if (t.nu1 > 0) {
            tail2d_smooth(t, l, sm, t.nu1, xzero, cur);
            xzero = false;
        }
        A* X0 = sm + t.off[l];
        const A* Xf = X0 + (long long)((cur >> (l)) & 1u) * gf.nx;
        A* Rf = X0 + (long long)(1 - ((cur >> (l)) & 1u)) * gf.nx;
        const A* Bv = X0 + 2 * gf.nx;
        for (int j = ty; j < gf.n1; j += by)
            for (int c = tx; c < gf.n0; c += bx) {
                const int p = j * gf.n0 + c;
                if (xzero) {
                    Rf[p] = Bv[p];
                } else {
                    A dg;
                    Rf[p] = Bv[p] - tail2d_apply(op, Xf, c, j, dg);
                }
            }
        __syncthreads();
        A* Xc = sm + t.off[l + 1];
        A* Bc = Xc + 2 * gc.nx;
        for (int J = ty; J < gc.n1; J += by)
            for (int I = tx; I < gc.n0; I += bx) {
                A acc = A(0);
#pragma unroll
                for (int dy = -1; dy <= 1; ++dy) {
                    const int fj = 2 * J + 1 + dy;
                    if (fj < 0 || fj >= gf.n1) continue;
                    const A wy = dy == 0 ? A(1) : A(0.5);
#pragma unroll
                    for (int dx = -1; dx <= 1; ++dx) {
                        const int fi = 2 * I + 1 + dx;
                        if (fi < 0 || fi >= gf.n0) continue;
                        const A wx = dx == 0 ? A(1) : A(0.5);
                        acc += wx * wy * Rf[fj * gf.n0 + fi];
                    }
                }
                Bc[J * gc.n0 + I] = acc;
                Xc[J * gc.n0 + I] = A(0);
            }
        __syncthreads();
        xzero = true;
    }
    {
        const Geo& g = t.op[L - 1].g;
        A* X = sm + t.off[L - 1] + (long long)((cur >> (L - 1)) & 1u) * g.nx;
        const A* Bv = sm + t.off[L - 1] + 2 * g.nx;
        const int nc = (int)g.nx;
        for (int p = tid; p < nc; p += nt) {
            A acc = A(0);
            for (int q = 0; q < nc; ++q) acc += t.Dinv[(long long)p * nc + q] * Bv[q];
            X[p] = acc;
        }
    }
    __syncthreads();
    for (int l = L - 2; l >= lc; --l) {
        const Geo& gf = t.op[l].g;
        const Geo& gc = t.op[l + 1].g;
        A* X = sm + t.off[l] + (long long)((cur >> (l)) & 1u) * gf.nx;
        const A* Xc = sm + t.off[l + 1] + (long long)((cur >> (l + 1)) & 1u) * gc.nx;
        for (int j = ty; j < gf.n1; j += by) {
            int Jy[2];
            float wy[2];
            const int my = interp_1d(j, gc.n1, Jy, wy);
            for (int c = tx; c < gf.n0; c += bx) {
                int Jx[2];
                float wx[2];
                const int mx = interp_1d(c, gc.n0, Jx, wx);
                A acc = X[j * gf.n0 + c];
                for (int q = 0; q < my; ++q)
                    for (int e = 0; e < mx; ++e) acc += A(wy[q]) * A(wx[e]) * Xc[Jy[q] * gc.n0 + Jx[e]];
                X[j * gf.n0 + c] = acc;
            }
        }
        __syncthreads();
        if (t.nu2 > 0) tail2d_smooth(t, l, sm, t.nu2, false, cur);
    }
    {
        const Geo& g = t.op[lc].g;
        const A* X = sm + t.off[lc] + (long long)((cur >> (lc)) & 1u) * g.nx;
        const int w = tid >> 5, lane = tid & 31, nw = nt >> 5;
        for (long long row = w; row < g.R; row += nw) {
            SI* o;
            float* osc;
            row_store_ptrs(xout, b, 0, row, g.n0, o, osc);
            row_store<SI>(o, osc, g.n0, lane, [&](int c) -> A { return X[row * g.n0 + c]; });
        }
    }
}

}  // namespace aao
