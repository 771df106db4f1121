// The FP64 all-at-once product of the finite-difference discretisation, apart from krylov.cuh so that its instances are
// compiled once (solver.cu).
#pragma once

#include <type_traits>

#include "common.cuh"
#include "krylov.cuh"

namespace aao {

// ---------------------------------------------------------------------------
// FP64 all-at-once matvec (FD, M = I), one thread per (time block n, point):
//   y_{v,0}   = v_0
//   y_{v,n+1} = v_{n+1} - v_n - tau sum_i b_i V_{n,i}
//   y_{V,n,i} = V_{n,i} + K v_n + tau sum_j a_ij K V_{n,j}
// and its transpose
//   y_{v,n}   = l_{v,n} - l_{v,n+1} + sum_i K l_{V,n,i}   (n < nt),  y_{v,nt} = l_{v,nt}
//   y_{V,n,i} = l_{V,n,i} - tau b_i l_{v,n+1} + tau sum_j a_ji K l_{V,n,j}.
// rhs != nullptr gives y = rhs - (A x).  Time block nt stands for v_0 / v_nt.
// skip != nullptr: the launch does nothing when *skip is nonzero (the relaxed outer product kept
// its FP32 result, k_relax_decide).
// Bound by FP64 arithmetic (two operations per cycle and SM): so tau a_ij and tau b_i are formed on the host,
// K's differences stay as they are (2 P - W - E is exact for smooth fields; merging the stages before K would
// save five operations of 41 but round those sums) and, where the mesh is square, the factor 1/h^2 is part of
// tau a_ij instead of multiplying every difference (36).  K v, the largest term of a stage's row, is added last, so one
// rounding of the row's size is left (rms error of the stages 0.89e-16; with K v first 1.21e-16).  Every load of a thread is issued
// before its arithmetic; a warp per row with its columns in a loop left the FP64 pipe idle for a third of the time.
// Measured: 256^2, s = 3, 128 steps 905 -> 655 us (36 operations per point and block: 0.46 TFMA/s of 0.60);
// 49 x 45 x 41 with faces, s = 2, 24 steps, transposed 256 -> 141 us; 32^2, 16 steps 5.5 -> 4.2 us.
// ---------------------------------------------------------------------------
constexpr int kMvThreads = 128;

struct MvTab {
    double A[kMaxS * kMaxS], b[kMaxS];   // tau a_ij (transpose: tau a_ji), on square meshes times 1 / h^2; tau b_i
    double h2;                           // square meshes: 1 / h^2 (the differences are unscaled), else 1
    double hx2, hy2, hz2;                // factors of the differences (square meshes: 1)
};

// Sum of the scaled differences of u at a point, from its P and neighbours.
template <int D, bool FACES, bool SQUARE>
__device__ __forceinline__ double mv_K(const double* nb, const double* f, const MvTab& t) {
    if constexpr (FACES) {
        double k = f[0] * (nb[0] - nb[1]);
#pragma unroll
        for (int q = 1; q < 2 * D; ++q) k += f[q] * (nb[0] - nb[q + 1]);
        return k;
    } else if constexpr (SQUARE) {
        double k = 2.0 * nb[0] - nb[1];
        k -= nb[2];
#pragma unroll
        for (int a = 1; a < D; ++a) k += (2.0 * nb[0] - nb[2 * a + 1]) - nb[2 * a + 2];
        return k;
    } else {
        double k = t.hx2 * ((2.0 * nb[0] - nb[1]) - nb[2]);
        k += t.hy2 * ((2.0 * nb[0] - nb[3]) - nb[4]);
        if (D == 3) k += t.hz2 * ((2.0 * nb[0] - nb[5]) - nb[6]);
        return k;
    }
}

template <int D, bool FACES, bool SQUARE, int TS, bool TRANS>
__global__ void __launch_bounds__(kMvThreads) k_matvec(Geo g, int nt, int stages, const __grid_constant__ MvTab tab,
                                                       Faces<double> faces, const double* x, double* y,
                                                       const double* rhs, const int* skip) {
    pdl_prologue();
    if (skip && *skip) return;
    // The stage count as a constant where that is faster.  In the forward product without faces and in the transposed one with
    // faces, checks against a variable keep every load ahead of the sums, which the compiler otherwise moves between them
    // to save registers (forward 40 instead of 56; 64^2, s = 3, 32 steps 19.2 us instead of 15.2; transposed with faces 24^3,
    // s = 2, 8 steps 13.8 instead of 11.8; from 128^2 on 1% either way).  The others: forward with faces 256^2, s = 2, 64
    // steps 254 us instead of 261; transposed without faces 64^2, s = 2 7.8 instead of 10.0.
    const int s = TS < kMaxS && FACES != TRANS ? TS : stages;
    const unsigned p = blockIdx.x * kMvThreads + threadIdx.x;
    if (p >= (unsigned)g.nx) return;
    const int n = blockIdx.y;
    const long long nx = g.nx;
    const long long voff = (long long)(nt + 1) * nx;
    if (n == nt) {   // y_{v,0} (forward) or y_{v,nt} (transpose)
        const long long i = (TRANS ? (long long)nt * nx : 0) + p;
        y[i] = rhs ? rhs[i] - x[i] : x[i];
        return;
    }
    const unsigned row = p / (unsigned)g.n0;
    const int c = (int)(p - row * g.n0);
    int j, k;
    row_jk(g, row, j, k);
    // neighbours west, east, south, north (down, up): inside the grid or zero
    bool in[2 * D];
    int off[2 * D];
    in[0] = c > 0;
    in[1] = c + 1 < g.n0;
    in[2] = j > 0;
    in[3] = j + 1 < g.n1;
    off[0] = -1;
    off[1] = 1;
    off[2] = -g.n0;
    off[3] = g.n0;
    if constexpr (D == 3) {
        in[4] = k > 0;
        in[5] = k + 1 < g.n2;
        off[4] = -g.n0 * g.n1;
        off[5] = g.n0 * g.n1;
    }
    auto load = [&](const double* u, double* nb) {
        nb[0] = u[0];
#pragma unroll
        for (int q = 0; q < 2 * D; ++q) nb[q + 1] = in[q] ? u[off[q]] : 0.0;
    };
    const double* xv = x + (long long)n * nx + p;
    const double* xV = x + voff + (long long)n * s * nx + p;
    double V[TS][2 * D + 1], v[2 * D + 1], f[2 * D];
    v[0] = xv[0];
    if constexpr (!TRANS) load(xv, v);
    const double v1 = xv[nx];
#pragma unroll
    for (int i = 0; i < TS; ++i)
        if (i < s) load(xV + (long long)i * nx, V[i]);
    if constexpr (FACES) {
        const long long fxi = (long long)row * (g.n0 + 1) + c;
        const long long fyi = ((long long)k * (g.n1 + 1) + j) * g.n0 + c;
        f[0] = faces.fx[fxi];
        f[1] = faces.fx[fxi + 1];
        f[2] = faces.fy[fyi];
        f[3] = faces.fy[fyi + g.n0];
        if constexpr (D == 3) {
            f[4] = faces.fz[p];
            f[5] = faces.fz[p + (long long)g.n1 * g.n0];
        }
    }
    double K[TS];
#pragma unroll
    for (int i = 0; i < TS; ++i)
        if (i < s) K[i] = mv_K<D, FACES, SQUARE>(V[i], f, tab);
    double Kv = 0.0;
    if constexpr (!TRANS) Kv = mv_K<D, FACES, SQUARE>(v, f, tab);
    auto put = [&](long long at, double a) { y[at] = rhs ? rhs[at] - a : a; };
    double acc;
    if constexpr (!TRANS) {
        acc = v1 - v[0];
#pragma unroll
        for (int i = 0; i < TS; ++i)
            if (i < s) acc -= tab.b[i] * V[i][0];
        put((long long)(n + 1) * nx + p, acc);
    } else {
        acc = 0.0;
#pragma unroll
        for (int i = 0; i < TS; ++i)
            if (i < s) acc += K[i];
        acc = v[0] - v1 + (SQUARE ? tab.h2 * acc : acc);
        put((long long)n * nx + p, acc);
    }
#pragma unroll
    for (int i = 0; i < TS; ++i)
        if (i < s) {
            double a = TRANS ? V[i][0] - tab.b[i] * v1 : V[i][0];
#pragma unroll
            for (int q = 0; q < TS; ++q)
                if (q < s) a += tab.A[i * s + q] * K[q];
            if constexpr (!TRANS) a += SQUARE ? tab.h2 * Kv : Kv;
            put(voff + ((long long)n * s + i) * nx + p, a);
        }
}

// The product's instance for a handle's grid and stages.
inline void launch_matvec(const Geo& g, int nt, const Tab& tab, double tau, const Faces<double>& faces, const double* x,
                          double* y, const double* rhs, int transpose, const int* skip, cudaStream_t st) {
    MvTab t{};
    const int s = tab.s;
    for (int i = 0; i < s; ++i) {
        t.b[i] = tau * tab.b[i];
        for (int q = 0; q < s; ++q) t.A[i * s + q] = tau * (transpose ? tab.A[q * s + i] : tab.A[i * s + q]);
    }
    const bool square = faces.fx == nullptr && g.hx2 == g.hy2 && (g.d == 2 || g.hz2 == g.hx2);
    if (square)
        for (int i = 0; i < s * s; ++i) t.A[i] *= g.hx2;
    t.h2 = g.hx2;
    t.hx2 = g.hx2;
    t.hy2 = g.hy2;
    t.hz2 = g.hz2;
    const dim3 grid((unsigned)((g.nx + kMvThreads - 1) / kMvThreads), (unsigned)nt + 1);
    auto pick = [&](auto d, auto fc, auto sq, auto ts, auto tr) {
        launch(k_matvec<decltype(d)::value ? 3 : 2, decltype(fc)::value, decltype(sq)::value, decltype(ts)::value,
                        decltype(tr)::value>,
               grid, kMvThreads, 0, st, g, nt, s, t, faces, x, y, rhs, skip);
    };
    auto by = [](bool v, auto&& f) {
        if (v) f(std::true_type{});
        else f(std::false_type{});
    };
    // An instance per stage count up to four: a stage's predicated-off operations take their turns of the FP64 pipe
    // too (s = 1 in an instance for up to three stages: 128^2, 32 steps 41.7 us instead of 28.2, transposed 36.7 instead
    // of 22.9; s = 4 in the one for up to eight: 106 instead of 66).
    auto stages = [&](auto&& f) {
        if (s == 1) f(std::integral_constant<int, 1>{});
        else if (s == 2) f(std::integral_constant<int, 2>{});
        else if (s == 3) f(std::integral_constant<int, 3>{});
        else if (s == 4) f(std::integral_constant<int, 4>{});
        else f(std::integral_constant<int, kMaxS>{});
    };
    by(g.d == 3, [&](auto d) {
        stages([&](auto ts) {
            by(transpose != 0, [&](auto tr) {
                if (faces.fx) pick(d, std::true_type{}, std::false_type{}, ts, tr);
                else by(square, [&](auto sq) { pick(d, std::false_type{}, sq, ts, tr); });
            });
        });
    });
}

}  // namespace aao
