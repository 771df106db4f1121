// The inner GMRES of P_tilde (Theta_tilde's batched solves and the steps of S_tilde) in three
// launches per Krylov step around the preconditioner:
//   k_theta_dots   w = Theta_hat z_k, with every inner product the orthogonalisation needs
//   k_arnoldi_upd  w -= sum_i h_i v_i and ||w||, then the Givens update of the item's least-squares
//                  problem and, when the item is done, its solution
//   k_scale_vec    v_{k+1} = w / ||w||
//
// Orthogonalisation.  Modified Gram--Schmidt takes h_i = v_i . (w - sum_{j<i} h_j v_j), one pass over
// w and two basis vectors per i.  Written out, (I + L) h = V^T w with L the strictly lower part of
// V^T V (the inverse compact WY form of modified Gram--Schmidt): the k + 1 products v_i . w and the
// k products v_k . v_i of the newest basis vector come from one pass, the triangular system is solved
// per item by the last block to finish, and a second pass applies all updates.  The same h as the
// step-by-step form for any stored basis, orthonormal or not.  Before: k + 2 launches and
// 4 k + 5 vector passes for step k; now 2 launches and 2 k + 4 passes.
//
// What bounds them: at large batches memory, at one item the launch and the reduction's two trips
// through L2.  FP64 runs at 1/58 of the FP32 rate on this GPU and conversions between the two share
// that pipe, so tableau coefficients are rounded once per block instead of per point, and in FP32 only the sums
// of a reduction and K z of S_tilde's recurrence are FP64.
#pragma once

#include <type_traits>

#include "krylov.cuh"

namespace aao {

constexpr int kArThreads = 128;
constexpr int kArWarps = kArThreads / kWarp;
constexpr int kArBlocks = 152 * 48;      // blocks of a reducing launch over the whole batch: beyond three or so
                                         // per thread slot, positions are chained per thread (128 blocks of 256^2
                                         // in k_theta_dots: 277 us with eight blocks per SM)
constexpr int kArSmallK = 5;             // inner iterations of the small instance (the defaults: 3 and 5)

// N consecutive stored values as arithmetic values: one 8- or 16-byte load where N values make one
// (the address aligned to it), else N loads.
template <int N, class S>
__device__ __forceinline__ void ld_n(const S* p, typename PT<S>::A* out) {
    if constexpr (N * sizeof(S) == 16) {
        const uint4 v = *reinterpret_cast<const uint4*>(p);
        const S* q = reinterpret_cast<const S*>(&v);
#pragma unroll
        for (int t = 0; t < N; ++t) out[t] = PT<S>::ld(q[t]);
    } else if constexpr (N * sizeof(S) == 8 && N > 1) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        const S* q = reinterpret_cast<const S*>(&v);
#pragma unroll
        for (int t = 0; t < N; ++t) out[t] = PT<S>::ld(q[t]);
    } else {
#pragma unroll
        for (int t = 0; t < N; ++t) out[t] = PT<S>::ld(p[t]);
    }
}
template <int N, class A> __device__ __forceinline__ void st_n(A* p, const A* v) {
    if constexpr (N * sizeof(A) == 16) {
        uint4 o;
        A* q = reinterpret_cast<A*>(&o);
#pragma unroll
        for (int t = 0; t < N; ++t) q[t] = v[t];
        *reinterpret_cast<uint4*>(p) = o;
    } else {
#pragma unroll
        for (int t = 0; t < N; ++t) p[t] = v[t];
    }
}

// One stage of one item: rows of n0 values with their scales.
template <class S> struct Field {
    const S* d;
    const float* sc;
    int n0;
    template <int N> __device__ __forceinline__ void row_n(int row, int c, typename PT<S>::A* out) const {
        ld_n<N>(d + (long long)row * n0 + c, out);
        if constexpr (PT<S>::scaled) {
            const float f = sc[row];
#pragma unroll
            for (int t = 0; t < N; ++t) out[t] *= f;
        }
    }
    __device__ __forceinline__ typename PT<S>::A at(int row, int c) const {
        typename PT<S>::A v = PT<S>::ld(d[(long long)row * n0 + c]);
        if constexpr (PT<S>::scaled) v *= sc[row];
        return v;
    }
};

// Stage i of item b; rows_b rows per item.
template <class S>
__device__ __forceinline__ Field<S> field_of(const Vec<S>& v, int b, long long rows_b, int i, const Geo& g) {
    Field<S> f;
    f.d = v.d + (long long)b * v.bs + (long long)i * g.nx;
    f.sc = PT<S>::scaled ? v.sc + (long long)b * rows_b + (long long)i * g.R : nullptr;
    f.n0 = g.n0;
    return f;
}

// (K u) at N consecutive columns of row (j, k), FD; P receives u there.  The arithmetic of fd_K.
template <int N, class S, class A>
__device__ __forceinline__ void fd_K_n(const Field<S>& u, const Geo& g, const InvH2<A>& h, const Faces<A>& f, int row,
                                       int j, int k, int c, A* P, A* K) {
    A So[N], No[N], Do[N], Up[N];
#pragma unroll
    for (int t = 0; t < N; ++t) So[t] = No[t] = Do[t] = Up[t] = A(0);
    u.template row_n<N>(row, c, P);
    if (j > 0) u.template row_n<N>(row - 1, c, So);
    if (j + 1 < g.n1) u.template row_n<N>(row + 1, c, No);
    if (g.d == 3) {
        if (k > 0) u.template row_n<N>(row - g.n1, c, Do);
        if (k + 1 < g.n2) u.template row_n<N>(row + g.n1, c, Up);
    }
    const A w = c > 0 ? u.at(row, c - 1) : A(0), e = c + N < g.n0 ? u.at(row, c + N) : A(0);
    if (f.fx == nullptr) {
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const A W = t == 0 ? w : P[t - 1], E = t == N - 1 ? e : P[t + 1];
            K[t] = h.x * (A(2) * P[t] - W - E) + h.y * (A(2) * P[t] - So[t] - No[t]);
            if (g.d == 3) K[t] += h.z * (A(2) * P[t] - Do[t] - Up[t]);
        }
    } else {
        const A* fx = f.fx + (long long)row * (g.n0 + 1) + c;
        const long long fyi = ((long long)k * (g.n1 + 1) + j) * g.n0 + c;
        A fs[N], fn[N];
        ld_n<N>(f.fy + fyi, fs);
        ld_n<N>(f.fy + fyi + g.n0, fn);
#pragma unroll
        for (int t = 0; t < N; ++t) {
            const A W = t == 0 ? w : P[t - 1], E = t == N - 1 ? e : P[t + 1];
            K[t] = fx[t] * (P[t] - W) + fx[t + 1] * (P[t] - E) + fs[t] * (P[t] - So[t]) + fn[t] * (P[t] - No[t]);
        }
        if (g.d == 3) {
            const long long fzi = ((long long)k * g.n1 + j) * g.n0 + c;
            A fd[N], fu[N];
            ld_n<N>(f.fz + fzi, fd);
            ld_n<N>(f.fz + fzi + (long long)g.n1 * g.n0, fu);
#pragma unroll
            for (int t = 0; t < N; ++t) K[t] += fd[t] * (P[t] - Do[t]) + fu[t] * (P[t] - Up[t]);
        }
    }
}

// M u and K u of Q1 at one point, one pass over the 3^d neighbours.
template <class S, class A>
__device__ __forceinline__ void q1_both(const Field<S>& u, const Geo& g, const Q1<A>& q, int row, int j, int k, int c,
                                        A& Mu, A& Ku) {
    Mu = A(0);
    Ku = A(0);
    const int zlo = g.d == 3 ? -1 : 0, zhi = g.d == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz) {
        if (k + dz < 0 || k + dz >= g.n2) continue;
        const A mz = g.d == 3 ? q.m[2][dz + 1] : A(1), kz = g.d == 3 ? q.k[2][dz + 1] : A(0);
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            if (j + dy < 0 || j + dy >= g.n1) continue;
            const A my = q.m[1][dy + 1], ky = q.k[1][dy + 1];
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                if (c + dx < 0 || c + dx >= g.n0) continue;
                const A mx = q.m[0][dx + 1], kx = q.k[0][dx + 1];
                A kc = kx * my * mz + mx * ky * mz;
                if (g.d == 3) kc += mx * my * kz;
                const A v = u.at(row + dy + dz * g.n1, c + dx);
                Mu += mx * my * mz * v;
                Ku += kc * v;
            }
        }
    }
}

// (M u, K u) at N columns: Q1 (N = 1) or FD (M = I).
template <int N, class S, class A>
__device__ __forceinline__ void op_MK_n(const Field<S>& u, const Geo& g, const InvH2<A>& h, const SpaceOp<A>& op,
                                        int row, int j, int k, int c, A* M, A* K) {
    if constexpr (N == 1) {
        if (op.q1) {
            q1_both(u, g, op.q, row, j, k, c, M[0], K[0]);
            return;
        }
    }
    fd_K_n<N>(u, g, h, op.faces, row, j, k, c, M, K);
}

// The Krylov basis of a batch: vector m of item b is v.d + m * stride + b * v.bs, `rows` rows of n0.
template <class S> struct Basis {
    Vec<S> v;
    long long stride, rows, srows;     // elements per basis vector; rows per item; stride / n0
    __device__ __forceinline__ const S* at(int m, int b) const { return v.d + m * stride + (long long)b * v.bs; }
    __device__ __forceinline__ const float* scale(int m, int b) const { return v.sc + m * srows + (long long)b * rows; }
};

// Reduction scratch of one preconditioner: nchunk blocks per item, up to nv values per block.
struct ArRed {
    double* part;          // items * nchunk * nv
    unsigned int* count;   // items, zero between launches
    int nchunk;
};

// float -> double by integer operations (an FP64 conversion costs as much as an FP64 operation).
__device__ __forceinline__ double to_fp64(float v) {
    const unsigned u = __float_as_uint(v), e = u >> 23 & 255u;
    if (e - 1u >= 254u) return (double)v;                     // zero, subnormal, infinity, NaN
    return __hiloint2double((int)((u & 0x80000000u) | (e + 896u) << 20 | (u >> 3 & 0xfffffu)), (int)(u << 29));
}
__device__ __forceinline__ double to_fp64(double v) { return v; }

// Sum the values chosen by `mask` over the blocks of item blockIdx.y: the last block to arrive has the
// sums in sum[] (shared memory) and gets true.  Partial sums are added in chunk order, so the result does
// not depend on scheduling.  preload() runs in that block beside the loads of the partial sums (all
// threads; visible to all on return): the item's state comes in the same trip to L2.
template <int MV, class A, class F>
__device__ __forceinline__ bool ar_reduce(const A* v, unsigned mask, const ArRed& red, double* sum, F&& preload) {
    // FP64 adds run at two per cycle and SM, and summing each value by shuffles in every warp would take longer than
    // the launch's other work (45 us of k_theta_dots on 128 items of 256^2): so the threads' FP32 values meet in
    // shared memory and one warp per value adds four per lane before its shuffles, 8 adds per value instead of 23.
    constexpr bool kF32 = std::is_same<A, float>::value;
    __shared__ A sh[MV][kF32 ? kArThreads : kArWarps];
    __shared__ bool last;
    const int w = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
#pragma unroll
    for (int i = 0; i < MV; ++i)
        if (mask >> i & 1u) {
            if constexpr (kF32) {
                sh[i][threadIdx.x] = v[i];
            } else {
                const double t = warp_sum(v[i]);
                if (lane == 0) sh[i][w] = t;
            }
        }
    __syncthreads();
    double* part = red.part + (long long)blockIdx.y * red.nchunk * MV;
    auto put = [&](int i, double t) {
        if (red.nchunk == 1) {
            sum[i] = t;                 // the block is the item's only one
        } else {
            part[(long long)blockIdx.x * MV + i] = t;
            __threadfence();
        }
    };
    if constexpr (kF32) {
        for (int i = w; i < MV; i += kArWarps) {
            if (!(mask >> i & 1u)) continue;
            static_assert(kArThreads == 4 * kWarp, "four values per lane");
            const A* s = sh[i] + lane;
            const double t = warp_sum((to_fp64(s[0]) + to_fp64(s[kWarp])) + (to_fp64(s[2 * kWarp]) + to_fp64(s[3 * kWarp])));
            if (lane == 0) put(i, t);
        }
    } else if (threadIdx.x < MV && (mask >> threadIdx.x & 1u)) {
        double t = 0.0;
        for (int i = 0; i < kArWarps; ++i) t += sh[threadIdx.x][i];
        put(threadIdx.x, t);
    }
    if (red.nchunk == 1) {
        preload();
        __syncthreads();
        return true;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(&red.count[blockIdx.y], 1u) == (unsigned)red.nchunk - 1;
        if (last) red.count[blockIdx.y] = 0;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    preload();
    for (int i = w; i < MV; i += kArWarps) {
        if (!(mask >> i & 1u)) continue;
        double t = 0.0;
        for (int c = lane; c < red.nchunk; c += kWarp) t += __ldcg(part + (long long)c * MV + i);
        t = warp_sum(t);
        if (lane == 0) sum[i] = t;
    }
    __syncthreads();
    return true;
}

// Per-item state of the batched inner GMRES (strides as in Precond).
struct ArItems {
    int kin;
    double *H, *cs, *sn, *g, *beta, *y, *gram;   // (kin+1)*kin, kin, kin, kin+1, 1, kin, kin*kin per item
    int *active, *its, *nonfinite, *breakdown;
    long long* count;                            // running total of iterations
    double tol;
};

// Start of an item with ||r|| = bt: done at once when it is zero (z = 0).
__device__ __forceinline__ void ar_init(const ArItems& it, int b, double bt) {
    const bool ok = isfinite(bt);
    if (!ok) atomicExch(it.nonfinite, 1);
    it.beta[b] = bt;
    it.its[b] = 0;
    it.g[(long long)b * (it.kin + 1)] = bt;
    const int act = ok && bt > 0.0;
    it.active[b] = act;
    if (!act)
        for (int i = 0; i < it.kin; ++i) it.y[(long long)b * it.kin + i] = 0.0;
}

// Shared-memory copy of an item's least-squares state: columns 0..k of the Hessenberg matrix, the
// rotations, the right-hand side.
template <int MK> struct ArState {
    double H[(MK + 1) * MK], cs[MK], sn[MK], g[MK + 1], beta;
    __device__ __forceinline__ void load(const ArItems& it, int b, int k) {
        const int kin = it.kin, tid = threadIdx.x;
        for (int i = tid; i < (k + 1) * kin; i += kArThreads) H[i] = it.H[(long long)b * (kin + 1) * kin + i];
        if (tid < k) {
            cs[tid] = it.cs[(long long)b * kin + tid];
            sn[tid] = it.sn[(long long)b * kin + tid];
        }
        if (tid <= k) g[tid] = it.g[(long long)b * (kin + 1) + tid];
        if (tid == 0) beta = it.beta[b];
    }
};

// Givens update of column k with h_{k+1,k} = hk1 (as k_givens), and the item's solution y = R^{-1} g when
// it is done.  One thread, a chain of FP64 operations on the state in shared memory.  hypot and two divisions, as
// in k_givens: products with one reciprocal square root would shorten the chain, but their rotations are less accurate
// (rms error of c 0.64 instead of 0.56 units of 2^-53).
template <int MK>
__device__ __forceinline__ void ar_givens(const ArItems& it, int b, int k, double hk1, ArState<MK>& s) {
    const int kin = it.kin;
    double* h = it.H + (long long)b * (kin + 1) * kin;
    double x = s.H[k];
    for (int i = 0; i < k; ++i) {
        const double lo = s.H[(i + 1) * kin + k];
        const double r = s.cs[i] * x + s.sn[i] * lo;
        x = -s.sn[i] * x + s.cs[i] * lo;
        s.H[i * kin + k] = r;
        h[i * kin + k] = r;
    }
    const double den = hypot(x, hk1);
    double cc = 1.0, ss = 0.0;
    if (den != 0.0) {
        cc = x / den;
        ss = hk1 / den;
    }
    const double gk = s.g[k], g1 = -ss * gk, g0 = cc * gk;
    s.H[k * kin + k] = den;
    h[k * kin + k] = den;
    h[(k + 1) * kin + k] = hk1;     // unrotated: the basis write divides by it
    it.cs[(long long)b * kin + k] = cc;
    it.sn[(long long)b * kin + k] = ss;
    it.g[(long long)b * (kin + 1) + k] = g0;
    it.g[(long long)b * (kin + 1) + k + 1] = g1;
    const double res = fabs(g1);
    it.its[b] = k + 1;
    const bool bad = !isfinite(res) || !isfinite(den);
    if (bad) atomicExch(it.nonfinite, 1);
    if (!(bad || res <= it.tol * s.beta || hk1 == 0.0 || k == kin - 1)) return;
    it.active[b] = 0;
    s.g[k] = g0;
    double* y = it.y + (long long)b * kin;
    for (int i = k; i >= 0; --i) {
        double t = s.g[i];
        for (int j = i + 1; j <= k; ++j) t -= s.H[i * kin + j] * s.g[j];
        const double d = s.H[i * kin + i];
        if (d == 0.0) {
            atomicExch(it.breakdown, 1);
            t = 0.0;
        } else {
            t /= d;
        }
        s.g[i] = t;                 // g_i is not read again: y takes its place
        y[i] = t;
    }
    for (int i = k + 1; i < kin; ++i) y[i] = 0.0;
    atomicAdd(reinterpret_cast<unsigned long long*>(it.count), (unsigned long long)(k + 1));
}

// ||src_b|| of contiguous items of n values and the start of their solves.
template <class SR>
__global__ void __launch_bounds__(kArThreads) k_ar_start(long long n, const SR* src, long long sbs, ArRed red,
                                                         ArItems it) {
    pdl_prologue();
    __shared__ double sum[1];
    const int b = blockIdx.y;
    const SR* x = src + (long long)b * sbs;
    const long long step = (long long)red.nchunk * kArThreads;
    SR acc = SR(0);
    long long i = (long long)blockIdx.x * kArThreads + threadIdx.x;
    for (; i + 3 * step < n; i += 4 * step) {
        SR v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = x[i + u * step];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc += v[u] * v[u];
    }
    for (; i < n; i += step) acc += x[i] * x[i];
    if (ar_reduce<1>(&acc, 1u, red, sum, [] {}) && threadIdx.x == 0) ar_init(it, b, sqrt(sum[0]));
}

// w = Theta_hat z_k:  w_i = M z_i + tau sum_j coef[i*s+j] K z_j  (coef = A_RK or its transpose), and
// h = (I + L)^{-1} V^T w into column k of the item's Hessenberg matrix.  A thread takes N consecutive
// columns of a row in every stage, so the s stages' loads are in flight together.  TS >= s stages and
// MK >= k + 1 basis vectors are unrolled.
template <class SZ, class SV, class A, int N, int TS, int MK>
__global__ void __launch_bounds__(kArThreads) k_theta_dots(Geo g, InvH2<A> hh, const int* active, Vec<SZ> Z, long long zrows,
                                                           A* wv, long long wbs, int s, const double* coef, A tau,
                                                           SpaceOp<A> sop, Basis<SV> V, int k, ArRed red,
                                                           ArItems it) {
    pdl_prologue();
    constexpr int MV = 2 * MK - 1;
    __shared__ A tc[TS * TS];
    __shared__ double sum[MV];
    const int b = blockIdx.y;
    if (!active[b]) return;
    for (int t = threadIdx.x; t < s * s; t += kArThreads) tc[t] = tau * (A)coef[t];
    __syncthreads();
    const unsigned nv = (unsigned)g.n0 / N;
    const unsigned npos = nv * (unsigned)g.R;
    A acc[MV];
#pragma unroll
    for (int i = 0; i < MV; ++i) acc[i] = A(0);
    for (unsigned q = blockIdx.x * kArThreads + threadIdx.x; q < npos; q += red.nchunk * kArThreads) {
        const int row = (int)(q / nv), c = (int)(q - row * nv) * N;
        int j, kk;
        row_jk(g, row, j, kk);
        A o[TS][N];
#pragma unroll
        for (int i = 0; i < TS; ++i)
#pragma unroll
            for (int t = 0; t < N; ++t) o[i][t] = A(0);
#pragma unroll
        for (int jj = 0; jj < TS; ++jj)
            if (jj < s) {
                A M[N], K[N];
                op_MK_n<N>(field_of(Z, b, zrows, jj, g), g, hh, sop, row, j, kk, c, M, K);
#pragma unroll
                for (int i = 0; i < TS; ++i)
                    if (i < s) {
                        const A a = tc[i * s + jj];
#pragma unroll
                        for (int t = 0; t < N; ++t) o[i][t] += i == jj ? M[t] + a * K[t] : a * K[t];
                    }
            }
        const long long p = (long long)row * g.n0 + c;
#pragma unroll
        for (int i = 0; i < TS; ++i)
            if (i < s) {
                st_n<N>(wv + (long long)b * wbs + (long long)i * g.nx + p, o[i]);
                A vk[N];
#pragma unroll
                for (int m = MK - 1; m >= 0; --m)
                    if (m <= k) {
                        A v[N];
                        const Field<SV> f{V.at(m, b) + (long long)i * g.nx,
                                          PT<SV>::scaled ? V.scale(m, b) + (long long)i * g.R : nullptr, g.n0};
                        f.template row_n<N>(row, c, v);
                        if (m == k) {
#pragma unroll
                            for (int t = 0; t < N; ++t) {
                                vk[t] = v[t];
                                acc[m] += v[t] * o[i][t];
                            }
                        } else {
#pragma unroll
                            for (int t = 0; t < N; ++t) {
                                acc[m] += v[t] * o[i][t];
                                if (m < MK - 1) acc[MK + m] += v[t] * vk[t];
                            }
                        }
                    }
            }
    }
    // values [0, k]: v_m . w; [MK, MK + k): v_k . v_m
    const unsigned mask = ((2u << k) - 1u) | (((1u << k) - 1u) << MK);
    const int kin = it.kin;
    double* gr = it.gram + (long long)b * kin * kin;
    double* h = it.H + (long long)b * (kin + 1) * kin;
    __shared__ double G[MK * MK], hc[MK];
    if (!ar_reduce<MV>(acc, mask, red, sum, [&] {
            for (int i = threadIdx.x; i < k * kin; i += kArThreads) G[i] = gr[i];
        }))
        return;
    if (threadIdx.x < k) gr[k * kin + threadIdx.x] = sum[MK + threadIdx.x];
    if (threadIdx.x == 0)
        for (int m = 0; m <= k; ++m) {
            double t = sum[m];
            for (int q = 0; q < m; ++q) t -= (m < k ? G[m * kin + q] : sum[MK + q]) * hc[q];
            hc[m] = t;
            h[m * kin + k] = t;
        }
}

// w -= sum_{m <= k} h_m v_m, ||w||, Givens.  Flat over the item's s*R rows.
template <class SV, class A, int N, int MK>
__global__ void __launch_bounds__(kArThreads) k_arnoldi_upd(int n0, unsigned rows, const int* active, A* wv, long long wbs,
                                                            Basis<SV> V, int k, ArRed red, ArItems it) {
    pdl_prologue();
    __shared__ double sum[1];
    __shared__ A hs[MK];
    const int b = blockIdx.y;
    if (!active[b]) return;
    if (threadIdx.x <= k) hs[threadIdx.x] = (A)it.H[(long long)b * (it.kin + 1) * it.kin + threadIdx.x * it.kin + k];
    __syncthreads();
    const unsigned nv = (unsigned)n0 / N, npos = nv * rows;
    A* w = wv + (long long)b * wbs;
    A acc[1] = {A(0)};
    for (unsigned q = blockIdx.x * kArThreads + threadIdx.x; q < npos; q += red.nchunk * kArThreads) {
        const unsigned row = q / nv;
        const long long p = (long long)q * N;       // rows are whole multiples of N
        A x[N];
        ld_n<N>(w + p, x);
#pragma unroll
        for (int m = 0; m < MK; ++m)
            if (m <= k) {
                A v[N];
                ld_n<N>(V.at(m, b) + p, v);
                if constexpr (PT<SV>::scaled) {
                    const float f = V.scale(m, b)[row];
#pragma unroll
                    for (int t = 0; t < N; ++t) v[t] *= f;
                }
#pragma unroll
                for (int t = 0; t < N; ++t) x[t] -= hs[m] * v[t];
            }
        st_n<N>(w + p, x);
#pragma unroll
        for (int t = 0; t < N; ++t) acc[0] += x[t] * x[t];
    }
    __shared__ ArState<MK> state;
    if (ar_reduce<1>(acc, 1u, red, sum, [&] { state.load(it, b, k); }) && threadIdx.x == 0)
        ar_givens(it, b, k, sqrt(sum[0]), state);
}

// out_b = src_b / denom[b * dstride] for unscaled storage, U vectors of N values per thread (all loads
// before the stores).  rep: the source is one stage of nx values that `rep` stages of out receive.
// sp: also advance the recurrence's step index (the launch that read it has finished).
template <class SO, class SR, int N, int U>
__global__ void __launch_bounds__(kArThreads) k_scale_vec(long long n, long long nx, int rep, const int* active,
                                                          const SR* src, long long sbs, const double* denom,
                                                          long long dstride, Vec<SO> out, StepPtrs* sp) {
    pdl_prologue();
    if (sp && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) sp->n += 1;
    static_assert(!PT<SO>::scaled, "unscaled storage only");
    using A = typename PT<SO>::A;
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    __shared__ A inv;
    if (threadIdx.x == 0) inv = denom ? A(1) / A(denom[(long long)b * dstride]) : A(1);
    __syncthreads();
    const SR* x = src + (long long)b * sbs;
    SO* o = out.d + (long long)b * out.bs;
    const long long i0 = ((long long)blockIdx.x * U * kArThreads + threadIdx.x) * N;
    A v[U][N];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const long long i = i0 + (long long)u * kArThreads * N;
        if (i < (rep ? nx : n)) {
            if constexpr (sizeof(SR) == sizeof(SO)) {
                SR t[N];
                ld_n<N>(x + i, t);
#pragma unroll
                for (int q = 0; q < N; ++q) v[u][q] = A(t[q]) * inv;
            } else {
#pragma unroll
                for (int q = 0; q < N; ++q) v[u][q] = A(x[i + q]) * inv;
            }
        }
    }
    for (int r = 0; r < (rep ? rep : 1); ++r)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long i = i0 + (long long)u * kArThreads * N;
            if (i < (rep ? nx : n)) st_n<N>(o + (long long)r * nx + i, v[u]);
        }
}

// ---------------------------------------------------------------------------
// Rana's stage sweep: out = V_stage - sum_j c_j K Z_j with c_j = tau (L D)_ij rounded on the host, j in
// [j0, j1).  Unscaled storage, N consecutive columns per thread.
// ---------------------------------------------------------------------------
template <class A> struct StageCoef {
    A c[kMaxS];
    int j0, j1;
};

template <class SV, class SZ, int N, int TS>
__global__ void __launch_bounds__(kArThreads) k_rana_vec(Geo g, InvH2<typename PT<SZ>::A> hh, const int* active,
                                                         Vec<SV> V, int stage, Vec<SZ> Z,
                                                         StageCoef<typename PT<SZ>::A> cf,
                                                         Faces<typename PT<SZ>::A> faces, Vec<SZ> out) {
    pdl_prologue();
    static_assert(!PT<SZ>::scaled && !PT<SV>::scaled, "unscaled storage only");
    using A = typename PT<SZ>::A;
    const int b = blockIdx.y;
    if (active && !active[b]) return;
    const unsigned nv = (unsigned)g.n0 / N;
    const unsigned q = blockIdx.x * kArThreads + threadIdx.x;
    if (q >= nv * (unsigned)g.R) return;
    const int row = (int)(q / nv), c = (int)(q - row * nv) * N;
    int j, kk;
    row_jk(g, row, j, kk);
    A acc[N];
    field_of(V, b, 0, stage, g).template row_n<N>(row, c, acc);
#pragma unroll
    for (int jj = 0; jj < TS; ++jj)
        if (jj >= cf.j0 && jj < cf.j1) {
            A P[N], K[N];
            fd_K_n<N>(field_of(Z, b, 0, jj, g), g, hh, faces, row, j, kk, c, P, K);
#pragma unroll
            for (int t = 0; t < N; ++t) acc[t] -= cf.c[jj] * K[t];
        }
    st_n<N>(out.d + (long long)b * out.bs + (long long)row * g.n0 + c, acc);
}

// The same in 16-bit storage: a thread per point of whole rows (the row's scale is a block reduction).
template <class SV, class SZ>
__global__ void __launch_bounds__(kPtMaxThreads) k_rana_pt(Geo g, InvH2<typename PT<SZ>::A> hh, PtMap pm, int B,
                                                           const int* active, Vec<SV> V, long long rows, int stage,
                                                           Vec<SZ> Z, StageCoef<typename PT<SZ>::A> cf,
                                                           Faces<typename PT<SZ>::A> faces, Vec<SZ> out) {
    pdl_prologue();
    using A = typename PT<SZ>::A;
    PtPos q = pt_pos(pm, B, g.R, active);
    const int row = (int)q.row;
    int j = 0, k = 0;
    if (q.valid) row_jk(g, row, j, k);
    SZ* o; float* osc;
    row_store_ptrs(out, q.b, 0, q.row, g.n0, o, osc);
    pt_store<SZ>(o, osc, pm, q.c0, q.valid, [&](int c) -> A {
        A acc;
        field_of(V, q.b, rows, stage, g).template row_n<1>(row, c, &acc);
#pragma unroll 2
        for (int jj = cf.j0; jj < cf.j1; ++jj) {
            A P, K;
            fd_K_n<1>(field_of(Z, q.b, rows, jj, g), g, hh, faces, row, j, k, c, &P, &K);
            acc -= cf.c[jj] * K;
        }
        return acc;
    });
}

// ---------------------------------------------------------------------------
// S_tilde's recurrence (one item, or B of MGRIT's intervals: item b at time index sp->n + b * stride).
// Its states are FP64 vectors that hold values of the arithmetic type A.
// ---------------------------------------------------------------------------

// double -> float for values a float holds exactly, by integer operations (an FP64 conversion costs as
// much as an FP64 operation); false where d is not a float of moderate size or zero.
__device__ __forceinline__ bool exact_float(double d, float& f) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d), mag = hi & 0x7fffffffu;
    // the exponent field minus 896 and the upper 23 bits of the fraction, then the sign
    const unsigned bits = (__funnelshift_l(lo, hi, 3) - (896u << 23)) | (hi & 0x80000000u);
    const bool zero = (mag | lo) == 0u;
    f = zero ? 0.f : __uint_as_float(bits);
    // 2^-83 <= |d| < 2^87, no fraction bits beyond a float's
    return zero || ((lo & 0x1fffffffu) == 0u && mag - (940u << 20) < (170u << 20));
}
__device__ __forceinline__ float to_arith(double d, float) {
    float f;
    return exact_float(d, f) ? f : (float)d;
}
__device__ __forceinline__ double to_arith(double d, double) { return d; }

// t = K z_{v,n} (every stage's right-hand side: one copy) and the start of the step's inner solves with
// ||r|| = sqrt(s) ||t||.  K z in FP64, rounded once to A: it cancels to 1e-4 of its terms on the finest grids.  (Q1 and FD
// apart: with both in one kernel 14 items of 256^2 took 48 us instead of 25; double-float sums took 18.)
template <class A, bool Q1M>
__global__ void __launch_bounds__(kArThreads) k_schur_start(Geo g, int s, const StepPtrs* sp, int stride, A* t,
                                                            SpaceOp<A> sop, ArRed red, ArItems it) {
    pdl_prologue();
    __shared__ double sum[1];
    const int b = blockIdx.y;
    const View<double> z{sp->z + (long long)(sp->n + b * stride) * g.nx, nullptr, g.n0};
    A* tb = t + (long long)b * g.nx;
    A acc = A(0);
#pragma unroll 1
    for (unsigned q = blockIdx.x * kArThreads + threadIdx.x; q < (unsigned)g.nx; q += red.nchunk * kArThreads) {
        const int row = (int)(q / (unsigned)g.n0), c = (int)(q - row * g.n0);
        int j, k;
        row_jk(g, row, j, k);
        A v;
        if constexpr (Q1M) v = (A)op_K(z, g, sop, row, j, k, c);
        else v = (A)fd_K(z, g, sop.faces, row, j, k, c);
        tb[q] = v;
        acc += v * v;
    }
    if (ar_reduce<1>(&acc, 1u, red, sum, [] {}) && threadIdx.x == 0) ar_init(it, b, sqrt((double)s * sum[0]));
}

// z_{v,n+1} = w_{n+1} + z_{v,n} - tau sum_i b_i q_i, q = sum_k y_k Z_k, n + 1 = sp->n + b * stride (the
// step index was advanced since the step's start).  res: the C-point residual w + Phi(z) - z_{n+1} into
// block b + 1 of res instead.  The its * s products tau b_i y_k are formed once per block.
template <class SZ, class A, int N>
__global__ void __launch_bounds__(kArThreads) k_schur_finish(Geo g, int s, const A* wbuf, const StepPtrs* sp, int stride,
                                                             Basis<SZ> Z, const double* y, int kin, const int* its,
                                                             const double* bw, double tau, A* res) {
    pdl_prologue();
    __shared__ A cf[kMaxInner * kMaxS];
    const int b = blockIdx.y;
    const int m = its[b], nc = m * s;
    for (int r = threadIdx.x; r < nc; r += kArThreads) {
        const int k = r / s;
        cf[r] = (A)(tau * bw[r - k * s] * y[(long long)b * kin + k]);
    }
    __syncthreads();
    const unsigned nv = (unsigned)g.n0 / N;
    const unsigned q = blockIdx.x * kArThreads + threadIdx.x;
    if (q >= nv * (unsigned)g.R) return;
    const int n1 = sp->n + b * stride;
    const unsigned row = q / nv;
    const long long p = (long long)q * N;
    const double* zn = sp->z + (long long)(n1 - 1) * g.nx + p;
    double* zn1 = sp->z + (long long)n1 * g.nx + p;
    A acc[N];
    ld_n<N>(wbuf + (long long)n1 * g.nx + p, acc);
#pragma unroll
    for (int t = 0; t < N; ++t) acc[t] += to_arith(zn[t], A(0));
    for (int k = 0; k < m; ++k) {
        const SZ* zk = Z.at(k, b) + p;
        const float* sc = PT<SZ>::scaled ? Z.scale(k, b) + row : nullptr;
#pragma unroll 3
        for (int i = 0; i < s; ++i) {
            A v[N];
            ld_n<N>(zk + (long long)i * g.nx, v);
            A a = cf[k * s + i];
            if constexpr (PT<SZ>::scaled) {
                const float f = sc[(long long)i * g.R];
#pragma unroll
                for (int t = 0; t < N; ++t) acc[t] -= a * (v[t] * f);
            } else {
#pragma unroll
                for (int t = 0; t < N; ++t) acc[t] -= a * v[t];
            }
        }
    }
    if (res) {
        A* r = res + (long long)(b + 1) * g.nx + p;
#pragma unroll
        for (int t = 0; t < N; ++t) r[t] = acc[t] - to_arith(zn1[t], A(0));
    } else {
#pragma unroll
        for (int t = 0; t < N; ++t) zn1[t] = to_fp64(acc[t]);
    }
}

// out_b = sum_{k < its[b]} y[b][k] Z_k, N consecutive columns per thread, over the item's s*R rows.
template <class SZ, class SO, int N>
__global__ void __launch_bounds__(kArThreads) k_combine_vec(int n0, unsigned rows, Basis<SZ> Z, const double* y, int kin,
                                                            const int* its, SO* out, long long obs) {
    pdl_prologue();
    using A = typename PT<SZ>::A;
    __shared__ A cf[kMaxInner];
    const int b = blockIdx.y;
    const int m = its[b];
    if (threadIdx.x < m) cf[threadIdx.x] = (A)y[(long long)b * kin + threadIdx.x];
    __syncthreads();
    const unsigned nv = (unsigned)n0 / N;
    const unsigned q = blockIdx.x * kArThreads + threadIdx.x;
    if (q >= nv * rows) return;
    const unsigned row = q / nv;
    const long long p = (long long)q * N;
    A acc[N];
#pragma unroll
    for (int t = 0; t < N; ++t) acc[t] = A(0);
#pragma unroll 3
    for (int k = 0; k < m; ++k) {
        A v[N];
        ld_n<N>(Z.at(k, b) + p, v);
        A a = cf[k];
        if constexpr (PT<SZ>::scaled) {
            const float f = Z.scale(k, b)[row];
#pragma unroll
            for (int t = 0; t < N; ++t) acc[t] += a * (v[t] * f);
        } else {
#pragma unroll
            for (int t = 0; t < N; ++t) acc[t] += a * v[t];
        }
    }
    SO* o = out + (long long)b * obs + p;
#pragma unroll
    for (int t = 0; t < N; ++t) {
        if constexpr (std::is_same<SO, A>::value) o[t] = acc[t];
        else o[t] = to_fp64(acc[t]);
    }
}

}  // namespace aao
