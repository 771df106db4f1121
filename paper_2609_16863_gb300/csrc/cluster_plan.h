// Plan of the cluster-resident V-cycles (cluster_mg.cuh) on the host: the shared-memory layout and the program of
// steps that every CTA of a cluster runs.  Plain C++, so that a test can compile it and check the
// exchanges of ghost rows against the barriers between them.
#pragma once

#include <algorithm>
#include <vector>

namespace aao {

constexpr int kClMax = 16;            // CTAs per cluster (16 needs the non-portable size)
constexpr int kClThreads = 512;
constexpr int kClMaxBatch = 32;       // 16-bit storage: batches of at most this many items run one cluster per item
constexpr int kClBatch8 = 8;          // 16-bit storage: batches of at least this many items take the 8-CTA plan
constexpr int kClPad = 4;             // columns before a row's first point and after its last vector: rows
                                      // start 16-byte aligned, the columns beside the grid are zero
constexpr int kClReach = 3;           // CTAs on either side whose ghost rows may hold a CTA's rows
constexpr int kClMaxLevels = 10;      // 2D levels of grids that fit a cluster

// Shape of a plan: what does not depend on the storage type.  Offsets and sizes count values of the arithmetic type.
struct ClShape {
    int C, L, T;                          // cluster size, levels, T = L-1 (the replicated coarsest level)
    int cycles, nu1, nu2;
    int fine0, has_faces;                 // level 0 is the FD operator; with faces of a kappa field
    int fuse0;                            // 1: level 0 takes two zero-guess sweeps at once (mode 3)
    int n0[kClMaxLevels], n1[kClMaxLevels];
    int nvp[kClMaxLevels];                // vectors per padded row
    unsigned magicv[kClMaxLevels];        // ceil(2^32 / nvp): tid / nvp = umulhi(tid, magicv)
    unsigned magic[kClMaxLevels];         // ceil(2^32 / n0)
    int per[kClMaxLevels];                // rows per thread
    int H[kClMaxLevels];                  // ghost rows
    int ix[kClMaxLevels];                 // rows of the x inbox per side
    int maxr[kClMaxLevels];               // own rows in the shared-memory layout
    int rlo[kClMaxLevels][kClMax + 1];    // CTA r owns rows [rlo[l][r], rlo[l][r+1]) (the coarsest: computes them)
    int off[kClMaxLevels];                // A-element offset of level l's X0 | X1 | B, each (maxr + 2H) x ld
    int ioff[kClMaxLevels];               // x inbox: 2 ix rows of ld
    int soff[kClMaxLevels];               // staged stencil, 9 x (maxr + 2(H-1)) x padded row (-1: none)
    int woff[kClMaxLevels];               // omega / a_PP, (maxr + 2H) x padded row (-1: the scalar w0)
    int sten_global[kClMaxLevels];        // 1: level l's stencil is read from global memory (L2), not staged
    int fxoff, fyoff;                     // level 0 faces: rows of ld | rows of the padded width
    int dinv_global;                      // 1: the rows of A_c^{-1} are read from global memory
    int dinv_off, boff;                   // this CTA's rows of A_c^{-1}, each padded to ncp; the coarsest b (ncp)
    int ncp;                              // unknowns of the coarsest level, rounded up to vectors
    int cs[kClMax + 1];                   // coarsest rows [cs[r], cs[r+1]) of A_c^{-1} b are computed by CTA r
    int img_off, img_len;                 // the staged constants: elements [img_off, img_off + img_len)
    int prog_off;                         // byte offset of the program in shared memory (part of the image)
    int pc[4];                            // operations of the first cycle, of odd and of even later cycles
    int kfin;                             // buffer of x_0 after the last cycle
};

// One operation of the cycle's program.
enum ClKind { kClStep, kClRestrict, kClRestrictLast, kClSolve, kClProlong, kClInbox, kClClear };
struct ClOp {
    unsigned char kind, lev;
    unsigned char mode;                   // step: 0 sweep, 1 sweep of a zero guess, 2 residual, 3 two sweeps of a
                                          // zero guess at once; restriction: also the first sweep (1)
    unsigned char kin;                    // buffer read (prolong: x_f's)
    unsigned char kc;                     // prolong: buffer of x_c; step: buffer written; restriction: of the sweep
    unsigned char ext;                    // ghost rows computed
    unsigned char depth;                  // ghost rows stored into the other CTAs (0: none)
    unsigned char flags;                  // 1: into the x inboxes; 2: cluster barrier
};
static_assert(sizeof(ClOp) == 8, "one 8-byte load");

// Ghost rows of the pre-smoothed x that are read: two by the residual of a ghost row, nu2 by the post-sweeps.
inline int cl_reach_after(int nu2) { return nu2 > 2 ? nu2 : 2; }

// The program of a plan: the operations of the first cycle, of an odd and of an even later one (the
// buffers alternate with the number of sweeps), and the buffer x_0 ends in.  Every CTA runs the same
// program, so its barriers match.  A step writes ghost rows of other CTAs' buffers (depth > 0 without
// the inbox flag) only where a cluster barrier separates it from the last read of those rows: with H = 1 an
// exchange follows every sweep; on levels with deeper ghost regions no sweep but the first post-sweep can be such a
// step (the interpolation covers all the post-sweeps' ghost rows, or one), and the buffer it writes was last read
// by the restriction.  b and the inboxes are read before the barriers of the steps in between.
inline std::vector<ClOp> cl_program(ClShape& t) {
    std::vector<ClOp> prog;
    const int T = t.T, nu1 = t.nu1, nu2 = t.nu2, left = cl_reach_after(nu2);
    auto emit = [&](int kind, int l, int mode, int kin, int kc, int ext, int depth, int flags) {
        prog.push_back(ClOp{(unsigned char)kind, (unsigned char)l, (unsigned char)mode, (unsigned char)kin,
                            (unsigned char)kc, (unsigned char)ext, (unsigned char)depth,
                            (unsigned char)(flags | (depth > 0 ? 2 : 0))});
    };
    int cur[kClMaxLevels] = {}, reach[kClMaxLevels] = {};     // buffer of x; valid ghost rows of the pre-smoothed x
    int after[3] = {};
    for (int part = 0; part < 3; ++part) {
        t.pc[part] = (int)prog.size();
        for (int l = 0; l < T; ++l) {
            const int H = t.H[l];
            int k = cur[l], v = H;
            bool zero = part == 0 || l > 0;
            int sw = 0;
            if (!zero) {
                emit(kClInbox, l, 0, k, 0, 0, 0, 0);
            } else if (l > 0 && nu1 > 0) {
                sw = 1;                        // the restriction has done the first sweep, into buffer k ^ 1
                zero = false;
                k ^= 1;
            } else if (l == 0 && nu1 > 1 && t.fuse0) {
                // two sweeps from b at once
                const int ext = std::min(v - 1, nu1 - 2 + left), depth = ext == 0 ? H : 0;
                emit(kClStep, l, 3, 2, k, ext, depth, 0);
                v = depth > 0 ? H : ext;
                sw = 2;
                zero = false;
            }
            for (; sw < nu1; ++sw) {
                // the result is read up to (sweeps left) + left rows beyond the own ones
                const int ext = std::min(zero ? v : v - 1, nu1 - 1 - sw + left);
                const int depth = ext == 0 ? H : 0;
                emit(kClStep, l, zero ? 1 : 0, k, k ^ 1, ext, depth, 0);
                v = depth > 0 ? H : ext;
                zero = false;
                k ^= 1;
            }
            int kr = 2;                        // no sweep on a zero guess: the residual is b
            if (zero) {
                emit(kClClear, l, 0, k, 0, 0, 0, 0);
            } else {
                emit(kClStep, l, 2, k, k ^ 1, v >= 2 ? 1 : 0, v >= 2 ? 0 : 1, 0);
                kr = k ^ 1;
            }
            cur[l] = k;
            reach[l] = v;
            emit(l + 1 < T ? kClRestrict : kClRestrictLast, l, nu1 > 0 ? 1 : 0, kr, cur[l + 1] ^ 1, 0, 0, 2);
        }
        emit(kClSolve, T, 0, 0, 0, 0, 0, 2);
        for (int l = T - 1; l >= 0; --l) {
            int k = cur[l];
            // interpolate on up to nu2 ghost rows: e of them need (e + 2) / 2 rows of x_c beyond the own ones
            int v = std::min(reach[l], nu2);
            if (l + 1 < T) v = std::min(v, 2 * t.ix[l + 1] - 1);
            if (v < nu2) v = std::min(v, 1);       // an exchange among the sweeps: after the first one
            emit(kClProlong, l, 0, k, l + 1 < T ? cur[l + 1] : 0, v, nu2 == 0 ? t.ix[l] : 0, 0);
            for (int sw = 0; sw < nu2; ++sw) {
                const bool fin = sw == nu2 - 1;
                const int e = std::min(v - 1, nu2 - 1 - sw);
                const int depth = fin ? t.ix[l] : (e == 0 ? t.H[l] : 0);
                emit(kClStep, l, 0, k, k ^ 1, e, depth, fin ? 1 : 0);
                v = depth > 0 ? t.H[l] : e;
                k ^= 1;
            }
            cur[l] = k;
        }
        after[part] = cur[0];
    }
    t.pc[3] = (int)prog.size();
    prog.push_back(ClOp{});
    const int last = t.cycles - 1;
    t.kfin = after[last == 0 ? 0 : 2 - (last & 1)];
    return prog;
}

// What a plan is made for and with.
struct ClSpec {
    int C;                                // CTAs per cluster
    int deep;                             // ghost rows for whole smoothing phases: 1: on the coarse levels, 2: on the finest
                                          // too; 0: one ghost row
    int lean;                             // read from global memory instead of being staged: 1: the rows of A_c^{-1},
                                          // 2: the first coarse stencil too, 3: every coarse stencil
    int L;                                // levels, n0 x n1 points each
    int n0[kClMaxLevels], n1[kClMaxLevels];
    int fine0, faces, fuse0;              // as in ClShape
    int cycles, nu1, nu2;
    int vn, size;                         // columns per thread; bytes of a value
};

// Lay out a plan; its bytes of shared memory, or -1 where the grid does not take it.
inline long long cl_layout(ClShape& t, const ClSpec& s) {
    if (s.n1[0] < s.C || s.L > kClMaxLevels) return -1;
    // ghost rows for up to three sweeps (an inbox of two rows of x_c serves three of the interpolation's ghost rows)
    if (s.deep > 0 && (s.nu2 > 3 || s.nu1 > 3)) return -1;
    const int C = s.C, L = s.L, T = L - 1, VN = s.vn, nu1 = s.nu1, nu2 = s.nu2, deep = s.deep, lean = s.lean;
    t = ClShape{};
    t.C = C;
    t.L = L;
    t.T = T;
    t.cycles = s.cycles;
    t.nu1 = nu1;
    t.nu2 = nu2;
    t.fine0 = s.fine0;
    t.has_faces = s.faces;
    t.fuse0 = s.fuse0;
    t.dinv_global = lean >= 1 ? 1 : 0;
    auto magic = [](long long d) { return (unsigned)((4294967296ULL + (unsigned long long)d - 1) / (unsigned long long)d); };

    long long o = 0;
    auto take = [&](long long n) {
        long long at = o;
        o += (n + 3) / 4 * 4;
        return (int)at;
    };
    for (int l = 0; l < L; ++l) {
        const int n0 = s.n0[l], n1 = s.n1[l], nvp = std::max((n0 + VN - 1) / VN, 2);
        if (nvp > kClThreads) return -1;
        t.n0[l] = n0;
        t.n1[l] = n1;
        t.nvp[l] = nvp;
        t.magicv[l] = magic(nvp);
        t.magic[l] = magic(std::max(n0, 2));
        for (int r = 0; r <= C; ++r)
            t.rlo[l][r] = l == 0 ? (int)((long long)r * n1 / C) : t.rlo[l - 1][r] / 2;
        // Every CTA must own at least one row of every distributed level (neighbours store edge rows
        // into the CTAs that own the rows beside theirs; grids with few rows for their width fail
        // this), and its ghost rows must belong to the kClReach CTAs on either side.
        int mr = 1;
        auto covered = [&](int need) {
            for (int r = 0; r < C; ++r) {
                if (std::max(t.rlo[l][r] - need, 0) < t.rlo[l][std::max(r - kClReach, 0)]) return false;
                const int top = r + 1 + kClReach >= C ? n1 : t.rlo[l][r + 1 + kClReach];
                if (std::min(t.rlo[l][r + 1] + need, n1) > top) return false;
            }
            return true;
        };
        for (int r = 0; r < C; ++r) {
            const int own = t.rlo[l][r + 1] - t.rlo[l][r];
            mr = std::max(mr, own);
            if (l < T && own < 1) return -1;
        }
        const int deepH = std::max((l == 0 ? nu1 : nu1 - 1) + cl_reach_after(nu2), 2);
        const bool dl = deep >= (l == 0 ? 2 : 1) && l < T && covered(deepH);
        if (deep == 2 && l == 0 && !dl) return -1;
        t.H[l] = dl ? deepH : 1;
        t.ix[l] = l >= T ? 0 : (l == 0 ? t.H[0] : (deep > 0 && covered(2) ? 2 : 1));
        t.maxr[l] = l < T ? mr : n1;
        const int groups = kClThreads / nvp;
        t.per[l] = (t.maxr[l] + 2 * t.H[l] + groups - 1) / groups;
        const long long ld = (long long)nvp * VN + 2 * kClPad;
        t.off[l] = take(3LL * (t.maxr[l] + 2 * t.H[l]) * ld);
        t.ioff[l] = take(2LL * t.ix[l] * ld);
    }
    const long long ncst = (long long)s.n0[T] * s.n1[T];
    t.ncp = (int)((ncst + VN - 1) / VN * VN);
    t.boff = take(t.ncp);
    // the image of constants, the program at its end
    t.img_off = (int)o;
    for (int l = 0; l < L; ++l) {
        t.soff[l] = t.woff[l] = -1;
        if (l >= T) continue;
        const long long np = (long long)t.nvp[l] * VN;
        const bool fd = l == 0 && s.fine0;
        if (!fd) {
            t.sten_global[l] = l >= 1 && (lean >= 3 || (lean == 2 && l == 1)) ? 1 : 0;
            if (t.sten_global[l] && s.n0[l] != np) return -1;     // read as whole vectors of the padded row
            if (!t.sten_global[l]) t.soff[l] = take(9LL * (t.maxr[l] + 2 * (t.H[l] - 1)) * np);
        }
        if (!fd || s.faces) t.woff[l] = take((long long)(t.maxr[l] + 2 * t.H[l]) * np);
    }
    if (s.faces) {
        const long long np = (long long)t.nvp[0] * VN, rows = t.maxr[0] + 2 * (t.H[0] - 1);
        t.fxoff = take(rows * (np + 2 * kClPad));
        t.fyoff = take((rows + 1) * np);
    }
    int msl = 0;
    for (int r = 0; r <= C; ++r) t.cs[r] = (int)((long long)r * ncst / C);
    for (int r = 0; r < C; ++r) msl = std::max(msl, t.cs[r + 1] - t.cs[r]);
    t.dinv_off = t.dinv_global ? -1 : take((long long)msl * t.ncp);
    const long long nprog = (long long)cl_program(t).size();
    t.prog_off = (int)(o * s.size);
    take((nprog * (long long)sizeof(ClOp) + s.size - 1) / s.size);
    t.img_len = (int)(o - t.img_off);
    return o * s.size;
}

}  // namespace aao
