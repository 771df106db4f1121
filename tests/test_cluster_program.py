"""The cluster V-cycle's plans (csrc/cluster_plan.h, compiled here with the host's C++ compiler): the program of steps, its
exchanges of ghost rows and its barriers, run on a model of a cluster's shared memories.

The model holds, per CTA, what csrc/cluster_mg.cuh holds: per distributed level three row blocks (two of x, one of
b) with H ghost rows, an inbox of x rows per side, the replicated coarsest level.  It restates the kernel's steps row
by row (cl_step, cl_restrict, cl_prolong, cl_push and the coarsest solve) and takes layout and program from the
header.  Checked for clusters of 2, 4, 8 and 16 CTAs, every depth of ghost regions, 0 to 4 sweeps before and after,
one to four cycles:
  * the result equals the oracle's V-cycles to 1e-11 (sums in another order, FP64), and every plan of a grid gives
    the same values bit for bit: a ghost row that is a sweep stale, or a row exchanged too late, would not;
  * between two cluster barriers no CTA stores into a row that its owner reads or writes or a third CTA stores into, and no
    store to another CTA follows the last cluster barrier (the CTA may have ended);
  * every access stays within the rows that the layout holds.
A program with one of its cluster barriers turned into a block's is reported as a race."""
import os
import random
import subprocess

import numpy as np
import pytest

import synth
from oracle.multigrid import Hierarchy, level_sizes
from oracle.operators import mass_fd, q1_matrices, stiffness_fd

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_16863_gb300", "csrc")
STEP, RESTRICT, RESTRICT_LAST, SOLVE, PROLONG, INBOX, CLEAR = range(7)
REACH = 3

MAIN = r"""
#include <cstdio>
#include "cluster_plan.h"
using namespace aao;
static void put(const char* k, const int* v, int n) {
    std::printf("%s", k);
    for (int i = 0; i < n; ++i) std::printf(" %d", v[i]);
    std::printf("\n");
}
int main() {
    ClSpec s{};
    while (std::scanf("%d %d %d %d %d %d %d %d %d %d %d", &s.C, &s.deep, &s.lean, &s.fine0, &s.faces, &s.fuse0, &s.cycles,
                      &s.nu1, &s.nu2, &s.vn, &s.L) == 11) {
        s.size = s.vn == 4 ? 4 : 8;
        for (int l = 0; l < s.L; ++l)
            if (std::scanf("%d %d", &s.n0[l], &s.n1[l]) != 2) return 1;
        ClShape t{};
        const long long bytes = cl_layout(t, s);
        std::printf("bytes %lld\n", bytes);
        if (bytes >= 0) {
            put("H", t.H, s.L); put("ix", t.ix, s.L); put("maxr", t.maxr, s.L); put("nvp", t.nvp, s.L);
            put("per", t.per, s.L); put("off", t.off, s.L); put("ioff", t.ioff, s.L); put("soff", t.soff, s.L);
            put("woff", t.woff, s.L); put("glob", t.sten_global, s.L);
            for (int l = 0; l < s.L; ++l) put("rlo", t.rlo[l], s.C + 1);
            put("cs", t.cs, s.C + 1); put("pc", t.pc, 4);
            const int misc[] = {t.kfin, t.boff, t.ncp, t.img_off, t.img_len, t.prog_off};
            put("misc", misc, 6);
            for (const ClOp& o : cl_program(t)) {
                const int v[] = {o.kind, o.lev, o.mode, o.kin, o.kc, o.ext, o.depth, o.flags};
                put("op", v, 8);
            }
        }
        std::printf("end\n");
    }
}
"""


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "t.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)

    def plan(ns, C, deep, nu1, nu2, cycles, fine0=1, faces=0, fuse0=1, lean=0, vn=4):
        """The plan as a dict, None where the grid does not take it."""
        sizes = level_sizes(ns)
        text = " ".join(str(v) for v in [C, deep, lean, fine0, faces, fuse0, cycles, nu1, nu2, vn, len(sizes)] +
                        [v for s in sizes for v in s])
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True, check=True).stdout
        p = dict(op=[], rlo=[], sizes=sizes, C=C, cycles=cycles, fine0=fine0, vn=vn)
        for line in out.splitlines():
            key, *v = line.split()
            v = [int(x) for x in v]
            if key in ("op", "rlo"):
                p[key].append(v)
            else:
                p[key] = v
        return p if p["bytes"][0] >= 0 else None
    return plan


class Cluster:
    """The shared memories of a cluster and the steps on them; `race` lists conflicting accesses."""

    def __init__(self, p, mg):
        self.p, self.mg, self.C, self.T = p, mg, p["C"], len(p["sizes"]) - 1
        self.rlo, self.H, self.ix = p["rlo"], p["H"], p["ix"]
        self.race, self.local, self.remote = [], set(), set()
        self.sten, self.w = [], []
        for l in range(self.T):
            n0, n1 = p["sizes"][l]
            A = mg.A[l].tocoo()
            S = np.zeros((9, n1, n0))
            r, c = A.row // n0, A.row % n0
            S[3 * (A.col // n0 - r + 1) + A.col % n0 - c + 1, r, c] = A.data
            self.sten.append(S)
            self.w.append(mg.omega / S[4])
        self.inv = np.linalg.inv(mg.A[-1].toarray())
        self.x, self.inb, self.xT, self.bT = [], [], [], []
        n0T, n1T = p["sizes"][-1]
        for r in range(self.C):
            self.x.append([np.zeros((3, self.nr(l, r) + 2 * self.H[l], p["sizes"][l][0] + 2)) for l in range(self.T)])
            self.inb.append([np.zeros((2 * self.ix[l], p["sizes"][l][0] + 2)) for l in range(self.T)])
            self.xT.append(np.zeros((n1T + 2, n0T + 2)))
            self.bT.append(np.zeros(n0T * n1T))

    def nr(self, l, r):
        return self.rlo[l][r + 1] - self.rlo[l][r] if 0 <= r < self.C else 0

    # -- accesses: objects are ("x", l, k, row), ("in", l, row), ("xT", row), ("bT", row) of a CTA
    def touch(self, r, *obj):
        self.local.add((r, obj))

    def store(self, src, dst, *obj):
        """A store by CTA src into CTA dst (which may be src itself: then a plain one)."""
        if src == dst:
            self.touch(dst, *obj)
            return
        self.remote.add((src, dst, obj))

    def barrier(self, cluster):
        if not cluster:
            return
        by = {}
        for src, dst, obj in self.remote:
            if (dst, obj) in self.local or by.setdefault((dst, obj), src) != src:
                self.race.append((src, dst, obj))
        self.local, self.remote = set(), set()

    def rows(self, r, l, k, lo, n):
        """Rows [lo, lo + n) of a block, relative to the CTA's first one."""
        assert lo >= -self.H[l] and lo + n <= self.nr(l, r) + self.H[l], (r, l, k, lo, n)
        for q in range(lo, lo + n):
            self.touch(r, "x", l, k, q)
        return self.x[r][l][k][lo + self.H[l]: lo + n + self.H[l]]

    def put(self, src, dst, l, k, row, value, inbox):
        if inbox:
            assert 0 <= row < 2 * self.ix[l]
            self.store(src, dst, "in", l, row)
            self.inb[dst][l][row] = value
        else:
            assert -self.H[l] <= row < self.nr(l, dst) + self.H[l]
            self.store(src, dst, "x", l, k, row)
            self.x[dst][l][k][row + self.H[l]] = value

    def push(self, r, l, k, lr, value, depth, inbox):
        """cl_push: own row lr into the ghost rows (or the inboxes) of the CTAs before and after."""
        prev = [self.nr(l, r - 1 - q) for q in range(REACH)]
        nxt = [self.nr(l, r + 1 + q) for q in range(REACH)]
        nr, ix, reach = self.nr(l, r), self.ix[l], max(self.H[l], self.ix[l])
        far = 0 < prev[0] < reach or 0 < nxt[0] < reach
        if lr < depth and prev[0] > 0:
            self.put(r, r - 1, l, k, ix + lr if inbox else lr + prev[0], value, inbox)
            between = prev[0]
            for q in range(1, REACH if far else 0):
                if lr >= depth - between or prev[q] == 0:
                    break
                self.put(r, r - 1 - q, l, k, ix + lr + between if inbox else lr + between + prev[q], value, inbox)
                between += prev[q]
        if lr >= nr - depth and nxt[0] > 0:
            self.put(r, r + 1, l, k, ix + lr - nr if inbox else lr - nr, value, inbox)
            between = nxt[0]
            for q in range(1, REACH if far else 0):
                if lr < nr - depth + between or nxt[q] == 0:
                    break
                self.put(r, r + 1 + q, l, k, ix + lr - nr - between if inbox else lr - nr - between, value, inbox)
                between += nxt[q]

    # -- steps
    def apply(self, l, x, j0, n):
        """A x on n grid rows from j0 on, x their rows and one more on each side."""
        n0 = self.p["sizes"][l][0]
        s = [sum(self.sten[l][3 * dy + dx, j0:j0 + n] * x[dy:dy + n, dx:dx + n0] for dx in range(3)) for dy in range(3)]
        return s[0] + s[1] + s[2]

    def step(self, r, l, mode, kin, kout, ext, depth, inbox):
        a, nr, n1 = self.rlo[l][r], self.nr(l, r), self.p["sizes"][l][1]
        lo, hi = max(-ext, -a), min(nr + ext, n1 - a)
        n, j0 = hi - lo, a + lo
        assert ext <= self.H[l] - (0 if mode == 1 else 1)           # rows of weights, of stencils
        b, w = self.rows(r, l, 2, lo, n)[:, 1:-1], self.w[l][j0:j0 + n]
        if mode == 1:
            out = w * b
        else:
            x = self.rows(r, l, kin, lo - 1, n + 2)
            if mode == 3:                                           # two sweeps of a zero guess, x = w b
                wide = np.zeros((n + 2, x.shape[1]))
                j = np.clip(np.arange(j0 - 1, j0 + n + 1), 0, n1 - 1)
                wide[:, 1:-1] = self.w[l][j] * x[:, 1:-1]
                x = wide
            d = b - self.apply(l, x, j0, n)
            out = d if mode == 2 else x[1:-1, 1:-1] + w * d
        self.rows(r, l, kout, lo, n)[:, 1:-1] = out
        if depth:
            for lr in range(nr):
                self.push(r, l, kout, lr, self.rows(r, l, kout, lr, 1)[0].copy(), depth, inbox)

    def restricted(self, r, l, kr, J):
        f = self.rows(r, l, kr, 2 * J - self.rlo[l][r], 3)
        nc = self.p["sizes"][l + 1][0]
        s = f[1] + 0.5 * (f[0] + f[2])
        return s[2:2 * nc + 1:2] + 0.5 * (s[1:2 * nc:2] + s[3:2 * nc + 2:2])

    def restrict(self, r, l, kr, kx):
        c = l + 1
        for q in range(self.nr(c, r)):
            J = self.rlo[c][r] + q
            for k, f in ((2, 1.0), (kx, self.w[c][J])):
                if k < 0:
                    continue
                row = self.rows(r, c, k, q, 1)[0]
                row[1:-1] = f * self.restricted(r, l, kr, J)
                self.push(r, c, k, q, row.copy(), self.H[c], False)

    def restrict_last(self, r, l, kr):
        n0 = self.p["sizes"][-1][0]
        for J in range(self.rlo[self.T][r], self.rlo[self.T][r + 1]):
            v = self.restricted(r, l, kr, J)
            for d in range(self.C):
                self.store(r, d, "bT", J)
                self.bT[d][J * n0:(J + 1) * n0] = v

    def solve(self, r):
        n0, n1 = self.p["sizes"][-1]
        for J in range(n1):
            self.touch(r, "bT", J)
        v = [float(self.inv[q] @ self.bT[r]) for q in range(self.p["cs"][r], self.p["cs"][r + 1])]
        for q, t in zip(range(self.p["cs"][r], self.p["cs"][r + 1]), v):
            for d in range(self.C):
                self.store(r, d, "xT", q)
                self.xT[d][q // n0 + 1, q % n0 + 1] = t

    def coarse_row(self, r, l, kc, y):
        if l == self.T:
            n0, n1 = self.p["sizes"][l]
            for q in range(max(y, 0) * n0, min(y + 1, n1) * n0):
                self.touch(r, "xT", q)
            return self.xT[r][y + 1]
        lr, nr = y - self.rlo[l][r], self.nr(l, r)
        if 0 <= lr < nr:
            return self.rows(r, l, kc, lr, 1)[0]
        row = self.ix[l] + (lr if lr < 0 else lr - nr)
        assert 0 <= row < 2 * self.ix[l]
        self.touch(r, "in", l, row)
        return self.inb[r][l][row]

    def prolong(self, r, l, kx, kc, ext, depth):
        a, nr, (n0, n1) = self.rlo[l][r], self.nr(l, r), self.p["sizes"][l]
        for q in range(max(-ext, -a), min(nr + ext, n1 - a)):
            g = a + q + 1
            y = (g // 2 - 1, g // 2 - 1) if g % 2 == 0 else ((g - 1) // 2 - 1, (g + 1) // 2 - 1)
            m = 0.5 * (self.coarse_row(r, l + 1, kc, y[0]) + self.coarse_row(r, l + 1, kc, y[1]))
            e = np.zeros(n0 + 2)
            e[2:-1:2] = m[1:1 + n0 // 2]
            e[1:-1:2] = (0.5 * (m[:-1] + m[1:]))[:(n0 + 1) // 2]
            row = self.rows(r, l, kx, q, 1)[0]
            row[1:-1] += e[1:-1]
            if depth and 0 <= q < nr:
                self.push(r, l, kx, q, row.copy(), depth, True)

    def inbox(self, r, k):
        H, nr = self.H[0], self.nr(0, r)
        for i in range(2 * H):
            self.touch(r, "in", 0, i)
            self.rows(r, 0, k, i - H if i < H else nr + i - H, 1)[0][:] = self.inb[r][0][i]

    def run(self, b):
        n0, n1 = self.p["sizes"][0]
        B = b.reshape(n1, n0)
        for r in range(self.C):
            a, nr, H = self.rlo[0][r], self.nr(0, r), self.H[0]
            for q in range(max(-H, -a), min(nr + H, n1 - a)):
                self.x[r][0][2][q + H, 1:-1] = B[a + q]
        for cyc in range(self.p["cycles"]):
            part = 0 if cyc == 0 else 2 - (cyc & 1)
            ops = self.p["op"][self.p["pc"][part]:self.p["pc"][part + 1]]
            for i, (kind, l, mode, kin, kc, ext, depth, flags) in enumerate(ops):
                if i == len(ops) - 1 and cyc == self.p["cycles"] - 1:
                    depth = flags = 0
                for r in range(self.C):
                    if kind == STEP:
                        self.step(r, l, mode, kin, kc, ext, depth, bool(flags & 1))
                    elif kind == RESTRICT:
                        self.restrict(r, l, kin, kc if mode else -1)
                    elif kind == RESTRICT_LAST:
                        self.restrict_last(r, l, kin)
                    elif kind == SOLVE:
                        self.solve(r)
                    elif kind == PROLONG:
                        self.prolong(r, l, kin, kc, ext, depth)
                    elif kind == INBOX:
                        self.inbox(r, kin)
                    else:
                        self.rows(r, l, kin, -self.H[l], self.nr(l, r) + 2 * self.H[l])[:] = 0.0
                self.barrier(bool(flags & 2))
        assert not self.remote, "a store into a CTA that may have ended"
        k = self.p["misc"][0]
        return np.concatenate([self.rows(r, 0, k, 0, self.nr(0, r))[:, 1:-1].ravel() for r in range(self.C)])


def hierarchy(ns, disc, nu1, nu2):
    if disc == "q1":
        M, K = q1_matrices(ns, (1.0, 1.0))
    else:
        M, K = mass_fd(ns), stiffness_fd(ns, (1.0, 1.0))
    return Hierarchy(M + 0.02 * K, ns, 0.8, nu1, nu2)


def plans(planner, ns, nu1, nu2, cycles, disc, fuse0):
    for C in (2, 4, 8, 16):
        for deep in (2, 1, 0):
            p = planner(ns, C, deep, nu1, nu2, cycles, fine0=int(disc == "fd"), fuse0=fuse0)
            if p:
                yield p


GRIDS = [(17, 17), (9, 100), (4, 70), (20, 33), (33, 64), (40, 129), (70, 66)]
RANDOM = random.Random(7)
CASES = [(ns, 2, 2, 3, "fd", 1) for ns in GRIDS] + [(ns, 2, 2, 2, "q1", 0) for ns in GRIDS[3:]] + [
    (RANDOM.choice(GRIDS), nu1, nu2, RANDOM.randint(1, 4), RANDOM.choice(["fd", "q1"]), 0)
    for nu1 in range(5) for nu2 in range(5)]


@pytest.mark.parametrize("ns,nu1,nu2,cycles,disc,fuse0", CASES)
def test_program_matches_the_v_cycles_without_races(planner, ns, nu1, nu2, cycles, disc, fuse0):
    mg = hierarchy(ns, disc, nu1, nu2)
    b = synth.random_vector(int(np.prod(ns)), 11)
    ref = mg.solve(b, cycles)
    first, count = None, 0
    for p in plans(planner, ns, nu1, nu2, cycles, disc, fuse0):
        c = Cluster(p, mg)
        x = c.run(b)
        assert not c.race, (p["C"], p["H"], c.race[:4])
        assert np.linalg.norm(x - ref) <= 1e-11 * np.linalg.norm(ref)
        first = x if first is None else first
        assert np.array_equal(x, first), (p["C"], p["H"])
        count += 1
    assert count >= 2


def test_missing_barriers_are_reported(planner):
    """Each exchange's cluster barrier in turn becomes a block's: the model finds a race."""
    ns = (40, 66)
    mg = hierarchy(ns, "fd", 2, 2)
    b = synth.random_vector(int(np.prod(ns)), 11)
    p = planner(ns, 8, 0, 2, 2, 2)
    found = []
    for i, o in enumerate(p["op"]):
        if not o[7] & 2 or i >= p["pc"][2] - 1:          # (the very last operation exchanges nothing)
            continue
        q = dict(p, op=[list(v) for v in p["op"]])
        q["op"][i][7] &= ~2
        c = Cluster(q, mg)
        try:
            c.run(b)
        except AssertionError:
            c.race.append("left over")
        found.append(bool(c.race))
    assert len(found) >= 10 and all(found)


@pytest.mark.parametrize("vn", [4, 1])
@pytest.mark.parametrize("lean", [0, 1, 2, 3])
def test_layout_regions_do_not_overlap(planner, vn, lean):
    """Blocks, inboxes and the image of constants are disjoint, aligned to four values, and rows hold whole vectors
    (two at least); a stencil read from global memory has rows of whole vectors."""
    taken = 0
    for ns in [(256, 256), (255, 257), (127, 95), (8, 200), (4, 100), (80, 72), (64, 64), (500, 40)]:
        for C in (2, 4, 8, 16):
            for deep in (0, 1, 2):
                for fine0, faces in ((1, 0), (1, 1), (0, 0)):
                    p = planner(ns, C, deep, 2, 2, 3, fine0=fine0, faces=faces, lean=lean, vn=vn)
                    if not p:
                        continue
                    taken += 1
                    spans = []
                    for l, (n0, _) in enumerate(p["sizes"]):
                        assert p["nvp"][l] == max(-(-n0 // vn), 2)
                        ld, rows = p["nvp"][l] * vn + 8, p["maxr"][l] + 2 * p["H"][l]
                        spans += [(p["off"][l], 3 * rows * ld), (p["ioff"][l], 2 * p["ix"][l] * ld)]
                        assert p["per"][l] * (512 // p["nvp"][l]) >= rows
                        if p["glob"][l]:
                            assert n0 == p["nvp"][l] * vn
                    _, boff, ncp, img, length, prog = p["misc"]
                    spans += [(boff, ncp), (img, length)]
                    spans.sort()
                    assert all(s % 4 == 0 for s, _ in spans)
                    assert all(s + n <= t for (s, n), (t, _) in zip(spans, spans[1:]))
                    size = 4 if vn == 4 else 8
                    assert (img + length) * size == p["bytes"][0] and img * size <= prog
                    assert prog + 8 * len(p["op"]) <= p["bytes"][0]
    assert taken > 20
