"""Grids whose rows are one 16-byte vector (n0 = 4) on thread-block clusters: the plan pads such rows to two
vectors, and the second one must neither be loaded from nor stored to global memory (it is the next row's
first).  Shifted solves and both stage sweeps against the oracle, batches against single items, in the
transposed sweep a store past a stage would overwrite a stage that is already done.  Tolerances as for the other
cluster plans: 8 u (1 + 8 c / h^2) per shifted solve, 32 u of it over a sweep's two stages, in FP64 at least
1e-13 and 4e-13."""
import numpy as np
import pytest

import synth
from oracle.precond import Preconditioner
from oracle.solve import build

from gpu_util import dev, host, to_dev, torch, zeros

pytestmark = pytest.mark.gpu

GRIDS = [(4, 100), (4, 65), (4, 300)]


@pytest.mark.parametrize("ns", GRIDS)
@pytest.mark.parametrize("pre", [2, 0])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_one_vector_rows(ns, pre, prec):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    B, s, T = 40, 2, 1.0
    S = Solver(ns, T, B, tableau=radau_iia(s), prec_P=prec, mg_pre=pre, restart=1, inner_maxit=1, inner_tol=0.0)
    op = build(ns, T, B, "radau", s)
    P = Preconditioner(op, ns, 1, 0.0, 3, pre, 2, 0.8)
    ratio = 1.0 + 8.0 * (op.tau * max(P.D)) * max(n + 1 for n in ns) ** 2
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    floor = 1e-13 if prec == "fp64" else 0.0

    def check(got, ref, f):
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= max(f * u * ratio, f * floor / 8)

    for i in range(s):
        b = synth.random_vector(op.nx, 80 + i)
        check(host(S.shifted_solve(i, to_dev(b), zeros(op.nx))), P.shifted_solve(i, b), 8)
    r = synth.random_vector(s * op.nx, 90)
    for tr in (False, True):
        check(host(S.pint_apply(to_dev(r), zeros(s * op.nx), transpose=tr)), (P.pint_apply_T if tr else P.pint_apply)(r), 32)
    n = s * op.nx
    r = to_dev(synth.random_vector(B * n, 91))
    one = zeros(n)
    for nb in (3, B):
        z = zeros(nb * n)
        S.inner_solve(nb, r[:nb * n], z)
        for b in (0, 1, nb - 1):
            S.inner_solve(1, r[b * n:(b + 1) * n].clone(), one)
            check(host(z[b * n:(b + 1) * n]), host(one), 32)
        again = zeros(nb * n)
        S.inner_solve(nb, r[:nb * n], again)
        assert torch.equal(z, again)
    S.close()
