"""Shifted solves on thread-block clusters at the edges of their plans: widths that are not whole vectors,
CTAs with a single row (ghost rows from several CTAs), few vectors per row, every number of sweeps the
ghost regions are planned for and the ones that fall back to single ghost rows, one to four cycles
(the program's parts for the first, odd and even cycles), kappa fields, Q1.  FP64 against the oracle's
V-cycles, both precisions to the unit roundoff times the diagonal's ratio 1 + 8 c / h^2 (the cancellation of
A x) with a factor 8 for the chain of sweeps, in FP64 at least 1e-13.  Launches repeat bit for bit (an exchange without its barrier
would show as differences)."""
import numpy as np
import pytest

import synth
from oracle.precond import Preconditioner
from oracle.solve import build

from gpu_util import dev, host, to_dev, zeros

pytestmark = pytest.mark.gpu

CASES = [  # grid, pre, post, cycles, disc, kappa
    ((17, 17), 2, 2, 3, "fd", False), ((33, 16), 2, 2, 2, "fd", False), ((65, 35), 2, 2, 4, "fd", True),
    ((80, 72), 2, 2, 3, "q1", False), ((127, 95), 2, 2, 1, "fd", False), ((70, 129), 1, 1, 3, "fd", False),
    ((66, 66), 3, 2, 3, "fd", True), ((48, 50), 2, 3, 3, "fd", False), ((64, 67), 0, 2, 2, "fd", False),
    ((64, 64), 2, 0, 3, "fd", False), ((37, 41), 1, 2, 4, "q1", False), ((5, 100), 2, 2, 3, "fd", False),
    ((250, 254), 2, 2, 3, "fd", False), ((256, 256), 2, 2, 2, "fd", True),
]


@pytest.mark.parametrize("ns,pre,post,cycles,disc,kap", CASES)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_cluster_plans_match_the_oracle(ns, pre, post, cycles, disc, kap, prec):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    nt, s, T = 4, 2, 0.25
    kappa = None
    if kap:
        kappa = np.exp(synth.gaussian_random_field(ns, 0.15, 0.5, synth.rng_for(5, "kappa"), with_boundary=True))
    S = Solver(ns, T, nt, tableau=radau_iia(s), prec_P=prec, mg_cycles=cycles, mg_pre=pre, mg_post=post, mg_omega=0.8,
               disc=disc, kappa=kappa, restart=1)
    op = build(ns, T, nt, "radau", s, disc=disc, kappa=kappa)
    P = Preconditioner(op, ns, 3, 0.0, cycles, pre, post, 0.8)
    for i in range(s):
        b = synth.random_vector(op.nx, 70 + i)
        bd, x = to_dev(b), zeros(op.nx)
        got = host(S.shifted_solve(i, bd, x)).copy()
        for _ in range(4):
            assert np.array_equal(host(S.shifted_solve(i, bd, x)), got)
        ref = P.shifted_solve(i, b)
        err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        c = op.tau * P.D[i] * (1.0 if kappa is None else kappa.max())
        ratio = 1.0 + 8.0 * c * max(n + 1 for n in ns) ** 2
        print(ns, prec, i, err)
        assert err <= (max(8 * 2.0 ** -53 * ratio, 1e-13) if prec == "fp64" else 8 * 2.0 ** -24 * ratio)
    S.close()
