"""The coarsest level's inverse (one cluster of 16 CTAs per matrix, rows dealt out cyclically): grids
that are a single multigrid level, where a shifted solve is that inverse alone, with fewer rows than
CTAs, one row each, a ragged last round and the largest size."""
import numpy as np
import pytest

import synth
from oracle.solve import build

from gpu_util import dev, host, to_dev, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [(3, 3), (4, 4), (5, 7), (16, 16), (17, 15), (3, 150), (6, 5, 8)])
def test_single_level_shifted_solve_is_the_inverse(ns):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    nt, s = 2, 3
    S = Solver(ns, 1.0, nt, tableau=radau_iia(s), prec_P="fp64", mg_cycles=1)
    op = build(ns, 1.0, nt, "radau", s)
    K = op.K.toarray()
    W, D = radau_iia(s)[0].copy(), []
    for k in range(s):                      # the pivots d_i of A_RK's LDU
        D.append(W[k, k])
        W[k + 1:, k:] -= np.outer(W[k + 1:, k] / W[k, k], W[k, k:])
    for i in range(s):
        M = np.eye(op.nx) + op.tau * D[i] * K
        b = synth.random_vector(op.nx, 60 + i)
        x = host(S.shifted_solve(i, to_dev(b), zeros(op.nx)))
        ref = np.linalg.solve(M, b)
        # n eps cond(M) bounds both sides' rounding; the matrices here have cond(M) <= 1e4
        assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
    S.close()
