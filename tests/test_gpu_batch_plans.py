"""Batched inner solves against single ones.  Grids that take clusters of 8, 4 or 2 CTAs in large batches (more than
32 items in FP32 and FP64) and grids too large for a cluster, whose batched 2D transfers run by vectors of columns
(n_1 odd and even, coarse levels of odd width).  Single items take the 16-CTA plan or the transfers a point at a time.
One inner step each, so a result is off by its two stages' shifted solves: 8 u (1 + 8 c / h^2) per solve (the
cancellation of A x and the chain of sweeps, as for a single cluster), two stages, two results: 32 u (1 + 8 c / h^2),
in FP64 at least 4e-13."""
import numpy as np
import pytest

import synth

from gpu_util import dev, host, to_dev, torch, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ns,B,kap", [
    ((64, 64), 40, False), ((37, 41), 80, False), ((127, 95), 16, True), ((128, 128), 64, True), ((33, 16), 150, False),
    ((512, 300), 16, False), ((516, 259), 17, True), ((500, 515), 16, False),
])
def test_batched_inner_solves_match_single_ones(ns, B, kap, prec):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    kappa = None
    if kap:
        kappa = np.exp(synth.gaussian_random_field(ns, 0.15, 0.5, synth.rng_for(5, "kappa"), with_boundary=True))
    s, T = 2, 1.0
    S = Solver(ns, T, B, tableau=radau_iia(s), prec_P=prec, kappa=kappa, restart=1, inner_maxit=1, inner_tol=0.0)
    n = s * S.nx
    r = to_dev(synth.random_vector(B * n, 7))
    z, one = zeros(B * n), zeros(n)
    S.inner_solve(B, r, z)
    c = T / B * (1.0 if kappa is None else kappa.max())
    ratio = 1.0 + 8.0 * c * max(m + 1 for m in ns) ** 2
    tol = max(32 * 2.0 ** -53 * ratio, 4e-13) if prec == "fp64" else 32 * 2.0 ** -24 * ratio
    for b in (0, 1, B // 2, B - 1):
        S.inner_solve(1, r[b * n:(b + 1) * n].clone(), one)
        ref = host(one)
        err = np.linalg.norm(host(z[b * n:(b + 1) * n]) - ref) / np.linalg.norm(ref)
        print(ns, B, prec, b, err, tol)
        assert err <= tol
    again = zeros(B * n)
    S.inner_solve(B, r, again)
    assert torch.equal(z, again)
    S.close()
