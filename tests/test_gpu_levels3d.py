"""The 3D level kernels at the edges of their tiles and vectors: shifted solves (one item) on grids whose rows
are shorter than a warp, of one warp, of four warps and beyond the tiles' 128 columns, with row and plane
counts that leave ragged tiles, constant and variable kappa, against the oracle's V-cycles (to the unit
roundoff times the diagonal's ratio 1 + 12 c / h^2, the cancellation of A x, with a factor 8 for the chain of
sweeps, in FP64 at least 1e-13)."""
import numpy as np
import pytest

import synth
from oracle.precond import Preconditioner
from oracle.solve import build

from gpu_util import dev, host, to_dev, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,kap", [((7, 9, 11), True), ((33, 9, 10), False), ((32, 12, 5), True), ((128, 12, 13), False),
                                    ((129, 12, 13), False), ((23, 24, 25), True), ((48, 20, 16), False)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_level_kernels_match_the_oracle(ns, kap, prec):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    nt, s, T = 3, 2, 0.25
    kappa = None
    if kap:
        kappa = np.exp(synth.gaussian_random_field(ns, 0.15, 0.5, synth.rng_for(6, "kappa"), with_boundary=True))
    S = Solver(ns, T, nt, tableau=radau_iia(s), prec_P=prec, kappa=kappa, restart=1)
    op = build(ns, T, nt, "radau", s, kappa=kappa)
    P = Preconditioner(op, ns, 3, 0.0, 3, 2, 2, 0.8)
    u = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    for i in range(s):
        b = synth.random_vector(op.nx, 90 + i)
        x = host(S.shifted_solve(i, to_dev(b), zeros(op.nx)))
        ref = P.shifted_solve(i, b)
        c = op.tau * P.D[i] * (1.0 if kappa is None else kappa.max())
        ratio = 1.0 + 12.0 * c * max(n + 1 for n in ns) ** 2
        err = np.linalg.norm(x - ref) / np.linalg.norm(ref)
        assert err <= max(8 * u * ratio, 1e-13 if prec == "fp64" else 0.0), (ns, i, err)
    S.close()


@pytest.mark.parametrize("ns,fmt", [((48, 40, 36), "bf16"), ((48, 40, 36), "fp16"), ((47, 22, 25), "bf16")])
def test_level_kernels_match_the_storage_emulation(ns, fmt):
    """16-bit storage at level sizes where every level kernel runs: in the 2-norm within half a unit of the format,
    the rounding of the stored result itself (entry by entry, flips of intermediate roundings on four levels
    reach many units of the smallest entries)."""
    import oracle.lowprec as lp
    from test_gpu_lowprec import emulation, make
    S, op, P = make(ns, 2, 2, fmt)
    E = emulation(P, fmt, fmt, 2, False)
    for i in range(2):
        b = synth.random_vector(op.nx, 160 + i)
        x = host(S.shifted_solve(i, to_dev(b), zeros(op.nx)))
        ref = E.mg[i].solve(lp.store_rows(b, ns[0], fmt), 3, E.plan_single).astype(np.float64)
        err = np.linalg.norm(x - ref) / np.linalg.norm(ref)
        assert err <= (2.0 ** -9 if fmt == "bf16" else 2.0 ** -12), (ns, i, err)
    S.close()
