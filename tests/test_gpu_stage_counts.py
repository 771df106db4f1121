"""Every stage count and long inner solves against the oracle: the products have an instance per stage count up to four
and one beyond, the inner GMRES's kernels one for up to three stages and five steps and ones for more of either.
Whole-vector rows and ragged ones, kappa, Q1, 2D and 3D.  Tolerances as elsewhere: products 1e-13; inner solves
1e-11 in FP64 and 2e-5 in FP32 for up to three steps, and as much again for every three more."""
import numpy as np
import pytest

import synth
from oracle.precond import Preconditioner, gmres_fixed
from oracle.solve import build

from gpu_util import dev, host, rel_max, to_dev, zeros

pytestmark = pytest.mark.gpu


def make(ns, nt, s, prec, kin, itol, disc="fd", kap=False):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    kappa = None
    if kap:
        kappa = np.exp(synth.gaussian_random_field(ns, 0.15, 0.5, synth.rng_for(5, "kappa"), with_boundary=True))
    S = Solver(ns, 1.0, nt, tableau=radau_iia(s), prec_P=prec, disc=disc, kappa=kappa, inner_maxit=kin, inner_tol=itol,
               restart=1)
    op = build(ns, 1.0, nt, "radau", s, disc=disc, kappa=kappa, tab=radau_iia(s))   # (the same coefficients to the last bit)
    return S, op, Preconditioner(op, ns, kin, itol, 3, 2, 2, 0.8)


@pytest.mark.parametrize("s", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("ns,kap", [((24, 24), False), ((23, 18), False), ((17, 20), True), ((8, 8, 8), False),
                                    ((7, 9, 6), True)])
def test_products(ns, kap, s):
    S, op, _ = make(ns, 3, s, "fp32", 3, 0.0, kap=kap)
    x = synth.random_vector(op.n_st, 21)
    assert rel_max(host(S.matvec(to_dev(x), zeros(op.n_st))), op.matvec(x)) <= 1e-13
    assert rel_max(host(S.matvec(to_dev(x), zeros(op.n_st), transpose=True)), op.rmatvec(x)) <= 1e-13
    S.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ns,disc,kap,s,kin,itol", [
    ((24, 20), "fd", False, 4, 6, 0.0), ((24, 20), "fd", False, 8, 6, 0.0), ((23, 21), "fd", True, 5, 16, 1e-9),
    ((24, 20), "fd", False, 3, 16, 1e-9), ((20, 18), "q1", False, 4, 8, 0.0), ((8, 10, 12), "fd", False, 8, 3, 0.0),
    ((9, 10, 7), "fd", True, 4, 8, 0.0), ((24, 20), "fd", False, 8, 16, 0.0),
])
def test_inner_solves(ns, disc, kap, s, kin, itol, prec):
    if prec == "fp32":
        itol = max(itol, 1e-4 if itol else 0.0)
        kin = min(kin, 8) if itol == 0.0 else kin
    nb = 3
    S, op, P = make(ns, nb, s, prec, kin, itol, disc, kap)
    n = s * op.nx
    R = synth.random_vector(nb * n, 50).reshape(nb, n)
    z, its = S.inner_solve(nb, to_dev(R.ravel()), zeros(nb * n))
    z = host(z).reshape(nb, n)
    for b in range(nb):
        ref, k = gmres_fixed(P.theta_apply, P.pint_apply, R[b], kin, itol)
        assert its[b] == k
        tol = -(-k // 3) * (1e-11 if prec == "fp64" else 2e-5)
        print(ns, disc, s, prec, k, rel_max(z[b], ref), tol)
        assert rel_max(z[b], ref) <= tol
    S.close()
