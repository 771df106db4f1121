"""The FP64 product against its own coefficients in extended precision: relative rms error of the stage rows.  K v, the
largest term, is added last: the error is then that of one rounding of the result's size, one of K v's differences (of
neighbours' size) and small ones, 0.9e-16 by host emulation; rounding every partial sum at the result's size gives 1.2e-16.
The bound lies between, 1.05e-16.  n + 1 is a power of two, so that 1 / h^2 is exact."""
import numpy as np
import pytest

import synth

from gpu_util import dev, host, to_dev, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,nt,s", [((63, 63), 16, 3), ((63, 31), 8, 3), ((31, 31, 31), 4, 2), ((127, 127), 32, 4)])
def test_stage_rows(ns, nt, s):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("no extended precision on this host")
    A, b, c = radau_iia(s)
    S = Solver(ns, 1.0, nt, tableau=(A, b, c), prec_P="fp32", restart=1)
    x = synth.random_vector(S.n_st, 31)
    y = host(S.matvec(to_dev(x), zeros(S.n_st)))
    L = np.longdouble
    nx, shape = S.nx, tuple(reversed(ns))

    def K(u):
        w = np.pad(u.reshape((-1,) + shape).astype(L), [(0, 0)] + [(1, 1)] * len(ns))
        core = tuple([slice(None)] + [slice(1, -1)] * len(ns))
        out = 0
        for a in range(1, len(ns) + 1):
            lo, hi = list(core), list(core)
            lo[a], hi[a] = slice(0, -2), slice(2, None)
            out = out + L((shape[a - 1] + 1) ** 2) * (2 * w[core] - w[tuple(lo)] - w[tuple(hi)])
        return out.reshape(u.shape)

    v, V = x[:(nt + 1) * nx].reshape(nt + 1, nx), x[(nt + 1) * nx:].reshape(nt, s, nx)
    KV, Kv = K(V.reshape(nt * s, nx)).reshape(nt, s, nx), K(v[:-1])
    ref = V + Kv[:, None] + sum(L(1.0 / nt * A[:, j])[None, :, None] * KV[:, j][:, None] for j in range(s))
    err = y[(nt + 1) * nx:].reshape(nt, s, nx) - ref
    rel = float(np.sqrt((err ** 2).sum() / (ref ** 2).sum()))
    print(ns, nt, s, rel)
    assert rel <= 1.05e-16
    S.close()
