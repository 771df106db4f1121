"""Sums of squares of the FP32 inner GMRES are FP64 beyond a thread's few values: vectors whose squared norm passes
FP32's range (but whose entries' squares do not) are solved as any other.  P_tilde is linear and every step
of it scales exactly with a power of two, so the scaled result is the unscaled one's multiple bit for bit."""
import numpy as np
import pytest

import synth
from oracle.solve import build

from gpu_util import dev, host, to_dev, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,nt,mgrit", [((64, 64), 6, 0), ((37, 41), 4, 0), ((48, 48), 8, 4)])
def test_squared_norms_beyond_the_fp32_range(ns, nt, mgrit):
    from paper_2609_16863_gb300 import Solver, radau_iia
    dev()
    S = Solver(ns, 1.0, nt, tableau=radau_iia(2), prec_P="fp32", restart=1, mgrit_m=mgrit)
    r = synth.random_vector(S.n_st, 3)
    z = host(S.precond_apply(to_dev(r), zeros(S.n_st))).copy()
    K = build(ns, 1.0, nt, "radau", 2).K
    t = max(np.sqrt(np.mean((K @ z[n * S.nx:(n + 1) * S.nx]) ** 2)) for n in range(nt))
    # rms |K z| about 2^60: a few squares sum to 2^123, a block's to 2^129 and an item's to more
    k = 60 - int(np.ceil(np.log2(t)))
    scaled = host(S.precond_apply(to_dev(r * 2.0 ** k), zeros(S.n_st)))
    assert np.array_equal(scaled, z * 2.0 ** k)
    S.close()
