"""Edges of the fixed-point reaction kernels that ordinary fields do not reach: directions whose sums
cancel.

Tolerance 1e-10 of the cancellation-aware scales, as for every derivative kernel here."""
import numpy as np
import pytest

import oracle
import paper_2409_06404_gb300 as nk
from paper_2409_06404_gb300 import synth
from conftest import gpu_mechanism, to_dev, host, scaled_err

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.mark.parametrize("K,R", [(9, 21), (53, 120)])
@pytest.mark.parametrize("d", [1e-18, 1e-22, 1e-26, 9e-31])
def test_jvp_cancelling_colliders(cuda, K, R, d):
    """Opposite entries of a direction in two species of equal efficiency and molar mass: their sum
    in d[M] is a rounding remainder far below a float's range."""
    el = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
    mech = synth.make_mechanism(K, R, R // 6, R // 6, elements=el, seed=700 + K).copy()
    mech.W[4] = mech.W[3]
    mech.eff[:, 3] = mech.eff[:, 4] = 3.7
    m = gpu_mechanism(mech)
    n = 96
    st = synth.states_uniform(K, n, seed=K)
    rng = np.random.default_rng(K)
    vT, vY = rng.standard_normal(n), np.zeros((K, n))
    vY[3] = d * (1.0 + rng.random(n))
    vY[4] = -vY[3]
    S = to_dev(st.T, st.p, st.Y, vT, vY)
    for got, want in ((nk.rates_jvp(m, *S), oracle.jvp(mech, st.T, st.p, st.Y, vT, vY, scales=True)),
                      (nk.rhs_jvp(m, *S), oracle.rhs_jvp(mech, st.T, st.p, st.Y, vT, vY, scales=True))):
        for a, o, s in zip(got, want[:2], want[2:]):
            assert scaled_err(host(a), o, s) <= TOL
    m.close()
