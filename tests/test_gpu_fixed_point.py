"""The FP64 rates and sources on fixed-point logarithms against the oracle: species counts at the
edges of the parts (8 species each), reaction counts at the edges of the chunks (48), ragged point
counts, and states at and beyond the form's ranges (T in (128, 4096) K, p in 2^+-100 Pa, sum |Y|
up to 1.5), which the fallback pass takes point by point.

Tolerance 1e-11 of the cancellation-aware scales: a rate term's exponent (up to about 700 in
natural units at the cold edge) carries some 2e-13 from the oracle's own double exponent and 2e-12
from the fallback's pairs; the fixed-point form itself about 1e-14."""
import numpy as np
import pytest

import oracle
import paper_2409_06404_gb300 as nk
from paper_2409_06404_gb300 import synth
from conftest import P_ATM, gpu_mechanism, to_dev, host, scaled_err

pytestmark = pytest.mark.gpu
TOL = 1e-11


def _check(mech, m, T, p, Y, dlnA=None):
    dA = None if dlnA is None else to_dev(dlnA)[0]
    w, h = nk.rates_eval(m, *to_dev(T, p, Y), dlnA=dA)
    wo, ho, ws, hs = oracle.rates(mech, T, p, Y, dlnA=dlnA, scales=True)
    assert scaled_err(host(w), wo, ws) <= TOL
    assert scaled_err(host(h), ho, hs) <= TOL


@pytest.mark.parametrize("K,R,n_tb,n_troe,n", [
    (8, 20, 1, 1, 1), (9, 47, 2, 3, 33), (16, 48, 3, 4, 64), (31, 49, 3, 3, 65), (32, 96, 6, 7, 31), (33, 97, 6, 7, 127),
    (64, 144, 9, 11, 95), (65, 250, 15, 19, 96),
    (128, 300, 18, 23, 40), (129, 310, 19, 23, 33)])
def test_parts_and_chunks(cuda, K, R, n_tb, n_troe, n):
    el = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
    mech = synth.make_mechanism(K, R, n_tb, n_troe, elements=el, seed=400 + K)
    m = gpu_mechanism(mech)
    st = synth.states_uniform(K, n, seed=K)
    _check(mech, m, st.T, st.p, st.Y)
    rng = np.random.default_rng(K)
    _check(mech, m, st.T, st.p, st.Y, dlnA=rng.standard_normal(R))
    m.close()


def test_range_edges(cuda):
    """One block after another with points inside, at and beyond the ranges, so that the fallback
    takes single points; the points inside keep the bits they have without such neighbours."""
    mech = synth.mechanism("ch4_53sp_325rx")
    m = gpu_mechanism("ch4_53sp_325rx")
    n = 200
    st = synth.states_uniform(mech.K, n, seed=8)
    T, p, Y = st.T.copy(), st.p.copy(), st.Y.copy()
    keep = np.ones(n, bool)

    def odd(i, **kw):
        keep[i] = False
        if "T" in kw:
            T[i] = kw["T"]
        if "p" in kw:
            p[i] = kw["p"]
        if "Y" in kw:
            Y[:, i] = kw["Y"]

    odd(3, T=128.0), odd(5, T=np.nextafter(128.0, 200.0)), odd(6, T=4096.0), odd(37, T=np.nextafter(4096.0, 0.0))
    odd(38, T=np.float64(1000.0)), odd(39, T=np.nextafter(1000.0, 2000.0)), odd(40, T=5000.0), odd(41, T=200.0)
    odd(64, p=0.01 * P_ATM), odd(65, p=50 * P_ATM), odd(66, p=1e-3)
    odd(99, Y=2.0 * Y[:, 99]), odd(100, Y=1.49 * Y[:, 100]), odd(101, Y=1e-6 * Y[:, 101])
    sub = Y[:, 130].copy()
    sub[:3] = [5e-324, 0.0, 1e-300]
    odd(130, Y=sub)
    neg = Y[:, 131].copy()
    neg[::5] *= -1e-3
    odd(131, Y=neg)
    one = np.zeros(mech.K)
    one[7] = 1.0
    odd(199, Y=one)
    _check(mech, m, T, p, Y)
    w = host(nk.rates_eval(m, *to_dev(T, p, Y))[0])
    w0 = host(nk.rates_eval(m, *to_dev(st.T, st.p, st.Y))[0])
    assert np.array_equal(w[:, keep], w0[:, keep])
    # the sources' form takes the same points
    fT, fY = nk.rhs_eval(m, *to_dev(T, p, Y))
    fTo, fYo, sT, sY = oracle.rhs(mech, T, p, Y, scales=True)
    assert scaled_err(host(fY), fYo, sY) <= TOL and scaled_err(host(fT), fTo, sT) <= TOL


def test_large_shift_and_nonfinite(cuda):
    """A shift of ln A beyond the fixed-point form scales the rates all the same; a NaN reaches
    every point; a NaN state stays in its point."""
    mech = synth.mechanism("h2_9sp_21rx")
    m = gpu_mechanism("h2_9sp_21rx")
    st = synth.states_uniform(mech.K, 70, seed=3)
    d = np.zeros(mech.R)
    d[2] = np.nan
    w, _ = nk.rates_eval(m, *to_dev(st.T, st.p, st.Y), dlnA=to_dev(d)[0])
    hit = sorted(set(mech.reac_sp[mech.reac_ptr[2]:mech.reac_ptr[3]]) | set(mech.prod_sp[mech.prod_ptr[2]:mech.prod_ptr[3]]))
    assert np.all(np.isnan(host(w)[hit]))
    d[2] = -3000.0
    w, _ = nk.rates_eval(m, *to_dev(st.T, st.p, st.Y), dlnA=to_dev(d)[0])
    d[2] = -2000.0
    w2, _ = nk.rates_eval(m, *to_dev(st.T, st.p, st.Y), dlnA=to_dev(d)[0])
    assert np.array_equal(host(w), host(w2))
    T = st.T.copy()
    T[[0, 33]] = [np.nan, -5.0]
    w3, h3 = nk.rates_eval(m, *to_dev(T, st.p, st.Y))
    w0, h0 = nk.rates_eval(m, *to_dev(st.T, st.p, st.Y))
    ok = np.ones(70, bool)
    ok[[0, 33]] = False
    assert np.all(np.isnan(host(w3)[:, 0])) and np.array_equal(host(w3)[:, ok], host(w0)[:, ok])
    assert np.array_equal(host(h3)[ok], host(h0)[ok])
