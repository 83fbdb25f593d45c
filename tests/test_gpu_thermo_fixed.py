"""Thermo and diffusion fluxes from the integer polynomials against the oracle: temperatures at the
ends of the polynomials' ranges (64 and 4096 K, T_mid, where doubles take over outside), species
whose T_mid differ, ragged point counts.  Relative tolerance 1e-13: the polynomials' terms reach
some hundred times their sum at the ends, with 2^-53 each, in the oracle as here."""
import numpy as np
import pytest

import oracle
import paper_2409_06404_gb300 as nk
from paper_2409_06404_gb300 import synth
from conftest import R_GAS, P_ATM, gpu_mechanism, to_dev, host, scaled_err

pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.mark.parametrize("K,n,mids", [(9, 1, False), (9, 63, True), (53, 65, False), (53, 129, True), (120, 40, False)])
def test_thermo_and_fluxes(cuda, K, n, mids):
    el = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
    mech = synth.make_mechanism(K, 2 * K, 1, 1, elements=el, seed=K).copy()
    rng = np.random.default_rng(K)
    if mids:
        mech.T_mid = rng.choice([800.0, 1000.0, 1023.5, 1400.0], K)
    m = gpu_mechanism(mech)
    st = synth.states_uniform(K, n, seed=n)
    T = st.T.copy()
    edges = [64.0, 63.99, 1000.0, np.nextafter(1000.0, 2e3), 4095.9, 4096.0, 6000.0, 20.0, 300.0, 1400.0, 800.0]
    T[:min(n, len(edges))] = edges[:min(n, len(edges))]
    o = nk.thermo_eval(m, *to_dev(T, st.p, st.Y))
    r = oracle.thermo(mech, T, st.p, st.Y)
    RT = R_GAS * T
    hs = np.sum(np.abs(st.Y * r["h_k"]) / mech.W[:, None], axis=0)
    # magnitudes of the polynomials' terms (they cancel far outside the fits)
    lo = (T[None, :] <= np.asarray(mech.T_mid)[:, None])[:, None, :]
    a = np.abs(np.where(lo, mech.nasa_lo[:, :, None], mech.nasa_hi[:, :, None]))
    cps = R_GAS * sum(a[:, j] * T ** j for j in range(5))
    for key, scale in (("cp_k", cps), ("h_k", T * cps + R_GAS * a[:, 5]), ("g_k", 10 * T * cps + R_GAS * a[:, 5] + RT * a[:, 6]),
                       ("cp_mix", np.sum(st.Y * cps / mech.W[:, None], axis=0)), ("Wbar", np.abs(r["Wbar"])),
                       ("h_mix", hs + np.sum(st.Y * T * cps / mech.W[:, None], axis=0)), ("rho", np.abs(r["rho"]))):
        assert scaled_err(host(o[key]), r[key], scale) <= TOL, key
    D = rng.uniform(1e-5, 1e-3, (K, n))
    G = rng.standard_normal((3, K, n))
    j, Vc, hf = nk.diffusion_fluxes(m, *to_dev(T, st.p, st.Y, D, G))
    jo, Vo, ho = oracle.diffusion(mech, T, st.p, st.Y, D, G)
    rho, Wb = r["rho"], r["Wbar"]
    av = rho * mech.W[:, None] / Wb * D * np.abs(G)
    js = av + st.Y * av.sum(axis=1)[:, None]
    assert scaled_err(host(j), jo, js) <= TOL
    assert scaled_err(host(Vc), Vo, av.sum(axis=1) / rho) <= TOL
    assert scaled_err(host(hf), ho, np.sum(cps / mech.W[:, None] * js, axis=1)) <= TOL
    m.close()
