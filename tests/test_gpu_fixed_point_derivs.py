"""The derivative kernels and the mixed rates on fixed-point logarithms at species counts on the
edges of their parts (32, 64 and 140 species), reaction counts on the edges of their chunks (36 and
48), ragged point counts, and with points that the fallback takes one by one (outside T in
(128, 4096) K, p in 2^+-100 Pa, sum |Y| up to 1.5, a zero and a negative mass fraction inside).

Tolerances: products and gradients 1e-10 of the cancellation-aware scales (as for every derivative
kernel here).  Single-precision products 2 (t + 8) u of the terms' magnitudes, u = 2^-24, t the
terms added (at most R).  Mixed rates: ln k_f and the falloff are sums of a few single-precision terms of magnitude
up to 400 (E_a/RT at the cold end), each rounded: 4 * 400 * 6e-8 = 1e-4, doubled for the falloff."""
import numpy as np
import pytest

import oracle
import paper_2409_06404_gb300 as nk
from paper_2409_06404_gb300 import synth
from conftest import gpu_mechanism, to_dev, host, scaled_err

pytestmark = pytest.mark.gpu
TOL = 1e-10
U = 2.0 ** -24


def _states(K, n):
    st = synth.states_uniform(K, n, seed=K)
    T, p, Y = st.T.copy(), st.p.copy(), st.Y.copy()
    if n >= 33:
        T[3], T[32] = 4500.0, 4095.0
        Y[:, 5] *= 2.0
        Y[K - 1, 6] = -1e-4
        Y[2, 7] = 0.0
    return T, p, Y


@pytest.mark.parametrize("K,R,n_tb,n_troe,n", [
    (8, 20, 1, 1, 33), (9, 48, 2, 3, 1), (32, 49, 3, 4, 64), (33, 36, 2, 3, 65), (64, 73, 4, 5, 33), (65, 97, 6, 7, 34),
    (140, 150, 9, 11, 33), (141, 150, 9, 11, 5)])
def test_parts_chunks_and_fallback(cuda, K, R, n_tb, n_troe, n):
    el = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
    mech = synth.make_mechanism(K, R, n_tb, n_troe, elements=el, seed=600 + K)
    m = gpu_mechanism(mech)
    T, p, Y = _states(K, n)
    vT, vY = synth.normal(n, 40 + K), synth.normal((K, n), 41 + K)
    wbar, hbar = synth.normal((K, n), 42 + K), synth.normal(n, 43 + K) * 1e-5
    dA = synth.normal(R, 44 + K) * 0.1
    S = to_dev(T, p, Y)
    vTt, vYt, wt, ht, dAt = to_dev(vT, vY, wbar, hbar, dA)
    dw_o, dh_o, dws, dhs = oracle.jvp(mech, T, p, Y, vT, vY, scales=True)

    def close(dw, dh):
        assert scaled_err(host(dw), dw_o, dws) <= TOL and scaled_err(host(dh), dh_o, dhs) <= TOL

    close(*nk.rates_jvp(m, *S, vTt, vYt))
    lin = nk.rates_linearize(m, *S)
    close(*nk.rates_jvp_linearized(m, *S, lin, vTt, vYt))
    lin, w, h = nk.rates_linearize_compact(m, *S, primal=True)
    close(*nk.rates_jvp_linearized_compact(m, *S, lin, vTt, vYt))
    w_o, h_o, ws, hs = oracle.rates(mech, T, p, Y, scales=True)
    assert scaled_err(host(w), w_o, ws) <= TOL and scaled_err(host(h), h_o, hs) <= TOL

    J, Js = oracle.jacobian(mech, T, p, Y, scales=True)
    u = np.vstack([wbar, hbar[None]])
    JTu, scale = np.einsum("nij,in->jn", J, u), np.einsum("nij,in->jn", Js, np.abs(u))
    gT, gY, _ = nk.rates_vjp(m, *S, wt, ht)
    assert scaled_err(host(gT), JTu[0], scale[0]) <= TOL and scaled_err(host(gY), JTu[1:], scale[1:]) <= TOL

    lin = nk.rates_linearize_f32(m, *S)
    dw, dh = nk.rates_jvp_linearized_f32(m, *S, lin, vTt, vYt)
    M = np.einsum("nrc,cn->rn", Js, np.abs(np.vstack([vT[None], vY])))
    bound = 2.0 * (R + 8) * U * M + 1e-25 * M.max(axis=0, keepdims=True)
    assert np.all(np.abs(host(dw) - dw_o) <= bound[:K]) and np.all(np.abs(host(dh) - dh_o) <= bound[K])

    w_o, h_o, ws, hs = oracle.rates(mech, T, p, Y, dlnA=dA, scales=True)
    w, h = nk.rates_eval(m, *S, dlnA=dAt)
    assert scaled_err(host(w), w_o, ws) <= TOL and scaled_err(host(h), h_o, hs) <= TOL
    w, h = nk.rates_eval(m, *S, dlnA=dAt, precision="mixed")
    assert scaled_err(host(w), w_o, ws) <= 2e-4 and scaled_err(host(h), h_o, hs) <= 2e-4
    m.close()
