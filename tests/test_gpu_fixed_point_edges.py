"""Edges of the fixed-point reaction kernels that ordinary fields do not reach: directions whose sums
cancel, fields with points outside the form in some or all blocks.

Tolerance 1e-10 of the cancellation-aware scales, as for every derivative kernel here."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2409_06404_gb300 as nk
from paper_2409_06404_gb300 import synth
from conftest import gpu_mechanism, to_dev, host, scaled_err, nu_matrix

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


@pytest.mark.parametrize("K,R", [(9, 21), (53, 120), (120, 200)])
@pytest.mark.parametrize("where", ["all", "one", "warm"])
def test_rejected_blocks(cuda, K, R, where):
    """Zero mass fractions in every point, in one point of the second block, or (no zero) temperatures
    above the form's in every point of the second block: all derivatives, with shifts of ln A."""
    el = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
    mech = synth.make_mechanism(K, R, R // 6, R // 6, elements=el, seed=800 + K)
    m = gpu_mechanism(mech)
    n = 97
    st = synth.states_uniform(K, n, seed=K)
    T, p, Y = st.T.copy(), st.p.copy(), st.Y.copy()
    if where == "warm":
        T[32:64] = 4200.0
    else:
        Y[K // 2, slice(None) if where == "all" else 40] = 0.0
    rng = np.random.default_rng(K)
    vT, vY, wb, hb = rng.standard_normal(n), rng.standard_normal((K, n)), rng.standard_normal((K, n)), 1e-5 * rng.standard_normal(n)
    dA = 0.1 * rng.standard_normal(R)
    S, (vTt, vYt, wbt, hbt, dAt) = to_dev(T, p, Y), to_dev(vT, vY, wb, hb, dA)

    dw, dh, dws, dhs = oracle.jvp(mech, T, p, Y, vT, vY, dlnA=dA, scales=True)
    lin, w, h = nk.rates_linearize_compact(m, *S, dlnA=dAt, primal=True)
    for a, b in (nk.rates_jvp(m, *S, vTt, vYt, dlnA=dAt), nk.rates_jvp_linearized_compact(m, *S, lin, vTt, vYt)):
        assert scaled_err(host(a), dw, dws) <= TOL and scaled_err(host(b), dh, dhs) <= TOL
    wo, ho, ws, hs = oracle.rates(mech, T, p, Y, dlnA=dA, scales=True)
    assert scaled_err(host(w), wo, ws) <= TOL and scaled_err(host(h), ho, hs) <= TOL
    for a, o, s in zip(nk.rhs_jvp(m, *S, vTt, vYt), *[oracle.rhs_jvp(mech, T, p, Y, vT, vY, scales=True)[i:i + 2] for i in (0, 2)]):
        assert scaled_err(host(a), o, s) <= TOL

    gT, gY, g = nk.rates_vjp(m, *S, wbt, hbt, dlnA=dAt)
    J, Js = oracle.jacobian(mech, T, p, Y, dlnA=dA, scales=True)
    u = np.vstack([wb, hb[None]])
    JTu, scale = np.einsum("nij,in->jn", J, u), np.einsum("nij,in->jn", Js, np.abs(u))
    assert scaled_err(host(gT), JTu[0], scale[0]) <= TOL and scaled_err(host(gY), JTu[1:], scale[1:]) <= TOL
    fwd, rev = oracle.rates_of_progress(mech, T, p, Y, dlnA=dA)
    qbar = np.abs(nu_matrix(mech)).T @ (np.abs(wb) + np.abs(hb * oracle.thermo(mech, T, p, Y)["h_k"]))
    assert scaled_err(host(g), oracle.grad_lnA(mech, T, p, Y, wb, hb, dlnA=dA), np.sum(qbar * (fwd + rev), axis=1)) <= TOL
    m.close()


def _median_ms(f):
    f()
    t = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t)[len(t) // 2]


def _pair_only(mech):
    """The same mechanism with five molecules on a side of one reaction, which keeps it off the
    fixed-point kernels."""
    other = mech.copy()
    other.reac_nu[0] = 5
    return other


@pytest.mark.parametrize("name", ["h2_9sp_21rx", "ch4_53sp_325rx"])
@pytest.mark.parametrize("call", ["jvp", "rhs_jvp", "linearize", "vjp"])
def test_rejected_blocks_cost_one_pass(cuda, name, call):
    """Fields all of whose blocks hold a point outside the form take the pair kernels' time: at most
    1.2 of what a mechanism that never enters the fixed-point kernels takes (the set-up that finds
    the points out is about a twentieth of a pass; a whole fixed-point pass is half of one)."""
    mech = synth.mechanism(name)
    n = 65536
    st = synth.states_uniform(mech.K, n, seed=2)
    st.Y[3, ::32] = 0.0
    T, p, Y = to_dev(st.T, st.p, st.Y)
    vT, vY = torch.randn_like(T), torch.randn_like(Y)
    ms = []
    for mm in (mech, _pair_only(mech)):
        m = gpu_mechanism(mm)
        lin = torch.empty((nk.linearization_slots_compact(m), n), dtype=torch.float64, device="cuda")
        ms.append(_median_ms({"jvp": lambda: nk.rates_jvp(m, T, p, Y, vT, vY), "rhs_jvp": lambda: nk.rhs_jvp(m, T, p, Y, vT, vY),
                              "vjp": lambda: nk.rates_vjp(m, T, p, Y, vY, vT),
                              "linearize": lambda: nk.rates_linearize_compact(m, T, p, Y, lin=lin, primal=True)}[call]))
        m.close()
    assert ms[0] <= 1.2 * ms[1], ms


@pytest.mark.parametrize("name", ["h2_9sp_21rx", "ch4_53sp_325rx"])
@pytest.mark.parametrize("T0", [110.0, 4500.0])
def test_rates_out_of_range_cost_one_pass(cuda, name, T0):
    """Rates and sources of fields wholly outside 128 .. 4096 K: as the derivatives above."""
    mech = synth.mechanism(name)
    n = 131072
    st = synth.states_uniform(mech.K, n, seed=2)
    _, p, Y = to_dev(st.T, st.p, st.Y)
    T = torch.full_like(p, T0)
    ms = []
    for mm in (mech, _pair_only(mech)):
        m = gpu_mechanism(mm)
        ms.append([_median_ms(lambda: nk.rates_eval(m, T, p, Y)), _median_ms(lambda: nk.rhs_eval(m, T, p, Y, precision="mixed"))])
        m.close()
    assert ms[0][0] <= 1.2 * ms[1][0] and ms[0][1] <= 1.2 * ms[1][1], ms


def test_noalloc_vjp_takes_two_rows_a_tile(cuda):
    """ln A partial sums take two rows of R per tile of 32 points: 2,000 points of 8,192 reactions fit
    the 8 MiB scratch.  Points of each of the VJP's three kernels share the rows."""
    mech = synth.make_mechanism(K=40, R=8192, n_tb=40, n_troe=40, seed=78)
    m = gpu_mechanism(mech)
    n = 2000
    assert nk.rates_vjp_workspace(m, n) == 2 * 63 * mech.R * 8
    st = synth.states_uniform(mech.K, n, seed=4)
    T, Y = st.T.copy(), st.Y.copy()
    T[320:640] = 4300.0
    Y[5, 640:960] = 0.0
    w = synth.normal((mech.K, n), 5)
    Tt, pt, Yt, wt = to_dev(T, st.p, Y, w)
    gT, gY, g1 = nk.rates_vjp(m, Tt, pt, Yt, wt)
    gT2, gY2, g2 = torch.empty_like(gT), torch.empty_like(gY), torch.empty_like(g1)
    P = lambda t: t.data_ptr()                                                                # noqa: E731
    status = nk.lib().nk_rates_vjp_noalloc(m.handle, n, n, P(Tt), P(pt), P(Yt), None, P(wt), None, P(gT2), P(gY2), P(g2), None)
    assert status == 0, nk.lib().nk_last_error()
    torch.cuda.synchronize()
    assert torch.equal(gT, gT2) and torch.equal(gY, gY2) and torch.equal(g1, g2)
    fwd, rev = oracle.rates_of_progress(mech, T, st.p, Y)
    scale = np.sum((np.abs(nu_matrix(mech)).T @ np.abs(w)) * (fwd + rev), axis=1)
    assert scaled_err(host(g1), oracle.grad_lnA(mech, T, st.p, Y, w), scale) <= TOL
    m.close()


def test_fluxes_of_few_points(cuda):
    """Few points: thermodynamics and diffusion fluxes both wait for one pass of loads per species, the
    fluxes for a second pass of loads that are independent of the first's sums (1.1 of the
    thermodynamics' time where loads of several species are in flight, 1.35 with one at a time)."""
    mech = synth.mechanism("ch4_53sp_325rx")
    m = gpu_mechanism("ch4_53sp_325rx")
    n = 5000
    st = synth.states_uniform(mech.K, n, seed=2)
    T, p, Y = to_dev(st.T, st.p, st.Y)
    D, G = torch.rand_like(Y), torch.randn((3, mech.K, n), dtype=torch.float64, device="cuda")
    many = lambda f: _median_ms(lambda: [f() for _ in range(20)])                             # noqa: E731
    flux, thermo = many(lambda: nk.diffusion_fluxes(m, T, p, Y, D, G)), many(lambda: nk.thermo_eval(m, T, p, Y))
    assert flux <= 1.15 * thermo, (flux, thermo)


@pytest.mark.parametrize("K,R,n", [(9, 21, 29184), (9, 21, 45000), (9, 21, 90000), (16, 48, 45000), (24, 60, 45000)])
def test_products_of_few_species(cuda, K, R, n):
    """Products from stored data at few species, where the number of points chooses between the chunked and
    the pair kernel: the compact ones against the oracle at 200 points, the single-precision ones bit
    for bit against blocks of 1,000 points, which the chunked kernel takes."""
    el = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
    mech = synth.make_mechanism(K, R, 2, 2, elements=el, seed=900 + K)
    m = gpu_mechanism(mech)
    st = synth.states_uniform(K, n, seed=K)
    vT, vY = synth.normal(n, 1), synth.normal((K, n), 2)
    S, (vTt, vYt) = to_dev(st.T, st.p, st.Y), to_dev(vT, vY)
    fT, fY = nk.rhs_eval(m, *S)
    lin = nk.rates_linearize_compact(m, *S)
    i = np.sort(np.random.default_rng(3).choice(n, 200, replace=False))
    sub = lambda a: np.ascontiguousarray(a[..., i])                                           # noqa: E731
    for got, ref in ((nk.rates_jvp_linearized_compact(m, *S, lin, vTt, vYt), oracle.jvp),
                     (nk.rhs_jvp_linearized_compact(m, *S, lin, fT, fY, vTt, vYt), oracle.rhs_jvp)):
        want = ref(mech, sub(st.T), sub(st.p), sub(st.Y), sub(vT), sub(vY), scales=True)
        for a, o, s in zip(got, want[:2], want[2:]):
            assert scaled_err(sub(host(a)), o, s) <= TOL
    lin = nk.rates_linearize_f32(m, *S)
    whole = nk.rates_jvp_linearized_f32(m, *S, lin, vTt, vYt) + nk.rhs_jvp_linearized_f32(m, *S, lin, fT, fY, vTt, vYt)
    for a in range(0, n, 10000):
        b = min(a + 1000, n)
        x = [t[..., a:b].contiguous() for t in (*S, lin, fT, fY, vTt, vYt)]
        part = nk.rates_jvp_linearized_f32(m, *x[:4], *x[6:]) + nk.rhs_jvp_linearized_f32(m, *x)
        assert all(torch.equal(q, w[..., a:b]) for q, w in zip(part, whole))
    m.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_mechanism_constants(cuda, bad):
    """A NaN or infinite polynomial coefficient, or efficiency of a falloff reaction, reaches what depends on
    it, as in the oracle, and nothing else."""
    base = synth.mechanism("h2_9sp_21rx")
    st = synth.states_uniform(base.K, 64, seed=6)
    T = np.linspace(400.0, 2200.0, 64)
    S = to_dev(T, st.p, st.Y)
    mech = base.copy()
    mech.nasa_hi[3, 2] = bad
    m = gpu_mechanism(mech)
    got, want = nk.thermo_eval(m, *S), oracle.thermo(mech, T, st.p, st.Y)
    for key in ("cp_k", "h_k", "g_k", "cp_mix", "h_mix"):
        a, o = host(got[key]), np.asarray(want[key])
        assert np.array_equal(np.isfinite(a), np.isfinite(o)), key
        ok = np.isfinite(o)
        assert np.allclose(a[ok], o[ok], rtol=1e-11), key
    m.close()
    mech = base.copy()
    r = int(np.flatnonzero(mech.rtype == 2)[0])
    mech.eff[r, 2] = bad
    m = gpu_mechanism(mech)
    w = host(nk.rates_eval(m, *S)[0])
    wo = oracle.rates(mech, T, st.p, st.Y)[0]
    assert np.array_equal(np.isfinite(w), np.isfinite(wo))
    m.close()


@pytest.mark.parametrize("K,R,n", [(9, 20, 33), (9, 48, 1), (32, 49, 64), (33, 36, 97), (53, 325, 160), (65, 97, 96), (140, 150, 65)])
def test_solver_linearization(cuda, K, R, n):
    """The per-entry linearization that the reactor keeps to itself (fixed-point pass, pair kernel for blocks
    outside its form: the second block here): products from it against the oracle."""
    el = ("H", "O", "N") if K < 20 else ("C", "H", "O", "N")
    mech = synth.make_mechanism(K, R, max(1, R // 16), max(1, R // 13), elements=el, seed=650 + K)
    m = gpu_mechanism(mech)
    st = synth.states_uniform(K, n, seed=K)
    T, Y = st.T.copy(), st.Y.copy()
    if n >= 64:
        T[33] = 4500.0
        Y[2, 34], Y[K - 1, 35] = 0.0, -1e-4
    if n >= 96:
        Y[K - 1, 70] = -1e-4
    vT, vY, dA = synth.normal(n, 1), synth.normal((K, n), 2), 0.1 * synth.normal(R, 3)
    S, (vTt, vYt, dAt) = to_dev(T, st.p, Y), to_dev(vT, vY, dA)
    lin = torch.empty((nk.linearization_slots(m), n), dtype=torch.float64, device="cuda")
    f = nk.lib()["_ZN2nk23launch_linearize_solverERKNS_7DevMechEllPKdS4_S4_S4_PdlP11CUstream_st"]
    f.argtypes = [ctypes.c_void_p] + [ctypes.c_int64] * 2 + [ctypes.c_void_p] * 5 + [ctypes.c_int64, ctypes.c_void_p]
    P = lambda t: t.data_ptr()                                                                # noqa: E731
    assert f(m.handle, n, n, *map(P, S), P(dAt), P(lin), n, torch.cuda.current_stream().cuda_stream) == 0
    a, b = nk.rates_jvp_linearized(m, *S, lin, vTt, vYt)
    dw, dh, dws, dhs = oracle.jvp(mech, T, st.p, Y, vT, vY, dlnA=dA, scales=True)
    assert scaled_err(host(a), dw, dws) <= TOL and scaled_err(host(b), dh, dhs) <= TOL
    m.close()


def test_noalloc_vjp_with_fewer_rows(cuda):
    """1,500 reactions on 20,000 points: more rows of ln A sums than the 8 MiB scratch holds at full grids;
    the call runs fewer blocks and gives the same gradients, marked points included."""
    mech = synth.make_mechanism(K=53, R=1500, n_tb=40, n_troe=40, seed=79)
    m = gpu_mechanism(mech)
    n = 20000
    assert nk.rates_vjp_workspace(m, n) > 8 * 2 ** 20
    st = synth.states_uniform(mech.K, n, seed=4)
    T, Y = st.T.copy(), st.Y.copy()
    T[3200:6400] = 4300.0
    Y[5, 9600:12800] = 0.0
    w = synth.normal((mech.K, n), 5)
    Tt, pt, Yt, wt = to_dev(T, st.p, Y, w)
    gT, gY, g1 = nk.rates_vjp(m, Tt, pt, Yt, wt)
    gT2, gY2, g2 = torch.empty_like(gT), torch.empty_like(gY), torch.empty_like(g1)
    P = lambda t: t.data_ptr()                                                                # noqa: E731
    status = nk.lib().nk_rates_vjp_noalloc(m.handle, n, n, P(Tt), P(pt), P(Yt), None, P(wt), None, P(gT2), P(gY2), P(g2), None)
    assert status == 0, nk.lib().nk_last_error()
    torch.cuda.synchronize()
    assert torch.equal(gT, gT2) and torch.equal(gY, gY2)
    fwd, rev = oracle.rates_of_progress(mech, T, st.p, Y)
    scale = np.sum((np.abs(nu_matrix(mech)).T @ np.abs(w)) * (fwd + rev), axis=1)
    assert scaled_err(host(g1), host(g2), scale) <= 1e-12
    m.close()
