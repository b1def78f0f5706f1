"""Which states the tile kernels keep: subnormal mass fractions and a third body's [M] of zero are
inside the tables, room temperature is for every workload mechanism, and a tile without any
state inside is left to the FP64 kernel at once, next to ordinary tiles and in every form of
the kernels.  Tolerances as in test_gpu_tile and test_gpu_jvp_tile (1e-11 of the gross scale)
and test_gpu_transport."""
import copy

import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COLD = slice(32, 96)                 # two whole tiles


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


@pytest.fixture(scope="module")
def load(mech_files):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    made = {}

    def get(idx, options=None):
        if (idx, options) not in made:
            made[idx, options] = (B.Mechanism(mech_files[0][idx], options), O.Oracle(mech_files[0][idx]))
            assert made[idx, options][0].stat("tile") == 1
            assert made[idx, options][0].stat("tile_t_lo") < 298.15
        return made[idx, options]
    return get


def _states(orc, idx, n, seed, cold):
    st = synth.config_states(idx, n=n, offset_seed=seed)
    T = st.T.copy()
    T[COLD] = np.linspace(*cold, T[COLD].size)
    T[5], T[6] = 298.15, 300.0
    return orc.density(st.p, T, st.Y), T, st.Y.copy()


def _check_rates(m, orc, rho, T, Y, w):
    ow, G = orc.net_production_rates(rho, T, Y, with_gross=True)
    assert np.all(np.abs(w.cpu().numpy() - ow) <= 1e-11 * G + 1e-300)


@pytest.mark.parametrize("idx,options,cold", [(0, None, (160.0, 200.0)), (1, None, (160.0, 200.0)),
                                              (4, "variant=warp", (240.0, 285.0))])
def test_rates_of_cold_tiles(load, idx, options, cold):
    m, orc = load(idx, options)
    rho, T, Y = _states(orc, idx, 140, 131, cold)
    w = m.net_production_rates(_t(rho), _t(Y), T=_t(T))
    _check_rates(m, orc, rho, T, Y, w)
    e = orc.internal_energy(T, Y)
    w, T1 = m.net_production_rates(_t(rho), _t(Y), e=_t(e))
    oT, _, bad = orc.temperature(e, Y)
    assert bad == 0 and m.nonconverged() == 0
    assert np.max(np.abs(T1.cpu().numpy() - oT) / oT) <= 1e-10
    _check_rates(m, orc, rho, T1.cpu().numpy(), Y, w)
    # alone, as beside others (a cluster of blocks per tile where the mechanism has chunks)
    for p in (5, 40):
        a = m.net_production_rates(_t(rho[p:p + 1]), _t(Y[:, p:p + 1]), T=_t(T[p:p + 1]))
        _check_rates(m, orc, rho[p:p + 1], T[p:p + 1], Y[:, p:p + 1], a)


@pytest.mark.parametrize("idx", [0, 1])
def test_derivatives_and_transport_of_cold_tiles(load, mech_files, idx):
    """Cold tiles have the bits of the FP64 kernels alone, the others their parity."""
    from paper_2503_24286_gb300 import binding as B
    m, orc = load(idx)
    fp64 = B.Mechanism(mech_files[0][idx], "tile=0")
    rho, T, Y = _states(orc, idx, 100, 132, (160.0, 200.0))
    warm = np.r_[0:32, 96:100]
    rng = np.random.default_rng(133)
    tangents = (0.1 * rho * rng.standard_normal(100), rng.standard_normal(100), 1e-3 * rng.standard_normal((orc.N, 100)))
    wb = rng.standard_normal((orc.N, 100))

    def check(call, ref, scale):
        a, b = (np.vstack([x.cpu().numpy().reshape(-1, 100) for x in call(h)]) for h in (m, fp64))
        assert np.array_equal(a[:, COLD], b[:, COLD], equal_nan=True)
        assert np.all(np.abs(a - ref)[:, warm] <= scale[:, warm])

    state = (rho, T, Y)
    dev = [_t(x) for x in state]
    check(lambda h: [h.jvp(*dev, *[_t(x) for x in tangents])], orc.jvp(*state, *tangents),
          1e-11 * orc.jvp_scale(*state, *tangents) + 1e-250)
    check(lambda h: h.vjp(*dev, _t(wb)), np.vstack([np.asarray(x).reshape(-1, 100) for x in orc.vjp(*state, wb)]),
          1e-11 * orc.vjp_scale(*state, wb) + 1e-250)
    NP = orc.N + 1
    check(lambda h: [h.jacobian(*dev)], orc.jacobian(*state).reshape(NP * NP, -1),
          1e-11 * orc.jacobian_gross(*state)[:, 1:].reshape(NP * NP, -1) + 1e-250)
    mu, kappa, D = orc.transport(T, Y)
    parts = {"mu": (mu[None], 1e-12), "kappa": (kappa[None], 1e-12), "diffusivities": (D, 2e-11)}
    for names in (("mu", "kappa", "diffusivities"), ("kappa", "diffusivities"), ("diffusivities",)):
        kw = {k: k in names for k in parts}
        ref = np.vstack([parts[k][0] for k in names])
        tol = np.vstack([parts[k][1] * np.abs(parts[k][0]) for k in names])
        check(lambda h: [x for x in h.transport(_t(T), _t(Y), **kw) if x is not None], ref, tol)


@pytest.mark.parametrize("idx", [0, 1])
def test_subnormal_fractions(load, idx):
    """Rates of states with subnormal fractions.  In double the oracle's own concentrations of
    those species are subnormal, with few bits or none, so the reference is its extended
    precision and the gross scale is that of fractions of at least 2^-1010 (concentrations of at
    least 2^-1022): 1e-11 of it, as elsewhere."""
    m, orc = load(idx)
    rho, T, Y = _states(orc, idx, 96, 134, (400.0, 2000.0))
    rng = np.random.default_rng(135)
    sub = rng.random(Y.shape) < 0.3
    sub[np.argmax(Y, axis=0), np.arange(96)] = False
    Y[sub] = rng.integers(1, 1 << 52, sub.sum()) * 2.0 ** -1074 * rng.choice([1.0, 2.0 ** -40], sub.sum())
    Y[sub & (rng.random(Y.shape) < 0.1)] = 5e-324
    Y[sub & (rng.random(Y.shape) < 0.1)] *= -1.0
    w = m.net_production_rates(_t(rho), _t(Y), T=_t(T)).cpu().numpy()
    _, G = orc.net_production_rates(rho, T, np.maximum(np.abs(Y), 2.0 ** -1010), with_gross=True)
    assert np.all(np.abs(w - orc.net_production_rates_ld(rho, T, Y)) <= 1e-11 * G + 1e-300)


@pytest.mark.parametrize("idx", [0])
def test_derivatives_without_third_bodies(load, tmp_path, idx):
    """[M] of zero in three-body reactions (efficiencies of 0 for all that is there): JVP, VJP and
    Jacobian against the oracle, whose sum of products is exactly zero; the kernels' sum is its
    rounding, 2 (N + 8) 2^-53 of the terms, so the tolerance adds that fraction of the scale
    with efficiencies of at least 1."""
    from paper_2503_24286_gb300 import binding as B
    load(idx)
    m = copy.deepcopy(synth.config_mechanism(idx))
    zero = np.arange(0, m.n_species, 2)
    for r in m.reactions:
        if r.kind == "falloff":
            r.kind, r.low, r.troe = "threebody", None, None
        if r.kind == "threebody":
            r.efficiencies.update({int(k): 0.0 for k in zero})
    full = copy.deepcopy(m)
    for r in full.reactions:
        r.efficiencies = {k: max(e, 1.0) for k, e in r.efficiencies.items()}
    paths = [str(tmp_path / s) for s in ("zero.txt", "full.txt")]
    for x, p in zip((m, full), paths):
        synth.write_mechanism(x, p)
    lib, orc, ofull = B.Mechanism(paths[0]), O.Oracle(paths[0]), O.Oracle(paths[1])
    st = synth.config_states(idx, n=40, offset_seed=136)
    T, Y = st.T, st.Y.copy()
    Y[1::2, ::3] = 0.0
    Y /= Y.sum(axis=0)
    rho = orc.density(st.p, T, Y)
    N, rng = orc.N, np.random.default_rng(137)
    a = (rho, T, Y, 0.1 * rho * rng.standard_normal(40), rng.standard_normal(40), 1e-3 * rng.standard_normal((N, 40)))
    noise = 2 * (N + 8) * 2.0 ** -53
    tol = lambda s, f: 1e-11 * s + noise * f + 1e-250  # noqa: E731
    assert np.all(np.abs(lib.jvp(*[_t(x) for x in a]).cpu().numpy() - orc.jvp(*a)) <= tol(orc.jvp_scale(*a), ofull.jvp_scale(*a)))
    wb = rng.standard_normal((N, 40))
    g = np.vstack([x.cpu().numpy().reshape(-1, 40) for x in lib.vjp(_t(rho), _t(T), _t(Y), _t(wb))])
    o = np.vstack([np.asarray(x).reshape(-1, 40) for x in orc.vjp(rho, T, Y, wb)])
    assert np.all(np.abs(g - o) <= tol(orc.vjp_scale(rho, T, Y, wb), ofull.vjp_scale(rho, T, Y, wb)))
    J = lib.jacobian(_t(rho), _t(T), _t(Y)).cpu().numpy().reshape(N + 1, N + 1, -1)
    Jo = orc.jacobian(rho, T, Y).reshape(J.shape)
    assert np.all(np.abs(J - Jo) <= tol(orc.jacobian_gross(rho, T, Y)[:, 1:], ofull.jacobian_gross(rho, T, Y)[:, 1:]))
