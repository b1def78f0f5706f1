"""The FP64 kernels by themselves (tile=0) against the oracle over the ordinary state space:
rates, temperature, JVP, VJP, dense Jacobian and transport, one thread and one warp per state.
With the tile kernels in front they evaluate only the few states those leave open, but they
are the whole path of mechanisms outside the tables (a fourth-order reaction, below).
Tolerances as in test_gpu_forward, test_gpu_derivatives and test_gpu_transport."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth
from tests import handmech

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

IDX = {"h2": 0, "gri": 1, "pdep": 7, "large": 4}


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


@pytest.fixture(scope="module")
def load(mech_files, mixed_reversibility_mech):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    made = {}

    def get(name, options):
        if (name, options) not in made:
            path = mixed_reversibility_mech if name == "pdep" else mech_files[0][IDX[name]]
            m = B.Mechanism(path, options)
            for key in ("tile", "jvp_tile", "vjp_tile", "jacobian_tile", "transport_tile"):
                assert m.stat(key) == 0
            made[name, options] = (m, O.Oracle(path))
        return made[name, options]
    return get


def _inputs(orc, idx, n, seed):
    st = synth.config_states(idx, n=n, offset_seed=seed)
    rng = np.random.default_rng(seed)
    rho = orc.density(st.p, st.T, st.Y)
    return [rho, st.T, st.Y, rng.standard_normal(n) * rho * 0.1, rng.standard_normal(n) * 10.0,
            rng.standard_normal((orc.N, n)) * 1e-3]


def _check_rates(m, orc, rho, T, Y):
    w = m.net_production_rates(_t(rho), _t(Y), T=_t(T)).cpu().numpy()
    ow, G = orc.net_production_rates(rho, T, Y, with_gross=True)
    assert np.all(np.abs(w - ow) <= 1e-11 * G + 1e-300)
    e = orc.internal_energy(T, Y)
    w, T1 = m.net_production_rates(_t(rho), _t(Y), e=_t(e))
    oT, _, bad = orc.temperature(e, Y)
    assert bad == 0 and m.nonconverged() == 0
    assert np.max(np.abs(T1.cpu().numpy() - oT) / oT) <= 1e-10
    ow, G = orc.net_production_rates(rho, oT, Y, with_gross=True)
    assert np.all(np.abs(w.cpu().numpy() - ow) <= 1e-11 * G + 1e-300)


def _check_products(m, orc, rho, T, Y, dr, dT, dY):
    a = (rho, T, Y, dr, dT, dY)
    g = m.jvp(*[_t(x) for x in a]).cpu().numpy()
    assert np.all(np.abs(g - orc.jvp(*a)) <= 1e-11 * orc.jvp_scale(*a) + 1e-250)
    wb = np.random.default_rng(7).standard_normal((orc.N, T.size))
    g = np.vstack([x.cpu().numpy().reshape(-1, T.size) for x in m.vjp(_t(rho), _t(T), _t(Y), _t(wb))])
    o = np.vstack([np.asarray(x).reshape(-1, T.size) for x in orc.vjp(rho, T, Y, wb)])
    assert np.all(np.abs(g - o) <= 1e-11 * orc.vjp_scale(rho, T, Y, wb) + 1e-250)


def _check_jacobian(m, orc, rho, T, Y):
    NP = orc.N + 1
    J = m.jacobian(_t(rho), _t(T), _t(Y)).cpu().numpy().reshape(NP, NP, -1)
    Jo = orc.jacobian(rho, T, Y).reshape(NP, NP, -1)
    assert np.all(np.abs(J - Jo) <= 1e-11 * orc.jacobian_gross(rho, T, Y)[:, 1:] + 1e-250)


@pytest.mark.parametrize("name,options,n", [("h2", "tile=0", 1001), ("gri", "tile=0", 1001), ("gri", "tile=0", 1),
                                            ("pdep", "tile=0", 333), ("gri", "tile=0;variant=warp", 333),
                                            ("large", "tile=0;variant=warp", 100)])
def test_rates_and_temperature(load, name, options, n):
    m, orc = load(name, options)
    _check_rates(m, orc, *_inputs(orc, IDX[name], n, 101)[:3])


@pytest.mark.parametrize("name", ["h2", "gri", "pdep"])
def test_products(load, name):
    m, orc = load(name, "tile=0")
    _check_products(m, orc, *_inputs(orc, IDX[name], 97, 102))


@pytest.mark.parametrize("name", ["h2", "gri", "pdep"])
def test_jacobian(load, name):
    m, orc = load(name, "tile=0")
    _check_jacobian(m, orc, *_inputs(orc, IDX[name], 65, 103)[:3])


@pytest.mark.parametrize("name,n", [("h2", 257), ("gri", 129)])
def test_transport(load, name, n):
    m, orc = load(name, "tile=0")
    st = synth.config_states(IDX[name], n=n, offset_seed=104)
    got = [x.cpu().numpy() for x in m.transport(_t(st.T), _t(st.Y))]
    for g, o, tol in zip(got, orc.transport(st.T, st.Y), (1e-12, 1e-12, 2e-11)):
        assert np.max(np.abs(g - o) / np.abs(o)) <= tol


@pytest.mark.parametrize("case", ["order4", "theta"])
def test_mechanisms_outside_the_tables(load, tmp_path, case):
    """Every call of a mechanism that the tile kernels refuse (a fourth-order reaction; an
    activation temperature beyond the coefficients' range)."""
    from paper_2503_24286_gb300 import binding as B
    if case == "order4":
        mech = handmech.abcd_mechanism()
        mech.reactions[0].reactants, mech.reactions[0].products = [(0, 2), (1, 2)], [(2, 2), (3, 2)]
    else:
        mech = handmech.abcd_mechanism(theta=3.0e6)
        mech.reactions.append(handmech.abcd_mechanism(A=1e9, theta=900.0).reactions[0])
    path = handmech.write(mech, str(tmp_path), case + ".txt")
    m, orc = B.Mechanism(path), O.Oracle(path)
    assert m.stat("tile") == 0
    rng = np.random.default_rng(105)
    n = 150
    T = rng.uniform(400.0, 2800.0, n)
    Y = rng.dirichlet(np.full(4, 0.5), n).T.copy()
    rho = orc.density(np.full(n, 101325.0), T, Y)
    _check_rates(m, orc, rho, T, Y)
    _check_products(m, orc, rho, T, Y, 0.1 * rho, rng.standard_normal(n), 1e-3 * rng.standard_normal((4, n)))
    _check_jacobian(m, orc, rho, T, Y)
