"""The transport tile kernel against the oracle where its dispatch or its number formats can go
wrong: ragged tiles, temperatures at and beyond the ends of its range beside ordinary ones,
nearly pure and slightly negative compositions, and each output alone.  Tolerances as in
test_gpu_transport (mu, kappa 1e-12, D 2e-11; relative)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mechs(mech_files):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    out = {}
    for i in (0, 1, 4):
        m = B.Mechanism(mech_files[0][i])
        assert m.stat("transport_tile") == 1
        out[i] = (m, O.Oracle(mech_files[0][i]))
    return out


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def _check(m, orc, T, Y):
    got = [x.cpu().numpy() for x in m.transport(_t(T), _t(Y))]
    for g, o, tol in zip(got, orc.transport(T, Y), (1e-12, 1e-12, 2e-11)):
        assert np.all(np.isfinite(g))
        assert np.max(np.abs(g - o) / np.abs(o)) <= tol
    return got


@pytest.mark.parametrize("idx,n", [(0, 1), (0, 33), (1, 31), (1, 64), (1, 97), (4, 35)])
def test_ragged_tiles(mechs, idx, n):
    m, orc = mechs[idx]
    st = synth.config_states(idx, n=n, offset_seed=51)
    _check(m, orc, st.T, st.Y)


@pytest.mark.parametrize("idx", [0, 1])
def test_open_states_and_single_outputs(mechs, idx):
    m, orc = mechs[idx]
    st = synth.config_states(idx, n=130, offset_seed=52)
    T, Y = st.T.copy(), st.Y.copy()
    T[[3, 40, 41, 42, 70]] = [199.0, 200.0, np.nextafter(200.0, 300.0), 5000.0, np.nextafter(5000.0, 0.0)]
    T[96:128] = np.linspace(150.0, 200.0, 32)
    mu, ka, D = _check(m, orc, T, Y)
    one = m.transport(_t(T), _t(Y), kappa=False, diffusivities=False)[0]
    two = m.transport(_t(T), _t(Y), mu=False, diffusivities=False)[1]
    three = m.transport(_t(T), _t(Y), mu=False, kappa=False)[2]
    assert np.array_equal(one.cpu().numpy(), mu) and np.array_equal(two.cpu().numpy(), ka)
    assert np.array_equal(three.cpu().numpy(), D)


@pytest.mark.parametrize("idx", [0, 1])
def test_nearly_pure_and_slightly_negative_compositions(mechs, idx):
    m, orc = mechs[idx]
    st = synth.config_states(idx, n=64, offset_seed=53)
    Y = st.Y.copy()
    N = orc.N
    rng = np.random.default_rng(54)
    for p in range(32):                                    # one species, traces of the others
        Y[:, p] = 10.0 ** rng.uniform(-14, -3, N)
        Y[p % N, p] = 0.0
        Y[p % N, p] = 1.0 - Y[:, p].sum()
    Y[:, 32:64] *= np.where(rng.random((N, 32)) < 0.1, -1e-9, 1.0)
    T = st.T
    got = [x.cpu().numpy() for x in m.transport(_t(T), _t(Y))]
    exp = orc.transport(T, Y)
    assert np.max(np.abs(got[0] - exp[0]) / exp[0]) <= 1e-12 and np.max(np.abs(got[1] - exp[1]) / exp[1]) <= 1e-12
    # (1 - Y_k) of the dominant species carries the rounding of Y itself on both sides
    scale = np.abs(exp[2]) * 2e-11 * np.maximum(1.0, 1e-5 / np.maximum(np.abs(1.0 - Y), 1e-300))
    assert np.all(np.abs(got[2] - exp[2]) <= scale)


def test_nan_stays_in_its_state(mechs):
    m, orc = mechs[1]
    st = synth.config_states(1, n=40, offset_seed=55)
    T, Y = st.T.copy(), st.Y.copy()
    T[5] = np.nan
    Y[3, 6] = np.nan
    mu, ka, D = (x.cpu().numpy() for x in m.transport(_t(T), _t(Y)))
    assert np.isnan(mu[[5, 6]]).all() and np.isnan(D[:, 5]).all()
    keep = np.setdiff1d(np.arange(40), [5, 6])
    for g, o, tol in zip((mu, ka, D), orc.transport(T[keep], np.ascontiguousarray(Y[:, keep])), (1e-12, 1e-12, 2e-11)):
        assert np.max(np.abs(g[..., keep] - o) / np.abs(o)) <= tol
