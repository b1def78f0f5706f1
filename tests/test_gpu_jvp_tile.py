"""The tile kernels of the JVP, the VJP and the dense Jacobian against the oracle where its dispatch or its number formats can go
wrong: ragged tiles, states outside its tables beside ordinary ones, absent, negative and tiny
mass fractions, zero and huge tangents, and every reaction class.  Tolerance: 1e-11 of each
entry's gross scale (as in test_gpu_derivatives), with that suite's absolute floor of 1e-250."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mechs(mech_files, mixed_reversibility_mech):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    out = {}
    for name, p in (("h2", mech_files[0][0]), ("gri", mech_files[0][1]), ("pdep", mixed_reversibility_mech)):
        out[name] = (B.Mechanism(p), O.Oracle(p))
        assert out[name][0].stat("jvp_tile") == 1
    return out


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def _inputs(orc, idx, n, seed):
    st = synth.config_states(idx, n=n, offset_seed=seed)
    rng = np.random.default_rng(seed)
    rho = orc.density(st.p, st.T, st.Y)
    return [rho, st.T.copy(), st.Y.copy(), rng.standard_normal(n) * rho * 0.1, rng.standard_normal(n) * 10.0,
            rng.standard_normal((orc.N, n)) * 1e-3]


def _check(m, orc, a, skip=()):
    g = m.jvp(*[_t(x) for x in a]).cpu().numpy()
    o, sc = orc.jvp(*a), orc.jvp_scale(*a)
    # states where the oracle's own numbers leave the double range ([M] = 0, 190 K) say nothing
    fine = np.isfinite(o).all(axis=0) & np.isfinite(sc).all(axis=0)
    keep = np.setdiff1d(np.arange(a[0].size)[fine], skip)
    assert keep.size >= 0.9 * a[0].size
    assert np.all(np.isfinite(g[:, keep]))
    assert np.all(np.abs(g - o)[:, keep] <= 1e-11 * sc[:, keep] + 1e-250)
    return g


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
@pytest.mark.parametrize("n", [1, 31, 33, 70])
def test_ragged_tiles(mechs, name, idx, n):
    m, orc = mechs[name]
    _check(m, orc, _inputs(orc, idx, n, 61 + n))


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
def test_open_states_and_compositions(mechs, name, idx):
    m, orc = mechs[name]
    a = _inputs(orc, idx, 128, 62)
    rho, T, Y, dr, dT, dY = a
    rng = np.random.default_rng(63)
    N = orc.N
    T[[3, 40, 41]] = [190.0, 5000.0, 5400.0]
    rho[5] = 1e-22
    Y[:, 32:64] = np.where(rng.random((N, 32)) < 0.6, 0.0, Y[:, 32:64])
    Y[:, 64:96] *= np.where(rng.random((N, 32)) < 0.3, -1e-6, 1.0)
    Y[:, 96:112] = 10.0 ** rng.uniform(-60, -1, (N, 16))
    dT[50], dr[51], dY[:, 52] = 0.0, 0.0, 0.0
    dY[:, 53] *= 1e30
    _check(m, orc, a)


def test_nan_stays_in_its_state(mechs):
    m, orc = mechs["gri"]
    a = _inputs(orc, 1, 64, 64)
    a[2][4, 10] = np.nan
    a[5][4, 11] = np.nan
    a[4][12] = np.inf
    g = _check(m, orc, a, skip=(10, 11, 12))
    assert np.isnan(g[4, 10]) and np.isnan(g[4, 11]) and not np.isfinite(g[:, 12]).all()


def _check_vjp(m, orc, rho, T, Y, wb, skip=()):
    g = np.vstack([x.cpu().numpy().reshape(-1, T.size) for x in m.vjp(_t(rho), _t(T), _t(Y), _t(wb))])
    o = np.vstack([np.asarray(x).reshape(-1, T.size) for x in orc.vjp(rho, T, Y, wb)])
    sc = orc.vjp_scale(rho, T, Y, wb)
    fine = np.isfinite(o).all(axis=0) & np.isfinite(sc).all(axis=0)
    keep = np.setdiff1d(np.arange(T.size)[fine], skip)
    assert keep.size >= 0.9 * T.size
    assert np.all(np.isfinite(g[:, keep]))
    assert np.all(np.abs(g - o)[:, keep] <= 1e-11 * sc[:, keep] + 1e-250)
    return g


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
@pytest.mark.parametrize("n", [1, 31, 33, 70])
def test_vjp_ragged_tiles(mechs, name, idx, n):
    m, orc = mechs[name]
    assert m.stat("vjp_tile") == 1
    rho, T, Y = _inputs(orc, idx, n, 71 + n)[:3]
    _check_vjp(m, orc, rho, T, Y, np.random.default_rng(n).standard_normal((orc.N, n)))


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
def test_vjp_open_states_and_compositions(mechs, name, idx):
    m, orc = mechs[name]
    rho, T, Y = _inputs(orc, idx, 128, 72)[:3]
    rng = np.random.default_rng(73)
    N = orc.N
    wb = rng.standard_normal((N, 128))
    T[[3, 40, 41]] = [190.0, 5000.0, 5400.0]
    rho[5] = 1e-22
    Y[:, 32:64] = np.where(rng.random((N, 32)) < 0.6, 0.0, Y[:, 32:64])
    Y[:, 64:96] *= np.where(rng.random((N, 32)) < 0.3, -1e-6, 1.0)
    Y[:, 96:112] = 10.0 ** rng.uniform(-60, -1, (N, 16))
    wb[:, 50] = 0.0
    wb[:, 51] *= 1e30
    _check_vjp(m, orc, rho, T, Y, wb)


def test_vjp_nan_stays_in_its_state(mechs):
    m, orc = mechs["gri"]
    rho, T, Y = _inputs(orc, 1, 64, 74)[:3]
    wb = np.random.default_rng(75).standard_normal((orc.N, 64))
    Y[4, 10] = np.nan
    wb[4, 11] = np.nan
    T[12] = np.nan
    g = _check_vjp(m, orc, rho, T, Y, wb, skip=(10, 11, 12))
    assert np.isnan(g[1, 10]) and np.isnan(g[1, 11]) and np.isnan(g[1, 12])


def _check_jac(m, orc, rho, T, Y, skip=()):
    NP = orc.N + 1
    J = m.jacobian(_t(rho), _t(T), _t(Y)).cpu().numpy().reshape(NP, NP, -1)
    Jo = orc.jacobian(rho, T, Y).reshape(NP, NP, -1)
    G = orc.jacobian_gross(rho, T, Y)[:, 1:]
    fine = np.isfinite(Jo).all(axis=(0, 1)) & np.isfinite(G).all(axis=(0, 1))
    keep = np.setdiff1d(np.arange(T.size)[fine], skip)
    assert keep.size >= 0.8 * T.size
    assert np.all(np.isfinite(J[..., keep]))
    assert np.all(np.abs(J - Jo)[..., keep] <= 1e-11 * G[..., keep] + 1e-250)
    return J


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
@pytest.mark.parametrize("n", [1, 31, 33])
def test_jacobian_ragged_tiles(mechs, name, idx, n):
    m, orc = mechs[name]
    assert m.stat("jacobian_tile") == 1
    _check_jac(m, orc, *_inputs(orc, idx, n, 81 + n)[:3])


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
def test_jacobian_open_states_and_compositions(mechs, name, idx):
    m, orc = mechs[name]
    rho, T, Y = _inputs(orc, idx, 48, 82)[:3]
    rng = np.random.default_rng(83)
    N = orc.N
    T[[3, 40, 41]] = [190.0, 5000.0, 5400.0]
    rho[5] = 1e-22
    Y[:, 8:20] = np.where(rng.random((N, 12)) < 0.6, 0.0, Y[:, 8:20])
    Y[:, 20:30] *= np.where(rng.random((N, 10)) < 0.3, -1e-6, 1.0)
    Y[:, 30:36] = 10.0 ** rng.uniform(-60, -1, (N, 6))
    _check_jac(m, orc, rho, T, Y)


def test_jacobian_nan_stays_in_its_state(mechs):
    m, orc = mechs["gri"]
    rho, T, Y = _inputs(orc, 1, 40, 84)[:3]
    Y[4, 10] = np.nan
    T[12] = np.nan
    J = _check_jac(m, orc, rho, T, Y, skip=(10, 12))
    # (the inert species takes part in no reaction: its row stays zero)
    assert np.isnan(J[..., 10]).any() and np.isnan(J[0, :, 12]).all()
