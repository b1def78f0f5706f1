"""The tile kernel of the net production rates against the oracle where its dispatch or its
number formats can go wrong: states outside its tables' range (left to the FP64 kernel)
beside states inside it, every ragged tile size, absent and slightly negative mass
fractions, tiny ones, NaN, and duplicates, SRI, PLOG and irreversible reactions.
Tolerance of every rate: 1e-11 of its gross scale (as in test_gpu_forward)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.fixture(scope="module")
def mechs(mech_files, mixed_reversibility_mech):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    paths = {"h2": mech_files[0][0], "gri": mech_files[0][1], "pdep": mixed_reversibility_mech}
    out = {k: (B.Mechanism(p), O.Oracle(p)) for k, p in paths.items()}
    for m, _ in out.values():
        assert m.stat("tile") == 1
    return out


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def _states(orc, idx, n, seed):
    st = synth.config_states(idx, n=n, offset_seed=seed)
    return orc.density(st.p, st.T, st.Y), st.T.copy(), st.Y.copy()


def _check(m, orc, rho, T, Y, skip=()):
    w = m.net_production_rates(_t(rho), _t(Y), T=_t(T)).cpu().numpy()
    ow, G = orc.net_production_rates(rho, T, Y, with_gross=True)
    keep = np.setdiff1d(np.arange(T.size), skip)
    assert np.all(np.isfinite(w[:, keep]))
    assert np.all(np.abs(w - ow)[:, keep] <= TOL * G[:, keep] + 1e-300)
    return w


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 95, 1025])
def test_ragged_tiles(mechs, name, idx, n):
    m, orc = mechs[name]
    _check(m, orc, *_states(orc, idx, n, 31 + n))


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
def test_open_states_go_to_the_fp64_kernel(mechs, name, idx):
    """Temperatures at and beyond both ends of the table's range, extreme densities and
    subnormal mass fractions, one state of each tile or a whole tile.  Below 140 K the
    synthetic rates leave the double range (the oracle's and the FP64 kernel's alike):
    such states only must not disturb the others."""
    m, orc = mechs[name]
    rho, T, Y = _states(orc, idx, 200, 33)
    lo = m.stat("tile_t_lo")
    T[[3, 40, 41, 70, 71, 72]] = [150.0, lo, np.nextafter(lo, 1e4), 5000.0, np.nextafter(5000.0, 0.0), 5600.0]
    T[96:128] = np.linspace(0.5 * lo, lo, 32)
    rho[[5, 130]] = [1e-25, 1e8]
    Y[0, 140] = 5e-310
    _check(m, orc, rho, T, Y, skip=np.where(T < 140.0)[0])


@pytest.mark.parametrize("name,idx", [("h2", 0), ("gri", 1), ("pdep", 7)])
def test_absent_negative_and_tiny_mass_fractions(mechs, name, idx):
    m, orc = mechs[name]
    rho, T, Y = _states(orc, idx, 160, 35)
    rng = np.random.default_rng(36)
    N = orc.N
    Y[:, 0:32] = np.where(rng.random((N, 32)) < 0.6, 0.0, Y[:, 0:32])
    Y[:, 32:64] *= np.where(rng.random((N, 32)) < 0.3, -1e-6, 1.0)
    Y[:, 64:96] = 10.0 ** rng.uniform(-290, -1, (N, 32))
    Y[:, 96] = 0.0
    Y[N // 2, 96] = 1.0
    w = _check(m, orc, rho, T, Y)
    ow, G = orc.net_production_rates(rho, T, Y, with_gross=True)
    assert np.all(w[G == 0.0] == 0.0)          # no reaction of these species runs: exactly zero


def test_split_tiles_give_the_same_bits(mech_files):
    """160 species: few tiles run one cluster of blocks per tile (a block per chunk of reactions),
    many run one block per tile; both give the same bits, open states included."""
    from paper_2503_24286_gb300 import binding as B
    m, orc = B.Mechanism(mech_files[0][4], "variant=warp"), O.Oracle(mech_files[0][4])
    assert m.stat("tile_chunks") > 1
    n = 32 * 200
    rho, T, Y = _states(orc, 4, n, 41)
    T[[7, 40]] = [280.0, 4990.0]
    assert m.stat("tile_t_lo") > 280.0
    e = orc.internal_energy(T, Y)
    full, Tf = m.net_production_rates(_t(rho), _t(Y), e=_t(e))
    for a, b in ((0, 1), (0, 33), (64, 640), (n - 95, n)):
        w, Ts = m.net_production_rates(_t(rho[a:b]), _t(Y[:, a:b]), e=_t(e[a:b]))
        assert torch.equal(w, full[:, a:b]) and torch.equal(Ts, Tf[a:b])
    m.nonconverged()
    _check(m, orc, rho[:100], T[:100], Y[:, :100])


def test_nan_stays_in_its_state(mechs):
    m, orc = mechs["gri"]
    rho, T, Y = _states(orc, 1, 100, 37)
    Y[4, 50] = np.nan
    T[60] = np.nan
    rho[61] = np.inf
    w = _check(m, orc, rho, T, Y, skip=(50, 60, 61))
    assert np.isnan(w[4, 50]) and np.isnan(w[:, 60]).any() and not np.isfinite(w[:, 61]).all()


def test_energy_input_with_an_unreachable_energy(mechs):
    """A state whose Newton iteration ends at the 5000 K clamp is counted and evaluated there;
    the others are solved as before."""
    m, orc = mechs["gri"]
    rho, T, Y = _states(orc, 1, 70, 39)
    e = orc.internal_energy(T, Y)
    e[33] = 1e12
    w, Tg = m.net_production_rates(_t(rho), _t(Y), e=_t(e))
    assert m.nonconverged() == 1
    w, Tg = w.cpu().numpy(), Tg.cpu().numpy()
    assert Tg[33] == 5000.0
    ok = np.arange(70) != 33
    assert np.max(np.abs(Tg - T)[ok] / T[ok]) <= 1e-12
    ow, G = orc.net_production_rates(rho, Tg, Y, with_gross=True)
    assert np.all(np.abs(w - ow) <= TOL * G + 1e-300)
