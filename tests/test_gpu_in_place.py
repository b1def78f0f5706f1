"""Outputs written over inputs: a call gives what it gives with separate arrays.  The tile kernels
read some inputs again after outputs have been written (and leave states open for an FP64
kernel that reads them then), so such calls take the FP64 kernels, which read a state before
they write it; temperatures over energies are the one form the tile kernel takes itself.
Tolerance against the separate arrays' results: 1e-11 of the gross scale (as between either
kernel and the oracle), bits where the same kernel runs."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    return B


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def _inputs(orc, idx, n, seed):
    st = synth.config_states(idx, n=n, offset_seed=seed)
    T = st.T.copy()
    T[::7] = 170.0                                   # open states among the others
    rho = orc.density(st.p, T, st.Y)
    rng = np.random.default_rng(seed)
    return rho, T, st.Y, rng.standard_normal(n), rng.standard_normal(n), rng.standard_normal((orc.N, n))


def test_rates_over_fractions_and_tangents_over_tangents(lib, mech_files):
    m, orc = lib.Mechanism(mech_files[0][1]), O.Oracle(mech_files[0][1])
    a = _inputs(orc, 1, 100, 121)
    rho, T, Y, dr, dT, dY = (_t(x) for x in a)
    open_ = np.arange(100) % 7 == 0
    _, G = orc.net_production_rates(*a[:3], with_gross=True)
    w, y = m.net_production_rates(rho, Y, T=T), Y.clone()
    m.net_production_rates(rho, y, T=T, out=y)
    g, v = m.jvp(rho, T, Y, dr, dT, dY), dY.clone()
    m.jvp(rho, T, Y, dr, dT, v, out=v)
    for x, ref, scale in ((y, w, 1e-11 * G), (v, g, 1e-11 * orc.jvp_scale(*a) + 1e-250)):
        x, ref = x.cpu().numpy(), ref.cpu().numpy()
        assert np.array_equal(x[:, open_], ref[:, open_])
        assert np.all(np.abs(x - ref)[:, ~open_] <= scale[:, ~open_] + 1e-300)


@pytest.mark.parametrize("idx,options", [(1, None), (4, "variant=warp")])
@pytest.mark.parametrize("n", [1, 33, 1000])
def test_temperatures_over_energies(lib, mech_files, idx, options, n):
    m, orc = lib.Mechanism(mech_files[0][idx], options), O.Oracle(mech_files[0][idx])
    st = synth.config_states(idx, n=n, offset_seed=122)
    rho, Y, e = _t(orc.density(st.p, st.T, st.Y)), _t(st.Y), _t(orc.internal_energy(st.T, st.Y))
    w, T = m.net_production_rates(rho, Y, e=e)
    a = e.clone()
    w2, T2 = m.net_production_rates(rho, Y, e=a, T_out=a)
    assert T2.data_ptr() == a.data_ptr() and torch.equal(T2, T) and torch.equal(w2, w)
