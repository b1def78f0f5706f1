"""Temperatures from energies against extended precision: the integer collapse of the species
polynomials (its scale depends on the number of species) may be no less precise on average
than the same solve with FP64 sums over the species in order."""
import numpy as np
import pytest

from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R_GAS = 8314.462618


def _polynomials(m, dtype):
    """e_k/R = d_0 + d_1 T + ... + d_5 T^5 of both ranges, [2][6][N], in double; then `dtype`."""
    weights = dict(m.elements)
    W = np.array([sum(weights[e] * c for e, c in s.composition.items()) for s in m.species])
    out = []
    for a in (np.array([s.nasa_low for s in m.species]).T, np.array([s.nasa_high for s in m.species]).T):
        out.append(np.stack([a[5], a[0] - 1.0, a[1] / 2, a[2] / 3, a[3] / 4, a[4] / 5]) / W)
    return np.stack(out).astype(dtype)


def _solve(d, t_mid, e, Y, T, dtype):
    """Newton from T, the sums over the species in order, in `dtype`."""
    B = np.zeros((2, 6, T.size), dtype)
    for k in range(Y.shape[0]):
        B += d[:, :, k, None] * Y[k].astype(dtype)
    T, eR = T.astype(dtype), e.astype(dtype) / dtype(R_GAS)
    for _ in range(8):
        b = np.where(T.astype(np.float64) < t_mid, B[0], B[1])
        f = b[0] + T * (b[1] + T * (b[2] + T * (b[3] + T * (b[4] + T * b[5]))))
        cv = b[1] + T * (2 * b[2] + T * (3 * b[3] + T * (4 * b[4] + T * 5 * b[5])))
        T = T - (f - eR) / cv
    return T


@pytest.mark.parametrize("idx,options", [(0, None), (1, None), (1, "newton=fp64"), (4, "variant=warp")])
def test_temperature_no_less_precise_than_fp64_sums(mech_files, idx, options):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    obj, lib = mech_files[1][idx], B.Mechanism(mech_files[0][idx], options)
    st = synth.config_states(idx, n=1000, offset_seed=77)
    keep = np.abs(st.T - obj.species[0].t_mid) > 1.0
    T0, Y = st.T[keep], np.ascontiguousarray(st.Y[:, keep])
    d = _polynomials(obj, np.longdouble)
    t_mid = obj.species[0].t_mid
    b = np.where(T0 < t_mid, *np.einsum("rqk,kn->rqn", d, Y.astype(np.longdouble)))
    e = (sum(b[q] * T0.astype(np.longdouble) ** q for q in range(6)) * np.longdouble(R_GAS)).astype(np.float64)
    exact = _solve(d, t_mid, e, Y, T0, np.longdouble)
    fp64 = _solve(_polynomials(obj, np.float64), t_mid, e, Y, T0, np.float64)
    err = lambda T: np.abs(T.astype(np.longdouble) / exact - 1).astype(np.float64)  # noqa: E731
    t = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda:0")  # noqa: E731
    rho = np.full_like(T0, 0.3)
    _, T1 = lib.net_production_rates(t(rho), t(Y), e=t(e))
    T2 = lib.temperature(t(e), t(Y))
    for T in (T1, T2):
        assert err(T.cpu().numpy()).mean() <= err(fp64).mean()
