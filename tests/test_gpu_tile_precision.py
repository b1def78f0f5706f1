"""The tile kernels may be no less precise than the FP64 kernels (tile=0): errors against the
oracle's extended precision, over the workloads' states (the coldest ones, whose exponents
are largest, among them) and for species with more than 128 reactions, whose sums are
rounded in two steps.  Both the mean over the states of each state's relative error (in the
norm of its outputs) and the error in the norm of all outputs are compared; the kernels differ
by a factor of two to ten, far more than the statistic's scatter."""
import copy

import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def _handles(path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    return B.Mechanism(path), B.Mechanism(path, "tile=0"), O.Oracle(path)


def _errors(got, ref):
    d = (got.astype(np.longdouble) - ref.astype(np.longdouble)).reshape(-1, got.shape[-1])
    r = ref.astype(np.longdouble).reshape(-1, got.shape[-1])
    state = np.sqrt((d ** 2).sum(axis=0) / (r ** 2).sum(axis=0))
    return float(state.mean()), float(np.sqrt((d ** 2).sum() / (r ** 2).sum()))


def _rates(path, idx, seed):
    tile, fp64, orc = _handles(path)
    assert tile.stat("tile") == 1 and fp64.stat("tile") == 0
    st = synth.config_states(idx, n=2000, offset_seed=seed)
    T = st.T.copy()
    T[::4] = 300.0 + (T[::4] - 300.0) * 0.1
    rho = orc.density(st.p, T, st.Y)
    ref = orc.net_production_rates_ld(rho, T, st.Y)
    a, b = (_errors(m.net_production_rates(_t(rho), _t(st.Y), T=_t(T)).cpu().numpy(), ref) for m in (tile, fp64))
    assert a[0] <= b[0] and a[1] <= b[1], (a, b)


@pytest.mark.parametrize("idx", [0, 1])
def test_rates(mech_files, idx):
    _rates(mech_files[0][idx], idx, 111)


def test_rates_of_long_lists(mech_files, tmp_path):
    m = copy.deepcopy(mech_files[1][0])
    third = [r for r in m.reactions if r.kind == "threebody"]
    rng = np.random.default_rng(112)
    for r in third:
        r.duplicate = True
        for _ in range(70):
            q = copy.deepcopy(r)
            q.A *= float(rng.uniform(0.2, 5.0))
            m.reactions.append(q)
    path = str(tmp_path / "long.txt")
    synth.write_mechanism(m, path)
    _rates(path, 0, 113)


@pytest.mark.parametrize("idx", [0, 1])
def test_transport(mech_files, idx):
    tile, fp64, orc = _handles(mech_files[0][idx])
    assert tile.stat("transport_tile") == 1 and fp64.stat("transport_tile") == 0
    st = synth.config_states(idx, n=100, offset_seed=114)
    ref = orc.transport(st.T, st.Y, long_double=True)
    out = [[x.cpu().numpy() for x in m.transport(_t(st.T), _t(st.Y))] for m in (tile, fp64)]
    for k in range(3):
        a, b = _errors(out[0][k], ref[k]), _errors(out[1][k], ref[k])
        assert a[0] <= b[0] and a[1] <= b[1], (k, a, b)
