"""The tile kernel of the net production rates where [M] of a reaction is not positive:
efficiencies of 0 whose species make up the state (a sum that cancels to rounding noise of
either sign), undershoots and negative densities.  A third body's [M] is a factor of its rate;
a state with a falloff reaction of [M] <= 0 belongs to the FP64 kernel.

Tolerance: 1e-11 of the gross scale as in test_gpu_forward, plus the rounding of [M] itself.
The kernels form [M]/rho as a sum of N + n_eff terms of at most sum_k max(eps, 1) |Y_k|/W_k,
so its error is below 2 (N + 8) 2^-53 of that, and the rate's error below the same fraction
of the gross scale G' with efficiencies max(eps, 1) at (|rho|, T, |Y|)."""
import copy
import os

import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def _mechanism(idx, falloff, zero):
    """Configuration idx with efficiencies of 0 for the species of `zero` in every reaction
    with a third body; falloff reactions become three-body reactions unless kept."""
    m = copy.deepcopy(synth.config_mechanism(idx))
    for r in m.reactions:
        if r.kind == "arrhenius":
            continue
        if r.kind == "falloff" and not falloff:
            r.kind, r.low, r.troe = "threebody", None, None
        r.efficiencies.update({k: 0.0 for k in zero})
    return m


def _load(m, directory, name):
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    full = copy.deepcopy(m)
    for r in full.reactions:
        r.efficiencies = {k: max(e, 1.0) for k, e in r.efficiencies.items()}
    paths = [os.path.join(directory, name + s) for s in (".txt", "_full.txt")]
    for x, p in zip((m, full), paths):
        synth.write_mechanism(x, p)
    return B.Mechanism(paths[0]), O.Oracle(paths[0]), O.Oracle(paths[1])


def _states(orc, idx, n, zero, seed):
    """Ordinary states with every fourth one special: only the species of efficiency 0; the same
    with traces of the others; clearly negative sums; negative densities."""
    st = synth.config_states(idx, n=n, offset_seed=seed)
    rho, T, Y = orc.density(st.p, st.T, st.Y), st.T.copy(), st.Y.copy()
    others = np.setdiff1d(np.arange(orc.N), zero)
    for p in range(0, n, 4):
        kind = (p // 4) % 4
        if kind < 3:
            y = Y[others, p].copy()
            Y[others, p] = (0.0, 1e-20, -0.2)[kind] * y
            Y[zero, p] *= (1.0 - Y[others, p].sum()) / Y[zero, p].sum()
        else:
            rho[p] = -rho[p]
    return rho, T, Y


def _check(orc, full, rho, T, Y, w):
    ow, G = orc.net_production_rates(rho, T, Y, with_gross=True)
    _, Gf = full.net_production_rates(np.abs(rho), T, np.abs(Y), with_gross=True)
    assert np.all(np.isfinite(w))
    assert np.all(np.abs(w - ow) <= 1e-11 * G + 2 * (orc.N + 8) * 2.0 ** -53 * Gf + 1e-300)


@pytest.mark.parametrize("idx", [0, 1])
def test_third_body_sums_of_either_sign(tmp_path, idx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N = synth.config_mechanism(idx).n_species
    zero = np.arange(0, N, 2)
    m, orc, full = _load(_mechanism(idx, False, zero), str(tmp_path), "third%d" % idx)
    assert m.stat("tile") == 1
    rho, T, Y = _states(orc, idx, 32 * 7, zero, 91)
    w = m.net_production_rates(_t(rho), _t(Y), T=_t(T)).cpu().numpy()
    _check(orc, full, rho, T, Y, w)
    for p in (0, 4, 8, 12):                       # alone, as beside others
        a = m.net_production_rates(_t(rho[p:p + 1]), _t(Y[:, p:p + 1]), T=_t(T[p:p + 1])).cpu().numpy()
        assert np.array_equal(a[:, 0], w[:, p])


def test_one_block_and_cluster_form_agree_on_open_states(mech_files):
    """160 species: states whose [M] is negative (densities, undershoots) go to the FP64 kernel in
    both forms of the tile kernel, bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    m, orc = B.Mechanism(mech_files[0][4], "variant=warp"), O.Oracle(mech_files[0][4])
    assert m.stat("tile_chunks") > 1
    n = 32 * 200
    rho, T, Y = _states(orc, 4, n, np.arange(0, orc.N, 2), 92)
    full = m.net_production_rates(_t(rho), _t(Y), T=_t(T))
    for a, b in ((0, 1), (8, 9), (12, 13), (0, 33), (64, 640), (n - 95, n)):
        w = m.net_production_rates(_t(rho[a:b]), _t(Y[:, a:b]), T=_t(T[a:b]))
        assert torch.equal(w.view(torch.int64), full[:, a:b].contiguous().view(torch.int64))


def test_falloff_states_without_third_bodies_are_the_fp64_kernel_s(tmp_path):
    """The same 53-species mechanism with one four-factor reaction of negligible rate does not
    fit the tile kernel's tables: its FP64 kernel gives the open states' values."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m0 = synth.config_mechanism(1)
    zero = np.arange(0, m0.n_species, 2)
    a = _mechanism(1, True, zero)
    key = lambda k: sorted(m0.species[k].composition.items())  # noqa: E731
    one, two = next((i, j) for i in range(m0.n_species) for j in range(m0.n_species)
                    if key(j) == [(e, 2 * c) for e, c in key(i)])
    b = copy.deepcopy(a)
    b.reactions.append(synth.Reaction("arrhenius", [(one, 4)], [(two, 2)], 1e-250, 0.0, 0.0, reversible=False))
    ma, orc, _ = _load(a, str(tmp_path), "fall1")
    mb, _, _ = _load(b, str(tmp_path), "fall1_fp64")
    assert ma.stat("tile") == 1 and mb.stat("tile") == 0
    rho, T, Y = _states(orc, 1, 32 * 3, zero, 93)
    wa, wb = (m.net_production_rates(_t(rho), _t(Y), T=_t(T)).cpu().numpy() for m in (ma, mb))
    special = np.arange(0, T.size, 4)
    M = np.array([sum((dict(r.efficiencies).get(k, 1.0)) * Y[k] / orc.W[k] for k in range(orc.N)) * rho
                  for r in a.reactions if r.kind == "falloff"])
    low = (M < 0).any(axis=0)
    assert set(np.where(low)[0]) <= set(special) and low[special].sum() >= special.size // 4
    # (codes of the same expressions: equal up to the contraction of products and sums)
    same = (wa == wb) | (np.isnan(wa) & np.isnan(wb)) | (np.abs(wa - wb) <= 1e-11 * np.nanmax(np.abs(wb), axis=0))
    assert same[:, low].all()
