"""Transport of compositions whose mole fractions have mixed signs and a large sum |X|, each
below 1.9 (undershoots that nearly cancel): the tile kernel's integer sums of Wilke's rule
hold while sum |X| < 2 and must leave other states to the FP64 kernel.

Thirty species, fifteen of weights 1..15 (negative fractions) and fifteen of 201..215
(positive): Wilke's coefficients 1/sqrt(8 (1 + W_k/W_j)) are then largest where X_j > 0, and
their sum passes 2^63 in the kernel's scale from sum |X| of about 30.

Tolerance of mu: 1e-12 as in test_gpu_transport, times the condition of its sums:
sum_k |X_k mu_k/d_k| (sum_j |Phi_kj X_j|/|d_k|), d_k = sum_j Phi_kj X_j."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth
from tests import handmech

torch = pytest.importorskip("torch")
HALF = 15


def _mechanism():
    sp = [handmech.const_cp_species("%s%d" % (e, k), {"L": k, **({"B": 1} if e == "B" else {})}, 2.5 + 0.1 * k, 0.0, 10.0)
          for e in ("L", "B") for k in range(1, HALF + 1)]
    r = synth.Reaction("arrhenius", [(0, 2)], [(1, 1)], 1e10, 0.0, 1000.0)
    m = synth.Mechanism("light_heavy", [("L", 1.0), ("B", 200.0)], sp, [r])
    N = len(sp)
    fit = lambda *shape: np.concatenate([np.full(shape + (1,), 1.0), np.zeros(shape + (4,))], axis=-1)  # noqa: E731
    m.transport = synth.Transport(1e-3 * fit(N), 1e-3 * fit(N), 1e-5 * fit(N, N))
    return m


def _states(W):
    """sum X = 1, sum |X| = s from 2.1 to 48 on every other state; 1 on the others."""
    N, n = 2 * HALF, 64
    rng = np.random.default_rng(58)
    X = rng.uniform(0.9, 1.1, (N, n))
    heavy = np.arange(N) >= HALF
    for p in range(n):
        s = np.linspace(2.1, 48.0, n)[p] if p % 2 == 0 else 1.0
        X[~heavy, p] *= -(s - 1.0) / 2.0 / X[~heavy, p].sum()
        X[heavy, p] *= (s + 1.0) / 2.0 / X[heavy, p].sum()
    T = rng.uniform(300.0, 2800.0, n)
    return T, X * W[:, None] / (X * W[:, None]).sum(axis=0)


def test_the_states_pass_the_integer_range(tmp_path):
    m = _mechanism()
    synth.write_mechanism(m, str(tmp_path / "m.txt"))
    W = np.asarray(O.Oracle(str(tmp_path / "m.txt")).W)
    _, Y = _states(W)
    X = Y / W[:, None] / (Y / W[:, None]).sum(axis=0)
    assert np.abs(X).max() < 1.9 and np.abs(X.sum(axis=0) - 1.0).max() < 1e-12
    c = 1.0 / np.sqrt(8.0 * (1.0 + W[:, None] / W[None, :]))
    # scale of the coefficients: the largest in [2^56, 2^57); X by 2^61; the sums in units of 2^57
    top = np.abs(c * 2.0 ** (56 - math.floor(math.log2(c.max()))) @ X).max(axis=0) * 2.0 ** 4
    assert (top >= 2.0 ** 63).sum() >= 8


@pytest.mark.gpu
def test_viscosity_of_mixed_signs(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    path = str(tmp_path / "m.txt")
    synth.write_mechanism(_mechanism(), path)
    m, orc = B.Mechanism(path), O.Oracle(path)
    assert m.stat("transport_tile") == 1
    W = np.asarray(orc.W)
    T, Y = _states(W)
    X = Y / W[:, None] / (Y / W[:, None]).sum(axis=0)
    t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")  # noqa: E731
    mu = m.transport(t(T), t(Y))[0].cpu().numpy()
    omu = orc.transport(T, Y)[0]
    for p in range(T.size):
        Phi = orc.wilke_phi(T[p])
        mk = np.array([orc.species_transport(k, T[p])[0] for k in range(orc.N)])
        d = Phi @ X[:, p]
        cond = (np.abs(Phi) @ np.abs(X[:, p])) / np.abs(d)
        assert abs(mu[p] - omu[p]) <= 1e-12 * (np.abs(X[:, p] * mk / d) * cond).sum()
