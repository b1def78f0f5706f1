"""The library called from a host thread that has made no CUDA call of its own."""
import threading

import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_24286_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_first_cuda_work_of_a_thread(mech_files):
    """As in a backward pass, whose thread may launch nothing before the library does."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_24286_gb300 import binding as B
    from paper_2503_24286_gb300 import build as BLD
    BLD.build()
    m, orc = B.Mechanism(mech_files[0][0]), O.Oracle(mech_files[0][0])
    m.prepare("jvp")
    st = synth.config_states(0, n=64, offset_seed=123)
    rng = np.random.default_rng(123)
    a = [torch.tensor(x, dtype=torch.float64, device="cuda:0")
         for x in (orc.density(st.p, st.T, st.Y), st.T, st.Y, rng.standard_normal(64), rng.standard_normal(64),
                   rng.standard_normal((orc.N, 64)))]
    ref = m.jvp(*a)
    out, failed = torch.empty_like(ref), []

    def work():
        try:
            m.jvp(*a, out=out)
        except Exception as e:  # noqa: BLE001
            failed.append(e)
    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not failed and torch.equal(out, ref)
