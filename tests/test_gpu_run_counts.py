"""nb_run reports the steps and interactions of a run that came to its end, also when
the context carries an error of an earlier call, which it then returns."""
import ctypes

import pytest

from paper_1812_00367_gb300 import ic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00367_gb300 import build as nbbuild
    nbbuild.build()
    from paper_1812_00367_gb300 import nb as nbmod
    nbmod.load()
    return nbmod


@pytest.mark.parametrize("max_steps", [-1, 1])
def test_counts_with_an_earlier_error(nb, max_steps):
    m, x, v = ic.plummer(200, seed=3)
    sim = nb.Simulation(m, x, v, eps=1e-2)
    act = torch.tensor([200], dtype=torch.int32, device="cuda")   # outside the cluster: flagged
    out = torch.zeros((10, 1), dtype=torch.float64, device="cuda")
    nb.nb_evaluate(sim.ctx, 0, act, 1, out)
    steps, inter = ctypes.c_int64(-1), ctypes.c_double(-1.0)
    rc = nb.load().nb_run(sim.ctx, ctypes.c_double(0.0), ctypes.c_int64(max_steps), ctypes.byref(steps),
                          ctypes.byref(inter))                    # no block time up to t = 0
    assert rc == 1 and steps.value == 0 and inter.value == 0.0
    sim.close()
