"""The 4th-order scheme has no snap: nb_evaluate's snap rows are zero whatever the
state, also where a position or a velocity that is not finite takes the other sums
(one-sided and each pair once)."""
import numpy as np
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


@pytest.mark.parametrize("n", [300, 8200])
def test_snap_rows_stay_zero(nb, n):
    m, x, v = ic.plummer(n, seed=2)
    z = np.zeros((n, 3))
    x[n // 2, 1] = np.nan
    sim = nb.Simulation(m, x, v, eps=1e-3, order=4, keep_state=True)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": z, "j": z, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    sim.predict(0.0, out=False)
    out = sim.evaluate(torch.arange(n, dtype=torch.int32, device="cuda")).cpu().numpy()
    sim.close()
    assert np.all(out[6:9] == 0.0)
    assert np.isnan(out[0:6]).all() and np.isnan(out[9]).all()
