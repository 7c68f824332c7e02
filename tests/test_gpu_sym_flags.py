"""Each pair once: a velocity or an acceleration that leaves the doubles' range in the
prediction, on a particle whose position does not.  As one by one: the velocity takes
every particle's jerk and snap, the acceleration every snap; the other sums stay
finite (the particle is massless, so its own distance from the others, out of the
potential's range, is its own potential's loss only).  Several bands of rows."""
import numpy as np
import pytest

from paper_1812_00367_gb300 import ic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BIG, H = 1.7e308, 2.0 ** -4


@pytest.fixture(scope="module")
def nb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00367_gb300 import build as nbbuild
    nbbuild.build()
    from paper_1812_00367_gb300 import nb as nbmod
    nbmod.load()
    return nbmod


@pytest.mark.parametrize("n", [8192, 30011])
@pytest.mark.parametrize("where", ["first", "middle", "last"])
@pytest.mark.parametrize("field", ["v", "a"])
def test_flags_reach_every_particle(nb, n, where, field):
    m, x, v = ic.plummer(n, seed=n)
    p = {"first": 0, "middle": n // 2, "last": n - 1}[where]
    m[p] = 0.0
    a, j, z = np.zeros((n, 3)), np.zeros((n, 3)), np.zeros((n, 3))
    (v if field == "v" else a)[p, 0] = BIG       # v + H a, or a + H j, overflows
    (a if field == "v" else j)[p, 0] = BIG
    sim = nb.Simulation(m, x, v, eps=1e-3, keep_state=True)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": a, "j": j, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    pred = sim.predict(H).cpu().numpy()
    assert np.isfinite(pred[0:3]).all() and not np.isfinite(pred[3 if field == "v" else 6, p])
    got = sim.evaluate(torch.arange(n, dtype=torch.int32, device="cuda")).cpu().numpy()
    one = sim.evaluate(torch.arange(n - 1, -1, -1, dtype=torch.int32, device="cuda")).cpu().numpy()[:, ::-1]
    sim.close()
    others = np.arange(n) != p
    for out in (got, one):
        assert np.isfinite(out[0:3]).all() and np.isfinite(out[9, others]).all()
        assert np.isnan(out[3:6]).all() if field == "v" else np.isfinite(out[3:6]).all()
        assert np.isnan(out[6:9]).all()
