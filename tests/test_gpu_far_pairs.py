"""Two particles at any separation, no softening: accelerations and energies keep to
the exact values; the potential of nb_evaluate, summed in pairs of floats, is exact
to 1e-12 or, where the floats' range ends, no number: never a finite wrong one."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("d", [1e-50, 1e-40, 1e-30, 1e-15, 1.0, 1e15, 1e25, 1e29, 1e33, 1e40, 1e60, 1e90])
def test_two_particles(nb, d):
    m = np.array([0.75, 2.5])
    x = np.array([[0.0, 0.0, 0.0], [0.48 * d, -0.6 * d, 0.64 * d]])
    v, z = np.zeros((2, 3)), np.zeros((2, 3))
    sim = nb.Simulation(m, x, v, eps=0.0, keep_state=True)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": z, "j": z, "s": z, "c": z, "t": np.zeros(2),
                         "dt": np.full(2, 2.0 ** -6), "pot": np.zeros(2)})
    sim.predict(0.0, out=False)
    out = sim.evaluate(torch.arange(2, dtype=torch.int32, device="cuda")).cpu().numpy()
    ekin, epot, _, _ = sim.energy(0.0)
    sim.close()
    r = np.linalg.norm(x[1] / d) * d
    for i in range(2):
        want = (x[1 - i] - x[i]) / d * (m[1 - i] / r / r) * (d / r)
        assert np.allclose(out[0:3, i], want, rtol=1e-12, atol=0.0)
        assert np.all(out[3:9, i] == 0.0)
    assert abs(epot + m[0] * m[1] / r) <= 1e-13 * m[0] * m[1] / r
    pot = -m[::-1] / r
    if 1e-37 < d < 1e29:
        assert np.allclose(out[9], pot, rtol=1e-12, atol=0.0)
    else:
        assert np.all(np.isnan(out[9]) | (np.abs(out[9] - pot) <= 1e-12 * np.abs(pot)))


def test_massless_and_padding_at_any_distance(nb):
    """Massless partners (and the padding of a tile) out of the floats' range change
    nothing: three particles about 1e31 from the origin."""
    m = np.array([1.0, 2.0, 0.0])
    x = np.array([[1e31, 0.0, 0.0], [1e31, 3e16, 4e16], [-1e40, 0.0, 0.0]])
    z = np.zeros((3, 3))
    sim = nb.Simulation(m, x, z, eps=0.0, keep_state=True)
    sim.set_state_numpy({"m": m, "x": x, "v": z, "a": z, "j": z, "s": z, "c": z, "t": np.zeros(3),
                         "dt": np.full(3, 2.0 ** -6), "pot": np.zeros(3)})
    sim.predict(0.0, out=False)
    out = sim.evaluate(torch.arange(2, dtype=torch.int32, device="cuda")).cpu().numpy()
    sim.close()
    assert np.allclose(out[9], [-2.0 / 5e16, -1.0 / 5e16], rtol=1e-12, atol=0.0)
