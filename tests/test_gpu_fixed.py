"""GPU parity of the FP64 evaluation's block fixed-point pair terms where they
could go wrong: pairs inside the softening length, cold systems, planar systems,
other units, tile edges; and what a non-finite velocity or acceleration does.
Tolerance: the FP64 path's 1e-12 per particle (norm of a vector)."""
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


def _evaluate(nb, m, x, v, a, eps, order=6, active=None):
    n = len(m)
    sim = nb.Simulation(m, x, v, eps=eps, keep_state=True, order=order)
    z = np.zeros((n, 3))
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": a, "j": z, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    sim.predict(0.0, out=False)
    act = np.arange(n, dtype=np.int32) if active is None else active
    out = sim.evaluate(torch.as_tensor(act, device="cuda")).cpu().numpy()
    sim.close()
    return out


def _check(out, ref, order):
    acc, jrk, snp, pot = ref
    rows = [(out[0:3].T, acc), (out[3:6].T, jrk)] + ([(out[6:9].T, snp)] if order == 6 else [])
    for got, want in rows:
        den = np.linalg.norm(want, axis=1)
        err = np.linalg.norm(got - want, axis=1)
        assert (err <= 1e-12 * np.where(den > 0, den, 1.0)).all(), float((err / np.maximum(den, 1e-300)).max())
    assert (np.abs(out[9] - pot) <= 1e-12 * np.abs(pot)).all()


@pytest.mark.parametrize("order", [6, 4])
@pytest.mark.parametrize("case", ["softened", "cold", "unsoftened", "units", "uneven masses"])
@pytest.mark.parametrize("n", [65, 700])
def test_fixed_point_parity(nb, oracle, n, case, order):
    m, x, v = ic.plummer(n, seed=n + order)
    rng = np.random.default_rng(n)
    eps, a = 1e-4, rng.normal(size=(n, 3))
    if case == "softened":      # most pairs lie inside the softening length
        eps = 1.0
    elif case == "cold":
        v = np.zeros((n, 3))
    elif case == "unsoftened":
        eps = 0.0
    elif case == "units":       # lengths in metres, speeds in metres per second, masses in kg
        m, x, v, a, eps = m * 2e30, x * 3e16, v * 300.0, a * 3e-12, 3e12
    elif case == "uneven masses":
        m = m * 10.0 ** rng.uniform(-8, 3, n) * np.where(rng.random(n) < 0.2, 0.0, 1.0)
        m[0] = 1.0
    _check(_evaluate(nb, m, x, v, a, eps, order), oracle.force(m, x, v, a, eps), order)


def test_planar_system_stays_planar(nb):
    n = 300
    m, x, v = ic.plummer(n, seed=5)
    a = np.random.default_rng(5).normal(size=(n, 3))
    x[:, 2] = v[:, 2] = a[:, 2] = 0.0
    out = _evaluate(nb, m, x, v, a, 1e-3)
    for row in (2, 5, 8):
        assert np.all(out[row] == 0.0)


def _evaluate_predicted(nb, m, x, v, a, eps):
    """nb_evaluate_noalloc: the predicted particles as they are given (a
    prediction of a non-finite velocity would spoil the position too)."""
    n = len(m)
    jpred = torch.as_tensor(np.concatenate([x.T, v.T, a.T, m[None]])).to("cuda").contiguous()
    act = torch.arange(n, dtype=torch.int32, device="cuda")
    out = torch.empty((10, n), dtype=torch.float64, device="cuda")
    rc = nb.load().nb_evaluate_noalloc(jpred.data_ptr(), n, eps, act.data_ptr(), n, out.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    return out.cpu().numpy()


def test_nonfinite_position_velocity_and_acceleration(nb):
    n = 130
    m, x, v = ic.plummer(n, seed=6)
    a = np.random.default_rng(6).normal(size=(n, 3))
    bad = v.copy()
    bad[3, 1] = np.nan
    out = _evaluate_predicted(nb, m, x, bad, a, 1e-3)
    assert np.isfinite(out[0:3]).all() and np.isfinite(out[9]).all()
    assert np.isnan(out[3:9]).all()
    bad = x.copy()
    bad[7, 0] = np.nan
    assert np.isnan(_evaluate_predicted(nb, m, bad, v, a, 1e-3)).all()
    bad = a.copy()
    bad[100, 2] = np.inf
    out = _evaluate_predicted(nb, m, x, v, bad, 1e-3)
    assert np.isfinite(out[0:6]).all() and np.isfinite(out[9]).all()
    assert not np.isfinite(out[6:9]).any()


@pytest.mark.parametrize("eps", [1e-4, 0.0, 2.0])
@pytest.mark.parametrize("n", [1, 2, 65, 1000])
def test_potential_parity(nb, oracle, n, eps):
    """The potential-only evaluation behind the energies, all particles."""
    m, x, v = ic.plummer(max(n, 2), seed=n)
    m, x, v = m[:n], x[:n], v[:n]
    a = np.zeros((n, 3))
    sim = nb.Simulation(m, x, v, eps=eps, keep_state=True)
    _, epot, _, _ = sim.energy(0.0)
    sim.close()
    ref = 0.5 * float(np.sum(m * oracle.force(m, x, v, a, eps)[3]))
    assert abs(epot - ref) <= 1e-13 * abs(ref)
