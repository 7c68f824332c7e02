"""Whole-cluster FP64 and EX evaluations that take each pair once: sizes at the edges of
rows (128) and columns (64), both orders, a list that is not every particle in
order, the start-up, the potential, and what is not finite.  Tolerances: the
arithmetics' per particle (FP64 1e-12, EX 1e-10)."""
import numpy as np
import pytest

from paper_1812_00367_gb300 import ic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [8192, 8193, 8255, 8256, 8319, 10007]
TOL = {"fp64": 1e-12, "ex": 1e-10}


@pytest.fixture(scope="module")
def nb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00367_gb300 import build as nbbuild
    nbbuild.build()
    from paper_1812_00367_gb300 import nb as nbmod
    nbmod.load()
    return nbmod


def _system(n, seed):
    masses = ic.kroupa_masses(n, seed=seed)
    masses[::97] = 0.0                       # massless particles feel, but do not pull
    m, x, v = ic.plummer(n, seed=seed, masses=masses)
    return m, x, v, np.random.default_rng(seed).normal(size=(n, 3))


def _sim(nb, m, x, v, a, **kw):
    n, z = len(m), np.zeros((len(m), 3))
    sim = nb.Simulation(m, x, v, keep_state=True, **kw)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": a, "j": z, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    sim.predict(0.0, out=False)
    return sim


def _check(got, ref, order, sel, tol):
    for lo, want in ((0, ref[0]), (3, ref[1]), (6, ref[2])):
        if lo == 6 and order == 4:
            assert np.all(got[6:9] == 0.0)
            continue
        err = np.linalg.norm(got[lo:lo + 3, sel].T - want, axis=1) / np.linalg.norm(want, axis=1)
        assert err.max() <= tol, (lo, float(err.max()))
    assert (np.abs(got[9, sel] - ref[3]) <= tol * np.abs(ref[3])).all()


@pytest.mark.parametrize("order", [6, 4])
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("precision", ["fp64", "ex"])
def test_whole_cluster_parity(nb, oracle, precision, n, order):
    eps, tol = 1e-4, TOL[precision]
    m, x, v, a = _system(n, n)
    sim = _sim(nb, m, x, v, a, eps=eps, order=order, precision=precision)
    every = torch.arange(n, dtype=torch.int32, device="cuda")
    got = sim.evaluate(every).cpu().numpy()
    np.testing.assert_array_equal(got, sim.evaluate(every).cpu().numpy())
    sel = np.unique(np.concatenate([[0, 1, 63, 64, 127, 128, n - 65, n - 2, n - 1],
                                    np.random.default_rng(n).choice(n, 150, replace=False)])).astype(np.int32)
    ref = oracle.force(m, x, v, a, eps, active=sel)
    _check(got, ref, order, sel, tol)
    # n entries that are not every particle in order: one by one, as listed
    perm = np.random.default_rng(n + 1).permutation(n).astype(np.int32)
    out = sim.evaluate(torch.as_tensor(perm, device="cuda")).cpu().numpy()
    back = np.empty_like(out)
    back[:, perm] = out
    _check(back, ref, order, sel, tol)
    dup = perm.copy()
    dup[1] = dup[0]
    out = sim.evaluate(torch.as_tensor(dup, device="cuda")).cpu().numpy()
    one = oracle.force(m, x, v, a, eps, active=dup[:2])
    _check(out, one, order, np.array([0, 1]), tol)
    sim.sync()
    sim.close()


@pytest.mark.parametrize("order", [6, 4])
@pytest.mark.parametrize("precision", ["fp64", "ex"])
def test_start_up_and_potential(nb, oracle, precision, order):
    n, eps = 8300, 1e-3
    m, x, v, _ = _system(n, 3)
    m = np.where(m > 0, m, 1e-9)
    sim = nb.Simulation(m, x, v, eps=eps, order=order, eta=0.4 if order == 6 else 0.02, precision=precision)
    ref = oracle.Sim(m, x, v, eps=eps, order=order, eta=0.4 if order == 6 else 0.02).init()
    st = sim.state_numpy()
    for f in ("a", "j", "s"):
        want = getattr(ref, f)
        den = np.maximum(np.linalg.norm(want, axis=1), 1e-300)
        assert (np.linalg.norm(st[f] - want, axis=1) <= TOL[precision] * den).all(), f
    if precision == "fp64":
        np.testing.assert_array_equal(st["dt"], ref.dt)
    _, epot, _, _ = sim.energy(0.0)
    want = 0.5 * float(np.sum(m * oracle.force(m, x, v, np.zeros((n, 3)), eps)[3]))
    assert abs(epot - want) <= 1e-13 * abs(want)
    sim.close()


@pytest.mark.parametrize("precision", ["fp64", "ex"])
def test_what_is_not_finite_spreads(nb, precision):
    n = 8200
    m, x, v, a = _system(n, 9)
    every = torch.arange(n, dtype=torch.int32, device="cuda")
    sim = _sim(nb, m, x, v, a, eps=1e-3, precision=precision)
    st = sim.state_numpy()
    st["x"][4711, 1] = np.nan
    sim.set_state_numpy(st)
    sim.predict(0.0, out=False)
    got = sim.evaluate(every).cpu().numpy()
    # EX takes each component by itself: the position's y component is lost
    assert np.isnan(got if precision == "fp64" else got[3:9]).all()
    sim.close()
