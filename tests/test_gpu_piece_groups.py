"""Evaluations whose i-tiles are summed from many pieces: just below, at and above
the 32 pieces from which each group of pieces is summed by its own last CTA, for
every tile width that reaches it, with stream-K ranges and with split items,
against the oracle and bit for bit against a repeat (another order of arrival).
Tolerances: the arithmetics' (FP64 1e-12, FP32X a 1e-10 and jerk, snap 2e-5)."""
import numpy as np
import pytest

from paper_1812_00367_gb300 import ic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-12, 1e-12), "fp32x": (1e-10, 2e-5)}


@pytest.fixture(scope="module")
def nb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00367_gb300 import build as nbbuild
    nbbuild.build()
    from paper_1812_00367_gb300 import nb as nbmod
    nbmod.load()
    return nbmod


# j-tiles: 31, 32, 33 (one per item), 41 (groups of 6 and 7), 313
@pytest.mark.parametrize("n", [31 * 64, 2048, 2049, 2600, 20011])
@pytest.mark.parametrize("precision", ["fp64", "fp32x"])
@pytest.mark.parametrize("streamk", [True, False])
def test_groups_of_pieces(nb, oracle, n, precision, streamk):
    eps = 1e-3
    m, x, v = ic.plummer(n, seed=n)
    rng = np.random.default_rng(n)
    a, z = rng.normal(size=(n, 3)), np.zeros((n, 3))
    sim = nb.Simulation(m, x, v, eps=eps, precision=precision, keep_state=True, streamk=streamk)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": a, "j": z, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    sim.predict(0.0, out=False)
    acts = [np.sort(rng.choice(n, A, replace=False)).astype(np.int32)
            for A in (1, 3, 4, 9, 30, 63, 64, 100, 129, 400, 1000)]
    every = np.unique(np.concatenate(acts)).astype(np.int32)
    ref = oracle.force(m, x, v, a, eps, active=every)
    for act in acts:
        at = torch.as_tensor(act, device="cuda")
        got = sim.evaluate(at).cpu().numpy()
        for _ in range(4):
            np.testing.assert_array_equal(got, sim.evaluate(at).cpu().numpy())
        k = np.searchsorted(every, act)
        for lo, want, tol in ((0, ref[0][k], 0), (3, ref[1][k], 1), (6, ref[2][k], 1)):
            err = np.linalg.norm(got[lo:lo + 3].T - want, axis=1) / np.linalg.norm(want, axis=1)
            assert err.max() <= TOL[precision][tol], (len(act), lo, float(err.max()))
        assert (np.abs(got[9] - ref[3][k]) <= TOL[precision][0] * np.abs(ref[3][k])).all()
    sim.close()
