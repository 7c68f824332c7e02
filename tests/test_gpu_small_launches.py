"""Evaluations of few active particles and of small clusters: every number of
lanes per i (1 to 32), ragged last tiles, one piece and many, with and without
stream-K, against the oracle and bit for bit against a repeat.  Tolerances: the
arithmetics' (FP64 1e-12, EX 1e-10, FP32 2e-5)."""
import numpy as np
import pytest

from paper_1812_00367_gb300 import ic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "ex": 1e-10, "fp32": 2e-5}


@pytest.fixture(scope="module")
def nb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00367_gb300 import build as nbbuild
    nbbuild.build()
    from paper_1812_00367_gb300 import nb as nbmod
    nbmod.load()
    return nbmod


@pytest.mark.parametrize("precision", ["fp64", "ex", "fp32"])
@pytest.mark.parametrize("n", [129, 1024, 8200])
@pytest.mark.parametrize("streamk", [True, False])
def test_small_launches(nb, oracle, precision, n, streamk):
    eps = 1e-3
    m, x, v = ic.plummer(n, seed=n)
    rng = np.random.default_rng(n)
    a, z = rng.normal(size=(n, 3)), np.zeros((n, 3))
    sim = nb.Simulation(m, x, v, eps=eps, precision=precision, keep_state=True, streamk=streamk)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": a, "j": z, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    sim.predict(0.0, out=False)
    sizes = [A for A in (1, 2, 3, 4, 5, 7, 9, 17, 31, 33, 63, 64, 65, 127, 129, 257, 511, 1023, 1025, 2500, 4097)
             if A <= n]
    acts = [np.sort(rng.choice(n, A, replace=False)).astype(np.int32) for A in sizes]
    every = np.unique(np.concatenate(acts))
    ref = oracle.force(m, x, v, a, eps, active=every.astype(np.int32))
    for act in acts:
        at = torch.as_tensor(act, device="cuda")
        got = sim.evaluate(at).cpu().numpy()
        np.testing.assert_array_equal(got, sim.evaluate(at).cpu().numpy())
        k = np.searchsorted(every, act)
        for lo, want in ((0, ref[0][k]), (3, ref[1][k]), (6, ref[2][k])):
            err = np.linalg.norm(got[lo:lo + 3].T - want, axis=1) / np.linalg.norm(want, axis=1)
            assert err.max() <= TOL[precision], (len(act), lo, float(err.max()))
        assert (np.abs(got[9] - ref[3][k]) <= TOL[precision] * np.abs(ref[3][k])).all()
    sim.close()
