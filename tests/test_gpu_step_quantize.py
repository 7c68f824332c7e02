"""A block step's corrector and time step (four lanes a particle, the criterion
as rough logarithms) against the same step through nb_predict, nb_evaluate and
nb_correct_and_timestep (one thread a particle, the criterion in FP64): every field equal bit
for bit.  Wide ranges of the derivatives and of eta, so that many steps fall near
powers of two, grow, shrink and reach both clamps; all tile widths."""
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


@pytest.mark.parametrize("order", [6, 4])
@pytest.mark.parametrize("n", [3, 30, 200, 1500, 7000])
@pytest.mark.parametrize("eta", [0.02, 0.37, 3.0])
def test_step_equals_correct(nb, order, n, eta):
    rng = np.random.default_rng(n)
    m, x, v = ic.plummer(n, seed=n)
    scale = 10.0 ** rng.uniform(-6, 6, (n, 1))
    dt = 2.0 ** rng.choice([-6.0, -7.0, -9.0], n)
    state = {"m": m, "x": x, "v": v, "a": rng.normal(size=(n, 3)), "j": rng.normal(size=(n, 3)) * scale,
             "s": rng.normal(size=(n, 3)) * scale ** 2, "c": rng.normal(size=(n, 3)),
             "t": np.full(n, 0.75) - dt, "dt": dt, "pot": np.zeros(n)}
    out = []
    for way in range(2):
        sim = nb.Simulation(m, x, v, eps=1e-2, eta=eta, order=order, keep_state=True,
                            dt_min=2.0 ** -20, dt_max=2.0 ** -6)
        sim.set_state_numpy(state)
        if way == 0:
            assert sim.run(0.75, 1)[0] == 1
        else:
            act = torch.arange(n, dtype=torch.int32, device="cuda")
            sim.predict(0.75, out=False)
            acc = sim.evaluate(act)
            nb.nb_correct_and_timestep(sim.ctx, 0, act, n, 0.75, acc)
            sim.sync()
        out.append((sim.state_numpy(), sim.counters()))
        sim.close()
    assert len(np.unique(out[0][0]["dt"])) >= (2 if n > 100 else 1)
    for f in ("x", "v", "a", "j", "s", "c", "t", "dt", "pot"):
        np.testing.assert_array_equal(out[0][0][f], out[1][0][f], err_msg=f)
