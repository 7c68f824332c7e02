"""Whole-cluster evaluations that take each pair once, in several bands of rows: every
particle against the same evaluation one by one (a list in another order), and
the device memory a context holds.  Tolerances: twice the arithmetics' per particle
(FP64 1e-12, EX 1e-10), each side being within one of them of the exact sums."""
import numpy as np
import pytest

from paper_1812_00367_gb300 import ic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 2e-12, "ex": 2e-10}


@pytest.fixture(scope="module")
def nb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00367_gb300 import build as nbbuild
    nbbuild.build()
    from paper_1812_00367_gb300 import nb as nbmod
    nbmod.load()
    return nbmod


# 1, 2 and 8 bands at the default scratch; 65601: the last row is half a row of one particle
@pytest.mark.parametrize("n", [10007, 30011, 65601])
@pytest.mark.parametrize("order", [6, 4])
@pytest.mark.parametrize("precision", ["fp64", "ex"])
def test_every_particle(nb, precision, order, n):
    m, x, v = ic.plummer(n, seed=n, masses=ic.kroupa_masses(n, seed=n))
    a, z = np.random.default_rng(n).normal(size=(n, 3)), np.zeros((n, 3))
    sim = nb.Simulation(m, x, v, eps=1e-4, precision=precision, order=order, keep_state=True)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": a, "j": z, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    sim.predict(0.0, out=False)
    every = torch.arange(n, dtype=torch.int32, device="cuda")
    got = sim.evaluate(every)
    assert torch.equal(got, sim.evaluate(every))
    want = sim.evaluate(every.flip(0)).flip(1)      # one by one
    for lo in (0, 3, 6):
        if lo == 6 and order == 4:
            assert not got[6:9].any() and not want[6:9].any()
            continue
        err = (got[lo:lo + 3] - want[lo:lo + 3]).norm(dim=0) / want[lo:lo + 3].norm(dim=0)
        assert err.max().item() <= TOL[precision], (lo, err.max().item(), int(err.argmax()))
    assert ((got[9] - want[9]).abs() <= TOL[precision] * want[9].abs()).all()
    _, epot, _, _ = sim.energy(0.0)
    ref = 0.5 * float((torch.as_tensor(m, device="cuda") * want[9]).sum())
    assert abs(epot - ref) <= TOL[precision] * abs(ref)
    sim.sync()
    sim.close()


@pytest.mark.parametrize("precision", ["fp64", "ex", "fp32"])
def test_device_memory(nb, precision):
    """A context of 65,536 particles: state 12 MB, records 7 MB and their FP64 copy
    5 MB, partial sums 199 MB with their counters 0.6 MB; 400 MB leave room for the
    allocator's granularity.  The partial sums of every column at once took 1.3 GB."""
    n = 65536
    m, x, v = ic.plummer(n, seed=1)
    nb.Simulation(m[:9000], x[:9000], v[:9000], eps=1e-4, precision=precision).close()  # modules loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    sim = nb.Simulation(m, x, v, eps=1e-4, precision=precision, keep_state=True)
    sim.sync()
    held = before - torch.cuda.mem_get_info()[0]
    sim.close()
    assert held < 400e6, held
