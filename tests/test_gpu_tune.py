"""The autotuner stores the lanes of the launch it timed, and a table timed for one
way of launching is not taken for another.  N = 4096, FP64, one cluster: up to 384
active particles every candidate is raised to 32 lanes (fewer units than stream-K
wants), so 32 is what was timed; a batch runs a table's own lanes and split items."""
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


def _table(path):
    lines = open(path).read().splitlines()
    return lines[0].split(), [tuple(map(int, x.split())) for x in lines[1:]]


def test_stored_lanes_and_cache_key(nb, tmp_path):
    path = str(tmp_path / "table.txt")
    m, x, v = ic.plummer(4096, seed=1)
    sim = nb.Simulation(m, x, v, eps=1e-3)
    sim.autotune(path)
    head, one = _table(path)
    assert len(one) == 32 and all(gl == 32 for gl, _ in one[:9])
    sim.autotune(path)                               # loads what it wrote
    assert _table(path) == (head, one)
    sim.close()
    batch = ic.plummer_batch(sizes=[4096, 512], seed=2)
    sim = nb.Simulation(batch.m, batch.x, batch.v, eps=1e-3, offsets=batch.offsets)
    sim.autotune(path)                               # times its own launches
    bhead, own = _table(path)
    assert bhead != head
    sim.autotune(path)
    assert _table(path) == (bhead, own)
    sim.run(1.0 / 64)
    sim.close()
    # one cluster with split items runs what a batch runs: the batch's table serves
    sim = nb.Simulation(m, x, v, eps=1e-3, streamk=False)
    sim.autotune(path)
    assert _table(path) == (bhead, own)
    sim.close()
    # a table without the fields is taken as given
    plain = "nbtune 0 0\n" + "8 64\n" * 32
    (tmp_path / "plain.txt").write_text(plain)
    sim = nb.Simulation(m, x, v, eps=1e-3)
    sim.autotune(str(tmp_path / "plain.txt"))
    assert (tmp_path / "plain.txt").read_text() == plain
    sim.close()
