"""Jerk and snap of the FP64 evaluation component by component, in systems thin
along z (1e-2 to 1e-8 of the extent), in both forms (one-sided and each pair
once), against sums in long double.  Tolerance: every component against the sum
of its own summands' absolute values,
    jerk  C1 = sum_j q (|v_k| + 3 A |r_k|),  A = sum_k |r_k v_k| / r^2,
    snap  C2 = sum_j q (|a_k| + 6 A (|v_k| + 3 A |r_k|) + 3 B |r_k|).
A pair term in doubles is within 12 roundings of its summands (difference, q: 5,
alpha or beta: 4, two FMAs), the sums of n <= 8320 terms add at most the partial
sums' roundings, sqrt(n) < 92 of them at random: 2^-53 (12 + 92) < 2^-46."""
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


def _sums(m, x, v, a, eps, i):
    """Jerk and snap of particle i and their summands' absolute sums, [3] each."""
    L = np.longdouble
    r, w, b = (np.asarray(f, dtype=L) - np.asarray(f[i], dtype=L) for f in (x, v, a))
    r2 = (r * r).sum(1) + L(eps * eps)
    q = np.asarray(m, dtype=L) / (r2 * np.sqrt(r2))
    q[i] = 0
    al = (r * w).sum(1) / r2
    be = ((w * w).sum(1) + (r * b).sum(1)) / r2 + al * al
    w1 = w - 3 * al[:, None] * r
    w2 = b - 6 * al[:, None] * w1 - 3 * be[:, None] * r
    aa = np.abs(r * w).sum(1) / r2
    ab = ((w * w).sum(1) + np.abs(r * b).sum(1)) / r2 + aa * aa
    c1 = np.abs(w) + 3 * aa[:, None] * np.abs(r)
    c2 = np.abs(b) + 6 * aa[:, None] * c1 + 3 * ab[:, None] * np.abs(r)
    aq = np.abs(q)[:, None]
    return (q[:, None] * w1).sum(0), (q[:, None] * w2).sum(0), (aq * c1).sum(0), (aq * c2).sum(0)


@pytest.mark.parametrize("order", [6, 4])
@pytest.mark.parametrize("thin", [1e-2, 1e-5, 1e-8])
@pytest.mark.parametrize("n", [300, 8320])   # 8320: every particle active takes each pair once
def test_thin_systems(nb, n, thin, order):
    eps = 1e-4
    m, x, v = ic.plummer(n, seed=n + order)
    a, z = np.random.default_rng(n).normal(size=(n, 3)), np.zeros((n, 3))
    for f in (x, v, a):
        f[:, 2] *= thin
    sim = nb.Simulation(m, x, v, eps=eps, keep_state=True, order=order)
    sim.set_state_numpy({"m": m, "x": x, "v": v, "a": a, "j": z, "s": z, "c": z, "t": np.zeros(n),
                         "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
    sim.predict(0.0, out=False)
    every = np.arange(n, dtype=np.int32)
    some = np.random.default_rng(1).choice(n, 40, replace=False).astype(np.int32)
    for act in (every, some):
        out = sim.evaluate(torch.as_tensor(act, device="cuda")).cpu().numpy()
        for i in some:
            j, s, cj, cs = _sums(m, x, v, a, eps, i)
            k = int(np.nonzero(act == i)[0][0])
            assert (np.abs(out[3:6, k] - j) <= 2.0 ** -46 * cj).all(), (n, i)
            if order == 6:
                assert (np.abs(out[6:9, k] - s) <= 2.0 ** -46 * cs).all(), (n, i)
    sim.close()
