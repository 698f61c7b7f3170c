"""Node charge of the FP32 path when the charges span its whole range: every node
as accurate as an FP64 sum over its own particles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
NR, NTH = 33, 45
GRID = dict(nr=NR, nth=NTH, r_min=1.0, r_max=3.0, r_map="log", th_map="linear", dt=0.004, n_filt=0, vacuum="none",
            precision="fp32", pusher="vay")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_1810_gb300 import build

    build.build()


def _f32(a):
    return np.asarray(a).astype(np.float32).astype(np.float64)


def _sums(p, g):
    """Node charge; its rounding on both sides: numpy rounds every product
    (twice) and partial sum, the library a share to 2^-54 of its own
    particle's charge, and the sum."""
    Q = np.zeros((NR + 2 * g + 1, NTH + 2))
    A, N, L = np.zeros_like(Q), np.zeros_like(Q), np.zeros_like(Q)
    i, j = np.floor(p["x1"]).astype(int), np.minimum(np.floor(p["x2"]).astype(int), NTH - 1)
    a, b = p["x1"] - i, p["x2"] - j
    for di, dj, w in ((0, 0, (1 - a) * (1 - b)), (1, 0, a * (1 - b)), (0, 1, (1 - a) * b), (1, 1, a * b)):
        np.add.at(Q, (i + g + di, j + dj), p["qw"] * w)
        np.add.at(A, (i + g + di, j + dj), np.abs(p["qw"]) * w)
        np.add.at(L, (i + g + di, j + dj), np.abs(p["qw"]))
        np.add.at(N, (i + g + di, j + dj), 1.0)
    return Q[:, :-1], ((N + 3) * EPS * A + 3 * 2.0 ** -54 * L)[:, :-1]


@pytest.mark.parametrize("small", [2.0 ** -6, 2.0 ** -8, 1.4 * 2.0 ** -9, 2.0 ** -20, 1.3 * 2.0 ** -34, 2.0 ** -50, 2.0 ** -70])
@pytest.mark.parametrize("flux_quantum", [0.0, 2.0 ** 10])
@pytest.mark.parametrize("stepped", [False, True])
def test_nodes_of_small_charges(small, flux_quantum, stepped):
    """Charges of about 1 at low x2, of about `small` beyond them; flux_quantum
    raises the fixed-point exponent by another 46 bits."""
    from paper_1407_1810_gb300 import picsar as P

    g = np.random.default_rng(5)
    n = 6000
    x1, x2 = g.integers(0, NR, n) + _f32(g.random(n)), g.integers(0, NTH, n) + _f32(g.random(n))
    q = np.where(g.random(n) < 0.5, 1.0, -1.0) * (1 + g.random(n)) * np.where(x2 < 20, 1.0, small)
    s = P.Simulation(P.make_desc(**GRID, flux_quantum=flux_quantum))
    s.load(x1, x2, *(_f32(v) for v in 0.3 * g.normal(size=(3, n))), _f32(q))
    if stepped:
        s.step(5)
    p = s.particles()
    ref, bound = _sums(p, s.g)
    d = np.abs(s.charge() - ref)
    assert np.all(d <= bound), float((d / np.maximum(bound, 1e-300)).max())


def test_the_step_after_a_charge_is_undisturbed():
    """The node charge borrows a plane of the deposit and clears it."""
    from paper_1407_1810_gb300 import picsar as P

    g = np.random.default_rng(6)
    n = 3000
    a = [g.integers(0, NR, n) + _f32(g.random(n)), g.integers(0, NTH, n) + _f32(g.random(n)),
         *(_f32(v) for v in 0.3 * g.normal(size=(3, n))), _f32(10.0 ** g.uniform(-20, 0, n))]
    out = []
    for ask in (False, True):
        s = P.Simulation(P.make_desc(**GRID))
        s.load(*a)
        s.step(2)
        if ask:
            s.charge()
            s.moments()
        s.step(2)
        out.append((s.flux(), s.fields()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
