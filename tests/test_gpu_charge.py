"""The FP32 path's exact node charge and its one-pass filter, against FP64 sums
over the particles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle as O
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


def _load(seed, nr, nth, n, dense):
    g = np.random.default_rng(seed)
    f = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    x1 = g.integers(-1, nr + 1, n) + f(g.random(n))
    x2 = g.integers(0, nth, n) + f(g.random(n))
    x1[:8], x2[8:16] = 3.0, 5.0               # on grid lines
    x2[16:24], x2[24:32] = 0.0, float(nth)     # on the axis
    x1[32:64] = 4 + f(2.0 ** -g.integers(1, 60, 32))   # offsets far below 2^-24
    u = f(g.normal(size=(3, n)))
    q = f(np.where(g.random(n) < 0.5, 1.0, -1.0) * 10.0 ** g.uniform(-9, 0, n))  # charges nine decades apart
    if dense:  # more than 2^13 particles in one cell, on its corner, of the largest charge
        x1 = np.concatenate([x1, np.full(dense, 6.0)])
        x2 = np.concatenate([x2, np.full(dense, 2.0)])
        u = np.concatenate([u, np.zeros((3, dense))], 1)
        q = np.concatenate([q, np.ones(dense)])
    return [np.ascontiguousarray(a) for a in (x1, x2, u[0], u[1], u[2], q)]


def _sums(p, nr, nth, g):
    """Node charge, and the bound of its rounding on both sides: numpy rounds
    every product (twice) and every partial sum, the library rounds a share to
    2^-54 of the largest charge and the sum once."""
    Q = np.zeros((nr + 2 * g + 1, nth + 2))
    A = np.zeros_like(Q)
    N = np.zeros_like(Q)
    i, j = np.floor(p["x1"]).astype(int), np.minimum(np.floor(p["x2"]).astype(int), nth - 1)
    a, b = p["x1"] - i, p["x2"] - j
    for di, dj, w in ((0, 0, (1 - a) * (1 - b)), (1, 0, a * (1 - b)), (0, 1, (1 - a) * b), (1, 1, a * b)):
        np.add.at(Q, (i + g + di, j + dj), p["qw"] * w)
        np.add.at(A, (i + g + di, j + dj), np.abs(p["qw"]) * w)
        np.add.at(N, (i + g + di, j + dj), 1.0)
    qmax = 2.0 ** np.ceil(np.log2(np.abs(p["qw"]).max()))
    return Q[:, :-1], ((N + 3) * EPS * A + N * 3 * 2.0 ** -54 * qmax)[:, :-1]


@pytest.mark.parametrize("tile_shape", [0, 1, 2])
@pytest.mark.parametrize("nr,nth,dense", [(16, 16, 0), (37, 45, 0), (20, 33, 20000)])
@pytest.mark.parametrize("stepped", [False, True])
def test_node_charge_is_the_sum_over_the_particles(tile_shape, nr, nth, dense, stepped):
    from paper_1407_1810_gb300 import picsar as P

    s = P.Simulation(P.make_desc(nr=nr, nth=nth, r_min=1.0, r_max=3.0, r_map="log", th_map="linear", dt=0.004,
                                 n_filt=0, vacuum="monopole", b0=3.0, precision="fp32", pusher="vay",
                                 tile_shape=tile_shape, sort_interval=50))
    s.load(*_load(nr, nr, nth, 5000, dense))
    if stepped:  # binned, then drifted; and some never binned
        s.step(30)
        s.load(*_load(1, nr, nth, 300, 0))
    Q = s.charge()
    m = s.moments()
    p = s.particles()
    ref, bound = _sums(p, nr, nth, s.g)
    d = np.abs(Q - ref)
    assert np.all(d <= bound), float((d / np.maximum(bound, 1e-300)).max())
    assert abs(m["total_charge"] - p["qw"].sum()) <= len(p["qw"]) * EPS * np.abs(p["qw"]).sum()
    # each term in FP32 (a few roundings of 2^-24), the sum in FP64
    u2 = p["ur"] ** 2 + p["uth"] ** 2 + p["uph"] ** 2
    k = (np.abs(p["qw"]) * u2 / (1 + np.sqrt(1 + u2))).sum()
    assert abs(m["kinetic_energy"] - k) <= 8 * 2.0 ** -24 * k
    assert m["live"] == len(p["qw"])


@pytest.mark.parametrize("n_filt", [1, 3, 4, 5])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_filtered_charge(n_filt, precision):
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    kw = dict(nr=19, nth=34, r_min=1.0, r_max=3.0, r_map="log", th_map="equal_area", dt=0.004, n_filt=n_filt,
              vacuum="none", pusher="vay")
    s = P.Simulation(P.make_desc(**kw, precision=precision))
    s.load(*_load(2, 19, 34, 4000, 0))
    s.step(2)
    a, F = s.charge(), s.charge(filtered=True)
    scale = np.abs(a).max()
    o = O.Oracle(O.params(**kw))
    for _ in range(n_filt):
        a = o.filter_pass(a, 0, 1)
    assert np.abs(F - a).max() <= n_filt * 18 * EPS * scale + 1e-13 * scale * (precision == "fp64")
