"""Grids of few tiles that hold millions of particles: the tile kernel's 32-bit
sums keep their room however the particles crowd."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_1810_gb300 import build

    build.build()


@pytest.mark.parametrize("members", [1, 2])
@pytest.mark.parametrize("n,dt,ur,spread", [(3_000_000, 0.05, 0.75, 1.0), (3_000_000, 0.1, 30.0, 0.02),
                                            (60_000, 0.1, 30.0, 0.02), (7_000, 0.1, 30.0, 0.02)])
def test_one_crowded_cell(members, n, dt, ur, spread):
    """A stream of n particles of one sign through one cell, each moving a
    quarter of it or most of it: in flux units every term is near the largest."""
    from paper_1407_1810_gb300 import picsar as P

    g = np.random.default_rng(1)
    f = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    x1, x2 = 8.0 + f(0.1 * g.random(n)), 8.0 + f(spread * g.random(n))
    z = np.zeros(n)
    c = dict(nr=16, nth=16, r_min=1.0, r_max=3.0, r_map="log", th_map="equal_area", dt=dt, n_filt=0, vacuum="none",
             pusher="vay", sort_interval=10)
    sims = {}
    for precision in ("fp32", "fp64"):
        s = [P.Simulation(P.make_desc(**c, precision=precision)) for _ in range(members)]
        for a in s:
            a.load(x1, x2, np.full(n, ur), z, z, np.ones(n))
        if members == 1:
            s[0].step(1)
        else:
            P.ensemble_step(s, 1)
        sims[precision] = s
    for a, b in zip(sims["fp32"], sims["fp64"]):
        a.moments()  # raises if the step reported an error
        fa, fb = a.flux(), b.flux()
        assert np.abs(fb[0]).max() > 0.1 * n
        for k in range(2):
            assert np.abs(fa[k] - fb[k]).max() <= 1e-5 * np.abs(fb[0]).max(), k
