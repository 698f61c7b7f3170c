"""The FP64 step at distances and displacements whose squares or reciprocals
leave the range of normal numbers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRID = dict(nr=20, nth=36, r_min=1.0, r_max=2.0, r_map="log", dt=0.01, n_filt=0, vacuum="none", pusher="vay")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle as O
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


def _pair(particle, **over):
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    c = dict(GRID, th_map="linear", **over)
    s, o = P.Simulation(P.make_desc(**c, precision="fp64")), O.Oracle(O.params(**c))
    for x in (s, o):
        x.load(*(np.array([v]) for v in particle))
        x.step(1)
    return s, o


@pytest.mark.parametrize("x2", [1e-150, 1e-153, 1e-154, 1e-155, 1e-156, 1e-157, 1e-160, 1e-200, 1e-300])
@pytest.mark.parametrize("turn", [0.0, 1.0, -0.3])
def test_next_to_the_axis(x2, turn):
    """u_ph displaces the particle by `turn` times its distance from the axis."""
    r = 2.0 ** (7.25 / 20)
    st = np.pi * x2 / 36
    up = turn * st * r / 0.01 * np.sqrt(1 + 0.5 ** 2)
    s, o = _pair([7.25, x2, 0.5, 0.0, up, 0.8])
    a, b = s.particles(), o.particles()  # raises if the step reported an error
    assert len(a["x1"]) == 1
    assert abs(a["x1"][0] - b["x1"][0]) <= 1e-13
    assert 0.0 <= a["x2"][0] <= 3 * x2
    assert abs(a["ur"][0] - 0.5) <= 1e-15 and abs(a["uth"][0]) <= 1e-140 and abs(a["uph"][0]) <= 1e-140
    # r_local stays 1 / (1 + a) of the turn on the way out: the swept azimuth
    g = np.sqrt(1 + 0.5 ** 2)
    phi = np.arctan2(up / g * 0.01 / r, st * (1 + 0.5 / g * 0.01 / r))
    assert abs(s.flux()[2].sum() - 0.8 * phi / (2 * np.pi)) <= 1e-13

