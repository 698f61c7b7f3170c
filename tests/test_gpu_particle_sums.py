"""Kinetic energy and total charge of the FP32 path at the ends of the range of
charges it accepts."""
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


@pytest.mark.parametrize("scale,u", [(1.2e30, 1.5e8), (1.0, 0.3), (2.0 ** -100, 2e-3), (2.0 ** -100, 3.0)])
def test_sums_at_the_ends_of_the_range(scale, u):
    """Accepted charges times energies that are FP32 numbers while the sum of
    eight of them is not, and ones next to the smallest."""
    from paper_1407_1810_gb300 import picsar as P

    g = np.random.default_rng(7)
    n = 1_500_000  # more than eight for every thread of the sum
    w = g.normal(size=(3, n))
    w *= u / np.sqrt((w * w).sum(0))
    q = _f32(scale * np.where(g.random(n) < 0.5, 1.0, -1.0) * (1 + 0.03 * g.random(n)))
    s = P.Simulation(P.make_desc(**GRID))
    s.load(g.random(n) * NR, g.random(n) * NTH, *(_f32(v) for v in w), q)
    m = s.moments()
    k = s.particles()
    u2 = k["ur"] ** 2 + k["uth"] ** 2 + k["uph"] ** 2
    e = (np.abs(k["qw"]) * u2 / (1 + np.sqrt(1 + u2))).sum()
    assert abs(m["kinetic_energy"] - e) <= 8 * 2.0 ** -24 * e
    assert abs(m["total_charge"] - k["qw"].sum()) <= n * EPS * np.abs(k["qw"]).sum()
