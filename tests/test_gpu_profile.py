"""The phases that pic_get_profile times: a phase with kernels of its own has a
time, one that runs inside another's kernel has none."""
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


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n_filt", [0, 4, 5, 6])
def test_phases(precision, n_filt):
    from paper_1407_1810_gb300 import picsar as P

    s = P.Simulation(P.make_desc(nr=40, nth=40, r_min=1.0, r_max=3.0, r_map="log", th_map="linear", dt=0.004,
                                 n_filt=n_filt, vacuum="monopole", b0=1.0, precision=precision, pusher="vay",
                                 sort_interval=3))
    g = np.random.default_rng(0)
    s.load(g.random(500) * 40, g.random(500) * 40, *(0.1 * g.normal(size=500) for _ in range(3)), np.ones(500))
    s.step(2)
    s.profile(True)
    s.step(6)
    ms, steps = s.get_profile()
    assert steps == 6
    assert ms["particles"] > 0 and ms["fields"] > 0 and ms["sort"] > 0 and ms["inject"] == 0
    assert (ms["reduce"] > 0) == (n_filt > 4 and precision == "fp32")
    assert (ms["filter"] > 0) == (n_filt > 4)
    assert max(ms.values()) < 1e3
