"""The azimuth a particle sweeps next to the axis, on a grid of the packed tile
kernel: from the displacement alone, however small."""
import numpy as np
import pytest

from paper_1407_1810_gb300 import configs

from gpu_common import setup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle as O
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


@pytest.mark.parametrize("nr", [64, 2051])
@pytest.mark.parametrize("uph", [1e-3, 1e-8, 1e-11, 1e-13, -1e-14, 1e-16])
def test_leaving_the_axis(nr, uph):
    """From x2 = 0 along r and phi: a quarter turn, whatever u_ph is."""
    cfg = dict(configs.CONFIGS["monopole-64x64"], nr=nr, nth=64, th_map="linear", vacuum="none", precision="fp32",
               pairs_per_cell=0, absorb_cells=4)
    one = {"x1": np.array([7.3]), "x2": np.array([0.0]), "ur": np.array([0.4]), "uth": np.array([0.0]),
           "uph": np.array([uph]), "qw": np.array([0.37])}
    s, o, _, _ = setup(cfg, plasma=one)
    s.step(1)
    o.step(1)
    assert s.flux()[2].sum() / 0.37 == pytest.approx(np.copysign(0.25, uph), abs=1e-5)
    assert o.flux()[2].sum() / 0.37 == pytest.approx(np.copysign(0.25, uph), abs=1e-5)
