"""FP64 charges near the end of the range on a pole node, through the filter's
one-pass form: finite sums as the passes taken one by one give them, and what
has overflowed stays infinite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRID = dict(nr=14, nth=34, r_min=1.0, r_max=3.0, r_map="log", th_map="equal_area", dt=0.004, vacuum="none",
            pusher="vay")
BIG = 1.5e308  # above 2^1023: twice it is infinite


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle as O
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


def _passes(a, n_filt):
    import oracle as O

    o = O.Oracle(O.params(**GRID, n_filt=n_filt))
    for _ in range(n_filt):
        a = o.filter_pass(a, 0, 1)
    return a


@pytest.mark.parametrize("n_filt", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("x2", [0.0, 1.0, 34.0])
@pytest.mark.parametrize("q", [BIG, -BIG])
def test_charge_on_one_node(n_filt, x2, q):
    from paper_1407_1810_gb300 import picsar as P

    s = P.Simulation(P.make_desc(**GRID, n_filt=n_filt, precision="fp64"))
    one = [np.array([6.0]), np.array([x2])] + [np.zeros(1)] * 3
    s.load(*one, np.array([q]))
    a = np.zeros((GRID["nr"] + 2 * s.g + 1, GRID["nth"] + 1))
    a[6 + s.g, int(x2)] = 1.0
    w = _passes(a, n_filt)  # exact: multiples of 16^-n_filt
    F = s.charge(filtered=True)
    # one term: the weight times the charge, a few roundings
    assert np.all(np.abs(F - q * w) <= 8 * 2.0 ** -53 * abs(q) * w)
    s.load(*one, np.array([q]))
    F = s.charge(filtered=True)
    assert np.array_equal(np.isinf(F) & (np.sign(F) == np.sign(q)), w != 0)
    assert np.all(F[w == 0] == 0.0)


@pytest.mark.parametrize("n_filt", [1, 3])
def test_flux_along_the_axis(n_filt):
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    c = dict(GRID, n_filt=n_filt, dt=0.07, th_map="linear")
    p = [np.array([6.05]), np.array([0.0]), np.array([20.0]), np.zeros(1), np.zeros(1), np.array([1.7e308])]
    s, o = P.Simulation(P.make_desc(**c, precision="fp64")), O.Oracle(O.params(**c))
    for x in (s, o):
        x.load(*p)
    s.step(1)
    o.step(1)
    b = o.flux()
    assert np.abs(b[0]).max() > 0.1 * 1.7e308 / 2 ** (2 * n_filt)
    assert np.all(np.abs(s.flux()[0] - b[0]) <= 1e-12 * np.abs(b[0]).max())
