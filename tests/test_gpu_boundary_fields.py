"""Fields set on the conductors and on the axis, which no update reaches: they
stay, the lossy layer scales those in its rows, and the curls and the gather
read them, as the oracle has it."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("th_map", ["linear", "equal_area"])
@pytest.mark.parametrize("profile,cells", [("none", 0), ("linear", 1), ("quadratic", 4), ("linear", 11)])
@pytest.mark.parametrize("n_filt", [0, 3, 5])
def test_values_on_the_boundaries(precision, th_map, profile, cells, n_filt):
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    nr, nth = 12, 40
    c = dict(nr=nr, nth=nth, r_min=1.0, r_max=1.8, r_map="log", th_map=th_map, dt=0.003, n_filt=n_filt,
             absorb_cells=cells, absorb_profile=profile, vacuum="none", pusher="vay")
    g = np.random.default_rng(3)
    f = g.normal(size=(6, nr + 1, nth + 1))
    f[0, -1] = f[4, -1] = f[5, -1] = 0.0       # beyond the components' rows
    f[[1, 3, 5], :, -1] = 0.0                  # and columns
    n = 400
    x1 = np.concatenate([g.random(n) * nr, g.random(40) * nr])
    x2 = np.concatenate([2 + g.random(n) * (nth - 4), g.choice([0.3, 0.6, nth - 0.4, nth - 0.7], 40)])
    x1 = np.floor(x1) + (x1 - np.floor(x1)).astype(np.float32)
    x2 = np.floor(x2) + (x2 - np.floor(x2)).astype(np.float32)
    u = (0.1 * g.normal(size=(3, n + 40))).astype(np.float32).astype(np.float64)
    s, o = P.Simulation(P.make_desc(**c, precision=precision)), O.Oracle(O.params(**c))
    for x in (s, o):
        x.load(x1, x2, *(np.ascontiguousarray(a) for a in u), np.full(n + 40, 2.0 ** -12))
        x.set_fields(f)
    bar = 1e-12 if precision == "fp64" else 1e-5
    for steps in (1, 4):
        s.step(steps)
        assert o.step(steps) == 0
        a, b = s.fields(), o.fields()
        for k in range(6):
            assert np.abs(a[k] - b[k]).max() <= bar * np.abs(b[k]).max(), (steps, k)
        p, q = s.particles(), o.particles()
        i, j = np.argsort(p["id"]), np.argsort(q["id"])
        assert np.array_equal(p["id"][i], q["id"][j])
        for k in ("ur", "uth", "uph"):
            # (next to the axis the turn of the basis divides a rounding by the distance)
            assert np.abs(p[k][i] - q[k][j]).max() <= 1e3 * bar * np.abs(u).max(), (steps, k)


@pytest.mark.parametrize("cells", [0, 4])
def test_the_gather_reads_the_axis(cells):
    """B_th on the axis alone, in the FP32 path's copies after the first step too."""
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    nr, nth = 12, 40
    c = dict(nr=nr, nth=nth, r_min=1.0, r_max=1.8, r_map="log", th_map="linear", dt=0.003, n_filt=0, absorb_cells=cells,
             absorb_profile="linear" if cells else "none", vacuum="none", pusher="vay")
    f = np.zeros((6, nr + 1, nth + 1))
    f[4, :-1, [0, -1]] = 40.0
    x1 = np.repeat(np.arange(nr) + 0.5, 2)
    x2 = np.tile([0.5, nth - 0.5], nr)
    u = [np.full(2 * nr, v) for v in (0.25, 0.0, 0.125)]
    s, o = P.Simulation(P.make_desc(**c, precision="fp32")), O.Oracle(O.params(**c))
    for x in (s, o):
        x.load(x1, x2, *u, np.full(2 * nr, 2.0 ** -20))
        x.set_fields(f)
        x.step(4)
    p, q = s.particles(), o.particles()
    i, j = np.argsort(p["id"]), np.argsort(q["id"])
    turned = 0.0
    for k, v in zip(("ur", "uth", "uph"), u):
        assert np.abs(p[k][i] - q[k][j]).max() <= 2e-6, k
        turned = max(turned, np.abs(q[k][j] - v).max())
    assert turned > 1e-2  # the field matters
