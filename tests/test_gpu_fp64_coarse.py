"""One FP64 step on grids that take the library functions (dxi > 1/16, nth < 32,
a step that moves r^2 by more than 1/16 of itself) while every move stays
within one cell, so that each map, pusher and analytic field is compared."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52
VACUA = ["none", "monopole", "monopole_rotator", "uniform_bz", "dipole_corot", "dipole_rotator"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle as O
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


@pytest.mark.parametrize("vacuum", VACUA)
@pytest.mark.parametrize("r_map,r_max", [("log", 6.0), ("linear", 2.0)])
@pytest.mark.parametrize("th_map", ["linear", "equal_area"])
@pytest.mark.parametrize("pusher", ["vay", "boris"])
def test_one_step(r_map, r_max, th_map, pusher, vacuum):
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    nr, nth = 8, 31
    c = dict(nr=nr, nth=nth, r_min=1.0, r_max=r_max, dt=0.04, r_map=r_map, th_map=th_map, pusher=pusher, n_filt=1,
             absorb_cells=1, absorb_profile="linear", b0=20.0, omega=0.3, t_spin=0.0, vacuum=vacuum)
    g = np.random.default_rng(11 + VACUA.index(vacuum))
    n = 4000
    x1 = g.random(n) * (nr + 2.0) - 1.0  # the conductors' first rows too
    x2 = np.clip(g.random(n) * nth, 0.01, nth - 0.01)
    x1[:20], x2[20:40] = np.round(x1[:20] * 2) / 2, np.clip(np.round(x2[20:40] * 2) / 2, 0.5, nth - 0.5)
    u = g.normal(size=(3, n)) * np.array([0.3, 2.0])[g.integers(0, 2, n)]
    u[:, :3] = 0.0
    qw = np.where(g.random(n) < 0.5, 0.7, -0.4)
    f = g.normal(size=(6, nr + 1, nth + 1)) * 3.0
    f[0, -1] = f[4, -1] = f[5, -1] = 0.0
    f[1, [0, -1]] = f[2, [0, -1]] = 0.0
    f[[1, 3, 5], :, -1] = 0.0
    f[2, :, [0, -1]] = f[4, :, [0, -1]] = 0.0
    s, o = P.Simulation(P.make_desc(**c, precision="fp64")), O.Oracle(O.params(**c))
    for x in (s, o):
        x.load(x1, x2, *(np.ascontiguousarray(a) for a in u), qw)
        x.set_fields(f)
    assert o.step(1) == 0
    s.step(1)
    a, b = s.particles(), o.particles()
    assert np.array_equal(a["id"], b["id"])
    i = a["id"]
    fr = lambda x: r_max ** (x / nr) if r_map == "log" else 1.0 + x * (r_max - 1.0) / nr  # noqa: E731
    r0, r1 = fr(x1[i]), fr(b["x1"])
    if r_map == "log":  # the large-argument branch of the radial move is taken
        assert np.abs((r1 / r0) ** 2 - 1).max() > 1 / 16
    # the oracle's angle has an absolute rounding of eps, which its basis
    # vectors divide by the distance from the axis, at both ends of the move
    ang = lambda x: np.arccos(np.clip(1 - 2 * x / nth, -1, 1)) if th_map == "equal_area" else np.pi * x / nth  # noqa: E731
    w = 1.0 + 1.0 / np.minimum(np.sin(ang(x2[i])), np.maximum(np.sin(ang(b["x2"])), 1e-3)) ** 2
    un = np.sqrt(b["ur"] ** 2 + b["uth"] ** 2 + b["uph"] ** 2) + np.sqrt((u[:, i] ** 2).sum(0)) + 1.0
    dxi = np.log(r_max) / nr if r_map == "log" else (r_max - 1.0) / nr
    for k, bar in (("x1", 16 * (nr + 4 / dxi) * np.ones(len(i))), ("x2", 64 * nth * w), ("ur", 64 * w * un),
                   ("uth", 64 * w * un), ("uph", 64 * w * un)):
        d = np.abs(a[k] - b[k])
        assert np.all(d <= EPS * bar), (k, float((d / (EPS * bar)).max()))
    fs, fo = s.flux(), o.flux()
    for k in range(3):
        assert np.linalg.norm(fs[k] - fo[k]) <= 1e-12 * np.linalg.norm(fo[k]), k
    Fs, Fo = s.fields(), o.fields()
    for k in range(6):
        assert np.linalg.norm(Fs[k] - Fo[k]) <= 1e-12 * max(np.linalg.norm(Fo[k]), 1.0), k
