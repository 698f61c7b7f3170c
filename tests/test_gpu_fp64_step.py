"""One step of the FP64 path's local-frame form against the oracle's global
one, on every map, pusher and analytic field, on grids fine enough for the
series and on grids that take the library functions instead (dxi > 1/16,
nth < 32, a step of a tenth of the radius)."""
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


GRIDS = {
    "fine": dict(nr=40, nth=48, r_max=2.0, dt=0.012),
    "edge": dict(nr=12, nth=32, r_max=2.1, dt=0.02),      # dxi just below 1/16 (log), nth = 32
    "coarse": dict(nr=8, nth=31, r_max=6.0, dt=0.09),      # dxi = 0.22, the library functions
    "smallest": dict(nr=3, nth=2, r_max=1.5, dt=0.03),
}


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("r_map", ["log", "linear"])
@pytest.mark.parametrize("th_map", ["linear", "equal_area"])
@pytest.mark.parametrize("pusher", ["vay", "boris"])
def test_one_step_against_the_oracle(grid, r_map, th_map, pusher):
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    cfg = dict(GRIDS[grid], r_min=1.0, r_map=r_map, th_map=th_map, pusher=pusher, n_filt=1, absorb_cells=1,
               absorb_profile="linear", b0=20.0, omega=0.3, t_spin=0.0)
    nr, nth = cfg["nr"], cfg["nth"]
    dr = (cfg["r_max"] - 1.0) / nr
    if r_map == "linear" and 1.0 - 3 * dr <= 0.0:
        pytest.skip("the ghost rows of this linear grid would reach r <= 0")
    for q, vacuum in enumerate(VACUA):
        g = np.random.default_rng(7 * q + nr)
        n = 4000
        x1 = g.random(n) * (nr + 2.0) - 1.0  # the conductors' first rows too
        # from a hundredth of a cell off the poles on; half a cell and the node
        # lines themselves among them
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
        c = dict(cfg, vacuum=vacuum)
        s = P.Simulation(P.make_desc(**c, precision="fp64"))
        o = O.Oracle(O.params(**c))
        for x in (s, o):
            x.load(x1, x2, *(np.ascontiguousarray(a) for a in u), qw)
            x.set_fields(f)
        s.step(1)
        if o.step(1):  # a particle crossed two grid lines: the GPU latches the same error
            with pytest.raises(P.PicError) as err:
                s.particles()
            assert err.value.code == P.PIC_ECOURANT
            continue
        a, b = s.particles(), o.particles()
        assert np.array_equal(a["id"], b["id"]), vacuum
        i = a["id"]
        th = np.arccos(1 - 2 * x2 / nth) if th_map == "equal_area" else np.pi * x2 / nth
        # the oracle's angle has an absolute rounding of eps, which its basis
        # vectors divide by the distance from the axis, at the start and at
        # the end of the move
        thn = np.arccos(np.clip(1 - 2 * b["x2"] / nth, -1, 1)) if th_map == "equal_area" else np.pi * b["x2"] / nth
        w = 1.0 + 1.0 / np.minimum(np.sin(th[i]), np.maximum(np.sin(thn), 1e-3)) ** 2
        un = np.sqrt(b["ur"] ** 2 + b["uth"] ** 2 + b["uph"] ** 2) + np.sqrt((u[:, i] ** 2).sum(0)) + 1.0
        dxi = np.log(cfg["r_max"]) / nr if r_map == "log" else dr
        for k, bar in (("x1", 16 * (nr + 4 / dxi) * np.ones(len(i))), ("x2", 64 * nth * w), ("ur", 64 * w * un),
                       ("uth", 64 * w * un), ("uph", 64 * w * un)):
            d = np.abs(a[k] - b[k])
            assert np.all(d <= EPS * bar), (vacuum, k, float((d / (EPS * bar)).max()))
        fs, fo = s.flux(), o.flux()
        for k in range(3):
            den = np.linalg.norm(fo[k])
            assert np.linalg.norm(fs[k] - fo[k]) <= 1e-12 * den, (vacuum, k, np.linalg.norm(fs[k] - fo[k]) / den)


def test_particles_on_the_axis_and_at_the_far_pole():
    """x2 = 0 and x2 = nth exactly, moving off the axis and along it."""
    import oracle as O
    from paper_1407_1810_gb300 import picsar as P

    for th_map in ("linear", "equal_area"):
        c = dict(nr=20, nth=36, r_min=1.0, r_max=2.0, r_map="log", th_map=th_map, dt=0.01, n_filt=0, vacuum="none",
                 pusher="vay")
        x1 = np.full(6, 7.25)
        x2 = np.array([0.0, 0.0, 0.0, 36.0, 36.0, 36.0])
        u = [np.array([0.5, 0.0, 0.3] * 2), np.array([0.0, 0.4, 0.2] * 2), np.array([0.0, 0.0, 0.1] * 2)]
        qw = np.ones(6)
        s = P.Simulation(P.make_desc(**c, precision="fp64"))
        o = O.Oracle(O.params(**c))
        for x in (s, o):
            x.load(x1, x2, *u, qw)
        s.step(1)
        o.step(1)
        a, b = s.particles(), o.particles()
        for k in ("x1", "x2"):
            assert np.allclose(a[k], b[k], rtol=0, atol=1e-12), (th_map, k, a[k] - b[k])
        assert np.allclose(a["ur"], b["ur"], rtol=0, atol=1e-14)
        # on the axis the azimuth of u is free: its size across r is not
        assert np.allclose(np.hypot(a["uth"], a["uph"]), np.hypot(b["uth"], b["uph"]), rtol=0, atol=1e-14)
