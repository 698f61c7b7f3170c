"""The fused grid kernels: the flux filter in one pass (64- and 128-bit
integers on the FP32 path, FP64 sums on the FP64 path, pass by pass above four
passes) and the B update that keeps the half-step field.
"""
import numpy as np
import pytest

from gpu_common import KEYS, setup  # noqa: F401

pytestmark = pytest.mark.gpu

BASE = dict(r_min=1.0, r_max=3.0, r_map="log", th_map="equal_area", absorb_cells=3, absorb_profile="linear",
            vacuum="monopole", b0=5.0, omega=0.0, t_spin=0.0, dt=0.004)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle as O
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


def _plasma(nr, nth, n, seed, dense=0):
    """FP32-representable particles over the whole grid (poles and both
    conductors' rows included), `dense` more in one polar cell, all moving
    outwards with the same sign."""
    g = np.random.default_rng(seed)
    f = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    x1 = g.integers(0, nr, n) + f(g.random(n))
    x2 = g.integers(0, nth, n) + f(g.random(n))
    u = f(g.normal(size=(3, n)) * 0.8)
    q = np.where(np.arange(n) % 2, 1.0, -1.0)
    if dense:
        x1 = np.concatenate([x1, 2 + f(0.3 + 0.1 * g.random(dense))])
        x2 = np.concatenate([x2, f(0.05 + 0.2 * g.random(dense))])
        u = np.concatenate([u, np.repeat(np.array([[3.0], [0.5], [0.25]]), dense, 1)], 1)
        q = np.concatenate([q, np.ones(dense)])
    return [np.ascontiguousarray(a) for a in (x1, x2, u[0], u[1], u[2], q)]


def _sim(nr, nth, n_filt, precision, plasma, **over):
    from paper_1407_1810_gb300 import picsar as P

    s = P.Simulation(P.make_desc(**dict(BASE, nr=nr, nth=nth, n_filt=n_filt, precision=precision, **over)))
    s.load(*plasma)
    return s


# sizes around the 32 x 8 tiles and the smallest grids; dense: sums beyond what
# 64 bits hold with the weights of three and four passes
@pytest.mark.parametrize("n_filt", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("nr,nth,dense", [(8, 2, 0), (9, 31, 0), (20, 33, 60000), (23, 64, 0)])
def test_fp32_filter_equals_the_passes_on_the_exact_deposit(n_filt, nr, nth, dense):
    """The deposit of one step does not depend on the filter: the filtered
    fluxes are the oracle's filter passes applied to the unfiltered run's, to
    the FP64 rounding of those passes (9 terms a pass, each with one rounding
    of the product and one of the sum, of values below the largest |F|)."""
    import oracle as O

    plasma = _plasma(nr, nth, 3000, seed=nr + nth, dense=dense)
    raw = _sim(nr, nth, 0, "fp32", plasma)
    raw.step(1)
    s = _sim(nr, nth, n_filt, "fp32", plasma)
    s.step(1)
    F0, F = raw.flux(), s.flux()
    o = O.Oracle(O.params(**dict(BASE, nr=nr, nth=nth, n_filt=n_filt)))
    bound = n_filt * 18 * 2.0 ** -53
    for k in range(3):
        a = np.zeros(F.shape[1:])
        a[n_filt:-n_filt] = F0[k]  # the ghost band is n_filt rows wider on each side
        for _ in range(n_filt):
            a = o.filter_pass(a, 1 if k == 1 else 0, -1 if k == 1 else 1)
        d = np.abs(F[k] - a)[:, : nth if k == 1 else nth + 1]
        assert d.max() <= bound * np.abs(F0[k]).max(), (k, d.max() / np.abs(F0[k]).max())


@pytest.mark.parametrize("n_filt", [0, 1, 4, 5, 6])
@pytest.mark.parametrize("nr,nth", [(9, 31), (20, 33)])
def test_fp64_steps_against_the_oracle(n_filt, nr, nth):
    import oracle as O

    plasma = _plasma(nr, nth, 2000, seed=nr * nth)
    s = _sim(nr, nth, n_filt, "fp64", plasma)
    o = O.Oracle(O.params(**dict(BASE, nr=nr, nth=nth, n_filt=n_filt)))
    o.load(*plasma)
    s.step(6)
    o.step(6)
    for a, b in ((s.fields(), o.fields()), (s.flux(), o.flux())):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_replaced_fields_restart_the_half_step(precision):
    """pic_set_fields between steps: the next step is that of a fresh context
    given the same fields and particles."""
    plasma = _plasma(20, 33, 2000, seed=4)
    a = _sim(20, 33, 2, precision, plasma)
    a.step(3)
    f = a.fields() * 1.25
    p = a.particles()
    b = _sim(20, 33, 2, precision, [p[k] for k in KEYS])
    for s in (a, b):
        s.set_fields(f)
        assert np.array_equal(s.fields(), f)
    a.step(2)
    b.step(2)
    fa, fb = a.fields(), b.fields()
    if precision == "fp32":
        assert np.array_equal(fa, fb)
    else:
        assert np.linalg.norm(fa - fb) <= 1e-13 * np.linalg.norm(fb)


def test_ensemble_members_with_any_number_of_filter_passes():
    from paper_1407_1810_gb300 import picsar as P

    ens, ref = [], []
    for k, n_filt in enumerate((0, 1, 3, 4, 5, 6)):
        plasma = _plasma(20 + k, 31 + k, 1500, seed=k)
        ens.append(_sim(20 + k, 31 + k, n_filt, "fp32", plasma))
        ref.append(_sim(20 + k, 31 + k, n_filt, "fp32", plasma))
    P.ensemble_step(ens, 25)
    for s in ref:
        s.step(25)
    for a, b in zip(ens, ref):
        assert np.array_equal(a.fields(), b.fields()) and np.array_equal(a.flux(), b.flux())
