"""The FP32 tile kernel with two particles a thread, which grids of more than
2^17 cells take: one-step replays against the oracle on every specialisation
and tile shape, and bit-for-bit agreement of its two copies (packed in the
tile's window, one particle a thread in global memory)."""
import numpy as np
import pytest

import oracle as O
from paper_1407_1810_gb300 import configs, synthetic

from gpu_common import KEYS, MAX_FP32, by_id, close, follow_ties, replay_compare_fp32, setup

pytestmark = pytest.mark.gpu
TAU = 2e-6

MONO = dict(configs.CONFIGS["monopole-64x64"], precision="fp32", r_max=40.0)
ROT = dict(configs.CONFIGS["rotator-1024x1024"], t_spin=0.05, absorb_cells=8)
CASES = {
    # just past the line, tall and wide; one and a half thousand odd tiles
    "monopole": dict(MONO, nr=514, nth=256),
    "monopole-wide": dict(MONO, nr=257, nth=513),
    "rotator": dict(ROT, nr=363, nth=362),
    # the general kernel: linear r, Boris; a coarse log grid that takes the
    # library functions; the other analytic fields
    "linear-boris": dict(MONO, nr=514, nth=256, r_map="linear", r_max=4.0, pusher="boris"),
    "linear-area": dict(MONO, nr=257, nth=512, r_map="linear", th_map="equal_area", r_max=3.0),
    "coarse": dict(MONO, nr=33, nth=3980, r_max=40.0),
    "coarse-area": dict(ROT, nr=41, nth=3200, r_max=40.0, inject=0),
    "dipole": dict(ROT, nr=363, nth=362, th_map="linear", vacuum="dipole_rotator", pusher="boris"),
    "uniform": dict(MONO, nr=514, nth=256, vacuum="uniform_bz", n_filt=1),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


def _plasma(cfg, qw, seed, T):
    """Pairs in the rows next to both conductors, next to both poles and in a
    block in between: hot, so that many cross one or both grid lines."""
    nr, nth = cfg["nr"], cfg["nth"]
    rows = [0, 1, 2, nr - 2, nr - 1]
    cells = [i * nth + j for i in rows for j in range(0, nth, max(1, nth // 200))]
    cells += [i * nth + j for i in range(0, nr, max(1, nr // 60)) for j in (0, 1, 2, nth - 2, nth - 1)]
    cells += [(nr // 3 + a) * nth + nth // 3 + b for a in range(18) for b in range(21)]
    return synthetic.pair_plasma_cells(nr, nth, np.array(cells), 7, T, qw, seed)


def _pair(cfg, seed=3, T=1.0, **over):
    p = O.params(**configs.oracle_kwargs(cfg, 0.0, 0.0))
    dt = O.oracle.courant_dt(p, cfg["courant"])
    _, qw = configs.physics(cfg, dt)
    return setup(cfg, plasma=_plasma(cfg, float(np.float32(qw)), seed, T), **over)


# (not the dipole: a hundredth of a cell from a pole its field turns a particle
# by radians a step, beyond the momentum bar with either form of the kernel)
@pytest.mark.parametrize("case", [c for c in CASES if c != "dipole"])
@pytest.mark.parametrize("tile_shape", [0, 1, 2])
def test_one_step_replay(case, tile_shape):
    if tile_shape and case not in ("monopole", "rotator", "linear-boris"):
        pytest.skip("the tile shapes are checked on one grid per specialisation")
    cfg = CASES[case]
    assert cfg["nr"] * cfg["nth"] > 1 << 17
    s, o, plasma, dt = _pair(cfg, tile_shape=tile_shape)
    s.step(3)
    st = s.particles()
    o2 = O.Oracle(o.p)
    o2.load(*(st[k] for k in KEYS), ids=st["id"])
    o2.set_fields(s.fields())
    nid = len(plasma["x1"]) + 3 * 2 * cfg.get("inject_pairs", 2) * cfg["nth"] * bool(cfg["inject"])
    o2.set_clock(3, nid)
    s.step(1)
    follow_ties(s, o2)
    o2.step(1)
    g, r = s.particles(), o2.particles()
    old = nid  # this step's injected pairs are compared by count
    g, r = ({k: v[d["id"] < old] for k, v in d.items()} for d in (g, r))
    replay_compare_fp32(g, r, TAU)
    close(s.flux(), o2.flux(), 1e-5, MAX_FP32)


def _slabs(cfg, dt, b0, rows):
    from paper_1407_1810_gb300 import picsar as P

    return P.Slabs(P.make_desc(**configs.desc_kwargs(cfg, dt, b0)), len(rows) - 1, rows)


@pytest.mark.parametrize("case,rows", [("monopole", [0, 97, 200, 514]), ("rotator", [0, 40, 210, 363]),
                                       ("coarse", [0, 12, 33]), ("dipole", [0, 150, 363]),
                                       ("linear-boris", [0, 257, 514]), ("coarse-area", [0, 20, 41])])
def test_window_and_global_copies_agree_bit_for_bit(case, rows):
    """Slabs start unbinned (the global-memory copy) and hand particles over
    unbinned; the whole-grid run steps them in their windows."""
    cfg = CASES[case]
    s, o, plasma, dt = _pair(cfg, T=0.6)
    g = _slabs(cfg, dt, s.desc.b0, rows)
    g.load(*(np.ascontiguousarray(plasma[k]) for k in KEYS))
    for n in (1, 8, 16):
        s.step(n)
        g.step(n)
        a, b = by_id(s.particles()), by_id(g.particles())
        assert np.array_equal(a["id"], b["id"])
        for k in KEYS:
            assert np.array_equal(a[k], b[k]), (n, k, int((a[k] != b[k]).sum()))
        assert np.array_equal(s.flux(), g.flux()), n
    assert np.array_equal(s.fields(), g.fields())


def test_packed_members_of_an_ensemble():
    """Members on both sides of the line step as their own runs do."""
    from paper_1407_1810_gb300 import picsar as P

    small = dict(MONO, nr=40, nth=33, pairs_per_cell=3)
    ens, ref = [], []
    for cfg in (CASES["monopole"], small, CASES["rotator"], CASES["dipole"]):
        if cfg is small:
            s1, _, plasma, _ = setup(cfg)
        else:
            s1, _, plasma, _ = _pair(cfg)
        s2, _, _, _ = setup(cfg, plasma=plasma)
        ens.append(s1)
        ref.append(s2)
    P.ensemble_step(ens, 24)
    for s in ref:
        s.step(24)
    for a, b in zip(ens, ref):
        assert np.array_equal(a.fields(), b.fields()) and np.array_equal(a.flux(), b.flux())
        pa, pb = by_id(a.particles()), by_id(b.particles())
        for k in ("id",) + KEYS:
            assert np.array_equal(pa[k], pb[k]), k


@pytest.mark.parametrize("uph,half", [(1e-9, 0.5), (-1e-9, -0.5)])
def test_axis_tie(uph, half):
    cfg = dict(configs.CONFIGS["monopole-64x64"], nr=2051, nth=64, th_map="linear", vacuum="none", precision="fp32",
               pairs_per_cell=0, absorb_cells=4)
    q = 0.37
    one = {"x1": np.array([7.3]), "x2": np.array([0.001]), "ur": np.array([0.0]), "uth": np.array([-3.0]),
           "uph": np.array([uph]), "qw": np.array([q])}
    s, o, _, _ = setup(cfg, plasma=one)
    s.step(1)
    o.step(1)
    t = s.axis_ties()
    assert list(t["step"]) == [0] and list(t["id"]) == [0] and list(t["sign"]) == [1 if half > 0 else -1]
    assert s.flux()[2].sum() / q == pytest.approx(half, abs=1e-5)
    assert s.flux()[2].sum() == pytest.approx(o.flux()[2].sum(), abs=1e-5 * q)


def test_errors_are_latched():
    """A particle that crosses more than one line is removed and reported."""
    from paper_1407_1810_gb300 import picsar as P

    d = P.make_desc(nr=514, nth=256, r_min=1.0, r_max=2.0, r_map="log", th_map="linear", dt=0.01, vacuum="none",
                    precision="fp32", pusher="vay")
    s = P.Simulation(d)
    s.load(*(np.array(a) for a in ([10.5, 20.5, 30.5], [100.5, 100.5, 100.5], [5.0, 0.01, 0.0], [0.0, 0.01, 0.0],
                                   [0.0, 0.0, 0.0], [1.0, 1.0, -1.0])))
    s.step(1)
    with pytest.raises(P.PicError) as err:
        s.moments()
    assert err.value.code == P.PIC_ECOURANT
