"""The two-particles-a-thread form of the FP32 tile kernel (grids of more than
2^17 cells) on plasmas of well under a particle a cell, which amplify rounding
most, against the FP64 path; and its one-step replay of a dipole's plasma away
from the poles."""
import numpy as np
import pytest

import oracle as O
from paper_1407_1810_gb300 import configs, synthetic

from gpu_common import KEYS, MAX_FP32, by_id, close, follow_ties, rel_l2, replay_compare_fp32, setup

pytestmark = pytest.mark.gpu

MONO = dict(configs.CONFIGS["monopole-64x64"], precision="fp32", T=0.3)
ROT = dict(configs.CONFIGS["rotator-1024x1024"], r_max=10.0, t_spin=0.05, absorb_cells=8)
DIP = dict(ROT, th_map="linear", vacuum="dipole_rotator", pusher="boris", wc_dt=1.0)
CASES = {
    "monopole": dict(MONO, nr=363, nth=362),
    "monopole-tall": dict(MONO, nr=514, nth=256),
    "rotator": dict(ROT, nr=363, nth=362),
    "dipole": dict(DIP, nr=363, nth=362, inject=0),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_1810_gb300 import build

    build.build()
    O.build_oracle()


def _plasma(cfg, cells, per_cell, seed):
    p = O.params(**configs.oracle_kwargs(cfg, 0.0, 0.0))
    dt = O.oracle.courant_dt(p, cfg["courant"])
    _, qw = configs.physics(dict(cfg, pairs_per_cell=1), dt)
    return synthetic.pair_plasma_cells(cfg["nr"], cfg["nth"], cells, per_cell, cfg["T"], float(np.float32(qw)), seed)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("seed", [0, 1])
def test_sparse_plasma_against_the_fp64_path(case, seed):
    """40 steps: the FP32 path's bar on the fields (1e-5, relative L2), and a
    typical particle within a few roundings of 2^-24 a step, random in sign."""
    cfg = CASES[case]
    n = cfg["nr"] * cfg["nth"]
    assert n > 1 << 17
    cells = np.random.default_rng(seed).choice(n, 10000, replace=False)
    pl = _plasma(cfg, np.sort(cells), 1, seed)
    a, _, pl, _ = setup(cfg, plasma=pl)
    b, _, _, _ = setup(cfg, plasma=pl, precision="fp64")
    a.step(40)
    follow_ties(a, b)
    b.step(40)
    assert rel_l2(a.fields(), b.fields()) < 1e-5
    p, q = by_id(a.particles()), by_id(b.particles())
    _, i, j = np.intersect1d(p["id"], q["id"], return_indices=True)
    assert len(i) >= 0.999 * max(len(p["id"]), len(q["id"]))
    um = np.sqrt(sum(q[k][j] ** 2 for k in ("ur", "uth", "uph"))) + 1e-2
    du = np.sqrt(sum((p[k][i] - q[k][j]) ** 2 for k in ("ur", "uth", "uph"))) / um
    dx = np.hypot(p["x1"][i] - q["x1"][j], p["x2"][i] - q["x2"][j])
    bar = 4 * np.sqrt(40) * 2.0 ** -24
    assert np.median(du) < bar, np.median(du)
    assert np.median(dx) < 2 * bar, np.median(dx)


@pytest.mark.parametrize("tile_shape", [0, 1, 2])
def test_dipole_replay_off_the_poles(tile_shape):
    """Particles from the tenth cell off the poles on: nearer, the dipole turns
    one by radians a step, in either form of the kernel."""
    cfg = dict(DIP, nr=363, nth=362, inject=0, T=1.0, r_max=40.0)
    nr, nth = cfg["nr"], cfg["nth"]
    rows = [0, 1, 2, 100, 101, 200, nr - 2, nr - 1]
    cells = np.array([i * nth + j for i in rows for j in range(10, nth - 10, 2)] +
                     [(nr // 3 + a) * nth + nth // 3 + b for a in range(18) for b in range(21)])
    s, o, plasma, _ = setup(cfg, plasma=_plasma(cfg, cells, 5, 4), tile_shape=tile_shape)
    s.step(3)
    st = s.particles()
    o2 = O.Oracle(o.p)
    o2.load(*(st[k] for k in KEYS), ids=st["id"])
    o2.set_fields(s.fields())
    o2.set_clock(3, len(plasma["x1"]))
    s.step(1)
    follow_ties(s, o2)
    o2.step(1)
    replay_compare_fp32(s.particles(), o2.particles(), 2e-6)
    close(s.flux(), o2.flux(), 1e-5, MAX_FP32)
