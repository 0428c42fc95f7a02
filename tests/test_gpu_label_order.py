"""Bubble numbers while the roots of many bubbles move past one another: the
step keeps the labels of cells and renumbers the bubbles by the order of
their roots (their smallest cell indices).  FP64 runs of many small bubbles
at nearly one height against the oracle, step by step: flags, labels, ids
and roots exact, volumes within 1e-10 (the bound of the other FP64 parity
cases); the order of the bubbles changes on the way, and a checkpoint taken
after it has changed resumes the run."""
import numpy as np
import pytest

from paper_1908_04262_gb300 import workloads as W
from tests._parity import rel_err

pytestmark = pytest.mark.gpu

# (nx, ny, nz), walls on every face, steps
CASES = [((45, 37, 22), True, 30), ((33, 40, 19), False, 24), ((97, 64, 1), True, 60), ((70, 41, 1), False, 60)]


def setup(shape, walled):
    nx, ny, nz = shape
    flat = nz == 1
    n_up = ny if flat else nz
    cfg = W.config(nx=nx, ny=ny, nz=nz, storage="fp64", tau=0.7, sigma=5e-3, d_max=3.0, k_pi=1e-3 / 3.0, D=0.05,
                   kH=0.3, c0=1.0, RT=0.15, accel=(2e-4, -1e-4, 0.0), walls=(0xF if flat else 0x3F) if walled else 0,
                   fill_height=n_up - 5.0 if walled else 1e9, atmosphere=int(walled))
    rng = np.random.default_rng(7)
    step = 8.0
    pts = [(x, y) for x in np.arange(6.0, nx - 5.0, step) for y in ([0.0] if flat else np.arange(6.0, ny - 5.0, step))]
    r = rng.uniform(2.0, 2.9, len(pts))
    low = 8.0 if walled else (12.0 if flat else 0.0)  # 3D periodic: bubbles lie across the lowest face
    c = [[x + rng.uniform(-0.4, 0.4), (low if flat else y) + rng.uniform(-0.4, 0.4),
          0.0 if flat else low + rng.uniform(-0.4, 0.4)] for x, y in pts]
    return cfg, np.array(c), r


@pytest.mark.parametrize("shape,walled,steps", CASES)
def test_numbers_follow_the_roots(oracle_mod, shape, walled, steps):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1908_04262_gb300 import build as B
    from paper_1908_04262_gb300 import lbf

    B.build()
    cfg, c, r = setup(shape, walled)
    sim, ora = lbf.Sim(cfg), oracle_mod.OracleSim(cfg)
    for s in (sim, ora):
        s.nucleate(c, r)
    saved, reordered = None, False
    for k in range(0, steps, 2):
        sim.step(2)
        ora.step(2)
        got, bg, bo = sim.fields(["flags", "label"]), sim.bubbles(), ora.bubbles()
        assert np.array_equal(got["flags"], ora.types()), k
        assert np.array_equal(got["label"], ora.labels()), k
        for name in ("id", "atm", "root"):
            assert np.array_equal(bg[name], bo[name]), (k, name)
        assert rel_err(bg["volume"], bo["volume"]) < 1e-10
        assert rel_err(bg["pressure"], bo["pressure"]) < 1e-10
        reordered |= not np.all(np.diff(bo["id"][bo["atm"] == 0]) > 0)
        if reordered and saved is None:
            saved = sim.checkpoint()
            fresh = lbf.Sim(cfg)
            fresh.restore(saved)
            assert np.array_equal(fresh.fields(["label"])["label"], ora.labels())
    assert reordered
    fresh.step(sim.step_count() - fresh.step_count())
    bf = fresh.bubbles()
    assert np.array_equal(fresh.fields(["label"])["label"], ora.labels())
    for name in ("id", "root"):
        assert np.array_equal(bf[name], bo[name])
    assert rel_err(bf["volume"], bo["volume"]) < 1e-10


def test_touching_bubbles_pool_their_gas():
    """Two bubbles behind one layer of interface cells (32^3, FP64): when
    their roots pass one another those cells go from one bubble to the other,
    so that old and new bubbles share cells and pool their gas; the larger
    keeps the smaller id, the other gets a fresh one.  Ids and pressures are
    those of the library whose labels were the ranks of the roots, where a
    change of order always took the full labelling."""
    import torch

    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1908_04262_gb300 import build as B
    from paper_1908_04262_gb300 import lbf

    B.build()
    cfg, c, _ = W.c2_crop_3d_32(storage="fp64")
    sim = lbf.Sim(cfg)
    sim.nucleate(np.concatenate([c, [[22.0, 20.0, 9.0]]]), [5.0, 3.0])
    sim.step(21)
    b = sim.bubbles()
    assert b["id"].tolist() == [1, 3, 0] and b["root"].tolist() == [7696, 7797, 25633]
    assert rel_err(b["pressure"], [0.33273405295113834, 0.3361376202527489, 1 / 3]) < 1e-10
    sim.step(9)
    b = sim.bubbles()
    assert b["id"].tolist() == [4, 1, 0] and b["root"].tolist() == [7797, 8655, 25633]
    assert rel_err(b["pressure"], [0.3356138194055036, 0.33639008142017535, 1 / 3]) < 1e-10
