"""Interface sweep and mass exchange over segment lists long enough to be
packed (longer than the grid's warps, for the single-precision and 16-bit
sweeps by a third: 2,433 and 3,243 segments on 152 SMs, 9,729 for the
exchange), and on a lattice that could list that many but does not: a lattice
made of copies of a small one, periodic or a closed box, against the small one,
whose list is walked segment by segment.  Rows end in a partial segment.  Bubbles add up their
volumes in any order, which moves pressures by FP64 rounding: FP64 within
1e-11, the other forms within a few units of their last place."""
import numpy as np
import pytest

from paper_1908_04262_gb300 import workloads as W
from tests._parity import rel_err

pytestmark = pytest.mark.gpu

SMALL = (35, 20, 15)
NAMES = ("rho", "u", "alpha", "mass", "conc", "kappa")


def box(walled):
    """Bubbles of radius 1.8 on a jittered cubic lattice of spacing 5: in
    nearly every row."""
    nx, ny, nz = SMALL
    rng = np.random.default_rng(17)
    g = np.stack(np.meshgrid(*(np.arange(2.0, n - 2.0, 5.0) for n in SMALL), indexing="ij"), -1).reshape(-1, 3)
    t, a = W.voxel_spheres(SMALL, g + rng.uniform(-0.3, 0.3, g.shape), rng.uniform(1.7, 1.9, len(g)), sub=3)
    t = t.reshape(nz, ny, nx)
    if walled:
        for face in (np.s_[0], np.s_[-1], np.s_[:, 0], np.s_[:, -1], np.s_[:, :, 0], np.s_[:, :, -1]):
            t[face] = 3
    N = nx * ny * nz
    u = 0.02 * (rng.random((N, 3)) - 0.5)
    return t.reshape(-1), 1.0 + 0.01 * rng.random(N), u, a, 0.1 * rng.random(N)


def copies(v, r):
    """A field of the small lattice repeated r times along x, y and z."""
    nx, ny, nz = SMALL
    v = np.asarray(v)
    w = v.reshape((nz, ny, nx) + v.shape[1:])
    return np.tile(w, (r[2], r[1], r[0]) + (1,) * (v.ndim - 1)).reshape((-1,) + v.shape[1:])


def listed(types, nx):
    t = types.reshape(-1, nx)
    return sum(int((t[:, x0:x0 + 32] == 2).any(-1).sum()) for x0 in range(0, nx, 32))


@pytest.mark.parametrize("collision", [0, 1])
@pytest.mark.parametrize("storage,tol", [("fp64", 1e-11), ("fp32", 1e-6), ("fp16s", 2e-3)])
@pytest.mark.parametrize("walled,r", [(True, (1, 5, 7)), (False, (1, 5, 7)), (True, (1, 2, 3))])
def test_long_lists_match_short_ones(storage, tol, walled, collision, r):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1908_04262_gb300 import build as B
    from paper_1908_04262_gb300 import lbf

    B.build()
    cfg = W.config(storage=storage, walls=0x3F if walled else 0, atmosphere=0, tau=0.8, sigma=5e-3, kH=0.1, D=0.05,
                   c0=0.1, RT=0.2, collision=collision)
    state = box(walled)
    small, large = (lbf.Sim(dict(cfg, nx=SMALL[0] * q[0], ny=SMALL[1] * q[1], nz=SMALL[2] * q[2]))
                    for q in ((1, 1, 1), r))
    small.set_cells(*state)
    large.set_cells(*[copies(v, r) for v in state])
    warps = 16 * torch.cuda.get_device_properties(0).multi_processor_count  # the sweep's; the exchange has four times as many
    for k in range(3):
        a, b = small.fields(NAMES + ("flags",)), large.fields(NAMES + ("flags",))
        assert np.array_equal(copies(a["flags"], r), b["flags"]), k
        for name in NAMES:
            assert rel_err(b[name], copies(a[name], r)) < tol, (k, name)
        assert listed(a["flags"], SMALL[0]) < warps
        n = listed(b["flags"], SMALL[0])
        if r == (1, 5, 7):
            assert 3 * n >= 4 * 4 * warps
        else:
            assert 3 * n < 4 * warps <= 3 * 2 * 20 * 15 * 6
        small.step(2)
        large.step(2)
