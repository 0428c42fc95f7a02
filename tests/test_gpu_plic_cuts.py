"""FP64 plane cuts over the whole range of normals and fill levels: the
exported offset of a cell against the exact inverse of the cut volume
(80-digit arithmetic) for the exported normal and fill level.  Smallest normal
components from 1e-10 to 1e-1, one or two of them small, and gas fractions at
and next to the bounds of the piecewise polynomial's branches.

The bound: with u = 2^-53 the normalised components carry at most 4 u each,
every branch amplifies that by less than 4 and adds at most 8 u of its own,
the components add up to at most sqrt(3), and scaling back adds 3 u: 45 u in
all; 64 u are allowed."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_1908_04262_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NB = 11  # blocks of 3 x 3 x 3 cells along each axis, one cut in each centre


def exact_offset(n, alpha):
    getcontext().prec = 80
    m = sorted(Decimal(abs(float(v))) for v in n)
    total = sum(m)
    m1, m2, m3 = (v / total for v in m)
    V = 1.0 - float(alpha)
    flip = V > 0.5
    V = Decimal(1.0 - V if flip else V)
    corners = [(1, Decimal(0)), (-1, m1), (-1, m2), (-1, m3), (1, m1 + m2), (1, m1 + m3), (1, m2 + m3)]
    six = 6 * m1 * m2 * m3
    lo, hi = Decimal(0), Decimal("0.5")
    for _ in range(90):  # 2^-91 is far below the bound
        a = (lo + hi) / 2
        if sum(s * (a - c) ** 3 for s, c in corners if a > c) < V * six:
            lo = a
        else:
            hi = a
    a = (lo + hi) / 2
    if flip:
        a = 1 - a
    return a * total - total / 2


def blocks(rng):
    """Gradients and gas fractions of the blocks' centres."""
    n = NB ** 3
    m = rng.uniform(0.05, 1.0, (n, 3))
    kind = np.arange(n) % 4
    m[kind == 1, 0] = 10.0 ** rng.uniform(-10, -1, (kind == 1).sum())
    m[kind == 2, :2] = 10.0 ** rng.uniform(-5, -0.5, ((kind == 2).sum(), 2))
    m[kind == 2, 2] = 1.0
    k3 = kind == 3  # the largest component near the sum of the others
    m[k3, 2] = m[k3, 0] + m[k3, 1] + rng.choice([-1, 1], k3.sum()) * 10.0 ** rng.uniform(-14, -1, k3.sum())
    m = np.abs(m)
    for row in m:
        rng.shuffle(row)
    g = 0.15 * m / m.max(1)[:, None] * rng.choice([-1.0, 1.0], m.shape)
    s = np.sort(np.abs(g), axis=1) / np.abs(g).sum(1)[:, None]
    m1, m2, m3 = s.T
    m12 = m1 + m2
    V2 = m1 * m1 / (6 * m2 * m3) + (m2 - m1) / (2 * m3)
    V3 = np.where(m3 < m12, (m3 * m3 * (3 * m12 - m3) + m1 * m1 * (m1 - 3 * m3) + m2 * m2 * (m2 - 3 * m3))
                  / (6 * m1 * m2 * m3), m12 / (2 * m3))
    V3 = np.clip(V3, V2, 0.5)
    near = rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-16, -3, n)
    pick = rng.integers(0, 4, n)
    V = np.select([pick == 0, pick == 1, pick == 2], [V2 + near, V3 + near, V2 + rng.random(n) * (V3 - V2)],
                  rng.uniform(0.01, 0.5, n))
    V = np.clip(V, 1e-9, 0.5)
    return g, np.where(rng.random(n) < 0.5, V, 1.0 - V), (V > V2) & ((V < V3) | (m3 < m12))


def test_cut_offsets_are_exact():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1908_04262_gb300 import build as B
    from paper_1908_04262_gb300 import lbf

    B.build()
    g, gas, cubic = blocks(np.random.default_rng(41))
    assert cubic.sum() > 400
    L = 3 * NB
    alpha = np.zeros((L, L, L))
    d = np.arange(3) - 1.0
    block = (0.5 + g[:, 2, None, None, None] * d[:, None, None] + g[:, 1, None, None, None] * d[:, None]
             + g[:, 0, None, None, None] * d)
    block[:, 1, 1, 1] = 1.0 - gas
    alpha = block.reshape(NB, NB, NB, 3, 3, 3).transpose(0, 3, 1, 4, 2, 5).reshape(-1)
    N = L ** 3
    sim = lbf.Sim(W.config(nx=L, ny=L, nz=L, storage="fp64", walls=0, atmosphere=0))
    sim.set_cells(np.full(N, 2, np.uint8), np.ones(N), np.zeros((N, 3)), alpha, np.zeros(N))
    f = sim.fields(["normal", "dstar", "alpha"])
    assert np.array_equal(f["alpha"], alpha)
    centre = np.arange(N).reshape(L, L, L)[1::3, 1::3, 1::3].reshape(-1)
    err = [abs(Decimal(float(f["dstar"][c])) - exact_offset(f["normal"][c], alpha[c])) for c in centre]
    assert max(float(e) for e in err) < 64 * 2.0 ** -53
