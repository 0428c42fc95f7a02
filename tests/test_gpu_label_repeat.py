"""The union-find passes give the same labels every time: fields whose
components run through many tiles (a snake of gas one cell wide, a percolating
random field, a headspace over bubbles), labelled again and again.  Every
label against a breadth-first search on the host."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

REPEATS = 400


def links(dim):
    r = (-1, 0, 1)
    e = [(x, y, z) for z in (r if dim == 3 else (0,)) for y in r for x in r]
    return [v for v in e if 0 < sum(abs(c) for c in v) <= 2]


def labels_by_search(types):
    """Gas components over the lattice links (periodic), numbered by their
    smallest cell; interface cells take the smallest number next to them."""
    nz, ny, nx = types.shape
    dim = 2 if nz == 1 else 3
    flat = types.reshape(-1)
    idx = np.arange(flat.size).reshape(types.shape)
    # [k][n]: the neighbours of every cell
    nb = np.stack([np.roll(idx, (-z, -y, -x), (0, 1, 2)).reshape(-1) for x, y, z in links(dim)])
    gas = flat == 0
    seen = np.zeros(flat.size, bool)
    comp = np.full(flat.size, -1)
    count = 0
    for n in np.flatnonzero(gas):
        if seen[n]:
            continue
        front = np.array([n])
        seen[n] = True
        while front.size:
            comp[front] = count
            nxt = np.unique(nb[:, front])
            nxt = nxt[gas[nxt] & ~seen[nxt]]
            seen[nxt] = True
            front = nxt
        count += 1
    around = np.where(comp[nb] >= 0, comp[nb], count).min(0)
    return np.where(flat == 2, np.where(around < count, around, -1), comp).astype(np.int32), count


def snake(nx, ny, nz):
    """One path through the whole lattice: rows along x, joined at alternate
    ends, layers joined at a corner."""
    t = np.full((nz, ny, nx), 1, np.uint8)
    for z in range(1, nz - 1, 3) if nz > 1 else [0]:
        for j, y in enumerate(range(1, ny - 1, 3)):
            t[z, y, 1:nx - 1] = 0
            if y + 3 < ny - 1:
                t[z, y:y + 4, nx - 2 if j % 2 == 0 else 1] = 0
        if z + 3 < nz - 1:
            t[z:z + 4, 1, 1] = 0
    return t


def random_field(nx, ny, nz, p, seed):
    r = np.random.default_rng(seed).random((nz, ny, nx))
    return np.where(r < p, 0, np.where(r < p + 0.2, 2, 1)).astype(np.uint8)


def headspace(nx, ny, nz, seed):
    rng = np.random.default_rng(seed)
    t = np.full((nz, ny, nx), 1, np.uint8)
    x, y, z = np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij")
    up = (y if nz == 1 else z).T
    for _ in range(30):
        c = rng.random(3) * (nx, ny, nz)
        d = np.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2 * (nz > 1)).T
        t[(d < 5) & (t == 1)] = 2
        t[d < 4] = 0
    top = 0.6 * (ny if nz == 1 else nz)
    t[up > top] = 0
    t[(up > top - 1) & (up <= top) & (t == 1)] = 2
    return t


CASES = [lambda: snake(101, 60, 40), lambda: snake(700, 90, 1), lambda: random_field(97, 64, 50, 0.16, 1),
         lambda: random_field(679, 54, 1, 0.42, 2), lambda: headspace(679, 54, 1, 3), lambda: headspace(96, 80, 60, 4)]


@pytest.mark.parametrize("case", CASES, ids=["snake3d", "snake2d", "random3d", "random2d", "headspace2d", "headspace3d"])
def test_labels_are_the_same_every_time(case):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1908_04262_gb300 import build as B
    from paper_1908_04262_gb300 import lbf

    B.build()
    t = case()
    nz, ny, nx = t.shape
    want, n = labels_by_search(t)
    assert n <= 4096
    want = torch.tensor(want, device="cuda")
    types = torch.tensor(t.reshape(-1), device="cuda")
    labels = torch.empty(t.size, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(REPEATS):
        labels.fill_(-7)
        lbf.label_gas_noalloc(types, nx, ny, nz, labels, count)
        wrong += (labels != want).sum() + (count[0] != n)
    assert wrong.item() == 0
