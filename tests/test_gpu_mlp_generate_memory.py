"""Generation of many training samples: its scratch stays bounded, and rows
past a chunk's end are those of their own shapes."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CHUNK = 1 << 20
USED_MEM_HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("the GPU tests need a CUDA device")
    from paper_1908_04262_gb300 import build as B
    from paper_1908_04262_gb300 import lbf as L

    B.build()
    return L, torch


def test_scratch_is_bounded(env):
    """20 doubles a sample are what the shapes alone take; a run of three
    chunks stays below that."""
    L, torch = env
    n = 3 * CHUNK + 5
    x, y = torch.empty(n, 27, device="cuda"), torch.empty(n, device="cuda")
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    pool = ctypes.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    high = ctypes.c_uint64(0)
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    L.mlp_generate(3, x, y)
    torch.cuda.synchronize()
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    assert 0 < high.value < 160 * n
    for k in range(1, 3):  # a chunk is not the one before again
        assert not torch.equal(x[:64], x[k * CHUNK:k * CHUNK + 64])
    assert bool((y != 0).all()) and float(y.abs().max()) < 4 * 1.25 / 0.75 ** 2 / 2.0 + 1e-5


def test_shapes_past_a_chunk(env):
    L, torch = env
    rng = np.random.default_rng(2)
    m = 40
    P = np.zeros((m, 20))
    P[:, 0:3] = rng.random((m, 3))
    P[:, 3:6] = rng.uniform(3, 12, (m, 1)) * rng.uniform(0.75, 1.25, (m, 3))
    P[:, 6] = P[:, 10] = P[:, 14] = 1.0
    P[:, 15] = 1.0
    d = rng.normal(size=(m, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    P[:, 16:19] = np.floor(P[:, :3] + d / np.sqrt(np.sum((d / P[:, 3:6]) ** 2, 1))[:, None] + 0.5)
    small = torch.empty(m, 27, device="cuda"), torch.empty(m, device="cuda")
    L.mlp_stencils_from_params(P, *small)
    n = CHUNK + m - 7
    many = torch.empty(n, 27, device="cuda"), torch.empty(n, device="cuda")
    L.mlp_stencils_from_params(np.concatenate([np.repeat(P[:1], n - m, 0), P]), *many)
    for a, b in zip(small, many):
        assert torch.equal(a, b[n - m:]) and torch.equal(a[:1].expand_as(b[:5]), b[:5])
