"""C and C^T for every plane size the pattern transform is instantiated for, and the single-point
kernels over chunk edges, on integer planes (every sum is exact in FP32, so equality is required),
also from a plane series that is not 16-byte aligned."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1605_00133_gb300 import presets  # noqa: E402
from paper_1605_00133_gb300.operators import PatOperator  # noqa: E402


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def fwht(v):
    n, h = v.shape[-1], 1
    while h < n:
        w = v.reshape(*v.shape[:-1], n // (2 * h), 2, h)
        v = np.stack([w[..., 0, :] + w[..., 1, :], w[..., 0, :] - w[..., 1, :]], axis=-2).reshape(v.shape)
        h *= 2
    return v


def shifted(a, dev, off):
    """a on the GPU, starting off floats past an aligned address"""
    buf = torch.zeros(a.size + off, dtype=torch.float32, device=dev)
    buf[off:] = torch.tensor(a.ravel(), dtype=torch.float32)
    return buf[off:].reshape(a.shape)


PLANES = [(8, 8), (8, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 256)]


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("ny,nx", PLANES)
def test_patterns_of_every_plane_size(dev, ny, nx, off):
    M, nt = ny * nx, 3
    rng = np.random.default_rng(M + off)
    for m in (1, M // 3, M):
        s = presets.make_sampling(presets.Grid(8, ny, nx), presets.KIND_SHD01, m, 5)
        with PatOperator(presets.Grid(8, ny, nx, T=4, pml_size=2), s) as op:
            pbar = rng.integers(-8, 9, (1, nt, M)).astype(np.float64)
            w = fwht(pbar[..., s.perm])
            got = op.sample(shifted(pbar, dev, off)).double().cpu().numpy()
            assert np.array_equal(got, 0.5 * (w[..., :1] + w[..., s.rows]))
            y = rng.integers(-8, 9, (1, nt, m)).astype(np.float64)
            e = np.zeros((1, nt, M))
            e[..., s.rows] = y
            ref = np.empty_like(e)
            ref[..., s.perm] = 0.5 * (y.sum(-1, keepdims=True) + fwht(e))
            assert np.array_equal(op.sample_adjoint(shifted(y, dev, off)).double().cpu().numpy(), ref)


@pytest.mark.parametrize("ny,nx,m", [(8, 8, 1), (8, 8, 64), (64, 64, 2048), (64, 64, 2049), (256, 256, 65536),
                                     (256, 256, 4097)])
def test_points_over_chunk_edges(dev, ny, nx, m):
    M = ny * nx
    s = presets.make_sampling(presets.Grid(8, ny, nx), presets.KIND_RSP, m, 9)
    rng = np.random.default_rng(m)
    with PatOperator(presets.Grid(8, ny, nx, T=4, pml_size=2, batch=2), s) as op:
        pbar = rng.standard_normal((2, 3, M)).astype(np.float32)
        assert np.array_equal(op.sample(shifted(pbar, dev, 1)).cpu().numpy(), pbar[..., s.indices])
        y = rng.standard_normal((2, 3, m)).astype(np.float32)
        ref = np.zeros((2, 3, M), np.float32)
        ref[..., s.indices] = y
        assert np.array_equal(op.sample_adjoint(shifted(y, dev, 1)).cpu().numpy(), ref)
