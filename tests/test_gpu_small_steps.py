"""Small grids do a time step in one launch, their spectrum in three parts, where the workspace limit leaves room for
the parts; elsewhere the three line passes run one after another.  Both give the same bits: over the line lengths (also
mixed), partly filled tiles, batches, one to a few steps, both kernels, and in the library's own scratch."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1605_00133_gb300 import _lib, presets  # noqa: E402
from paper_1605_00133_gb300.operators import PatOperator  # noqa: E402


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def sequential(grid, sampling):
    """The operator under the smallest workspace limit that admits it: without room for the parts."""
    L = _lib.load()
    lo, hi = 0, 1 << 30  # refused, admitted
    try:
        while hi - lo > 1:
            mid = (lo + hi) // 2
            L.pat_set_workspace_limit(mid)
            try:
                PatOperator(grid, sampling).close()
                hi = mid
            except Exception as e:  # noqa: BLE001
                assert "limit" in str(e)
                lo = mid
        L.pat_set_workspace_limit(hi)
        return PatOperator(grid, sampling)
    finally:
        L.pat_set_workspace_limit(0)


@pytest.mark.parametrize("shape,T,batch,m", [
    ((8, 8, 8), 2, 1, 0), ((16, 32, 8), 3, 2, 70), ((32, 32, 32), 12, 1, 200), ((8, 16, 256), 5, 1, 0),
    ((128, 16, 64), 4, 3, 0), ((64, 64, 64), 6, 1, 500), ((16, 128, 128), 5, 1, 900), ((256, 32, 32), 4, 1, 0),
    ((32, 128, 128), 4, 1, 0), ((64, 64, 64), 4, 3, 300), ((16, 16, 16), 1, 1, 0)])
def test_one_launch_equals_three(dev, shape, T, batch, m):
    g = presets.Grid(*shape, T=T, pml_size=2, batch=batch)
    s = presets.make_sampling(g, 1, m, 0) if m else presets.Sampling()
    a, b = PatOperator(g, s), sequential(g, s)
    assert T == 1 or a.workspace_bytes > b.workspace_bytes or m  # (with samples the parts may fit in their series)
    r = torch.Generator(device=dev).manual_seed(T)
    p0 = torch.randn(a.image_shape, generator=r, device=dev)
    f = a.forward(p0)
    assert torch.equal(f, b.forward(p0))
    d = torch.randn(f.shape, generator=r, device=dev)
    assert torch.equal(a.adjoint(d), b.adjoint(d))
    assert torch.equal(f, a.forward(p0))
    e = torch.full_like(f, float("nan"))
    st = _lib.load().pat_forward_noalloc(a._h, ctypes.c_void_p(p0.data_ptr()), ctypes.c_void_p(e.data_ptr()),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st != 0 or torch.equal(f, e)
