"""The TV prox's two forms agree bit for bit: pairs of iterations in one launch (16-byte aligned images) and
one iteration per launch (anything else), on grids that exercise the pair kernel's tiles (lines of 8 voxels up
to split lines of 256, fewer rows than a tile, runs of one plane, batches), odd and even iteration counts, out
of place and in place; and an infinite voxel does not spread further than the iterations reach."""
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


@pytest.mark.parametrize("shape,batch", [((8, 8, 8), 1), ((16, 32, 8), 2), ((32, 32, 32), 1), ((64, 128, 128), 1),
                                         ((8, 64, 256), 2), ((256, 16, 64), 1), ((16, 8, 128), 3)])
def test_pairs_equal_single_iterations(dev, shape, batch):
    op = PatOperator(presets.Grid(*shape, T=2, pml_size=2, batch=batch), presets.Sampling())
    g = torch.Generator(device=dev).manual_seed(sum(shape))
    x = torch.rand(op.image_shape, generator=g, device=dev)
    u = torch.empty(x.numel() + 1, device=dev)[1:].view(op.image_shape).copy_(x)  # 4 bytes past an aligned address
    for alpha in (0.01, 0.4, 2e-15):
        for iters in (1, 2, 3, 4, 9, 16):
            a = op.tv_prox(x, alpha, iters)
            assert torch.equal(a, op.tv_prox(u, alpha, iters)), (alpha, iters)
            y = x.clone()
            assert torch.equal(a, op.tv_prox(y, alpha, iters, out=y)), (alpha, iters)


def test_infinite_input_stays_local(dev):
    """One iteration reaches one voxel: an infinite voxel (whose dual is then undefined) leaves the rest alone."""
    op = PatOperator(presets.Grid(16, 16, 16, T=2, pml_size=2), presets.Sampling())
    x = torch.rand(op.image_shape, device=dev)
    x[0, 8, 8, 8] = float("inf")
    out = op.tv_prox(x, 0.1, 2)
    x[0, 8, 8, 8] = 0.5
    near = op.tv_prox(x, 0.1, 2)
    assert torch.equal(out[0, :5], near[0, :5]) and torch.equal(out[0, 12:], near[0, 12:])
    assert bool(torch.isfinite(near).all())
