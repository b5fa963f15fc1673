"""The TV prox's two forms (test_gpu_prox_tiles.py) agree bit for bit on values of every size that FP32 has: images
scaled down until they are subnormal, images whose voxels spread over all exponents, and a point source, whose front
decays through the subnormals as it spreads into the zeros around it."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1605_00133_gb300 import presets  # noqa: E402
from paper_1605_00133_gb300.operators import PatOperator  # noqa: E402


@pytest.mark.parametrize("shape", [(16, 32, 32), (8, 16, 256)])
@pytest.mark.parametrize("what", [2.0 ** -96, 2.0 ** -104, 2.0 ** -120, 2.0 ** -130, 2.0 ** -140, "spread", "point", "large"])
def test_forms_agree(shape, what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    dev = torch.device("cuda", 0)
    op = PatOperator(presets.Grid(*shape, T=2, pml_size=2), presets.Sampling())
    g = torch.Generator(device=dev).manual_seed(1)
    x = torch.rand(op.image_shape, generator=g, device=dev)
    if what == "spread":
        x = (x + 0.5) * 2.0 ** torch.randint(-149, 60, x.shape, generator=g, device=dev)
    elif what == "large":
        x = x * 2.0 ** 60
    elif what == "point":
        x = torch.zeros_like(x)
        x[0, 2, 5, 7] = 1.0
    else:
        x = (x.double() * what).float()
    u = torch.empty(x.numel() + 1, device=dev)[1:].view(op.image_shape).copy_(x)  # 4 bytes past an aligned address
    for alpha in (2e-15, 0.02, 1e14):
        for iters in (2, 8, 60):
            a, b = op.tv_prox(x, alpha, iters), op.tv_prox(u, alpha, iters)
            assert torch.equal(a.view(torch.int32), b.view(torch.int32)), (alpha, iters)
