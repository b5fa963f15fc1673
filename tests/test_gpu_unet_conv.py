"""The convolution and its weight gradient where their tilings change: volumes large enough for the
persistent kernel (partial last columns and lines, z runs that start inside a column, one to five output
tiles), long lines whose boxes overlap, channel counts that are not a whole number of operand rows, and
the weight gradient's groups of M tiles and output channels.  Inputs are exactly BF16, so the
convolution differs from FP64 by the FP32 accumulation and the final BF16 rounding (relative 2^-9, 4e-3)
and the weight gradient by FP32 accumulation only (1e-5), the tolerances of the layers' other tests."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def rel(a, b):
    return float((a.double() - b).norm() / b.norm())


def conv64(x, w, dims):
    """x [V][cin], w [27][cout][cin] -> [V][cout], FP64 on the GPU"""
    D, H, W = dims
    xp = torch.nn.functional.pad(x.reshape(D, H, W, -1), (0, 0, 1, 1, 1, 1, 1, 1))
    return sum(xp[t // 9:t // 9 + D, (t // 3) % 3:(t // 3) % 3 + H, t % 3:t % 3 + W].reshape(D * H * W, -1) @ w[t].T
               for t in range(27))


def inputs(cin, cout, dims, ldx, ldy, dev):
    g = torch.Generator(device=dev).manual_seed(cin + 7 * cout)
    V = dims[0] * dims[1] * dims[2]
    x = torch.randn((V, cin), generator=g, device=dev).bfloat16()
    w = (torch.randn((27, cout, cin), generator=g, device=dev) / (27 * cin) ** 0.5).bfloat16()
    dy = torch.randn((V, cout), generator=g, device=dev).bfloat16()
    xb = torch.full((V, ldx), float("nan"), dtype=torch.bfloat16, device=dev)
    xb[:, ldx - cin:] = x
    db = torch.full((V, ldy), float("nan"), dtype=torch.bfloat16, device=dev)
    db[:, ldy - cout:] = dy
    return x, w, dy, xb, db


@pytest.mark.parametrize("cin,cout,dims,ldx,ldy", [
    (16, 16, (40, 17, 128), 16, 16), (48, 16, (33, 20, 101), 64, 32), (16, 48, (13, 50, 128), 32, 48),
    (32, 32, (20, 64, 64), 32, 96), (32, 96, (17, 56, 40), 48, 96), (16, 16, (160, 55, 8), 16, 16),
    (48, 80, (12, 70, 72), 48, 80), (64, 16, (20, 31, 66), 64, 16), (32, 16, (13, 50, 65), 48, 16), (32, 16, (9, 70, 127), 32, 16), (16, 64, (700, 3, 17), 16, 64),
    (16, 16, (3, 4, 260), 16, 16), (80, 32, (4, 6, 129), 80, 32), (112, 112, (3, 9, 20), 112, 112)])
def test_convolution_over_its_kernels(dev, cin, cout, dims, ldx, ldy):
    from paper_1605_00133_gb300 import _lib
    L = _lib.load()
    st = torch.cuda.current_stream().cuda_stream
    x, w, _, xb, _ = inputs(cin, cout, dims, ldx, ldy, dev)
    ref = conv64(x.double(), w.double(), dims)
    for relu in (1, 0):
        yb = torch.full((x.shape[0], ldy), 7.0, dtype=torch.bfloat16, device=dev)
        _lib.check(L.pat_unet_conv3(xb.data_ptr() + 2 * (ldx - cin), ldx, cin, w.data_ptr(), cout,
                                    yb.data_ptr() + 2 * (ldy - cout), ldy, *dims, relu, st))
        _lib.check(L.pat_unet_device_status(st))
        y = yb[:, ldy - cout:]
        assert rel(y, ref.relu() if relu else ref) < 4e-3
        # every voxel of the volume's edges too, not only on average
        assert float((y.double() - (ref.relu() if relu else ref)).abs().max() / ref.abs().max()) < 1e-2
        assert bool((yb[:, :ldy - cout] == 7.0).all())


@pytest.mark.parametrize("cin,cout,dims,ldx,ldy", [
    (16, 16, (40, 17, 128), 16, 16), (48, 16, (13, 20, 101), 64, 32), (80, 48, (5, 9, 33), 80, 48),
    (96, 32, (8, 16, 40), 96, 32), (112, 112, (3, 9, 20), 112, 112), (256, 96, (2, 3, 9), 256, 96),
    (32, 128, (2, 70, 3), 32, 128)])
def test_weight_gradient_over_its_groups(dev, cin, cout, dims, ldx, ldy):
    from paper_1605_00133_gb300 import _lib
    L = _lib.load()
    st = torch.cuda.current_stream().cuda_stream
    x, _, dy, xb, db = inputs(cin, cout, dims, ldx, ldy, dev)
    w = torch.zeros((27, cout, cin), dtype=torch.float64, device=dev, requires_grad=True)
    (conv64(x.double(), w, dims) * dy.double()).sum().backward()
    scratch = torch.full((L.pat_unet_wgrad_scratch(cin, cout, *dims),), float("nan"), device=dev)
    dw = torch.full((27, cout, cin), float("nan"), device=dev)
    _lib.check(L.pat_unet_conv3_wgrad(xb.data_ptr() + 2 * (ldx - cin), ldx, cin, db.data_ptr() + 2 * (ldy - cout), ldy,
                                      cout, *dims, scratch.data_ptr(), dw.data_ptr(), st))
    _lib.check(L.pat_unet_device_status(st))
    assert rel(dw, w.grad) < 1e-5
