"""The persistent convolution where its window of three accumulators moves: more planes than the ring has
accumulators (16 of 16 columns, 6 of 80), runs of one and two planes, runs that start inside a column, several groups of
output channels, both forms of lines.  Tolerances as the layers' other tests (BF16 rounding of the result)."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,dims", [
    (16, 16, (64, 16, 100)), (16, 80, (9, 80, 70)), (48, 48, (7, 100, 128)), (16, 16, (1, 640, 65)),
    (16, 32, (2, 400, 80)), (32, 64, (37, 64, 33)), (32, 32, (20, 64, 64))])
def test_ring_of_accumulators(cin, cout, dims):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, dev, (D, H, W) = _lib.load(), torch.device("cuda", 0), dims
    st = torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device=dev).manual_seed(cin + cout + D)
    x = torch.randn((D * H * W, cin), generator=g, device=dev).bfloat16()
    w = (torch.randn((27, cout, cin), generator=g, device=dev) / (27 * cin) ** 0.5).bfloat16()
    xp = torch.nn.functional.pad(x.double().reshape(D, H, W, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    ref = sum(xp[t // 9:t // 9 + D, (t // 3) % 3:(t // 3) % 3 + H, t % 3:t % 3 + W].reshape(-1, cin) @ w[t].double().T
              for t in range(27))
    y = torch.full((D * H * W, cout), float("nan"), dtype=torch.bfloat16, device=dev)
    for _ in range(2):
        _lib.check(L.pat_unet_conv3(x.data_ptr(), cin, cin, w.data_ptr(), cout, y.data_ptr(), cout, D, H, W, 0, st))
    _lib.check(L.pat_unet_device_status(st))
    d = y.double() - ref
    assert float(d.norm() / ref.norm()) < 4e-3
    assert float(d.abs().max() / ref.abs().max()) < 1e-2
