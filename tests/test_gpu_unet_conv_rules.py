"""The convolution by boxes chooses its operand rows and output channels per CTA by the number of tiles.  A volume on one
side of a rule gives the bits of the volume it is cut from on the other, where both see the same voxels, and both agree
with FP64 (BF16 rounding of the output: 4e-3, as the layers' other tests)."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,dims,cut", [
    (64, 64, (16, 32, 32), 9),     # 128 tiles, 72: channels halved
    (128, 32, (16, 32, 32), 4),
    (192, 64, (20, 32, 32), 2),    # 160 tiles, 16
    (96, 32, (24, 32, 32), 8),     # over 152 CTAs, 64
    (96, 128, (21, 31, 30), 3),
    (160, 64, (24, 32, 32), 12)])
def test_rules_do_not_change_results(cin, cout, dims, cut):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, dev, (D, H, W) = _lib.load(), torch.device("cuda", 0), dims
    st = torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device=dev).manual_seed(cin + cout)
    x = torch.randn((D * H * W, cin), generator=g, device=dev).bfloat16()
    w = (torch.randn((27, cout, cin), generator=g, device=dev) / (27 * cin) ** 0.5).bfloat16()
    out = []
    for d in (D, cut):
        y = torch.zeros((d * H * W, cout), dtype=torch.bfloat16, device=dev)
        _lib.check(L.pat_unet_conv3(x.data_ptr(), cin, cin, w.data_ptr(), cout, y.data_ptr(), cout, d, H, W, 0, st))
        _lib.check(L.pat_unet_device_status(st))
        out.append(y)
    same = (cut - 1) * H * W  # the last plane of the cut volume has zeros above it
    assert torch.equal(out[0][:same], out[1][:same])
    xp = torch.nn.functional.pad(x.double().reshape(D, H, W, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    ref = sum(xp[t // 9:t // 9 + D, (t // 3) % 3:(t // 3) % 3 + H, t % 3:t % 3 + W].reshape(-1, cin) @ w[t].double().T
              for t in range(27))
    assert float((out[0].double() - ref).norm() / ref.norm()) < 4e-3
