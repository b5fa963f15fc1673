"""The weight gradient of layers with few channels, fetched by lines: lines and rows shorter than a block of it, one
voxel, volumes of one plane, one to three channel blocks of both widths, one to three groups of M tiles.  Inputs are
exactly BF16, so it differs from FP64 by FP32 accumulation only (1e-5, as the layers' other tests)."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,dims,ldx,ldy", [
    (16, 16, (1, 1, 1), 16, 16), (16, 32, (2, 3, 17), 32, 48), (32, 16, (3, 1, 100), 32, 16), (48, 32, (4, 30, 15), 48, 32),
    (64, 16, (5, 9, 33), 80, 16), (80, 32, (3, 7, 70), 80, 32), (96, 16, (2, 40, 20), 96, 16), (16, 16, (9, 33, 65), 16, 16)])
def test_weight_gradient_by_lines(cin, cout, dims, ldx, ldy):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, dev, (D, H, W) = _lib.load(), torch.device("cuda", 0), dims
    st = torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device=dev).manual_seed(cin + 7 * cout)
    # what lies beside the operands' channels must not be read
    xb = torch.full((D * H * W, ldx), float("nan"), dtype=torch.bfloat16, device=dev)
    db = torch.full((D * H * W, ldy), float("nan"), dtype=torch.bfloat16, device=dev)
    xb[:, ldx - cin:] = torch.randn((D * H * W, cin), generator=g, device=dev)
    db[:, ldy - cout:] = torch.randn((D * H * W, cout), generator=g, device=dev)
    xp = torch.nn.functional.pad(xb[:, ldx - cin:].double().reshape(D, H, W, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    ref = torch.stack([db[:, ldy - cout:].double().T @ xp[t // 9:t // 9 + D, (t // 3) % 3:(t // 3) % 3 + H,
                                                         t % 3:t % 3 + W].reshape(-1, cin) for t in range(27)])
    scratch = torch.full((L.pat_unet_wgrad_scratch(cin, cout, *dims),), float("nan"), device=dev)
    dw = torch.full((27, cout, cin), float("nan"), device=dev)
    _lib.check(L.pat_unet_conv3_wgrad(xb.data_ptr() + 2 * (ldx - cin), ldx, cin, db.data_ptr() + 2 * (ldy - cout), ldy,
                                      cout, *dims, scratch.data_ptr(), dw.data_ptr(), st))
    _lib.check(L.pat_unet_device_status(st))
    assert float((dw.double() - ref).norm() / ref.norm()) < 1e-5
