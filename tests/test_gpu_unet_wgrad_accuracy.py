"""The weight gradient at the network's volumes against FP64, on the inputs it meets there: activations behind a ReLU,
and gradients that do or do not cancel.  The tensor core truncates as it adds, so a long sum of one sign comes out low by
a share that grows with the sum's length; the bound is the 1e-5 of the layers' other tests.  The shapes cover both
kernels, one and several accumulators in turn, and sums in one and in several segments."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,dims", [
    (16, 16, (64, 128, 128)), (48, 16, (64, 128, 128)), (16, 32, (32, 64, 64)), (32, 32, (64, 128, 128)),
    (96, 32, (32, 64, 64)), (16, 16, (64, 256, 256)), (64, 64, (16, 32, 32)), (192, 64, (16, 32, 32)), (16, 48, (64, 64, 128))])
def test_weight_gradient_of_activations(cin, cout, dims):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, dev, (D, H, W) = _lib.load(), torch.device("cuda", 0), dims
    st = torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device=dev).manual_seed(cin + 7 * cout)
    x = torch.randn((D * H * W, cin), generator=g, device=dev).relu().bfloat16()
    noise = torch.randn((D * H * W, cout), generator=g, device=dev)
    xp = torch.nn.functional.pad(x.double().reshape(D, H, W, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    scratch = torch.empty(L.pat_unet_wgrad_scratch(cin, cout, *dims), device=dev)
    dw = torch.empty((27, cout, cin), device=dev)
    for dy in (noise.bfloat16(), noise.relu().bfloat16()):
        ref = torch.stack([dy.double().T @ xp[t // 9:t // 9 + D, (t // 3) % 3:(t // 3) % 3 + H,
                                              t % 3:t % 3 + W].reshape(-1, cin) for t in range(27)])
        _lib.check(L.pat_unet_conv3_wgrad(x.data_ptr(), cin, cin, dy.data_ptr(), cout, cout, *dims, scratch.data_ptr(),
                                          dw.data_ptr(), st))
        _lib.check(L.pat_unet_device_status(st))
        assert float((dw.double() - ref).norm() / ref.norm()) < 1e-5
