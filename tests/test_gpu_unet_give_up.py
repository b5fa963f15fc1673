"""The bounded waits of the convolution ring and of the two weight-gradient kernels run out cleanly.  The test hook lets
each CTA issue only its first copies: the wait for the next one gives up after a few polls, nothing is in flight, the
tensor memory is freed, pat_unet_device_status reports PAT_ERR_TIMEOUT once, and with the hook off the same call, and a
convolution that needs the tensor memory of every SM, give the results of before, bit for bit."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call,cin,cout,dims,stops", [
    ("conv", 16, 16, (16, 40, 128), (0, 1, 4)),   # ring, lines with a halo
    ("conv", 48, 16, (64, 16, 101), (2, 3)),      # the same in three parts
    ("conv", 16, 16, (160, 16, 32), (0, 3)),      # ring, three copies of a plane; several z runs a CTA
    ("conv", 64, 64, (8, 16, 16), (0, 5)),        # by boxes
    ("grad", 48, 16, (64, 30, 15), (0, 1)),       # by lines, two blocks a CTA
    ("grad", 16, 16, (64, 256, 256), (3, 30)),    # by lines, in the first and in the second segment
    ("grad", 64, 64, (16, 32, 32), (0, 2))])      # general form
def test_waits_that_run_out(call, cin, cout, dims, stops):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, dev = _lib.load(), torch.device("cuda", 0)
    st = torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device=dev).manual_seed(5)

    def conv(cin, cout, dims):
        V = dims[0] * dims[1] * dims[2]
        x, w = (torch.randn(s, generator=g, device=dev).bfloat16() for s in ((V, cin), (27, cout, cin)))

        def run():
            y = torch.zeros((V, cout), dtype=torch.bfloat16, device=dev)
            _lib.check(L.pat_unet_conv3(x.data_ptr(), cin, cin, w.data_ptr(), cout, y.data_ptr(), cout, *dims, 0, st))
            return y
        return run

    def grad(cin, cout, dims):
        V = dims[0] * dims[1] * dims[2]
        x, d = (torch.randn(s, generator=g, device=dev).bfloat16() for s in ((V, cin), (V, cout)))
        scratch = torch.zeros(L.pat_unet_wgrad_scratch(cin, cout, *dims), device=dev)

        def run():
            dw = torch.zeros((27, cout, cin), device=dev)
            _lib.check(L.pat_unet_conv3_wgrad(x.data_ptr(), cin, cin, d.data_ptr(), cout, cout, *dims, scratch.data_ptr(),
                                              dw.data_ptr(), st))
            return dw
        return run

    run, everywhere = {"conv": conv, "grad": grad}[call](cin, cout, dims), conv(16, 16, (32, 64, 64))
    want, want_all = run(), everywhere()
    _lib.check(L.pat_unet_device_status(st))
    for stop in stops:
        try:
            _lib.check(L.pat_unet_debug_copy_fault(stop, 4))
            run()
            with pytest.raises(_lib.PatError) as e:
                _lib.check(L.pat_unet_device_status(st))
            assert e.value.status == 4
        finally:
            _lib.check(L.pat_unet_debug_copy_fault(-1, 0))
        _lib.check(L.pat_unet_device_status(st))  # cleared
        assert torch.equal(run(), want) and torch.equal(everywhere(), want_all)
        _lib.check(L.pat_unet_device_status(st))
