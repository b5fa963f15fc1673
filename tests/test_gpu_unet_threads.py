"""Host threads that run layers of different shapes at the same time, each on a stream of its own: every call is
accepted, whatever the other thread launches between its preparation and its launch, and gives the results it gives
alone."""
import threading

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_threads_with_different_shapes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, dev = _lib.load(), torch.device("cuda", 0)

    def layer(cin, cout, dims, seed):
        g = torch.Generator(device=dev).manual_seed(seed)
        V = dims[0] * dims[1] * dims[2]
        x, w, d = (torch.randn(s, generator=g, device=dev).bfloat16() for s in ((V, cin), (27, cout, cin), (V, cout)))
        y, dw = torch.empty((V, cout), dtype=torch.bfloat16, device=dev), torch.empty((27, cout, cin), device=dev)
        scratch = torch.empty(L.pat_unet_wgrad_scratch(cin, cout, *dims), device=dev)

        def run(st, conv, grad):
            if conv:
                _lib.check(L.pat_unet_conv3(x.data_ptr(), cin, cin, w.data_ptr(), cout, y.data_ptr(), cout, *dims, 0, st))
            if grad:
                _lib.check(L.pat_unet_conv3_wgrad(x.data_ptr(), cin, cin, d.data_ptr(), cout, cout, *dims,
                                                  scratch.data_ptr(), dw.data_ptr(), st))
            return y, dw
        return run

    # shapes of one kernel whose shared memory differs: the convolution ring, the weight gradient by lines, its
    # general form, and the convolution by boxes
    pairs = [((16, 16, (16, 40, 128)), (16, 16, (210, 40, 8)), True, False),
             ((48, 16, (4, 16, 16)), (16, 16, (4, 4, 16)), False, True),
             ((112, 48, (2, 4, 16)), (192, 64, (2, 4, 16)), False, True),
             ((64, 128, (4, 64, 160)), (64, 16, (2, 4, 16)), True, False)]
    for a, b, conv, grad in pairs:
        errors, results = [], {}
        layers = [layer(*a, 1), layer(*b, 2)]
        st = torch.cuda.current_stream().cuda_stream
        want = [[t.clone() for t in run(st, conv, grad)] for run in layers]
        torch.cuda.synchronize()
        gate = threading.Barrier(2)

        def work(i):
            try:
                stream = torch.cuda.Stream(dev)
                torch.zeros(1, device=dev)
                gate.wait()
                for _ in range(1500):
                    results[i] = layers[i](stream.cuda_stream, conv, grad)
                stream.synchronize()
            except Exception as e:  # noqa: BLE001
                errors.append(e)
        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert not errors, errors
        for i in range(2):
            if conv:
                assert torch.equal(results[i][0], want[i][0])
            if grad:
                assert torch.equal(results[i][1], want[i][1])
        _lib.check(L.pat_unet_device_status(st))


def test_a_thread_whose_first_call_is_a_layer():
    """Nothing else of CUDA has run in the thread: the call finds the device's context by itself."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, dev = _lib.load(), torch.device("cuda", 0)
    x, w = torch.ones((64, 16), device=dev).bfloat16(), torch.ones((27, 16, 16), device=dev).bfloat16()
    y, dw = torch.zeros((64, 16), device=dev).bfloat16(), torch.zeros((27, 16, 16), device=dev)
    scratch, z = torch.empty(L.pat_unet_wgrad_scratch(16, 16, 4, 4, 4), device=dev), torch.zeros_like(y)
    torch.cuda.synchronize()
    status = []

    def conv():
        status.append(L.pat_unet_conv3(x.data_ptr(), 16, 16, w.data_ptr(), 16, y.data_ptr(), 16, 4, 4, 4, 0, None))

    def grad():
        status.append(L.pat_unet_conv3_wgrad(x.data_ptr(), 16, 16, x.data_ptr(), 16, 16, 4, 4, 4, scratch.data_ptr(),
                                             dw.data_ptr(), None))
    def captured():
        stream, graph = torch.cuda.Stream(dev), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            status.append(L.pat_unet_conv3(x.data_ptr(), 16, 16, w.data_ptr(), 16, z.data_ptr(), 16, 4, 4, 4, 0,
                                           stream.cuda_stream))
        graph.replay()
        torch.cuda.synchronize()
    for f in (conv, grad, captured):
        t = threading.Thread(target=f)
        t.start()
        t.join()
    torch.cuda.synchronize()
    assert status == [0, 0, 0] and torch.equal(y, z)
    assert float(y[21, 0]) == 27 * 16 and float(dw[13, 0, 0]) == 64  # an inner voxel; the centre tap
