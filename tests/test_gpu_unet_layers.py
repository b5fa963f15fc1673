"""The elementwise layers' vector forms against their scalar forms (taken when a stride is not a multiple
of 8, or a pointer not 16-byte aligned): bit for bit, on odd channel octets and small volumes; the masked
calls against the plain call followed by the ReLU backward, bit for bit; the output layer's backward
against FP64."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    lib = _lib.load()

    def call(name, *args):
        _lib.check(getattr(lib, name)(*args, torch.cuda.current_stream().cuda_stream))
    return call


def buf(V, C, ld, seed):
    """[V][ld] BF16 with C live channels (the rest a sentinel)"""
    g = torch.Generator(device="cuda").manual_seed(seed)
    b = torch.full((V, ld), 7.0, dtype=torch.bfloat16, device="cuda")
    b[:, :C] = torch.randn((V, C), generator=g, device="cuda").bfloat16()
    return b


@pytest.mark.parametrize("C,dims", [(8, (2, 2, 2)), (24, (4, 6, 10)), (48, (2, 8, 34)), (128, (6, 2, 4))])
def test_vector_forms_equal_scalar_forms(L, C, dims):
    D, H, W = dims
    V, P = D * H * W, D * H * W // 8
    res = []
    for ld in (C + 8, C + 1):  # 16-byte rows, and odd ones
        big, small, act, sact = buf(V, C, ld, 1), buf(P, C, ld, 2), buf(V, C, ld, 3), buf(P, C, ld, 4)
        out = []
        y = buf(P, C, ld, 5)
        L("pat_unet_pool", big.data_ptr(), ld, C, D, H, W, y.data_ptr(), ld)
        out.append(y)
        y = buf(V, C, ld, 6)
        L("pat_unet_pool_bwd_add", small.data_ptr(), ld, C, D, H, W, y.data_ptr(), ld)
        out.append(y.clone())
        L("pat_unet_relu_bwd", y.data_ptr(), ld, act.data_ptr(), ld, C, V)
        out.append(y)
        m = buf(V, C, ld, 6)
        L("pat_unet_pool_bwd_add_masked", small.data_ptr(), ld, C, D, H, W, m.data_ptr(), ld, act.data_ptr(), ld)
        assert torch.equal(m, y)
        y = buf(V, C, ld, 7)
        L("pat_unet_up", small.data_ptr(), ld, C, D // 2, H // 2, W // 2, y.data_ptr(), ld)
        out.append(y)
        y = buf(P, C, ld, 8)
        L("pat_unet_up_bwd", big.data_ptr(), ld, C, D // 2, H // 2, W // 2, y.data_ptr(), ld)
        out.append(y.clone())
        L("pat_unet_relu_bwd", y.data_ptr(), ld, sact.data_ptr(), ld, C, P)
        m = buf(P, C, ld, 8)
        L("pat_unet_up_bwd_masked", big.data_ptr(), ld, C, D // 2, H // 2, W // 2, m.data_ptr(), ld, sact.data_ptr(), ld)
        assert torch.equal(m, y)
        for o in out:
            assert bool((o[:, C:] == 7.0).all())
        res.append([o[:, :C].clone() for o in out])
    for a, b in zip(*res):
        assert torch.equal(a, b)


@pytest.mark.parametrize("V", [1, 255, 70001])
def test_output_layer_and_its_backward(L, V):
    g = torch.Generator(device="cuda").manual_seed(V)
    head = torch.randn(17, generator=g, device="cuda")
    x = torch.randn(V, generator=g, device="cuda")
    t = torch.randn(V, generator=g, device="cuda")
    res = []
    for off in (0, 1):  # aligned, and one channel past an aligned address
        h = torch.zeros(16 * V + 8, dtype=torch.bfloat16, device="cuda")
        h[off:off + 16 * V] = torch.randn(16 * V, generator=torch.Generator(device="cuda").manual_seed(V + 1),
                                          device="cuda").bfloat16()
        hv = h[off:off + 16 * V].reshape(V, 16)
        out = torch.empty(V, device="cuda")
        L("pat_unet_head", hv.data_ptr(), head.data_ptr(), V, out.data_ptr())
        x16 = torch.empty(16 * V + 8, dtype=torch.bfloat16, device="cuda")[off:off + 16 * V]
        L("pat_unet_input", x.data_ptr(), 0.5, V, x16.data_ptr())
        grads = []
        for name in ("pat_unet_head_bwd", "pat_unet_head_bwd_masked"):
            dh = torch.zeros(16 * V + 8, dtype=torch.bfloat16, device="cuda")
            gh, loss = torch.empty(17, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
            part = torch.empty(304 * 18, dtype=torch.float64, device="cuda")
            L(name, hv.data_ptr(), head.data_ptr(), out.data_ptr(), t.data_ptr(), V, dh.data_ptr() + 2 * off, gh.data_ptr(),
              loss.data_ptr(), part.data_ptr())
            grads += [dh[off:off + 16 * V].reshape(V, 16).clone(), gh, loss]
        assert torch.equal(grads[3], torch.where(hv > 0, grads[0], torch.zeros_like(grads[0])))
        res.append([out, x16.clone(), grads[0]])
        e = out.double() - t.double()
        gv = (2.0 / V * e).float().double()
        ref = torch.cat([hv.double().T @ gv, gv.sum()[None]])
        scale = torch.cat([hv.double().abs().T @ gv.abs(), gv.abs().sum()[None]])
        # FP64-grade sums rounded once to FP32: half an ulp of the value, plus 2^-40 of the terms' magnitude
        assert bool(((grads[1].double() - ref).abs() <= 2.0 ** -24 * ref.abs() + 2.0 ** -40 * scale).all())
        assert abs(float(grads[2]) - float((e * e).mean())) <= 1e-12 * float((e * e).mean())
    for a, b in zip(*res):
        assert torch.equal(a, b)
