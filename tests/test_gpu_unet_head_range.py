"""The output layer's backward keeps its sums in FP64, with its range: squared errors beyond FP32's largest and below
its smallest value, an infinite prediction, and channels that are infinite, NaN or subnormal.  Each against plain FP64
(a sum of n terms is within n 2^-53 of the terms' magnitude, a gradient rounded once to FP32), and the result does not
depend on the alignment of h and dh, bit for bit."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [1, 300, 70001])
@pytest.mark.parametrize("what", ["ordinary", "large", "tiny", "infinite prediction", "odd channels", "subnormal channels"])
def test_sums_have_the_range_of_fp64(V, what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_00133_gb300 import _lib
    L, st = _lib.load(), torch.cuda.current_stream().cuda_stream
    r = torch.Generator(device="cuda").manual_seed(V)
    scale = {"large": 1e25, "tiny": 1e-24}.get(what, 1.0)
    out, target = (scale * torch.randn(V, generator=r, device="cuda") for _ in range(2))
    head = torch.randn(17, generator=r, device="cuda")
    hv = torch.randn((V, 16), generator=r, device="cuda").bfloat16()
    if what == "infinite prediction":
        out[V // 2] = float("inf")
    if what == "odd channels":
        hv[V // 2, 3], hv[V // 3, 5] = float("inf"), float("nan")
    if what == "subnormal channels":
        hv[:, 1::2] = (hv[:, 1::2].double() * 2.0 ** -130).bfloat16()
        out, target = out * 1e30, target * 1e30
    res = []
    for off in (0, 1):  # aligned, and one channel past an aligned address
        h, dh = (torch.zeros(16 * V + 8, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        h[off:off + 16 * V] = hv.reshape(-1)
        gh, loss = torch.empty(17, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
        part = torch.empty(L.pat_unet_head_scratch(V), dtype=torch.float64, device="cuda")
        _lib.check(L.pat_unet_head_bwd(h.data_ptr() + 2 * off, head.data_ptr(), out.data_ptr(), target.data_ptr(), V,
                                       dh.data_ptr() + 2 * off, gh.data_ptr(), loss.data_ptr(), part.data_ptr(), st))
        res.append((gh, loss, dh[off:off + 16 * V].clone()))
    for a, b in zip(*res):
        assert torch.equal(torch.nan_to_num(a, nan=7.0), torch.nan_to_num(b, nan=7.0))
        assert torch.equal(a.isnan(), b.isnan())
    e = out.double() - target.double()
    ref = (e * e).mean()
    loss = res[0][1][0]
    assert loss == ref or abs(float(loss - ref)) <= 2.0 ** -52 * V * float(ref)
    g = (2.0 / V * e).float().double()
    terms = torch.cat([hv.double() * g[:, None], g[:, None]], 1)
    want, got = terms.sum(0), res[0][0].double()
    tol = 2.0 ** -24 * want.abs() + 2.0 ** -53 * V * terms.abs().sum(0) + 2.0 ** -150
    finite = want.isfinite()
    assert bool(((got - want).abs() <= tol)[finite].all())
    assert torch.equal(torch.nan_to_num(got[~finite], nan=7.0, posinf=8.0, neginf=9.0),
                       torch.nan_to_num(want[~finite], nan=7.0, posinf=8.0, neginf=9.0))
