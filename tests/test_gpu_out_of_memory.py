"""A prox or a solve that runs out of device memory while it allocates its workspace reports it, and the same call
works once there is room: with what the first attempt got and the rest."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1605_00133_gb300 import _lib, presets  # noqa: E402
from paper_1605_00133_gb300.operators import PatOperator  # noqa: E402


@pytest.mark.parametrize("what", ["prox", "solve"])
def test_a_call_that_ran_out_of_memory_can_be_repeated(what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    dev = torch.device("cuda", 0)
    g, s = presets.Grid(64, 128, 128, T=4, pml_size=3), presets.Sampling()
    op, other = PatOperator(g, s), PatOperator(g, s)
    x = torch.rand(op.image_shape, generator=torch.Generator(device=dev).manual_seed(1), device=dev)
    f = op.forward(x)

    def call(o):
        if what == "prox":
            return o.tv_prox(x, 0.05, 6, out=out)
        return o.bregman_solve(f, 1e-3, outer=1, inner=2, prox_iters=6, L=1.0)[0]
    out = torch.empty_like(x)
    if what == "solve":
        op.tv_prox(x, 0.05, 2, out=out)  # its workspace is there: the solver's own is what fails
    want = call(other).clone()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # the image is 4 MB; of the prox's 44 MB and the solver's 17 MB or more, leave room for the first buffers
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (11 << 20), dtype=torch.uint8, device=dev)
    try:
        with pytest.raises(_lib.PatError) as e:
            call(op)
        assert "out of memory" in str(e.value)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(call(op), want)
