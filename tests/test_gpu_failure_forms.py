"""The failure path of test_gpu_failure.py on every form of the time step: one launch a step (small grids, also with the
rolled loop body of lines of 64), three launches a step on a small grid (a workspace limit without room for the parts),
the rolled line passes of 64x128x128, the same with states streamed past the L2 (four volumes), and a grid with a
256-voxel axis, whose 16 KB tiles the hook leaves alone.  With one state's copies left out the calls return, the status
names the copy and is cleared, and with the hook off both operators give the bits of before."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1605_00133_gb300 import _lib, presets  # noqa: E402
from paper_1605_00133_gb300.operators import PatOperator  # noqa: E402
from test_gpu_small_steps import sequential  # noqa: E402


@pytest.mark.parametrize("shape,batch,limited", [
    ((16, 32, 32), 1, False), ((64, 64, 64), 1, False), ((16, 32, 32), 1, True), ((64, 64, 64), 1, True),
    ((64, 128, 128), 1, False), ((64, 128, 128), 4, False), ((16, 64, 256), 1, False), ((16, 64, 256), 1, True)])
def test_every_form_reports_a_copy_that_never_lands(shape, batch, limited):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    lib, dev = _lib.load(), torch.device("cuda", 0)
    g, s = presets.Grid(*shape, T=6, pml_size=3, batch=batch), presets.Sampling()
    op = sequential(g, s) if limited else PatOperator(g, s)
    r = torch.Generator(device=dev).manual_seed(2)
    x = torch.randn(op.image_shape, generator=r, device=dev)
    y = torch.randn(op.data_shape, generator=r, device=dev)
    want = op.forward(x), op.adjoint(y)
    op.device_status(dev)
    for mask, what in ((2, "state-1 tile"), (4, "state-2 tile")):
        for call in (lambda: op.forward(x), lambda: op.adjoint(y)):
            try:
                assert lib.pat_debug_copy_fault(op._h, mask, 4) == 0
                call()
                with pytest.raises(_lib.PatError) as e:
                    op.device_status(dev)
                assert e.value.status == 4 and what in str(e.value)
                op.device_status(dev)  # cleared
            finally:
                assert lib.pat_debug_copy_fault(op._h, 0, 0) == 0
        assert torch.equal(op.forward(x), want[0]) and torch.equal(op.adjoint(y), want[1])
        op.device_status(dev)
    op.close()
