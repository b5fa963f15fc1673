"""What test_gpu_small_steps.py compares are two forms: the operator without a limit holds the parts of the spectrum and
the one under the smallest limit does not, on every grid of it; and the library's own scratch serves exactly the grids
whose workspace without the parts fits it, with the same bits."""
import ctypes
import re

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1605_00133_gb300 import _lib, presets  # noqa: E402
from paper_1605_00133_gb300.operators import PatOperator  # noqa: E402
from test_gpu_small_steps import sequential  # noqa: E402

SCRATCH = 64 << 20


def spectrum_bytes(shape, batch):
    return (batch * shape[0] * shape[1] * (shape[2] // 2 + 1) * 8 + 255) // 256 * 256


@pytest.mark.parametrize("shape,T,batch,m", [
    ((8, 8, 8), 2, 1, 0), ((16, 32, 8), 3, 2, 70), ((32, 32, 32), 12, 1, 200), ((8, 16, 256), 5, 1, 0),
    ((128, 16, 64), 4, 3, 0), ((64, 64, 64), 6, 1, 500), ((16, 128, 128), 5, 1, 900), ((256, 32, 32), 4, 1, 0),
    ((32, 128, 128), 4, 1, 0), ((64, 64, 64), 4, 3, 300), ((16, 16, 16), 1, 1, 0), ((64, 128, 128), 500, 1, 2048)])
def test_the_two_forms_are_two(shape, T, batch, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    L, dev = _lib.load(), torch.device("cuda", 0)
    g = presets.Grid(*shape, T=T, pml_size=2, batch=batch)
    s = presets.make_sampling(g, 1, m, 0) if m else presets.Sampling()
    a, b = PatOperator(g, s), sequential(g, s)
    large = shape == (64, 128, 128)  # more tiles than one launch serves: no parts
    assert a.workspace_bytes - b.workspace_bytes == (0 if large else 4 * spectrum_bytes(shape, batch))
    # the smallest limit that admits the grid is its workspace without the parts
    L.pat_set_workspace_limit(1)
    try:
        with pytest.raises(_lib.PatError) as e:
            PatOperator(g, s)
    finally:
        L.pat_set_workspace_limit(0)
    need = int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))
    p0 = torch.randn(a.image_shape, generator=torch.Generator(device=dev).manual_seed(T), device=dev)
    f = a.forward(p0)
    out = torch.full_like(f, float("nan"))
    st = L.pat_forward_noalloc(a._h, ctypes.c_void_p(p0.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if need <= SCRATCH:
        assert st == 0 and torch.equal(f, out)
    else:
        assert st == 1 and f"needs {need} bytes" in L.pat_last_error().decode()
