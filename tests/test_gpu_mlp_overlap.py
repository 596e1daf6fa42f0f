"""Forward pass with the output over the input: tiles of 256 rows read 24 bytes and write 8 a sample, so
without a copy one tile's outputs would overwrite another's inputs.  One tile, several, more than one per CTA."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [100, 3000, 100003])
@pytest.mark.parametrize("at", [0, 1, 4])
def test_output_over_input(n, at):
    """The output at `at` floats of the input per sample (4: its last third)."""
    mlp = gf.MLP(seed=8)
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand(n, 6, generator=g, device="cuda")
    ref = mlp.forward(x)
    buf = x.clone().reshape(-1)
    out = buf[at * n:at * n + 2 * n]
    st = gf.lib().gf_mlp_forward(mlp._h, ctypes.c_void_p(buf.data_ptr()), n, ctypes.c_void_p(out.data_ptr()),
                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == gf.GF_OK
    assert torch.equal(out.view(n, 2), ref)
    mlp.close()
