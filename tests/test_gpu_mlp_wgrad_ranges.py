"""Length of the float sums in the weight gradients of large batches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as R
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rows", [(32768, 512), (65536, 1024)])
def test_sums_of_large_batches(n, rows):
    """Against the mean, in double, of calls of 512 rows (whose sums run over 64): n is a power of two times 512, so
    every rounding but the sums' is the same.  A range of `rows` rows is rows/16 additions in the tensor cores, each
    losing at most an ulp (2^-23) of the running sum, half of one on average; the running sum is half of the
    final one on average: rows 2^-29 of a weight's gradient, asked of each layer's root mean square."""
    mlp = gf.MLP(seed=1)
    g = torch.Generator(device="cuda").manual_seed(5)
    lo = torch.tensor([-np.pi, -np.pi, -0.6, -0.5, -0.5, 1.0], device="cuda")
    hi = torch.tensor([np.pi, np.pi, 0.6, 0.5, 0.5, 4.0], device="cuda")
    x = (lo + (hi - lo) * torch.rand(n, 6, generator=g, device="cuda")).contiguous()
    t = torch.randn(n, 2, generator=g, device="cuda")
    whole = mlp.gradients(x, t)[0].astype(np.float64)
    parts = np.zeros_like(whole)
    for i in range(0, n, 512):
        parts += mlp.gradients(x[i:i + 512], t[i:i + 512])[0]
    parts /= n // 512
    off = 0
    for l in range(5):
        m = R.DIMS[l + 1] * R.DIMS[l] + R.DIMS[l + 1]
        d, r = whole[off:off + m] - parts[off:off + m], parts[off:off + m]
        assert np.sqrt((d * d).mean()) < rows * 2.0 ** -29 * np.sqrt((r * r).mean()), l
        off += m
    mlp.close()
