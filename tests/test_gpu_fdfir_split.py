"""Full-length FD-FIR as 1024 x P/1024: the largest array of each transform length (outputs in both
halves of the last transform), template counts that end on either scratch buffer, and a shorter
array after a longer one, against the overlap-save plane to the FP32 tolerance."""
import numpy as np
import pytest

from parity import TOL_FP32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("log2p", [21, 22, 23])
@pytest.mark.parametrize("m,k", [(1, 33), (2, 5), (3, 421)])
def test_largest_array(log2p, m, k):
    import paper_1805_12280_gb300 as fd
    fd.load()
    rng = np.random.default_rng(log2p * 10 + m)
    h = ((rng.standard_normal((m, k)) + 1j * rng.standard_normal((m, k))) / np.sqrt(2 * k)).astype(np.complex64)
    n_max = (1 << log2p) - k + 1
    g = torch.Generator(device="cuda").manual_seed(log2p)
    x = torch.randn(n_max, 2, device="cuda", generator=g).view(torch.complex64).reshape(-1)
    with fd.FdFir(h, n_max=n_max) as ff, fd.Plan(h, n_max=n_max) as plan:
        assert ff.length == 1 << log2p
        for n in (n_max, (1 << (log2p - 1)) + 4097, 1):
            a = ff.convolve(x[:n])
            b = plan.convolve(x[:n])
            plan.status()
            assert float((a - b).abs().max()) <= TOL_FP32 * max(float(b.max()), 1.0)
