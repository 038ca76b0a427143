"""The two-stage tensor-core form leaves out the output runs that the discard of K - 1 outputs
removes: the kernel for several arrays, which leaves them out, against the kernel for one short
array, which computes them all, bit for bit, at the filter lengths where the first kept run moves
past a quarter of a chunk, a chunk and the last chunk."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("k", [1, 2, 33, 384, 385, 416, 417, 480, 481, 512, 513, 896, 897, 1408, 1409, 1537, 1920, 1921, 2033])
def test_skipped_runs(k):
    import paper_1805_12280_gb300 as fd
    fd.load()
    rng = np.random.default_rng(k)
    h = ((rng.standard_normal((3, k)) + 1j * rng.standard_normal((3, k))) / np.sqrt(2 * k)).astype(np.complex64)
    ns = [5001, 1, 2 * (2049 - k) + 1]
    xs = [torch.from_numpy((rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)).cuda() for n in ns]
    with fd.Plan(h, n_max=max(ns), precision=fd.FDAS_PREC_TC_DFT2) as plan:
        singles = [plan.convolve(x) for x in xs]
        outs = [torch.full((3, n), -1.0, device="cuda") for n in ns]
        torch.cuda.synchronize()
        fd.fdas_convolve_batch_noalloc(plan.handle, [x.data_ptr() for x in xs], ns, [o.data_ptr() for o in outs])
        plan.status()
    for o, s in zip(outs, singles):
        assert torch.equal(o, s)


@pytest.mark.parametrize("k", [1, 384, 385, 416, 417, 512, 513, 897, 1408, 1409, 1920, 1921])
def test_skipped_runs_of_a_long_array(k):
    # the kernel for one long array (equal unit shares of at least 12 per block) against the one for
    # several arrays
    import paper_1805_12280_gb300 as fd
    fd.load()
    rng = np.random.default_rng(k)
    h = ((rng.standard_normal((3, k)) + 1j * rng.standard_normal((3, k))) / np.sqrt(2 * k)).astype(np.complex64)
    n = 2200 * (2049 - k) + 77            # 2201 segments, 1101 segment pairs x 2 template pairs
    g = torch.Generator(device="cuda").manual_seed(k)
    x = torch.randn(n, 2, device="cuda", generator=g).view(torch.complex64).reshape(-1)
    with fd.Plan(h, n_max=n, precision=fd.FDAS_PREC_TC_DFT2) as plan:
        a, b = (torch.full((3, n), -1.0, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        plan.convolve(x, out=a)
        fd.fdas_convolve_batch_noalloc(plan.handle, [x.data_ptr()], [n], [b.data_ptr()])
        plan.status()
    assert torch.equal(a, b) and bool((a >= 0).all())
