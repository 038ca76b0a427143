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
