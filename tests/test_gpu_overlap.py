"""Launches that overlap on one stream (programmatic dependent launch): a call whose input the call
before writes, or whose output the call before still reads, gives the bits it gives when the GPU is
waited for in between."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fd():
    import paper_1805_12280_gb300 as m
    m.load()
    return m


@pytest.fixture(scope="module")
def bank():
    import synth
    return synth.template_bank()[0]


def _rand(n, seed):
    rng = np.random.default_rng(seed)
    return torch.from_numpy((rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)).cuda()


def _sync(wait):
    if wait:
        torch.cuda.synchronize()


@pytest.mark.parametrize("precision", ["FDAS_PREC_FP32", "FDAS_PREC_TC_DFT2"])
@pytest.mark.parametrize("n", [1, 1629, 1 << 14, 70_001])
def test_chained_planes(fd, bank, precision, n):
    # the second call's input is the first call's plane (its first 2n floats as n complex values)
    xs = [_rand(n, 10 + i) for i in range(2)]
    with fd.Plan(bank, n_max=n, precision=getattr(fd, precision)) as plan:
        first = torch.zeros((85, n), device="cuda")
        link = torch.view_as_complex(first.reshape(-1)[: 2 * n].reshape(n, 2))

        def run(wait, reps):
            outs = [torch.full((85, n), -1.0, device="cuda") for _ in xs]
            torch.cuda.synchronize()
            for _ in range(reps):
                for x, o in zip(xs, outs):
                    plan.convolve(x, out=first)
                    _sync(wait)
                    plan.convolve(link, out=o)
                    _sync(wait)
            torch.cuda.synchronize()
            return outs

        ref = run(True, 1)
        for r, g in zip(ref, run(False, 25)):
            assert torch.equal(r, g)
        plan.status()


@pytest.mark.parametrize("precision", ["FDAS_PREC_FP32", "FDAS_PREC_TC_DFT2"])
@pytest.mark.parametrize("max_harm", [1, 8, 32])
def test_harmonic_sums_then_next_plane(fd, bank, precision, max_harm):
    # the plane is overwritten by the call that follows its harmonic sums
    n = 40_001
    xs = [_rand(n, 20 + i) for i in range(2)]
    with fd.Plan(bank, n_max=n, precision=getattr(fd, precision)) as plan:
        P = torch.empty((85, n), device="cuda")
        bufs = [(torch.empty((1 << 17, 3), dtype=torch.int64, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda"))
                for _ in xs]

        def run(wait, reps):
            for _ in range(reps):
                for x, (buf, count) in zip(xs, bufs):
                    plan.convolve(x, out=P)
                    _sync(wait)
                    fd.harmonic_sum(P, 210, max_harm, [14.0 * (1 << j) for j in range(max_harm.bit_length())], buf=buf, count=count)
                    _sync(wait)
            torch.cuda.synchronize()
            recs = [fd.harmonic_to_numpy(buf, count) for buf, count in bufs]
            return [r[np.lexsort((r["nharm"], r["bin"], r["tpl"]))] for r in recs]

        ref = run(True, 1)
        assert ref[0].size > 100
        for r, g in zip(ref, run(False, 25)):
            np.testing.assert_array_equal(r, g)


def test_fdfir_calls_back_to_back(fd, bank):
    # consecutive calls share the plan's scratch; the last call's plane feeds an overlap-save plane
    n, h = 60_001, bank[::21]
    xs = [_rand(n, 30 + i) for i in range(2)]
    with fd.FdFir(h, n) as f, fd.Plan(bank, n_max=n) as plan:
        outs = [torch.empty((h.shape[0], n), device="cuda") for _ in xs]
        tail = torch.empty((85, n), device="cuda")

        def run(wait, reps):
            for _ in range(reps):
                for x, o in zip(xs, outs):
                    f.convolve(x, out=o)
                    _sync(wait)
                plan.convolve(torch.view_as_complex(outs[1].reshape(-1)[: 2 * n].reshape(n, 2)), out=tail)
                _sync(wait)
            torch.cuda.synchronize()
            return [t.clone() for t in (*outs, tail)]

        ref = run(True, 1)
        for r, g in zip(ref, run(False, 10)):
            assert torch.equal(r, g)
