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


def _link(plane, n):
    # the first 2n floats of a plane as n complex values
    return torch.view_as_complex(plane.reshape(-1)[: 2 * n].reshape(n, 2))


def _records(buf, count, fields):
    c = buf[: int(count.item())].cpu().numpy().reshape(-1)
    return np.sort(c.view(fields).reshape(-1), order=["tpl", "bin"])


@pytest.mark.parametrize("precision", ["FDAS_PREC_FP32", "FDAS_PREC_TC_DFT2"])
@pytest.mark.parametrize("n", [1 << 14, 300_001])   # 300001 FP32 points: equal shares
def test_thresholds_of_the_plane_before(fd, bank, precision, n):
    # a threshold call right after the plane that is its input, then the plane of another input
    xs = [_rand(n, 40 + i) for i in range(2)]
    with fd.Plan(bank, n_max=n, precision=getattr(fd, precision)) as plan:
        first = torch.zeros((85, n), device="cuda")
        bufs = [(torch.empty((85 * n, 2), dtype=torch.int64, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda"))
                for _ in xs]   # room for every output: a truncated list may hold any of the crossings

        def run(wait, reps):
            for _ in range(reps):
                for x, (buf, count) in zip(xs, bufs):
                    plan.convolve(x, out=first)
                    _sync(wait)
                    plan.candidates(_link(first, n), 60.0, max_cand=buf.shape[0], buf=buf, count=count)
                    _sync(wait)
            torch.cuda.synchronize()
            return [_records(buf, count, fd.fdas.CANDIDATE_DTYPE) for buf, count in bufs]

        ref = run(True, 1)
        assert ref[0].size > 100
        for r, g in zip(ref, run(False, 25)):
            np.testing.assert_array_equal(r, g)
        plan.status()


@pytest.mark.parametrize("precision", ["FDAS_PREC_FP32", "FDAS_PREC_TC_DFT2"])
def test_captured_chain(fd, bank, precision):
    # every launch reads what the one before writes: in a graph, replayed, as when waited for in between
    n, m = 60_001, 5
    xs = [_rand(n, 50 + i) for i in range(2)]
    x = torch.empty_like(xs[0])
    with fd.Plan(bank, n_max=n, precision=getattr(fd, precision)) as plan, fd.FdFir(bank[::21], n) as f:
        a, b, tail = (torch.zeros((85, n), device="cuda") for _ in range(3))
        full = torch.zeros((m, n), device="cuda")
        hbuf, hcount = torch.empty((1 << 18, 3), dtype=torch.int64, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda")
        cbuf, ccount = torch.empty((1 << 18, 2), dtype=torch.int64, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda")

        def chain(wait):
            plan.convolve(x, out=a)
            _sync(wait)
            plan.convolve(_link(a, n), out=b)
            _sync(wait)
            f.convolve(_link(b, n), out=full)
            _sync(wait)
            plan.convolve(_link(full, n), out=tail)
            _sync(wait)
            fd.harmonic_sum(tail, 210, 8, thr, max_cand=hbuf.shape[0], buf=hbuf, count=hcount)
            _sync(wait)
            plan.candidates(_link(tail, n), cthr, max_cand=cbuf.shape[0], buf=cbuf, count=ccount)
            _sync(wait)

        def result():
            torch.cuda.synchronize()
            h = hbuf[: int(hcount.item())].cpu().numpy().view(fd.fdas.HARMONIC_DTYPE).reshape(-1)
            return [t.clone() for t in (a, b, full, tail)], np.sort(h, order=["nharm", "tpl", "bin"]), \
                _records(cbuf, ccount, fd.fdas.CANDIDATE_DTYPE)

        # thresholds from the data: about 2e-3 of the sums and of the last plane
        thr, cthr = [float("inf")] * 4, float("inf")
        x.copy_(xs[0])
        chain(True)
        q = float(torch.quantile(tail[::7].reshape(-1)[:1 << 20], 0.998))
        thr = [q * h for h in (1, 2, 4, 8)]
        last = plan.convolve(_link(tail, n))
        cthr = float(torch.quantile(last[::7].reshape(-1)[:1 << 20], 0.998))
        ref = []
        for v in xs:
            x.copy_(v)
            chain(True)
            ref.append(result())
        assert ref[0][1].size > 100 and ref[0][2].size > 100
        side = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=side):
            chain(False)
        for _ in range(10):
            for v, (planes, h, c) in zip(xs, ref):
                for t in (a, b, full, tail):
                    t.fill_(-1.0)
                x.copy_(v)
                for _ in range(3):
                    g.replay()
                got = result()
                assert all(torch.equal(p, r) for p, r in zip(planes, got[0]))
                np.testing.assert_array_equal(h, got[1])
                np.testing.assert_array_equal(c, got[2])
        plan.status()


@pytest.mark.parametrize("precision", ["FDAS_PREC_FP32", "FDAS_PREC_TC_DFT2"])
@pytest.mark.parametrize("n", [1 << 14, 300_001])
def test_input_from_another_stream(fd, bank, precision, n):
    # between two planes of one stream, that stream waits for the event of another, which writes the
    # second plane's input late; a third stream runs planes of its own on the SMs meanwhile
    xs = [_rand(n, 60 + i) for i in range(3)]
    slow = torch.zeros(64 << 20, device="cuda")
    with fd.Plan(bank, n_max=n, precision=getattr(fd, precision)) as plan:
        ref = [plan.convolve(x).clone() for x in xs]
        x = torch.empty_like(xs[0])
        s1, s2, s3 = (torch.cuda.Stream() for _ in range(3))
        outs = [torch.full((85, n), -1.0, device="cuda") for _ in range(24)]
        o0, o3 = (torch.empty((85, n), device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        for i, o in enumerate(outs):
            plan.convolve(xs[2], out=o0, stream=s1)
            with torch.cuda.stream(s2):
                slow.add_(1.0)
                x.copy_(xs[i % 2])
            plan.convolve(xs[1], out=o3, stream=s3)
            s1.wait_stream(s2)
            plan.convolve(x, out=o, stream=s1)
            s2.wait_stream(s1)
        torch.cuda.synchronize()
        for i, o in enumerate(outs):
            assert torch.equal(o, ref[i % 2])
        assert torch.equal(o0, ref[2]) and torch.equal(o3, ref[1])
        plan.status()
