"""FP32 planes whose blocks take equal shares of the (segment, template) units: bit for bit the plane
of whole template groups, at the ends of the range that takes shares (7 units per block; 45 for
2048-point segments), with shares inside one segment, across one boundary and over several."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _bank(m, k, seed):
    rng = np.random.default_rng(seed)
    return ((rng.standard_normal((m, k)) + 1j * rng.standard_normal((m, k))) / np.sqrt(2 * k)).astype(np.complex64)


@pytest.mark.parametrize("L", [1024, 2048, 4096])
@pytest.mark.parametrize("m,k,group", [(20, 100, 0), (85, 421, 0), (131, 33, 0), (150, 211, 1)])
def test_equal_shares_match_groups(L, m, k, group):
    import paper_1805_12280_gb300 as fd
    fd.load()
    h = _bank(m, k, m)
    if group:   # supports of different length
        for z in range(m):
            h[z, k - z:] = 0
    with fd.Plan(h, n_max=1 << 22, seg_len=L, group_support=group) as auto, \
            fd.Plan(h, n_max=1 << 22, seg_len=L, group_support=group, tpl_per_cta=5) as fixed:
        slots, S = auto.desc.batch_blocks, auto.desc.seg_step
        first = -(-7 * slots // m)          # segments from which shares are taken
        last = 45 * slots // m
        for nseg in (first - 1, first, first + 1, 2 * first + 1, last, last + 1, 3 * slots // 2):
            n = min((nseg - 1) * S + 1 + nseg % 7, 1 << 22)
            g = torch.Generator(device="cuda").manual_seed(nseg)
            x = torch.randn(n, 2, device="cuda", generator=g).view(torch.complex64).reshape(-1)
            a, b = (torch.full((m, n), -1.0, device="cuda") for _ in range(2))
            torch.cuda.synchronize()
            for _ in range(3):              # launches that overlap
                auto.convolve(x, out=a)
            fixed.convolve(x, out=b)
            auto.status()
            fixed.status()
            assert torch.equal(a, b)


def test_the_split_a_call_takes_is_reported():
    # the resident blocks where a call takes equal shares, at both ends of their range; 0: template groups
    import paper_1805_12280_gb300 as fd
    fd.load()
    h = _bank(85, 421, 1)
    with fd.Plan(h, n_max=1 << 22) as plan, fd.Plan(h, n_max=1 << 22, tpl_per_cta=17) as fixed, \
            fd.Plan(h, n_max=1 << 22, precision=fd.FDAS_PREC_TC_DFT2) as tc:
        slots, S = plan.desc.batch_blocks, plan.desc.seg_step
        first = -(-7 * slots // 85)
        for nseg, shares in ((1, 0), (first - 1, 0), (first, slots), (45 * slots // 85, slots), (45 * slots // 85 + 1, 0)):
            assert fd.fdas_plan_share_blocks(plan.handle, nseg * S) == shares
            assert fd.fdas_plan_tpl_per_cta(plan.handle, nseg * S) >= 1
            for other in (fixed, tc):
                assert fd.fdas_plan_share_blocks(other.handle, nseg * S) == 0
        for bad in (0, (1 << 22) + 1):
            with pytest.raises(fd.FdasError) as e:
                fd.fdas_plan_share_blocks(plan.handle, bad)
            assert e.value.code == fd.fdas.FDAS_ERR_INVALID_ARG
    with fd.Plan(h, n_max=1 << 22, group_support=1) as plan:
        assert fd.fdas_plan_share_blocks(plan.handle, 1) == 0
