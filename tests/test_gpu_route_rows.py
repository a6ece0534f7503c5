"""A query's probe list does not depend on the batch it is in: few queries run
in wider blocks and give a large batch's lists, for every form of the threshold
enumeration and its fallbacks (many equal costs, subtrees beyond the capacity),
at the ends of the rule's range. Where few buckets are occupied, a non-empty
budget takes the larger enumeration or the heap: the oracle's lists."""
import numpy as np
import pytest

import oracle
from gpu_util import build_small, need_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case(tmp_path_factory):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    path, base, _ = build_small(tmp_path_factory.mktemp("route"), "tiny", n=20_000, bits=16, name="route")
    ix = nr.Index(path, 0)
    lg = np.random.default_rng(3).normal(size=(600, 16)).astype(np.float32)
    lg[1::3] = np.round(lg[1::3] * 2) / 2      # many equal costs
    lg[2::7] = ix.thresholds()   # every deviation zero
    return torch, ix, torch.from_numpy(lg).cuda()


@pytest.mark.parametrize("P", [1, 2, 64, 129, 1024, 4096])
@pytest.mark.parametrize("kw", [{}, dict(nonempty_budget=1), dict(l_sel=9), dict(s_max=1.5),
                                dict(nonempty_budget=1, l_sel=12, s_max=2.5)], ids=str)
def test_few_queries_equal_a_large_batch(case, P, kw):
    torch, ix, lg = case
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if not kw:
        ix.set_params()
    ix.set_params(**kw)
    codes, n = ix.route(lg, P)
    for a, b in ((0, 1), (1, 2), (2, 3), (5, 5 + sms), (5, 6 + sms), (20, 60)):
        c, m = ix.route(lg[a:b].contiguous(), P)
        assert torch.equal(m, n[a:b])
        assert torch.equal(c, codes[a:b])
    ix.set_params()


# 16 bits over 3,000 rows: one bucket in some twenty is occupied, so 2 P flip
# sets never hold P non-empty ones
@pytest.mark.parametrize("P", [4, 60, 512, 1024, 1536, 2048])
@pytest.mark.parametrize("kw", [{}, dict(l_sel=11), dict(s_max=2.0)], ids=str)
def test_non_empty_budget_over_few_buckets(tmp_path, P, kw):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    path, base, _ = build_small(tmp_path, "tiny", n=3_000, bits=16, name="sparse")
    ix, orc = nr.Index(path, 0), oracle.Index(path)
    lg = np.random.default_rng(4).normal(size=(300, 16)).astype(np.float32)
    lg[1::5] = np.round(lg[1::5] * 2) / 2
    ix.set_params(nonempty_budget=1, **kw)
    codes, n = ix.route(torch.from_numpy(lg).cuda(), P)
    few, nfew = ix.route(torch.from_numpy(lg[:100]).cuda(), P)
    assert torch.equal(few, codes[:100]) and torch.equal(nfew, n[:100])
    codes, n = codes.cpu().numpy().view(np.uint32), n.cpu().numpy()
    p = oracle.params(nonempty_budget=1, **kw)
    for i in range(0, 300, 7):
        exp, _ = orc.probe_list(lg[i], P, p)
        assert n[i] == len(exp) and np.array_equal(codes[i, :n[i]], exp), i
        assert np.all(codes[i, n[i]:] == 0xFFFFFFFF)
    ix.close()
    orc.close()
