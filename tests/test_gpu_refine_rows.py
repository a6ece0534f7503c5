"""Every row size's tile, as spans (few queries) and as whole streams (many, by
length and by code): a query's answer is the oracle's and does not depend on the
batch it is in, nor on the batch being pipelined."""
import numpy as np
import pytest

import oracle
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu

# uint8 rows of 128 bytes, up to 512 and above; short fp32 rows, 96 values, up to
# 128 and 256; rows in pieces of 4, 8 and 16 chunks
ROWS = [("u8", 128), ("u8", 48), ("u8", 512), ("u8", 528), ("f32", 20), ("f32", 96), ("f32", 128),
        ("f32", 200), ("f32", 272), ("f32", 288), ("f32", 320)]
NQ = 4200


@pytest.fixture(scope="module", params=ROWS, ids=lambda r: f"{r[0]}-{r[1]}")
def index(request, tmp_path_factory):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr
    from paper_2608_15438_gb300.builder import build_index, config

    dtype, D = request.param
    rng = np.random.default_rng(D)
    centres = rng.normal(size=(64, D))
    x = centres[rng.integers(0, 64, 16_000)] + 0.4 * rng.normal(size=(16_000, D))
    base = (np.clip(x * 40 + 128, 0, 255).astype(np.uint8) if dtype == "u8" else x.astype(np.float32))
    W = (rng.normal(size=(64, D)).astype(np.float32) / np.sqrt(D).astype(np.float32), np.zeros(64, np.float32),
         rng.normal(size=(9, 64)).astype(np.float32) / 8, np.zeros(9, np.float32))
    path = str(tmp_path_factory.mktemp("rows") / "rows.nrix")
    build_index(config(dtype, D, 64, 9, 4, 32), base, W, path)
    q = base[rng.integers(0, len(base), NQ)]
    if dtype == "f32":
        q = (q + 0.05 * rng.normal(size=q.shape)).astype(np.float32)
    orc = oracle.Index(path)
    return torch, nr.Index(path, 0), orc, np.ascontiguousarray(q), orc.encode(q)


# (k, P, C, t_low): both shapes of the uint8 x 128 tile, the block's commit and the warp's
@pytest.mark.parametrize("k,P,C,t_low", [(10, 64, 1024, 0), (10, 64, 64, 4), (100, 64, 128, 16), (33, 256, 512, 0)])
def test_answers_do_not_depend_on_the_batch(index, k, P, C, t_low):
    torch, ix, orc, q, lg = index
    dq, dl = torch.from_numpy(q).cuda(), torch.from_numpy(lg).cuda()
    ix.set_params(t_low=t_low)
    try:
        ids, d = ix.search_logits(dq, dl, k, P, C)
        st = ix.query_stats(NQ).clone()
        for a, n in ((0, 1), (3, 40), (100, 150), (300, 700)):
            i, e = ix.search_logits(dq[a:a + n].contiguous(), dl[a:a + n].contiguous(), k, P, C)
            assert torch.equal(i, ids[a:a + n]) and torch.equal(e, d[a:a + n]), (a, n)
            assert torch.equal(ix.query_stats(n), st[a:a + n]), (a, n)
        for pc in (60, 1000):
            ix.set_params(t_low=t_low, pipe_chunk=pc)
            i, e = ix.search_logits(dq[:1100].contiguous(), dl[:1100].contiguous(), k, P, C)
            torch.cuda.synchronize()
            assert torch.equal(i, ids[:1100]) and torch.equal(e, d[:1100]), pc
    finally:
        ix.set_params()
    n = 40
    ids_o, d_o, st_o = orc.search(q[:n], k, P, C, oracle.params(t_low=t_low), logits=lg[:n])
    assert np.array_equal(ids[:n].cpu().numpy(), ids_o)
    assert np.array_equal(d[:n].cpu().numpy(), d_o)
    assert np.array_equal(st[:n].cpu().numpy(), st_o)
