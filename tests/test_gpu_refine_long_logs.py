"""Streams of which nearly every row enters the top-k: the logs of their spans are
longer than a commit stages, and together longer than the pool, so that the
spans without room for one are refined again when their turn comes. For k up to
32 a warp commits, above the block; ids, distances, rows and rounds equal the
oracle's sequential refinement."""
import numpy as np
import pytest

import oracle
from gpu_util import need_cuda
from nrix_writer import write_nrix

pytestmark = pytest.mark.gpu

N = 150_000  # rows of the one cluster, each nearer to the queries than those before it
NQ = 12
# entries of the log pool of at most 128 queries
POOL = {k: 4096 * k for k in (1, 20, 33, 100)}


@pytest.fixture(scope="module", params=[("u8", 128), ("u8", 48), ("f32", 96), ("f32", 20), ("f32", 288)],
                ids=lambda p: f"{p[0]}-{p[1]}")
def index(request, tmp_path_factory):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    dtype, D = request.param
    b, rng = 4, np.random.default_rng(D)
    vec = np.zeros((N, D), np.uint8 if dtype == "u8" else np.float32)
    # few distances: the ids fall along the stream and order the rows of one
    vec[:, 0] = 255 - np.arange(N) * 256 // N
    vec[:, 1] = rng.integers(0, 2, N)  # every second row or so a little further away
    q = np.zeros((NQ, D), vec.dtype)
    q[:, 2] = np.arange(NQ)
    path = str(tmp_path_factory.mktemp("logs") / "logs.nrix")
    off = np.zeros((1 << b) + 1, np.int64)
    off[1:] = 1
    write_nrix(path, vec, np.arange(N)[::-1], off, [0, N], np.zeros((1, b)), np.zeros(b) + 0.5,
               np.zeros((16, D)), np.zeros(16), np.zeros((b, 16)), np.zeros(b), K_max=1)
    return torch, nr.Index(path, 0), oracle.Index(path), q, np.zeros((NQ, b), np.float32)


# no stop, and one after 1,500 and after 300 rounds
@pytest.mark.parametrize("kw", [dict(t_low=0, round_size=32), dict(t_low=0, round_size=256),
                                dict(t_low=1500, round_size=32, u_min=1 << 20, f_min=1 << 20),
                                dict(t_low=300, round_size=64, u_min=1 << 20, f_min=1 << 20)],
                         ids=["r32", "r256", "r32-stop", "r64-stop"])
@pytest.mark.parametrize("k", sorted(POOL))
def test_logs_longer_than_their_pool(index, k, kw):
    torch, ix, orc, q, lg = index
    # members logged: of a round's rows at least a quarter enter, and k stay
    R = kw["round_size"]
    assert NQ * (N // R) * min(k, R // 4) > POOL[k]
    ix.set_params(**kw)
    try:
        ids, d = ix.search_logits(torch.from_numpy(q).cuda(), torch.from_numpy(lg).cuda(), k, 4, 1)
        st = ix.query_stats(NQ).cpu().numpy()
    finally:
        ix.set_params()
    ids_o, d_o, st_o = orc.search(q, k, 4, 1, oracle.params(**kw), logits=lg)
    assert np.array_equal(ids.cpu().numpy(), ids_o)
    assert np.array_equal(d.cpu().numpy(), d_o)
    assert np.array_equal(st, st_o)
