"""Streams of one-row clusters with clusters without rows between them, as a
file may hold them (the builders drop such clusters): every stream row is the
one of the last segment that begins at or before it, so ids, distances, rows
and rounds equal the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import need_cuda
from nrix_writer import write_nrix

pytestmark = pytest.mark.gpu


def write_index(path, dtype, D, lens, order):
    """One cluster a bucket; cluster c holds lens[c] rows and is the
    order[c]-th nearest to logits that equal the first centroid."""
    b = 10
    n, rng = len(lens), np.random.default_rng(3)
    assert n == 1 << b
    cl_off = np.concatenate([[0], np.cumsum(lens)])
    # rows past the last cluster: a row read from a segment without rows is
    # inside the array as well
    N = int(cl_off[-1]) + 4
    vec = (rng.integers(0, 256, (N, D)).astype(np.uint8) if dtype == "u8"
           else rng.normal(size=(N, D)).astype(np.float32))
    cent = np.zeros((n, b), np.float32)
    cent[:, 0] = 1.0 + np.asarray(order, np.float32) / n
    cl = np.concatenate([cl_off[:-1], [N]])  # the last cluster holds them
    write_nrix(path, vec, rng.permutation(N), np.arange(n + 1), cl, cent, np.zeros(b),
               np.zeros((16, D)), np.zeros(16), np.zeros((b, 16)), np.zeros(b), K_max=1)
    return vec


# rows of the clusters in list order. The first: a warp's 32 segments of which
# the last has no rows and is followed by the one with the warp's last row
def pattern(name, n):
    rng = np.random.default_rng(11)
    if name == "crafted":
        lens = np.ones(n, np.int64)
        lens[31::33] = 0
    elif name == "sparse":
        lens = (rng.random(n) > 0.04).astype(np.int64)
    else:
        lens = rng.choice([0, 1, 2, 40], n, p=[0.3, 0.6, 0.05, 0.05])
    return lens


@pytest.mark.parametrize("dtype,D", [("u8", 128), ("u8", 32), ("f32", 96), ("f32", 20)])
@pytest.mark.parametrize("name", ["crafted", "sparse", "mixed"])
def test_rows_behind_segments_without_rows(tmp_path, dtype, D, name):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    n, b, nq = 1 << 10, 10, 12
    rng = np.random.default_rng(7)
    order = rng.permutation(n)  # of the clusters as stored
    lens = pattern(name, n)[order]
    path = str(tmp_path / "empty.nrix")
    vec = write_index(path, dtype, D, lens, order)
    ix, orc = nr.Index(path, 0), oracle.Index(path)
    lg = np.full((nq, b), 1e-3, np.float32)
    lg[:, 0] = 1.0
    lg[nq // 2:, 0] = 1.0 + rng.random(nq - nq // 2)  # another order of the clusters
    q = vec[rng.integers(0, len(vec), nq)].copy()
    for kw in (dict(t_low=0), dict(t_low=0, round_size=32), dict(t_low=2)):
        ix.set_params(**kw)
        ids, d = ix.search_logits(torch.from_numpy(q).cuda(), torch.from_numpy(lg).cuda(), 256, n, n)
        st = ix.query_stats(nq).cpu().numpy()
        ids_o, d_o, st_o = orc.search(q, 256, n, n, oracle.params(**kw), logits=lg)
        assert np.array_equal(ids.cpu().numpy(), ids_o)
        assert np.array_equal(d.cpu().numpy(), d_o)
        assert np.array_equal(st, st_o)
    ix.close()
