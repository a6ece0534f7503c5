"""Small batches, whose candidate streams are cut into spans refined by many
blocks and committed in stream order: ids, distances, rows and rounds equal the
oracle's sequential refinement (whole numbers and a fixed fp32 chain: exact)."""
import numpy as np
import pytest

import oracle
from gpu_util import build_small, need_cuda
from test_gpu_mlp import mlp_case

pytestmark = pytest.mark.gpu

# (queries, k, parameters): streams of one span and of many; rounds shorter
# than a tile, of a tile's multiple and longer than a stream; a stop in the
# first span, in a later one and never; front and first-round rules; k = 1 with
# short rounds logs more entries than their pool holds (those spans are
# refined again when they are committed)
CASES = [(1, 10, dict(t_low=0)), (1, 10, dict(t_low=20)), (3, 10, dict(t_low=4)), (2, 1, dict(t_low=0)),
         (5, 100, dict(t_low=16)), (2, 256, dict(t_low=0, round_size=64)),
         (64, 1, dict(t_low=0, round_size=32)), (64, 1, dict(t_low=200, round_size=32)),
         (7, 10, dict(t_low=3, round_size=4096)), (9, 10, dict(t_low=2, round_size=1024, r_min=6)),
         (4, 20, dict(t_low=5, round_size=128, u_min=3, f_min=2, alpha_front=0.7)),
         (4, 10, dict(t_low=2, u_min=0, f_min=1)), (100, 10, dict(t_low=8))]
IDS = [f"nq{n}-k{k}-" + "-".join(f"{a}{v}" for a, v in kw.items()) for n, k, kw in CASES]


@pytest.fixture(scope="module", params=["u8", "f32", "long", "wide"])
def index(request, tmp_path_factory):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr
    from paper_2608_15438_gb300.builder import build_index, config

    d = tmp_path_factory.mktemp(f"spans_{request.param}")
    rng = np.random.default_rng(5)
    if request.param == "u8":
        path, base, _ = build_small(d, "tiny", n=60_000, bits=10, name="u8")
    elif request.param == "f32":
        path, base, _ = build_small(d, "f32-10m", n=30_000, bits=9, name="f32")
    elif request.param == "long":
        base, _, weights, widths, b = mlp_case(512, (256, 128, 64), 8, 12_000)
        path = str(d / "long.nrix")
        build_index(config("f32", 512, widths[0], b, 4, 16, mid=widths[1:]), base, weights, path)
    else:  # uint8 rows of 640 bytes: the generic tile
        base = rng.integers(0, 256, (20_000, 640), dtype=np.uint8)
        path = str(d / "wide.nrix")
        W = (rng.normal(size=(64, 640)).astype(np.float32) / 25, np.zeros(64, np.float32),
             rng.normal(size=(8, 64)).astype(np.float32) / 8, np.zeros(8, np.float32))
        build_index(config("u8", 640, 64, 8, 4, 32), base, W, path)
    orc = oracle.Index(path)
    # queries near stored rows, so that early rounds fill the top-k and later ones still change it
    q = base[rng.integers(0, len(base), 100)]
    if request.param in ("f32", "long"):
        q = (q + rng.normal(size=q.shape) * 0.02).astype(np.float32)
    return torch, nr.Index(path, 0), orc, np.ascontiguousarray(q), orc.encode(q)


@pytest.mark.parametrize("case", CASES, ids=IDS)
def test_spans_equal_the_sequential_refinement(index, case):
    torch, ix, orc, q, lg = index
    nq, k, kw = case
    P, C = 256, 1024
    ix.set_params(**kw)
    try:
        ids, d = ix.search_logits(torch.from_numpy(q[:nq]).cuda(), torch.from_numpy(lg[:nq]).cuda(), k, P, C)
        st = ix.query_stats(nq).cpu().numpy()
    finally:
        ix.set_params()
    ids_o, d_o, st_o = orc.search(q[:nq], k, P, C, oracle.params(**kw), logits=lg[:nq])
    assert np.array_equal(ids.cpu().numpy(), ids_o)
    assert np.array_equal(d.cpu().numpy(), d_o)
    assert np.array_equal(st, st_o)
