"""Small searches launch their kernels early, each waiting for the one before:
back to back on one stream, on two streams at once, and captured into a graph
and replayed, they give the large batch's results."""
import pytest

from gpu_util import build_small, need_cuda
from test_gpu_mlp import mlp_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=["fused", "layers"])
def case(request, tmp_path_factory):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr
    from paper_2608_15438_gb300.builder import build_index, config

    d = tmp_path_factory.mktemp("chain")
    path = str(d / "chain.nrix")
    if request.param == "fused":
        path, base, _ = build_small(d, "tiny", n=20_000, bits=10, name="chain")
    else:
        base, _, weights, widths, b = mlp_case(128, (256, 128, 64), 10, 20_000)
        build_index(config("f32", 128, widths[0], b, 4, 16, mid=widths[1:]), base, weights, path)
    ix = [nr.Index(path, 0) for _ in range(2)]
    q = torch.from_numpy(base[:600].copy()).cuda()
    ids, dist = ix[0].search(q, 10, 64, 128)
    torch.cuda.synchronize()
    return torch, ix, q, ids.clone(), dist.clone()


@pytest.mark.parametrize("n", [1, 40, 128, 129, 152, 153])
def test_back_to_back_and_two_streams(case, n):
    torch, ix, q, ids, dist = case
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = []
    torch.cuda.synchronize()
    for r in range(20):
        for j in range(2):
            a = (37 * r + 11 * j) % (600 - n)
            with torch.cuda.stream(streams[j]):
                i, d = ix[j].search(q[a:a + n], 10, 64, 128)
                got.append((a, i, d))
    torch.cuda.synchronize()
    for a, i, d in got:
        assert torch.equal(i, ids[a:a + n]) and torch.equal(d, dist[a:a + n])


@pytest.mark.parametrize("entry", ["search", "search_static"])
def test_captured_and_replayed(case, entry):
    torch, (ix, _), q, ids, dist = case
    call = getattr(ix, entry)
    x = q[:40].clone()
    call(x, 10, 64, 128)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        i, d = call(x, 10, 64, 128)
    for a in (0, 100, 333):
        x.copy_(q[a:a + 40])
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(i, ids[a:a + 40]) and torch.equal(d, dist[a:a + 40])


@pytest.mark.parametrize("n", [1, 7, 40, 128, 153, 300])
def test_cut_streams_back_to_back(case, n):
    """Without an early stop these batches' streams are cut into spans, whose
    logs one block commits for another (the batch of 600 keeps them whole)."""
    torch, ix, q, _, _ = case
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = []
    for x in ix:
        x.set_params(t_low=0)
    try:
        ids, dist = (v.clone() for v in ix[0].search(q, 10, 256, 1024))
        torch.cuda.synchronize()
        for r in range(20):
            for j in range(2):
                a = (37 * r + 11 * j) % (600 - n)
                with torch.cuda.stream(streams[j]):
                    i, d = ix[j].search(q[a:a + n], 10, 256, 1024)
                    got.append((a, i, d))
        torch.cuda.synchronize()
    finally:
        for x in ix:
            x.set_params()
    for a, i, d in got:
        assert torch.equal(i, ids[a:a + n]) and torch.equal(d, dist[a:a + n])
