"""The search workspace: a batch whose streams stay whole takes no room for spans
beyond what the largest cut batch needs, a smaller batch after a larger one needs
no more, and a capture that would need more keeps its streams whole, as does a
call for whose spans there is no device memory."""
import numpy as np
import pytest

from gpu_util import build_small, need_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture
def index(tmp_path):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    path, base, _ = build_small(tmp_path, "tiny", n=20_000, bits=10, name="ws")
    ix = nr.Index(path, 0)
    q = torch.from_numpy(np.tile(base, (2, 1))[:30_000].copy()).cuda()
    yield torch, ix, q
    ix.close()


def used(torch, call):
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    call()
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0]


def buffers(torch, nq, k):
    return (torch.empty((nq, k), dtype=torch.int64, device="cuda"),
            torch.empty((nq, k), dtype=torch.float32, device="cuda"))


def test_whole_streams_take_no_room_for_spans(index):
    torch, ix, q = index
    ix.search(q[:1], 1, 8, 16)  # modules are loaded
    out = buffers(torch, 30_000, 100)
    # 30,000 queries with their lists are some 15 MB; logs and flags for all were
    # 300 MB, those of the queries that may be cut some 60 MB at most
    assert used(torch, lambda: ix.search(q, 100, 8, 16, out=out)) < 120 << 20
    # smaller batches, cut or not, fit it (a kernel may be loaded at its first launch)
    ix.set_params(t_low=0)
    assert used(torch, lambda: [ix.search(q[:n], 100, 8, 16, out=tuple(o[:n] for o in out))
                                for n in (1, 100, 300, 600, 2_000)]) < 8 << 20
    ix.set_params()


def test_captured_after_calls_of_a_smaller_k(index, tmp_path):
    torch, ix, q = index
    from paper_2608_15438_gb300 import neuroute as nr

    ids, dist = (v.clone() for v in ix.search(q[:2_000], 100, 64, 128))
    fresh = nr.Index(str(tmp_path / "ws.nrix"), 0)
    x, out = q[:40].clone(), buffers(torch, 40, 100)
    fresh.search(x, 1, 64, 128)  # its workspace: too small to cut at k = 100
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fresh.search(x, 100, 64, 128, out=out)
    for a in (0, 300):
        x.copy_(q[a:a + 40])
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out[0], ids[a:a + 40]) and torch.equal(out[1], dist[a:a + 40])
    fresh.close()


def test_without_memory_for_spans(index, tmp_path):
    torch, ix, q = index
    from paper_2608_15438_gb300 import neuroute as nr

    k, P, C = 100, 8, 16
    ix.set_params(t_low=0)
    # both kinds of kernels are loaded: 2,000 queries stay whole, 400 are cut
    ids, dist = (v[:400].clone() for v in ix.search(q[:2_000], k, P, C))
    ix.search(q[:400], k, P, C)
    fresh = nr.Index(str(tmp_path / "ws.nrix"), 0)
    fresh.set_params(t_low=0)
    fresh.search(q[:1], 1, P, C)
    out = buffers(torch, 400, k)
    torch.cuda.synchronize()
    # the logs of 400 queries take 20 MB, the batch without them 1 MB or so
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (12 << 20), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        for o in out:
            o.zero_()
        fresh.search(q[:400], k, P, C, out=out)
        torch.cuda.synchronize()
        assert torch.equal(out[0], ids) and torch.equal(out[1], dist)
    del fill
    torch.cuda.empty_cache()
    fresh.search(q[:400], k, P, C, out=out)
    torch.cuda.synchronize()
    assert torch.equal(out[0], ids) and torch.equal(out[1], dist)
    fresh.close()
