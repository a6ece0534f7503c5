"""nr_index_locate with few ids (found through the filters) and many (searched
directly, or where the device has no memory for the filters): repeats, ids that
are not stored, negative and 2^32-range ids."""
import numpy as np
import pytest

from gpu_util import build_small, need_cuda
from nrix_reader import read_nrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 7_499, 7_500, 40_000])
def test_locate_matches_the_stored_order(tmp_path, n):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    path, _, _ = build_small(tmp_path, "tiny", n=30_000, bits=10, name="loc")
    a = read_nrix(path)
    rng = np.random.default_rng(n)
    ids = rng.integers(0, 30_000, n)
    odd = rng.random(n) < 0.2
    ids[odd] = rng.choice(np.array([-1, -5, 30_000, 2**19, 2**19 + 3, 2**27 + 7, 2**32 - 1, 2**33 + 1]), odd.sum())
    ix = nr.Index(path, 0)
    got = ix.locate(torch.from_numpy(ids).cuda()).cpu().numpy()
    ix.close()
    pos = np.full(30_000, -1)
    pos[a["ids"].astype(np.int64)] = np.arange(30_000)
    ok = (ids >= 0) & (ids < 30_000)
    p = pos[np.where(ok, ids, 0)]
    c = np.searchsorted(a["cl_off"], p, side="right") - 1
    u = np.searchsorted(a["bkt_off"], c, side="right") - 1
    first, last = a["bkt_off"][u].astype(np.int64), a["bkt_off"][u + 1].astype(np.int64)
    exp = np.stack([c, u, first, last - first], 1)
    exp[~ok] = (-1, -1, -1, 0)
    assert np.array_equal(got, exp)


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_locate_into_a_buffer_at_any_int32(tmp_path, offset):
    """d_out need be no more aligned than int32; nothing beside it is written."""
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    path, _, _ = build_small(tmp_path, "tiny", n=30_000, bits=10, name="loc")
    ix = nr.Index(path, 0)
    ids = torch.randint(-10, 30_010, (5_000,), device="cuda")
    exp = ix.locate(ids)
    buf = torch.full((5_000 * 4 + 4,), 7, dtype=torch.int32, device="cuda")
    assert buf.data_ptr() % 16 == 0
    out = buf[offset:offset + 5_000 * 4]
    assert nr.lib().nr_index_locate(ix.h, ids.data_ptr(), 5_000, out.data_ptr(), None) == 0
    ix.close()
    assert torch.equal(out.view(-1, 4), exp)
    assert buf[:offset].eq(7).all() and buf[offset + 5_000 * 4:].eq(7).all()


def test_locate_without_memory_for_the_filters(tmp_path):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    path, _, _ = build_small(tmp_path, "tiny", n=30_000, bits=10, name="loc")
    ix = nr.Index(path, 0)
    ids = torch.randint(-10, 30_010, (7_499,), device="cuda")
    exp = ix.locate(ids)
    out = torch.zeros_like(exp)
    torch.cuda.synchronize()
    # the filters of 7,499 ids take 4.1 MB, the rest 0.2
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (4 << 20), dtype=torch.uint8, device="cuda")
    assert nr.lib().nr_index_locate(ix.h, ids.data_ptr(), 7_499, out.data_ptr(), None) == 0
    assert torch.cuda.mem_get_info()[0] < 4_100_000
    del fill
    torch.cuda.empty_cache()
    ix.close()
    assert torch.equal(out, exp)
