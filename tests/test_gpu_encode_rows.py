"""A row's logits do not depend on the batch it is in: small batches (narrower
column tiles, shorter copies) give a large batch's rows bit for bit, for the
fused encoder and the layer-by-layer one."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import build_small, need_cuda
from paper_2608_15438_gb300.builder import build_index, config
from test_gpu_mlp import mlp_case
from test_gpu_tc_shapes import _rows, _weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=["fused", (512, (256, 128, 64), 12), (1536, (512, 256, 128, 64), 16),
                                        (128, (704, 192, 96 + 32), 20)], ids=str)
def case(request, tmp_path_factory):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    d = tmp_path_factory.mktemp("rows")
    if request.param == "fused":
        path, base, _ = build_small(d, "tiny", n=5_000, bits=12, name="rows")
        return torch, nr.Index(path, 0), base
    D, widths, b = request.param
    base, _, weights, widths, b = mlp_case(D, widths, b, 5_000)
    path = str(d / "rows.nrix")
    build_index(config("f32", D, widths[0], b, 4, 16, mid=widths[1:]), base, weights, path)
    return torch, nr.Index(path, 0), base


@pytest.mark.parametrize("n", [1, 4, 8, 9, 64, 127, 128, 129, 300, 1500])
def test_small_batches_equal_the_large_one(case, n):
    torch, ix, base = case
    x = torch.from_numpy(base).cuda()
    full = ix.encode(x)
    part = ix.encode(x[: n].contiguous())
    tail = ix.encode(x[3000: 3000 + n].clone())
    assert torch.equal(part, full[:n])
    assert torch.equal(tail, full[3000: 3000 + n])
    ix.last_stats()  # no wait expired


# one, two and three hidden chunks a tile against one, two and four tiles a CTA;
# fp32 rows of 12 and 16 pieces a thread (batches of six), the narrowest rows
@pytest.mark.parametrize("dtype,D,H,b", [("f32", 128, 384, 20), ("f32", 96, 128, 24), ("u8", 16, 256, 5)])
def test_fused_hand_offs(tmp_path, dtype, D, H, b):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    path = str(tmp_path / "enc.nrix")
    build_index(config(dtype, D, H, b, 4, 32), _rows(dtype, 4000, D, 1), _weights(D, H, b, 5), path)
    ix, orc = nr.Index(path, 0), oracle.Index(path)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    x = _rows(dtype, 4 * sms * 128 - 5, D, 2)
    dx = torch.from_numpy(x).cuda()
    full = ix.encode(dx)
    ref = orc.encode(x[:2000]).astype(np.float64)
    err = np.abs(full[:2000].cpu().numpy() - ref).max(1)
    assert (err <= 1e-2 * np.abs(ref).max(1)).all()  # the encoder's normwise bound
    for n in (1, 129, sms * 128 + 1, 2 * sms * 128):
        assert torch.equal(ix.encode(dx[:n].contiguous()), full[:n])
    ix.last_stats()  # no wait expired
    ix.close()
