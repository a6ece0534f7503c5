"""A row's logits do not depend on the batch it is in: small batches (narrower
column tiles, shorter copies) give a large batch's rows bit for bit, for the
fused encoder and the layer-by-layer one."""
import numpy as np
import pytest

import synth
from gpu_util import build_small, need_cuda
from test_gpu_mlp import mlp_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=["fused", (512, (256, 128, 64), 12), (1536, (512, 256, 128, 64), 16),
                                        (128, (704, 192, 96 + 32), 20)], ids=str)
def case(request, tmp_path_factory):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr
    from paper_2608_15438_gb300.builder import build_index, config

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
