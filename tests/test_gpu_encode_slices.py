"""The layer kernel's fp32 first layer, slice by slice: rows that hold s + 1 in
every value of 64-value slice s, and a hidden unit per slice that sums it. Each
logit is then the exact 64 (s + 1): a value taken from another slice (of a
stage refilled too early, or read before its copy landed) shows in it, on any
of the repeated calls. 64 and 256 columns run with four and two raw stages;
192 columns leave room for three."""
import numpy as np
import pytest

from gpu_util import need_cuda
from paper_2608_15438_gb300.builder import build_index, config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,n", [(64, 4000), (256, 4000), (192, 20_000)])
def test_every_slice_is_its_own(tmp_path, hidden, n):
    torch = need_cuda()
    from paper_2608_15438_gb300 import neuroute as nr

    D, S = 1536, 24
    W1, W2, W3 = (np.zeros(s, np.float32) for s in ((hidden, D), (64, hidden), (S, 64)))
    for s in range(S):
        W1[s, 64 * s:64 * s + 64] = 1.0
        W2[s, s] = W3[s, s] = 1.0
    zeros = [np.zeros(k, np.float32) for k in (hidden, 64, S)]
    base = np.random.default_rng(1).normal(size=(4000, D)).astype(np.float32)
    path = str(tmp_path / "slices.nrix")
    build_index(config("f32", D, hidden, S, 4, 16, mid=(64,)), base,
                (W1, zeros[0], W3, zeros[2], ((W2, zeros[1]),)), path)
    ix = nr.Index(path, 0)
    x = (torch.arange(D, device="cuda") // 64 + 1).float().expand(n, D).contiguous()
    want = 64.0 * (torch.arange(S, device="cuda") + 1).float()
    wrong = sum((ix.encode(x) != want).sum() for _ in range(100))
    assert int(wrong) == 0
    ix.close()
