"""The GPU build's k-means at the edges of its bucket classes (a warp up to 256
rows, a CTA up to 1,024, a larger CTA above, sums folded every 65,536 rows) and
of its fixed point (scales that fp32 holds and one it does not, subnormal
logits, widths that are and are not multiples of four): the same bytes as the
host builder's."""
import numpy as np
import pytest

from gpu_util import need_cuda
from paper_2608_15438_gb300.builder import config
from test_gpu_build import same_as_host

pytestmark = pytest.mark.gpu


def sized_logits(sizes, b, scale, seed):
    """Logits whose buckets hold about these rows: a bucket and its complement
    get the same number, so every column's median lies between the signs."""
    rng = np.random.default_rng(seed)
    codes = np.concatenate([np.full(n, u, np.int64) for c, n in enumerate(sizes) for u in (c, (1 << b) - 1 - c)])
    rng.shuffle(codes)
    bits = (codes[:, None] >> np.arange(b)) & 1
    # a few groups per bucket, so that clusters differ in size
    mag = rng.integers(1, 5, (len(codes), b)) + 0.2 * rng.random((len(codes), b))
    return (np.where(bits == 1, mag, -mag) * scale).astype(np.float32)


@pytest.mark.parametrize("sizes,b,kmax,t,scale", [
    ((255, 256, 257, 258, 40, 1, 2), 4, 16, 32, 1.0),
    ((1023, 1024, 1025, 1026), 3, 8, 64, 1e-3),
    ((70_000, 300), 2, 4, 64, 1.0),
    ((66_000, 600), 2, 1, 64, 1e30),
    ((300, 1100, 30), 5, 16, 16, 1e-31),
    ((300, 1100), 4, 8, 16, 1e-40),
    ((500, 90, 260), 20, 16, 16, 100.0),
    ((400, 1500), 24, 64, 8, 1.0),
])
def test_bucket_classes_same_bytes_as_host_builder(tmp_path, sizes, b, kmax, t, scale):
    torch = need_cuda()
    logits = sized_logits(sizes, b, scale, seed=b)
    n = len(logits)
    rng = np.random.default_rng(1)
    base = rng.integers(0, 256, (n, 16), dtype=np.uint8)
    weights = (np.zeros((8, 16), np.float32), np.zeros(8, np.float32), np.zeros((b, 8), np.float32),
               np.zeros(b, np.float32))
    same_as_host(tmp_path, torch, config("u8", 16, 8, b, kmax, t), base, logits, weights)
