"""Device encoder against the host encoder for rows that are mostly padding and
rows that are not: lengths around the 16-byte pieces, the last row's padding
not there, a partial last tile, N in the reads."""
import numpy as np
import pytest
import torch

from paper_2103_14978_gb300 import gk
from tests.gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stride", [160, 192, 512, 1024])
@pytest.mark.parametrize("m", [1, 15, 16, 17, 76, 80, 81, 96, 160])
def test_padded_rows(m, stride):
    require_gpu()
    sw = 3 if m <= 96 else 5  # no power of two: rows staged in tiles
    for n in (1, 2, 1001):
        rng = np.random.default_rng(1000 * m + stride + n)
        buf = rng.choice(np.frombuffer(b"ACGTacgtN", np.uint8), (n - 1) * stride + m)
        dev = torch.from_numpy(buf).cuda()
        host = torch.from_numpy(buf)
        got = gk.gk_encode(dev, n, stride, fixed_len=m, stride_words=sw)
        want = gk.gk_encode(host, n, stride, fixed_len=m, stride_words=sw)
        torch.cuda.synchronize()
        assert torch.equal(got[0].cpu(), want[0]) and torch.equal(got[1].cpu(), want[1]), (m, stride, n)
        full = torch.from_numpy(np.concatenate([buf, np.full(stride - m, 67, np.uint8)]))
        lens = torch.from_numpy(rng.integers(0, m + 1, n).astype(np.int16))
        got = gk.gk_encode(full.cuda(), n, stride, lens=lens.cuda(), stride_words=sw)
        want = gk.gk_encode(full, n, stride, lens=lens, stride_words=sw)
        torch.cuda.synchronize()
        assert torch.equal(got[0].cpu(), want[0]) and torch.equal(got[1].cpu(), want[1]), ("lens", m, stride, n)
