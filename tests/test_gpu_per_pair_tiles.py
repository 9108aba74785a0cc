"""Per-pair thresholds at every tile size (128 to 1024 pairs, chosen by the
number of pairs), with tiles that are sorted and tiles that keep their order, a
partial last tile, N, invalid pairs and their count, against the oracle on a
sample, the last tile and the tile edges (tolerance 0)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2103_14978_gb300 import device_data as dd, gk
from tests.gpu_helpers import GpuRun, oracle_run, require_gpu, small_workload

pytestmark = pytest.mark.gpu

THRESHOLDS = {
    "one": [2], "close": [0, 1, 2], "spread": [3, 8, 15, 25, 30], "past 30": [2, 30, 31, 32, 33, 46, 47, 62, 63, 64, 126,
                                                                           127, 200, 254, 255],
}


@pytest.mark.parametrize("m", [20, 33, 50, 64, 76, 100, 128, 150, 157, 170, 200, 250, 256, 300, 330, 512])
@pytest.mark.parametrize("n", [400_003, 700_001, 1_200_001, 2_300_001, 4_100_001])
def test_every_tile_size(m, n):
    require_gpu()
    if n == 4_100_001 and not 32 < m <= 64:  # from there on those sort as well
        n = 3
    w = small_workload(m, 40_000, seed=6000 + m, n_frac=0.0005 if m < 300 else 0.002, read_n_frac=0.0005, cands=5)
    rng = np.random.default_rng(m + n)
    pick = rng.integers(0, w.n_pairs, n)
    w.pair_read, w.pair_off = w.pair_read[pick].copy(), w.pair_off[pick].copy()
    w.pair_read[rng.integers(0, n, 9)] = w.n_reads
    w.pair_off[rng.integers(0, n, 9)] = w.ref.shape[0] - m + 1
    run = GpuRun(w)
    r = run.reads
    idx = np.unique(np.concatenate([rng.integers(0, n, 4000), np.arange(max(0, n - 1500), n), np.arange(min(n, 300))]))
    for name, values in THRESHOLDS.items():
        w.pair_e = rng.choice(np.array(values, np.uint8), n)
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        acc, ed = gk.gk_filter(run.ref, r.packed, r.stride_words, r.n_reads, r.nflag, m, run.pairs.pair_read,
                               run.pairs.pair_off, torch.from_numpy(w.pair_e).cuda(), err_count=err)
        torch.cuda.synchronize()
        acc, ed = acc.cpu().numpy(), dd.edits_u16(ed)
        want_a, want_e = oracle_run(w, idx=idx)
        bad = np.nonzero((acc[idx] != want_a) | (ed[idx] != want_e))[0]
        assert bad.size == 0, (m, n, name, idx[bad[:5]], ed[idx[bad[:5]]], want_e[bad[:5]])
        assert int(err.item()) == int((ed == O.INVALID).sum()) == int(
            ((w.pair_read >= w.n_reads) | (w.pair_off > w.ref.shape[0] - m)).sum())
