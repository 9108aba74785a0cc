"""The batched filter's routes (one pair per lane) on both sides of every size
at which they change: tile sizes of launches filtered in their tiles, the first
sizes that go through records, one filter launch for all lengths and one per
range; mixed lengths, thresholds far above 30, the edge OR off, the popcount.
Compared with the oracle on a sample, the first pairs and the last tiles;
result bytes with the counts of every pair (tolerance 0)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2103_14978_gb300 import batch, device_data as dd, gk, synth
from tests.gpu_helpers import assert_same, oracle_run, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def workload(lengths, n, seed):
    """n pairs drawn from 60 thousand of mixed lengths: thresholds of 0 to 20% of
    the length and, one in eight, anywhere up to 255."""
    ref = synth.reference(300_000, seed, 0.05, 0.0004)
    w = synth.pairs_workload("routes", seed=seed, ref=ref, n_pairs=60_000, m=lengths, cands=6,
                             e_rates=(0.0, 0.02, 0.05, 0.10, 0.2), read_n_frac=0.0004, shuffle=True)
    rng = np.random.default_rng(seed + n)
    pick = rng.integers(0, w.n_pairs, n)
    w.pair_read, w.pair_off, w.pair_e = w.pair_read[pick].copy(), w.pair_off[pick].copy(), w.pair_e[pick].copy()
    far = rng.integers(0, n, n // 8)
    w.pair_e[far] = rng.integers(20, 256, far.size)
    w.read_len[rng.integers(0, w.n_reads, 3)] = 0
    w.pair_read[rng.integers(0, n, 11)] = w.n_reads + 2
    return w


class Launch:
    def __init__(self, w):
        self.w = w
        self.ref = gk.gk_load_reference(w.ref)
        self.sw = -(-w.stride // 32)
        self.reads = dd.upload_reads(w.reads, w.read_len, w.stride, stride_words=self.sw)
        self.len = dd.as_i16(w.read_len).cuda()
        self.p = dd.upload_pairs(w.pair_read, w.pair_off, w.pair_e)
        self.ws = torch.empty(gk.gk_filter_batched_workspace(w.n_pairs), dtype=torch.uint8, device="cuda")

    def run(self, flags=0, mode=gk.GK_COUNT_RUNS4):
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        acc, ed = gk.gk_filter_batched(self.ref, self.reads.packed, self.sw, self.reads.n_reads, self.len,
                                       self.reads.nflag, self.p.pair_read, self.p.pair_off, self.p.pair_e,
                                       gk.Tiling(1, 256, 4, 8), self.ws, count_mode=mode, flags=flags, err_count=err)
        torch.cuda.synchronize()
        return acc.cpu().numpy(), None if ed is None else dd.edits_u16(ed), int(err.item())


def check(w, full=False):
    n = w.n_pairs
    rng = np.random.default_rng(n)
    idx = np.arange(n) if full else np.unique(
        np.concatenate([rng.integers(0, n, 6000), np.arange(min(n, 300)), np.arange(max(0, n - 1500), n)]))
    L = Launch(w)
    for flags, mode, oflags, omode in ((0, gk.GK_COUNT_RUNS4, 0, O.RUNS4),
                                       (gk.GK_FLAG_NO_EDGE_FIX, gk.GK_COUNT_POPCOUNT, O.FLAG_NO_EDGE_FIX, O.POPCOUNT)):
        acc, ed, err = L.run(flags, mode)
        assert_same((acc[idx], ed[idx]), oracle_run(w, mode=omode, flags=oflags, idx=idx), f"n={n} flags={flags}")
        assert err == int((ed == O.INVALID).sum())
        res, _, _ = L.run(flags | gk.GK_FLAG_RESULT_BYTE, mode)
        want = np.where(ed == O.UNDEFINED, gk.GK_RESULT_UNDEFINED,
                        np.where(ed == O.INVALID, gk.GK_RESULT_INVALID, np.minimum(ed, gk.GK_RESULT_MAX_COUNT)))
        assert (res == want.astype(np.uint8)).all()


@pytest.mark.parametrize("lengths,n", [
    ((1, 128), 150_001), ((1, 128), 300_001), ((1, 128), 700_001), ((1, 128), 1_300_001), ((1, 128), 2_000_000),
    ((90, 256), 70_001), ((90, 256), 100_001), ((90, 256), 300_000), ((50, 300), 160_001),
    ((120, 512), 30_001), ((120, 512), 50_001), ((36, 512), 100_001), ((120, 512), 300_000)])
def test_in_tiles(lengths, n):
    check(workload(lengths, n, 7000 + lengths[1]))


@pytest.mark.parametrize("lengths,n", [
    ((1, 128), 2_000_001), ((90, 256), 300_001), ((50, 300), 300_001), ((50, 300), 1_000_003), ((36, 512), 300_001),
    ((200, 512), 458_752), ((36, 512), 1_100_017)])
def test_through_records_all_lengths_in_one(lengths, n):
    check(workload(lengths, n, 7100 + lengths[1]))


@pytest.mark.parametrize("lengths", [(40, 128), (90, 256), (50, 300), (36, 512)])
def test_through_records_by_range(lengths):
    """Above 8 million pairs, one filter launch per range of lengths."""
    check(workload(lengths, 8_000_003, 7200 + lengths[1]))


def test_full_size_default_tiling():
    """50 million pairs of 50-300 bp through the default tiling, as a graph."""
    w = synth.config4()
    ref = gk.gk_load_reference(w.ref)
    reads = dd.upload_reads(w.reads, w.read_len, w.stride)
    pairs = dd.upload_pairs(w.pair_read, w.pair_off, w.pair_e)
    bf = batch.BatchedFilter(ref, reads.packed, reads.stride_words, reads.n_reads, dd.as_i16(w.read_len).cuda(),
                             reads.nflag, pairs.pair_read, pairs.pair_off, pairs.pair_e)
    bf.capture()
    bf.accept.fill_(7)
    bf.edits.fill_(-1)
    bf.replay()
    torch.cuda.synchronize()
    acc, ed = bf.accept.cpu().numpy(), dd.edits_u16(bf.edits)
    valid = ed < gk.GK_EDITS_INVALID
    assert np.array_equal(acc[valid], (ed[valid] <= w.pair_e[valid]).astype(np.uint8))
    idx = np.sort(np.random.default_rng(7).choice(w.n_pairs, 60_000, replace=False))
    assert_same((acc[idx], ed[idx]), oracle_run(w, idx=idx), "50 million pairs")
