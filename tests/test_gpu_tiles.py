"""Bit-exact parity of the batched filter's sorted tiles (one pair per lane) with
the CPU oracle: launches filtered in their tiles and launches that go through
records, at tile remainders, over row strides that select each compiled range
of read lengths (integer work, tolerance 0)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2103_14978_gb300 import device_data as dd, gk, synth
from tests.gpu_helpers import assert_same, oracle_run, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def workload(lengths, n_pairs, seed, n_frac=0.0005):
    ref = synth.reference(300_000, seed, 0.05, n_frac)
    w = synth.pairs_workload("tiles", seed=seed, ref=ref, n_pairs=n_pairs, m=lengths, cands=7,
                             e_rates=(0.0, 0.02, 0.05, 0.10, 0.2), read_n_frac=n_frac, shuffle=True)
    rng = np.random.default_rng(seed)
    w.pair_e[rng.integers(0, n_pairs, n_pairs // 50)] = rng.integers(28, 256, n_pairs // 50)
    w.read_len[rng.integers(0, w.n_reads, 5)] = 0
    w.pair_read[rng.integers(0, n_pairs, 11)] = w.n_reads + 2
    return w


def run(w, flags=0, mode=gk.GK_COUNT_RUNS4):
    ref = gk.gk_load_reference(w.ref)
    sw = -(-w.stride // 32)
    reads = dd.upload_reads(w.reads, w.read_len, w.stride, stride_words=sw)
    p = dd.upload_pairs(w.pair_read, w.pair_off, w.pair_e)
    ws = torch.empty(gk.gk_filter_batched_workspace(w.n_pairs), dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    acc, ed = gk.gk_filter_batched(ref, reads.packed, sw, reads.n_reads, dd.as_i16(w.read_len).cuda(), reads.nflag,
                                   p.pair_read, p.pair_off, p.pair_e, gk.Tiling(1, 256, 2, 8), ws, count_mode=mode,
                                   flags=flags, err_count=err)
    torch.cuda.synchronize()
    return acc.cpu().numpy(), None if ed is None else dd.edits_u16(ed), int(err.item())


@pytest.mark.parametrize("lengths", [(1, 128), (90, 256), (33, 320), (120, 512)])
@pytest.mark.parametrize("n_pairs", [1, 255, 257, 30_011])
def test_filtered_in_tiles(lengths, n_pairs):
    w = workload(lengths, n_pairs, 4000 + lengths[1] + n_pairs % 100)
    acc, ed, err = run(w)
    want = oracle_run(w)
    assert_same((acc, ed), want, f"{lengths} n={n_pairs}")
    assert err == int((want[1] == O.INVALID).sum())
    acc, ed, _ = run(w, flags=gk.GK_FLAG_NO_EDGE_FIX, mode=gk.GK_COUNT_POPCOUNT)
    assert_same((acc, ed), oracle_run(w, mode=O.POPCOUNT, flags=O.FLAG_NO_EDGE_FIX), f"{lengths} n={n_pairs} no edge")


@pytest.mark.parametrize("lengths", [(1, 128), (90, 256), (50, 300), (120, 512)])
def test_through_records(lengths):
    """Above 2 million pairs, the last tile partly filled: every 53rd pair
    against the oracle, result bytes against the counts on every pair."""
    w = workload(lengths, 2_000_357, 4100 + lengths[1])
    acc, ed, err = run(w)
    idx = np.arange(0, w.n_pairs, 53)
    assert_same((acc[idx], ed[idx]), oracle_run(w, idx=idx), f"{lengths}")
    assert err == int((ed == O.INVALID).sum())
    res, _, _ = run(w, flags=gk.GK_FLAG_RESULT_BYTE)
    want = np.where(ed == O.UNDEFINED, gk.GK_RESULT_UNDEFINED,
                    np.where(ed == O.INVALID, gk.GK_RESULT_INVALID, np.minimum(ed, gk.GK_RESULT_MAX_COUNT)))
    assert (res == want.astype(np.uint8)).all()


@pytest.mark.parametrize("lengths", [(150, 150), (250, 250)])
@pytest.mark.parametrize("n_pairs", [600_001, 2_000_357, 8_004_099])
def test_records_of_one_length(lengths, n_pairs):
    """One group holds nearly every pair, so its items are cut into slices; one
    filter launch up to 8 million pairs, one per range of lengths above."""
    w = workload(lengths, n_pairs, 4200 + lengths[1])
    acc, ed, err = run(w)
    idx = np.concatenate([np.arange(0, w.n_pairs, 211), np.arange(w.n_pairs - 500, w.n_pairs)])
    assert_same((acc[idx], ed[idx]), oracle_run(w, idx=idx), f"{lengths} n={n_pairs}")
    assert err == int((ed == O.INVALID).sum())
