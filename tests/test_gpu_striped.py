"""Bit-exact parity of the striped kernels with the CPU oracle at the read
lengths where the number of stripes changes and where the last row is full,
nearly full or just begun (integer work, tolerance 0)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2103_14978_gb300 import device_data as dd, gk
from tests.gpu_helpers import GpuRun, assert_same, oracle_run, require_gpu, small_workload

pytestmark = pytest.mark.gpu

EDGES = [33, 63, 64, 65, 91, 92, 93, 96, 97, 100, 101, 125, 126, 127, 128, 129, 150, 155, 156, 157, 160, 161, 192,
         224, 248, 253, 254, 255, 256, 257, 300, 319, 320, 321]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("m", EDGES)
def test_sweep_at_stripe_edges(m):
    """Neighbouring pairs that share a read (an odd pair count, so that the
    last one is alone) and pairs in random order; both counts; a genome with
    few and with many N (one thread per pair, the queue of defined pairs)."""
    for cands, n_frac, mode in ((4, 0.0, gk.GK_COUNT_RUNS4), (5, 0.0, gk.GK_COUNT_POPCOUNT),
                                (1, 0.0, gk.GK_COUNT_RUNS4), (6, 0.002, gk.GK_COUNT_RUNS4)):
        w = small_workload(m, 1501, seed=3000 + m + cands, n_frac=n_frac, read_n_frac=n_frac, cands=cands)
        if cands == 5:
            perm = np.random.default_rng(m).permutation(w.n_pairs)
            w.pair_read, w.pair_off = w.pair_read[perm].copy(), w.pair_off[perm].copy()
        run = GpuRun(w)
        r = run.reads
        acc, ed = gk.gk_filter_sweep(run.ref, r.packed, r.stride_words, r.n_reads, r.nflag, m, run.pairs.pair_read,
                                     run.pairs.pair_off, 0, 30, count_mode=mode)
        torch.cuda.synchronize()
        for e in range(31):
            assert_same((acc[e].cpu().numpy(), dd.edits_u16(ed[e])),
                        oracle_run(w, e, O.RUNS4 if mode == gk.GK_COUNT_RUNS4 else O.POPCOUNT),
                        f"m={m} cands={cands} e={e}")


@pytest.mark.parametrize("m", [m for m in EDGES if m >= 65])
def test_one_threshold_at_stripe_edges(m):
    """Shift counts around those from which one threshold runs striped, and
    the largest (30); neighbours that share a read and pairs in random order;
    the queue of defined pairs."""
    for cands, n_frac, mode in ((4, 0.0, gk.GK_COUNT_RUNS4), (5, 0.0, gk.GK_COUNT_POPCOUNT),
                                (6, 0.002, gk.GK_COUNT_RUNS4)):
        w = small_workload(m, 1501, seed=3500 + m + cands, n_frac=n_frac, read_n_frac=n_frac, cands=cands)
        if cands == 5:
            perm = np.random.default_rng(m).permutation(w.n_pairs)
            w.pair_read, w.pair_off = w.pair_read[perm].copy(), w.pair_off[perm].copy()
        run = GpuRun(w)
        for e in (7, 8, 9, 12, 14, 16, 17, 25, 30):
            assert_same(run.filter(e=e, mode=mode),
                        oracle_run(w, e, O.RUNS4 if mode == gk.GK_COUNT_RUNS4 else O.POPCOUNT),
                        f"m={m} cands={cands} e={e}")


@pytest.mark.parametrize("m", [1, 2, 31, 33, 96, 100, 126, 127, 150, 156, 157, 254, 255, 300, 349, 512])
def test_per_pair_thresholds_sorted_in_tiles(m):
    """Thresholds on both sides of the largest deferred shift count (30) and
    past m; launches of one pair, a partial warp, whole and partial tiles; N
    in genome and reads; invalid pairs, counted once."""
    w = small_workload(m, 5001, seed=3900 + m, n_frac=0.001, read_n_frac=0.001, cands=3, e_rates=(0.02,))
    rng = np.random.default_rng(m)
    w.pair_e = rng.choice(np.array([0, 1, 2, 5, 9, 15, 29, 30, 31, 32, 60, 255], np.uint8), w.n_pairs)
    w.pair_read[rng.integers(0, w.n_pairs, 9)] = w.n_reads
    run = GpuRun(w)
    want = oracle_run(w)
    r, p = run.reads, run.pairs
    for n in (1, 31, 128, 129, 1000, 5001):
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        acc, ed = gk.gk_filter(run.ref, r.packed, r.stride_words, r.n_reads, r.nflag, m, p.pair_read[:n],
                               p.pair_off[:n], p.pair_e[:n], err_count=err)
        torch.cuda.synchronize()
        assert_same((acc.cpu().numpy(), dd.edits_u16(ed)), (want[0][:n], want[1][:n]), f"m={m} n={n}")
        assert int(err.item()) == int((want[1][:n] == O.INVALID).sum())


@pytest.mark.parametrize("m", [8, 9, 100, 120, 150, 250])
@pytest.mark.parametrize("e_lo,e_hi", [(0, 7), (5, 8), (6, 7), (7, 8), (6, 9)])
def test_sliced_sweep_range_ends(m, e_lo, e_hi):
    """Sliced sweeps that end at 7, 8 and above; thresholds past m - 1."""
    w = small_workload(m, 700, seed=3300 + m)
    run = GpuRun(w)
    r = run.reads
    buf = gk.gk_slice(run.ref, r.packed, r.stride_words, r.n_reads, r.nflag, m, run.pairs.pair_read,
                      run.pairs.pair_off)
    acc, ed = gk.gk_filter_sliced_sweep(buf, w.n_pairs, m, e_lo, e_hi)
    torch.cuda.synchronize()
    for e in range(e_lo, e_hi + 1):
        assert_same((acc[e - e_lo].cpu().numpy(), dd.edits_u16(ed[e - e_lo])), oracle_run(w, e), f"m={m} e={e}")


@pytest.mark.parametrize("m", [33, 59, 60, 61, 65, 89, 90, 91, 97, 101, 119, 120, 121, 129, 149, 150, 151, 161, 180, 181,
                               193, 210, 225, 240, 241])
def test_overlapping_words_at_their_limits(m):
    """Every shift count of the overlapping words and the first beyond, at
    read lengths around those W words hold; neighbours that share a read and
    pairs in random order; packed reads and ASCII rows."""
    for cands, mode in ((4, gk.GK_COUNT_RUNS4), (5, gk.GK_COUNT_POPCOUNT)):
        w = small_workload(m, 1203, seed=3700 + m + cands, cands=cands)
        if cands == 5:
            perm = np.random.default_rng(m).permutation(w.n_pairs)
            w.pair_read, w.pair_off = w.pair_read[perm].copy(), w.pair_off[perm].copy()
        run = GpuRun(w)
        asc = torch.from_numpy(np.ascontiguousarray(w.reads)).cuda()
        for e in (0, 1, 2, 3, 5, 7, 8, 10):
            want = oracle_run(w, e, O.RUNS4 if mode == gk.GK_COUNT_RUNS4 else O.POPCOUNT)
            assert_same(run.filter(e=e, mode=mode), want, f"m={m} cands={cands} e={e}")
            acc, ed = gk.gk_filter_ascii(run.ref, asc, w.stride, w.n_reads, m, run.pairs.pair_read, run.pairs.pair_off,
                                         e, count_mode=mode)
            torch.cuda.synchronize()
            assert_same((acc.cpu().numpy(), dd.edits_u16(ed)), want, f"ascii m={m} cands={cands} e={e}")
