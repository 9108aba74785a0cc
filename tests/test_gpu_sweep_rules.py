"""Threshold sweeps around the rules that choose between the striped and the
linear form (few thresholds at the end of many steps, the queue of defined
pairs) and sweeps of one threshold, against the oracle (tolerance 0)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2103_14978_gb300 import device_data as dd, gk
from tests.gpu_helpers import GpuRun, accept_of_result_bytes, assert_same, oracle_run, require_gpu, small_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("m", [40, 64, 92, 96, 100, 128, 150, 160, 180, 200, 250, 288, 300, 320])
def test_ranges_on_both_sides_of_the_rules(m):
    for cands, n_frac in ((4, 0.0), (1, 0.0), (6, 0.002)):
        w = small_workload(m, 1203, seed=5000 + m + cands, n_frac=n_frac, read_n_frac=n_frac, cands=cands)
        run = GpuRun(w)
        r = run.reads
        want = {e: oracle_run(w, e) for e in range(31)}
        for lo, hi in ((2, 3), (5, 10), (8, 12), (8, 15), (12, 15), (20, 25), (20, 30), (0, 10), (0, 13), (0, 30)):
            acc, ed = gk.gk_filter_sweep(run.ref, r.packed, r.stride_words, r.n_reads, r.nflag, m,
                                         run.pairs.pair_read, run.pairs.pair_off, lo, hi)
            torch.cuda.synchronize()
            for e in range(lo, hi + 1):
                assert_same((acc[e - lo].cpu().numpy(), dd.edits_u16(ed[e - lo])), want[e], f"m={m} {lo}..{hi} e={e}")


@pytest.mark.parametrize("m", [0, 1, 20, 33, 100, 128, 160, 300, 400])
def test_one_threshold(m):
    """One row: the same as gk_filter's results, also as result bytes and with
    pairs counted as invalid; thresholds past m - 1 as well."""
    if m == 0:  # empty reads: accepted with no edits
        w = small_workload(1, 100, seed=1)
        ref = gk.gk_load_reference(w.ref)
        p = dd.upload_pairs(w.pair_read, w.pair_off, None)
        acc, ed = gk.gk_filter_sweep(ref, torch.zeros(2, dtype=torch.int32, device="cuda"), 1, w.n_reads, None, 0,
                                     p.pair_read, p.pair_off, 3, 3)
        torch.cuda.synchronize()
        assert acc.cpu().numpy().all() and not dd.edits_u16(ed).any()
        return
    w = small_workload(m, 1001, seed=5200 + m, n_frac=0.002, read_n_frac=0.002)
    w.pair_read[np.random.default_rng(m).integers(0, w.n_pairs, 7)] = w.n_reads + 1
    run = GpuRun(w)
    r = run.reads
    for e in (0, 5, 15, 25, 30) if m > 31 else (0, 5, 200):
        want = oracle_run(w, e)
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        args = (run.ref, r.packed, r.stride_words, r.n_reads, r.nflag, m, run.pairs.pair_read, run.pairs.pair_off, e, e)
        acc, ed = gk.gk_filter_sweep(*args, err_count=err)
        res, _ = gk.gk_filter_sweep(*args, flags=gk.GK_FLAG_RESULT_BYTE)
        torch.cuda.synchronize()
        assert_same((acc[0].cpu().numpy(), dd.edits_u16(ed[0])), want, f"m={m} e={e}")
        assert int(err.item()) == int((want[1] == O.INVALID).sum())
        ok = want[1] != O.INVALID
        assert (accept_of_result_bytes(res[0], e)[ok] == want[0][ok]).all()
