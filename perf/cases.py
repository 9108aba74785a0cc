"""The work whose time this repository answers for: filtering passes through
the public entry points, over the sizes its configurations, benchmark and tests
use (10 thousand to 50 million pairs, reads of 36 to 512 bases, thresholds up
to 10% of the read length).

A case is a dict of plain values:
  kind      the entry points of one pass: "filter" (gk_filter), "sweep"
            (gk_filter_sweep), "sliced" (gk_slice, gk_filter_sliced_sweep),
            "ascii" (gk_filter_ascii), "batched" (gk_filter_batched as a
            captured graph), "round" (one round of the server on the device:
            gk_expand_pairs and gk_filter_batched per read-row stride) and
            "pipe" (gk_pipe_*, host buffers to host buffers)
  m, m_hi   read length, or a range of lengths (m_hi > m)
  pairs     pairs of one pass
  c, c_hi   candidates per read, c_hi > c: uniform in that range
  e_lo, e   thresholds e_lo..e, or the one threshold e; e_rate > 0: per-pair
            thresholds ceil(rate * m), rates 0.02, 0.05, 0.10
  encode    the pass starts from ASCII reads on the device (gk_encode)
  n_frac    share of 'N' in the genome and in the reads
  shuffle   pairs in random order, so that neighbours name different reads
  genome    bases of the genome
  popcount, no_edge, result_byte   the entry points' options

Outputs are whole numbers (accept bits and counts, or result bytes).
"""
import math

import numpy as np
import torch

from paper_2103_14978_gb300 import batch, gk

RATES = (0.02, 0.05, 0.10)
DEFAULTS = {"m_hi": 0, "c": 4, "c_hi": 0, "e_lo": 0, "e_rate": False, "encode": False, "n_frac": 0.0,
            "shuffle": False, "genome": 100_000_000, "popcount": False, "no_edge": False, "result_byte": False}


def listed():
    return [
        # A single small batch, as a mapper hands over the candidates of a few
        # thousand reads: latency, launches and the host path count.
        {"name": "small_100bp_e2", "kind": "filter", "m": 100, "pairs": 10_000, "c": 1, "e": 2, "genome": 1_040_000},
        # The paper's headline filtration: one threshold, 100 bp, encoded
        # reads resident.
        {"name": "filter_100bp_e2", "kind": "filter", "m": 100, "pairs": 20_000_000, "e": 2},
        # The same at its other threshold in the device-encoded mode.
        {"name": "encode_filter_100bp_e5", "kind": "filter", "m": 100, "pairs": 20_000_000, "e": 5, "encode": True},
        # A threshold study: every threshold 0..10 of a batch (the benchmark's step).
        {"name": "sweep_100bp_e0_10", "kind": "sweep", "m": 100, "pairs": 20_000_000, "e": 10, "encode": True},
        # The same for 150 bp reads with many candidates each and N in genome and reads.
        {"name": "sweep_150bp_e0_15_n", "kind": "sweep", "m": 150, "pairs": 10_000_000, "c": 8, "c_hi": 64, "e": 15,
         "n_frac": 0.001},
        # Long reads at the largest threshold (10% of the length), N in genome and reads.
        {"name": "filter_250bp_e25_n", "kind": "filter", "m": 250, "pairs": 10_000_000, "c": 8, "c_hi": 64, "e": 25,
         "n_frac": 0.001},
        # A threshold per pair, as mappers ask that scale it by pair.
        {"name": "per_pair_e_150bp", "kind": "filter", "m": 150, "pairs": 10_000_000, "e": 0, "e_rate": True},
        # Mixed read lengths and per-pair thresholds in random order, one graph.
        {"name": "batched_50_300bp", "kind": "batched", "m": 50, "m_hi": 300, "pairs": 50_000_000, "e": 0,
         "e_rate": True, "shuffle": True},
        # One round of the continuous-batching server: requests of 100, 150 and 250 bp.
        {"name": "server_round", "kind": "round", "m": 100, "m_hi": 250, "pairs": 3_000_000, "e": 0, "e_rate": True,
         "result_byte": True},
        # The bit-sliced form, sliced once and filtered at thresholds 0..7, a ragged batch.
        {"name": "sliced_150bp_e0_7", "kind": "sliced", "m": 150, "pairs": 5_000_011, "e": 7},
        # Reads of an odd length straight from their ASCII rows, odd row stride.
        {"name": "ascii_101bp_e3", "kind": "ascii", "m": 101, "pairs": 3_000_001, "e": 3},
        # Host buffers to host buffers: four batches through the streamed pipeline.
        {"name": "pipe_100bp_e0_5", "kind": "pipe", "m": 100, "pairs": 4_000_000, "e": 5, "result_byte": True},
    ]


def draw(rng):
    kind = rng.choice(["filter", "filter", "filter", "sweep", "sweep", "sliced", "ascii", "batched", "round", "pipe"])
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    m = log(36, 250 if kind == "sliced" else 400)
    e = max(0, math.ceil(rng.choice((0.0,) + RATES) * m))
    if kind in ("sweep", "pipe"):
        e = min(e, gk.GK_SWEEP_MAX_SHIFT)
    if kind == "sliced":
        e = min(e, gk.GK_SLICED_MAX_SHIFT)
    case = {"kind": kind, "m": m, "e": e, "pairs": log(10_000, 5_000_000 if kind in ("pipe", "round") else 20_000_000)}
    case["pairs"] = min(case["pairs"], int(2e9 / ((m + 31) // 32 * (e + 3))))
    if kind == "filter":
        case["encode"] = rng.random() < 0.3
        case["popcount"] = rng.random() < 0.15
        case["no_edge"] = rng.random() < 0.15
        case["e_rate"] = rng.random() < 0.25
        case["result_byte"] = not case["e_rate"] and rng.random() < 0.25
    if kind == "sweep":
        case["e_lo"] = rng.choice((0, 0, e // 2))
        case["encode"] = rng.random() < 0.5
        case["result_byte"] = rng.random() < 0.25
    if kind in ("batched", "round"):
        case.update(m=rng.randint(36, 100), m_hi=rng.randint(150, 320), e_rate=True, shuffle=kind == "batched",
                    result_byte=kind == "round")
    elif kind != "pipe":
        case["shuffle"] = rng.random() < 0.2
        if rng.random() < 0.4:
            case.update(c=8, c_hi=64)
        if rng.random() < 0.3:
            case["n_frac"] = 0.001
    else:
        case["result_byte"] = rng.random() < 0.5
    return case


# ---- inputs ----------------------------------------------------------------

LETTERS = torch.tensor(list(b"ACGT"), dtype=torch.uint8)


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device="cuda")


def _genome(g, n):
    """Uniform bases (0..3), 5% of them copies of other places at 2% substitutions."""
    codes = torch.randint(0, 4, (n,), generator=g, device="cuda", dtype=torch.uint8)
    length = max(1, min(5_000, n // 40))
    k = max(1, n // 20 // length)
    src = (_rand(g, k) * (n - length)).long()
    # copies land on a grid, so that no two of them overlap
    dst = torch.randperm(n // length, generator=g, device="cuda")[:k] * length
    cols = torch.arange(length, device="cuda")
    copy = codes[src[:, None] + cols]
    other = (_rand(g, k, length) < 0.02).to(torch.uint8)
    codes[dst[:, None] + cols] = (copy + other) & 3
    return codes


def _reads(g, codes, lens, stride, rate):
    """ASCII rows of reads sampled from the genome with up to rate x length
    edits each (substitutions, insertions, deletions), and their origins."""
    n, letters = lens.numel(), LETTERS.cuda()
    margin = math.ceil(rate * stride) + 2
    origin = margin + (_rand(g, n).double() * (codes.numel() - stride - 2 * margin)).long()
    out = torch.empty((n, stride), dtype=torch.uint8, device="cuda")
    cols = torch.arange(stride, device="cuda")
    for a in range(0, n, 1_000_000):
        b = min(n, a + 1_000_000)
        k = (_rand(g, b - a) * (torch.floor(rate * lens[a:b]) + 1)).long()
        kmax = max(1, int(rate * stride))
        kind = torch.randint(0, 3, (b - a, kmax), generator=g, device="cuda")
        kind = torch.where(torch.arange(kmax, device="cuda") < k[:, None], kind, 3)
        pos = (_rand(g, b - a, kmax) * lens[a:b, None]).long()
        shift = torch.zeros((b - a, stride + 1), dtype=torch.int32, device="cuda")
        shift.scatter_add_(1, pos, (kind == 2).int())
        shift.scatter_add_(1, pos + 1, -(kind == 1).int())
        changed = torch.zeros((b - a, stride + 1), dtype=torch.bool, device="cuda")
        changed.scatter_(1, torch.where(kind < 2, pos, stride), True)
        idx = origin[a:b, None] + cols + torch.cumsum(shift[:, :stride], 1, dtype=torch.int32)
        c = codes[idx]
        out[a:b] = letters[torch.where(changed[:, :stride], (c + 1 + (idx % 3).to(torch.uint8)) & 3, c).int()]
    return out, origin


def _some_n(g, ascii_, frac):
    """'N' at a share of the positions."""
    if frac > 0:
        flat = ascii_.view(-1)
        flat[(_rand(g, int(flat.numel() * frac)).double() * flat.numel()).long()] = ord("N")


def _counts(g, pairs, c, c_hi):
    """Candidates of each read, `pairs` in all."""
    if c_hi <= c:
        n = -(-pairs // c)
        counts = torch.full((n,), c, dtype=torch.int64, device="cuda")
    else:
        est = int(pairs / ((c + c_hi) / 2) * 1.2) + 64
        counts = torch.randint(c, c_hi + 1, (est,), generator=g, device="cuda")
        n = int(torch.searchsorted(torch.cumsum(counts, 0), pairs).item()) + 1
        counts = counts[:n].clone()
    counts[-1] += pairs - counts.sum()
    return counts


class Inputs:
    """Genome, reads and pairs of one case, on the device."""

    def __init__(self, case, seed):
        g = self.g = torch.Generator(device="cuda").manual_seed(int(seed))
        codes = _genome(g, case["genome"])
        ref = LETTERS.cuda()[codes.int()]
        _some_n(g, ref, case["n_frac"])
        self.ref = gk.gk_load_reference(ref)
        counts = _counts(g, case["pairs"], case["c"], case["c_hi"])
        n = self.n_reads = counts.numel()
        self.stride = max(case["m"], case["m_hi"])
        lens = torch.full((n,), case["m"], dtype=torch.int64, device="cuda")
        if case["kind"] == "round":  # the server's lengths, each request of one
            lens = None
        elif case["m_hi"] > case["m"]:
            lens = torch.randint(case["m"], case["m_hi"] + 1, (n,), generator=g, device="cuda")
        if lens is not None:
            self._pairs(case, codes, lens, counts)
        self.codes = codes if lens is None else None

    def _pairs(self, case, codes, lens, counts):
        g, n = self.g, counts.numel()
        self.ascii, origin = _reads(g, codes, lens, self.stride, 0.02)
        _some_n(g, self.ascii, case["n_frac"])
        ids = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
        m = lens[ids]
        off = (_rand(g, ids.numel()).double() * (codes.numel() - m + 1)).long()
        self.starts = torch.cumsum(counts, 0) - counts
        off[self.starts] = origin
        e = None
        if case["e_rate"]:
            rates = torch.tensor(RATES, device="cuda", dtype=torch.float64)
            r = rates[torch.randint(0, 3, (ids.numel(),), generator=g, device="cuda")]
            e = torch.ceil(r * m - 1e-9).clamp(max=255).to(torch.uint8)
        if case["shuffle"]:
            p = torch.randperm(ids.numel(), generator=g, device="cuda")
            ids, off, e = ids[p], off[p], None if e is None else e[p]
        self.lens, self.ids, self.off, self.pair_e = lens.to(torch.int16), ids.int(), off.int(), e

    def packed(self, fixed, sw):
        return gk.gk_encode(self.ascii, self.n_reads, self.stride, lens=None if fixed else self.lens,
                            fixed_len=self.stride if fixed else 0, stride_words=sw)


# ---- states ----------------------------------------------------------------


class Plain:
    """Reads (ASCII or packed) and pairs of one length, resident."""

    def __init__(self, case, seed):
        x = Inputs(case, seed)
        self.kind, self.m, self.n = case["kind"], case["m"], x.n_reads
        self.ref, self.ids, self.off = x.ref, x.ids, x.off
        self.sw = gk.words_for(self.m)
        self.e_lo, self.e = case["e_lo"], case["e"] if x.pair_e is None else x.pair_e
        self.mode = gk.GK_COUNT_POPCOUNT if case["popcount"] else gk.GK_COUNT_RUNS4
        self.flags = ((gk.GK_FLAG_NO_EDGE_FIX if case["no_edge"] else 0) |
                      (gk.GK_FLAG_RESULT_BYTE if case["result_byte"] else 0))
        self.ascii = x.ascii if case["encode"] or self.kind == "ascii" else None
        if self.kind != "ascii":
            self.packed, self.nflag = x.packed(True, self.sw)
        if self.kind == "sliced":
            self.sliced = torch.empty(gk.gk_sliced_bytes(self.ids.numel(), self.m), dtype=torch.uint8, device="cuda")

    def run(self):
        if self.kind == "ascii":
            return gk.gk_filter_ascii(self.ref, self.ascii, self.m, self.n, self.m, self.ids, self.off, self.e,
                                      count_mode=self.mode, flags=self.flags)
        if self.ascii is not None:
            gk.gk_encode(self.ascii, self.n, self.m, fixed_len=self.m, stride_words=self.sw, packed=self.packed,
                         nflag=self.nflag)
        reads = (self.ref, self.packed, self.sw, self.n, self.nflag, self.m, self.ids, self.off)
        if self.kind == "filter":
            return gk.gk_filter(*reads, self.e, count_mode=self.mode, flags=self.flags)
        if self.kind == "sweep":
            return gk.gk_filter_sweep(*reads, self.e_lo, self.e, count_mode=self.mode, flags=self.flags)
        gk.gk_slice(*reads, out=self.sliced)
        return gk.gk_filter_sliced_sweep(self.sliced, self.ids.numel(), self.m, self.e_lo, self.e,
                                         count_mode=self.mode, flags=self.flags)


class Batched:
    """Mixed lengths and per-pair thresholds, the call captured in a graph."""

    def __init__(self, case, seed):
        x = Inputs(case, seed)
        sw = gk.words_for(x.stride)
        packed, nflag = x.packed(False, sw)
        self.filter = batch.BatchedFilter(x.ref, packed, sw, x.n_reads, x.lens, nflag, x.ids, x.off, x.pair_e)
        self.filter.capture()

    def run(self):
        return self.filter.replay()


class Round:
    """A round of the server: per read-row stride the requests' packed reads,
    one start per read, offsets and one threshold per request."""

    def __init__(self, case, seed):
        x = Inputs(case, seed)
        self.ref, self.lanes = x.ref, []
        lengths = sorted({case["m"], (case["m"] + case["m_hi"]) // 2 // 10 * 10, case["m_hi"]})
        rng = np.random.default_rng(case["pairs"])  # the requests' sizes are the case's, the seed's their contents
        sizes, left = [], case["pairs"]
        while left > 0:  # log-uniform, as requests come
            sizes.append(min(left, int(np.exp(rng.uniform(np.log(1_000), np.log(1_000_000))))))
            left -= sizes[-1]
        which = rng.integers(0, len(lengths), len(sizes))
        dev = lambda a, t: torch.tensor(a, dtype=t, device="cuda")  # noqa: E731
        for k, m in enumerate(lengths):
            mine = [s for s, w in zip(sizes, which) if w == k]
            if not mine:
                continue
            part = dict(case, pairs=sum(mine), m=m, m_hi=0, e_rate=False, shuffle=False, kind="lane")
            reads = [-(-s // case["c"]) for s in mine]
            counts = torch.full((sum(reads),), case["c"], dtype=torch.int64, device="cuda")
            last = np.cumsum(reads) - 1
            counts[dev(last, torch.int64)] = dev([s - (r - 1) * case["c"] for s, r in zip(mine, reads)], torch.int64)
            x.n_reads, x.stride = sum(reads), m
            x._pairs(part, x.codes, torch.full((x.n_reads,), m, dtype=torch.int64, device="cuda"), counts)
            sw = gk.words_for(m)
            packed, _ = x.packed(True, sw)
            pair_end, read_end = np.cumsum(mine), np.cumsum(reads)
            first = np.repeat(pair_end - np.array(mine), reads)
            n = sum(mine)
            e = np.ceil(np.array(RATES)[rng.integers(0, 3, len(mine))] * m - 1e-9).astype(np.uint8)
            self.lanes.append(dict(
                n_reads=x.n_reads, sw=sw, packed=packed, off=x.off, starts=x.starts.int() - dev(first, torch.int32),
                ids=torch.empty(n, dtype=torch.int32, device="cuda"), e=torch.empty(n, dtype=torch.uint8, device="cuda"),
                out=torch.empty(n, dtype=torch.uint8, device="cuda"),
                lens=torch.empty(x.n_reads, dtype=torch.int16, device="cuda"),
                nflag=torch.empty(x.n_reads, dtype=torch.uint8, device="cuda"),
                read_end=dev(read_end, torch.int64), pair_end=dev(pair_end, torch.int64),
                slot=dev(read_end - np.array(reads), torch.int64),
                base=torch.zeros(len(mine), dtype=torch.int32, device="cuda"), seg_e=dev(e, torch.uint8),
                info=torch.full((len(mine),), m | gk.GK_SEG_NO_N, dtype=torch.int32, device="cuda"),
                ws=torch.empty(max(256, gk.gk_filter_batched_workspace(n)), dtype=torch.uint8, device="cuda")))
        self.tiling = gk.Tiling(1, 256, 3, 8)  # the server's

    def run(self):
        for v in self.lanes:
            gk.gk_expand_pairs(v["ids"], v["e"], v["starts"], v["read_end"], v["pair_end"], v["slot"], v["base"],
                               v["seg_e"], n_reads=v["n_reads"], seg_read_info=v["info"], read_len=v["lens"],
                               read_nflag=v["nflag"])
            gk.gk_filter_batched(self.ref, v["packed"], v["sw"], v["n_reads"], v["lens"], v["nflag"], v["ids"],
                                 v["off"], v["e"], self.tiling, v["ws"], flags=gk.GK_FLAG_RESULT_BYTE, accept=v["out"])
        return [v["out"] for v in self.lanes]


class Streamed:
    """Pinned host buffers of four batches and the pipe that filters them."""

    BATCHES = 4

    def __init__(self, case, seed):
        x = Inputs(case, seed)
        step = -(-x.n_reads // self.BATCHES)
        th = list(range(case["e_lo"], case["e"] + 1))
        first = x.starts.tolist()[::step] + [case["pairs"]]
        self.ref, self.batches = x.ref, []
        for b in range(len(first) - 1):
            r0, r1 = b * step, min(x.n_reads, (b + 1) * step)
            n = first[b + 1] - first[b]
            pin = lambda t: t.cpu().contiguous().pin_memory()  # noqa: E731
            acc = torch.zeros(len(th) * n, dtype=torch.uint8).pin_memory()
            ed = None if case["result_byte"] else torch.zeros(len(th) * n, dtype=torch.int16).pin_memory()
            self.batches.append((pin(x.ascii[r0:r1]).view(-1), r1 - r0, pin(x.starts[r0:r1].int() - first[b]),
                                 pin(x.off[first[b]:first[b + 1]]), acc, ed))
        self.pipe = gk.Pipe(x.ref, step, x.stride, case["m"], max(b[3].numel() for b in self.batches), th,
                            flags=gk.GK_PIPE_READ_STARTS | (gk.GK_FLAG_RESULT_BYTE if case["result_byte"] else 0))

    def run(self):
        for b in self.batches:
            last = self.pipe.submit(*b)
        self.pipe.wait(last)
        return [b[4:] for b in self.batches]

    def __del__(self):
        if hasattr(self, "pipe"):
            self.pipe.close()


def prepare(case, seed):
    case = {**DEFAULTS, **case}
    return {"batched": Batched, "round": Round, "pipe": Streamed}.get(case["kind"], Plain)(case, seed)


def run(state):
    return state.run()


def work(case):
    """Bytes of the inputs and outputs, each once, at the widths the entry
    points take them; the path has no floating-point operations."""
    case = {**DEFAULTS, **case}
    n, m = case["pairs"], (case["m"] + max(case["m"], case["m_hi"])) / 2
    reads = n / ((case["c"] + max(case["c"], case["c_hi"])) / 2)
    one_e = case["kind"] not in ("sweep", "sliced", "pipe")
    rows = 1 if one_e else case["e"] - case["e_lo"] + 1
    link = 4 * reads if case["kind"] in ("round", "pipe") else 4 * n
    per_read = m if case["encode"] or case["kind"] in ("ascii", "pipe") else m / 4
    genome = min(case["genome"] / 4, n * m / 4)
    return {"bytes": genome + reads * per_read + link + 4 * n + (n if case["e_rate"] and case["kind"] != "round" else 0) +
            rows * n * (1 if case["result_byte"] else 3), "flops": 0.0}
