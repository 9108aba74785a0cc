"""The per-pair filter's striped and overlapping forms (stripe.cuh, overlap.cuh)
compiled for the host and compared with the oracle (integer work, tolerance 0):
every combination of words and stripes that the launchers pick, at the read
lengths where they begin and end, all shift counts, both counts."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import oracle as O
from tests.conftest import ROOT

SOURCE = r"""
#include "overlap.cuh"
#include "stripe.cuh"
using namespace gk;

struct Planes { const uint32_t *rh, *rl, *gh, *gl; };

template <int W, int S, bool WHOLE>
static void sweep(uint32_t m, uint32_t K, int mode, const Planes &p, uint16_t *out) {
  uint32_t x[W], rh[S], rl[S], gh[1][S], gl[1][S];
  auto stripes = [&](const uint32_t *from, uint32_t (&to)[S]) {
    for (int w = 0; w < W; ++w) x[w] = from[w];
    stripe_linear<W, S>(x, to);
  };
  stripes(p.rh, rh);
  stripes(p.rl, rl);
  stripes(p.gh, gh[0]);
  stripes(p.gl, gl[0]);
  striped_exact<W, S, 1, WHOLE>(m, 0u, K, mode, rh, rl, gh, gl,
                                [&](uint32_t k, const uint32_t (&c)[1]) { out[k] = (uint16_t)c[0]; });
}

template <int W, int S, bool WHOLE>
static void single(uint32_t m, uint32_t K, int mode, const Planes &p, uint16_t *out) {
  uint32_t h[W], l[W], wh[W], wl[W], rh[S], rl[S], gh[1][S], gl[1][S], lo[1], hi[1], c[1];
  for (int w = 0; w < W; ++w) {
    h[w] = p.rh[w];
    l[w] = p.rl[w];
    wh[w] = p.gh[w];
    wl[w] = p.gl[w];
  }
  stripe_linear<W, S>(h, rh);
  stripe_linear<W, S>(l, rl);
  stripe_linear<W, S>(wh, gh[0]);
  stripe_linear<W, S>(wl, gl[0]);
  for (uint32_t k = 0; k <= K; ++k) {
    end_corrections<W>(m, k, h, l, wh, wl, lo[0], hi[0]);
    striped_deferred<W, S, 1, WHOLE>(m, k, mode, rh, rl, gh, gl, lo, hi, c);
    out[k] = (uint16_t)c[0];
  }
}

template <int W>
static void overlap(uint32_t m, uint32_t K, int mode, const Planes &p, uint16_t *out) {
  uint32_t rh[W], rl[W], gh[1][W], gl[1][W], c[1];
  for (int w = 0; w < W; ++w) {
    rh[w] = p.rh[w];
    rl[w] = p.rl[w];
    gh[0][w] = p.gh[w];
    gl[0][w] = p.gl[w];
  }
  for (uint32_t k = 0; k <= K; ++k) {
    if (k == 0)
      overlap_counts<W, 1, 0>(m, k, mode, rh, rl, gh, gl, c);
    else if (k == 1)
      overlap_counts<W, 1, 1>(m, k, mode, rh, rl, gh, gl, c);
    else if (k == 2)
      overlap_counts<W, 1, 2>(m, k, mode, rh, rl, gh, gl, c);
    else
      overlap_counts<W, 1, -1>(m, k, mode, rh, rl, gh, gl, c);
    out[k] = (uint16_t)c[0];
  }
}

// n pairs' counts at shift counts 0..K; planes: n rows of W words each.  form 0
// sweep, 1 one threshold, in S stripes; 2 overlapping words.
extern "C" int run(int form, int W, int S, uint32_t m, uint32_t K, int mode, uint64_t n, const uint32_t *rh,
                   const uint32_t *rl, const uint32_t *gh, const uint32_t *gl, uint16_t *out) {
  for (uint64_t i = 0; i < n; ++i) {
    const Planes p{rh + i * W, rl + i * W, gh + i * W, gl + i * W};
    uint16_t *o = out + i * (K + 1);
    bool done = false;
#define STRIPES(w, s)                                                                  \
  if (form < 2 && W == w && S == s) {                                                  \
    done = true;                                                                       \
    if (m % s == 0)                                                                    \
      form == 0 ? sweep<w, s, true>(m, K, mode, p, o) : single<w, s, true>(m, K, mode, p, o); \
    else                                                                               \
      form == 0 ? sweep<w, s, false>(m, K, mode, p, o) : single<w, s, false>(m, K, mode, p, o); \
  }
    STRIPES(2, 3) STRIPES(3, 3) STRIPES(3, 4) STRIPES(4, 4) STRIPES(4, 5) STRIPES(5, 5) STRIPES(5, 8) STRIPES(6, 8)
    STRIPES(7, 8) STRIPES(8, 8) STRIPES(9, 11) STRIPES(10, 11)
#define WORDS(w)                   \
  if (form == 2 && W == w) {       \
    done = true;                   \
    overlap<w>(m, K, mode, p, o);  \
  }
    WORDS(2) WORDS(3) WORDS(4) WORDS(5) WORDS(6) WORDS(7) WORDS(8)
    if (!done) return 1;
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    cuda = next((d for d in (os.environ.get("CUDA_HOME"), "/usr/local/cuda") if d and os.path.isdir(d)), None)
    if shutil.which("g++") is None or cuda is None:
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("forms")
    (d / "forms.cpp").write_text(SOURCE)
    so = str(d / "forms.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-w", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2103_14978_gb300", "csrc"), "-I",
                           os.path.join(cuda, "include"), "-o", so, str(d / "forms.cpp")])
    return ctypes.CDLL(so)


def planes(codes, W):
    """n x m base codes (A C G T = 0 1 2 3) -> high and low planes, W words a row."""
    n, m = codes.shape
    out = []
    for bit in (1, 0):
        b = np.zeros((n, 32 * W), np.uint8)
        b[:, :m] = codes >> bit & 1
        out.append(np.ascontiguousarray(np.packbits(b, axis=1, bitorder="little")).view(np.uint32).reshape(n, W))
    return out


def pairs(m, n, seed):
    """Reads and windows: unrelated, the read with a few edits and shifts, and
    windows rich in 'A' (code 00, which vacated positions compare as)."""
    rng = np.random.default_rng(seed)
    read = rng.integers(0, 4, (n, m)).astype(np.uint8)
    win = rng.integers(0, 4, (n, m)).astype(np.uint8)
    for i in range(n):
        kind = i % 4
        if kind == 3:
            continue
        s = int(rng.integers(-12, 13)) if kind else 0
        lo, hi = max(0, s), min(m, m + s)
        win[i, lo:hi] = read[i, lo - s:hi - s]
        for p in rng.integers(0, m, int(rng.integers(0, 6))):
            win[i, p] = rng.integers(0, 4)
        if kind == 2:
            win[i, rng.random(m) < 0.4] = 0
            read[i, :3] = 0
            win[i, -3:] = 0
    return read, win


def combinations():
    for m in (33, 40, 63, 64, 65, 91, 92, 93, 95, 96, 97, 100, 124, 125, 126, 127, 128, 129, 150, 155, 156, 157, 160, 161,
              170, 192, 193, 200, 223, 224, 225, 248, 250, 253, 254, 257, 288, 289, 300, 319, 320):
        W = -(-m // 32)
        stripes = [3, 3, 4, 5, 8, 8, 8, 11, 11][W - 2] if W <= 10 else 0
        limit = lambda S: 32 * S - (4 if S & 1 else 2)  # noqa: E731
        if m > limit(stripes):
            stripes = {3: 4, 4: 5, 5: 8}.get(W, 0)
        if stripes:
            yield m, W, stripes, 0
        if W >= 3 and stripes == (W if W <= 5 else 8 if W <= 8 else 11):
            yield m, W, stripes, 1
        if W <= 8 and m <= 30 * W:
            yield m, W, 0, 2


@pytest.mark.parametrize("m,W,S,form", list(combinations()))
def test_host_build_matches_the_oracle(forms, m, W, S, form):
    n, K = 64, 7 if form == 2 else 30
    K = min(K, m - 1)
    read, win = pairs(m, n, 100 * m + form)
    letters = np.frombuffer(b"ACGT", np.uint8)
    # every window in a genome of its own: the windows side by side
    ref = letters[win].reshape(-1)
    rp, gp = planes(read, W), planes(win, W)
    for mode in (0, 1):
        got = np.zeros((n, K + 1), np.uint16)
        assert forms.run(form, W, S, ctypes.c_uint32(m), ctypes.c_uint32(K), mode, ctypes.c_uint64(n),
                         *(ctypes.c_void_p(p.ctypes.data) for p in rp + gp), ctypes.c_void_p(got.ctypes.data)) == 0
        for k in range(K + 1):
            _, want, _ = O.filter_batch(letters[read].reshape(-1), np.arange(n) * m, np.full(n, m), ref, np.arange(n),
                                        np.arange(n) * m, k, mode)
            bad = np.nonzero(got[:, k] != want)[0]
            assert bad.size == 0, (m, W, S, form, mode, k, bad[:5], got[bad[:5], k], want[bad[:5]])
