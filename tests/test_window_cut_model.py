"""The window cut as the scan kernels apply it returns exactly the best g, on adversarial scores.

test_selection_model.py models a window that always histograms its scores on 12-bit bins. The scan goes through up to
three rules first: a bound from the query's histogram H (bins of csrc/bound_bins.cuh, compiled for the host here), a
cut guessed from a sample of the window when there is no bound, and all slots when the window's budget holds them; only
then the full cut. This file models these rules, the merge's floor and the zero rule, and checks on the CPU that for any
order in which windows finish and any snapshot of H the result is exactly the top g by (score desc, id asc). Mistakes
planted in the model have to fail."""
import ctypes
import os
import subprocess
import zlib

import numpy as np
import pytest

from test_selection_model import find_bin, keys_of, order_bits, score_pattern, truth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_08395_gb300", "csrc")
SRC = r"""
#include "bound_bins.cuh"
extern "C" {
int bins_n() { return sindi::kHBins; }
int bins_rest() { return sindi::kHRest; }
int bins_top(uint32_t m, int terms) { return sindi::hbin_top(m, terms); }
void bins_of(const uint32_t* ob, int n, int top, int64_t* out) { for (int i = 0; i < n; i++) out[i] = sindi::hbin(ob[i], top); }
uint32_t bins_floor(int b, int top) { return sindi::hbin_floor((uint32_t)b, top); }
}
"""
U64 = np.uint64


@pytest.fixture(scope="module")
def bins(tmp_path_factory):
    d = tmp_path_factory.mktemp("bins")
    (d / "b.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "b.cpp"), "-o",
                           str(d / "b.so")])
    lib = ctypes.CDLL(str(d / "b.so"))
    lib.bins_floor.restype = ctypes.c_uint32
    return lib


class Model:
    """One query: its largest product bound M and number of terms give H's bins. wrong: a planted mistake."""

    def __init__(self, lib, M, terms, wrong=None):
        self.lib, self.wrong = lib, wrong
        self.top = lib.bins_top(ctypes.c_uint32(int(order_bits(np.float32(M)))), terms)
        self.n, self.rest = lib.bins_n(), lib.bins_rest()

    def bin(self, keys):
        ob = np.ascontiguousarray(keys >> U64(32), np.uint32)
        out = np.empty(len(ob), np.int64)
        self.lib.bins_of(ob.ctypes.data_as(ctypes.c_void_p), len(ob), self.top, out.ctypes.data_as(ctypes.c_void_p))
        return out

    def floor(self, b):
        return U64(self.lib.bins_floor(int(b), self.top))

    def threshold(self, b, skip_zero):
        """Least order bits that count when g candidates lie in bin b and above."""
        f = self.floor(b + 1 if self.wrong == "bound a bin too high" and 0 < b < self.n - 1 else b)
        return U64(0x80000001) if skip_zero and f <= U64(0x80000000) else f

    def window(self, K, s, g, bound, skip_zero):
        """What a window with keys K and scores s emits. bound: H's bin of the g-th emitted candidate, or None."""
        n, g_w = len(K), min(g, len(K))
        cap = 2 * min(g, self.lam)
        ob, need, bits = K >> U64(32), 0, U64(0)
        direct = True
        if bound is not None:
            bits = self.floor(bound)
            thr = self.threshold(bound, skip_zero)
        elif n <= cap:
            thr = self.threshold(0, skip_zero)
        else:  # the sampled cut: every 2^sh-th span of 128 slots
            over = 7 * g_w // (5 * 32)
            sh = 3 if over >= 8 else 2 if over >= 4 else 1 if over >= 2 else 0
            want = (7 * g_w // 5) >> sh if sh else g_w
            seen = ((np.arange(n) >> 7) % (1 << sh) == 0) & (s > 0)
            b = self.bin(K[seen])
            b, _, _, total = find_bin(np.bincount(b[b > self.rest], minlength=self.n), want)
            found = total >= want
            thr = self.threshold(b if found else 0, skip_zero)
            need = 0 if skip_zero and thr == U64(0x80000001) else g_w if found else None
            if self.wrong == "any sample will do" and need is not None:
                need = 0
            direct = need is not None
        if direct:
            out = K[ob >= thr]
            if need <= len(out) <= cap:
                return out
        # the full cut: 12-bit bins from the window's best down, 8 more bits, an exact select
        b12 = (K >> U64(52)).astype(np.int64)
        rel = np.minimum(b12.max() - b12, 255)
        cut, above, _, _ = find_bin(np.bincount(255 - rel, minlength=256), g_w)
        relative, bw = 255 - cut < 255, b12.max() - (255 - cut)
        lo = max(bw, int(bits) >> 20)
        t = U64(lo) << U64(52)
        exact = not relative
        if relative and lo == bw:
            sub = ((K[b12 == bw] >> U64(44)) & U64(255)).astype(np.int64)
            b2, a2, o2, _ = find_bin(np.bincount(sub, minlength=256), g_w - above)
            t = U64((int(bw) << 8) | b2) << U64(44)
            exact = above + a2 + o2 > cap
        if exact:
            t = np.sort(K)[-g_w]
        return K[K >= max(t, bits << U64(32))]

    def search(self, s, lam, g, schedule, rng):
        self.lam = lam
        n, sigma = len(s), -(-len(s) // lam)
        keys, nonneg = keys_of(s, np.arange(len(s))), bool(np.all(s >= 0))
        H, emitted = np.zeros(self.n, np.int64), []
        history = [H.copy()]

        def run(w, snapshot):
            bound = None
            if snapshot is not None:
                b, _, _, total = find_bin(snapshot, g)
                bound = b if total >= g else None
            skip = nonneg and (w * lam >= g or (self.wrong == "zeros never count" and w > 0))
            lo, hi = w * lam, min(n, (w + 1) * lam)
            out = self.window(keys[lo:hi], s[lo:hi], g, bound, skip)
            assert len(out) <= max(2 * min(g, lam), min(g, hi - lo))
            emitted.append(out)
            np.add.at(H, self.bin(out), 1)
            history.append(H.copy())

        first = sigma if schedule == "none" else 0 if schedule == "batched" else max(2, -(-sigma // 8))
        first = min(first, sigma)
        for w in rng.permutation(first):
            run(int(w), None)
        done = len(history) - 1
        for w in rng.permutation(np.arange(first, sigma)):
            run(int(w), history[int(rng.integers(done if schedule == "split" else 0, len(history)))])
        C = np.concatenate(emitted)
        g_m = min(g, len(C))
        b, _, _, _ = find_bin(H, g_m)
        return np.sort(C[(C >> U64(32)) >= self.floor(b)])[::-1][:g_m]


def scores(kind, n, rng):
    """Scores, and the largest product bound and number of terms of a query that can have them."""
    if kind == "binary":  # sums of up to 100 equal products
        return rng.binomial(100, 0.3, n).astype(np.float32), 1.0, 100
    if kind == "dense":  # sums of many similar products
        return rng.normal(1000.0, 40.0, n).astype(np.float32), 1.5, 2048
    if kind == "below-zero":
        return (-rng.gamma(4.0, 2.0, n)).astype(np.float32), 3.0, 20
    if kind == "mostly-below-zero":
        return (rng.gamma(4.0, 2.0, n) * np.where(rng.random(n) < 0.01, 1, -1)).astype(np.float32), 3.0, 20
    if kind == "outlier":  # one product bound far above everything that scores
        return rng.lognormal(0, 1, n).astype(np.float32), 1e20, 3
    if kind == "spans":  # the best slots in spans that the sample does not read, or only there
        return ((np.arange(n) >> 7) % 8 == rng.integers(0, 2)).astype(np.float32) + rng.random(n).astype(np.float32), 2.0, 1
    s = score_pattern(kind, n, rng)
    return s, float(np.abs(s).max()), int(rng.choice([1, 8, 50, 700]))


KINDS = ["binary", "dense", "below-zero", "mostly-below-zero", "outlier", "spans", "sparse", "ties", "zeros", "one_bin",
         "one_subbin", "signed"]


def _trials(kind, schedule, count):
    rng = np.random.default_rng(zlib.crc32(f"{kind}/{schedule}".encode()))
    for _ in range(count):
        lam = int(rng.choice([64, 1000, 2048, 4096]))
        n = int(rng.choice([1, lam - 1, lam, 3 * lam + 5, 9 * lam + 1]))
        g = int(rng.choice([1, 10, 50, 300, 700]))
        yield rng, lam, n, g, *scores(kind, n, rng)


@pytest.mark.parametrize("schedule", ["none", "batched", "split"])
@pytest.mark.parametrize("kind", KINDS)
def test_the_best_g_are_found(bins, kind, schedule):
    for rng, lam, n, g, s, M, terms in _trials(kind, schedule, 25):
        got = Model(bins, M, terms).search(s, lam, g, schedule, rng)
        assert np.array_equal(got, truth(s, g)), (kind, schedule, lam, n, g)


@pytest.mark.parametrize("wrong", ["bound a bin too high", "any sample will do", "zeros never count"])
def test_planted_mistakes_fail(bins, wrong):
    for kind in KINDS:
        for schedule in ("none", "batched", "split"):
            for rng, lam, n, g, s, M, terms in _trials(kind, schedule, 25):
                if not np.array_equal(Model(bins, M, terms, wrong).search(s, lam, g, schedule, rng), truth(s, g)):
                    return
    pytest.fail("not one answer was wrong")
