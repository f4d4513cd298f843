"""Host model of the pipelined column pass for pencils of 2^11 points
(fft_col_pipe.cuh, col_pipe2_kernel), without a GPU: the stages on one pencil
against numpy (one cycle of 2048 rows, two cycles of 64 x 32), the two-round
exchange, the sheared walk and its two output rounds, for every thread."""
import random

import numpy as np
import pytest

L, T, P, R = 2048, 4, 64, 32


@pytest.mark.parametrize("two", [True, False], ids=["64x32", "2048"])
def test_stages_equal_the_dft(two):
    rng = np.random.default_rng(7)
    x = rng.standard_normal(L) + 1j * rng.standard_normal(L)
    pos = np.empty(L, complex)
    for p in range(P):  # the radix-2 stage folded into the reads, then stage 0 (Ns = 2)
        j = (p >> 1) + 32 * np.arange(R)
        v = x[j] - x[j + 1024] if p & 1 else x[j] + x[j + 1024]
        y = np.fft.fft(v * np.exp(-2j * np.pi * (p & 1) / 64) ** np.arange(R))
        pos[((p >> 1) << 6) | (np.arange(R) << 1) | (p & 1)] = y
    ref = np.fft.fft2(x.reshape(64, 32)).reshape(-1) if two else np.fft.fft(x)
    for p in range(P):  # stage 1 (Ns = 64); with two cycles its table holds floor(k / 64) = 0
        w = 1.0 if two else np.exp(-2j * np.pi * p / L)
        out = np.fft.fft(pos[(np.arange(R) << 6) | p] * w ** np.arange(R))
        rows = 32 * p + np.arange(R) if two else p + P * np.arange(R)
        assert np.allclose(out, ref[rows])


def test_exchange_rounds():
    seen = set()
    for h in (0, 1):
        X = {}
        for p in range(P):
            for i in range(16):
                r = 16 * (h ^ ((p >> 5) & 1)) + i
                slot = (((p >> 1) & 15) << 6) | (r << 1) | (p & 1)
                assert slot < 1024 and slot not in X
                X[slot] = ((p >> 1) << 6) | (r << 1) | (p & 1)
        for p in range(P):
            for i in range(16):
                r = 16 * (h ^ ((p >> 5) & 1)) + i
                assert X[((r & 15) << 6) | p] == (r << 6) | p
                seen.add((r, p))
    assert len(seen) == L


@pytest.mark.parametrize("two", [True, False], ids=["64x32", "2048"])
@pytest.mark.parametrize("seed", range(4))
def test_walk_and_output_rounds(two, seed):
    rng = random.Random(seed)
    al0, al1 = rng.randrange(64 if two else L), rng.randrange(32)
    for c in range(T):
        off0, off1 = (c * al0) % (64 if two else L), (c * al1) % 32

        def walk(p, j):
            if two:
                return ((((p >> 5) + off0 + 2 * j) & 63) << 5) | ((p + off1) & 31)
            return (p + off0 + 64 * j) & (L - 1)

        assert sorted(walk(p, j) for p in range(P) for j in range(32)) == list(range(L))
        for h in (0, 1):
            X = {}
            for p in range(P):
                u = (p - off0) & 63
                for r in range(R):
                    if two:
                        if u >> 5 != h:
                            continue
                        slot, row = ((u & 31) << 5) + ((r - off1) & 31), 32 * p + r
                    else:
                        t = (r - (((u + off0) & (L - 1)) >> 6) - 16 * h) & 31
                        if t >= 16:
                            continue
                        slot, row = 64 * t + p, p + 64 * r
                    assert slot < 1024 and slot not in X
                    X[slot] = row
            assert len(X) == 1024
            for p in range(P):
                for t in range(16):
                    assert X[64 * t + (p if two else (p + off0) & 63)] == walk(p, 16 * h + t)
