"""The mixed-radix passes (fft_mixed.cuh): a host model of their index
arithmetic, and GPU parity against the FP64 oracle at the sizes where a tile
can go wrong -- every register radix, the smallest and largest direct primes,
one and several pencils per tile, a last tile that is not full, whole signals
up to the size where they stop fitting, split last cycles with few rows
lambda_a, pencils over one, two and three axes, d = 1 .. 4.  Tolerances are
those of the parity bar (1e-5 complex64, 1e-12 complex128)."""
import random

import numpy as np
import pytest
import torch

import oracle
from oracle import lattice as L
import paper_1107_5415_gb300 as pf
import seeded_inputs as SI
from parity_util import TOL, rel_l2

ORDER = [15, 13, 11, 9, 16, 14, 12, 10, 8, 7, 6, 5, 4, 3, 2]  # kMixOrder


def _radices(n, rng):
    out = []
    for R in range(16, 1, -1):
        while n % R == 0 and rng.random() < 0.7:
            out.append(R)
            n //= R
    for R in (2, 3, 5, 7, 11, 13, 17, 19, 23):
        while n % R == 0:
            out.append(R)
            n //= R
    return out if n == 1 else None


def test_padded_stages_are_one_to_one_and_affine():
    """mix_configure's padded steps: element r of a butterfly lies at its first
    element plus r steps, and the reads and writes of a stage each cover the
    tile's positions exactly once."""
    rng = random.Random(1)
    done = 0
    while done < 120:
        naxes = rng.randint(1, 3)
        axes = [rng.randint(2, 40 if naxes > 1 else 1200) for _ in range(naxes)]
        rads = [_radices(a, rng) for a in axes]
        T = rng.choice([1, 1, 2, 4, 8, 16, 32])
        n = T * int(np.prod(axes))
        if n > 8192 or any(r is None for r in rads):
            continue
        done += 1
        stages = [(R, i) for i, r in enumerate(rads) for R in r]
        stages.sort(key=lambda x: ORDER.index(x[0]) if x[0] < 17 else -1)
        sigma = [int(np.prod(axes[:i])) for i in range(naxes)]
        Ns, unit = [1] * naxes, 0
        for R, i in stages:
            sig, aR = sigma[i] * T, axes[i] // R
            first = sigma[i] == 1 and Ns[i] == 1 and R % 2 == 0 and T < 16
            istep, ostep = aR * sig, Ns[i] * sig
            ipad = T if unit else 0
            if unit:
                istep += istep // unit * T
            uin = unit
            if first:
                unit = R * T
            opad = T if unit else 0
            if unit and not first:
                ostep += ostep // unit * T
            size = n + (n // unit * T if unit else 0)
            b = np.arange(n // R)
            t, low = b // sig, b % sig
            j = t % aR
            base = t // aR * (aR * R * sig) + low
            k = j % Ns[i]
            x, y = base + j * sig, base + ((j - k) * R + k) * sig
            src = x + (x // uin * ipad if ipad else 0)
            dst = y + (y // unit * opad if opad else 0)
            reads, writes = [], []
            for r in range(R):
                xr, yr = x + r * aR * sig, y + r * Ns[i] * sig
                reads.append(src + r * istep)
                writes.append(dst + r * ostep)
                assert np.array_equal(reads[-1], xr + (xr // uin * ipad if ipad else 0))
                assert np.array_equal(writes[-1], yr + (yr // unit * opad if opad else 0))
            for s in (reads, writes):
                s = np.concatenate(s)
                assert len(np.unique(s)) == n and s.min() >= 0 and s.max() < size
            Ns[i] *= R


def test_box_walk_steps_by_a_fixed_point():
    """BoxWalk: the slot of a box point after any number of additions of a fixed
    box point, d = 2 and 3."""
    rng = random.Random(2)

    def wrap(x, n):
        return x + n if x < 0 else x - n if x >= n else x

    for _ in range(600):
        d = rng.choice([2, 3])
        H = [[0] * d for _ in range(d)]
        for r in range(d):
            H[r][r] = rng.randint(1, 9)
        for r in range(d):
            for c in range(r + 1, d):
                H[r][c] = rng.randrange(H[r][r])
        m = int(np.prod([H[r][r] for r in range(d)]))
        st = [int(np.prod([H[i][i] for i in range(r + 1, d)])) for r in range(d)]
        y = [rng.randrange(H[r][r]) for r in range(d)]
        c = [rng.randrange(H[r][r]) for r in range(d)]
        point, slot = list(y), sum(a * b for a, b in zip(y, st))
        if d == 2:
            y1, h1 = y[1], H[1][1]
            d0 = c[0] * st[0] + c[1]
            d1 = wrap(c[0] - H[0][1], H[0][0]) * st[0] + c[1] - h1
        else:
            y1, y2, h1, h2, H0 = y[1], y[2], H[1][1], H[2][2], H[0][0]
            r1 = c[1] - H[1][2]
            c1c = r1 + h1 if r1 < 0 else r1
            x0 = wrap(c[0] - H[0][2], H0)
            x0c = wrap(x0 + H[0][1], H0) if r1 < 0 else x0
            d0 = c[0] * st[0] + c[1] * st[1] + c[2]
            d1 = x0c * st[0] + c1c * st[1] + c[2] - h2
            d2 = wrap(c[0] - H[0][1], H0) * st[0] + (c[1] - h1) * st[1] + c[2]
            d3 = wrap(x0c - H[0][1], H0) * st[0] + (c1c - h1) * st[1] + c[2] - h2
        for _ in range(25):
            assert slot == sum(a * b for a, b in zip(point, st))
            point = [a + b for a, b in zip(point, c)]
            for r in range(d - 1, -1, -1):
                q = point[r] // H[r][r]
                for i in range(r + 1):
                    point[i] -= q * H[i][r]
            if d == 2:
                y1 += c[1]
                p = y1 >= h1
                y1 -= h1 if p else 0
                slot += d1 if p else d0
            else:
                y2 += c[2]
                p = y2 >= h2
                y2 -= h2 if p else 0
                y1 += c1c if p else c[1]
                q = y1 >= h1
                y1 -= h1 if q else 0
                slot += (d3 if q else d1) if p else (d2 if q else d0)
            slot -= m if slot >= m else 0


# (M, batch)
PATTERNS = [
    ([[r, 0], [0, 2 * r]], 3) for r in range(2, 17)  # every radix, whole signals
] + [
    ([[17, 0], [0, 17]], 1),            # smallest direct prime, both cycles
    ([[2584]], 2),                      # two direct primes on one axis (8 17 19)
    ([[1021, 3], [0, 4]], 1),           # largest direct prime
    ([[60]], 67),                       # many signals per tile, the last tile not full
    ([[64, 0], [0, 128]], 1),           # 8192 points: the largest whole signal of a small batch
    ([[120, 8], [0, 120]], 65),         # 14400 points: whole from 64 signals on
    ([[120, 8], [0, 120]], 2),          # and two passes below
    ([[15200]], 1),                     # one row of 19 800: narrow direct items
    ([[1200, 240], [0, 1080]], 1),      # one row of 10800 per tile
    ([[135, 0], [0, 1215]], 2),         # a last column tile that is not full
    ([[9, 0], [0, 1350]], 2),           # several rows per tile, a last tile that is not full
    ([[300, 7], [0, 450]], 1),          # a split cycle of 135000
    ([[509, 3], [0, 503]], 1),          # a split cycle of two direct primes
    ([[131072]], 1),                    # d = 1, split power of two
    ([[27, 1], [0, 729]], 2),           # 3^9, split
    ([[2, 0, 0], [0, 6, 0], [0, 0, 30000]], 1),  # split, pencils over three axes
    ([[96, 0, 0], [0, 48, 0], [0, 0, 12]], 1),   # pencils over two axes
    ([[2, 1, 0, 0], [0, 3, 1, 0], [0, 0, 5, 1], [0, 0, 0, 700]], 1),  # d = 4
]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128], ids=["c64", "c128"])
@pytest.mark.parametrize("M,batch", PATTERNS, ids=[str(i) for i in range(len(PATTERNS))])
def test_mixed_passes(M, batch, dtype):
    m = abs(L.det(M))
    plan = pf.PatternFFT(M, batch, dtype)
    tol = TOL["c64" if dtype == torch.complex64 else "c128"]
    c = SI.complex_normal(batch, m, seed=m % 97, dtype=np.complex64 if dtype == torch.complex64 else np.complex128)
    y = plan.forward(torch.from_numpy(c).cuda())
    yh = y.cpu().numpy()
    last = batch - 1
    slots = SI.sample_slots(m, 1024 if m > 4096 else m, seed=3)
    assert rel_l2(yh[last:, slots], oracle.pattern_fft(M, c[last:], out_slots=slots)) <= tol
    assert np.allclose(np.linalg.norm(yh, axis=1), np.linalg.norm(c, axis=1), rtol=1e-5)
    back = plan.inverse(y).cpu().numpy()
    assert rel_l2(back, c) <= tol
    ref = oracle.pattern_fft(M, yh[:1].astype(np.complex128), inverse=True, out_slots=slots)
    assert rel_l2(back[:1, slots], ref) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("M", [[[300, 7], [0, 450]], [[135, 0], [0, 1215]], [[40, 3], [0, 60]],
                               [[2, 0, 0], [0, 6, 0], [0, 0, 30000]]], ids=["split", "rows", "whole", "three"])
def test_transposed_route(M):
    """Both directions through the plan of M^T equal the direct passes (the
    adjoint passes of a mixed-radix plan without and with conjugations)."""
    m = abs(L.det(M))
    x = torch.from_numpy(SI.complex_normal(2, m, seed=8)).cuda()
    a, b = pf.PatternFFT(M, 2), pf.PatternFFT(M, 2, route="transposed")
    assert b.route == (True, True)
    for f in ("forward", "inverse"):
        u, v = getattr(a, f)(x).cpu().numpy(), getattr(b, f)(x).cpu().numpy()
        assert rel_l2(v, u) <= TOL["c64"]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128], ids=["c64", "c128"])
@pytest.mark.parametrize("M", [[[160, 150], [0, 270]], [[480, 60], [0, 540]], [[240, 48], [0, 216]],
                               [[720, 16], [0, 720]], [[1200, 240], [0, 1080]]],
                         ids=["step16", "step8", "rows", "several", "step40"])
def test_strided_column_order(M, dtype):
    """Rows whose column order steps by multiples of the banks: the workspace
    side of a row tile is padded by a unit of its own (pad_unit)."""
    test_mixed_passes(M, 2, dtype)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128], ids=["c64", "c128"])
def test_one_launch_tile_limit(dtype):
    """A single-launch batch plans tiles of at most 512 threads; columns of 96^2
    points have no such tile in complex64 and keep the larger one."""
    n = 96 if dtype == torch.complex64 else 64
    Ms = [[[n, 0, 0], [0, n, 0], [0, 0, n]], [[16, 3], [0, 30]], [[10800]]]
    A = pf.PatternBatch(Ms, None, dtype=dtype)
    Q = pf.PatternBatch(Ms, None, dtype=dtype, flags=pf.PFFT_BATCH_ONE_LAUNCH)
    x = SI.complex_normal(1, A.total, seed=5, dtype=np.complex64 if dtype == torch.complex64 else np.complex128)
    x = torch.from_numpy(x[0]).cuda()
    want, got = A.forward(x), Q.forward(x)
    Q.check_device_status()
    tol = TOL["c64" if dtype == torch.complex64 else "c128"]
    off = 0
    for M in Ms:
        m = abs(L.det(M))
        assert rel_l2(got[off:off + m].cpu().numpy(), want[off:off + m].cpu().numpy()) <= tol
        off += m
