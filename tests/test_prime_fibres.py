"""GPU parity of the built-in band system on its int32 index path: the primes
that a thread holds whole (2, 3, 5, 7) and those split into chunks of bands, d =
1 .. 3, fibres on the symbol's boundary (even sides), several signals per
thread, and matrices whose numerators need 64 bits.  Tolerances are those
of the parity bar."""
import numpy as np
import pytest
import torch

import oracle
from oracle import lattice as L
import paper_1107_5415_gb300 as pf
import seeded_inputs as SI
from parity_util import TOL, rel_l2

pytestmark = pytest.mark.gpu

CASES = [
    ([[34]], [[17]]),
    ([[30]], [[5]]),
    ([[12, 4], [0, 10]], [[2, 0], [0, 1]]),
    ([[12, 3], [0, 10]], [[3, 0], [0, 1]]),
    ([[40, 10], [0, 12]], [[5, 0], [0, 1]]),
    ([[42, 7], [0, 10]], [[7, 0], [0, 1]]),
    ([[26, 13], [0, 8]], [[13, 0], [0, 1]]),
    ([[34, 17], [0, 6]], [[17, 0], [0, 1]]),
    ([[6, 3, 0], [0, 4, 1], [0, 0, 6]], [[3, 0, 0], [0, 1, 0], [0, 0, 1]]),
    ([[10, 5, 0], [0, 4, 1], [0, 0, 6]], [[5, 0, 0], [0, 1, 0], [0, 0, 1]]),
    ([[14, 7, 7], [0, 4, 1], [0, 0, 2]], [[7, 0, 0], [0, 1, 0], [0, 0, 1]]),
    ([[22, 11, 0], [0, 4, 1], [0, 0, 2]], [[11, 0, 0], [0, 1, 0], [0, 0, 1]]),
    ([[27, 16000011], [0, 27]], [[3, 0], [0, 1]]),  # numerators above 2^29
]


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128], ids=["c64", "c128"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_prime_bands(case, dtype):
    M, J = CASES[case]
    m, p, batch = abs(L.det(M)), abs(L.det(J)), 5
    c = SI.complex_normal(batch, m, 300 + case, dtype=np.complex128)
    tol = TOL["c64" if dtype == torch.complex64 else "c128"]
    parts = pf.split_general(M, J, None, torch.from_numpy(c).to(dtype).cuda()).cpu().numpy()
    ref = oracle.wavelet_level_p(M, J, c_hat=c)
    assert rel_l2(parts.transpose(1, 0, 2).reshape(batch, -1), ref.transpose(1, 0, 2).reshape(batch, -1)) <= tol
    back = pf.merge_general(M, J, None, torch.from_numpy(np.ascontiguousarray(ref)).to(dtype).cuda()).cpu().numpy()
    assert rel_l2(back, c) <= tol


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128], ids=["c64", "c128"])
@pytest.mark.parametrize("M", [[[32, 16000002], [0, 27]], [[-32, 16000002], [0, 27]]], ids=["pos", "neg"])
def test_two_band_split_with_large_numerators(M, dtype):
    """Numerators between 2^29 and 2^60: the 64-bit multiply-high path of the
    weights and phases, both symbols, split and inverse."""
    J, batch = [[2, 0], [0, 1]], 3
    m, tol = abs(L.det(M)), TOL["c64" if dtype == torch.complex64 else "c128"]
    c = SI.complex_normal(batch, m, 77, dtype=np.complex128)
    x = torch.from_numpy(c).to(dtype).cuda()
    plan = pf.WaveletSplit(M, [J], pf.PWT_DIRICHLET, 0.125, batch, dtype)
    s, w = plan.decompose(x)
    s_ref, w_ref = oracle.wavelet_cascade(M, [J], c)
    assert rel_l2(s.cpu().numpy(), s_ref) <= tol and rel_l2(w[0].cpu().numpy(), w_ref[0]) <= tol
    plan = pf.WaveletSplit(M, [J], pf.PWT_DLVP, 0.125, batch, dtype)
    assert rel_l2(plan.reconstruct(*plan.decompose(x)).cpu().numpy(), c) <= tol


def test_zero_weight_members_stay_apart():
    """An infinite coefficient of a member without weight reaches its own band
    only: the other bands of the fibre do not see it."""
    M, J = [[15, 0], [0, 15]], [[3, 0], [0, 1]]
    c = torch.ones((1, 225), dtype=torch.complex64, device="cuda")
    base = pf.split_general(M, J, None, c)
    c[0, 100] = float("inf")
    got = pf.split_general(M, J, None, c)
    assert int((~torch.isfinite(torch.view_as_real(got)).all(-1)).sum()) in (1, 3)
    same = torch.isfinite(torch.view_as_real(got)).all(-1)
    assert torch.equal(got[same], base[same])
