"""GPU parity of the synthesis in fused launches: every split of the levels into
groups of three, two and one, odd batches (a last signal alone), both symbols,
reconstruct and adjoint, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1107_5415_gb300 as pf
import seeded_inputs as SI
from parity_util import TOL, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("symbol", [pf.PWT_DIRICHLET, pf.PWT_DLVP], ids=["dirichlet", "dlvp"])
@pytest.mark.parametrize("levels,batch", [(1, 1), (2, 3), (3, 1), (4, 5), (5, 2), (6, 4), (7, 3)])
def test_synthesis(levels, batch, symbol):
    M, Js = [[24, 24], [-24, 24]], SI.wavelet_dilations(levels)
    plan = pf.WaveletSplit(M, Js, symbol, 0.125, batch)
    c = SI.complex_normal(batch, plan.sizes[0], 40 + levels)
    s, w = plan.decompose(torch.from_numpy(c).cuda())
    back = plan.reconstruct(s, w).cpu().numpy()
    assert rel_l2(back, c) <= TOL["c64"]
    # adjoint: <decompose x, y> = <x, adjoint y> for random parts y
    ys = [SI.complex_normal(batch, n, 60 + i) for i, n in enumerate([plan.sizes[-1]] + list(plan.sizes[1:]))]
    adj = plan.adjoint(torch.from_numpy(ys[0]).cuda(), [torch.from_numpy(y).cuda() for y in ys[1:]]).cpu().numpy()
    parts = [s.cpu().numpy()] + [x.cpu().numpy() for x in w]
    for b in range(batch):
        lhs = sum(np.vdot(y[b], p[b].astype(np.complex128)) for y, p in zip(ys, parts))
        rhs = np.vdot(adj[b].astype(np.complex128), c[b])
        assert abs(lhs - rhs) <= TOL["c64"] * np.linalg.norm(adj[b]) * np.linalg.norm(c[b])
    if symbol == pf.PWT_DIRICHLET:
        # the Dirichlet split is unitary: its adjoint is its inverse, checked against the oracle's cascade
        s_ref, w_ref = oracle.wavelet_cascade(M, Js, c)
        ref = [torch.from_numpy(np.ascontiguousarray(x)).to(torch.complex64).cuda() for x in [s_ref] + list(w_ref)]
        assert rel_l2(plan.adjoint(ref[0], ref[1:]).cpu().numpy(), c) <= TOL["c64"]
        assert rel_l2(plan.reconstruct(ref[0], ref[1:]).cpu().numpy(), c) <= TOL["c64"]
