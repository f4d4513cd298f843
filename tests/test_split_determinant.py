"""|det J| of the plan-free splits (_det_int): exact up to the four dimensions
that the library takes, and no slower to refuse more."""
import random
import time

import numpy as np

from oracle import lattice as L
import paper_1107_5415_gb300 as pf


def test_exact_up_to_four_dimensions():
    rng = random.Random(5)
    for d in (1, 2, 3, 4):
        for bound in (3, 1 << 15):
            A = [[rng.randint(-bound, bound) for _ in range(d)] for _ in range(d)]
            assert pf._det_int(A) == abs(L.det(A))


def test_more_dimensions_take_no_longer():
    """The library refuses them; eleven rows by expansion took about ten seconds."""
    A = np.arange(121).reshape(11, 11) % 7 + np.eye(11, dtype=np.int64)
    t = time.perf_counter()
    assert pf._det_int(A) == round(abs(np.linalg.det(A.astype(np.float64))))
    assert time.perf_counter() - t < 1.0
