"""Host side of plan creation against a stand-in for the CUDA runtime
(fake_cudart.cpp): what is still in flight when a plan is handed out."""
import ctypes
import os
import shutil
import subprocess

import pytest
import torch

import oracle
from oracle import lattice as L
import paper_1107_5415_gb300 as pf
from paper_1107_5415_gb300 import _capi, build_lib
import seeded_inputs as SI
from parity_util import TOL, rel_l2

CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """The library's objects linked with the stand-in runtime."""
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INCLUDE):
        pytest.skip("needs g++ and the CUDA headers")
    pf.library_path()
    objs = [os.path.join(build_lib.BUILD, os.path.basename(s) + ".o") for s in build_lib._sources()]
    if not all(os.path.exists(o) for o in objs):
        build_lib.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "libpfft_fake.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fake_cudart.cpp")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-O1", "-I", CUDA_INCLUDE, "-Wl,-Bsymbolic", "-Wl,-z,defs",
                    src, *objs, "-o", out], check=True)
    lib = ctypes.CDLL(out)
    for name, (res, args) in _capi._SIGS.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    lib.fake_kernel.restype = ctypes.c_char_p
    return lib


def _create(lib, M, batch=1, dtype=0, flags=0):
    """(status, plan handle) of pfft_plan_create."""
    d, (_, p) = _capi._mat(M)
    h = ctypes.c_void_p()
    lib.fake_reset()
    return lib.pfft_plan_create(ctypes.byref(h), d, p, batch, dtype, flags), h


PLANS = {
    "whole": ([[64, 16], [-16, 64]], 1), "whole-many": ([[60]], 67), "whole-direct": ([[17, 0], [0, 34]], 1),
    "two-mixed": ([[1200, 240], [0, 1080]], 2), "one-mixed-row": ([[15200]], 1), "split": ([[300, 7], [0, 450]], 1),
    "fast": ([[512, 128], [0, 512]], 2), "fast-row": ([[2048, 0], [0, 3]], 2),
    "three": ([[2, 0, 0], [0, 6, 0], [0, 0, 30000]], 1),
    "trivial": ([[1]], 1),
}


@pytest.mark.parametrize("flags", [0, pf.PFFT_FLAG_LAYOUT_SNF, pf.PFFT_FLAG_TRANSPOSED, pf.PFFT_FLAG_AUTOTUNE],
                         ids=["direct", "snf", "transposed", "autotune"])
@pytest.mark.parametrize("dtype", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("name", PLANS)
def test_plan_tables_are_built_when_the_plan_is(fake, name, dtype, flags):
    """The first call may come on a stream that does not wait for the default
    one, where the tables are built: nothing is in flight any more."""
    M, batch = PLANS[name]
    st, h = _create(fake, M, batch, dtype, flags)
    assert st == 0 or (st == 5 and flags == pf.PFFT_FLAG_TRANSPOSED)
    if st == 0:
        assert fake.fake_pending() == 0
        fake.pfft_plan_destroy(h)


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["whole", "whole-direct", "two-mixed", "split", "fast"])
def test_first_call_on_a_side_stream(name):
    """A plan made while the default stream is busy, called at once on a stream
    that does not wait for it."""
    M, batch = PLANS[name]
    m = abs(L.det(M))
    c = SI.complex_normal(batch, m, seed=m % 89)
    x = torch.from_numpy(c).cuda()
    side = torch.cuda.Stream()
    busy = torch.ones(1 << 28, device="cuda")
    torch.cuda.synchronize()
    for _ in range(20):
        busy.mul_(1.0)
    plan = pf.PatternFFT(M, batch)
    with torch.cuda.stream(side):
        y = plan.forward(x)
    side.synchronize()
    slots = SI.sample_slots(m, 1024 if m > 4096 else m, seed=3)
    assert rel_l2(y.cpu().numpy()[:, slots], oracle.pattern_fft(M, c, out_slots=slots)) <= TOL["c64"]
