"""Host side of plan creation against a stand-in for the CUDA runtime
(fake_cudart.cpp): what is still in flight when a plan is handed out, which
kernels a call launches, which lengths have a plan; and on a GPU the calls that
these decide."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
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


@pytest.mark.parametrize("flags", [0, pf.PFFT_BATCH_RADIX8, pf.PFFT_BATCH_AUTOTUNE, pf.PFFT_BATCH_ONE_LAUNCH],
                         ids=["grouped", "radix8", "autotune", "one-launch"])
def test_batch_tables_are_built_when_the_batch_is(fake, flags):
    """The schedule, the stage tables of its radices and the split tables, for
    launches on streams that do not wait for the default one."""
    Ms = [[[96, 0], [0, 96]], [[64, 2], [0, 256]], [[1200, 240], [0, 1080]], [[60]]]
    Js = [[[2, 0], [0, 1]], [[2, 0], [0, 1]], [[3, 0], [0, 1]], [[2]]]
    flat = [x for A in Ms for r in A for x in r], [x for A in Js for r in A for x in r]
    (_, m), (_, j) = _capi._i64(flat[0]), _capi._i64(flat[1])
    h = ctypes.c_void_p()
    fake.fake_reset()
    d = (ctypes.c_int * len(Ms))(*[len(A) for A in Ms])
    assert fake.pfft_batch_create(ctypes.byref(h), len(Ms), d, m, j, pf.PWT_DIRICHLET, 0.0, 0, flags) == 0
    assert fake.fake_pending() == 0
    fake.pfft_batch_destroy(h)


def _launches(lib):
    """(kernel, grid x, grid y, threads) of the launches since fake_reset()."""
    return [(lib.fake_kernel(i).decode(), lib.fake_grid_x(i), lib.fake_grid_y(i), lib.fake_threads(i))
            for i in range(lib.fake_launches())]


def _synthesis(lib, size, levels, batch, dtype=0):
    """Launches of a reconstruction of a quincunx cascade."""
    d, (_, m) = _capi._mat([[size, size], [-size, size]])
    _, j = _capi._i64([x for J in SI.wavelet_dilations(levels) for r in J for x in r])
    h = ctypes.c_void_p()
    assert lib.pwt_plan_create(ctypes.byref(h), d, m, levels, j, pf.PWT_DLVP, 0.25, batch, dtype, 0) == 0
    lib.fake_reset()
    assert lib.pwt_reconstruct(h, 4096, _capi._ptr_array([4096] * levels), 8192, None) == 0
    lib.pwt_plan_destroy(h)
    return _launches(lib)


def test_synthesis_is_fused_where_symbol_tables_exist(fake):
    """Fewer than four signals have none: one level a launch."""
    assert ["fused" in k for k, *_ in _synthesis(fake, 64, 7, 3)] == [False] * 7
    assert ["fused" in k for k, *_ in _synthesis(fake, 64, 7, 4)] == [False, True, True]


def _band_kernel(lib, p, mode, dtype=0):
    """The kernel that splits (0) or merges (1) a pattern by diag(p, 1)."""
    d, (_, m) = _capi._mat([[8 * p, 0], [0, 64]])
    _, j = _capi._i64([p, 0, 0, 1])
    lib.fake_reset()
    f = lib.pwt_merge_general if mode else lib.pwt_split_general
    assert f(d, m, j, 4, dtype, None, 4096, 8192, None) == 0
    (k, *_), = _launches(lib)
    return k


@pytest.mark.parametrize("mode", [0, 1], ids=["split", "merge"])
def test_large_primes_run_in_a_kernel_of_their_own(fake, mode):
    """Beside the code of the small fibres their loop is slower."""
    assert "split_prime_small" in _band_kernel(fake, 5, mode)
    small, wide = _band_kernel(fake, 1021, mode), _band_kernel(fake, 1031, mode)
    assert "split_prime_kernel" in small and "split_prime_kernel" in wide and small != wide


def test_fibres_of_seven_in_registers_where_they_fit(fake):
    """A split by seven in double precision takes the chunks of the larger primes."""
    assert "split_prime_small" in _band_kernel(fake, 7, 0) and "split_prime_small" in _band_kernel(fake, 7, 1, 1)
    assert "split_prime_kernel" in _band_kernel(fake, 7, 0, 1)


ROWS = {2048: [[512, 128], [0, 512]], 4096: [[8, 0], [0, 4096]], 8192: [[4, 0], [0, 8192]], 16384: [[4, 0], [0, 16384]]}


@pytest.mark.parametrize("inverse", [False, True], ids=["forward", "inverse"])
@pytest.mark.parametrize("n", ROWS)
def test_bulk_copies_only_where_they_are_aligned(fake, n, inverse):
    """A bulk copy starts on 16 bytes: rows of a signal that begins 8 bytes past
    such an address are read and written element by element."""
    st, h = _create(fake, ROWS[n])
    assert st == 0
    f = fake.pfft_inverse if inverse else fake.pfft_forward
    for src, dst, bulk in ((4096, 8192, True), (4104, 8192, inverse), (4096, 8200, not inverse), (4104, 8200, False)):
        fake.fake_reset()
        assert f(h, src, dst, None) == 0
        rows = fake.fake_kernel(1 if inverse else 0).decode()
        assert ("row_tma" in rows or "row_pipe" in rows) if bulk else "row_fast" in rows
    fake.pfft_plan_destroy(h)


@pytest.mark.gpu
def test_long_cycle_beside_a_long_pencil():
    """Cycles 1024 and 32768: rows of 8192, columns over axes of 1024 and 4."""
    M = [[4096, 1024], [0, 8192]]
    m = abs(L.det(M))
    plan = pf.PatternFFT(M, 1)
    c = SI.complex_normal(1, m, seed=67)
    y = plan.forward(torch.from_numpy(c).cuda())
    slots = SI.sample_slots(m, 16, seed=3)
    assert rel_l2(y.cpu().numpy()[:, slots], oracle.pattern_fft(M, c, out_slots=slots)) <= TOL["c64"]
    assert rel_l2(plan.inverse(y).cpu().numpy(), c) <= TOL["c64"]

# matrix, signals, complex128, whole signals in one tile
WHOLE = [([[512]], 4096, 0, True), ([[1024]], 304, 0, True), ([[1024]], 305, 0, False), ([[4096]], 1, 0, False),
         ([[16384]], 70, 0, False), ([[8192]], 1, 0, False), ([[4096]], 1, 1, True), ([[90, 0], [0, 90]], 1, 0, True),
         ([[64, 0], [0, 128]], 1, 0, True), ([[128, 0], [0, 128]], 100, 0, False), ([[128, 0], [0, 128]], 101, 0, True),
         ([[120, 0], [0, 120]], 64, 0, True), ([[120, 0], [0, 120]], 63, 0, False), ([[8, 0], [0, 2048]], 64, 0, True),
         ([[64, 0], [0, 64]], 100, 1, False), ([[64, 0], [0, 64]], 101, 1, True), ([[32, 0], [0, 64]], 1, 1, True),
         ([[64, 0], [0, 128]], 64, 1, False), ([[16, 0, 0], [0, 16, 0], [0, 0, 32]], 200, 1, False),
         ([[60, 0], [0, 72]], 64, 1, True), ([[8192]], 64, 1, True)]


@pytest.mark.parametrize("M,batch,c128,whole", WHOLE)
def test_whole_signals_in_a_tile(fake, M, batch, c128, whole):
    st, h = _create(fake, M, batch, c128)
    assert st == 0
    fake.fake_reset()
    assert fake.pfft_forward(h, 4096, 8192, None) == 0
    kernels = [k for k, *_ in _launches(fake)]
    assert (len(kernels) == 1 and "mixed_kernel" in kernels[0]) == whole
    fake.pfft_plan_destroy(h)


@pytest.mark.gpu
@pytest.mark.parametrize("M,batch,c128,whole", WHOLE)
def test_transform_of_many_signals(M, batch, c128, whole):
    m = abs(L.det(M))
    plan = pf.PatternFFT(M, batch, torch.complex128 if c128 else torch.complex64)
    tol = TOL["c128" if c128 else "c64"]
    c = SI.complex_normal(batch, m, seed=m % 71, dtype=np.complex128 if c128 else np.complex64)
    y = plan.forward(torch.from_numpy(c).cuda())
    slots = SI.sample_slots(m, 64, seed=3)
    assert rel_l2(y.cpu().numpy()[-2:, slots], oracle.pattern_fft(M, c[-2:], out_slots=slots)) <= tol
    assert rel_l2(plan.inverse(y).cpu().numpy(), c) <= tol


def test_complex128_cycles_with_factors_11_and_13(fake):
    """Two equal cycles of n points, 11 or 13 dividing n: the row and the column
    each take a tile of 512 threads, 16 points a thread, wherever the other
    factors do (15 points in radices 3 and 5, 14 in radix 7)."""
    tried = 0
    for n in range(11 * 400, 8193):
        if n % 11 and n % 13:
            continue
        primes = [p for p in range(2, 1022) if n % p == 0 and all(p % q for q in range(2, p))]
        rest = n
        for p in primes:
            while rest % p == 0:
                rest //= p
        if rest > 1 or n > 512 * min([16] + [{3: 15, 5: 15, 7: 14}[p] for p in primes if p in (3, 5, 7)]):
            continue
        tried += 1
        st, h = _create(fake, [[n, 0], [0, n]], 1, 1)
        assert st == 0, n
        fake.pfft_plan_destroy(h)
    assert tried > 300


@pytest.mark.gpu
@pytest.mark.parametrize("M,batch", [([[77, 0, 0], [0, 77, 0], [0, 0, 77]], 2),      # column 7 7 11 11
                                     ([[26, 0, 0], [0, 286, 0], [0, 0, 286]], 1),   # column 2 2 11 13 13
                                     ([[88, 0, 0], [0, 88, 0], [0, 0, 88]], 1),     # column 2^6 11 11
                                     ([[6006, 0], [0, 6006]], 1)],                  # row and column
                         ids=["77", "26-286", "88", "6006"])
def test_complex128_direct_11_and_13(M, batch):
    m = abs(L.det(M))
    plan = pf.PatternFFT(M, batch, torch.complex128)
    c = SI.complex_normal(batch, m, seed=m % 79, dtype=np.complex128)
    y = plan.forward(torch.from_numpy(c).cuda())
    yh = y.cpu().numpy()
    slots = SI.sample_slots(m, 16 if m > 1 << 24 else 256, seed=3)
    assert rel_l2(yh[:, slots], oracle.pattern_fft(M, c, out_slots=slots)) <= TOL["c128"]
    assert rel_l2(plan.inverse(y).cpu().numpy(), c) <= TOL["c128"]
    ref = oracle.pattern_fft(M, yh, inverse=True, out_slots=slots)
    assert rel_l2(c[:, slots], ref) <= TOL["c128"]


@pytest.mark.parametrize("n,batch", [(1021, 4), (1004, 8), (1124, 1), (727, 4)])
def test_complex128_direct_sums_share_an_sm(fake, n, batch):
    """A tile of direct sums has its SM alone only when it must: at 128 registers a
    thread, 256 threads leave room for a second one."""
    st, h = _create(fake, [[n, 0], [0, n]], batch, 1)
    assert st == 0
    fake.fake_reset()
    assert fake.pfft_forward(h, 4096, 8192, None) == 0
    assert [t <= 256 for *_, t in _launches(fake)] == [True, True]
    fake.pfft_plan_destroy(h)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128], ids=["c64", "c128"])
@pytest.mark.parametrize("M,batch", [([[37, 0], [0, 74]], 5), ([[101, 0], [0, 101]], 3), ([[281, 0], [0, 1124]], 1),
                                     ([[997]], 5), ([[643, 0], [0, 283]], 2), ([[1021, 0], [0, 127]], 1),
                                     ([[17, 0], [0, 323]], 2), ([[29, 1], [0, 4 * 29 * 31]], 1)],
                         ids=["37", "101", "281", "997", "643-283", "1021-127", "17-19", "29-31"])
def test_direct_sums(M, batch, dtype):
    """One to three turns of items, one to sixteen pencils a tile."""
    m = abs(L.det(M))
    plan = pf.PatternFFT(M, batch, dtype)
    tol = TOL["c64" if dtype == torch.complex64 else "c128"]
    c = SI.complex_normal(batch, m, seed=m % 73, dtype=np.complex64 if dtype == torch.complex64 else np.complex128)
    y = plan.forward(torch.from_numpy(c).cuda())
    slots = SI.sample_slots(m, min(m, 512), seed=3)
    assert rel_l2(y.cpu().numpy()[:, slots], oracle.pattern_fft(M, c, out_slots=slots)) <= tol
    assert rel_l2(plan.inverse(y).cpu().numpy(), c) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("n", ROWS)
def test_transform_of_a_view_aligned_to_one_element(n):
    M = ROWS[n]
    m = abs(L.det(M))
    plan = pf.PatternFFT(M, 2)
    c = SI.complex_normal(2, m, seed=m % 83)

    def view():
        return torch.empty(2 * m + 1, dtype=torch.complex64, device="cuda")[1:].view(2, m)

    x = view().copy_(torch.from_numpy(c))
    y, z = view(), view()
    assert x.data_ptr() % 16 == 8
    plan.forward(x, out=y)
    plan.inverse(y, out=z)
    slots = SI.sample_slots(m, 1024, seed=3)
    assert rel_l2(y.cpu().numpy()[:, slots], oracle.pattern_fft(M, c, out_slots=slots)) <= TOL["c64"]
    assert rel_l2(z.cpu().numpy(), c) <= TOL["c64"]


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
