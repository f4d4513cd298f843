"""What the framework is timed on: the work that its users have it do.

``listed()`` holds the named cases, ``draw(rng)`` one more of the same ranges,
``prepare`` what a program has in hand before the call (inputs on the GPU and
the plan it keeps), ``run`` one pass through the public entry points, ``work``
the bytes and operations that a pass cannot do without, and ``exact`` the
outputs in 64 bits from the definitions, without the library.

Matrices are written as text, rows separated by ";" ("64 16; -16 64").
"""
import itertools
import math

import torch

import paper_1107_5415_gb300 as pf

DIAG_A, DIAG_B = "1 1; -1 1", "1 -1; 1 1"  # the two dilations of the quincunx cascade


def _case(kind, matrix, batch=1, dtype="complex64", **more):
    return dict(kind=kind, matrix=matrix, batch=batch, dtype=dtype, **more)


def listed():
    out = []

    def add(name, case):
        out.append(dict(case, name=name))

    # one small signal there and back: latency, four launches
    add("small_2d", _case("transform", "64 16; -16 64"))
    # sixteen images of 2^18 points, resident in the L2: the ordinary call
    add("image_2d", _case("transform", "512 128; 0 512", 16))
    # sides that are no powers of two (2, 3 and 5 as factors)
    add("smooth_2d", _case("transform", "1200 240; 0 1080", 8))
    # cycles (8, 2^19): the long cycle is split over both passes
    add("long_cycle_2d", _case("transform", "2048 8; 0 2048", 8))
    # the batched 2-D workload of the benchmark, the largest call
    add("batched_2d", _case("transform", "4096 1024; 0 4096", 8))
    # double precision, for callers who validate against it
    add("double_2d", _case("transform", "1024 256; 0 1024", 4, "complex128"))
    # a gradient step through a 3-D transform (forward and backward)
    add("grad_3d", _case("gradient", "256 64 0; 0 256 32; 0 0 256", 4))
    # the twelve-level decomposition of a batch of coefficient sets, and its inverse
    add("cascade", _case("decompose", "1024 1024; -1024 1024", 16, levels=12, symbol="dirichlet"))
    add("cascade_back", _case("reconstruct", "1024 1024; -1024 1024", 16, levels=12, symbol="dlvp"))
    # one level of a directional analysis, forward and gradient of the split
    add("directional", _case("split_gradient", "512 0; 0 512", 16, dilation="2 0; 0 1", symbol="dirichlet"))
    # one split by an odd determinant and its inverse, planned in the call
    add("thirds", _case("bands", "768 96; 0 729", 8, dilation="3 0; 0 1"))
    # a serving mix of many patterns of uneven size, each transformed and split once
    add("mix", dict(kind="mix", patterns=512, mix=4, dtype="complex64"))
    return out


# Side lengths of the drawn patterns: powers of two, products of small primes
# and some with a larger prime.
_SIDES = [16, 20, 24, 27, 32, 36, 45, 48, 60, 64, 75, 80, 96, 100, 105, 120, 125, 128, 135, 144, 160, 180, 192, 200,
          210, 225, 240, 243, 256, 270, 288, 300, 320, 343, 352, 360, 375, 384, 400, 416, 420, 432, 450, 480, 500, 512,
          540, 576, 600, 625, 640, 720, 729, 768, 800, 864, 900, 960, 1000, 1024, 1080, 1152, 1200, 1280, 1440, 1536,
          1600, 1728, 1800, 1920, 2000, 2048, 2160, 2400, 2560, 2880, 3072, 3600, 4096]


def _triangular(rng, d, max_points):
    """An upper-triangular pattern matrix, its number of points log-uniform."""
    goal = math.exp(rng.uniform(math.log(1024), math.log(max_points)))
    side = goal ** (1.0 / d)
    while True:
        diag = [rng.choice([s for s in _SIDES if side / 3 <= s <= max(side * 3, 20)]) for _ in range(d)]
        if not 512 <= math.prod(diag) <= max_points:
            continue
        M = [[0] * d for _ in range(d)]
        for r in range(d):
            M[r][r] = diag[r]
            if r + 1 < d:  # off-diagonal: a multiple of a divisor of the sides, so that the cycles vary
                g = math.gcd(diag[r], diag[r + 1])
                g //= rng.choice([f for f in (1, 2, 4, 8, 3, 5) if g % f == 0])
                M[r][r + 1] = g * rng.randrange(max(1, diag[r] // g))
        eps = _smith(M)[1]
        if math.prod(eps[:-1]) <= 2048 and eps[-1] < 1 << 22:
            return M


def _text(M):
    return "; ".join(" ".join(str(x) for x in row) for row in M)


def draw(rng):
    kind = rng.choice(["transform", "transform", "transform", "gradient", "decompose", "reconstruct",
                       "split_gradient", "bands", "mix"])
    if kind == "mix":
        return dict(kind="mix", patterns=int(math.exp(rng.uniform(math.log(16), math.log(512)))),
                    mix=rng.randrange(1000), dtype="complex64")
    batch = int(math.exp(rng.uniform(0.0, math.log(24.99))))
    dtype = "complex128" if rng.random() < 0.25 else "complex64"
    if kind in ("transform", "gradient"):
        M = _triangular(rng, rng.choice([2, 2, 3]), (1 << 26) // (batch * (4 if dtype == "complex128" else 1)))
        return _case(kind, _text(M), batch, dtype)
    symbol = rng.choice(["dirichlet", "dlvp"])
    if kind == "bands":
        p = rng.choice([3, 5, 7])
        a, b = p * rng.randrange(20, 1200 // p), rng.randrange(60, 1200)
        return _case(kind, f"{a} {p * rng.randrange(a // p)}; 0 {b}", batch, dtype, dilation=f"{p} 0; 0 1")
    if kind == "split_gradient":
        a, b = 2 * rng.randrange(30, 600), 2 * rng.randrange(30, 600)
        return _case(kind, f"{a} 0; 0 {b}", batch, dtype, dilation=rng.choice(["2 0; 0 1", "1 0; 0 2", DIAG_B]),
                     symbol=symbol)
    # cascades: c 2^e [[1, 1], [-1, 1]] can be split 2 e + 1 times
    e = rng.randrange(3, 10)
    c = rng.choice([1, 1, 3, 5, 7])
    while c << e > 1024:
        e -= 1
    s = c << e
    return _case(kind, f"{s} {s}; {-s} {s}", batch, dtype, levels=rng.randrange(2, min(12, 2 * e + 1) + 1), symbol=symbol)


def _matrix(text):
    return [[int(x) for x in row.split()] for row in text.split(";")]


def _dilations(case):
    if "dilation" in case:
        return [_matrix(case["dilation"])]
    return [_matrix((DIAG_A, DIAG_B)[l % 2]) for l in range(case["levels"])]


def _mix(case):
    """The patterns of a serving mix and their dilations: upper-triangular, d
    uniform in {2, 3}, diagonals uniform in [16, 512], off-diagonals below the
    diagonal entry of their row, at most 2^20 points; each is split by a
    dilation whose determinant is the smallest prime in its size."""
    import random
    rng = random.Random(case["mix"])
    Ms, Js = [], []
    while len(Ms) < case["patterns"]:
        d = rng.randint(2, 3)
        M = [[0] * d for _ in range(d)]
        for r in range(d):
            M[r][r] = rng.randint(16, 512)
        for r in range(d):
            for c in range(r + 1, d):
                M[r][c] = rng.randrange(M[r][r])
        m = math.prod(M[r][r] for r in range(d))
        if m > 1 << 20:
            continue
        p = next(f for f in range(2, m + 1) if m % f == 0)
        # v with v^T M = 0 mod p, v_r = 1, zero before r = the last row with
        # p | M_rr; J Z^d = {x : v . x = 0 mod p}
        r = max(i for i in range(d) if M[i][i] % p == 0)
        v = [0] * d
        v[r] = 1
        for j in range(r + 1, d):
            v[j] = -sum(v[i] * M[i][j] for i in range(r, j)) * pow(M[j][j], -1, p) % p
        J = [[int(i == j) for j in range(d)] for i in range(d)]
        for j in range(d):
            J[r][j] = p if j == r else -v[j]
        Ms.append(M)
        Js.append(J)
    return Ms, Js


def _det(M):
    if len(M) == 1:
        return M[0][0]
    return sum((-1) ** j * M[0][j] * _det([row[:j] + row[j + 1:] for row in M[1:]]) for j in range(len(M)) if M[0][j])


def _normal(shape, dtype, gen):
    """Complex values, real and imaginary parts i.i.d. N(0, 1)."""
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    return torch.view_as_complex(torch.randn((*shape, 2), dtype=real, device="cuda", generator=gen))


def _inputs(case, seed):
    """The input tensors of a case, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype = getattr(torch, case["dtype"])
    if case["kind"] == "mix":
        return [_normal((sum(abs(_det(M)) for M in _mix(case)[0]),), dtype, gen)]
    M = _matrix(case["matrix"])
    m, batch = abs(_det(M)), case["batch"]
    x = _normal((batch, m), dtype, gen)
    if case["kind"] == "transform":
        return [x]
    if case["kind"] == "gradient":
        return [x, _normal((batch, m), dtype, gen)]
    # Fourier coefficients: N(0, 1) weighted by 1 / (1 + |h|^2), h the centred frequency
    T = torch.tensor(_transpose(M), dtype=torch.float64, device="cuda")
    k = _points(_hermite(_transpose(M))).double()
    h = k - torch.round(k @ torch.linalg.inv(T).T) @ T.T
    c = (x / (1 + (h * h).sum(1))).to(dtype)
    if case["kind"] in ("decompose", "bands"):
        return [c]
    # parts on every level, of the same energy
    sizes = [m >> (l + 1) for l in range(len(_dilations(case)))]
    parts = [_normal((batch, n), dtype, gen) for n in [sizes[-1]] + sizes]
    return parts if case["kind"] == "reconstruct" else [c] + parts


def prepare(case, seed):
    state = dict(kind=case["kind"], x=_inputs(case, seed))
    dtype = getattr(torch, case["dtype"])
    if case["kind"] == "mix":
        Ms, Js = _mix(case)
        state["plan"] = pf.PatternBatch(Ms, Js, pf.PWT_DIRICHLET, dtype=dtype)
    elif case["kind"] in ("transform", "gradient"):
        state["plan"] = pf.PatternFFT(_matrix(case["matrix"]), case["batch"], dtype)
    elif case["kind"] == "bands":
        state["M"], state["J"] = _matrix(case["matrix"]), _matrix(case["dilation"])
    else:
        symbol = pf.PWT_DIRICHLET if case["symbol"] == "dirichlet" else pf.PWT_DLVP
        state["plan"] = pf.WaveletSplit(_matrix(case["matrix"]), _dilations(case), symbol, 0.125, case["batch"], dtype)
    if case["kind"] in ("gradient", "split_gradient"):
        state["x"][0].requires_grad_(True)
    return state


def run(state):
    kind, x, plan = state["kind"], state["x"], state.get("plan")
    if kind == "transform":
        y = plan.forward(x[0])
        return [y, plan.inverse(y)]
    if kind == "gradient":
        y = pf.pattern_fft(x[0], plan)
        return [y.detach(), *torch.autograd.grad(y, x[0], x[1])]
    if kind == "decompose":
        scaling, wavelets = plan.decompose(x[0])
        return [scaling, *wavelets]
    if kind == "reconstruct":
        return [plan.reconstruct(x[0], x[1:])]
    if kind == "split_gradient":
        scaling, wavelets = pf.wavelet_decompose(x[0], plan)
        grad = torch.autograd.grad([scaling, *wavelets], x[0], x[1:])
        return [scaling.detach(), *(w.detach() for w in wavelets), *grad]
    if kind == "bands":
        parts = pf.split_general(state["M"], state["J"], None, x[0])
        return [parts, pf.merge_general(state["M"], state["J"], None, parts)]
    return list(plan.forward(x[0]))


def work(case):
    esize = 8 if case["dtype"] == "complex64" else 16
    if case["kind"] == "mix":
        sizes = [abs(_det(M)) for M in _mix(case)[0]]
        total = sum(sizes)
        # the signal in, the coefficients out, the split parts out
        return dict(bytes=3 * esize * total, flops=sum(5 * m * math.log2(m) for m in sizes) + 10 * total)
    m = abs(_det(_matrix(case["matrix"])))
    n = m * case["batch"]
    if case["kind"] in ("transform", "gradient"):  # two transforms
        return dict(bytes=4 * esize * n, flops=2 * 5 * n * math.log2(m))
    if case["kind"] in ("decompose", "reconstruct"):
        return dict(bytes=2 * esize * n, flops=10 * sum(n >> l for l in range(case["levels"])))
    return dict(bytes=4 * esize * n, flops=20 * n)


# ---- the outputs in 64 bits, from the definitions


def _transpose(M):
    return [list(r) for r in zip(*M)]


def _mul(A, B):
    return [[sum(a * b for a, b in zip(row, col)) for col in zip(*B)] for row in A]


def _adjugate(M):
    d = len(M)
    if d == 1:
        return [[1]]
    return [[(-1) ** (i + j) * _det([row[:i] + row[i + 1:] for k, row in enumerate(M) if k != j]) for j in range(d)]
            for i in range(d)]


def _hermite(A):
    """Column-style Hermite normal form: upper triangular, positive diagonal,
    0 <= H_rc < H_rr for c > r."""
    d = len(A)
    cols = _transpose(A)
    for r in range(d - 1, -1, -1):
        while any(cols[c][r] for c in range(r)):
            c = min((c for c in range(r + 1) if cols[c][r]), key=lambda c: abs(cols[c][r]))
            cols[c], cols[r] = cols[r], cols[c]
            for c in range(r):
                q = cols[c][r] // cols[r][r]
                cols[c] = [a - q * b for a, b in zip(cols[c], cols[r])]
        if cols[r][r] < 0:
            cols[r] = [-a for a in cols[r]]
        for c in range(r + 1, d):
            q = cols[c][r] // cols[r][r]
            cols[c] = [a - q * b for a, b in zip(cols[c], cols[r])]
    return _transpose(cols)


def _smith(M):
    """(U, eps, V) with U M V = diag(eps), U and V unimodular, eps_j | eps_{j+1}."""
    d = len(M)
    A = [list(r) for r in M]
    U = [[int(i == j) for j in range(d)] for i in range(d)]
    V = [[int(i == j) for j in range(d)] for i in range(d)]

    def row_op(i, j, q):  # row i -= q row j
        for X in (A, U):
            X[i] = [a - q * b for a, b in zip(X[i], X[j])]

    def col_op(i, j, q):  # column i -= q column j
        for X in (A, V):
            for row in X:
                row[i] -= q * row[j]

    for t in range(d):
        while True:
            i, j = min(((i, j) for i in range(t, d) for j in range(t, d) if A[i][j]), key=lambda p: abs(A[p[0]][p[1]]))
            for X in (A, U):
                X[t], X[i] = X[i], X[t]
            for X in (A, V):
                for row in X:
                    row[t], row[j] = row[j], row[t]
            for i in range(t + 1, d):
                row_op(i, t, A[i][t] // A[t][t])
            for j in range(t + 1, d):
                col_op(j, t, A[t][j] // A[t][t])
            if any(A[i][t] for i in range(t + 1, d)) or any(A[t][t + 1:]):
                continue
            bad = next((i for i in range(t + 1, d) if any(x % A[t][t] for x in A[i][t + 1:])), None)
            if bad is None:
                break
            row_op(t, bad, -1)
        if A[t][t] < 0:
            for X in (A, U):
                X[t] = [-a for a in X[t]]
    return U, [A[t][t] for t in range(d)], V


def _points(H):
    """The box points of H, [m, d], row-major."""
    d = len(H)
    axes = [torch.arange(H[r][r], device="cuda") for r in range(d)]
    return torch.stack(torch.meshgrid(*axes, indexing="ij"), -1).reshape(-1, d)


def _slots(H, y):
    """Slots of the points y [n, d] reduced into the box of H."""
    y = y.clone()
    s, stride = 0, 1
    for r in range(len(H) - 1, -1, -1):
        q = torch.div(y[:, r], H[r][r], rounding_mode="floor")
        for i in range(r + 1):
            y[:, i] -= q * H[i][r]
        s = s + y[:, r] * stride
        stride *= H[r][r]
    return s


def _smith_index(rows, eps, points):
    """Row-major index over the cycles of the coordinates (rows . point) mod eps."""
    s = 0
    for row, e in zip(rows, eps):
        t = sum((a % e) * points[:, c] for c, a in enumerate(row)) % e
        s = s * e + t
    return s


def _transform(M, c, inverse=False):
    """The unitary transform on the pattern of M, [batch, m]: k^T M^{-1} y =
    sum_j mu_j lambda_j / eps_j with lambda = U y, mu = V^T k."""
    U, eps, V = _smith(M)
    m = c.shape[-1]
    lam = _smith_index(U, eps, _points(_hermite(M)))
    mu = _smith_index(_transpose(V), eps, _points(_hermite(_transpose(M))))
    src, dst, fft = (mu, lam, torch.fft.ifftn) if inverse else (lam, mu, torch.fft.fftn)
    dims = list(range(1, len(eps) + 1))
    out = torch.empty(c.shape, dtype=torch.complex128, device=c.device)
    for b in range(c.shape[0]):
        x = torch.empty(m, dtype=torch.complex128, device=c.device)
        x[src] = c[b].to(torch.complex128)
        out[b] = fft(x.reshape(1, *eps), dim=dims, norm="ortho").reshape(-1)[dst]
    return out


def _fibres(M, J, symbol):
    """One split level M = J N: slots of the fibre members [p, n], their
    periodised weights [p, n], the wavelet phase [n] and N."""
    d, detJ, detM = len(M), _det(J), _det(M)
    p, q = abs(detJ), abs(detM)
    N = [[x // detJ for x in row] for row in _mul(_adjugate(J), M)]
    HM, HN = _hermite(_transpose(M)), _hermite(_transpose(N))
    # v: J v = 0 mod p, scaled to 1 at its first non-zero entry i (the generator is e_i)
    v = next(col for col in ([x % p for x in c] for c in zip(*_adjugate(J))) if any(col))
    i = next(i for i in range(d) if v[i])
    v = [x * pow(v[i], -1, p) % p for x in v]
    z = [x - p if 2 * x >= p else x for x in v]  # p times the centred generator of the pattern of J
    u = [sum(a * b for a, b in zip(row, z)) // p for row in J]
    sign = 1 if detM > 0 else -1
    phase = [sign * sum(a * b for a, b in zip(row, u)) % q for row in _adjugate(M)]
    K = [[sign * x for x in row] for row in _mul(_transpose(J), _adjugate(_transpose(M)))]
    g = _points(HN)
    e = sum(phase[c] * g[:, c] for c in range(d)) % q
    e = torch.polar(torch.ones_like(e, dtype=torch.float64), -2 * math.pi * e.double() / q)
    step = torch.tensor(N[i], device="cuda")  # N^T e_i
    slots, weights = [], []
    for t in range(p):
        h = g + t * step
        slots.append(_slots(HM, h))
        B, k = [], []
        for r in range(d):
            a = sum(K[r][c] * h[:, c] for c in range(d))
            k0 = -torch.div(2 * a + q, 2 * q, rounding_mode="floor")
            for_r, ks = [], []
            for o in (-1, 0, 1):
                s = (a + (k0 + o) * q).abs()
                if symbol == "dirichlet":
                    for_r.append((2 * s < q).double() + 0.5 * (2 * s == q).double())
                else:
                    for_r.append(((0.5 * (1 + 0.125) - s.double() / q) / 0.125).clamp(0, 1))
                ks.append((k0 + o) * v[r])
            B.append(for_r)
            k.append(ks)
        w = 0
        for combo in itertools.product(range(3), repeat=d):
            inside = sum(k[r][combo[r]] for r in range(d)) % p == 0
            w = w + inside * math.prod(B[r][combo[r]] for r in range(d))
        weights.append(w)
    return torch.stack(slots), torch.stack(weights), e, N


def _bands(w, e, c=None, d=None):
    """The unitary band system of a fibre, [batch, p, n]: the analysis of the
    members c or the synthesis of the bands d."""
    p = w.shape[0]
    V = w.sqrt()
    V[0] += 1
    ej = torch.stack([e ** j for j in range(p)])
    x = c if c is not None else ej * d
    x = 2 * V * ((V * x).sum(1) / (V * V).sum(0)).unsqueeze(1) - x
    return ej.conj() * x if c is not None else x


def _split(M, J, symbol, c):
    slots, w, e, N = _fibres(M, J, symbol)
    c = c.to(torch.complex128)[:, slots]
    if symbol == "dirichlet":
        return _bands(w, e, c=c), N
    A = math.sqrt(2) * w
    return torch.stack([A[0] * c[:, 0] + A[1] * c[:, 1], e.conj() * (A[1] * c[:, 0] - A[0] * c[:, 1])], 1) / math.sqrt(2), N


def _merge(M, J, symbol, parts, adjoint):
    """parts [batch, 2, n] back to the coefficients: the inverse or the adjoint of the split."""
    slots, w, e, _ = _fibres(M, J, symbol)
    A = (2 * w).sqrt() if symbol == "dirichlet" else math.sqrt(2) * w
    scale = 1 / math.sqrt(2) if adjoint else math.sqrt(2) / (A * A).sum(0)
    a, b = parts[:, 0], e * parts[:, 1]
    out = torch.empty((parts.shape[0], slots.numel()), dtype=torch.complex128, device=parts.device)
    out[:, slots[0]] = scale * (A[0] * a + A[1] * b)
    out[:, slots[1]] = scale * (A[1] * a - A[0] * b)
    return out


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "mix":
        coeffs, scaling, wavelet, off = [], [], [], 0
        for M, J in zip(*_mix(case)):
            m = abs(_det(M))
            c = _transform(M, x[0][off:off + m].unsqueeze(0))
            off += m
            parts, _ = _split(M, J, "dirichlet", c)
            coeffs.append(c[0])
            scaling.append(parts[0, 0])
            wavelet.append(parts[0, 1:].reshape(-1))
        return [torch.cat(coeffs), torch.cat(scaling), torch.cat(wavelet)]
    M = _matrix(case["matrix"])
    if kind == "transform":
        return [_transform(M, x[0]), x[0].to(torch.complex128)]
    if kind == "gradient":
        return [_transform(M, x[0]), _transform(M, x[1], inverse=True)]
    if kind == "bands":
        parts, _ = _split(M, _matrix(case["dilation"]), "dirichlet", x[0])
        return [parts.transpose(0, 1).contiguous(), x[0].to(torch.complex128)]
    Js, symbol = _dilations(case), case["symbol"]
    if kind == "reconstruct":
        Ms = [M]
        for J in Js:
            Ms.append([[v // _det(J) for v in row] for row in _mul(_adjugate(J), Ms[-1])])
        c = x[0].to(torch.complex128)
        for l in range(len(Js) - 1, -1, -1):
            c = _merge(Ms[l], Js[l], symbol, torch.stack([c, x[1 + l].to(torch.complex128)], 1), False)
        return [c]
    c, wavelets, N = x[0], [], M
    for J in Js:
        parts, N = _split(N, J, symbol, c)
        c = parts[:, 0]
        wavelets.append(parts[:, 1])
    if kind == "decompose":
        return [c, *wavelets]
    grad = _merge(M, Js[0], symbol, torch.stack([x[1], x[2]], 1).to(torch.complex128), True)
    return [c, *wavelets, grad]
