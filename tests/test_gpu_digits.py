"""Large FP64 GETTs as exact digits on the tensor cores (FP32: by SIMT): exact on
integers, within the stated bound of |A||B| on uniform entries (and closer than
one rounding per term), one panel of B and several, and what the digits leave
to the SIMT chains bit for bit: single results and patches of C where large
terms cancel, tiles with wide ranges and zeros along K, infinities and NaN,
exponents near the ends."""
import numpy as np
import pytest

from paper_1409_8608_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NP = {"f64": np.float64, "f32": np.float32}
U = {"f64": 2.0 ** -53, "f32": 2.0 ** -24}
# M, N, K large enough for the digits to be the faster estimate
SIZES = {"f64": [(300, 4000, 257), (129, 9001, 130)], "f32": [(700, 16001, 301), (513, 30000, 256)]}


@pytest.fixture(scope="module")
def tcmod():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1409_8608_gb300 import tc
    tc.load()
    return tc


def execute(tc, dtype, A, B, C0=None, alpha=1.0, beta=0.0, spec="ab=ai,ib"):
    """A (M, K) and B (K, N) as the spec's dense operands; returns C (M, N)
    and the same product by SIMT (a plan whose strides give B a batch index
    of extent 1, which only the SIMT tiles take)."""
    M, K = A.shape
    N = B.shape[1]
    lay = {"ab=ai,ib": (A.T, B.T), "ab=ia,bi": (A, B)}[spec]  # reversed modes, C order
    dA, dB = (torch.from_numpy(np.ascontiguousarray(x)).cuda().reshape(-1) for x in lay)
    out = []
    for s, ext in ((spec, {"a": M, "b": N, "i": K}),
                   (spec.replace("=", "h=").replace(",", "h,") + "h", {"a": M, "b": N, "i": K, "h": 1})):
        plan = tc.Plan(s, [ext[c] for c in synth.index_order(s)], dtype=dtype)
        dC = torch.full((N, M), float("nan"), dtype=dA.dtype, device="cuda:0") if C0 is None else \
            torch.from_numpy(np.ascontiguousarray(C0.T)).cuda()
        plan.execute(dA, dB, dC, alpha=alpha, beta=beta)
        torch.cuda.synchronize()
        plan.device_status()
        plan.close()
        out.append(dC.cpu().numpy().T)
    return out


@pytest.mark.parametrize("spec", ["ab=ai,ib", "ab=ia,bi"])
@pytest.mark.parametrize("dtype,size", [(d, s) for d in SIZES for s in SIZES[d]])
def test_exact_on_integers(tcmod, dtype, size, spec):
    M, N, K = size
    rng = np.random.default_rng(5)
    top = 2 ** 22 if dtype == "f64" else 100  # sums below 2^53 and 2^24
    A, B = rng.integers(-top, top + 1, (M, K)), rng.integers(-top, top + 1, (K, N))
    A[3] = 0  # a row of zeros
    want = (torch.from_numpy(A).double().cuda() @ torch.from_numpy(B).double().cuda()).cpu().numpy()
    got, simt = execute(tcmod, dtype, A.astype(NP[dtype]), B.astype(NP[dtype]), spec=spec)
    assert np.array_equal(got, want) and np.array_equal(simt, want)
    C0 = rng.integers(-50, 50, (M, N)).astype(NP[dtype])
    got, _ = execute(tcmod, dtype, A.astype(NP[dtype]), B.astype(NP[dtype]), C0, 0.5, -2.0, spec=spec)
    assert np.array_equal(got, (0.5 * want - 2.0 * C0).astype(NP[dtype]))


@pytest.mark.parametrize("dtype,size", [("f64", s) for s in SIZES["f64"]])
def test_error_on_uniform(tcmod, dtype, size):
    M, N, K = size
    rng = np.random.default_rng(6)
    A, B = (rng.uniform(-1, 1, s).astype(NP[dtype]) for s in ((M, K), (K, N)))
    got, simt = execute(tcmod, dtype, A, B)
    i, j = rng.integers(0, M, 2000), rng.integers(0, N, 2000)
    terms = A[i].astype(np.longdouble) * B[:, j].T.astype(np.longdouble)
    want, scale = terms.sum(1), np.abs(terms).sum(1)
    err = np.abs(got[i, j] - want)
    # rounded once: half a unit in the last place, and the digits left out
    # (2^-59 of at most |x|, |y| < 1 per term)
    left = K * 2.0 ** -59
    assert np.all(err <= U[dtype] * np.abs(want) * 1.01 + left), float(np.max(err / scale))
    # and no further off than the chain of fused multiply-adds
    assert np.linalg.norm(err) <= np.linalg.norm(simt[i, j] - want)


@pytest.mark.parametrize("dtype", ["f64"])
def test_extreme_digits(tcmod, dtype):
    # every digit at its end: the level sums reach their bound
    M, N, K = SIZES[dtype][0]
    x = np.nextafter(NP[dtype](1), NP[dtype](0))
    for a, b in ((x, x), (-x, x), (x, NP[dtype](0.50390625)), (NP[dtype](-0.50196), x)):
        A, B = np.full((M, K), a, NP[dtype]), np.full((K, N), b, NP[dtype])
        got, _ = execute(tcmod, dtype, A, B)
        want = np.longdouble(a) * np.longdouble(b) * K
        left = K * 2.0 ** -59
        assert np.all(np.abs(got - want) <= U[dtype] * abs(want) * 1.01 + left)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_left_to_simt(tcmod, dtype):
    M, N, K = SIZES[dtype][0]
    rng = np.random.default_rng(7)
    A, B = (rng.uniform(0.5, 1, s).astype(NP[dtype]) for s in ((M, K), (K, N)))
    tiny, huge = (1e-310, 1e300) if dtype == "f64" else (1e-42, 1e37)
    A[5, 1], A[6, 2] = np.inf, np.nan
    B[3, 70] = -np.inf
    A[7] = tiny
    A[8, :] = huge
    A[280, : K // 2 + 9] = 0              # mostly zeros along K
    A[281] *= NP[dtype](2.0) ** -np.arange(K, dtype=NP[dtype])  # wide range along K
    B[:, N - 1] = 0
    B[0, N - 1] = 1
    got, simt = execute(tcmod, dtype, A, B)
    bad = np.zeros((M, N), bool)
    bad[[5, 6, 7, 8, 280, 281]] = True
    bad[:, [70, N - 1]] = True
    assert np.array_equal(got[bad], simt[bad], equal_nan=True)
    C0 = rng.uniform(-1, 1, (M, N)).astype(NP[dtype])
    got2, simt2 = execute(tcmod, dtype, A, B, C0, 0.5, -2.0)
    assert np.array_equal(got2[bad], simt2[bad], equal_nan=True)
    i, j = np.nonzero(~bad)
    pick = rng.integers(0, len(i), 2000)
    i, j = i[pick], j[pick]
    want = (A[i].astype(np.longdouble) * B[:, j].T.astype(np.longdouble)).sum(1)
    assert np.all(np.abs(got[i, j] - want) <= K * U[dtype] * np.abs(want))


@pytest.mark.parametrize("dtype,small", [("f32", 2.0 ** -26), ("f64", 2.0 ** -56)])
def test_large_terms_cancel(tcmod, dtype, small):
    # pairs of terms that cancel exactly, beside entries far below them: a
    # chain keeps the small terms to their last bit, K roundings at most
    M, N, K = SIZES[dtype][0][0], SIZES[dtype][0][1], 256
    rng = np.random.default_rng(9)
    A = np.empty((M, K), NP[dtype])
    A[:, 0:128:2], A[:, 1:128:2] = 1, -1
    A[:, 128:] = small * rng.uniform(0.5, 1, (M, 128))
    B = rng.uniform(0.5, 1, (K, N)).astype(NP[dtype])
    B[1:128:2] = B[0:128:2]
    got, _ = execute(tcmod, dtype, A, B)
    i, j = rng.integers(0, M, 2000), rng.integers(0, N, 2000)
    want = (A[i, 128:].astype(np.longdouble) * B[128:, j].T.astype(np.longdouble)).sum(1)
    assert np.all(np.abs(got[i, j] - want) <= K * U[dtype] * np.abs(want))


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (0.5, -2.0)])
@pytest.mark.parametrize("spec", ["ab=ai,ib", "ab=ia,bi"])
def test_small_results_by_the_chain(tcmod, spec, alpha, beta):
    """Results below 2^-10 of the scales of their row and column come from the
    chain bit for bit -- single ones, a row of a patch of 32 x 32, patches with
    more than an eighth of them --, all others within half a unit in the last
    place and K 2^-48.9 of the result."""
    M, N, K = 300, 4000, 258
    rng = np.random.default_rng(10)
    A, B = rng.uniform(-1, 1, (M, K)), rng.uniform(-1, 1, (K, N))
    for rows in (slice(32, 75), slice(200, 201)):
        A[rows, 0::2], A[rows, 1::2] = 1, -1
    B[1::2, 100:300] = B[0::2, 100:300]
    A[250] = 0
    C0 = rng.uniform(-1, 1, (M, N)) if beta else None
    got, simt = execute(tcmod, "f64", A, B, C0, alpha, beta, spec=spec)
    want = A @ B
    scale = np.exp2(np.frexp(np.abs(A).max(1))[1])[:, None] * np.exp2(np.frexp(np.abs(B).max(0))[1])
    v = np.abs(want) / scale
    few = v < 2.0 ** -10.1
    few[250] = False
    assert few[:32].sum() > 5 and few[32:75, 100:300].all() and few[200, 100:300].all()
    assert np.array_equal(got[few], simt[few])
    assert not np.array_equal(got, simt)  # the digits ran
    strong = v > 2.0 ** -9.9
    strong[32:96, 96:320] = False  # patches there are left as a whole
    i, j = np.nonzero(strong)
    pick = rng.integers(0, len(i), 3000)
    i, j = i[pick], j[pick]
    v = (A[i].astype(np.longdouble) * B[:, j].T.astype(np.longdouble)).sum(1)
    want = alpha * v + (beta * C0[i, j].astype(np.longdouble) if beta else 0)
    u = U["f64"] * 1.01
    bound = abs(alpha) * (K * 2.0 ** -48.9 + u) * np.abs(v) + u * np.abs(want)
    if beta:
        bound += u * np.abs(beta * C0[i, j])
    assert np.all(np.abs(got[i, j] - want) <= bound)


@pytest.mark.parametrize("alpha", [float("inf"), float("-inf"), float("nan"), 0.0, -0.0])
def test_special_alpha(tcmod, alpha):
    M, N, K = SIZES["f64"][0]
    rng = np.random.default_rng(11)
    A, B = rng.uniform(-1, 1, (M, K)), rng.uniform(-1, 1, (K, N))
    A[17], A[18] = np.abs(A[17]), 0
    B[:, 40] = np.abs(B[:, 40])
    got, simt = execute(tcmod, "f64", A, B, None, alpha, 0.0)
    assert np.array_equal(got, simt, equal_nan=True)
    assert np.array_equal(np.signbit(got), np.signbit(simt)) or np.isnan(simt).any()


def test_panels(tcmod):
    """Three panels of B, the last one ragged: exact on integers in all of them;
    with rows and columns that the digits refuse in the later ones, listed and
    digit tiles side by side."""
    M, N, K = 600, 64 * 484 + 17, 257
    rng = np.random.default_rng(12)
    A, B = rng.integers(-(2 ** 22), 2 ** 22, (M, K)), rng.integers(-(2 ** 22), 2 ** 22, (K, N))
    want = (torch.from_numpy(A).double().cuda() @ torch.from_numpy(B).double().cuda()).cpu().numpy()
    got, _ = execute(tcmod, "f64", A.astype(np.float64), B.astype(np.float64))
    assert np.array_equal(got, want)
    A, B = rng.uniform(-1, 1, (M, K)), rng.uniform(-1, 1, (K, N))
    A[530] *= 2.0 ** -np.arange(K)        # the third row tile: listed in every panel
    B[0, 16000] = np.inf                  # second panel
    B[:, 25000] = 1e300
    B[: K // 2 + 9, N - 1] = 0            # the last, ragged tile
    B[1:256:2, 30000:30040] = B[0:256:2, 30000:30040]  # third panel: results that cancel
    A[10, 0:256:2], A[10, 1:256:2], A[10, 256] = 1, -1, 2.0 ** -50
    listed = np.zeros((M, N), bool)
    listed[512:] = True
    for n in (16000, 25000, N - 1):
        listed[:, n // 64 * 64: n // 64 * 64 + 64] = True
    got, simt = execute(tcmod, "f64", A, B)
    assert np.array_equal(got[listed], simt[listed], equal_nan=True)
    assert np.array_equal(got[10, 30000:30040], simt[10, 30000:30040])
    for m0 in (0, 256):  # every other tile by the digits
        for n0 in range(0, N, 64):
            if not listed[m0, n0]:
                assert not np.array_equal(got[m0:m0 + 256, n0:n0 + 64], simt[m0:m0 + 256, n0:n0 + 64]), (m0, n0)
    i, j = np.nonzero(~listed)
    pick = rng.integers(0, len(i), 4000)
    i, j = i[pick], j[pick]
    terms = A[i].astype(np.longdouble) * B[:, j].T.astype(np.longdouble)
    v = terms.sum(1)
    small = np.abs(v) < 2.0 ** -9  # some of these by the chain
    bound = (K * 2.0 ** -48.9 + 1.01 * U["f64"]) * np.abs(v) + np.where(small, K * U["f64"] * np.abs(terms).sum(1), 0)
    assert np.all(np.abs(got[i, j] - v) <= bound)


def test_long_k(tcmod):
    # few tiles of B to a panel, many accumulations to a tile
    M, N, K = 500, 600, 10001
    gen = torch.Generator().manual_seed(13)
    A, B = (torch.randint(-(2 ** 15), 2 ** 15, s, generator=gen).double() for s in ((M, K), (K, N)))
    want = (A.cuda() @ B.cuda()).cpu().numpy()  # exact: sums below 2^44
    got, _ = execute(tcmod, "f64", A.numpy(), B.numpy())
    assert np.array_equal(got, want)
    A, B = (torch.empty(s, dtype=torch.float64).uniform_(-1, 1, generator=gen) for s in ((M, K), (K, N)))
    got, simt = execute(tcmod, "f64", A.numpy(), B.numpy())
    assert not np.array_equal(got, simt)
    i, j = torch.arange(0, 500, 5), torch.arange(0, 600, 6)
    terms = A[i].numpy().astype(np.longdouble) * B[:, j].T.numpy().astype(np.longdouble)
    v = terms.sum(1)
    assert np.all(np.abs(got[i, j] - v) <= 1.01 * U["f64"] * np.abs(v) + K * 2.0 ** -58.9)
    assert np.linalg.norm(got[i, j] - v) < np.linalg.norm(simt[i, j] - v)


def test_marks_in_groups(tcmod):
    """More results than marks are kept for at a time: the chain runs between
    the panels too (beta = 1, so results left to it would keep the old C)."""
    M, N, K = 33000, 8300, 40
    gen = torch.Generator(device="cuda").manual_seed(14)
    A, B, C = (torch.randint(-(2 ** 20), 2 ** 20, (n,), device="cuda", generator=gen).double()
               for n in (M * K, K * N, M * N))
    want = C.view(N, M) + B.view(N, K) @ A.view(K, M)  # exact: sums below 2^46
    plan = tcmod.Plan("ab=ai,ib", [M, N, K], dtype="f64")
    plan.execute(A, B, C, alpha=1.0, beta=1.0)
    torch.cuda.synchronize()
    plan.device_status()
    plan.close()
    assert torch.equal(C.view(N, M), want)


def test_benchmark_counts_every_launch(tcmod):
    from bench import kernels_of
    stream = torch.cuda.Stream()
    for N, panels in ((4000, 1), (64 * 484 + 17, 3)):
        M, K = 600, 257
        A, B, C = (torch.ones(n, dtype=torch.float64, device="cuda") for n in (M * K, K * N, M * N))
        torch.cuda.synchronize()
        plan = tcmod.Plan("ab=ai,ib", [M, N, K], dtype="f64")
        plan.execute(A, B, C, stream=stream)
        torch.cuda.synchronize()
        # a pre-pass and a GETT per panel, and one launch for what they leave
        assert kernels_of(lambda: plan.execute(A, B, C, stream=stream), stream) == 2 * panels + 1
        plan.close()


@pytest.mark.parametrize("size", [(2148, 218, 2150), (300, 4000, 257)])
def test_refused_tiles_spread_over_the_sms(tcmod, size):
    # everything left to the chain: little more than the SIMT GETT takes
    M, N, K = size
    gen = torch.Generator(device="cuda").manual_seed(15)
    A, B = (torch.empty(n, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=gen) for n in (M * K, K * N))
    A.view(K, M)[: K // 2 + 9] = 0
    C = torch.empty(M * N, dtype=torch.float64, device="cuda")
    st, times, out = torch.cuda.current_stream(), [], []
    for mode in (1, 0):
        plan = tcmod.Plan("ab=ai,ib", [M, N, K], dtype="f64")
        plan.set_gett_pack(mode)
        ts = []
        for _ in range(7):
            e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
            e0.record(st)
            plan.execute(A, B, C, stream=st)
            e1.record(st)
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        plan.close()
        times.append(sorted(ts)[3])
        out.append(C.clone())
    assert torch.equal(out[0], out[1])
    assert times[0] < 1.5 * times[1], times
