"""Calls that a rule sends to a newer kernel, against the general one: the
tensor-core GETT on images of both inputs by default, the FP64 / FP32 GETT on
digits, loop nests with short contracted indices, FP64 batches whose tiles are
chosen by padding -- over orders and strides of the modes, at the rules' edges,
and inside a stream capture before and after the scratch exists."""
import numpy as np
import pytest

from oracle import contraction as oc
from paper_1409_8608_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NP = {"f64": np.float64, "f32": np.float32}


@pytest.fixture(scope="module")
def tcmod():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1409_8608_gb300 import tc
    tc.load()
    return tc


def padded(spec, e, pad):
    """Strides (C, A, B) of operands with `pad` elements of gap after the
    first mode and after the second, their lengths, and the strides as a list."""
    lay, length = [], []
    for modes in oc.parse_spec(spec):
        st, s = [], 1
        for n, c in enumerate(modes):
            st.append(s)
            s = s * e[c] + (pad if n < 2 else 0)
        lay.append(st)
        length.append(1 + sum((e[c] - 1) * x for c, x in zip(modes, st)))
    return lay, length, [x for st in lay for x in st]


IMAGES = [
    ("ab=ia,bi", {"a": 65, "b": 70, "i": 47}),      # below, at and past the rule's edges along K
    ("ab=ia,bi", {"a": 65, "b": 70, "i": 48}),
    ("ab=ai,ib", {"a": 129, "b": 257, "i": 127}),
    ("ab=ai,ib", {"a": 129, "b": 257, "i": 128}),
    ("bca=iaj,jbic", {"a": 70, "b": 33, "c": 9, "i": 20, "j": 8}),
    ("cab=ija,bjic", {"a": 131, "b": 5, "c": 30, "i": 13, "j": 11}),
    ("dacb=aijd,cjbi", {"a": 17, "b": 6, "c": 40, "d": 9, "i": 30, "j": 9}),  # K = 270: past a chunk
    ("abc=ai,ibc", {"a": 74, "b": 371, "c": 50, "i": 52}),   # one tile of M, many columns
    ("abc=ai,ibc", {"a": 74, "b": 371, "c": 50, "i": 128}),
    ("ab=ai,ib", {"a": 4200, "b": 4100, "i": 50}),  # a result of more than 2^24
]


@pytest.mark.parametrize("dtype", ["bf16x3", "tf32x3", "tf32", "bf16", "f16", "e4m3"])
@pytest.mark.parametrize("pad", [0, 3])
@pytest.mark.parametrize("spec,e", IMAGES)
def test_images_by_default(tcmod, spec, e, pad, dtype):
    ext = [e[c] for c in synth.index_order(spec)]
    lay, length, strides = padded(spec, e, pad)
    rng = np.random.default_rng(4)
    C0, A, B = (rng.integers(-8, 9, n).astype(np.float64) for n in length)
    in_t = {"bf16": torch.bfloat16, "f16": torch.float16}.get(dtype, torch.float32)
    dA, dB = (torch.from_numpy(x).to(in_t).cuda() for x in (A, B))
    out = []
    for mode in (1, 0):
        plan = tcmod.Plan(spec, ext, strides=strides, dtype=dtype)
        plan.set_gett_pack(mode)
        dC = torch.from_numpy(C0).float().cuda()
        plan.execute(dA, dB, dC, alpha=2.0, beta=-0.5)
        torch.cuda.synchronize()
        plan.device_status()
        plan.close()
        out.append(dC.double().cpu().numpy())
    assert np.array_equal(out[0], out[1])  # products and sums are exact in every form
    if e["a"] * e["b"] < 1 << 22:
        assert np.array_equal(out[0], oc.contract(spec, ext, A, B, C=C0.copy(), alpha=2.0, beta=-0.5, strides=strides))


def test_image_panels(tcmod):
    """Images of B past 512 MiB: two panels, the second one ragged, against the
    inputs as they are; integers, so exact in every form."""
    M, N, K = 200, 600011, 160
    gen = torch.Generator(device="cuda").manual_seed(3)
    A, B = (torch.randint(-8, 9, (n,), device="cuda", generator=gen).float() for n in (M * K, K * N))
    out = []
    for mode in (1, 0):
        plan = tcmod.Plan("ab=ai,ib", [M, N, K], dtype="bf16x3")
        plan.set_gett_pack(mode)
        C = torch.full((M * N,), float("nan"), device="cuda")
        free = torch.cuda.mem_get_info()[0]
        plan.execute(A, B, C)
        torch.cuda.synchronize()
        scratch = free - torch.cuda.mem_get_info()[0]
        assert (scratch > 256 << 20) == (mode == 1), scratch  # the images ran
        plan.device_status()
        plan.close()
        out.append(C)
    assert torch.equal(out[0], out[1])
    want = B.view(N, K).double() @ A.view(K, M).double()
    assert torch.equal(out[0].double().view(N, M), want)


DIGITS = [
    ("cab=iaj,jbic", {"a": 300, "b": 40, "c": 100, "i": 17, "j": 16}),
    ("bac=jai,cibj", {"a": 300, "b": 80, "c": 60, "i": 30, "j": 9}),
    ("adbc=dija,bcji", {"a": 20, "b": 100, "c": 50, "d": 15, "i": 16, "j": 17}),
]


def digit_operands(dtype, spec, e, pad, integers):
    lay, length, strides = padded(spec, e, pad)
    rng = np.random.default_rng(8)
    if integers:
        top = 2 ** 20 if dtype == "f64" else 100
        vals = [rng.integers(-top, top + 1, n).astype(NP[dtype]) for n in length]
    else:
        vals = [rng.uniform(-1, 1, n).astype(NP[dtype]) for n in length]
    C0, A, B = (torch.from_numpy(v).cuda() for v in vals)
    views = [torch.as_strided(x, [e[c] for c in m], st)
             for x, m, st in zip((C0, A, B), oc.parse_spec(spec), lay)]
    return strides, C0, A, B, views


def simt_plan(tc, spec, e, strides, dtype):
    """The same contraction with a batch index of extent 1: SIMT tiles."""
    c, a, b = oc.parse_spec(spec)
    s = f"{''.join(c)}h={''.join(a)}h,{''.join(b)}h"
    x = dict(e, h=1)
    st = strides[:len(c)] + [1 << 40] + strides[len(c):len(c) + len(a)] + [1] + strides[len(c) + len(a):] + [1]
    return tc.Plan(s, [x[i] for i in synth.index_order(s)], strides=st, dtype=dtype)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("pad", [0, 5])
@pytest.mark.parametrize("spec,e", DIGITS)
def test_digits_layouts(tcmod, spec, e, pad, dtype):
    if dtype == "f32":
        e = dict(e, a=e["a"] * 3, c=e["c"] * 4)
    strides, C0, A, B, (vc, va, vb) = digit_operands(dtype, spec, e, pad, True)
    plan = tcmod.Plan(spec, [e[c] for c in synth.index_order(spec)], strides=strides, dtype=dtype)
    c, a, b = ("".join(m) for m in oc.parse_spec(spec))
    want = C0.double().clone()
    view = torch.as_strided(want, vc.shape, vc.stride())
    view.copy_(0.5 * torch.einsum(f"{a},{b}->{c}", va.double(), vb.double()) - 2 * view)  # exact: sums below 2^53
    plan.execute(A, B, C0, alpha=0.5, beta=-2.0)  # and the gaps in C stay as they were
    torch.cuda.synchronize()
    plan.device_status()
    plan.close()
    assert torch.equal(C0.double(), want.to(C0.dtype).double())


@pytest.mark.parametrize("dtype", ["f64"])
def test_digits_and_capture(tcmod, dtype):
    """A first execute inside a capture takes no scratch: the chains run.
    After one outside, the digits run, also in a capture."""
    spec, e = DIGITS[0]
    strides, C0, A, B, _ = digit_operands(dtype, spec, e, 0, False)
    ext = [e[c] for c in synth.index_order(spec)]
    simt = simt_plan(tcmod, spec, e, strides, dtype)
    want = torch.zeros_like(C0)
    simt.execute(A, B, want)
    torch.cuda.synchronize()
    simt.close()
    plan = tcmod.Plan(spec, ext, strides=strides, dtype=dtype)
    small = next(a["id"] for a in plan.algorithms() if a["kernel"] == "gemm")
    stream = torch.cuda.Stream()

    def captured():
        g = torch.cuda.CUDAGraph()
        out = torch.zeros_like(C0)
        with torch.cuda.graph(g, stream=stream):
            plan.execute(A, B, out, stream=stream)
        return g, out

    plan.select(small)
    plan.execute(A, B, C0, stream=stream)  # the plan's status word, but no scratch
    torch.cuda.synchronize()
    plan.select(0)
    before, out1 = captured()
    before.replay()
    torch.cuda.synchronize()
    assert torch.equal(out1, want)
    digits = torch.zeros_like(C0)
    plan.execute(A, B, digits, stream=stream)
    torch.cuda.synchronize()
    assert not torch.equal(digits, want)
    K = e["i"] * e["j"]
    u = 2.0 ** -53
    assert float((digits.double() - want.double()).abs().max()) <= (K + 2) * u * K  # |x|, |y| < 1
    after, out2 = captured()
    for _ in range(2):
        out2.zero_()
        after.replay()
        torch.cuda.synchronize()
        assert torch.equal(out2, digits)
    before.replay()
    torch.cuda.synchronize()
    assert torch.equal(out1, want)
    plan.device_status()
    plan.close()


def test_pack_mode_0_keeps_the_chain(tcmod):
    """FP64 with tc_plan_set_gett_pack(0): the SIMT tiles' bits, no scratch."""
    spec, e = DIGITS[0]
    strides, C0, A, B, _ = digit_operands("f64", spec, e, 0, False)
    simt = simt_plan(tcmod, spec, e, strides, "f64")
    want = torch.zeros_like(C0)
    simt.execute(A, B, want)
    simt.close()
    plan = tcmod.Plan(spec, [e[c] for c in synth.index_order(spec)], strides=strides, dtype="f64")
    plan.set_gett_pack(0)
    plan.execute(A, B, C0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert torch.equal(C0, want)
    plan.set_gett_pack(1)
    plan.execute(A, B, C0)
    torch.cuda.synchronize()
    assert not torch.equal(C0, want) and torch.cuda.mem_get_info()[0] < free
    plan.set_gett_pack(0)
    plan.execute(A, B, C0)
    torch.cuda.synchronize()
    assert torch.equal(C0, want)
    plan.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("K", [1, 3, 4, 5, 31, 32, 33])
@pytest.mark.parametrize("a", [97, 100])  # either side of 64 outputs per SM
def test_nests_short_contracted(tcmod, a, K, dtype):
    spec = "abc=ibj,jaic"
    e = {"a": a, "b": 50, "c": 2, "i": K, "j": 2}
    ext = [e[c] for c in synth.index_order(spec)]
    A, B, C0 = synth.integer_operands(spec, ext, seed=K, with_c=True)
    S = oc.contract(spec, ext, A, B, threads=4)
    dA, dB, dC0 = (torch.from_numpy(x.astype(NP[dtype])).cuda() for x in (A, B, C0))
    plan = tcmod.Plan(spec, ext, dtype=dtype)
    seen = set()
    for alg in plan.algorithms():
        key = (alg["kernel"], alg["name"][-8:])
        if alg["kernel"] == "gett" or key in seen:
            continue
        seen.add(key)
        plan.select(alg["id"])
        dC = dC0.clone()
        plan.execute(dA, dB, dC, alpha=2.0, beta=-1.0)
        torch.cuda.synchronize()
        assert np.array_equal(dC.double().cpu().numpy(), 2 * S - C0), alg["name"]
    plan.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("K", [2, 4, 5, 11, 16, 17, 31])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (0.7, 1.0), (1.0, -0.3)])
def test_nests_sum_in_the_same_order(tcmod, alpha, beta, K, dtype):
    """Few outputs go to groups of lanes, a hundred per SM to a thread each:
    the same sums, so a slice of the larger contraction has the same bits."""
    spec = "ab=ija,ijb"
    N = 128
    rng = np.random.default_rng(K)
    A, B, C0 = (torch.from_numpy(rng.uniform(-1, 1, n).astype(NP[dtype])).cuda()
                for n in (K * 9 * N, K * 9 * N, N * N))
    out = []
    for b in (N, 64):  # 16384 outputs, and 8192: fewer than 64 per SM
        plan = tcmod.Plan(spec, [N, b, K, 9], dtype=dtype)
        ids = {}
        for alg in plan.algorithms():
            if alg["kernel"] not in ("gemm", "gett") and alg["n_phases"] == 1:
                ids[alg["name"]] = alg["id"]
        res = {}
        for name, i in ids.items():
            plan.select(i)
            dC = C0[:N * b].clone()
            plan.execute(A, B[:K * 9 * b], dC, alpha=alpha, beta=beta)
            torch.cuda.synchronize()
            res[name] = dC.cpu().numpy()
        plan.close()
        out.append(res)
    assert out[0].keys() == out[1].keys() and len(out[0]) >= 2
    for name, c in out[1].items():
        assert np.array_equal(out[0][name][:N * 64], c), name


@pytest.mark.parametrize("K", [1, 15, 17])
def test_batch_f64_tiles(tcmod, K):
    spec = "abc=ai,ibc"
    sizes = [1, 7, 8, 9, 31, 33, 64, 65, 127, 129]
    rows = [[{"a": m, "b": n, "c": 3, "i": K}[c] for c in synth.index_order(spec)] for m in sizes for n in sizes]
    host = [synth.integer_operands(spec, r, seed=q) for q, r in enumerate(rows)]
    As, Bs = ([torch.from_numpy(h[o]).cuda() for h in host] for o in (0, 1))
    Cs = [torch.full((synth.dense_sizes(spec, r)[0],), float("nan"), dtype=torch.float64, device="cuda") for r in rows]
    batch = tcmod.Batch(spec, rows, "f64")
    batch.set_operands(As, Bs, Cs)
    batch.execute()
    torch.cuda.synchronize()
    for r, h, C in zip(rows, host, Cs):
        assert np.array_equal(C.cpu().numpy(), oc.contract(spec, r, h[0], h[1])), r
    batch.close()
