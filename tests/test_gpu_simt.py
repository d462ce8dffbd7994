"""The SIMT tile shapes (FP64 64 / 32 / 16, FP32 128 / 64 / 32 rows and
columns, chosen by how many tiles a result has): exact on integer inputs,
whose products and sums are exact in FP32, with edges one past a tile, K one
past a stage and below one, both copy mappings, alpha through registers and
beta read from C."""
import numpy as np
import pytest

from oracle import contraction as oc
from paper_1409_8608_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def tcmod():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_1409_8608_gb300 import tc
    tc.load()
    return tc


# (M, N): enough tiles of the largest shape, of the second, and few
SIZES = {"f64": [(129, 30000), (129, 9000), (17, 40)], "f32": [(257, 14000), (129, 6500), (33, 70)]}


@pytest.mark.parametrize("spec", ["ab=ai,ib", "ab=ia,bi", "ab=ia,ib", "ba=ai,bi"])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("size", [0, 1, 2])
@pytest.mark.parametrize("K", [3, 17])
def test_tile_shapes_exact_on_integers(tcmod, spec, dtype, size, K):
    M, N = SIZES[dtype][size]
    e = {"a": M, "b": N, "i": K}
    ext = [e[c] for c in synth.index_order(spec)]
    A, B, C0 = synth.integer_operands(spec, ext, seed=K, with_c=True)
    S = oc.contract(spec, ext, A, B, threads=4)
    np_t = {"f64": np.float64, "f32": np.float32}[dtype]
    dA, dB = (torch.from_numpy(x.astype(np_t)).cuda() for x in (A, B))
    for alpha, beta in ((1.0, 0.0), (1.0, 1.0), (-2.0, 0.5)):
        plan = tcmod.Plan(spec, ext, dtype=dtype)
        dC = torch.from_numpy((2 * C0).astype(np_t)).cuda() if beta else \
            torch.full((M * N,), float("nan"), dtype=dA.dtype, device="cuda:0")
        plan.execute(dA, dB, dC, alpha=alpha, beta=beta)
        torch.cuda.synchronize()
        plan.close()
        assert np.array_equal(dC.double().cpu().numpy(), alpha * S + beta * 2 * C0), (alpha, beta)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("size", [(129, 300, 37), (40, 1000, 7), (1, 500, 20), (500, 1, 20)])
def test_order_of_c_does_not_change_the_sums(tcmod, dtype, size):
    """Tiles store C along its fastest index, A's or B's: the same bits either
    way, alpha multiplying A's entries (uniform values, alpha and beta inexact)."""
    M, N, K = size
    np_t = {"f64": np.float64, "f32": np.float32}[dtype]
    rng = np.random.default_rng(1)
    A, B, C0 = (torch.from_numpy(rng.uniform(-1, 1, n).astype(np_t)).cuda() for n in (M * K, K * N, M * N))
    out = []
    for spec in ("ab=ai,ib", "ba=ai,ib"):
        e = {"a": M, "b": N, "i": K}
        plan = tcmod.Plan(spec, [e[c] for c in synth.index_order(spec)], dtype=dtype)
        first = spec[0] == "a"
        gemm = next(a["id"] for a in plan.algorithms() if a["kernel"] == "gemm" and not a["loops"])
        for alg in (0, gemm):
            plan.select(alg)
            C = (C0.view(N, M) if first else C0.view(N, M).T.contiguous()).clone().reshape(-1)
            plan.execute(A, B, C, alpha=0.7, beta=0.3)
            torch.cuda.synchronize()
            out.append(C.view(N, M) if first else C.view(M, N).T)
        plan.close()
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])
