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
