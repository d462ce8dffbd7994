"""The GETT with both inputs pre-converted, at the edges of its tiles: rows and
columns one past and one short of a tile, K below and one past a stage, free
indices of B that do not chain in C, and the pair and lone-CTA forms -- exact
on integer inputs (every product and sum is exact in every form)."""
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


CASES = [
    ("ab=ai,ib", {"a": 1, "b": 1, "i": 1}),
    ("ab=ai,ib", {"a": 129, "b": 33, "i": 7}),
    ("ab=ia,bi", {"a": 257, "b": 255, "i": 65}),
    ("ab=aij,jib", {"a": 1025, "b": 1040, "i": 5, "j": 13}),     # default route: M, N >= 1024
    ("ab=aij,jib", {"a": 300, "b": 700, "i": 11, "j": 29}),      # K = 319: compensated in the split forms
    ("bac=ai,ibc", {"a": 130, "b": 100, "c": 7, "i": 33}),       # B's free indices do not chain in C
    ("abc=iaj,jbic", {"a": 127, "b": 19, "c": 31, "i": 9, "j": 7}),
]


@pytest.mark.parametrize("dtype", ["bf16x3", "tf32x3", "tf32", "bf16", "f16", "e4m3"])
@pytest.mark.parametrize("spec,e", CASES)
def test_packed_exact_on_integers(tcmod, spec, e, dtype):
    ext = [e[c] for c in synth.index_order(spec)]
    A, B, C0 = synth.integer_operands(spec, ext, seed=3, with_c=True)
    S = oc.contract(spec, ext, A, B, threads=4)
    in_t = {"bf16": torch.bfloat16, "f16": torch.float16}.get(dtype, torch.float32)
    dA, dB = (torch.from_numpy(x).to(in_t).cuda() for x in (A, B))
    for pair in (0, 1):
        for alpha, beta in ((1.0, 0.0), (2.0, -0.5)):
            plan = tcmod.Plan(spec, ext, dtype=dtype)
            plan.set_gett_pack(3)
            plan.set_gett_pair(pair)
            dC = torch.from_numpy(C0).float().cuda() if beta else \
                torch.full((S.size,), float("nan"), dtype=torch.float32, device="cuda:0")
            plan.execute(dA, dB, dC, alpha=alpha, beta=beta)
            torch.cuda.synchronize()
            plan.device_status()
            plan.close()
            assert np.array_equal(dC.double().cpu().numpy(), alpha * S + beta * C0), (pair, alpha, beta)
