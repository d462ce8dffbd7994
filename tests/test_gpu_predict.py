"""GPU checks of the predictor (Section 3 on the device), the ranking and
the autotuner.  Timings have no oracle: these tests check that every
prediction is a positive time, that the ranking agrees with measurement
(rank correlation), that selection picks the smallest prediction, and that
the tuner and its cache behave."""
import numpy as np
import pytest

from paper_1409_8608_gb300 import ranking

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


def test_rank_statistics_helpers():
    assert ranking.spearman([1, 2, 3, 4], [10, 20, 30, 40]) == pytest.approx(1.0)
    assert ranking.spearman([1, 2, 3, 4], [4, 3, 2, 1]) == pytest.approx(-1.0)
    assert ranking.kendall([1, 2, 3], [1, 3, 2]) == pytest.approx(1 / 3)


def test_predictions_are_positive_and_selection_uses_them(tcmod):
    plan = tcmod.Plan("abc=ai,ibc", [64, 64, 64, 8])
    pred = plan.predict()  # scratch operands
    assert len(pred) == 37 and all(p > 0 for p in pred)
    best = plan.select_best()
    assert best == int(np.argmin(pred)) and plan.selected == best
    plan.close()


def test_small_plain_workload_ranking(tcmod):
    # the plain small workload (a=b=c=64, i=8, FP64): all 37 algorithms
    r = ranking.study("abc=ai,ibc", [64, 64, 64, 8], "f64", reps=5)
    assert len(r["algorithms"]) == 37
    assert r["spearman"] > 0.6, r
    assert r["prediction_seconds"] > 0


def test_permuted_workload_ranking(tcmod):
    r = ranking.study("abc=iaj,jbic", [96, 96, 96, 16, 16], "f64", reps=3)
    assert len(r["algorithms"]) == 177
    assert r["spearman"] > 0.6, {k: v for k, v in r.items() if k != "algorithms"}


@pytest.mark.parametrize("dtype,ext", [("f64", [2048, 30000, 512]), ("bf16x3", [2048, 60000, 512]),
                                       ("f32", [700, 16001, 301])])
def test_gett_prediction_scales_what_shrinks(tcmod, dtype, ext):
    """The GETT's probe cuts the columns, not the pre-pass over A nor the
    launches: prediction within a fifth of the time of the whole."""
    plan = tcmod.Plan("ab=ai,ib", ext, dtype=dtype)
    dt = torch.float64 if dtype == "f64" else torch.float32
    M, N, K = ext
    gen = torch.Generator(device="cuda").manual_seed(0)
    A, B = (torch.empty(n, dtype=dt, device="cuda").uniform_(-1, 1, generator=gen) for n in (M * K, K * N))
    C = torch.empty(M * N, dtype=dt, device="cuda")
    st = torch.cuda.current_stream()
    times = []
    for _ in range(12):
        e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
        e0.record(st)
        plan.execute(A, B, C, stream=st)
        e1.record(st)
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1) * 1e-3)
    want = sorted(times)[5]
    got = plan.predict([0])[0]
    plan.close()
    assert 0.8 * want < got < 1.2 * want, (got, want)


def test_prediction_without_operands_has_entries(tcmod):
    """Scratch operands hold uniform entries, not zeros, which the digits of an
    FP64 GETT never leave to the chain: the prediction is that on uniform ones."""
    plan = tcmod.Plan("ab=ai,ib", [300, 4000, 257], dtype="f64")
    gen = torch.Generator(device="cuda").manual_seed(0)
    A, B = (torch.empty(n, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=gen)
            for n in (300 * 257, 257 * 4000))
    C = torch.empty(300 * 4000, dtype=torch.float64, device="cuda")
    zero = plan.predict([0], torch.zeros_like(A), torch.zeros_like(B), C)[0]
    uniform = plan.predict([0], A, B, C)[0]
    own = plan.predict([0])[0]
    plan.close()
    assert zero < 0.95 * uniform and abs(own - uniform) < abs(own - zero), (zero, uniform, own)


def test_tensor_dtype_ranks_gemm_nests_and_gett(tcmod):
    # at tensor-core dtypes the gemm nests and the GETT are predicted (the
    # other kernels cannot run there), and the best prediction is one of them
    plan = tcmod.Plan("abc=iaj,jbic", [256, 256, 8, 16, 16], dtype="bf16x3")
    algs = plan.algorithms()
    gemm_ids = [a["id"] for a in algs if a["kernel"] == "gemm"]
    other = next(a["id"] for a in algs if a["kernel"] == "gemv")
    pred = plan.predict([0, other] + gemm_ids)
    assert pred[0] > 0 and pred[1] < 0 and all(t > 0 for t in pred[2:])
    best = plan.select_best()
    assert best in [0] + gemm_ids
    plan.close()


def test_autotune_and_cache(tcmod, tmp_path):
    spec, ext = "abc=iaj,jbic", [256, 512, 4, 16, 16]
    plan = tcmod.Plan(spec, ext, dtype="bf16x3")
    width, tma = plan.autotune()
    assert width in (128, 256) and tma in (0, 1)
    path = tmp_path / "tune.jsonl"
    tcmod.tc_tuning_cache_save(path)
    text = path.read_text()
    assert "gett_tile" in text and spec in text
    tcmod.tc_tuning_cache_load(path)
    plan2 = tcmod.Plan(spec, ext, dtype="bf16x3")
    assert plan2.autotune() == (width, tma)  # answered from the cache
    plan.close()
    plan2.close()


def test_autotuned_is_no_slower_than_the_default(tcmod):
    # 16-bit inputs, both as images by default: among the candidates too
    spec, ext = "ab=aij,jib", [700, 900, 16, 40]
    M, N, K = 700, 900, 640
    A, B = (torch.ones(n, dtype=torch.bfloat16, device="cuda") for n in (M * K, K * N))
    C = torch.empty(M * N, device="cuda")
    st = torch.cuda.current_stream()

    def time(plan):
        ts = []
        for _ in range(20):
            e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
            e0.record(st)
            plan.execute(A, B, C, stream=st)
            e1.record(st)
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        return sorted(ts)[5]

    plan = tcmod.Plan(spec, ext, dtype="bf16")
    default = time(plan)
    plan.autotune()
    tuned = time(plan)
    plan.close()
    assert tuned < 1.3 * default, (tuned, default)
