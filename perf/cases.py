"""What users of the contraction library run, as cases that can be timed and
compared: single contractions through ``tc.Plan``, batches through
``tc.Batch`` and request mixes through ``tc.Server``.

A case is a dict of plain values.  ``kind`` "contract": one
``Plan.execute`` of ``spec`` over device operands (``algorithm`` names a loop
nest, "gett" the fused kernel), alpha and beta given; with beta != 0 a pass
first puts the starting values back into C, as a program does that adds a
contraction to a fresh copy of a right-hand side.  "batch": one
``Batch.execute`` over ``count`` problems.  "serving": ``requests`` requests
submitted at once to a server and waited for, host buffers in and out.
``shapes`` seeds the sizes of a batch or a request mix.
"""
import math
import random

import numpy as np
import torch

from paper_1409_8608_gb300 import tc

DEVICE = "cuda:0"
IN_TYPES = {"f64": torch.float64, "f32": torch.float32, "tf32": torch.float32, "bf16x3": torch.float32,
            "tf32x3": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
SERVING_SPECS = ("abc=ai,ibc", "abc=iaj,jbic", "ab=aij,jib")
SERVING_DTYPES = ("f64", "f32", "f32", "bf16x3", "bf16x3")
SERVING_MAX_C = 1 << 24  # elements of one request's result


def _contract(name, spec, extents, dtype, algorithm="gett", alpha=1.0, beta=0.0, values="uniform"):
    case = {"kind": "contract", "spec": spec, "extents": ",".join(str(e) for e in extents), "dtype": dtype,
            "algorithm": algorithm, "alpha": alpha, "beta": beta, "values": values}
    return {"name": name, **case} if name else case


def listed():
    return [
        # the paper's worked size in its own precision: one small call, where
        # launch and host time are all there is
        _contract("plain_f64_64", "abc=ai,ibc", (64, 64, 64, 8), "f64"),
        # the headline contraction (both inputs permuted against C) in the
        # paper's precision and in the precisions a user trades down to
        _contract("permuted_f64_512", "abc=iaj,jbic", (512, 512, 512, 16, 16), "f64"),
        _contract("permuted_f32_512", "abc=iaj,jbic", (512, 512, 512, 16, 16), "f32"),
        _contract("permuted_bf16x3_512", "abc=iaj,jbic", (512, 512, 512, 16, 16), "bf16x3"),
        # short contracted index, large result: memory traffic bounds it;
        # slices of very different size, as unscaled data has
        _contract("outer_bf16x3_512", "abc=ai,ibc", (512, 512, 512, 64), "bf16x3", values="lognormal"),
        # long contracted indices, square result: arithmetic bounds it, at
        # FP32-level accuracy and in plain 16-bit inputs
        _contract("matrix_bf16x3_4096", "ab=aij,jib", (4096, 4096, 64, 64), "bf16x3"),
        _contract("matrix_bf16_4096", "ab=aij,jib", (4096, 4096, 64, 64), "bf16"),
        # sizes that no tile divides, added to an existing result
        _contract("ragged_bf16x3_update", "abc=iaj,jbic", (301, 203, 97, 13, 11), "bf16x3", alpha=-1.0, beta=1.0),
        # a loop nest around gemm calls, chosen by name as the planner's
        # users do
        _contract("nest_gemm_f32_256", "abc=iaj,jbic", (256, 256, 256, 16, 16), "f32", algorithm="bi'-gemm"),
        # thousands of small uneven contractions in one launch
        {"name": "batch_f32_4096", "kind": "batch", "count": 4096, "dtype": "f32", "shapes": 0},
        {"name": "batch_bf16x3_4096", "kind": "batch", "count": 4096, "dtype": "bf16x3", "shapes": 0},
        # a burst of mixed requests to the server, host memory to host memory
        {"name": "serving_mix_24", "kind": "serving", "requests": 24, "shapes": 3},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    pick = rng.choice(("plain", "permuted", "permuted", "outer", "matrix", "matrix", "nest", "batch", "serving"))
    beta = rng.choice((0.0, 0.0, 0.0, 1.0))
    alpha = 1.0 if beta == 0.0 else rng.choice((-1.0, 0.5))
    values = rng.choice(("uniform", "uniform", "lognormal"))
    if pick == "plain":
        ext = [_log_int(rng, 8, 128) for _ in range(3)] + [_log_int(rng, 4, 32)]
        return _contract(None, "abc=ai,ibc", ext, rng.choice(("f64", "f32", "bf16x3")), alpha=alpha, beta=beta)
    if pick == "permuted":
        ext = [_log_int(rng, 64, 512) for _ in range(3)] + [rng.choice((16, 16, rng.randint(5, 16))) for _ in range(2)]
        return _contract(None, "abc=iaj,jbic", ext, rng.choice(("f64", "f32", "bf16x3", "tf32")), alpha=alpha,
                         beta=beta, values=values)
    if pick == "outer":
        ext = [_log_int(rng, 64, 512) for _ in range(3)] + [_log_int(rng, 8, 64)]
        return _contract(None, "abc=ai,ibc", ext, rng.choice(("f32", "bf16x3", "tf32", "bf16", "f16")), alpha=alpha,
                         beta=beta, values=values)
    if pick == "matrix":
        ext = [_log_int(rng, 256, 4096) for _ in range(2)] + [_log_int(rng, 8, 64) for _ in range(2)]
        return _contract(None, "ab=aij,jib", ext, rng.choice(("f32", "bf16x3", "tf32", "bf16", "f16", "tf32x3")),
                         alpha=alpha, beta=beta, values=values)
    if pick == "nest":
        ext = [_log_int(rng, 24, 160) for _ in range(3)] + [rng.choice((8, 16, rng.randint(5, 16))) for _ in range(2)]
        return _contract(None, "abc=iaj,jbic", ext, rng.choice(("f64", "f32")), alpha=alpha, beta=beta,
                         algorithm=rng.choice(("bi'-gemm", "cj'-gemm", "i'c-gemm", "bci'-gemv", "cij-ger",
                                               "cbaj-dot", "bcji-axpy")))
    if pick == "batch":
        return {"kind": "batch", "count": _log_int(rng, 64, 4096), "dtype": rng.choice(("f32", "bf16x3", "f64")),
                "shapes": rng.randint(1, 10 ** 6)}
    return {"kind": "serving", "requests": _log_int(rng, 4, 24), "shapes": rng.randint(1, 10 ** 6)}


# ------------------------------------------------------------------ inputs
def _modes(spec):
    lhs, rhs = spec.split("=")
    return (lhs, *rhs.split(","))


def _sizes(spec, extents):
    """Extent of each index and element counts of C, A, B."""
    modes = _modes(spec)
    ext = dict(zip(dict.fromkeys("".join(modes)), extents))
    return ext, [math.prod(ext[m] for m in ms) for ms in modes]


def _extents(case):
    return [int(x) for x in case["extents"].split(",")]


def _fill(n, dtype, gen):
    """n entries uniform in [-1, 1], drawn in 32 bits (FP64: in 64) and rounded to the type."""
    wide = torch.float64 if dtype == torch.float64 else torch.float32
    return torch.empty(n, dtype=wide, device=DEVICE).uniform_(-1.0, 1.0, generator=gen).to(dtype)


def _contract_inputs(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    ext, (nc, na, nb) = _sizes(case["spec"], _extents(case))
    dt = IN_TYPES[case["dtype"]]
    out_t = torch.float64 if case["dtype"] == "f64" else torch.float32
    ops = []
    for n, ms in ((na, _modes(case["spec"])[1]), (nb, _modes(case["spec"])[2])):
        x = _fill(n, dt, gen)
        if case["values"] == "lognormal":
            # one scale per value of the operand's last mode, 1e-4 to 1e4
            last = ext[ms[-1]]
            scale = torch.empty(last, dtype=torch.float64, device=DEVICE)
            scale.normal_(0.0, 4.0 * math.log(10.0) / 3.0, generator=gen).exp_().clamp_(1e-4, 1e4)
            x = (x.view(last, -1) * scale.view(last, 1).to(dt)).reshape(-1).contiguous()
        ops.append(x)
    c0 = _fill(nc, out_t, gen) if case["beta"] != 0.0 else None
    return ops[0], ops[1], c0, nc, out_t


def _batch_rows(case):
    rng = np.random.default_rng(case["shapes"])
    abc = np.rint(np.exp(rng.uniform(math.log(8), math.log(128), (case["count"], 3)))).astype(int)
    ks = rng.choice([4, 8, 16, 32], case["count"])
    return [[int(a), int(b), int(c), int(k)] for (a, b, c), k in zip(abc, ks)]


def _aligned(n):
    return (n + 63) // 64 * 64  # operands start on 256-byte boundaries, as allocations do


def _batch_inputs(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    dt = IN_TYPES[case["dtype"]]
    rows = _batch_rows(case)
    offs, tot = [], [0, 0, 0]
    for a, b, c, k in rows:
        offs.append(tuple(tot))
        for o, n in enumerate((a * k, k * b * c, a * b * c)):
            tot[o] += _aligned(n)
    return rows, offs, _fill(tot[0], dt, gen), _fill(tot[1], dt, gen), tot[2], dt


def _requests(case):
    rng = random.Random(case["shapes"])
    out = []
    while len(out) < case["requests"]:
        spec = rng.choice(SERVING_SPECS)
        order = list(dict.fromkeys("".join(_modes(spec))))
        ext = [_log_int(rng, 8, 128) if m in "ij" else _log_int(rng, 16, 384) for m in order]
        dtype = rng.choice(SERVING_DTYPES)
        sizes = _sizes(spec, ext)[1]
        if max(sizes) <= SERVING_MAX_C:
            out.append((spec, ext, dtype, sizes))
    return out


def _serving_inputs(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    out = []
    for spec, ext, dtype, (nc, na, nb) in _requests(case):
        dt = IN_TYPES[dtype]
        out.append((spec, ext, dtype, _fill(na, dt, gen), _fill(nb, dt, gen), nc))
    return out


# --------------------------------------------------------------- the cases
def prepare(case, seed):
    if case["kind"] == "contract":
        A, B, c0, nc, out_t = _contract_inputs(case, seed)
        plan = tc.Plan(case["spec"], _extents(case), dtype=case["dtype"])
        if case["algorithm"] != "gett":
            plan.select({a["name"]: a["id"] for a in plan.algorithms()}[case["algorithm"]])
        return {"case": case, "plan": plan, "A": A, "B": B, "C0": c0,
                "C": torch.empty(nc, dtype=out_t, device=DEVICE)}
    if case["kind"] == "batch":
        rows, offs, A, B, nc, dt = _batch_inputs(case, seed)
        C = torch.zeros(nc, dtype=dt, device=DEVICE)
        size = A.element_size()
        batch = tc.Batch("abc=ai,ibc", rows, case["dtype"])
        batch.set_operands(*([x.data_ptr() + o[i] * size for o in offs] for i, x in enumerate((A, B, C))))
        batch.prepare()
        return {"case": case, "batch": batch, "A": A, "B": B, "C": C}
    host = []
    for spec, ext, dtype, A, B, nc in _serving_inputs(case, seed):
        host.append((spec, ext, dtype, A.cpu().pin_memory(), B.cpu().pin_memory(),
                     torch.empty(nc, dtype=A.dtype, pin_memory=True)))
    return {"case": case, "server": tc.Server(budget_bytes=4 << 30, slots=32, streams=8), "requests": host}


def run(state):
    case = state["case"]
    if case["kind"] == "contract":
        if state["C0"] is not None:
            state["C"].copy_(state["C0"])
        state["plan"].execute(state["A"], state["B"], state["C"], alpha=case["alpha"], beta=case["beta"],
                              stream=torch.cuda.current_stream())
        return state["C"]
    if case["kind"] == "batch":
        state["batch"].execute(stream=torch.cuda.current_stream())
        return state["C"]
    server = state["server"]
    ids = [server.submit(*request) for request in state["requests"]]
    for rid in ids:
        server.wait(rid)
    return [request[-1] for request in state["requests"]]


def work(case):
    if case["kind"] == "contract":
        ext, (nc, na, nb) = _sizes(case["spec"], _extents(case))
        size = IN_TYPES[case["dtype"]].itemsize
        out = 8 if case["dtype"] == "f64" else 4
        return {"bytes": (na + nb) * size + nc * out * (2 if case["beta"] != 0.0 else 1),
                "flops": 2 * math.prod(ext.values())}
    if case["kind"] == "batch":
        size = IN_TYPES[case["dtype"]].itemsize
        rows = _batch_rows(case)
        return {"bytes": sum(size * (a * k + k * b * c + a * b * c) for a, b, c, k in rows),
                "flops": sum(2 * a * b * c * k for a, b, c, k in rows)}
    reqs = _requests(case)
    return {"bytes": sum(sum(sizes) * IN_TYPES[dtype].itemsize for _, _, dtype, sizes in reqs),
            "flops": sum(2 * math.prod(ext) for _, ext, _, _ in reqs)}


# Largest relative error of another correct implementation, by the type the
# products are taken in: about four times what was measured over these ranges
# -- one chain of roundings against the same chain run backwards (FP64 7e-16
# at 256 terms, FP32 1.6e-6 at 4096), and the library against 64 bits (split
# BF16 and 3xTF32 1.8e-6, BF16 and FP16 4e-6 at 4096 terms, their inputs being
# exact; TF32 2.6e-4, its inputs rounded to 11 bits).
TOLERANCE = {"f64": 4e-15, "f32": 6e-6, "bf16x3": 8e-6, "tf32x3": 8e-6, "tf32": 1.2e-3, "bf16": 1.6e-5, "f16": 1.6e-5}


def tolerance(case):
    if case["kind"] == "serving":  # requests of several types: the widest of them
        return {"rel": TOLERANCE["bf16x3"]}
    return {"rel": TOLERANCE[case["dtype"]]}


def _product(spec, ext, A, B):
    """The contraction in 64 bits, flat and first index fastest like C."""
    e = _sizes(spec, ext)[0]
    c, a, b = _modes(spec)
    x = A.double().view([e[m] for m in reversed(a)])
    y = B.double().view([e[m] for m in reversed(b)])
    return torch.einsum(f"{a[::-1]},{b[::-1]}->{c[::-1]}", x, y).reshape(-1)


def exact(case, seed):
    if case["kind"] == "contract":
        A, B, c0, _, _ = _contract_inputs(case, seed)
        out = case["alpha"] * _product(case["spec"], _extents(case), A, B)
        return out if c0 is None else out + case["beta"] * c0.double()
    if case["kind"] == "batch":
        rows, offs, A, B, nc, _ = _batch_inputs(case, seed)
        C = torch.zeros(nc, dtype=torch.float64, device=DEVICE)
        for (a, b, c, k), (oa, ob, oc) in zip(rows, offs):
            x = A[oa:oa + a * k].double().view(k, a)
            y = B[ob:ob + k * b * c].double().view(b * c, k)
            C[oc:oc + a * b * c] = (y @ x).view(-1)
        return C
    return [_product(spec, ext, A, B).cpu() for spec, ext, _, A, B, _ in _serving_inputs(case, seed)]
