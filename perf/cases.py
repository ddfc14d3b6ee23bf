"""The work a user of this framework has it do, as measurable cases.

A case is one QPE problem (or one batch of them, or one readout of a state a
program already holds), sized after this repository's named workloads
(workloads.py: c1 .. c5), the shapes of Tables 1-2 that scaling_study.py runs
and the benchmark. A pass is what a program does per problem: load U and psi,
run, read the histogram and both estimators.

The bins of complex64 plans (complex64 state, or one of the split precisions)
are kept as float32, the precision they are computed in; the bins of FP64 plans
stay float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_17175_gb300 import qpe

PREC = {"fp64": qpe.FP64, "c64": qpe.C64_FP32, "fp16x2": qpe.C64_FP16X2, "tf32x3": qpe.C64_TF32X3}


def _case(kind, prec, nmat, nmeas, support, **more):
    """``support``: how many eigenvectors of U psi is a superposition of."""
    return {"kind": kind, "prec": prec, "nmat": nmat, "nmeas": nmeas, "support": support, **more}


def listed():
    return [
        # The smallest problem (workload c1): a 2-qubit U, 6 measurement qubits,
        # host arrays in and out. Latency and launches.
        _case("small", "fp64", 2, 6, 1, name="small_fp64_2_6"),
        # Workload c2, captured as a graph and replayed with new inputs: the
        # ordinary complex64 call.
        _case("fused_graph", "c64", 6, 16, 1, name="fused_c64_6_16"),
        # The complex64 schedule at size, an odd register.
        _case("fused", "c64", 3, 25, 5, name="fused_c64_3_25"),
        # Sec. 4.2's study of both estimators: FP64, a 16 x 16 U, eigenvector inputs.
        _case("fused", "fp64", 4, 19, 1, name="fused_fp64_4_19"),
        # The benchmark's headline problem (workload c5) at 32 qubits: FP64
        # accuracy with the levels on the tensor cores.
        _case("levels_tc", "fp64", 4, 28, 16, name="levels_fp64_4_28"),
        # The same problem in split precision.
        _case("levels_tc", "fp16x2", 4, 28, 16, name="levels_fp16x2_4_28"),
        # A large target register (workload c3's kind): gates and squarings as
        # GEMMs on the tensor cores.
        _case("gemm_tc", "fp16x2", 11, 18, 1, name="gemm_fp16x2_11_18"),
        # The same kind at FP64 accuracy.
        _case("gemm_tc", "fp64", 10, 17, 1, name="gemm_fp64_10_17"),
        # Table 1's largest shape with no option set: complex64, CUDA cores.
        _case("plain", "c64", 8, 13, 1, name="plain_c64_8_13"),
        # Small registers with the final statevector kept (the paper's output
        # file): passes over a state in memory.
        _case("state", "c64", 2, 25, 3, name="state_c64_2_25"),
        # A batch of uneven problems (workload c4's ranges), one graph.
        {"kind": "batch", "prec": "fp16x2", "count": 41, "shapes": 12345, "name": "batch_fp16x2_41"},
        # Histogram and readout of a state that another program computed.
        _case("readout", "c64", 5, 21, 3, name="readout_c64_5_21"),
    ]


# kind: (precisions, Nmat range, Nmeas range, bound on Nmat + Nmeas, bound on 2 Nmat + Nmeas)
RANGES = {
    "small": (("fp64", "c64"), (1, 4), (1, 10), 14, 18),
    "fused_graph": (("c64", "fp64"), (2, 6), (8, 18), 24, 28),
    "fused": (("c64", "fp64"), (1, 6), (10, 25), 28, 31),
    "levels_tc": (("fp64", "fp16x2", "tf32x3"), (4, 4), (11, 28), 32, 36),
    "gemm_tc": (("fp16x2", "tf32x3", "fp64"), (8, 11), (8, 18), 29, 40),
    "plain": (("c64",), (7, 9), (6, 15), 23, 32),
    "state": (("c64", "fp64"), (1, 3), (14, 25), 27, 31),
    "readout": (("c64", "fp64"), (1, 12), (8, 21), 26, 40),
}
FP64_BOUND = {"fused": 28, "fused_graph": 24, "gemm_tc": 37, "state": 28, "readout": 38}


def draw(rng):
    kind = rng.choice(sorted(RANGES) + ["batch"])
    if kind == "batch":
        prec = rng.choice(("fp16x2", "tf32x3", "c64"))
        return {"kind": kind, "prec": prec, "count": rng.randint(3, 36 if prec == "fp16x2" else 18),
                "shapes": rng.randrange(1 << 30)}
    precs, mat, meas, both, cost = RANGES[kind]
    prec = rng.choice(precs)
    if prec == "fp64":
        cost = min(cost, FP64_BOUND.get(kind, cost))
    while True:
        nmat, nmeas = rng.randint(*mat), rng.randint(*meas)
        if nmat + nmeas <= both and 2 * nmat + nmeas <= cost:
            break
    return _case(kind, prec, nmat, nmeas, rng.randint(1, 1 << nmat if kind != "readout" else 6))


def _shapes(case):
    """(Nmat, Nmeas) of a batch's instances: Nmat in 3..10, Nmeas in 8..18."""
    rng = np.random.default_rng(case["shapes"])
    return [(int(rng.integers(3, 11)), int(rng.integers(8, 19))) for _ in range(case["count"])]


def _problem(nmat, support, seed):
    """U = V diag(exp(2 pi i phi)) V^dagger with a Haar V and uniform phases, and
    a normalised superposition of ``support`` eigenvectors, on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    d = 1 << nmat
    z = torch.randn((d, d), generator=gen, dtype=torch.complex128, device="cuda")
    q, r = torch.linalg.qr(z)
    diag = torch.diagonal(r)
    V = q * (diag / diag.abs())
    lam = torch.exp(2j * math.pi * torch.rand(d, generator=gen, dtype=torch.float64, device="cuda"))
    U = (V * lam) @ V.mH
    c = torch.randn(support, generator=gen, dtype=torch.complex128, device="cuda")
    psi = V[:, :support] @ (c / c.norm())
    return U.contiguous(), psi.contiguous()


def _final_state(case, seed):
    """A final statevector as QPE leaves it: peaks of sin(pi x) / (N sin(pi x / N))
    over the outcomes, one for each eigenvector in the input."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    N, d, k = 1 << case["nmeas"], 1 << case["nmat"], case["support"]
    phases = torch.rand(k, generator=gen, dtype=torch.float64, device="cuda")
    vec = torch.randn((k, d), generator=gen, dtype=torch.complex128, device="cuda")
    vec = vec / vec.norm()
    y = torch.arange(N, dtype=torch.float64, device="cuda")
    S = torch.zeros((N, d), dtype=torch.complex64 if case["prec"] == "c64" else torch.complex128, device="cuda")
    for j in range(k):
        x = N * phases[j] - y
        amp = torch.sin(math.pi * x) / (N * torch.sin(math.pi * x / N)) * torch.exp(1j * math.pi * x * (N - 1) / N)
        S += (amp[:, None] * vec[j][None, :]).to(S.dtype)
    return S


FLAGS = {"small": 0, "fused": 0, "fused_graph": qpe.FLAG_GRAPH, "levels_tc": qpe.FLAG_LEVEL_TC | qpe.FLAG_GRAPH,
         "gemm_tc": qpe.FLAG_SQUARE_TC | qpe.FLAG_LEVEL_TC, "plain": 0, "state": qpe.FLAG_PLAIN,
         "batch": qpe.FLAG_SQUARE_TC | qpe.FLAG_GRAPH}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        shapes = _shapes(case)
        inputs = [_problem(nmat, 1, seed * 1000 + i) for i, (nmat, _) in enumerate(shapes)]
        plan = qpe.BatchedPlan(shapes, PREC[case["prec"]], FLAGS[kind])
        sizes = [1 << nmeas for _, nmeas in shapes]
        bins = torch.empty(sum(sizes), dtype=torch.float64, device="cuda")
        return {"case": case, "plan": plan, "inputs": inputs, "bins": bins, "hist": bins.split(sizes)}
    nmat, nmeas = case["nmat"], case["nmeas"]
    if kind == "readout":
        return {"case": case, "state": _final_state(case, seed),
                "hist": torch.empty(1 << nmeas, dtype=torch.float64, device="cuda"),
                "readout": torch.empty(4, dtype=torch.float64, device="cuda")}
    U, psi = _problem(nmat, case["support"], seed)
    if kind == "small":
        U, psi = U.cpu().numpy(), psi.cpu().numpy()
        hist = np.empty(1 << nmeas, dtype=np.float64)
    else:
        hist = torch.empty(1 << nmeas, dtype=torch.float64, device="cuda")
    state = {"case": case, "plan": qpe.Plan(nmat, nmeas, PREC[case["prec"]], FLAGS[kind]), "U": U, "psi": psi, "hist": hist}
    if kind == "state":
        state["final"] = torch.empty((1 << nmeas, 1 << nmat), dtype=torch.complex128 if case["prec"] == "fp64" else torch.complex64,
                                     device="cuda")
    return state


def _bins(case, hist):
    if case["prec"] == "fp64":
        return hist
    return hist.astype(np.float32) if isinstance(hist, np.ndarray) else hist.to(torch.float32)


def run(state):
    case = state["case"]
    if case["kind"] == "readout":
        status = qpe.readout_static(state["state"], case["nmat"], case["nmeas"], PREC[case["prec"]], state["hist"],
                                    state["readout"])
        if status != qpe.OK:
            raise RuntimeError(qpe.status_string(status))
        return {"hist": _bins(case, state["hist"]), "argmax": state["readout"][:1].view(torch.int64),
                "estimators": _bins(case, state["readout"][1:])}
    plan = state["plan"]
    if case["kind"] == "batch":
        for i, (U, psi) in enumerate(state["inputs"]):
            plan.load(i, U, psi)
        plan.run()
        read = [plan.probs(i, out) for i, out in enumerate(state["hist"])]
        return {"hist": _bins(case, state["bins"]), "argmax": np.array([r[1] for r in read]),
                "phase_mean": np.array([r[3] for r in read], dtype=np.float32)}
    plan.load(state["U"], state["psi"])
    plan.run()
    hist, argmax, _, mean = plan.probs(state["hist"])
    out = {"hist": _bins(case, hist), "argmax": argmax, "phase_mean": mean}
    if case["kind"] == "state":
        out["state"] = plan.state(state["final"])
    return out


def work(case):
    if case["kind"] == "batch":
        parts = [_one_work(a, b, 4) for a, b in _shapes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    esize = 16 if case["prec"] == "fp64" else 8
    nmat, nmeas = case["nmat"], case["nmeas"]
    points = 1 << (nmat + nmeas)
    if case["kind"] == "readout":
        return {"bytes": points * esize + ((esize // 2) << nmeas), "flops": 4 * points}
    w = _one_work(nmat, nmeas, esize // 2)
    if case["kind"] == "state":
        w["bytes"] += points * esize
    return w


def _one_work(nmat, nmeas, bin_bytes):
    """U and psi in, the bins out; the squarings, one gate row per outcome, the
    transform of every column and the squared magnitudes."""
    d, N = 1 << nmat, 1 << nmeas
    return {"bytes": 16 * d * (d + 1) + bin_bytes * N,
            "flops": 8 * (nmeas - 1) * d ** 3 + 8 * N * d * d + 5 * N * nmeas * d + 4 * N * d}


def _exact_problem(U, psi, nmeas, keep=False):
    """Histogram, weighted mean (and the final state) of one problem in 64 bits:
    the rows U^m psi by doubling, one FFT per column, squared magnitudes. The most
    probable outcome follows from the bins and has no value of its own."""
    N, d = 1 << nmeas, U.shape[0]
    S = torch.empty((d, N), dtype=torch.complex128, device="cuda")
    S[:, 0] = psi / math.sqrt(N)
    P = U
    for j in range(nmeas):
        h = 1 << j
        for a in range(0, h, 1 << 24):
            b = min(h, a + (1 << 24))
            S[:, h + a:h + b] = P @ S[:, a:b]
        if j + 1 < nmeas:
            P = P @ P
    hist = torch.zeros(N, dtype=torch.float64, device="cuda")
    for t in range(d):
        X = torch.fft.fft(S[t], norm="ortho")
        if keep:
            S[t] = X
        hist += X.real.square() + X.imag.square()
    y = torch.arange(N, dtype=torch.float64, device="cuda")
    mean = float((hist * (y / N)).sum())
    return hist, mean, (S.T.contiguous() if keep else None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        parts = [_exact_problem(*_problem(nmat, 1, seed * 1000 + i), nmeas) for i, (nmat, nmeas) in enumerate(_shapes(case))]
        return {"hist": torch.cat([p[0] for p in parts]), "argmax": None,
                "phase_mean": np.array([p[1] for p in parts])}
    if kind == "readout":
        S = _final_state(case, seed).to(torch.complex128)
        hist = (S.real.square() + S.imag.square()).sum(1)
        y = torch.arange(hist.numel(), dtype=torch.float64, device="cuda") / hist.numel()
        return {"hist": hist, "argmax": None,
                "estimators": torch.stack([y[int(hist.argmax())], (hist * y).sum(), hist.sum()])}
    U, psi = _problem(case["nmat"], case["support"], seed)
    hist, mean, final = _exact_problem(U, psi, case["nmeas"], kind == "state")
    out = {"hist": hist, "argmax": None, "phase_mean": mean}
    if kind == "state":
        out["state"] = final
    return out
