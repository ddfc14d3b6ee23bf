"""QFT^-1 passes and the reordering of their output: every split of the passes'
points over registers and shared memory (1 .. 9 bits), narrow rows (several
blocks per CTA), wide ones, and both read-back routes (16-byte pieces, and
elements for an output on an 8-byte boundary).

Tolerance (derived): a transform of 2^n points in n radix-2 steps errs by at most
n (4 sqrt 2 u + mu) |x| in the 2-norm, mu <= 6 u for twiddles that are products of
two table entries: 12 n u."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2507_17175_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2507_17175_gb300 import qpe
    return qpe


SHAPES = [(1, 1), (2, 2), (1, 3), (3, 4), (2, 5), (1, 6), (4, 7), (1, 8), (2, 9), (1, 10), (2, 11), (3, 12), (4, 13),
          (1, 14), (2, 15), (5, 11), (1, 17), (2, 18), (1, 19), (6, 10), (8, 6), (9, 12)]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nmat,nmeas", SHAPES)
def test_transform_and_read_back(q, prec, nmat, nmeas):
    import torch
    N, d = 1 << nmeas, 1 << nmat
    dt = np.complex128 if prec == 0 else np.complex64
    S = W.random_state(np.random.default_rng(nmat * 100 + nmeas), N, d).astype(dt)
    plan = q.Plan(nmat, nmeas, prec, q.FLAG_PLAIN)
    plan.load_state(S)
    plan.run_stages(q.STAGE_FFT, q.STAGE_REDUCE)
    ref = np.fft.fft(S.astype(np.complex128), axis=0, norm="ortho")
    u = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    tol = 12 * nmeas * u * np.linalg.norm(ref)
    flat = torch.zeros(N * d + 2, dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
    for offset in (0, 1):  # 1: complex64 output on an 8-byte boundary
        out = flat[offset:offset + N * d]
        out.zero_()
        plan.state(out)
        torch.cuda.synchronize()
        assert np.linalg.norm(out.cpu().numpy().reshape(N, d) - ref) <= tol
    P, am, _, _ = plan.probs()
    p = (np.abs(ref) ** 2).sum(1)
    # |X|^2 of values off by tol in all: 2 tol sqrt(max) + the sum's own roundings
    assert np.abs(P - p).max() <= 3 * tol * np.sqrt(p.max()) + 64 * u * p.max()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nmat,nmeas", [(1, 9), (2, 9), (2, 1)])
def test_rows_of_small_registers(q, prec, nmat, nmeas):
    """d = 2 and 4: a thread per row, on both schedules (doubling, gate by gate)."""
    inst = W.haar_instance(np.random.default_rng(nmat + nmeas), nmat, nmeas, superposition=True)
    u = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    ref = [inst.psi / np.sqrt(inst.N)]
    for m in range(1, inst.N):
        ref.append(inst.U @ ref[-1])
    # entries of U^m carry the rounding of U's squarings (2^n u) and of n gates
    tol = 32 * (inst.N * 2.0 ** -53 + nmeas * inst.d * u) / np.sqrt(inst.N)
    for flags in (q.FLAG_PLAIN, q.FLAG_GATE_SWEEP):
        plan = q.Plan(nmat, nmeas, prec, flags)
        plan.load(inst.U, inst.psi)
        plan.run_stages(q.STAGE_POWERS, q.STAGE_SWEEP)
        assert np.abs(plan.state() - np.array(ref)).max() <= tol
