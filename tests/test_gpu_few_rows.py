"""Doubling levels of few rows (warps share the inner index instead of 64 x 64
tiles): the rows after the controlled gates against numpy products with the
plan's own powers, on both sides of the rule that picks the kernel.

Tolerance (derived): a level's dot product of 2 d real terms with a unit row of
P_j errs by at most 2 d u |row|, so after n levels an entry is within
2 n d u of the exact row's norm (u = 2^-53, complex64 2^-24; complex64 adds its
rounding of P_j, 2 d u more per level)."""
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


def rows_by_doubling(plan, psi, nmeas):
    S = psi[None, :] / np.sqrt(1 << nmeas)
    for k in range(nmeas):
        S = np.concatenate([S, S @ plan.power(k).T])
    return S


def check(got, ref, nmeas, d, prec):
    u = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    tol = (1 if prec == 0 else 2) * 2 * nmeas * d * u / np.sqrt(1 << nmeas)
    assert np.abs(got - ref).max() <= tol


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nmat,nmeas", [(6, 1), (6, 4), (6, 10), (7, 2), (7, 8), (8, 3), (8, 9), (9, 7), (10, 5), (11, 3)])
def test_rows_after_the_gates(q, prec, nmat, nmeas):
    inst = W.haar_instance(np.random.default_rng(100 * nmat + nmeas), nmat, nmeas, superposition=True)
    plan = q.Plan(nmat, nmeas, prec, q.FLAG_PLAIN)
    plan.load(inst.U, inst.psi)
    plan.run_stages(q.STAGE_POWERS, q.STAGE_SWEEP)
    check(plan.state(), rows_by_doubling(plan, inst.psi, nmeas), nmeas, 1 << nmat, prec)


@pytest.mark.parametrize("prec", [0, 1])
def test_grouped_levels_match_the_single_plan(q, prec):
    """A batch that mixes sizes on both sides of the rule gives each instance
    the histogram of its own plan (the squarings' tiles may differ: a rounding bound)."""
    shapes = [(7, 9), (8, 5), (9, 7), (10, 4), (6, 6), (11, 2), (7, 1)]
    insts = [W.haar_instance(np.random.default_rng(i), a, b, superposition=True) for i, (a, b) in enumerate(shapes)]
    bp = q.BatchedPlan(shapes, prec, q.FLAG_PLAIN)
    for i, inst in enumerate(insts):
        bp.load(i, inst.U, inst.psi)
    bp.run()
    for i, inst in enumerate(insts):
        plan = q.Plan(inst.nmat, inst.nmeas, prec, q.FLAG_PLAIN)
        plan.load(inst.U, inst.psi)
        plan.run()
        P, am, _, _ = plan.probs()
        Pb, amb, _, _ = bp.probs(i)
        tol = 64 * inst.d * inst.nmeas * (2.0 ** -53 if prec == 0 else 2.0 ** -24)
        assert np.abs(P - Pb).max() <= tol and am == amb
