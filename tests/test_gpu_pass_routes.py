"""QFT^-1 passes on both sides of the rule between short and long transforms, narrow
rows with wide tiles, and batches that mix them; grouped gate levels by the norm of
the final state.

Tolerances (2-norm of the whole state, whose norm is 1): the transform's 12 n u of
test_gpu_passes.py; rows through n gate levels off by at most 2 sqrt(2) d u each;
powers from different squaring tiles by 8 d N 2^-53 in all."""
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


def unit(prec):
    return 2.0 ** -53 if prec == 0 else 2.0 ** -24


# the last shape below and the first above 2^17 and 2^18 points, parts of a tile, 3 and
# 4 bits, and narrow rows in tiles of more than 128 bytes
SHAPES = [(1, 3), (2, 3), (1, 4), (3, 4), (2, 7), (3, 7), (3, 9), (8, 8), (8, 9), (3, 13), (1, 16), (3, 14), (1, 17),
          (4, 14), (2, 19), (1, 20), (1, 21), (2, 20)]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nmat,nmeas", SHAPES)
def test_transform(q, prec, nmat, nmeas):
    N, d = 1 << nmeas, 1 << nmat
    S = W.random_state(np.random.default_rng(nmat * 100 + nmeas), N, d).astype(np.complex128 if prec == 0 else np.complex64)
    plan = q.Plan(nmat, nmeas, prec, q.FLAG_PLAIN)
    plan.load_state(S)
    plan.run_stages(q.STAGE_FFT, q.STAGE_FFT)
    ref = np.fft.fft(S.astype(np.complex128), axis=0, norm="ortho")
    assert np.linalg.norm(plan.state() - ref) <= 12 * nmeas * unit(prec) * np.linalg.norm(ref)


BATCHES = {
    "short": [(1, 8), (2, 9), (3, 6), (1, 3)],
    "nine_bits": [(1, 9), (3, 9), (2, 5)],
    "mixed": [(3, 14), (1, 9), (2, 13), (1, 19), (1, 3), (4, 14)],
    "gates": [(7, 9), (8, 5), (9, 7), (10, 4), (6, 6), (11, 2), (7, 1)],
}


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("batch", BATCHES)
def test_batched_final_states(q, prec, batch):
    insts = [W.haar_instance(np.random.default_rng(i), a, b, superposition=True)
             for i, (a, b) in enumerate(BATCHES[batch])]
    bp = q.BatchedPlan(BATCHES[batch], prec, q.FLAG_PLAIN)
    for i, inst in enumerate(insts):
        bp.load(i, inst.U, inst.psi)
    bp.run()
    for i, inst in enumerate(insts):
        one = q.Plan(inst.nmat, inst.nmeas, prec, q.FLAG_PLAIN)
        one.load(inst.U, inst.psi)
        one.run_stages(q.STAGE_POWERS, q.STAGE_POWERS)
        S = inst.psi[None, :] / np.sqrt(inst.N)
        for k in range(inst.nmeas):
            S = np.concatenate([S, S @ one.power(k).T])
        ref = np.fft.fft(S, axis=0, norm="ortho")
        tol = (12 + 4 * inst.d) * inst.nmeas * unit(prec) + 8 * inst.d * inst.N * 2.0 ** -53
        assert np.linalg.norm(bp.state(i) - ref) <= tol
