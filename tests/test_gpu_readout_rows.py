"""qpe_readout_static's row sums: complex64 rows are summed in error-free FP32
parts, so every bin has to be within a few FP64 roundings of the exact sum
whatever the row's length, range of magnitudes or address.

Tolerances (derived): a complex64 bin loses at most 2^-54 of the row's largest
square per step it drops (three-part sums) and two FP64 roundings when the
parts meet, 4 * 2^-53 in all; a complex128 bin is a chain of at most 16 FP64
FMAs per lane, 5 lane sums and 15 pieces: 40 * 2^-53."""
from __future__ import annotations

import numpy as np
import pytest

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


def bins(q, S, prec, offset):
    import torch
    N, d = S.shape
    flat = torch.zeros(S.size + 2, dtype=torch.complex64 if prec == q.C64_FP32 else torch.complex128, device="cuda")
    view = flat[offset:offset + S.size]  # offset 1: complex64 data on an 8-byte boundary
    view.copy_(torch.from_numpy(S.reshape(-1)))
    probs = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
    ro = torch.zeros(4, dtype=torch.float64, device="cuda")
    st = q.readout_static(view, int(np.log2(d)), int(np.log2(N)), prec, probs, ro)
    assert st == q.OK
    torch.cuda.synchronize()
    r = ro.cpu().numpy()
    return probs.cpu().numpy(), int(r[:1].view(np.int64)[0]), r[2], r[3]


def exact(S):
    """Row sums of |x|^2 in double-double (numpy): squares by Dekker splits."""
    import math
    x = np.stack([S.real, S.imag], -1).reshape(S.shape[0], -1).astype(np.float64)
    c = x * 134217729.0
    h = c - (c - x)
    l = x - h
    p = x * x
    e = ((h * h - p) + 2 * h * l) + l * l
    return np.array([math.fsum(np.concatenate([a, b])) for a, b in zip(p, e)])


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nmat,nmeas", [(1, 1), (1, 10), (2, 9), (3, 8), (4, 9), (5, 3), (5, 9), (6, 8), (7, 7), (8, 5),
                                        (9, 5), (10, 6), (12, 4)])
def test_row_sums_are_fp64_accurate(q, prec, nmat, nmeas, offset):
    rng = np.random.default_rng(1000 * nmat + nmeas)
    N, d = 1 << nmeas, 1 << nmat
    S = rng.standard_normal((N, d)) + 1j * rng.standard_normal((N, d))
    S *= 10.0 ** rng.uniform(-9, 0, (N, d))           # magnitudes mixed within a row
    S *= 10.0 ** rng.uniform(-14, 14, (N, 1))         # and across rows, past FP32's range when squared
    S[N // 2] = 0.0
    S = np.ascontiguousarray(S.astype(np.complex64 if prec == 1 else np.complex128))
    if prec == 1 and N > 2:
        S[1] = np.complex64(1e-42)                    # a row of subnormal numbers
    P, am, mean, total = bins(q, S, prec, offset)
    ref = exact(S)
    tol = (4 if prec == 1 else 40) * 2.0 ** -53
    assert np.all(np.abs(P - ref) <= tol * ref)
    assert P[N // 2] == 0.0
    assert am == int(np.argmax(ref))
    assert abs(total - ref.sum()) <= 1e-12 * ref.sum()
    assert abs(mean - (ref * np.arange(N)).sum() / N) <= 1e-12 * ref.sum()


@pytest.mark.parametrize("nmat", [2, 5, 9])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_rows_stay_apart(q, nmat, bad):
    """One bad value spoils its own bin and the readout, and no other bin."""
    rng = np.random.default_rng(5)
    S = (rng.standard_normal((64, 1 << nmat)) + 1j * rng.standard_normal((64, 1 << nmat))).astype(np.complex64)
    S[17, 1] = bad
    P, am, _, total = bins(q, S, q.C64_FP32, 0)
    assert am == -1 and not np.isfinite(total) and not np.isfinite(P[17])
    keep = np.arange(64) != 17
    ref = exact(S[keep])
    assert np.all(np.abs(P[keep] - ref) <= 4 * 2.0 ** -53 * ref)
