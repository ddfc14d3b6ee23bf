"""States on any boundary of their real type: read back and read out as on one of 16
bytes; pointers that no load of the real type can take are refused before a launch."""
import ctypes

import numpy as np
import pytest

from paper_2507_17175_gb300 import qpe
from paper_2507_17175_gb300 import workloads as W

BASE = 1 << 20  # never dereferenced: the checks come first


@pytest.mark.parametrize("prec,state,probs,readout", [(qpe.FP64, 4, 0, 0), (qpe.C64_FP32, 2, 0, 0), (qpe.FP64, 0, 4, 0),
                                                      (qpe.C64_FP16X2, 0, 0, 4), (qpe.FP64, 9, 0, 0)])
def test_misaligned_pointers_are_refused(prec, state, probs, readout):
    st = qpe._lib.qpe_readout_static(BASE + state, 2, 3, prec, BASE + 4096 + probs, BASE + 8192 + readout, None)
    assert st == qpe.ERR_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("nmat,nmeas", [(1, 6), (2, 11), (5, 8), (9, 7)])
@pytest.mark.parametrize("prec,offset", [(qpe.FP64, 8), (qpe.C64_FP32, 8), (qpe.C64_FP32, 4), (qpe.C64_FP32, 12)])
def test_offset_states(prec, offset, nmat, nmeas):
    import torch
    N, d = 1 << nmeas, 1 << nmat
    dt = np.complex128 if prec == qpe.FP64 else np.complex64
    S = W.random_state(np.random.default_rng(7 * nmat + nmeas), N, d).astype(dt)
    plan = qpe.Plan(nmat, nmeas, prec, qpe.FLAG_PLAIN)
    plan.load_state(S)
    plan.run_stages(qpe.STAGE_FFT, qpe.STAGE_FFT)
    ref = plan.state()  # through the host
    raw = torch.zeros(S.nbytes + 32, dtype=torch.uint8, device="cuda")
    assert raw.data_ptr() % 16 == 0
    assert qpe._lib.qpe_state(plan.handle, 0, raw.data_ptr() + offset, 1) == qpe.OK
    torch.cuda.synchronize()
    assert raw.cpu().numpy()[offset:offset + S.nbytes].tobytes() == ref.tobytes()
    if (prec == qpe.FP64) and offset % 8 == 0:
        assert qpe._lib.qpe_state(plan.handle, 0, raw.data_ptr() + 4, 1) == qpe.ERR_ARG
    both = []
    for at in (0, offset):
        raw[at:at + S.nbytes] = torch.from_numpy(np.frombuffer(ref.tobytes(), dtype=np.uint8).copy()).cuda()
        probs = torch.empty(N, dtype=torch.float64, device="cuda")
        out = torch.empty(4, dtype=torch.float64, device="cuda")
        assert qpe._lib.qpe_readout_static(raw.data_ptr() + at, nmat, nmeas, prec, probs.data_ptr(), out.data_ptr(),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == qpe.OK
        torch.cuda.synchronize()
        both.append((probs, out))
    assert torch.equal(both[0][0], both[1][0]) and torch.equal(both[0][1], both[1][1])
