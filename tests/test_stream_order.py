"""Plans on a stream of their own and the caller's CUDA tensors.

Host part: the enqueue order of Plan / BatchedPlan against a recording library,
recording streams and tensors that call themselves CUDA tensors. GPU part: inputs
that the current stream still computes.
"""
import numpy as np
import pytest
import torch

from paper_2507_17175_gb300 import qpe


class _Stream:
    def __init__(self, handle, log):
        self.cuda_stream, self.log = handle, log

    def wait_event(self, event):
        self.log.append(("wait", self.cuda_stream, event.recorded))


class _Event:
    def record(self, stream):
        self.recorded = stream.cuda_stream


class _Tensor(torch.Tensor):
    """A host tensor that says it lies on the GPU."""
    is_cuda = True

    def record_stream(self, stream):
        stream.log.append(("record", stream.cuda_stream, self.data_ptr()))


class _Lib:
    def __init__(self, log):
        self.log = log

    def __getattr__(self, name):
        def call(*args):
            self.log.append((name,))
            return 0
        return call


OWN, CURRENT = 7, 3


def _tensor(*shape, dtype=torch.complex128):
    return torch.zeros(shape, dtype=dtype).as_subclass(_Tensor)


@pytest.fixture
def recorded(monkeypatch):
    """(plan maker, log, capture switch) without a GPU."""
    log, capturing = [], [False]
    monkeypatch.setattr(qpe, "_lib", _Lib(log))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: _Stream(CURRENT, log))
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: capturing[0])
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "Event", _Event)

    def make(cls=qpe.Plan, handle=OWN):
        p = object.__new__(cls)
        p._h, p.prec, p.flags = 1, qpe.C64_FP32, qpe.FLAG_GRAPH
        p.nmat, p.nmeas, p.d, p.N = 1, 2, 2, 4
        p.shapes, p._keep_inputs = [(1, 2)], {}
        p.stream, p.device = _Stream(handle, log), torch.device("cuda")
        p._device_index, p._order = 0, _Event()
        return p
    yield make, log, capturing
    log.clear()


INPUTS = {
    "load": lambda p: p.load(_tensor(2, 2), _tensor(2)),
    "load_state": lambda p: p.load_state(_tensor(4, 2, dtype=torch.complex64)),
    "batched_load": lambda p: p.load(0, _tensor(2, 2), _tensor(2)),
}


@pytest.mark.parametrize("call", INPUTS)
def test_device_inputs_are_ordered_after_the_current_stream(recorded, call):
    make, log, _ = recorded
    INPUTS[call](make(qpe.BatchedPlan if call.startswith("batched") else qpe.Plan))
    enqueue = ("qpe_load_state",) if call == "load_state" else ("qpe_load",)
    assert ("wait", OWN, CURRENT) in log[:log.index(enqueue)]


@pytest.mark.parametrize("call", INPUTS)
def test_memory_of_dropped_inputs_waits_for_the_copy(recorded, call):
    make, log, _ = recorded
    INPUTS[call](make(qpe.BatchedPlan if call.startswith("batched") else qpe.Plan))
    assert sum(entry[:2] == ("record", OWN) for entry in log) == (1 if call == "load_state" else 2)


@pytest.mark.parametrize("cls,args", [(qpe.Plan, (1, 2, qpe.C64_FP32, qpe.FLAG_GRAPH)),
                                      (qpe.ShardedPlan, (1, 2, qpe.C64_FP32, qpe.FLAG_GRAPH, 0, 2)),
                                      (qpe.BatchedPlan, ([(1, 2)], qpe.C64_FP32, qpe.FLAG_GRAPH))])
def test_workspace_of_a_dropped_plan_waits_for_its_run(recorded, cls, args):
    _, log, _ = recorded
    ws = _tensor(64, dtype=torch.uint8)
    cls(*args, stream=_Stream(OWN, log), workspace=ws)
    assert ("record", OWN, ws.data_ptr()) in log
    assert log.index(("wait", OWN, CURRENT)) < log.index(("qpe_bind",))


@pytest.mark.parametrize("call", INPUTS)
def test_no_wait_on_the_same_stream_or_while_it_is_captured(recorded, call):
    make, log, capturing = recorded
    cls = qpe.BatchedPlan if call.startswith("batched") else qpe.Plan
    INPUTS[call](make(cls, CURRENT))
    capturing[0] = True
    INPUTS[call](make(cls))
    assert not any(entry[0] == "wait" for entry in log)


OUTPUTS = {
    "probs": lambda p: p.probs(_tensor(4, dtype=torch.float64)),
    "state": lambda p: p.state(_tensor(4, 2, dtype=torch.complex64)),
    "batched_probs": lambda p: p.probs(0, _tensor(4, dtype=torch.float64)),
    "batched_state": lambda p: p.state(0, _tensor(4, 2, dtype=torch.complex64)),
}


@pytest.mark.parametrize("call", OUTPUTS)
def test_device_outputs_are_ordered_with_the_current_stream(recorded, call):
    """A buffer the current stream still reads is not overwritten, and what that stream
    does next with a state that is only enqueued waits for it (qpe_probs returns when
    the bins are there)."""
    make, log, _ = recorded
    OUTPUTS[call](make(qpe.BatchedPlan if call.startswith("batched") else qpe.Plan))
    at = log.index(("qpe_" + call.split("_")[-1],))
    assert ("wait", OWN, CURRENT) in log[:at]
    assert ("wait", CURRENT, OWN) in log[at:] or call.endswith("probs")


def test_host_inputs_do_not_wait(recorded):
    make, log, _ = recorded
    plan = make()
    plan.load(np.eye(2, dtype=np.complex128), np.array([1, 0], dtype=np.complex128))
    assert log == [("qpe_load",)]


def _late(tensors, filler):
    """Copies that the current stream makes only after some 10 ms of other work;
    their memory holds NaN until then."""
    out = [torch.full_like(x, float("nan")) for x in tensors]
    torch.cuda.synchronize()
    filler @ filler
    for o, x in zip(out, tensors):
        o.copy_(x)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("batched", [False, True])
def test_inputs_still_being_computed(batched):
    """A graph plan replayed with inputs that are not there yet: the bins are those of
    the same inputs after a synchronisation, exactly."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    z = torch.randn((16, 16), generator=gen, dtype=torch.complex128, device="cuda")
    U, _ = torch.linalg.qr(z)
    U = U.contiguous()
    psi = U[:, 0].contiguous()
    filler = torch.eye(8192, device="cuda")
    if batched:
        plan = qpe.BatchedPlan([(4, 9)] * 2, qpe.FP64, qpe.FLAG_GRAPH)
        loads = [lambda a, b, i=i: plan.load(i, a, b) for i in range(2)]
    else:
        plan = qpe.Plan(4, 9, qpe.FP64, qpe.FLAG_GRAPH)
        loads = [plan.load]

    def bins():
        return [plan.probs(i)[0] if batched else plan.probs()[0] for i in range(len(loads))]

    torch.cuda.synchronize()
    for load in loads:
        load(U, psi)
    plan.run()
    want = bins()
    late = _late([U, psi] * len(loads), filler)
    for i, load in enumerate(loads):
        load(*late[2 * i:2 * i + 2])
    plan.run()
    for got, ref in zip(bins(), want):
        np.testing.assert_array_equal(got, ref)


@pytest.mark.gpu
def test_outputs_still_being_read():
    """The current stream's late copy of the last run's outputs is not overtaken by the next
    run's, and its copies of the next outputs see them whole."""
    gen = torch.Generator(device="cuda").manual_seed(6)
    Us = [torch.linalg.qr(torch.randn((4, 4), generator=gen, dtype=torch.complex128, device="cuda"))[0].contiguous()
          for _ in range(2)]
    plan = qpe.Plan(2, 16, qpe.FP64, qpe.FLAG_GRAPH | qpe.FLAG_PLAIN)
    filler = torch.eye(8192, device="cuda")
    hist = torch.empty(plan.N, dtype=torch.float64, device="cuda")
    state = torch.empty((plan.N, plan.d), dtype=torch.complex128, device="cuda")

    def run(U):
        plan.load(U, U[:, 0].contiguous())
        plan.run()
        plan.probs(hist)
        plan.state(state)
        return hist.clone(), state.clone()

    want = [run(U) for U in Us]
    torch.cuda.synchronize()
    run(Us[0])
    torch.cuda.synchronize()
    filler @ filler  # the copies below come late
    got = [(hist.clone(), state.clone()), run(Us[1])]
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        assert torch.equal(g[0], w[0]) and torch.equal(g[1], w[1])
