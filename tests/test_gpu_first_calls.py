"""A plan can be used on any stream as soon as it has been made (GPU).

Tables go to the device on the legacy stream, which nothing orders before a call on a
non-blocking stream.  The legacy stream is kept busy here while the plan is made, so that
a copy that is still queued when the maker returns would be missed by the first call.
"""
import threading

import numpy as np
import pytest

from paper_2108_06831_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


class _BusyLegacyStream:
    """A thread that always keeps a few short kernels queued on the legacy stream."""

    def __enter__(self):
        self._stop = threading.Event()
        self._busy = threading.Event()
        self._thread = threading.Thread(target=self._run)
        self._thread.start()
        self._busy.wait()
        return self

    def _run(self):
        queued = []
        while not self._stop.is_set():
            torch.cuda._sleep(2_000_000)  # about a millisecond
            e = torch.cuda.Event()
            e.record(torch.cuda.default_stream())
            queued.append(e)
            self._busy.set()
            if len(queued) >= 4:
                queued.pop(0).synchronize()

    def __exit__(self, *exc):
        self._stop.set()
        self._thread.join()
        torch.cuda.synchronize()


def _empty(*shape, dtype=torch.complex64):
    return torch.empty(shape, dtype=dtype, device="cuda")


def _state(n, **kw):
    from paper_2108_06831_gb300 import tn
    ctr = tn.Contractor(C.brickwork(n, 6, 5)[0], **kw)
    return lambda out, st: tn.contract_state(ctr.plan, None, out, ctr.workspace, stream=st)


def _q428(n):
    from paper_2108_06831_gb300 import tn
    plan = tn.Plan(tn.CircuitHandle(C.brickwork(n, 6, 5)[0]), q428=True)
    return lambda out, st: tn.contract_state_q428(plan, out, stream=st)


def _network(ws, bits):
    from paper_2108_06831_gb300 import tn
    plan = tn.Plan(tn.CircuitHandle(C.grid(3, 4, 6, 3)), target=tn.TARGET_AMPLITUDES, network_bitstrings=8)
    assert plan.workspace_bytes <= ws.numel()
    return lambda out, st: tn.contract_amplitudes(plan, None, bits, out, ws, stream=st)


def _batch(ws):
    from paper_2108_06831_gb300 import tn
    b = tn.Batch([tn.Plan(tn.CircuitHandle(C.brickwork(n, 6, n)[0]), specialize=False) for n in (8, 10)])
    assert b.workspace_bytes <= ws.numel()
    return lambda out, st: tn.batch_run(b, out, ws, stream=st)


def _energy(state, ws):
    from paper_2108_06831_gb300 import tn
    obs = tn.Observable(C.tfim(12))
    nb = tn.state_expectation_workspace_bytes(obs, 1)
    assert nb <= ws.numel()
    return lambda out, st: tn.state_expectation(obs, 1, state, out, ws, nb, stream=st)


@pytest.mark.parametrize("kind", ["state20", "state9", "q428", "blocks", "network", "batch", "energy"])
def test_first_call_on_a_non_blocking_stream(kind):
    ws = torch.zeros(1 << 26, dtype=torch.uint8, device="cuda")
    bits = torch.arange(8, dtype=torch.int64, device="cuda")
    psi = torch.zeros(1 << 12, dtype=torch.complex64, device="cuda")
    psi[5] = 1
    make, out = {
        "state20": (lambda: _state(20), _empty(1, 1 << 20)),
        "state9": (lambda: _state(9), _empty(1, 1 << 9)),
        "q428": (lambda: _q428(14), _empty(1 << 14, 2, dtype=torch.int32)),
        "blocks": (lambda: _state(14, block_qubits=6), _empty(1, 1 << 14)),
        "network": (lambda: _network(ws, bits), _empty(1, 8)),
        "batch": (lambda: _batch(ws), _empty((1 << 8) + (1 << 10))),
        "energy": (lambda: _energy(psi, ws), _empty(1, dtype=torch.float64)),
    }[kind]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with _BusyLegacyStream():
        call = make()
        call(out, side)
        side.synchronize()
        with torch.cuda.stream(side):
            first = out.cpu()
    call(out, side)
    torch.cuda.synchronize()
    assert np.array_equal(first.numpy(), out.cpu().numpy())
    assert np.abs(first.numpy()).max() > 0
