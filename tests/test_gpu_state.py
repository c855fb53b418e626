"""Parity of the CUDA contraction path with the FP64 oracle (GPU).

Bar (complex64 states and amplitude vectors): relative L2 error <= 1e-5 against the
oracle's complex128 result; expectations |E - E_ref| <= 1e-4 max(1, |E_ref|).
"""
import numpy as np
import pytest

from paper_2108_06831_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STATE_TOL = 1e-5


def _tn():
    from paper_2108_06831_gb300 import tn
    return tn


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def gpu_state(circ, params=None, batch=1, tile=0, specialize=True):
    tn = _tn()
    ctr = tn.Contractor(circ, target=tn.TARGET_STATE, batch=batch, tile_qubits=tile, specialize=specialize)
    p = None if params is None else torch.as_tensor(np.asarray(params, dtype=np.float64).reshape(batch, -1),
                                                    device="cuda").contiguous()
    out = ctr.state(p)
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    return out.cpu().numpy()


@pytest.mark.parametrize("specialize", [True, False])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 8, 9, 11, 12])
def test_random_circuits_small(n, specialize):
    """Every gate kind, both the plan-specialised kernels and the interpreting kernel."""
    from oracle.statevector import simulate_state
    for seed in range(3):
        c = C.random_circuit(n, 12 * n + 5, 100 * n + seed)
        c.init_basis = (seed * 7919) % (1 << n)
        ref = simulate_state(c)
        got = gpu_state(c, specialize=specialize)[0]
        assert rel_l2(got, ref) <= STATE_TOL, (n, seed)


@pytest.mark.parametrize("specialize", [True, False])
@pytest.mark.parametrize("n,tile", [(13, 6), (14, 6), (15, 8), (16, 10), (17, 12), (18, 13), (16, 7)])
def test_random_circuits_multipass(n, tile, specialize):
    """Several tiles and passes; tile sizes from the smallest allowed upwards."""
    from oracle.statevector import simulate_state
    c = C.random_circuit(n, 10 * n, 7 * n + tile)
    c.init_basis = (n * 104729) % (1 << n)
    ref = simulate_state(c)
    got = gpu_state(c, tile=tile, specialize=specialize)[0]
    assert rel_l2(got, ref) <= STATE_TOL


def test_cfg1_brickwork_10q_depth8():
    from oracle.statevector import simulate_state
    c, _ = C.brickwork(10, 8, 1000)
    ref = simulate_state(c)
    got = gpu_state(c)[0]
    assert rel_l2(got, ref) <= STATE_TOL


@pytest.mark.parametrize("maker", [
    lambda: C.brickwork(16, 12, 5)[0],
    lambda: C.qft(16, 12345),
    lambda: C.paper_fig31(16, 6, 3),
    lambda: C.grid(4, 4, 10, 8),
    lambda: C.ghz(14),
])
def test_workload_families(maker):
    from oracle.statevector import simulate_state
    c = maker()
    ref = simulate_state(c)
    for tile in (0, 9):
        got = gpu_state(c, tile=tile)[0]
        assert rel_l2(got, ref) <= STATE_TOL


def test_parameterized_batch():
    """Per-batch parameters: every batch element matches the oracle with its own angles."""
    from oracle.statevector import simulate_state
    c, p0 = C.brickwork(12, 6, 77, parameterized=True)
    rng = np.random.default_rng(5)
    params = np.stack([p0] + [rng.uniform(0, 2 * np.pi, size=p0.shape) for _ in range(4)])
    got = gpu_state(c, params, batch=5)
    for b in range(5):
        assert rel_l2(got[b], simulate_state(c, params[b])) <= STATE_TOL


def test_cfg2_full_size_sampled():
    """24-qubit brickwork, depth 20, in the bench's launch configuration (parameterised
    U3 angles, plan-specialised kernels): sampled amplitudes against the oracle's network
    contraction, plus the norm."""
    from oracle.tn import contract_amplitude
    c, params = C.brickwork(24, 20, 1001, parameterized=True)
    got = gpu_state(c, params)[0]
    c, _ = C.brickwork(24, 20, 1001)
    assert abs(np.linalg.norm(got.astype(np.complex128)) - 1.0) < 1e-5
    xs = C.random_bitstrings(24, 10, 4242)
    ref = np.array([contract_amplitude(c, int(x)) for x in xs])
    assert rel_l2(got[xs.astype(np.int64)], ref) <= STATE_TOL


def test_amplitudes_gather():
    from oracle.statevector import simulate_state
    tn = _tn()
    c = C.grid(4, 4, 8, 11)
    ref = simulate_state(c)
    ctr = tn.Contractor(c, target=tn.TARGET_AMPLITUDES)
    xs = C.random_bitstrings(16, 300, 9)
    got = ctr.amplitudes(torch.as_tensor(xs.astype(np.int64), device="cuda")).cpu().numpy()[0]
    assert rel_l2(got, ref[xs.astype(np.int64)]) <= STATE_TOL
    # empty batch of bitstrings is a no-op
    ctr.amplitudes(torch.empty(0, dtype=torch.int64, device="cuda"))
    torch.cuda.synchronize()


def test_empty_circuit_and_basis():
    c = C.Circuit(7, [], init_basis=93)
    got = gpu_state(c)[0]
    ref = np.zeros(128, dtype=np.complex128)
    ref[93] = 1
    assert np.abs(got - ref).max() == 0


def test_invalid_arguments_rejected():
    tn = _tn()
    with pytest.raises(tn.TnError):
        tn.CircuitHandle(C.Circuit(3, [C.Gate("H", (3,))]))
    with pytest.raises(tn.TnError):
        tn.CircuitHandle(C.Circuit(3, [C.Gate("CZ", (1, 1))]))
    with pytest.raises(tn.TnError):
        tn.CircuitHandle(C.Circuit(3, [], init_basis=8))
    ctr = tn.Contractor(C.brickwork(6, 2, 1, parameterized=True)[0])
    with pytest.raises(tn.TnError):
        ctr.state(None)  # parameterised circuit without parameters


@pytest.mark.parametrize("n,k", [(2, 14), (6, 2), (14, 8), (20, 14)])
def test_fig31_sweep_points(n, k):
    """Points of the paper-shaped sweep (Fig. 3.1 circuits) against the FP64 oracle."""
    from oracle.statevector import simulate_state
    from paper_2108_06831_gb300 import tn
    c = C.paper_fig31(n, k, 6000 + n + k)
    ctr = tn.Contractor(c)
    out = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    tn.contract_state(ctr.plan, None, out, ctr.workspace)
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    ref = simulate_state(c)
    got = out.cpu().numpy().astype(np.complex128)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5


def test_fig31_largest_point_against_stored_oracle():
    """n = 28, k = 14 (2 GiB state), the largest point of the Fig. 3.1 grid, in the bench's
    launch configuration: 8 amplitudes against the oracle's FP64 greedy network contraction
    (stored: ~1 min and 9 GB of host memory per amplitude), plus the norm."""
    import os
    from paper_2108_06831_gb300 import tn
    c = C.paper_fig31(28, 14, 6042)
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "oracle_fig31_n28_k14_s6042.txt")
    rows = [l.split() for l in open(path) if l.strip() and not l.startswith("#")]
    xs = np.array([int(r[0]) for r in rows], dtype=np.int64)
    ref = np.array([complex(float(r[1]), float(r[2])) for r in rows])
    assert np.array_equal(xs.astype(np.uint64), C.random_bitstrings(28, 8, 6242))
    a = tn.Contractor(c)
    x = torch.empty(1 << 28, dtype=torch.complex64, device="cuda")
    tn.contract_state(a.plan, None, x, a.workspace)
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    nx = torch.linalg.vector_norm(x.to(torch.complex128)).item()
    assert abs(nx - 1.0) <= 1e-5
    got = x[torch.as_tensor(xs, device="cuda")].cpu().numpy()
    # amplitudes of a 2^28-entry state are ~2^-14: compare them against the state's RMS scale
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err <= 1e-5, err


def test_max_size_32_qubits_closed_form():
    """32 qubits (a 32 GiB complex64 state): U3 on every qubit, then CZ on every neighbour pair.
    Every amplitude has a closed form, amp(x) = prod_q (U3_q|0>)[x_q] * (-1)^(sum_q x_q x_{q+1}),
    evaluated in FP64 on 4096 sampled indices."""
    from oracle.gates import matrix
    from paper_2108_06831_gb300 import tn
    n = 32
    rng = np.random.default_rng(3232)
    angles = rng.uniform(0.0, 2.0 * np.pi, size=(n, 3))
    gates = [C.Gate("U3", (q,), tuple(float(a) for a in angles[q])) for q in range(n)]
    gates += [C.Gate("CZ", (q, q + 1)) for q in range(n - 1)]
    c = C.Circuit(n, gates)
    ctr = tn.Contractor(c)
    out = torch.empty((1, 1 << n), dtype=torch.complex64, device="cuda")
    tn.contract_state(ctr.plan, None, out, ctr.workspace)
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    xs = rng.integers(0, 1 << n, size=4096, dtype=np.int64)
    got = out[0, torch.as_tensor(xs, device="cuda")].cpu().numpy().astype(np.complex128)
    col = np.array([matrix("U3", tuple(angles[q]))[:, 0] for q in range(n)])  # U3_q |0>
    bits = (xs[:, None] >> (n - 1 - np.arange(n))[None, :]) & 1  # bit of qubit q (MSB first)
    ref = np.prod(col[np.arange(n)[None, :], bits], axis=1)
    ref = ref * (-1.0) ** np.sum(bits[:, :-1] * bits[:, 1:], axis=1)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= STATE_TOL


def test_tile_autotuner_single_plan():
    """tn_plan_contraction_tuned: the circuit planned at each candidate tile size, each plan's
    contraction timed, the fastest returned; its tile is a candidate and its state matches the
    oracle (parameterised circuit, batch of 2)."""
    from oracle.statevector import simulate_state
    tn = _tn()
    c, p0 = C.brickwork(16, 10, 91, parameterized=True)
    params = np.stack([p0, np.random.default_rng(92).uniform(0, 2 * np.pi, size=p0.shape)])
    ctr = tn.Contractor(c, batch=2, tune={"candidates": (8, 10, 12), "reps": 2})
    assert ctr.plan.tuned_tile in (8, 10, 12)
    assert ctr.plan.stats()["tile_qubits"] == ctr.plan.tuned_tile
    got = ctr.state(torch.as_tensor(params, device="cuda")).cpu().numpy()
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    for b in range(2):
        assert rel_l2(got[b], simulate_state(c, params[b])) <= STATE_TOL
    with pytest.raises(tn.TnError):  # tile_qubits is the tuner's choice
        tn.Plan(tn.CircuitHandle(c), tile_qubits=10, tune={})


@pytest.mark.parametrize("n,depth,batch,parameterized", [
    (6, 5, 3, True), (8, 4, 1215, True), (9, 3, 1216, True), (12, 6, 2, True), (13, 4, 3, True), (14, 4, 2, True),
    (6, 8, 1, False), (12, 8, 1, False), (13, 6, 1, False), (16, 5, 1, False), (18, 4, 1, False)])
def test_small_states_take_few_amplitudes_per_thread(n, depth, batch, parameterized):
    """Plans of few warps run four (or eight) amplitudes per thread: one tile and several, either side of the
    rule's limits, tables staged and constant, the gate tables of few and of many slots; as amplitudes too."""
    from oracle.statevector import simulate_state
    tn = _tn()
    c, _ = C.brickwork(n, depth, 50 + n, parameterized=parameterized)
    c.init_basis = (n * 977) % (1 << n)
    params = np.random.default_rng(n).uniform(0, 2 * np.pi, size=(batch, c.n_params)) if parameterized else None
    got = gpu_state(c, params, batch=batch)
    xs = np.arange(0, 1 << n, 37)
    ctr = tn.Contractor(c, target=tn.TARGET_AMPLITUDES, batch=batch)
    p = None if params is None else torch.as_tensor(params, device="cuda")
    amps = ctr.amplitudes(torch.as_tensor(xs, device="cuda"), p).cpu().numpy()
    for b in sorted({0, batch // 2, batch - 1}):
        ref = simulate_state(c, None if params is None else params[b])
        assert rel_l2(got[b], ref) <= STATE_TOL
        assert rel_l2(amps[b], ref[xs]) <= STATE_TOL


@pytest.mark.parametrize("n,batch,parameterized", [(5, 1, False), (6, 1, True), (9, 1215, True), (9, 1216, True),
                                                   (13, 1, False), (14, 2, True), (18, 1, False), (19, 1, True)])
def test_host_only_plans_describe_the_plans_that_run(n, batch, parameterized):
    tn = _tn()
    ch = tn.CircuitHandle(C.brickwork(n, 6, n, parameterized=parameterized)[0])
    host, run = (tn.Plan(ch, batch=batch, host_only=h) for h in (True, False))
    differ = {k for k, v in run.stats().items() if host.stats()[k] != v}
    assert differ <= {"specialized"} and host.workspace_bytes == run.workspace_bytes


@pytest.mark.parametrize("parameterized", [False, True])
@pytest.mark.parametrize("n,tile", [(3, 0), (7, 0), (12, 0), (13, 6), (14, 8), (17, 12), (18, 0)])
def test_runs_of_diagonal_gates(n, tile, parameterized):
    """Runs of diagonal gates of every kind between mixing gates on single qubits: operands in the registers,
    in the tile and outside it, both operands of a pair anywhere, runs that end at a mix or at the phase."""
    from oracle.statevector import simulate_state
    rng = np.random.default_rng(31 * n + tile)
    gates, n_params = [C.Gate("H", (q,)) for q in range(n)], 0
    one, two = ["Z", "S", "SDG", "T", "TDG", "RZ"], ["CZ", "CP"]
    for _ in range(6):
        for _ in range(3 * n):
            if rng.uniform() < 0.6:
                kind = two[int(rng.integers(0, 2))]
                qs = tuple(int(q) for q in rng.choice(n, size=2, replace=False))
            else:
                kind, qs = one[int(rng.integers(0, len(one)))], (int(rng.integers(0, n)),)
            angles, at = (), -1
            if kind in ("RZ", "CP"):
                angles = (float(rng.uniform(0, 2 * np.pi)),)
                if parameterized:
                    at, n_params = n_params, n_params + 1
            gates.append(C.Gate(kind, qs, angles, at))
        for q in rng.choice(n, size=2, replace=False):  # one mixed, one mixed under a control
            gates.append(C.Gate("SX", (int(q),)))
        a, b = (int(q) for q in rng.choice(n, size=2, replace=False))
        gates.append(C.Gate("CNOT", (a, b)))
    c = C.Circuit(n, gates, n_params=n_params)
    batch = 2 if parameterized else 1
    params = rng.uniform(0, 2 * np.pi, size=(batch, n_params)) if parameterized else None
    got = gpu_state(c, params, batch=batch, tile=tile)
    for b in range(batch):
        assert rel_l2(got[b], simulate_state(c, None if params is None else params[b])) <= STATE_TOL


@pytest.mark.parametrize("n,tile", [(7, 0), (12, 0), (14, 8), (18, 0)])
def test_diagonal_gates_leave_what_their_condition_excludes(n, tile):
    """Amplitudes that a MAT1 drove to infinity stay infinite under phases and signs whose condition is false
    for them (no inf * 0), wherever the condition's bit lies; the others stay exact."""
    from oracle.statevector import simulate_state
    tn = _tn()
    big = float(2.0 ** 100)
    for q in (0, n // 2, n - 1):
        h = [C.Gate("H", (k,)) for k in range(n)]
        scale = [C.Gate("MAT1", (q,), mat=(big, 0, 0, 1))] * 2
        phases = [C.Gate(kind, (q,)) for kind in ("S", "T", "SDG", "TDG", "Z")]
        for k in range(n):
            if k != q:
                phases += [C.Gate("CP", (q, k), (0.1 + k,)), C.Gate("CZ", (k, q))]
        ctr = tn.Contractor(C.Circuit(n, h + scale + phases), tile_qubits=tile, fuse=False)
        got = ctr.state().cpu().numpy()[0].reshape(1 << q, 2, -1)
        ref = simulate_state(C.Circuit(n, h + phases)).reshape(1 << q, 2, -1)
        assert np.all(np.isposinf(got[:, 0].real)) and np.all(got[:, 0].imag == 0), q
        assert rel_l2(got[:, 1], ref[:, 1]) <= STATE_TOL, q


@pytest.mark.parametrize("n,tile,batch", [(18, 6, 1), (20, 7, 1), (19, 7, 1), (12, 6, 77), (17, 6, 2)])
def test_small_tiles_share_ctas(n, tile, batch):
    """CTAs of a few threads that take several tiles each: shares that divide the tiles and that do not, several
    batch elements (whose tables change within a CTA's share)."""
    from oracle.statevector import simulate_state
    c, _ = C.brickwork(n, 3, 60 + n, parameterized=batch > 1)
    c.init_basis = (n * 7919) % (1 << n)
    params = np.random.default_rng(n).uniform(0, 2 * np.pi, size=(batch, c.n_params)) if batch > 1 else None
    got = gpu_state(c, params, batch=batch, tile=tile)
    for b in sorted({0, batch // 2, batch - 1}):
        assert rel_l2(got[b], simulate_state(c, None if params is None else params[b])) <= STATE_TOL
