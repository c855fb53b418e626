"""Expectation values and adjoint gradients against the FP64 oracle (GPU).

Bars: |E - E_ref| <= 1e-4 max(1, |E_ref|); per parameter set
||g - g_ref|| / max(||g_ref||, 1e-3) <= 1e-4, with g_ref the oracle's parameter-shift
gradient (cross-checked there against finite differences).
"""
import numpy as np
import pytest

from paper_2108_06831_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _tn():
    from paper_2108_06831_gb300 import tn
    return tn


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("n,layers,tile", [(4, 2, 0), (8, 3, 0), (12, 2, 7), (14, 3, 9)])
def test_hea_tfim_expectation_and_gradient(n, layers, tile):
    from oracle import gradients as GR
    from oracle import observables as OB
    tn = _tn()
    c = C.hea(n, layers)
    H = C.tfim(n)
    batch = 3
    params = C.hea_params(c.n_params, batch, 40 + n)
    ctr = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=batch, tile_qubits=tile)
    obs = tn.Observable(H)
    E = ctr.expectation(obs, _dev(params)).cpu().numpy()
    G = ctr.expectation_backward(obs, _dev(params)).cpu().numpy()
    for b in range(batch):
        Eref = OB.expectation(c, H, params[b])
        assert abs(E[b] - Eref) <= 1e-4 * max(1.0, abs(Eref))
        gref = GR.param_shift_grad(c, H, params[b])
        assert np.linalg.norm(G[b] - gref) / max(np.linalg.norm(gref), 1e-3) <= 1e-4


@pytest.mark.parametrize("n,layers,tile,ham", [(6, 3, 0, "tfim"), (13, 2, 8, "tfim"), (11, 2, 8, "pauli")])
def test_value_and_grad_matches_separate_calls_and_oracle(n, layers, tile, ham):
    """tn_expectation_value_and_grad contracts the forward state once; energies and gradients
    equal the two-call path and the oracle (parameter shift).  Its energy is Re <psi|H psi> summed
    from lambda = H psi, the two-call path's the direct term sum: both in FP32 per amplitude, so they
    agree to FP32 rounding of the state's norm-sized sums, not bit for bit."""
    from oracle import gradients as GR
    from oracle import observables as OB
    tn = _tn()
    c = C.hea(n, layers)
    H = C.tfim(n) if ham == "tfim" else C.random_pauli_sum(n, 30, 90 + n)  # X, Y and Z factors
    batch = 2
    params = C.hea_params(c.n_params, batch, 70 + n)
    ctr = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=batch, tile_qubits=tile)
    obs = tn.Observable(H)
    e1, g1 = ctr.expectation_value_and_grad(obs, _dev(params))
    e0 = ctr.expectation(obs, _dev(params))
    g0 = ctr.expectation_backward(obs, _dev(params))
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    E, G = e1.cpu().numpy(), g1.cpu().numpy()
    assert np.allclose(E, e0.cpu().numpy(), rtol=1e-5, atol=1e-5)
    assert np.allclose(G, g0.cpu().numpy(), rtol=1e-9, atol=1e-12)
    for b in range(batch):
        Eref = OB.expectation(c, H, params[b])
        assert abs(E[b] - Eref) <= 1e-4 * max(1.0, abs(Eref))
        gref = GR.param_shift_grad(c, H, params[b])
        assert np.linalg.norm(G[b] - gref) / max(np.linalg.norm(gref), 1e-3) <= 1e-4


def test_theta_zero_energy_20q():
    tn = _tn()
    n = 20
    c = C.hea(n, 10)
    ctr = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=2)
    obs = tn.Observable(C.tfim(n))
    E = ctr.expectation(obs, _dev(np.zeros((2, c.n_params)))).cpu().numpy()
    assert np.abs(E + 19.0).max() <= 1e-4 * 19


def test_cfg4_full_size_sampled():
    """20-qubit HEA, 400 parameters, batch 64 (bench launch configuration); the oracle checks
    the energy of two batch elements and, by parameter shift, three sampled gradient entries
    (a full 400-parameter shift at 2^20 amplitudes would take the oracle minutes)."""
    from oracle import observables as OB
    from oracle.statevector import simulate_state
    tn = _tn()
    n, layers, batch = 20, 10, 64
    c = C.hea(n, layers)
    H = C.tfim(n)
    params = C.hea_params(c.n_params, batch, 4000)
    ctr = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=batch)
    obs = tn.Observable(H)
    E = ctr.expectation(obs, _dev(params)).cpu().numpy()
    G = ctr.expectation_backward(obs, _dev(params)).cpu().numpy()
    e2, g2 = ctr.expectation_value_and_grad(obs, _dev(params))  # the call the benchmark times
    E2, G2 = e2.cpu().numpy(), g2.cpu().numpy()
    assert np.allclose(G2, G, rtol=1e-9, atol=1e-12)
    rng = np.random.default_rng(1)
    for b in (0, 37):
        Eref = OB.expectation(c, H, params[b])
        assert abs(E[b] - Eref) <= 1e-4 * max(1.0, abs(Eref))
        assert abs(E2[b] - Eref) <= 1e-4 * max(1.0, abs(Eref))
    for b in (37,):
        ks = rng.choice(c.n_params, size=3, replace=False)
        for k in ks:
            gate_idx = [i for i, g in enumerate(c.gates) if g.param_idx == k]
            vals = []
            for sgn in (1, -1):
                ov = {gi: (params[b][k] + sgn * np.pi / 2,) for gi in gate_idx}
                vals.append(OB.expectation_of_state(simulate_state(c, params[b], ov), H))
            gk = 0.5 * (vals[0] - vals[1])
            assert abs(G[b, k] - gk) <= 1e-4 * max(np.linalg.norm(G[b]), 1e-3)


def test_random_pauli_sum_state_expectation():
    from oracle import observables as OB
    from oracle.statevector import simulate_state
    tn = _tn()
    n = 11
    c = C.random_circuit(n, 120, 3)
    H = C.random_pauli_sum(n, 25, 8)
    psi = simulate_state(c)
    ctr = tn.Contractor(c)
    st = ctr.state()
    obs = tn.Observable(H)
    ws_bytes = tn.state_expectation_workspace_bytes(obs, 1)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    tn.state_expectation(obs, 1, st, out, ws, ws_bytes)
    Eref = OB.expectation_of_state(psi, H)
    assert abs(out.item() - Eref) <= 1e-4 * max(1.0, abs(Eref))


def test_autograd_function():
    tn = _tn()
    from oracle import gradients as GR
    n = 6
    c = C.hea(n, 2)
    H = C.tfim(n)
    params = C.hea_params(c.n_params, 2, 9)
    ctr = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=2)
    obs = tn.Observable(H)
    th = torch.tensor(params, device="cuda", requires_grad=True)
    E = tn.expectation_autograd(th, ctr, obs)
    (E * torch.tensor([1.0, -2.0], device="cuda", dtype=torch.float64)).sum().backward()
    g = th.grad.cpu().numpy()
    for b, w in ((0, 1.0), (1, -2.0)):
        gref = w * GR.param_shift_grad(c, H, params[b])
        assert np.linalg.norm(g[b] - gref) / max(np.linalg.norm(gref), 1e-3) <= 1e-4


def _mixed_sum(n, n_terms, seed):
    """Random Pauli strings: dense ones up to 10 qubits, on three qubits beyond (their flips fit a tile);
    several terms share their flips, some have none."""
    rng = np.random.default_rng(seed)
    H = C.PauliSum(n)
    for k in range(n_terms):
        if n <= 10:
            s = "".join("IXYZ"[int(v)] for v in rng.integers(0, 4, size=n))
            H.coef.append(float(rng.normal()))
            H.strings.append(s)
            if k % 4 == 0:  # the same flips with other signs, and a Z string
                H.coef.append(float(rng.normal()))
                H.strings.append(s.translate(str.maketrans("XYIZ", "YXZI")))
                H.coef.append(float(rng.normal()))
                H.strings.append(s.translate(str.maketrans("XY", "ZI")))
        else:
            qs = rng.choice(n, size=3, replace=False)
            for ops in ("XYZ", "YXZ", "XXI", "YYI", "ZZZ", "IIY"):
                H.add(float(rng.normal()), [(int(q), p) for q, p in zip(qs, ops) if p != "I"])
    return H


@pytest.mark.parametrize("n", [1, 2, 4, 7, 8, 9, 10, 11, 12, 13, 16])
def test_pauli_sums_over_tile_sizes(n):
    """Tiles of every size (one row of fewer than 256 amplitudes up to 16 rows), flips on thread bits and
    on row bits, Z masks on both and outside the tile: the direct energy and the one summed from H psi,
    within the stated FP32 bound (terms + 16) 2^-24 sum |c| plus the state's own FP32 error."""
    from oracle import observables as OB
    tn = _tn()
    c = C.hea(n, 2)
    H = _mixed_sum(n, 12, 300 + n)
    batch = 2
    params = C.hea_params(c.n_params, batch, 20 + n)
    ctr = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=batch)
    obs = tn.Observable(H)
    e, _ = ctr.expectation_value_and_grad(obs, _dev(params))
    direct = ctr.expectation(obs, _dev(params)).cpu().numpy()
    bound = (len(H.coef) + 16 + len(c.gates)) * 2.0 ** -24 * float(np.abs(H.coef).sum())
    for b in range(batch):
        ref = OB.expectation(c, H, params[b])
        assert abs(direct[b] - ref) <= bound
        assert abs(e[b].item() - ref) <= bound


@pytest.mark.parametrize("n,tile", [(2, 0), (5, 0), (8, 0), (9, 6), (10, 7), (11, 8)])
def test_gradients_of_every_parameterised_gate(n, tile):
    """Gates of one, two-qubit and three angles in mixed order on every qubit: the dots of a phase come in
    groups of every size, first and last phases with and without the tile's lowest bits in the registers."""
    from oracle import gradients as GR
    from oracle import observables as OB
    tn = _tn()
    rng = np.random.default_rng(17 * n + tile)
    gates, at = [], 0
    for _ in range(5 * n):
        kind = ["RX", "RY", "RZ", "U3", "U3", "CP", "CZ", "CNOT"][int(rng.integers(0, 8))]
        arity, angles = C.GATE_ARITY[kind]
        qs = tuple(int(q) for q in rng.choice(n, size=arity, replace=False))
        gates.append(C.Gate(kind, qs, (0.0,) * angles, at if angles else -1))
        at += angles
    c = C.Circuit(n, gates, n_params=at)
    H = C.random_pauli_sum(n, 12, 5 + n)
    params = rng.uniform(0, 2 * np.pi, size=(2, at))
    ctr = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=2, tile_qubits=tile)
    E, G = ctr.expectation_value_and_grad(tn.Observable(H), _dev(params))
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    for b in range(2):
        Eref = OB.expectation(c, H, params[b])
        assert abs(float(E[b]) - Eref) <= 1e-4 * max(1.0, abs(Eref))
        gref = GR.param_shift_grad(c, H, params[b])
        assert np.linalg.norm(G[b].cpu().numpy() - gref) / max(np.linalg.norm(gref), 1e-3) <= 1e-4


@pytest.mark.parametrize("n,tile", [(3, 0), (6, 0), (9, 6), (11, 7), (12, 8)])
def test_register_permutations_among_mixing_gates(n, tile):
    """CNOT, SWAP and X runs between diagonal, mixing and parameterised gates: controls in the registers, in the
    tile and outside it, exchanges that reach a phase's loads or stores and ones that a gate in between stops."""
    from oracle import gradients as GR
    from oracle import observables as OB
    from oracle.statevector import simulate_state
    tn = _tn()
    rng = np.random.default_rng(131 * n + tile)
    gates, at = [], 0
    for _ in range(14 * n):
        kind = ["CNOT", "CNOT", "CNOT", "SWAP", "X", "H", "RZ", "RY", "CZ", "T", "CP", "SX"][int(rng.integers(0, 12))]
        arity, angles = C.GATE_ARITY[kind]
        qs = tuple(int(q) for q in rng.choice(n, size=arity, replace=False))
        free = angles and rng.uniform() < 0.3
        gates.append(C.Gate(kind, qs, tuple(float(x) for x in rng.uniform(0, 2 * np.pi, size=angles)), at if free else -1))
        at += angles if free else 0
    c = C.Circuit(n, gates, n_params=at)
    H = C.random_pauli_sum(n, 9, 3 + n)
    params = rng.uniform(0, 2 * np.pi, size=(2, at))
    psi = tn.Contractor(c, target=tn.TARGET_STATE, batch=2, tile_qubits=tile).state(_dev(params)).cpu().numpy()
    E, G = tn.Contractor(c, target=tn.TARGET_EXPECTATION, batch=2, tile_qubits=tile).expectation_value_and_grad(
        tn.Observable(H), _dev(params))
    torch.cuda.synchronize()
    assert tn.sync_status() == tn.OK
    for b in range(2):
        ref = simulate_state(c, params[b])
        assert np.linalg.norm(psi[b] - ref) / np.linalg.norm(ref) <= 1e-5
        Eref = OB.expectation(c, H, params[b])
        assert abs(float(E[b]) - Eref) <= 1e-4 * max(1.0, abs(Eref))
        gref = GR.param_shift_grad(c, H, params[b])
        assert np.linalg.norm(G[b].cpu().numpy() - gref) / max(np.linalg.norm(gref), 1e-3) <= 1e-4
