"""What is timed when this framework is made faster: its public calls, over the sizes users bring.

Every case is one call (or the few calls) a user's program makes through
``paper_2108_06831_gb300.tn`` on inputs it already holds on the device, with the plan,
observable and workspace such a program keeps.  The structure of a case (gates, legs,
shapes) comes from the case alone, its numbers (angles, matrices, bitstrings, operands)
from the seed.  ``exact`` evaluates the same inputs with plain torch in complex128.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2108_06831_gb300 import circuits as C
from paper_2108_06831_gb300 import tn

DEV = "cuda"


def listed():
    return [
        # one small circuit for one parameter set: the shortest call there is
        {"name": "state_9q_one", "kind": "state", "family": "brickwork", "n": 9, "depth": 6, "batch": 1},
        # many parameter sets of a small circuit in one call (a parameter scan)
        {"name": "state_10q_512sets", "kind": "state", "family": "brickwork", "n": 10, "depth": 8, "batch": 512},
        # the headline workload: a 24-qubit brickwork's full state vector
        {"name": "state_24q", "kind": "state", "family": "brickwork", "n": 24, "depth": 20, "batch": 1},
        # one training step of a variational circuit: energies and gradients of 64 parameter sets
        {"name": "grad_20q_64sets", "kind": "grad", "n": 20, "layers": 10, "batch": 64, "model": "tfim"},
        # energies alone (a line search, a measurement), a Hamiltonian with several flip patterns
        {"name": "energy_22q_4sets", "kind": "energy", "n": 22, "layers": 4, "batch": 4, "model": "heisenberg"},
        # a server's batch of circuits of uneven width and depth in one call
        {"name": "serving_128", "kind": "serving", "count": 128, "n_min": 8, "n_max": 22, "d_max": 30, "mix": 5000},
        # amplitudes by network contraction at the default precision
        {"name": "amps_grid5x5_fp32", "kind": "amps", "rows": 5, "cols": 5, "depth": 12, "bits": 64, "prec": 0},
        # amplitudes of a circuit too wide for a state vector, merges on the tensor cores
        {"name": "amps_grid6x6_3xtf32", "kind": "amps", "rows": 6, "cols": 6, "depth": 12, "bits": 64, "prec": 1},
        # one large complex matrix product on the tensor cores
        {"name": "gemm_4096_3xtf32", "kind": "gemm", "batch": 1, "m": 4096, "nn": 4096, "k": 4096, "prec": 1},
        # a batch of complex matrix products of odd sizes in plain FP32
        {"name": "gemm_ragged_fp32", "kind": "gemm", "batch": 3, "m": 1999, "nn": 1023, "k": 777, "prec": 0},
        # regrouping the legs of a large tensor
        {"name": "permute_27legs", "kind": "permute", "n": 27, "batch": 1, "perm": 11},
        # the fixed-point emulation of the paper's datapath on the headline circuit
        {"name": "q428_24q", "kind": "q428", "family": "brickwork", "n": 24, "depth": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["state", "state", "grad", "energy", "serving", "amps", "gemm", "gemm", "permute", "q428"])
    if kind == "state":
        n = rng.randint(6, 24)
        family = rng.choice(["brickwork", "brickwork", "fig31", "qft"])
        batch = _log_int(rng, 1, max(1, min(512, 1 << (23 - n)))) if n <= 22 and family == "brickwork" else 1
        return {"kind": kind, "family": family, "n": n, "depth": rng.randint(2, 16), "batch": batch}
    if kind == "grad":
        n = rng.randint(6, 18)
        return {"kind": kind, "n": n, "layers": rng.randint(2, 8), "batch": _log_int(rng, 1, min(64, 1 << (23 - n))),
                "model": rng.choice(["tfim", "heisenberg"])}
    if kind == "energy":
        n = rng.randint(6, 23)
        return {"kind": kind, "n": n, "layers": rng.randint(2, 6), "batch": _log_int(rng, 1, min(64, 1 << (24 - n))),
                "model": rng.choice(["tfim", "heisenberg"])}
    if kind == "serving":
        return {"kind": kind, "count": _log_int(rng, 8, 96), "n_min": 8, "n_max": rng.randint(12, 21),
                "d_max": rng.randint(8, 24), "mix": rng.randint(1, 9999)}
    if kind == "amps":
        return {"kind": kind, "rows": rng.randint(3, 5), "cols": rng.randint(4, 6), "depth": rng.randint(6, 12),
                "bits": 1 << rng.randint(0, 6), "prec": rng.randint(0, 2)}
    if kind == "gemm":
        prec = rng.randint(0, 2)
        if prec == 0:
            m, nn, k = (_log_int(rng, 16, 2048) for _ in range(3))
        else:  # the tensor-core tiles: rows in 128s, columns in 64s, 16-byte operand rows
            m, nn, k = 128 * _log_int(rng, 1, 32), 64 * _log_int(rng, 1, 64), 4 * _log_int(rng, 4, 1024)
        most = max(1, min(64, (1 << 33) // (m * nn * k + 1), (1 << 27) // (m * nn + m * k + nn * k)))
        return {"kind": kind, "batch": _log_int(rng, 1, most), "m": m, "nn": nn, "k": k, "prec": prec}
    if kind == "permute":
        n = rng.randint(8, 27)
        return {"kind": kind, "n": n, "batch": _log_int(rng, 1, min(16, 1 << (27 - n))), "perm": rng.randint(1, 9999)}
    return {"kind": "q428", "family": rng.choice(["brickwork", "fig31", "qft"]), "n": rng.randint(6, 23),
            "depth": rng.randint(2, 16)}


# ------------------------------------------------------------------ inputs

def _state_circuit(case, seed):
    """(circuit, number of parameters): brickwork angles are parameters, the other families' fixed."""
    n, depth = case["n"], case["depth"]
    if case["family"] == "brickwork":
        return C.brickwork(n, depth, seed, parameterized=case["kind"] == "state")[0]
    if case["family"] == "qft":
        return C.qft(n, C.random_basis(n, seed))
    return C.paper_fig31(n, max(1, depth // 2), seed)


def _params(batch, count, seed):
    return torch.from_numpy(np.random.default_rng(seed).uniform(0.0, 2.0 * math.pi, size=(batch, count)))


def _hamiltonian(case, seed):
    n, rng = case["n"], np.random.default_rng(seed + 77)
    H = C.PauliSum(n)
    j, h = rng.uniform(0.5, 1.5, size=2)
    if case["model"] == "tfim":
        return C.tfim(n, float(j), float(h))
    for i in range(n - 1):
        for p in "XYZ":
            H.add(float(j), [(i, p), (i + 1, p)])
    for i in range(n):
        H.add(float(h), [(i, "Z")])
    return H


def _serving(case, seed):
    """(circuits, parameters of all of them back to back): widths and depths from the case, angles
    and the transforms' basis states from the seed."""
    circs, _ = C.serving_mix_params(case["count"], case["mix"], n_min=case["n_min"], n_max=case["n_max"], d_max=case["d_max"])
    rng = np.random.default_rng(seed)
    for c in circs:
        if c.n_params == 0:
            c.init_basis = int(rng.integers(0, 1 << c.n_qubits))
    return circs, torch.from_numpy(rng.uniform(0.0, 2.0 * math.pi, size=sum(c.n_params for c in circs)))


def _grid_bits(case, seed):
    n = case["rows"] * case["cols"]
    return C.grid(case["rows"], case["cols"], case["depth"], seed), C.random_bitstrings(n, case["bits"], seed + 1)


def _operands(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)

    def normal(*shape):
        return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV))

    if case["kind"] == "permute":
        return normal(case["batch"], 1 << case["n"])
    return normal(case["batch"], case["m"], case["k"]), normal(case["batch"], case["nn"], case["k"])


def _perm(case):
    return [int(v) for v in np.random.default_rng(case["perm"]).permutation(case["n"])]


def _workspace(nbytes):
    return torch.empty(max(int(nbytes), 16), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "state":
        circ = _state_circuit(case, seed)
        ctr = tn.Contractor(circ, batch=case["batch"])
        params = _params(case["batch"], circ.n_params, seed).to(DEV) if circ.n_params else None
        out = torch.empty((case["batch"], 1 << case["n"]), dtype=torch.complex64, device=DEV)
        return {"kind": kind, "ctr": ctr, "params": params, "out": out}
    if kind in ("grad", "energy"):
        circ = C.hea(case["n"], case["layers"])
        ctr = tn.Contractor(circ, target=tn.TARGET_EXPECTATION, batch=case["batch"])
        return {"kind": kind, "ctr": ctr, "obs": tn.Observable(_hamiltonian(case, seed)),
                "params": _params(case["batch"], circ.n_params, seed).to(DEV)}
    if kind == "serving":
        circs, params = _serving(case, seed)
        # generated kernels where the batch runs them (wide circuits), the shared executor for the rest
        batch = tn.Batch([tn.Plan(tn.CircuitHandle(c), specialize=c.n_qubits >= 19) for c in circs])
        return {"kind": kind, "batch": batch, "params": params.to(DEV), "ws": _workspace(batch.workspace_bytes),
                "out": torch.empty(batch.state_elems, dtype=torch.complex64, device=DEV)}
    if kind == "amps":
        circ, bits = _grid_bits(case, seed)
        plan = tn.Plan(tn.CircuitHandle(circ), target=tn.TARGET_AMPLITUDES, precision=case["prec"],
                       network_bitstrings=case["bits"])
        return {"kind": kind, "plan": plan, "bits": torch.from_numpy(bits.astype(np.int64)).to(DEV),
                "ws": _workspace(plan.workspace_bytes),
                "out": torch.empty((1, case["bits"]), dtype=torch.complex64, device=DEV)}
    if kind == "gemm":
        a, b = _operands(case, seed)
        nbytes = tn.cgemm_workspace_bytes(case["prec"], case["batch"], case["m"], case["nn"], case["k"])
        return {"kind": kind, "case": dict(case), "a": a, "b": b, "ws": _workspace(nbytes), "nbytes": nbytes,
                "out": torch.empty((case["batch"], case["m"], case["nn"]), dtype=torch.complex64, device=DEV)}
    if kind == "permute":
        x = _operands(case, seed)
        return {"kind": kind, "n": case["n"], "batch": case["batch"], "perm": _perm(case), "x": x, "out": torch.empty_like(x)}
    plan = tn.Plan(tn.CircuitHandle(_state_circuit(case, seed)), q428=True)
    return {"kind": kind, "plan": plan, "out": torch.empty((1 << case["n"], 2), dtype=torch.int32, device=DEV)}


def run(s):
    kind = s["kind"]
    if kind == "state":
        return s["ctr"].state(s["params"], out=s["out"])
    if kind == "grad":
        return s["ctr"].expectation_value_and_grad(s["obs"], s["params"])
    if kind == "energy":
        return s["ctr"].expectation(s["obs"], s["params"])
    if kind == "serving":
        tn.batch_run(s["batch"], s["out"], s["ws"], params=s["params"])
    elif kind == "amps":
        tn.contract_amplitudes(s["plan"], None, s["bits"], s["out"], s["ws"])
    elif kind == "gemm":
        c = s["case"]
        tn.cgemm_batched(c["prec"], c["batch"], c["m"], c["nn"], c["k"], s["a"], s["b"], s["out"], s["ws"], s["nbytes"])
    elif kind == "permute":
        tn.permute(s["n"], s["perm"], s["batch"], s["x"], s["out"])
    else:
        tn.contract_state_q428(s["plan"], s["out"])
    return s["out"]


# ------------------------------------------------------------------ what a pass cannot do without

# real operations per amplitude of one gate (a U3 up to a phase, rotations with real or imaginary
# entries; sign flips and exchanges none)
_GATE_FLOPS = {"U3": 10, "RX": 6, "RY": 6, "H": 6, "SX": 6, "SY": 6, "SW": 10, "RZ": 6, "CP": 1.5}


def _circuit_flops(circ):
    return sum(_GATE_FLOPS.get(g.kind, 0) for g in circ.gates) * 2.0 ** circ.n_qubits


def work(case):
    kind = case["kind"]
    if kind in ("state", "q428"):
        circ = _state_circuit(case, 1)
        batch = case.get("batch", 1)
        return {"bytes": 8.0 * batch * (2.0 ** case["n"] + circ.n_params), "flops": batch * _circuit_flops(circ)}
    if kind in ("grad", "energy"):
        circ = C.hea(case["n"], case["layers"])
        terms, amps, batch = len(_hamiltonian(case, 1).coef), 2.0 ** case["n"], case["batch"]
        flops = _circuit_flops(circ) + 4.0 * terms * amps
        if kind == "grad":  # both states swept back, one overlap per parameter
            flops += 2.0 * _circuit_flops(circ) + 4.0 * circ.n_params * amps
        return {"bytes": 8.0 * batch * (circ.n_params * (2 if kind == "grad" else 1) + 1), "flops": batch * flops}
    if kind == "serving":
        circs, _ = _serving(case, 1)
        return {"bytes": sum(8.0 * (2.0 ** c.n_qubits + c.n_params) for c in circs),
                "flops": sum(_circuit_flops(c) for c in circs)}
    if kind == "amps":
        # an estimate: a frontier across the grid's shorter side (a bond per coupled pair and period of
        # the four edge patterns), extended over the rest of the network for every bitstring
        cut = min(case["rows"], case["cols"]) * max(1, case["depth"] // 4)
        return {"bytes": 16.0 * case["bits"], "flops": 8.0 * case["bits"] * 2.0 ** (cut + 12)}
    if kind == "gemm":
        m, nn, k = case["m"], case["nn"], case["k"]
        return {"bytes": 8.0 * case["batch"] * (m * k + nn * k + m * nn), "flops": 8.0 * case["batch"] * m * nn * k}
    return {"bytes": 16.0 * case["batch"] * 2.0 ** case["n"], "flops": 0.0}


# ------------------------------------------------------------------ the same in 64 bits, plain torch

def _matrix(kind, a):
    """2x2 matrix of a one-qubit gate, entries numpy arrays over the parameter sets."""
    one, r2 = np.ones_like(a[0]) if a else np.ones(1), math.sqrt(0.5)
    if kind == "SX":
        kind, a = "RX", [one * math.pi / 2]
    if kind == "SY":
        kind, a = "RY", [one * math.pi / 2]
    if kind == "H":
        return r2 * one, r2 * one, r2 * one, -r2 * one
    if kind == "SW":
        return r2 * one, (-0.5 - 0.5j) * one, (0.5 - 0.5j) * one, r2 * one
    c, s = np.cos(a[0] / 2), np.sin(a[0] / 2)
    if kind == "RX":
        return c, -1j * s, -1j * s, c
    if kind == "RY":
        return c, -s, s, c
    if kind == "RZ":
        return c - 1j * s, 0 * c, 0 * c, c + 1j * s
    assert kind == "U3", kind
    return c, -np.exp(1j * a[2]) * s, np.exp(1j * a[1]) * s, np.exp(1j * (a[1] + a[2])) * c


def _angles(g, params):
    """Angles of a gate: arrays over the parameter sets (one entry where the gate's are fixed)."""
    if g.param_idx >= 0:
        return [params[:, g.param_idx + i] for i in range(g.n_angles)]
    return [np.full(1, v) for v in g.angles]


def _gate(psi, n, g, a, inverse=False):
    """One gate applied in place to psi [sets, 2^n] (complex128); a: its angles."""
    sets = psi.shape[0]
    if g.kind in ("CZ", "CP", "CNOT", "SWAP"):
        p, q = g.qubits
        lo, hi = min(p, q), max(p, q)
        v = psi.view(sets, 1 << lo, 2, 1 << (hi - lo - 1), 2, 1 << (n - 1 - hi))
        if g.kind == "CZ":
            v[:, :, 1, :, 1] *= -1
        elif g.kind == "CP":
            v[:, :, 1, :, 1] *= complex(np.exp((-1j if inverse else 1j) * a[0][0]))
        else:
            if g.kind == "SWAP":
                x, y = v[:, :, 0, :, 1], v[:, :, 1, :, 0]
            else:
                x, y = (v[:, :, 1, :, 0], v[:, :, 1, :, 1]) if p < q else (v[:, :, 0, :, 1], v[:, :, 1, :, 1])
            t = x.clone()
            x.copy_(y)
            y.copy_(t)
        return
    m = _matrix(g.kind, a)
    if inverse:
        m = (np.conj(m[0]), np.conj(m[2]), np.conj(m[1]), np.conj(m[3]))
    u = [torch.from_numpy(np.asarray(e, dtype=np.complex128)).to(psi.device).view(-1, 1, 1) for e in m]
    q = g.qubits[0]
    v = psi.view(sets, 1 << q, 2, 1 << (n - 1 - q))
    if g.kind == "RZ":
        v[:, :, 0] *= u[0]
        v[:, :, 1] *= u[3]
        return
    x, y = v[:, :, 0], v[:, :, 1]
    nx = u[0] * x
    nx += u[1] * y
    y *= u[3]
    y += u[2] * x
    x.copy_(nx)


def _exact_state(circ, params):
    sets = params.shape[0] if circ.n_params else 1
    psi = torch.zeros((sets, 1 << circ.n_qubits), dtype=torch.complex128, device=DEV)
    psi[:, circ.init_basis] = 1
    for g in circ.gates:
        _gate(psi, circ.n_qubits, g, _angles(g, params))
    return psi


def _pauli_sum(psi, n, H):
    """H psi."""
    out = torch.zeros_like(psi)
    x = torch.arange(1 << n, device=psi.device)
    diag = torch.zeros(1 << n, dtype=torch.float64, device=psi.device)
    for c, s in zip(H.coef, H.strings):
        sign = torch.full_like(diag, c)
        flip, ny = 0, 0
        for q, p in enumerate(s):
            bit = n - 1 - q
            if p in "YZ":
                sign *= 1.0 - 2.0 * ((x >> bit) & 1)
            if p in "XY":
                flip |= 1 << bit
            ny += p == "Y"
        if flip == 0:
            diag += sign
        else:  # P|x> = i^ny (-1)^(x . z) |x ^ flip>
            at = x ^ flip
            out += (1j ** ny) * (sign * psi)[:, at]
    return out.addcmul_(diag.to(psi.dtype).expand_as(psi), psi)


def _exact_energy(case, seed, grad):
    circ, H, n = C.hea(case["n"], case["layers"]), _hamiltonian(case, seed), case["n"]
    params = _params(case["batch"], circ.n_params, seed).numpy()
    energies, grads = [], []
    per = max(1, (1 << 24) >> n)  # parameter sets at a time
    for b0 in range(0, case["batch"], per):
        p = params[b0:b0 + per]
        psi = _exact_state(circ, p)
        lam = _pauli_sum(psi, n, H)
        energies.append(torch.linalg.vecdot(psi, lam).real)
        if not grad:
            continue
        out = torch.zeros(p.shape, dtype=torch.float64, device=DEV)
        for g in reversed(circ.gates):
            a = _angles(g, p)
            if g.param_idx >= 0:  # d/dt exp(-i t P / 2): 2 Re <lam| (-i/2) P |psi> = Im <lam| P |psi>
                q = g.qubits[0]
                v, l = (t.view(p.shape[0], 1 << q, 2, 1 << (n - 1 - q)) for t in (psi, lam))

                def dot(i, j):
                    return (l[:, :, i].conj() * v[:, :, j]).sum(dim=(1, 2))

                over = dot(0, 0) - dot(1, 1) if g.kind == "RZ" else 1j * (dot(1, 0) - dot(0, 1))
                out[:, g.param_idx] = over.imag
            _gate(psi, n, g, a, inverse=True)
            _gate(lam, n, g, a, inverse=True)
        grads.append(out)
    e = torch.cat(energies)
    return (e, torch.cat(grads)) if grad else e


def exact(case, seed):
    kind = case["kind"]
    if kind == "state":
        circ = _state_circuit(case, seed)
        return _exact_state(circ, _params(case["batch"], circ.n_params, seed).numpy())
    if kind in ("grad", "energy"):
        return _exact_energy(case, seed, kind == "grad")
    if kind == "serving":
        circs, params = _serving(case, seed)
        out, at = [], 0
        for c in circs:
            out.append(_exact_state(c, params[None, at:at + c.n_params].numpy()).reshape(-1))
            at += c.n_params
        return torch.cat(out)
    if kind == "amps":
        circ, bits = _grid_bits(case, seed)
        if circ.n_qubits > 30:
            return None
        return _exact_state(circ, np.zeros((1, 0)))[:, torch.from_numpy(bits.astype(np.int64)).to(DEV)]
    if kind == "gemm":
        a, b = _operands(case, seed)
        return torch.matmul(a.to(torch.complex128), b.to(torch.complex128).transpose(1, 2))
    if kind == "permute":
        n, perm = case["n"], _perm(case)
        y = torch.arange(1 << n, device=DEV)
        x = torch.zeros_like(y)
        for j, p in enumerate(perm):  # output leg j holds input leg p (first leg most significant)
            x |= ((y >> (n - 1 - j)) & 1) << (n - 1 - p)
        return _operands(case, seed).to(torch.complex128)[:, x]
    return None  # whole numbers
