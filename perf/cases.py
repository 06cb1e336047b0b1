"""Performance cases of the state-vector framework: whole calls through its
public entry points, over the range of sizes a user brings.

A case names a ``family`` (what the user does) and its sizes:

  ansatz      the 12-qubit class of small complex128 circuits, run and read out
  ladder      a serving request: U3 layers and CNOT ladders on a middle-sized state
  layered     the fused layered circuit, U3 on every qubit and CZ on neighbours
  random      Haar-random one- and two-qubit matrices on random qubits
  packed      many small independent circuits in one call
  adjoint     values and gradients of a hardware-efficient ansatz, a batch of parameter vectors
  batchlayer  the torch layer inside a training step, forward and backward
  expect      a Hamiltonian of Pauli strings on a finished state
  sample      finite shots from a finished state
  readout     per-qubit <Z> and the probability vector of a finished state

Complex64 is the bulk precision of the framework and complex128 its exact mode.
"""

import math
from collections import namedtuple

import numpy as np
import torch

import paper_2608_09733_gb300 as sv

Gate = namedtuple("Gate", "name targets controls control_states params slots matrix")
Term = namedtuple("Term", "paulis qubits coeff")

TORCH_DTYPE = {"c64": torch.complex64, "c128": torch.complex128}
SV_DTYPE = {"c64": sv.SV_C64, "c128": sv.SV_C128}
AMP_BYTES = {"c64": 8, "c128": 16}


def gate(name, targets, controls=(), params=(), slots=None, matrix=None):
    return Gate(name, list(targets), list(controls), [1] * len(controls), [float(p) for p in params],
                list(slots) if slots is not None else [-1] * len(params), matrix)


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest thing a user runs: a 12-qubit ansatz in double precision, one circuit at a time
        {"name": "ansatz_12q_c128", "family": "ansatz", "n": 12, "layers": 10, "dtype": "c128"},
        # one serving request of the middle of the stream's range (8 to 26 qubits, depth 5 to 40)
        {"name": "ladder_17q_c64", "family": "ladder", "n": 17, "depth": 22, "dtype": "c64"},
        # the layered benchmark circuit on a state that fits a few times into L2 ...
        {"name": "layered_24q_c64", "family": "layered", "n": 24, "layers": 20, "dtype": "c64"},
        # ... and on the 8 GiB state of the headline figure
        {"name": "layered_30q_c64", "family": "layered", "n": 30, "layers": 20, "dtype": "c64"},
        # the exact mode on the precision sweep's circuit
        {"name": "random_24q_c128", "family": "random", "n": 24, "n1": 400, "n2": 200, "dtype": "c128"},
        # small serving requests, packed into one call
        {"name": "packed_256_c64", "family": "packed", "requests": 256, "dtype": "c64"},
        # variational training: 400 parameters, 64 parameter vectors a step
        {"name": "adjoint_20q_b64_c64", "family": "adjoint", "n": 20, "layers": 10, "batch": 64, "dtype": "c64"},
        # a quantum layer in a classifier, a batch of 256 input rows
        {"name": "batchlayer_16q_b256_c64", "family": "batchlayer", "n": 16, "layers": 4, "batch": 256, "dtype": "c64"},
        # energy of a ring model (ZZ on neighbours, X on every site)
        {"name": "expect_ring_24q_c64", "family": "expect", "n": 24, "terms": "ring", "count": 48, "dtype": "c64"},
        # energy of a molecule-like sum of strings with X, Y and Z, in the exact mode
        {"name": "expect_strings_21q_c128", "family": "expect", "n": 21, "terms": "strings", "count": 96, "dtype": "c128"},
        # a million shots
        {"name": "sample_28q_c64", "family": "sample", "n": 28, "shots": 1 << 20, "dtype": "c64"},
        # marginals and distribution of a finished state
        {"name": "readout_26q_c64", "family": "readout", "n": 26, "dtype": "c64"},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["ansatz", "ladder", "layered", "random", "packed", "adjoint", "batchlayer", "expect",
                         "sample", "readout"])
    either = rng.choice(["c64", "c128"])
    if family == "ansatz":
        return {"family": family, "n": rng.randint(6, 16), "layers": rng.randint(2, 20), "dtype": "c128"}
    if family == "ladder":
        return {"family": family, "n": rng.randint(13, 23), "depth": rng.randint(5, 40), "dtype": "c64"}
    if family == "layered":
        return {"family": family, "n": rng.randint(14, 28 if either == "c64" else 24), "layers": rng.randint(4, 20),
                "dtype": either}
    if family == "random":
        n1 = log_int(40, 400)
        return {"family": family, "n": rng.randint(10, 24), "n1": n1, "n2": n1 // 2, "dtype": either}
    if family == "packed":
        return {"family": family, "requests": log_int(3, 600), "dtype": "c64"}
    if family == "adjoint":
        return {"family": family, "n": rng.randint(8, 20), "layers": rng.randint(2, 10), "batch": log_int(1, 64),
                "dtype": "c64"}
    if family == "batchlayer":
        return {"family": family, "n": rng.randint(4, 16), "layers": rng.randint(1, 4), "batch": log_int(9, 300),
                "dtype": "c64"}
    if family == "expect":
        n, terms = rng.randint(10, 26), rng.choice(["ring", "strings"])
        return {"family": family, "n": n, "terms": terms, "count": 2 * n if terms == "ring" else log_int(4, 200),
                "dtype": either}
    if family == "sample":
        return {"family": family, "n": rng.randint(8, 28), "shots": log_int(5, 1 << 20), "dtype": either}
    return {"family": family, "n": rng.randint(5, 27), "dtype": either}


# ---------------------------------------------------------------- circuits

def _generator(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _haar_u3(rng):
    return math.acos(1.0 - 2.0 * rng.random()), rng.random() * 2.0 * math.pi, rng.random() * 2.0 * math.pi


def _haar_unitary(rng, dim):
    z = rng.standard_normal((dim, dim)) + 1j * rng.standard_normal((dim, dim))
    q, r = np.linalg.qr(z)
    d = np.diagonal(r)
    return np.ascontiguousarray(q * (d / np.abs(d)))


def ansatz_circuit(case, seed):
    rng, n = _generator(seed), case["n"]
    gates = []
    for _ in range(case["layers"]):
        for q in range(n):
            gates += [gate("ry", [q], params=[rng.random() * 2.0 * math.pi]),
                      gate("rz", [q], params=[rng.random() * 2.0 * math.pi])]
        gates += [gate("x", [q + 1], [q]) for q in range(n - 1)]
    return gates


def ladder_circuit(n, angles):
    gates = []
    for layer in angles:
        gates += [gate("u3", [q], params=layer[q]) for q in range(n)]
        gates += [gate("x", [q + 1], [q]) for q in range(n - 1)]
    return gates


def ladder_angles(n, depth, rng):
    u = rng.random((depth, n, 3))
    return np.stack([np.arccos(1.0 - 2.0 * u[..., 0]), 2.0 * math.pi * u[..., 1], 2.0 * math.pi * u[..., 2]], axis=-1)


def layered_circuit(case, seed):
    rng, n = _generator(seed), case["n"]
    gates = []
    for _ in range(case["layers"]):
        gates += [gate("u3", [q], params=_haar_u3(rng)) for q in range(n)]
        gates += [gate("z", [q + 1], [q]) for q in list(range(0, n - 1, 2)) + list(range(1, n - 1, 2))]
    return gates


def random_circuit(case, seed):
    """Which qubits the gates act on belongs to the case (it is the circuit);
    the matrices come from the seed."""
    place, rng, n = _generator(case["n"] + 1000 * case["n1"]), _generator(seed), case["n"]
    kinds = np.array([1] * case["n1"] + [2] * case["n2"])
    place.shuffle(kinds)
    gates = []
    for k in kinds:
        qubits = [int(q) for q in place.permutation(n)[:k]]
        gates.append(gate("unitary", qubits, matrix=_haar_unitary(rng, 2 ** int(k))))
    return gates


def packed_requests(case, seed):
    """(n, angles) of every request: 8 to 12 qubits, depth 5 to 40."""
    rng = _generator(seed)
    out = []
    for _ in range(case["requests"]):
        n, depth = int(rng.integers(8, 13)), int(rng.integers(5, 41))
        out.append((n, ladder_angles(n, depth, rng)))
    return out


def adjoint_template(n, layers):
    gates, slot = [], 0
    for _ in range(layers):
        for q in range(n):
            gates += [gate("ry", [q], params=[0.0], slots=[slot]), gate("rz", [q], params=[0.0], slots=[slot + 1])]
            slot += 2
        gates += [gate("x", [(q + 1) % n], [q]) for q in range(n)]
    return gates


def batchlayer_template(n, layers):
    gates, slot = [gate("ry", [q], params=[0.0], slots=[q]) for q in range(n)], n
    for _ in range(layers):
        for q in range(n):
            gates += [gate("ry", [q], params=[0.0], slots=[slot]), gate("rz", [q], params=[0.0], slots=[slot + 1])]
            slot += 2
        gates += [gate("x", [(q + 1) % n], [q]) for q in range(n)]
    return gates


def ring_terms(n):
    return [Term("ZZ", [q, (q + 1) % n], 1.0) for q in range(n)] + [Term("X", [q], 0.7) for q in range(n)]


def string_terms(case):
    """The Hamiltonian is the model's, not the seed's: weights 1 to 4, letters X, Y, Z."""
    rng, n = _generator(7 * case["n"] + case["count"]), case["n"]
    terms = []
    for _ in range(case["count"]):
        w = int(rng.integers(1, 5))
        qubits = [int(q) for q in rng.permutation(n)[:w]]
        terms.append(Term("".join("XYZ"[int(v)] for v in rng.integers(0, 3, size=w)), qubits,
                          float(rng.standard_normal())))
    return terms


def case_terms(case):
    return ring_terms(case["n"]) if case["family"] != "expect" or case["terms"] == "ring" else string_terms(case)


# ---------------------------------------------------------------- states and parameters

def deep_state(n, dtype, seed):
    """The state a deep circuit leaves: Gaussian amplitudes, norm one."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    psi = torch.randn(2 ** n, dtype=TORCH_DTYPE[dtype], device="cuda", generator=g)
    return psi.mul_(1.0 / float(torch.linalg.vector_norm(psi)))


def ansatz_state(n, dtype, seed):
    """The state a shallow variational circuit leaves: mostly a product of
    one-qubit states, partly spread, so that local terms have values of order one."""
    rng = _generator(seed)
    psi = torch.ones(1, dtype=torch.complex128, device="cuda")
    for _ in range(n):
        th, ph = rng.random() * math.pi, rng.random() * 2.0 * math.pi
        one = torch.tensor([math.cos(th / 2), complex(math.cos(ph), math.sin(ph)) * math.sin(th / 2)],
                           dtype=torch.complex128, device="cuda")
        psi = torch.outer(one, psi).reshape(-1)
    psi = psi.to(TORCH_DTYPE[dtype]) + 0.3 * deep_state(n, dtype, seed)
    return psi.mul_(1.0 / float(torch.linalg.vector_norm(psi)))


def batch_params(case, count, seed):
    p = _generator(seed).random((case["batch"], count)) * 2.0 * math.pi
    return torch.tensor(p, dtype=torch.float32, device="cuda")


def batchlayer_inputs(case, seed):
    rng, n = _generator(seed), case["n"]
    x = torch.tensor(rng.random((case["batch"], n)) * math.pi, dtype=torch.float32, device="cuda")
    up = torch.tensor(rng.standard_normal((case["batch"], n)), dtype=torch.float32, device="cuda")
    w = torch.tensor(rng.random(2 * n * case["layers"]) * 2.0 * math.pi, dtype=torch.float32, device="cuda")
    return x, up, w


# ---------------------------------------------------------------- prepare and run

CIRCUITS = {"ansatz": ansatz_circuit, "layered": layered_circuit, "random": random_circuit,
            "ladder": lambda case, seed: ladder_circuit(
                case["n"], ladder_angles(case["n"], case["depth"], _generator(seed)))}


def prepare(case, seed):
    s = dict(case)
    f = case["family"]
    if f in CIRCUITS:
        s["gates"] = sv.Gates(CIRCUITS[f](case, seed))
        s["psi"] = torch.empty(2 ** case["n"], dtype=TORCH_DTYPE[case["dtype"]], device="cuda")
    elif f == "packed":
        req = packed_requests(case, seed)
        s["sizes"] = [n for n, _ in req]
        s["sets"] = [sv.layered_u3_cnot_gates(n, a) for n, a in req]
    elif f == "adjoint":
        n = case["n"]
        s["gates"] = sv.Gates(adjoint_template(n, case["layers"]))
        s["hamiltonian"] = ring_terms(n)
        s["params"] = batch_params(case, 2 * n * case["layers"], seed)
    elif f == "batchlayer":
        n = case["n"]
        x, up, w = batchlayer_inputs(case, seed)
        layer = sv.BatchLayer(batchlayer_template(n, case["layers"]), n, n_data=n, n_weights=w.numel(),
                              dtype=SV_DTYPE[case["dtype"]]).float().cuda()
        layer.weight.data.copy_(w)
        s["layer"], s["x"], s["up"] = layer, x, up
    elif f == "expect":
        s["psi"] = ansatz_state(case["n"], case["dtype"], seed)
        s["hamiltonian"] = sv.pauli_terms(case_terms(case))
    else:
        s["psi"] = deep_state(case["n"], case["dtype"], seed)
        if f == "sample":
            s["uniforms"] = _generator(seed).random(case["shots"])
    return s


def run(s):
    f = s["family"]
    if f in CIRCUITS:
        sv.sv_init_basis(s["psi"], 0)
        sv.sv_apply_circuit(s["psi"], s["gates"], fuse_max_k=5 if f == "layered" else 0)
        if f == "ansatz":
            return {"state": s["psi"], "z": sv.sv_expect_z_all(s["psi"])}
        return {"state": s["psi"]}
    if f == "packed":
        return {"sum_z": sv.sv_run_batch_small(s["sizes"], s["sets"], dtype=SV_DTYPE[s["dtype"]])}
    if f == "adjoint":
        p = s["params"].detach().requires_grad_()
        values = sv.adjoint_expectation(p, s["n"], s["gates"], s["hamiltonian"], dtype=SV_DTYPE[s["dtype"]],
                                        checkpoint_every=2 * 3 * s["n"])
        values.sum().backward()
        return {"values": values.detach(), "gradients": p.grad}
    if f == "batchlayer":
        x = s["x"].detach().requires_grad_()
        s["layer"].zero_grad()
        z = s["layer"](x)
        z.backward(s["up"])
        return {"z": z.detach(), "dx": x.grad, "dw": s["layer"].weight.grad}
    if f == "expect":
        return {"terms": sv.sv_expect(s["psi"], s["hamiltonian"])}
    if f == "sample":
        return {"indices": sv.sv_sample(s["psi"], s["uniforms"])}
    return {"z": sv.sv_expect_z_all(s["psi"]), "p": sv.sv_probabilities(s["psi"])}


# ---------------------------------------------------------------- the work of one pass

# real operations per amplitude of one gate: a one-qubit matrix takes two
# complex products and a sum, a two-qubit one four and three sums, a real
# rotation two scalings and a sum per part, a diagonal one complex product;
# sign and bit flips take none
GATE_FLOPS = {"ry": 6, "rz": 6, "u3": 14, "x": 0, "z": 0}


def work(case):
    f = case["family"]
    amp = AMP_BYTES[case["dtype"]]
    if f == "packed":
        flops = 0
        for n, a in packed_requests(case, 0):
            flops += 2 ** n * (a.shape[0] * n * GATE_FLOPS["u3"] + 4)
        return {"bytes": 8 * case["requests"] + 24 * sum(a.size // 3 for _, a in packed_requests(case, 0)),
                "flops": flops}
    n = case["n"]
    size = 2 ** n
    if f in CIRCUITS:
        layer = {"ansatz": (GATE_FLOPS["ry"] + GATE_FLOPS["rz"]) * n, "ladder": GATE_FLOPS["u3"] * n,
                 "layered": GATE_FLOPS["u3"] * n}
        flops = 14 * case["n1"] + 30 * case["n2"] if f == "random" else \
            layer[f] * (case["depth"] if f == "ladder" else case["layers"])
        return {"bytes": amp * size, "flops": size * flops}
    if f in ("adjoint", "batchlayer"):
        # forward once, the gates undone on two states, a product per gradient
        rotations = 2 * n * case["layers"] + (n if f == "batchlayer" else 0)
        flops = case["batch"] * size * rotations * (6 + 2 * 6 + 4)
        io = 4 * case["batch"] * (2 * n * case["layers"] if f == "adjoint" else 3 * n) * 2
        return {"bytes": io, "flops": flops}
    if f == "expect":
        return {"bytes": amp * size, "flops": size * (8 + 2 * case["count"])}
    if f == "sample":
        return {"bytes": amp * size + 16 * case["shots"], "flops": 4 * size}
    return {"bytes": amp * size + 8 * size, "flops": size * (4 + n)}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch and numpy

def _u3(th, ph, la):
    c, s = math.cos(th / 2), math.sin(th / 2)
    e = np.exp
    return np.array([[c, -e(1j * la) * s], [e(1j * ph) * s, e(1j * (ph + la)) * c]])


def _matrix(g):
    if g.name == "u3":
        return _u3(*g.params)
    if g.name == "ry":
        return _u3(g.params[0], 0.0, 0.0)
    if g.name == "rz":
        return np.diag(np.exp([-0.5j * g.params[0], 0.5j * g.params[0]]))
    return g.matrix


def _axis(psi, n, q):
    """psi as (..., above, bit q, below)."""
    return psi.view(*psi.shape[:-1], 2 ** (n - 1 - q), 2, 2 ** q)


def _pair(psi, n, a, b):
    """The four quarters of psi by (bit b, bit a), as views."""
    lo, hi = min(a, b), max(a, b)
    v = psi.view(*psi.shape[:-1], 2 ** (n - 1 - hi), 2, 2 ** (hi - lo - 1), 2, 2 ** lo)
    pick = lambda i, j: v[..., i, :, j, :] if hi == b else v[..., j, :, i, :]  # noqa: E731
    return [pick(0, 0), pick(0, 1), pick(1, 0), pick(1, 1)]


def _apply1(psi, n, q, u00, u01, u10, u11):
    v = _axis(psi, n, q)
    a, b = v[..., 0, :].clone(), v[..., 1, :].clone()
    v[..., 0, :] = u00 * a + u01 * b
    v[..., 1, :] = u10 * a + u11 * b


def _apply_gate(psi, n, g):
    if g.name == "x":
        quarters = _pair(psi, n, g.targets[0], g.controls[0])
        keep = quarters[2].clone()
        quarters[2].copy_(quarters[3])
        quarters[3].copy_(keep)
    elif g.name == "z":
        _pair(psi, n, g.targets[0], g.controls[0])[3].neg_()
    elif len(g.targets) == 1:
        m = _matrix(g)
        _apply1(psi, n, g.targets[0], *[complex(m[i, j]) for i in (0, 1) for j in (0, 1)])
    else:
        m = g.matrix
        quarters = _pair(psi, n, g.targets[0], g.targets[1])
        old = [x.clone() for x in quarters]
        for i in range(4):
            quarters[i].copy_(sum(complex(m[i, j]) * old[j] for j in range(4)))


def _run_exact(n, gates):
    psi = torch.zeros(2 ** n, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    for g in gates:
        _apply_gate(psi, n, g)
    return psi


def _z_exact(p, n):
    """(<Z_q> of every qubit, their sum) of probabilities p (..., 2^n)."""
    z = [(v[..., 0, :].sum(dim=(-1, -2)) - v[..., 1, :].sum(dim=(-1, -2)))
         for v in (_axis(p, n, q) for q in range(n))]
    return torch.stack(z + [sum(z)], dim=-1)


def _packed_exact(case, seed):
    out = []
    for n, angles in packed_requests(case, seed):
        psi = np.zeros(2 ** n, dtype=np.complex128)
        psi[0] = 1.0
        index = np.arange(2 ** n)
        ladder = index.copy()  # where amplitude i of the ladder's result comes from
        for q in range(n - 2, -1, -1):
            ladder = ladder ^ (((ladder >> q) & 1) << (q + 1))
        for layer in angles:
            for q in range(n):
                v = psi.reshape(-1, 2, 2 ** q)
                psi = np.matmul(_u3(*layer[q]), v).reshape(-1)
            psi = psi[ladder]
        ones = sum((index >> q) & 1 for q in range(n))
        out.append(float(np.sum(np.abs(psi) ** 2 * (n - 2 * ones))))
    return {"sum_z": np.array(out)}


def _strings_exact(psi, n, terms):
    index = torch.arange(2 ** n, device="cuda")
    out = []
    for t in terms:
        x = sum(1 << q for p, q in zip(t.paulis, t.qubits) if p in "XY")
        z = sum(1 << q for p, q in zip(t.paulis, t.qubits) if p in "ZY")
        par = index & z
        for shift in (16, 8, 4, 2, 1):
            par = par ^ (par >> shift)
        sign = 1.0 - 2.0 * (par & 1).to(torch.float64)
        value = (psi[index ^ x].conj() * psi * sign).sum() * 1j ** t.paulis.count("Y")
        out.append(value.real)
    return torch.stack(out)


def _ring_times(psi, n):
    """H psi for the ring model, over the batch."""
    index = torch.arange(2 ** n, device="cuda")
    diag = torch.zeros(2 ** n, dtype=torch.float64, device="cuda")
    for q in range(n):
        diag += 1.0 - 2.0 * (((index >> q) ^ (index >> ((q + 1) % n))) & 1).to(torch.float64)
    out = diag * psi
    for q in range(n):
        _axis(out, n, q).add_(_axis(psi, n, q).flip(-2), alpha=0.7)
    return out


def _template_exact(n, gates, params, hpsi):
    """f and its gradients (batch, slots) by the adjoint recursion, for a
    template of RY, RZ and CNOT; ``hpsi(psi)`` gives H psi per row."""
    batch = params.shape[0]
    psi = torch.zeros(batch, 2 ** n, dtype=torch.complex128, device="cuda")
    psi[:, 0] = 1.0
    half = (params.to(torch.float64) / 2)[:, :, None, None]
    c, s = torch.cos(half), torch.sin(half)

    def turn(v, g, back):
        k, sg = g.slots[0], -1.0 if back else 1.0
        if g.name == "ry":
            _apply1(v, n, g.targets[0], c[:, k], -sg * s[:, k], sg * s[:, k], c[:, k])
        else:
            w = _axis(v, n, g.targets[0])
            w[..., 0, :] *= torch.complex(c[:, k], -sg * s[:, k])
            w[..., 1, :] *= torch.complex(c[:, k], sg * s[:, k])

    for g in gates:
        _apply_gate(psi, n, g) if g.name == "x" else turn(psi, g, False)
    lam = hpsi(psi)
    values = (psi.conj() * lam).real.sum(dim=-1)
    final = psi.clone()
    grad = torch.zeros(batch, params.shape[1], dtype=torch.float64, device="cuda")
    for g in reversed(gates):
        if g.name == "x":
            _apply_gate(psi, n, g)
            _apply_gate(lam, n, g)
            continue
        v, w = _axis(psi, n, g.targets[0]), _axis(lam, n, g.targets[0])
        if g.name == "ry":  # Y v = (-i v1, i v0)
            dot = (w[..., 1, :].conj() * v[..., 0, :] - w[..., 0, :].conj() * v[..., 1, :]).real
        else:
            dot = (w[..., 0, :].conj() * v[..., 0, :] - w[..., 1, :].conj() * v[..., 1, :]).imag
        grad[:, g.slots[0]] += dot.sum(dim=(-1, -2))
        turn(psi, g, True)
        turn(lam, g, True)
    return values, grad, final


def exact(case, seed):
    f, n = case["family"], case.get("n", 0)
    if f == "packed":
        return _packed_exact(case, seed)
    if f in CIRCUITS:
        if n > 26:  # a pass over the state per gate takes too long
            return None
        psi = _run_exact(n, CIRCUITS[f](case, seed))
        if f != "ansatz":
            return {"state": psi}
        return {"state": psi, "z": _z_exact(psi.abs().square(), n)}
    if f == "adjoint":
        if case["batch"] * 2 ** n > 2 ** 26:  # as above
            return None
        params = batch_params(case, 2 * n * case["layers"], seed)
        values, grad, _ = _template_exact(n, adjoint_template(n, case["layers"]), params,
                                          lambda psi: _ring_times(psi, n))
        return {"values": values, "gradients": grad}
    if f == "batchlayer":
        x, up, w = batchlayer_inputs(case, seed)
        params = torch.cat([x, w.expand(x.shape[0], -1)], dim=1)
        index = torch.arange(2 ** n, device="cuda")
        signs = torch.stack([1.0 - 2.0 * ((index >> q) & 1).to(torch.float64) for q in range(n)])
        diag = up.to(torch.float64) @ signs
        _, grad, psi = _template_exact(n, batchlayer_template(n, case["layers"]), params, lambda psi: diag * psi)
        return {"z": _z_exact(psi.abs().square(), n)[:, :n], "dx": grad[:, :n], "dw": grad[:, n:].sum(dim=0)}
    if f == "expect":
        psi = ansatz_state(n, case["dtype"], seed).to(torch.complex128)
        return {"terms": _strings_exact(psi, n, case_terms(case))}
    if f == "sample":
        return None  # whole numbers
    psi = deep_state(n, case["dtype"], seed).to(torch.complex128)
    p = torch.view_as_real(psi).square().sum(dim=-1)
    return {"z": _z_exact(p, n), "p": p / p.sum()}
