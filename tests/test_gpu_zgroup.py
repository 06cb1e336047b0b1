"""Groups of one-qubit diagonals in the batched adjoint passes, against the
oracle's gradients: several rotations of one qubit, members on register slots,
thread bits and bits outside the tile, more than four gradient members,
constant diagonals, and diagonals that must stay out (controls, generators
other than Z); compiled and interpreted passes give the same bits."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import Gate, Term

pytestmark = pytest.mark.gpu

TOL = {sv.SV_C64: 1e-4, sv.SV_C128: 1e-10}  # the gradient tolerances of the other adjoint tests


def _template(n, layers, seed):
    rng = np.random.default_rng(seed)
    gates, slot = [], 0

    def rot(name, targets, controls=()):
        nonlocal slot
        gates.append(Gate(name, list(targets), list(controls), slots=[slot], params=[0.0]))
        slot += 1

    for _ in range(layers):
        for q in range(n):
            if rng.integers(3):
                rot("ry", [q])
            for _ in range(int(rng.integers(0, 3))):
                rot("rz", [q])
            if not rng.integers(4):
                gates.append(Gate(["s", "t", "z"][int(rng.integers(3))], [q]))
        for q in range(n):
            other = (q + 1 + int(rng.integers(n - 1))) % n
            kind = rng.integers(6)
            if kind < 2:
                gates.append(Gate("x", [other], [q]))
            elif kind == 2:
                rot("rz", [other], [q])
            elif kind == 3:
                rot("p", [q])
            elif kind == 4:
                rot("rzz", [q, other])
    return gates, slot


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n,layers,ckpt", [(3, 3, 0), (4, 2, 0), (6, 3, 10), (13, 2, 0), (14, 2, 25)])
def test_gradients(svlib, cuda_dev, n, layers, ckpt, dtype):
    gates, npar = _template(n, layers, seed=n)
    terms = [Term("Z", [q], 1.0) for q in range(n)] + [Term("X", [0], 0.5), Term("XY", [0, n - 1], 0.3)]
    th = np.random.default_rng(n).uniform(-np.pi, np.pi, size=(3, npar))
    out = []
    try:
        for mode in (0, 2):
            sv.sv_jit_set_mode(mode)
            out.append(sv.sv_adjoint_grad(n, dtype, gates, th, terms, checkpoint_every=ckpt))
    finally:
        sv.sv_jit_set_mode(-1)
    (v, g), (v2, g2) = out
    assert np.array_equal(v, v2) and np.array_equal(g, g2)
    for b in range(3):
        v_ref, g_ref = oracle.adjoint_grad(n, gates, th[b], terms, npar)
        assert abs(v[b] - v_ref) < TOL[dtype] and np.abs(g[b] - g_ref).max() < TOL[dtype]


@pytest.mark.parametrize("qubits", [[11], [0, 5, 11]])
def test_a_callers_matrix_keeps_its_modulus(svlib, cuda_dev, qubits):
    # accepted within 1e-6 of unitary: modulus 1 + 4e-7 forty times over is
    # 3.2e-5 in a value of order one, three times the single precision bound
    # of its 120 operations (120 x 2^-24, of a norm squared)
    n, tol = 12, 1e-5
    big = np.diag([1.0 + 4e-7, (1.0 + 4e-7) * 1j])
    gates = [Gate("ry", [q], slots=[q], params=[0.0]) for q in range(n)]
    for k in range(40):
        q = qubits[k % len(qubits)]
        gates += [Gate("rz", [(q + 1) % n], slots=[n], params=[0.0]), Gate("unitary", [q], matrix=big)]
    terms = [Term("ZZ", [1, 2], 1.0)]
    th = np.full((2, n + 1), 0.3)
    v, _ = sv.sv_adjoint_grad(n, sv.SV_C64, gates, th, terms)
    v_ref, _ = oracle.adjoint_grad(n, gates, th[0], terms, n + 1)
    assert np.abs(v - v_ref).max() < tol
