"""One-qubit gates joined into two-qubit matrices (planner), run on the host
against the oracle: every order of gate and neighbour, both matrix orders of a
pair, the same pair twice, controls and diagonals in between."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import Gate, haar_unitary


def _circuit(n, count, seed):
    rng = np.random.default_rng(seed)
    gates = []
    for _ in range(count):
        a, b, c = (int(q) for q in rng.permutation(n)[:3])
        kind = rng.integers(9)
        if kind < 3:
            gates.append(Gate("unitary", [a], matrix=haar_unitary(rng, 2, special=False)))
        elif kind < 5:
            gates.append(Gate("unitary", [a, b], matrix=haar_unitary(rng, 4)))
            if rng.integers(2):  # the same pair again, in either order
                gates.append(Gate("unitary", [b, a] if rng.integers(2) else [a, b], matrix=haar_unitary(rng, 4)))
        else:
            gates.append([Gate("rz", [a], params=[float(rng.uniform(-3, 3))]), Gate("x", [a]),
                          Gate("y", [a], controls=[b]), Gate("rzz", [a, b], params=[float(rng.uniform(-3, 3))])][kind - 5])
            if kind == 8 and rng.integers(2):
                gates.append(Gate("unitary", [a, b], controls=[c], matrix=haar_unitary(rng, 4)))
    return gates


@pytest.mark.parametrize("dtype,tol", [(sv.SV_C64, 2e-6), (sv.SV_C128, 1e-12)])  # the program tests' tolerances
@pytest.mark.parametrize("n", [3, 6, 17])
@pytest.mark.parametrize("fuse", [0, 2])
def test_joined_circuits_match_oracle(n, dtype, tol, fuse):
    circ = _circuit(n, 80, seed=10 * n + fuse)
    st = np.zeros(2 ** n, dtype=np.complex128)
    st[0] = 1.0
    sv.sv_emulate_apply(st, n, dtype, circ, fuse_max_k=fuse)
    assert np.abs(st - oracle.run(n, circ)).max() <= tol


def test_joining_leaves_blocks_and_plain_path_alone():
    # the block boundaries name source gates; one operation per pass keeps every gate
    n = 6
    circ = _circuit(n, 30, seed=1)
    blocks, passes, starts = sv.sv_plan_info(n, sv.SV_C128, circ, ops_per_pass=1)
    assert blocks == len(circ) == passes and starts == list(range(len(circ) + 1))
    assert sv.sv_plan_info(n, sv.SV_C128, circ)[2] == starts
