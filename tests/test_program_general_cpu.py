"""The general pass's programs of small states, run on the host against the
oracle.  By default states of 5 to 16 qubits take the cluster pass's programs;
with a tile width they take the general ones, which also serve larger states,
states beside a live session and devices without large clusters: the planner's
own widths (13 qubits complex64, 11 complex128) and a narrower one (several
tiles)."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from test_program_cpu import CASES, TOL, _closing_phase_circuit, _emulate
from workloads import hea_params, hea_ring, random_circuit, serving_circuit

MORE = [
    ("ladder", 14, lambda: serving_circuit(14, 8, 1)),
    ("closing_phases", 13, lambda: _closing_phase_circuit(13, 5, seed=4)),
    ("wide_unitaries", 12, lambda: random_circuit(12, 120, seed=3, max_controls=1, max_unitary_k=5)),
]
WIDTHS = {sv.SV_C64: (13, 10), sv.SV_C128: (11, 8)}


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("name,n,make", CASES + MORE, ids=[c[0] for c in CASES + MORE])
@pytest.mark.parametrize("fuse", [0, 5])
def test_general_programs_match_oracle(name, n, make, dtype, fuse):
    circ = make()
    ref = oracle.run(n, circ)
    for tile in WIDTHS[dtype]:
        got = _emulate(n, circ, dtype, fuse_max_k=fuse, tile_qubits=tile)
        assert np.abs(got - ref).max() <= TOL[dtype], tile


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
def test_general_programs_bound_parameters(dtype):
    n = 12
    circ = hea_ring(n, 4)
    params = hea_params(1, 2 * n * 4, seed=9)[0]
    ref = oracle.run(n, circ, params)
    for tile in WIDTHS[dtype]:
        got = _emulate(n, circ, dtype, params=params, tile_qubits=tile)
        assert np.abs(got - ref).max() <= TOL[dtype], tile
