"""Which pass a complex64 state of 15 and 16 qubits takes: short circuits of
one-qubit gates and diagonals the general one, others and smaller states the
cluster pass; either way the oracle's state, on both sides of the rule."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import Gate, fused_layered_u3_cz, layered_ry_rz_cnot

torch = pytest.importorskip("torch")

DT = {sv.SV_C64: torch.complex64, sv.SV_C128: torch.complex128}


def _with_flip(n):
    return fused_layered_u3_cz(n, 2, 1) + [Gate("x", [0], [1])]


CASES = [  # n, circuit, dtype, takes the cluster pass
    (14, lambda: fused_layered_u3_cz(14, 2, 1), sv.SV_C64, True),
    (15, lambda: fused_layered_u3_cz(15, 2, 1), sv.SV_C64, False),
    (15, lambda: fused_layered_u3_cz(15, 6, 1), sv.SV_C64, False),  # 174 operations
    (15, lambda: fused_layered_u3_cz(15, 7, 1), sv.SV_C64, True),   # 203
    (16, lambda: fused_layered_u3_cz(16, 5, 1), sv.SV_C64, False),
    (16, lambda: fused_layered_u3_cz(16, 7, 1), sv.SV_C64, True),
    (16, lambda: _with_flip(16), sv.SV_C64, True),
    (16, lambda: layered_ry_rz_cnot(16, 1, 1), sv.SV_C64, True),
    (16, lambda: fused_layered_u3_cz(16, 2, 1), sv.SV_C128, True),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("fuse", [0, 5])
def test_host_execution(case, fuse):
    n, make, dtype, _ = CASES[case]
    circ = make()
    st = np.zeros(2 ** n, dtype=np.complex128)
    st[0] = 1.0
    got = sv.sv_emulate_apply(st, n, dtype, circ, fuse_max_k=fuse)
    # the coefficients' rounding, as in the other program tests
    assert np.abs(got - oracle.run(n, circ)).max() <= {sv.SV_C128: 1e-12, sv.SV_C64: 2e-6}[dtype]


@pytest.mark.gpu
@pytest.mark.parametrize("case", range(len(CASES)))
def test_pass_and_state(svlib, cuda_dev, case):
    n, make, dtype, lane = CASES[case]
    circ = make()
    st = torch.empty(2 ** n, dtype=DT[dtype], device="cuda")
    sv.sv_init_basis(st, 0)
    sv.sv_profile_enable(True)
    sv.sv_apply_circuit(st, circ, fuse_max_k=5)
    torch.cuda.synchronize()
    fam = set(sv.sv_profile_read())
    sv.sv_profile_enable(False)
    assert (fam == {"sweep_lane"}) == lane
    # the state tolerances of the other parity tests
    assert np.abs(st.cpu().numpy() - oracle.run(n, circ)).max() < {sv.SV_C64: 1e-5, sv.SV_C128: 1e-12}[dtype]
