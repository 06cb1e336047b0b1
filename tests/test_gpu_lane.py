"""The cluster pass of small states (5 to 16 qubits) against the oracle: every
spread of a tile over CTAs, warps and groups (each size has its own), several
tiles, every op kind, and the general pass on the same circuits."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import fused_layered_u3_cz, layered_ry_rz_cnot, random_circuit, serving_circuit

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DT = {sv.SV_C64: torch.complex64, sv.SV_C128: torch.complex128}
TOL = {sv.SV_C64: 1e-5, sv.SV_C128: 1e-12}  # the state tolerances of the other parity tests


def _run(n, dtype, circ, **kw):
    st = torch.empty(2 ** n, dtype=DT[dtype], device="cuda")
    sv.sv_init_basis(st, 0)
    sv.sv_profile_enable(True)
    sv.sv_apply_circuit_ex(st, circ, **kw)
    torch.cuda.synchronize()
    fam = sv.sv_profile_read()
    sv.sv_profile_enable(False)
    return st.cpu().numpy().astype(np.complex128), set(fam)


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", list(range(5, 17)))
def test_every_size(svlib, cuda_dev, n, dtype):
    circ = random_circuit(n, 150, seed=n, max_controls=2, max_unitary_k=min(4, n))
    got, fam = _run(n, dtype, circ)
    assert fam == {"sweep_lane"}
    assert np.abs(got - oracle.run(n, circ)).max() < TOL[dtype]


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", [7, 14, 16])
@pytest.mark.parametrize("kind", ["ansatz", "ladder", "layered", "dense"])
def test_circuits(svlib, cuda_dev, n, kind, dtype):
    circ = {"ansatz": lambda: layered_ry_rz_cnot(n, 6, 1), "ladder": lambda: serving_circuit(n, 8, 2),
            "layered": lambda: fused_layered_u3_cz(n, 8, 3), "dense": lambda: fused_layered_u3_cz(n, 3, 4)}[kind]()
    kw = dict(fuse_max_k=5, block_mode=sv.SV_BLOCK_DENSE) if kind == "dense" else dict(fuse_max_k=0)
    got, fam = _run(n, dtype, circ, **kw)
    assert fam == {"sweep_lane"}
    assert np.abs(got - oracle.run(n, circ)).max() < TOL[dtype]


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
def test_other_sizes_and_options_keep_the_general_pass(svlib, cuda_dev, dtype):
    for n, kw in ((4, {}), (17, {}), (12, dict(tile_qubits=10)), (12, dict(ops_per_pass=1))):
        circ = random_circuit(n, 40, seed=n, max_controls=1, max_unitary_k=2)
        got, fam = _run(n, dtype, circ, **kw)
        assert "sweep_lane" not in fam
        assert np.abs(got - oracle.run(n, circ)).max() < TOL[dtype]


def test_live_session_keeps_the_general_pass(svlib, cuda_dev):
    # a session's resident CTAs could keep a cluster of 16 waiting
    from paper_2608_09733_gb300.binding import SmallSession, SvError
    s = SmallSession(sv.SV_C64, wait_limit_s=0.2)
    try:
        circ = serving_circuit(12, 4, 5)
        got, fam = _run(12, sv.SV_C64, circ)
        assert fam == {"sweep"}
        assert np.abs(got - oracle.run(12, circ)).max() < 1e-5
    finally:
        try:
            s.stop()
        except SvError:
            pass  # it sat idle
    got, fam = _run(12, sv.SV_C64, circ)
    assert fam == {"sweep_lane"}
