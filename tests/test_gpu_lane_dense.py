"""Unitaries of three to five targets in the cluster pass, against the oracle:
the matrix on lane bits in every order, controls on lane bits, on the group's
bits and outside the tile, one, two and four groups a warp."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import Gate, haar_unitary, random_circuit

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DT = {sv.SV_C64: torch.complex64, sv.SV_C128: torch.complex128}
TOL = {sv.SV_C64: 1e-5, sv.SV_C128: 1e-12}  # the state tolerances of the other parity tests


def _check(n, dtype, circ, **kw):
    st = torch.empty(2 ** n, dtype=DT[dtype], device="cuda")
    sv.sv_init_basis(st, 0)
    sv.sv_profile_enable(True)
    sv.sv_apply_circuit_ex(st, circ, **kw)
    torch.cuda.synchronize()
    fam = set(sv.sv_profile_read())
    sv.sv_profile_enable(False)
    assert fam == {"sweep_lane"}
    assert np.abs(st.cpu().numpy() - oracle.run(n, circ)).max() < TOL[dtype]


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", [5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16])
def test_random_wide(svlib, cuda_dev, n, dtype):
    _check(n, dtype, random_circuit(n, 60, seed=n, max_controls=2, max_unitary_k=5))


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("k", [3, 4, 5])
@pytest.mark.parametrize("n", [8, 13, 16])
def test_targets_in_every_order_with_controls(svlib, cuda_dev, n, k, dtype):
    rng = np.random.Generator(np.random.PCG64(10 * n + k))
    gates = [Gate("u3", [q], params=list(rng.uniform(0.3, 2.8, 3))) for q in range(n)]
    for _ in range(12):
        qs = [int(q) for q in rng.permutation(n)]
        nc = int(rng.integers(0, min(3, n - k) + 1))
        gates.append(Gate("unitary", qs[:k], qs[k:k + nc], [int(b) for b in rng.integers(0, 2, nc)],
                          matrix=haar_unitary(rng, 2 ** k)))
    _check(n, dtype, gates)


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", [6, 14, 16])
def test_wide_diagonals(svlib, cuda_dev, n, dtype):
    rng = np.random.Generator(np.random.PCG64(n))
    gates = [Gate("u3", [q], params=list(rng.uniform(0.3, 2.8, 3))) for q in range(n)]
    for k in (3, 4, 5, 3):
        qs = [int(q) for q in rng.permutation(n)]
        nc = min(1, n - k)
        gates.append(Gate("unitary", qs[:k], qs[k:k + nc], [1] * nc,
                          matrix=np.diag(np.exp(1j * rng.uniform(-3, 3, 2 ** k)))))
        gates.append(Gate("h", [qs[0]]))
    _check(n, dtype, gates)
