"""H|psi> over tiles: Z strings within the low local bits, within the high ones
and across both, X terms alone with and without Z on the tile, more terms than
one launch takes; one Hamiltonian and one per state, against the oracle's
gradients."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import Gate, Term

pytestmark = pytest.mark.gpu

# |g| <= sum |c_j| <= 12: 64 roundings of float there are 4.6e-5, of double 8.5e-14
TOL = {sv.SV_C64: 1e-4, sv.SV_C128: 1e-10}


def _terms(n, count, seed):
    rng = np.random.default_rng(seed)
    low, high = list(range(min(n, 7))), list(range(7, n))
    terms = [Term("Z", [q], 0.2) for q in range(n)]
    for i in range(count):
        pool = [low, high or low, list(range(n))][i % 3]
        qs = list(rng.choice(pool, size=int(rng.integers(1, len(pool) + 1)), replace=False))
        kind = ["Z", "Z", "Z", "ZX", "Y"][int(rng.integers(5))] if i % 4 else "X"
        ps = "".join(kind[int(rng.integers(len(kind)))] if j < 3 else "Z" for j in range(len(qs)))
        if kind == "X":
            qs, ps = qs[:1], "X"
        terms.append(Term(ps, [int(q) for q in qs], float(rng.uniform(-0.1, 0.1))))
    return terms


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n,count", [(1, 1), (3, 9), (6, 20), (7, 30), (8, 40), (12, 60), (14, 120)])
def test_h_psi(svlib, cuda_dev, n, count, dtype):
    gates, npar = [], 0
    for q in range(n):
        for name in ("ry", "rz"):
            gates.append(Gate(name, [q], slots=[npar], params=[0.0]))
            npar += 1
    gates += [Gate("x", [q + 1], [q]) for q in range(n - 1)]
    for q in range(n):
        gates.append(Gate("rx", [q], slots=[npar], params=[0.0]))
        npar += 1
    terms = _terms(n, count, seed=n)
    rng = np.random.default_rng(100 + n)
    th = rng.uniform(-np.pi, np.pi, size=(2, npar))
    v, g = sv.sv_adjoint_grad(n, dtype, gates, th, terms)
    rows = np.array([[t.coeff for t in terms]] * 2) * np.array([[1.0], [-0.5]])
    _, grows = sv.sv_adjoint_grad_rows(n, dtype, gates, th, terms, rows)
    for b in range(2):
        v_ref, g_ref = oracle.adjoint_grad(n, gates, th[b], terms, npar)
        assert abs(v[b] - v_ref) < TOL[dtype] and np.abs(g[b] - g_ref).max() < TOL[dtype]
        assert np.abs(grows[b] - [1.0, -0.5][b] * g_ref).max() < TOL[dtype]
