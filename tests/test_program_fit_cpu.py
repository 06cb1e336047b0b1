"""Circuits of wide unitaries whose passes hold more than one device program
can (its ops, phase tables and merged matrices): the pass is cut in parts, not
refused.  Host execution of every part against the oracle, in the two program
forms (the cluster pass and, with a tile width, the general one)."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import random_circuit

TOL = {sv.SV_C128: 1e-12, sv.SV_C64: 2e-6}  # float: the coefficients' rounding, as in the other program tests
# more ops than one device program holds fit one tile of each size
SIZES = [(6, 18), (6, 3), (12, 7), (12, 41), (13, 10), (14, 5)]


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n,seed", SIZES)
def test_wide_unitaries_are_cut_not_refused(n, seed, dtype):
    circ = random_circuit(n, 150, seed=seed, max_controls=1, max_unitary_k=5)
    ref = oracle.run(n, circ)
    for kw in ({}, dict(tile_qubits=10), dict(fuse_max_k=5)):
        st = np.zeros(2 ** n, dtype=np.complex128)
        st[0] = 1.0
        got = sv.sv_emulate_apply(st, n, dtype, circ, **kw)
        assert np.abs(got - ref).max() <= TOL[dtype], kw


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
def test_every_seed_is_planned(dtype):
    # sv_plan_info counts the programs that run, so it builds each of them
    for n in (6, 12, 13):
        for seed in range(60):
            circ = sv.Gates(random_circuit(n, 150, seed=seed, max_controls=1, max_unitary_k=5))
            _, passes, _ = sv.sv_plan_info(n, dtype, circ)
            assert passes >= 1
