"""Batched <Z> (one launch for all states of a batch) where the states are cut
into chunks over several blocks: fewer chunks than blocks wanted, more, and
blocks of one to eight warps; large batches and then small ones on one stream."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import Gate

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# complex64: about sixty roundings of 2^-24 by the gates and 70 by the read-out's
# runs, of values of order one; complex128 as many of 2^-53
TOL = {sv.SV_C64: 2e-5, sv.SV_C128: 1e-12}


def _template(n):
    gates = [Gate("ry", [q], slots=[q]) for q in range(n)]
    gates += [Gate("x", [q + 1], controls=[q]) for q in range(n - 1)]
    return gates + [Gate("rx", [q], slots=[n + q]) for q in range(n)]


def _check(n, dtype, batch, seed):
    gates = _template(n)
    params = np.random.default_rng(seed).uniform(0, 2 * np.pi, size=(batch, 2 * n))
    z = sv.sv_batch_expect_z(n, dtype, gates, params)
    for b in sorted({0, 1, batch // 2, batch - 1}):
        per, s = oracle.expect_z_all(oracle.run(n, gates, params[b]), n)
        assert np.abs(z[b, :n] - per).max() < TOL[dtype], b
        assert abs(z[b, n] - s) < n * TOL[dtype], b


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", [11, 12, 14, 16])
@pytest.mark.parametrize("batch", [2, 3, 300])
def test_batch_z_over_several_blocks(svlib, cuda_dev, n, dtype, batch):
    _check(n, dtype, batch, 100 * n + batch)


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
def test_large_batch_then_small(svlib, cuda_dev, dtype):
    for n, batch in ((12, 500), (14, 2), (11, 3), (16, 5)):
        _check(n, dtype, batch, n + batch)
