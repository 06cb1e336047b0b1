"""The reduction and measurement kernels at the sizes where their splits
change: terms per X mask around the accumulator counts, the read-out around
one warp chunk, chunks and shot groups of the draws, and the integer form of
p = x^2 + y^2 over every class of float."""
import numpy as np
import pytest

import oracle
import paper_2608_09733_gb300 as sv
from workloads import Term, random_circuit

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DT = {sv.SV_C64: torch.complex64, sv.SV_C128: torch.complex128}


def _random_state(n, dtype, seed):
    rng = np.random.default_rng(seed)
    psi = rng.standard_normal(2 ** n) + 1j * rng.standard_normal(2 ** n)
    psi /= np.linalg.norm(psi)
    st = torch.tensor(psi, dtype=DT[dtype], device="cuda")
    return st, st.cpu().numpy().astype(np.complex128)


# complex64: a run of 64 float adds and one product are off by at most about
# 70 * 2^-24 of the sum of |terms| (= 1); complex128 by as many 2^-53
TOL = {sv.SV_C64: 5e-6, sv.SV_C128: 1e-13}


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", [1, 2, 9, 18])
@pytest.mark.parametrize("count", [1, 2, 3, 4, 5, 8, 9, 16, 17, 150])
def test_terms_per_mask(svlib, cuda_dev, dtype, n, count):
    st, host = _random_state(n, dtype, n)
    rng = np.random.default_rng(1000 * n + count)
    terms = []
    for letters in ("IZ", "XY"):  # no X bit; the same X mask with X or Y letters
        flip = rng.random(n) < 0.5
        flip[-1] = True
        for _ in range(count):
            qs = [q for q in range(n) if letters == "IZ" or flip[q]]
            ps = "".join(letters[int(rng.integers(0, 2))] for _ in qs)
            zs = [q for q in range(n) if q not in qs and rng.random() < 0.5]
            keep = [(p, q) for p, q in zip(ps + "Z" * len(zs), qs + zs) if p != "I"]
            terms.append(Term("".join(p for p, _ in keep), [q for _, q in keep], 1.0))
    got = sv.sv_expect(st, terms)
    assert np.abs(got - oracle.expect_terms(host, n, terms)[1]).max() < TOL[dtype]


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
def test_many_masks_fill_several_launches(svlib, cuda_dev, dtype):
    n = 10
    st, host = _random_state(n, dtype, 3)
    terms = [Term("X" * bin(x).count("1"), [q for q in range(n) if (x >> q) & 1], 1.0) for x in range(1, 400)]
    got = sv.sv_expect(st, terms)
    assert np.abs(got - oracle.expect_terms(host, n, terms)[1]).max() < TOL[dtype]


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", [1, 3, 5, 6, 8, 9, 10, 11, 12, 15, 20, 21])
def test_z_all_sizes(svlib, cuda_dev, dtype, n):
    st, host = _random_state(n, dtype, 50 + n)
    z = sv.sv_expect_z_all(st)
    per, s = oracle.expect_z_all(host, n)
    assert np.abs(z[:n] - per).max() < TOL[dtype]
    assert abs(z[n] - s) < n * TOL[dtype]


def test_probability_bits_of_every_float_class(svlib, cuda_dev):
    n = 20
    rng = np.random.default_rng(11)
    bits = rng.integers(0, 2 ** 32, size=2 ** (n + 1), dtype=np.uint64).astype(np.uint32)
    near = rng.integers(0, 2 ** 32, size=2 ** n, dtype=np.uint64).astype(np.uint32)
    re, im = bits[0::2].copy(), bits[1::2].copy()
    half = 2 ** (n - 1)  # half of the pairs with exponents close to each other, where rounding decides
    e = (re[:half] >> 23 & 255).astype(np.int64) + (near[:half] % 33).astype(np.int64) - 16
    im[:half] = (im[:half] & np.uint32(0x807FFFFF)) | (np.clip(e, 0, 255).astype(np.uint32) << np.uint32(23))
    im[half:half + 4096] &= np.uint32(0x807FFFFF)  # subnormal
    re[half:half + 2048] &= np.uint32(0x807FFFFF)
    im[-4096:] = 0
    re[-2048:] = 0
    psi = np.empty(2 ** n, dtype=np.complex64)
    psi.view(np.float32)[0::2], psi.view(np.float32)[1::2] = re.view(np.float32), im.view(np.float32)
    st = torch.from_numpy(psi).cuda()
    got = sv.sv_probabilities(st, normalise=False).cpu().numpy()
    x, y = re.view(np.float32).astype(np.float64), im.view(np.float32).astype(np.float64)
    with np.errstate(invalid="ignore", over="ignore"):
        want = x * x + y * y
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.array_equal(got[ok], want[ok])


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n", [1, 2, 7, 17])
def test_normalised_probabilities(svlib, cuda_dev, dtype, n):
    st, host = _random_state(n, dtype, n)
    p = sv.sv_probabilities(st * 3.0).cpu().numpy()
    want = oracle.probabilities((st * 3.0).cpu().numpy().astype(np.complex128), n)
    assert np.allclose(p, want, rtol=1e-13, atol=0.0)
    zero = torch.zeros_like(st)
    assert not sv.sv_probabilities(zero).any()  # no mass: left as it is


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n,shots", [(5, 1), (6, 33), (7, 64), (8, 3000), (13, 20000), (19, 400001)])
def test_draws_across_chunks_and_groups(svlib, cuda_dev, dtype, n, shots):
    st = torch.empty(2 ** n, dtype=DT[dtype], device="cuda")
    sv.sv_init_basis(st, 0)
    sv.sv_apply_circuit(st, random_circuit(n, 60, seed=n, max_controls=1, max_unitary_k=2))
    st[2 ** n // 4: 2 ** n // 2] = 0  # empty chunks
    u = np.random.default_rng(n).random(shots)
    u[0] = 1.0 - 2.0 ** -53
    assert (sv.sv_sample(st, u) == oracle.sample(st.cpu().numpy().astype(np.complex128), n, u)).all()


def test_draws_from_large_amplitudes(svlib, cuda_dev):
    # |x| >= 2 takes the FP64 form of q (not normalised states)
    n = 9
    st = torch.zeros(2 ** n, dtype=torch.complex64, device="cuda")
    st[5], st[300] = 2.25, 1.5j
    u = np.random.default_rng(0).random(5000)
    assert (sv.sv_sample(st, u) == oracle.sample(st.cpu().numpy().astype(np.complex128), n, u)).all()
