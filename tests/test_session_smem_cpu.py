"""What a resident session CTA leaves of its SM's shared memory: the large
kernels of other streams have to fit beside it, or a session on every SM would
hold them back until it goes idle."""
import pytest

import paper_2608_09733_gb300 as sv
from paper_2608_09733_gb300 import binding

SM = 228 * 1024       # shared memory of an SM
RESERVED = 1024       # of every CTA, by the system
STATIC = 1024         # the session kernel's own static arrays, rounded up
# (dynamic + static) bytes of one CTA of the large kernels, complex64
BESIDE = {
    # two 2^12 tiles, 256 gather offsets, coefficients, the gradient accumulators (64 x 8 doubles)
    "reverse batched sweep": 2 * 8 * 2 ** 12 + 1024 + 8 * 1024 + 64 * 8 * 8 + 2048,
    # a 2^13 tile, offsets, the terms' masks, coefficients and sums
    "H|psi> tiles": 8 * 2 ** 13 + 2048 + 8 * 1024,
    # a 2^13 tile, offsets and a full coefficient pool
    "general pass, 13-qubit tile": 8 * 2 ** 13 + 8 * 256 + 24 * 1024,
}


def test_a_session_cta_holds_its_largest_state_and_no_more(svlib):
    f = svlib.sv_small_session_shared_bytes
    assert f(sv.SV_C64) == 8 << 14
    assert f(sv.SV_C128) == 16 << 12
    assert f(7) == 0
    assert "sv_small_session_shared_bytes" in binding.EXPORTS


@pytest.mark.parametrize("kernel", sorted(BESIDE))
def test_large_kernels_fit_beside_a_session(svlib, kernel):
    left = SM - svlib.sv_small_session_shared_bytes(sv.SV_C64) - RESERVED - STATIC
    assert BESIDE[kernel] + RESERVED <= left
