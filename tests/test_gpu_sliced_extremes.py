"""Sliced FP64 products at the edge of the tensor core's exact sums: operands whose digits are 64, -128, -128, ... everywhere, so
that every digit product has the largest size and one sign.

rsfd_transmission with Gamma_R = I and Gamma_L = e_a e_a^T is one element of G_RL^H G_RL: with G_RL = x (1 + i) in column a (and random
signs, which cancel) T = 2 ns x^2, computed here in exact rational arithmetic.  Tolerance: the result's rounding (2^-53) and, per
128 rows, at most 2^-46.7 on a sum of 256 x^2: together below 2^-52 of T."""

from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1502_00081_gb300.build_lib import build
    build()
    import paper_1502_00081_gb300 as m
    m.load_library()
    return m


@pytest.mark.parametrize("ns", [208, 256, 1000])
@pytest.mark.parametrize("digits", [6, 4, 1])
def test_largest_digits(rs, ns, digits):
    x = 1.0 - sum(2.0 ** (1 - 8 * s) for s in range(1, digits + 1))   # digits 64, then -128 `digits` times
    a, rng = 5, np.random.Generator(np.random.PCG64(ns))
    G = np.zeros((1, 2 * ns, 2 * ns), complex)
    G[0, ns:, a] = x * (1 + 1j) * rng.choice([-1.0, 1.0], size=ns)
    SL = np.zeros((1, ns, ns), complex)
    SL[0, a, a] = -0.5j
    SR = -0.5j * np.eye(ns)[None]
    up = lambda M: torch.from_numpy(np.ascontiguousarray(M.transpose(0, 2, 1))).cuda()   # noqa: E731
    with rs.Handle((ns, 1, 4), 0.5, 2, np.zeros(4 * ns), n_face=1, precision=rs.RSFD_FP64) as h:
        T = rs.rsfd_transmission(h.ptr, up(G), up(SL), up(SR))[0]
    exact = 2 * ns * Fraction(x) ** 2
    assert abs(Fraction(float(T)) - exact) <= exact / 2 ** 52
