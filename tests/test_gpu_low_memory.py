"""Calls on a device whose memory another allocation nearly fills: the lead decimation takes its two leads one after the other,
and products and solves of the Dyson step without room for digit planes or block inverses run on their plain forms.  The
results agree with those of an empty device to FP64 round-off of n-term sums (n 2^-46 allowed)."""

import contextlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MIB = 1 << 20
FP64, TC = 1, 2


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1502_00081_gb300.build_lib import build
    build()
    import paper_1502_00081_gb300 as m
    m.load_library()
    return m


@contextlib.contextmanager
def _left(mib):
    """An allocation that leaves this much device memory."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    filler = torch.empty(free - mib * MIB, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del filler
        torch.cuda.empty_cache()


def _rel(a, b):
    return float((a - b).norm() / b.norm())


def test_lead_decimation_one_lead_after_the_other(rs):
    """800 rows: 10 MiB a matrix, 26 of them for both leads of one energy, 13 for one."""
    nx, E = 20, np.array([0.7, 1.1])
    V = np.random.Generator(np.random.PCG64(3)).uniform(-0.5, 0.0, size=(2, 2, nx, nx))
    def handle():
        return rs.Handle((nx, nx, 6), 0.5, 4, np.zeros(6 * nx * nx), precision=rs.RSFD_FP64)
    with handle() as h:
        ref = rs.rsfd_lead_sigma_decimation(h.ptr, E, 2e-2, V[0], V[1])
    with handle() as h, _left(310):
        got = rs.rsfd_lead_sigma_decimation(h.ptr, E, 2e-2, V[0], V[1])
    assert got[2] == ref[2]
    assert _rel(got[0], ref[0]) <= 800 * 2.0 ** -46 and _rel(got[1], ref[1]) <= 800 * 2.0 ** -46


# FP64: five matrices of 64 MiB; tensor-core form: four; the digits of the smallest large product take 8 MiB
@pytest.mark.parametrize("kind,mib", [(FP64, 5 * 64 + 10), (TC, 4 * 64 + 10)])
def test_dyson_without_room_for_digits(rs, kind, mib):
    nb = 2048
    g = torch.Generator(device="cuda").manual_seed(3)
    G0 = torch.randn((1, nb, nb), dtype=torch.complex128, device="cuda", generator=g) * (0.3 / nb ** 0.5)
    S = torch.randn((1, nb // 2, nb // 2), dtype=torch.complex128, device="cuda", generator=g) * (1.0 / nb ** 0.5)
    S2, out = S.transpose(1, 2).contiguous(), []
    for low in (False, True):
        G = torch.zeros_like(G0)
        with rs.Handle((nb // 2, 1, 4), 0.5, 2, np.zeros(2 * nb), n_face=1, precision=rs.RSFD_FP64) as h:
            rs.rsfd_set_solve_options(h.ptr, dyson_kind=kind)
            with _left(mib) if low else contextlib.nullcontext():
                ref = rs.rsfd_dyson_boundary(h.ptr, G0, S, S2, G)
        assert (ref <= nb * 2.0 ** -50).all()
        out.append(G)
    assert not torch.equal(out[0], out[1])   # the plain forms round differently
    assert _rel(out[1], out[0]) <= nb * 2.0 ** -46
