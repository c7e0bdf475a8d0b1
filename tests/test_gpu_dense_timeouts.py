"""Expired bounded waits inside the sliced tensor-core products (solve option wait_cap = -1: no attempts), without a GPU fault:
every CTA of the product gives up as a whole, lets its copies and matrix instructions in flight end, gives its tensor memory
back and returns; the call reports RSFD_ERR_TIMEOUT.  The same handle then gives what a fresh one gives.  One tile per CTA
and several, FP64 and FP32 digits."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

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


def _inputs(nb, K):
    g = torch.Generator(device="cuda").manual_seed(nb)
    G0 = torch.randn((K, nb, nb), dtype=torch.complex128, device="cuda", generator=g) * (0.2 / nb ** 0.5)
    S = torch.randn((K, nb // 2, nb // 2), dtype=torch.complex128, device="cuda", generator=g) * (1.0 / nb ** 0.5)
    return G0, S, S.transpose(1, 2).contiguous()


def _expires(rs, h, call):
    rs.rsfd_set_solve_options(h.ptr, wait_cap=-1, **h.kind)
    with pytest.raises(rs.RsfdError) as e:
        call()
    assert e.value.status == rs.RSFD_ERR_TIMEOUT and "wait expired" in str(e.value)
    torch.cuda.synchronize()
    rs.rsfd_set_solve_options(h.ptr, **h.kind)


@pytest.mark.parametrize("kind", [FP64, TC])
@pytest.mark.parametrize("nb,K", [(258, 4), (1026, 4)])   # 4 x 129^3 is above the rule for slicing
def test_dyson_and_transmission(rs, nb, K, kind):
    G0, SL, SR = _inputs(nb, K)
    out = []
    for expire in (True, False):
        with rs.Handle((nb // 2, 1, 4), 0.5, 2, np.zeros(2 * nb), n_face=1, precision=rs.RSFD_FP64) as h:
            h.kind = dict(dyson_kind=kind)
            rs.rsfd_set_solve_options(h.ptr, **h.kind)
            G = torch.zeros_like(G0)
            if expire:
                _expires(rs, h, lambda: rs.rsfd_dyson_boundary(h.ptr, G0, SL, SR, G))
                _expires(rs, h, lambda: rs.rsfd_transmission(h.ptr, G0, SL, SR))
            rs.rsfd_dyson_boundary(h.ptr, G0, SL, SR, G)
            out.append((G.cpu().numpy(), rs.rsfd_transmission(h.ptr, G, SL, SR)))
    assert np.isfinite(out[0][0]).all()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_lead_decimation(rs):
    n, E = 8, np.linspace(0.3, 2.0, 8)
    out = []
    for expire in (True, False):
        with rs.Handle((n, n, 4), 0.5, 2, np.zeros(4 * n * n), n_face=1, precision=rs.RSFD_FP64) as h:
            h.kind = {}
            if expire:
                _expires(rs, h, lambda: rs.rsfd_lead_sigma_decimation(h.ptr, E, 2e-2, maxit=30))
            out.append(rs.rsfd_lead_sigma_decimation(h.ptr, E, 2e-2))
    for a, b in zip(out[0][:2], out[1][:2]):
        assert torch.isfinite(torch.view_as_real(a)).all() and torch.equal(a, b)
