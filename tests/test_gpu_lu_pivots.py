"""Pivot search of the FP64 panels where the squared measures are denormal: a tiny element is a pivot, a zero is not."""

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


def _up(M):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(M, complex)[None].transpose(0, 2, 1))).cuda()


@pytest.mark.parametrize("alloc", [True, False])
@pytest.mark.parametrize("t", [1e-100, 1e-158, 1e-160])
def test_tiny_pivot_below_a_zero(rs, t, alloc):
    """I - G0 Sigma = [[0, 1], [t, 0]] with Sigma = 1: G = [[-1, 1 / t], [1, -1]]."""
    G0, S = _up([[1.0, -1.0], [-t, 1.0]]), _up([[1.0]])
    G = torch.zeros_like(G0)
    if alloc:
        with rs.Handle((1, 1, 4), 0.5, 2, np.zeros(4), n_face=1, precision=rs.RSFD_FP64) as h:
            rs.rsfd_dyson_boundary(h.ptr, G0, S, S.clone(), G)
    else:
        rs.rsfd_dyson_boundary_noalloc(G0, S, S.clone(), G)
    got = G.cpu().numpy()[0].T
    ref = np.array([[-1.0, 1.0 / t], [1.0, -1.0]])
    assert (np.abs(got - ref) <= 4e-16 * np.abs(ref)).all()


def test_zero_column_is_singular(rs):
    with rs.Handle((1, 1, 4), 0.5, 2, np.zeros(4), n_face=1, precision=rs.RSFD_FP64) as h:
        G0, S = _up([[1.0, -1.0], [0.0, 1.0]]), _up([[1.0]])
        with pytest.raises(rs.RsfdError) as e:
            rs.rsfd_dyson_boundary(h.ptr, G0, S, S.clone(), torch.zeros_like(G0))
        assert e.value.status == rs.RSFD_ERR_BREAKDOWN
