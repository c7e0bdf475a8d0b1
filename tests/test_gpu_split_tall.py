"""Narrow, tall cross-sections through the automatic pass: the tiles stay within the TMA box's 256 rows and leave room for the
deepest prefetch.  Double-float and complex64 results are the stored pass's bit for bit, FP64 within 1e-9 of it."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from workloads import small_problem   # noqa: E402


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1502_00081_gb300.build_lib import build
    build()
    import paper_1502_00081_gb300 as m
    m.load_library()
    return m


def _solve(rs, p, prec, **opts):
    with rs.Handle(p.grid, p.h, p.fd_order, p.V, n_face=p.n_face, precision=prec) as h:
        rs.rsfd_set_solve_options(h.ptr, **opts)
        G = torch.zeros((p.K, p.cols.size, h.nb), dtype=h.complex_dtype, device="cuda")
        rs.rsfd_shifted_cocg(h.ptr, p.cols, p.energies, p.eta, 1e-30, 30, G)
        return G.cpu().numpy()


@pytest.mark.parametrize("grid,order", [((2, 256, 6), 4), ((1, 300, 5), 2), ((2, 127, 9), 4), ((1, 64, 8), 2), ((3, 401, 4), 4),
                                        ((4, 130, 7), 4), ((6, 253, 5), 2)])
def test_narrow_and_tall(rs, grid, order):
    p = small_problem(grid=grid, h=0.45, fd_order=order, n_wells=3, n_energies=4, e_range=(0.3, 2.0), eta=1e-1, cols=4)
    for prec in (rs.RSFD_FP64, rs.RSFD_DF64, rs.RSFD_MIXED):
        b = _solve(rs, p, prec, pass_kind=rs.RSFD_PASS_STORED)
        assert np.abs(b).max() > 0
        for opts in (dict(), dict(pass_kind=rs.RSFD_PASS_SPLIT, prefetch=7)):
            a = _solve(rs, p, prec, **opts)
            if prec == rs.RSFD_FP64:
                assert np.linalg.norm(a - b) <= 1e-9 * np.linalg.norm(b)
            elif not opts:
                assert np.array_equal(a, b)
