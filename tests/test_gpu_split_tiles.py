"""Tiles of the split pass cut to the grid, and the automatic pass.

With double-float vectors the automatic pass runs the split kernels with the sums in the stored pass's blocks, so its
result is the stored pass's bit for bit, at every width and height (rows of up to 8, 16 and 32 columns, a
remainder joined to the last 32-wide tile or not, odd heights, z-chunks, slot refill, tracked planes).  FP64 and
complex64 use tiles of their own; FP64 is compared with the stored pass within 1e-9, the mode's stated bound."""

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


def _solve(rs, p, prec, planes=(), **opts):
    with rs.Handle(p.grid, p.h, p.fd_order, p.V, n_face=p.n_face, proj=p.proj, precision=prec) as h:
        rs.rsfd_set_solve_options(h.ptr, **opts)
        rs.rsfd_set_tracked_planes(h.ptr, list(planes))
        nr = rs.rsfd_tracked_rows(h.ptr).size
        G = torch.zeros((p.K, p.cols.size, nr), dtype=h.complex_dtype, device="cuda")
        # 40 iterations, or fewer where the grid has so few points that the Krylov space is exhausted
        rs.rsfd_shifted_cocg(h.ptr, p.cols, p.energies, p.eta, 1e-30, 40, G)
        return G.cpu().numpy()


GRIDS = [((2, 3, 6), 2), ((8, 5, 40), 4), ((7, 9, 12), 4), ((16, 16, 48), 4), ((13, 21, 9), 2), ((31, 6, 10), 4),
         ((33, 18, 16), 4), ((37, 26, 19), 4), ((48, 24, 20), 4), ((60, 17, 11), 2), ((62, 9, 12), 4), ((72, 16, 13), 4),
         ((65, 8, 8), 4)]


@pytest.mark.parametrize("grid,order", GRIDS)
def test_automatic_double_float_pass_is_the_stored_pass(rs, grid, order):
    p = small_problem(grid=grid, h=0.45, fd_order=order, n_wells=3, n_energies=4, e_range=(0.3, 2.0), eta=5e-2, cols=5)
    planes = [z for z in (grid[2] // 2,) if p.n_face <= z < grid[2] - p.n_face]
    a = _solve(rs, p, rs.RSFD_DF64, planes, slots=3)
    b = _solve(rs, p, rs.RSFD_DF64, planes, slots=3, pass_kind=rs.RSFD_PASS_STORED)
    assert np.abs(b).max() > 0 and np.array_equal(a, b)


def test_automatic_pass_with_projectors(rs):
    p = small_problem(grid=(40, 18, 17), h=0.45, fd_order=4, n_wells=3, projectors=6, n_energies=4, e_range=(0.3, 2.0),
                      eta=5e-2, cols=5)
    a = _solve(rs, p, rs.RSFD_DF64)
    b = _solve(rs, p, rs.RSFD_DF64, pass_kind=rs.RSFD_PASS_STORED)
    assert np.array_equal(a, b)


@pytest.mark.parametrize("grid,order", GRIDS)
def test_automatic_fp64_pass(rs, grid, order):
    p = small_problem(grid=grid, h=0.45, fd_order=order, n_wells=3, n_energies=4, e_range=(0.3, 2.0), eta=5e-2, cols=5)
    a = _solve(rs, p, rs.RSFD_FP64, slots=3)
    b = _solve(rs, p, rs.RSFD_FP64, slots=3, pass_kind=rs.RSFD_PASS_STORED)
    assert np.linalg.norm(a - b) <= 1e-9 * np.linalg.norm(b)


@pytest.mark.parametrize("tile_y,z_chunk,kind", [(1, 0, 3), (7, 9, 3), (7, 0, 4), (16, 5, 4), (3, 17, 4)])
def test_given_tiles_of_the_split_passes(rs, tile_y, z_chunk, kind):
    """Odd heights and short z-chunks of the double-float split passes against FP64 (their stated bound, 1e-6)."""
    p = small_problem(grid=(38, 23, 18), h=0.45, fd_order=4, n_wells=3, n_energies=4, e_range=(0.3, 2.0), eta=5e-2,
                      cols=4)
    a = _solve(rs, p, rs.RSFD_DF64, slots=2, pass_kind=kind, tile_y=tile_y, z_chunk=z_chunk)
    b = _solve(rs, p, rs.RSFD_FP64, slots=2, pass_kind=rs.RSFD_PASS_STORED)
    assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)
