"""The automatic pass of complex64 handles: the split kernels with the stored pass's products and its sums in that pass's
blocks, so that its result is the stored pass's bit for bit (launches of at most one CTA per SM run the stored pass itself: the
numbers of columns below are above that where a grid has so many).  The recurrence amplifies a changed last bit of a dot product to
1e-5 of G0_bb (1e-3 of the rms in single elements), so any other bound would leave the choice of the pass visible."""

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


def _solve(rs, p, prec, planes=(), maxit=40, **opts):
    with rs.Handle(p.grid, p.h, p.fd_order, p.V, n_face=p.n_face, proj=p.proj, precision=prec) as h:
        rs.rsfd_set_solve_options(h.ptr, **opts)
        rs.rsfd_set_tracked_planes(h.ptr, list(planes))
        nr = rs.rsfd_tracked_rows(h.ptr).size
        G = torch.zeros((p.K, p.cols.size, nr), dtype=h.complex_dtype, device="cuda")
        _, info, _ = rs.rsfd_shifted_cocg(h.ptr, p.cols, p.energies, p.eta, 1e-30, maxit, G)
        return G.cpu().numpy(), info["iters"].copy()


# widths around the 4-point granularity of the potential's boxes and the 32-column blocks, a remainder joined to the
# last 32-wide tile (28 columns at most) or not, odd heights, one to several z-chunks
GRIDS = [((1, 4, 9), 2), ((2, 3, 6), 2), ((5, 7, 10), 2), ((8, 5, 40), 4), ((7, 9, 12), 4), ((16, 16, 48), 4), ((13, 28, 37), 4),
         ((13, 21, 9), 2), ((31, 6, 10), 4), ((33, 18, 16), 4), ((37, 26, 19), 4), ((48, 24, 20), 4), ((56, 12, 20), 4),
         ((60, 17, 11), 2), ((61, 9, 12), 4), ((72, 16, 13), 4), ((65, 8, 8), 4), ((90, 5, 34), 2)]


@pytest.mark.parametrize("grid,order", GRIDS)
def test_automatic_pass_is_the_stored_pass(rs, grid, order):
    p = small_problem(grid=grid, h=0.45, fd_order=order, n_wells=3, n_energies=4, e_range=(0.3, 2.0), eta=1e-1,
                      cols=min(170, 2 * grid[0] * grid[1]))
    planes = [z for z in (grid[2] // 2,) if p.n_face <= z < grid[2] - p.n_face]
    a, ia = _solve(rs, p, rs.RSFD_MIXED, planes, slots=160)
    b, ib = _solve(rs, p, rs.RSFD_MIXED, planes, slots=160, pass_kind=rs.RSFD_PASS_STORED)
    assert np.abs(b).max() > 0 and np.array_equal(a, b) and np.array_equal(ia, ib)


def test_automatic_pass_with_projectors(rs):
    p = small_problem(grid=(42, 18, 17), h=0.45, fd_order=4, n_wells=3, projectors=6, n_energies=4, e_range=(0.3, 2.0),
                      eta=1e-1, cols=40)
    a, _ = _solve(rs, p, rs.RSFD_MIXED)
    b, _ = _solve(rs, p, rs.RSFD_MIXED, pass_kind=rs.RSFD_PASS_STORED)
    assert np.array_equal(a, b)


@pytest.mark.parametrize("tile_y,z_chunk", [(1, 0), (7, 9), (16, 5), (3, 17)])
def test_given_tiles_of_the_split_pass(rs, tile_y, z_chunk):
    """Against FP64 within the bound that the other complex64 tests use."""
    p = small_problem(grid=(38, 23, 18), h=0.45, fd_order=4, n_wells=3, n_energies=4, e_range=(0.3, 2.0), eta=1e-1,
                      cols=4)
    a, _ = _solve(rs, p, rs.RSFD_MIXED, slots=2, pass_kind=rs.RSFD_PASS_SPLIT, tile_y=tile_y, z_chunk=z_chunk)
    b, _ = _solve(rs, p, rs.RSFD_FP64, slots=2, pass_kind=rs.RSFD_PASS_STORED)
    assert np.linalg.norm(a - b) <= 5e-5 * np.linalg.norm(b)
