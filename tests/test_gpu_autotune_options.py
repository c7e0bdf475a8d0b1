"""rsfd_autotune sets the launch shape only: a handle served from the process-wide cache keeps its own other options, whatever
options the handle had that was timed."""

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


def _tuned(rs, p, call, **opts):
    with rs.Handle(p.grid, p.h, p.fd_order, p.V, n_face=p.n_face, precision=rs.RSFD_FP64) as h:
        rs.rsfd_set_solve_options(h.ptr, **opts)
        o, us = rs.rsfd_autotune(h.ptr, p.energies, p.eta, slots=6, iters=64)
        return o, us, call(h)


def test_cached_shape_leaves_the_other_options(rs):
    p = small_problem(grid=(22, 14, 17), h=0.5, fd_order=2, n_wells=3, n_energies=5, e_range=(0.5, 2.0), eta=5e-2, cols=4)
    ns = 22 * 14
    g = torch.Generator(device="cuda").manual_seed(1)
    G0 = torch.randn((2, 2 * ns, 2 * ns), dtype=torch.complex128, device="cuda", generator=g) * 0.01
    S = torch.randn((2, ns, ns), dtype=torch.complex128, device="cuda", generator=g) * 0.01

    def dyson(h):
        G = torch.zeros_like(G0)
        rs.rsfd_dyson_boundary(h.ptr, G0, S, S.clone(), G)
        return G.cpu().numpy()

    first = dict(dyson_cols=1, dyson_refine=3, dyson_kind=2, breakdown_tol=1e-20, use_graphs=-1, wait_cap=4000)
    o1, us1, left = _tuned(rs, p, dyson, **first)
    o2, us2, full = _tuned(rs, p, dyson)
    shape = ("pass_kind", "tile_y", "tile_x", "rows_per_thread", "z_chunk", "reg_budget", "slots")
    assert us1 == us2 and all(o1[k] == o2[k] for k in shape)          # the second came from the cache
    assert all(o1[k] == v for k, v in first.items())
    assert all(o2[k] == 0 for k in first)
    assert np.all(left[:, ns:] == 0)                                  # G[k][column][row]
    assert np.abs(full[:, ns:]).max() > 0 and np.allclose(full[:, :ns], left[:, :ns], rtol=1e-10, atol=1e-14)
    # another chunk length, or other recorded rows, is another measurement and keeps its own length
    o3, _, _ = _tuned(rs, p, lambda h: None, iters_per_sync=16)
    assert o3["iters_per_sync"] == 16 and o2["iters_per_sync"] == 32


def test_tuning_knows_the_untuned_pass(rs):
    """FP64 on a grid 37 wide: tiles cut to the grid are 9 % faster than the best tile of at most 32 columns, and they are what
    an untuned handle runs (the split pass without a height has the automatic pass's tiles and sums)."""
    p = small_problem(grid=(37, 26, 19), h=0.45, fd_order=4, n_wells=3, n_energies=8, e_range=(0.3, 2.0), eta=1e-1, cols=24)
    out = []
    with rs.Handle(p.grid, p.h, p.fd_order, p.V, n_face=p.n_face, precision=rs.RSFD_FP64) as h:
        picks = [rs.rsfd_autotune(h.ptr, p.energies, p.eta, slots=n, iters=64)[0] for n in (24, 23, 22)]   # three measurements
        assert any(o["pass_kind"] == rs.RSFD_PASS_SPLIT and o["tile_y"] == 0 for o in picks)
        for opts in (dict(), dict(pass_kind=rs.RSFD_PASS_SPLIT)):
            rs.rsfd_set_solve_options(h.ptr, **opts)
            G = torch.zeros((p.K, p.cols.size, h.nb), dtype=h.complex_dtype, device="cuda")
            rs.rsfd_shifted_cocg(h.ptr, p.cols, p.energies, p.eta, 1e-30, 60, G)
            out.append(G)
    assert torch.equal(out[0], out[1])
