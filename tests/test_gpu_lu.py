"""The batched LU and triangular solves of the Dyson step (Eq. sec3-01a) at the sizes where their blocking
changes: panels of 16 columns, row tiles of 64, column tiles of 16, substitution blocks of 64 (FP64) and 128
(FP32), outer blocks of 128, one to eight CTAs per panel, two and four rows per thread, and the panel kept
in global memory.  M = I - G0 Sigma is built to need row exchanges: a cyclic shift of the rows of a well-conditioned
matrix, so the largest entry of every column is far from the diagonal."""

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


def _problem(nb, K, seed=5):
    """G0, Sigma_L, Sigma_R (ABI layout) with I - G0 Sigma = P (I + E), |E| about 0.3 (spectral), P a shift."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ns = nb // 2
    E = torch.randn((K, nb, nb), dtype=torch.complex128, device="cuda", generator=g) * (0.15 / nb ** 0.5)
    M = E
    M.diagonal(dim1=1, dim2=2).add_(1.0)
    M = torch.roll(M, max(1, nb // 3), dims=1)                       # [K, row, col]
    # Sigma = -i s I (retarded): G0 = (I - M) Sigma^{-1}
    s = 0.5
    G0 = -M
    G0.diagonal(dim1=1, dim2=2).add_(1.0)
    G0 *= 1j / s
    S = torch.zeros((K, ns, ns), dtype=torch.complex128, device="cuda")
    S.diagonal(dim1=1, dim2=2).fill_(-1j * s)
    return G0.transpose(1, 2).contiguous(), S, S.clone(), s


def _residual(G0, G, s, cols):
    """|| G0 - (I - G0 Sigma) G || / ||G0|| on some columns, Sigma = -i s I."""
    A = G0.transpose(1, 2)
    x, b = G.transpose(1, 2)[:, :, cols], A[:, :, cols]
    r = b - (x - A @ (-1j * s * x))
    return float(r.norm() / b.norm())


def _solve(rs, prec, kind, G0, SL, SR):
    nb = G0.shape[1]
    with rs.Handle((nb // 2, 1, 4), 0.5, 2, np.zeros(nb * 2), n_face=1, precision=prec) as h:
        rs.rsfd_set_solve_options(h.ptr, dyson_kind=kind)
        G = torch.empty_like(G0)
        ref = rs.rsfd_dyson_boundary(h.ptr, G0, SL, SR, G)
    return G, ref


# the condition number of I + E is below 2, so FP64 residuals of n-term sums stay below about n 2^-53 times a
# few; the FP32 factorisation with one FP64 refinement leaves (n 2^-24 x growth)^2, far below 1e-8
@pytest.mark.parametrize("kind", [FP64, TC])
@pytest.mark.parametrize("nb,K", [(2, 3), (14, 2), (16, 5), (18, 2), (62, 3), (66, 2), (126, 2), (128, 3), (130, 2),
                                  (144, 1), (254, 2), (258, 9), (386, 1), (514, 2), (1026, 2)])
def test_dyson_with_row_exchanges(rs, nb, K, kind):
    G0, SL, SR, s = _problem(nb, K)
    G, ref = _solve(rs, rs.RSFD_FP64, kind, G0, SL, SR)
    bound = max(nb, 8) * 2.0 ** -50
    assert _residual(G0, G, s, slice(0, nb)) <= bound
    assert (ref <= bound).all()


@pytest.mark.parametrize("kind,nb", [(FP64, 4104), (TC, 4104), (FP64, 8200), (TC, 8200), (TC, 16392)])
def test_tall_panels(rs, kind, nb):
    G0, SL, SR, s = _problem(nb, 1)
    G, _ = _solve(rs, rs.RSFD_FP64, kind, G0, SL, SR)
    assert _residual(G0, G, s, [0, 1, nb // 2, nb - 1]) <= nb * 2.0 ** -50


@pytest.mark.parametrize("kind", [FP64, TC])
def test_singular_energy_is_named(rs, kind):
    G0, SL, SR, s = _problem(130, 3)
    # a zero column of I - G0 Sigma at energy 1
    G0[1, 70, :] = 0.0
    G0[1, 70, 70] = 1j / s
    with pytest.raises(rs.RsfdError) as e:
        _solve(rs, rs.RSFD_FP64, kind, G0, SL, SR)
    assert e.value.status == rs.RSFD_ERR_BREAKDOWN and "energy 1" in str(e.value)


@pytest.mark.parametrize("nb,K", [(2, 7), (4, 40), (34, 3), (130, 4), (258, 9)])
def test_without_allocations(rs, nb, K):
    G0, SL, SR, s = _problem(nb, K)
    G = torch.empty_like(G0)
    ref = rs.rsfd_dyson_boundary_noalloc(G0, SL, SR, G)
    bound = max(nb, 8) * 2.0 ** -50
    assert _residual(G0, G, s, slice(0, nb)) <= bound and (ref <= bound).all()
