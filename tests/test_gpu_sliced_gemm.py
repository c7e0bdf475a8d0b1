"""The FP64 products of the Dyson step and the transmission on the tensor cores (digit slices, 64-bit integer
sums), reached through rsfd_transmission (Eq. TF): T = Tr[Gamma_L G_RL^H Gamma_R G_RL] is one product with
a plain and one with a conjugate-transposed left operand, G_RL being a block of a larger matrix.

Tolerance: two FP64 products and a trace of ns x ns matrices err by at most about
4 ns 2^-53 |Gamma_L| |G_RL|^2 |Gamma_R| (Frobenius norms) in ordinary FP64 arithmetic; the slices must not
be worse."""

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


def _inputs(ns, K, scale):
    rng = np.random.Generator(np.random.PCG64(ns))
    def mat(n):
        return rng.normal(size=(K, n, n)) + 1j * rng.normal(size=(K, n, n))
    G, SL, SR = mat(2 * ns), mat(ns), mat(ns)
    # graded rows and columns: magnitudes over 2^scale
    g = 2.0 ** rng.integers(-scale, scale + 1, size=(K, 2 * ns, 1))
    return G * g * g.transpose(0, 2, 1), SL, SR


def _T(rs, ns, G, SL, SR):
    up = lambda M: torch.from_numpy(np.ascontiguousarray(M.transpose(0, 2, 1))).cuda()   # noqa: E731
    with rs.Handle((ns, 1, 4), 0.5, 2, np.zeros(ns * 4), n_face=1, precision=rs.RSFD_FP64) as h:
        return rs.rsfd_transmission(h.ptr, up(G), up(SL), up(SR))


# below and above the rule of 8e6 multiply-adds; rows around the 128-row tile, columns around the 32-column
# tile, k around the 16-deep step and the 128-deep chunk
@pytest.mark.parametrize("ns,K,scale", [(33, 40, 0), (96, 16, 0), (127, 5, 0), (128, 4, 20), (129, 4, 0), (161, 2, 8),
                                        (257, 1, 0), (300, 1, 30)])
def test_sliced_products_match_fp64(rs, ns, K, scale):
    G, SL, SR = _inputs(ns, K, scale)
    T = _T(rs, ns, G, SL, SR)
    for k in range(K):
        gl, gr = (1j * (S - S.conj().T) for S in (SL[k], SR[k]))
        A = G[k][ns:, :ns]
        ref = np.trace(gl @ A.conj().T @ gr @ A).real
        bound = 4 * ns * 2.0 ** -53 * np.linalg.norm(gl) * np.linalg.norm(A) ** 2 * np.linalg.norm(gr)
        assert abs(T[k] - ref) <= bound, (k, T[k] - ref, bound)


def test_non_finite_elements_stay_in_their_energy(rs):
    ns, K = 129, 6
    G, SL, SR = _inputs(ns, K, 0)
    clean = _T(rs, ns, G, SL, SR)
    G[1, ns + 5, 7] = np.nan
    G[3, ns + 1, 2] = np.inf
    T = _T(rs, ns, G, SL, SR)
    assert not np.isfinite(T[[1, 3]]).any()
    assert np.array_equal(T[[0, 2, 4, 5]], clean[[0, 2, 4, 5]])


def test_zero_matrices(rs):
    ns, K = 130, 4
    z = np.zeros((K, ns, ns), complex)
    assert (_T(rs, ns, np.zeros((K, 2 * ns, 2 * ns), complex), z, z) == 0).all()
