"""Dyson step, interior planes and transmission where the slabs hardly couple: wires with uniform leads at energies below the
first subband, against the closed form (an infinite perfect chain per transverse mode: G(a, b) = lam^|a-b| / (t (1/lam - lam))).
The block G_RL falls to 1e-25 of G_LL with the wire's length; every block is compared by itself, since a norm of the whole
matrix, or of the whole residual, does not see it.

Tolerance: every element of a block is a sum of nb products of like magnitude, solved for with one or two FP64 refinements of
a system whose condition number is of order 1, so an error of about nb 2^-53 times a few; nb 2^-48 is allowed (the reference
transforms modes to the grid with sums of the same kind).  T is quadratic in G_RL, and Gamma (eta 1e-2 of the self-energy)
loses two digits to cancellation: 1e-10."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

H = 0.5
HOP = -0.5 / H ** 2
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


def _modes(n):
    return np.linalg.eigh(np.diag(np.full(n, 1.0 / H ** 2)) + np.diag(np.full(n - 1, HOP), 1) + np.diag(np.full(n - 1, HOP), -1))


class Wire:
    """Closed forms on planes 1 .. nz: lam [K, mode], g0(a, b) of the isolated wire and g(a, b) with its leads."""

    def __init__(self, nx, ny, nz, E, eta=1e-2):
        (ex, ux), (ey, uy) = _modes(nx), _modes(ny)
        e = (ey[:, None] + ex[None, :]).ravel()
        self.U = np.einsum("ya,xb->yxab", uy, ux).reshape(nx * ny, nx * ny)
        q = (np.asarray(E)[:, None] + 1j * eta - e[None, :] - 1.0 / H ** 2).astype(np.clongdouble)
        s = np.sqrt(q * q - 4 * HOP * HOP)
        lam = (q + s) / (2 * HOP)
        self.lam = np.where(np.abs(lam) < 1, lam, (q - s) / (2 * HOP))
        self.nz = nz

    def g0(self, a, b):
        a, b = min(a, b), max(a, b)
        p = lambda m: 1 - self.lam ** (2 * m)   # noqa: E731
        return self.lam ** (b - a + 1) * p(a) * p(self.nz + 1 - b) / (p(1) * p(self.nz + 1)) / HOP

    def g(self, a, b):
        return self.lam ** abs(a - b) / (HOP * (1 / self.lam - self.lam))

    def dense(self, v):
        return (self.U[None] * v.astype(complex)[:, None, :]) @ self.U.T

    def blocks(self, f, planes):
        return [[self.dense(f(a, b)) for b in planes] for a in planes]


def _up(M):
    return torch.from_numpy(np.ascontiguousarray(M.transpose(0, 2, 1))).cuda()


def _check(G, ref, planes, bound):
    n = ref[0][0].shape[1]
    for i in range(len(planes)):
        for j in range(len(planes)):
            d, r = G[:, i * n:(i + 1) * n, j * n:(j + 1) * n] - ref[i][j], ref[i][j]
            err = np.linalg.norm(d, axis=(1, 2)) / np.linalg.norm(r, axis=(1, 2))
            assert (err <= bound).all(), (i, j, err.max(), np.linalg.norm(r[0]) / np.linalg.norm(ref[0][0][0]))


# lengths: G_RL / G_LL of about 1e-10, 1e-16 and 1e-25; nb and K on both sides of the rule for sliced products, slabs that
# are and are not whole substitution blocks (64 rows in FP64, 128 in FP32)
@pytest.mark.parametrize("kind", [FP64, TC])
@pytest.mark.parametrize("nx,ny,K", [(6, 6, 1), (6, 6, 24), (8, 8, 3), (8, 8, 16), (10, 9, 16), (13, 11, 1), (13, 11, 16), (16, 8, 16)])
@pytest.mark.parametrize("nz", [25, 40, 62])
def test_weakly_coupled_slabs(rs, nx, ny, K, nz, kind):
    w = Wire(nx, ny, nz, np.linspace(-1.0, -0.9, K))
    ns, nb, planes = nx * ny, 2 * nx * ny, (1, nz)
    G0, ref, S = np.block(w.blocks(w.g0, planes)), w.blocks(w.g, planes), w.dense(HOP * w.lam)
    with rs.Handle((nx, ny, 6), H, 2, np.zeros(6 * ns), n_face=1, precision=rs.RSFD_FP64) as h:
        rs.rsfd_set_solve_options(h.ptr, dyson_kind=kind)
        dS = _up(S)
        G = torch.empty((K, nb, nb), dtype=torch.complex128, device="cuda")
        rs.rsfd_dyson_boundary(h.ptr, _up(G0), dS, dS.clone(), G)
        T = rs.rsfd_transmission(h.ptr, G, dS, dS)
    _check(G.cpu().numpy().transpose(0, 2, 1), ref, planes, nb * 2.0 ** -48)
    gam = -2 * (HOP * w.lam).imag
    T_ref = (gam ** 2 * np.abs(w.g(1, nz)) ** 2).sum(1).astype(float)
    assert (np.abs(T - T_ref) <= 1e-10 * T_ref).all(), (T / T_ref)


@pytest.mark.parametrize("nx,ny,K", [(6, 6, 24), (9, 9, 8), (16, 8, 4)])
@pytest.mark.parametrize("nz", [25, 62])
def test_interior_planes_of_weakly_coupled_slabs(rs, nx, ny, K, nz):
    w = Wire(nx, ny, nz, np.linspace(-1.0, -0.9, K))
    n, zs = nx * ny, (nz // 4, nz // 2, (7 * nz) // 8)
    planes = (1, nz) + tuple(z + 1 for z in zs)
    G0, ref, S = np.block(w.blocks(w.g0, planes)), w.blocks(w.g, planes), w.dense(HOP * w.lam)
    with rs.Handle((nx, ny, nz), H, 2, np.zeros(nz * n), n_face=1, precision=rs.RSFD_FP64) as h:
        rs.rsfd_set_tracked_planes(h.ptr, list(zs))
        dS = _up(S)
        G = torch.empty((K, 5 * n, 5 * n), dtype=torch.complex128, device="cuda")
        rs.rsfd_dyson_tracked(h.ptr, _up(G0), dS, dS.clone(), G)
    _check(G.cpu().numpy().transpose(0, 2, 1), ref, planes, 5 * n * 2.0 ** -48)
