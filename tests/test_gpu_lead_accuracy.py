"""Lead decimation of small cross-sections is as accurate as the same iteration with LAPACK's FP64 solves: the errors of both
against the closed form (V = 0), as geometric means over energy sets, differ by less than 30 % (other orders of
summation and elimination move single sets by more than that, a mean of 48 by 10 to 20 %)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.leads import _layer_blocks, sigma_bloch   # noqa: E402


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1502_00081_gb300.build_lib import build
    build()
    import paper_1502_00081_gb300 as m
    m.load_library()
    return m


def _lapack(H00, H01, Z):
    n = len(H00)
    one, eps_s, eps = np.eye(n), H00.astype(complex), H00.astype(complex)
    a, b = H01.astype(complex), H01.T.astype(complex)
    while max(np.abs(a).max(), np.abs(b).max()) >= 1e-15 * max(1.0, np.abs(H01).max()):
        Y = np.linalg.solve(Z * one - eps, np.hstack([a, b]))
        ga, gb = Y[:, :n], Y[:, n:]
        agb = a @ gb
        eps_s, eps, a, b = eps_s + agb, eps + agb + b @ ga, a @ ga, b @ gb
    return H01 @ np.linalg.solve(Z * one - eps_s, H01.T.astype(complex))


def test_small_leads_are_as_accurate_as_lapack(rs):
    rng, ratios = np.random.default_rng(1), []
    for nx in (8, 9):
        H00, H01 = _layer_blocks(nx, nx, 0.5, 2)
        for rep in range(24):
            eta, E = (1e-2, 2e-2, 5e-2)[rep % 3], np.linspace(0.3, 2.0, 8) + rng.uniform(0, 0.1)
            with rs.Handle((nx, nx, 4), 0.5, 2, np.zeros(4 * nx * nx), precision=rs.RSFD_FP64) as h:
                S = rs.rsfd_lead_sigma_decimation(h.ptr, E, eta)[1].cpu().numpy().transpose(0, 2, 1)
            ref = np.array([sigma_bloch(nx, nx, 0.5, 2, e + 1j * eta)[1] for e in E])
            lap = np.array([_lapack(H00, H01, e + 1j * eta) for e in E])
            ratios.append(np.linalg.norm(S - ref) / np.linalg.norm(lap - ref))
    assert np.exp(np.mean(np.log(ratios))) <= 1.3
